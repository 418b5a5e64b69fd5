"""The allocation-free plain step at the edges of its row split: one receiver, ragged receiver tiles, windows
of one step, ring wrap-around, fewer rows than the GPU has warps, against the FP64 sum in torch."""
import pytest

from paper_1903_02118_gb300 import fdph

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,W,hist_len,step", [(1, 1, 1, 0), (1, 300, 300, 299), (31, 7, 9, 40), (33, 64, 64, 63), (100, 3, 5, 1),
                                               (257, 65, 70, 131), (500, 2, 2, 7)])
def test_plain_step_equals_the_sum(n, W, hist_len, step):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_02118_gb300 import build
    build.build()
    gen = torch.Generator(device="cuda").manual_seed(n * 1000 + W)
    K = torch.randn((W, n, n), dtype=torch.float64, device="cuda", generator=gen)
    D = torch.randn((hist_len, n), dtype=torch.float64, device="cuda", generator=gen)
    T = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
    kmax = min(step + 1, W)
    rows = torch.tensor([(step - k) % hist_len for k in range(kmax)], device="cuda")
    ref = torch.einsum("kji,kj->i", K[:kmax], D[rows])
    scale = torch.einsum("kji,kj->i", K[:kmax].abs(), D[rows].abs())
    for _ in range(2):
        fdph.plain_step_noalloc(K, n, W, D, hist_len, step, T)
        torch.cuda.synchronize()
        # each sum of kmax n products, rounded at most once per product on either side
        assert bool(((T - ref).abs() <= 2.0 * kmax * n * 2.0 ** -53 * scale).all())
