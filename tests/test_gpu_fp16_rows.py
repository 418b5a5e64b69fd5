"""FP16 windows on the tensor cores: slip rates of any size, one right-hand side included.

The slip rates go in as FP16 parts under a power-of-two scale per step and leaf, so a march scaled by 1e-30 or
1e30 must stay as close to the oracle as an unscaled one.  Bound (the one of test_gpu_tensor_cores.py; it
scales with the slip rates):

    |dT_i,n| <= 2^-11 sum_window |K_ijk| |D_j,n-k| + 2^-20 sum |Kc_ijk| |D_j,n-k| + 5e-6 max |T|

against the oracle's compressed operator (FP64).  A second test compares the FP32 near field with its tail
slices in one item per leaf (many leaves) and in two (few) with the FP64 plan: FP32 products and sums of at
most 2^8 terms per item, 1e-5 of the largest traction.
"""
import numpy as np
import pytest

from oracle import dense
from oracle import fdph as ofd
from oracle import kernel as kn
from paper_1903_02118_gb300 import fdph, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_02118_gb300 import build
    build.build()


def _march(plan, D):
    Dd = torch.from_numpy(np.ascontiguousarray(D)).cuda()
    Td = torch.empty_like(Dd)
    torch.cuda.synchronize()
    plan.run(D.shape[0], Dd, Td)
    plan.synchronize()
    return Td.cpu().numpy()


@pytest.mark.parametrize("R", [1, 2, 8])
@pytest.mark.parametrize("geom,N,leaf", [("curved", 192, 32), ("kinked", 181, 13)])
def test_fp16_rows_of_any_scale(geom, N, leaf, R):
    _need_gpu()
    M, steps, eps = 800, 300, 1e-5
    xy = inputs.curved_fault(N, inputs.seed_for(1, 0)) if geom == "curved" else inputs.kinked_fault(N)
    kw = dict(eta=0.5, eps_st=1e-4, soe_terms=16, amp_window=1)
    el = kn.element_table(xy)
    oplan = ofd.build_plan(el, ofd.Params(leaf=leaf, eps=eps, M=M, **kw))
    Kc = ofd.operator_rows(el, oplan, np.arange(N))
    Kw = np.zeros_like(Kc)
    for d in oplan["near"]:
        I, J, W = d["I"], d["J"], d["W"]
        Kw[:W][:, I[:, None], J[None, :]] = np.abs(d["K"][:W])
    plan = fdph.Plan(xy, 0.5, M, eps, leaf_size=leaf, precision=fdph.FP16, nrhs=R, **kw)
    D0 = inputs.gaussian_filtered_history(N, steps, 7)
    T0 = dense.march_rows_fft(Kc[:steps], D0)
    B = (2.0 ** -11 * dense.march_rows_fft(Kw[:steps], np.abs(D0)) + 2.0 ** -20 * dense.march_rows_fft(np.abs(Kc[:steps]), np.abs(D0))
         + 5e-6 * np.abs(T0).max())
    scale = [1e-30, 1.0, 1e30, 3e-20, 1e-5, 7e15, 2e-33, 40.0]
    for base in range(0, 3 if R == 1 else 1):
        D = np.stack([D0 * scale[(base + r) % len(scale)] for r in range(R)], 1)
        plan.reset()
        T = _march(plan, D if R > 1 else D[:, 0]).reshape(steps, R, N)
        for r in range(R):
            err = np.abs(T[:, r] / scale[(base + r) % len(scale)] - T0)
            assert np.all(err <= B), (base, r, float((err / B).max()))
    plan.close()


@pytest.mark.parametrize("leaf", [32, 3])     # 3: more than 152 x 4 leaves
def test_fp32_tail_items_agree_with_fp64(leaf):
    _need_gpu()
    N, M, steps = 640, 1000, 160
    xy = inputs.curved_fault(N, inputs.seed_for(1, 0))
    D = inputs.gaussian_filtered_history(N, steps, 11)
    out = []
    for prec in (fdph.FP64, fdph.FP32):
        plan = fdph.Plan(xy, 0.5, M, 1e-5, eta=0.5, eps_st=1e-4, leaf_size=leaf, soe_terms=16, amp_window=1, precision=prec)
        assert (plan.stats()["n_near"] >= 4 * 152) == (leaf == 3)
        out.append(_march(plan, D))
        plan.close()
    assert np.abs(out[1] - out[0]).max() <= 1e-5 * np.abs(out[0]).max()
