"""Tractions that only quiet elements of a leaf have reached.

One leaf of 32 elements: the first four slip at 1, the last twelve q times as fast, q down to 1e-12, and the
receivers at the far end are watched until the waves of the loud ones arrive.  What they see is bounded by
the rounding of its own terms, whatever the loud ones do:

    |dT_i,n| <= u sum_k,j |K_ijk| |D_j,n-k|

with u = 2^-11 + 2^-20 for FP16 windows (rounding of the stored coefficients; FP32 products and sums), 2^-20 for
FP32, and for FP64 1e-11 (2^-46 for 12 x 46 terms, and the closed form of the kernel on the host and the device).
"""
import numpy as np
import pytest

from oracle import kernel as kn
from paper_1903_02118_gb300 import fdph, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _check(prec, u, q):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_02118_gb300 import build
    build.build()
    N, steps = 32, 46
    xy = inputs.straight_fault(N)
    rng = np.random.default_rng(2)
    D = np.zeros((steps, N))
    D[:, :4] = rng.uniform(0.5, 1.0, (steps, 4))
    D[:, 20:] = q * rng.uniform(0.5, 1.0, (steps, 12))
    K = kn.discrete_kernel(kn.element_table(xy), 0.5, steps, 1.0, 1.0)
    far = np.arange(29, 32)                       # 25 elements and more from the loud ones: 49 steps at CFL 1/2
    assert not np.any(K[:, far][:, :, :4])
    T0, B = (np.array([np.einsum("kij,kj->i", f(K[:n + 1, far]), f(D[n::-1][:n + 1])) for n in range(steps)])
             for f in (np.asarray, np.abs))
    plan = fdph.Plan(xy, 0.5, steps, 0.0, eta=0.0, eps_st=0.0, precision=prec)
    for cut in (steps, 1):
        plan.reset()
        Dd = torch.from_numpy(D).cuda()
        T = torch.empty_like(Dd)
        torch.cuda.synchronize()
        for n in range(0, steps, cut):
            plan.run(cut, Dd[n:], T[n:])
        plan.synchronize()
        err = np.abs(T.cpu().numpy()[:, far] - T0)
        assert np.all(err <= u * B), float((err / B).max())
    plan.close()


@pytest.mark.parametrize("q", [1e-4, 1e-8, 1e-12])
@pytest.mark.parametrize("prec,u", [(fdph.FP64, 1e-11), (fdph.FP32, 2.0 ** -20), (fdph.FP16, 2.0 ** -11 + 2.0 ** -20)])
def test_quiet_sources(prec, u, q):
    _check(prec, u, q)
