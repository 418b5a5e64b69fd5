"""The near field's FP32 sums lose no more than sums of one slice at a time.

Slip-rate pulses on the plain operator of N = 300 elements (no approximation), where a sum over the lags of a few
sources is much larger than one over the sources of a lag.  FP32 against FP64 storage: 2.48e-7 (relative, L2) with
every slice of a work item summed over its 32 sources in four FP32 chains, up to 16 slices in FP32 and the
rest in FP64; 1.5e-7 of it is the rounding of coefficients and slip rates.
"""
import numpy as np
import pytest

from paper_1903_02118_gb300 import fdph, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_02118_gb300 import build
    build.build()


def _pulses(steps, n, seed):
    rng = np.random.default_rng(seed)
    s, t = np.arange(n), np.arange(steps) + 0.5
    D = np.zeros((steps, n))
    for _ in range(4):
        D += rng.uniform(0.25, 1.0) * np.exp(-(s[None] - rng.uniform(0, n)) ** 2 / 512
                                             - (t[:, None] - rng.uniform(0, steps)) ** 2 / 128)
    return D


def _march(D, precision, **kw):
    steps, nrhs, n = D.shape
    plan = fdph.Plan(inputs.straight_fault(n), 0.5, steps, 1e-4, eta=0.0, eps_st=0.0, precision=precision, nrhs=nrhs, **kw)
    Dd = torch.from_numpy(np.ascontiguousarray(D)).cuda()
    T = torch.empty_like(Dd)
    torch.cuda.synchronize()
    plan.run(steps, Dd, T)
    plan.synchronize()
    plan.close()
    return T.cpu().numpy()


@pytest.mark.parametrize("R", [1, 2])
def test_fp32_sums(R):
    _need_gpu()
    D = np.stack([_pulses(200, 300, 5 + r) for r in range(R)], 1)
    T64, T32 = _march(D, fdph.FP64), _march(D, fdph.FP32)
    assert np.linalg.norm(T32[:, 0] - T64[:, 0]) <= 2.48e-7 * np.linalg.norm(T64[:, 0])


@pytest.mark.parametrize("R", [2, 4])
def test_sums_behind_the_tensor_cores(R):
    """FP16 windows of several right-hand sides against exact sums of the stored coefficients, white noise: the
    MMAs' own sums are 9e-8 off, 16 additions in two levels of up to 8 add 2^-24 sqrt(8) / 2 to that (together
    1.25e-7); one sum over all slices of a work item was 1.35e-7 off."""
    _need_gpu()
    from oracle import kernel as kn
    n, steps = 300, 200
    D = np.random.default_rng(0).standard_normal((steps, 4, n)).astype(np.float32).astype(np.float64)
    K = kn.discrete_kernel(kn.element_table(inputs.straight_fault(n)), 0.5, steps, 1.0, 1.0)
    K = torch.from_numpy((K * 2.0 ** 14).astype(np.float16).astype(np.float64) / 2.0 ** 14).cuda()   # (largest 1 / 2)
    Dd = torch.from_numpy(D).cuda()
    E = torch.zeros_like(Dd)
    for k in range(steps):
        E[k:] += torch.einsum("ij,trj->tri", K[k], Dd[:steps - k])
    T = np.concatenate([_march(D[:, r:r + R], fdph.FP16) for r in range(0, 4, R)], 1)
    E = E.cpu().numpy()
    assert np.linalg.norm(T - E) <= 1.25e-7 * np.linalg.norm(E)
