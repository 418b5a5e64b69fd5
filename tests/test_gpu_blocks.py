"""Steps run in blocks of up to 16: a march gives the same bits however it is cut into calls.

Every output is summed in an order that depends on its step alone, so marches cut at odd places (blocks
of 16, remainders, single steps), runs in place, through overlapping rows, through host buffers and
from a state saved in the middle of a block must agree bit for bit; the uncut march is compared with the
oracle in test_gpu_parity.py and test_gpu_tensor_cores.py.
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


def _march(plan, D, cuts):
    """T of the march over D cut into calls of the given lengths (repeated), from rest."""
    plan.reset()
    Dd = torch.from_numpy(D).cuda()
    Td = torch.zeros_like(Dd)
    torch.cuda.synchronize()
    n = k = 0
    while n < D.shape[0]:
        m = min(cuts[k % len(cuts)], D.shape[0] - n)
        if m == 1:
            plan.step(Dd[n], Td[n])
        else:
            plan.run(m, Dd[n:], Td[n:])
        n, k = n + m, k + 1
    plan.synchronize()
    return Td.cpu().numpy()


# leaves of 32, 13 (ragged, half a warp) and 3 (many lane groups); both near kernels, all storage types
@pytest.mark.parametrize("prec", [fdph.FP64, fdph.FP32, fdph.FP16])
@pytest.mark.parametrize("R,leaf,soe", [(1, 32, 16), (1, 13, 0), (1, 3, 16), (2, 32, 16), (4, 13, 16), (8, 32, 0)])
def test_cut_marches_give_the_same_bits(prec, R, leaf, soe):
    _need_gpu()
    N, M = 187, 830
    xy = inputs.kinked_fault(N) if R == 1 else inputs.curved_fault(N, inputs.seed_for(1, 0))
    plan = fdph.Plan(xy, 0.5, M, 1e-5, eta=0.5, eps_st=1e-4, leaf_size=leaf, soe_terms=soe, precision=prec, nrhs=R,
                     amp_window=1)
    steps = 150
    D = np.stack([inputs.gaussian_filtered_history(N, steps, 40 + r) for r in range(R)], 1)
    whole = _march(plan, D, [steps])
    assert np.isfinite(whole).all() and np.abs(whole).max() > 0
    for cuts in ([1], [16], [15, 1, 17], [7, 33, 2]):
        assert np.array_equal(_march(plan, D, cuts), whole), cuts
    # host buffers, and a state saved in the middle of a block (rings at another phase)
    plan.reset()
    out = plan.run_host(np.ascontiguousarray(D[:37]))
    buf = plan.save_state()
    tail = plan.run_host(np.ascontiguousarray(D[37:]))
    assert np.array_equal(np.concatenate([out, tail]), whole)
    plan.load_state(buf)
    assert np.array_equal(plan.run_host(np.ascontiguousarray(D[37:])), whole[37:])
    plan.close()


def test_rows_in_place_and_overlapping():
    """T over D's own rows; and T one row behind D, where step n's traction becomes the slip rate of
    step n + 1 (such a march is taken step by step)."""
    _need_gpu()
    N, M = 150, 64
    plan = fdph.Plan(inputs.kinked_fault(N), 0.5, M, 1e-5, eta=0.5, eps_st=1e-4, leaf_size=16)
    D = inputs.gaussian_filtered_history(N, M, 3)
    ref = _march(plan, D, [M])
    plan.reset()
    X = torch.from_numpy(D).cuda()
    torch.cuda.synchronize()
    plan.run(M, X, X)
    plan.synchronize()
    assert np.array_equal(X.cpu().numpy(), ref)
    fed = []
    for run in (True, False):
        plan.reset()
        X = torch.zeros((M + 1, N), dtype=torch.float64, device="cuda")
        X[0] = torch.from_numpy(D[5])
        torch.cuda.synchronize()
        if run:
            plan.run(M, X, X[1:])
        else:
            for n in range(M):
                plan.step(X[n], X[n + 1])
        plan.synchronize()
        fed.append(X.cpu().numpy())
    assert np.array_equal(fed[0], fed[1]) and np.abs(fed[0][10]).max() > 0


# eps_st = 0.05: windows shorter than a block (rupture steps then taken singly); leaf 3: far blocks that
# act within a block
@pytest.mark.parametrize("prec,leaf,eps_st,cfl", [(fdph.FP64, 32, 1e-4, 0.5), (fdph.FP32, 13, 1e-4, 0.25),
                                                  (fdph.FP16, 32, 1e-4, 0.5), (fdph.FP32, 16, 0.05, 0.5),
                                                  (fdph.FP64, 3, 1e-4, 0.5)])
def test_cut_ruptures_give_the_same_bits(prec, leaf, eps_st, cfl):
    _need_gpu()
    N, M = 203, 140
    xy = inputs.kinked_fault(N)
    tau0 = np.full(N, 0.45)
    tau0[N // 2 - 8:N // 2 + 8] = 0.61
    t0 = torch.from_numpy(tau0).cuda()
    torch.cuda.synchronize()
    outs = []
    for cuts in ([M], [1], [5, 30, 16, 1], [16]):
        plan = fdph.Plan(xy, cfl, M, 1e-5, eta=0.5, eps_st=eps_st, leaf_size=leaf, precision=prec)
        plan.rupture_init(t0, 1.0, 0.6, 0.3, 2.0, law=1)
        D = torch.zeros((M, N), dtype=torch.float64, device="cuda")
        T = torch.zeros_like(D)
        torch.cuda.synchronize()
        n = k = 0
        while n < M:
            m = min(cuts[k % len(cuts)], M - n)
            plan.rupture_run(m, D[n:], T[n:])
            n, k = n + m, k + 1
        slip = torch.zeros(N, dtype=torch.float64, device="cuda")
        plan.rupture_slip(slip)
        plan.synchronize()
        outs.append([x.cpu().numpy() for x in (D, T, slip)])
        plan.close()
    assert (outs[0][0] > 0).mean() > 0.05
    for o in outs[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(o, outs[0]))


@pytest.mark.parametrize("prec,eps_st,cfl", [(fdph.FP64, 0.05, 0.5), (fdph.FP32, 1e-3, 0.25), (fdph.FP64, 1e-3, 0.25)])
def test_short_windows_rupture_equals_predict_and_commit(prec, eps_st, cfl):
    """Leaves whose window is shorter than a block: their static terms act within the block.  Against the
    same law solved by the caller between predict and commit (FP64 to rounding, FP32 products to 1e-5)."""
    _need_gpu()
    N, M = 240, 100
    plan = fdph.Plan(inputs.kinked_fault(N), cfl, M, 1e-6, eta=0.5, eps_st=eps_st, leaf_size=16, precision=prec)
    tau0 = np.full(N, 0.45)
    tau0[N // 2 - 8:N // 2 + 8] = 0.61
    t0 = torch.from_numpy(tau0).cuda()
    plan.rupture_init(t0, 1.0, 0.6, 0.3, 2.0)
    D = torch.zeros((M, N), dtype=torch.float64, device="cuda")
    T = torch.zeros_like(D)
    torch.cuda.synchronize()
    plan.rupture_run(M, D, T)
    plan.synchronize()
    plan.reset()
    k0 = torch.from_numpy(plan.self_coefficients()).cuda()
    slip = torch.zeros(N, dtype=torch.float64, device="cuda")
    Du, Tu = torch.zeros_like(D), torch.zeros_like(T)
    for n in range(M):
        plan.predict(Tu[n])
        plan.synchronize()
        tau = t0 + Tu[n]
        strength = 0.6 - 0.3 * torch.clamp(slip / 2.0, max=1.0)
        v = torch.where(tau > strength, (tau - strength) / (-k0), torch.zeros_like(tau))
        Du[n] = v
        Tu[n] = tau + k0 * v
        slip += v * cfl
        torch.cuda.synchronize()
        plan.commit(Du[n])
    plan.synchronize()
    tol = 1e-10 if prec == fdph.FP64 else 1e-5
    assert (D > 0).double().mean().item() > 0.05
    assert ((D - Du).norm() / Du.norm()).item() < tol and ((T - Tu).norm() / Tu.norm()).item() < tol
