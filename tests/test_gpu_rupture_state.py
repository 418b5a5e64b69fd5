"""What a rupture takes from its plan's state: the friction law last given."""
import numpy as np
import pytest

from paper_1903_02118_gb300 import fdph, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LAWS = [(1.0, 0.6, 0.3, 6.4, 0), (1.1, 0.55, 0.2, 2.0, 1)]   # sigma_n, mu_s, mu_d, Dc, law


def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_02118_gb300 import build
    build.build()


def _tau0(N):
    tau0 = np.full(N, 0.45)
    tau0[N // 2 - 8:N // 2 + 8] = 0.63
    return torch.from_numpy(tau0).cuda()


def _plan(N, prec=fdph.FP32, **kw):
    args = dict(eta=0.5, eps_st=1e-4, leaf_size=16, precision=prec)
    args.update(kw)
    return fdph.Plan(inputs.kinked_fault(N), 0.5, 256, 1e-5, **args)


@pytest.mark.parametrize("batch", [False, True])
def test_the_friction_law_is_the_one_last_given(batch):
    """Two laws in turn on the same plans and buffers, over whole blocks and a remainder (captured and
    direct steps): each run is that of fresh plans under its law."""
    _need_gpu()
    steps, sizes = 37, (181, 130)
    plans = [_plan(N) for N in sizes]
    taus = [_tau0(N) for N in sizes]
    Ds = [torch.zeros((steps, N), dtype=torch.float64, device="cuda") for N in sizes]
    Ts = [torch.zeros_like(D) for D in Ds]
    torch.cuda.synchronize()
    group = fdph.Batch(plans) if batch else None

    def run(ps, law, batch_of):
        for p, t in zip(ps, taus):
            p.reset()
            p.rupture_init(t, *law)
        if batch_of:
            batch_of.rupture_run(steps, Ds, Ts)
            batch_of.synchronize()
        else:
            for p, D, T in zip(ps, Ds, Ts):
                p.rupture_run(steps, D, T)
                p.synchronize()
        return [(D.cpu().numpy(), T.cpu().numpy()) for D, T in zip(Ds, Ts)]

    results = []
    for k in (0, 1):
        got = run(plans, LAWS[k], group)
        fresh = [_plan(N) for N in sizes]
        ref = run(fresh, LAWS[k], None)
        for p in fresh:
            p.close()
        for (D, T), (Dr, Tr) in zip(got, ref):
            assert np.array_equal(D, Dr) and np.array_equal(T, Tr), k
            assert D.max() > 0
        results.append(got)
    assert not np.array_equal(results[0][0][0], results[1][0][0])
    if group:
        group.close()
    for p in plans:
        p.close()


# Domain-S thresholds at which no window is longer than a few steps (0.5: none is kept at all)
@pytest.mark.parametrize("prec", [fdph.FP64, fdph.FP32, fdph.FP16])
@pytest.mark.parametrize("eps_st", [0.02, 0.05, 0.5])
def test_short_windows(eps_st, prec):
    """Rupture blocks of an operator whose windows are shorter than a block: the same bits step by step, and
    from a state saved in the middle of a block; FP64 against predict / commit with the same law."""
    _need_gpu()
    N, M = 150, 90
    law = (1.0, 0.6, 0.3, 2.0, 0)
    tau0 = _tau0(N)

    def plan():
        p = _plan(N, prec, eps_st=eps_st)
        assert p.stats()["max_window"] < 16
        assert eps_st < 0.5 or p.stats()["max_window"] == 0
        p.rupture_init(tau0, *law)
        return p

    def march(p, cuts, first=0):
        D = torch.zeros((M, N), dtype=torch.float64, device="cuda")
        T = torch.zeros_like(D)
        torch.cuda.synchronize()
        n = first
        for m in cuts:
            p.rupture_run(m, D[n:], T[n:])
            n += m
        p.synchronize()
        return D.cpu().numpy(), T.cpu().numpy()

    p = plan()
    D, T = march(p, [M])
    assert (D > 0).mean() > 0.05 and np.isfinite(T).all()
    q = plan()
    D1, T1 = march(q, [1] * M)
    assert np.array_equal(D, D1) and np.array_equal(T, T1)
    q.close()
    for at in (21, 47):
        q = plan()
        march(q, [at])
        state = q.save_state()
        q.close()
        q = plan()
        q.load_state(state)
        D2, T2 = march(q, [M - at], at)
        assert np.array_equal(D[at:], D2[at:]) and np.array_equal(T[at:], T2[at:]), at
        q.close()
    if prec == fdph.FP64:
        q = plan()
        k0 = q.self_coefficients()
        X = torch.zeros(N, dtype=torch.float64, device="cuda")
        slip = np.zeros(N)
        sigma_n, mu_s, mu_d, Dc, _ = law
        for n in range(M):
            q.predict(X)
            q.synchronize()
            tau = tau0.cpu().numpy() + X.cpu().numpy()
            strength = sigma_n * (mu_s - (mu_s - mu_d) * np.minimum(slip / Dc, 1.0))
            d = np.where(tau > strength, (tau - strength) / -k0, 0.0)
            assert np.abs(d - D[n]).max() < 1e-9, n
            q.commit(torch.from_numpy(d).cuda())
            q.synchronize()
            slip += d * 0.5
        q.close()
    p.close()
