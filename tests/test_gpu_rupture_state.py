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
