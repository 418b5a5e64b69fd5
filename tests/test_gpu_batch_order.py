"""A batch call is ordered with the streams of all its plans."""
import numpy as np
import pytest

from paper_1903_02118_gb300 import fdph, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("rupture", [False, True])
def test_all_buffers_prepared_and_read_on_the_first_plans_stream(rupture):
    """The first plan is the smallest and done first; its stream fills the inputs of all plans late (behind
    a long kernel) and copies all outputs right after the call."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_02118_gb300 import build
    build.build()
    steps, sizes = 64, (64, 900, 400)
    plans = [fdph.Plan(inputs.kinked_fault(N), 0.5, 512, 1e-5, eta=0.5, eps_st=1e-4, precision=fdph.FP32) for N in sizes]
    src = [torch.from_numpy(inputs.gaussian_filtered_history(N, steps, 7)).cuda() for N in sizes]
    taus = []
    for N in sizes:
        tau0 = torch.full((N,), 0.45, dtype=torch.float64, device="cuda")
        tau0[N // 2 - 8:N // 2 + 8] = 0.63
        taus.append(tau0)
    Ds = [torch.zeros_like(d) for d in src]
    Ts = [torch.zeros_like(d) for d in src]
    torch.cuda.synchronize()
    first = torch.cuda.ExternalStream(plans[0].stream)

    def start():
        for p, t in zip(plans, taus):
            p.reset()
            if rupture:
                p.rupture_init(t, 1.0, 0.6, 0.3, 2.0)
    start()
    for p, s, D, T in zip(plans, src, Ds, Ts):   # alone
        if rupture:
            p.rupture_run(steps, D, T)
        else:
            p.run(steps, s, T)
        p.synchronize()
    ref = [(D if rupture else s).clone() for D, s in zip(Ds, src)], [T.clone() for T in Ts]
    for x in Ds + Ts:
        x.zero_()
    start()
    batch = fdph.Batch(plans)
    torch.cuda.synchronize()
    with torch.cuda.stream(first):
        torch.cuda._sleep(40_000_000)
        for D, T, s in zip(Ds, Ts, src):
            D.copy_(s)
            T.fill_(7.0)
    (batch.rupture_run if rupture else batch.run)(steps, Ds, Ts)
    with torch.cuda.stream(first):
        out = [D.clone() for D in Ds], [T.clone() for T in Ts]
    first.synchronize()
    for got, want in zip(out[0] + out[1], ref[0] + ref[1]):
        assert np.array_equal(got.cpu().numpy(), want.cpu().numpy())
    batch.close()
    for p in plans:
        p.close()
