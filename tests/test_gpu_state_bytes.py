"""Saved states: the same bytes come back from a plan that restored them, whatever the rings' phase."""
import numpy as np
import pytest

from paper_1903_02118_gb300 import fdph, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("kw", [dict(soe_terms=16), dict(soe_terms=0, nrhs=2), dict(far_mode=1), dict(eps_q=1e-3, leaf_size=13),
                                dict(eta=0.0, eps_st=0.0)])
def test_saved_bytes_survive_a_restore(kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_02118_gb300 import build
    build.build()
    N, M = 220, 900
    args = dict(dict(eta=0.5, eps_st=1e-4, precision=fdph.FP32), **kw)
    a, b = (fdph.Plan(inputs.kinked_fault(N), 0.5, M, 1e-5, **args) for _ in range(2))
    R = args.get("nrhs", 1)
    D = np.stack([inputs.gaussian_filtered_history(N, 400, 3 + r) for r in range(R)], 1)
    Dd = torch.from_numpy(D).cuda()
    T, U = torch.empty_like(Dd), torch.empty_like(Dd)
    torch.cuda.synchronize()
    n = 0
    for steps in (0, 1, 22, 300):
        a.run(steps, Dd[n:], T[n:])
        n += steps
        state = a.save_state()
        b.load_state(state)
        assert np.array_equal(b.save_state(), state), n
        # the newest row of the slip-rate ring stands where the state says: slot n - 1 modulo the rows saved
        if n:
            body = state[8:].view(np.float64)
            perm = fdph.tree_export(inputs.kinked_fault(N), 0.5, eta=args["eta"], leaf_size=args.get("leaf_size", 32))["perm"]
            row = D[n - 1, 0][perm]
            hits = [r for r in range(0, min(body.size // N, M + 1)) if np.array_equal(body[r * N:(r + 1) * N], row)]
            assert hits, n
        b.run(20, Dd[n:], U[n:])
        b.synchronize()
    a.run(20, Dd[n:], T[n:])
    a.synchronize()
    assert np.array_equal(T[n:n + 20].cpu().numpy(), U[n:n + 20].cpu().numpy())
    a.close()
    b.close()
