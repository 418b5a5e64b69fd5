"""What admission counts: the plan's statistics cover its device allocations, and the estimate covers the plan."""
import pytest

from paper_1903_02118_gb300 import fdph, inputs, serving

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", [fdph.FP32, fdph.FP16, fdph.FP64])
@pytest.mark.parametrize("N,cfl,soe", [(512, 0.5, 16), (1500, 0.25, 16), (1500, 0.5, 0)])
def test_estimate_covers_the_plan_and_its_statistics_the_device(N, cfl, soe, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_02118_gb300 import build
    build.build()
    xy = inputs.curved_fault(N, inputs.seed_for(3, inputs.GEOMETRY))
    M = int(round(N / cfl))
    kw = dict(eta=0.5, eps_st=1e-4, leaf_size=32, soe_terms=soe, precision=prec, amp_window=1, aca_min=4096)
    warm = fdph.Plan(xy, cfl, M, 1e-4, **kw)          # (the context's own allocations)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    plan = fdph.Plan(xy, cfl, M, 1e-4, **kw)
    used = free - torch.cuda.mem_get_info()[0]
    st = plan.stats()
    counted = st["arena_bytes"] + st["state_bytes"]
    # (the driver hands out pieces of 2 MB, small allocations share one)
    assert counted >= 0.85 * used, (counted, used)
    assert serving.footprint_model(xy, cfl, M, soe_terms=soe, precision=prec) >= counted
    plan.close()
    warm.close()
