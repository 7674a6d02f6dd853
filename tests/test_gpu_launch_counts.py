"""The launch counts of fdas_profile against the kernels that the CUDA profiler
records for the same search: by bounds (4 kernels of the harmonic sum where the
correlation writes the pooled plane itself, else 5, statistics included) and plain
(2), one series and three.
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HARMONIC = ("finalize_stats", "pool_kernel", "harmonic_")


@pytest.mark.parametrize("series", [1, 3])
@pytest.mark.parametrize("prec,corr,interbin,sigma,harmonic", [
    (0, 1, False, 6.0, 5),   # overlap-save plane, pooled by a kernel of its own
    (0, 1, False, 4.0, 2),
    (1, 2, False, 6.0, 4),   # pooled by the tensor-core correlation
    (1, 2, False, 4.0, 2),
    (1, 2, True, 6.0, 4),
])
def test_counts_are_the_launches(series, prec, corr, interbin, sigma, harmonic):
    import paper_2211_13517_gb300 as pkg
    pkg.build()
    from paper_2211_13517_gb300 import capi
    from torch.profiler import ProfilerActivity, profile
    plan = capi.Plan(1 << 15, 64e-6, 24.0, 1.0, 2048, 8, precision=prec, correlator=corr,
                     interbin=interbin, threshold_sigma=sigma)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    xs = [torch.randn(1 << 15, generator=g, device="cuda") for _ in range(series)]
    plan.search(xs)
    with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]):
        plan.search(xs)   # (a process's first records may lack the kernels)
    plan.profile(False)   # resets the counts
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as prof:
        plan.search(xs)
        torch.cuda.synchronize()
    counts = plan.profile()
    plan.close()
    # (the checked build's guard checks are not the search's)
    names = [e.name for e in prof.events()
             if e.device_type == torch.autograd.DeviceType.CUDA and "fdas::" in e.name
             and "canary" not in e.name]
    if not names:
        pytest.skip("the profiler records no kernels here")
    of_sum = [n for n in names if any(k in n for k in HARMONIC)]
    assert len(of_sum) == harmonic * series == counts["harmonic"][0]
    assert len(names) == sum(counts[k][0] for k in capi.PROFILE_GROUPS)
