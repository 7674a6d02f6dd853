"""Dedispersion by channel groups at the sizes where its tables can go wrong:
channel counts that leave groups of 1 to 3, one DM tile and a row of the next,
DM steps from "all trials alike" to mostly ungrouped, output tiles of one sample
and of one past a tile, more groups than one set of 16-bit partial sums, samples
past the end.  8-bit sums equal the oracle's; FP32 sums stay within the
summation bound (n_chan - 1) 2^-24 sum |in| (any order of the additions).
"""
import numpy as np
import pytest

import oracle as O
import synthetic as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# n_chan, n_t, n_out, df, dm_lo, dm_step, n_dm
CASES = [
    (7, 1024, 1, 8.0, 0.0, 0.05, 33),
    (258, 4096, 513, 1.0, 30.0, 0.1, 65),
    (259, 4096, 4096, 1.0, 0.0, 0.3, 31),       # n_out = n_t: zeros past the end
    (300, 8192, 4000, 0.85, 200.0, 0.0, 40),    # every trial alike
    (128, 8192, 5121, 2.0, 5.0, 0.9, 34),       # groups of 1, 2 and 4
    (1030, 2048, 1100, 0.25, 1.0, 0.25, 3),     # more than 64 groups, few trials
]


@pytest.fixture(scope="module")
def capi():
    import paper_2211_13517_gb300 as pkg
    pkg.build()
    from paper_2211_13517_gb300 import capi as c
    c.lib()
    return c


@pytest.mark.parametrize("n_chan,n_t,n_out,df,dm_lo,dm_step,n_dm", CASES)
@pytest.mark.parametrize("bits", [8, 32])
def test_grouped_sums(capi, bits, n_chan, n_t, n_out, df, dm_lo, dm_step, n_dm):
    delays = O.dm_delays(n_chan, 1670.0, df, 64e-6, dm_lo, dm_step, n_dm)
    plan = capi.DedispPlan(n_chan, n_t, 1670.0, df, 64e-6, dm_lo, dm_step, n_dm, n_out)
    fb = S.filterbank_u8(n_chan, n_t, 3) if bits == 8 else S.filterbank_noise(n_chan, n_t, 3)
    if bits == 8:
        fb[n_chan // 2] = 255   # the largest partial sums
    guard = torch.full((n_dm * n_out + 64,), -7.0, device="cuda")
    out = plan.dedisperse(torch.from_numpy(fb).cuda(), out=guard[:n_dm * n_out].view(n_dm, n_out))
    torch.cuda.synchronize()
    assert torch.all(guard[n_dm * n_out:] == -7.0)
    got = out.cpu().numpy().astype(np.float64)
    ref = O.dedisperse(fb.astype(np.float64), delays, n_out)
    if bits == 8:
        assert np.array_equal(got, ref)
    else:
        bound = O.dedisperse(np.abs(fb.astype(np.float64)), delays, n_out) * (n_chan - 1) * 2.0 ** -24
        assert np.all(np.abs(got - ref) <= bound + 1e-6)
    plan.close()


@pytest.mark.parametrize("off", [0, 1, 3])   # the filterbank's first sample, in elements past 16 bytes
@pytest.mark.parametrize("n_t", [2048, 2049, 2050, 2051])
def test_rows_on_any_4_byte_boundary(capi, n_t, off):
    """FP32 filterbanks whose rows start on any multiple of 4 bytes, with the
    trials' windows partly and wholly past the end of their rows."""
    n_chan, n_dm = 64, 40
    args = (1670.0, 4.0, 64e-6, 20.0, 0.2)
    delays = O.dm_delays(n_chan, *args, n_dm)
    plan = capi.DedispPlan(n_chan, n_t, *args, n_dm, n_t)
    assert plan.info.workspace_bytes > 4 * n_chan * n_dm   # summed by groups
    fb = S.filterbank_noise(n_chan, n_t, n_t + off)
    # the samples around the filterbank must not be summed
    buf = torch.full((n_chan * n_t + 8,), 1e6, device="cuda")
    view = buf[off:off + n_chan * n_t].view(n_chan, n_t)
    view.copy_(torch.from_numpy(fb))
    got = plan.dedisperse(view).cpu().numpy().astype(np.float64)
    ref = O.dedisperse(fb.astype(np.float64), delays, n_t)
    bound = O.dedisperse(np.abs(fb.astype(np.float64)), delays, n_t) * (n_chan - 1) * 2.0 ** -24
    assert np.all(np.abs(got - ref) <= bound + 1e-6)
    plan.close()
