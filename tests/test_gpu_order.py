"""Ordering and conversion of the crossings in one kernel (up to 8192 records) at
its edges: none, one, one more than a CTA's or the eager copy's share, the most it
takes, and the first count that the sorting kernels take over.  The records are
those of the sorting kernels for the same cells, bit for bit.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [0, 1, 255, 257, 2048, 2049, 8191, 8192, 8193])
@pytest.mark.parametrize("capacity", [1 << 14, 2000])
def test_records_of_a_few_cells_are_those_of_many(n, capacity):
    import paper_2211_13517_gb300 as pkg
    pkg.build()
    from paper_2211_13517_gb300 import capi
    plan = capi.Plan(1 << 14, 64e-6, 8.0, 1.0, 2048, 1, max_candidates=1 << 16)
    rng = np.random.RandomState(n)
    n_z, cols = plan.info.n_z, plan.info.plane_cols
    cells = rng.permutation(n_z * cols)[:20000]
    power = rng.uniform(30.0, 400.0, cells.size).astype(np.float32)
    power[::3] = 55.5   # equal powers
    stats = torch.tensor([1.0, 1.0], dtype=torch.float64, device="cuda")

    def records(count, capacity):
        plane = np.zeros(n_z * cols, dtype=np.float32)
        plane[cells[:count]] = power[:count]
        t = torch.from_numpy(plane.reshape(n_z, cols)).cuda()
        return plan.threshold(t, stats, trial_id=7, capacity=capacity)

    st, many, nf = records(cells.size, 1 << 16)   # by the sorting kernels
    assert st == capi.FDAS_OK and nf == cells.size
    flat = many["iz"].astype(np.int64) * cols + many["ir"]
    assert np.array_equal(flat, np.sort(cells))
    want = many[np.isin(flat, cells[:n])]
    assert len(want) == n
    st, got, nf = records(n, capacity)
    assert nf == n
    assert st == (capi.FDAS_OK if n <= capacity else capi.FDAS_ERR_CAND_OVERFLOW)
    assert got.tobytes() == want[:capacity].tobytes()
    plan.close()
