"""The device build's layouts (padded D, its beam segments, D by beams, D^T) at the
edges of its tiles.  D, x, pi and the masks are small integers, so every FP32 sum is
exact and the products through each layout must equal the oracle's."""
import numpy as np
import pytest

import oracle as O
from _helpers import need_cuda, random_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = need_cuda()
    from paper_1003_5402_gb300 import build
    build.build()
    return t


@pytest.mark.parametrize("V,rows,cols,mean_row", [
    (1, [1], [1], 1.0), (31, [2], [3], 2.0), (33, [4, 1, 5], [3, 1, 7], 6.0),
    (256, [4, 6], [5, 5], 1.5),                         # many empty rows, one window of the placement
    (257, [4, 6], [5, 5], 20.0), (515, [9, 8], [9, 8], 60.0),
    (1030, [1] * 300, [2] * 300, 12.0),                 # more beams than shared memory keeps offsets of
    (300, [120, 120], [30, 30], 900.0),                  # 7200 beamlets: two tiles of the placement
    (77824, [4], [6], 2.0), (77825, [4], [6], 2.0),     # 16 rows to each of the dose's warps, and units of 32 from there
    (550000, [270], [30], 1.0),                         # chunks of more rows than one window
])
def test_layouts_hold_every_entry(torch, V, rows, cols, mean_row):
    from paper_1003_5402_gb300 import Plan
    case = random_case(500 + V, V, rows=rows, cols=cols, mean_row=mean_row)
    rng = np.random.default_rng(V)
    case.data = rng.integers(1, 4, len(case.data)).astype(np.float32)
    N = case.n_beamlets
    x = rng.integers(0, 3, N).astype(np.float32)
    pi = rng.integers(-2, 3, V).astype(np.float32)
    D = O.csr64(case)
    off = np.concatenate([[0], np.cumsum(case.rows.astype(np.int64) * case.cols)])
    with Plan(case) as plan:
        z, g = (torch.empty(V, dtype=torch.float32, device="cuda") for _ in range(2))
        plan.k_dose(torch.from_numpy(x).cuda(), z, g)
        assert np.array_equal(z.cpu().numpy(), O.dose(D, x.astype(np.float64)))
        w = torch.empty(N, dtype=torch.float32, device="cuda")
        plan.k_beamlet_prices(torch.from_numpy(pi).cuda(), w)
        assert np.array_equal(w.cpu().numpy(), O.beamlet_prices(D, pi.astype(np.float64)))
        for b in {0, case.n_beams // 2, case.n_beams - 1}:
            R, Cb = int(case.rows[b]), int(case.cols[b])
            lv = np.sort(rng.integers(0, Cb + 1, (R, 2)), axis=1).astype(np.int32)
            lv[0] = (0, Cb)
            m = np.zeros(N)
            for r in range(R):
                m[off[b] + r * Cb + lv[r, 0]: off[b] + r * Cb + lv[r, 1]] = 1.0
            plan.k_aperture_column(b, lv, z)
            assert np.array_equal(z.cpu().numpy(), O.dose(D, m))


@pytest.mark.parametrize("row", [0, 31, 32, 63, 64, 99])
@pytest.mark.parametrize("what", ["order", "equal", "column", "nan", "across"])
def test_faults_in_any_row_of_a_warp(torch, row, what):
    """A fault in the first, a middle or the last row of a warp's 32 is named; a row
    that starts below the end of the one before ("across") is none."""
    from paper_1003_5402_gb300 import DaoError, Plan
    V, N = 100, 24
    case = random_case(91, V, rows=[4], cols=[6], mean_row=5.0)
    ip = np.arange(V + 1, dtype=np.int64) * 3
    ix = np.tile(np.array([2, 5, 11], np.int32), V)
    d = np.ones(3 * V, np.float32)
    if what == "order":
        ix[3 * row + 1: 3 * row + 3] = (11, 5)
    elif what == "equal":
        ix[3 * row + 1] = 2
    elif what == "column":
        ix[3 * row + 2] = N
    elif what == "nan":
        d[3 * row] = np.nan
    else:
        ix[3 * row: 3 * row + 3] = (21, 22, 23)
    case.indptr, case.indices, case.data = ip.astype(case.indptr.dtype), ix, d
    if what == "across":
        with Plan(case):
            return
    with pytest.raises(DaoError) as e:
        Plan(case)
    assert {"order": f"in row {row}", "equal": f"in row {row}", "column": f"entry {3 * row + 2}",
            "nan": f"entry {3 * row}"}[what] in str(e.value)
