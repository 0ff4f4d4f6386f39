"""The single-kernel calls (dose, prices, the allocation-free dose) at the edges of
their tiles and limits, against the FP64 oracle."""
import numpy as np
import pytest

import oracle as O
from _helpers import U32, need_cuda, random_case, sum_abs_cols, sum_abs_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = need_cuda()
    from paper_1003_5402_gb300 import build
    build.build()
    return t


@pytest.mark.parametrize("threads", [64, 128])
def test_prices_with_either_default_block(torch, threads):
    """64 and 128 threads to a row of D^T, consecutive entries on consecutive
    threads: a thread adds ceil(n / threads) <= ceil(n / 64) products, then a warp
    tree of 5 levels, FP64 over the warps and one rounding."""
    from paper_1003_5402_gb300 import Plan
    case = random_case(71, 3001, rows=[3, 7], cols=[5, 9], mean_row=23.0)
    pi = np.random.default_rng(3).normal(size=case.n_voxels).astype(np.float32)
    with Plan(case, dt_threads=threads, dt_map="consecutive") as plan:
        w = torch.empty(case.n_beamlets, dtype=torch.float32, device="cuda")
        plan.k_beamlet_prices(torch.from_numpy(pi).cuda(), w)
        w = w.cpu().numpy().astype(np.float64)
    ref = O.beamlet_prices(O.csr64(case), pi.astype(np.float64))
    bound, n = sum_abs_cols(case, pi)
    assert np.all(np.abs(w - ref) <= (np.ceil(n / 64) + 7) * U32 * bound + U32 * np.abs(ref))


def test_dose_ticket_over_repeated_calls(torch):
    """The unit form's last block adds the objective: the ticket is back at 0 after
    every call, with and without a gradient, and equal calls give equal bits."""
    from paper_1003_5402_gb300 import Plan
    case = random_case(72, 2050, rows=[6, 4], cols=[8, 5], mean_row=19.0)
    rng = np.random.default_rng(4)
    xs = [torch.from_numpy(rng.uniform(0, 2, case.n_beamlets).astype(np.float32)).cuda() for _ in range(2)]
    D, vt = O.csr64(case), O.voxel_terms(case)
    got = [[], []]
    with Plan(case, dose_form="units") as plan:
        z = torch.empty(case.n_voxels, dtype=torch.float32, device="cuda")
        g = torch.empty_like(z)
        for r in range(6):
            got[r % 2].append(plan.k_dose(xs[r % 2], z, g if r < 4 else None))
    for i in range(2):
        assert len(set(got[i])) == 1
        F = O.objective(O.dose(D, xs[i].cpu().numpy().astype(np.float64)), vt)
        assert abs(got[i][0] - F) <= 1e-5 * abs(F)


@pytest.mark.parametrize("V,rows,cols,mean_row,weight", [
    (1, [2], [3], 3.0, 1.0), (31, [4], [5], 9.0, 1.0), (33, [4], [5], 9.0, 1.0), (1000, [16, 9], [16, 9], 33.0, 1.0),
    (515, [32, 31], [32, 31], 90.0, 1.0),      # units of more entries than a warp holds at a time
    (700, [96], [96], 40.0, 1.0),              # x in shared memory, the last size
    (700, [96, 1], [96, 1], 40.0, 1.0),        # x read from memory
    (700, [9], [9], 6.0, np.inf),              # inf * 0 is a NaN in every voxel of the structure
])
def test_noalloc_dose_edges(torch, V, rows, cols, mean_row, weight):
    from paper_1003_5402_gb300 import binding
    case = random_case(73 + V, V, rows=rows, cols=cols, mean_row=mean_row)
    N = case.n_beamlets
    x = np.random.default_rng(5).uniform(0, 2, N).astype(np.float32)
    terms = np.stack([case.under_w, case.under_t, case.over_w, case.over_t], axis=1).astype(np.float64)
    terms[-1, 2] = weight
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a, t)).cuda()
    z = torch.full((V,), float("nan"), dtype=torch.float32, device="cuda")
    g = torch.full_like(z, float("nan"))
    F = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
    binding.dose_objective_noalloc(dev(case.indptr, np.int32), dev(case.indices, np.int32), dev(case.data, np.float32),
                                   dev(x, np.float32), dev(case.voxel_struct, np.int32), terms, z, g, F)
    torch.cuda.synchronize()
    z, g, F = z.cpu().numpy(), g.cpu().numpy(), float(F.item())
    ref = O.dose(O.csr64(case), x.astype(np.float64))
    bound, n = sum_abs_rows(case, x)
    assert np.all(np.abs(z - ref) <= (n + 6) * U32 * bound + U32 * np.abs(ref))
    t, zd = terms[case.voxel_struct], z.astype(np.float64)
    under, over = np.maximum(0, t[:, 1] - zd), np.maximum(0, zd - t[:, 3])
    with np.errstate(invalid="ignore"):
        gref, Fref = 2 * (t[:, 2] * over - t[:, 0] * under), np.sum(t[:, 0] * under**2 + t[:, 2] * over**2)
    # FP64 from the FP32 dose, the gradient rounded once
    bad = ~np.isfinite(gref)
    assert np.array_equal(np.isnan(gref), np.isnan(g)) and np.all(g[bad & ~np.isnan(gref)] == np.inf)
    assert np.all(np.abs(g[~bad] - gref[~bad]) <= 2 * U32 * np.abs(gref[~bad]) + 1e-45)
    assert abs(F - Fref) <= 1e-11 * Fref if np.isfinite(Fref) else not np.isfinite(F)
