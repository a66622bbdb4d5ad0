"""Edges of the cell sort's runs, the paint's crowded bins and the L-BFGS passes."""
import numpy as np
import pytest
import torch

from gpu_util import context, rel_l2, to_dev, to_np
from oracle import pm as opm

pytestmark = pytest.mark.gpu


def _in_cells(keys, N, rng):
    """One particle per entry of keys, anywhere in that cell."""
    keys = np.asarray(keys)
    corner = np.stack([keys // (N * N), (keys // N) % N, keys % N]).astype(np.float64)
    return (corner + rng.uniform(0.02, 0.98, size=corner.shape)).astype(np.float32)


# particles in the leading runs. 512-cell runs (N^3 < 2^21) are sorted in registers up to
# 1536 particles and in perm beyond; 2048-cell runs in registers up to 3072, in shared
# memory up to 5632, in perm beyond. 18^3 and 162^3 end in a run of fewer cells.
@pytest.mark.parametrize("N,counts", [(16, [1536, 1537, 0, 1, 512]), (18, [1535, 2200, 3, 0, 1409]),
                                      (128, [3072, 3073, 0, 5632, 5633, 1, 2048, 20000]), (162, [5633, 3073, 1])])
def test_cell_sort_run_sizes(N, counts):
    rng = np.random.default_rng(N)
    RS = 2048 if N**3 >= 1 << 21 else 512
    keys = [RS * r + rng.integers(0, RS, size=n) for r, n in enumerate(counts)]
    last = (N**3 - 1) // RS * RS
    keys.append(rng.integers(last, N**3, size=300))
    keys = rng.permutation(np.concatenate(keys))
    x = _in_cells(keys, N, rng)
    ctx, _ = context(N=N, nsteps=1, lbfgs_m=1)
    got_keys, perm, start = ctx.cell_sort(to_dev(x))
    want_perm, want_start = opm.sort_by_cell(opm.cell_keys(x, N), N)
    assert np.array_equal(opm.cell_keys(x, N), keys)
    assert np.array_equal(to_np(got_keys).view(np.uint32), keys)
    assert np.array_equal(to_np(perm).view(np.uint32), want_perm)
    assert np.array_equal(to_np(start).view(np.uint32), want_start)


def test_empty_catalogue_on_a_mesh_of_long_runs():
    N = 128
    ctx, _ = context(N=N, nsteps=1, lbfgs_m=1)
    assert float(ctx.paint(torch.empty(3, 0, device="cuda")).abs().max()) == 0.0


# A bin of more than 24 particles is summed by its warp if at most 4 of the warp's 32 bins
# are so crowded, else by its lane, in the same order: the cells around the bins of a row
# do not change by a bit when crowded bins elsewhere in the row make the rule turn.
@pytest.mark.parametrize("masses", [False, True])
@pytest.mark.parametrize("counts", [(24, 25), (25, 32, 33, 200), (26, 64, 65, 511)])
def test_crowded_bins_are_summed_in_one_order(counts, masses):
    N = 32
    rng = np.random.default_rng(sum(counts))
    row = (5 * N + 7) * N  # bins z = 0, 2, 4, 6 of the row (5, 7)
    few = np.concatenate([np.full(n, row + 2 * i) for i, n in enumerate(counts)])
    more = np.concatenate([np.full(40, row + 14 + 2 * i) for i in range(5)])
    xf, xm = _in_cells(rng.permutation(few), N, rng), _in_cells(more, N, rng)
    x = np.concatenate([xf, xm], axis=1)
    m = rng.uniform(0.5, 2.0, x.shape[1]).astype(np.float32) if masses else None
    mf = None if m is None else to_dev(m[:xf.shape[1]])
    ctx, _ = context(N=N, nsteps=1, lbfgs_m=1)
    by_warp, by_lane = to_np(ctx.paint(to_dev(xf), mf)), to_np(ctx.paint(to_dev(x), None if m is None else to_dev(m)))
    assert np.array_equal(by_warp[:, :, :10], by_lane[:, :, :10])
    # a cell adds up to sum(counts) products rounded to 2^-24 of the partial sums
    want = opm.paint(x.astype(np.float64), N, m, f32_wrap=True)
    assert rel_l2(by_lane, want) <= (sum(counts) + 8) * 2.0**-24


# Vectors of odd length put every second pair on an 8-byte boundary (no 16-byte loads).
# Tolerance: float64 sums over k <= 5 well-conditioned pairs, as for even lengths.
@pytest.mark.parametrize("n,k,shift", [(3, 1, 0), (1001, 5, 0), (4097, 2, 1), (4096, 5, 1), (16384, 5, 0)])
def test_lbfgs_direction_of_odd_and_shifted_vectors(n, k, shift):
    from oracle import lbfgs as olb
    ctx, _ = context(N=32, nsteps=1)
    rng = np.random.default_rng(n + k)
    S = [rng.standard_normal(n) for _ in range(k)]
    Y = [s + 0.3 * rng.standard_normal(n) for s in S]
    g = rng.standard_normal(n)
    gbuf = torch.zeros(n + 1, device="cuda", dtype=torch.float64)
    gbuf[shift:shift + n] = torch.from_numpy(g)
    d = ctx.lbfgs_direction(gbuf[shift:shift + n], torch.tensor(np.stack(S), device="cuda"),
                            torch.tensor(np.stack(Y), device="cuda"))
    assert rel_l2(to_np(d), olb.two_loop(g, S, Y)) <= 1e-12
