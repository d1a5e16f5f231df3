"""The curve -> grid map's tiles: widths 4 to 32, chosen by how much of a tile
lies outside the grid.

Tolerances as in test_gpu_parity.py: FP64 1e-12, FP32 + refinement 1e-5, both
of max |u|."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_11041_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _problem(nx, ny, seed=5):
    rng = np.random.default_rng(seed)
    one = np.ones((ny, nx))
    return W.Problem(nx, ny, 3e-3, 0.8, 0.8 * one, 0.6 * one, W.random_field(rng, nx, ny), W.make_mask("square", nx, ny),
                     y1=(ny - 1) / (nx - 1))


# more nodes than the one-launch iteration takes: the separate map kernel
SHAPES = [(5, 33000), (9, 18000), (17, 9600), (33, 5000), (48, 3400), (129, 1300), (33000, 5), (5000, 33), (450, 371)]


@pytest.mark.parametrize("nx,ny", SHAPES)
@pytest.mark.parametrize("prec", [0, 1])
def test_thin_grids_match_oracle(nx, ny, prec):
    from paper_2411_11041_gb300 import Solver
    p = _problem(nx, ny)
    s = Solver(p, tol=0.0, max_iter=3, prec=prec)
    u, it, st, _ = s.solve_stationary(want_iter=True)
    ref, refit, k, rel, _ = O.Oracle(p).solve_stationary(tol=0.0, max_iter=3)
    tol = 1e-12 if prec == 0 else 1e-5
    assert st["iters"] == k == 3
    assert np.abs(u.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()
    assert np.abs(it.cpu().numpy() - refit).max() <= tol * np.abs(refit).max()
    assert abs(st["rel_update"] - rel) <= (1e-9 if prec == 0 else 1e-3) * rel + 1e-13


def test_batch_of_thin_grids_matches_single_solves():
    import torch
    from paper_2411_11041_gb300 import Batch, Solver
    ps = [_problem(nx, ny, seed=k) for k, (nx, ny) in enumerate([(5, 900), (33, 700), (129, 60), (900, 5), (64, 64)])]
    hs = [Solver(p, tol=0.0, max_iter=4) for p in ps]
    ref = [h.solve_stationary()[0].clone() for h in hs]
    outs, stats, _ = Batch(hs).solve()
    for u, r, st in zip(outs, ref, stats):
        assert st["iters"] == 4 and torch.equal(u, r)


def test_thin_grids_cost_no_more_than_wide_ones():
    """Maps of 5 x 60000 nodes against those of 60000 x 5, the same work: below
    2.5 times their time (tiles of 32 x 8 for both: 4.7)."""
    from paper_2411_11041_gb300 import Solver

    def maps(nx, ny):
        s = Solver(_problem(nx, ny))
        return min(t[2] + t[5] for t in (s.time_kernels(20) for _ in range(3)))

    tall, wide = maps(5, 60000), maps(60000, 5)
    assert tall < 2.5 * wide, (tall, wide)


@pytest.mark.parametrize("count,nx,ny", [(2, 64, 64), (6, 200, 150), (8, 257, 257)])  # 1, 2 and 4 tiles a block
@pytest.mark.parametrize("prec", [0, 1])
def test_batches_of_every_block_size_match_single_solves(count, nx, ny, prec):
    import torch
    from paper_2411_11041_gb300 import Batch, Solver
    hs = [Solver(_problem(nx, ny, seed=k), tol=0.0, max_iter=5, prec=prec) for k in range(count)]
    one = [h.solve_stationary() for h in hs]
    ref = [(r[0].clone(), r[2]["rel_update"]) for r in one]
    outs, stats, _ = Batch(hs).solve()
    for u, (r, rel), st in zip(outs, ref, stats):
        assert st["iters"] == 5 and torch.equal(u, r)
        # the same squares summed in another order: n - 1 additions each rounding by 2^-53 at most
        assert abs(st["rel_update"] - rel) <= nx * ny * 2.0 ** -53 * rel
