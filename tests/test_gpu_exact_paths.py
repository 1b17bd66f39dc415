"""Paths whose results other tests compare only with one another or within wide bounds: that the one-launch
Arnoldi cycle really is one launch where the step kernels are compared with it, the FP64 fit against a
host solution in FP64, and the weights within the error of their sums."""

import numpy as np
import pytest

from gpu_util import need_gpu
from test_gpu_tile_edges import _level, _walk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("nx,ny", [(40, 40), (257, 255), (261, 259), (1030, 1021)])
def test_arnoldi_tiles_match_a_cycle_that_ran_in_one_launch(nx, ny):
    """Row tiles of 256 rows, of 512, and beyond what shared memory keeps (4096): the iterates of the captured step
    and of the one-launch cycle, bit for bit, and the latter with fewer launches.  Seven steps do not converge."""
    import torch

    import paper_1004_1451_gb300 as bamg

    A = _walk(nx, ny)
    xs, launches = [], []
    for persistent in (0, 1):
        s = bamg.Solver(*A, r=10, levels=20, grid=(nx, ny), precision="mixed", max_it=7, mle_restart=0, device_loop=0,
                        persistent=persistent)
        x = torch.full((nx * ny,), float("nan"), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        before = bamg.launch_count()
        with pytest.raises(bamg.BamgError) as e:
            s.solve(1e-15, out=x)
        launches.append(bamg.launch_count() - before)
        assert e.value.code == -5 and e.value.stats["iterations"] == 7  # not converged
        xs.append(x)
        s.close()
    assert launches[1] < launches[0] / 2, launches
    assert bool(torch.isfinite(xs[0]).all()) and torch.equal(xs[0], xs[1])


@pytest.mark.parametrize("kind,n", [("grid", 9001), ("ring", 2001), ("hubs", 1500)])
@pytest.mark.parametrize("ncols,c", [(4, 1), (8, 2), (12, 2), (16, 3), (21, 2), (30, 2), (9, 4), (32, 4)])
def test_fp64_weights_solve_the_least_squares_problem(kind, n, ncols, c):
    """Every fine row's weights against a solution on the host in FP64 of the ridge problem over the row's own
    coarse points.  The ridge (1e-4 of the mean diagonal) keeps the condition number below 4 / 1e-4, and an FP64
    elimination of order 4 loses at most a few hundred roundings of that: 1e-9 of the largest weight."""
    import torch

    import paper_1004_1451_gb300 as bamg

    B, cf, cidx, X, w = _level(kind, n, ncols, ncols + ncols % 2, "fp64", 0, seed=n + ncols)
    pcol, pval, pcnt = (t.cpu().numpy() for t in bamg.interp_ls(B, cf, cidx, X, ncols, w, z=2, mmax=16, c=c, ridge=1e-4))
    Xh, wh = X[:, :ncols].cpu().numpy(), w[:ncols].cpu().numpy()
    fine = np.flatnonzero(cf.cpu().numpy() == 0)
    at = np.flatnonzero(cf.cpu().numpy())  # the fine-level index of every coarse point
    seen = 0
    for m in range(1, c + 1):
        rows = fine[pcnt[fine] == m]
        if rows.size == 0:
            continue
        S = Xh[at[pcol[rows, :m]]]  # rows x m x ncols
        G = np.einsum("iak,k,ibk->iab", S, wh, S)
        G += (1e-4 * np.trace(G, axis1=1, axis2=2) / m)[:, None, None] * np.eye(m)
        b = np.einsum("iak,k,ik->ia", S, wh, Xh[rows])
        want = np.linalg.solve(G, b[..., None])[..., 0]
        err = np.abs(pval[rows, :m] - want).max(1)
        assert (err <= 1e-9 * np.maximum(np.abs(want).max(1), 1e-3)).all()
        seen += rows.size
    assert seen > 0.9 * fine.size


@pytest.mark.parametrize("nx,ny,ncols", [(2, 1, 1), (17, 19, 31), (300, 250, 10), (1100, 600, 5)])
def test_weights_within_the_error_of_their_sums(nx, ny, ncols):
    """The weights 1 / ||B x||^2 over their largest, in FP64: a row of B x has at most five products (10 units of its
    sum of magnitudes), the sums of squares at most n + 64 additions of positive terms."""
    import torch

    import paper_1004_1451_gb300 as bamg

    ptr, col, val = _walk(nx, ny)
    n = nx * ny
    i = torch.arange(n, device="cuda")
    rows = torch.cat([torch.repeat_interleave(i, (ptr[1:] - ptr[:-1]).long()), i])
    cols, vals = torch.cat([col.long(), i]), torch.cat([-val, torch.ones(n, dtype=torch.float64, device="cuda")])
    order = torch.argsort(rows * n + cols)
    unit = 2.0 ** -53
    B = ((ptr + torch.arange(n + 1, device="cuda")).int(), cols[order].int(), vals[order].contiguous())
    X = 1.0 + torch.rand(n, ncols + ncols % 2, dtype=torch.float64, device="cuda",
                         generator=torch.Generator(device="cuda").manual_seed(n))
    count = (B[0][1:] - B[0][:-1]).long()
    x, b = X[:, :ncols].clone(), B[2]
    bx = torch.stack([torch.segment_reduce(b * x[:, c].contiguous()[B[1].long()], "sum", lengths=count) for c in range(ncols)], 1)
    mag = torch.stack([torch.segment_reduce(b.abs() * x[:, c].contiguous()[B[1].long()], "sum", lengths=count)
                       for c in range(ncols)], 1)
    xx, s = x.square().sum(0), bx.square().sum(0)
    want = xx / s
    # relative error of sum (B x)^2: 2 |bx| 10 u mag summed over the rows, and its square
    e = (2 * (bx.abs() * 10 * unit * mag).sum(0) + ((10 * unit * mag) ** 2).sum(0)) / s + 2 * (n + 64) * unit + 4 * unit
    w = bamg.tv_weights(B, X, ncols)
    top = int(want.argmax())
    err = (w - want / want[top]).abs() / (want / want[top])
    assert bool((err <= (e + e[top]) * 1.01).all())
