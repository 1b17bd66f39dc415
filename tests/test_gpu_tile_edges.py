"""Kernels at the sizes where their tiling can go wrong: tile edges, remainders, the smallest
and the largest launch shapes, and the alignments their wide loads distinguish."""

import numpy as np
import pytest

from gpu_util import need_gpu
from oracle import learned as ol

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def _network(rows, seed=3):
    """A model with random parameters, its FP32 parameters as FP64 arrays, and features."""
    import torch

    import paper_1004_1451_gb300 as bamg

    rng = np.random.default_rng(seed)
    p = ol.init_params(seed)
    for k in ("b1", "b2", "b3"):
        p[k] = rng.standard_normal(p[k].shape) * 0.05
    flat = np.concatenate([p[k].ravel() for k in ("W1", "b1", "W2", "b2", "W3", "b3")]).astype(np.float32)
    m = bamg.Model(0)
    m.set(flat)
    p32 = {k: v.astype(np.float32).astype(np.float64) for k, v in p.items()}
    feat = rng.standard_normal((rows, 112)).astype(np.float32) * 0.5
    feat[:, 0:96:6] = np.arange(16)[None, :] < rng.integers(1, 17, rows)[:, None]
    return torch, m, p32, feat


@pytest.mark.parametrize("rows", [1, 15, 16, 17, 33, 16 * 152 * 12 - 1, 16 * 152 * 12 + 17])
def test_forward_at_tile_edges(rows):
    """Every row equals the row on its own, bit for bit (a row's arithmetic does not depend on its
    place), also from storage that is only 8-byte aligned; the first rows agree with the oracle, whose
    sums are exact: a difference is a bf16 rounding that fell the other way (2^-8 of an activation)."""
    base = min(rows, 40)
    torch, m, p, f = _network(base)
    idx = np.arange(rows) % base
    Fd = torch.tensor(f, device="cuda")[torch.tensor(idx, device="cuda")].contiguous()
    y = m.forward(Fd)
    alone = torch.cat([m.forward(Fd[k:k + 1].contiguous()) for k in range(base)])
    assert torch.equal(y, alone[torch.tensor(idx, device="cuda")])
    shifted = torch.empty(rows * 112 + 2, dtype=torch.float32, device="cuda")[2:].view(rows, 112)
    shifted.copy_(Fd)
    assert shifted.data_ptr() % 16 == 8
    assert torch.equal(m.forward(shifted), y)
    y_o, _ = ol.forward(p, f.astype(np.float64), use_bf16=True)
    err = np.abs(alone.cpu().numpy() - y_o)
    scale = max(1.0, np.abs(y_o).max())
    assert err.max() <= 1e-2 * scale and err.mean() <= 1e-4 * scale


@pytest.mark.parametrize("rows", [1, 16, 17, 127, 129, 16 * 152 + 3, 16 * 152 * 8 + 5])
def test_gradients_at_tile_edges(rows):
    """Loss and gradients against the oracle with the same roundings.  A bf16 rounding that falls the
    other way moves an entry by at most 2^-8 of itself, so each gradient by at most 2^-8 of its norm;
    the targets lie at an odd 4-byte address."""
    torch, m, p, f = _network(rows, seed=rows)
    T = np.random.default_rng(1).standard_normal((rows, 16)).astype(np.float32) * 0.3
    Td = torch.empty(rows * 16 + 1, dtype=torch.float32, device="cuda")[1:].view(rows, 16)
    Td.copy_(torch.tensor(T))
    g, loss = m.gradients(torch.tensor(f, device="cuda"), Td)
    f64 = f.astype(np.float64)
    y, cache = ol.forward(p, f64, use_bf16=True)
    mask = ol.slot_mask(f64)
    g_o = ol.backward(p, cache, y, T.astype(np.float64), mask, bf16_grads=True)
    assert loss == pytest.approx(ol.loss(y, T, mask), rel=1e-3)
    at = 0
    for k in ("W1", "b1", "W2", "b2", "W3", "b3"):
        part = g[at:at + g_o[k].size].reshape(g_o[k].shape)
        at += g_o[k].size
        assert np.linalg.norm(part - g_o[k]) <= 2.0 ** -8 * max(np.linalg.norm(g_o[k]), 1e-30), k


def _walk(nx, ny):
    """A grid walk's CSR arrays on the GPU (uniform 1/degree), without the host's sort."""
    import torch

    off = torch.tensor([-nx, -1, 1, nx], device="cuda")
    i = torch.arange(nx * ny, device="cuda")
    x, y = i % nx, i // nx
    ok = torch.stack([y > 0, x > 0, x < nx - 1, y < ny - 1], 1)
    deg = ok.sum(1)
    col = (i[:, None] + off)[ok]
    ptr = torch.zeros(nx * ny + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = deg.cumsum(0)
    return ptr.int(), col.int(), 1.0 / deg[col].double()


@pytest.mark.parametrize("nx,ny", [(40, 40), (257, 255), (261, 259), (1030, 1021)])
def test_arnoldi_tiles_match_persistent_cycle(nx, ny):
    """The step kernels against the one-launch cycle, which adds in the same order with other
    thread counts: row tiles of 256, 512 and beyond what shared memory keeps (4096 rows), ragged
    last tiles, odd and even column counts.  Same iterates bit for bit."""
    import torch

    import paper_1004_1451_gb300 as bamg

    A = _walk(nx, ny)
    xs = []
    for persistent in (0, 1):
        s = bamg.Solver(*A, r=10, levels=20, grid=(nx, ny), precision="mixed", max_it=7, mle_restart=0,
                        persistent=persistent)
        x = torch.empty(nx * ny, dtype=torch.float64, device="cuda")
        try:
            s.solve(1e-15, out=x)
        except bamg.BamgError:
            pass
        xs.append(x)
        s.close()
    assert torch.equal(xs[0], xs[1]) and bool(torch.isfinite(xs[0]).all())


def _level(kind, n, ncols, ld, dtype, offset, seed):
    """B (pattern with unit diagonal), a C/F split and test vectors whose rows start `offset` elements
    into their storage."""
    import scipy.sparse as sp
    import torch

    rng = np.random.default_rng(seed)
    if kind == "grid":  # five entries a row, neighbours a multiple of 512 apart
        nx = 512
        i = np.arange(n)
        pairs = [(i[:-1], i[1:]), (i[:-nx], i[nx:])] if n > nx else [(i[:-1], i[1:])]
    elif kind == "ring":  # about 12 entries a row
        i = np.arange(n)
        pairs = [(i, (i + rng.integers(1, 40, n)) % n) for _ in range(6)]
    else:  # hubs: a few rows of hundreds of entries, so that searches overflow the first list
        i = np.arange(n)
        pairs = [(i, rng.integers(0, n, n)) for _ in range(2)] + [(np.full(300, h), rng.integers(0, n, 300)) for h in range(4)]
    a, b = (np.concatenate([p[k] for p in pairs]) for k in (0, 1))
    A = sp.coo_matrix((np.ones(a.size), (a, b)), shape=(n, n))
    A = sp.csr_matrix(A + A.T + sp.identity(n))
    A.data[:] = -0.1
    A.setdiag(1.0)
    A.sort_indices()
    cf = rng.random(n) < 0.3
    cf[0] = True
    cidx = np.where(cf, np.cumsum(cf) - 1, -1)
    td = torch.float64 if dtype == "fp64" else torch.float32
    X = torch.empty(n * ld + offset, dtype=td, device="cuda")[offset:].view(n, ld)
    X.copy_(torch.tensor(rng.random((n, ld)) + 0.5))
    X[:, ncols:] = float("nan")  # columns beyond ncols are not read into a result
    B = tuple(torch.tensor(v, device="cuda") for v in (A.indptr.astype(np.int32), A.indices.astype(np.int32)))
    B += (torch.tensor(A.data, dtype=td, device="cuda"),)
    w = torch.tensor(np.concatenate([rng.random(ncols), np.zeros(32 - ncols)]), device="cuda")
    return B, torch.tensor(cf.astype(np.uint8), device="cuda"), torch.tensor(cidx.astype(np.int32), device="cuda"), X, w


@pytest.mark.parametrize("kind,n", [("grid", 1), ("grid", 1023), ("grid", 9001), ("ring", 2001), ("hubs", 1500),
                                    ("hubs", 7000)])
@pytest.mark.parametrize("ncols,ld,offset,c,z,mmax,dtype", [
    (1, 4, 0, 1, 1, 16, "fp32"), (8, 8, 0, 2, 2, 16, "fp32"), (9, 12, 0, 2, 2, 5, "fp32"), (16, 17, 0, 2, 2, 16, "fp32"),
    (20, 20, 1, 2, 2, 16, "fp32"), (24, 24, 0, 2, 3, 16, "fp32"), (31, 32, 0, 2, 2, 16, "fp32"), (12, 12, 0, 4, 2, 16, "fp32"),
    (10, 10, 0, 2, 2, 16, "fp64"), (17, 18, 0, 3, 1, 16, "fp64"), (5, 5, 1, 2, 3, 1, "fp64")])
def test_interpolation_rows_equal_the_recording_path(kind, n, ncols, ld, offset, c, z, mmax, dtype):
    """interp_ls (searches and fits in two kernels, two points a warp) against interp_features, whose
    kernel takes a point a warp and also writes its rows by candidate: the same rows bit for bit, over
    short and long rows, lists that overflow, odd sizes, alignments and column counts."""
    import torch

    import paper_1004_1451_gb300 as bamg

    B, cf, cidx, X, w = _level(kind, n, ncols, ld, dtype, offset, seed=n + ncols)
    pcol, pval, pcnt = bamg.interp_ls(B, cf, cidx, X, ncols, w, z=z, mmax=mmax, c=c, ridge=1e-4)
    _, tgt, cand = bamg.interp_features(B, cf, cidx, X, ncols, w, z=z, mmax=mmax, c=c, ridge=1e-4, targets=True)
    pcol, pval, pcnt, tgt, cand = (t.cpu().numpy() for t in (pcol, pval, pcnt, tgt, cand))
    cidx_h, cf_h = cidx.cpu().numpy(), cf.cpu().numpy().astype(bool)
    assert (pcnt[cf_h] == 1).all() and (pcol[cf_h, 0] == cidx_h[cf_h]).all() and (pval[cf_h, 0] == 1).all()
    for i in np.flatnonzero(~cf_h):
        slots = np.flatnonzero(tgt[i])
        assert len(slots) == pcnt[i] and (pcol[i, pcnt[i]:] == -1).all() and (pval[i, pcnt[i]:] == 0).all()
        cols = cidx_h[cand[i, slots]]
        order = np.argsort(cols)
        assert np.array_equal(cols[order], pcol[i, :pcnt[i]])
        assert np.array_equal(tgt[i, slots][order], pval[i, :pcnt[i]].astype(np.float32))


def test_kept_memory_is_bounded_and_given_back():
    """Handles made, used and freed on several threads and streams keep at most the pool's 512 MiB and
    their streams; release_memory gives it back.  (The first handle loads kernels and pages.)"""
    import threading

    import torch

    import paper_1004_1451_gb300 as bamg

    A = _walk(160, 150)
    results = {}

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(3):
                s = bamg.Solver(*A, r=8, levels=20, grid=(160, 150), precision="mixed")
                x, _ = s.solve(1e-10)
                s.close()
            torch.cuda.current_stream().synchronize()
            results[k] = x

    work(-1)
    bamg.release_memory()
    torch.cuda.empty_cache()
    free0 = torch.cuda.mem_get_info()[0]
    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    assert free0 - torch.cuda.mem_get_info()[0] <= (640 << 20)
    assert all(torch.equal(results[k], results[-1]) for k in range(4))
    bamg.release_memory()
    assert free0 - torch.cuda.mem_get_info()[0] <= (64 << 20)


@pytest.mark.parametrize("dtype", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny,ncols", [(150, 100, 12), (700, 301, 16)])
def test_odd_sweep_counts_write_every_row(dtype, nx, ny, ncols):
    """An odd number of sweeps ends in the work buffer and is copied back: three sweeps in one call and
    one sweep three times (each copied back) and two and one give the same bits, on every row."""
    import torch

    import paper_1004_1451_gb300 as bamg

    ptr, col, val = _walk(nx, ny)
    td = torch.float64 if dtype == "fp64" else torch.float32
    n = nx * ny
    # B = I - A with the diagonal last in each row's order of columns put in its place
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), (ptr[1:] - ptr[:-1]).long())
    rows = torch.cat([row, torch.arange(n, device="cuda")])
    cols = torch.cat([col.long(), torch.arange(n, device="cuda")])
    vals = torch.cat([-val, torch.ones(n, dtype=torch.float64, device="cuda")])
    order = torch.argsort(rows * n + cols)
    B = ((ptr + torch.arange(n + 1, device="cuda")).int(), cols[order].int(), vals[order].to(td))
    X0 = torch.rand(n, ncols, dtype=td, device="cuda")
    once, thrice, split = X0.clone(), X0.clone(), X0.clone()
    bamg.relax(B, once, ncols, 0, 0.7, 3)
    for _ in range(3):
        bamg.relax(B, thrice, ncols, 0, 0.7, 1)
    bamg.relax(B, split, ncols, 0, 0.7, 2)
    assert torch.equal((split != X0).any(1), torch.ones(n, dtype=torch.bool, device="cuda"))
    bamg.relax(B, split, ncols, 0, 0.7, 1)
    assert torch.equal(once, split) and torch.equal(once, thrice)


@pytest.mark.parametrize("shift", [False, True])
@pytest.mark.parametrize("rows_entries,n,ncols,nu", [(3, 1, 4, 1), (5, 1000, 10, 2), (5, 400001, 16, 3), (14, 3001, 7, 2),
                                                     (14, 300000, 12, 1)])
def test_first_sweep_forms_the_diagonals(shift, rows_entries, n, ncols, nu):
    """FP32 sweeps whose first one reads the diagonals off the rows, against sweeps one call at a time
    with the diagonals at hand (relax_noalloc where it fits, else single-sweep calls): same bits, the
    diagonal among the first entries of a row or beyond them, small levels and tuned ones."""
    import torch

    import paper_1004_1451_gb300 as bamg

    g = torch.Generator(device="cuda").manual_seed(n)
    m = min(rows_entries, n)
    i = torch.arange(n, device="cuda")
    off = torch.arange(m, device="cuda") - (m - 1 if rows_entries == 14 else m // 2)  # the last entry, or the middle
    col = (i[:, None] + off[None, :]).clamp(0, n - 1)
    col = torch.where(col == torch.cat([col[:, 1:], col[:, -1:] + n], 1), torch.full_like(col, -1), col)  # unique
    ok = col >= 0
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = ok.sum(1).cumsum(0)
    val = torch.where(col == i[:, None], 1.0 + torch.rand(n, m, generator=g, device="cuda"),
                      -0.1 * torch.rand(n, m, generator=g, device="cuda"))[ok]
    B = (ptr.int(), col[ok].int(), val.contiguous())
    T = (0.5 + 0.1 * torch.rand(val.numel(), generator=g, device="cuda")) if shift else None
    lam = (0.01 * torch.rand(ncols, generator=g, device="cuda")).double() if shift else None
    ld = (ncols + 3) // 4 * 4
    X = torch.rand(n, ld, generator=g, device="cuda")
    Y = X.clone()
    bamg.relax(B, X, ncols, 0, 0.7, nu, T_val=T, lam=lam)
    if n * (ld + 3) * 4 <= (8 << 20) - 4096:
        bamg.relax_noalloc(B, Y, ncols, 0, 0.7, nu, T_val=T, lam=lam)
    else:
        d = torch.zeros(n, device="cuda")
        row = torch.repeat_interleave(i, ok.sum(1))
        at = B[1].long() == row
        d[row[at]] = val[at]
        for _ in range(nu):
            bamg.relax(B, Y, ncols, 0, 0.7, 1, T_val=T, lam=lam)
        Z = torch.rand(n, ld, generator=g, device="cuda")
        R = Z.double()
        v = val.double() if not shift else None
        bamg.relax(B, Z, ncols, 0, 0.7, 1, T_val=T, lam=lam)
        for c in range(ncols):  # one sweep in FP64: 14 products and a quotient in FP32, 2^-24 each
            l = lam[c] if shift else 0.0
            w = val.double() - l * T.double() if shift else v
            s = torch.segment_reduce(w * R[:, c][B[1].long()], "sum", lengths=ok.sum(1))
            dd = torch.zeros(n, dtype=torch.float64, device="cuda")
            dd[row[at]] = w[at]
            ref = R[:, c] - 0.7 * s / dd
            assert float((Z[:, c].double() - ref).abs().max()) <= 40 * 2.0 ** -24 * 4.0
    assert torch.equal(X, Y)


@pytest.mark.parametrize("nx,ny,ncols", [(2, 1, 1), (17, 19, 32), (300, 250, 10), (1100, 600, 5)])
def test_weights_over_many_partials(nx, ny, ncols):
    """Column norms and LS weights in FP64 (one to 512 partial blocks, summed by several blocks) against
    torch: sums of positive terms, n 2^-53 relative at most, and a quotient."""
    import torch

    import paper_1004_1451_gb300 as bamg

    ptr, col, val = _walk(nx, ny)
    n = nx * ny
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), (ptr[1:] - ptr[:-1]).long())
    i = torch.arange(n, device="cuda")
    rows, cols = torch.cat([row, i]), torch.cat([col.long(), i])
    vals = torch.cat([-val, torch.ones(n, dtype=torch.float64, device="cuda")])
    order = torch.argsort(rows * n + cols)
    B = ((ptr + torch.arange(n + 1, device="cuda")).int(), cols[order].int(), vals[order].contiguous())
    X = 1.0 + torch.rand(n, ncols + ncols % 2, dtype=torch.float64, device="cuda")
    ref = X[:, :ncols] / torch.linalg.vector_norm(X[:, :ncols], dim=0)
    count = (B[0][1:] - B[0][:-1]).long()
    bx = torch.stack([torch.segment_reduce(B[2] * ref[:, c].contiguous()[B[1].long()], "sum", lengths=count)
                      for c in range(ncols)], 1)
    wr = 1.0 / bx.square().sum(0)
    w = bamg.tv_weights(B, X, ncols)
    tol = 64 * n * 2.0 ** -53 + 1e-14
    assert float(((w - wr / wr.max()).abs() / (wr / wr.max())).max()) <= 1e3 * tol
    assert float((X[:, :ncols] - ref).abs().max()) <= tol


@pytest.mark.parametrize("kind,n", [("path", 2), ("path", 5000), ("grid", 70000), ("star", 3000), ("dense", 700),
                                    ("hub", 2000), (30, 900), (150, 301)])
def test_independent_set_is_the_greedy_one(kind, n):
    """The splitting before any relaxation round (max_rounds 0) is the greedy independent set by
    descending (priority, index): long chains of waiting neighbours, more than 64 neighbours a state
    (their states are then looked up again), rows of one direction only, every number of lanes a row
    (by the mean row length; a hub's row is longer than its lanes remember)."""
    import torch

    import paper_1004_1451_gb300 as bamg
    from oracle import bamg as ob

    rng = np.random.default_rng(n)
    if kind == "path":
        a, b = np.arange(n - 1), np.arange(1, n)
    elif kind == "grid":
        i = np.arange(n)
        a, b = np.concatenate([i[:-1], i[:-250]]), np.concatenate([i[1:], i[250:]])
    elif kind == "star":
        a, b = np.concatenate([np.zeros(n - 1, int), np.ones(n - 2, int)]), np.concatenate([np.arange(1, n), np.arange(2, n)])
    else:
        a = np.repeat(np.arange(n), {"dense": 60, "hub": 14}.get(kind, kind))
        b = rng.integers(0, n, a.size)
        if kind == "hub":
            a, b = np.concatenate([a, np.full(n - 1, n - 1)]), np.concatenate([b, np.arange(n - 1)])
    import scipy.sparse as sp

    A = sp.csr_matrix((np.full(a.size, -0.01), (a, b)), shape=(n, n))  # edges stored one way
    A.setdiag(1.0)
    A = sp.csr_matrix(A)
    A.sort_indices()
    B = (torch.tensor(A.indptr.astype(np.int32), device="cuda"), torch.tensor(A.indices.astype(np.int32), device="cuda"),
         torch.tensor(A.data, device="cuda"))
    cf, _, nc, _ = bamg.coarsen_cr(B, 3, 11, max_rounds=0)
    pri = ob.counter_u64(11, (1 << 23) + (3 << 8), np.arange(n, dtype=np.uint64))
    S = sp.csr_matrix(A + A.T)
    want = np.zeros(n, dtype=bool)
    gone = np.zeros(n, dtype=bool)
    for i in sorted(range(n), key=lambda k: (int(pri[k]), k), reverse=True):
        if not gone[i]:
            want[i] = True
            gone[S.indices[S.indptr[i]:S.indptr[i + 1]]] = True
            gone[i] = True
    assert np.array_equal(cf.cpu().numpy().astype(bool), want) and nc == want.sum()


@pytest.mark.parametrize("per_row", [4, 20])
def test_entries_of_coarse_columns_take_no_part(per_row):
    """F-relaxation leaves out the columns of C: an infinite entry there changes no splitting (one lane
    and several lanes a row).  The first set does not depend on the values, so its columns are known."""
    import scipy.sparse as sp
    import torch

    import paper_1004_1451_gb300 as bamg

    n = 1500
    rng = np.random.default_rng(per_row)
    A = sp.random(n, n, density=per_row / n, random_state=rng, format="csr")
    A.data[:] = -1.0
    A = sp.csr_matrix(A + A.T)
    A.setdiag(0.0)
    A.setdiag(-np.asarray(A.sum(1)).ravel() + 0.01)
    A = sp.csr_matrix(A)
    A.sort_indices()
    rp, ci = (torch.tensor(v.astype(np.int32), device="cuda") for v in (A.indptr, A.indices))
    val = torch.tensor(A.data, device="cuda")
    first = bamg.coarsen_cr((rp, ci, val), 0, 5, max_rounds=0)[0].bool()
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
    hit = first[ci.long()] & ~first[row]
    want, _, nc, rounds = bamg.coarsen_cr((rp, ci, val), 0, 5, theta=0.3)
    assert rounds > 0
    for bad in (float("inf"), float("nan")):
        got, _, nc2, rounds2 = bamg.coarsen_cr((rp, ci, torch.where(hit, torch.full_like(val, bad), val)), 0, 5, theta=0.3)
        assert torch.equal(got, want) and nc2 == nc and rounds2 == rounds
