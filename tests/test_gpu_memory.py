"""Calls on a device with little free memory: what fits is not refused."""

import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


class _Only:
    """Holds the device's memory but for `free` bytes."""

    def __init__(self, free):
        self.free = free

    def __enter__(self):
        import torch

        import paper_1004_1451_gb300 as bamg

        bamg.release_memory()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        at_hand = torch.cuda.mem_get_info()[0]
        if at_hand < self.free:
            pytest.skip("less memory free than the test leaves")
        self.held = torch.empty(at_hand - self.free, dtype=torch.uint8, device="cuda")

    def __exit__(self, *exc):
        import torch

        import paper_1004_1451_gb300 as bamg

        self.held = None
        torch.cuda.empty_cache()
        bamg.release_memory()


def _walk(nx, ny):
    import torch

    off = torch.tensor([-nx, -1, 1, nx], device="cuda")
    i = torch.arange(nx * ny, device="cuda")
    x, y = i % nx, i // nx
    ok = torch.stack([y > 0, x > 0, x < nx - 1, y < ny - 1], 1)
    deg = ok.sum(1)
    col = (i[:, None] + off)[ok]
    ptr = torch.zeros(nx * ny + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = deg.cumsum(0)
    return (ptr.int(), col.int(), 1.0 / deg[col].double()), deg.double() / deg.sum()


def test_batch_leaves_fewer_in_flight_where_memory_is_short():
    """Twelve chains of about 1 GiB with 6 GiB free and the number of threads left to the library: one thread per four
    chains fits, one per chain does not."""
    import torch

    import paper_1004_1451_gb300 as bamg

    A, want = _walk(724, 724)
    opts = {"grid": (724, 724), "precision": "fp64"}
    bamg.solve_batch([A], 8, 20, 1e-10, opts=opts)  # loads the kernels
    with _Only(6 << 30):
        xs, stats = bamg.solve_batch([A] * 12, 8, 20, 1e-10, opts=opts)
        assert all(s["status"] == 0 for s in stats)
        assert all(float((x - want).abs().sum()) <= 1e-3 and torch.equal(x, xs[0]) for x in xs)
        del xs


def _features(rows):
    import torch

    g = torch.Generator(device="cuda").manual_seed(rows)
    feat = torch.randn(rows, 112, device="cuda", generator=g)
    feat[:, 0:96:6] = (torch.rand(rows, 16, device="cuda", generator=g) < 0.7).float()
    return feat, torch.randn(rows, 16, device="cuda", generator=g)


def test_gradients_of_a_large_batch_in_little_memory():
    """A batch of 4,000,000 rows with 7 GiB free beside its features: activations and gradients take 6104 MiB as long
    as every number is kept once, 8160 with the rounded gradients beside the unrounded ones."""
    import torch

    import paper_1004_1451_gb300 as bamg

    rows = 4000000
    feat, target = _features(rows)
    m = bamg.Model(3)
    m.gradients(feat[:300000], target[:300000])  # loads the kernels
    with _Only(7 << 30):
        g, loss = m.gradients(feat, target)
    d = torch.cat([m.forward(c) for c in feat.split(500000)]).double() - target
    d *= feat[:, 0:96:6] > 0
    assert loss == pytest.approx(float(d.square().sum()) / rows, rel=1e-6)
    # 15,625 additions a partial sum and 13 to join the 256 of a column, each to 2^-24 of the sum of magnitudes
    err = (torch.tensor(g[-16:], dtype=torch.float64) - (2 * d.sum(0) / rows).cpu()).abs()
    assert bool((err <= (15625 + 13) * 2.0 ** -24 * (2 * d.abs().sum(0) / rows).cpu()).all())


@pytest.mark.parametrize("rows", [2 ** 18, 2 ** 18 + 1, 2 ** 18 + 256 * 7 + 17])
def test_gradients_where_the_rounded_ones_are_not_kept(rows):
    """On both sides of the row count from which the rounded gradients have no place of their own, against the network
    with the same roundings in 64 bits: a bf16 rounding that falls the other way moves an entry by at most 2^-8 of
    itself, so each gradient by at most 2^-8 of its norm."""
    import torch

    import paper_1004_1451_gb300 as bamg

    def bf(x):
        return x.to(torch.bfloat16).double()

    feat, target = _features(rows)
    m = bamg.Model(3)
    p = torch.tensor(m.get(), device="cuda").double()
    p += 0.02 * torch.rand(p.shape, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    m.set(p.cpu().numpy())
    p = p.float().double()
    W1, b1, W2, b2, W3, b3 = (t for t in torch.split(p, [128 * 112, 128, 128 * 128, 128, 16 * 128, 16]))
    W1, W2, W3 = W1.view(128, 112), W2.view(128, 128), W3.view(16, 128)
    x = bf(feat)
    h1 = bf((x @ bf(W1).T + b1).relu().float())
    h2 = bf((h1 @ bf(W2).T + b2).relu().float())
    d3 = 2 * ((h2 @ bf(W3).T + b3) - target) * (feat[:, 0:96:6] > 0) / rows
    d2 = (bf(d3.float()) @ bf(W3)) * (h2 > 0)
    d1 = (bf(d2.float()) @ bf(W2)) * (h1 > 0)
    want = [bf(d1.float()).T @ x, d1.sum(0), bf(d2.float()).T @ h1, d2.sum(0), bf(d3.float()).T @ h2, d3.sum(0)]
    g, _ = m.gradients(feat, target)
    at = 0
    for w in want:
        part = torch.tensor(g[at:at + w.numel()], device="cuda").double().view(w.shape)
        at += w.numel()
        assert float((part - w).norm()) <= 2.0 ** -8 * float(w.norm())


def test_calls_after_one_that_ran_out_of_memory():
    """A call that the device has no memory for says so; the calls after it, on the same thread, run."""
    import torch

    import paper_1004_1451_gb300 as bamg

    big, _ = _walk(1400, 1400)
    small, want = _walk(60, 50)
    opts = {"grid": (60, 50), "precision": "fp64"}
    bamg.solve_batch([small], 8, 20, 1e-10, opts=opts)  # loads the kernels
    with _Only(1 << 30):
        with pytest.raises(bamg.BamgError) as e:
            bamg.Solver(*big, r=8, levels=20, grid=(1400, 1400), precision="fp64")
        assert e.value.code == -4
        x, _ = bamg.Solver(*small, r=8, levels=20, **opts).solve(1e-10)
        assert float((x - want).abs().sum()) <= 1e-6
        with pytest.raises(bamg.BamgError) as e:
            bamg.solve_batch([small, big, small], 8, 20, 1e-10, workers=1,
                             opts=[opts, {"grid": (1400, 1400), "precision": "fp64"}, opts])
        assert e.value.code == -4 and [s["status"] for s in e.value.stats] == [0, -4, 0]
        assert torch.equal(e.value.xs[0], e.value.xs[2]) and float((e.value.xs[0] - want).abs().sum()) <= 1e-6


@pytest.mark.parametrize("nx,ny,count,mib", [(20, 10, 200, 1.0), (64, 64, 100, 9.2), (200, 200, 40, 89.0)])
def test_a_kept_handle_holds_little_beyond_its_buffers(nx, ny, count, mib):
    """Device memory of a hierarchy that has solved: its buffers (0.4, 7.4 and 73 MiB in FP64) and a quarter more, with what
    the pool rounds up to shared by all."""
    import torch

    import paper_1004_1451_gb300 as bamg

    A, _ = _walk(nx, ny)

    def make():
        s = bamg.Solver(*A, r=8, levels=20, grid=(nx, ny), precision="fp64")
        s.solve(1e-8)
        return s

    make().close()
    bamg.release_memory()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    handles = [make() for _ in range(count)]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = free - torch.cuda.mem_get_info()[0]
    for s in handles:
        s.close()
    bamg.release_memory()
    assert held <= (count * mib + 64) * 2 ** 20


def test_a_handle_does_not_grow_with_the_cycles_of_its_setup():
    """Setups of more cycles rebuild the coarse operators more often in the same memory."""
    import torch

    import paper_1004_1451_gb300 as bamg

    A, _ = _walk(64, 64)
    held = []
    for cycles in (2, 16):
        bamg.release_memory()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        handles = [bamg.Solver(*A, r=8, levels=20, grid=(64, 64), precision="fp64", setup_cycles=cycles) for _ in range(64)]
        torch.cuda.synchronize()
        held.append(free - torch.cuda.mem_get_info()[0])
        for s in handles:
            s.close()
    bamg.release_memory()
    assert held[1] <= held[0] + (32 << 20)
