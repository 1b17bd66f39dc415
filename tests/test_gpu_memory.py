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
