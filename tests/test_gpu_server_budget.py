"""Budgets that a request server accepts.

`smallest_budget` is the smallest budget of the server's earlier memory layout (two
preparation streams with its Lanczos scratch, shares of <out, X - out> in rows of their
own): budgets that were accepted stay accepted, and serve their largest order.
"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2507_09165_gb300 import binding as b, synth  # noqa: E402


def _up(v, m):
    return (v + m - 1) // m * m


def smallest_budget(max_order, max_batch):
    n, npad, nb = max_order, _up(max_order, 256), (max_order + 127) // 128
    npart, nctas = (n + 31) // 32, (n + 255) // 256
    lanczos = sum(_up(v, 256) for v in (8 * 21 * npad, 8 * 3 * npad, 4 * 2 * npad, 8 * 2 * nb * npad, 8 * 32 * npart,
                                        8 * 32 * npart, 8 * max(npart, nctas), 8 * (nb * (nb + 1) // 2), 8))
    lane = _up(1024 + lanczos, 1024)
    ldm = _up(n, 64)
    wide = (n + 255) // 256
    rows_needed = 4 * n + (32 * wide * (wide + 1) + 2 * ldm - 1) // (2 * ldm)

    def fixed(tile_cap):
        # per-step staging: block records (112 bytes) of 4 products, finished records (16), tiles, reports (64)
        stage = _up(4 * 112 * max_batch, 256) + _up(16 * max_batch, 256) + _up(16 * 4 * tile_cap, 256) + \
            _up(64 * max_batch, 256)
        return 1024 + _up(1280 * max_batch, 1024) + 2 * lane + 2 * _up(stage, 1024)

    tile_cap = 2 * max_batch + (max_order // 256 + 3) * (rows_needed // 1024 + 1)
    return fixed(tile_cap) + rows_needed * 2 * ldm


@pytest.mark.parametrize("max_order,max_batch", [(64, 1024), (257, 64), (1024, 8), (2048, 32), (4096, 1)])
def test_smallest_budget_serves_its_largest_order(max_order, max_batch):
    h = b.psd_server_create(smallest_budget(max_order, max_batch), 0, max_order, max_batch)
    try:
        jobs = []
        for i, n in enumerate((max_order, 1, max_order - 1, max_order // 2)):
            X = torch.from_numpy(synth.wigner(n, 60 + i)).cuda()
            out, ref = torch.empty_like(X), torch.empty_like(X)
            b.psd_project(n, X, n, ref, "fp16")
            jobs.append((n, out, ref, X, b.psd_server_submit(h, n, X, n, out, n, "fp16")))
        for n, out, ref, X, t in jobs:
            info, _ = b.psd_server_wait(h, t, 60000)
            assert info["status"] == 0
        torch.cuda.synchronize()
        for n, out, ref, X, t in jobs:
            assert torch.equal(out, ref), n
        assert b.psd_server_stats(h)["arena_rows"] >= 4 * max_order
    finally:
        b.psd_server_destroy(h)


def test_many_small_requests_at_once():
    # a request of order 500 has 48 final tiles where a stage product has 6: the final
    # products of many of them together are more than one step's staging holds
    n, count = 500, 64
    h = b.psd_server_create(150 << 20, 0, n, count)
    try:
        X = torch.from_numpy(synth.wigner(n, 5)).cuda()
        ref = torch.empty_like(X)
        b.psd_project(n, X, n, ref, "bf16")
        outs = [torch.empty_like(X) for _ in range(count)]
        tickets = [b.psd_server_submit(h, n, X, n, o, n, "bf16") for o in outs]
        for t in tickets:
            info, _ = b.psd_server_wait(h, t, 60000)
            assert info["status"] == 0
        torch.cuda.synchronize()
        assert all(torch.equal(o, ref) for o in outs)
    finally:
        b.psd_server_destroy(h)
