"""The bench's serving leg and the serving workload end when the server does not: on CPU,
with a server that never completes a request."""
import importlib.util
import os
import types

import pytest

torch = pytest.importorskip("torch")

from paper_2507_09165_gb300 import admm, binding as b  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _bench():
    spec = importlib.util.spec_from_file_location("bench_mod", os.path.join(ROOT, "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


class _Server:
    """Takes requests and never completes one."""

    def __init__(self, monkeypatch):
        self.calls = []
        for name in ("create", "submit", "wait", "poll", "stats", "destroy"):
            monkeypatch.setattr(b, "psd_server_" + name, getattr(self, name))

    def create(self, *a):
        return self

    def submit(self, *a, **k):
        return 1

    def wait(self, server, ticket, timeout_ms=0):
        assert timeout_ms > 0, "a wait without a limit"
        raise b.PsdError(6, "psd_server_wait")

    def poll(self, server, ticket):
        return False, None, 0.0

    def stats(self, server):
        return {}

    def destroy(self, server):
        self.calls.append("destroy")


def test_serving_leg_reports_a_stalled_server_and_leaves_it(monkeypatch):
    server = _Server(monkeypatch)
    from paper_2507_09165_gb300 import synth
    monkeypatch.setattr(synth, "er_laplacian", lambda n, seed, *a: torch.zeros(4, 4).double().numpy())
    args = types.SimpleNamespace(serve_rate=8.0, serve_seconds=1.0, serve_iters=5)
    res = _bench().serving_leg(torch.device("cpu"), args)
    assert "PSD_ERR_TIMEOUT" in res["unfinished"]
    assert server.calls == []  # destroying it would wait for the stalled work


def test_serving_workload_gives_up_on_a_request(monkeypatch):
    _Server(monkeypatch)
    monkeypatch.setattr(torch.cuda, "Stream", lambda *a: None)
    monkeypatch.setattr(admm, "Solve", lambda C, sig, iters, stream: types.SimpleNamespace(
        n=4, S=None, ready=None, sigma=sig, make_input=lambda: None))
    with pytest.raises(TimeoutError):
        admm.run_serving(object(), {4: None}, solve_rate=100.0, arrival_seconds=0.1, max_solves=1,
                         request_limit_s=0.05)


def test_the_serving_leg_comes_last():
    with open(os.path.join(ROOT, "bench.py")) as f:
        code = f.read().split("def run_ours(")[1]
    legs = [code.index('leg("%s"' % k) for k in ("batched", "bands", "deflation", "accuracy", "cpu baseline", "serving")]
    assert legs == sorted(legs)
