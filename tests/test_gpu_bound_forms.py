"""The norm bound's forms give the same bits at the orders where the form changes.

A direct call runs the bound as one cluster (n <= 1152), as the persistent kernel
with one or two tiles per CTA on chip (n <= 3072, n <= 4352 on 152 SMs) or with
streamed tiles; a served request runs the multi-launch form.  Rows that take no
16-byte loads go other ways: scalar loads, and a packed copy where tiles stream.
"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2507_09165_gb300 import binding as b  # noqa: E402

DEV = torch.device("cuda")
GB = 1 << 30


def _matrix(n, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    G = torch.randn(n, n, generator=g, device=DEV)
    return (G + G.T) * (0.5 / n ** 0.5)


def _bound(X, n, ld):
    A = torch.full((n, ld), float("nan"), device=DEV)
    A[:, :n] = X
    info = torch.zeros(b.INFO_BYTES, dtype=torch.uint8, device=DEV)
    b.psd_norm_bound(n, A, ld, info)
    torch.cuda.synchronize()
    d = b.info_from_bytes(info.cpu().numpy())
    d.pop("compl_resid")  # NaN: no projection ran
    return d


@pytest.mark.parametrize("n", [1, 31, 128, 129, 384, 1152, 1153, 3072, 3073, 4352, 4353])
def test_rows_without_16_byte_loads_give_the_same_bound(n):
    X = _matrix(n, n)
    aligned = _bound(X, n, (n + 3) // 4 * 4)
    odd = _bound(X, n, n + 1 if n % 2 == 0 else n)
    assert aligned["status"] == 0 and aligned == odd


@pytest.mark.parametrize("n", [19, 128, 129, 700, 1152, 1153, 3073, 4353])
def test_direct_and_served_reports_agree(n):
    X = _matrix(n, 7 + n)
    out, served = torch.empty_like(X), torch.empty_like(X)
    info = torch.zeros(b.INFO_BYTES, dtype=torch.uint8, device=DEV)
    b.psd_project_ex(n, X, n, out, n, "fp16", info)
    torch.cuda.synchronize()
    h = b.psd_server_create(2 * GB, 0, 4480, 4)
    try:
        got, _ = b.psd_server_wait(h, b.psd_server_submit(h, n, X, n, served, n, "fp16"), 60000)
    finally:
        b.psd_server_destroy(h)
    assert got == b.info_from_bytes(info.cpu().numpy()) and got["status"] == 0
    assert torch.equal(out, served)
