"""A wait limit of 0 (psd_debug_set) reaches every form of a direct norm bound: one
thread-block cluster (n <= 1152), and the persistent kernel above.  The waits give up at
once and nothing hangs or faults; with the limit restored the same call gives the same bits.
"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2507_09165_gb300 import binding as b  # noqa: E402
from paper_2507_09165_gb300 import synth  # noqa: E402

DEV = torch.device("cuda")
PSD_ERR_TIMEOUT = 6


def _project(X, prec):
    n = X.shape[0]
    out = torch.full_like(X, float("nan"))
    info = torch.zeros(b.INFO_BYTES, dtype=torch.uint8, device=DEV)
    b.psd_project_ex(n, X, n, out, n, prec, info)
    torch.cuda.synchronize()
    return out, b.info_from_bytes(info.cpu().numpy())


@pytest.mark.parametrize("n", [33, 129, 700, 1152, 1153])
@pytest.mark.parametrize("prec", ["fp16", "fp32"])
def test_zero_limit_is_reported(n, prec):
    X = torch.from_numpy(synth.wigner(n, n)).to(DEV)
    ref, info0 = _project(X, prec)
    assert info0["status"] == 0
    try:
        b.psd_debug_set(b.DEBUG_BARRIER_LIMIT_NS, 0)
        _, info = _project(X, prec)
    finally:
        b.psd_debug_set(b.DEBUG_BARRIER_LIMIT_NS, 4e9)
    assert info["status"] == PSD_ERR_TIMEOUT, info
    again, info1 = _project(X, prec)
    assert info1 == info0 and torch.equal(again, ref)
