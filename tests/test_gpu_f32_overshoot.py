"""A norm bound below ||X||_2 on the FP32 path: the report says so, with a finite size.

The bound is scaled down on the host (psd_debug_set); the iterates then leave the range of
their FP16 pairs within a few stages.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2507_09165_gb300 import binding as b  # noqa: E402
from paper_2507_09165_gb300 import synth  # noqa: E402

DEV = torch.device("cuda")
PSD_ERR_NONFINITE, PSD_ERR_BOUND = 4, 5


def _project(X):
    n = X.shape[0]
    out = torch.full_like(X, float("nan"))
    info = torch.zeros(b.INFO_BYTES, dtype=torch.uint8, device=DEV)
    b.psd_project_ex(n, X, n, out, n, "fp32", info)
    torch.cuda.synchronize()
    return out.cpu(), b.info_from_bytes(info.cpu().numpy())


@pytest.mark.parametrize("n", [1, 33, 700, 1500])
@pytest.mark.parametrize("factor", [0.2, 0.5, 0.9])
def test_small_bound_is_reported_as_overshoot(n, factor):
    X = torch.from_numpy(synth.wigner(n, 31 + n)).to(DEV)
    ref, info0 = _project(X)
    assert info0["status"] == 0 and info0["overshoot_max"] <= 1.01
    try:
        b.psd_debug_set(b.DEBUG_BOUND_SCALE, factor)
        out, info = _project(X)
    finally:
        b.psd_debug_set(b.DEBUG_BOUND_SCALE, 1.0)
    assert info["status"] == PSD_ERR_BOUND, info
    assert np.isfinite(info["overshoot_max"]) and info["overshoot_max"] > 1.01
    assert torch.isfinite(out).all()
    again, info1 = _project(X)
    assert info1["status"] == 0 and torch.equal(again.view(torch.int32), ref.view(torch.int32))


def test_nan_stays_nonfinite():
    X = torch.from_numpy(synth.wigner(300, 5)).to(DEV)
    X[7, 9] = X[9, 7] = float("nan")
    _, info = _project(X)
    assert info["status"] == PSD_ERR_NONFINITE
