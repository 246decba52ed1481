"""The FP32 path's product kernel at the edges of its tiles and accumulation chunks.

Orders around the 32-column chunks, the 128-row halves and 256 x 256 tiles, the
128-element accumulation chunks and the 32-element pipeline stages, in a padded
array and at small and large scales of X, against the oracle's exact filter output.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2507_09165_gb300 import binding as b  # noqa: E402
from paper_2507_09165_gb300 import synth  # noqa: E402

from _bars import TOL_F  # noqa: E402

DEV = torch.device("cuda")


def _project(X, ld):
    n = X.shape[0]
    Xd = torch.full((n, ld), float("nan"), dtype=torch.float32)
    Xd[:, :n] = torch.from_numpy(X)
    Xd = Xd.to(DEV)
    out = torch.full((n, ld), float("nan"), dtype=torch.float32, device=DEV)
    info = torch.zeros(b.INFO_BYTES, dtype=torch.uint8, device=DEV)
    b.psd_project_ex(n, Xd, ld, out, ld, "fp32", info)
    torch.cuda.synchronize()
    return out.cpu().numpy(), b.info_from_bytes(info.cpu().numpy())


@pytest.mark.parametrize("n,pad,scale", [(31, 0, 1.0), (33, 3, 1.0), (96, 0, 1.0), (127, 0, 1.0), (129, 7, 1.0),
                                         (255, 0, 1.0), (257, 0, 1e-6), (385, 1, 1e6), (511, 0, 1.0),
                                         (640, 0, 1.0)])
def test_fp32_products_at_their_edges(n, pad, scale):
    X = (synth.gaussian_symmetric(n, 40 + n).astype(np.float64) * scale).astype(np.float32)
    o, info = _project(X, n + pad)
    assert info["status"] == 0
    assert np.isnan(o[:, n:]).all()  # nothing is written past the order
    o = o[:, :n].astype(np.float64)
    assert np.array_equal(o, o.T)
    lam, Q = np.linalg.eigh(X.astype(np.float64))
    coefs, scales = oracle.schedules.schedule("single")
    F = oracle.filter_from_eig(lam, Q, info["lambda_bound"], coefs, scales)
    # the FP32 bar: 31 products whose operands carry 22 bits and whose sums are rounded every 128 terms
    assert oracle.rel_err(o, F) <= TOL_F["fp32"]
