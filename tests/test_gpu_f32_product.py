"""The FP32 path's product kernel, element by element, at every tile width it runs with.

Through psd_symm_product with EPI_SCALED_PAIR: FP16 hi/lo pairs of the values times powers of
two.  The orders give tile widths of 32 to 256 columns with remainders on both sides of a
32-column chunk, a 128-row half, a 64-element stage and a 128-element accumulation chunk.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2507_09165_gb300 import binding as b  # noqa: E402

DEV = torch.device("cuda")
SA, SB, SY, SC = 2.0 ** 14, 2.0 ** 12, 2.0 ** 11, 2.0 ** 13


def tile_width(n):
    """The width with the least rounds of tiles over the SM pairs times (290 + width)."""
    pairs = torch.cuda.get_device_properties(0).multi_processor_count // 2
    cost = {w: -(-sum(-(-(n - m) // w) for m in range(0, n, 256)) // pairs) * (290 + w) for w in range(256, 0, -32)}
    return min(cost, key=cost.get)


def _sym(n, seed):
    G = np.random.default_rng(seed).standard_normal((n, n))
    return (G + G.T) * (0.5 / np.sqrt(n))


def _pair(A, scale, ld):
    """(device pair, its value in FP64)."""
    n = A.shape[0]
    v = (A * scale).astype(np.float32)
    hi = v.astype(np.float16)
    lo = (v - hi.astype(np.float32)).astype(np.float16)
    P = np.full((2, n, ld), np.nan, dtype=np.float16)
    P[0, :, :n], P[1, :, :n] = hi, lo
    return torch.from_numpy(P).to(DEV), (hi.astype(np.float64) + lo.astype(np.float64)) / scale


@pytest.mark.parametrize("n,width", [(1, 32), (33, 32), (129, 32), (385, 32), (1000, 64), (1037, 64), (1499, 96),
                                     (1501, 96), (1793, 128), (2001, 128), (2177, 160), (2307, 192), (2529, 224),
                                     (2753, 256), (3001, 160), (4097, 160)])
def test_elements_of_every_epilogue(n, width):
    # A sum's terms leave out lo * lo (2^-22 of |A||B|); the tensor cores add into FP32 without
    # rounding to nearest, 24 instructions a chunk of 128 (2^-22 each), the chunks are added
    # rounded to nearest (2^-24 each), and the output is split into 22 bits with a floor of
    # 2^-25 / scale.
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert tile_width(n) == width
    ld = (n + 7) // 8 * 8
    A, Av = _pair(_sym(n, n), SA, ld)
    B, Bv = _pair(_sym(n, n + 1), SB, ld)
    Y, Yv = _pair(_sym(n, n + 2), SY, ld)
    prod = Av @ Bv
    mass = (25.0 * 2.0 ** -22 + (n / 128.0 + 1.0) * 2.0 ** -24) * (np.abs(Av) @ np.abs(Bv))
    iu = np.triu_indices(n)
    scales = (1.0 / (SA * SB), 1.0 / SY, SC)
    a, bb, c, s, lam = 1.5, -0.7, 0.3, 1.0 / 1.001, 2.5
    for epi, own, D, tol in ((0, (), prod, mass),
                             (1, (a, bb, c), a * np.eye(n) + bb * Yv + c * prod,
                              c * mass + 2.0 ** -23 * (abs(bb) * np.abs(Yv) + 2.0 * a * np.eye(n))),
                             (2, (s,), s * prod, s * mass)):
        C = torch.full((2, n, ld), float("nan"), dtype=torch.float16, device=DEV)
        amax = torch.zeros(1, device=DEV)
        b.psd_symm_product(n, A, B, ld, C, 0, "fp32", epi | b.EPI_SCALED_PAIR, params=own + scales, aux=Y, ld_aux=ld,
                           d_absmax=amax)
        torch.cuda.synchronize()
        P = C.cpu().numpy().astype(np.float64)
        assert np.isnan(P[:, :, n:]).all()
        got = (P[0] + P[1])[:, :n] / SC
        assert np.array_equal(got, got.T)
        err = np.abs(got - D)[iu]
        assert np.all(err <= (tol + 2.0 ** -22 * np.abs(D))[iu] + 2.0 ** -25 / SC + 2.0 ** -23 * np.abs(D)[iu]), epi
        if n > 64:
            assert np.linalg.norm(err) <= 1.5e-6 * np.linalg.norm(D[iu])
        assert amax.item() == pytest.approx(np.abs(got).max(), rel=1e-6)
    Xf = np.triu(_sym(n, n + 3)).astype(np.float32)
    X = torch.from_numpy(Xf).to(DEV)
    # column-major upper triangle: element (i, j), i <= j, at j * ld + i
    Xc = X.T.contiguous()
    out = torch.full((n, n + 1), float("nan"), device=DEV)
    b.psd_symm_product(n, A, B, ld, out, n + 1, "fp32", 3 | b.EPI_SCALED_PAIR, params=(lam,) + scales, aux=Xc, ld_aux=n)
    torch.cuda.synchronize()
    o = out.cpu().numpy().astype(np.float64)
    assert np.isnan(o[:, n:]).all()
    o = o[:, :n]
    assert np.array_equal(o, o.T)
    D = 0.5 * (Xf.astype(np.float64) + lam * prod)
    err = np.abs(o - D)[iu]
    assert np.all(err <= (0.5 * lam * mass + 2.0 ** -23 * (np.abs(D) + lam * np.abs(prod)))[iu])


def test_rejects_what_it_does_not_run():
    A = torch.zeros((2, 64, 64), dtype=torch.float16, device=DEV)
    for prec, flags, params in (("mixed", 0, (1.0,) * 3), ("fp32", b.EPI_CTA_PAIR, (1.0,) * 3),
                                ("fp32", b.EPI_GROUPED, (1.0,) * 3), ("fp16", 0, (1.0,) * 3)):
        with pytest.raises(b.PsdError):
            b.psd_symm_product(64, A, A, 64, torch.empty_like(A), 0, prec, b.EPI_SCALED_PAIR | flags, params=params)
    with pytest.raises(ValueError):
        b.psd_symm_product(64, A, A, 64, torch.empty_like(A), 0, "fp32", b.EPI_SCALED_PAIR)
