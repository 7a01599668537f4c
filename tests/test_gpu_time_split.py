"""Short of CTAs, the gridding and column kernels split a launch's samples: block lengths around the splits (parts of one
pass, empty parts, the smallest split block) against the FP64 oracle at the FP32 path's 1e-5, with a beam pixel whose
samples are written by different CTAs; and the built-in gridding shape (cell pairs on wide stripes) against the
narrow one, whose sums run in the same order (bit-identical)."""
import numpy as np
import pytest

import oracle
import paper_0812_3669_gb300 as moff
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    moff.build()
    yield


def case(seed, A, N, P, C, T, K=3):
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0, N, size=(A, 2))
    taps = (rng.normal(size=(A, P, K, K)) + 1j * rng.normal(size=(A, P, K, K))).astype(np.complex64).astype(np.complex128)
    codes = synth.pack_4bit(rng.integers(-8, 8, size=(T, C, A, P)), rng.integers(-8, 8, size=(T, C, A, P)))
    return pos, taps, codes, synth.gains_random(rng, C, A, P).astype(np.complex64).astype(np.complex128)


@pytest.mark.parametrize("N,P", [(32, 1), (64, 2), (128, 2), (256, 1), (512, 2)])
@pytest.mark.parametrize("T", [1, 15, 16, 17, 33, 127, 130])
def test_short_blocks(N, P, T):
    pos, taps, codes, gains = case(5 * T + N, 24, N, P, 1, T)
    with moff.Plan(pos, taps, N, 1, P) as pl:
        pl.set_gains(gains)
        pl.set_beams([N // 3], [N // 5])
        pl.submit(codes)
        beams = pl.read_beams()
        img, n = pl.read_image()
    assert n == T
    assert oracle.max_norm_err(img, oracle.moff_image(codes, gains, pos, taps, N, P)).max() <= 1e-5
    # the beam's power summed over the samples is the image at its pixel
    power = (np.abs(beams[:, 0, 0].astype(np.complex128)) ** 2).sum(axis=0)
    np.testing.assert_allclose(power, img[0, :P, N // 5, N // 3] if P == 2 else img[0, :1, N // 5, N // 3],
                               atol=1e-5 * img[0, :P].max(), rtol=0)


@pytest.mark.parametrize("N", [32, 64, 128, 256, 512])
@pytest.mark.parametrize("C,T", [(1, 1), (2, 100), (80, 5), (80, 130)])
def test_fp16_field(N, C, T):
    """The FP16 field's column kernels, split and whole, at odd sample counts (3e-3, the reduced-precision bar)."""
    if N == 512 and C == 80:
        C = 20
    pos, taps, codes, gains = case(N + T, 12, N, 2, C, T)
    with moff.Plan(pos, taps, N, C, 2, fp16tc=True) as pl:
        assert pl.route() == "fp16_rowspec"
        pl.set_gains(gains)
        pl.set_beams([N // 3], [N // 5])
        pl.submit(codes)
        beams = pl.read_beams()
        img, _ = pl.read_image()
    pick = [0, C - 1]
    ref = oracle.moff_image(np.ascontiguousarray(codes[:, pick]), gains[pick], pos, taps, N, 2)
    assert oracle.max_norm_err(img[pick], ref).max() <= 3e-3
    power = (np.abs(beams[:, :, 0].astype(np.complex128)) ** 2).sum(axis=0)
    np.testing.assert_allclose(power, img[:, :2, N // 5, N // 3], atol=1e-5 * img[:, :2].max(), rtol=0)


@pytest.mark.parametrize("A,N,P,K", [(64, 32, 1, 5), (300, 128, 2, 5), (700, 128, 2, 9), (700, 256, 2, 5), (3000, 256, 2, 9),
                                     (10000, 512, 2, 9)])
def test_wide_and_narrow_stripes_agree(monkeypatch, A, N, P, K):
    pos, taps, codes, gains = case(3, A, N, P, 2, 13, K=K)

    def image():
        with moff.Plan(pos, taps, N, 2, P) as pl:
            pl.set_gains(gains)
            pl.submit(codes)
            return pl.tuning(), pl.read_image()[0]

    monkeypatch.delenv("MOFF_GRID_WIDE", raising=False)
    wide, a = image()
    monkeypatch.setenv("MOFF_GRID_WIDE", "0")
    narrow, b = image()
    assert narrow["wide_rows"] == 0 and wide["wide_rows"] == 1
    np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("N,P", [(64, 1), (128, 2), (256, 2)])
@pytest.mark.parametrize("large", [False, True])
def test_scales_outside_fp32(N, P, large):
    """Gains and kernels so small (or large) together that the row-spectrum route's FP32 scale of a channel is 0 (or
    infinite): a fold that puts the product's bits together must not wrap its exponent.  The image is 0 (the true one lies
    below FP32's range), or nowhere finite."""
    A, C, T = 12, 2, 40
    pos, taps, codes, gains = case(N + 3, A, N, P, C, T)
    gains /= np.abs(gains)
    if large:
        gains, taps = gains * 1e30, taps * 1e15
    else:   # one antenna without signal sets the channel's scale, so that the others' sums are far below 1
        codes[:, :, 0] = 0
        gains, taps = gains * 2e-38, taps * 1e-12
        gains[:, 0] *= 5e5
    with moff.Plan(pos, taps.astype(np.complex64), N, C, P, fp16tc=True) as pl:
        assert pl.route() == "fp16_rowspec"
        pl.set_gains(gains.astype(np.complex64))
        pl.submit(codes)
        img, _ = pl.read_image()
    if large:
        assert not np.isfinite(img).any()
    else:
        assert np.array_equal(img, np.zeros_like(img))
