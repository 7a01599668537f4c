"""The column kernel's role pipeline (k_cols_pipe) and its FP64 fold, at the block lengths where a ring of
four strips and double-buffered accumulators can go wrong, on both grids, both widths and both pol counts.

The tolerance against the FP64 oracle is the reduced-precision route's (3e-3 max-normalised, see
test_gpu_dft.py).  Scaling the gains by a power of two changes no rounding anywhere (every FP16 scale is a power
of two chosen from the gains), so the image scales by its square exactly: that pins the fold's exponent arithmetic.
"""
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


def case(seed, A, N, P, C, T, K=5):
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0, 0.6 * N, size=(A, 2)) + 0.33 * N          # some rows out of reach, some windows wrapping
    taps = (rng.normal(size=(A, P, K, K)) + 1j * rng.normal(size=(A, P, K, K))).astype(np.complex64).astype(np.complex128)
    codes = synth.pack_4bit(rng.integers(-8, 8, size=(T, C, A, P)), rng.integers(-8, 8, size=(T, C, A, P)))
    gains = synth.gains_random(rng, C, A, P).astype(np.complex64).astype(np.complex128)
    return pos, taps, codes, gains


def image(pos, taps, N, codes, gains):
    T, C, A, P = codes.shape
    with moff.Plan(pos, taps, N, C, P, fp16tc=True) as pl:
        assert pl.route() == "fp16_tcgrid"
        pl.set_gains(gains)
        pl.submit(np.ascontiguousarray(codes))
        img, n = pl.read_image()
    assert n == T
    return img


@pytest.mark.parametrize("N,width", [(512, 8), (256, 8), (256, 16)])
@pytest.mark.parametrize("P", [1, 2])
@pytest.mark.parametrize("T", [1, 2, 4, 5, 129])
def test_block_lengths(monkeypatch, N, width, P, T):
    monkeypatch.setenv("MOFF_TC_DFT", "1")
    monkeypatch.setenv("MOFF_COLS_W", str(width))
    pos, taps, codes, gains = case(31 + T + P, 90, N, P, 2, T)
    img = image(pos, taps, N, codes, gains)
    assert np.isfinite(img).all()
    assert oracle.max_norm_err(img, oracle.moff_image(codes, gains, pos, taps, N, P)).max() <= 3e-3


@pytest.mark.parametrize("shift", [-30, 30])
def test_power_of_two_gains_scale_exactly(monkeypatch, shift):
    monkeypatch.setenv("MOFF_TC_DFT", "1")
    pos, taps, codes, gains = case(77, 90, 256, 2, 1, 6)
    a = image(pos, taps, 256, codes, gains)
    b = image(pos, taps, 256, codes, gains * 2.0 ** shift)
    assert np.array_equal(b, np.ldexp(a, 2 * shift))


@pytest.mark.parametrize("N,P,C", [(256, 1, 64), (256, 2, 64), (512, 1, 16), (512, 2, 16)])
def test_hand_overs_hold_over_full_waves(monkeypatch, N, P, C):
    """One pol of one stage-1 tile (the 256 grid at 8 columns per CTA) leaves four of the twiddle warps without
    rows; they must not stand in for the four that write the operand.  Several waves of CTAs, blocks of
    four launches of 128 samples, repeated: the images equal each other bit for bit, and those of 16 columns per CTA (on
    the 512 grid a kernel of its own, without roles), whose arithmetic and order of sums are the same."""
    monkeypatch.setenv("MOFF_TC_DFT", "1")
    T = 512
    pos, taps, codes, gains = case(5 + P, 90, N, P, C, T)
    dev = torch.from_numpy(codes).cuda()
    images = {}
    for width in (8, 16):
        monkeypatch.setenv("MOFF_COLS_W", str(width))
        with moff.Plan(pos, taps, N, C, P, fp16tc=True) as pl:
            assert pl.route() == "fp16_tcgrid" and pl.dft_tuning()["cols_width"] == width
            pl.set_gains(gains)
            images[width] = []
            for _ in range(6):
                pl.submit(dev)
                images[width].append(pl.read_image(reset=True)[0])
    for width in (8, 16):
        for img in images[width]:
            assert np.array_equal(img, images[16][0])
    pick = [0, C - 1]
    ref = oracle.moff_image(np.ascontiguousarray(codes[:, pick]), gains[pick], pos, taps, N, P)
    assert oracle.max_norm_err(images[8][0][pick], ref).max() <= 3e-3
