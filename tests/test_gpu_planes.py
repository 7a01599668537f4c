"""The voltage-plane kernels at the edges of their dispatch: every plane value is the decoded voltage times the
channel's power of two exactly (unit gains), whatever kernel makes it -- 32 staged samples per CTA (odd voltage counts,
rows past the last voltage, block lengths that are no multiple of 32), one thread per row in raster order, and 8 or 16
staged samples for large arrays in another order."""
import numpy as np
import pytest

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


# (antennas, grid, pols, shuffled): A P of 33 and 66 (not whole 16-byte pieces), 2560 and 2562 (either side of the raster
# rule), 6112 and 6144 (either side of the largest staged block), in the lattice's order or another
@pytest.mark.parametrize("A,N,P,shuffle", [(33, 64, 1, False), (33, 64, 2, True), (1280, 256, 2, False), (1281, 256, 2, False),
                                           (1296, 256, 2, False), (3056, 256, 2, True), (3072, 256, 2, True)])
@pytest.mark.parametrize("T", [1, 33, 128])
def test_planes_are_the_decoded_voltages(monkeypatch, A, N, P, shuffle, T):
    if N == 256:
        monkeypatch.setenv("MOFF_TC_DFT", "1")
    rng = np.random.default_rng(A + T)
    nx = int(np.ceil(np.sqrt(A)))
    pos = synth.positions_lattice(rng, nx, nx, 1.0, 0.05, (N / 2 - nx, N / 2 - nx))[:A]
    if shuffle:
        pos = pos[rng.permutation(A)]
    taps = synth.taps_gaussian(rng, pos, 5, 1.2, n_pol=P).astype(np.complex64)
    re, im = (rng.integers(-8, 8, size=(T, 2, A, P)) for _ in range(2))
    with moff.Plan(pos, taps, N, 2, P, fp16tc=True) as pl:
        pl.set_gains(np.ones((2, A, P), dtype=np.complex64))
        planes, scale = pl.voltage_planes(synth.pack_4bit(re, im), 1)
    assert scale == 512.0
    np.testing.assert_array_equal(planes.real, 512.0 * re[:, 1])
    np.testing.assert_array_equal(planes.imag, 512.0 * im[:, 1])
