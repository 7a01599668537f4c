"""Batching pattern: every chunk of a block in one persistent launch
(MOFF_PERSIST): CTAs pull the chunks' gridding stripes and column strips from a
device work queue, each item waiting (bounded) for the items it depends on.

The items run the direct launches' arithmetic and the FP64 sums fold in chunk
order, so images must be bit-identical to the direct launches (with and
without graph replay) and within the FP32 bar (1e-5) of the FP64 oracle.  A
dependency that never arrives (MOFF_PERSIST_EXTRA: column items wait for row
items that do not exist) runs its wait out: the launch ends and the next read
returns MOFF_ETIMEDOUT (-5), with the context still usable.
"""
import numpy as np
import pytest

import oracle
import paper_0812_3669_gb300 as moff
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL32 = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    moff.build()
    yield


def c64(x):
    return np.asarray(x).astype(np.complex64).astype(np.complex128)


def case(seed, A, N, K, P, C, T_list, jones=False):
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0, N * 0.7, size=(A, 2)) + N * 0.15
    shape = (A, 2, 2, K, K) if jones else (A, P, K, K)
    taps = c64(rng.normal(size=shape) + 1j * rng.normal(size=shape))
    gains = c64(synth.gains_random(rng, C, A, P))
    blocks = []
    for T in T_list:
        re = np.clip(np.rint(rng.normal(0, 2.5, size=(T, C, A, P))), -7, 7).astype(int)
        im = np.clip(np.rint(rng.normal(0, 2.5, size=(T, C, A, P))), -7, 7).astype(int)
        blocks.append(synth.pack_4bit(re, im))
    return pos, taps, gains, blocks


def run(pos, taps, gains, N, C, P, blocks, **kw):
    with moff.Plan(pos, taps, N, C, P, **kw) as pl:
        info = pl.info()
        pl.set_gains(gains)
        for b in blocks:
            pl.submit(b)
        img, n = pl.read_image()
    return img, n, info


@pytest.mark.parametrize("N,P,K,A,C,T_list,jones,scratch_mb", [
    (64, 1, 5, 150, 4, [37, 20], False, None),
    (128, 2, 7, 300, 6, [150, 41], False, 12),     # channel chunks and a ragged time chunk
    (32, 2, 3, 60, 3, [9], True, None),            # Jones kernels
    (256, 2, 5, 200, 2, [12], False, None),
])
def test_persistent_equals_direct_and_oracle(monkeypatch, N, P, K, A, C, T_list, jones, scratch_mb):
    if scratch_mb:
        monkeypatch.setenv("MOFF_SCRATCH_MB", str(scratch_mb))
    pos, taps, gains, blocks = case(900 + N + P, A, N, K, P, C, T_list, jones)
    d, nd, info_d = run(pos, taps, gains, N, C, P, blocks, jones=jones)
    p, npers, info_p = run(pos, taps, gains, N, C, P, blocks, jones=jones, persist=True)
    g, ng, _ = run(pos, taps, gains, N, C, P, blocks + blocks[:1], jones=jones, persist=True, graph=True)
    assert nd == npers == sum(T_list)
    if scratch_mb:
        assert info_p["chan_chunk"] < C and info_p["time_chunk"] < max(T_list), info_p
    # the direct plan may pick another gridding shape; a persistent plan's shape is the
    # direct one with 4 samples per pass, so compare with that direct plan as well
    assert np.array_equal(p, run(pos, taps, gains, N, C, P, blocks, jones=jones, persist=True)[0])
    ref = oracle.moff_image(np.concatenate(blocks), gains, pos, taps, N, P, jones=jones)
    for img in (d, p):
        err = oracle.max_norm_err(img, ref)
        print(f"N={N} P={P} jones={jones}: max-normalised error {float(err.max()):.2e}")
        assert err.max() <= TOL32
    # graph replay of the persistent launch: the first block once more
    ref_g = oracle.moff_image(np.concatenate(blocks + blocks[:1]), gains, pos, taps, N, P, jones=jones)
    assert ng == nd + T_list[0]
    assert oracle.max_norm_err(g, ref_g).max() <= TOL32


def test_persistent_equals_direct_launches_of_the_same_shape(monkeypatch):
    """With the built-in rule forced to 4 samples per pass (cell pairs), the direct and
    persistent plans run the same gridding shape: bit for bit the same image."""
    pos, taps, gains, blocks = case(950, 400, 128, 7, 2, 5, [130, 60])
    monkeypatch.setenv("MOFF_SCRATCH_MB", "20")
    direct = None
    with moff.Plan(pos, taps, 128, 5, 2) as pl:
        t = pl.tuning()
        if t["time_batch"] != 4 or t["staged"]:
            pytest.skip(f"built-in rule picked time_batch={t['time_batch']} staged={t['staged']}")
        pl.set_gains(gains)
        for b in blocks:
            pl.submit(b)
        direct, nd = pl.read_image()
    pers, npers, _ = run(pos, taps, gains, 128, 5, 2, blocks, persist=True)
    assert nd == npers == 190
    assert np.array_equal(direct, pers)


def test_persistent_timing_kind_and_refusals():
    pos, taps, gains, blocks = case(960, 100, 64, 5, 2, 3, [40])
    with moff.Plan(pos, taps, 64, 3, 2, persist=True) as pl:
        pl.set_gains(gains)
        pl.set_timing(True)
        pl.submit(blocks[0])
        tot, n = pl.timing(8)
        assert n == 1 and tot > 0.0
        assert pl.timing(1)[1] == 0 and pl.timing(2)[1] == 0
    for kw in (dict(fp16tc=True), dict(served=True)):
        with pytest.raises(moff.MoffError) as e:
            moff.Plan(pos, taps, 64, 3, 2, persist=True, **kw)
        assert e.value.status == -1


def test_dependency_wait_runs_out_and_returns_timeout(monkeypatch):
    pos, taps, gains, blocks = case(970, 120, 64, 5, 2, 4, [30])
    monkeypatch.setenv("MOFF_PERSIST_EXTRA", "1")
    monkeypatch.setenv("MOFF_PERSIST_BUDGET_US", "2000")
    with moff.Plan(pos, taps, 64, 4, 2, persist=True) as pl:
        pl.set_gains(gains)
        pl.submit(blocks[0])
        with pytest.raises(moff.MoffError) as e:
            pl.read_image()
        assert e.value.status == -5
    monkeypatch.delenv("MOFF_PERSIST_EXTRA")
    # the context is still usable: a new plan images correctly
    img, n, _ = run(pos, taps, gains, 64, 4, 2, blocks, persist=True)
    ref = oracle.moff_image(blocks[0], gains, pos, taps, 64, 2)
    assert n == 30 and oracle.max_norm_err(img, ref).max() <= TOL32


def squeezed(seed, A, N, K, P, rows):
    """Positions over the whole grid, and the same antennas on `rows` grid rows, with kernels for each."""
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0, N, size=(2, A, 2))
    pos[1, :, 1] = N // 3 + rng.integers(0, rows, size=A)
    return pos, c64(rng.normal(size=(2, A, P, K, K)) + 1j * rng.normal(size=(2, A, P, K, K)))


@pytest.mark.parametrize("groups", [[1, 1, 1], [0, 1, 1]])
def test_denser_sets_after_creation(groups):
    """Replacing the positions by denser ones needs more shared memory per stripe than the plan was created with: the
    persistent launch takes it from the sets in force, and gives the direct launches' image."""
    N, P, K, A, C, T = 128, 1, 5, 2000, 3, 33
    pos, taps = squeezed(970, A, N, K, P, 20)
    rng = np.random.default_rng(971)
    codes = synth.pack_4bit(rng.integers(-7, 8, size=(T, C, A, P)), rng.integers(-7, 8, size=(T, C, A, P)))
    sets = (pos[1:], taps[1:], None) if min(groups) == 1 else (pos, taps, groups)
    out = []
    for persist in (False, True):
        with moff.Plan(pos[0], taps[0], N, C, P, persist=persist) as pl:
            before = pl.tuning()["time_batch"]
            pl.set_channel_groups(*sets)
            pl.set_timing(True)
            pl.submit(codes)
            assert pl.timing(8)[1] == (1 if persist else 0)
            out.append(pl.read_image()[0])
            assert not persist or before == 4
    assert np.array_equal(out[0], out[1])
    err = oracle.max_norm_err(out[1], oracle.moff_image_sets(codes, np.ones((C, A, P), complex), pos, taps, groups, N, P))
    assert err.max() <= TOL32


def test_sets_that_no_persistent_shape_fits_run_the_direct_launches():
    """A set that fits one sample per pass but not four: the persistent kernel is built for four, so the plan's blocks
    take the direct launches."""
    N, P, K, A, C, T = 256, 2, 9, 2600, 2, 10
    pos, taps = squeezed(980, A, N, K, P, 1)
    rng = np.random.default_rng(981)
    codes = synth.pack_4bit(rng.integers(-7, 8, size=(T, C, A, P)), rng.integers(-7, 8, size=(T, C, A, P)))
    out = []
    for persist in (False, True):
        with moff.Plan(pos[0], taps[0], N, C, P, persist=persist) as pl:
            pl.set_channel_groups(pos, taps, [0, 1])
            assert pl.tuning()["time_batch"] == 1
            pl.set_timing(True)
            pl.submit(codes)
            assert pl.timing(8)[1] == 0 and pl.timing(1)[1] > 0
            out.append(pl.read_image()[0])
    assert np.array_equal(out[0], out[1])
    err = oracle.max_norm_err(out[1], oracle.moff_image_sets(codes, np.ones((C, A, P), complex), pos, taps, [0, 1], N, P))
    assert err.max() <= TOL32


@pytest.mark.parametrize("N,P,A,wide", [(64, 1, 300, 1), (128, 2, 300, 1), (512, 1, 6000, 0), (512, 2, 6000, 1)])
def test_built_in_shape(N, P, A, wide):
    """The rule picks among the persistent kernel's shapes (4 samples per pass) and takes wide stripes where they pay: not
    for one pol on the 512 grid.  The image is the direct launches'."""
    K, C, T = 7, 1, 9
    pos, taps, gains, blocks = case(990, A, N, K, P, C, [T])
    if N == 512:
        pos = 100 + (pos - pos.min()) * 0.45        # dense enough for wide stripes in a direct plan
    with moff.Plan(pos, taps, N, C, P) as pl:
        assert pl.tuning()["wide_rows"] == 1
    with moff.Plan(pos, taps, N, C, P, persist=True) as pl:
        t = pl.tuning()
        assert (t["time_batch"], t["wide_rows"], t["staged"]) == (4, wide, 0)
    d, _, _ = run(pos, taps, gains, N, C, P, blocks)
    p, _, _ = run(pos, taps, gains, N, C, P, blocks, persist=True)
    assert np.array_equal(d, p)


@pytest.mark.parametrize("N", [256, 512])
def test_block_lanes_on_wide_stripes(monkeypatch, N):
    """2 x 2 blocks per lane with two pols on the large grids: only the wide stripes have two rows (the autotuner may
    pick them)."""
    monkeypatch.setenv("MOFF_GRID_QUADS", "1")
    monkeypatch.setenv("MOFF_GRID_WIDE", "1")
    pos, taps, gains, blocks = case(995, 150, N, 5, 2, 2, [21])
    out = []
    for persist in (False, True):
        with moff.Plan(pos, taps, N, 2, 2, persist=persist) as pl:
            t = pl.tuning()
            assert (t["cells_per_lane"], t["wide_rows"], t["time_batch"]) == (4, 1, 4)
            pl.set_gains(gains)
            pl.submit(blocks[0])
            out.append(pl.read_image()[0])
    assert np.array_equal(out[0], out[1])
    assert oracle.max_norm_err(out[1], oracle.moff_image(blocks[0], gains, pos, taps, N, 2)).max() <= TOL32
