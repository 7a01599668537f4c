"""Performance cases of the imaging library: the calls a user's program makes, over the range of sizes it makes them at.

Each case is one array with its plan, a block of device-resident input and one pass through the public entry points
(submit a block, read the image sums back into a device buffer and start the next integration).  Array layouts, kernel
sizes, grids, channel counts and block lengths are those of the repository's workloads: the tiny uniform array, the
dual-pol hexagonal core with and without its polyphase filter bank, the filled aperture, the wide-field Jones lattice
and the sub-arrays of the serving mix.  Fields of a case:

    entry   "submit" (4-bit voltages), "adc" (F-stage first), "calibrate" (submit with calibrator pixel, beams and
            autocorrelations) or "serve" (several sub-arrays through one server)
    prec    "fp32" or "fp16" (the tensor-core plan flag)
    layout  "uniform", "hex" or "lattice"; ``A`` antennas on an ``N`` x ``N`` grid, ``K`` x ``K`` kernels, ``P`` pols
    C, T    channels and samples of the block
"""
import math

import numpy as np
import torch

import paper_0812_3669_gb300 as moff

N_PFB_TAPS = 8
BEAMS = ((3, 5), (17, 120), (64, 64), (101, 9))
CALIBRATOR = (37, 90)
SERVER_BYTES = 24 << 30


def _case(name, **kw):
    c = dict(name=name, entry="submit", prec="fp32", layout="lattice", K=7, P=2, jones=False, graph=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: the 64-antenna single-pol array, one shared 3 x 3 kernel; launches and waits count
        _case("tiny_fp32", layout="uniform", A=64, N=32, K=3, P=1, C=16, T=256, graph=True),
        # a short block of the smallest serving sub-array on the reduced-precision route
        _case("subarray256_fp16", prec="fp16", A=256, N=64, C=64, T=100),
        # a serving sub-array too dense for the reduced-precision routes on its grid; ragged block length
        _case("dense128_fp32", A=4096, N=128, C=64, T=300),
        # the dual-pol core on the default (FP32) path: one 1000-sample integration replayed as a graph
        _case("dualpol_fp32", layout="hex", A=1024, N=128, C=64, T=1000, graph=True),
        # the same core on the reduced-precision row-spectrum route
        _case("dualpol_fp16", prec="fp16", layout="hex", A=1024, N=128, C=256, T=1000),
        # the same core from 8-bit ADC streams: 1024-channel filter bank, then imaging
        _case("dualpol_adc_fp16", entry="adc", prec="fp16", layout="hex", A=1024, N=128, C=1024, T=96),
        # a dense serving sub-array on the 256 grid, odd block length
        _case("dense256_fp16", prec="fp16", A=4096, N=256, C=96, T=333),
        # the filled aperture on the FP32 path
        _case("filled512_fp32", A=16384, N=512, C=8, T=100),
        # the filled aperture on the tensor-core gridding route, ragged second chunk
        _case("filled512_fp16", prec="fp16", A=16384, N=512, C=24, T=250),
        # the wide-field lattice with Jones kernels and a w-phase (x extent wraps the grid): the largest array
        _case("widefield_fp16", prec="fp16", A=32768, N=512, K=9, jones=True, C=24, T=256),
        # calibration and beam-forming beside the imaging: every per-sample tap in use
        _case("calibrate_fp32", entry="calibrate", layout="hex", A=1024, N=128, C=32, T=200),
        # a request stream: blocks of uneven sub-arrays admitted by one server, reduced and full precision mixed
        _case("serving_mix", entry="serve", A=16384, N=512, C=64, T=100, prec="mixed"),
    ]


def _subarrays(case):
    """The sub-arrays of a served stream: the case's own largest array and three smaller ones."""
    N, A, C, T = case["N"], case["A"], case["C"], case["T"]
    mk = lambda prec, a, n, c, t: _case("", prec=prec, A=a, N=n, C=c, T=t)
    return [
        mk("fp16", A, N, max(1, C // 8), T),
        mk("fp16", max(256, A // 4), N // 2, C, T + 57),
        mk("fp16", max(64, A // 16), max(64, N // 4), 2 * C, 3 * T),
        mk("fp32", max(64, A // 64), max(64, N // 8), C, 2 * T + 31),
    ]


def draw(rng):
    """One more case of the listed ones' ranges (serving channel counts, block lengths and grids; odd sizes)."""

    def lg(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    top = max((work(c)["flops"], work(c)["bytes"]) for c in listed())
    while True:
        kind = rng.choice(["tiny", "sparse16", "sparse32", "adc", "dense16", "dense32", "wide", "calibrate", "serve"])
        if kind == "tiny":
            c = _case("", layout="uniform", A=lg(16, 64), N=rng.choice([32, 64]), K=rng.choice([1, 3, 5]),
                      P=rng.choice([1, 2]), C=lg(1, 64), T=lg(16, 512), graph=rng.random() < 0.5)
        elif kind in ("sparse16", "sparse32"):
            n = rng.choice([64, 128, 128, 256])
            c = _case("", prec="fp16" if kind == "sparse16" else "fp32", layout=rng.choice(["hex", "lattice"]),
                      A=lg(100, {64: 256, 128: 1024, 256: 1024}[n]), N=n, K=rng.choice([5, 7]), P=rng.choice([1, 2, 2]),
                      C=lg(16, 1024), T=lg(50, 1000), graph=rng.random() < 0.3)
        elif kind == "adc":
            c = _case("", entry="adc", prec=rng.choice(["fp16", "fp32"]), layout="hex", A=lg(100, 1024), N=128,
                      C=rng.choice([256, 512, 1024, 1024]), T=lg(16, 96))
        elif kind == "dense16":
            n = rng.choice([256, 512])
            c = _case("", prec="fp16", A=lg(3000 if n == 256 else 9000, 4096 if n == 256 else 16384), N=n,
                      K=rng.choice([5, 7]), P=2, C=lg(4, 96 if n == 256 else 24), T=lg(100, 333))
        elif kind == "dense32":
            n = rng.choice([128, 256, 512])
            c = _case("", A=lg(1000, {128: 4096, 256: 8000, 512: 16384}[n]), N=n, C=lg(4, 64 if n < 512 else 8),
                      T=lg(50, 300))
        elif kind == "wide":
            c = _case("", prec="fp16", A=256 * rng.randint(64, 128), N=512, K=rng.choice([7, 9]), jones=True, C=lg(4, 24),
                      T=lg(100, 256))
        elif kind == "calibrate":
            c = _case("", entry="calibrate", layout=rng.choice(["hex", "lattice"]), A=lg(100, 1024), N=128, C=lg(8, 64),
                      T=lg(50, 300))
        else:
            c = _case("", entry="serve", A=16384, N=512, C=8 * rng.randint(2, 8), T=lg(50, 100), prec="mixed")
        w = work(c)
        out_mb = c["C"] * (4 if c["P"] == 2 else 1) * c["N"] ** 2 * 4 / 1e6
        if (w["flops"], w["bytes"]) <= top and out_mb <= 270 and w["bytes"] < 6e9:
            del c["name"]
            return c


# ------------------------------------------------------------------------------------------------ inputs

def _rng(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) % (1 << 62))
    return g


def _positions(case, seed):
    """Antenna positions in cells of half a wavelength (float64, CUDA)."""
    A, N = case["A"], case["N"]
    g = _rng(seed, 1)
    if case["layout"] == "uniform":            # at least one wavelength (2 cells) apart: jittered 2-cell raster
        n = N // 2
        cells = torch.randperm(n * n, generator=g, device="cuda")[:A]
        return torch.stack([cells % n, cells // n], 1).double() * 2 + 0.3 * torch.randn((A, 2), generator=g, device="cuda",
                                                                                        dtype=torch.float64)
    if case["layout"] == "hex":                # the A points of a 1.5-wavelength hexagonal lattice nearest the centre
        m = int(math.ceil(math.sqrt(A))) + 4
        jj, ii = torch.meshgrid(torch.arange(-m, m + 1, device="cuda"), torch.arange(-m, m + 1, device="cuda"), indexing="ij")
        x = ((ii + 0.5 * (jj % 2)) * 3.0).double().flatten()
        y = (jj * (math.sqrt(3.0) / 2) * 3.0).double().flatten()
        near = torch.argsort(x * x + y * y + 1e-6 * x + 1e-9 * y)[:A]
        p = torch.stack([x[near], y[near]], 1) + N / 2.0
        return p + 0.15 * torch.randn((A, 2), generator=g, device="cuda", dtype=torch.float64)
    if case["jones"]:                          # 256 antennas along x at one wavelength: the extent wraps the grid
        nx, ny = 256, (A + 255) // 256
        ox, oy = 0.0, N / 2.0 - ny
    else:
        nx = ny = int(math.ceil(math.sqrt(A)))
        ox = oy = N / 2.0 - nx
    k = torch.arange(A, device="cuda")
    p = torch.stack([(k % nx).double() * 2 + ox, (k // nx).double() * 2 + oy], 1)
    return p + 0.1 * torch.randn((A, 2), generator=g, device="cuda", dtype=torch.float64)


def _taps(case, pos, seed):
    """Gridding kernels, complex64 on the GPU: [A][P][K][K], or [A][2][2][K][K] for Jones kernels."""
    A, K, P = case["A"], case["K"], case["P"]
    g = _rng(seed, 2)
    uni = lambda shape, lo, hi: lo + (hi - lo) * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)
    d = torch.arange(K, device="cuda", dtype=torch.float64) - K // 2
    if case["layout"] == "uniform":            # one real Gaussian kernel shared by all antennas
        k = torch.exp(-(d[:, None] ** 2 + d[None, :] ** 2) / (2 * 0.5 ** 2))
        return (k / k.sum()).to(torch.complex64).expand(A, P, K, K).contiguous()
    off = torch.floor(pos + 0.5) - pos
    dx = d[None, None, :] + off[:, 0, None, None]
    dy = d[None, :, None] + off[:, 1, None, None]
    sigma = 1.5 if case["jones"] else 1.2
    b = torch.exp(-(dx ** 2 + dy ** 2) / (2 * sigma ** 2))
    b = b / b.sum((1, 2), keepdim=True)
    if not case["jones"]:
        ph = (uni((A, P, 1, 1), 0, 2 * math.pi) + uni((A, P, 1, 1), -0.3, 0.3) * d[None, None, None, :]
              + uni((A, P, 1, 1), -0.3, 0.3) * d[None, None, :, None])
        return (b[:, None] * torch.exp(1j * ph)).to(torch.complex64)
    h = K // 2 + 1
    s = uni((A, 2, 1, 1), -1, 1) + uni((A, 2, 1, 1), -1, 1) * (dx / h)[:, None] + uni((A, 2, 1, 1), -1, 1) * (dy / h)[:, None]
    leak = 0.05 * torch.exp(1j * uni((A, 2, 1, 1), 0, 2 * math.pi))
    w = torch.exp(1j * uni((A, 1, 1), -0.3, 0.3) * (dx ** 2 + dy ** 2))
    J = torch.empty((A, 2, 2, K, K), dtype=torch.complex128, device="cuda")
    J[:, 0, 0] = b * (1 + 0.1 * s[:, 0])
    J[:, 1, 1] = b * (1 + 0.1 * s[:, 1])
    J[:, 0, 1] = b * leak[:, 0]
    J[:, 1, 0] = b * leak[:, 1]
    return (J * w[:, None, None]).to(torch.complex64)


def _gains(case, seed):
    shape = (case["C"], case["A"], case["P"])
    g = _rng(seed, 3)
    amp = 0.8 + 0.4 * torch.rand(shape, generator=g, device="cuda")
    return torch.polar(amp, 2 * math.pi * torch.rand(shape, generator=g, device="cuda"))


def _codes(case, pos, seed):
    """4-bit voltages: receiver noise of sigma 2 and two point sources, rounded and clipped to [-7, 7]."""
    T, C, A, P, N = case["T"], case["C"], case["A"], case["P"], case["N"]
    g = _rng(seed, 4)
    out = torch.empty((T, C, A, P), dtype=torch.uint8, device="cuda")
    src = torch.randint(0, N, (2, 2), generator=g, device="cuda").double()
    ph = torch.exp(-2j * math.pi * (pos @ src.T) / N).to(torch.complex64)      # [A][2 sources]
    step = max(1, (1 << 26) // (C * A * P))
    for t in range(0, T, step):
        n = min(step, T - t)
        v = 2.0 * torch.view_as_complex(torch.randn((n, C, A, P, 2), generator=g, device="cuda"))
        for k in range(2):
            v += torch.randn((n, C, 1, P), generator=g, device="cuda", dtype=torch.complex64) * ph[:, k, None]
        q = torch.view_as_real(v).round_().clamp_(-7, 7).to(torch.int16)
        out[t:t + n] = (((q[..., 0] & 15) << 4) | (q[..., 1] & 15)).to(torch.uint8)
    return out


def _adc(case, seed):
    """8-bit ADC streams [A][P][S]: Gaussian noise of sigma 20 and one tone."""
    S = (case["T"] + N_PFB_TAPS - 1) * 2 * case["C"]
    g = _rng(seed, 5)
    out = torch.empty((case["A"], case["P"], S), dtype=torch.int8, device="cuda")
    tone = 8.0 * torch.cos(2 * math.pi * 0.2123 * torch.arange(S, device="cuda", dtype=torch.float64)).float()
    step = max(1, (1 << 26) // (case["P"] * S))
    for a in range(0, case["A"], step):
        n = min(step, case["A"] - a)
        x = 20.0 * torch.randn((n, case["P"], S), generator=g, device="cuda") + tone
        out[a:a + n] = x.round_().clamp_(-127, 127).to(torch.int8)
    return out


def _pfb_coeffs(C):
    """Hann-windowed sinc of the 8-tap filter bank, float32 [8 M], and the scale that leaves noise at sigma 2."""
    M = 2 * C
    n = np.arange(N_PFB_TAPS * M, dtype=np.float64)
    L = N_PFB_TAPS * M - 1
    h = np.sinc((n - L / 2) / M) * (0.5 - 0.5 * np.cos(2 * np.pi * n / L))
    return h.astype(np.float32), float(np.float32(2.0 / (20.0 * math.sqrt(float((h ** 2).sum()) / 2))))


def _array(case, seed):
    pos = _positions(case, seed)
    return pos, _taps(case, pos, seed)


# ------------------------------------------------------------------------------------------------ prepare and run

def _plan(case, pos, taps, seed, served=False):
    p = moff.Plan(pos.cpu().numpy(), taps.cpu().numpy(), case["N"], case["C"], case["P"], jones=case["jones"],
                  fp16tc=case["prec"] == "fp16", fstage=case["entry"] == "adc", graph=case["graph"], served=served)
    p.set_gains(_gains(case, seed))
    return p


def _image_buffer(case):
    return torch.empty((case["C"], 4 if case["P"] == 2 else 1, case["N"], case["N"]), dtype=torch.float32, device="cuda")


def prepare(case, seed):
    if case["entry"] == "serve":
        subs = _subarrays(case)
        st = {"case": case, "server": moff.Server(SERVER_BYTES, 4), "plans": [], "codes": [], "images": []}
        for k, sub in enumerate(subs):
            pos, taps = _array(sub, seed + k)
            st["plans"].append(_plan(sub, pos, taps, seed + k, served=True))
            st["codes"].append(_codes(sub, pos, seed + k))
            st["images"].append(_image_buffer(sub))
        torch.cuda.synchronize()
        return st
    pos, taps = _array(case, seed)
    st = {"case": case, "plan": _plan(case, pos, taps, seed), "image": _image_buffer(case)}
    if case["entry"] == "adc":
        h, scale = _pfb_coeffs(case["C"])
        st["plan"].set_fstage(N_PFB_TAPS, h, scale)
        st["adc"] = _adc(case, seed)
    else:
        st["codes"] = _codes(case, pos, seed)
    if case["entry"] == "calibrate":
        st["plan"].set_calibrator(*CALIBRATOR)
        st["plan"].set_beams([b[0] for b in BEAMS], [b[1] for b in BEAMS])
        st["plan"].set_autocorr(True)
        st["cross"] = _image_buffer(case)
    torch.cuda.synchronize()
    return st


def _parts(image):
    """The whole image as views of at most 2^24 elements (several outputs instead of a very large one)."""
    per = max(1, (1 << 24) // image[0].numel())
    return [image[c:c + per] for c in range(0, image.shape[0], per)]


def run(state):
    case = state["case"]
    if case["entry"] == "serve":
        for p, codes in zip(state["plans"], state["codes"]):
            state["server"].submit(p, codes)
        state["server"].wait()
        out = []
        for p, image in zip(state["plans"], state["images"]):
            p.read_image(reset=True, out=image)
            out += _parts(image)
        return out
    plan = state["plan"]
    if case["entry"] == "adc":
        plan.submit_adc(state["adc"])
    else:
        plan.submit(state["codes"])
    if case["entry"] == "calibrate":
        corr, power, _ = plan.read_feedback(reset=True)
        beams = plan.read_beams()
        plan.read_image_cross(out=state["cross"])
        plan.read_image(reset=True, out=state["image"])
        return [corr, power, beams, state["cross"]] + _parts(state["image"])
    plan.read_image(reset=True, out=state["image"])
    return _parts(state["image"])


# ------------------------------------------------------------------------------------------------ work

def work(case):
    """Bytes: inputs (voltages or ADC samples, gains) and outputs once.  Operations: weights (6 per voltage), kernel
    taps (8 per complex multiply-add), the 2D transform (5 n log2 n) and the products, FIR and transform of the F-stage."""
    if case["entry"] == "serve":
        w = [work(s) for s in _subarrays(case)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    A, P, N, K, C, T = (case[k] for k in ("A", "P", "N", "K", "C", "T"))
    snap = C * T
    flops = snap * (6 * A * P + 8 * A * P * K * K * (2 if case["jones"] else 1) + P * 10 * N * N * math.log2(N)
                    + (16 if P == 2 else 4) * N * N)
    image = 4 * C * (4 if P == 2 else 1) * N * N
    nbytes = 8 * C * A * P + image
    if case["entry"] == "adc":
        M = 2 * C
        nbytes += A * P * (T + N_PFB_TAPS - 1) * M
        flops += A * P * T * (2 * N_PFB_TAPS * M + 5 * C * math.log2(C) + 16 * C)
    else:
        nbytes += snap * A * P
    if case["entry"] == "calibrate":
        nbytes += image + 8 * C * A * P + 8 * C * P + 8 * T * C * len(BEAMS) * P
        flops += snap * A * P * (8 + 7)
    return {"bytes": int(nbytes), "flops": int(flops)}


# ------------------------------------------------------------------------------------------------ exact

def _operator(case, pos, taps):
    """The gridding operator as a sparse complex128 matrix [P N N][A P]."""
    A, P, N, K = case["A"], case["P"], case["N"], case["K"]
    anchor = torch.floor(pos + 0.5).long()
    d = torch.arange(K, device="cuda") - K // 2
    ix = (anchor[:, 0, None] + d) % N
    iy = (anchor[:, 1, None] + d) % N
    cell = iy[:, :, None] * N + ix[:, None, :]                                   # [A][K][K]
    a = torch.arange(A, device="cuda")[:, None, None].expand(A, K, K)
    rows, cols, vals = [], [], []
    for po in range(P):
        for pi in range(P):
            if case["jones"] or po == pi:
                rows.append((po * N * N + cell).flatten())
                cols.append((a * P + pi).flatten())
                vals.append((taps[:, po, pi] if case["jones"] else taps[:, po]).reshape(-1).to(torch.complex128))
    m = torch.sparse_coo_tensor(torch.stack([torch.cat(rows), torch.cat(cols)]), torch.cat(vals), (P * N * N, A * P))
    return m.coalesce().to_sparse_csr()


def _unpack64(codes):
    b = codes.to(torch.int16)
    s = lambda u: (u - ((u & 8) << 1)).double()
    return torch.complex(s((b >> 4) & 15), s(b & 15))


def _codes64(case, seed):
    """The F-stage in 64 bits: 4-bit codes [T][C][A][P] of the ADC streams, round half to even."""
    T, C, A, P = case["T"], case["C"], case["A"], case["P"]
    M = 2 * C
    h, scale = _pfb_coeffs(C)
    h = torch.from_numpy(h).cuda().double().reshape(N_PFB_TAPS, M)
    adc = _adc(case, seed)
    out = torch.empty((T, C, A, P), dtype=torch.uint8, device="cuda")
    for a in range(0, A, 64):
        x = adc[a:a + 64].double().reshape(-1, P, T + N_PFB_TAPS - 1, M)
        s = sum(h[p] * x[:, :, p:p + T] for p in range(N_PFB_TAPS))
        X = torch.fft.rfft(s, dim=-1)[..., :C] * scale                           # [a][P][T][C]
        q = torch.view_as_real(X).round().clamp(-7, 7).to(torch.int16)
        out[:, :, a:a + 64] = (((q[..., 0] & 15) << 4) | (q[..., 1] & 15)).to(torch.uint8).permute(2, 3, 0, 1)
    return out


def _exact_one(case, seed):
    N, P, C, T, A = (case[k] for k in ("N", "P", "C", "T", "A"))
    pos, taps = _array(case, seed)
    op = _operator(case, pos, taps)
    gains = _gains(case, seed).to(torch.complex128)
    codes = _codes64(case, seed) if case["entry"] == "adc" else _codes(case, pos, seed)
    image = torch.zeros((C, 4 if P == 2 else 1, N, N), dtype=torch.float64, device="cuda")
    cal = case["entry"] == "calibrate"
    if cal:
        khat = torch.empty((A, P, N * N), dtype=torch.complex128, device="cuda")   # every antenna's kernel on the sky
        dense = torch.zeros((P * N * N, 64), dtype=torch.complex128, device="cuda")
        for a in range(0, A, 64):
            n = min(64, A - a)
            for p in range(P):
                pick = torch.zeros((A * P, n), dtype=torch.complex128, device="cuda")
                pick[(a + torch.arange(n, device="cuda")) * P + p, torch.arange(n, device="cuda")] = 1
                col = (op @ pick).reshape(P, N, N, n)[p].permute(2, 0, 1)
                khat[a:a + n, p] = torch.fft.ifft2(col, norm="forward").reshape(n, N * N)
        del dense
        pix = CALIBRATOR[1] * N + CALIBRATOR[0]
        corr = torch.empty((C, A, P), dtype=torch.complex128, device="cuda")
        power = torch.empty((C, P), dtype=torch.float64, device="cuda")
        beams = torch.empty((T, C, len(BEAMS), P), dtype=torch.complex128, device="cuda")
        cross = torch.empty_like(image)
    step = max(1, (1 << 25) // (P * N * N))
    for c in range(C):
        y = (_unpack64(codes[:, c]) * gains[c]).reshape(T, A * P)
        field = torch.empty((T, P), dtype=torch.complex128, device="cuda") if cal else None
        for t in range(0, T, step):
            E = torch.fft.ifft2((op @ y[t:t + step].T.contiguous()).reshape(P, N, N, -1).permute(3, 0, 1, 2), norm="forward")
            image[c, 0] += (E[:, 0].abs() ** 2).sum(0)
            if P == 2:
                image[c, 1] += (E[:, 1].abs() ** 2).sum(0)
                xy = (E[:, 0] * E[:, 1].conj()).sum(0)
                image[c, 2] += xy.real
                image[c, 3] += xy.imag
            if cal:
                field[t:t + step] = E[:, :, CALIBRATOR[1], CALIBRATOR[0]]
                for k, (bx, by) in enumerate(BEAMS):
                    beams[t:t + step, c, k] = E[:, :, by, bx]
        if cal:
            y = y.reshape(T, A, P)
            corr[c] = khat[:, :, pix].conj() * torch.einsum("tp,tap->ap", field, y.conj())
            power[c] = (field.abs() ** 2).sum(0)
            auto = [torch.einsum("a,an->n", (y[:, :, p] * y[:, :, q].conj()).sum(0), khat[:, p] * khat[:, q].conj())
                    .reshape(N, N) for p, q in ((0, 0), (1, 1), (0, 1))]
            cross[c] = image[c] - torch.stack([auto[0].real, auto[1].real, auto[2].real, auto[2].imag])
    if cal:
        return [corr, power, beams, cross] + _parts(image)
    return _parts(image)


def exact(case, seed):
    if case["entry"] == "serve":
        out = []
        for k, sub in enumerate(_subarrays(case)):
            out += _exact_one(sub, seed + k)
        return out
    return _exact_one(case, seed)
