// moff_dft_kernels.cu -- the row and column transforms of Eq. m6 step 3 (Morales, arXiv
// 0812.3669) as factored DFT contractions on the tensor cores, the columns fused with step 4
// (|E|^2 and the cross-pol products summed over a chunk, then added to the FP64
// accumulators), for the dense FP16 path.  (The FP32 gather's row transform runs inside the
// gridding kernel: k_grid_rows_dft, moff_dft.cuh.)
//
//   k_rows_dft8  one CTA = a stripe of grid rows of one channel walking a chunk of samples.
//   k_cols_pipe  one CTA = 8 (or 16) columns of one channel walking a chunk of samples, each
//                step on warps of its own.
//   k_cols_dft   the same work with block barriers between the steps: 16 columns on the 512
//                grid, whose accumulators leave no TMEM for a second buffer.  Per sample: the FP16
//                field's strip (cp.async) lands as the stage-1 A operand (rows (b, x), k = (a,
//                re/im)); stage 1 on the tensor cores; the twiddled FP32 result is written back as
//                the stage-2 A operand (128-byte swizzled, rows (c, x)); stage 2 leaves E in TMEM,
//                where the epilogue squares and sums it.  Loads of sample t + 1 and stage 1 of
//                sample t run while the epilogue of sample t - 1 works.
#include <cuda_fp16.h>

#include <cmath>
#include <cstdlib>
#include <cstring>

#include "moff_dft.cuh"
#include "moff_fft.cuh"
#include "moff_internal.h"
#include "moff_tc.cuh"

namespace moff {
namespace {

// exp(2 pi i m / L) with the angle reduced exactly (m mod L), in FP64.
void unit_root(long long m, long long L, double *c, double *s) {
    long long r = m % L;
    if (r < 0) r += L;
    const double ang = 2.0 * 3.14159265358979323846264338327950288 * (double)r / (double)L;
    *c = std::cos(ang);
    *s = std::sin(ang);
}

// Byte offset of element (n, k) of a K-major operand image with K columns
// (8 x 8 core matrices of 128 bytes; along K 128 bytes apart, along rows (K/8) * 128).
size_t kmajor_at(int n, int k, int K) {
    return (size_t)(n >> 3) * (K >> 3) * 128 + (size_t)(k >> 3) * 128 + (n & 7) * 16 + (k & 7) * 2;
}

template <int N, int P, int W>
struct ColDftShape {
    using S = DftShape<N>;
    static_assert(W == 8 || W == 16, "columns per CTA");
    static constexpr int N2 = S::N2;
    static constexpr int H = W / 8;                    // 16-byte pieces per (pol, row, re/im) of the strip
    static constexpr int M1 = W * N2;                  // stage-1 rows per pol: m = W b + x
    static constexpr int T1 = M1 / 128;
    static constexpr int MH = S::K1 * 128;             // stage-1 A: bytes of 64 rows m (128-byte swizzled)
    static constexpr int A1P = M1 * S::K1 * 2;         // bytes of one pol's stage-1 A
    static constexpr int M2 = 16 * W;                  // stage-2 rows per pol: m2 = 8 W c_hi + 8 x + c_lo
    static constexpr int T2 = M2 / 128;
    static constexpr int A2P = M2 * S::K2 * 2;         // bytes of one pol's stage-2 A (128-byte swizzled)
    static constexpr int D1 = P * T1 * S::C1;          // TMEM columns: stage-1 accumulators
    static constexpr int D2 = P * T2 * S::C2;          // then stage-2 accumulators
    static constexpr int TC_ = D1 + D2;
    static constexpr int TCOLS = TC_ <= 32 ? 32 : (TC_ <= 64 ? 64 : (TC_ <= 128 ? 128 : (TC_ <= 256 ? 256 : 512)));
    static constexpr int NPIECE = P * N * 2 * H;       // 16-byte pieces per sample: (p, ry, re/im, h)
    static constexpr int ITER = NPIECE / kBlock;
    static constexpr int ROWS_K = kBlock / (2 * H);    // grid rows covered by one piece round of the block
    // warp groups per stage-2 tile: with one tile (W = 8) the two groups split the d range
    static constexpr int DSPLIT = 2 / T2;
    static constexpr int ND = N2 / DSPLIT;             // d values per thread
    static constexpr size_t SMEM = 1024 + (size_t)P * A2P + 2 * (size_t)P * A1P + S::TAB_BYTES + 32;
    static_assert(T2 >= 1 && T2 <= 2 && T1 >= 1 && TC_ <= 512 && NPIECE % kBlock == 0 && ITER <= 32 && ND % 8 == 0 &&
                      (2 * H * N) % kBlock == 0 && ROWS_K % N2 == 0 && SMEM <= 225 * 1024,
                  "column-kernel shape");
};

template <int P>
__global__ void __launch_bounds__(kBlock, 1) k_cols_dft(const ColDftArgs a) {
    constexpr int N = 512, W = 16;
    using S = DftShape<N>;
    using CS = ColDftShape<N, P, W>;
    constexpr int N2 = S::N2, K2 = S::K2, C2 = S::C2, H = CS::H, ND = CS::ND;
    constexpr int NPROD = P == 1 ? 1 : 4;
    const int x0 = blockIdx.x * W, cl = blockIdx.y, c = a.c0 + cl;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q = warp & 3;

    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // the swizzled stage-2 operand needs a 1024-byte aligned base (the size includes the slack)
    unsigned char *smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    unsigned char *sA2 = smem;                                   // [P][A2P]
    unsigned char *sA1 = sA2 + P * CS::A2P;                      // [2 buffers][P][A1P]
    unsigned char *sTab = sA1 + 2 * P * CS::A1P;
    const unsigned char *sB1 = sTab, *sB2 = sTab + S::B1_BYTES;
    const float4 *sTw = reinterpret_cast<const float4 *>(sB2 + S::B2_BYTES);   // [c pair][b]
    uint64_t *mbar = reinterpret_cast<uint64_t *>(sTab + S::TAB_BYTES);   // [0] stage 1, [1] stage 2
    uint32_t *tslot = reinterpret_cast<uint32_t *>(mbar + 2);

    dftc::load_table(sTab, a.dft_tab, S::TAB_BYTES);
    if (tid == 0) {
        tc::mbar_init(&mbar[0], 1);
        tc::mbar_init(&mbar[1], 1);
    }
    if (warp == 0) {
        tc::tmem_alloc(tslot, CS::TCOLS);
        tc::tmem_relinquish();
    }
    // Piece i = k kBlock + tid of a sample: pol p, row ry, re/im ri, column piece h (16 bytes = 8 columns).  With
    // kBlock a divisor of 2 H N, k fixes p and ry's multiple of ROWS_K (PK, RYK below, compile-time) and the
    // thread fixes ry mod ROWS_K = r0, ri and h, consecutive lanes consecutive rows.  In the stage-1 operand (128-byte swizzle) the piece is the 8 rows
    // m = W b + 8 h + (0..7) at k = 2 a + ri (ry = N2 a + b): eight consecutive b share 128 bytes, so the copies'
    // shared-memory writes meet no bank conflict either.  Rows no kernel reaches are zero: cleared once in both
    // buffers and never loaded.
    const int r0 = tid % CS::ROWS_K, ri0 = (tid / CS::ROWS_K) & 1, h0 = tid / (2 * CS::ROWS_K);
    const int a0 = r0 / N2, b0 = r0 - a0 * N2, kt = 2 * a0 + ri0;
    const int cg0 = (H * b0 + h0) & 7, mh0 = (H * b0 + h0) >> 3;
    const uint32_t dst_t = (uint32_t)(mh0 * CS::MH + kt * 128 + ((cg0 ^ (kt & 7)) << 4));
    const int src_t = field_offset(N, r0, ri0, blockIdx.x * H + h0);
    auto piece_dst = [&](int k) -> uint32_t {      // k compile-time after unrolling
        const int PK = (k * kBlock) / (2 * H * N), RYK = ((k * kBlock) % (2 * H * N)) / (2 * H), AK = RYK / N2;
        // 2 AK is a multiple of 4: its bit 2 flips that of the swizzle (kt < 4)
        return (uint32_t)(PK * CS::A1P + 2 * AK * 128) + (dst_t ^ (uint32_t)(((2 * AK) & 4) << 4));
    };
    auto piece_src = [&](int k) -> long long {
        const int PK = (k * kBlock) / (2 * H * N), RYK = ((k * kBlock) % (2 * H * N)) / (2 * H);
        return (long long)PK * N * 2 * N + RYK * 2 * N + src_t;
    };
    uint32_t act = 0;
#pragma unroll
    for (int k = 0; k < CS::ITER; ++k) {
        const int ry = (((k * kBlock) % (2 * H * N)) / (2 * H)) + r0;
        if ((a.row_nz[ry >> 5] >> (ry & 31)) & 1u) {
            act |= 1u << k;
        } else {
            const uint32_t d = piece_dst(k);
            *reinterpret_cast<uint4 *>(sA1 + d) = make_uint4(0u, 0u, 0u, 0u);
            *reinterpret_cast<uint4 *>(sA1 + P * CS::A1P + d) = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = *tslot;

    auto stage = [&](int tt, int buf) {
        const __half *src = a.H + ((long long)tt * a.slab_t + (long long)cl * a.slab_c) * P * N * 2 * N;
        unsigned char *dst = sA1 + buf * P * CS::A1P;
#pragma unroll
        for (int k = 0; k < CS::ITER; ++k)
            if ((act >> k) & 1u) cp_async16(dst + piece_dst(k), src + piece_src(k));
        cp_async_commit();
    };
    auto issue_s1 = [&](int buf) {
        tc::fence_after_sync();
        const uint32_t id1 = tc::idesc_f16(128, S::C1, true, false);
        const uint32_t a0 = tc::smem_u32(sA1 + buf * P * CS::A1P), b0 = tc::smem_u32(sB1);
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
            for (int j = 0; j < CS::T1; ++j)
#pragma unroll
                for (int ks = 0; ks < 2; ++ks)
                    tc::mma_f16(tbase + (uint32_t)((p * CS::T1 + j) * S::C1),
                                tc::smem_desc_sw128(a0 + p * CS::A1P + j * 2 * CS::MH + ks * 2048, CS::MH, 1024),
                                tc::smem_desc(b0 + ks * 256, 128, 512), id1, ks > 0);
        tc::mma_commit(&mbar[0]);
    };
    auto issue_s2 = [&]() {
        tc::fence_after_sync();
        const uint32_t id2 = tc::idesc_f16(128, C2, true, false);
        const uint32_t a0 = tc::smem_u32(sA2), b0 = tc::smem_u32(sB2);
        constexpr uint32_t SBOB = (K2 / 8) * 128;
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
            for (int j = 0; j < CS::T2; ++j)
#pragma unroll
                for (int ks = 0; ks < K2 / 16; ++ks)
                    tc::mma_f16(tbase + (uint32_t)(CS::D1 + (p * CS::T2 + j) * C2),
                                tc::smem_desc_sw128(a0 + p * CS::A2P + j * 2 * K2 * 128 + ks * 2048, K2 * 128, 1024),
                                tc::smem_desc(b0 + ks * 256, 128, SBOB), id2, ks > 0);
        tc::mma_commit(&mbar[1]);
    };
    // Twiddle stage 1's result and write it as stage 2's A: thread (b, x) of tile (p, j) writes, for
    // c = 8 ch .. 8 ch + 7 (one TMEM load of 16 columns each: real parts, then imaginary parts), the
    // re piece at k = b and the im piece at k = N2 + b of row group m2 = 8 W ch + 8 x.  Outputs c and
    // c + 1 go through packed FP32 arithmetic as a pair (t = (re w, -im w) / 16 of both):
    //   re = Xr re w - Xi im w,   im = Xi re w + Xr im w.
    auto epi1 = [&]() {
        for (int idx = warp >> 2; idx < P * CS::T1; idx += kBlock / 128) {
            const int p = idx / CS::T1, j = idx - p * CS::T1;
            const int m = 128 * j + 32 * q + lane, b = m / W, x = m % W;
            unsigned char *a2 = sA2 + p * CS::A2P;
#pragma unroll
            for (int ch = 0; ch < 2; ++ch) {
                float v[16];
                tc::tmem_ld16(tbase + ((uint32_t)(32 * q) << 16) + (uint32_t)(idx * S::C1 + 16 * ch), v);
                uint32_t re[4], im[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 t = sTw[(4 * ch + i) * N2 + b];
                    const float2 xr = make_float2(v[2 * i], v[2 * i + 1]), xi = make_float2(v[8 + 2 * i], v[9 + 2 * i]);
                    const float2 wr = make_float2(t.x, t.y), nwi = make_float2(t.z, t.w);
                    const float2 yr = dftc::fma2(xi, nwi, dftc::mul2(xr, wr));
                    const float2 yi = dftc::sub2(dftc::mul2(xi, wr), dftc::mul2(xr, nwi));
                    re[i] = dftc::pack_hh(yr.x, yr.y);
                    im[i] = dftc::pack_hh(yi.x, yi.y);
                }
                const int m2 = ch * 8 * W + x * 8;
                const int hb = (m2 >> 6) * K2 * 128, cg = (m2 & 63) >> 3;
                const int kr = b, ki = N2 + b;
                *reinterpret_cast<uint4 *>(a2 + hb + kr * 128 + ((cg ^ (kr & 7)) << 4)) =
                    make_uint4(re[0], re[1], re[2], re[3]);
                *reinterpret_cast<uint4 *>(a2 + hb + ki * 128 + ((cg ^ (ki & 7)) << 4)) =
                    make_uint4(im[0], im[1], im[2], im[3]);
            }
        }
    };
    // Square and sum: warp group j2 = warp / 4 takes stage-2 tile j2; lane quarter q's row l = 32 q + lane of the tile is
    // m2 = 128 j2 + l = 8 W c_hi + 8 x + c_lo: pixels (ky = 8 c_hi + c_lo + 16 d, kx = x0 + x) for every d.
    const int j2 = warp >> 2;
    // sums of d and d + 1 side by side (packed FP32)
    float2 acc[NPROD][ND / 2];
#pragma unroll
    for (int pq = 0; pq < NPROD; ++pq)
#pragma unroll
        for (int d = 0; d < ND / 2; ++d) acc[pq][d] = make_float2(0.f, 0.f);
    auto epi2 = [&]() {
#pragma unroll
        for (int db = 0; db < ND / 8; ++db) {         // 8 d per TMEM load of each pol: real parts, then imaginary
            const uint32_t col = (uint32_t)(CS::D1 + j2 * C2 + 16 * db);
            float ex[16];
            tc::tmem_ld16(tbase + ((uint32_t)(32 * q) << 16) + col, ex);
            if constexpr (P == 1) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 xr = make_float2(ex[2 * i], ex[2 * i + 1]), xi = make_float2(ex[8 + 2 * i], ex[9 + 2 * i]);
                    float2 &s0 = acc[0][4 * db + i];
                    s0 = dftc::fma2(xr, xr, dftc::fma2(xi, xi, s0));
                }
            } else {
                float ey[16];
                tc::tmem_ld16(tbase + ((uint32_t)(32 * q) << 16) + col + (uint32_t)(CS::T2 * C2), ey);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 xr = make_float2(ex[2 * i], ex[2 * i + 1]), xi = make_float2(ex[8 + 2 * i], ex[9 + 2 * i]);
                    const float2 yr = make_float2(ey[2 * i], ey[2 * i + 1]), yi = make_float2(ey[8 + 2 * i], ey[9 + 2 * i]);
                    const int dp = 4 * db + i;
                    acc[0][dp] = dftc::fma2(xr, xr, dftc::fma2(xi, xi, acc[0][dp]));
                    acc[1][dp] = dftc::fma2(yr, yr, dftc::fma2(yi, yi, acc[1][dp]));
                    acc[2][dp] = dftc::fma2(xr, yr, dftc::fma2(xi, yi, acc[2][dp]));
                    acc[3][dp] = dftc::sub2(dftc::fma2(xi, yr, acc[3][dp]), dftc::mul2(xr, yi));
                }
            }
        }
    };

    bool ok = true;
    if (a.nt > 0) stage(0, 0);
    for (int t = 0; t < a.nt; ++t) {
        const int buf = t & 1;
        cp_async_wait<0>();                    // sample t's strip has landed
        tc::fence_async_smem();
        tc::fence_before_sync();
        ok = __syncthreads_and(ok);
        if (!ok) break;
        if (tid == 0) issue_s1(buf);
        if (t + 1 < a.nt) stage(t + 1, buf ^ 1);   // its buffer was read by stage 1 of t - 1 (done)
        if (t > 0) {
            ok &= tc::mbar_wait_bounded(&mbar[1], (uint32_t)((t - 1) & 1), dftc::kWaitCycles);
            tc::fence_after_sync();
            epi2();
        }
        ok &= tc::mbar_wait_bounded(&mbar[0], (uint32_t)(t & 1), dftc::kWaitCycles);
        tc::fence_after_sync();
        epi1();
        tc::fence_async_smem();
        tc::fence_before_sync();
        ok = __syncthreads_and(ok);
        if (!ok) break;
        if (tid == 0) issue_s2();
    }
    if (ok && a.nt > 0) {
        ok &= tc::mbar_wait_bounded(&mbar[1], (uint32_t)((a.nt - 1) & 1), dftc::kWaitCycles);
        tc::fence_after_sync();
        epi2();
    }
    cp_async_wait<0>();
    tc::fence_before_sync();
    ok = __syncthreads_and(ok);
    tc::fence_after_sync();
    if (ok) {
        // undo the field's scale s_G / (16 N) (exact powers of two), squared, and fold into FP64
        const double un = 16.0 * (double)N / ((double)a.sy[c] * (double)a.s_t);
        const double sc2 = un * un;
        const int m2 = 128 * j2 + 32 * q + lane;
        const int x = (m2 % (8 * W)) >> 3, cy = 8 * (m2 / (8 * W)) + (m2 & 7);
#pragma unroll
        for (int pq = 0; pq < NPROD; ++pq) {
            double *dst = a.acc + ((long long)c * NPROD + pq) * N * N + x0 + x;
#pragma unroll
            for (int d = 0; d < ND; ++d)
                dst[(long long)(cy + 16 * d) * N] += (double)((d & 1) ? acc[pq][d >> 1].y : acc[pq][d >> 1].x) * sc2;
        }
    } else if (tid == 0) {
        atomicExch(a.err, tc::kErrWaitTimeout);
    }
    if (warp == 0) tc::tmem_dealloc(tbase, CS::TCOLS);
}

// ---------------------------------------------------------------------------------------------
// The column kernel as a pipeline of roles (one CTA per SM).  k_cols_dft's per-sample chain -- stage 1,
// twiddle, barrier, stage 2, square and sum, barrier -- left the SM waiting for MMA and TMEM latencies (issue 32 %,
// DRAM 26 % with two such CTAs per SM).  Here each step has warps of its own and hands over through
// mbarriers, every accumulator and operand double-buffered (all 512 TMEM columns for two pols), so the steps of
// neighbouring samples overlap:
//   warps 0-7    twiddle stage 1's result (their 16 twiddles stay in registers: a thread keeps its b for every
//                sample) and write the stage-2 operand
//   warps 8-15   square and sum stage 2's result in registers; at the end fold into the FP64 accumulators
//   warps 16, 19 cp.async of the strip into a ring of kCpStages samples (32 rows x 16 bytes per instruction; the
//                swizzled operand's writes are conflict-free)
//   warps 17, 18 issue the MMAs of stage 1 and of stage 2 (one elected lane each)
// The arithmetic and the order of each pixel's sums are k_cols_dft's, so the images are bit-identical.
// Measured (two pols; k_cols_dft with 8 columns -> this): 512 grid, 24 channels x 250 samples of 16384 antennas 3599 ->
// 2660 us; 256 grid, 96 x 333 of 4096 antennas 4796 -> 3521 us.  About 1600 cycles per sample and SM, against 2660
// before; no role waits long on one other: shared-memory traffic (about 1100 of them) binds next.
// Every wait is bounded (shared abort flag); the status word is set and every role unwinds.
constexpr int kCpThreads = 20 * 32;   // whole warpgroups (register shares below); 
constexpr int kCpStages = 4;

// Register shares of the warpgroups (launched with 96 a thread, 640 threads: 61,440): 2 x 128 threads squaring at
// 128, 2 x 128 twiddling at 88, 128 at 40 = 60,416, so every increase is covered by the decreases.
constexpr int kCpRegsSquare = 128, kCpRegsTwiddle = 88, kCpRegsIssue = 40;
static_assert(256 * kCpRegsSquare + 256 * kCpRegsTwiddle + 128 * kCpRegsIssue <= kCpThreads * 96, "register shares");
template <int R>
__device__ __forceinline__ void regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(R)); }
template <int R>
__device__ __forceinline__ void regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(R)); }

template <int N, int P, int W>
struct ColPipeShape {
    using S = DftShape<N>;
    using CS = ColDftShape<N, P, W>;
    static constexpr int D1 = P * CS::T1 * S::C1, D2 = P * CS::T2 * S::C2;   // TMEM columns of one buffer
    static constexpr int TC_ = 2 * (D1 + D2);
    static constexpr int TCOLS = TC_ <= 128 ? 128 : (TC_ <= 256 ? 256 : 512);
    static constexpr int A1 = P * CS::A1P, A2 = P * CS::A2P;                  // operand bytes of one sample
    static constexpr int TAB = S::B1_BYTES + S::B2_BYTES;                     // twiddles go to registers
    static constexpr int NBAR = 2 * kCpStages + 12;
    // Groups of four twiddle warps with rows to twiddle: two tiles, or two pols of one tile; one pol of one tile leaves
    // the second group without any.  That group keeps out of the hand-overs: only a warp that waits for the
    // operand buffer's release (a2_empty) may arrive on a2_full, or two arrivals of its own could complete a phase that
    // the other group, still writing, has not arrived for.
    static constexpr int TGROUPS = CS::T1 * P >= 2 ? 2 : 1;
    static constexpr size_t SMEM = 1024 + (size_t)kCpStages * A1 + 2 * (size_t)A2 + TAB + NBAR * 8 + 16;
    static_assert(TC_ <= 512 && SMEM <= 227 * 1024 && CS::T1 <= 2, "column pipeline shape");
};

template <int N, int P, int W>
__global__ void __launch_bounds__(kCpThreads, 1) k_cols_pipe(const ColDftArgs a) {
    using S = DftShape<N>;
    using CS = ColDftShape<N, P, W>;
    using CP = ColPipeShape<N, P, W>;
    constexpr int N2 = S::N2, K2 = S::K2, C2 = S::C2, H = CS::H, ND = CS::ND;
    constexpr int NPROD = P == 1 ? 1 : 4;
    const int x0 = blockIdx.x * W, cl = blockIdx.y, c = a.c0 + cl;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q = warp & 3;

    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    unsigned char *sA1 = smem;                                   // [kCpStages][P][A1P]
    unsigned char *sA2 = sA1 + kCpStages * CP::A1;               // [2][P][A2P]
    unsigned char *sB1 = sA2 + 2 * CP::A2, *sB2 = sB1 + S::B1_BYTES;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sB1 + CP::TAB);
    uint64_t *full = bars, *empty = full + kCpStages;            // strip ring
    uint64_t *d1_full = empty + kCpStages, *d1_empty = d1_full + 2, *a2_full = d1_full + 4, *a2_empty = d1_full + 6,
             *d2_full = d1_full + 8, *d2_empty = d1_full + 10;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + CP::NBAR);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);

    dftc::load_table(sB1, a.dft_tab, CP::TAB);
    if (tid == 0) {
        for (int s = 0; s < kCpStages; ++s) {
            tc::mbar_init(&full[s], 2);          // the two producer warps
            tc::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&d1_full[b], 1);
            tc::mbar_init(&d1_empty[b], 4 * CP::TGROUPS);
            tc::mbar_init(&a2_full[b], 4 * CP::TGROUPS);
            tc::mbar_init(&a2_empty[b], 1);
            tc::mbar_init(&d2_full[b], 1);
            tc::mbar_init(&d2_empty[b], 8);
        }
        *abort_flag = 0;
    }
    if (warp == 0) {
        tc::tmem_alloc(tslot, CP::TCOLS);
        tc::tmem_relinquish();
    }
    tc::fence_async_smem();   // the tables, written by generic stores, read by the tensor core
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = *tslot;

    if (warp < 8) {
        // ---------------- twiddle: row m = 128 j + 32 q + lane of tile j (b = m / W, x = m % W) of each pol
        if constexpr (P == 2) regs_dec<kCpRegsTwiddle>();
        constexpr int PW = CS::T1 == 2 ? 1 : 2;                  // warp groups per (tile, set of pols)
        const int g = warp >> 2, j = CS::T1 == 2 ? g : 0, p0 = CS::T1 == 2 ? 0 : g;
        const int m = 128 * j + 32 * q + lane, b = m / W, x = m % W;
        const float4 *gtw = reinterpret_cast<const float4 *>(a.dft_tab + CP::TAB);   // [c pair][b]
        float4 tw[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) tw[i] = __ldg(gtw + i * N2 + b);
        // piece (c group ch, k) at a2_t + ch * (8 W / 64) * K2 * 128 + k * 128, k = b and N2 + b (same k mod 8)
        const int cgx = W == 8 ? x : (x & 7);
        const uint32_t a2_t = (uint32_t)((W == 16 ? (x >> 3) * K2 * 128 : 0) + b * 128 + ((cgx ^ (b & 7)) << 4));
        for (int t = 0; t < a.nt && g < CP::TGROUPS; ++t) {
            const int buf = t & 1;
            const uint32_t ph = (uint32_t)((t >> 1) & 1);
            if (!tc::mbar_wait_abortable(&d1_full[buf], ph, dftc::kWaitCycles, abort_flag)) break;
            tc::fence_after_sync();
            bool ok = true;
#pragma unroll
            for (int p = 0; p < P; ++p) {
                if (PW == 2 && p != p0) continue;
                float v[32];
                tc::tmem_ld32(tbase + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * CP::D1 + (p * CS::T1 + j) * S::C1), v);
                if (PW == 2 || p == P - 1) {                     // the warp's last read of this accumulator
                    tc::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&d1_empty[buf]);
                }
                uint32_t re[8], im[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float *u = v + 16 * (i >> 2);
                    const int e = 2 * (i & 3);
                    const float2 xr = make_float2(u[e], u[e + 1]), xi = make_float2(u[8 + e], u[9 + e]);
                    const float2 wr = make_float2(tw[i].x, tw[i].y), nwi = make_float2(tw[i].z, tw[i].w);
                    const float2 yr = dftc::fma2(xi, nwi, dftc::mul2(xr, wr));
                    const float2 yi = dftc::sub2(dftc::mul2(xi, wr), dftc::mul2(xr, nwi));
                    re[i] = dftc::pack_hh(yr.x, yr.y);
                    im[i] = dftc::pack_hh(yi.x, yi.y);
                }
                // stage 2 of sample t - 2 has read this operand buffer
                if ((PW == 2 || p == 0) && !tc::mbar_wait_abortable(&a2_empty[buf], ph ^ 1u, dftc::kWaitCycles, abort_flag)) { ok = false; break; }
                unsigned char *o = sA2 + buf * CP::A2 + p * CS::A2P + a2_t;
#pragma unroll
                for (int ch = 0; ch < 2; ++ch) {
                    *reinterpret_cast<uint4 *>(o + ch * (W / 8) * K2 * 128) =
                        make_uint4(re[4 * ch], re[4 * ch + 1], re[4 * ch + 2], re[4 * ch + 3]);
                    *reinterpret_cast<uint4 *>(o + ch * (W / 8) * K2 * 128 + N2 * 128) =
                        make_uint4(im[4 * ch], im[4 * ch + 1], im[4 * ch + 2], im[4 * ch + 3]);
                }
            }
            if (!ok) break;
            tc::fence_async_smem();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&a2_full[buf]);
        }
    } else if (warp < 16) {
        // ---------------- square and sum (as k_cols_dft): warp group g takes stage-2 tile j2 or half the d range
        if constexpr (P == 2) regs_inc<kCpRegsSquare>();
        const int g = (warp - 8) >> 2;
        const int j2 = CS::T2 == 2 ? g : 0, dbase = CS::T2 == 2 ? 0 : g * ND;
        float2 acc[NPROD][ND / 2];
#pragma unroll
        for (int pq = 0; pq < NPROD; ++pq)
#pragma unroll
            for (int d = 0; d < ND / 2; ++d) acc[pq][d] = make_float2(0.f, 0.f);
        bool ok = true;
        for (int t = 0; t < a.nt; ++t) {
            const int buf = t & 1;
            if (!(ok = tc::mbar_wait_abortable(&d2_full[buf], (uint32_t)((t >> 1) & 1), dftc::kWaitCycles, abort_flag))) break;
            tc::fence_after_sync();
            const uint32_t col0 = tbase + ((uint32_t)(32 * q) << 16) +
                                  (uint32_t)(2 * CP::D1 + buf * CP::D2 + j2 * C2 + 2 * dbase);
#pragma unroll
            for (int db = 0; db < ND / 8; ++db) {     // 8 d per TMEM load of each pol: real parts, then imaginary
                float ex[16];
                tc::tmem_ld16(col0 + 16 * db, ex);
                if constexpr (P == 1) {
                    if (db == ND / 8 - 1) {
                        tc::fence_before_sync();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(&d2_empty[buf]);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float2 xr = make_float2(ex[2 * i], ex[2 * i + 1]), xi = make_float2(ex[8 + 2 * i], ex[9 + 2 * i]);
                        float2 &s0 = acc[0][4 * db + i];
                        s0 = dftc::fma2(xr, xr, dftc::fma2(xi, xi, s0));
                    }
                } else {
                    float ey[16];
                    tc::tmem_ld16(col0 + 16 * db + (uint32_t)(CS::T2 * C2), ey);
                    if (db == ND / 8 - 1) {
                        tc::fence_before_sync();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(&d2_empty[buf]);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float2 xr = make_float2(ex[2 * i], ex[2 * i + 1]), xi = make_float2(ex[8 + 2 * i], ex[9 + 2 * i]);
                        const float2 yr = make_float2(ey[2 * i], ey[2 * i + 1]), yi = make_float2(ey[8 + 2 * i], ey[9 + 2 * i]);
                        const int dp = 4 * db + i;
                        acc[0][dp] = dftc::fma2(xr, xr, dftc::fma2(xi, xi, acc[0][dp]));
                        acc[1][dp] = dftc::fma2(yr, yr, dftc::fma2(yi, yi, acc[1][dp]));
                        acc[2][dp] = dftc::fma2(xr, yr, dftc::fma2(xi, yi, acc[2][dp]));
                        acc[3][dp] = dftc::sub2(dftc::fma2(xi, yr, acc[3][dp]), dftc::mul2(xr, yi));
                    }
                }
            }
        }
        if (ok) {   // undo the field's scale s_G / (16 N) (exact powers of two), squared, and fold into FP64
            const double un = 16.0 * (double)N / ((double)a.sy[c] * (double)a.s_t);
            const double sc2 = un * un;
            const int se = pow2_exp(sc2);
            const int m2 = 128 * j2 + 32 * q + lane;
            const int x = (m2 % (8 * W)) >> 3, cy = 8 * (m2 / (8 * W)) + (m2 & 7);
#pragma unroll
            for (int pq = 0; pq < NPROD; ++pq) {
                double *dst = a.acc + ((long long)c * NPROD + pq) * N * N + x0 + x + (long long)(cy + 16 * dbase) * N;
#pragma unroll
                for (int d = 0; d < ND; ++d)
                    red_scaled(dst + 16 * d * N, (d & 1) ? acc[pq][d >> 1].y : acc[pq][d >> 1].x, se, sc2);
            }
        }
    } else {
        if constexpr (P == 2) regs_dec<kCpRegsIssue>();
        if (warp == 16 || warp == 19) {
        // ---------------- producers (one warp per part, re / im): piece (p, h, i) = rows ry = 32 i + lane; in the
        // operand row group H b + h at k = 2 a + ri (ry = N2 a + b), 16-byte chunk XOR-ed with k mod 8.  Rows
        // no kernel reaches are zero: cleared once in every stage and never loaded.  Every offset is one of four
        // swizzled thread constants plus a compile-time one (a copy is one instruction: with addresses computed
        // per copy the issue itself was the slowest role, about 1500 cycles per sample).
        constexpr int NI = N / 32, AI = 32 / N2;                 // a = AI i + al
        const int ri = warp == 19;
        const int al = lane / N2, b = lane % N2;
        const uint32_t base = (uint32_t)(((H * b) >> 3) * CS::MH + al * 256 + ((((H * b) & 7) ^ (2 * al) ^ ri) << 4) + ri * 128);
        uint32_t dt[4];                                          // variants: XOR with 2 v (N2 = 32: i mod 4), or 4 (i mod 2) + h
#pragma unroll
        for (int v = 0; v < 4; ++v) dt[v] = tc::smem_u32(sA1) + (base ^ (uint32_t)((AI == 1 ? 2 * v : 4 * (v >> 1) + (v & 1)) << 4));
        uint32_t rows = 0;
#pragma unroll
        for (int i = 0; i < NI; ++i) rows |= ((a.row_nz[i] >> lane) & 1u) << i;
        auto for_pieces = [&](auto &&f) {                        // f(i, smem offset, source offset in halves)
#pragma unroll
            for (int i = 0; i < NI; ++i)
#pragma unroll
                for (int p = 0; p < P; ++p)
#pragma unroll
                    for (int h = 0; h < H; ++h)
                        f(i, AI == 1 ? i & 3 : 2 * (i & 1) + h, p * CS::A1P + 2 * AI * i * 128, p * N * 2 * N + field_offset(N, 32 * i, 0, h));
        };
        for (int s = 0; s < kCpStages; ++s)
            for_pieces([&](int i, int v, int off, int) {
                if (!((rows >> i) & 1u))
                    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};\n" ::"r"(dt[v] + s * CP::A1 + off), "r"(0u) : "memory");
            });
        const __half *src = a.H + (long long)cl * a.slab_c * P * N * 2 * N + field_offset(N, lane, ri, blockIdx.x * H);
        const long long tstep = a.slab_t * P * N * 2 * N;
        auto landed = [&](int t) {                               // this warp's copies of sample t are complete
            tc::fence_async_smem();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&full[t % kCpStages]);
        };
        // two samples stay in flight: a third would tie each hand-over to the stage freed right before it
        constexpr int LAG = kCpStages - 2;
        for (int t = 0; t < a.nt; ++t, src += tstep) {
            const int st = t % kCpStages;
            if (!tc::mbar_wait_abortable(&empty[st], (uint32_t)(((t / kCpStages) & 1) ^ 1), dftc::kWaitCycles, abort_flag)) break;
            uint32_t d[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) d[v] = dt[v] + st * CP::A1;
            for_pieces([&](int i, int v, int off, int so) { cp_async16_if((rows >> i) & 1u, d[v] + off, src + so); });
            cp_async_commit();
            if (t >= LAG) {
                cp_async_wait<LAG>();
                landed(t - LAG);
            }
        }
        cp_async_wait<0>();
        for (int t = a.nt > LAG ? a.nt - LAG : 0; t < a.nt; ++t) landed(t);
        } else if (warp == 17) {
        // ---------------- stage-1 MMAs (the whole warp runs it, one elected lane issues)
        const uint32_t one = tc::elect_one(), id1 = tc::idesc_f16(128, S::C1, true, false), b1 = tc::smem_u32(sB1);
        for (int t = 0; t < a.nt; ++t) {
            const int st = t % kCpStages, buf = t & 1;
            if (!tc::mbar_wait_warp(&full[st], (uint32_t)((t / kCpStages) & 1), dftc::kWaitCycles, abort_flag)) break;
            if (!tc::mbar_wait_warp(&d1_empty[buf], (uint32_t)(((t >> 1) & 1) ^ 1), dftc::kWaitCycles, abort_flag)) break;
            tc::fence_after_sync();
            const uint32_t a0 = tc::smem_u32(sA1 + st * CP::A1);
#pragma unroll
            for (int p = 0; p < P; ++p)
#pragma unroll
                for (int j = 0; j < CS::T1; ++j)
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks)
                        tc::mma_f16_warp(one, tbase + (uint32_t)(buf * CP::D1 + (p * CS::T1 + j) * S::C1),
                                         tc::smem_desc_sw128(a0 + p * CS::A1P + j * 2 * CS::MH + ks * 2048, CS::MH, 1024),
                                         tc::smem_desc(b1 + ks * 256, 128, 512), id1, ks > 0);
            tc::mma_commit_warp(one, &d1_full[buf]);
            tc::mma_commit_warp(one, &empty[st]);
        }
        } else {
        // ---------------- stage-2 MMAs
        const uint32_t one = tc::elect_one(), id2 = tc::idesc_f16(128, C2, true, false), b2 = tc::smem_u32(sB2);
        constexpr uint32_t SBOB = (K2 / 8) * 128;
        for (int t = 0; t < a.nt; ++t) {
            const int buf = t & 1;
            const uint32_t ph = (uint32_t)((t >> 1) & 1);
            if (!tc::mbar_wait_warp(&a2_full[buf], ph, dftc::kWaitCycles, abort_flag)) break;
            if (!tc::mbar_wait_warp(&d2_empty[buf], ph ^ 1u, dftc::kWaitCycles, abort_flag)) break;
            tc::fence_after_sync();
            const uint32_t a0 = tc::smem_u32(sA2 + buf * CP::A2);
#pragma unroll
            for (int p = 0; p < P; ++p)
#pragma unroll
                for (int j = 0; j < CS::T2; ++j)
#pragma unroll
                    for (int ks = 0; ks < K2 / 16; ++ks)
                        tc::mma_f16_warp(one, tbase + (uint32_t)(2 * CP::D1 + buf * CP::D2 + (p * CS::T2 + j) * C2),
                                         tc::smem_desc_sw128(a0 + p * CS::A2P + j * 2 * K2 * 128 + ks * 2048, K2 * 128, 1024),
                                         tc::smem_desc(b2 + ks * 256, 128, SBOB), id2, ks > 0);
            tc::mma_commit_warp(one, &d2_full[buf]);
            tc::mma_commit_warp(one, &a2_empty[buf]);
        }
        }
    }
    __syncwarp();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (*abort_flag && tid == 0) atomicExch(a.err, tc::kErrWaitTimeout);
    if (warp == 0) tc::tmem_dealloc(tbase, CP::TCOLS);
}

template <int N, int P, int W>
cudaError_t launch_cols_pipe_t(const ColDftArgs &a, cudaStream_t st) {
    auto k = k_cols_pipe<N, P, W>;
    const size_t smem = ColPipeShape<N, P, W>::SMEM;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<dim3(N / W, a.nc), kCpThreads, smem, st>>>(a);
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_cols_dft_t(const ColDftArgs &a, cudaStream_t st) {
    using CS = ColDftShape<512, P, 16>;
    auto k = k_cols_dft<P>;
    const size_t smem = CS::SMEM;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<dim3(512 / 16, a.nc), kBlock, smem, st>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Row transform of the tensor-core gridding's tile-major field as N1 x N2 (8 x 64 on the 512 grid,
// 16 x 16 on the 256 grid) with the second stage transposed.  One CTA = a stripe of RS grid rows of one channel
// (512 grid: eight rows of one pol, whole 256-byte tile samples in and whole 128-byte lines of every strip out; 256
// grid: eight rows of both pols or sixteen of the one) walking a chunk of samples.  With n = b + N2 a (a < N1, b < N2): stage 1 is the
// N1-point DFT over a, [F N2 rows (f, b)] x [2 N1 (a, re/im)] -> 2 N1 columns per row; the twiddle
// exp(+2 pi i b c / N) / N1 is applied in FP32 and the result rounded to FP16 into the stage-2 operand Y'
// (MN-major); stage 2 is the N2-point DFT over b with the DFT matrix in real form as the K-major A operand.
//   N = 512: D[(re/im, d) 128][(f, c) 64], K = (re/im, b).  The matrix's four 64 x 64 blocks are C, -S / S, C
//            (C, S the cosine and sine matrices), kept once as [-S; C; S]: the real-input k-steps read
//            rows C, S from the middle block on, the imaginary-input ones -S, C from the top.
//   N = 256: the 16-point matrix X in real form is 32 x 32, so the 16 rows of a stripe are taken as four
//            quarters h of four: D[(h, re/im, d) 128][(f mod 4, c) 64], K = (h, re/im, b), A = diag(X, X, X, X)
//            kept once as [0; 0; 0; X; 0; 0; 0], the k-steps of quarter h reading from block 3 - h on.
// A TMEM lane then holds N1 consecutive outputs k = c + N1 d of one part for consecutive grid rows, which the
// field's layout (field_offset) takes as whole 32-byte stores.  Output scale 1/N.
// At most 73 KB of shared memory and 128 TMEM columns: three CTAs per SM.  Bound by DRAM (field in and out).
// Measured: 256 grid, 96 channels x 333 samples of 4096 antennas 3017 us (3934 us for a 16 x 16 kernel whose stage 2
// was not transposed and whose rows left as half2 pairs swapped by shuffles); 512 grid, 24 x 250 of 16384 antennas
// 1942 us (2046 us with rows of [re N][im N]; 2010 us and, on the 256 grid, 3851 us with kFieldRows = 4).
template <int N_, int P>
struct RowDft8Shape {
    static constexpr int PC = N_ == 512 ? 1 : P;          // pols per CTA: eight (or sixteen) grid rows of one pol or both
    static constexpr int N = N_, N1 = N == 512 ? 8 : 16, N2 = N / N1;
    static constexpr int HV = 64 / N2;                    // parts of the stripe's rows sharing one product
    static constexpr int F = N == 512 ? 8 : 16, RS = F / PC;   // transform rows per stripe, f = p RS + rl
    static constexpr int FH = F / HV;                     // rows f per part: f = h FH + f'
    static constexpr int M1 = F * N2, T1 = M1 / 128;      // stage-1 rows (f, b)
    static constexpr int K1 = 2 * N1, C1 = 2 * N1;        // (a, re/im) -> stage-1 columns
    static constexpr int LBO1 = (M1 / 8) * 128;
    static constexpr int A1B = M1 * K1 * 2;
    static constexpr int NB = FH * N1;                    // stage-2 N: (f', c)
    static constexpr int K2 = 2 * N2 * HV;                // stage-2 K: (h, re/im, b)
    static constexpr int LBOB = (NB / 8) * 128;           // K-direction stride of the stage-2 B operand
    static constexpr int BB = NB * K2 * 2;
    static constexpr int B1_BYTES = C1 * K1 * 2;
    static constexpr int KT = N == 512 ? 64 : 32;         // contraction of the stored blocks
    static constexpr int TSBO = (KT / 8) * 128;           // their row-group stride
    static constexpr int T_BYTES = (N == 512 ? 192 : 224) * KT * 2;
    static constexpr int W_BYTES = N == 512 ? N2 * 8 : N1 * N2 * 8;   // float2 w_b, or exp(2 pi i b c / N) / 16 [c][b]
    static constexpr int TAB_BYTES = B1_BYTES + T_BYTES + W_BYTES;
    static constexpr int D1 = T1 * C1;                    // TMEM: stage-1 accumulators, then NB stage-2 columns
    static constexpr int TCOLS = 128;
    static constexpr int B8 = N2 / 8;                     // 16-byte pieces (8 b) per (f, a, re/im)
    static constexpr int ITER = F * N1 * 2 * B8 / kBlock; // pieces per thread and sample
    static constexpr size_t SMEM = 16 + 2 * (size_t)A1B + BB + TAB_BYTES + 32;
    static_assert(D1 + NB <= TCOLS && NB == 64 && K2 == 128 && kBlock == 256 && F % 8 == 0 && ITER == 4 &&
                      TAB_BYTES % 16 == 0 && SMEM * 3 <= 226 * 1024,
                  "row-transform shape");
};

__device__ __forceinline__ float2 cmul8(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// 32 contiguous bytes (32-byte aligned) in one store: a whole L2 sector.
__device__ __forceinline__ void st_sector(__half *dst, const uint32_t (&w)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                 "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}

template <int N, int P>
__global__ void __launch_bounds__(kBlock) k_rows_dft8(const RowDftArgs a) {
    using RD = RowDft8Shape<N, P>;
    constexpr int N1 = RD::N1, N2 = RD::N2, RS = RD::RS, FH = RD::FH;
    const int s = blockIdx.x / (P / RD::PC), pc = blockIdx.x % (P / RD::PC), cl = blockIdx.y;   // pc: the first pol
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q = warp & 3;
    const int ry0 = s * RS;
    {   // stripes no kernel reaches carry no field: nothing to transform or store
        bool any = false;
        for (int rl = 0; rl < RS; ++rl) any |= ((a.row_nz[(ry0 + rl) >> 5] >> ((ry0 + rl) & 31)) & 1u) != 0;
        if (!any) return;
    }
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned char *sA1 = smem;                                   // [2][A1B]
    unsigned char *sB = sA1 + 2 * RD::A1B;                       // stage-2 B operand Y'
    unsigned char *sTab = sB + RD::BB;
    const unsigned char *sB1 = sTab, *sT = sTab + RD::B1_BYTES;
    const float2 *sW = reinterpret_cast<const float2 *>(sT + RD::T_BYTES);
    uint64_t *mbar = reinterpret_cast<uint64_t *>(sTab + RD::TAB_BYTES);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(mbar + 2);

    dftc::load_table(sTab, a.dft_tab, RD::TAB_BYTES);
    if (tid == 0) {
        tc::mbar_init(&mbar[0], 1);
        tc::mbar_init(&mbar[1], 1);
    }
    if (warp == 0) {
        tc::tmem_alloc(tslot, RD::TCOLS);
        tc::tmem_relinquish();
    }
    // Piece (f, tile column tx, re/im ri): 8 consecutive b of a row.  Sixteen consecutive threads take the sixteen
    // pieces of one tile (256 contiguous bytes; with the tiles across the lanes every 16-byte piece was half a sector
    // of a line of its own, and the row kernel 25 % slower), rounds k of the block the next sixteen tiles.  In the
    // stage-1 operand (N2 aa + 8 b8 = 8 tx) the piece is the 8 rows m = N2 f + 8 b8 + (0..7) at kk = 2 aa + ri; pieces
    // of tiles no kernel reaches are zero, cleared once.
    constexpr int B8 = RD::B8, NTX = N / 8;
    const int ri = tid & 1, rl = (tid >> 1) & 7, e0 = tid >> 4;
    auto piece_dst = [&](int k) -> uint32_t {
        const int e = 16 * k + e0, tx = e % NTX, kk = 2 * (tx / B8) + ri, f = (e / NTX) * 8 + rl;
        return (uint32_t)((f * B8 + tx % B8) * 128 + (kk >> 3) * RD::LBO1 + (kk & 7) * 16);
    };
    // input piece: the tile-major field, [channel][pol][tile row][tile col][sample][cy][re/im][cx]
    const long long tstride = (long long)a.Tb * 128;
    long long src_k[RD::ITER];
    uint32_t act = 0;
#pragma unroll
    for (int k = 0; k < RD::ITER; ++k) {
        const int e = 16 * k + e0, tx = e % NTX, f = (e / NTX) * 8 + rl, p = f / RS, ty = (ry0 + f % RS) >> 3;
        src_k[k] = ((((long long)cl * P + pc + p) * NTX + ty) * NTX + tx) * tstride + (rl * 2 + ri) * 8;
        if (a.active[ty * NTX + tx]) {
            act |= 1u << k;
        } else {
            *reinterpret_cast<uint4 *>(sA1 + piece_dst(k)) = make_uint4(0u, 0u, 0u, 0u);
            *reinterpret_cast<uint4 *>(sA1 + RD::A1B + piece_dst(k)) = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = *tslot;
    const float sc = 1.0f / (float)N2;
    const uint32_t one = tc::elect_one();

    auto load = [&](int tt, int buf) {
        const uint32_t dst = tc::smem_u32(sA1 + buf * RD::A1B);
#pragma unroll
        for (int k = 0; k < RD::ITER; ++k) cp_async16_if((act >> k) & 1u, dst + piece_dst(k), a.G + src_k[k] + (long long)tt * 128);
        cp_async_commit();
    };
    auto issue_s1 = [&](int buf) {   // by warp 0, one elected lane
        tc::fence_after_sync();
        const uint32_t id1 = tc::idesc_f16(128, RD::C1, true, false);
        const uint32_t a0 = tc::smem_u32(sA1 + buf * RD::A1B), b0 = tc::smem_u32(sB1);
#pragma unroll
        for (int j = 0; j < RD::T1; ++j)
#pragma unroll
            for (int ks = 0; ks < RD::K1 / 16; ++ks)
                tc::mma_f16_warp(one, tbase + (uint32_t)(j * RD::C1),
                            tc::smem_desc(a0 + j * 2048 + ks * 2 * RD::LBO1, RD::LBO1, 128),
                            tc::smem_desc(b0 + ks * 256, 128, (RD::K1 / 8) * 128), id1, ks > 0);
        tc::mma_commit_warp(one, &mbar[0]);
    };
    auto issue_s2 = [&]() {
        tc::fence_after_sync();
        const uint32_t id2 = tc::idesc_f16(128, RD::NB, false, true);
        const uint32_t t0 = tc::smem_u32(sT), b0 = tc::smem_u32(sB);
#pragma unroll
        for (int ks = 0; ks < RD::K2 / 16; ++ks) {
            // N = 512: real parts of Y' (k-steps 0-3) meet rows C, S, imaginary ones -S, C; N = 256: quarter ks / 2
            const uint32_t ta = t0 + (N == 512 ? (ks < 4 ? (uint32_t)(8 * RD::TSBO) : 0u) + (uint32_t)((ks & 3) * 256)
                                               : (uint32_t)((3 - (ks >> 1)) * 4 * RD::TSBO + (ks & 1) * 256));
            tc::mma_f16_warp(one, tbase + (uint32_t)RD::D1, tc::smem_desc(ta, 128, RD::TSBO),
                        tc::smem_desc(b0 + ks * 2 * RD::LBOB, RD::LBOB, 128), id2, ks > 0);
        }
        tc::mma_commit_warp(one, &mbar[1]);
    };
    // twiddle, then the stage-2 operand: thread (f, b) writes its row's N1 outputs c at k = (h, re, b)
    // and (h, im, b) of n-group f'
    auto epi1 = [&]() {
        for (int u = warp >> 2; u < RD::T1; u += kBlock / 128) {
            const int m = 128 * u + 32 * q + lane, f = m / N2, b = m - f * N2;
            const int h = f / FH, fp = f - h * FH, kr = h * 2 * N2 + b, ki = kr + N2;
            float v[2 * N1];
            float2 w[N1];
            if constexpr (N == 512) {   // columns: the eight real parts, then the imaginary ones
                tc::tmem_ld16(tbase + ((uint32_t)(32 * q) << 16) + (uint32_t)(u * RD::C1), v);
                w[0] = make_float2(1.f, 0.f);
                w[1] = sW[b];
                w[2] = cmul8(w[1], w[1]);
                w[3] = cmul8(w[2], w[1]);
                w[4] = cmul8(w[2], w[2]);
                w[5] = cmul8(w[4], w[1]);
                w[6] = cmul8(w[3], w[3]);
                w[7] = cmul8(w[4], w[3]);
            } else {                    // columns: (re, im) of each c
                tc::tmem_ld32(tbase + ((uint32_t)(32 * q) << 16) + (uint32_t)(u * RD::C1), v);
#pragma unroll
                for (int c = 0; c < N1; ++c) w[c] = sW[c * N2 + b];
            }
            uint32_t re[N1 / 2], im[N1 / 2];
#pragma unroll
            for (int cc = 0; cc < N1; cc += 2) {
                const float2 t0 = w[cc], t1 = w[cc + 1];
                if constexpr (N == 512) {
                    re[cc >> 1] = dftc::pack_hh((v[cc] * t0.x - v[8 + cc] * t0.y) * 0.125f,
                                                (v[cc + 1] * t1.x - v[9 + cc] * t1.y) * 0.125f);
                    im[cc >> 1] = dftc::pack_hh((v[cc] * t0.y + v[8 + cc] * t0.x) * 0.125f,
                                                (v[cc + 1] * t1.y + v[9 + cc] * t1.x) * 0.125f);
                } else {
                    re[cc >> 1] = dftc::pack_hh(v[2 * cc] * t0.x - v[2 * cc + 1] * t0.y,
                                                v[2 * cc + 2] * t1.x - v[2 * cc + 3] * t1.y);
                    im[cc >> 1] = dftc::pack_hh(v[2 * cc] * t0.y + v[2 * cc + 1] * t0.x,
                                                v[2 * cc + 2] * t1.y + v[2 * cc + 3] * t1.x);
                }
            }
#pragma unroll
            for (int ch = 0; ch < N1 / 8; ++ch) {
                unsigned char *o = sB + (fp * (N1 / 8) + ch) * 128;
                *reinterpret_cast<uint4 *>(o + (kr >> 3) * RD::LBOB + (kr & 7) * 16) =
                    make_uint4(re[4 * ch], re[4 * ch + 1], re[4 * ch + 2], re[4 * ch + 3]);
                *reinterpret_cast<uint4 *>(o + (ki >> 3) * RD::LBOB + (ki & 7) * 16) =
                    make_uint4(im[4 * ch], im[4 * ch + 1], im[4 * ch + 2], im[4 * ch + 3]);
            }
        }
    };
    // stage-2 accumulators -> FP16 (x 1/N2): lane (h, re/im, d) of warp group g holds columns 32 g .. 32 g + 31 =
    // (f', c): N = 512 the eight c of four consecutive grid rows (64 contiguous bytes of strip d), N = 256 the
    // sixteen c of two (32 bytes of strips 2 d and 2 d + 1)
    const int m2 = 32 * q + lane, hh = m2 / (2 * N2), part = (m2 / N2) & 1, d = m2 % N2;
    const int f0o = hh * FH + 32 * (warp >> 2) / N1, po = f0o / RS;
    const int out_t = (pc + po) * N * 2 * N + field_offset(N, ry0 + f0o - po * RS, part, d * (N1 / 8));
    auto epi2 = [&](int tt) {
        float v[32];
        tc::tmem_ld32(tbase + ((uint32_t)(32 * q) << 16) + (uint32_t)(RD::D1 + 32 * (warp >> 2)), v);
        __half *o = a.H + ((long long)tt * a.slab_t + (long long)cl * a.slab_c) * P * N * 2 * N + out_t;
#pragma unroll
        for (int k = 0; k < 2; ++k) {   // N = 512: row pair k; N = 256: strip 2 d + k
            uint32_t w[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = N == 512 ? 16 * k + 2 * u : 16 * (u >> 2) + 8 * k + 2 * (u & 3);
                w[u] = dftc::pack_hh(v[i] * sc, v[i + 1] * sc);
            }
            st_sector(o + (N == 512 ? field_offset(N, 2 * k, 0, 0) : field_offset(N, 0, 0, k)), w);
        }
    };

    bool ok = true;
    if (a.nt > 0) load(0, 0);
    for (int t = 0; t < a.nt; ++t) {
        const int buf = t & 1;
        cp_async_wait<0>();
        tc::fence_async_smem();
        tc::fence_before_sync();
        ok = __syncthreads_and(ok);
        if (!ok) break;
        if (warp == 0) issue_s1(buf);
        if (t + 1 < a.nt) load(t + 1, buf ^ 1);
        if (t > 0) {
            ok &= tc::mbar_wait_bounded(&mbar[1], (uint32_t)((t - 1) & 1), dftc::kWaitCycles);
            tc::fence_after_sync();
            epi2(t - 1);
        }
        ok &= tc::mbar_wait_bounded(&mbar[0], (uint32_t)(t & 1), dftc::kWaitCycles);
        tc::fence_after_sync();
        epi1();
        tc::fence_async_smem();
        tc::fence_before_sync();
        ok = __syncthreads_and(ok);
        if (!ok) break;
        if (warp == 0) issue_s2();
    }
    if (ok && a.nt > 0) {
        ok &= tc::mbar_wait_bounded(&mbar[1], (uint32_t)((a.nt - 1) & 1), dftc::kWaitCycles);
        tc::fence_after_sync();
        epi2(a.nt - 1);
    }
    cp_async_wait<0>();
    tc::fence_before_sync();
    ok = __syncthreads_and(ok);
    tc::fence_after_sync();
    if (!ok && tid == 0) atomicExch(a.err, tc::kErrWaitTimeout);
    if (warp == 0) tc::tmem_dealloc(tbase, RD::TCOLS);
}

template <int N, int P>
cudaError_t launch_rows_dft8_t(const RowDftArgs &a, cudaStream_t st) {
    auto k = k_rows_dft8<N, P>;
    const size_t smem = RowDft8Shape<N, P>::SMEM;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<dim3(N / RowDft8Shape<N, P>::RS * (P / RowDft8Shape<N, P>::PC), a.nc), kBlock, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace

// B1 [n = 2c + re/im][k = 2a + re/im] = the real form of exp(+2 pi i a c / 16);
// B2 [n = 2d + re/im][k = re/im N2 + b] = that of exp(+2 pi i b d / N2) (both K-major
// images); twiddles [c][b] = exp(+2 pi i b c / N) / 16.  All in FP64, then rounded once.
// cols: the column kernel's image.  Output columns grouped by eight: n = 16 (c / 8) + 8 re/im
// + c mod 8 (and the same for d), so one 16-column TMEM load returns the real parts of eight
// outputs, then their imaginary parts, and neighbouring outputs pair up for packed FP32 arithmetic;
// twiddles as float4 (re w_c, re w_{c+1}, -im w_c, -im w_{c+1}) / 16 per (c pair, b).
std::vector<unsigned char> build_dft_table(int N, bool cols) {
    const int N2 = N / 16, K2 = 2 * N2;
    std::vector<unsigned char> img((size_t)dft_table_bytes(N), 0);
    auto put = [&](size_t off, double v) {
        const __half h = __float2half_rn((float)v);
        std::memcpy(img.data() + off, &h, 2);
    };
    auto col = [&](int o, int ri) { return cols ? 16 * (o >> 3) + 8 * ri + (o & 7) : 2 * o + ri; };
    for (int cc = 0; cc < 16; ++cc)
        for (int aa = 0; aa < 16; ++aa) {
            double wc, ws;
            unit_root((long long)aa * cc, 16, &wc, &ws);
            put(kmajor_at(col(cc, 0), 2 * aa, 32), wc);
            put(kmajor_at(col(cc, 0), 2 * aa + 1, 32), -ws);
            put(kmajor_at(col(cc, 1), 2 * aa, 32), ws);
            put(kmajor_at(col(cc, 1), 2 * aa + 1, 32), wc);
        }
    const size_t b2 = 2048;
    for (int d = 0; d < N2; ++d)
        for (int b = 0; b < N2; ++b) {
            double vc, vs;
            unit_root((long long)b * d, N2, &vc, &vs);
            put(b2 + kmajor_at(col(d, 0), b, K2), vc);
            put(b2 + kmajor_at(col(d, 0), N2 + b, K2), -vs);
            put(b2 + kmajor_at(col(d, 1), b, K2), vs);
            put(b2 + kmajor_at(col(d, 1), N2 + b, K2), vc);
        }
    const size_t tw = b2 + (size_t)K2 * K2 * 2;
    for (int cc = 0; cc < 16; ++cc)
        for (int b = 0; b < N2; ++b) {
            double wc, ws;
            unit_root((long long)b * cc, N, &wc, &ws);
            if (cols) {
                float *q = reinterpret_cast<float *>(img.data() + tw + ((size_t)(cc >> 1) * N2 + b) * 16);
                q[cc & 1] = (float)(wc / 16.0);
                q[2 + (cc & 1)] = (float)(-ws / 16.0);
            } else {
                const float2 v = make_float2((float)(wc / 16.0), (float)(ws / 16.0));
                std::memcpy(img.data() + tw + ((size_t)cc * N2 + b) * 8, &v, 8);
            }
        }
    return img;
}

// Tables of the row transform, all in FP64 then rounded once.  N = 512: B1 [n = 8 re/im + c][k = 2 a +
// re/im] = the real form of exp(+2 pi i a c / 8) (K-major, 16 x 16), the stage-2 blocks [-S; C; S] (S, C
// [d][b] = sin, cos of 2 pi b d / 64; K-major, 192 rows x 64), w_b = exp(+2 pi i b / 512).  N = 256: B1
// [n = 2 c + re/im][k = 2 a + re/im] (32 x 32), the blocks [0; 0; 0; X; 0; 0; 0] with X [re/im 16 + d][re/im 16 + b]
// the real form of exp(+2 pi i b d / 16) (224 rows x 32), twiddles [c][b] = exp(+2 pi i b c / 256) / 16.
std::vector<unsigned char> build_rows8_table(int N) {
    const int N1 = N == 512 ? 8 : 16, N2 = N / N1, K1 = 2 * N1, KT = N == 512 ? 64 : 32;
    const size_t b1 = (size_t)K1 * K1 * 2, tb = (size_t)(N == 512 ? 192 : 224) * KT * 2;
    std::vector<unsigned char> img(b1 + tb + (size_t)(N == 512 ? N2 : N1 * N2) * 8, 0);
    auto put = [&](size_t off, double v) {
        const __half h = __float2half_rn((float)v);
        std::memcpy(img.data() + off, &h, 2);
    };
    auto col = [&](int c, int ri) { return N == 512 ? 8 * ri + c : 2 * c + ri; };
    for (int c = 0; c < N1; ++c)
        for (int aa = 0; aa < N1; ++aa) {
            double wc, ws;
            unit_root((long long)aa * c, N1, &wc, &ws);
            put(kmajor_at(col(c, 0), 2 * aa, K1), wc);
            put(kmajor_at(col(c, 0), 2 * aa + 1, K1), -ws);
            put(kmajor_at(col(c, 1), 2 * aa, K1), ws);
            put(kmajor_at(col(c, 1), 2 * aa + 1, K1), wc);
        }
    for (int d = 0; d < N2; ++d)
        for (int b = 0; b < N2; ++b) {
            double vc, vs;
            unit_root((long long)b * d, N2, &vc, &vs);
            if (N == 512) {
                put(b1 + kmajor_at(d, b, KT), -vs);
                put(b1 + kmajor_at(64 + d, b, KT), vc);
                put(b1 + kmajor_at(128 + d, b, KT), vs);
            } else {
                put(b1 + kmajor_at(96 + d, b, KT), vc);
                put(b1 + kmajor_at(96 + d, 16 + b, KT), -vs);
                put(b1 + kmajor_at(112 + d, b, KT), vs);
                put(b1 + kmajor_at(112 + d, 16 + b, KT), vc);
            }
        }
    for (int i = 0; i < (N == 512 ? N2 : N1 * N2); ++i) {
        double wc, ws;
        if (N == 512) {
            unit_root(i, N, &wc, &ws);
        } else {
            unit_root((long long)(i / N2) * (i % N2), N, &wc, &ws);
            wc /= 16.0;
            ws /= 16.0;
        }
        const float2 v = make_float2((float)wc, (float)ws);
        std::memcpy(img.data() + b1 + tb + (size_t)i * 8, &v, 8);
    }
    return img;
}

cudaError_t launch_rows_dft8(int N, int P, const RowDftArgs &a, cudaStream_t st) {
    if (N == 512) return P == 1 ? launch_rows_dft8_t<512, 1>(a, st) : launch_rows_dft8_t<512, 2>(a, st);
    if (N == 256) return P == 1 ? launch_rows_dft8_t<256, 1>(a, st) : launch_rows_dft8_t<256, 2>(a, st);
    return cudaErrorInvalidValue;
}

// Columns per CTA by default: 8 (k_cols_pipe) unless MOFF_COLS_W=16; MOFF_AUTOTUNE times both.
int cols_dft_width() { return (getenv("MOFF_COLS_W") && atoi(getenv("MOFF_COLS_W")) == 16) ? 16 : 8; }
bool cols_dft_width_forced() { return getenv("MOFF_COLS_W") != nullptr; }

cudaError_t launch_cols_dft(int N, int P, int W, const ColDftArgs &a, cudaStream_t st) {
    if (W == 16) {
        if (N == 512) return P == 1 ? launch_cols_dft_t<1>(a, st) : launch_cols_dft_t<2>(a, st);
        if (N == 256) return P == 1 ? launch_cols_pipe_t<256, 1, 16>(a, st) : launch_cols_pipe_t<256, 2, 16>(a, st);
    } else {
        if (N == 512) return P == 1 ? launch_cols_pipe_t<512, 1, 8>(a, st) : launch_cols_pipe_t<512, 2, 8>(a, st);
        if (N == 256) return P == 1 ? launch_cols_pipe_t<256, 1, 8>(a, st) : launch_cols_pipe_t<256, 2, 8>(a, st);
    }
    return cudaErrorInvalidValue;
}

size_t grid_smem_bytes_dft(int N, int P, int TB, int rows, int max_nloc) {
    const int ldr = N + N / 16;
    const int F = TB * P * rows;
    size_t b = (dft_row_region_bytes(N, F) + 15) / 16 * 16;
    b += (size_t)F * ldr * 8 + 8;                       // one row buffer (+ alignment)
    b += (size_t)volt_stride(TB) * max_nloc * P * 8;    // calibrated voltages of TB samples
    b += (size_t)max_nloc * P * 8 + 8;                  // gains (+ padding)
    b += (size_t)max_nloc * 4;                          // antenna indices
    return (b + 15) & ~(size_t)15;
}

cudaError_t launch_grid_dft(int N, int P, int TB, int CPL, const GridArgs &a, int n_stripes, size_t smem,
                            cudaStream_t st) {
    if (N == 512) return launch_grid_dft_n512(P, TB, CPL, a, n_stripes, smem, st);
    if (N == 256) return launch_grid_dft_n256(P, TB, CPL, a, n_stripes, smem, st);
    return cudaErrorInvalidValue;
}

}  // namespace moff
