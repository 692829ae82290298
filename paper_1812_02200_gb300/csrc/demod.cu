// demod.cu -- direct multi-tone demodulation (Sec. III.B of arXiv:1812.02200)
// as the dense contraction it is, on the tcgen05 tensor cores.
//
// Definition (per tone t with NCO word w_t, frame k, b_k = first sample of
// the frame, taps h[0..L)):
//   out[t][k] = sum_n h[n] x[b_k+n] exp(-i*phi_t(b_k+n)),  phi_t(m) = 2*pi*(w_t*m mod 2^64)/2^64.
// Because w_t*(b+n) = w_t*b + w_t*n (mod 2^64) exactly,
//   out[t][k] = exp(-i*phi_t(b_k)) * sum_n x[b_k+n] * C_t[n],   C_t[n] = h[n] exp(-i*phi_t(n)),
// i.e. a GEMM of the Toeplitz matrix A[k][n] = x[b_k+n] (row stride D) with
// the modulated taps C (plan constant), followed by a per-(t,k) rotation.
//
// Precision.  x is a 14-bit integer: x = xh + xl with xh = fp16(x) and
// xl = x - xh, both exact in FP16.  C (scaled by 2^e so max|C| is in
// [2^14, 2^15)) is split into ch = fp16(C) and cl = fp16(C - ch).  The MMAs
// accumulate xh*ch + xh*cl + xl*ch (the dropped xl*cl is ~2^-22 relative) in
// FP32.  To keep the tensor cores' internal accumulation error small, each
// TMEM accumulator collects only a short chunk of K and the epilogue warps add
// the chunks into FP32 register sums (the accumulator is double-buffered, so
// the MMAs of the next chunk overlap the drain of the previous one).
//
// Real embedding: K' = 2L (re, im of x interleaved), N' = 2*tones with
//   B'[2t][2n] = Re C, B'[2t][2n+1] = -Im C, B'[2t+1][2n] = Im C, B'[2t+1][2n+1] = Re C
// so column 2t of the product is Re(x.C_t) and column 2t+1 is Im(x.C_t).
//
// Kernels:
//   build_taps  (plan time) FP64 modulated taps -> FP16 hi/lo, K-major B'.
//   rot         (per push)  FP64 rotation anchors exp(-i*phi_t(b)) at every
//                           128-frame tile start and steps exp(-i*w_t*D*j).
//   presplit    (per push)  int16 IQ of [carry | buffer] -> FP16 hi/lo rows of D
//                           samples (the Toeplitz view's 2-D tensor).
//   gemm        (per push)  TMA -> smem (128B swizzle) -> tcgen05.mma -> TMEM
//                           -> register sums -> rotation -> [tone][frame] out.
//   prep3       (per push)  the three-product form's rotation tables and planes
//   *3 variants             the Gauss three-product form (see below), a plan
//                           option (rfr_plan_set_demod_products).
#include <cuda.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <vector>

#include "dev_common.cuh"
#include "rfr_internal.h"
#include "umma.cuh"

namespace rfr {

// the CUDA driver API's cuTensorMapEncodeTiled, looked up once (nullptr if absent)
void* tmap_encode_tiled_fn() {
    static void* fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = p;
    });
    return fn;
}

namespace {

constexpr int BM = kDemodBM, BN = kDemodBN, BK = kDemodBK;
constexpr int STAGES = 2;
constexpr uint32_t A_BYTES = BM * BK * 2;
constexpr uint32_t B_BYTES = BN * BK * 2;
constexpr uint32_t STAGE_BYTES = 2 * A_BYTES + 2 * B_BYTES;
constexpr int EPI_WARPS = 8;
constexpr int GEMM_THREADS = (EPI_WARPS + 2) * 32;
constexpr uint32_t TMEM_COLS = 512;       // two 256-column FP32 accumulators
constexpr size_t GEMM_SMEM = 1024 + STAGES * STAGE_BYTES + 256;

__device__ __forceinline__ float2 expmi_u64(uint64_t phase) {
    // exp(-i * 2*pi*phase/2^64) in FP64, rounded to FP32
    const double xs = static_cast<double>(static_cast<int64_t>(phase)) * 0x1p-63;   // in [-1, 1)
    double s, c;
    sincospi(xs, &s, &c);
    return make_float2(static_cast<float>(c), static_cast<float>(-s));
}

__device__ __forceinline__ void split_store(__half* hi, __half* lo, size_t i, double v) {
    const __half h = __double2half(v);
    hi[i] = h;
    lo[i] = __double2half(v - static_cast<double>(__half2float(h)));
}

__global__ void build_taps_kernel(const double* __restrict__ h, const uint64_t* __restrict__ words,
                                  int n_tones, int ntp, int L, int Lpad, double scale,
                                  __half* __restrict__ bh, __half* __restrict__ bl) {
    const int64_t total = static_cast<int64_t>(ntp) * Lpad;
    const size_t ldk = static_cast<size_t>(2) * Lpad;
    for (int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; idx < total;
         idx += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int t = static_cast<int>(idx / Lpad);
        const int n = static_cast<int>(idx - static_cast<int64_t>(t) * Lpad);
        double cr = 0.0, ci = 0.0;
        if (t < n_tones && n < L) {
            const uint64_t ph = words[t] * static_cast<uint64_t>(n);
            const double xs = static_cast<double>(static_cast<int64_t>(ph)) * 0x1p-63;
            double s, c;
            sincospi(xs, &s, &c);
            const double a = h[n] * scale;
            cr = a * c;      // C = h * exp(-i*theta) = h*(cos - i sin)
            ci = -a * s;
        }
        const size_t r0 = static_cast<size_t>(2 * t) * ldk, r1 = r0 + ldk;
        split_store(bh, bl, r0 + 2 * n, cr);
        split_store(bh, bl, r0 + 2 * n + 1, -ci);
        split_store(bh, bl, r1 + 2 * n, ci);
        split_store(bh, bl, r1 + 2 * n + 1, cr);
    }
}

// Rotation factors on ABSOLUTE frame indices K = 128*A + i (so a stream split
// into pushes rotates every frame by the same FP32 factors):
//   anchors[a] = exp(-i*phi_t(b(128*(A0 + a)))),  steps[t][i] = exp(-i*w_t*D*i),
// with b(K) = (K+1)*D - L the first sample of frame K and A0 = F0/128.
__global__ void rot_kernel(const uint64_t* __restrict__ words, int n_tones, int ntp, int64_t A0, int L,
                           int D, int n_anch, float2* __restrict__ anchors, float2* __restrict__ steps) {
    const int64_t na = static_cast<int64_t>(n_anch) * ntp;
    const int64_t total = na + static_cast<int64_t>(ntp) * BM;
    for (int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; idx < total;
         idx += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        if (idx < na) {
            const int a = static_cast<int>(idx / ntp);
            const int t = static_cast<int>(idx - static_cast<int64_t>(a) * ntp);
            float2 r = make_float2(0.f, 0.f);
            if (t < n_tones) {
                const int64_t K = (A0 + a) * BM;
                const int64_t b = (K + 1) * D - L;
                r = expmi_u64(words[t] * static_cast<uint64_t>(b));
            }
            anchors[idx] = r;
        } else {
            const int64_t j = idx - na;
            const int t = static_cast<int>(j / BM);
            const int i = static_cast<int>(j - static_cast<int64_t>(t) * BM);
            float2 r = make_float2(0.f, 0.f);
            if (t < n_tones) r = expmi_u64(words[t] * static_cast<uint64_t>(static_cast<int64_t>(i) * D));
            steps[j] = r;
        }
    }
}

// Sample s of the virtual stream [carry | buffer] -> FP16 hi/lo pairs.
__global__ void presplit_kernel(const uint32_t* __restrict__ carry, int64_t cl,
                                const uint32_t* __restrict__ buf, int64_t lv, int64_t total,
                                __half2* __restrict__ hi, __half2* __restrict__ lo) {
    for (int64_t s = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; s < total;
         s += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        uint32_t w = 0;
        if (s < lv) w = s < cl ? carry[s] : buf[s - cl];
        const float2 f = iq_to_f2(w);
        const __half hr = __float2half_rn(f.x), hq = __float2half_rn(f.y);
        hi[s] = __halves2half2(hr, hq);
        lo[s] = __halves2half2(__float2half_rn(f.x - __half2float(hr)),
                               __float2half_rn(f.y - __half2float(hq)));
    }
}

struct GemmArgs {
    int raster;           // tile order: groups of `raster` M tiles sweep all N tiles
    int64_t F;
    int64_t F0;           // frames of the stream before this push
    int n_tones, ntp, KB, kchunk, two_d, n_mt, n_nt;
    const float2* anchors;
    const float2* steps;
    float inv_scale;
    float2* out;
    int64_t ld, fo;
    int* status;
};

// Tile index -> (M tile, N tile): groups of g.raster M tiles are swept
// N-tile-major, so concurrently running CTAs share the same tap slices in L2.
__device__ __forceinline__ void tile_coords_of(int raster, int n_mt, int n_nt, int tile, int& mt, int& nt) {
    const int r = raster > 1 ? raster : 1;
    if (r == 1) {
        mt = tile / n_nt;
        nt = tile % n_nt;
        return;
    }
    const int per_group = r * n_nt;
    const int grp = tile / per_group, in = tile % per_group;
    const int m_base = grp * r;
    const int rows = min(r, n_mt - m_base);
    nt = in / rows;
    mt = m_base + in % rows;
}
__device__ __forceinline__ void tile_coords(const GemmArgs& g, int tile, int& mt, int& nt) {
    tile_coords_of(g.raster, g.n_mt, g.n_nt, tile, mt, nt);
}

__global__ void __launch_bounds__(GEMM_THREADS, 1)
demod_gemm_kernel(const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmAl,
                  const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ CUtensorMap tmBl,
                  const GemmArgs g) {
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    unsigned char* smem = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* tfull = empty + STAGES;
    uint64_t* tempty = tfull + 2;
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(tempty + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], EPI_WARPS * 32);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == EPI_WARPS + 1) {
        umma::alloc(tmem_holder, TMEM_COLS);
        umma::relinquish();
    }
    if (warp == EPI_WARPS && lane == 0) {
        tma_prefetch_desc(&tmAh);
        tma_prefetch_desc(&tmAl);
        tma_prefetch_desc(&tmBh);
        tma_prefetch_desc(&tmBl);
    }
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    const uint32_t tmem = *tmem_holder;
    const int n_tiles = g.n_mt * g.n_nt;
    constexpr uint32_t IDESC = umma::idesc_f16_f32(BM, BN);

    if (warp == EPI_WARPS) {
        // ------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t it = 0;
            for (int tile = blockIdx.x; tile < n_tiles && !*abort_flag; tile += gridDim.x) {
                int tm, tn;
                tile_coords(g, tile, tm, tn);
                const int m0 = tm * BM, n0 = tn * BN;
                for (int kb = 0; kb < g.KB; ++kb, ++it) {
                    const int s = it % STAGES;
                    const uint32_t ph = (it / STAGES) & 1;
                    if (!mbar_wait(&empty[s], ph ^ 1, g.status)) { *abort_flag = 1; break; }
                    unsigned char* st = smem + s * STAGE_BYTES;
                    mbar_arrive_expect_tx(&full[s], STAGE_BYTES);
                    const int kh = kb * BK;
                    const int c0 = kh % g.two_d, c1 = m0 + kh / g.two_d;
                    tma_load_2d(st, &tmAh, c0, c1, &full[s]);
                    tma_load_2d(st + A_BYTES, &tmAl, c0, c1, &full[s]);
                    tma_load_2d(st + 2 * A_BYTES, &tmBh, kh, n0, &full[s]);
                    tma_load_2d(st + 2 * A_BYTES + B_BYTES, &tmBl, kh, n0, &full[s]);
                }
            }
            // wait for the copies still in flight before leaving
            for (uint32_t k = 0; k < STAGES && it > 0; ++k) {
                const uint32_t j = it - 1 - k;
                if (static_cast<int32_t>(j) < 0) break;
                // the last STAGES fills: their full barriers complete on arrival
                mbar_wait(&full[j % STAGES], (j / STAGES) & 1, g.status);
            }
        }
    } else if (warp == EPI_WARPS + 1) {
        // ------------------------------------------------ MMA issuer
        if (lane == 0) {
            uint32_t it = 0, cc = 0;
            for (int tile = blockIdx.x; tile < n_tiles && !*abort_flag; tile += gridDim.x) {
                for (int kb0 = 0; kb0 < g.KB && !*abort_flag; kb0 += g.kchunk, ++cc) {
                    const uint32_t ab = cc & 1, aph = (cc >> 1) & 1;
                    if (!mbar_wait(&tempty[ab], aph ^ 1, g.status)) { *abort_flag = 1; break; }
                    umma::fence_after_sync();
                    const uint32_t d_tmem = tmem + ab * BN;
                    const int kb1 = min(kb0 + g.kchunk, g.KB);
                    for (int kb = kb0; kb < kb1; ++kb, ++it) {
                        const int s = it % STAGES;
                        const uint32_t ph = (it / STAGES) & 1;
                        if (!mbar_wait(&full[s], ph, g.status)) { *abort_flag = 1; break; }
                        umma::fence_after_sync();
                        const uint32_t sa = smem_u32(smem + s * STAGE_BYTES);
                        const uint32_t ah = sa, al = sa + A_BYTES;
                        const uint32_t bh = sa + 2 * A_BYTES, bl = bh + B_BYTES;
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k) {
                            const uint32_t off = k * 32;   // 16 fp16 of K = 32 bytes
                            const uint32_t acc = (kb > kb0 || k > 0) ? 1u : 0u;
                            umma::mma_f16(d_tmem, umma::desc_k_sw128(ah + off), umma::desc_k_sw128(bh + off), IDESC, acc);
                            umma::mma_f16(d_tmem, umma::desc_k_sw128(ah + off), umma::desc_k_sw128(bl + off), IDESC, 1u);
                            umma::mma_f16(d_tmem, umma::desc_k_sw128(al + off), umma::desc_k_sw128(bh + off), IDESC, 1u);
                        }
                        umma::commit(&empty[s]);
                    }
                    umma::commit(&tfull[ab]);
                }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ epilogue (8 warps)
        const int q = warp & 3, half_sel = warp >> 2;
        const int row = q * 32 + lane;
        uint32_t cc = 0;
        for (int tile = blockIdx.x; tile < n_tiles && !*abort_flag; tile += gridDim.x) {
            int mt, tn;
            tile_coords(g, tile, mt, tn);
            const int m0 = mt * BM, n0 = tn * BN;
            float sums[128];
#pragma unroll
            for (int i = 0; i < 128; ++i) sums[i] = 0.f;
            bool ok = true;
            for (int kb0 = 0; kb0 < g.KB; kb0 += g.kchunk, ++cc) {
                const uint32_t ab = cc & 1, aph = (cc >> 1) & 1;
                if (!mbar_wait(&tfull[ab], aph, g.status)) { *abort_flag = 1; ok = false; break; }
                umma::fence_after_sync();
                const uint32_t base = tmem + (static_cast<uint32_t>(q * 32) << 16) + ab * BN + half_sel * 128;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t r[32];
                    umma::ld_32x32b_x32(base + j * 32, r);
                    umma::wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; ++i) sums[j * 32 + i] += __uint_as_float(r[i]);
                }
                umma::fence_before_sync();
                mbar_arrive(&tempty[ab]);
            }
            if (!ok) break;
            const int64_t k = static_cast<int64_t>(m0) + row;
            if (k < g.F) {
                const int tb = n0 / 2 + half_sel * 64;
                const int64_t K = g.F0 + k;                       // absolute frame
                const int64_t arow = K / BM - g.F0 / BM;          // anchor row of this push
                const int si = static_cast<int>(K % BM);
#pragma unroll
                for (int tl = 0; tl < 64; ++tl) {
                    const int t = tb + tl;
                    if (t < g.n_tones) {
                        const float2 an = __ldg(g.anchors + arow * g.ntp + t);
                        const float2 sp = __ldg(g.steps + static_cast<int64_t>(t) * BM + si);
                        const float2 rot = cmul(an, sp);
                        const float2 acc = make_float2(sums[2 * tl] * g.inv_scale, sums[2 * tl + 1] * g.inv_scale);
                        g.out[static_cast<int64_t>(t) * g.ld + g.fo + k] = cmul(acc, rot);
                    }
                }
            }
        }
    }
    umma::fence_before_sync();
    __syncthreads();
    if (warp == EPI_WARPS + 1) {
        umma::fence_after_sync();
        umma::dealloc(tmem, TMEM_COLS);
    }
}

// ---------------------------------------------- Gauss three-product form
//
// With x = xr + i xi and C = cr + i ci, the three real contractions
//   P1 = sum ((xr + xi)/2) cr,   P2 = sum xr (ci - cr),   P3 = sum xi (cr + ci)
// give Re(x.C) = 2 P1 - P3 and Im(x.C) = 2 P1 + P2: three real products per
// complex multiply-add instead of the four of the real embedding.  Each A
// plane ((xr+xi)/2, xr, xi) and B plane (cr, ci-cr, cr+ci) is split into FP16
// hi/lo as above ((xr+xi)/2 has at most 17 significant bits, exact as hi+lo);
// each product again takes the three MMAs hi.hi + hi.lo + lo.hi.
//
// What bounds it.  Per 16 taps a CTA's shared memory takes the MMAs' operand
// reads and the TMA's writes at 128 bytes a clock, and the SM takes at most
// 64 bytes a clock from L2.  A tile of 128 frames x 128 tones on one SM needs
// 36-40 KB of shared-memory traffic and 16 KB from L2 for 192 clocks of
// tensor work: both limits lie above the tensor time, and the tensor pipe
// measured 62 % active.  PAIR therefore gives two SMs one tile of 256 frames
// (cta_group::2 MMAs, M = 256): each SM holds its 128 frames and half the
// tones' tap rows.  At 256 tones (WIDE) it reads 8 KB per MMA of 128 clocks,
// 40 KB and 16 KB from L2 for 384 clocks of tensor work; at 128, 24 KB of reads
// and 12 KB of writes for 192.
//
// WIDE leaves no room for both FP32 sums (re and im) of every output in
// registers, so a tile runs its three products one after the other over all
// of K: the epilogue warps hold ONE product's FP32 sums (64 tones a thread)
// and park each product in a scratch of the CTA (L2-resident).  Finisher warps
// fetch a parked tile back by bulk copies, combine, rotate and store it while
// the next tile's first two products run.  (Done by the epilogue warps at the
// tile's end it stalled the MMAs, which run at most two chunks ahead, by about
// 50,000 clocks of 400,000 per tile; finishers with register loads could not
// keep enough bytes in flight either.)  Two finisher warps take some 120,000
// clocks a tile, more than the MMAs of filters up to 2500 taps, so short filters
// take tiles of up to 128 tones instead: the first product's sums wait in
// TMEM (its last 128 columns, beside three accumulators), the epilogue holds
// im = 2 P1 + P2 and P3 of 32 tones a thread and stores the outputs itself.
//
// Measured, 2^27 samples x 2048 tones, L = 4096, D = 2048, whole push: 7.6 ms
// with tiles of 128 x 128 on one SM, 6.0 ms with pairs (short runs; 6.4 ms in
// seconds-long runs under the power cap).  The MMAs alone would take 3.84 ms
// at 2.07 GHz.  2^24 samples x 1000 tones, L = 1024, D = 512: 579 us with tiles
// of 128 x 128 on one SM, 630 with wide pairs, 447 with pairs of 128 tones;
// L = 256, D = 64: 1650, 3540 and 1280 us.
//
// Precision: the three MMAs of a term set go to the same FP32 TMEM
// accumulator, which collects a chunk of K (128 taps by default) before the
// epilogue adds it into the FP32 sums; two (WIDE) or three accumulators take turns.
// Every form sums each output in the same order (16 taps hi.hi, hi.lo, lo.hi;
// chunks; products), so tile shape, form and the plans sharing a launch never
// change a result.
//
// Forms.  Pairs, wide or of up to 128 tones, as above; the tone tile is narrowed
// (in steps of 32) so that a plan's tones divide evenly.  One CTA per tile of 128
// frames x at most 128 tones where that fills the chip's waves better.  Any form
// may be SPLIT when tiles are few: a work item is then one product of a tile,
// the products go to planes in the scratch and combine3_kernel finishes.
// G3Form::clocks and g3_choose pick by size.
//
// Fused pre-split (FUSED, single-CTA form): instead of TMA loads of the six
// pre-split source planes (written to HBM by prep3_kernel, 12 bytes per
// sample), three producer warps read the int16 stream view [carry | buffer] and
// write each stage's A hi/lo tiles themselves, in the 128-byte swizzled layout
// the TMA would produce, with the same FP32 -> FP16 hi/lo rounding as the
// pre-split kernel (bit-identical planes, so bit-identical results); only the
// B tiles arrive by TMA.  A launch choice the autotuner times.
//
// The kernel is persistent over a list of plans: one launch runs the work
// items of every demodulation stream of a batched step (or of one push), each
// CTA (or pair) striding over the global item index; an item's plan is found
// from the plans' first-item offsets.
constexpr int G3_BK = 64;                                  // complex taps per K-block
constexpr uint32_t G3_OP_BYTES = 128 * G3_BK * 2;          // one operand tile: 128 rows x 64 fp16
constexpr int G3_SLOTS_MAX = 4;
constexpr uint32_t G3_TMEM_COLS = 512;
constexpr int G3_EPI_WARPS = 16;          // 4 lane quadrants x 4 tone groups
constexpr int G3_FUSED_PRODUCERS = 3;                       // producer warps of the fused form
constexpr int G3_WIDE_TONES = 256, G3_TONES = 128;          // widest tone tiles
// scratch of one CTA: a ring of products, [tone][128 frames] FP32 each
constexpr int G3_PLANES = 4;   // a ring: 3 measured 0.8 % slower (6.02 against 5.97 ms, 2^27 samples)
constexpr int64_t G3_PLANE = int64_t(G3_WIDE_TONES) * 128;
constexpr int64_t G3_CTA_SCRATCH = G3_PLANES * G3_PLANE;
// finisher staging: chunks of two tones (three products of 128 frames, then the
// tones' 128 rotation steps), FIN_BUFS chunks per warp in flight
constexpr int G3_FIN_BUFS = 3, G3_FINISHERS = 2;
constexpr uint32_t G3_FIN_BYTES = 3 * 2 * 128 * 4 + 2 * 128 * 8;
constexpr uint32_t G3_BARS_BYTES = 256;
// What the kernel's forms differ in (see the Gauss form's comment).
template <bool PAIR, bool FUSED, bool WIDE>
struct G3Cfg {
    static constexpr int TW = WIDE ? G3_WIDE_TONES : G3_TONES;             // columns of a TMEM slot
    static constexpr int SLOTS = WIDE ? 2 : 3;
    static constexpr uint32_t PARK = 3 * G3_TONES;                         // not WIDE: the first product's columns
    static constexpr uint32_t B_BYTES = PAIR ? TW / 2 * G3_BK * 2 : TW * G3_BK * 2;   // of a CTA's rows of B
    static constexpr uint32_t STAGE_BYTES = 2 * G3_OP_BYTES + 2 * B_BYTES;  // A hi, A lo, B hi, B lo
    static constexpr int STAGES = STAGE_BYTES > 48 * 1024 ? 3 : 4;
    static constexpr int FINISHERS = WIDE ? G3_FINISHERS : 0;
    static constexpr int MMA_WARP = G3_EPI_WARPS + (FUSED ? G3_FUSED_PRODUCERS : 1);
    static constexpr int THREADS = (MMA_WARP + 1 + FINISHERS) * 32;
    static constexpr size_t SMEM = 1024 + STAGES * STAGE_BYTES + G3_BARS_BYTES + FINISHERS * G3_FIN_BUFS * G3_FIN_BYTES;
};

struct G3Plan {
    CUtensorMap a[6];   // (x sum/2, xr, xi) x (hi, lo): [rows][D] fp16, Toeplitz view (unused when fused)
    CUtensorMap b[6];   // (cr, ci - cr, cr + ci) x (hi, lo): [ntp][Lpad] fp16, K-major
    GemmArgs g;         // n_mt, n_nt: tiles (of a pair in the pair form); kchunk: half K-blocks per chunk
    int unit0;          // first global work item of this plan
    int bw;             // tones per tile
    int split;          // work items are single products, written to planes
    float* scratch;     // wide form: [CTA][4][256][128]; split: planes [3][n_tones][pld]
    int64_t pld;
    // fused form: the int16 stream view v[s] = s < cl ? carry[s] : buf[s - cl]
    // for s < lv (0 beyond); vec: the buffer part may be read 16 bytes at a time
    const uint32_t* carry;
    const uint32_t* buf;
    int64_t cl, lv;
    int vec;
};
constexpr int kG3MaxPlans = 16;
struct G3Batch {
    int n_plans, total_units;
    G3Plan p[kG3MaxPlans];
};
static_assert(sizeof(G3Batch) <= 32000, "kernel parameter space");
static_assert(sizeof(G3Plan) <= kDemodJobBytes, "job storage");

__device__ __forceinline__ const G3Plan& g3_plan_of(const G3Batch& bt, int unit) {
    int pi = 0;
    while (pi + 1 < bt.n_plans && unit >= bt.p[pi + 1].unit0) ++pi;
    return bt.p[pi];
}

// A work item: frame tile origin (of this CTA), tone tile origin and width,
// products [q0, q1).  `width` is a multiple of the MMA's N step.
struct G3Unit {
    int64_t m0;
    int n0, width, q0, q1;
};
template <bool PAIR>
__device__ __forceinline__ G3Unit g3_unit(const G3Plan& P, int unit, int rank) {
    int local = unit - P.unit0;
    G3Unit u;
    u.q0 = 0;
    u.q1 = 3;
    if (P.split) {
        u.q0 = local % 3;
        u.q1 = u.q0 + 1;
        local /= 3;
    }
    int mt, nt;
    tile_coords(P.g, local, mt, nt);
    u.m0 = PAIR ? static_cast<int64_t>(mt) * 256 + rank * 128 : static_cast<int64_t>(mt) * BM;
    u.n0 = nt * P.bw;
    constexpr int step = PAIR ? 32 : 16;
    u.width = min(P.bw, (P.g.n_tones - u.n0 + step - 1) / step * step);
    return u;
}

__global__ void build_taps3_kernel(const double* __restrict__ h, const uint64_t* __restrict__ words,
                                   int n_tones, int ntp, int L, int Lpad, double scale,
                                   __half* __restrict__ planes) {
    const int64_t total = static_cast<int64_t>(ntp) * Lpad;
    for (int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; idx < total;
         idx += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int t = static_cast<int>(idx / Lpad);
        const int n = static_cast<int>(idx - static_cast<int64_t>(t) * Lpad);
        double cr = 0.0, ci = 0.0;
        if (t < n_tones && n < L) {
            const uint64_t ph = words[t] * static_cast<uint64_t>(n);
            const double xs = static_cast<double>(static_cast<int64_t>(ph)) * 0x1p-63;
            double sn, cs;
            sincospi(xs, &sn, &cs);
            const double a = h[n] * scale;
            cr = a * cs;
            ci = -a * sn;
        }
        const double v[3] = {cr, ci - cr, cr + ci};
#pragma unroll
        for (int q = 0; q < 3; ++q) split_store(planes + (2 * q) * total, planes + (2 * q + 1) * total, idx, v[q]);
    }
}

// Plane q ((xr+xi)/2, xr or xi; exact in FP32) of two samples -> packed FP16 hi and lo.
__device__ __forceinline__ void g3_split_pair(uint32_t w0, uint32_t w1, int q, uint32_t& hi, uint32_t& lo) {
    const float2 f0 = iq_to_f2(w0), f1 = iq_to_f2(w1);
    const float v0 = q == 0 ? 0.5f * (f0.x + f0.y) : (q == 1 ? f0.x : f0.y);
    const float v1 = q == 0 ? 0.5f * (f1.x + f1.y) : (q == 1 ? f1.x : f1.y);
    const __half h0 = __float2half_rn(v0), h1 = __float2half_rn(v1);
    const __half l0 = __float2half_rn(v0 - __half2float(h0));
    const __half l1 = __float2half_rn(v1 - __half2float(h1));
    hi = static_cast<uint32_t>(__half_as_ushort(h0)) | (static_cast<uint32_t>(__half_as_ushort(h1)) << 16);
    lo = static_cast<uint32_t>(__half_as_ushort(l0)) | (static_cast<uint32_t>(__half_as_ushort(l1)) << 16);
}

// What a three-product push needs ahead of its GEMM, in one launch: the first
// rot_blocks blocks write the rotation tables (FP64-bound), the others the six
// source planes (memory-bound), so the two overlap.
//   anchors, steps: as rot_kernel, in runs of 8 absolute indices from one exact
// FP64 evaluation each, the others by FP64 products with the run's step (within
// 8 x 2^-52 of exact, far inside the FP32 rounding; runs start at absolute
// multiples of 8, so every push of a stream gets the same values).  FP64 issues
// one warp instruction in 16 clocks on an SM, so a block takes `rot_items` threads'
// worth of runs, few enough that all SMs share a small push's.
//   planes: eight samples s of [carry | buffer] per thread -> ((xr+xi)/2, xr,
// xi) x (hi, lo), one 16-byte store per plane.
// Measured: 300 tones x 10^6 samples 47.0 -> 38.6 us a push (two launches, 11.4 us,
// before); of a push of 2^27 samples x 2048 tones 555 -> 343 us (its bytes: 316).
constexpr int kRotRun = 8;
struct Prep3Args {
    const uint64_t* words;
    int n_tones, ntp, L, D, n_anch, rot_blocks, rot_items;
    int64_t A0;                      // first anchor's absolute index
    float2* anchors;
    float2* steps;
    const uint32_t* carry;
    const uint32_t* buf;
    int64_t cl, lv, total;           // total: samples of a plane (a multiple of 64); 0: no planes
    __half* planes;
};
__global__ void __launch_bounds__(256) prep3_kernel(const Prep3Args a) {
    if (static_cast<int>(blockIdx.x) < a.rot_blocks) {
        const int64_t runs0 = a.A0 / kRotRun;
        const int64_t n_runs = (a.A0 + a.n_anch - 1) / kRotRun - runs0 + 1;
        const int64_t na = n_runs * a.ntp, total = na + static_cast<int64_t>(a.ntp) * (BM / kRotRun);
        if (static_cast<int>(threadIdx.x) >= a.rot_items) return;
        for (int64_t idx = static_cast<int64_t>(blockIdx.x) * a.rot_items + threadIdx.x; idx < total;
             idx += static_cast<int64_t>(a.rot_blocks) * a.rot_items) {
            const bool anchor = idx < na;
            const int64_t j = anchor ? idx : idx - na;
            const int t = static_cast<int>(j % a.ntp);
            const int64_t run = j / a.ntp;                   // of anchors (from runs0) or of steps
            double c = 0.0, sn = 0.0, dc = 0.0, ds = 0.0;
            if (t < a.n_tones) {
                const uint64_t w = a.words[t];
                const int64_t K = (runs0 + run) * kRotRun * BM;
                const uint64_t ph = w * static_cast<uint64_t>(anchor ? (K + 1) * a.D - a.L : run * kRotRun * a.D);
                const uint64_t dp = w * static_cast<uint64_t>(anchor ? static_cast<int64_t>(BM) * a.D : static_cast<int64_t>(a.D));
                sincospi(static_cast<double>(static_cast<int64_t>(ph)) * 0x1p-63, &sn, &c);
                sincospi(static_cast<double>(static_cast<int64_t>(dp)) * 0x1p-63, &ds, &dc);
            }
#pragma unroll 4
            for (int i = 0; i < kRotRun; ++i) {
                const float2 r = make_float2(static_cast<float>(c), static_cast<float>(-sn));
                if (anchor) {
                    const int64_t row = (runs0 + run) * kRotRun + i - a.A0;
                    if (row >= 0 && row < a.n_anch) a.anchors[row * a.ntp + t] = r;
                } else {
                    a.steps[static_cast<int64_t>(t) * BM + run * kRotRun + i] = r;
                }
                const double nc = fma(c, dc, -sn * ds);
                sn = fma(c, ds, sn * dc);
                c = nc;
            }
        }
        return;
    }
    const int64_t nb = gridDim.x - a.rot_blocks;
    for (int64_t g = (blockIdx.x - a.rot_blocks) * 256 + threadIdx.x; g < a.total / 8; g += nb * 256) {
        const int64_t s0 = g * 8;
        uint32_t w[8];
        const uint32_t* bp = a.buf + (s0 - a.cl);
        if (s0 >= a.cl && s0 + 8 <= a.lv && (reinterpret_cast<uintptr_t>(bp) & 15) == 0) {
            const uint4 u0 = __ldg(reinterpret_cast<const uint4*>(bp)), u1 = __ldg(reinterpret_cast<const uint4*>(bp) + 1);
            w[0] = u0.x; w[1] = u0.y; w[2] = u0.z; w[3] = u0.w;
            w[4] = u1.x; w[5] = u1.y; w[6] = u1.z; w[7] = u1.w;
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int64_t s = s0 + e;
                w[e] = s < a.lv ? (s < a.cl ? __ldg(a.carry + s) : __ldg(a.buf + (s - a.cl))) : 0u;
            }
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int e = 0; e < 8; e += 2) g3_split_pair(w[e], w[e + 1], q, hi[e / 2], lo[e / 2]);
            *reinterpret_cast<uint4*>(a.planes + (2 * q) * a.total + s0) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4*>(a.planes + (2 * q + 1) * a.total + s0) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
    }
}

// Fused pre-split: chunk c (8 samples) of row i of a stage's A hi/lo tiles of plane q,
// the samples from s on, in the 128-byte swizzled layout of the TMA loads (16-byte
// chunk c of row i at chunk c ^ (i & 7)).  Eight lanes take a row, so that a warp
// reads runs of 256 bytes.
__device__ __forceinline__ void g3_fill_chunk(const G3Plan& P, int q, int64_t s, unsigned char* ahi, unsigned char* alo,
                                              int i, int c) {
    uint32_t w[8];
    const uint32_t* bp = P.buf + (s - P.cl);
    if (P.vec && s >= P.cl && s + 8 <= P.lv && (reinterpret_cast<uintptr_t>(bp) & 15) == 0) {
        const uint4 u0 = __ldg(reinterpret_cast<const uint4*>(bp)), u1 = __ldg(reinterpret_cast<const uint4*>(bp) + 1);
        w[0] = u0.x; w[1] = u0.y; w[2] = u0.z; w[3] = u0.w;
        w[4] = u1.x; w[5] = u1.y; w[6] = u1.z; w[7] = u1.w;
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int64_t sv = s + e;
            w[e] = sv < P.lv ? (sv < P.cl ? __ldg(P.carry + sv) : __ldg(P.buf + (sv - P.cl))) : 0u;
        }
    }
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 8; e += 2) g3_split_pair(w[e], w[e + 1], q, hi[e / 2], lo[e / 2]);
    const uint32_t off = static_cast<uint32_t>(i) * 128u + (static_cast<uint32_t>(c ^ (i & 7)) << 4);
    *reinterpret_cast<uint4*>(ahi + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(alo + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
}

// An output from its products (re, im) and rotation factors.
__device__ __forceinline__ float2 g3_rotate(float re, float im, float inv_scale, float2 an, float2 sp) {
    return cmul(make_float2(re * inv_scale, im * inv_scale), cmul(an, sp));
}
__device__ __forceinline__ float2 g3_output(float p1, float p2, float p3, float inv_scale, float2 an, float2 sp) {
    return g3_rotate(fmaf(2.f, p1, -p3), fmaf(2.f, p1, p2), inv_scale, an, sp);
}

// Outputs of a CTA's last tile, by all its epilogue and finisher warps (in 16-byte
// loads: frames l + 32 r a lane in 4-byte ones took 20 us more, 237 -> 256 for a push
// of one wave with L = 4096): lane l
// takes frames 4 l .. 4 l + 3, warp w of nw (less the `skip` producer and MMA
// warps between the two kinds) every tone of its number, FT in flight.
__device__ __noinline__ void g3_finish(const G3Plan& P, const G3Unit u, const float* scr_cta, uint32_t tile, int lane,
                                          int w, int nw, int skip) {
    constexpr int FT = 2;
    const GemmArgs& g = P.g;
    if (w >= G3_EPI_WARPS) w -= skip;
    nw -= skip;
    const float* pl[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) pl[q] = scr_cta + ((3 * tile + q) % G3_PLANES) * G3_PLANE + 4 * lane;
    const int64_t k = u.m0 + 4 * lane;               // the lane's first frame
    const int64_t K = g.F0 + k;
    const int rows = static_cast<int>(k < g.F ? (g.F - k < 4 ? g.F - k : 4) : 0);
    if (rows == 0) return;
    // four frames of one anchor row, with aligned steps; 16-byte stores
    const bool near = (g.F0 & 3) == 0;
    const bool vec = rows == 4 && ((reinterpret_cast<uintptr_t>(g.out + g.fo + k) | static_cast<uintptr_t>(g.ld * 8)) & 15) == 0;
    const int n = min(u.width, g.n_tones - u.n0);
#pragma unroll 1
    for (int c0 = w; c0 < n; c0 += nw * FT) {
        float p[FT][3][4];
        float2 an[FT][4], sp[FT][4];
#pragma unroll
        for (int f = 0; f < FT; ++f) {
            const int c = c0 + f * nw, t = u.n0 + c;
            if (c >= n) continue;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float4 v = __ldcg(reinterpret_cast<const float4*>(pl[q] + c * 128));
                p[f][q][0] = v.x;
                p[f][q][1] = v.y;
                p[f][q][2] = v.z;
                p[f][q][3] = v.w;
            }
            const float2* anc = g.anchors + t - (g.F0 / BM) * g.ntp;
            const float2* stp = g.steps + static_cast<int64_t>(t) * BM;
            if (near) {
                an[f][0] = __ldg(anc + (K / BM) * g.ntp);
                an[f][1] = an[f][2] = an[f][3] = an[f][0];
                const float4* s4 = reinterpret_cast<const float4*>(stp + static_cast<int>(K % BM));
                const float4 s0 = __ldg(s4), s1 = __ldg(s4 + 1);
                sp[f][0] = make_float2(s0.x, s0.y);
                sp[f][1] = make_float2(s0.z, s0.w);
                sp[f][2] = make_float2(s1.x, s1.y);
                sp[f][3] = make_float2(s1.z, s1.w);
            } else {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int64_t Kr = r < rows ? K + r : K;
                    an[f][r] = __ldg(anc + (Kr / BM) * g.ntp);
                    sp[f][r] = __ldg(stp + static_cast<int>(Kr % BM));
                }
            }
        }
#pragma unroll
        for (int f = 0; f < FT; ++f) {
            const int c = c0 + f * nw, t = u.n0 + c;
            if (c >= n) continue;
            float2* o = g.out + static_cast<int64_t>(t) * g.ld + g.fo + k;
            float2 y[4];
#pragma unroll
            for (int r = 0; r < 4; ++r)
                y[r] = g3_output(p[f][0][r], p[f][1][r], p[f][2][r], g.inv_scale, an[f][r], sp[f][r]);
            if (vec) {
                reinterpret_cast<float4*>(o)[0] = make_float4(y[0].x, y[0].y, y[1].x, y[1].y);
                reinterpret_cast<float4*>(o)[1] = make_float4(y[2].x, y[2].y, y[3].x, y[3].y);
            } else {
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    if (r < rows) o[r] = y[r];
            }
        }
    }
}

// PAIR: launched in clusters of two CTAs on one tile of 256 frames.  Both CTAs
// load their own operand halves, counted on the full barriers of CTA 0, whose
// MMA thread issues for both; its commits arrive on both CTAs' barriers, and
// the epilogue warps of both report drained slots to CTA 0.  The CTAs meet at
// cluster barriers after initialising their mbarriers and before leaving.
// The mbarriers order tensor-core and TMA work only (no ordinary loads or
// stores pass between the CTAs), so plain waits do; acquiring at cluster
// scope put a memory barrier into every wait.
template <bool PAIR, bool FUSED, bool WIDE>
__global__ void __launch_bounds__(G3Cfg<PAIR, FUSED, WIDE>::THREADS, 1)
demod3m_gemm_kernel(const __grid_constant__ G3Batch bt) {
    static_assert(!(FUSED && PAIR), "the pair form loads its A tiles by TMA");
    static_assert(PAIR || !WIDE, "wide tiles are a pair's");
    using Cfg = G3Cfg<PAIR, FUSED, WIDE>;
    constexpr int STAGES = Cfg::STAGES, TW = Cfg::TW, SLOTS = Cfg::SLOTS;
    constexpr uint32_t STAGE_BYTES = Cfg::STAGE_BYTES, B_BYTES = Cfg::B_BYTES;
    constexpr int TPG = TW / 4;                                             // tones per epilogue thread, at most
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    unsigned char* smem = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* sfull = empty + STAGES;
    uint64_t* sempty = sfull + G3_SLOTS_MAX;
    uint64_t* parked = sempty + G3_SLOTS_MAX;                               // a tile's products are in the scratch
    uint64_t* finished = parked + 1;                                        // ... and its outputs stored
    uint64_t* fbar = finished + 1;                                          // finisher staging, per warp and buffer
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(fbar + G3_FINISHERS * G3_FIN_BUFS);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
    unsigned char* const fin_stage = smem + STAGES * STAGE_BYTES + G3_BARS_BYTES;
    int* const status0 = bt.p[0].g.status;
    constexpr int PROD_WARP = G3_EPI_WARPS;                                  // first producer warp
    constexpr int MMA_WARP = Cfg::MMA_WARP, FIN_WARP = MMA_WARP + 1, FINISHERS = Cfg::FINISHERS;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = PAIR ? static_cast<int>(cluster_ctarank()) : 0;
    const int first = PAIR ? static_cast<int>(blockIdx.x >> 1) : static_cast<int>(blockIdx.x);
    const int stride = PAIR ? static_cast<int>(gridDim.x >> 1) : static_cast<int>(gridDim.x);
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], FUSED ? G3_FUSED_PRODUCERS * 32 : 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < SLOTS; ++b) {
            mbar_init(&sfull[b], 1);
            mbar_init(&sempty[b], (PAIR ? 2 : 1) * G3_EPI_WARPS);
        }
        if constexpr (WIDE) {
            mbar_init(parked, G3_EPI_WARPS);
            mbar_init(finished, FINISHERS);
            for (int b = 0; b < FINISHERS * G3_FIN_BUFS; ++b) mbar_init(&fbar[b], 1);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == MMA_WARP) {
        umma::alloc<PAIR>(tmem_holder, G3_TMEM_COLS);
        umma::relinquish<PAIR>();
    }
    if (warp == PROD_WARP && lane < bt.n_plans) {
        for (int i = 0; i < 6; ++i) {
            if (!FUSED) tma_prefetch_desc(&bt.p[lane].a[i]);
            tma_prefetch_desc(&bt.p[lane].b[i]);
        }
    }
    umma::fence_before_sync();
    __syncthreads();
    if (PAIR) cluster_sync();          // both CTAs' barriers exist before anything arrives on them
    umma::fence_after_sync();
    const uint32_t tmem = *tmem_holder;
    const int n_units = bt.total_units;
    allow_dependents();
    float* const scr_cta = WIDE ? bt.p[0].scratch + static_cast<int64_t>(blockIdx.x) * G3_CTA_SCRATCH : nullptr;

    if (FUSED && warp >= PROD_WARP && warp < MMA_WARP) {
        // ------------------------------------------------ fused producers
        const int pt = threadIdx.x - PROD_WARP * 32;                         // 0 .. 95
        uint32_t it = 0;
        bool stop = false;
        for (int unit = first; unit < n_units && !stop; unit += stride) {
            const G3Plan& P = g3_plan_of(bt, unit);
            const G3Unit u = g3_unit<PAIR>(P, unit, rank);
            const int64_t D = P.g.two_d;
            for (int q = u.q0; q < u.q1 && !stop; ++q) {
                for (int kb = 0; kb < P.g.KB; ++kb, ++it) {
                    const int s = it % STAGES;
                    const uint32_t ph = (it / STAGES) & 1;
                    if (*abort_flag || !mbar_wait(&empty[s], ph ^ 1, status0)) {
                        *abort_flag = 1;
                        stop = true;
                        break;
                    }
                    unsigned char* st = smem + s * STAGE_BYTES;
                    const int kt = kb * G3_BK;
                    if (pt == 0) {
                        mbar_expect_tx(&full[s], 2u * P.bw * (G3_BK * 2));
                        tma_load_2d(st + 2 * G3_OP_BYTES, &P.b[2 * q], kt, u.n0, &full[s]);
                        tma_load_2d(st + 2 * G3_OP_BYTES + B_BYTES, &P.b[2 * q + 1], kt, u.n0, &full[s]);
                    }
#pragma unroll 2
                    for (int e = pt; e < BM * (G3_BK / 8); e += G3_FUSED_PRODUCERS * 32) {
                        const int i = e / (G3_BK / 8), c = e % (G3_BK / 8);
                        g3_fill_chunk(P, q, (u.m0 + i) * D + kt + 8 * c, st, st + G3_OP_BYTES, i, c);
                    }
                    fence_proxy_async_smem();                 // the MMAs read the tiles through the async proxy
                    mbar_arrive(&full[s]);
                }
            }
        }
        // the B copies still in flight complete before the CTA exits
        if (pt == 0) {
            for (uint32_t k = 0; k < static_cast<uint32_t>(STAGES) && it > 0; ++k) {
                const uint32_t j = it - 1 - k;
                if (static_cast<int32_t>(j) < 0) break;
                mbar_wait(&full[j % STAGES], (j / STAGES) & 1, status0);
            }
        }
    } else if (!FUSED && warp == PROD_WARP) {
        // ------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t it = 0;
            bool stop = false;
            for (int unit = first; unit < n_units && !stop; unit += stride) {
                const G3Plan& P = g3_plan_of(bt, unit);
                const G3Unit u = g3_unit<PAIR>(P, unit, rank);
                // rows of a B box: the tile's tones, or this CTA's half of them
                const uint32_t box = PAIR ? P.bw / 2 : P.bw;
                const uint32_t bytes = 2 * G3_OP_BYTES + 2 * box * (G3_BK * 2);
                const int b0 = PAIR ? u.n0 + rank * (u.width / 2) : u.n0;
                for (int q = u.q0; q < u.q1 && !stop; ++q) {
                    for (int kb = 0; kb < P.g.KB; ++kb, ++it) {
                        const int s = it % STAGES;
                        const uint32_t ph = (it / STAGES) & 1;
                        if (*abort_flag || !mbar_wait(&empty[s], ph ^ 1, status0)) {
                            *abort_flag = 1;
                            stop = true;
                            break;
                        }
                        unsigned char* st = smem + s * STAGE_BYTES;
                        const int kt = kb * G3_BK;
                        const int c0 = kt % P.g.two_d, c1 = static_cast<int>(u.m0) + kt / P.g.two_d;
                        if constexpr (PAIR) {
                            // both CTAs' bytes are counted on CTA 0's barrier
                            if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * bytes);
                            const uint32_t fb = cluster_addr(&full[s], 0);
                            tma_load_2d_2sm(st, &P.a[2 * q], c0, c1, fb);
                            tma_load_2d_2sm(st + G3_OP_BYTES, &P.a[2 * q + 1], c0, c1, fb);
                            tma_load_2d_2sm(st + 2 * G3_OP_BYTES, &P.b[2 * q], kt, b0, fb);
                            tma_load_2d_2sm(st + 2 * G3_OP_BYTES + B_BYTES, &P.b[2 * q + 1], kt, b0, fb);
                        } else {
                            mbar_arrive_expect_tx(&full[s], bytes);
                            tma_load_2d(st, &P.a[2 * q], c0, c1, &full[s]);
                            tma_load_2d(st + G3_OP_BYTES, &P.a[2 * q + 1], c0, c1, &full[s]);
                            tma_load_2d(st + 2 * G3_OP_BYTES, &P.b[2 * q], kt, b0, &full[s]);
                            tma_load_2d(st + 2 * G3_OP_BYTES + B_BYTES, &P.b[2 * q + 1], kt, b0, &full[s]);
                        }
                    }
                }
            }
            // wait for the copies still in flight before leaving (CTA 0 of a
            // pair for both CTAs' copies)
            for (uint32_t k = 0; rank == 0 && k < static_cast<uint32_t>(STAGES) && it > 0; ++k) {
                const uint32_t j = it - 1 - k;
                if (static_cast<int32_t>(j) < 0) break;
                mbar_wait(&full[j % STAGES], (j / STAGES) & 1, status0);
            }
            // pair form: and for the last commits to this CTA's empty
            // barriers, so that nothing arrives here after the CTA has left
            for (uint32_t k = 0; PAIR && k < static_cast<uint32_t>(STAGES) && it > 0; ++k) {
                const uint32_t j = it - 1 - k;
                if (static_cast<int32_t>(j) < 0) break;
                mbar_wait(&empty[j % STAGES], (j / STAGES) & 1, status0);
            }
        }
    } else if (warp == MMA_WARP) {
        // ------------------------------------------------ MMA issuer
        // The whole warp runs the loops and one elected thread issues, so that control
        // flow, descriptors and addresses stay in uniform registers.  (Run by one thread
        // alone, every MMA took about 115 clocks to issue whatever its width: 1370 a
        // K-block, where tiles of 128 tones need 960.)  Wide tiles' MMAs take 128 each:
        // there one thread runs alone.
        if (rank == 0 && (!WIDE || lane == 0)) {
            const bool leader = WIDE || umma::elect_one();
            auto agreed = [](bool ok) {
                if constexpr (WIDE) return ok;
                else return static_cast<bool>(__all_sync(0xffffffffu, ok));
            };
            const uint64_t desc0 = umma::desc_k_sw128(smem_u32(smem));
            uint32_t phase = 0, s = 0, par = 0;             // chunk; stage and the parity of its use
            bool go = true;
            for (int unit = first; unit < n_units && go; unit += stride) {
                const G3Plan& P = g3_plan_of(bt, unit);
                const GemmArgs& g = P.g;
                const G3Unit u = g3_unit<PAIR>(P, unit, rank);
                const uint32_t idesc = umma::idesc_f16_f32(PAIR ? 256 : 128, u.width);
                const int H = 2 * g.KB, chunk = g.kchunk;
                for (int q = u.q0; q < u.q1 && go; ++q) {
                    // chunks of half K-blocks (32 taps); chunks of whole blocks have their own
                    // loop (a block's twelve MMAs in two pieces: 800 us where this took 733,
                    // 2^24 samples x 2048 tones)
                    for (int h0 = 0; h0 < H && go; h0 += chunk, ++phase) {
                        const int h1 = min(h0 + chunk, H);
                        const uint32_t slot = phase % SLOTS, use = phase / SLOTS;
                        go = agreed(!*abort_flag && mbar_wait(&sempty[slot], (use & 1) ^ 1, status0));
                        if (!go) break;
                        umma::fence_after_sync();
                        const uint32_t d_tmem = tmem + slot * TW;
                        auto arrived = [&] {                            // the block's operands
                            go = agreed(mbar_wait(&full[s], par, status0));
                            umma::fence_after_sync();
                            return go;
                        };
                        auto release = [&] {                            // its stage, in both CTAs of a pair
                            if (leader) {
                                if constexpr (PAIR) umma::commit_2sm(&empty[s]);
                                else umma::commit(&empty[s]);
                            }
                            if (++s == STAGES) {
                                s = 0;
                                par ^= 1u;
                            }
                        };
                        auto steps = [&](auto n, uint32_t from, bool fresh) {   // n steps of 16 taps
                            const uint64_t ah = desc0 + ((s * STAGE_BYTES + from) >> 4);
                            const uint64_t al = ah + (G3_OP_BYTES >> 4), bh = ah + (2 * G3_OP_BYTES >> 4), bl = bh + (B_BYTES >> 4);
                            if (leader) {
#pragma unroll
                                for (int k = 0; k < n; ++k) {
                                    const uint32_t acc = (!fresh || k > 0) ? 1u : 0u;
                                    if constexpr (PAIR) {
                                        umma::mma_f16_2sm(d_tmem, ah + 2 * k, bh + 2 * k, idesc, acc);
                                        umma::mma_f16_2sm(d_tmem, ah + 2 * k, bl + 2 * k, idesc, 1u);
                                        umma::mma_f16_2sm(d_tmem, al + 2 * k, bh + 2 * k, idesc, 1u);
                                    } else {
                                        umma::mma_f16(d_tmem, ah + 2 * k, bh + 2 * k, idesc, acc);
                                        umma::mma_f16(d_tmem, ah + 2 * k, bl + 2 * k, idesc, 1u);
                                        umma::mma_f16(d_tmem, al + 2 * k, bh + 2 * k, idesc, 1u);
                                    }
                                }
                            }
                        };
                        if ((chunk & 1) == 0) {
                            for (int h = h0; h < h1; h += 2) {
                                if (!arrived()) break;
                                steps(std::integral_constant<int, G3_BK / 16>{}, 0, h == h0);
                                release();
                            }
                        } else {
                            for (int h = h0; h < h1; ++h) {
                                if ((h & 1) == 0 && !arrived()) break;
                                steps(std::integral_constant<int, G3_BK / 32>{}, (h & 1) * G3_BK, h == h0);
                                if (h & 1) release();
                            }
                        }
                        if (leader) {
                            if constexpr (PAIR) umma::commit_2sm(&sfull[slot]);
                            else umma::commit(&sfull[slot]);
                        }
                    }
                }
            }
            if (!go) *abort_flag = 1;
        }
        __syncwarp();
    } else if (warp < G3_EPI_WARPS) {
        // ------------------------------------------------ epilogue (16 warps)
        const int qd = warp & 3, grp = warp >> 2;          // lane quadrant, tone group
        const int row = qd * 32 + lane;
        const uint32_t lanes = tmem + (static_cast<uint32_t>(qd * 32) << 16);
        uint32_t phase = 0, tile = 0;
        bool ok = true;
        // this thread's column of the CTA's scratch planes
        float* const scr = WIDE ? scr_cta + grp * TPG * 128 + row : nullptr;
        for (int unit = first; unit < n_units && ok; unit += stride) {
            const G3Plan& P = g3_plan_of(bt, unit);
            const GemmArgs& g = P.g;
            const G3Unit u = g3_unit<PAIR>(P, unit, rank);
            // this thread's tones (cols: a multiple of 16, or <= 0), from c0 on
            const int tpg = WIDE || u.width > 64 ? TPG : 16, c0 = grp * tpg, cols = min(tpg, u.width - c0);
            const int64_t k = u.m0 + row;                             // and its frame
            float sum[TPG], im[WIDE ? 1 : TPG];
            for (int q = u.q0; q < u.q1 && ok; ++q) {
#pragma unroll
                for (int i = 0; i < TPG; ++i) sum[i] = 0.f;
                for (int h0 = 0; h0 < 2 * g.KB; h0 += g.kchunk, ++phase) {
                    const uint32_t slot = phase % SLOTS, use = phase / SLOTS;
                    if (*abort_flag || !mbar_wait(&sfull[slot], use & 1, status0)) {
                        *abort_flag = 1;
                        ok = false;
                        break;
                    }
                    umma::fence_after_sync();
                    const uint32_t ta = lanes + slot * TW + c0;
#pragma unroll
                    for (int h = 0; h < TPG; h += 16) {
                        if (h < cols) {
                            uint32_t r0[16];
                            umma::ld_32x32b_x16(ta + h, r0);
                            umma::wait_ld_regs(r0);
#pragma unroll
                            for (int i = 0; i < 16; ++i) sum[h + i] += __uint_as_float(r0[i]);
                        }
                    }
                    umma::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) {
                        if constexpr (PAIR) mbar_arrive_cluster(cluster_addr(&sempty[slot], 0));
                        else mbar_arrive(&sempty[slot]);
                    }
                }
                if (!ok) break;
                if (P.split) {
                    const int tb = u.n0 + c0;
                    if (k < g.F) {
                        float* pl = P.scratch + (static_cast<int64_t>(q) * g.n_tones + tb) * P.pld + k;
#pragma unroll
                        for (int i = 0; i < TPG; ++i, pl += P.pld)
                            if (i < cols && tb + i < g.n_tones) *pl = sum[i];
                    }
                    continue;
                }
                if constexpr (WIDE) {
                    // the first product to reuse a plane of the tile before, which
                    // has to be finished by then
                    if (q == G3_PLANES - 3 && tile > 0 && !mbar_wait(finished, (tile - 1) & 1, status0)) {
                        *abort_flag = 1;
                        ok = false;
                        break;
                    }
                    float* const pl = scr + ((3 * tile + q) % G3_PLANES) * G3_PLANE;
#pragma unroll
                    for (int i = 0; i < TPG; ++i)
                        if (i < cols) pl[i * 128] = sum[i];
                } else if (q == 0) {
                    // P1 waits in this thread's own TMEM columns
                    if (cols > 0) {
                        uint32_t w[TPG];
#pragma unroll
                        for (int i = 0; i < TPG; ++i) w[i] = __float_as_uint(sum[i]);
                        umma::st_32x32b_x32(lanes + Cfg::PARK + grp * TPG, w);
                        umma::wait_st();
                    }
                } else {
                    // im = 2 P1 + P2; re = 2 P1 - P3 and the outputs, their
                    // arithmetic that of g3_output
#pragma unroll
                    for (int h = 0; h < TPG; h += 16) {
                        if (h < cols) {
                            uint32_t p1[16];
                            umma::ld_32x32b_x16(lanes + Cfg::PARK + grp * TPG + h, p1);
                            umma::wait_ld_regs(p1);
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                if (q == 1) im[h + i] = fmaf(2.f, __uint_as_float(p1[i]), sum[h + i]);
                                else sum[h + i] = fmaf(2.f, __uint_as_float(p1[i]), -sum[h + i]);
                            }
                        }
                    }
                    const int n = min(cols, g.n_tones - u.n0 - c0);
                    if (q == 2 && k < g.F && n > 0) {
                        const float2* const anc = g.anchors + ((g.F0 + k) / BM - g.F0 / BM) * g.ntp + u.n0 + c0;
                        const float2* const stp = g.steps + static_cast<int64_t>(u.n0 + c0) * BM + static_cast<int>((g.F0 + k) % BM);
                        float2* const out = g.out + static_cast<int64_t>(u.n0 + c0) * g.ld + g.fo + k;
                        // (loads four tones at a time, unconditional: one by one their
                        // latency adds up to more than the MMAs run ahead)
#pragma unroll
                        for (int h = 0; h < TPG; h += 4) {
                            if (h >= n) break;
                            float2 an[4], sp[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const int t = min(h + i, n - 1);
                                an[i] = __ldg(anc + t);
                                sp[i] = __ldg(stp + t * BM);
                            }
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                if (h + i < n) out[(h + i) * g.ld] = g3_rotate(sum[h + i], im[h + i], g.inv_scale, an[i], sp[i]);
                        }
                    }
                }
            }
            if constexpr (WIDE) {
                if (ok && !P.split) {
                    fence_proxy_async_global();              // the finishers read the planes by bulk copies
                    __syncwarp();
                    if (lane == 0) mbar_arrive(parked);
                    if (unit + stride >= n_units && mbar_wait(parked, tile & 1, status0))
                        g3_finish(P, u, scr_cta, tile, lane, warp, Cfg::THREADS / 32, FIN_WARP - G3_EPI_WARPS);
                    ++tile;
                }
            }
        }
    } else if constexpr (WIDE) {
        // ------------------------------------------------ finishers
        const int w = warp - FIN_WARP;
        unsigned char* const stage = fin_stage + w * G3_FIN_BUFS * G3_FIN_BYTES;
        uint64_t* const bars = fbar + w * G3_FIN_BUFS;
        uint32_t tile = 0, fills = 0;                         // chunks consumed so far (buffer and phase)
        bool ok = true;
        for (int unit = first; unit < n_units && ok; unit += stride) {
            const G3Plan& P = g3_plan_of(bt, unit);
            if (P.split) continue;
            if (*abort_flag || !mbar_wait(parked, tile & 1, status0)) {
                *abort_flag = 1;
                break;
            }
            const G3Unit u = g3_unit<PAIR>(P, unit, rank);
            if (unit + stride >= n_units) {
                // the CTA's last tile: every warp that is free takes part
                g3_finish(P, u, scr_cta, tile, lane, warp, Cfg::THREADS / 32, FIN_WARP - G3_EPI_WARPS);
            } else {
                const GemmArgs& g = P.g;
                const int n = min(u.width, g.n_tones - u.n0);
                // the warp's chunks: tones 2 (w + i FINISHERS), 2 (w + i FINISHERS) + 1
                const int chunks = ((n + 1) / 2 - w + FINISHERS - 1) / FINISHERS;
                // chunk i into its buffer: lanes 0 .. 2 copy the products, lane 3 the steps
                auto fetch = [&](int i) {
                    const uint32_t b = (fills + i) % G3_FIN_BUFS;
                    const int c = 2 * (w + i * FINISHERS);
                    if (lane == 0) mbar_arrive_expect_tx(&bars[b], G3_FIN_BYTES);
                    __syncwarp();
                    if (lane < 4) {
                        const void* src = lane < 3 ? static_cast<const void*>(scr_cta + ((3 * tile + lane) % G3_PLANES) * G3_PLANE + c * 128)
                                                   : g.steps + static_cast<int64_t>(u.n0 + c) * BM;
                        tma_bulk_g2s(stage + b * G3_FIN_BYTES + lane * 1024, src, lane < 3 ? 1024u : 2048u, &bars[b]);
                    }
                };
                for (int i = 0; i < min(chunks, G3_FIN_BUFS); ++i) fetch(i);
                // lane l: frames l + 32 r, so that a warp's loads and stores are runs of
                // frames whatever the rows' alignment (four consecutive frames a lane took
                // 480 clocks a tone in 16-byte stores and more in 8-byte ones); anchor rows
                // a0 and, from row `turn` of the tile on, a0 + 1
                const int64_t k = u.m0 + lane;
                const int f0 = static_cast<int>(g.F0 % BM), turn = BM - f0;
                const float2* const anc = g.anchors + ((g.F0 + u.m0) / BM - g.F0 / BM) * g.ntp + u.n0;
                float2 a_lo = make_float2(0.f, 0.f), a_hi = a_lo;
                for (int i = 0; i < chunks; ++i) {
                    if ((i & 15) == 0) {
                        // anchors of the next 16 chunks, a tone per lane
                        const int c = 2 * (w + (i + (lane >> 1)) * FINISHERS) + (lane & 1);
                        const bool on = c < n;
                        a_lo = on ? __ldg(anc + c) : make_float2(0.f, 0.f);
                        a_hi = on && f0 > 0 && u.m0 + turn < g.F ? __ldg(anc + g.ntp + c) : make_float2(0.f, 0.f);
                    }
                    const uint32_t fi = fills + i;
                    if (!mbar_wait(&bars[fi % G3_FIN_BUFS], (fi / G3_FIN_BUFS) & 1, status0)) {
                        *abort_flag = 1;
                        ok = false;
                        break;
                    }
                    const unsigned char* src = stage + (fi % G3_FIN_BUFS) * G3_FIN_BYTES;
                    float p[2][3][4];
                    float2 sp[2][4], al[2], ah[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int from = ((i & 15) << 1) + h;
                        al[h] = make_float2(__shfl_sync(0xffffffffu, a_lo.x, from), __shfl_sync(0xffffffffu, a_lo.y, from));
                        ah[h] = make_float2(__shfl_sync(0xffffffffu, a_hi.x, from), __shfl_sync(0xffffffffu, a_hi.y, from));
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
#pragma unroll
                            for (int q = 0; q < 3; ++q)
                                p[h][q][r] = *reinterpret_cast<const float*>(src + q * 1024 + h * 512 + r * 128 + lane * 4);
                            sp[h][r] = *reinterpret_cast<const float2*>(src + 3072 + h * 1024 + ((lane + 32 * r + f0) & (BM - 1)) * 8);
                        }
                    }
                    __syncwarp();                             // the buffer has been read
                    if (i + G3_FIN_BUFS < chunks) fetch(i + G3_FIN_BUFS);
                    const int c = 2 * (w + i * FINISHERS);
                    float2* const o = g.out + static_cast<int64_t>(u.n0 + c) * g.ld + g.fo + k;
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const float2 y = g3_output(p[h][0][r], p[h][1][r], p[h][2][r], g.inv_scale,
                                                       lane + 32 * r < turn ? al[h] : ah[h], sp[h][r]);
                            if (c + h < n && k + 32 * r < g.F) o[h * g.ld + 32 * r] = y;
                        }
                }
                fills += chunks;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(finished);
            ++tile;
        }
    }
    umma::fence_before_sync();
    __syncthreads();
    if (PAIR) cluster_sync();          // neither CTA leaves while the other may still signal it
    if (warp == MMA_WARP) {
        umma::fence_after_sync();
        umma::dealloc<PAIR>(tmem, G3_TMEM_COLS);
    }
}

// The split form's last step: planes P1, P2, P3 [n_tones][pld] -> outputs,
// with the arithmetic of the GEMM's own last step.  One thread per output,
// frames along the warp.
__global__ void combine3_kernel(const float* __restrict__ planes, int64_t pld, const GemmArgs g) {
    const int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    allow_dependents();
    if (k >= g.F) return;
    const int64_t K = g.F0 + k;
    const int64_t arow = K / BM - g.F0 / BM;
    const int si = static_cast<int>(K % BM);
    const int64_t plane = static_cast<int64_t>(g.n_tones) * pld;
    for (int t = blockIdx.y; t < g.n_tones; t += gridDim.y) {
        const float* p = planes + t * pld + k;
        g.out[static_cast<int64_t>(t) * g.ld + g.fo + k] =
            g3_output(p[0], p[plane], p[2 * plane], g.inv_scale, __ldg(g.anchors + arow * g.ntp + t),
                      __ldg(g.steps + static_cast<int64_t>(t) * BM + si));
    }
}

// ------------------------------------------------------------ host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(tmap_encode_tiled_fn());
}

// 2-D fp16 tensor [rows][cols] (cols contiguous), box [box_rows][64], 128B swizzle.
bool make_map(CUtensorMap* m, const void* base, uint64_t cols, uint64_t rows, uint32_t box_rows) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {cols * 2};
    cuuint32_t box[2] = {static_cast<cuuint32_t>(BK), box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

unsigned grid_for(int64_t work, int n_sms) {
    return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>((work + 255) / 256, int64_t(n_sms) * 16)));
}

}  // namespace

int demod_anchor_rows(int64_t F0, int64_t F) {
    return static_cast<int>((F0 + F - 1) / BM - F0 / BM + 1);
}

size_t demod_xs_rows(int64_t F, int Lpad, int D) {
    // frame F-1 reads rows F-1 .. F-1 + (Lpad-1)/D
    return static_cast<size_t>(F + (Lpad - 1) / D);
}

namespace {
// Rows of the split form's planes, and whether three planes stay within what the
// unsplit forms may need at most.
int64_t g3_plane_ld(int64_t F) { return (F + 31) / 32 * 32; }
bool g3_planes_fit(int n_tones, int64_t F, int n_sms) {
    return 3 * n_tones * g3_plane_ld(F) * 4 <= static_cast<int64_t>(demod3_scratch_bytes(n_sms));
}
}  // namespace
size_t demod3_scratch_bytes(int ctas) { return static_cast<size_t>(ctas) * G3_CTA_SCRATCH * 4; }
// Wide tiles: 256 frames x 256 tones at most on two CTAs (evened out, no more tiles
// than that).
int demod3_ctas(int n_tones, int64_t F, int n_sms) {
    if (n_tones <= G3_TONES) return 0;
    return static_cast<int>(std::min<int64_t>(
        n_sms, 2 * ((F + 255) / 256) * ((n_tones + G3_WIDE_TONES - 1) / G3_WIDE_TONES)));
}
size_t demod3_scratch_need(int n_tones, int64_t F, int n_sms) {
    const int64_t planes = g3_planes_fit(n_tones, F, n_sms) ? 3 * n_tones * g3_plane_ld(F) * 4
                                                            : static_cast<int64_t>(demod3_scratch_bytes(n_sms));
    return std::max(demod3_scratch_bytes(demod3_ctas(n_tones, F, n_sms)), static_cast<size_t>(planes));
}

size_t demod3_xs_rows(int64_t F, int Lpad, int D) { return static_cast<size_t>(F + (Lpad - 1) / D); }

cudaError_t demod_build_taps(const double* d_h, const uint64_t* d_words, int n_tones, int ntp, int L,
                             int Lpad, int e, void* b_hi, void* b_lo, cudaStream_t st) {
    const int64_t total = static_cast<int64_t>(ntp) * Lpad;
    build_taps_kernel<<<grid_for(total, 152), 256, 0, st>>>(d_h, d_words, n_tones, ntp, L, Lpad,
                                                             std::ldexp(1.0, e), static_cast<__half*>(b_hi),
                                                             static_cast<__half*>(b_lo));
    return cudaGetLastError();
}

cudaError_t demod_launch(const DemodLaunch& L, cudaStream_t st) {
    if (L.F <= 0) return cudaSuccess;
    if (L.D % 32 != 0 || L.Lpad % 32 != 0) return cudaErrorInvalidValue;
    const int64_t rows = static_cast<int64_t>(demod_xs_rows(L.F, L.Lpad, L.D));
    if (rows > L.xs_rows) return cudaErrorInvalidValue;
    const int n_mt = static_cast<int>((L.F + BM - 1) / BM);
    const int n_nt = (2 * L.ntp) / BN;
    const int n_anch = demod_anchor_rows(L.F0, L.F);
    float2* anchors = static_cast<float2*>(L.rot);
    float2* steps = anchors + static_cast<int64_t>(n_anch) * L.ntp;
    // rotation tables
    const int64_t nrot = static_cast<int64_t>(n_anch) * L.ntp + static_cast<int64_t>(L.ntp) * BM;
    rot_kernel<<<grid_for(nrot, L.n_sms), 256, 0, st>>>(L.words, L.n_tones, L.ntp, L.F0 / BM, L.L, L.D,
                                                         n_anch, anchors, steps);
    // pre-split of the Toeplitz source rows
    const int64_t total = rows * L.D;
    presplit_kernel<<<grid_for(total, L.n_sms), 256, 0, st>>>(
        reinterpret_cast<const uint32_t*>(L.carry), L.cl, reinterpret_cast<const uint32_t*>(L.buf),
        L.cl + L.n, total, static_cast<__half2*>(L.xs_hi), static_cast<__half2*>(L.xs_lo));
    // tensor maps
    CUtensorMap mAh, mAl, mBh, mBl;
    const uint64_t two_d = static_cast<uint64_t>(2) * L.D;
    if (!make_map(&mAh, L.xs_hi, two_d, rows, BM) || !make_map(&mAl, L.xs_lo, two_d, rows, BM) ||
        !make_map(&mBh, L.b_hi, static_cast<uint64_t>(2) * L.Lpad, static_cast<uint64_t>(2) * L.ntp, BN) ||
        !make_map(&mBl, L.b_lo, static_cast<uint64_t>(2) * L.Lpad, static_cast<uint64_t>(2) * L.ntp, BN))
        return cudaErrorInvalidValue;
    GemmArgs g{};
    g.raster = L.raster_group;
    g.F = L.F;
    g.F0 = L.F0;
    g.n_tones = L.n_tones;
    g.ntp = L.ntp;
    g.KB = 2 * L.Lpad / BK;
    g.kchunk = L.kchunk > 0 ? L.kchunk : 2;
    g.two_d = static_cast<int>(two_d);
    g.n_mt = n_mt;
    g.n_nt = n_nt;
    g.anchors = anchors;
    g.steps = steps;
    g.inv_scale = static_cast<float>(L.inv_scale);
    g.out = static_cast<float2*>(L.tones);
    g.ld = L.tones_ld;
    g.fo = L.frame_offset;
    g.status = L.status;
    cudaError_t e = cudaFuncSetAttribute(demod_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(GEMM_SMEM));
    if (e != cudaSuccess) return e;
    const int tiles = n_mt * n_nt;
    const int grid = std::min(tiles, L.n_sms);
    demod_gemm_kernel<<<grid, GEMM_THREADS, GEMM_SMEM, st>>>(mAh, mAl, mBh, mBl, g);
    return cudaGetLastError();
}

cudaError_t demod3_build_taps(const double* d_h, const uint64_t* d_words, int n_tones, int ntp, int L, int Lpad,
                              int e, void* planes, cudaStream_t st) {
    const int64_t total = static_cast<int64_t>(ntp) * Lpad;
    build_taps3_kernel<<<grid_for(total, 152), 256, 0, st>>>(d_h, d_words, n_tones, ntp, L, Lpad, std::ldexp(1.0, e),
                                                              static_cast<__half*>(planes));
    return cudaGetLastError();
}

namespace {
// Clocks that a work item takes.  A K-block (64 taps of one product) of a pair: its
// MMAs, 12 of w / 2 clocks and 15 % for their gaps, or the shared-memory traffic of the
// MMAs and the TMA at 128 bytes a clock (see the Gauss form's comment); of a single
// CTA, fitted: 900, 1000 and 1180 clocks at w = 16, 64 and 128.  Finishing: wide tiles
// beside the next tile's first two products, by two warps, 480 clocks a tone; others in
// the epilogue, 75 clocks a tone of which the next tile's MMAs do not run beside.
// Measured, 2^24 samples, D = 512, 1000 tones, L = 256 / 1024 / 2048 / 4096, in us: wide
// 468 / 603 / 782 / 1337, pairs of 128 tones 217 / 447 / 756 / 1387, single CTAs of 128
// 229 / 523 / 924 / 1717.
struct G3Form {
    bool pair = false, split = false;
    int bw = 128;
    bool wide() const { return bw > G3_TONES; }
    double clocks(int64_t KB) const {
        constexpr double kFinish = 480.0, kExposed = 75.0;
        const double block = pair ? std::max(6.9 * bw, 640.0 + 2.5 * bw) : 860.0 + 2.5 * bw;
        if (split) return KB * block;
        if (wide()) return std::max(3 * KB * block, KB * block + kFinish * bw);
        return 3 * KB * block + kExposed * bw;
    }
};
int g3_even_width(int n_tones, int widest, int step) {
    const int tiles = (n_tones + widest - 1) / widest;
    return ((n_tones + tiles - 1) / tiles + step - 1) / step * step;
}
// The form of a push: the least time of those its plan allows (any, or the pinned
// pair, tone width or fused pre-split), counting whole waves of work items over the
// chip (a batched step's launch shares its waves between plans, so there only the
// work counts, and nothing is split).  kSplitClocks: the planes' round trip and
// combine3_kernel's launch.
G3Form g3_choose(const DemodLaunch& L, bool shared_launch) {
    constexpr double kSplitClocks = 8000.0;
    G3Form best;
    double best_t = 1e300;
    const int64_t KB = L.Lpad / G3_BK;
    const bool pinned = !L.auto_form, pinned_pair = pinned && L.pair && !L.fused_presplit;
    for (int pair = 0; pair < 2; ++pair) {
        if (pinned && pair != (pinned_pair ? 1 : 0)) continue;
        int widths[2];
        if (pair) {
            widths[0] = g3_even_width(L.n_tones, G3_WIDE_TONES, 32);
            widths[1] = g3_even_width(L.n_tones, G3_TONES, 32);
        } else if (pinned) {
            widths[0] = widths[1] = L.tone_tile == 64 ? 64 : 128;
        } else {
            widths[0] = g3_even_width(L.n_tones, G3_TONES, 16);
            widths[1] = g3_even_width(L.n_tones, 64, 16);
        }
        for (int w : widths) {
            const int64_t tiles = (L.F + (pair ? 255 : 127)) / (pair ? 256 : 128) * ((L.n_tones + w - 1) / w);
            const int64_t places = pair ? L.n_sms / 2 : L.n_sms;
            for (int split = 0; split < 2; ++split) {
                if (split && (shared_launch || !g3_planes_fit(L.n_tones, L.F, L.n_sms))) continue;
                G3Form f;
                f.pair = pair != 0;
                f.split = split != 0;
                f.bw = w;
                const int64_t units = tiles * (split ? 3 : 1);
                const double waves = shared_launch ? static_cast<double>(units) / places
                                                   : static_cast<double>((units + places - 1) / places);
                const double t = waves * f.clocks(KB) + (split ? kSplitClocks : 0.0);
                if (t < best_t) {
                    best_t = t;
                    best = f;
                }
            }
        }
    }
    return best;
}
}  // namespace

cudaError_t demod3_prepare(const DemodLaunch& L, cudaStream_t st, DemodGemmJob* job, bool shared_launch) {
    job->n_units = 0;
    if (L.F <= 0) return cudaSuccess;
    if (L.D % G3_BK != 0 || L.Lpad % G3_BK != 0 || L.ntp % 128 != 0) return cudaErrorInvalidValue;
    const G3Form form = g3_choose(L, shared_launch);
    job->kind = form.wide() ? 0 : form.pair ? 1 : !L.auto_form && L.fused_presplit ? 3 : 2;
    const bool fused = job->kind == 3;
    const int64_t rows = static_cast<int64_t>(demod3_xs_rows(L.F, L.Lpad, L.D));
    if (!fused && rows > L.xs_rows) return cudaErrorInvalidValue;
    if (form.split && 3 * static_cast<size_t>(L.n_tones) * g3_plane_ld(L.F) * 4 > L.scratch_bytes) return cudaErrorInvalidValue;
    const int bm = form.pair ? 256 : BM;
    const int n_mt = static_cast<int>((L.F + bm - 1) / bm);
    const int n_nt = (L.n_tones + form.bw - 1) / form.bw;
    const int n_anch = demod_anchor_rows(L.F0, L.F);
    float2* anchors = static_cast<float2*>(L.rot);
    float2* steps = anchors + static_cast<int64_t>(n_anch) * L.ntp;
    G3Plan* P = reinterpret_cast<G3Plan*>(job->bytes);
    std::memset(P, 0, sizeof(G3Plan));
    const __half* bp = static_cast<const __half*>(L.b_hi);
    const int64_t bplane = static_cast<int64_t>(L.ntp) * L.Lpad;
    const int64_t total = rows * L.D;
    __half* xp = static_cast<__half*>(L.xs_hi);
    if (fused) {
        // the GEMM's producers read the stream view themselves
        P->carry = reinterpret_cast<const uint32_t*>(L.carry);
        P->buf = reinterpret_cast<const uint32_t*>(L.buf);
        P->cl = L.cl;
        P->lv = L.cl + L.n;
        P->vec = (reinterpret_cast<uintptr_t>(L.buf) % 16 == 0) && ((L.cl % 4) + 4) % 4 == 0 ? 1 : 0;
    }
    Prep3Args pa{};
    pa.words = L.words;
    pa.n_tones = L.n_tones;
    pa.ntp = L.ntp;
    pa.L = L.L;
    pa.D = L.D;
    pa.n_anch = n_anch;
    pa.A0 = L.F0 / BM;
    pa.anchors = anchors;
    pa.steps = steps;
    pa.carry = reinterpret_cast<const uint32_t*>(L.carry);
    pa.buf = reinterpret_cast<const uint32_t*>(L.buf);
    pa.cl = L.cl;
    pa.lv = L.cl + L.n;
    pa.total = fused ? 0 : total;
    pa.planes = xp;
    const int64_t rot_items = ((pa.A0 + n_anch - 1) / kRotRun - pa.A0 / kRotRun + 1 + BM / kRotRun) * L.ntp;
    pa.rot_items = static_cast<int>(std::min<int64_t>(256, (rot_items / (2 * L.n_sms) + 31) / 32 * 32));
    if (pa.rot_items < 32) pa.rot_items = 32;
    pa.rot_blocks = static_cast<int>(std::min<int64_t>((rot_items + pa.rot_items - 1) / pa.rot_items, int64_t(L.n_sms) * 8));
    const unsigned plane_blocks = pa.total ? grid_for(pa.total / 8, L.n_sms) : 0;
    prep3_kernel<<<pa.rot_blocks + plane_blocks, 256, 0, st>>>(pa);
    const uint32_t b_box = static_cast<uint32_t>(form.pair ? form.bw / 2 : form.bw);
    for (int i = 0; i < 6; ++i) {
        if ((!fused && !make_map(&P->a[i], xp + i * total, static_cast<uint64_t>(L.D),
                                      static_cast<uint64_t>(rows), BM)) ||
            !make_map(&P->b[i], bp + i * bplane, static_cast<uint64_t>(L.Lpad), static_cast<uint64_t>(L.ntp), b_box))
            return cudaErrorInvalidValue;
    }
    P->bw = form.bw;
    P->split = form.split ? 1 : 0;
    P->scratch = static_cast<float*>(L.scratch);
    P->pld = g3_plane_ld(L.F);
    GemmArgs& g = P->g;
    g.raster = L.raster_group;
    g.F = L.F;
    g.F0 = L.F0;
    g.n_tones = L.n_tones;
    g.ntp = L.ntp;
    g.KB = L.Lpad / G3_BK;
    // the three MMAs of a tap set share one accumulator, where two would take them
    // apart (hi.hi + lo.hi beside hi.lo); a chunk is half as long for that, as many
    // half K-blocks as the plan says blocks: the accumulator takes fewer additions of
    // smaller partial sums
    g.kchunk = std::max(L.kchunk, 1);
    g.two_d = L.D;                 // columns of a Toeplitz source row (one plane)
    g.n_mt = n_mt;
    g.n_nt = n_nt;
    g.anchors = anchors;
    g.steps = steps;
    g.inv_scale = static_cast<float>(L.inv_scale);
    g.out = static_cast<float2*>(L.tones);
    g.ld = L.tones_ld;
    g.fo = L.frame_offset;
    g.status = L.status;
    job->n_units = n_mt * n_nt * (form.split ? 3 : 1);
    job->unit_cost = form.clocks(g.KB);
    return cudaGetLastError();
}

namespace {
// room: bytes of the scratch that unsplit CTAs park their products in.
template <bool PAIR, bool FUSED, bool WIDE>
cudaError_t g3_run(const G3Batch& b, int n_sms, size_t room, cudaStream_t st) {
    using Cfg = G3Cfg<PAIR, FUSED, WIDE>;
    bool parks = false;
    for (int k = 0; WIDE && k < b.n_plans; ++k) parks = parks || !b.p[k].split;
    auto fits = [&](int grid) { return !parks || demod3_scratch_bytes(grid) <= room; };
    auto kern = demod3m_gemm_kernel<PAIR, FUSED, WIDE>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(Cfg::SMEM));
    if (e != cudaSuccess) return e;
    const int threads = Cfg::THREADS;
    if (!PAIR) {
        const int grid = std::max(1, std::min(b.total_units, n_sms));
        if (!fits(grid)) return cudaErrorInvalidValue;
        kern<<<grid, threads, Cfg::SMEM, st>>>(b);
        return cudaGetLastError();
    }
    // clusters of two CTAs: as many as can be resident at once (one CTA per SM)
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    static std::atomic<int> max_clusters{0};      // queried once
    int mc = max_clusters.load();
    if (mc <= 0) {
        cfg.gridDim = dim3(static_cast<unsigned>(2 * (n_sms / 2)), 1, 1);
        if (cudaOccupancyMaxActiveClusters(&mc, kern, &cfg) != cudaSuccess || mc <= 0) {
            cudaGetLastError();
            mc = n_sms / 2;
        }
        max_clusters.store(mc);
    }
    const int clusters = std::max(1, std::min(b.total_units, std::min(mc, n_sms / 2)));
    if (!fits(2 * clusters)) return cudaErrorInvalidValue;
    cfg.gridDim = dim3(static_cast<unsigned>(2 * clusters), 1, 1);
    e = cudaLaunchKernelEx(&cfg, kern, b);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}
}  // namespace

cudaError_t demod3_gemm(const DemodGemmJob* const* jobs, int n, int n_sms, void* scratch, size_t room, cudaStream_t st,
                        int only) {
    // costliest work items first, so that the launch ends on short ones
    std::vector<const DemodGemmJob*> order(jobs, jobs + n);
    std::stable_sort(order.begin(), order.end(),
                     [](const DemodGemmJob* x, const DemodGemmJob* y) { return x->unit_cost > y->unit_cost; });
    // one persistent launch per group of up to kG3MaxPlans jobs of the same kind
    for (int kind = 0; kind < kDemodKinds; ++kind) {
        if (only >= 0 && kind != only) continue;
        G3Batch b;
        b.n_plans = 0;
        b.total_units = 0;
        for (int i = 0; i <= n; ++i) {
            const bool flush = i == n || b.n_plans == kG3MaxPlans;
            if (flush && b.n_plans > 0) {
                // the launch's CTAs, whatever plans' tiles they take, park products in the one
                // scratch of the call (the kernel finds it at its first plan's)
                for (int k = 0; k < b.n_plans; ++k)
                    if (!b.p[k].split) b.p[k].scratch = static_cast<float*>(scratch);
                const cudaError_t e = kind == 0   ? g3_run<true, false, true>(b, n_sms, room, st)
                                      : kind == 1 ? g3_run<true, false, false>(b, n_sms, room, st)
                                      : kind == 2 ? g3_run<false, false, false>(b, n_sms, room, st)
                                                  : g3_run<false, true, false>(b, n_sms, room, st);
                if (e != cudaSuccess) return e;
                for (int k = 0; k < b.n_plans; ++k)
                    if (b.p[k].split) {
                        const GemmArgs& g = b.p[k].g;
                        const dim3 grid(static_cast<unsigned>((g.F + 255) / 256), static_cast<unsigned>(std::min(g.n_tones, 65535)));
                        combine3_kernel<<<grid, 256, 0, st>>>(b.p[k].scratch, b.p[k].pld, g);
                        const cudaError_t ce = cudaGetLastError();
                        if (ce != cudaSuccess) return ce;
                    }
                b.n_plans = 0;
                b.total_units = 0;
            }
            if (i == n) break;
            if (order[i]->kind != kind || order[i]->n_units <= 0) continue;
            std::memcpy(&b.p[b.n_plans], order[i]->bytes, sizeof(G3Plan));
            b.p[b.n_plans].unit0 = b.total_units;
            b.total_units += order[i]->n_units;
            ++b.n_plans;
        }
    }
    return cudaSuccess;
}

cudaError_t demod3_launch(const DemodLaunch& L, cudaStream_t st) {
    DemodGemmJob job;
    cudaError_t e = demod3_prepare(L, st, &job, false);
    if (e != cudaSuccess || job.n_units <= 0) return e;
    const DemodGemmJob* jp = &job;
    return demod3_gemm(&jp, 1, L.n_sms, L.scratch, L.scratch_bytes, st);
}

}  // namespace rfr

// ====================================================================
// Allocation-free one-shot demodulation (rfr_demod_noalloc).
//
// For callers that must not allocate device memory once they are running:
// a real-time processing thread that cannot afford the device-wide
// synchronisation and allocator locks that cudaMalloc/cudaFree can take, or a
// host application whose device-memory budget is owned by another allocator.
// The working memory of this path -- the modulated taps, the FP16 split of
// the samples, the rotation tables, a zero history block and the status word
// -- lives in one file-scope device array of kNaBytes (about 6.7 MB), which
// every GPU that loads this library holds until the process exits.
// ====================================================================
#include <mutex>

namespace rfr {
namespace {

constexpr int64_t kNaMaxSamples = int64_t(1) << 18;   // samples per call
constexpr int kNaMaxTones = 256;
constexpr int kNaMaxTaps = 1024;

constexpr size_t na_align(size_t v) { return (v + 255) / 256 * 256; }
constexpr size_t kNaStatus = 0;
constexpr size_t kNaWords = 256;
constexpr size_t kNaTaps = na_align(kNaWords + kNaMaxTones * 8);
constexpr size_t kNaZero = na_align(kNaTaps + kNaMaxTaps * 8);                 // zero history
constexpr size_t kNaBhi = na_align(kNaZero + kNaMaxTaps * 4);
constexpr size_t kNaBBytes = static_cast<size_t>(2) * kNaMaxTones * 2 * kNaMaxTaps * 2;
constexpr size_t kNaBlo = na_align(kNaBhi + kNaBBytes);
constexpr size_t kNaXsBytes = static_cast<size_t>(kNaMaxSamples + kNaMaxTaps) * 4;
constexpr size_t kNaXhi = na_align(kNaBlo + kNaBBytes);
constexpr size_t kNaXlo = na_align(kNaXhi + kNaXsBytes);
constexpr int64_t kNaMaxAnchRows = kNaMaxSamples / 32 / BM + 2;
constexpr size_t kNaRot = na_align(kNaXlo + kNaXsBytes);
constexpr size_t kNaRotBytes = static_cast<size_t>(kNaMaxAnchRows + BM) * kNaMaxTones * 8;
constexpr size_t kNaBytes = na_align(kNaRot + kNaRotBytes);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaBytes];

// Device address of g_noalloc_scratch per device, looked up once per device
// (the host-side name of the array is not a device address).
constexpr int kNaMaxDevices = 64;
unsigned char* g_na_ptr[kNaMaxDevices] = {};
std::mutex g_na_mu;

cudaError_t na_scratch(unsigned char** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kNaMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_na_mu);
    if (!g_na_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_na_ptr[dev] = static_cast<unsigned char*>(p);
    }
    *out = g_na_ptr[dev];
    return cudaSuccess;
}

}  // namespace
}  // namespace rfr

extern "C" rfr_status rfr_demod_noalloc(const int16_t* iq, int64_t n_samples, const double* taps,
                                        int32_t L, int32_t D, const uint64_t* words, int32_t n_tones,
                                        void* tones, int64_t tones_ld, void* stream) {
    using namespace rfr;
    if (n_samples < 0 || n_samples > kNaMaxSamples) return RFR_E_INVALID;   // beyond the static scratch
    if (L < 1 || L > kNaMaxTaps || D < 32 || D % 32 != 0 || D > kNaMaxSamples) return RFR_E_INVALID;
    if (n_tones < 1 || n_tones > kNaMaxTones || !taps || !words) return RFR_E_INVALID;
    const int64_t F = n_samples / D;
    if (F > 0 && (!iq || !tones || tones_ld < F)) return RFR_E_INVALID;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char* base = nullptr;
    if (na_scratch(&base) != cudaSuccess) return RFR_E_CUDA;
    if (F == 0) return RFR_OK;
    // tap scale 2^e with max|h| * 2^e in [2^14, 2^15) (same rule as a plan)
    double hmax = 0.0;
    for (int j = 0; j < L; ++j) hmax = std::max(hmax, std::fabs(taps[j]));
    if (!(hmax > 0.0) || !std::isfinite(hmax)) return RFR_E_INVALID;
    int e2 = 0;
    std::frexp(hmax, &e2);
    const int tap_exp = 15 - e2;
    const int Lpad = (L + 31) / 32 * 32;
    const int ntp = (n_tones + BN / 2 - 1) / (BN / 2) * (BN / 2);
    int* status = reinterpret_cast<int*>(base + kNaStatus);
    uint64_t* d_words = reinterpret_cast<uint64_t*>(base + kNaWords);
    double* d_taps = reinterpret_cast<double*>(base + kNaTaps);
    const uint32_t* zero = reinterpret_cast<const uint32_t*>(base + kNaZero);
    __half* bh = reinterpret_cast<__half*>(base + kNaBhi);
    __half* bl = reinterpret_cast<__half*>(base + kNaBlo);
    __half2* xh = reinterpret_cast<__half2*>(base + kNaXhi);
    __half2* xl = reinterpret_cast<__half2*>(base + kNaXlo);
    float2* anchors = reinterpret_cast<float2*>(base + kNaRot);
    // contents left by the previous call are overwritten or cleared here
    if (cudaMemsetAsync(base, 0, kNaTaps, st) != cudaSuccess ||
        cudaMemsetAsync(base + kNaZero, 0, static_cast<size_t>(kNaMaxTaps) * 4, st) != cudaSuccess ||
        cudaMemcpyAsync(d_words, words, static_cast<size_t>(n_tones) * 8, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(d_taps, taps, static_cast<size_t>(L) * 8, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return RFR_E_CUDA;
    build_taps_kernel<<<grid_for(static_cast<int64_t>(ntp) * Lpad, 152), 256, 0, st>>>(
        d_taps, d_words, n_tones, ntp, L, Lpad, std::ldexp(1.0, tap_exp), bh, bl);
    const int n_mt = static_cast<int>((F + BM - 1) / BM);
    const int n_anch = demod_anchor_rows(0, F);
    float2* steps = anchors + static_cast<int64_t>(n_anch) * ntp;
    rot_kernel<<<grid_for(static_cast<int64_t>(n_anch + BM) * ntp, 152), 256, 0, st>>>(
        d_words, n_tones, ntp, 0, L, D, n_anch, anchors, steps);
    // zero history: the stream view starts L - D samples before sample 0
    const int64_t cl = static_cast<int64_t>(L) - D;
    const int64_t rows = static_cast<int64_t>(demod_xs_rows(F, Lpad, D));
    presplit_kernel<<<grid_for(rows * D, 152), 256, 0, st>>>(zero, cl, reinterpret_cast<const uint32_t*>(iq),
                                                             cl + n_samples, rows * D, xh, xl);
    CUtensorMap mAh, mAl, mBh, mBl;
    const uint64_t two_d = static_cast<uint64_t>(2) * D;
    if (!make_map(&mAh, xh, two_d, rows, BM) || !make_map(&mAl, xl, two_d, rows, BM) ||
        !make_map(&mBh, bh, static_cast<uint64_t>(2) * Lpad, static_cast<uint64_t>(2) * ntp, BN) ||
        !make_map(&mBl, bl, static_cast<uint64_t>(2) * Lpad, static_cast<uint64_t>(2) * ntp, BN))
        return RFR_E_CUDA;
    GemmArgs g{};
    g.raster = 1;
    g.F = F;
    g.F0 = 0;
    g.n_tones = n_tones;
    g.ntp = ntp;
    g.KB = 2 * Lpad / BK;
    g.kchunk = 2;
    g.two_d = static_cast<int>(two_d);
    g.n_mt = n_mt;
    g.n_nt = (2 * ntp) / BN;
    g.anchors = anchors;
    g.steps = steps;
    g.inv_scale = static_cast<float>(std::ldexp(1.0, -tap_exp));
    g.out = static_cast<float2*>(tones);
    g.ld = tones_ld;
    g.fo = 0;
    g.status = status;
    if (cudaFuncSetAttribute(demod_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(GEMM_SMEM)) != cudaSuccess)
        return RFR_E_CUDA;
    int n_sms = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev);
    demod_gemm_kernel<<<std::min(n_mt * g.n_nt, std::max(n_sms, 1)), GEMM_THREADS, GEMM_SMEM, st>>>(mAh, mAl, mBh, mBl, g);
    return cudaGetLastError() == cudaSuccess ? RFR_OK : RFR_E_CUDA;
}

extern "C" rfr_status rfr_demod_noalloc_status(void* stream, int32_t* device_status) {
    using namespace rfr;
    unsigned char* base = nullptr;
    if (na_scratch(&base) != cudaSuccess) return RFR_E_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int v = 0;
    if (cudaMemcpyAsync(&v, base + kNaStatus, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return RFR_E_CUDA;
    if (device_status) *device_status = v;
    if (v == DEV_TIMEOUT) return RFR_E_TIMEOUT;
    return v == DEV_OK ? RFR_OK : RFR_E_CUDA;
}
