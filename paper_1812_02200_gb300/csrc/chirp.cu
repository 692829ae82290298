// chirp.cu -- the chirped readout (Sec. III.C, Eq. 1).
//
// Eq. 1, phi_t = 2*pi*(f0*t + k*t^2), in sample units t = m/fs becomes the
// exact uint64 phase  p(m) = s*m + r*m^2 (mod 2^64)  in units of 2*pi/2^64,
// s = f0/fs*2^64 (start word), r = k/fs^2*2^64 (rate word).
//
// chirp_synth_kernel: the transmit buffer generated on the GPU in real time
// (instead of a stored table): round-half-even of A*cos, A*sin of the phase,
// as complex int16.  The sine and cosine are computed in FP32 (the paper's
// "32 bit precision"); a component whose FP32 value lies within twice its
// error bound of a rounding tie is recomputed in FP64, so every int16 is the
// FP64 decision.
//
// chirp_demod_kernel: demodulation of the Rx stream against chirps ("using
// the algorithm outlined in section III.B"): for chirp c and frame k,
//   out[c][k] = sum_{n<L} h[n] x[b_k+n] exp(-i*2*pi*p_c(b_k+n)/2^64),
// the mix fused into the filter (the mixer depends on the frame through the
// quadratic term, so there is no fixed modulated-tap matrix to multiply).
// One CTA per frame, all chirps: each thread mixes and filters L/256 taps per
// chirp in FP32; the partial sums are reduced in FP32 within a warp and in FP64
// across the warps.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "dev_common.cuh"
#include "rfr_internal.h"

namespace rfr {

namespace {

__device__ __forceinline__ uint64_t chirp_phase(uint64_t s, uint64_t r, int64_t m) {
    const uint64_t um = static_cast<uint64_t>(m);
    return s * um + r * (um * um);
}

// ---------------------------------------------------------------- synthesis
//
// A sample is A*exp(i*2*pi*p/2^64).  The phase is reduced exactly to the
// nearest quarter turn q and an offset x in [-1/4, 1/4] (angle / pi), taken
// from the top 32 phase bits and rounded to 24 significant bits (error
// <= 2^-27 + 2^-31).  Error of the FP32 value v = fl(fl(A) * sincospif(x))
// against A*sin (or cos) of the exact angle, |v - v_exact| <= e with
//   e = A*(pi*(2^-27 + 2^-31) + 2^-24 + 2^-24) + |fl(A) - A|
// (argument rounding, 1 ulp of sincospif for results below 1 in magnitude,
// product rounding).  When |v - rint(v)| <= 1/2 - 2e, rint(v) is the rounding
// of the exact value; every other component goes to a per-tile queue in
// shared memory and is recomputed in FP64 (sincos_phase_f64) by the whole
// CTA, so the FP64 pipe only ever runs full warps (its throughput is counted
// per warp instruction, active lanes or not).
constexpr int kSynThreads = 256;
constexpr int kSynTile = 2048;          // samples per tile (8 per thread)

__device__ __forceinline__ int16_t clamp16(float v) {
    return static_cast<int16_t>(fminf(fmaxf(v, -32768.f), 32767.f));
}

// FP64 sine and cosine of the exact phase for the near-tie recompute, from
// the angle-addition formula: the phase is reduced in integer arithmetic to a
// quarter turn q, an offset i/1024 of a half turn (|i| <= 256, table of FP64
// sin and cos of pi*i/1024) and a remainder delta, |delta| <= pi/2048, whose
// sine and cosine come from their Taylor series (terms to delta^7 and
// delta^8: truncation below 1e-25).
struct SinCos1024 {
    double s[513], c[513];
};
__device__ SinCos1024 g_sc1024;

__device__ __forceinline__ void sincos_phase_f64(uint64_t p, const double2* __restrict__ tab, double* sn,
                                                 double* cs) {
    const uint32_t q = static_cast<uint32_t>((p + (1ull << 61)) >> 62);
    const int64_t f = static_cast<int64_t>(p - (static_cast<uint64_t>(q) << 62));     // x = f / 2^63
    const int64_t i = (f + (int64_t(1) << 52)) >> 53;                                 // nearest i/1024
    const int64_t r = f - i * (int64_t(1) << 53);                                     // |r| <= 2^52
    const double d = static_cast<double>(r) * 3.4061215800865545e-19;                 // pi * 2^-63
    const double d2 = d * d;
    const double sd = d * (1.0 + d2 * (-1.0 / 6 + d2 * (1.0 / 120 + d2 * (-1.0 / 5040))));
    const double cd = 1.0 + d2 * (-0.5 + d2 * (1.0 / 24 + d2 * (-1.0 / 720 + d2 * (1.0 / 40320))));
    const double2 t = tab[i + 256];                                                   // (sin, cos)
    double sx = fma(t.x, cd, t.y * sd), cx = fma(t.y, cd, -(t.x * sd));
    if (q & 1) {
        const double u = sx;
        sx = cx;
        cx = -u;
    }
    if (q & 2) {
        sx = -sx;
        cx = -cx;
    }
    *sn = sx;
    *cs = cx;
}

__global__ void __launch_bounds__(kSynThreads) chirp_synth_kernel(uint64_t s, uint64_t r, float ampf,
                                                                  double amp, float tie_lo, int64_t m0,
                                                                  int64_t n, short2* __restrict__ out) {
    __shared__ __align__(16) short2 tile[kSynTile];
    __shared__ uint16_t fix[2 * kSynTile];
    __shared__ int nfix;
    __shared__ double2 tab[513];
    const int tid = threadIdx.x;
    for (int i = tid; i < 513; i += kSynThreads) tab[i] = make_double2(g_sc1024.s[i], g_sc1024.c[i]);
    for (int64_t base = static_cast<int64_t>(blockIdx.x) * kSynTile; base < n;
         base += static_cast<int64_t>(gridDim.x) * kSynTile) {
        if (tid == 0) nfix = 0;
        __syncthreads();
        const int cnt = static_cast<int>(n - base < kSynTile ? n - base : kSynTile);
        // p(m + 256) = p(m) + d(m), d(m + 256) = d(m) + 2*256^2*r  (all mod 2^64)
        const uint64_t m = static_cast<uint64_t>(m0 + base + tid);
        uint64_t p = chirp_phase(s, r, static_cast<int64_t>(m));
        uint64_t d = s * 256ull + r * (512ull * m + 65536ull);
        const uint64_t dd = r * 131072ull;
        for (int i = tid; i < cnt; i += kSynThreads) {
            // quarter turn q and offset from the top 32 phase bits:
            // x = fi * 2^-31 in [-1/4, 1/4] (angle / pi)
            const uint32_t hi = static_cast<uint32_t>(p >> 32);
            const uint32_t q = ((hi + (1u << 29)) >> 30) & 3u;
            const int32_t fi = static_cast<int32_t>(hi - (q << 30));
            float sx, cx;
            sincospif(static_cast<float>(fi) * 0x1p-31f, &sx, &cx);
            float c = cx, sn = sx;                 // rotate by q quarter turns
            if (q & 1) {
                c = -sx;
                sn = cx;
            }
            if (q & 2) {
                c = -c;
                sn = -sn;
            }
            const float vc = ampf * c, vs = ampf * sn;
            const float rc = rintf(vc), rs = rintf(vs);
            if (fabsf(vc - rc) > tie_lo) fix[atomicAdd(&nfix, 1)] = static_cast<uint16_t>(i << 1);
            if (fabsf(vs - rs) > tie_lo) fix[atomicAdd(&nfix, 1)] = static_cast<uint16_t>((i << 1) | 1);
            tile[i] = make_short2(clamp16(rc), clamp16(rs));
            p += d;
            d += dd;
        }
        __syncthreads();
        const int nf = nfix;
        int16_t* comp = reinterpret_cast<int16_t*>(tile);
        for (int j = tid; j < nf; j += kSynThreads) {
            const int e = fix[j];
            double sd, cd;
            sincos_phase_f64(chirp_phase(s, r, m0 + base + (e >> 1)), tab, &sd, &cd);
            comp[e] = clamp16(static_cast<float>(rint(amp * ((e & 1) ? sd : cd))));
        }
        __syncthreads();
        short2* dst = out + base;
        if (cnt == kSynTile && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
            const uint4* src4 = reinterpret_cast<const uint4*>(tile);
            uint4* dst4 = reinterpret_cast<uint4*>(dst);
            for (int i = tid; i < kSynTile / 4; i += kSynThreads) dst4[i] = src4[i];
        } else {
            for (int i = tid; i < cnt; i += kSynThreads) dst[i] = tile[i];
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------- demodulation
//
// One CTA per frame (grid-stride): the frame's L samples are converted to FP32
// once into shared memory and reused by every chirp.  For chirp c a thread
// walks its taps n = tid, tid + 256, ... with the exact phase recurrence
// p(m + 256) = p(m) + d, d += 2*256^2*r; the mixer is that of the phase's top 32
// bits in FP32 and the products are summed in FP32 per thread and across the
// warp (shuffles); the 8 warp sums are added in FP64 (through shared memory,
// a group of 32 chirps at a time).
constexpr int kChirpThreads = 256;
constexpr int kChirpGroup = 32;

// cos and sin of 2 pi ph / 2^32.  The quadrant comes off the integer phase, the
// rest |r| <= 2^29 (converted to FP32 with an error of at most 2^-27 of a half
// turn; the whole phase would lose 2^-25) goes through the Taylor series of sin(pi
// x) and cos(pi x), |x| <= 1/4: the first terms left out are below 2e-9 and
// 2e-10.  (sincospif of the whole phase: 303 us where this takes 282,
// 2^24 samples, 8 chirps, L = 4096, D = 2048.)
__device__ __forceinline__ void mixer(uint32_t ph, float& cs, float& sn) {
    const uint32_t u = ph + 0x20000000u, q = u >> 30;
    const float x = static_cast<float>(static_cast<int32_t>(u & 0x3fffffffu) - 0x20000000) * 0x1p-31f;
    const float t = x * x;
    // pi^(2 n + 1) / (2 n + 1)!, pi itself in two parts, and pi^(2 n) / (2 n)!
    constexpr double P = 3.14159265358979323846;
    constexpr float s1 = static_cast<float>(P), s1l = static_cast<float>(P - static_cast<double>(s1));
    constexpr float s3 = static_cast<float>(-P * P * P / 6), s5 = static_cast<float>(P * P * P * P * P / 120);
    constexpr float s7 = static_cast<float>(-P * P * P * P * P * P * P / 5040);
    constexpr float s9 = static_cast<float>(P * P * P * P * P * P * P * P * P / 362880);
    constexpr float c2 = static_cast<float>(-P * P / 2), c4 = static_cast<float>(P * P * P * P / 24);
    constexpr float c6 = static_cast<float>(-P * P * P * P * P * P / 720);
    constexpr float c8 = static_cast<float>(P * P * P * P * P * P * P * P / 40320);
    constexpr float c10 = static_cast<float>(-P * P * P * P * P * P * P * P * P * P / 3628800);
    const float ps = fmaf(x, s1, x * fmaf(t, fmaf(t, fmaf(t, fmaf(t, s9, s7), s5), s3), s1l));
    const float pc = fmaf(t, fmaf(t, fmaf(t, fmaf(t, fmaf(t, c10, c8), c6), c4), c2), 1.0f);
    const bool odd = (q & 1u) != 0;
    cs = __uint_as_float(__float_as_uint(odd ? ps : pc) ^ (((q + 1u) & 2u) << 30));
    sn = __uint_as_float(__float_as_uint(odd ? pc : ps) ^ ((q & 2u) << 30));
}

struct ChirpArgs {
    const uint32_t* carry;
    int64_t cl;
    const uint32_t* buf;
    int64_t F;
    int64_t a0;             // absolute sample index of v[0]
    int L, D;
    const float* h;
    const uint64_t* s;
    const uint64_t* r;
    int n_chirps;
    float2* out;
    int64_t ld, fo;
};

__global__ void __launch_bounds__(kChirpThreads) chirp_demod_kernel(const ChirpArgs a) {
    extern __shared__ float2 xs[];                      // [L]
    __shared__ double2 red[kChirpGroup][kChirpThreads / 32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    allow_dependents();
    for (int64_t k = blockIdx.x; k < a.F; k += gridDim.x) {
        __syncthreads();                                // previous frame's readers are done
        for (int n = tid; n < a.L; n += kChirpThreads) {
            const int64_t vi = k * a.D + n;             // index in [carry | buffer]
            xs[n] = iq_to_f2(vi < a.cl ? __ldg(a.carry + vi) : __ldg(a.buf + (vi - a.cl)));
        }
        __syncthreads();
        const uint64_t m = static_cast<uint64_t>(a.a0 + k * a.D + tid);
        for (int c0 = 0; c0 < a.n_chirps; c0 += kChirpGroup) {
            const int cn = a.n_chirps - c0 < kChirpGroup ? a.n_chirps - c0 : kChirpGroup;
            for (int cc = 0; cc < cn; ++cc) {
                const uint64_t s = __ldg(a.s + c0 + cc), r = __ldg(a.r + c0 + cc);
                uint64_t p = chirp_phase(s, r, static_cast<int64_t>(m));
                uint64_t d = s * 256ull + r * (512ull * m + 65536ull);
                const uint64_t dd = r * 131072ull;
                float ar = 0.f, ai = 0.f;
                for (int n = tid; n < a.L; n += kChirpThreads) {
                    const float2 x = xs[n];
                    float sn, cs;
                    mixer(static_cast<uint32_t>(p >> 32), cs, sn);
                    // x * exp(-i*theta) = (x.re*cos + x.im*sin, x.im*cos - x.re*sin)
                    const float mr = fmaf(x.x, cs, x.y * sn), mi = fmaf(x.y, cs, -x.x * sn);
                    const float hn = __ldg(a.h + n);
                    ar = fmaf(hn, mr, ar);
                    ai = fmaf(hn, mi, ai);
                    p += d;
                    d += dd;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    ar += __shfl_xor_sync(0xffffffffu, ar, o);
                    ai += __shfl_xor_sync(0xffffffffu, ai, o);
                }
                if (lane == 0) red[cc][warp] = make_double2(ar, ai);
            }
            __syncthreads();
            if (tid < cn) {
                double tr = 0.0, ti = 0.0;
                for (int w = 0; w < kChirpThreads / 32; ++w) {
                    tr += red[tid][w].x;
                    ti += red[tid][w].y;
                }
                a.out[static_cast<int64_t>(c0 + tid) * a.ld + a.fo + k] =
                    make_float2(static_cast<float>(tr), static_cast<float>(ti));
            }
            __syncthreads();
        }
    }
}

// Overlapping frames (L > D, D a multiple of 256): a sample's mixer value does
// not depend on the frame, so each is evaluated once for the J = ceil(L / D)
// frames that use it.  The sine and cosine bound the kernel above (about 40
// issue slots per evaluation), so this divides its time by almost J.
//
// A CTA takes a run of frames on one SM, in segments whose samples fit its
// shared memory (packed int16, converted at use).  Four workers of 256 threads
// share a segment: a work item is a chirp over `sub` of the segment's frames,
// walked block by block (block b: the D samples from v[b D]) with one pair of
// sums per frame in progress: block b adds taps jD .. jD + D - 1 to frame b - j.
// A thread's samples are those the kernel above gives it, in the same order,
// and the reduction is the same, so the frames are bit-identical to its frames.
// Measured, 2^24 samples, 8 chirps, L = 4096, D = 2048: 467 -> 303 us (then 282 with
// the mixer above).
constexpr int kOvWorkers = 4;
constexpr int kOvSub = 32;                              // frames per work item at most
struct ChirpOverlap {
    int seg, sub;                                       // frames per segment, per work item
    int64_t per_cta;                                    // frames per CTA
};
template <int J, bool FULL>                             // FULL: L == J * D; J == 1: items of one frame
__global__ void __launch_bounds__(kOvWorkers * kChirpThreads, 1)
    chirp_overlap_kernel(const ChirpArgs a, const ChirpOverlap o) {
    extern __shared__ uint32_t xs32[];                  // [(seg + J - 1) * D]
    __shared__ double2 red[kOvWorkers][kOvSub][kChirpThreads / 32];
    const int wk = threadIdx.x / kChirpThreads, tid = threadIdx.x % kChirpThreads;
    const int warp = tid >> 5, lane = tid & 31;
    allow_dependents();
    auto worker_sync = [&] { asm volatile("bar.sync %0, 256;" ::"r"(1 + wk) : "memory"); };
    const int64_t k_end = a.F < (blockIdx.x + 1) * o.per_cta ? a.F : (blockIdx.x + 1) * o.per_cta;
    for (int64_t k0 = blockIdx.x * o.per_cta; k0 < k_end; k0 += o.seg) {
        const int seg = static_cast<int>(k_end - k0 < o.seg ? k_end - k0 : o.seg);
        // the segment's samples: those of its last frame end L - 1 past its start
        const int need = (seg - 1) * a.D + a.L;
        __syncthreads();                                // previous segment's readers are done
        for (int n = threadIdx.x; n < need; n += kOvWorkers * kChirpThreads) {
            const int64_t vi = k0 * a.D + n;
            xs32[n] = vi < a.cl ? __ldg(a.carry + vi) : __ldg(a.buf + (vi - a.cl));
        }
        __syncthreads();
        const int subs = (seg + o.sub - 1) / o.sub;
        for (int item = wk; item < a.n_chirps * subs; item += kOvWorkers) {
            const int c = item / subs, f0 = (item - c * subs) * o.sub;
            const int nf = seg - f0 < o.sub ? seg - f0 : o.sub;
            const uint64_t s = __ldg(a.s + c), r = __ldg(a.r + c);
            const uint64_t m = static_cast<uint64_t>(a.a0 + (k0 + f0) * a.D + tid);
            uint64_t p = chirp_phase(s, r, static_cast<int64_t>(m));
            uint64_t d = s * 256ull + r * (512ull * m + 65536ull);
            const uint64_t dd = r * 131072ull;
            // the sums of frame f (of the item) over the warp
            auto reduce = [&](int f, float tr, float ti) {
#pragma unroll
                for (int w = 16; w > 0; w >>= 1) {
                    tr += __shfl_xor_sync(0xffffffffu, tr, w);
                    ti += __shfl_xor_sync(0xffffffffu, ti, w);
                }
                if (lane == 0) red[wk][f][warp] = make_double2(tr, ti);
            };
            if constexpr (J == 1) {
                // one frame: its L samples straight through
                const uint32_t* xb = xs32 + f0 * a.D;
                float sr = 0.f, si = 0.f;
#pragma unroll 2
                for (int n = tid; n < a.L; n += kChirpThreads) {
                    const float2 x = iq_to_f2(xb[n]);
                    float sn, cs;
                    mixer(static_cast<uint32_t>(p >> 32), cs, sn);
                    const float mr = fmaf(x.x, cs, x.y * sn), mi = fmaf(x.y, cs, -x.x * sn);
                    const float hn = __ldg(a.h + n);
                    sr = fmaf(hn, mr, sr);
                    si = fmaf(hn, mi, si);
                    p += d;
                    d += dd;
                }
                reduce(0, sr, si);
            } else {
                float ar[J], ai[J];                          // frame b - j
#pragma unroll
                for (int j = 0; j < J; ++j) ar[j] = ai[j] = 0.f;
                for (int b = 0; b < nf + J - 1; ++b) {
                    const uint32_t* xb = xs32 + (f0 + b) * a.D;
                    const int limit = (nf - 1 - b) * a.D + a.L;  // samples of the item from this block on
                    for (int n = tid; n < a.D && (FULL || n < limit); n += kChirpThreads) {
                        const float2 x = iq_to_f2(xb[n]);
                        float sn, cs;
                        mixer(static_cast<uint32_t>(p >> 32), cs, sn);
                        const float mr = fmaf(x.x, cs, x.y * sn), mi = fmaf(x.y, cs, -x.x * sn);
#pragma unroll
                        for (int j = 0; j < J; ++j) {
                            if (FULL || j * a.D + n < a.L) {
                                const float hn = __ldg(a.h + j * a.D + n);
                                ar[j] = fmaf(hn, mr, ar[j]);
                                ai[j] = fmaf(hn, mi, ai[j]);
                            }
                        }
                        p += d;
                        d += dd;
                    }
                    // frame b - (J - 1) is complete
                    if (b >= J - 1) reduce(b - (J - 1), ar[J - 1], ai[J - 1]);
#pragma unroll
                    for (int j = J - 1; j > 0; --j) {
                        ar[j] = ar[j - 1];
                        ai[j] = ai[j - 1];
                    }
                    ar[0] = ai[0] = 0.f;
                }
            }
            worker_sync();
            if (tid < nf) {
                double tr = 0.0, ti = 0.0;
                for (int w = 0; w < kChirpThreads / 32; ++w) {
                    tr += red[wk][tid][w].x;
                    ti += red[wk][tid][w].y;
                }
                a.out[static_cast<int64_t>(c) * a.ld + a.fo + k0 + f0 + tid] =
                    make_float2(static_cast<float>(tr), static_cast<float>(ti));
            }
            worker_sync();
        }
    }
}

}  // namespace

namespace {
// The FP64 sine/cosine table of the near-tie recompute, uploaded once per
// device (the first synthesis on a device; call it outside stream capture).
std::mutex g_sc_mu;
bool g_sc_done[64] = {};

cudaError_t ensure_sincos_table() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_sc_mu);
    if (g_sc_done[dev]) return cudaSuccess;
    SinCos1024 t;
    for (int i = -256; i <= 256; ++i) {
        t.s[i + 256] = std::sin(3.14159265358979323846 * i / 1024.0);
        t.c[i + 256] = std::cos(3.14159265358979323846 * i / 1024.0);
    }
    e = cudaMemcpyToSymbol(g_sc1024, &t, sizeof(t));
    if (e == cudaSuccess) g_sc_done[dev] = true;
    return e;
}
}  // namespace

cudaError_t chirp_synth(uint64_t s, uint64_t r, double amp, int64_t m0, int64_t n, void* out,
                        cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const float ampf = static_cast<float>(amp);
    // argument rounding, 1 ulp of sincospif (results below 1 in magnitude:
    // 2^-24), product rounding, amplitude rounding
    const double e = amp * (3.14159265358979 * (0x1p-27 + 0x1p-31) + 0x1p-24 + 0x1p-24) +
                     std::fabs(static_cast<double>(ampf) - amp);
    cudaError_t ce = ensure_sincos_table();
    if (ce != cudaSuccess) return ce;
    const float tie_lo = static_cast<float>(0.5 - 2.0 * e);
    const int64_t tiles = (n + kSynTile - 1) / kSynTile;
    const int64_t blocks = std::min<int64_t>(tiles, 152 * 8);
    chirp_synth_kernel<<<static_cast<unsigned>(blocks), kSynThreads, 0, st>>>(
        s, r, ampf, amp, tie_lo, m0, n, static_cast<short2*>(out));
    return cudaGetLastError();
}

cudaError_t chirp_demod_launch(const ChirpLaunch& L, cudaStream_t st) {
    if (L.F <= 0 || L.n_chirps <= 0) return cudaSuccess;
    ChirpArgs a{};
    a.carry = reinterpret_cast<const uint32_t*>(L.carry);
    a.cl = L.cl;
    a.buf = reinterpret_cast<const uint32_t*>(L.buf);
    a.F = L.F;
    a.a0 = L.a0;
    a.L = L.L;
    a.D = L.D;
    a.h = L.h32;
    a.s = L.start_words;
    a.r = L.rate_words;
    a.n_chirps = L.n_chirps;
    a.out = static_cast<float2*>(L.tones);
    a.ld = L.tones_ld;
    a.fo = L.frame_offset;
    // overlapping frames: each mixer value once for all its frames, where at
    // least a segment of two frames fits and it pays
    const int J = (L.L + L.D - 1) / L.D;
    const size_t smem = static_cast<size_t>(L.L) * sizeof(float2);      // of the single-frame kernel
    const int single_per_sm = std::max(1, std::min(8, static_cast<int>((220u * 1024u) / (smem + 5u * 1024u))));
    constexpr int kOvSamples = 48 * 1024;               // of a segment: 192 KB
    const int jt = J <= 2 ? 2 : (J <= 4 ? 4 : 8);       // compiled widths; the blocks past L add nothing
    if (J >= 2 && J <= 8 && L.D % kChirpThreads == 0 && (jt + 1) * L.D <= kOvSamples) {
        const bool full = L.L == jt * L.D;
        ChirpOverlap o{};
        const int64_t grid = std::min<int64_t>(L.F, L.n_sms);
        o.per_cta = (L.F + grid - 1) / grid;
        const int64_t widest = kOvSamples / L.D - (jt - 1) > 0 ? kOvSamples / L.D - (jt - 1) : 1;
        const int64_t n_seg = (o.per_cta + widest - 1) / widest;
        o.seg = static_cast<int>((o.per_cta + n_seg - 1) / n_seg);
        // Frames per work item, at most kOvSub (so from ceil(seg / kOvSub) items a chirp
        // on), or the kernel above: the least of these times, in issue slots, fitted to
        // 1500 shapes of L = 307 .. 16384, D = 256 .. 4096, 1 .. 16 chirps, 20 .. 10^4
        // frames (12 % RMS).  An item of several frames: 26 a sample and 5.6 for each
        // frame it may belong to (8.8 where taps end inside a block), 52 a block, 95 in
        // all; of one frame: 31 a sample, 220 in all; the kernel above: 44 and 45 a frame
        // and chirp.  Four workers share an SM's slots, one alone gets two thirds.  (Rounds
        // of block walks alone chose up to 1.8 times what the kernel above takes, where
        // a CTA has one or two frames or a sample's frames are few.)
        constexpr double kAlone = 1.5;
        const double walk = (L.L + kChirpThreads - 1) / kChirpThreads;      // a thread's samples of a frame
        double best = 1e300;
        auto consider = [&](int sub) {
            const int64_t items = static_cast<int64_t>(a.n_chirps) * ((o.seg + sub - 1) / sub);
            const double samples = (static_cast<double>(sub - 1) * L.D + L.L) / kChirpThreads;
            const double item = sub == 1 ? 31.0 * walk + 220.0
                                         : samples * (26.0 + (full ? 5.6 : 8.8) * jt) + 52.0 * (sub + jt - 1) + 95.0;
            const int64_t rest = items % kOvWorkers;
            const double cost = n_seg * item * ((items - rest) + (rest ? std::max(kAlone, static_cast<double>(rest)) : 0.0));
            if (cost < best) {
                best = cost;
                o.sub = sub;
            }
        };
        for (int parts = (o.seg + kOvSub - 1) / kOvSub; parts < o.seg; parts = parts < 4 ? parts + 1 : parts * 3 / 2)
            consider((o.seg + parts - 1) / parts);
        consider(1);
        const double per_sm = static_cast<double>(L.F) / L.n_sms;
        const double alone = a.n_chirps * (44.0 * walk + 45.0) *
                             std::max(per_sm, kAlone * std::ceil(static_cast<double>(L.F) / (L.n_sms * single_per_sm)));
        if (best <= alone) {
            const size_t bytes = static_cast<size_t>(o.seg + jt - 1) * L.D * 4;
            auto run = [&](auto kern) {
                const cudaError_t e = allow_smem(kern, kOvSamples * 4);
                if (e != cudaSuccess) return e;
                kern<<<static_cast<unsigned>((L.F + o.per_cta - 1) / o.per_cta), kOvWorkers * kChirpThreads, bytes, st>>>(a, o);
                return cudaGetLastError();
            };
            if (o.sub == 1) return run(chirp_overlap_kernel<1, false>);
            switch (jt) {
            case 2: return full ? run(chirp_overlap_kernel<2, true>) : run(chirp_overlap_kernel<2, false>);
            case 4: return full ? run(chirp_overlap_kernel<4, true>) : run(chirp_overlap_kernel<4, false>);
            default: return full ? run(chirp_overlap_kernel<8, true>) : run(chirp_overlap_kernel<8, false>);
            }
        }
    }
    constexpr int kMostTaps = 16384;                    // of a plan
    const cudaError_t e = allow_smem(chirp_demod_kernel, kMostTaps * static_cast<int>(sizeof(float2)));
    if (e != cudaSuccess) return e;
    const int64_t blocks = std::min<int64_t>(L.F, static_cast<int64_t>(L.n_sms) * single_per_sm);
    chirp_demod_kernel<<<static_cast<unsigned>(blocks), kChirpThreads, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace rfr
