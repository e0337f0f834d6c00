// Readouts with FP64 accumulation: probabilities |a_i|^2 (Sec. II.A), norm, Pauli-word
// expectation values and inverse-CDF sampling (per-range sums, their prefix sums, the search of
// each shot).
//
// GB300 issues 2 FP64 operations per clock and SM, conversions to FP64 included, so these passes
// are bound by the FP64 pipe unless an amplitude takes at most two of them (complex64: one state
// read at the copy rate takes as long as 0.75 FP64 operations per amplitude).  Hence complex64
// components are widened by integer operations (widen), products go straight into fused
// accumulations, and the two terms that a Pauli word pairs up are summed as one.  n = 28 complex64:
// a word takes 0.47 ms (0.32 at the copy rate), the range sums 0.95, all probabilities 0.95 (0.63);
// norm, four words, 4096 shots and all probabilities together 30.2 -> 4.3 ms.
#include <type_traits>

#include "sv_internal.h"

namespace sv {
namespace {

constexpr int kThreads = 256;

// Exact widening without the FP64 pipe: FAST moves a normal float's sign, exponent and mantissa to
// their places in a double.  Zeros, subnormals, infinities and NaN (odd) take the conversion.
__device__ __forceinline__ bool odd(float x) { return ((__float_as_uint(x) + 0x00800000u) & 0x7F000000u) == 0u; }
__device__ __forceinline__ bool odd(double) { return false; }
template <bool FAST>
__device__ __forceinline__ double widen(float x) {
    if (!FAST) return (double)x;
    const unsigned b = __float_as_uint(x);
    const unsigned hi = (b & 0x80000000u) | (((b >> 3) & 0x0FFFFFFFu) + 0x38000000u);
    return __hiloint2double((int)hi, (int)(b << 29));
}
template <bool FAST>
__device__ __forceinline__ double widen(double x) { return x; }

template <bool FAST, typename T2>
__device__ __forceinline__ double p2_of(const T2 &v) {
    const double x = widen<FAST>(v.x), y = widen<FAST>(v.y);
    return fma(x, x, y * y);
}
template <typename T2>
__device__ __forceinline__ double p2(const T2 &v) {
    return (odd(v.x) || odd(v.y)) ? p2_of<false>(v) : p2_of<true>(v);
}

// Two amplitudes per load (complex64: 16 bytes in, 16 out), kProbs loads in flight per thread;
// VEC: out is 16-byte aligned.
constexpr int kProbs = 4;
template <typename T2, bool VEC>
__global__ void __launch_bounds__(kThreads) k_probs(const T2 *__restrict__ a, double *__restrict__ out, int64_t pairs) {
    const int64_t i0 = (int64_t)blockIdx.x * (kProbs * kThreads) + threadIdx.x;
    T2 u[kProbs][2];
#pragma unroll
    for (int k = 0; k < kProbs; ++k) {
        const int64_t i = i0 + k * kThreads;
        u[k][0] = u[k][1] = T2{1, 1};
        if (i >= pairs) continue;
        if constexpr (sizeof(T2) == 8) {
            const float4 q = *reinterpret_cast<const float4 *>(a + 2 * i);
            u[k][0] = make_float2(q.x, q.y);
            u[k][1] = make_float2(q.z, q.w);
        } else {
            u[k][0] = a[2 * i];
            u[k][1] = a[2 * i + 1];
        }
    }
    // one branch for the whole batch: predicated conversions would keep the FP64 pipe busy
    bool slow = false;
#pragma unroll
    for (int k = 0; k < kProbs; ++k)
#pragma unroll
        for (int e = 0; e < 2; ++e) slow = slow || odd(u[k][e].x) || odd(u[k][e].y);
    auto store = [&](auto fast) {
#pragma unroll
        for (int k = 0; k < kProbs; ++k) {
            const int64_t i = i0 + k * kThreads;
            if (i >= pairs) continue;
            const double p = p2_of<decltype(fast)::value>(u[k][0]), q = p2_of<decltype(fast)::value>(u[k][1]);
            if (VEC) {
                reinterpret_cast<double2 *>(out)[i] = make_double2(p, q);
            } else {
                out[2 * i] = p;
                out[2 * i + 1] = q;
            }
        }
    };
    if (slow) store(std::false_type{});
    else store(std::true_type{});
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int NT>
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double red[NT / 32];
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0;
    if (threadIdx.x < 32) {
        s = threadIdx.x < NT / 32 ? red[threadIdx.x] : 0.0;
        s = warp_sum(s);
    }
    __syncthreads();
    return s;
}

// Each CTA sums a contiguous range of the state (the partials are added in CTA order, so the
// result does not depend on scheduling).  complex64: threads read 16-byte vectors (two
// amplitudes); squares are summed in FP32 over runs of 8 vectors per thread (16 terms, all
// non-negative) and the runs accumulated in FP64 -- FP64 arithmetic on every element would
// make this pass FP64-bound instead of HBM-bound on GB300.  complex128: FP64 throughout.
__global__ void __launch_bounds__(kThreads) k_partial_norm_c64(const float4 *__restrict__ v, int64_t nv,
                                                               double *partials) {
    const int64_t per = (nv + gridDim.x - 1) / gridDim.x;
    const int64_t lo = (int64_t)blockIdx.x * per, hi = lo + per < nv ? lo + per : nv;
    double s = 0;
    for (int64_t base = lo + threadIdx.x; base < hi; base += 8 * kThreads) {
        float f = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int64_t i = base + (int64_t)k * kThreads;
            if (i < hi) {
                const float4 q = v[i];
                f = fmaf(q.x, q.x, fmaf(q.y, q.y, fmaf(q.z, q.z, fmaf(q.w, q.w, f))));
            }
        }
        s += (double)f;
    }
    s = block_sum<kThreads>(s);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

__global__ void __launch_bounds__(kThreads) k_partial_norm_c128(const double2 *__restrict__ a, int64_t len,
                                                                double *partials) {
    const int64_t per = (len + gridDim.x - 1) / gridDim.x;
    const int64_t lo = (int64_t)blockIdx.x * per, hi = lo + per < len ? lo + per : len;
    double s = 0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += kThreads) {
        const double2 v = a[i];
        s = fma(v.y, v.y, fma(v.x, v.x, s));
    }
    s = block_sum<kThreads>(s);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

// Norm restoration after a tensor-core circuit: d = sqrt(n_in / n_out) - 1 from the two sets of
// norm partials (input at part[0, nb), output at part[nb, 2 nb)), applied only when every fused
// group was unitary (*flag != 0).
__global__ void k_renorm_factor(const double *__restrict__ part, int nb, const int *__restrict__ flag,
                                float *__restrict__ out) {
    double nin = 0, nout = 0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        nin += part[b];
        nout += part[nb + b];
    }
    nin = block_sum<kThreads>(nin);
    nout = block_sum<kThreads>(nout);
    if (threadIdx.x == 0) out[0] = (*flag != 0 && nout > 0) ? (float)(sqrt(nin / nout) - 1.0) : 0.f;
}

// a <- a (1 + d), applied as a small correction so that the factor's FP32 rounding next to 1
// does not become the error.
template <typename V>
__global__ void __launch_bounds__(kThreads) k_renorm_apply(V *__restrict__ v, int64_t nv, const float *__restrict__ dp) {
    const float d = *dp;
    if (d == 0.f) return;
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < nv; i += (int64_t)gridDim.x * kThreads) {
        V q = v[i];
        q.x = fmaf(q.x, d, q.x);
        q.y = fmaf(q.y, d, q.y);
        q.z = fmaf(q.z, d, q.z);
        q.w = fmaf(q.w, d, q.w);
        v[i] = q;
    }
}

// sum_j conj(a_{j^x}) a_j (-1)^{popc(j & z)}; the phase i^{popc(x&z)} is applied on the host.
//
// j and j ^ x carry conjugate terms with signs that differ by (-1)^{popc(x & z)}, so for x != 0 the
// pair sums to twice a real (EVEN) or twice an imaginary part (ODD): half the loads and a quarter of
// the products of summing every j.  NORM (x = 0): +-|a_j|^2.  t enumerates the pairs (index j = t
// with a zero inserted at x's highest bit) in tiles of 4 x 256; j & z has the parity of t & zt, zt
// the mask z without that bit, so the signs of tile, step and thread combine by exclusive or.
enum : int { NORM = 0, EVEN = 1, ODD = 2 };

template <int MODE, bool FAST, typename T>
__device__ __forceinline__ void add_term(double &s, T ux, T uy, T vx, T vy, unsigned sign) {
    // the sign goes onto u before widening: integer work
    double a = widen<FAST>(ux), b = widen<FAST>(uy);
    a = __hiloint2double(__double2hiint(a) ^ (int)sign, __double2loint(a));
    b = __hiloint2double(__double2hiint(b) ^ (int)sign, __double2loint(b));
    const double c = widen<FAST>(vx), d = widen<FAST>(vy);
    if (MODE == ODD) {  // Im(conj(u) v)
        s = fma(a, d, s);
        s = fma(-b, c, s);
    } else {  // Re(conj(u) v)
        s = fma(a, c, s);
        s = fma(b, d, s);
    }
}

// |x| in FP32, for the sum of the terms' magnitudes (a double's to 12 %, out of FP32's range as 0 or huge).
__device__ __forceinline__ float magnitude(float x) { return fabsf(x); }
__device__ __forceinline__ float magnitude(double x) {
    return __int_as_float(min(max((__double2hiint(x) & 0x7FFFFFFF) - (896 << 20), 0), 254 << 20) << 3);
}

// Per CTA its sum, and at partials[gridDim.x ..] the magnitudes of its products.
template <typename T2, int MODE>
__global__ void __launch_bounds__(kThreads) k_partial_expval(const T2 *__restrict__ a, int64_t terms, uint64_t x,
                                                             uint64_t zt, int hb, double *partials) {
    constexpr int kSteps = 4, kTile = kSteps * kThreads;
    unsigned step_sign[kSteps];
#pragma unroll
    for (int k = 0; k < kSteps; ++k)
        step_sign[k] = (unsigned)((__popcll(((uint64_t)k * kThreads + threadIdx.x) & zt) & 1) << 31);
    double s = 0;
    float w = 0;
    for (int64_t t0 = (int64_t)blockIdx.x * kTile; t0 < terms; t0 += (int64_t)gridDim.x * kTile) {
        const unsigned tile_sign = (unsigned)((__popcll((uint64_t)t0 & zt) & 1) << 31);
        T2 u[kSteps], v[kSteps];
        bool slow = false;
#pragma unroll
        for (int k = 0; k < kSteps; ++k) {
            const int64_t t = t0 + k * kThreads + threadIdx.x;
            u[k] = v[k] = T2{0, 0};
            if (t < terms) {
                if (MODE == NORM) {
                    u[k] = v[k] = a[t];
                } else {
                    const int64_t j = ((t >> hb) << (hb + 1)) | (t & ((int64_t(1) << hb) - 1));
                    v[k] = a[j];
                    u[k] = a[(uint64_t)j ^ x];
                }
            }
        }
#pragma unroll
        for (int k = 0; k < kSteps; ++k) slow = slow || odd(u[k].x) || odd(u[k].y) || odd(v[k].x) || odd(v[k].y);
        if (slow) {
#pragma unroll
            for (int k = 0; k < kSteps; ++k)
                add_term<MODE, false>(s, u[k].x, u[k].y, v[k].x, v[k].y, tile_sign ^ step_sign[k]);
        } else {
#pragma unroll
            for (int k = 0; k < kSteps; ++k)
                add_term<MODE, true>(s, u[k].x, u[k].y, v[k].x, v[k].y, tile_sign ^ step_sign[k]);
        }
#pragma unroll
        for (int k = 0; k < kSteps; ++k) {
            w = fmaf(magnitude(u[k].x), magnitude(MODE == ODD ? v[k].y : v[k].x), w);
            w = fmaf(magnitude(u[k].y), magnitude(MODE == ODD ? v[k].x : v[k].y), w);
        }
    }
    s = block_sum<kThreads>(s);
    const double total = block_sum<kThreads>((double)w);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = MODE == NORM ? s : 2 * s;
        partials[gridDim.x + blockIdx.x] = MODE == NORM ? total : 2 * total;
    }
}

// The sum term by term: for words whose paired sum vanishes, where the result is the rounding residue
// of the order of summation (6 FP64 operations and conversions more per amplitude).
template <typename T2>
__global__ void __launch_bounds__(kThreads) k_partial_expval_direct(const T2 *__restrict__ a, int64_t len, uint64_t x,
                                                                    uint64_t z, double *partials) {
    const int64_t per = (len + gridDim.x - 1) / gridDim.x;
    const int64_t lo = (int64_t)blockIdx.x * per, hi = lo + per < len ? lo + per : len;
    double sr = 0, si = 0;
    for (int64_t j = lo + threadIdx.x; j < hi; j += kThreads) {
        const T2 u = a[(uint64_t)j ^ x], v = a[j];
        // conj(u) * v
        double tr = (double)u.x * (double)v.x + (double)u.y * (double)v.y;
        double ti = (double)u.x * (double)v.y - (double)u.y * (double)v.x;
        if (__popcll((unsigned long long)j & z) & 1) { tr = -tr; ti = -ti; }
        sr += tr;
        si += ti;
    }
    sr = block_sum<kThreads>(sr);
    si = block_sum<kThreads>(si);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = sr;
        partials[2 * blockIdx.x + 1] = si;
    }
}

// Sum of the partials, of the weights behind them if there are any, and the handle's error word, into the
// caller's result words (host memory the GPU writes directly, or device memory).
__global__ void __launch_bounds__(kThreads) k_finish(const double *__restrict__ partials, int nb, bool weights,
                                                     const int *__restrict__ err, Readout *out) {
    double s = 0, w = 0;
    for (int b = threadIdx.x; b < nb; b += kThreads) {
        s += partials[b];
        if (weights) w += partials[nb + b];
    }
    s = block_sum<kThreads>(s);
    w = block_sum<kThreads>(w);
    if (threadIdx.x == 0) {
        out->value = s;
        out->weight = w;
        out->err = *err;
    }
}

// sums[b] = sum of |a_i|^2 over i in [b 2^sb, (b+1) 2^sb), one warp per range, summed in
// index order within each lane then across lanes.
template <typename T2>
__global__ void __launch_bounds__(kThreads) k_block_sums(const T2 *__restrict__ a, int sb, int64_t nb, double *sums) {
    const int64_t w = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= nb) return;
    const int64_t lo = w << sb;
    const int64_t len = int64_t(1) << sb;
    double s = 0;
    constexpr int kBatch = 8;
    for (int64_t i0 = lane; i0 < len; i0 += 32 * kBatch) {
        T2 v[kBatch];
        bool slow = false;
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            v[k] = T2{0, 0};
            if (i0 + 32 * k < len) v[k] = a[lo + i0 + 32 * k];
            slow = slow || odd(v[k].x) || odd(v[k].y);
        }
        auto add = [&](auto fast) {
#pragma unroll
            for (int k = 0; k < kBatch; ++k) {
                const double x = widen<decltype(fast)::value>(v[k].x), y = widen<decltype(fast)::value>(v[k].y);
                s = fma(y, y, fma(x, x, s));
            }
        };
        if (slow) add(std::false_type{});
        else add(std::true_type{});
    }
    s = warp_sum(s);
    if (lane == 0) sums[w] = s;
}

// Prefix sums of the range sums in two levels: inclusive within blocks of kScan ranges (in place),
// then inclusive over the blocks' totals (one CTA).
constexpr int kScan = 1024;

__device__ __forceinline__ double warp_scan(double v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

template <int NT>
__device__ __forceinline__ double block_scan(double v) {
    __shared__ double red[NT / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    v = warp_scan(v, lane);
    if (lane == 31) red[w] = v;
    __syncthreads();
    if (w == 0) {
        const double r = warp_scan(lane < NT / 32 ? red[lane] : 0.0, lane);
        if (lane < NT / 32) red[lane] = r;
    }
    __syncthreads();
    if (w > 0) v += red[w - 1];
    __syncthreads();
    return v;
}

__global__ void __launch_bounds__(kThreads) k_scan_blocks(double *sums, int64_t nb, double *totals) {
    constexpr int kPer = kScan / kThreads;
    const int64_t at = (int64_t)blockIdx.x * kScan + threadIdx.x * kPer;
    double v[kPer], own = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        v[k] = own += at + k < nb ? sums[at + k] : 0.0;
    }
    const double incl = block_scan<kThreads>(own), before = incl - own;
#pragma unroll
    for (int k = 0; k < kPer; ++k)
        if (at + k < nb) sums[at + k] = before + v[k];
    if (threadIdx.x == kThreads - 1) totals[blockIdx.x] = incl;
}

__global__ void __launch_bounds__(kThreads) k_scan_totals(double *totals, int count, const int *__restrict__ err,
                                                          Readout *out) {
    const int per = (count + kThreads - 1) / kThreads;
    const int lo = min(count, (int)threadIdx.x * per), hi = min(count, lo + per);
    double own = 0;
    for (int i = lo; i < hi; ++i) own += totals[i];
    double run = block_scan<kThreads>(own) - own;
    for (int i = lo; i < hi; ++i) totals[i] = run += totals[i];
    __syncthreads();
    if (threadIdx.x == 0) {
        out->value = totals[count - 1];
        out->err = *err;
    }
}

// Output s of the SplitMix64 stream (Steele, Lea & Flood, OOPSLA 2014) seeded with `seed`: mixes
// seed + (s+1) * 0x9E3779B97F4A7C15; the uniform takes its top 53 bits.
__device__ __forceinline__ double uniform_of(uint64_t seed, uint64_t s) {
    uint64_t z = seed + (s + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);
}

// One warp per shot: the smallest range whose inclusive prefix exceeds the target, in it the first
// of 32 segments whose inclusive prefix does (each lane sums one), and in that the first amplitude
// whose running sum does -- or the last non-zero one of the range, or segment, where rounding leaves
// the sum short.  (A warp that ran through the range one amplitude at a time took 456 us for 4096
// shots, a thread alone longer still.)
template <typename T2>
__global__ void __launch_bounds__(kThreads) k_sample(const T2 *__restrict__ a, int sb, const double *__restrict__ incl,
                                                     int64_t nb, const double *__restrict__ totals, int count,
                                                     uint64_t seed, int64_t shots, uint64_t *out) {
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int64_t k = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5; k < shots; k += (int64_t)gridDim.x * (kThreads / 32)) {
        const double total = totals[count - 1];
        if (!(total > 0)) continue;  // the host reports it
        const double t = uniform_of(seed, (uint64_t)k) * total;
        int lo = 0, hi = count - 1;
        while (lo < hi) {
            const int mid = lo + (hi - lo) / 2;
            if (totals[mid] > t) hi = mid; else lo = mid + 1;
        }
        const double base = lo > 0 ? totals[lo - 1] : 0.0;
        const int64_t first = (int64_t)lo * kScan, last = min(nb, first + kScan) - 1;
        int64_t bl = first, bh = last;
        while (bl < bh) {
            const int64_t mid = bl + (bh - bl) / 2;
            if (base + incl[mid] > t) bh = mid; else bl = mid + 1;
        }
        double acc = bl > first ? base + incl[bl - 1] : base;  // at most t
        const int len = 1 << sb, seg = len > 32 ? len / 32 : 1;  // amplitudes per lane
        double upto = 0;
        unsigned over = 0, any = 0;
        for (bool chosen = true;; chosen = false, --bl) {
            double own = 0;
            bool nz = false;
            if (lane * seg < len)
                for (int i = 0; i < seg; ++i) {
                    const double p = p2(a[(bl << sb) + lane * seg + i]);
                    nz = nz || p > 0;
                    own += p;
                }
            upto = warp_scan(own, lane);
            over = chosen ? __ballot_sync(kAll, acc + upto > t) : 0u;
            any = __ballot_sync(kAll, nz);
            // a range of zeros is met only where two prefix sums that should be equal differ in
            // their last bit: the nearest non-zero index below it is the shot
            if (any || bl == 0) break;
        }
        const int64_t start = bl << sb;
        // without a prefix over the target: the last segment that is not all zero
        const int pick = over ? __ffs((int)over) - 1 : any ? 31 - __clz((int)any) : 0;
        const double before = __shfl_sync(kAll, upto, max(pick - 1, 0));
        if (pick > 0) acc += before;  // tested: at most t
        int64_t found = -1, last_nz = start + pick * seg;
        const double p = lane < seg ? p2(a[start + pick * seg + lane]) : 0.0;
        const unsigned pos = __ballot_sync(kAll, p > 0);
        if (pos) last_nz = start + pick * seg + 31 - __clz((int)pos);
        for (int l = 0; over && l < seg; ++l) {
            acc += __shfl_sync(kAll, p, l);
            if (acc > t && found < 0) found = start + pick * seg + l;
        }
        if (lane == 0) out[k] = (uint64_t)(found >= 0 ? found : last_nz);
    }
}

}  // namespace

void launch_probs(int dtype, const void *state, int n, double *out, int64_t first, int64_t count, cudaStream_t st) {
    (void)n;  // first and count are even (n >= 1)
    const int64_t pairs = count / 2;
    const unsigned grid = (unsigned)((pairs + kProbs * kThreads - 1) / (kProbs * kThreads));
    const bool vec = reinterpret_cast<uintptr_t>(out) % 16 == 0;
    if (dtype == SV_C64) {
        const float2 *a = (const float2 *)state + first;
        if (vec) k_probs<float2, true><<<grid, kThreads, 0, st>>>(a, out, pairs);
        else k_probs<float2, false><<<grid, kThreads, 0, st>>>(a, out, pairs);
    } else {
        const double2 *a = (const double2 *)state + first;
        if (vec) k_probs<double2, true><<<grid, kThreads, 0, st>>>(a, out, pairs);
        else k_probs<double2, false><<<grid, kThreads, 0, st>>>(a, out, pairs);
    }
    check_cuda(cudaGetLastError(), "probabilities kernel launch");
}

void launch_partial_norm(int dtype, const void *state, int n, double *partials, int nblocks, cudaStream_t st) {
    const int64_t len = int64_t(1) << n;
    if (dtype == SV_C64)  // n >= 1: an even number of amplitudes
        k_partial_norm_c64<<<nblocks, kThreads, 0, st>>>((const float4 *)state, len / 2, partials);
    else
        k_partial_norm_c128<<<nblocks, kThreads, 0, st>>>((const double2 *)state, len, partials);
    check_cuda(cudaGetLastError(), "norm kernel launch");
}

void launch_renorm(int dtype, void *state, int n, const double *partials, int nblocks, const int *flag, float *d,
                   cudaStream_t st) {
    k_renorm_factor<<<1, kThreads, 0, st>>>(partials, nblocks, flag, d);
    check_cuda(cudaGetLastError(), "renorm factor launch");
    const int64_t nv = (int64_t(1) << n) / (dtype == SV_C64 ? 2 : 1);
    const int grid = (int)std::min<int64_t>((nv + kThreads - 1) / kThreads, (int64_t)num_sms() * 8);
    if (dtype == SV_C64)
        k_renorm_apply<float4><<<grid, kThreads, 0, st>>>((float4 *)state, nv, d);
    else
        fail(SV_ERR_UNSUPPORTED, "norm restoration is for complex64 tensor-core circuits");
    check_cuda(cudaGetLastError(), "renorm launch");
}

template <typename T2>
static void expval_of(const void *state, int n, uint64_t x, uint64_t z, double *partials, int nblocks, cudaStream_t st) {
    const T2 *a = (const T2 *)state;
    if (x == 0) {
        k_partial_expval<T2, NORM><<<nblocks, kThreads, 0, st>>>(a, int64_t(1) << n, 0, z, 0, partials);
        return;
    }
    const int hb = 63 - __builtin_clzll(x);
    const uint64_t zt = (z & ((uint64_t(1) << hb) - 1)) | ((z >> (hb + 1)) << hb);
    const int64_t terms = int64_t(1) << (n - 1);
    if (__builtin_popcountll(x & z) & 1)
        k_partial_expval<T2, ODD><<<nblocks, kThreads, 0, st>>>(a, terms, x, zt, hb, partials);
    else
        k_partial_expval<T2, EVEN><<<nblocks, kThreads, 0, st>>>(a, terms, x, zt, hb, partials);
}

void launch_partial_expval(int dtype, const void *state, int n, uint64_t x, uint64_t z, double *partials, int nblocks,
                           cudaStream_t st) {
    if (dtype == SV_C64) expval_of<float2>(state, n, x, z, partials, nblocks, st);
    else expval_of<double2>(state, n, x, z, partials, nblocks, st);
    check_cuda(cudaGetLastError(), "expval kernel launch");
}

void pauli_phase(uint64_t x, uint64_t z, double sr, double si, double *out) {
    switch (__builtin_popcountll(x & z) & 3) {
        case 1: out[0] = -si; out[1] = sr; break;
        case 2: out[0] = -sr; out[1] = -si; break;
        case 3: out[0] = si; out[1] = -sr; break;
        default: out[0] = sr; out[1] = si; break;
    }
}

void launch_partial_expval_direct(int dtype, const void *state, int n, uint64_t x, uint64_t z, double *partials,
                                  int nblocks, cudaStream_t st) {
    const int64_t len = int64_t(1) << n;
    if (dtype == SV_C64)
        k_partial_expval_direct<float2><<<nblocks, kThreads, 0, st>>>((const float2 *)state, len, x, z, partials);
    else
        k_partial_expval_direct<double2><<<nblocks, kThreads, 0, st>>>((const double2 *)state, len, x, z, partials);
    check_cuda(cudaGetLastError(), "expval kernel launch");
}

void launch_finish(const double *partials, int nblocks, bool weights, const int *err, Readout *out, cudaStream_t st) {
    k_finish<<<1, kThreads, 0, st>>>(partials, nblocks, weights, err, out);
    check_cuda(cudaGetLastError(), "readout kernel launch");
}

int64_t sample_totals(int n, int sb) { return ((int64_t(1) << (n - sb)) + kScan - 1) / kScan; }

void launch_sample(int dtype, const void *state, int n, int sb, double *sums, double *totals, uint64_t seed, int64_t shots,
                   uint64_t *out, const int *err, Readout *total, cudaStream_t st) {
    const int64_t nb = int64_t(1) << (n - sb);
    const int count = (int)sample_totals(n, sb);
    const unsigned sgrid = (unsigned)((nb * 32 + kThreads - 1) / kThreads);
    const unsigned kgrid = (unsigned)std::min<int64_t>((shots * 32 + kThreads - 1) / kThreads, (int64_t)num_sms() * 8);
    if (dtype == SV_C64) k_block_sums<float2><<<sgrid, kThreads, 0, st>>>((const float2 *)state, sb, nb, sums);
    else k_block_sums<double2><<<sgrid, kThreads, 0, st>>>((const double2 *)state, sb, nb, sums);
    k_scan_blocks<<<(unsigned)count, kThreads, 0, st>>>(sums, nb, totals);
    k_scan_totals<<<1, kThreads, 0, st>>>(totals, count, err, total);
    if (dtype == SV_C64)
        k_sample<float2><<<kgrid, kThreads, 0, st>>>((const float2 *)state, sb, sums, nb, totals, count, seed, shots, out);
    else
        k_sample<double2><<<kgrid, kThreads, 0, st>>>((const double2 *)state, sb, sums, nb, totals, count, seed, shots, out);
    check_cuda(cudaGetLastError(), "sampling kernel launch");
}

}  // namespace sv
