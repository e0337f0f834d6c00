// Per-gate path: one HBM sweep per gate (the paper's baseline, Sec. V.A; gate update of
// Sec. II.A).  A 1-qubit gate on qubit k updates every pair (i, i XOR 2^k) (Fig. 2); a 2-qubit
// gate every quadruple of indices that differ only in its two bits.
//
// Memory access: every thread moves whole 16-byte units.  For complex64 a unit holds the two
// amplitudes that differ in bit 0, so when bit 0 is not a gate qubit each unit carries two
// independent groups, and when it is, the unit holds both members of a pair.  For complex128
// a unit is one amplitude.  Consecutive threads take consecutive groups, so each warp reads
// and writes whole 128-byte lines.
//
// A sweep touches only the amplitudes that its gate can change: local basis states whose row and
// column are those of the identity are left out, so a controlled gate moves half of the state and a
// controlled phase a quarter, and an exchange (X, CNOT, SWAP) moves amplitudes without arithmetic.
// (Complex64 gates on qubit 0 sweep the whole state: every unit holds both values of it.)
// Complex128 products run in block fixed point on the integer pipe (fixed64.cuh) where that is as exact,
// amplitude by amplitude (apply_fx).  480 gates of random layers on 16 qubits, complex128: 3.94 ms with
// every gate dense in FP64, 1.97 ms so (before after_last_gate).
#include <cmath>

#include "fixed64.cuh"
#include "sv_internal.h"

namespace sv {
namespace {

constexpr int kThreads = 256;
constexpr int kUnroll = 2;

// Gates of a circuit are launched with programmatic dependence (launch_after): a gate's blocks may be
// placed while the last gate's are finishing, and wait here, before their first access to the state,
// until it has completed and its writes are visible.  (480 gates on 16 qubits,
// complex128: 1.97 ms without, 1.07 so, 1.11 since apply_fx judges every group.)
__device__ __forceinline__ void after_last_gate() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ int64_t insert0(int64_t x, int p) {
    const int64_t low = x & ((int64_t(1) << p) - 1);
    return ((x >> p) << (p + 1)) | low;
}

template <typename T>
struct C2 { T re, im; };

template <typename T>
__device__ __forceinline__ void cmac(T &ore, T &oim, T mre, T mim, T xre, T xim) {
    ore = fma(mre, xre, ore);
    ore = fma(-mim, xim, ore);
    oim = fma(mre, xim, oim);
    oim = fma(mim, xre, oim);
}

template <typename T>
__device__ __forceinline__ void apply1(const T *m, T &x0r, T &x0i, T &x1r, T &x1i) {
    T y0r = 0, y0i = 0, y1r = 0, y1i = 0;
    cmac(y0r, y0i, m[0], m[1], x0r, x0i);
    cmac(y0r, y0i, m[2], m[3], x1r, x1i);
    cmac(y1r, y1i, m[4], m[5], x0r, x0i);
    cmac(y1r, y1i, m[6], m[7], x1r, x1i);
    x0r = y0r; x0i = y0i; x1r = y1r; x1i = y1i;
}

template <typename T>
__device__ __forceinline__ void apply2(const T *m, T (&xr)[4], T (&xi)[4]) {
    T yr[4], yi[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        yr[r] = 0; yi[r] = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) cmac(yr[r], yi[r], m[2 * (4 * r + c)], m[2 * (4 * r + c) + 1], xr[c], xi[c]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) { xr[r] = yr[r]; xi[r] = yi[r]; }
}

// ---- complex64, 1 qubit, k == 0: each unit is one pair.
__global__ void __launch_bounds__(kThreads) k_gate1_c64_lo(float4 *a, int64_t units, Mat1 M) {
    after_last_gate();
    const int64_t g0 = (int64_t)blockIdx.x * kThreads * kUnroll + threadIdx.x;
    float4 A[kUnroll];
#pragma unroll
    for (int s = 0; s < kUnroll; ++s)
        if (g0 + s * kThreads < units) A[s] = a[g0 + s * kThreads];
#pragma unroll
    for (int s = 0; s < kUnroll; ++s) {
        if (g0 + s * kThreads >= units) continue;
        apply1(M.m, A[s].x, A[s].y, A[s].z, A[s].w);
        a[g0 + s * kThreads] = A[s];
    }
}

// ---- complex64, 2 qubits, one of them is qubit 0: 2 units per group.  `zero_is_q0` says
// whether the gate's q[0] (low local bit) is qubit 0.
__global__ void __launch_bounds__(kThreads) k_gate2_c64_lo(float4 *a, int64_t groups, int po, int zero_is_q0, Mat2 M) {
    after_last_gate();
    const int64_t g0 = (int64_t)blockIdx.x * kThreads * kUnroll + threadIdx.x;
    float4 U0[kUnroll], U1[kUnroll];
    int64_t base[kUnroll];
#pragma unroll
    for (int s = 0; s < kUnroll; ++s) {
        const int64_t g = g0 + s * kThreads;
        base[s] = insert0(g, po);
        if (g < groups) { U0[s] = a[base[s]]; U1[s] = a[base[s] | (int64_t(1) << po)]; }
    }
#pragma unroll
    for (int s = 0; s < kUnroll; ++s) {
        if (g0 + s * kThreads >= groups) continue;
        float xr[4], xi[4];
        if (zero_is_q0) {  // local b: bit0 -> element in unit, bit1 -> unit
            xr[0] = U0[s].x; xi[0] = U0[s].y; xr[1] = U0[s].z; xi[1] = U0[s].w;
            xr[2] = U1[s].x; xi[2] = U1[s].y; xr[3] = U1[s].z; xi[3] = U1[s].w;
        } else {           // local b: bit0 -> unit, bit1 -> element in unit
            xr[0] = U0[s].x; xi[0] = U0[s].y; xr[2] = U0[s].z; xi[2] = U0[s].w;
            xr[1] = U1[s].x; xi[1] = U1[s].y; xr[3] = U1[s].z; xi[3] = U1[s].w;
        }
        apply2(M.m, xr, xi);
        if (zero_is_q0) {
            U0[s] = make_float4(xr[0], xi[0], xr[1], xi[1]);
            U1[s] = make_float4(xr[2], xi[2], xr[3], xi[3]);
        } else {
            U0[s] = make_float4(xr[0], xi[0], xr[2], xi[2]);
            U1[s] = make_float4(xr[1], xi[1], xr[3], xi[3]);
        }
        a[base[s]] = U0[s];
        a[base[s] | (int64_t(1) << po)] = U1[s];
    }
}

// ---- the general sweep: 16-byte units at base | off[j], j < NA, form a group; the base runs over
// the group number with the gate's unit bits lo < hi inserted as zeros (hi < 0: one bit).
template <int NA, typename M>
struct GateArgs {
    int64_t groups;
    int lo, hi;
    int64_t off[NA];
    M m;
};

__device__ __forceinline__ int64_t group_base(int64_t g, int lo, int hi) {
    const int64_t x = insert0(g, lo);
    return hi < 0 ? x : insert0(x, hi);
}

// Exchange: unit j of a group takes unit from[j]; complex128 units also take a factor 1, i, -1 or -i
// (turn[j] quarter turns), by swapping the components' words and flipping sign bits.
struct Moves {
    int from[4], turn[4];
};

__device__ __forceinline__ uint4 quarter_turns(uint4 u, int turn) {
    if (turn & 1) u = make_uint4(u.z, u.w ^ 0x80000000u, u.x, u.y);  // i (a + i b) = -b + i a
    if (turn & 2) {
        u.y ^= 0x80000000u;
        u.w ^= 0x80000000u;
    }
    return u;
}

template <int NA>
__global__ void __launch_bounds__(kThreads) k_gate_move(uint4 *a, const __grid_constant__ GateArgs<NA, Moves> P) {
    after_last_gate();
    const int64_t g0 = (int64_t)blockIdx.x * kThreads * kUnroll + threadIdx.x;
    uint4 U[kUnroll][NA];
    int64_t base[kUnroll];
#pragma unroll
    for (int s = 0; s < kUnroll; ++s) {
        const int64_t g = g0 + s * kThreads;
        base[s] = group_base(g, P.lo, P.hi);
        if (g < P.groups) {
#pragma unroll
            for (int j = 0; j < NA; ++j) U[s][j] = a[base[s] | P.off[P.m.from[j]]];
        }
    }
#pragma unroll
    for (int s = 0; s < kUnroll; ++s) {
        if (g0 + s * kThreads >= P.groups) continue;
#pragma unroll
        for (int j = 0; j < NA; ++j) a[base[s] | P.off[j]] = quarter_turns(U[s][j], P.m.turn[j]);
    }
}

// Dense on the NA touched local states, complex64 (both halves of a unit are independent groups).
template <int NA>
struct MatC64 {
    float m[2 * NA * NA];
};

template <int NA>
__device__ __forceinline__ void apply_n(const float *m, float (&xr)[NA], float (&xi)[NA]) {
    float yr[NA], yi[NA];
#pragma unroll
    for (int r = 0; r < NA; ++r) {
        yr[r] = 0; yi[r] = 0;
#pragma unroll
        for (int c = 0; c < NA; ++c) cmac(yr[r], yi[r], m[2 * (NA * r + c)], m[2 * (NA * r + c) + 1], xr[c], xi[c]);
    }
#pragma unroll
    for (int r = 0; r < NA; ++r) { xr[r] = yr[r]; xi[r] = yi[r]; }
}

template <int NA>
__global__ void __launch_bounds__(kThreads) k_gate_c64(float4 *a, const __grid_constant__ GateArgs<NA, MatC64<NA>> P) {
    after_last_gate();
    const int64_t g0 = (int64_t)blockIdx.x * kThreads * kUnroll + threadIdx.x;
    float4 U[kUnroll][NA];
    int64_t base[kUnroll];
#pragma unroll
    for (int s = 0; s < kUnroll; ++s) {
        const int64_t g = g0 + s * kThreads;
        base[s] = group_base(g, P.lo, P.hi);
        if (g < P.groups) {
#pragma unroll
            for (int j = 0; j < NA; ++j) U[s][j] = a[base[s] | P.off[j]];
        }
    }
#pragma unroll
    for (int s = 0; s < kUnroll; ++s) {
        if (g0 + s * kThreads >= P.groups) continue;
        float xr[NA], xi[NA];
#pragma unroll
        for (int j = 0; j < NA; ++j) { xr[j] = U[s][j].x; xi[j] = U[s][j].y; }
        apply_n<NA>(P.m.m, xr, xi);
#pragma unroll
        for (int j = 0; j < NA; ++j) { U[s][j].x = xr[j]; U[s][j].y = xi[j]; xr[j] = U[s][j].z; xi[j] = U[s][j].w; }
        apply_n<NA>(P.m.m, xr, xi);
#pragma unroll
        for (int j = 0; j < NA; ++j) {
            U[s][j].z = xr[j]; U[s][j].w = xi[j];
            a[base[s] | P.off[j]] = U[s][j];
        }
    }
}

// Dense on the NA touched local states, complex128: FP64 values, and the fixed-point factors and
// moduli of a unitary gate (FX).
template <int NA>
struct MatC128 {
    double m[2 * NA * NA];
    int32_t e[4 * NA * NA];
    float w[NA * NA];  // non-zero ones at least kLeast
};
constexpr float kLeast = 0x1p-60f;

template <int NA>
__device__ __forceinline__ void apply_fp64(const double *m, double2 (&U)[NA]) {
    double2 y[NA];
#pragma unroll
    for (int r = 0; r < NA; ++r) {
        double yr = 0, yi = 0;
#pragma unroll
        for (int c = 0; c < NA; ++c) cmac(yr, yi, m[2 * (NA * r + c)], m[2 * (NA * r + c) + 1], U[c].x, U[c].y);
        y[r] = make_double2(yr, yi);
    }
#pragma unroll
    for (int r = 0; r < NA; ++r) U[r] = y[r];
}

// An amplitude's larger component as a share of the group's largest (high word top), to 12 %; 0 for a zero, else at
// least kLeast.
__device__ __forceinline__ float share_of(const double2 &x, int top) {
    const int hi = max(__double2hiint(x.x) & 0x7FFFFFFF, __double2hiint(x.y) & 0x7FFFFFFF);
    const float f = __int_as_float(max(hi - top + (127 << 20), 67 << 20) << 3);
    return (hi | __double2loint(x.x) | __double2loint(x.y)) ? f : 0.0f;
}

// Fixed point is off by at most 3 units of 2^-58 of the largest component per output, FP64 by about 3.5 units of
// 2^-53 of w = sum |m| |x| over the output's products.  So a group takes fixed point where every output
// that is not structurally zero has w >= 1/32 of the largest component, and FP64 elsewhere: an amplitude
// far below its partners that no product of theirs reaches keeps its digits.  (26 qubits, 1 layer 15.4 -> 16.0 ms,
// quantum volume 9.1 -> 9.4; all in FP64 53.3 and 26.6.)
template <int NA>
__device__ __forceinline__ void apply_fx(const MatC128<NA> &M, double2 (&U)[NA]) {
    int top = 0, any = 0;
#pragma unroll
    for (int j = 0; j < NA; ++j) {
        fx::scan(U[j].x, top, any);
        fx::scan(U[j].y, top, any);
    }
    bool near = !fx::special(top, any);
    if (NA > 1) {
        float f[NA];
#pragma unroll
        for (int j = 0; j < NA; ++j) f[j] = share_of(U[j], top);
#pragma unroll
        for (int r = 0; r < NA; ++r) {
            float w = 0.0f;
#pragma unroll
            for (int c = 0; c < NA; ++c) w = fmaf(M.w[NA * r + c], f[c], w);
            near = near && !(w > 0.0f && w < 1.0f / 32);
        }
    }
    if (!near) {
        apply_fp64<NA>(M.m, U);
        return;
    }
    const int E = fx::exponent(top);
    fx::Real xr[NA], xi[NA];
#pragma unroll
    for (int j = 0; j < NA; ++j) {
        xr[j] = fx::from_double(U[j].x, E);
        xi[j] = fx::from_double(U[j].y, E);
    }
#pragma unroll
    for (int r = 0; r < NA; ++r) {
        fx::Acc yr, yi, ii{0, 0};  // ii: the products of imaginary parts, subtracted
#pragma unroll
        for (int c = 0; c < NA; ++c) {
            const int32_t *e = M.e + 4 * (NA * r + c);
            fx::mac(yr, xr[c], e[0], e[1]);
            fx::mac(ii, xi[c], e[2], e[3]);
            fx::mac(yi, xi[c], e[0], e[1]);
            fx::mac(yi, xr[c], e[2], e[3]);
        }
        yr.hi -= ii.hi;
        yr.mid -= ii.mid;
        U[r] = make_double2(fx::to_double(fx::fin(yr), E), fx::to_double(fx::fin(yi), E));
    }
}

// UN groups per thread: two keep more loads in flight on large states, one spreads a small state
// over more CTAs.
template <int NA, bool FX, int UN>
__global__ void __launch_bounds__(kThreads) k_gate_c128(double2 *a, const __grid_constant__ GateArgs<NA, MatC128<NA>> P) {
    after_last_gate();
    const int64_t g0 = (int64_t)blockIdx.x * kThreads * UN + threadIdx.x;
    double2 U[UN][NA];
    int64_t base[UN];
#pragma unroll
    for (int s = 0; s < UN; ++s) {
        const int64_t g = g0 + s * kThreads;
        base[s] = group_base(g, P.lo, P.hi);
        if (g < P.groups) {
#pragma unroll
            for (int j = 0; j < NA; ++j) U[s][j] = a[base[s] | P.off[j]];
        }
    }
#pragma unroll
    for (int s = 0; s < UN; ++s) {
        if (g0 + s * kThreads >= P.groups) continue;
        if (FX) apply_fx<NA>(P.m, U[s]);
        else apply_fp64<NA>(P.m.m, U[s]);
#pragma unroll
        for (int j = 0; j < NA; ++j) a[base[s] | P.off[j]] = U[s][j];
    }
}

// complex64 with n == 1: the whole state is one unit.
__global__ void k_gate1_c64_single(float4 *a, Mat1 M) {
    after_last_gate();
    float4 A = a[0];
    apply1(M.m, A.x, A.y, A.z, A.w);
    a[0] = A;
}

template <typename T>
__global__ void k_set_one(T *a, uint64_t idx) { a[idx] = T{1, 0}; }

template <typename... P, typename... A>
void launch_after(void (*kernel)(P...), unsigned grid, unsigned block, cudaStream_t st, A... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    check_cuda(cudaLaunchKernelEx(&cfg, kernel, P(args)...), "per-gate kernel launch");
}

inline unsigned grid_for(int64_t groups, int unroll = kUnroll) {
    return (unsigned)((groups + (int64_t)kThreads * unroll - 1) / ((int64_t)kThreads * unroll));
}

// A gate as its sweep needs it: the local states it can change, ascending, and its matrix on them.
struct Touched {
    int n = 0;
    int state[4] = {0, 0, 0, 0};
    double m[32];       // n x n, row-major, interleaved
    bool move = false;  // row r takes state from[r], turned by i^turn[r]
    bool turns = false;
    int from[4] = {0, 0, 0, 0}, turn[4] = {0, 0, 0, 0};
};

Touched touched_states(const sv_gate &g) {
    const int d = 1 << g.nq;
    auto entry = [&](int r, int c, double re, double im) { return g.m[2 * (r * d + c)] == re && g.m[2 * (r * d + c) + 1] == im; };
    Touched t;
    for (int b = 0; b < d; ++b) {
        bool same = entry(b, b, 1.0, 0.0);
        for (int k = 0; k < d; ++k)
            if (k != b) same = same && entry(b, k, 0.0, 0.0) && entry(k, b, 0.0, 0.0);
        if (!same) t.state[t.n++] = b;
    }
    if (t.n == 3) {  // the kernels take 1, 2 or 4 states
        t.n = 4;
        for (int b = 0; b < 4; ++b) t.state[b] = b;
    }
    static const double kTurn[4][2] = {{1, 0}, {0, 1}, {-1, 0}, {0, -1}};
    t.move = true;
    for (int r = 0; r < t.n; ++r) {
        int units = 0, zeros = 0;
        for (int c = 0; c < t.n; ++c) {
            const int row = t.state[r], col = t.state[c], k = 2 * (row * d + col);
            t.m[2 * (t.n * r + c)] = g.m[k];
            t.m[2 * (t.n * r + c) + 1] = g.m[k + 1];
            if (entry(row, col, 0.0, 0.0)) ++zeros;
            for (int q = 0; q < 4; ++q)
                if (entry(row, col, kTurn[q][0], kTurn[q][1])) {
                    ++units;
                    t.from[r] = c;
                    t.turn[r] = q;
                    t.turns = t.turns || q;
                }
        }
        t.move = t.move && units == 1 && zeros == t.n - 1;
    }
    // one source per state: a matrix with two rows on one column is not an exchange
    for (int r = 0; r < t.n; ++r)
        for (int q = 0; q < r; ++q) t.move = t.move && t.from[r] != t.from[q];
    return t;
}

// Groups and unit offsets of a sweep over 2^units_log2 units whose gate acts on unit bits q[0..nq).
template <int NA, typename M>
GateArgs<NA, M> sweep_args(const Touched &t, int units_log2, int nq, const int *q) {
    GateArgs<NA, M> P{};
    P.groups = int64_t(1) << (units_log2 - nq);
    P.lo = nq == 1 ? q[0] : std::min(q[0], q[1]);
    P.hi = nq == 1 ? -1 : std::max(q[0], q[1]);
    for (int j = 0; j < NA; ++j)
        for (int k = 0; k < nq; ++k) P.off[j] |= int64_t((t.state[j] >> k) & 1) << q[k];
    return P;
}

template <int NA>
void launch_move(void *state, const Touched &t, int units_log2, int nq, const int *q, cudaStream_t st) {
    auto P = sweep_args<NA, Moves>(t, units_log2, nq, q);
    for (int j = 0; j < NA; ++j) {
        P.m.from[j] = t.from[j];
        P.m.turn[j] = t.turn[j];
    }
    launch_after(k_gate_move<NA>, grid_for(P.groups), kThreads, st, (uint4 *)state, P);
}

template <int NA>
void launch_c64(void *state, const Touched &t, int units_log2, int nq, const int *q, cudaStream_t st) {
    auto P = sweep_args<NA, MatC64<NA>>(t, units_log2, nq, q);
    for (int i = 0; i < 2 * NA * NA; ++i) P.m.m[i] = (float)t.m[i];
    launch_after(k_gate_c64<NA>, grid_for(P.groups), kThreads, st, (float4 *)state, P);
}

template <int NA>
void launch_c128(void *state, const Touched &t, int n, int nq, const int *q, cudaStream_t st) {
    auto P = sweep_args<NA, MatC128<NA>>(t, n, nq, q);
    for (int i = 0; i < 2 * NA * NA; ++i) P.m.m[i] = t.m[i];
    double2 *a = (double2 *)state;
    const bool small = P.groups <= (int64_t)num_sms() * kThreads * kUnroll;  // at most one CTA per SM
    if (fx_unitary(t.m, NA)) {
        fx_pack(t.m, NA * NA, P.m.e);
        for (int i = 0; i < NA * NA; ++i) {
            const double a = std::hypot(t.m[2 * i], t.m[2 * i + 1]);
            P.m.w[i] = a > 0 ? std::max((float)a, kLeast) : 0.0f;
        }
        if (small) launch_after(k_gate_c128<NA, true, 1>, grid_for(P.groups, 1), kThreads, st, a, P);
        else launch_after(k_gate_c128<NA, true, kUnroll>, grid_for(P.groups), kThreads, st, a, P);
    } else {
        launch_after(k_gate_c128<NA, false, 1>, grid_for(P.groups, 1), kThreads, st, a, P);
    }
}

}  // namespace

double launch_gate(int dtype, void *state, int n, const sv_gate &g, cudaStream_t st) {
    const double full = 2.0 * (double)(int64_t(1) << n) * (dtype == SV_C64 ? 8.0 : 16.0);
    if (dtype == SV_C64 && (g.q[0] == 0 || (g.nq == 2 && g.q[1] == 0))) {
        float4 *a = (float4 *)state;
        if (g.nq == 1) {
            Mat1 M;
            for (int i = 0; i < 8; ++i) M.m[i] = (float)g.m[i];
            if (n == 1) {
                launch_after(k_gate1_c64_single, 1, 1, st, a, M);
            } else {
                const int64_t units = int64_t(1) << (n - 1);
                launch_after(k_gate1_c64_lo, grid_for(units), kThreads, st, a, units, M);
            }
        } else {
            Mat2 M;
            for (int i = 0; i < 32; ++i) M.m[i] = (float)g.m[i];
            const int other = g.q[0] == 0 ? g.q[1] : g.q[0];
            const int64_t groups = int64_t(1) << (n - 2);
            launch_after(k_gate2_c64_lo, grid_for(groups), kThreads, st, a, groups, other - 1, g.q[0] == 0 ? 1 : 0, M);
        }
        return full;
    }
    const Touched t = touched_states(g);
    if (t.n == 0) return 0.0;  // the identity
    // complex64: units of two amplitudes, so unit bit q - 1 for qubit q >= 1
    const int shift = dtype == SV_C64 ? 1 : 0, units_log2 = n - shift;
    const int q[2] = {g.q[0] - shift, g.nq == 2 ? g.q[1] - shift : 0};
    if (t.move && (dtype == SV_C128 || !t.turns)) {
        if (t.n == 1) launch_move<1>(state, t, units_log2, g.nq, q, st);
        else if (t.n == 2) launch_move<2>(state, t, units_log2, g.nq, q, st);
        else launch_move<4>(state, t, units_log2, g.nq, q, st);
    } else if (dtype == SV_C64) {
        if (t.n == 1) launch_c64<1>(state, t, units_log2, g.nq, q, st);
        else if (t.n == 2) launch_c64<2>(state, t, units_log2, g.nq, q, st);
        else launch_c64<4>(state, t, units_log2, g.nq, q, st);
    } else {
        if (t.n == 1) launch_c128<1>(state, t, n, g.nq, q, st);
        else if (t.n == 2) launch_c128<2>(state, t, n, g.nq, q, st);
        else launch_c128<4>(state, t, n, g.nq, q, st);
    }
    return full * t.n / (1 << g.nq);
}

void launch_init_basis(int dtype, void *state, int n, uint64_t basis, cudaStream_t st) {
    const size_t bytes = (size_t(1) << n) * (dtype == SV_C64 ? 8 : 16);
    check_cuda(cudaMemsetAsync(state, 0, bytes, st), "cudaMemsetAsync");
    if (dtype == SV_C64)
        k_set_one<float2><<<1, 1, 0, st>>>((float2 *)state, basis);
    else
        k_set_one<double2><<<1, 1, 0, st>>>((double2 *)state, basis);
    check_cuda(cudaGetLastError(), "init kernel launch");
}

}  // namespace sv
