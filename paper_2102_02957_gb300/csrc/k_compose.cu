// Gate fusion for the tensor-core path: every register group of r bits (r = 3, 4, 5) in a
// blocking section becomes one dense 2^r x 2^r complex unitary, composed in FP64 on the GPU, then
// written as the B operand of a real GEMM in the tensor cores' canonical shared-memory layout,
// split into TF32 high and low parts.
//
// Real embedding: a register group holds NA = 2^r amplitudes x_c, stored interleaved as the row
// [re x_0, im x_0, re x_1, ...] (K = 2 NA).  The fused unitary U maps it to y_s = sum_c U_sc x_c,
// i.e. D = A B with
//     B[2c][2s] = Re U_sc,  B[2c+1][2s] = -Im U_sc,  B[2c][2s+1] = Im U_sc,  B[2c+1][2s+1] = Re U_sc.
// B (K rows x N = K columns) is stored K-major without swizzle: 8-row x 16-byte core matrices,
// element (k, n) at byte (n / 8) * SBO + (k / 4) * 128 + (n % 8) * 16 + (k % 4) * 4, SBO = 32 K;
// B_lo follows B_hi directly, so that the pair reads as one K x 2K operand [B_hi | B_lo].
// The high part is B rounded to TF32 (round to nearest), the low part the remainder, also
// rounded to nearest TF32 (the tensor cores would otherwise truncate it, a one-sided error).
#include <cuda_fp16.h>

#include "fixed64.cuh"
#include "sv_internal.h"

namespace sv {
namespace {

__device__ __forceinline__ uint32_t tf32_rna(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

// One CTA per register group; every thread owns elements (row r, column j) of the running product
// U, kept in two shared-memory copies that a gate reads and writes in turn.  (With one thread per
// column walking its gates alone the kernel was a serial chain of FP64 latencies, 209 us for the
// 69 groups of a 20-qubit ansatz; so it takes 22 us.)  Gate records are fetched kGates at a
// time, so that their latency is paid once per batch.
template <int R>
__global__ void __launch_bounds__(256) k_compose_f64(const ComposeSeg *__restrict__ segs,
                                                     const DevGate<double> *__restrict__ gates,
                                                     unsigned char *__restrict__ prog, int *__restrict__ all_unitary) {
    constexpr int NA = 1 << R, K = 2 * NA, SBO = 32 * K, NE = NA * NA, kGates = 16;
    extern __shared__ __align__(16) unsigned char smem[];
    double2 *U = reinterpret_cast<double2 *>(smem);  // [2][NE], element r * NA + j
    __shared__ __align__(16) DevGate<double> sg_gates[kGates];
    __shared__ unsigned long long dev_bits;
    const ComposeSeg sg = segs[blockIdx.x];
    const int tid = threadIdx.x, nt = blockDim.x;
    if (tid == 0) dev_bits = 0;
    for (int e = tid; e < NE; e += nt) U[e] = make_double2((e >> R) == (e & (NA - 1)) ? 1.0 : 0.0, 0.0);
    int cur = 0;
    for (int base = sg.g0; base < sg.g1; base += kGates) {
        const int count = min(kGates, sg.g1 - base);
        __syncthreads();  // the last batch's records are used up
        const uint4 *src = reinterpret_cast<const uint4 *>(gates + base);
        for (int k = tid; k < count * (int)(sizeof(DevGate<double>) / 16); k += nt)
            reinterpret_cast<uint4 *>(sg_gates)[k] = src[k];
        __syncthreads();
        for (int gi = 0; gi < count; ++gi) {
            const DevGate<double> &g = sg_gates[gi];
            const double2 *x = U + cur * NE;
            double2 *y = U + (cur ^ 1) * NE;
            const int ba = 1 << g.a;
            for (int e = tid; e < NE; e += nt) {
                const int r = e >> R, j = e & (NA - 1);
                double2 out;
                if (g.op == OP_DENSE1 || g.op == OP_X1) {
                    const double *m = g.m + ((r & ba) ? 4 : 0);
                    const double2 p = x[((r & ~ba) << R) | j], q = x[((r | ba) << R) | j];
                    out.x = m[0] * p.x - m[1] * p.y + m[2] * q.x - m[3] * q.y;
                    out.y = m[0] * p.y + m[1] * p.x + m[2] * q.y + m[3] * q.x;
                } else if (g.op == OP_DIAG1 || g.op == OP_DIAG2) {
                    const int l = ((r >> g.a) & 1) | (g.op == OP_DIAG2 ? ((r >> g.b) & 1) << 1 : 0);
                    const double dr = g.m[2 * l], di = g.m[2 * l + 1];
                    out = x[e];
                    if (!(dr == 1.0 && di == 0.0)) out = make_double2(dr * out.x - di * out.y, dr * out.y + di * out.x);
                } else {
                    const int bb = 1 << g.b, l = ((r >> g.a) & 1) | (((r >> g.b) & 1) << 1);
                    const int r0 = r & ~(ba | bb);
                    auto row = [&](int c) { return r0 | ((c & 1) ? ba : 0) | ((c & 2) ? bb : 0); };
                    if (g.op == OP_DENSE2) {
                        out = make_double2(0.0, 0.0);
                        for (int c = 0; c < 4; ++c) {
                            const double2 p = x[(row(c) << R) | j];
                            const double mr = g.m[2 * (4 * l + c)], mi = g.m[2 * (4 * l + c) + 1];
                            out.x += mr * p.x - mi * p.y;
                            out.y += mr * p.y + mi * p.x;
                        }
                    } else {  // an exchange: row l takes row m[l]
                        out = x[(row((int)g.m[l]) << R) | j];
                    }
                }
                y[e] = out;
            }
            cur ^= 1;
            __syncthreads();
        }
    }
    __syncthreads();
    const double2 *x = U + cur * NE;
    // unitarity of the fused matrix: max |(U^H U - I)_ij| over all i <= j (the rest is conjugate)
    double worst = 0.0;
    for (int e = tid; e < NE; e += nt) {
        const int i = e >> R, j = e & (NA - 1);
        if (i > j) continue;
        double gr = 0.0, gi = 0.0;  // <U e_i, U e_j>
        for (int r = 0; r < NA; ++r) {
            const double2 p = x[(r << R) | i], q = x[(r << R) | j];
            gr += p.x * q.x + p.y * q.y;
            gi += p.x * q.y - p.y * q.x;
        }
        const double d = fabs(gr - (i == j ? 1.0 : 0.0)) + fabs(gi);
        worst = d > worst || !(d == d) ? d : worst;
    }
    // non-negative values (and NaN above them all) order as integers
    atomicMax(&dev_bits, (unsigned long long)__double_as_longlong(worst) & 0x7FFFFFFFFFFFFFFFull);
    __syncthreads();
    const bool unitary = __longlong_as_double((long long)dev_bits) <= 1e-10;
    if (tid == 0 && !unitary && all_unitary) atomicAnd(all_unitary, 0);
    if (tid == 0 && sg.flag_off != kNoFlag) *reinterpret_cast<int *>(prog + sg.flag_off) = unitary ? 1 : 0;
    unsigned char *bhi = prog + sg.b_off, *blo = bhi + 4 * K * K;
    auto b_offset = [](int k, int n) {
        return (uint32_t)((n >> 3) * SBO + (k >> 2) * 128 + (n & 7) * 16 + (k & 3) * 4);
    };
    for (int e = tid; e < NE; e += nt) {
        const int r = e >> R, j = e & (NA - 1);
        const double u_re = x[e].x, u_im = x[e].y;
        const double val[4] = {u_re, -u_im, u_im, u_re};  // (k, n) = (2j, 2r), (2j+1, 2r), (2j, 2r+1), (2j+1, 2r+1)
        const int kk[4] = {2 * j, 2 * j + 1, 2 * j, 2 * j + 1};
        const int nn[4] = {2 * r, 2 * r, 2 * r + 1, 2 * r + 1};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float f = (float)val[q];
            const uint32_t hi = tf32_rna(f);
            const uint32_t lo = tf32_rna((float)(val[q] - (double)__uint_as_float(hi)));
            *reinterpret_cast<uint32_t *>(bhi + b_offset(kk[q], nn[q])) = hi;
            *reinterpret_cast<uint32_t *>(blo + b_offset(kk[q], nn[q])) = lo;
        }
    }
}

// Fused unitary of a complex128 group (block_oz.cuh), in block fixed point with the fixed scale 2^59
// (all entries of unitaries are at most 1), from the section's own gate area; then
// M = round(U 2^(54 + s)) in balanced base-256 digits as FP16 B operands, s the most (up to 2) that
// keeps |M| within 0.99 * 2^55.  One CTA per group, one thread
// per element (row r, column j); element products read and write two shared copies in turn.
__global__ void __launch_bounds__(256) k_compose_fx(const OzCompose *__restrict__ groups, unsigned char *__restrict__ prog,
                                                    unsigned char *__restrict__ operands) {
    constexpr int NA = 16;
    __shared__ fx::Real Ur[2][NA * NA], Ui[2][NA * NA];
    const OzCompose sg = groups[blockIdx.x];
    const unsigned char *gates = prog + sg.gates_off;
    const int e = threadIdx.x, r = e >> 4, j = e & 15;
    int cur = 0;
    Ur[0][e] = r == j ? fx::pack(1ll << 59) : fx::Real{0, 0};
    Ui[0][e] = fx::Real{0, 0};
    __syncthreads();
    for (int gi = sg.g0; gi < sg.g1; ++gi) {
        const int4 hd = reinterpret_cast<const int4 *>(gates)[gi];  // op, payload offset, -, code
        const int op = hd.x, code = hd.w;
        const int4 *pay = reinterpret_cast<const int4 *>(gates + hd.y);
        const bool one = op == OP_DENSE1 || op == OP_REAL1 || op == OP_DIAG1 || op == OP_X1;
        const int ba = one ? 1 << code : 1 << (code >> 3), bb = one ? 0 : 1 << (code & 7);
        const int l = ((r & ba) ? 1 : 0) | ((r & bb) ? 2 : 0), r0 = r & ~(ba | bb);
        auto at = [&](int c) { return ((r0 | ((c & 1) ? ba : 0) | ((c & 2) ? bb : 0)) << 4) | j; };
        fx::Acc yr, yi;
        auto term = [&](int c, int4 m) {
            const fx::Real xr = Ur[cur][at(c)], xi = Ui[cur][at(c)];
            fx::mac(yr, xr, m.x, m.y);
            fx::mac(yr, xi, -m.z, -m.w);
            fx::mac(yi, xi, m.x, m.y);
            fx::mac(yi, xr, m.z, m.w);
        };
        int from = -1;
        if (op == OP_DENSE1) {
            for (int c = 0; c < 2; ++c) term(c, pay[2 * l + c]);
        } else if (op == OP_REAL1) {
            const int4 row = pay[l];
            term(0, make_int4(row.x, row.y, 0, 0));
            term(1, make_int4(row.z, row.w, 0, 0));
        } else if (op == OP_DENSE2) {
            for (int c = 0; c < 4; ++c) term(c, pay[4 * l + c]);
        } else if (op == OP_DIAG1 || op == OP_DIAG2) {
            term(l, pay[l]);
        } else if (op == OP_X1) {
            from = l ^ 1;
        } else if (op == OP_CXA) {
            from = (l & 1) ? l ^ 2 : l;
        } else if (op == OP_CXB) {
            from = (l & 2) ? l ^ 1 : l;
        } else if (op == OP_SWAP2) {
            from = ((l & 1) << 1) | (l >> 1);
        } else {
            from = reinterpret_cast<const int *>(pay)[l];
        }
        const int nx = cur ^ 1;
        Ur[nx][e] = from >= 0 ? Ur[cur][at(from)] : fx::fin(yr);
        Ui[nx][e] = from >= 0 ? Ui[cur][at(from)] : fx::fin(yi);
        cur = nx;
        __syncthreads();
    }
    // entries (k, n) = (2j, 2r), (2j + 1, 2r), (2j, 2r + 1), (2j + 1, 2r + 1) = re, -im, im, re
    constexpr long long kBias = 0x0080808080808080ll;
    const long long ure = fx::value(Ur[cur][e]), uim = fx::value(Ui[cur][e]);
    __shared__ int top;  // largest |entry| in units of 2^-27
    if (e == 0) top = 0;
    __syncthreads();
    atomicMax(&top, (int)(llabs(ure) >> 32));
    atomicMax(&top, (int)(llabs(uim) >> 32));
    __syncthreads();
    const double most = (double)(top + 1) * 0x1p-27;
    const int s = most <= 0.495 ? 2 : most <= 0.99 ? 1 : 0;
    if (e == 0) *reinterpret_cast<int *>(prog + sg.scale_off) = s;
    const long long half = 16 >> s;
    const long long re = (ure + half) >> (5 - s), im = (uim + half) >> (5 - s);
    unsigned char *b = operands + sg.b_off + (r >> 3) * (kOzBBytes / 2);
#pragma unroll
    for (int part = 0; part < 2; ++part) {
        const int n = 2 * (r & 7) + part;  // output real within its half row
        const unsigned long long lo = (unsigned long long)((part ? im : re) + kBias), hi = (unsigned long long)((part ? re : -im) + kBias);
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            const int row = 16 * d + n;  // N row of digit block d
            __half2 v = __floats2half2_rn(0.f, 0.f);
            if (d < 7) {
                const int at = 8 * (6 - d);
                v = __floats2half2_rn((float)((int)((lo >> at) & 255) - 128), (float)((int)((hi >> at) & 255) - 128));
            }
            *reinterpret_cast<__half2 *>(b + (row >> 3) * 512 + (j >> 2) * 128 + (row & 7) * 16 + (j & 3) * 4) = v;
        }
    }
}

}  // namespace

void launch_compose_oz(const void *dev_groups, int ngroups, void *dev_prog, void *dev_operands, cudaStream_t st) {
    if (ngroups <= 0) return;
    k_compose_fx<<<ngroups, 256, 0, st>>>((const OzCompose *)dev_groups, (unsigned char *)dev_prog, (unsigned char *)dev_operands);
    check_cuda(cudaGetLastError(), "compose kernel launch");
}

void launch_compose(const void *dev_segs, int nseg, const void *dev_gates, void *dev_prog, int *all_unitary, int r,
                    cudaStream_t st) {
    if (nseg <= 0) return;
    const ComposeSeg *sg = (const ComposeSeg *)dev_segs;
    const DevGate<double> *g = (const DevGate<double> *)dev_gates;
    unsigned char *p = (unsigned char *)dev_prog;
    const size_t smem = (size_t)32 << (2 * r);  // two copies of the 2^r x 2^r product (at most 32 KiB)
    if (r == 3) k_compose_f64<3><<<nseg, 64, smem, st>>>(sg, g, p, all_unitary);
    else if (r == 4) k_compose_f64<4><<<nseg, 256, smem, st>>>(sg, g, p, all_unitary);
    else if (r == 5) k_compose_f64<5><<<nseg, 256, smem, st>>>(sg, g, p, all_unitary);
    else fail(SV_ERR_UNSUPPORTED, "fused groups have 3, 4 or 5 bits");
    check_cuda(cudaGetLastError(), "compose kernel launch");
}

}  // namespace sv
