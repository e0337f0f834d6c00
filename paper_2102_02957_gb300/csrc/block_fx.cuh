// Register-group engine of complex128 sections on the integer pipe (arithmetic: fixed64.cuh).
//
// Same shape as run_segment: a thread loads the 16 amplitudes spanned by the group's 4 chunk bits,
// applies every gate of the group, stores them back.  In between the components are block
// fixed-point integers with one exponent per thread, converted once each way per group -- or, in a
// group that only exchanges amplitudes and flips signs (kSegRaw), the doubles' own words, and in one of
// diagonals alone (kSegDiag) doubles.
//
// Bound by the multiply-add pipe (57 % busy on random-layer sections, where run_segment kept the
// FP64 pipe full) and by the dependent chains that two warps per scheduler leave exposed: 168
// registers a thread allow no more, and 3 x 128 threads of 128 registers spill (217 ms against 166
// for the first line below).  Measured against FP64 register groups, n qubits, 12-bit chunks:
//   27, 8 random layers (12 sections, 44 groups)       417 -> 169 ms
//   28, QFT with diagonals outside the chunk           393 -> 239 ms, with merged runs 160 ms
//   25, quantum volume of 10 layers, gathered chunks   108 -> 38.6 ms
// (all of them before the chunks were looked over, ChunkRange: two passes over a chunk in shared memory)
//
// The section's gate area is a table of 16-byte headers {op, payload offset, outside bits, code},
// then the payloads (encode_fx writes them):
//   OP_DENSE1 / OP_DENSE2  4 / 16 entries {re h, re l, im h, im l}     OP_REAL1  4 x {h, l}
//   OP_DIAG1 / OP_DIAG2    2 / 4 entries   OP_DIAGX  2 or 4 OP_DIAG1   OP_PERM2  4 ints
//   OP_DIAGRUN  the run's gates and kFxRunBytes of tables, filled per chunk (fx_merge): a
//   QFT section has up to 16 controlled phases from outside the chunk on each of its qubits
#pragma once
#include "block_core.cuh"
#include "fixed64.cuh"

namespace sv {
namespace {

// Real and imaginary component of every amplitude of the thread's group.
template <int NA>
struct FxGroup {
    fx::Real re[NA], im[NA];
};

struct FxEntry {
    int rh, rl, ih, il;
};
__device__ __forceinline__ FxEntry lds_entry(uint32_t a) {
    FxEntry e;
    ldc_i4(a, e.rh, e.rl, e.ih, e.il);
    return e;
}

// (yr, yi) accumulators += entry * (xr + i xi)
__device__ __forceinline__ void fx_cmac(fx::Acc &yr, fx::Acc &yi, const FxEntry &m, const fx::Real &xr, const fx::Real &xi) {
    fx::mac(yr, xr, m.rh, m.rl);
    fx::mac(yr, xi, -m.ih, -m.il);
    fx::mac(yi, xi, m.rh, m.rl);
    fx::mac(yi, xr, m.ih, m.il);
}

template <int NA, int A>
__device__ __forceinline__ void fx_dense1(FxGroup<NA> &v, uint32_t ma) {
    const FxEntry m0 = lds_entry(ma), m1 = lds_entry(ma + 16), m2 = lds_entry(ma + 32), m3 = lds_entry(ma + 48);
#pragma unroll
    for (int x = 0; x < NA; ++x) {
        if (x & (1 << A)) continue;
        const int y = x | (1 << A);
        fx::Acc pr, pi, qr, qi;
        fx_cmac(pr, pi, m0, v.re[x], v.im[x]);
        fx_cmac(pr, pi, m1, v.re[y], v.im[y]);
        fx_cmac(qr, qi, m2, v.re[x], v.im[x]);
        fx_cmac(qr, qi, m3, v.re[y], v.im[y]);
        v.re[x] = fx::fin(pr); v.im[x] = fx::fin(pi);
        v.re[y] = fx::fin(qr); v.im[y] = fx::fin(qi);
    }
}

// Real matrix (RY, H): half the products.
template <int NA, int A>
__device__ __forceinline__ void fx_real1(FxGroup<NA> &v, uint32_t ma) {
    const FxEntry r0 = lds_entry(ma), r1 = lds_entry(ma + 16);  // rows {m0 h, m0 l, m1 h, m1 l}
#pragma unroll
    for (int x = 0; x < NA; ++x) {
        if (x & (1 << A)) continue;
        const int y = x | (1 << A);
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            fx::Real &a = part ? v.im[x] : v.re[x], &b = part ? v.im[y] : v.re[y];
            fx::Acc p, q;
            fx::mac(p, a, r0.rh, r0.rl);
            fx::mac(p, b, r0.ih, r0.il);
            fx::mac(q, a, r1.rh, r1.rl);
            fx::mac(q, b, r1.ih, r1.il);
            a = fx::fin(p);
            b = fx::fin(q);
        }
    }
}

template <int NA, int A, int B>
__device__ __forceinline__ void fx_dense2(FxGroup<NA> &v, uint32_t ma) {
#pragma unroll
    for (int x = 0; x < NA; ++x) {
        if (x & ((1 << A) | (1 << B))) continue;
        const int id[4] = {x, x | (1 << A), x | (1 << B), x | (1 << A) | (1 << B)};
        fx::Real xr[4], xi[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) { xr[k] = v.re[id[k]]; xi[k] = v.im[id[k]]; }
#pragma unroll
        for (int rr = 0; rr < 4; ++rr) {
            fx::Acc yr, yi, ii{0, 0};  // ii: the products of imaginary parts, subtracted
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                const FxEntry m = lds_entry(ma + 16 * (4 * rr + cc));
                fx::mac(yr, xr[cc], m.rh, m.rl);
                fx::mac(ii, xi[cc], m.ih, m.il);
                fx::mac(yi, xi[cc], m.rh, m.rl);
                fx::mac(yi, xr[cc], m.ih, m.il);
            }
            yr.hi -= ii.hi;
            yr.mid -= ii.mid;
            v.re[id[rr]] = fx::fin(yr);
            v.im[id[rr]] = fx::fin(yi);
        }
    }
}

// Diagonal entry l on the amplitudes whose gate bits read l; entries of exactly 1 and -1 take no
// products (uniform over the warp).
template <int NA, int A, int B, int NL>
__device__ __forceinline__ void fx_diag(FxGroup<NA> &v, uint32_t ma, bool raw) {
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        const FxEntry d = lds_entry(ma + 16 * l);
        const bool real = d.rl == 0 && d.ih == 0 && d.il == 0;
        if (real && d.rh == fx::kOne) continue;
        if (real && d.rh == -fx::kOne) {
#pragma unroll
            for (int x = 0; x < NA; ++x)
                if ((((x >> A) & 1) | (NL == 4 ? ((x >> B) & 1) << 1 : 0)) == l) {
                    v.re[x] = raw ? fx::flip_sign(v.re[x]) : fx::negate(v.re[x]);
                    v.im[x] = raw ? fx::flip_sign(v.im[x]) : fx::negate(v.im[x]);
                }
            continue;
        }
#pragma unroll
        for (int x = 0; x < NA; ++x)
            if ((((x >> A) & 1) | (NL == 4 ? ((x >> B) & 1) << 1 : 0)) == l) {
                fx::Acc yr, yi;
                fx_cmac(yr, yi, d, v.re[x], v.im[x]);
                v.re[x] = fx::fin(yr);
                v.im[x] = fx::fin(yi);
            }
    }
}

template <int NA, int A>
__device__ __forceinline__ void fx_x1(FxGroup<NA> &v) {
#pragma unroll
    for (int x = 0; x < NA; ++x) {
        if (x & (1 << A)) continue;
        const int y = x | (1 << A);
        fx::Real t = v.re[x]; v.re[x] = v.re[y]; v.re[y] = t;
        t = v.im[x]; v.im[x] = v.im[y]; v.im[y] = t;
    }
}

template <int NA, int A, int B, int U, int V>
__device__ __forceinline__ void fx_xchg2(FxGroup<NA> &v) {
#pragma unroll
    for (int x = 0; x < NA; ++x) {
        if (x & ((1 << A) | (1 << B))) continue;
        const int id[4] = {x, x | (1 << A), x | (1 << B), x | (1 << A) | (1 << B)};
        fx::Real t = v.re[id[U]]; v.re[id[U]] = v.re[id[V]]; v.re[id[V]] = t;
        t = v.im[id[U]]; v.im[id[U]] = v.im[id[V]]; v.im[id[V]] = t;
    }
}

template <int NA, int A, int B>
__device__ __forceinline__ void fx_perm2(FxGroup<NA> &v, uint32_t ma) {
    int p[4];
    ldc_i4(ma, p[0], p[1], p[2], p[3]);
#pragma unroll
    for (int x = 0; x < NA; ++x) {
        if (x & ((1 << A) | (1 << B))) continue;
        const int id[4] = {x, x | (1 << A), x | (1 << B), x | (1 << A) | (1 << B)};
        fx::Real xr[4], xi[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) { xr[k] = v.re[id[k]]; xi[k] = v.im[id[k]]; }
#pragma unroll
        for (int rr = 0; rr < 4; ++rr) {
            const int s = p[rr];
            v.re[id[rr]] = s == 0 ? xr[0] : s == 1 ? xr[1] : s == 2 ? xr[2] : xr[3];
            v.im[id[rr]] = s == 0 ? xi[0] : s == 1 ? xi[1] : s == 2 ? xi[2] : xi[3];
        }
    }
}

template <int NA, int A>
__device__ __forceinline__ void fx_one(int op, FxGroup<NA> &v, uint32_t m, bool raw) {
    if (op == OP_DENSE1) fx_dense1<NA, A>(v, m);
    else if (op == OP_REAL1) fx_real1<NA, A>(v, m);
    else if (op == OP_X1) fx_x1<NA, A>(v);
    else fx_diag<NA, A, 0, 2>(v, m, raw);
}

template <int NA, int A, int B>
__device__ __forceinline__ void fx_two(int op, FxGroup<NA> &v, uint32_t m, bool raw) {
    if (op == OP_DENSE2) fx_dense2<NA, A, B>(v, m);
    else if (op == OP_DIAG2) fx_diag<NA, A, B, 4>(v, m, raw);
    else if (op == OP_CXA) fx_xchg2<NA, A, B, 1, 3>(v);
    else if (op == OP_CXB) fx_xchg2<NA, A, B, 2, 3>(v);
    else if (op == OP_SWAP2) fx_xchg2<NA, A, B, 1, 2>(v);
    else fx_perm2<NA, A, B>(v, m);
}

__device__ __forceinline__ void fx_diag16(FxGroup<16> &v, uint32_t ma);

__device__ __forceinline__ void fx_apply(int op, int code, uint32_t m, FxGroup<16> &v, bool raw) {
    if (op == OP_DIAGRUN) {
        fx_diag16(v, m);
    } else if (op == OP_DENSE1 || op == OP_REAL1 || op == OP_DIAG1 || op == OP_X1) {
        switch (code) {
            case 0: fx_one<16, 0>(op, v, m, raw); break;
            case 1: fx_one<16, 1>(op, v, m, raw); break;
            case 2: fx_one<16, 2>(op, v, m, raw); break;
            default: fx_one<16, 3>(op, v, m, raw); break;
        }
    } else {
        switch (code) {
            case 0 * 8 + 1: fx_two<16, 0, 1>(op, v, m, raw); break;
            case 0 * 8 + 2: fx_two<16, 0, 2>(op, v, m, raw); break;
            case 0 * 8 + 3: fx_two<16, 0, 3>(op, v, m, raw); break;
            case 1 * 8 + 2: fx_two<16, 1, 2>(op, v, m, raw); break;
            case 1 * 8 + 3: fx_two<16, 1, 3>(op, v, m, raw); break;
            default: fx_two<16, 2, 3>(op, v, m, raw); break;
        }
    }
}

// Diagonal of all 16 amplitudes (a merged run).
__device__ __forceinline__ void fx_diag16(FxGroup<16> &v, uint32_t ma) {
#pragma unroll
    for (int x = 0; x < 16; ++x) {
        FxEntry d;  // rewritten for every chunk: not a pure load like the program's
        asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(d.rh), "=r"(d.rl), "=r"(d.ih), "=r"(d.il) : "r"(ma + 16u * x));
        if (d.rh == fx::kOne && d.rl == 0 && d.ih == 0 && d.il == 0) continue;
        fx::Acc yr, yi;
        fx_cmac(yr, yi, d, v.re[x], v.im[x]);
        v.re[x] = fx::fin(yr);
        v.im[x] = fx::fin(yi);
    }
}

// Payload of a gate of group [g0, g1) once its outside bits are read off the chunk's origin.
struct FxGate {
    int op, code;
    uint32_t m;
    int more;  // further headers that belong to it
};
__device__ __forceinline__ uint32_t fx_variant(int outside, int64_t origin) {
    const int e0 = outside & 0xFF, e1 = (outside >> 8) & 0xFF;
    int v = (int)((origin >> e0) & 1);
    if (e1 != 0xFF) v |= (int)((origin >> e1) & 1) << 1;
    return (uint32_t)(32 * v);
}
__device__ __forceinline__ FxGate fx_gate(uint32_t gates, int gi, int64_t origin, int cg) {
    int op, off, rb, code;
    ldc_i4(gates + 16u * (uint32_t)gi, op, off, rb, code);
    uint32_t m = gates + (uint32_t)off;
    int more = 0;
    if (op == OP_DIAGX) {
        m += fx_variant(rb, origin);
        op = OP_DIAG1;
    } else if (op == OP_DIAGRUN) {
        more = rb - 1;
        m += (uint32_t)(16 + 16 * rb + kFxRunBytes / kFxGroups * cg);
    }
    return FxGate{op, code, m, more};
}

// Product of two values of the scale 2^59 of fixed64.cuh, both at most 1 in modulus.
__device__ __forceinline__ void fx_product(fx::Real &ar, fx::Real &ai, const fx::Real &br, const fx::Real &bi) {
    // b in the entries' scale 2^61, its low part negatable
    fx::Real er = fx::pack(fx::value(br) * 4), ei = fx::pack(fx::value(bi) * 4);
    er.l += er.l == (int)0x80000000;
    ei.l += ei.l == (int)0x80000000;
    fx::Acc yr, yi;
    fx_cmac(yr, yi, FxEntry{er.h, er.l, ei.h, ei.l}, ar, ai);
    ar = fx::fin(yr);
    ai = fx::fin(yi);
}

// Tables of the merged runs of gates [g0, g1) for this chunk (NC threads, ends in a barrier).  The run
// is cut into a part per half warp: lane x of a half multiplies entry x over every eighth gate,
// the halves join by shuffle, and a half warp multiplies the warps' parts.  (One half warp alone took
// a chain of up to 64 products per group, longer than the group's own work.)
// as_double: the tables' entries are doubles, for a group of diagonals alone.
template <int NC>
__device__ __forceinline__ void fx_merge(uint32_t gates, int g0, int g1, int64_t origin, int cg, int ctid, int bar_id,
                                         bool as_double) {
    constexpr int W = NC / 32;
    const int lane = ctid & 31, warp = ctid >> 5, x = lane & 15;
    auto store = [](uint32_t a, const fx::Real &r, const fx::Real &i) {
        asm volatile("st.shared.v4.s32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(r.h), "r"(r.l), "r"(i.h), "r"(i.l) : "memory");
    };
    for (int pass = 0; pass < 2; ++pass) {
        for (int gi = g0; gi < g1; ++gi) {
            int op, off, count, code;
            ldc_i4(gates + 16u * (uint32_t)gi, op, off, count, code);
            if (op != OP_DIAGRUN) continue;
            gi += count - 1;
            const uint32_t list = gates + (uint32_t)off + 16;
            const uint32_t table = list + (uint32_t)(16 * count + kFxRunBytes / kFxGroups * cg), parts = table + 256;
            fx::Real pr = fx::pack(1ll << 59), pi{0, 0};
            if (pass == 0) {
                for (int k = 2 * warp; k < count; k += 2 * W) {  // whole warps: the vote
                    const int mine = k + (lane >> 4);
                    FxEntry d{fx::kOne, 0, 0, 0};
                    if (mine < count) {
                        int goff, outside, bit, unused;
                        ldc_i4(list + 16u * (uint32_t)mine, goff, outside, bit, unused);
                        d = lds_entry(gates + (uint32_t)goff + fx_variant(outside, origin) + 16u * (uint32_t)((x >> bit) & 1));
                    }
                    // an outside qubit that reads 0 leaves a controlled phase out
                    if (!__any_sync(0xFFFFFFFFu, d.rh != fx::kOne || d.rl || d.ih || d.il)) continue;
                    fx::Acc yr, yi;
                    fx_cmac(yr, yi, d, pr, pi);
                    pr = fx::fin(yr);
                    pi = fx::fin(yi);
                }
                fx::Real qr, qi;
                qr.h = __shfl_xor_sync(0xFFFFFFFFu, pr.h, 16);
                qr.l = __shfl_xor_sync(0xFFFFFFFFu, pr.l, 16);
                qi.h = __shfl_xor_sync(0xFFFFFFFFu, pi.h, 16);
                qi.l = __shfl_xor_sync(0xFFFFFFFFu, pi.l, 16);
                fx_product(pr, pi, qr, qi);
                if (lane < 16) store(parts + 256u * (uint32_t)warp + 16u * (uint32_t)x, pr, pi);
            } else if (warp == 0) {
                for (int w = 0; w < W; ++w) {
                    fx::Real qr, qi;
                    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(qr.h), "=r"(qr.l), "=r"(qi.h), "=r"(qi.l)
                                 : "r"(parts + 256u * (uint32_t)w + 16u * (uint32_t)x));
                    fx_product(pr, pi, qr, qi);
                }
                const long long vr = fx::value(pr), vi = fx::value(pi);
                fx::Real er = fx::pack(vr * 4), ei = fx::pack(vi * 4);
                er.l += er.l == (int)0x80000000;
                ei.l += ei.l == (int)0x80000000;
                if (lane < 16 && as_double) SM<double>::st(table + 16u * (uint32_t)x, (double)vr * 0x1p-59, (double)vi * 0x1p-59);
                else if (lane < 16) store(table + 16u * (uint32_t)x, er, ei);
            }
        }
        ptx::named_bar_sync(bar_id, NC);
    }
}

// What a chunk's amplitudes look like, for the engines that give a whole register group (here) or chunk
// (block_oz.cuh) one exponent.  Their error is a unit of the chunk's largest component, so they may run a chunk
//   DENSE  of which few enough amplitudes (Dense, sv_internal.h) are small beside that component; or
//   TRIAL  whose results are all within kNearOrders binary orders of it (chunk_filled): states that gates
//          fill from a few amplitudes.  Tried where at most one amplitude in 64 is small and not zero, and only
//          with gates like Hadamards (Dense::trial).
//   ZERO   chunks stay as they are, and so do OTHER ones (and failed trials), which FP64 register groups run
//          next (SweepArgs): components that are not finite or near the ends of the exponent range, states with
//          most of their weight on few amplitudes.
struct ChunkRange {
    int top, zeros, small, near;  // largest high word, amplitudes that are zero, below Dense's line, and below kNearOrders
    int least_out, filled;        // of the results: smallest non-zero, number of non-zero ones,
    unsigned any_bits, all_bits;  // or and and of their indices
    __device__ void clear() volatile {
        top = zeros = small = near = filled = 0;
        least_out = 0x7FFFFFFF;
        any_bits = 0;
        all_bits = ~0u;
    }
};
enum : int { CHUNK_DENSE = 0, CHUNK_TRIAL = 1, CHUNK_ZERO = 2, CHUNK_OTHER = 3 };
constexpr int kMinTop = 200 << 20, kMaxTop = 2030 << 20;

// High word of an amplitude's larger component; some: the amplitude is not zero.
__device__ __forceinline__ int amp_top(uint32_t a, bool &some) {
    double x, y;
    SM<double>::ld(a, x, y);
    const int hi = max(__double2hiint(x) & 0x7FFFFFFF, __double2hiint(y) & 0x7FFFFFFF);
    some = (hi | __double2loint(x) | __double2loint(y)) != 0;
    return hi;
}

// NC threads; sh was cleared before a barrier of theirs.  top: the largest component's high word.
template <int NC>
__device__ __forceinline__ int chunk_range(uint32_t buf, int c, int ctid, int bar_id, volatile ChunkRange *sh, const Dense &d,
                                           int &top) {
    int most = 0, zeros = 0;
    for (int i = ctid; i < (1 << c); i += NC) {
        bool some;
        most = max(most, amp_top(buf + 16u * (uint32_t)i, some));
        zeros += some ? 0 : 1;
    }
    most = __reduce_max_sync(0xFFFFFFFFu, most);
    zeros = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)zeros);
    if ((ctid & 31) == 0) {
        atomicMax(const_cast<int *>(&sh->top), most);
        if (zeros) atomicAdd(const_cast<int *>(&sh->zeros), zeros);
    }
    ptx::named_bar_sync(bar_id, NC);
    top = sh->top;
    zeros = sh->zeros;
    if (zeros == 1 << c) return CHUNK_ZERO;
    if (d.orders < 0) return CHUNK_DENSE;
    if (top < kMinTop || top >= kMaxTop) return CHUNK_OTHER;
    const int line = top - (d.orders << 20), near = top - (kNearOrders << 20);
    int below = 0;  // in two halves: of `line`, of `near`
    for (int i = ctid; i < (1 << c); i += NC) {
        bool some;
        const int hi = amp_top(buf + 16u * (uint32_t)i, some);
        below += (hi < line ? 1 : 0) + (hi < near ? 0x10000 : 0);
    }
    below = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)below);
    if ((ctid & 31) == 0 && below) {
        atomicAdd(const_cast<int *>(&sh->small), below & 0xFFFF);
        atomicAdd(const_cast<int *>(&sh->near), below >> 16);
    }
    ptx::named_bar_sync(bar_id, NC);
    if (sh->small <= d.most) return CHUNK_DENSE;
    return d.trial && (sh->near - zeros) * 64 <= (1 << c) ? CHUNK_TRIAL : CHUNK_OTHER;
}

// Whether the results of a TRIAL (in the natural layout, behind a barrier of the group) are within the orders.
// A zero among them is one whose inputs are zero, not a small result lost, where the non-zero ones fill a
// cube of the index space in which every bit that a dense gate touched (dense_bits) runs free.
template <int NC>
__device__ __forceinline__ bool chunk_filled(uint32_t buf, int c, int ctid, int bar_id, volatile ChunkRange *sh, int top,
                                             unsigned dense_bits) {
    int least = 0x7FFFFFFF, filled = 0;
    unsigned any_bits = 0, all_bits = ~0u;
    for (int i = ctid; i < (1 << c); i += NC) {
        bool some;
        const int hi = amp_top(buf + 16u * (uint32_t)i, some);
        if (!some) continue;
        least = min(least, hi);
        ++filled;
        any_bits |= (unsigned)i;
        all_bits &= (unsigned)i;
    }
    least = __reduce_min_sync(0xFFFFFFFFu, least);
    filled = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)filled);
    any_bits = __reduce_or_sync(0xFFFFFFFFu, any_bits);
    all_bits = __reduce_and_sync(0xFFFFFFFFu, all_bits);
    if ((ctid & 31) == 0) {
        atomicMin(const_cast<int *>(&sh->least_out), least);
        atomicAdd(const_cast<int *>(&sh->filled), filled);
        atomicOr(const_cast<unsigned *>(&sh->any_bits), any_bits);
        atomicAnd(const_cast<unsigned *>(&sh->all_bits), all_bits);
    }
    ptx::named_bar_sync(bar_id, NC);
    const unsigned free_bits = sh->any_bits & ~sh->all_bits;
    return sh->least_out >= top - (kNearOrders << 20) && sh->filled == 1 << __popc(free_bits) && (dense_bits & ~free_bits) == 0;
}

// A group of diagonals in FP64: they mix nothing, so every amplitude keeps an exponent of its own, and a merged
// run is one product of 4 FP64 operations an amplitude, fewer than the conversions to fixed point and back.
__device__ __forceinline__ void fx_diagonals(double (&re)[16], double (&im)[16], uint32_t gates, int g0, int g1, int64_t origin, int cg) {
    auto entry = [](uint32_t a) { return ((double)lds_s32(a) * 4294967296.0 + (double)lds_s32(a + 4)) * 0x1p-61; };
    for (int gi = g0; gi < g1; ++gi) {
        const FxGate g = fx_gate(gates, gi, origin, cg);
        gi += g.more;
        const int a = g.op == OP_DIAG2 ? g.code >> 3 : g.code, b = g.code & 7;
#pragma unroll
        for (int x = 0; x < 16; ++x) {
            double tr, ti;
            if (g.op == OP_DIAGRUN) {
                SM<double>::ld(g.m + 16u * (uint32_t)x, tr, ti);
            } else {
                const uint32_t e = g.m + 16u * (uint32_t)(((x >> a) & 1) | (g.op == OP_DIAG2 ? ((x >> b) & 1) << 1 : 0));
                tr = entry(e);
                ti = entry(e + 8);
            }
            if (tr == 1.0 && ti == 0.0) continue;
            scale_amp(re[x], im[x], tr, ti);
        }
    }
}

// One register group of 4 bits over the chunk in shared memory (see run_segment for the addressing).
template <int NC>
__device__ __forceinline__ void run_segment_fx(uint32_t buf, uint32_t seg, uint32_t gates, int ctid, const int *swz,
                                               int c, int64_t origin, int cg, int bar_id) {
    constexpr int R = 4, NA = 1 << R;
    int po[R], pf[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const int p = lds_s8(seg + j);
        po[j] = 1 << p;
        pf[j] = po[j] ^ swz[p];
    }
    const int lane = ctid & 31;
    int lbase = 0, lfb = 0;
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const int p = lds_s8(seg + 8 + j);
        if ((lane >> j) & 1) { lbase |= 1 << p; lfb ^= swz[p]; }
    }
    const int nrest = lds_s8(seg + 13), flags = lds_s8(seg + 14);
    const int g0 = lds_s16(seg + 32), g1 = lds_s16(seg + 34);
    const int G = 1 << (c - R);
    bool merged = false;  // uniform: whether the group has merged runs
    for (int gi = g0; gi < g1; ++gi) merged = merged || lds_s32(gates + 16u * (uint32_t)gi) == OP_DIAGRUN;
    const bool diagonal = (flags & kSegDiag) != 0;
    if (merged) fx_merge<NC>(gates, g0, g1, origin, cg, ctid, bar_id, diagonal);
    uint32_t ld_step[R], st_step[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
        ld_step[j] = (uint32_t)((flags & 1) ? po[j] : pf[j]) << 4;
        st_step[j] = (uint32_t)((flags & 2) ? po[j] : pf[j]) << 4;
    }
    for (int gb = ctid; gb < G; gb += NC) {
        int bs = lbase, fb = lfb;
        for (int j = 0; j < nrest; ++j)
            if ((gb >> (5 + j)) & 1) {
                const int p = lds_s8(seg + 16 + j);
                bs |= 1 << p;
                fb ^= swz[p];
            }
        const uint32_t ld0 = (uint32_t)((flags & 1) ? bs : bs ^ fb) << 4, st0 = (uint32_t)((flags & 2) ? bs : bs ^ fb) << 4;
        double dr[NA], di[NA];
        int top = 0, any = 0;
        uint32_t off = ld0;
#pragma unroll
        for (int b = 0; b < NA; ++b) {
            if (b) off ^= ld_step[low_bit(b)];
            const int g = b ^ (b >> 1);
            SM<double>::ld(buf + off, dr[g], di[g]);
        }
#pragma unroll
        for (int b = 0; b < NA; ++b) {
            fx::scan(dr[b], top, any);
            fx::scan(di[b], top, any);
        }
        if (diagonal) {
            fx_diagonals(dr, di, gates, g0, g1, origin, cg);
        } else {
            const bool raw = (flags & kSegRaw) != 0;
            const int E = fx::exponent(top);
            FxGroup<NA> v;
#pragma unroll
            for (int b = 0; b < NA; ++b) {
                v.re[b] = raw ? fx::from_bits(dr[b]) : fx::from_double(dr[b], E);
                v.im[b] = raw ? fx::from_bits(di[b]) : fx::from_double(di[b], E);
            }
            for (int gi = g0; gi < g1; ++gi) {
                const FxGate g = fx_gate(gates, gi, origin, cg);
                fx_apply(g.op, g.code, g.m, v, raw);
                gi += g.more;
            }
#pragma unroll
            for (int b = 0; b < NA; ++b) {
                dr[b] = raw ? fx::to_bits(v.re[b]) : fx::to_double(v.re[b], E);
                di[b] = raw ? fx::to_bits(v.im[b]) : fx::to_double(v.im[b], E);
            }
        }
        off = st0;
#pragma unroll
        for (int b = 0; b < NA; ++b) {
            if (b) off ^= st_step[low_bit(b)];
            const int g = b ^ (b >> 1);
            SM<double>::st(buf + off, dr[g], di[g]);
        }
    }
}

}  // namespace
}  // namespace sv
