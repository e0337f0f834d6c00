// Register-group engine of complex128 sections on the tensor cores: exact products of integer
// digits (the splitting scheme of Ozaki, Ogita, Oishi and Rump 2012).
//
// A section's chunk becomes block fixed point with one exponent: X = x 2^-e, |X| < 2^55, int64 in
// place of every double.  A register group is one 2^4 x 2^4 unitary U, M = round(U 2^(54 + s)), s = 0, 1
// or 2 as its largest entry allows, composed by k_compose_fx to 2^-59.  X and M are written in balanced base-256 digits, seven each (digit 0
// the most significant), which FP16 holds exactly; as in the complex64 path a row is the group's 16
// amplitudes as K = 32 reals, a tile is 128 rows, and
//     D_d = sum_{i + j = d} A_i B_j,   d = 0..7,   |D_d| <= 7 * 32 * 2^14 < 2^22,
// so FP32 accumulation is exact.  D_8 and beyond are left out (below 2^-4 units of X in the rms).
// B's blocks j = 0..6 and one of zeros lie side by side along N, so digit i is one MMA of
// N = 16 (8 - i) per K step for 16 output reals (a half row), its D columns shifted by 16 i:
// 14 MMAs per half, 1120 cycles per tile at the FP16 rate.  The thread that drains a row sums
//     V = sum_d D_d 2^{8 (6 - d) - 4} = X U 2^(2 + s)
// in int64 and stores it to the chunk; the largest V of the chunk sets the shift back to 55 bits
// that the next group's staging applies, with rounding.  Only a section's first group reads
// doubles and only its last writes them.
//
// Bound by the latency of the integer work (digits out, sums back), so all 512 consumer threads
// work on one chunk, four to a row, and the MMAs run under them: a tile's digits have two buffers
// (112 columns each), its two halves of D one each (128), the next tile is staged while this
// one's MMAs run, and a half's MMAs for the next tile start as soon as it is read.
//
// Measured against the integer-pipe sections (block_fx.cuh) and the FP64 ones before them, 12-bit
// chunks: n = 27, 8 random layers (44 groups) on a dense state 169 and 417 ms, here 57 to 63; n = 25, quantum volume of
// 10 layers (44 groups) from a basis state 108 ms in FP64, here 20 to 21 (12.8 with the first sections, of few
// amplitudes, here too; they are FP64's).  A group costs about 2.3 clocks per amplitude and
// SM whatever its gates are; a dense one-qubit gate on the integer pipe alone takes 1.4, and the
// conversions of a group there 1.5.
//
// Precision: a unit of X is 2^-54 to 2^-55 of the chunk's largest component; each group rounds once to it,
// and U is within 2^-(55 + s), where FP64 rounds four to eight times per gate.  That holds for the chunk as
// a whole, so chunks run here only where ChunkRange finds them dense; FP64 register groups run the others
// from memory, where they were left.  Relative error of single amplitudes against extended precision, here and in
// FP64, after 8 layers on 13 qubits from a dense state: median 3.2e-16 and 7.4e-16, one in 1000 above 1.2e-14 and
// 4.0e-14, largest 1.1e-13 and 2.5e-13; quantum volume 3.5e-16 and 7.0e-16, 1.0e-14 and 2.5e-14, 3.1e-14 and 6.7e-14.
#pragma once
#include "block_fx.cuh"

namespace sv {
namespace {

constexpr int kOzMaxSegs = 16;  // register groups per sweep (shared memory allows about six)

// Per consumer group, in shared memory.
struct OzShared {
    ChunkRange range;
    int skip;                    // the chunk does not run: no MMAs
    unsigned high[kOzMaxSegs];   // largest magnitude's high word after each group
};

enum : int { OZ_LD = 0, OZ_ST = 256, OZ_SCALE = 512 };  // byte offsets of OzSeg's tables

__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));  // program data: read-only after the first barrier
    return v;
}
__device__ __forceinline__ void lds_i64x2(uint32_t a, long long &x, long long &y) {
    asm volatile("ld.shared.v2.s64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "r"(a));
}
__device__ __forceinline__ void sts_i64x2(uint32_t a, long long x, long long y) {
    asm volatile("st.shared.v2.s64 [%0], {%1, %2};" ::"r"(a), "l"(x), "l"(y) : "memory");
}

constexpr unsigned long long kOzBias = 0x0080808080808080ull;  // makes all seven digits non-negative

// X + bias of a double whose chunk has exponent E: X = x * 2^(1077 - E).
__device__ __forceinline__ unsigned long long oz_from_double(double x, int E) {
    const int hi = __double2hiint(x);
    const int d = min(E - ((hi >> 20) & 0x7FF), 63);
    const unsigned long long m =
        ((unsigned long long)(unsigned)((hi & 0xFFFFF) | 0x100000) << 32) | (unsigned)__double2loint(x);
    const unsigned long long v = ((m << 2) + ((1ull << d) >> 1)) >> d;  // magnitude, rounded
    const unsigned long long s = (unsigned long long)(long long)(hi >> 31);
    return (v ^ s) - s + kOzBias;
}

// v * 2^e as a double.
__device__ __forceinline__ double oz_to_double(long long v, int e) {
    const long long s = v >> 63;
    unsigned long long a = ((unsigned long long)v ^ (unsigned long long)s) - (unsigned long long)s;
    const int ah = (int)(a >> 32), al = (int)a;
    const int lz = ah ? __clz(ah) : 32 + __clz(al);
    a <<= lz & 63;
    unsigned long long b = (a >> 11) + ((a >> 10) & 1);
    b += (unsigned long long)(unsigned)(e + 1085 - lz) << 52;  // exponent 63 - lz + e + 1023, less the hidden bit
    b |= (unsigned long long)s & 0x8000000000000000ull;
    return __longlong_as_double((ah | al) ? (long long)b : 0);
}

// Digit b (byte, 0 the least significant) of two biased components as a pair of FP16 integers
// in [-128, 127]: 1024 + byte by its bit pattern, less 1152.
__device__ __forceinline__ uint32_t oz_half2(uint32_t t) {
    uint32_t r;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(t), "r"(0x64806480u));
    return r;
}
__device__ __forceinline__ void oz_digits(unsigned long long re, unsigned long long im, uint32_t (&a)[7]) {
    const uint32_t rl = (uint32_t)re, rh = (uint32_t)(re >> 32), il = (uint32_t)im, ih = (uint32_t)(im >> 32);
    const uint32_t q0 = __byte_perm(rl, il, 0x5140), q1 = __byte_perm(rl, il, 0x7362);  // (re, im) bytes 0, 1; 2, 3
    const uint32_t q2 = __byte_perm(rh, ih, 0x5140), q3 = __byte_perm(rh, ih, 0x7362);
    constexpr uint32_t k64 = 0x64646464u;
    a[6] = oz_half2(__byte_perm(q0, k64, 0x4140));
    a[5] = oz_half2(__byte_perm(q0, k64, 0x4342));
    a[4] = oz_half2(__byte_perm(q1, k64, 0x4140));
    a[3] = oz_half2(__byte_perm(q1, k64, 0x4342));
    a[2] = oz_half2(__byte_perm(q2, k64, 0x4140));
    a[1] = oz_half2(__byte_perm(q2, k64, 0x4342));
    a[0] = oz_half2(__byte_perm(q3, k64, 0x4140));
}

// Two FP32 values (an amplitude's components, adjacent accumulator columns) per instruction.
__device__ __forceinline__ void add2(uint32_t x, uint32_t y, float c, uint32_t &ox, uint32_t &oy) {
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %4};\n\t"
        "add.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=r"(ox), "=r"(oy)
        : "r"(x), "r"(y), "r"(__float_as_uint(c)));
}
__device__ __forceinline__ void fma2(uint32_t x, uint32_t y, float m, uint32_t cx, uint32_t cy, uint32_t &ox, uint32_t &oy) {
    asm("{\n\t.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %4};\n\tmov.b64 c, {%5, %6};\n\t"
        "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=r"(ox), "=r"(oy)
        : "r"(x), "r"(y), "r"(__float_as_uint(m)), "r"(cx), "r"(cy));
}

// V = sum_d D_d 2^{8 (6 - d) - 4} of an amplitude's two components, D_d exact FP32 integers below
// 2^22 in magnitude.  Adding 1.5 * 2^23 leaves u = D + 2^22 in the low 23 bits of b; for a pair of
// diagonals P = (b_k << 8) + b_{k+1} = 256 D_k + D_{k+1} + kOff without wrapping (the shift drops
// the exponent bits), so all offsets are one constant of the 64-bit sum.  D_6 + D_7 / 256 is summed in
// FP32 (to 2^-3) and rounded to V's unit.
__device__ __forceinline__ void oz_sum(const uint32_t (&dr)[8], const uint32_t (&di)[8], long long &vr, long long &vi) {
    constexpr float kMagic = 12582912.0f;
    constexpr uint32_t kMagicBits = 0x4B400000u;
    constexpr unsigned long long kOff = 0x4B000000ull + 257ull * (1ull << 22);
    constexpr unsigned long long kConst =
        0ull - (kOff * ((1ull << 36) + (1ull << 20) + (1ull << 4)) + (unsigned long long)kMagicBits);
    uint32_t br[6], bi[6], fr, fi, lr, li;
#pragma unroll
    for (int k = 0; k < 6; ++k) add2(dr[k], di[k], kMagic, br[k], bi[k]);
    fma2(dr[7], di[7], 1.0f / 256, dr[6], di[6], fr, fi);
    fma2(fr, fi, 0.0625f, kMagicBits, kMagicBits, lr, li);
    auto total = [&](const uint32_t (&b)[6], uint32_t low) {
        unsigned long long t = kConst + low;
        t += (unsigned long long)((b[4] << 8) + b[5]) * 16u;
        t += (unsigned long long)((b[2] << 8) + b[3]) * (1u << 20);
        const uint32_t p0 = (b[0] << 8) + b[1];
        return (long long)(t + ((unsigned long long)(p0 << 4) << 32));
    };
    vr = total(br, lr);
    vi = total(bi, li);
}

// MMA issue of half rows `half`, one warp: an MMA holds its issuing thread for about 88 cycles (14
// of them in a row 1210), so the halves have a warp each and the threads that stage and drain
// have none of it (with one of those issuing, a section of n = 24 took 645 us instead of 545).
__device__ __forceinline__ void oz_issue(int half, uint32_t bops, int nseg, int c, int64_t count, uint32_t tcol,
                                         uint64_t *mbar, volatile int *abort_flag, int *err, const uint64_t *wait_ns,
                                         const OzShared *sh) {
    constexpr int kDCols = 128, kACols = 112;
    const int T = 1 << (c - 4 - 7);
    const uint32_t d = tcol + (uint32_t)(half * kDCols);
    uint32_t phase = 0;
    for (int64_t it = 0; it < count; ++it) {
        for (int k = 0; k < nseg * T; ++k) {
            const bool ok = ptx::mbar_wait(&mbar[2 + half], phase, *(volatile const uint64_t *)wait_ns) && !*abort_flag;
            phase ^= 1;
            if (__any_sync(0xFFFFFFFFu, !ok)) {
                if ((threadIdx.x & 31) == 0) {
                    atomicCAS(err, DEV_OK, DEV_ERR_TIMEOUT);
                    *abort_flag = 1;
                }
                return;
            }
            ptx::tc_fence_after();
            const bool skip = *(volatile const int *)&sh->skip != 0;  // only with a chunk's first tile
            __syncwarp();  // every lane has read it before the commit below lets the consumers clear it for their next chunk
            if ((threadIdx.x & 31) == 0) {
                const uint32_t a = tcol + 2 * kDCols + (uint32_t)((k % T & 1) * kACols);
                const uint64_t bd = ptx::smem_desc_kmajor(bops + (uint32_t)(k / T) * kOzBBytes, 128, 512) +
                                    (uint64_t)(half * (kOzBBytes / 2 / 16));
                if (!skip) {
#pragma unroll
                    for (int i = 0; i < 7; ++i)
#pragma unroll
                        for (int s = 0; s < 2; ++s)
                            ptx::mma_f16_ts(d + 16 * i, a + 56 * s + 8 * i, bd + 16 * s, ptx::idesc_f16(128, 16 * (8 - i)),
                                            i > 0 || s > 0);
                }
                ptx::mma_commit(&mbar[half]);
            }
            __syncwarp();
            if (skip) break;
        }
    }
}

// All register groups of a section on one chunk; kind (uniform): CHUNK_DENSE where the results stand, else
// how the chunk was left.  Returns false (uniformly) when a wait expired.
template <int NC>
__device__ __forceinline__ bool run_chunk_oz(uint32_t buf, uint32_t tabs, int nseg, int ctid, int c, const Dense &dense,
                                             uint32_t tcol, int bar_id, uint64_t *mbar, uint32_t (&phase)[2],
                                             volatile int *abort_flag, const uint64_t *wait_ns, OzShared *sh, int &kind) {
    static_assert(NC == 512, "four threads per row of a 128-row tile");
    constexpr int kDCols = 128, kACols = 112;  // D half 0, D half 1, digits 0, digits 1
    // exponent search (sh was cleared before the barrier that opened this chunk)
    int top;
    kind = chunk_range<NC>(buf, c, ctid, bar_id, &sh->range, dense, top);
    auto ready = [&](int half) {  // this warp's part of a tile's half: digits staged, last sums read
        ptx::tc_fence_before();
        __syncwarp();
        if ((ctid & 31) == 0) ptx::mbar_arrive(&mbar[2 + half]);
    };
    bool failed = false;
    auto wait_mma = [&](int half) {
        if (!ptx::mbar_wait(&mbar[half], phase[half], *(volatile const uint64_t *)wait_ns)) {
            failed = true;
            *abort_flag = 1;
        }
        phase[half] ^= 1;
        ptx::tc_fence_after();
    };
    if (kind >= CHUNK_ZERO) {
        if (ctid == 0) sh->skip = 1;
        ptx::named_bar_sync(bar_id, NC);
        for (int half = 0; half < 2; ++half) {
            ready(half);
            wait_mma(half);
        }
        return !ptx::named_bar_or(bar_id, NC, failed);
    }
    // |X| <= 0.985 * 2^55: seven balanced digits reach 0.996 * 2^55
    const int E = (top >> 20) + ((top & 0xFFFFF) >= 0xF8000 ? 1 : 0);
    int e = E - 1077, scale = 0;  // value = X 2^e
    const int lane = ctid & 31, quarter = (threadIdx.x >> 5) & 3, sub = ctid >> 7;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    const uint32_t acol = tcol + 2 * kDCols;  // digits: [half of K][digit][8 columns]
    const int T = 1 << (c - 4 - 7);
    for (int si = 0; si < nseg; ++si) {
        const uint32_t tab = tabs + (uint32_t)(si * sizeof(OzSeg));
        const bool first = si == 0, last = si == nseg - 1;
        // byte offsets in the chunk are exclusive ors of a lane's, a row block's and an amplitude's
        const uint32_t ld_lane = lds_u32(tab + OZ_LD + 4 * lane) ^ lds_u32(tab + OZ_LD + 4 * (48 + 4 * sub));
        const uint32_t ld1 = lds_u32(tab + OZ_LD + 4 * 49), ld2 = lds_u32(tab + OZ_LD + 4 * 50);
        const uint32_t st_lane = lds_u32(tab + OZ_ST + 4 * lane) ^ lds_u32(tab + OZ_ST + 4 * (48 + 2 * sub));
        const uint32_t st1 = lds_u32(tab + OZ_ST + 4 * 49), st8 = lds_u32(tab + OZ_ST + 4 * 56);
        // shift of the last group's sums (scale: its s) back to 0.992 * 2^55, with its rounding and the digits' bias
        int shift = 0;
        unsigned long long add = kOzBias;
        if (!first) {
            const unsigned high = *(volatile unsigned *)&sh->high[si - 1];  // below 2^30: sums are below 2^61.5
            shift = max(0, 9 - __clz((int)high));
            shift += (high >> shift) >= 0x7EF000u;
            add = (kOzBias << shift) + ((1ull << shift) >> 1);
            e += shift - 2 - scale;
        }
        scale = (int)lds_u32(tab + OZ_SCALE);
        int vmax = 0, vmin = 0;  // extreme high words of the group's sums
        // this thread's 4 amplitudes of tile t (group bits 3, 2 = sub) to digit buffer t & 1
        auto stage = [&](int t) {
            const uint32_t at0 = ld_lane ^ lds_u32(tab + OZ_LD + 4 * (32 + quarter + 4 * t));
            uint32_t dig[7][4];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const uint32_t off = at0 ^ ((g & 1) ? ld1 : 0u) ^ ((g & 2) ? ld2 : 0u);
                unsigned long long re, im;
                if (first) {
                    double x, y;
                    SM<double>::ld(buf + off, x, y);
                    re = oz_from_double(x, E);
                    im = oz_from_double(y, E);
                } else {
                    long long x, y;
                    lds_i64x2(buf + off, x, y);
                    re = ((unsigned long long)x + add) >> shift;
                    im = ((unsigned long long)y + add) >> shift;
                }
                uint32_t a[7];
                oz_digits(re, im, a);
#pragma unroll
                for (int i = 0; i < 7; ++i) dig[i][g] = a[i];
            }
            const uint32_t to = acol + (uint32_t)((t & 1) * kACols) + lane_off + 56 * (sub >> 1) + 4 * (sub & 1);
#pragma unroll
            for (int i = 0; i < 7; ++i) ptx::tmem_st4(to + 8 * i, dig[i]);
            ptx::tmem_wait_st();
        };
        // wait for half `half` of tile t and write its amplitudes (group bit 3 = half, bits 2, 1 = sub)
        auto drain = [&](int t, int half) {
            const uint32_t at0 = st_lane ^ lds_u32(tab + OZ_ST + 4 * (32 + quarter + 4 * t)) ^ (half ? st8 : 0u);
            wait_mma(half);
            uint32_t d[8][4];
#pragma unroll
            for (int k = 0; k < 8; ++k) ptx::tmem_ld4(tcol + (uint32_t)(half * kDCols) + lane_off + 16 * k + 4 * sub, d[k]);
            ptx::tmem_wait_ld();
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t dr[8], di[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) { dr[k] = d[k][2 * q]; di[k] = d[k][2 * q + 1]; }
                long long vr, vi;
                oz_sum(dr, di, vr, vi);
                const uint32_t at = buf + (q ? at0 ^ st1 : at0);
                if (last) {
                    SM<double>::st(at, oz_to_double(vr, e - 2 - scale), oz_to_double(vi, e - 2 - scale));
                } else {
                    vmax = __vimax3_s32(vmax, (int)(vr >> 32), (int)(vi >> 32));
                    vmin = __vimin3_s32(vmin, (int)(vr >> 32), (int)(vi >> 32));
                    sts_i64x2(at, vr, vi);
                }
            }
        };
        stage(0);
        ready(0);
        ready(1);
        for (int t = 0; t < T; ++t) {
            if (t + 1 < T) stage(t + 1);  // its buffer's MMAs (tile t - 1) were waited for
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                drain(t, half);
                if (t + 1 < T) ready(half);
            }
        }
        if (!last) {
            const unsigned high = __reduce_max_sync(0xFFFFFFFFu, (unsigned)max(vmax, ~vmin));
            if (lane == 0) atomicMax(&sh->high[si], high);
        }
        if (ptx::named_bar_or(bar_id, NC, failed)) return false;  // the group's sums are in the chunk
    }
    if (kind == CHUNK_TRIAL) kind = chunk_filled<NC>(buf, c, ctid, bar_id, &sh->range, top, dense.bits) ? CHUNK_DENSE : CHUNK_OTHER;
    return true;
}

}  // namespace
}  // namespace sv
