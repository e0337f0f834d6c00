// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/sv.h"

namespace sv {

// ------------------------------------------------------------------ errors
struct Error {
    sv_status code;
    std::string msg;
};
void set_error(const std::string &msg);
[[noreturn]] void fail(sv_status code, const std::string &msg);
void check_cuda(cudaError_t e, const char *what);

// Device-side error codes written to the handle's error word.
enum : int { DEV_OK = 0, DEV_ERR_TIMEOUT = 1, DEV_ERR_BOUNDS = 2 };

// ------------------------------------------------------------------ plan (host)
struct BlockGate {
    int64_t gi;      // index into the caller's gate list
    int32_t nq;
    int32_t phys[2]; // physical bit of the gate's q[0], q[1] (gate's own order); after
                     // localize_gates: the chunk-local bit, or -1 for a qubit outside the chunk
    int32_t label[2];
    int32_t ext[2] = {-1, -1};  // after localize_gates: state bit of a qubit outside the chunk
};

struct PlanOp {
    int32_t kind;  // 1 = chunk_swap round, 2 = block, 3 = output-reordering round, 4 = gathered block
    std::vector<std::pair<int32_t, int32_t>> pairs;
    std::vector<BlockGate> gates;
    uint64_t mask = 0;  // chunk bits of a gathered block
    int32_t seg_bits = 0;  // tensor-core register-group width of this block (0: the plan's)
};

struct GateKey {
    int32_t nq, q0, q1, flags;
    bool operator==(const GateKey &o) const {
        return nq == o.nq && q0 == o.q0 && q1 == o.q1 && (flags & SV_GATE_SWAP) == (o.flags & SV_GATE_SWAP);
    }
};

struct HostSeg;

}  // namespace sv

struct sv_plan {
    int32_t n = 0, c = 0, reserve = 0, restore = 1, seg_bits = 4, use_tc = 0, pinned = 0;
    int32_t tc_no_renorm = 0, wait_limit_ms = 0, fp64 = 0;  // executor options carried by the plan
    std::vector<sv::PlanOp> ops;
    std::vector<int32_t> final_map;
    std::vector<sv::GateKey> keys;  // structure of the gate list it was made from
    // Register groups of the sections, searched when first executed and kept with the plan (they follow
    // from its structure alone, like the sections): plan_groups.  A plan may serve several threads.
    // (20-qubit ansatz, 69 groups: a repeated evaluation 1.09 ms with a search each time, 0.90 without.)
    mutable std::mutex groups_mu;
    mutable std::map<std::array<int, 4>, std::shared_ptr<const std::vector<sv::HostSeg>>> groups;
};

namespace sv {

// Cost-model steering of the transpiler's QB_CHUNK choice (gathered chunks only): for every
// section the planner lists candidate chunk sets -- candidates[0] is always the paper's rule --
// with the gates each would take and its features, and a chooser picks one.
constexpr int kNumFeatures = 16;
struct SectionCandidate {
    uint64_t chosen = 0;  // qubits of the chunk
    int absorbed = 0;     // gates the section takes
    int ce = 0;           // chunk bits
    int seg_bits = 0;     // register-group width the features assume (0: the plan's)
    float f[kNumFeatures] = {0};
};
struct SectionChooser {
    virtual ~SectionChooser() = default;
    virtual int choose(const std::vector<SectionCandidate> &cands) = 0;
};

sv_plan *plan_blocking(int n, const sv_gate *gates, int64_t n_gates, const sv_options &o,
                       SectionChooser *chooser = nullptr, int dtype = SV_C64);
// The 16 features of a blocking section (kind 2 or 4) as the cost model sees it.
void section_features(const sv_plan &plan, const PlanOp &op, const sv_gate *gates, int dtype, float *out);

// ------------------------------------------------------------------ block programs
constexpr int SEG_BITS = 4;      // default register-group width (amplitudes per group = 2^SEG_BITS)
constexpr int MAX_SEG_BITS = 5;

// Shared-memory swizzle of a chunk: amplitude i lives in slot i ^ F(i), F(i) = XOR of V[k] over
// the set bits k >= SB of i (SB = 4 for complex64, 3 for complex128).  The V are distinct
// non-powers-of-two below 2^SB where possible, so that any SB of the chunk bits outside a
// register group, plus the low bits, enumerate distinct banks.
#define SV_SWZ64_LIST 0, 0, 0, 0, 3, 5, 6, 7, 9, 10, 11, 12, 13, 14, 15, 3, 5, 6, 7, 9, 10, 11, 12, 13
#define SV_SWZ128_LIST 0, 0, 0, 3, 5, 6, 7, 3, 5, 6, 7, 3, 5, 6, 7, 3, 5, 6, 7, 3, 5, 6, 7, 3
constexpr int kSwz64[24] = {SV_SWZ64_LIST};
constexpr int kSwz128[24] = {SV_SWZ128_LIST};

// Gate op-codes inside a segment.  The exchange codes (bit flip, the two CNOT orientations,
// SWAP) also carry their general form in m[] (dense 2x2 for OP_X1, the permutation of OP_PERM2
// for the others) for consumers that do not special-case them.
enum : int32_t {
    OP_DENSE1 = 0, OP_DENSE2 = 1, OP_DIAG1 = 2, OP_DIAG2 = 3, OP_PERM2 = 4,
    OP_CXA = 5,    // exchange local states 1 <-> 3: control = lower bit a, target = b
    OP_CXB = 6,    // exchange 2 <-> 3: control = b, target = a
    OP_SWAP2 = 7,  // exchange 1 <-> 2
    OP_X1 = 8,     // 1-qubit bit flip
    OP_REAL1 = 10, // dense 1-qubit gate with real entries (fixed-point programs only)
    OP_DIAGRUN = 11, // the next `b` gates, all OP_DIAGX, as one 16-entry diagonal per chunk (likewise)
    OP_DIAGX = 9   // diagonal gate with qubits outside the chunk: b = e0 | e1 << 8 (state bits,
                   // 0xFF = none); variant v = bit e0 + 2 bit e1 of the chunk's origin selects
                   // m[4v..4v+3], a diagonal (d0, d1) on register bit a (a phase: d0 = d1, a = 0)
};

// Register group as the kernel reads it.  A thread's group index g enumerates the chunk bits
// outside the group: g bits 0..4 land on lane[0..4], the higher bits on rest[0..nrest).
struct DevSeg {
    int8_t pos[8];    // group bits (ascending); r of them used
    int8_t lane[5];
    int8_t nrest;
    int8_t flags;     // 1: read the natural (unswizzled) layout, 2: write the natural layout, kSegRaw
    int8_t r;
    int8_t rest[16];
    int16_t g0, g1;   // gate range [g0, g1) in the section's gate array
};
static_assert(sizeof(DevSeg) == 36, "DevSeg layout");

constexpr int kSegRaw = 4;   // fixed-point programs: every gate of the group is exact_gate()
constexpr int kSegDiag = 8;  // ... or diagonal_gate(): in FP64, amplitude by amplitude

template <typename T>
struct DevGate {
    int32_t op;     // OP_*
    int32_t a, b;   // local register bits (a < b for 2-qubit ops)
    int32_t code;   // a for 1-qubit ops, a * 8 + b for 2-qubit ops
    T m[32];        // row-major complex matrix in local basis bit a + 2*bit b (diag: the diagonal)
};

struct HostSeg {
    int r = SEG_BITS;
    int32_t pos[8] = {0};
    int32_t lane[5] = {0};
    int32_t rest[16] = {0};
    int nrest = 0;
    int flags = 0;
    std::vector<int32_t> gates;  // indices into the section's gate list
};

// Split a section's gates (physical bits < width) into register groups of at most r bits,
// and choose each group's lane layout for elements of elem_bytes bytes.
// search = false: the greedy groups only (the cost model's cheap feature).
std::vector<HostSeg> segment_block(const std::vector<BlockGate> &gates, int width, int r, int elem_bytes,
                                   bool search = true);
int plan_segment_count(const sv_plan &plan);
using Groups = std::shared_ptr<const std::vector<HostSeg>>;
// The groups kept for a section (null before keep_groups): by plan op, group width and element size, and
// the gates they are of.
enum : int { ALL_GATES = 0, INSIDE_GATES = 1, OUTSIDE_GATES = 2 };  // without / only the ones with qubits outside the chunk
Groups plan_groups(const sv_plan &plan, int op_index, int r, int elem_bytes, int gates = ALL_GATES);
Groups keep_groups(const sv_plan &plan, int op_index, int r, int elem_bytes, std::vector<HostSeg> segs, int gates = ALL_GATES);

template <typename T>
void encode_gate(const sv_gate &g, const BlockGate &bg, const HostSeg &seg, DevGate<T> &out);

// Block fixed-point programs of complex128 sections (fixed64.cuh, block_fx.cuh).
// Whether the dim x dim matrix is unitary to 1e-9, as the fixed-point ranges need.
bool fx_unitary(const double *m, int dim);
// Clocks per amplitude and SM that a gate takes in FP64 register groups, at 2 FP64 operations a clock.
double fp64_clocks(const DevGate<double> &g);
// Square of the ratio of the largest to the smallest non-zero entry of a gate that mixes amplitudes, else 1.
double entry_ratio(const DevGate<double> &g);
// Whether a gate's entries are all real.
bool real_gate(const DevGate<double> &g);
// Local bits of a gate that its matrix mixes (bit 0: a, bit 1: b), see Dense.
int mixed_bits(const DevGate<double> &g);
// Fixed-point factors of `count` complex entries (4 ints each).
void fx_pack(const double *m, int count, int32_t *entries);
// Whether a gate only exchanges amplitudes or multiplies them by 1 or -1.
bool exact_gate(const DevGate<double> &g);
// Tensor-core programs of complex128 sections (block_oz.cuh): address tables (OzSeg) of the register groups, and
// in device memory of their own per group the B operand of its unitary in base-256 digits, two halves of 16
// output reals, each 8 digit blocks side by side (the last zero), K-major FP16.
constexpr int kOzBBytes = 16384;
// Addresses of a register group's rows in the chunk, loading and storing side: byte offsets of the 32
// lanes, of the 16 row blocks (quarter | tile << 2) and of the 16 amplitudes, to be combined by
// exclusive or (both the natural and the swizzled layout are linear).
struct OzSeg {
    uint32_t ld[64], st[64];
    int32_t scale, unused[3];  // s of the group's operand (written by the composer)
};
OzSeg oz_addresses(const HostSeg &seg, int width, bool natural_ld, bool natural_st);
// One group to compose: gates [g0, g1) of the gate area at gates_off of the program, its scale's word at
// scale_off; B at b_off of the operands.
struct OzCompose {
    uint32_t gates_off, b_off, scale_off;
    int32_t g0, g1;
};
void launch_compose_oz(const void *dev_groups, int ngroups, void *dev_prog, void *dev_operands, cudaStream_t st);
// Whether a gate is diagonal.
bool diagonal_gate(const DevGate<double> &g);
// Moves the OP_DIAGX gates of a register group's list as far back as they commute (a diagonal on a
// register bit passes every gate that is diagonal or acts on other bits, a phase every gate), so
// that they meet in few runs.
void gather_outside_diagonals(std::vector<DevGate<double>> &gates, size_t first);
// The gate area of a section's program: header table and payloads.  false (out untouched) when a
// gate is not unitary.  Runs of OP_DIAGX gates within a group (group_starts: each group's first gate)
// are merged where `merge` is set.
bool encode_fx(const std::vector<DevGate<double>> &gates, const std::vector<int> &group_starts, bool merge,
               std::vector<unsigned char> &out);
constexpr int kFxGroups = 2;  // consumer groups of the integer-pipe kernel, each with its own merged diagonals:
// 16 entries and a part of each for its four warps
constexpr int kFxRunBytes = kFxGroups * 5 * 256;

// Gathered chunk: the state is viewed as a tensor of rank <= 5 whose dimension d covers the
// index bits [s[d], s[d+1]); each dimension starts with a run of chunk bits (its box, at most
// 8 bits), the bits above it up to the next dimension are addressed by coordinates.  Chunk bits
// outside the boxes are "loop" bits: one tensor copy per value.  Chunk-local bit order: the
// box bits of dimension 0, 1, ..., then the loop bits.
struct GatherArgs {
    int32_t rank;
    int32_t s[6];          // dimension start bits; s[rank] = n
    int32_t nouter, nloop;
    int32_t box_amps;      // amplitudes per tensor copy (2^(box bits))
    int8_t outer[64];      // chunk-index bit -> state bit
    int8_t loop[16];       // copy-index bit -> state bit
};

struct GatherLayout {
    GatherArgs args{};
    int box_len[5] = {0};
    int local_of[64];      // state bit -> chunk-local bit (-1 outside the chunk)
    int ce = 0;            // chunk bits
};

GatherLayout gather_layout(uint64_t mask, int n, int elem_bytes);

// A section's gates on chunk-local bits: bits < min(c, n) for a contiguous chunk (kind 2), the
// gathered layout's local order for kind 4 (`lay` non-null).  A qubit outside the chunk (only
// diagonal gates, diag_outside) gets phys = -1 and its state bit in ext.
std::vector<BlockGate> localize_gates(const PlanOp &op, int n, int c, const GatherLayout *lay);

// Tensor-core path: per register group, the gates to fuse and where its B operand goes.
struct ComposeSeg {
    int32_t g0, g1;     // gate range in the FP64 gate array
    uint32_t b_off;     // byte offset of the group's B_hi (B_lo follows at + tc_b_bytes(r) / 2) in the program
    uint32_t flag_off;  // where to write an int: 1 if the fused matrix is unitary (kNoFlag: none)
};
constexpr uint32_t kNoFlag = 0xFFFFFFFFu;
constexpr int TC_B_BYTES = 8192;  // B_hi + B_lo of one 4-bit register group (2 x 32 x 32 TF32)
// B_hi + B_lo of an r-bit group: two K x K TF32 matrices, K = 2^(r+1) reals per row.
constexpr int tc_b_bytes(int r) { return 8 << (2 * (r + 1)); }
static_assert(tc_b_bytes(4) == TC_B_BYTES, "B operand size");

// Batched execution: one blocking section of one state.  Chunk-local bit k is state bit k for
// k < low (the contiguous low run of the chunk) and high[k - low] above it; the chunk index
// enumerates the state bits outside the chunk, outer[] ascending.  The section's program is
// npiece consecutive pieces at prog_off, each {nseg, ngate, bytes, 0} + DevSeg[] + DevGate[].
struct BatchOp {
    int32_t state, op, ce, low;
    int64_t nchunks, first;  // chunks of this section; first global work-item index
    uint32_t prog_off, prog_bytes;
    int32_t npiece, tc;  // tc: tensor-core groups (pieces hold B operands instead of gate records)
    int32_t nhigh, nouter;
    int8_t high[24];
    int8_t outer[40];
};
constexpr int kBatchMaxChunkBits = 13;
constexpr int kBatchMaxProgBytes = 24 * 1024;    // program piece of a SIMT batch
constexpr int kBatchMaxProgBytesTc = 32 * 1024;  // ... of a batch with tensor-core sections (per pool)
// Tensor-core batches whose chunks have at most kBatchTc3ChunkBits bits run three pools per CTA
// (one tile buffer each) with program pieces of at most kBatchMaxProgBytesTc3 bytes.
constexpr int kBatchTc3ChunkBits = 12;
constexpr int kBatchMaxProgBytesTc3 = 38 * 1024;
constexpr int kBatchTcGroupBytes = TC_B_BYTES + 16;  // B operand + unitarity flag per group
// wait_ns bounds every device wait; stall_state >= 0 (a failure-path test) keeps that state's first
// section from releasing the later ones.
void launch_batch(const void *dev_ops, int nops, const void *dev_progs, void *const *dev_amps, int *dev_ops_done,
                  int *dev_chunks_done, unsigned long long *dev_next, int64_t total, int from_zero, int use_tc,
                  int *dev_err, cudaStream_t st, uint64_t wait_ns, int stall_state);
// Fuse register groups of r bits in FP64; *all_unitary (1 on entry; may be null) is cleared when
// a fused matrix is not unitary to 1e-10 (max |U^H U - I|).
void launch_compose(const void *dev_segs, int nseg, const void *dev_gates, void *dev_prog, int *all_unitary, int r,
                    cudaStream_t st);

// cost-model network kernels (k_mlp.cu)
int mlp_param_count();
int mlp_grad_blocks(int64_t B);
void launch_mlp_fwd(const float *P, const float *X, int64_t B, float *Y, cudaStream_t st);
void launch_mlp_grad(const float *P, const float *X, const float *T, const int32_t *idx, int64_t start, int64_t B,
                     float *part, double *lpart, cudaStream_t st);
void launch_mlp_reduce(const float *part, int nblk, const double *lpart, double *loss, int mode, float *grad, float *P,
                       float *M, float *V, float lr, float c1, float c2, cudaStream_t st);

// ------------------------------------------------------------------ kernels (launchers)
struct Mat1 { float m[8]; };
struct Mat2 { float m[32]; };

// Returns the bytes that the sweep reads and writes (0: the identity, nothing is launched).
double launch_gate(int dtype, void *state, int n, const sv_gate &g, cudaStream_t st);
void launch_init_basis(int dtype, void *state, int n, uint64_t basis, cudaStream_t st);
// When a chunk is dense enough for one exponent: at most `most` of its amplitudes (zeros too) are more than
// `orders` binary orders below its largest component.  A unit is 2^-54 of that component, and FP64 is as
// inexact only for results that draw on amplitudes near it.  So it depends on what the sweep's gates mix:
// a bit is mixed where every row of some gate has at least 1/16 of its norm on either value of the
// bit.  With kMixedBits of them or more, up to half of the 2^bits amplitudes that every result draws on
// may be small (and at most 1 in 32 of the chunk): a chunk of 2^12 of a state as random circuits leave it has 1 amplitude
// below 8 orders where it is complex, 45 where it is real, so that practically none falls out.  Else
// (phases, small angles) all have to be within kNearOrders.
struct Dense {
    int orders, most;  // orders < 0: every chunk but one of zeros
    unsigned bits;  // chunk bits that dense gates act on
    int trial;      // whether gates may fill a chunk within kNearOrders from one amplitude
};
constexpr int kNearOrders = 4, kFarOrders = 8, kMixedBits = 6;
// Section programs of a plan with SIMT register groups (complex128: tensor-core sweeps where they
// apply), laid out as one device upload (api.cu).
struct SimtPrograms {
    struct Prog {
        size_t off;
        int nseg, gate_bytes, op_index;
        bool fixed, oz, gathered;  // complex128 off FP64: on the integer pipe, or the tensor cores (block_oz.cuh)
        bool redo;                 // ... with an FP64 program for the chunks it leaves
        size_t redo_off;
        int redo_bytes;
        Dense dense;
        int oz_first;      // of its nseg groups to compose
        size_t b_off;      // their operands
        GatherLayout lay;  // gathered chunks
    };
    std::vector<unsigned char> host;
    std::vector<Prog> progs;
    size_t oz_off = 0;  // groups to compose once uploaded (launch_compose_oz)
    int noz = 0;
    size_t b_bytes = 0;  // device memory for their operands
    int seg_bits = 4;
};
void build_simt_programs(const sv_plan *plan, const sv_gate *gates, int dtype, SimtPrograms &out);
// Device memory that launch_section's `list` needs for a state of 2^n amplitudes in chunks of c bits (0: none),
// its first LIST_FIRST ints zeroed.  One list serves one stream at a time.
size_t redo_list_bytes(const SimtPrograms &sp, int n, int c);
// Launch one section of 2^n amplitudes (chunks of c bits) from its program at base + p.off and operands
// + p.b_off; returns the number of kernels.
int launch_section(int dtype, void *state, int n, int c, const unsigned char *base, const unsigned char *operands,
                   const SimtPrograms::Prog &p, int seg_bits, int *list, int *dev_err, cudaStream_t st, uint64_t wait_ns);
// Amplitudes with bit `bit` == value, in index order, to / from a buffer of 2^(n-1) (k_shard.cu).
void launch_shard_half(bool pack, int dtype, void *state, int n, int bit, int value, void *buf, cudaStream_t st);

struct PermPlan;  // defined in k_permute.cu
void launch_permute(int dtype, void *state, int n, const std::vector<std::pair<int32_t, int32_t>> &pairs,
                    cudaStream_t st);

// Bounded device waits: wait_ns (kDefaultWaitNs unless the plan sets wait_limit_ms).
constexpr uint64_t kDefaultWaitNs = 4000000000ull;
// Chunks of a complex128 section that a fixed-point or tensor-core pass leaves to FP64 (block_fx.cuh,
// ChunkRange): the pass appends their numbers to `to` (device memory), and an FP64 pass with `from` set runs
// those alone and empties the list.  to null: the section's gates keep the amplitudes apart, every chunk runs.
struct SweepArgs {
    int *to = nullptr;
    Dense dense;
    int *from = nullptr;
    const void *operands = nullptr;  // B operands of a tensor-core sweep
};
enum : int { LIST_COUNT = 0, LIST_READERS = 1, LIST_FIRST = 2 };  // both 0 in an empty list; then room for every chunk
// SIMT sections: the program is nseg register groups and a gate area of gate_bytes bytes, gate
// records (DevGate) or, `fixed` (complex128), a fixed-point area (encode_fx).
void launch_block(int dtype, void *state, int n, int c, const void *dev_prog, int nseg, int gate_bytes, bool fixed,
                  int *dev_err, int seg_bits, cudaStream_t st, uint64_t wait_ns = kDefaultWaitNs, const SweepArgs &sa = SweepArgs{});
// Blocking section over a gathered chunk (bits in `mask`), fetched and written back with
// tensor copies.
void launch_block_gather(int dtype, void *state, int n, const GatherLayout &lay, const void *dev_prog, int nseg,
                         int gate_bytes, bool fixed, int *dev_err, int seg_bits, cudaStream_t st,
                         uint64_t wait_ns = kDefaultWaitNs, const SweepArgs &sa = SweepArgs{});
// Chunk buffers that a complex128 SIMT section of 2^ce amplitudes gets beside its program (0: it does not fit).
int simt_buffers(int ce, int nseg, size_t gate_bytes);
// Register groups (at most) that one tensor-core sweep of a complex128 chunk of ce bits takes; 0: the
// chunk cannot run there.
int oz_max_segs(int ce);
// Tensor-core blocking section of a complex128 state; `lay` null for a contiguous chunk of c bits.
void launch_block_oz(void *state, int n, int c, const GatherLayout *lay, const void *dev_prog, int nseg, int *dev_err,
                     cudaStream_t st, uint64_t wait_ns, const SweepArgs &sa);
// Tensor-core blocking section (complex64, register groups of seg_bits = 3, 4 or 5 bits, B
// operands in the program, tc_b_bytes(seg_bits) each); `lay` null for a contiguous chunk of c bits.
void launch_block_tc(void *state, int n, int c, const GatherLayout *lay, const void *dev_prog, int nseg, int *dev_err,
                     int seg_bits, cudaStream_t st, uint64_t wait_ns = kDefaultWaitNs);

// readouts
void launch_probs(int dtype, const void *state, int n, double *out, int64_t first, int64_t count,
                  cudaStream_t st);
void launch_partial_norm(int dtype, const void *state, int n, double *partials, int nblocks,
                         cudaStream_t st);
// state <- state * sqrt(n_in / n_out) (complex64) when *flag != 0; partials: n_in's nblocks
// partial sums, then n_out's; d: one float of device scratch.
void launch_renorm(int dtype, void *state, int n, const double *partials, int nblocks, const int *flag, float *d,
                   cudaStream_t st);
// nblocks partial sums of a Pauli word's paired terms, then as many of the magnitudes of their products.
void launch_partial_expval(int dtype, const void *state, int n, uint64_t x, uint64_t z,
                           double *partials, int nblocks, cudaStream_t st);
// (re, im) partial sums of the word's terms in index order, nblocks pairs.
void launch_partial_expval_direct(int dtype, const void *state, int n, uint64_t x, uint64_t z, double *partials,
                                  int nblocks, cudaStream_t st);
// Result words of a readout: a value, the magnitude of what was summed to it, the handle's error word.
struct Readout {
    double value, weight;
    int err;
};
// out->value = sum of the partials, out->weight (weights) that of the nblocks behind them.
void launch_finish(const double *partials, int nblocks, bool weights, const int *err, Readout *out, cudaStream_t st);
// Whether a Pauli word's sum cancels to nothing beside its products (a real state under a word with an odd number of
// Y's): callers then get the residue of the term-by-term sum, as they always have.
inline bool expval_cancels(const Readout &r) { return !(std::fabs(r.value) > 0x1p-40 * r.weight); }
// (sr + i si) i^{popcount(x & z)}
void pauli_phase(uint64_t x, uint64_t z, double sr, double si, double *out);
// Inverse-CDF sampling over ranges of 2^sb amplitudes: sums holds 2^(n-sb) doubles, totals
// sample_totals(n, sb); total->value receives the squared norm.
int64_t sample_totals(int n, int sb);
void launch_sample(int dtype, const void *state, int n, int sb, double *sums, double *totals, uint64_t seed, int64_t shots,
                   uint64_t *out, const int *err, Readout *total, cudaStream_t st);

int num_sms();

}  // namespace sv
struct sv_state;
namespace sv {
// Synchronise the handle's stream and turn its device error word into a status (clearing it).
void check_dev_error(sv_state *h);

}  // namespace sv

// ------------------------------------------------------------------ state handle
struct sv_state {
    int32_t n = 0;
    int32_t dtype = SV_C64;
    void *amp = nullptr;      // device amplitudes
    bool owns_amp = false;
    cudaStream_t stream = nullptr;
    int *dev_err = nullptr;   // device error word, then (16 bytes on) a Readout
    sv::Readout *slot = nullptr;  // pinned result words (api.cu's pool)
    double *scratch = nullptr;  // device scratch for reductions
    size_t scratch_bytes = 0;
    void *prog = nullptr;     // device block programs
    size_t prog_bytes = 0;
    void *prog_host = nullptr;  // pinned staging for programs
    size_t prog_host_bytes = 0;
    cudaEvent_t prog_event = nullptr;
    sv_apply_stats stats{};
    int device = 0;
    bool profiling = false;
    std::vector<cudaEvent_t> ev_pool;                 // reusable timing events
    struct Mark {
        int kind, ev, op;  // launch kind, index of its start event, plan op (-1: per-gate)
    };
    std::vector<Mark> ev_marks;
    bool stats_timed = false;
};
