// Gate fusion inside a register group of complex64 SIMT sections.
//
// A gate costs a thread its products and, whatever it does, about 90 integer instructions for its 16
// amplitudes (reading the record, branching to its bits, moving results back), nearly as many as the
// products of a dense one-qubit gate.  So gates whose fused matrix costs no more than they do apart
// become one record: a one-qubit gate joins the last dense gate on its bit, a two-qubit gate takes up
// the one-qubit gates waiting on its bits if they are dense on both or it is dense itself, and
// two-qubit gates on the same pair, one of them dense, are multiplied.  So a record mixes only
// amplitudes that the separate gates mix (a non-finite one spreads as far as before).  Matrices are
// multiplied in FP64 and rounded to FP32 once.  n = 27, 10 random layers in sections of 13 bits: 34.4 ->
// 28.9 ms.
#include <cstring>
#include <vector>

#include "sv_internal.h"

namespace sv {
namespace {

using Gate = DevGate<double>;

// c = a b for d x d row-major interleaved complex matrices.
void multiply(int d, const double *a, const double *b, double *c) {
    for (int r = 0; r < d; ++r)
        for (int k = 0; k < d; ++k) {
            double re = 0, im = 0;
            for (int j = 0; j < d; ++j) {
                const double *x = a + 2 * (r * d + j), *y = b + 2 * (j * d + k);
                re += x[0] * y[0] - x[1] * y[1];
                im += x[0] * y[1] + x[1] * y[0];
            }
            c[2 * (r * d + k)] = re;
            c[2 * (r * d + k) + 1] = im;
        }
}

bool one_bit(const Gate &g) { return g.op == OP_DENSE1 || g.op == OP_DIAG1 || g.op == OP_X1; }

// The gate's matrix, dense: 2 x 2 or 4 x 4 on (a, b).
void dense(const Gate &g, double *m) {
    std::memset(m, 0, (one_bit(g) ? 8 : 32) * sizeof(double));
    switch (g.op) {
        case OP_DENSE1: case OP_X1: std::memcpy(m, g.m, 8 * sizeof(double)); break;
        case OP_DIAG1:
            m[0] = g.m[0]; m[1] = g.m[1]; m[6] = g.m[2]; m[7] = g.m[3];
            break;
        case OP_DENSE2: std::memcpy(m, g.m, 32 * sizeof(double)); break;
        case OP_DIAG2:
            for (int r = 0; r < 4; ++r) { m[10 * r] = g.m[2 * r]; m[10 * r + 1] = g.m[2 * r + 1]; }
            break;
        default:  // an exchange: row r takes column m[r]
            for (int r = 0; r < 4; ++r) m[2 * (4 * r + (int)g.m[r])] = 1.0;
    }
}

// u on bit `high` (0: a, 1: b) of a two-qubit gate's local basis, as a 4 x 4 matrix.
void expand(const double *u, int high, double *m) {
    std::memset(m, 0, 32 * sizeof(double));
    for (int r = 0; r < 4; ++r)
        for (int c = 0; c < 4; ++c) {
            const int rb = high ? r >> 1 : r & 1, cb = high ? c >> 1 : c & 1;
            if ((high ? (r & 1) == (c & 1) : r >> 1 == c >> 1)) {
                m[2 * (4 * r + c)] = u[2 * (2 * rb + cb)];
                m[2 * (4 * r + c) + 1] = u[2 * (2 * rb + cb) + 1];
            }
        }
}

void make_dense(Gate &g, const double *m) {
    const bool one = one_bit(g);
    g.op = one ? OP_DENSE1 : OP_DENSE2;
    std::memcpy(g.m, m, (one ? 8 : 32) * sizeof(double));
}

}  // namespace

void fuse_gates(std::vector<DevGate<double>> &gates, size_t first) {
    std::vector<Gate> out;
    int last[MAX_SEG_BITS];     // the last record on each bit, or -1
    Gate wait[MAX_SEG_BITS];    // one-qubit gate waiting on each bit
    bool waiting[MAX_SEG_BITS];
    for (int b = 0; b < MAX_SEG_BITS; ++b) { last[b] = -1; waiting[b] = false; }
    double x[32], y[32], z[32];
    auto emit = [&](const Gate &g) {
        out.push_back(g);
        last[g.a] = (int)out.size() - 1;
        if (!one_bit(g) && g.op != OP_DIAGX) last[g.b] = last[g.a];
    };
    auto flush = [&](int b) {
        if (waiting[b]) emit(wait[b]);
        waiting[b] = false;
    };
    // g <- u on bit `bit` after g, for a dense two-qubit record
    auto join = [&](Gate &g, const Gate &u, int bit) {
        dense(u, x);
        expand(x, bit == g.b, y);
        dense(g, x);
        multiply(4, y, x, z);
        make_dense(g, z);
    };
    for (size_t i = first; i < gates.size(); ++i) {
        const Gate &g = gates[i];
        if (one_bit(g)) {
            if (waiting[g.a] && wait[g.a].op == OP_DIAG1 && g.op == OP_DIAG1) {
                for (int l = 0; l < 4; l += 2) {
                    const double re = wait[g.a].m[l], im = wait[g.a].m[l + 1];
                    wait[g.a].m[l] = g.m[l] * re - g.m[l + 1] * im;
                    wait[g.a].m[l + 1] = g.m[l] * im + g.m[l + 1] * re;
                }
            } else if (waiting[g.a]) {
                dense(g, x);
                dense(wait[g.a], y);
                multiply(2, x, y, z);
                make_dense(wait[g.a], z);
            } else if (last[g.a] >= 0 && out[(size_t)last[g.a]].op == OP_DENSE2) {
                join(out[(size_t)last[g.a]], g, g.a);
            } else {
                wait[g.a] = g;
                waiting[g.a] = true;
            }
            continue;
        }
        if (g.op == OP_DIAGX) {
            flush(g.a);
            emit(g);
            continue;
        }
        // the same pair's last record, with nothing waiting in between
        if (!waiting[g.a] && !waiting[g.b] && last[g.a] >= 0 && last[g.a] == last[g.b] &&
            (out[(size_t)last[g.a]].op == OP_DENSE2 || g.op == OP_DENSE2)) {
            Gate &p = out[(size_t)last[g.a]];
            dense(g, x);
            dense(p, y);
            multiply(4, x, y, z);
            make_dense(p, z);
            continue;
        }
        const bool both = waiting[g.a] && waiting[g.b] && wait[g.a].op == OP_DENSE1 && wait[g.b].op == OP_DENSE1;
        Gate f = g;
        if (both || (g.op == OP_DENSE2 && (waiting[g.a] || waiting[g.b]))) {
            dense(g, x);
            for (int b : {g.a, g.b})
                if (waiting[b]) {
                    double u[8];
                    dense(wait[b], u);
                    expand(u, b == g.b, y);
                    multiply(4, x, y, z);
                    std::memcpy(x, z, sizeof(x));
                    waiting[b] = false;
                }
            make_dense(f, x);
        } else {
            flush(g.a);
            flush(g.b);
        }
        emit(f);
    }
    for (int b = 0; b < MAX_SEG_BITS; ++b) flush(b);
    for (Gate &g : out) g.code = one_bit(g) || g.op == OP_DIAGX ? g.a : g.a * 8 + g.b;
    gates.resize(first);
    gates.insert(gates.end(), out.begin(), out.end());
}

DevGate<float> narrow(const DevGate<double> &g) {
    DevGate<float> f;
    f.op = g.op;
    f.a = g.a;
    f.b = g.b;
    f.code = g.code;
    for (int k = 0; k < 32; ++k) f.m[k] = (float)g.m[k];
    return f;
}

}  // namespace sv
