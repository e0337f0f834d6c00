// Host side of the block fixed-point path (fixed64.cuh): which gates it takes and their payloads.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "sv_internal.h"

namespace sv {
namespace {

// Gate entry as two signed 32-bit factors: m * 2^61 = h * 2^32 + l, |l| < 2^31.
void split(double m, int32_t &h, int32_t &l) {
    int64_t M = std::llrint(m * 0x1p61);
    if ((int32_t)(uint32_t)(uint64_t)M == INT32_MIN) ++M;  // keep -l representable
    l = (int32_t)(uint32_t)(uint64_t)M;
    h = (int32_t)((M - l) / (int64_t(1) << 32));
}

}  // namespace

bool fx_unitary(const double *m, int dim) {
    for (int i = 0; i < dim; ++i)
        for (int j = 0; j < dim; ++j) {
            double re = i == j ? -1.0 : 0.0, im = 0.0;
            for (int r = 0; r < dim; ++r) {
                const double *a = m + 2 * (r * dim + i), *b = m + 2 * (r * dim + j);
                re += a[0] * b[0] + a[1] * b[1];
                im += a[0] * b[1] - a[1] * b[0];
            }
            if (!(std::fabs(re) + std::fabs(im) <= 1e-9)) return false;  // NaN entries too
        }
    return true;
}

void fx_pack(const double *m, int count, int32_t *entries) {
    for (int k = 0; k < 2 * count; ++k) split(m[k], entries[2 * k], entries[2 * k + 1]);
}

bool exact_gate(const DevGate<double> &g) {
    int entries = 0;
    switch (g.op) {
        case OP_X1: case OP_CXA: case OP_CXB: case OP_SWAP2: case OP_PERM2: return true;
        case OP_DIAG1: entries = 2; break;
        case OP_DIAG2: entries = 4; break;
        case OP_DIAGX: entries = ((g.b >> 8) & 0xFF) == 0xFF ? 4 : 8; break;
        default: return false;
    }
    for (int l = 0; l < entries; ++l)
        if (std::fabs(g.m[2 * l]) != 1.0 || g.m[2 * l + 1] != 0.0) return false;
    return true;
}

bool diagonal_gate(const DevGate<double> &g) { return g.op == OP_DIAG1 || g.op == OP_DIAG2 || g.op == OP_DIAGX; }

double fp64_clocks(const DevGate<double> &g) {
    int entries = 0;
    switch (g.op) {
        case OP_DENSE1: return 4.0;  // 8 multiply-adds an amplitude
        case OP_DENSE2: return 8.0;
        case OP_DIAG1: entries = 2; break;
        case OP_DIAG2: entries = 4; break;
        case OP_DIAGX: entries = ((g.b >> 8) & 0xFF) == 0xFF ? 4 : 8; break;
        default: return 0.0;
    }
    int used = 0;  // entries of exactly 1 are skipped, the others take 4 multiply-adds
    for (int l = 0; l < entries; ++l) used += g.m[2 * l] != 1.0 || g.m[2 * l + 1] != 0.0;
    return 2.0 * used / entries;
}

double entry_ratio(const DevGate<double> &g) {
    const int entries = g.op == OP_DENSE1 ? 4 : g.op == OP_DENSE2 ? 16 : 0;
    double least = 4.0, most = 0.0;
    for (int l = 0; l < entries; ++l) {
        const double a = g.m[2 * l] * g.m[2 * l] + g.m[2 * l + 1] * g.m[2 * l + 1];
        if (a > 0.0) least = std::min(least, a);
        most = std::max(most, a);
    }
    return entries ? most / least : 1.0;
}

bool real_gate(const DevGate<double> &g) {
    const int entries = g.op == OP_DENSE1 ? 4 : g.op == OP_DENSE2 ? 16 : g.op == OP_DIAG1 ? 2 : g.op == OP_DIAG2 ? 4 : g.op == OP_DIAGX ? 8 : 0;
    for (int l = 0; l < entries; ++l)
        if (g.m[2 * l + 1] != 0.0) return false;
    return true;
}

int mixed_bits(const DevGate<double> &g) {
    const int nb = g.op == OP_DENSE1 ? 1 : g.op == OP_DENSE2 ? 2 : 0, d = 1 << nb;
    int mixed = 0;
    for (int b = 0; b < nb; ++b) {
        bool all = true;
        for (int r = 0; r < d; ++r) {
            double part[2] = {0, 0};  // squared moduli on columns with either value of the bit
            for (int c = 0; c < d; ++c) {
                const double *e = g.m + 2 * (r * d + c);
                part[(c >> b) & 1] += e[0] * e[0] + e[1] * e[1];
            }
            all = all && part[0] >= 1.0 / 256 && part[1] >= 1.0 / 256;
        }
        if (all) mixed |= 1 << b;
    }
    return mixed;
}

void gather_outside_diagonals(std::vector<DevGate<double>> &gates, size_t first) {
    std::vector<DevGate<double>> out, pending;
    for (size_t i = first; i < gates.size(); ++i) {
        const DevGate<double> &g = gates[i];
        if (g.op == OP_DIAGX) {
            pending.push_back(g);
            continue;
        }
        if (g.op != OP_DIAG1 && g.op != OP_DIAG2) {
            const bool one = g.op == OP_DENSE1 || g.op == OP_X1;
            std::vector<DevGate<double>> keep;
            for (const DevGate<double> &d : pending) {
                bool phase = true;  // equal entries in every variant
                for (int v = 0; v < 4; ++v) phase = phase && d.m[4 * v] == d.m[4 * v + 2] && d.m[4 * v + 1] == d.m[4 * v + 3];
                if (!phase && (d.a == g.a || (!one && d.a == g.b))) out.push_back(d);
                else keep.push_back(d);
            }
            pending.swap(keep);
        }
        out.push_back(g);
    }
    out.insert(out.end(), pending.begin(), pending.end());
    std::copy(out.begin(), out.end(), gates.begin() + (ptrdiff_t)first);
}

bool encode_fx(const std::vector<DevGate<double>> &gates, const std::vector<int> &group_starts, bool merge,
               std::vector<unsigned char> &out) {
    std::vector<unsigned char> body;
    std::vector<int32_t> head;
    const size_t table = gates.size() * 16;
    auto put = [&](const void *p, size_t bytes) {
        const unsigned char *b = static_cast<const unsigned char *>(p);
        body.insert(body.end(), b, b + bytes);
    };
    auto put_entries = [&](const double *m, int count) {
        int32_t e[64];
        fx_pack(m, count, e);
        put(e, (size_t)count * 16);
    };
    auto put_diag = [&](const double *d, int count) {
        for (int l = 0; l < count; ++l)
            if (!(std::fabs(d[2 * l] * d[2 * l] + d[2 * l + 1] * d[2 * l + 1] - 1.0) <= 1e-9)) return false;
        put_entries(d, count);
        return true;
    };
    for (const DevGate<double> &g : gates) {
        int32_t op = g.op;
        const size_t off = table + body.size();
        switch (g.op) {
            case OP_DENSE1:
                if (!fx_unitary(g.m, 2)) return false;
                if (g.m[1] == 0.0 && g.m[3] == 0.0 && g.m[5] == 0.0 && g.m[7] == 0.0) {
                    op = OP_REAL1;
                    const double re[4] = {g.m[0], g.m[2], g.m[4], g.m[6]};
                    put_entries(re, 2);
                } else {
                    put_entries(g.m, 4);
                }
                break;
            case OP_DENSE2:
                if (!fx_unitary(g.m, 4)) return false;
                put_entries(g.m, 16);
                break;
            case OP_DIAG1:
                if (!put_diag(g.m, 2)) return false;
                break;
            case OP_DIAG2:
                if (!put_diag(g.m, 4)) return false;
                break;
            case OP_DIAGX: {
                // variants that the gate has: 2 for one outside qubit, 4 for two
                const int nv = ((g.b >> 8) & 0xFF) == 0xFF ? 2 : 4;
                if (!put_diag(g.m, 2 * nv)) return false;
                break;
            }
            case OP_PERM2: {
                int32_t p[4];
                for (int r = 0; r < 4; ++r) p[r] = (int32_t)g.m[r];
                put(p, sizeof(p));
                break;
            }
            default: break;  // register exchanges: no payload
        }
        head.insert(head.end(), {op, (int32_t)off, g.b, g.code});
    }
    // merged runs: {count, 0, 0, 0}, {payload offset, outside bits, code, 0} per gate, then the
    // consumer groups' tables; the run's first header points here
    for (size_t i = 0; merge && i < gates.size();) {
        size_t j = i;
        while (j < gates.size() && gates[j].op == OP_DIAGX &&
               (j == i || std::find(group_starts.begin(), group_starts.end(), (int)j) == group_starts.end()))
            ++j;
        // runs of signs alone stay apart: groups that only exchange and flip signs work on doubles' words
        if (j - i >= 2 && !std::all_of(gates.begin() + (ptrdiff_t)i, gates.begin() + (ptrdiff_t)j, exact_gate)) {
            const size_t off = table + body.size();
            const int32_t count[4] = {(int32_t)(j - i), 0, 0, 0};
            put(count, sizeof(count));
            for (size_t k = i; k < j; ++k) {
                const int32_t row[4] = {head[4 * k + 1], head[4 * k + 2], head[4 * k + 3], 0};
                put(row, sizeof(row));
            }
            body.resize(body.size() + (size_t)kFxRunBytes, 0);
            head[4 * i] = OP_DIAGRUN;
            head[4 * i + 1] = (int32_t)off;
            head[4 * i + 2] = (int32_t)(j - i);
        }
        i = std::max(j, i + 1);
    }
    const unsigned char *h = reinterpret_cast<const unsigned char *>(head.data());
    out.assign(h, h + table);
    out.insert(out.end(), body.begin(), body.end());
    return true;
}

OzSeg oz_addresses(const HostSeg &seg, int width, bool natural_ld, bool natural_st) {
    OzSeg out{};
    auto slot = [&](int index, bool natural) {
        int s = index;
        for (int k = 3; !natural && k < width; ++k)
            if ((index >> k) & 1) s ^= kSwz128[k];
        return (uint32_t)s * 16u;
    };
    for (int side = 0; side < 2; ++side) {
        uint32_t *t = side ? out.st : out.ld;
        const bool natural = side ? natural_st : natural_ld;
        // both layouts are linear: an entry is the exclusive or of its bits'
        auto fill = [&](int at, int count, const int32_t *bits) {
            t[at] = 0;
            for (int k = 0; (1 << k) < count; ++k) {
                const uint32_t step = slot(1 << bits[k], natural);
                for (int v = 1 << k; v < std::min(count, 2 << k); ++v) t[at + v] = t[at + v - (1 << k)] ^ step;
            }
        };
        fill(0, 32, seg.lane);
        fill(32, std::min(16, 1 << seg.nrest), seg.rest);
        fill(48, 16, seg.pos);
    }
    return out;
}

}  // namespace sv
