// Pauli expectation value that allocates no memory (sv_expval_pauli_noalloc).
//
// Some callers cannot allocate device memory at the moment they need a readout: code running
// under a memory pool or budget they do not own, real-time loops where cudaMalloc/cudaFree
// would synchronise the device, or hosts that hand this library a pre-sized arena and forbid
// allocations afterwards.  This entry point computes the same quantity as sv_expval_pauli
// but keeps its partial sums in a fixed array compiled into the library instead of the
// handle's lazily allocated scratch buffer.
//
// The array lives in device memory for as long as the library is loaded, on every GPU that
// loads it.  Its host-side name is only a stand-in, so the host fetches the device address
// with cudaGetSymbolAddress once per device (on the first call made on that device, with that
// device current) and passes it to the kernels.  All calls share the array: two calls whose
// kernels overlap on the GPU (for example on different streams) race on it.
#include <array>
#include <mutex>

#include "sv_internal.h"

namespace sv {
namespace {

constexpr int kMaxPartials = 4096;  // up to 4096 CTAs of partial sums (64 KiB of scratch)
constexpr int kMaxDevices = 64;

// Two doubles for each of up to kMaxPartials CTAs, then the final (re, im) pair and the paired sum's words.
static __device__ __align__(256) double g_expval_scratch[2 * kMaxPartials + 2 + (sizeof(Readout) + 7) / 8];

std::mutex g_mu;
std::array<double *, kMaxDevices> g_addr{};

double *scratch_address(int dev) {
    if (dev < 0 || dev >= kMaxDevices) fail(SV_ERR_UNSUPPORTED, "sv_expval_pauli_noalloc: device index too large");
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_addr[dev]) {
        double *p = nullptr;
        check_cuda(cudaGetSymbolAddress(reinterpret_cast<void **>(&p), g_expval_scratch),
                   "cudaGetSymbolAddress(expval scratch)");
        g_addr[dev] = p;
    }
    return g_addr[dev];
}

// One thread adds the partials in CTA order into the final pair.
__global__ void k_expval_final_noalloc(double *scratch, int nparts) {
    double r = 0, i = 0;
    for (int b = 0; b < nparts; ++b) {
        r += scratch[2 * b];
        i += scratch[2 * b + 1];
    }
    scratch[2 * kMaxPartials] = r;
    scratch[2 * kMaxPartials + 1] = i;
}

}  // namespace
}  // namespace sv

using namespace sv;

extern "C" sv_status sv_expval_pauli_noalloc(sv_handle h, uint64_t x, uint64_t z, double *out) {
    try {
        if (!h || !out) fail(SV_ERR_ARG, "sv_expval_pauli_noalloc: null argument");
        if ((x >> h->n) || (z >> h->n)) fail(SV_ERR_ARG, "sv_expval_pauli_noalloc: Pauli mask outside the register");
        int dev = -1;
        check_cuda(cudaGetDevice(&dev), "cudaGetDevice");
        if (dev != h->device) fail(SV_ERR_ARG, "sv_expval_pauli_noalloc: the handle's device is not current");
        const int64_t len = int64_t(1) << h->n;
        const int64_t nb = std::max<int64_t>(1, std::min<int64_t>((int64_t)num_sms() * 8, len / 256));
        if (nb > kMaxPartials)
            fail(SV_ERR_UNSUPPORTED, "sv_expval_pauli_noalloc: needs " + std::to_string(nb) +
                                         " partial sums, more than the fixed scratch holds (4096)");
        double *scratch = scratch_address(dev);
        // the same kernels and the same order of summation as sv_expval_pauli's
        Readout *words = reinterpret_cast<Readout *>(scratch + 2 * kMaxPartials + 2), r;
        launch_partial_expval(h->dtype, h->amp, h->n, x, z, scratch, (int)nb, h->stream);
        launch_finish(scratch, (int)nb, true, h->dev_err, words, h->stream);
        check_cuda(cudaMemcpyAsync(&r, words, sizeof(r), cudaMemcpyDeviceToHost, h->stream), "cudaMemcpyAsync(expval result)");
        // synchronise and report a failure an earlier kernel on this handle left in its error word
        check_dev_error(h);
        const bool odd = __builtin_popcountll(x & z) & 1;
        double res[2] = {odd ? 0.0 : r.value, odd ? r.value : 0.0};
        if (expval_cancels(r)) {
            launch_partial_expval_direct(h->dtype, h->amp, h->n, x, z, scratch, (int)nb, h->stream);
            k_expval_final_noalloc<<<1, 1, 0, h->stream>>>(scratch, (int)nb);
            check_cuda(cudaGetLastError(), "expval (no-alloc) final kernel launch");
            check_cuda(cudaMemcpyAsync(res, scratch + 2 * kMaxPartials, sizeof(res), cudaMemcpyDeviceToHost, h->stream),
                       "cudaMemcpyAsync(expval result)");
            check_dev_error(h);
        }
        pauli_phase(x, z, res[0], res[1], out);
        return SV_OK;
    } catch (const sv::Error &e) {
        sv::set_error(e.msg);
        return e.code;
    }
}
