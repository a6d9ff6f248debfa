// af_step_host_bands: a step of a state kept in host memory, in bands whose
// copies in, step and copies back overlap on three streams.  Native because
// the enqueueing itself was the bottleneck: seven calls and four event
// operations per band took 90 us of Python, more than a 6 MB band's copies
// (2048^2 cells in 32 bands: 2.97 ms a step from Python, 1.57 now; the copies
// alone take 1.2 at the link's rate both ways).
#include <cuda_runtime.h>

#include <new>

#include "af_internal.h"

namespace {

// A failed call's error is reported by the return value, and not once more by
// whatever call reads the runtime's last error next.
bool ok(cudaError_t e) {
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess;
}

// Events of one call, destroyed on return (the driver keeps what is pending).
struct Events {
    cudaEvent_t *e = nullptr;
    int n = 0;
    explicit Events(int want) {
        e = new (std::nothrow) cudaEvent_t[want];
        if (!e) return;
        while (n < want && ok(cudaEventCreateWithFlags(&e[n], cudaEventDisableTiming))) ++n;
        if (n < want) {
            clear();
        }
    }
    void clear() {
        for (int k = 0; k < n; ++k) cudaEventDestroy(e[k]);
        n = 0;
    }
    ~Events() {
        clear();
        delete[] e;
    }
    Events(const Events &) = delete;
    Events &operator=(const Events &) = delete;
};

}  // namespace

extern "C" af_status af_step_host_bands(const af_config *cfg, int32_t tiling, int32_t nband, const af_band *h_band,
                                        int32_t owned, void *h_state, void *d_up, void *d_down, void *d_a, void *d_b,
                                        double dt0, double dx0, double dy0, double *d_flux_reg, void *stream,
                                        void *s_in, void *s_cmp, void *s_out) {
    if (!cfg || nband < 1 || !h_band || !h_state || !d_a || !d_b) return AF_ERR_ARG;
    if (owned && (!d_up || !d_down)) return AF_ERR_ARG;
    if (cfg->n < 2 || cfg->n > 64 || (cfg->prec != AF_F64 && cfg->prec != AF_F32)) return AF_ERR_ARG;
    if (cfg->ncomp != (cfg->eq == AF_ADVECTION ? 1 : 3)) return AF_ERR_ARG;
    for (int b = 0; b < nband; ++b)
        if (h_band[b].p0 < 0 || h_band[b].p1 <= h_band[b].p0 || h_band[b].nwork < 0) return AF_ERR_ARG;
    // a step that would be refused is, before the first copy
    for (int b = 0; b < nband; ++b) {
        const af_status st = af::step_check(cfg, tiling, h_band[b].nwork, h_band[b].d_work, d_a, d_b, dt0, dx0, dy0, d_flux_reg);
        if (st != AF_OK) return st;
    }
    const size_t esz = cfg->prec == AF_F64 ? 8 : 4;
    const size_t dev = (size_t)af_patch_words(cfg->n, cfg->ncomp) * esz;
    const size_t host = owned ? (size_t)cfg->ncomp * 4 * cfg->n * cfg->n * esz : dev;
    cudaStream_t cur = static_cast<cudaStream_t>(stream), in = static_cast<cudaStream_t>(s_in);
    cudaStream_t cmp = static_cast<cudaStream_t>(s_cmp), out = static_cast<cudaStream_t>(s_out);
    auto at = [](void *base, size_t patch, size_t bytes) { return static_cast<char *>(base) + patch * bytes; };

    Events ev(2 * nband + 4);  // uploaded [nband], stepped [nband], start, ends of s_out, s_cmp, s_in
    if (ev.n == 0) return AF_ERR_CUDA;
    cudaEvent_t *const up = ev.e, *const done = ev.e + nband, start = ev.e[2 * nband];
    if (!ok(cudaEventRecord(start, cur)) || !ok(cudaStreamWaitEvent(in, start, 0)) ||
        !ok(cudaStreamWaitEvent(cmp, start, 0)) || !ok(cudaStreamWaitEvent(out, start, 0)))
        return AF_ERR_CUDA;
    af_status st = AF_OK;
    // copies only, back to back: the link stays busy
    for (int b = 0; b < nband && st == AF_OK; ++b) {
        const af_band &B = h_band[b];
        const size_t p0 = B.p0, bytes = (size_t)(B.p1 - B.p0) * host;
        if (!ok(cudaMemcpyAsync(at(owned ? d_up : d_a, p0, host), at(h_state, p0, host), bytes, cudaMemcpyHostToDevice, in)) ||
            !ok(cudaEventRecord(up[b], in)))
            st = AF_ERR_CUDA;
    }
    int ready = -1;  // bands 0 .. ready have arrived on cmp
    for (int k = 1; k <= nband && st == AF_OK; ++k) {
        const int b = k == nband ? 0 : k;  // 1, 2, .., nband - 1, 0: the band above is the last to arrive
        while (ready < (b + 1 < nband ? b + 1 : nband - 1) && st == AF_OK) {
            const af_band &U = h_band[++ready];
            if (!ok(cudaStreamWaitEvent(cmp, up[ready], 0)))
                st = AF_ERR_CUDA;
            else if (owned)
                st = af_unpack_owned(cfg, U.p1 - U.p0, at(d_up, U.p0, host), at(d_a, U.p0, dev), cmp);
        }
        if (st != AF_OK) break;
        const af_band &B = h_band[b];
        st = af_patch_step_tiled(cfg, tiling, B.nwork, B.d_work, d_a, d_b, dt0, dx0, dy0, d_flux_reg, cmp);
        if (st == AF_OK && owned)
            st = af_pack_owned(cfg, B.p1 - B.p0, at(d_b, B.p0, dev), at(d_down, B.p0, host), cmp);
        if (st != AF_OK) break;
        const size_t p0 = B.p0, bytes = (size_t)(B.p1 - B.p0) * host;
        if (!ok(cudaEventRecord(done[b], cmp)) || !ok(cudaStreamWaitEvent(out, done[b], 0)) ||
            !ok(cudaMemcpyAsync(at(h_state, p0, host), at(owned ? d_down : d_b, p0, host), bytes, cudaMemcpyDeviceToHost, out)))
            st = AF_ERR_CUDA;
    }
    // joined even after an error, by every join that can still be made: what was
    // enqueued stays ordered before `stream`.  (s_cmp has waited for all uploads
    // unless a band was left out.)
    const cudaStream_t last[3] = {out, cmp, in};
    for (int k = 0; k < (st == AF_OK ? 2 : 3); ++k) {
        cudaEvent_t end = ev.e[2 * nband + 1 + k];
        if ((!ok(cudaEventRecord(end, last[k])) || !ok(cudaStreamWaitEvent(cur, end, 0))) && st == AF_OK) st = AF_ERR_CUDA;
    }
    return st;
}
