"""CPU model of af_step_host_bands' stream order: its source compiled against a
fake CUDA runtime that keeps, for every stream, which copies and kernels a wait
for it would cover.  Whatever fails on the way -- a copy, an event, the step of
a band -- every copy that was enqueued is ordered before the caller's stream
when the call returns, no runtime error is left pending, and a step that would
be refused is refused before the first copy."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda/include"

FAKE = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <set>
#include "af.h"

static std::map<void *, std::set<int>> before;  // operations a stream or event comes after
static int ops = 0, copies = 0, pending = 0, events = 0;
static int fail_kind = 0, fail_at = 0, seen[6];   // the fail_at-th call of a kind fails
enum { kCopy = 1, kRecord, kWait, kStep, kPack };

static bool fails(int kind) { return ++seen[kind] == fail_at && kind == fail_kind; }
static cudaError_t bad() { pending = 1; return cudaErrorInvalidValue; }
static void op(void *s) { before[s].insert(ops++); }

extern "C" {
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = (cudaEvent_t)malloc(1); ++events; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { before.erase(e); free(e); --events; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    if (fails(kRecord)) return bad();
    before[e] = before[s];
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    if (fails(kWait)) return bad();
    before[s].insert(before[e].begin(), before[e].end());
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t s) {
    if (fails(kCopy)) return bad();
    op(s);
    ++copies;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { const int p = pending; pending = 0; return p ? cudaErrorInvalidValue : cudaSuccess; }
int64_t af_patch_words(int32_t, int32_t) { return 64; }
af_status af_patch_step_tiled(const af_config *, int32_t, int32_t, const af_work *, const void *, void *, double, double,
                              double, double *, void *s) {
    if (fails(kStep)) return AF_ERR_UNIMPLEMENTED;
    op(s);
    return AF_OK;
}
af_status af_pack_owned(const af_config *, int32_t, const void *, void *, void *s) {
    if (fails(kPack)) return AF_ERR_CUDA;
    op(s);
    return AF_OK;
}
af_status af_unpack_owned(const af_config *, int32_t, const void *, void *, void *s) { op(s); return AF_OK; }
}
namespace af {
af_status step_check(const af_config *, int32_t, int32_t, const af_work *, const void *, const void *, double dt, double,
                     double, const double *) {
    return dt < 1.0 ? AF_OK : AF_ERR_CFL;
}
}

int main(int argc, char **argv) {
    const int nband = atoi(argv[1]), owned = atoi(argv[2]);
    fail_kind = atoi(argv[3]);
    fail_at = atoi(argv[4]);
    const double dt = atof(argv[5]);
    af_config cfg = {};
    cfg.eq = AF_ACOUSTICS;
    cfg.prec = AF_F32;
    cfg.n = 8;
    cfg.ncomp = 3;
    af_band *b = new af_band[nband];
    for (int k = 0; k < nband; ++k) b[k] = {k, k + 1, 1, 0, (const af_work *)64};
    static char buf[5][1 << 16], stream[4];
    const af_status st = af_step_host_bands(&cfg, 0, nband, b, owned, buf[0], buf[1], buf[2], buf[3], buf[4], dt, 1.0, 1.0,
                                            nullptr, &stream[0], &stream[1], &stream[2], &stream[3]);
    // status, copies, operations, those that the caller's stream comes after, error left pending, events left
    printf("%d %d %d %d %d %d\n", (int)st, copies, ops, (int)before[&stream[0]].size(), pending, events);
    return 0;
}
"""


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("host_step")
    (d / "fake.cpp").write_text(FAKE)
    csrc = os.path.join(ROOT, "paper_2205_07572_gb300", "csrc")
    exe = str(d / "model")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CUDA, "-I", os.path.join(ROOT, "include"), "-I", csrc,
                    str(d / "fake.cpp"), os.path.join(csrc, "af_host_step.cpp"), "-o", exe], check=True)

    def run(nband, owned, kind=0, at=0, dt=0.1):
        out = subprocess.run([exe] + [str(v) for v in (nband, owned, kind, at, dt)], check=True, capture_output=True, text=True)
        return [int(v) for v in out.stdout.split()]
    return run


@pytest.mark.parametrize("owned", [0, 1])
@pytest.mark.parametrize("nband", [1, 2, 7])
def test_every_enqueued_operation_is_ordered_before_the_callers_stream(model, nband, owned):
    st, copies, ops, covered, pending, events = model(nband, owned)
    assert st == 0 and copies == 2 * nband and covered == ops and events == 0
    # the k-th copy, step or pack fails; event records and waits up to the joins
    # themselves (start and its three waits before anything is enqueued)
    kinds = {1: 2 * nband, 4: nband, 5: nband if owned else 0, 2: 1 + 2 * nband, 3: 3 + 2 * nband}
    for kind, calls in kinds.items():
        for at in range(1, calls + 1):
            st, copies, ops, covered, pending, events = model(nband, owned, kind, at)
            assert st != 0 and covered == ops and events == 0, (kind, at)


@pytest.mark.parametrize("owned", [0, 1])
def test_a_refused_step_copies_nothing(model, owned):
    st, copies, ops, covered, pending, events = model(5, owned, dt=2.0)
    assert st != 0 and copies == 0 and ops == 0


@pytest.mark.parametrize("kind", [1, 2, 3])
def test_no_runtime_error_is_left_pending(model, kind):
    """The failed call's error is returned, and the call that reads the
    runtime's last error next does not see it again."""
    for at in range(1, 5):  # two bands: four copies, at least as many event operations
        st, _, _, _, pending, _ = model(2, 1, kind, at)
        assert st != 0 and pending == 0, (kind, at)


@pytest.mark.gpu
def test_a_refused_launch_is_reported_once(tmp_path):
    """launch_chained returns a launch's error (1 MB of shared memory: refused
    by the host; nothing runs) and does not leave it to the next call that reads
    the last error.  (A machine without a driver reports that at every call.)"""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("needs nvcc")
    (tmp_path / "launch.cu").write_text(r"""
#include <cstdio>
#include "af_launch.cuh"
__global__ void kern(int *out) { *out = (int)af::chain_begin(); }
int main() {
    const cudaError_t e = af::launch_chained(true, kern, 1, 32, 1 << 20, nullptr, (int *)nullptr);
    printf("%d %d\n", (int)e, (int)cudaPeekAtLastError());
    return 0;
}
""")
    exe = str(tmp_path / "launch")
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2205_07572_gb300", "csrc"), str(tmp_path / "launch.cu"), "-o", exe], check=True)
    e, pending = (int(v) for v in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert e != 0 and pending == 0
