"""Work on a context's side stream is joined on every way out of a call: the
host side of the library (api.cu, as built) is linked against a fake of the
CUDA runtime and of the kernels' launchers, which writes down what is queued
where and fails the n-th launch of a call.  Whatever fails, the context's own
stream has waited for everything queued on the side stream when the call
returns, and the caller's for that."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2503_20605_gb300")

RUNTIME = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <vector>
#include <cuda_runtime_api.h>
#include "iblb.h"

// a stream's clock counts what was queued on it; known[s][t]: how much of stream t comes before s's next work
static int streams = 0, events = 0, launches = 0, fail_at = 0;
static long clk[8], known[8][8];
static std::map<void *, std::vector<long>> ev;
static int id(cudaStream_t s) { return (int)(intptr_t)s; }
static void queue(cudaStream_t s) { known[id(s)][id(s)] = ++clk[id(s)]; }
// the n-th launch of a call fails, after its work was queued in part
cudaError_t fake_launch(cudaStream_t s)
{
    queue(s);
    return ++launches == fail_at ? cudaErrorLaunchOutOfResources : cudaSuccess;
}
extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { *p = calloc(n ? n : 1, 1); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t t) { memcpy(d, s, n); queue(t); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t t) { memset(d, v, n); queue(t); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)(intptr_t)++streams; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) { *s = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)(intptr_t)++events; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    ev[e].assign(known[id(s)], known[id(s)] + 8);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned)
{
    for (int t = 0; t < 8; ++t)
        if (!ev[e].empty() && ev[e][t] > known[id(s)][t])
            known[id(s)][t] = ev[e][t];
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
}

int main()
{
    iblb_lattice_desc lat{};
    lat.nx = lat.ny = lat.nz = 24;
    lat.tau_out = 1.0;
    lat.lambda = 5.0;
    lat.rho0 = 1.0;
    lat.walls = 1;
    iblb_physics_desc phys{};
    phys.sigma = 0.01;
    const double x[12] = {8, 8, 8, 14, 8, 8, 8, 14, 8, 8, 8, 14};
    const int32_t tri[12] = {0, 2, 1, 0, 1, 3, 0, 3, 2, 1, 2, 3};
    // streams: the caller's is 7, the context's own and its side stream the first two made
    for (int call = 0; call < 3; ++call)
        for (int n = 0; n <= 12; ++n) {
            iblb_ctx *c = nullptr;
            streams = events = launches = fail_at = 0;
            memset(clk, 0, sizeof(clk));
            memset(known, 0, sizeof(known));
            ev.clear();
            if (iblb_create(&lat, &phys, (void *)(intptr_t)7, &c) || iblb_set_membrane(c, 0, x, 4, tri, 4) ||
                iblb_set_option(c, IBLB_OPT_SPLIT_LB, call == 2))
                return 1;
            const long side0 = clk[2];
            launches = 0;
            fail_at = n;
            iblb_obs o;
            const int r = call == 0 ? iblb_observe(c, 0, 0.3, 0.2, &o)
                                    : (call == 1 ? iblb_observe_all(c, 0.3, 0.2, &o) : iblb_step(c, 1));
            std::printf("%d %d %d %d %ld %ld %ld %d\n", call, n, r, launches, clk[2] - side0, clk[2] - known[1][2],
                        clk[2] - known[7][2], streams);
            iblb_destroy(c);
        }
    return 0;
}
"""
LAUNCHERS = r"""
#include <cstring>
#include "iblb_internal.h"
cudaError_t fake_launch(cudaStream_t s);
static cudaError_t launch(cudaStream_t s) { return fake_launch(s); }
namespace iblb {
int lb_consumers(int) { return 224; }
int lb_items_per_row(int p, int sb) { return sb == 2 ? p / 2 : p; }
int64_t observe_scratch_doubles(int, int) { return 64; }
void obs_mesh_plan(ObsMesh &m) { m.nc = m.fpc = m.npc = 1; }
void finish_observe(const double *, double, double *h) { memset(h, 0, sizeof(double) * 14); }
cudaError_t launch_init_populations(const Arrays &, int, void *, cudaStream_t s) { return launch(s); }
cudaError_t launch_mass(const Arrays &, int, const void *, double *, int, int, int, int, cudaStream_t s)
{
    const cudaError_t e = launch(s);         // two kernels
    return e == cudaSuccess ? launch(s) : e;
}
cudaError_t launch_corrected_positions(const Arrays &, cudaStream_t s, double *, int, int) { return launch(s); }
cudaError_t enqueue_observe(const ObsMesh *, const ObsMesh *, int, int, double, double, cudaStream_t s) { return launch(s); }
cudaError_t enqueue_observe_result(const ObsMesh *, const ObsMesh *, int, const double *, const int *, int, double *, cudaStream_t s) { return launch(s); }
cudaError_t launch_classify(const Arrays &, cudaStream_t s) { return launch(s); }
cudaError_t launch_node_force(const Arrays &, cudaStream_t s) { return launch(s); }
cudaError_t launch_spread(const Arrays &, cudaStream_t s, bool) { return launch(s); }
cudaError_t launch_inout(const Arrays &, cudaStream_t s, bool) { return launch(s); }
cudaError_t launch_interp_advect(const Arrays &, cudaStream_t s) { return launch(s); }
cudaError_t launch_volume_correction(const Arrays &, int, cudaStream_t s) { return launch(s); }
cudaError_t launch_lb(const Arrays &, int, const void *, void *, bool, const LaunchCfg &, cudaStream_t s, const int *, const int *, bool, int, bool) { return launch(s); }
}
"""


def test_side_stream_is_joined_whatever_fails(tmp_path):
    from paper_2503_20605_gb300 import build
    build.build()
    rt, la, exe = tmp_path / "rt.cpp", tmp_path / "la.cu", tmp_path / "fake"
    rt.write_text(RUNTIME)
    la.write_text(LAUNCHERS)
    inc = [f"-I{os.path.join(ROOT, 'include')}", f"-I{os.path.join(PKG, 'csrc')}"]
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, *inc, "-c", str(la), "-o", str(tmp_path / "la.o")], check=True)
    subprocess.run(["g++", "-std=c++17", *inc, "-I", cuda, "-c", str(rt), "-o", str(tmp_path / "rt.o")], check=True)
    # (what is not called here stays unresolved)
    subprocess.run(["g++", "-no-pie", "-Wl,--unresolved-symbols=ignore-all", "-o", str(exe), str(tmp_path / "rt.o"),
                    str(tmp_path / "la.o"), os.path.join(PKG, "_build", "api.o"), "-ldl", "-lpthread"], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rows = [[int(v) for v in line.split()] for line in out.splitlines()]
    assert len(rows) == 39
    failed = 0
    for call, n, r, launches, side, behind, caller, streams in rows:
        assert streams == 2
        assert (r != 0) == (0 < n <= launches), (call, n)
        if r == 0:
            assert side > 0, (call, n)               # the side stream is used at all
        failed += r != 0 and side > 0
        assert behind == 0, (call, n, "the context's stream runs ahead of the side stream")
        assert caller == 0, (call, n, "the caller's stream runs ahead of the side stream")
    assert failed >= 12
