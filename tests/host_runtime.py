"""The handle runtime (csrc/pt_capi.cu) compiled with the host compiler against a CUDA runtime of a
few lines, for tests of its bookkeeping and error paths without a GPU.

Device memory is host memory.  Every copy is checked against the allocations it touches, every sweep
launch against what its bundles need (threads, shared memory, the launch's mapping), and the n-th
allocation or launch from now on can be made to fail.  Kernels compute nothing: set_spins leaves
records by their index, a TTS reduction zeros, so every evaluation counts as decided.
"""
import ctypes as C
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1605_03607_gb300", "csrc")

RUNTIME = r"""
#include <unistd.h>
#include <atomic>
#include <cstring>
#include <map>
#include <vector>
#include "pt_capi.cu"

namespace {
std::map<char*, size_t> device;
std::atomic<long> overruns{0}, down{0};
long launches = 0, allocs = 0;
long fail_launch = 0, launch_last = 0, fail_alloc = 0, alloc_last = 0;     // failing range, counted from 1
int fast_team = 0, fast_block = -1, last_team = 0, last_block = 0, last_ctas = 0;
std::vector<int> seen;                        // runs covered by the last launch: instance * 4096 + run
bool bad_launch = false;
int wait_us = 0;                              // length of a stream synchronisation
bool inside(const void* p, size_t n)
{
    auto it = device.upper_bound((char*)p);
    if (it == device.begin()) return false;
    --it;
    return (char*)p + n <= it->first + it->second;
}
bool fails(long& count, long first, long last) { ++count; return first > 0 && count >= first && count <= last; }
}

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n)
{
    *p = nullptr;
    if (fails(allocs, fail_alloc, alloc_last)) return cudaErrorMemoryAllocation;
    *p = std::calloc(1, n);
    device[(char*)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) { device.erase((char*)p); std::free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t)
{
    if (n && !inside(k == cudaMemcpyHostToDevice ? d : s, n)) { ++overruns; return cudaSuccess; }
    if (k == cudaMemcpyDeviceToHost) down += (long)n;
    if (n) std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) { return cudaMemcpyAsync(d, s, n, k, 0); }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t)
{
    if (n && !inside(d, n)) { ++overruns; return cudaSuccess; }
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t)
{
    *ms = last_team == fast_team && last_block == fast_block ? 1.0f : 2.0f;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)1; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { if (wait_us) usleep(wait_us); return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "made to fail"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
int sg_forward(sg_model*, int32_t, int32_t, const int8_t*, float*) { return PT_ERR_STATE; }
const char* sg_last_error(const sg_model*) { return ""; }

void host_fail_launches(long first, long last) { launches = 0; fail_launch = first; launch_last = last; }
void host_fail_allocs(long first, long last) { allocs = 0; fail_alloc = first; alloc_last = last; }
void host_fastest(int team, int block) { fast_team = team; fast_block = block; }
long host_launches() { return launches; }
long host_allocs() { return allocs; }
long host_overruns() { return overruns; }
long host_downloaded() { return down.exchange(0); }
void host_wait(int us) { wait_us = us; }
int host_last_team() { return last_team; }
int host_last_block() { return last_block; }
int host_last_ctas() { return last_ctas; }
// 1 if the last sweep launch covered runs 0 .. runs - 1 of n instances once each and its bundles fitted it
int host_last_launch_ok(int n, int runs)
{
    if (bad_launch || (int)seen.size() != n * runs) return 0;
    std::vector<char> hit((size_t)n * runs, 0);
    for (int x : seen) {
        const int i = x / 4096, r = x % 4096;
        if (i >= n || r >= runs || hit[(size_t)i * runs + r]) return 0;
        hit[(size_t)i * runs + r] = 1;
    }
    return 1;
}
}

namespace ptg {
cudaError_t sweep_smem_capacity(int* b) { *b = 232448 - 16; return cudaSuccess; }
cudaError_t set_sweep_smem_limit(int, int, bool, int, int) { return cudaSuccess; }
cudaError_t launch_init(const InstDesc*, const int2*, int, bool, cudaStream_t) { return cudaSuccess; }
// a state that can be told apart: records by their index, slots in reverse order
cudaError_t launch_energy(const InstDesc* insts, const int2* items, int nitems, int32_t, cudaStream_t)
{
    for (int i = 0; i < nitems; ++i) {
        const InstDesc& d = insts[items[i].x];
        const int r = items[i].y, np = d.NT > 1 ? d.NT - 1 : 1;
        for (int t = 0, x = r * d.NT; t < d.NT; ++t, ++x) {
            d.E[x] = 7 * x + 3;
            d.perm[x] = (uint8_t)(d.NT - 1 - t);
            d.macc[x] = 11 * x;
        }
        for (int t = 0; t < np; ++t) d.xacc[r * np + t] = 13 * (r * np + t);
        d.best[r] = -r;
        d.first[r] = r + 1;
    }
    return cudaSuccess;
}
cudaError_t launch_hamming(const InstDesc*, int, const int32_t*, const int32_t*, int32_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_tts(const InstDesc*, int n, int32_t, int32_t, int32_t* out, cudaStream_t, const int32_t*)
{
    if (!inside(out, 12 * (size_t)n)) { ++overruns; return cudaSuccess; }
    std::memset(out, 0, 12 * (size_t)n);
    return cudaSuccess;
}
cudaError_t launch_sweeps(const InstDesc* insts, const Bundle* bundles, int nb, int grid, int block, int smem, uint32_t, int, int,
                          int, int*, cudaStream_t, int team, bool walk, int)
{
    if (fails(launches, fail_launch, launch_last)) return cudaErrorLaunchOutOfResources;
    seen.clear();
    bad_launch = smem > 232448 - 16 || block > 1024;
    last_team = team;
    last_block = block;
    last_ctas = grid;
    if (!inside(bundles, sizeof(Bundle) * (size_t)nb)) { ++overruns; bad_launch = true; return cudaSuccess; }
    for (int i = 0; i < nb; ++i) {
        const Bundle& b = bundles[i];
        const InstDesc& d = insts[b.inst];
        int64_t threads, need;
        if ((b.team < 0) != (team < 0) || (b.team > 0) != (team > 0) || walk != (d.wstate != nullptr)) bad_launch = true;
        if (b.team < 0) {
            const int gr = -b.team, ng = (b.nitems + gr - 1) / gr + (b.nitems2 + gr - 1) / gr;
            const LaneLayout l = lane_layout(d.L, d.NT, d.kt, gr, ng, walk, b.nitems2 > 0 ? 2 : 1);
            threads = 32 * b.sp * l.ncols * ng;
            need = l.bytes;
        } else {
            threads = (int64_t)b.nitems * (b.team > 0 ? b.sp * b.team : b.sp * d.L * d.L);
            need = bundle_smem_bytes(d.L, d.NT, b.nitems, b.team, walk, d.kt);
        }
        if (threads > block || need > smem) bad_launch = true;
        for (int r = 0; r < b.nitems; ++r) seen.push_back(b.inst * 4096 + b.run0 + r);
        for (int r = 0; r < b.nitems2; ++r) seen.push_back(b.inst2 * 4096 + r);
    }
    return cudaSuccess;
}
bool debug_build() { return false; }
cudaError_t debug_check(cudaStream_t, const char*) { return cudaSuccess; }
unsigned debug_take() { return 0; }
}
"""


def build(folder):
    """Compiles the runtime into `folder` and loads it; None without a host compiler or CUDA headers."""
    from paper_1605_03607_gb300 import _lib
    from paper_1605_03607_gb300 import build as B
    gxx = shutil.which("g++")
    headers = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    if gxx is None or not os.path.exists(os.path.join(headers, "cuda_runtime.h")):
        return None
    src, so = os.path.join(str(folder), "runtime.cpp"), os.path.join(str(folder), "libhost_runtime.so")
    with open(src, "w") as f:
        f.write(RUNTIME)
    # -Bsymbolic: these definitions, not those of a CUDA runtime that the process has loaded
    subprocess.run([gxx, "-std=c++17", "-O1", "-w", "-fPIC", "-shared", "-Wl,-Bsymbolic", f"-I{headers}", f"-I{CSRC}",
                    f"-I{os.path.join(ROOT, 'include')}", src, "-o", so], check=True)
    lib = C.CDLL(so)
    for name, res, args in _lib.SIGNATURES:
        if hasattr(lib, name):
            f = getattr(lib, name)
            f.restype, f.argtypes = res, args
    for name in ("launches", "allocs", "overruns", "downloaded"):
        getattr(lib, "host_" + name).restype = C.c_long
    for name in ("launches", "allocs"):
        getattr(lib, "host_fail_" + name).argtypes = [C.c_long, C.c_long]
    return lib
