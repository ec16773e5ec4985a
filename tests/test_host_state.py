"""The host side of klb_set_state and klb_get_state, over a stand-in for the CUDA runtime (device memory is host
memory, kernel launches do nothing).  Without host memory for the conversions, each allocation failing in turn:
KLB_ENOMEM, and the lattice's buffers and step stay as they were.  States of narrow, ragged and full rows, whose
species go in one copy (up to 1 MB) or one by one, come back as they went in, 0 where a species has no cell, with
zero padding; a lattice starts from rest."""
import os
import subprocess

import pytest

from paper_2403_15768_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2403_15768_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "klb.h"
#include "klb_internal.h"

static int left = -1;  // allocations until one fails; < 0: none fails

void *operator new[](std::size_t n, const std::nothrow_t &) noexcept
{
    return left >= 0 && left-- == 0 ? nullptr : std::malloc(n ? n : 1);
}
void operator delete[](void *p) noexcept { std::free(p); }

extern "C" {
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { return std::memmove(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { return std::memmove(d, s, n), cudaSuccess; }
cudaError_t cudaMemset(void *d, int v, size_t n) { return std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return cudaErrorNotSupported; }
cudaError_t cudaEventCreate(cudaEvent_t *) { return cudaErrorNotSupported; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventElapsedTime(float *, cudaEvent_t, cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "stand-in"; }
}

namespace klb {
cudaError_t launch(int, int, const void *, int, int, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_ref(int, int, const void *, float *const[3], float *const[3], cudaStream_t) { return cudaSuccess; }
cudaError_t launch_finalize(const double *, int, double *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_count_period(uint32_t *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_batch(int, int, const BatchLaunch &, cudaStream_t) { return cudaSuccess; }
cudaError_t static_scratch(double **, double **, size_t *) { return cudaErrorNotSupported; }
}

#define NEED(c) do { if (!(c)) return std::printf("storage %d, allocation %d: %s\n", storage, fail, #c), 1; } while (0)

static int round_trip(int nx, int storage)
{
    const int fail = nx;
    klb_desc d;
    std::memset(&d, 0, sizeof d);
    d.kind = KLB_D3Q19;
    d.nx = nx;
    d.ny = d.nz = 11;
    d.geom = KLB_GEOM_PIPE;
    d.radius = 3;
    d.shell = 1;
    d.tau_w = d.tau_e = d.tau_p = 0.8;
    d.rho0 = 1.0;
    d.storage = storage;
    const size_t bytes = klb_lattice_bytes(&d), cells = (size_t)nx * 11 * 11, nxp = (nx + 31) / 32 * 32;
    char *buf = static_cast<char *>(std::aligned_alloc(256, (bytes + 255) / 256 * 256));
    std::memset(buf, 0x7f, bytes);
    klb_lattice *L = nullptr;
    klb_info info;
    NEED(klb_create_lattice(&d, buf, bytes, nullptr, &L) == KLB_OK && klb_lattice_info(&d, &info) == KLB_OK);
    std::vector<double> g(3 * 19 * cells), u(9 * cells), h(g.size(), 9.0), v(u.size(), 9.0), w(u.size(), 9.0);
    NEED(klb_get_state(L, h.data(), v.data(), w.data()) == KLB_OK);  // from rest, over a buffer of 0x7f
    for (double x : h) NEED(x == 0.0);
    for (double x : v) NEED(x == 0.0);
    for (double x : w) NEED(x == 0.0);
    h.assign(h.size(), 9.0);
    for (size_t k = 0; k < g.size(); ++k) g[k] = (float)(1e-4 * (double)(k % 97 + 1));
    for (size_t k = 0; k < u.size(); ++k) u[k] = (float)(1e-4 * (double)(k % 89 + 1));
    NEED(klb_set_state(L, g.data(), u.data(), u.data(), 2) == KLB_OK);
    NEED(klb_get_state(L, h.data(), v.data(), w.data()) == KLB_OK);
    size_t live = 0, faces = 0;
    for (size_t k = 0; k < g.size(); ++k) {
        NEED(h[k] == g[k] || h[k] == 0.0);
        live += h[k] != 0.0;
    }
    for (size_t k = 0; k < u.size(); ++k) {
        NEED((v[k] == u[k] || v[k] == 0.0) && w[k] == v[k]);
        faces += v[k] != 0.0;
    }
    NEED(live == 19 * (size_t)(info.species_cells[0] + 2 * info.species_cells[1]));
    NEED(faces == 3 * (size_t)nx * (size_t)(info.iface_cs[0] + 2 * info.iface_cs[1]));
    const size_t size = storage == KLB_FP64 ? 8 : 4;  // padding of the first state buffer's first rows
    for (size_t r = 0; r < (size_t)info.fluid_cs; ++r)
        for (size_t b = (r * nxp + nx) * size; b < (r + 1) * nxp * size; ++b) NEED(buf[b] == 0);
    klb_destroy(L);
    std::free(buf);
    return 0;
}

int main()
{
    for (int nx : {1, 5, 25, 26, 31, 32, 33, 51, 52, 64, 130, 700})
        for (int storage : {KLB_FP64, KLB_FP32})
            if (round_trip(nx, storage)) return 1;
    for (int storage = 0; storage < 4; ++storage) {
        int fail = -1;
        klb_desc d;
        std::memset(&d, 0, sizeof d);
        d.kind = KLB_D3Q19;
        d.nx = 5;
        d.ny = d.nz = 12;
        d.geom = KLB_GEOM_PIPE;
        d.radius = 3;
        d.shell = 1;
        d.tau_w = d.tau_e = d.tau_p = 0.8;
        d.rho0 = 1.0;
        d.storage = storage;
        const size_t bytes = klb_lattice_bytes(&d), cells = 5 * 12 * 12;
        NEED(bytes > 0);
        char *buf = static_cast<char *>(std::aligned_alloc(256, (bytes + 255) / 256 * 256));
        std::memset(buf, 0, bytes);
        klb_lattice *L = nullptr;
        NEED(klb_create_lattice(&d, buf, bytes, nullptr, &L) == KLB_OK);
        std::vector<double> g(3 * 19 * cells), u(9 * cells);
        for (size_t k = 0; k < g.size(); ++k) g[k] = 1e-4 * (double)(k % 97);
        for (size_t k = 0; k < u.size(); ++k) u[k] = 1e-4 * (double)(k % 89);
        NEED(klb_set_state(L, g.data(), u.data(), u.data(), 3) == KLB_OK);
        NEED(klb_step(L, 4) == KLB_OK && klb_get_step(L) == 7);
        const std::vector<char> before(buf, buf + bytes);
        int failed = 0;
        for (fail = 0; fail < 20; ++fail) {
            left = fail;
            const klb_status st = klb_set_state(L, g.data(), u.data(), u.data(), 50);
            left = -1;
            if (st == KLB_OK) break;
            ++failed;
            NEED(st == KLB_ENOMEM);
            NEED(klb_get_step(L) == 7);
            NEED(std::memcmp(before.data(), buf, bytes) == 0);
        }
        NEED(failed >= 3 && klb_get_step(L) == 50);
        klb_destroy(L);
        std::free(buf);
    }
    return 0;
}
"""


def test_state_on_the_host(tmp_path):
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    if not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                           "-I", include, str(src), os.path.join(CSRC, "klb_api.cpp"),
                           os.path.join(CSRC, "klb_geometry.cpp"), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
