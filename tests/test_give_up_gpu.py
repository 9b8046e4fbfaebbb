"""The plane loop's way out when its copies' waits run out, without a fault: the
loop runs on a ring whose barriers want one arrival more than the copies give, so
that every wait gives up after its limit (1 s; three more while the copies in flight
are drained). The segment must end and say so, the timeout status be set, and the same
launch on proper barriers give the same field before and after it."""
import subprocess

import pytest

from paper_1912_00695_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cstdio>
#include <cstring>
#include <vector>
#include "fd_tma.cuh"
using namespace fdgb;
constexpr int R = 2, LZ = 8, W = 4, Nx = 13, Ny = 20, Nz = 40, PZ = 64;
using G = TmaShape<R, LZ, W, float>;

// one segment per tile over all planes, its barriers set up for `arrivals` arrivals each
__global__ void __launch_bounds__(32 * W) segment_kernel(const __grid_constant__ TmaMaps maps,
                                                         const __grid_constant__ StepArgs a, int arrivals,
                                                         unsigned *gave_up) {
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char *base = smem + ((128u - (smem_addr(smem) & 127u)) & 127u);
    if (threadIdx.x == 0) {
        uint64_t *bars = reinterpret_cast<uint64_t *>(base);
        for (int s = 0; s < TmaPipe<R>::STAGES; ++s) mbar_init(smem_addr(&bars[s]), arrivals);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    int g = 0;
    TmaAcc acc;
    const ScaleState sc = read_scales<float>(a);
    const bool ok = tma_segment<R, kFactored, LZ, W, float>(&maps, a, sc, blockIdx.x, blockIdx.y, 0, a.Nx, base + 128,
                                                            g, acc);
    if (!ok) atomicAdd(gave_up, 1u);
}

using Encode = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                            const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                            CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static bool box(Encode fn, void *base, int w, int h, CUtensorMap *out) {
    const cuuint64_t dims[3] = {Nz, Ny, Nx}, strides[2] = {PZ * 4, cuuint64_t(PZ) * Ny * 4};
    const cuuint32_t b[3] = {cuuint32_t(w), cuuint32_t(h), 1}, e[3] = {1, 1, 1};
    return fn(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, b, e, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int main() {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess)
        return 1;
    const Encode fn = reinterpret_cast<Encode>(p);
    const size_t n = size_t(Nx) * Ny * PZ;
    float *u, *up, *w;
    unsigned *words;  // status, segments that gave up
    if (cudaMalloc(&u, 4 * n) != cudaSuccess || cudaMalloc(&up, 4 * n) != cudaSuccess ||
        cudaMalloc(&w, 4 * n) != cudaSuccess || cudaMalloc(&words, 8) != cudaSuccess)
        return 1;
    std::vector<float> h(n), hw(n, 3.0f), got(n), first(n);
    for (size_t i = 0; i < n; ++i) h[i] = i % PZ < Nz ? float((i * 2654435761u >> 20) & 1023u) / 512.0f - 1.0f : 0.0f;
    TmaMaps maps;
    if (!box(fn, u, G::SW, G::SH, &maps.u_halo) || !box(fn, u, G::TZ, G::TY, &maps.u_pt) ||
        !box(fn, up, G::TZ, G::TY, &maps.up_pt) || !box(fn, w, G::TZ, G::TY, &maps.f1_pt) ||
        !box(fn, w, G::TZ, G::TY, &maps.f2_pt))
        return 1;
    StepArgs a{};
    a.u = u, a.up = up, a.f1 = a.f2 = w;
    a.Nx = a.x_hi = a.x_block = Nx, a.Ny = Ny, a.Nz = Nz, a.pz = PZ, a.plane = (long long)Ny * PZ;
    a.bx1 = a.by1 = a.bz1 = 1 << 20;  // no damping anywhere
    a.coef[1] = 0.02f, a.coef[2] = -0.001f;
    a.rec_sample = -1;
    a.status = words;
    if (cudaFuncSetAttribute(segment_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM_BYTES) != cudaSuccess)
        return 1;
    const dim3 grid((Nz + G::TZ - 1) / G::TZ, (Ny + G::TY - 1) / G::TY);
    for (int run = 0; run < 3; ++run) {
        unsigned out[2];
        cudaEvent_t e0, e1;
        float ms = 0.0f;
        cudaMemcpy(u, h.data(), 4 * n, cudaMemcpyHostToDevice);
        cudaMemcpy(up, h.data(), 4 * n, cudaMemcpyHostToDevice);
        cudaMemcpy(w, hw.data(), 4 * n, cudaMemcpyHostToDevice);
        cudaMemset(words, 0, 8);
        cudaEventCreate(&e0), cudaEventCreate(&e1);
        cudaEventRecord(e0);
        segment_kernel<<<grid, 32 * W, G::SMEM_BYTES>>>(maps, a, run == 1 ? 2 : 1, words + 1);
        cudaEventRecord(e1);
        if (cudaDeviceSynchronize() != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) return 2;
        cudaMemcpy(out, words, 8, cudaMemcpyDeviceToHost);
        cudaMemcpy(got.data(), up, 4 * n, cudaMemcpyDeviceToHost);
        std::printf("run %d: status %u, threads that were told %u, %.0f ms\n", run, out[0], out[1], ms);
        const unsigned threads = grid.x * grid.y * 32 * W;
        if (run == 1 && (out[0] != kStatusTimeout || out[1] != threads || ms < 900.0f || ms > 20000.0f)) return 3;
        if (run != 1 && (out[0] != 0 || out[1] != 0 || ms > 900.0f)) return 4;
        if (run == 0) first = got;
        if (run == 2 && std::memcmp(first.data(), got.data(), 4 * n) != 0) return 5;
        if (run == 0 && std::memcmp(h.data(), got.data(), 4 * n) == 0) return 6;
    }
    return 0;
}
"""


def test_a_segment_whose_waits_run_out_ends_and_says_so(tmp_path):
    (tmp_path / "t.cu").write_text(SRC)
    subprocess.run([build.nvcc(), str(tmp_path / "t.cu"), "-o", str(tmp_path / "t")] + build.NVCC_FLAGS, check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=120)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr
