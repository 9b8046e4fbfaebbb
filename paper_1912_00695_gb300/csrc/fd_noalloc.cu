// fd_forward_noalloc: time steps on caller-owned device buffers with no device
// allocation at all. The step kernel's scratch (the running maximum of |u| over
// the call) lives in one file-scope __device__ array instead of a cudaMalloc'd
// buffer; the caller passes every input and output.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <utility>

#include "../../include/fd_acoustic.h"
#include "fd_launch_count.h"
#include "fd_tma.cuh"

// sources this entry point accepts (its documented limit)
constexpr int kNoallocSources = 4;
// space orders this entry point accepts (its documented limit)
constexpr int kNoallocMaxRadius = 8;

namespace fdgb {
void set_last_error(const char *msg);  // fd_api.cu: the fd_last_error() text

namespace {

constexpr int kNoAllocMaxTiles = 16384;  // 8 x 32 tiles a y-z plane may hold (a documented limit)
constexpr int kNoAllocMaxDevices = 64;

// Scratch: word 0 = running max |u| (float bits) over the call's steps. Held by
// every GPU that loads the library until the process exits.
static __device__ __align__(256) unsigned g_noalloc_scratch[64];

std::mutex g_noalloc_mu;
unsigned *g_noalloc_ptr[kNoAllocMaxDevices] = {};
int g_noalloc_sms[kNoAllocMaxDevices] = {};  // multiprocessors of each device, read with its address

// Asynchronous copy of VEC floats (both sides aligned to them) into shared memory; zeros
// where !ok.
template <int VEC>
__device__ __forceinline__ void copy_async(uint32_t dst, const float *src, bool ok) {
    const int n = ok ? 4 * VEC : 0;
    if constexpr (VEC == 4)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(4 * VEC), "r"(n)
                     : "memory");
}

__device__ __forceinline__ float2 pair(float v) { return make_float2(v, v); }

// CTAs of the step kernel per multiprocessor. Above radius 5 four would leave 128 registers a
// thread and spills (one GB300, 186^3 damped, 150 steps: space order 12 69.9 us a step at four,
// 62.3 at three; 16 81.8 and 70.8)
constexpr int noalloc_ctas_per_sm(int r) { return r <= 5 ? 4 : 3; }

template <int R>
struct NoallocShape {
    static constexpr int TZ = 32, TY = 16, W = 4;  // tile: 8 x 4 threads of 4 z points per warp
    static constexpr int RZ = (R + 3) / 4 * 4;     // z halo: windows start 16-byte aligned
    static constexpr int SW = TZ + 2 * RZ, SH = TY + 2 * R;
    static constexpr int HALO = SW * SH, PT = TZ * TY;  // floats
    static constexpr int STAGE = HALO + 4 * PT;         // halo tile, front, u^{n-1}, m, eta
    static constexpr int S = 4;
    static constexpr int SMEM_BYTES = S * STAGE * 4;
};

// Streaming step (expanded form, FP32 storage, dense [Nx][Ny][Nz] layout): the
// schedule of the TMA step kernel (fd_tma.cuh: 4 z points per thread, x taps from
// a register queue, every input of a plane in a shared ring several planes
// ahead), with the planes fetched by cp.async in pieces of VEC floats instead of
// tensor copies, which need 16-byte row pitches that a caller's dense rows seldom
// have. VEC is the widest of 4, 2, 1 that divides Nz and the buffers' addresses.
// The per-point arithmetic is the expanded form's of the other kernels.
// Bound: instruction issue and latency at 12 to 16 warps per multiprocessor (the copies in
// pieces add to the arithmetic), not memory. It replaces one point per thread with halos
// staged through registers and a second launch per step for the maximum. Time a step,
// before -> now (one GB300, a damped 10-point layer on every side, 150 steps): 186^3 at
// space order 2 / 8 / 12 / 16 55.1 / 79.5 / 87.0 / 95.4 -> 35.4 / 45.2 / 62.1 / 70.7 us;
// 276^3 at 8 287 -> 106 us; 84^3 at 4 18.6 -> 10.3 us; rows of 16 / 4 bytes alignment
// (186 x 186 x 188 / 185 at 8) 80.3 / 78.4 -> 37.4 / 53.9 us. Without damping (no divisions)
// 186^3 at 8 65.7 -> 34.9 us, 276^3 279 -> 92.3 us.
template <int R, int VEC>
__global__ void __launch_bounds__(128, noalloc_ctas_per_sm(R)) noalloc_step_kernel(const StepArgs a, unsigned *scratch) {
    using G = NoallocShape<R>;
    constexpr int TZ = G::TZ, TY = G::TY, SW = G::SW, SH = G::SH, RZ = G::RZ, S = G::S, W = G::W;
    constexpr int U = TmaUnroll<R, kExpanded>::U, Q = 2 * R + U, NWIN = 4 + 2 * RZ;
    extern __shared__ __align__(16) float ring[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int lz = lane & 7, ty = warp * 4 + (lane >> 3);
    const int z0 = blockIdx.x * TZ, y0 = blockIdx.y * TY;
    const int z4 = z0 + 4 * lz, y = y0 + ty;
    const int xb = blockIdx.z * a.x_block, xe = min(xb + a.x_block, a.Nx);
    const bool own = y < a.Ny && z4 < a.Nz;
    const float *__restrict__ u = static_cast<const float *>(a.u);
    float *up = static_cast<float *>(a.up);
    const float *f1 = a.f1, *f2 = a.f2;
    const long long P = a.plane;
    const int Ny = a.Ny, Nz = a.Nz, Nx = a.Nx, pz = a.pz;
    const bool damped = f2 != nullptr;

    // Copies of plane x into its stage. Halo rows: row j of the tile by warp j mod 4, the
    // lanes along z. Point tiles: each warp its own four rows.
    auto issue = [&](int x, int stage) {
        float *st = ring + stage * G::STAGE;
        const uint32_t sb = smem_addr(st);
        const float *pu = u + x * P;
#pragma unroll
        for (int k = 0; k < (SH + W - 1) / W; ++k) {
            const int j = warp + k * W, yy = y0 - R + j;
            if (SH % W != 0 && j >= SH) break;
            const bool row = yy >= 0 && yy < Ny;
            const float *pr = pu + (long long)yy * pz;
#pragma unroll
            for (int c0 = 0; c0 < SW; c0 += 32 * VEC) {
                const int c = c0 + lane * VEC, zz = z0 - RZ + c;
                if (c < SW) {
                    const bool ok = row && zz >= 0 && zz < Nz;
                    copy_async<VEC>(sb + 4 * (j * SW + c), ok ? pr + zz : u, ok);
                }
            }
        }
        const bool front = x + R < Nx;
#pragma unroll
        for (int k = 0; k < 4 / VEC; ++k) {
            const int i = (k * 32 + lane) * VEC;  // element of the warp's 4 x 32 points
            const int yy = y0 + warp * 4 + i / TZ, zz = z0 + i % TZ;
            const bool ok = yy < Ny && zz < Nz;
            const long long o = ok ? (long long)yy * pz + zz : 0;
            const uint32_t d = sb + 4 * (G::HALO + warp * 4 * TZ + i);
            copy_async<VEC>(d, front ? pu + R * P + o : u, ok && front);
            copy_async<VEC>(d + 4 * G::PT, up + x * P + o, ok);
            copy_async<VEC>(d + 8 * G::PT, f1 + x * P + o, ok);
            if (damped) copy_async<VEC>(d + 12 * G::PT, f2 + x * P + o, ok);
        }
    };
#pragma unroll
    for (int s = 0; s < S - 1; ++s) {
        if (xb + s < xe) issue(xb + s, s);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }

    unsigned src_mask = 0;
    int src_p[kFusedSources];
#pragma unroll
    for (int s = 0; s < kFusedSources; ++s) {
        src_p[s] = 0;
        if (own && s < a.ns && a.sy[s] == y && a.sz[s] >= z4 && a.sz[s] < z4 + 4 && a.sx[s] >= xb && a.sx[s] < xe) {
            src_mask |= 1u << s;
            src_p[s] = a.sz[s] - z4;
        }
    }
    const unsigned in_row = own ? min(Nz - z4, 4) : 0;  // the thread's points inside the row
    const long long col = (long long)y * pz + z4;
    // VEC floats at a time between global memory and the thread's four points
    auto load4 = [&](const float *p) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (VEC == 4) {
            if (in_row) v = __ldg(reinterpret_cast<const float4 *>(p));
        } else if constexpr (VEC == 2) {
            if (in_row > 0) { const float2 t = __ldg(reinterpret_cast<const float2 *>(p)); v.x = t.x, v.y = t.y; }
            if (in_row > 2) { const float2 t = __ldg(reinterpret_cast<const float2 *>(p + 2)); v.z = t.x, v.w = t.y; }
        } else {
            if (in_row > 0) v.x = __ldg(p);
            if (in_row > 1) v.y = __ldg(p + 1);
            if (in_row > 2) v.z = __ldg(p + 2);
            if (in_row > 3) v.w = __ldg(p + 3);
        }
        return v;
    };
    auto store4 = [&](float *p, float4 v) {
        if constexpr (VEC == 4) {
            if (in_row) *reinterpret_cast<float4 *>(p) = v;
        } else if constexpr (VEC == 2) {
            if (in_row > 0) *reinterpret_cast<float2 *>(p) = make_float2(v.x, v.y);
            if (in_row > 2) *reinterpret_cast<float2 *>(p + 2) = make_float2(v.z, v.w);
        } else {
            if (in_row > 0) p[0] = v.x;
            if (in_row > 1) p[1] = v.y;
            if (in_row > 2) p[2] = v.z;
            if (in_row > 3) p[3] = v.w;
        }
    };
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 q[Q];
#pragma unroll
    for (int k = 0; k < 2 * R; ++k) {
        const int x = xb - R + k;
        q[k] = x >= 0 && x < Nx ? load4(u + x * P + col) : zero4;
    }
    float cj[R + 1];
#pragma unroll
    for (int j = 1; j <= R; ++j) cj[j] = a.coef[j];
    const float half_dt = a.half_dt, dt2 = a.dt2;
    unsigned amax_bits = 0;
    int stage = 0;

    for (int xo = xb; xo < xe; xo += U) {
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int x = xo + i;
            if (x >= xe) break;
            asm volatile("cp.async.wait_group %0;" ::"n"(S - 2) : "memory");
            __syncthreads();  // plane x has landed for every thread; plane x - 1 is read
            if (x + S - 1 < xe) issue(x + S - 1, stage == 0 ? S - 1 : stage - 1);
            asm volatile("cp.async.commit_group;" ::: "memory");
            const float *st = ring + stage * G::STAGE;
            const float *pt = st + G::HALO + ty * TZ + 4 * lz;
            if (++stage == S) stage = 0;
            q[2 * R + i] = *reinterpret_cast<const float4 *>(pt);
            if (!own) continue;
            const float4 um = *reinterpret_cast<const float4 *>(pt + G::PT);
            const float4 cm = *reinterpret_cast<const float4 *>(pt + 2 * G::PT);
            const float4 ce = damped ? *reinterpret_cast<const float4 *>(pt + 3 * G::PT) : zero4;
            const float *rowp = st + (ty + R) * SW + 4 * lz;
            float win[NWIN];
#pragma unroll
            for (int m = 0; m < NWIN / 4; ++m) {
                // (the window's middle is the thread's own points)
                const float4 v = 4 * m == RZ ? q[R + i] : *reinterpret_cast<const float4 *>(rowp + 4 * m);
                win[4 * m] = v.x, win[4 * m + 1] = v.y, win[4 * m + 2] = v.z, win[4 * m + 3] = v.w;
            }
            const float2 hdt = pair(half_dt), ucA = lo2(q[R + i]), ucB = hi2(q[R + i]);
            const float2 r0A = fma2(hdt, lo2(ce), lo2(cm)), r0B = fma2(hdt, hi2(ce), hi2(cm));
            const float2 invA = make_float2(expanded_inv(r0A.x), expanded_inv(r0A.y));
            const float2 invB = make_float2(expanded_inv(r0B.x), expanded_inv(r0B.y));
            float2 lapA = pair(0.f), lapB = pair(0.f);
#pragma unroll
            for (int j = 1; j <= R; ++j) {
                const float4 xm = q[R + i - j], xp = q[R + i + j];
                const float4 ym = *reinterpret_cast<const float4 *>(rowp + RZ - j * SW);
                const float4 yp = *reinterpret_cast<const float4 *>(rowp + RZ + j * SW);
                const float2 cA = mul2(pair(cj[j]), invA), cB = mul2(pair(cj[j]), invB);
                lapA = fma2(cA, sub2(lo2(xm), ucA), lapA);
                lapA = fma2(cA, sub2(lo2(xp), ucA), lapA);
                lapA = fma2(cA, sub2(lo2(ym), ucA), lapA);
                lapA = fma2(cA, sub2(lo2(yp), ucA), lapA);
                lapA = fma2(cA, zdiff_pair<RZ>(win, -j, ucA), lapA);
                lapA = fma2(cA, zdiff_pair<RZ>(win, j, ucA), lapA);
                lapB = fma2(cB, sub2(hi2(xm), ucB), lapB);
                lapB = fma2(cB, sub2(hi2(xp), ucB), lapB);
                lapB = fma2(cB, sub2(hi2(ym), ucB), lapB);
                lapB = fma2(cB, sub2(hi2(yp), ucB), lapB);
                lapB = fma2(cB, zdiff_pair<RZ + 2>(win, -j, ucB), lapB);
                lapB = fma2(cB, zdiff_pair<RZ + 2>(win, j, ucB), lapB);
            }
            // u+ = L + (2a) u + (1 - 2a) u-, a = m / r0 correctly rounded: exactly 1 without damping
            float2 vA, vB;
            if (ce.x == 0.f && ce.y == 0.f && ce.z == 0.f && ce.w == 0.f) {
                vA = fma2(pair(-1.f), lo2(um), fma2(pair(2.f), ucA, lapA));
                vB = fma2(pair(-1.f), hi2(um), fma2(pair(2.f), ucB, lapB));
            } else {
                const float am[4] = {__fdiv_rn(cm.x, r0A.x), __fdiv_rn(cm.y, r0A.y), __fdiv_rn(cm.z, r0B.x),
                                     __fdiv_rn(cm.w, r0B.y)};
                vA = fma2(make_float2(1.0f - 2.0f * am[0], 1.0f - 2.0f * am[1]), lo2(um),
                          fma2(make_float2(2.0f * am[0], 2.0f * am[1]), ucA, lapA));
                vB = fma2(make_float2(1.0f - 2.0f * am[2], 1.0f - 2.0f * am[3]), hi2(um),
                          fma2(make_float2(2.0f * am[2], 2.0f * am[3]), ucB, lapB));
            }
            float4 o = make_float4(vA.x, vA.y, vB.x, vB.y);
            if (src_mask) {
#pragma unroll
                for (int s = 0; s < kFusedSources; ++s)
                    if (((src_mask >> s) & 1u) && a.sx[s] == x) {
                        const float qv = source_value(a, s);
                        if (src_p[s] == 0) o.x = fmaf(dt2 * invA.x, qv, o.x);
                        if (src_p[s] == 1) o.y = fmaf(dt2 * invA.y, qv, o.y);
                        if (src_p[s] == 2) o.z = fmaf(dt2 * invB.x, qv, o.z);
                        if (src_p[s] == 3) o.w = fmaf(dt2 * invB.y, qv, o.w);
                    }
            }
            amax_bits = max(amax_bits, __float_as_uint(fabsf(o.x)));
            if (in_row > 1) amax_bits = max(amax_bits, __float_as_uint(fabsf(o.y)));
            if (in_row > 2) amax_bits = max(amax_bits, __float_as_uint(fabsf(o.z)));
            if (in_row > 3) amax_bits = max(amax_bits, __float_as_uint(fabsf(o.w)));
            store4(up + x * P + col, o);
        }
#pragma unroll
        for (int k = 0; k < 2 * R; ++k) q[k] = q[k + U];
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax_bits = max(amax_bits, __shfl_xor_sync(0xffffffffu, amax_bits, o));
    if (lane == 0) atomicMax(scratch, amax_bits);  // float bits: NaN above Inf above finite
}

__global__ void noalloc_clear_kernel(unsigned *scratch) {
    if (threadIdx.x == 0) scratch[0] = 0u;
}

template <int R, int VEC>
cudaError_t launch_noalloc_v(const StepArgs &a, unsigned *scratch, int dev, cudaStream_t s) {
    using G = NoallocShape<R>;
    static std::atomic<unsigned long long> attr_set{0};  // bit per device
    static_assert(kNoAllocMaxDevices <= 64, "one bit per device");
    if (!((attr_set.load(std::memory_order_relaxed) >> dev) & 1u)) {
        const cudaError_t e = cudaFuncSetAttribute(noalloc_step_kernel<R, VEC>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM_BYTES);
        if (e != cudaSuccess) return e;
        attr_set.fetch_or(1ull << dev, std::memory_order_relaxed);
    }
    const dim3 grid((a.Nz + G::TZ - 1) / G::TZ, (a.Ny + G::TY - 1) / G::TY, (a.Nx + a.x_block - 1) / a.x_block);
    noalloc_step_kernel<R, VEC><<<grid, 128, G::SMEM_BYTES, s>>>(a, scratch);
    return counted(cudaGetLastError(), s);
}

template <int R>
cudaError_t launch_noalloc(const StepArgs &a, int vec, unsigned *scratch, int dev, cudaStream_t s) {
    return vec == 4 ? launch_noalloc_v<R, 4>(a, scratch, dev, s)
                    : vec == 2 ? launch_noalloc_v<R, 2>(a, scratch, dev, s)
                               : launch_noalloc_v<R, 1>(a, scratch, dev, s);
}

cudaError_t launch_noalloc_r(int r, const StepArgs &a, int vec, unsigned *scratch, int dev, cudaStream_t s) {
    switch (r) {
        case 1: return launch_noalloc<1>(a, vec, scratch, dev, s);
        case 2: return launch_noalloc<2>(a, vec, scratch, dev, s);
        case 3: return launch_noalloc<3>(a, vec, scratch, dev, s);
        case 4: return launch_noalloc<4>(a, vec, scratch, dev, s);
        case 5: return launch_noalloc<5>(a, vec, scratch, dev, s);
        case 6: return launch_noalloc<6>(a, vec, scratch, dev, s);
        case 7: return launch_noalloc<7>(a, vec, scratch, dev, s);
        case 8: return launch_noalloc<8>(a, vec, scratch, dev, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace
}  // namespace fdgb

using namespace fdgb;

extern "C" int fd_forward_noalloc(float *d_u, float *d_u_prev, const float *d_m, const float *d_eta,
                                  int Nx, int Ny, int Nz, int space_order, double h, double dt, int ns,
                                  const int *src_xyz, const float *d_wavelet, int ld, long long step0,
                                  int nt, void *stream, float *amax_out) {
    char msg[256];
    auto fail = [&](int code, const char *text) {
        std::snprintf(msg, sizeof msg, "fd_forward_noalloc: %s", text);
        fdgb::set_last_error(msg);
        return code;
    };
    if (!d_u || !d_u_prev || !d_m) return fail(FD_EINVAL, "u, u_prev and m must be device pointers");
    if (Nx < 1 || Ny < 1 || Nz < 1 || Nx > kMaxDim || Ny > kMaxDim || Nz > kMaxDim)
        return fail(FD_EINVAL, "extents must be in [1, 65535]");
    // the library's weight generator (Fornberg's recursion on fixed-size arrays: no heap use)
    double c[kMaxRadiusHost + 1];
    if (space_order > 2 * kNoallocMaxRadius || !fornberg_second_derivative(space_order, c))
        return fail(FD_EINVAL, "space_order must be even in [2, 16]");
    if (!(h > 0) || !std::isfinite(h) || !(dt > 0) || !std::isfinite(dt))
        return fail(FD_EINVAL, "h and dt must be positive and finite");
    if (ns < 0 || ns > kNoallocSources) return fail(FD_EINVAL, "ns must be in [0, 4]");
    if (ns > 0 && (!src_xyz || !d_wavelet || ld < 1)) return fail(FD_EINVAL, "sources need src_xyz, wavelet, ld >= 1");
    if (nt < 0 || step0 < 0) return fail(FD_EINVAL, "nt and step0 must be >= 0");
    const int r = space_order / 2;
    const int tiles_z = (Nz + kTileZ - 1) / kTileZ;
    if ((long long)tiles_z * ((Ny + 7) / 8) > kNoAllocMaxTiles)
        return fail(FD_EINVAL, "Ny*Nz too large: a y-z plane may hold at most 16384 tiles of 8 x 32 points");
    // per-device set-up: the address of this device's copy of the scratch array
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices)
        return fail(FD_ECUDA, "no usable current device");
    unsigned *scratch = nullptr;
    int sms = 0;
    {
        std::lock_guard<std::mutex> lk(g_noalloc_mu);
        if (!g_noalloc_ptr[dev]) {
            void *p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess) return fail(FD_ECUDA, cudaGetErrorString(e));
            int n_sm = 0;
            e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess) return fail(FD_ECUDA, cudaGetErrorString(e));
            g_noalloc_sms[dev] = n_sm > 0 ? n_sm : 1;
            g_noalloc_ptr[dev] = static_cast<unsigned *>(p);
        }
        scratch = g_noalloc_ptr[dev];
        sms = g_noalloc_sms[dev];
    }
    // x-chunks: as many as fill the resident CTA slots once, and no longer than 24 planes
    // (276^3 damped, space order 8: one wave of 92-plane chunks 124.3 us a step, this rule's 23
    // planes 105.9, 24 planes 100.5, 12 planes 104.6), but none shorter than 8 unless the domain
    // is: a chunk also loads its 2r neighbouring planes
    const long long tiles = (long long)tiles_z * ((Ny + 15) / 16);
    const long long slots = (long long)noalloc_ctas_per_sm(r) * sms;
    const long long chunks = std::max<long long>(
        1, std::min<long long>(std::max<long long>(slots / tiles, (Nx + 23) / 24), Nx / 8));
    const int x_block = int((Nx + chunks - 1) / chunks);
    // the widest copies that the rows and the buffers allow
    const uintptr_t at = reinterpret_cast<uintptr_t>(d_u) | reinterpret_cast<uintptr_t>(d_u_prev) |
                         reinterpret_cast<uintptr_t>(d_m) | reinterpret_cast<uintptr_t>(d_eta) | uintptr_t(4) * Nz;
    const int vec = at % 16 == 0 ? 4 : at % 8 == 0 ? 2 : 1;

    StepArgs a{};
    a.f1 = d_m;
    a.f2 = d_eta;
    a.Nx = Nx;
    a.Ny = Ny;
    a.Nz = Nz;
    a.pz = Nz;
    a.plane = (long long)Ny * Nz;
    a.x_block = x_block;
    const double scale = dt * dt / (h * h);
    for (int j = 1; j <= r; ++j) a.coef[j] = float(c[j] * scale);
    a.half_dt = float(0.5 * dt);
    a.dt2 = float(dt * dt);
    a.ns = ns;
    for (int s = 0; s < ns; ++s) {
        const int x = src_xyz[3 * s], y = src_xyz[3 * s + 1], z = src_xyz[3 * s + 2];
        if (x < 0 || x >= Nx || y < 0 || y >= Ny || z < 0 || z >= Nz)
            return fail(FD_ERANGE, "source node outside the domain");
        a.sx[s] = x;
        a.sy[s] = y;
        a.sz[s] = z;
    }
    a.wavelet = d_wavelet;
    a.ld = ld;

    cudaStream_t s = static_cast<cudaStream_t>(stream);
    noalloc_clear_kernel<<<1, 32, 0, s>>>(scratch);
    cudaError_t e = counted(cudaGetLastError(), s);
    float *cur = d_u, *prev = d_u_prev;
    for (int i = 0; i < nt && e == cudaSuccess; ++i) {
        a.u = cur;
        a.up = prev;
        a.step = step0 + i;
        e = launch_noalloc_r(r, a, vec, scratch, dev, s);
        std::swap(cur, prev);
    }
    if (e != cudaSuccess) return fail(FD_ECUDA, cudaGetErrorString(e));
    if (amax_out) {
        unsigned bits = 0;
        e = cudaMemcpyAsync(&bits, scratch, sizeof bits, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return fail(FD_ECUDA, cudaGetErrorString(e));
        float v;
        std::memcpy(&v, &bits, sizeof v);
        *amax_out = v;
        if (bits >= 0x7f800000u) return fail(FD_ENONFINITE, "wavefield reached NaN/Inf");
    }
    return FD_OK;
}
