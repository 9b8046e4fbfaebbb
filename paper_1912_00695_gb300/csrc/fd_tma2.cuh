// Two time steps per launch (temporal blocking along the streaming direction),
// FP32 storage, factored form, stencil radius R <= 2. Included by the radius-1
// and radius-2 translation units after fd_tma.cuh.
//
// Schedule. A CTA of 256 threads owns an extended y-z tile E of 64 (z) x 16 (y)
// points and its interior T (z in [4, 60), y in [R, 16 - R)); neighbouring
// CTAs' extended tiles overlap by their halos. Marching x over the chunk's
// planes extended by R on both sides, at step-1 plane x every thread
//  * computes u^{n+1}(x) at its 4 points of E from u^n (register queue for the
//    x taps, the TMA-fed halo box for y and z, exactly the single-step
//    kernel's per-point arithmetic) and puts it in a shared ring of
//    u^{n+1} planes (zero outside the domain: the Dirichlet halo of u^{n+1});
//    points of T inside [xb, xe) are also stored to global memory (u^{n+1});
//  * after a CTA barrier, computes u^{n+2}(x - R) at its points of T from the
//    u^{n+1} ring (y and z taps; the x taps are the thread's own results, at R = 1
//    kept in registers), u^n(x - R) (the oldest queue entry), and
//    w, g of plane x - R (a register queue of R+1 planes), and stores it.
// Per pair of steps HBM sees u^n, u^{n-1}, w (g in the layer) read and
// u^{n+1}, u^{n+2} written: 20 B per point (plus g in the layer) instead of 32
// for two single steps (halo and overlap re-reads come from L2). The extended tile costs
// 64x16 / (56 x (16-2R)) more first-step work. Outputs go to two other
// buffers: u^{n+1} cannot overwrite u^{n-1}, which overlapping CTAs still read.
// Sources of both steps are fused; receivers and the other storages are not
// supported here.
// Bound: latency at 16 warps per SM (two CTAs; shared memory and registers allow no third)
// and two CTA barriers per plane, well above the HBM time of its 10.4 B per point and
// step. The barriers carry no vote, the sources sit out of line, the L2 prefetches are
// issued by a second warp, and four stages are in flight: 276^3, space order 2, 300 steps,
// one GB300 407 -> 463 Gpts/s (three stages and ring x taps: 442); 84^3 115 -> 144;
// 343 x 220 x 350 385 -> 460.
#pragma once

#include "fd_tma.cuh"

namespace fdgb {

template <int R>
struct Tb2Shape {
    static_assert(R >= 1 && R <= 2, "two-step kernel: radius 1 or 2");
    static constexpr int EZ = 64, EY = 16;   // extended tile (z points, y rows)
    static constexpr int HZ = 4;             // z halo of E around T, and of u^n around E (>= R, 16 B)
    static constexpr int TZ = EZ - 2 * HZ;   // 56 output points along z
    static constexpr int TY = EY - 2 * R;    // output rows along y
    static constexpr int SW = EZ + 2 * HZ;   // u^n box width
    static constexpr int SH = EY + 2 * R;    // u^n box height
    static constexpr int HALO_RAW = SW * SH * 4;
    static constexpr int PT_RAW = EZ * EY * 4;
    static constexpr int HALO = (HALO_RAW + 127) / 128 * 128;
    static constexpr int OFF_FRONT = HALO, OFF_UP = HALO + PT_RAW, OFF_F1 = HALO + 2 * PT_RAW,
                         OFF_F2 = HALO + 3 * PT_RAW;
    static constexpr int STAGE_BYTES = HALO + 4 * PT_RAW;
    static constexpr int STAGES = 4;
    // The second step's x taps are the thread's own earlier results: at R = 1 they stay in
    // registers and the ring holds the planes that the y and z taps still read (at R = 2 the
    // registers are worth more: 359.7 against 355.9 Gpts/s at 276^3, space order 4)
    static constexpr bool OWN_X = R == 1;
    static constexpr int NU1 = OWN_X ? R + 1 : 2 * R + 1;  // u^{n+1} planes in the ring
    static constexpr int U1_OFF = STAGES * STAGE_BYTES;
    static constexpr int BAR_OFF = U1_OFF + NU1 * PT_RAW;
    static constexpr int SMEM_BYTES = BAR_OFF + 64 + 128;
    static constexpr int THREADS = 256;
    static constexpr int U = R + 1;  // x unroll: the w/g delay queue indexes statically
};

// Factored FP32 update of 4 points (the single-step kernel's association order):
// L = sum_j c_j ((xm+xp + ym+yp) + z pair - 6 u_c); u+ = w L + (2u - u-) - 2 g (u - u-).
// XT(j, m, p) gives the x taps (m = minus side) as float4; YP(j) the y rows' window
// base (y - j and y + j rows at offsets -j*SW, +j*SW of `rowp`).
template <int R, int RZ, int SWROW, typename XT>
__device__ __forceinline__ float4 tb2_update(const float *rowp, const float *win, XT xtap, float4 uc, float4 cum,
                                             float4 cf1, float4 cf2, const float2 *cz2) {
    float2 lapA = f2(0.f, 0.f), lapB = f2(0.f, 0.f);
    const float2 nsixA = mul2(f2(-6.f, -6.f), lo2(uc)), nsixB = mul2(f2(-6.f, -6.f), hi2(uc));
#pragma unroll
    for (int j = 1; j <= R; ++j) {
        const float4 ym = *reinterpret_cast<const float4 *>(rowp + RZ - j * SWROW);
        const float4 yp = *reinterpret_cast<const float4 *>(rowp + RZ + j * SWROW);
        const float4 xm = xtap(j, true), xp = xtap(j, false);
        const float2 sA = add2(add2(add2(lo2(xm), lo2(xp)), add2(lo2(ym), lo2(yp))), ztap_pair<RZ>(win, j));
        const float2 sB = add2(add2(add2(hi2(xm), hi2(xp)), add2(hi2(ym), hi2(yp))), ztap_pair<RZ + 2>(win, j));
        lapA = fma2(cz2[j], add2(sA, nsixA), lapA);
        lapB = fma2(cz2[j], add2(sB, nsixB), lapB);
    }
    const float2 ucA = lo2(uc), ucB = hi2(uc), umA = lo2(cum), umB = hi2(cum);
    const float2 m2gA = mul2(f2(-2.f, -2.f), lo2(cf2)), m2gB = mul2(f2(-2.f, -2.f), hi2(cf2));
    const float2 dA = fma2(f2(-1.f, -1.f), umA, ucA), dB = fma2(f2(-1.f, -1.f), umB, ucB);
    float2 vA = fma2(lo2(cf1), lapA, add2(ucA, dA));
    float2 vB = fma2(hi2(cf1), lapB, add2(ucB, dB));
    vA = fma2(m2gA, dA, vA);
    vB = fma2(m2gB, dB, vB);
    return make_float4(vA.x, vA.y, vB.x, vB.y);
}

// u^{n+1} into out1 and u^{n+2} into out2 from u^n = a.u, u^{n-1} = a.up (read
// through `maps`), global step n = a.step. CTA (bz, by, bx): T origin
// (bz*56, by*(16-2R)), planes [bx x_block, (bx+1) x_block).
template <int R>
__global__ void __launch_bounds__(256, 2) fd_tma2_kernel(const __grid_constant__ TmaMaps maps, const __grid_constant__ StepArgs a,
                                                          float *out1, float *out2, int check) {
    using G = Tb2Shape<R>;
    constexpr int S = G::STAGES, U = G::U, Q = 2 * R + U, NWIN = 4 + 2 * G::HZ, EZ = G::EZ, SW = G::SW;
    extern __shared__ __align__(128) unsigned char smem_dyn[];
    // aligned by pointer arithmetic on the shared array (keeps its address space)
    unsigned char *ring = smem_dyn + ((128u - (smem_addr(smem_dyn) & 127u)) & 127u);
    float *u1ring = reinterpret_cast<float *>(ring + G::U1_OFF);
    uint64_t *bars = reinterpret_cast<uint64_t *>(ring + G::BAR_OFF);

    const int tid = threadIdx.x;
    const int lz = tid & 15, ty = tid >> 4;
    const int zt0 = blockIdx.x * G::TZ, yt0 = blockIdx.y * G::TY;
    const int ze0 = zt0 - G::HZ, ye0 = yt0 - R;  // E origin
    const int z4 = ze0 + 4 * lz, y = ye0 + ty;
    const bool dom = y >= 0 && y < a.Ny && z4 >= 0 && z4 < a.Nz;
    const bool inT = lz >= 1 && lz <= 14 && ty >= R && ty < G::EY - R;
    const int xb = blockIdx.z * a.x_block, xe = min(xb + a.x_block, a.Nx);
    const int xs = xb - R, xend = xe + R;  // first-step planes
    const long long P = a.plane;
    const long long col = (long long)y * a.pz + z4;
    const float *u = static_cast<const float *>(a.u) + col;
    float *o1 = out1 + col, *o2 = out2 + col;

    if (tid == 0) {
        for (int s = 0; s < S; ++s) mbar_init(smem_addr(&bars[s]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    wait_previous_launch();
    // the extended tile lies where the damping field vanishes (in y and z)
    const bool tile_yz_box = ye0 >= a.by0 && ye0 + G::EY <= a.by1 && ze0 >= a.bz0 && ze0 + EZ <= a.bz1;
    auto g_free = [&](int x) { return tile_yz_box && x >= a.bx0 && x < a.bx1; };
    auto issue = [&](int x, int stage) {
        const uint32_t bar = smem_addr(&bars[stage]);
        unsigned char *st = ring + stage * G::STAGE_BYTES;
        const bool need_g = !g_free(x);
        mbar_expect_tx(bar, uint32_t(G::HALO_RAW + (need_g ? 4 : 3) * G::PT_RAW));
        tma_load_3d(smem_addr(st), &maps.u_halo, bar, ze0 - G::HZ, ye0 - R, x);
        tma_load_3d(smem_addr(st + G::OFF_FRONT), &maps.u_pt, bar, ze0, ye0, x + R);
        tma_load_3d(smem_addr(st + G::OFF_UP), &maps.up_pt, bar, ze0, ye0, x);
        tma_load_3d(smem_addr(st + G::OFF_F1), &maps.f1_pt, bar, ze0, ye0, x);
        if (need_g) tma_load_3d(smem_addr(st + G::OFF_F2), &maps.f2_pt, bar, ze0, ye0, x);
    };
    // the same boxes of plane x into L2, further ahead
    auto prefetch = [&](int x) {
        if (x < xend) {
            tma_prefetch_3d(&maps.up_pt, ze0, ye0, x);
            tma_prefetch_3d(&maps.f1_pt, ze0, ye0, x);
            if (!g_free(x)) tma_prefetch_3d(&maps.f2_pt, ze0, ye0, x);
            if (x + R < a.Nx) tma_prefetch_3d(&maps.u_pt, ze0, ye0, x + R);
        }
    };
    const int n_planes = xend - xs;
    if (tid == 0)
        for (int s = 0; s < S - 1 && s < n_planes; ++s) issue(xs + s, s);

    // planes on which E has a fused source: [src_lo, src_hi] (empty for nearly every tile)
    int src_lo = a.Nx, src_hi = -1;
#pragma unroll
    for (int s = 0; s < kFusedSources; ++s)
        if (s < a.ns && a.sy[s] >= ye0 && a.sy[s] < ye0 + G::EY && a.sz[s] >= ze0 && a.sz[s] < ze0 + EZ) {
            src_lo = min(src_lo, a.sx[s]);
            src_hi = max(src_hi, a.sx[s]);
        }

    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    auto load_u = [&](int x) -> float4 {
        return (dom && x >= 0 && x < a.Nx) ? __ldg(reinterpret_cast<const float4 *>(u + x * P)) : zero4;
    };
    float4 q[Q];  // u^n at planes xo - R .. xo + R + U - 1 (xo: first plane of the unrolled group)
#pragma unroll
    for (int k = 0; k < 2 * R; ++k) q[k] = load_u(xs - R + k);
    float4 wq[U], gq[U];  // w, g of the last R+1 planes (slot = plane offset within the group)
#pragma unroll
    for (int k = 0; k < U; ++k) wq[k] = gq[k] = zero4;
    float2 cz2[R + 1];
#pragma unroll
    for (int j = 1; j <= R; ++j) cz2[j] = f2(a.coef[j], a.coef[j]);
    const int pt_off = ty * EZ + 4 * lz;  // this thread's 4 points in an E plane
    float4 u1q[2 * R + 1];  // OWN_X: the thread's u^{n+1} at planes x - 2R .. x
#pragma unroll
    for (int k = 0; k <= 2 * R; ++k) u1q[k] = zero4;
    float2 nonfinite = f2(0.f, 0.f);
    // false once this thread's wait has given up: it then runs on without waiting or issuing,
    // and the results are void (as in tma_segment)
    bool alive = true;
    int issued = min(S - 1, n_planes), it_failed = 0;
    // ring planes of u^{n+1}: the slots of planes x - NU1 + 1 .. x, rotated once per plane
    float *u1p[G::NU1];
#pragma unroll
    for (int k = 0; k < G::NU1; ++k) u1p[k] = u1ring + k * (EZ * G::EY);
    int stage = 0;
    uint32_t phase = 0;

    for (int xo = xs; xo < xend; xo += U) {
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int x = xo + i;
            if (x >= xend) break;
            const int it = x - xs;
            if (!mbar_try_wait(smem_addr(&bars[stage]), phase))
                if (alive && !mbar_wait_slow(smem_addr(&bars[stage]), phase)) {
                    alive = false;
                    it_failed = it;
                }
            __syncthreads();
            if (tid == 0 && alive && x + S - 1 < xend) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                issue(x + S - 1, stage == 0 ? S - 1 : stage - 1);
                ++issued;
            }
            if (tid == 32) prefetch(x + 1 + kPrefetchAhead);
            const unsigned char *st = ring + stage * G::STAGE_BYTES;
            q[2 * R + i] = *reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(st + G::OFF_FRONT) + pt_off);
            // ---- step 1: u^{n+1}(x) at this thread's points of E
            float4 u1 = zero4;
            const float4 cf1 = *reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(st + G::OFF_F1) + pt_off);
            const float4 cf2 = g_free(x) ? zero4
                                         : *reinterpret_cast<const float4 *>(
                                               reinterpret_cast<const float *>(st + G::OFF_F2) + pt_off);
            wq[i] = cf1;
            gq[i] = cf2;
            if (dom && x >= 0 && x < a.Nx) {
                const float4 cum = *reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(st + G::OFF_UP) + pt_off);
                const float *rowp = reinterpret_cast<const float *>(st) + (ty + R) * SW + 4 * lz;
                float win[NWIN];
#pragma unroll
                for (int m = 0; m < NWIN / 4; ++m) {
                    // (the window's middle is the thread's own points)
                    const float4 v = 4 * m == G::HZ ? q[R + i] : *reinterpret_cast<const float4 *>(rowp + 4 * m);
                    win[4 * m] = v.x;
                    win[4 * m + 1] = v.y;
                    win[4 * m + 2] = v.z;
                    win[4 * m + 3] = v.w;
                }
                u1 = tb2_update<R, G::HZ, SW>(rowp, win, [&](int j, bool minus) { return minus ? q[R + i - j] : q[R + i + j]; },
                                             q[R + i], cum, cf1, cf2, cz2);
                if (x >= src_lo && x <= src_hi)
                    u1 = tma_add_sources<kFactored>(a, u1, x, y, z4, a.step,
                                                    reinterpret_cast<const float *>(st + G::OFF_F1) + pt_off, nullptr,
                                                    1.0f);
                if (z4 + 3 >= a.Nz) {  // beyond the row's end: zero (the Dirichlet halo and the pitch padding)
                    if (z4 + 1 >= a.Nz) u1.y = 0.f;
                    if (z4 + 2 >= a.Nz) u1.z = 0.f;
                    if (z4 + 3 >= a.Nz) u1.w = 0.f;
                }
                if (inT && x >= xb && x < xe) *reinterpret_cast<float4 *>(o1 + x * P) = u1;
            }
            *reinterpret_cast<float4 *>(u1p[G::NU1 - 1] + pt_off) = u1;
            if constexpr (G::OWN_X) u1q[2 * R] = u1;
            __syncthreads();  // the ring's plane x is complete
            // ---- step 2: u^{n+2}(x - R) at this thread's points of T
            const int x2 = x - R;
            if (inT && dom && x2 >= xb && x2 < xe) {
                const float *plane_c = u1p[G::NU1 - 1 - R];  // plane x - R
                float4 uc;
                if constexpr (G::OWN_X) uc = u1q[R];
                else uc = *reinterpret_cast<const float4 *>(plane_c + pt_off);
                const float *rowp = plane_c + ty * EZ + 4 * lz - G::HZ;  // z window from 4 points before
                float win[NWIN];
#pragma unroll
                for (int m = 0; m < NWIN / 4; ++m) {
                    const float4 v = 4 * m == G::HZ ? uc : *reinterpret_cast<const float4 *>(rowp + 4 * m);
                    win[4 * m] = v.x;
                    win[4 * m + 1] = v.y;
                    win[4 * m + 2] = v.z;
                    win[4 * m + 3] = v.w;
                }
                auto xtap = [&](int j, bool minus) {
                    if constexpr (G::OWN_X) return u1q[minus ? R - j : R + j];
                    else return *reinterpret_cast<const float4 *>(u1p[minus ? R - j : R + j] + pt_off);
                };
                const float4 w2 = wq[(i + 1) % U], g2 = gq[(i + 1) % U];  // plane x - R
                float4 u2 = tb2_update<R, G::HZ, EZ>(rowp, win, xtap, uc, q[i], w2, g2, cz2);
                if (x2 >= src_lo && x2 <= src_hi) {
                    const float w4[4] = {w2.x, w2.y, w2.z, w2.w};
                    u2 = tma_add_sources<kFactored>(a, u2, x2, y, z4, a.step + 1, w4, nullptr, 1.0f);
                }
                if (z4 + 3 >= a.Nz) {
                    if (z4 + 1 >= a.Nz) u2.y = 0.f;
                    if (z4 + 2 >= a.Nz) u2.z = 0.f;
                    if (z4 + 3 >= a.Nz) u2.w = 0.f;
                }
                // x * 0 is 0 for finite x and NaN otherwise
                nonfinite = fma2(lo2(u2), f2(0.f, 0.f), nonfinite);
                nonfinite = fma2(hi2(u2), f2(0.f, 0.f), nonfinite);
                *reinterpret_cast<float4 *>(o2 + x2 * P) = u2;
            }
            {
                float *oldest = u1p[0];  // the next plane takes the oldest one's slot
#pragma unroll
                for (int k = 0; k < G::NU1 - 1; ++k) u1p[k] = u1p[k + 1];
                u1p[G::NU1 - 1] = oldest;
            }
            if constexpr (G::OWN_X) {
#pragma unroll
                for (int k = 0; k < 2 * R; ++k) u1q[k] = u1q[k + 1];
            }
            if (++stage == S) {
                stage = 0;
                phase ^= 1u;
            }
        }
#pragma unroll
        for (int k = 0; k < 2 * R; ++k) q[k] = q[k + U];
    }
    if (__syncthreads_or(!alive)) {
        if (tid == 0) {
            if (a.status) atomicOr(a.status, kStatusTimeout);
            if (alive) it_failed = issued;  // this thread has waited for every copy it issued
            for (int it = it_failed; it < issued; ++it) mbar_wait_bounded(smem_addr(&bars[it % S]), uint32_t(it / S) & 1u);
        }
        return;
    }
    // as bits: NaN sorts above every finite magnitude (the status test)
    if (check) reduce_amax(a, nonfinite.x == 0.f && nonfinite.y == 0.f ? 0u : 0x7fc00000u, false);
}

template <int R>
cudaError_t tma2_launch(const TmaMaps &maps, const StepArgs &a, float *out1, float *out2, bool check,
                        cudaStream_t s) {
    using G = Tb2Shape<R>;
    auto kernel = fd_tma2_kernel<R>;
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM_BYTES);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const dim3 grid((a.Nz + G::TZ - 1) / G::TZ, (a.Ny + G::TY - 1) / G::TY, (a.Nx + a.x_block - 1) / a.x_block);
    return launch_step(kernel, grid, G::THREADS, G::SMEM_BYTES, true, s, maps, a, out1, out2, check ? 1 : 0);
}

}  // namespace fdgb

#define FDGB_INSTANTIATE_TMA2_RADIUS(R)                                                           \
    namespace fdgb {                                                                              \
    cudaError_t tma2_step_radius_##R(const TmaMaps &map, const StepArgs &a, float *out1, float *out2, \
                                     bool check, cudaStream_t s) {                                \
        return tma2_launch<R>(map, a, out1, out2, check, s);                                      \
    }                                                                                             \
    void tma2_geometry_radius_##R(int *tz, int *ty, int *box_w, int *box_h, int *ez, int *ey) {   \
        *tz = Tb2Shape<R>::TZ;                                                                    \
        *ty = Tb2Shape<R>::TY;                                                                    \
        *box_w = Tb2Shape<R>::SW;                                                                 \
        *box_h = Tb2Shape<R>::SH;                                                                 \
        *ez = Tb2Shape<R>::EZ;                                                                    \
        *ey = Tb2Shape<R>::EY;                                                                    \
    }                                                                                             \
    }
