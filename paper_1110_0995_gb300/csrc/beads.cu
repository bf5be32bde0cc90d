// Magnetic bead assembly (Sec. 2.5): the dipole-dipole force between beads,
// a harmonic contact force, and overdamped bead motion, all pairs on the GPU.
//
// One launch per step.  A block takes BEAD_TILE beads, one per thread, and a
// share of the partners: it stages their positions and moments in shared
// memory as pairs and evaluates two partners at a time with packed FP32
// (add / mul / fma.f32x2), then writes its partial forces.  The last block of a
// tile to finish adds the tile's partials in a fixed order and moves the beads
// by mobility * F * dt into the other position buffer (every bead sees the
// positions of the same step), so results do not vary from run to run.
//
// What bounds it is the FP32 pipe: about 50 packed operations per two partners
// in a periodic box (41 in an open one), 805 G pairs/s at 128 lanes per SM; one
// partner at a time it was issue (47 instructions per pair) and, at a few
// thousand beads, 13 warps per SM.  The partners are split so that about eight
// blocks per SM are there from a thousand beads on; six or eight resident
// blocks, two or four partner pairs unrolled make no difference beyond 10 %.
// Measured on GB300, periodic box, per step: 256 beads 39 us (force and move
// launches) -> 4.4, 1,024 beads 39 -> 6.5, 4,096 beads 53 -> 32 (526 G pairs/s),
// 16,384 beads 575 -> 438 (613 G pairs/s; open box 372).
#include "lbibm.h"
#include "lbibm_internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

namespace lbibm {
lb_status context_free_error(lb_status s, const char* msg);   // lbibm_api.cu

namespace {

constexpr int BEAD_TILE = 128;    // beads (threads) per block
constexpr int BEAD_STAGE = 256;   // partners staged at a time

struct BeadDev {
    float c3;         // 3 mu0 / (4 pi)
    float two_r;      // contact distance 2R
    float k;          // contact stiffness
    float mob_dt;     // mobility * dt
    float box[3];     // 0 on open axes
    float inv_box[3];
    int per[3];
    int n;
    int share;        // partners per block (even)
};

typedef float2 F2;
__device__ __forceinline__ F2 f2s(float a) { return make_float2(a, a); }
__device__ __forceinline__ F2 add2(F2 a, F2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ F2 mul2(F2 a, F2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) { return __ffma2_rn(a, b, c); }

// The bead of a thread with its constants, each in both halves of a pair.
struct BeadSelf {
    F2 x, y, z, mx, my, mz;
};

// r minus its periods, for both halves: t = rint(r / box) by the addition of
// 1.5 2^23 (round to nearest even, exact for |t| < 2^22).
__device__ __forceinline__ F2 nearest(F2 r, float box, float inv) {
    const F2 magic = f2s(12582912.0f);
    const F2 t = add2(fma2(r, f2s(inv), magic), f2s(-12582912.0f));
    return fma2(t, f2s(-box), r);
}

// Force on the bead from a pair of partners, added to (fx, fy, fz): half by
// half the dipole interaction and the contact force; a partner at distance 0
// (the bead itself) adds nothing.
template <bool PER>
__device__ __forceinline__ void bead_pair(const BeadSelf& b, float4 p0, float4 p1, float4 p2, const BeadDev& p, F2& fx,
                                          F2& fy, F2& fz) {
    // (x, y), (z, mx), (my, mz) of the two partners
    const F2 ax = make_float2(-p0.x, -p0.y), ay = make_float2(-p0.z, -p0.w), az = make_float2(-p1.x, -p1.y);
    const F2 ma = make_float2(p1.z, p1.w), mb = make_float2(p2.x, p2.y), mc = make_float2(p2.z, p2.w);
    // r = x_b - x_a (force on b from a), minimum image on periodic axes
    F2 r0 = add2(b.x, ax), r1 = add2(b.y, ay), r2 = add2(b.z, az);
    if (PER) {
        r0 = nearest(r0, p.box[0], p.inv_box[0]);
        r1 = nearest(r1, p.box[1], p.inv_box[1]);
        r2 = nearest(r2, p.box[2], p.inv_box[2]);
    }
    const F2 rr = fma2(r2, r2, fma2(r1, r1, mul2(r0, r0)));
    const F2 inv = make_float2(rr.x > 0.f ? rsqrtf(rr.x) : 0.f, rr.y > 0.f ? rsqrtf(rr.y) : 0.f);
    const F2 inv2 = mul2(inv, inv);
    const F2 pre = mul2(mul2(f2s(p.c3), inv2), mul2(inv2, inv));   // 3c / |r|^5
    const F2 mar = fma2(mc, r2, fma2(mb, r1, mul2(ma, r0)));
    const F2 mbr = fma2(b.mz, r2, fma2(b.my, r1, mul2(b.mx, r0)));
    const F2 mab = fma2(mc, b.mz, fma2(mb, b.my, mul2(ma, b.mx)));
    const F2 s = fma2(mul2(f2s(-5.0f), mar), mul2(mbr, inv2), mab);
    // contact: k (2R - d) / d below 2R
    const F2 gap = fma2(rr, make_float2(-inv.x, -inv.y), f2s(p.two_r));
    const F2 c = mul2(mul2(f2s(p.k), inv), make_float2(fmaxf(gap.x, 0.f), fmaxf(gap.y, 0.f)));
    const F2 kr = fma2(pre, s, c), ka = mul2(pre, mbr), kb = mul2(pre, mar);
    fx = fma2(kr, r0, fma2(ka, ma, fma2(kb, b.mx, fx)));
    fy = fma2(kr, r1, fma2(ka, mb, fma2(kb, b.my, fy)));
    fz = fma2(kr, r2, fma2(ka, mc, fma2(kb, b.mz, fz)));
}

// One step: forces of every bead; with x_out also the overdamped move
// x_out = x + mobility dt F, wrapped on periodic axes, otherwise the forces to
// F.  Grid (bead tiles, shares of the partners); part: [shares][tiles *
// BEAD_TILE] partial forces; done: a zeroed counter per tile, left at zero.
template <bool PER>
__global__ void __launch_bounds__(BEAD_TILE, 6) k_bead_step(const float4* __restrict__ x, const float4* __restrict__ m,
                                                         BeadDev p, float4* part, unsigned* done, float4* F,
                                                         float4* __restrict__ x_out) {
    __shared__ float4 st[3][BEAD_STAGE / 2];
    __shared__ bool last;
    pdl_entry();   // the previous step's positions
    const int b = blockIdx.x * BEAD_TILE + threadIdx.x;
    const bool live = b < p.n;
    const float4 xb = live ? x[b] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 mb = live ? m[b] : make_float4(0.f, 0.f, 0.f, 0.f);
    const BeadSelf self{f2s(xb.x), f2s(xb.y), f2s(xb.z), f2s(mb.x), f2s(mb.y), f2s(mb.z)};
    F2 fx = f2s(0.f), fy = fx, fz = fx;
    const int j1 = min(p.n, (int)(blockIdx.y + 1) * p.share);
    for (int j0 = blockIdx.y * p.share; j0 < j1; j0 += BEAD_STAGE) {
        const int cnt = min(BEAD_STAGE, j1 - j0);
        __syncthreads();
        for (int k = threadIdx.x; 2 * k < cnt; k += BEAD_TILE) {
            // (an odd end is paired with itself; that half is dropped below)
            const int a0 = j0 + 2 * k, a1 = 2 * k + 1 < cnt ? a0 + 1 : a0;
            const float4 u = x[a0], v = x[a1], mu = m[a0], mv = m[a1];
            st[0][k] = make_float4(u.x, v.x, u.y, v.y);
            st[1][k] = make_float4(u.z, v.z, mu.x, mv.x);
            st[2][k] = make_float4(mu.y, mv.y, mu.z, mv.z);
        }
        __syncthreads();
        if (live) {
            const int pairs = cnt >> 1;
#pragma unroll 2
            for (int k = 0; k < pairs; ++k) bead_pair<PER>(self, st[0][k], st[1][k], st[2][k], p, fx, fy, fz);
            if (cnt & 1) {
                F2 ox = f2s(0.f), oy = ox, oz = ox;
                bead_pair<PER>(self, st[0][pairs], st[1][pairs], st[2][pairs], p, ox, oy, oz);
                fx.x += ox.x;
                fy.x += oy.x;
                fz.x += oz.x;
            }
        }
    }
    const int stride = gridDim.x * BEAD_TILE;
    part[(size_t)blockIdx.y * stride + b] = make_float4(fx.x + fx.y, fy.x + fy.y, fz.x + fz.y, 0.f);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(done + blockIdx.x, 1u) + 1 == gridDim.y;
    __syncthreads();
    if (!last) return;
    __threadfence();
    float3 f = make_float3(0.f, 0.f, 0.f);
#pragma unroll 8
    for (int c = 0; c < (int)gridDim.y; ++c) {
        const float4 q = __ldcg(part + (size_t)c * stride + b);
        f.x += q.x; f.y += q.y; f.z += q.z;
    }
    if (threadIdx.x == 0) done[blockIdx.x] = 0u;
    if (!live) return;
    if (!x_out) {
        F[b] = make_float4(f.x, f.y, f.z, 0.f);
        return;
    }
    float v[3] = {xb.x + p.mob_dt * f.x, xb.y + p.mob_dt * f.y, xb.z + p.mob_dt * f.z};
#pragma unroll
    for (int d = 0; d < 3; ++d)
        if (p.per[d]) v[d] -= p.box[d] * floorf(v[d] / p.box[d]);
    x_out[b] = make_float4(v[0], v[1], v[2], 0.f);
}

// Grid of a step: (bead tiles, shares of the partners) with about eight blocks
// per SM, a share no smaller than 32 beads.
dim3 step_grid(int n, int& share) {
    int sms = 152, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaGetLastError();
    const int tiles = (n + BEAD_TILE - 1) / BEAD_TILE;
    const int want = std::max(1, std::min((n + 31) / 32, (8 * std::max(sms, 1) + tiles - 1) / tiles));
    share = ((n + want - 1) / want + 1) & ~1;
    return dim3((unsigned)tiles, (unsigned)((n + share - 1) / share));
}

bool params_ok(const bead_params* p, int n) {
    if (!p || n < 1) return false;
    const double v[5] = {p->mu0_4pi, p->radius, p->k_contact, p->mobility, p->dt};
    for (double x : v)
        if (!std::isfinite(x)) return false;
    if (p->radius < 0 || p->k_contact < 0) return false;
    for (int d = 0; d < 3; ++d)
        if (p->periodic[d] && !(p->box[d] > 0 && std::isfinite(p->box[d]))) return false;
    for (int k = 0; k < 5; ++k)
        if (p->reserved[k]) return false;
    return true;
}

BeadDev dev_params(const bead_params* p, int n) {
    BeadDev d;
    d.c3 = (float)(3.0 * p->mu0_4pi);
    d.two_r = (float)(2.0 * p->radius);
    d.k = (float)p->k_contact;
    d.mob_dt = (float)(p->mobility * p->dt);
    for (int k = 0; k < 3; ++k) {
        d.box[k] = p->periodic[k] ? (float)p->box[k] : 0.f;
        d.inv_box[k] = p->periodic[k] ? (float)(1.0 / p->box[k]) : 0.f;
        d.per[k] = p->periodic[k] ? 1 : 0;
    }
    d.n = n;
    d.share = 0;
    return d;
}

// Device buffers of one call in one allocation: the uploaded part (positions,
// moments, zeroed tile counters), then the other positions, forces and partial
// forces.
struct BeadBuffers {
    char* base = nullptr;
    float4* x[2] = {nullptr, nullptr};
    float4* m = nullptr;
    float4* F = nullptr;
    float4* part = nullptr;
    unsigned* done = nullptr;
    std::vector<float4> up;   // host image of the uploaded part, alive until the call has synchronised
    ~BeadBuffers() { cudaFree(base); }
};

lb_status upload(const double* xyz, const double* moments, int n, dim3 grid, BeadBuffers& B, cudaStream_t s) {
    const size_t row = (size_t)n, counters = (grid.x + 3) / 4, parts = (size_t)grid.x * BEAD_TILE * grid.y;
    B.up.resize(2 * row + counters, make_float4(0.f, 0.f, 0.f, 0.f));
    for (int i = 0; i < n; ++i) {
        B.up[i] = make_float4((float)xyz[3 * i], (float)xyz[3 * i + 1], (float)xyz[3 * i + 2], 0.f);
        B.up[row + i] = make_float4((float)moments[3 * i], (float)moments[3 * i + 1], (float)moments[3 * i + 2], 0.f);
    }
    if (cudaMalloc(&B.base, sizeof(float4) * (B.up.size() + 2 * row + parts)) != cudaSuccess) {
        cudaGetLastError();
        return context_free_error(LB_ERR_OOM, "bead buffers: device allocation failed");
    }
    B.x[0] = (float4*)B.base;
    B.m = B.x[0] + row;
    B.done = (unsigned*)(B.m + row);
    B.x[1] = B.m + row + counters;
    B.F = B.x[1] + row;
    B.part = B.F + row;
    if (cudaMemcpyAsync(B.base, B.up.data(), sizeof(float4) * B.up.size(), cudaMemcpyHostToDevice, s) != cudaSuccess)
        return context_free_error(LB_ERR_CUDA, "bead upload: CUDA error");
    return LB_OK;
}

cudaError_t launch_step(const BeadDev& d, dim3 grid, const BeadBuffers& B, int from, float4* out, bool pdl, cudaStream_t s) {
    const bool per = d.per[0] || d.per[1] || d.per[2];
    auto* kern = per ? k_bead_step<true> : k_bead_step<false>;
    return launch_ex(kern, grid, BEAD_TILE, 0, s, pdl, (const float4*)B.x[from], (const float4*)B.m, d, B.part, B.done, B.F, out);
}

lb_status download(const float4* d, int n, double* out, cudaStream_t s) {
    std::vector<float4> h(n);
    if (cudaMemcpyAsync(h.data(), d, sizeof(float4) * (size_t)n, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return context_free_error(LB_ERR_CUDA, "bead readback: CUDA error");
    for (int i = 0; i < n; ++i) {
        out[3 * i] = h[i].x;
        out[3 * i + 1] = h[i].y;
        out[3 * i + 2] = h[i].z;
    }
    return LB_OK;
}

}  // namespace
}  // namespace lbibm

using namespace lbibm;

extern "C" {

lb_status bead_forces(const double* xyz, const double* moments, int n, const bead_params* p, double* F,
                      void* cuda_stream) {
    if (!xyz || !moments || !F || !params_ok(p, n))
        return context_free_error(LB_ERR_ARG, "null array, n < 1 or invalid bead parameters");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    BeadDev d = dev_params(p, n);
    const dim3 grid = step_grid(n, d.share);
    BeadBuffers B;
    lb_status st = upload(xyz, moments, n, grid, B, s);
    if (st != LB_OK) return st;
    if (launch_step(d, grid, B, 0, nullptr, false, s) != cudaSuccess) {
        cudaGetLastError();
        return context_free_error(LB_ERR_CUDA, "bead forces: launch failed");
    }
    return download(B.F, n, F, s);
}

lb_status bead_relax(double* xyz, const double* moments, int n, const bead_params* p, int steps, void* cuda_stream) {
    if (!xyz || !moments || steps < 0 || !params_ok(p, n))
        return context_free_error(LB_ERR_ARG, "null array, n < 1, steps < 0 or invalid bead parameters");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    BeadDev d = dev_params(p, n);
    const dim3 grid = step_grid(n, d.share);
    BeadBuffers B;
    lb_status st = upload(xyz, moments, n, grid, B, s);
    if (st != LB_OK) return st;
    // each step a programmatic dependent of the one before
    for (int k = 0; k < steps; ++k)
        if (launch_step(d, grid, B, k & 1, B.x[(k + 1) & 1], k > 0, s) != cudaSuccess) {
            cudaGetLastError();
            return context_free_error(LB_ERR_CUDA, "bead relax: launch failed");
        }
    return download(B.x[steps & 1], n, xyz, s);
}

}  // extern "C"
