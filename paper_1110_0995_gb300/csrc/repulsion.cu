// Collisions between cells and with walls and beads (Gusenbauer et al.,
// arXiv:1110.0995, Sec. 2.4: a soft potential between mesh nodes of different
// cells and between cells and walls, cut at an interaction radius; form and
// constants not printed).  Reading: harmonic soft sphere, a force
// k (d_c - d) along the separation for d < d_c, between
//   * nodes of different cells of the same channel (equal and opposite,
//     x minimum image on a periodic axis),
//   * a node and a bead surface (d = |x - c| - r),
//   * a node and a wall of a non-periodic axis (walls half a link outside the
//     first and last lattice node).
// Per step three launches, each a programmatic dependent of the one before:
// each cell's bounding sphere and its candidate beads, one block per cell
// (k_rep_cells); candidate cell pairs from the bounding spheres and, beside
// them, every node's bead and wall forces, which start its R (k_rep_pairs);
// node-node forces of the candidate pairs, added to R (k_rep_nodes).  R joins
// the membrane forces in the spreading kernel.  Distances come from exact
// fixed-point differences.
//
// What bounds it: launches while few cells touch (seven launches and clears in
// a row took 28 us of the 98 us cycle of the 16-slit experiment, GB300; these
// three 16), and node pairs when cells touch.  A pair of cells is cut into
// units of RN_THREADS nodes, so that two 2562-node tumor cells spread over 22
// blocks rather than two, and both sides first drop the nodes outside the other
// cell's bounding sphere, which leaves a few per cent of the pairs: two such
// cells beside a red cell in a 32x108x19 channel 4586 -> 36 us per cycle,
// the 62-cell 256x128x64 filter with collisions 410 -> 84.
#include "lbibm_internal.cuh"

namespace lbibm {

// v * 2^-40: the nearest multiple of 2^32 and the rest, each rounded to FP32,
// and their sum (below 2^-9 lu one rounding, beyond at most three quarters of
// an ulp), over the whole range and with no 64-bit conversion.
__device__ __forceinline__ float rfx(long long v) {
    const int lo = (int)v;
    const int hi = (int)((v + 0x80000000LL) >> 32);
    return fmaf((float)hi, 0.00390625f, (float)lo * FIX_INV_F);   // 2^-8
}

__device__ __forceinline__ const ChannelDev& rchan(const RepArgs& a, int c) {
    return c < MAXCH_P ? a.chp[c] : a.ch[c];
}

// Minimum image along one axis: n and 1 / n, or zeros when it is not periodic.
struct Image {
    float n, inv;
};
__device__ __forceinline__ Image image(const ChannelDev& C, int d) {
    const int n = d == 0 ? C.nx : d == 1 ? C.ny : C.nz;
    return C.per[d] ? Image{(float)n, 1.0f / (float)n} : Image{0.f, 0.f};
}
__device__ __forceinline__ float min_image(float d, Image m) { return fmaf(-m.n, rintf(d * m.inv), d); }

// Positions are never wrapped; every absolute coordinate of a cell is taken
// less the whole periods of its reference node (RepArgs::home, exact), so that
// it is about a box at most and its FP32 rounding does not grow with the
// distance travelled.
__device__ __forceinline__ int home(long long q, Image m) { return (int)rintf(rfx(q) * m.inv); }
__device__ __forceinline__ long long shift(int periods, Image m) {
    return (long long)periods * ((long long)(int)m.n << FIX_BITS);
}

// Periods between a coordinate and the image of it next to `to`.
__device__ __forceinline__ int periods(float from, float to, Image m) { return (int)rintf((from - to) * m.inv); }
// A fixed-point difference wrapped into half a period, exactly.
__device__ __forceinline__ long long wrapped(long long d, Image m) {
    return d - shift(home(d, m), m);
}

constexpr int RC_THREADS = 512;

// (1) bounding sphere of every cell: centre (relative to the reference node,
// plus the reference node's position less its periods) and radius; the beads
// within reach.  Margin 0.5 lu covers the float rounding of the centres (on an
// axis without periods up to 2^20 lu from the origin).
__global__ void __launch_bounds__(RC_THREADS) k_rep_cells(const __grid_constant__ RepArgs a) {
    const CellDev& C = a.cells[blockIdx.x];
    const ChannelDev& Ch = rchan(a, C.ch);
    const int ch = C.ch, node0 = C.node0, nn = C.n_nodes;
    pdl_entry();
    const Q4 qr = a.q[C.ref];
    float sx = 0.f, sy = 0.f, sz = 0.f;
    for (int i = threadIdx.x; i < nn; i += RC_THREADS) {
        const Q4 q = a.q[node0 + i];
        sx += rfx(q.x - qr.x); sy += rfx(q.y - qr.y); sz += rfx(q.z - qr.z);
    }
    __shared__ float sh[3][RC_THREADS / 32];
    __shared__ int near;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
        sy += __shfl_xor_sync(0xffffffffu, sy, o);
        sz += __shfl_xor_sync(0xffffffffu, sz, o);
    }
    if (lane == 0) { sh[0][wid] = sx; sh[1][wid] = sy; sh[2][wid] = sz; }
    if (threadIdx.x == 0) near = 0;
    __syncthreads();
    float cen[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int w = 0; w < RC_THREADS / 32; ++w)
        for (int d = 0; d < 3; ++d) cen[d] += sh[d][w];
    for (int d = 0; d < 3; ++d) cen[d] /= (float)nn;
    float r2 = 0.f;
    for (int i = threadIdx.x; i < nn; i += RC_THREADS) {
        const Q4 q = a.q[node0 + i];
        const float dx = rfx(q.x - qr.x) - cen[0], dy = rfx(q.y - qr.y) - cen[1], dz = rfx(q.z - qr.z) - cen[2];
        r2 = fmaxf(r2, dx * dx + dy * dy + dz * dz);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, o));
    __syncthreads();
    if (lane == 0) sh[0][wid] = r2;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < RC_THREADS / 32; ++w) r2 = fmaxf(r2, sh[0][w]);
    // centre as float (a coarse test with a margin; distances between nodes
    // themselves use fixed point)
    const Image ix = image(Ch, 0), iy = image(Ch, 1), iz = image(Ch, 2);
    const int hx = home(qr.x, ix), hy = home(qr.y, iy), hz = home(qr.z, iz);
    const float4 A = make_float4(rfx(qr.x - shift(hx, ix)) + cen[0], rfx(qr.y - shift(hy, iy)) + cen[1],
                                 rfx(qr.z - shift(hz, iz)) + cen[2], sqrtf(r2));
    if (threadIdx.x == 0) {
        a.bounds[blockIdx.x] = A;
        a.home[blockIdx.x] = make_int4(hx, hy, hz, 0);
    }
    for (int b = threadIdx.x; b < a.n_beads; b += RC_THREADS) {
        if (a.bead_ch[b] != ch) continue;
        const Q4 bq = a.bead_q[b];
        const float dx = min_image(A.x - rfx(bq.x), ix), dy = min_image(A.y - rfx(bq.y), iy),
                    dz = min_image(A.z - rfx(bq.z), iz);
        const float lim = A.w + a.bead_r[b] + a.dc + 0.5f;
        if (dx * dx + dy * dy + dz * dz < lim * lim) {
            const int k = atomicAdd(&near, 1);
            if (k < REP_NEARB) a.near[blockIdx.x * REP_NEARB + k] = b;
            else atomicAdd(a.err, 1);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a.near_count[blockIdx.x] = near;
        if (blockIdx.x == 0) *a.pair_count = 0;   // counted by the next kernel
    }
}

// Node-bead (the cell's candidate beads) and node-wall forces of node i.
__device__ __forceinline__ void rep_walls_beads(const RepArgs& a, int i) {
    const int c = a.info[i].x;
    const CellDev& C = a.cells[c];
    const ChannelDev& Ch = rchan(a, C.ch);
    const Q4 q = a.q[i];
    const float k = a.k, dc = a.dc;
    const Image ix = image(Ch, 0), iy = image(Ch, 1), iz = image(Ch, 2);
    // the image of the cell in the middle of the box (exact: the distances below
    // keep their FP32 accuracy however far the cell has travelled)
    const float4 S = a.bounds[c];
    const int4 H = a.home[c];
    const long long px = q.x - shift(H.x + periods(S.x, 0.5f * ix.n, ix), ix),
                    py = q.y - shift(H.y + periods(S.y, 0.5f * iy.n, iy), iy),
                    pz = q.z - shift(H.z + periods(S.z, 0.5f * iz.n, iz), iz);
    float fx = 0.f, fy = 0.f, fz = 0.f;
    const int nb = min(a.near_count[c], REP_NEARB);
    for (int t = 0; t < nb; ++t) {
        const int b = a.near[c * REP_NEARB + t];
        const Q4 bq = a.bead_q[b];
        const float dx = rfx(wrapped(px - bq.x, ix));
        const float dy = rfx(wrapped(py - bq.y, iy));
        const float dz = rfx(wrapped(pz - bq.z, iz));
        const float d2 = dx * dx + dy * dy + dz * dz;
        const float rr = a.bead_r[b] + dc;
        if (d2 < rr * rr && d2 > 0.f) {
            const float d = sqrtf(d2);
            const float f = k * (dc - (d - a.bead_r[b])) / d;
            fx += f * dx; fy += f * dy; fz += f * dz;
        }
    }
    // walls at -1/2 and n - 1/2 on the non-periodic axes
    const long long half = 1LL << (FIX_BITS - 1);
    const long long qq[3] = {q.x, q.y, q.z};
    const int n[3] = {Ch.nx, Ch.ny, Ch.nz};
    float fw[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (Ch.per[d]) continue;
        const float lo = rfx(qq[d] + half);
        const float hi = rfx(((long long)n[d] << FIX_BITS) - half - qq[d]);
        if (lo < dc) fw[d] += k * (dc - lo);
        if (hi < dc) fw[d] -= k * (dc - hi);
    }
    a.R[i] = make_float4(fx + fw[0], fy + fw[1], fz + fw[2], 0.f);
}

// (2) blocks [0, pair_blocks): ordered cell pairs (a != b, same channel) whose
// bounding spheres come within the cut-off; the others: bead and wall forces.
constexpr int RP_THREADS = 128;
__global__ void __launch_bounds__(RP_THREADS) k_rep_pairs(const __grid_constant__ RepArgs a, int pair_blocks) {
    pdl_entry();
    if ((int)blockIdx.x >= pair_blocks) {
        const int i = ((int)blockIdx.x - pair_blocks) * RP_THREADS + threadIdx.x;
        if (i < a.n_nodes) rep_walls_beads(a, i);
        return;
    }
    const long long t = (long long)blockIdx.x * RP_THREADS + threadIdx.x;
    const long long nC = a.n_cells;
    if (t >= nC * nC) return;
    const int ca = (int)(t / nC), cb = (int)(t - (t / nC) * nC);
    if (ca == cb || a.cells[ca].ch != a.cells[cb].ch) return;
    const ChannelDev& Ch = rchan(a, a.cells[ca].ch);
    const float4 A = a.bounds[ca], B = a.bounds[cb];
    const float dx = min_image(A.x - B.x, image(Ch, 0)), dy = min_image(A.y - B.y, image(Ch, 1)),
                dz = min_image(A.z - B.z, image(Ch, 2));
    const float lim = A.w + B.w + a.dc + 0.5f;
    if (dx * dx + dy * dy + dz * dz < lim * lim) {
        const int k = atomicAdd(a.pair_count, 1);
        if (k < a.pair_cap) a.pairs[k] = make_int2(ca, cb);
        else atomicAdd(a.err, 1);
    }
}

// (3) node-node forces of ordered candidate pairs (a, b): forces on a's nodes.
// A unit is RN_THREADS nodes of a; b's nodes near a's sphere are collected in
// shared memory a tile at a time, relative to a's reference node.
constexpr int RN_THREADS = 128;
constexpr int RN_TILE = 512;

__global__ void __launch_bounds__(RN_THREADS) k_rep_nodes(const __grid_constant__ RepArgs a, int units_per_pair) {
    pdl_entry();
    __shared__ float3 tile[RN_TILE];
    __shared__ int count;
    const int n_units = min(*a.pair_count, a.pair_cap) * units_per_pair;
    const float k = a.k, dc = a.dc, dc2 = a.dc * a.dc;
    for (int u = blockIdx.x; u < n_units; u += gridDim.x) {
        const int2 pr = a.pairs[u / units_per_pair];
        const CellDev& A = a.cells[pr.x];
        const CellDev& B = a.cells[pr.y];
        const int i = (u % units_per_pair) * RN_THREADS + threadIdx.x;
        if (i - (int)threadIdx.x >= A.n_nodes) continue;   // (the whole block)
        const ChannelDev& Ch = rchan(a, A.ch);
        const Image ix = image(Ch, 0), iy = image(Ch, 1), iz = image(Ch, 2);
        const Q4 qr = a.q[A.ref];
        // the spheres relative to a's reference node (less its periods); margin as in the pair test
        const float4 SA = a.bounds[pr.x], SB = a.bounds[pr.y];
        const int4 HA = a.home[pr.x], HB = a.home[pr.y];
        const long long hx = qr.x - shift(HA.x, ix), hy = qr.y - shift(HA.y, iy), hz = qr.z - shift(HA.z, iz);
        const float rx = rfx(hx), ry = rfx(hy), rz = rfx(hz);
        // b's image next to a, as exact fixed-point periods
        const long long ox = hx + shift(HB.x + periods(SB.x, SA.x, ix), ix),
                        oy = hy + shift(HB.y + periods(SB.y, SA.y, iy), iy),
                        oz = hz + shift(HB.z + periods(SB.z, SA.z, iz), iz);
        auto within = [&](float3 x, float4 S) {
            const float dx = min_image(x.x - (S.x - rx), ix), dy = min_image(x.y - (S.y - ry), iy),
                        dz = min_image(x.z - (S.z - rz), iz);
            const float lim = S.w + dc + 0.5f;
            return dx * dx + dy * dy + dz * dz < lim * lim;
        };
        float3 xi = make_float3(0.f, 0.f, 0.f);
        bool live = false;
        if (i < A.n_nodes) {
            const Q4 q = a.q[A.node0 + i];
            xi = make_float3(rfx(q.x - qr.x), rfx(q.y - qr.y), rfx(q.z - qr.z));
            live = within(xi, SB);
        }
        if (!__syncthreads_or(live)) continue;
        float fx = 0.f, fy = 0.f, fz = 0.f;
        for (int j0 = 0; j0 < B.n_nodes; j0 += RN_TILE) {
            if (threadIdx.x == 0) count = 0;
            __syncthreads();
            for (int j = threadIdx.x; j < RN_TILE && j0 + j < B.n_nodes; j += RN_THREADS) {
                const Q4 q = a.q[B.node0 + j0 + j];
                const float3 xj = make_float3(rfx(q.x - ox), rfx(q.y - oy), rfx(q.z - oz));
                if (within(xj, SA)) tile[atomicAdd(&count, 1)] = xj;
            }
            __syncthreads();
            const int nj = count;
            if (live) {
                for (int j = 0; j < nj; ++j) {
                    const float3 xj = tile[j];
                    const float dx = min_image(xi.x - xj.x, ix);
                    const float dy = min_image(xi.y - xj.y, iy);
                    const float dz = min_image(xi.z - xj.z, iz);
                    const float d2 = dx * dx + dy * dy + dz * dz;
                    if (d2 < dc2 && d2 > 0.f) {
                        const float d = sqrtf(d2);
                        const float f = k * (dc - d) / d;
                        fx += f * dx; fy += f * dy; fz += f * dz;
                    }
                }
            }
            __syncthreads();   // every thread is done with the tile and its count
        }
        if (live && (fx != 0.f || fy != 0.f || fz != 0.f)) atomicAdd(a.R + A.node0 + i, make_float4(fx, fy, fz, 0.f));
    }
}

cudaError_t launch_repulsion(const RepArgs& a, int sm_count, cudaStream_t s) {
    if (a.n_cells <= 0) return cudaSuccess;
    cudaError_t e = launch_ex(k_rep_cells, a.n_cells, RC_THREADS, 0, s, a.pdl, a);
    const int pair_blocks = (int)(((long long)a.n_cells * a.n_cells + RP_THREADS - 1) / RP_THREADS);
    if (e == cudaSuccess)
        e = launch_ex(k_rep_pairs, pair_blocks + (a.n_nodes + RP_THREADS - 1) / RP_THREADS, RP_THREADS, 0, s, a.pdl, a,
                      pair_blocks);
    if (e == cudaSuccess)
        e = launch_ex(k_rep_nodes, 8 * sm_count, RN_THREADS, 0, s, a.pdl, a, (a.max_nodes + RN_THREADS - 1) / RN_THREADS);
    return e;
}

}  // namespace lbibm
