// Membrane forces per patch (Gusenbauer et al., arXiv:1110.0995, Sec. 2.3.1:
// stretching, bending, local / global area, volume).
//
// Each cell mesh is cut once, by its connectivity, into patches of at most
// PATCH_NODES nodes.  One block takes one patch of one cell: it loads the
// positions of the patch's nodes and of the nodes around them into shared
// memory, evaluates every triangle and edge that touches the patch from there
// (elements on a patch border are evaluated by both sides), and then gathers
// each node's ring from shared memory in a fixed order.  What leaves is three
// vectors per node: the local forces, the sum of the area directions and the
// sum of the normals, to which the spreading kernel applies the cell's global
// area and volume terms once all patches of the cell have added their share of
// them.
//
// What bounds this: two passes with the elements' forces in memory between
// them (98 MB written and read per cycle on the 512x256x128 filter, 30 gathered
// 16-byte pieces per node) kept 24 to 36 warps per SM waiting on L2.  From
// shared memory a patch's elements cost 1.2 evaluations each and 17 KB of
// input per block, half of it tables shared by all cells of a mesh; now it is
// the shared-memory pipe (59 % busy; 8 wavefronts per 128-bit access of random
// nodes), the block's three dependent rounds of loads and issue (32 %).
// Measured on GB300, element pass + spreading before, this kernel + spreading
// now: 512x256x128 (404 cells) 49 + 52 us, 47.7 + 22.4; 24-channel sweep (621
// cells) 70 + 76, 63 + 33; 256x128x64 (62 cells) 14.9 + 13.2, 15.1 + 9.3.
#include "lbibm_internal.cuh"

#include <algorithm>
#include <vector>

namespace lbibm {

namespace {

constexpr int MB = 256;                 // threads per block
constexpr int ROUNDS = 3;               // element rounds whose tables are loaded before the wait
constexpr int RING_ROWS = 4;            // the same for the ring table
constexpr unsigned RING_END = 0xffffffffu;

__device__ __forceinline__ float3 operator+(float3 a, float3 b) { return make_float3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ float3 operator-(float3 a, float3 b) { return make_float3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float3 operator*(float s, float3 a) { return make_float3(s * a.x, s * a.y, s * a.z); }
__device__ __forceinline__ float dot(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ float3 cross(float3 a, float3 b) {
    return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float sqrt_fast(float x) { return x * rsqrtf(x); }

// A node in shared memory: position x relative to the cell's reference node
// and displacement d from rest (minus the reference node's), each the sum of
// two FP32 numbers: hi a multiple of the cell's grid 2^-g (differences of two
// are exact), lo the remainder (exact for g = 16).  So an edge, (hi_b - hi_a) +
// (lo_b - lo_a), carries one rounding, as the fixed-point difference would,
// however far the cell has moved.
struct Node {
    float3 xh, xl, dh, dl;
};
struct Nodes {
    float4 *A, *B, *C;   // (xh, xl.x), (xl.yz, dh.xy), (dh.z, dl)
};

__device__ __forceinline__ Node node_full(const Nodes& S, int k) {
    const float4 a = S.A[k], b = S.B[k], c = S.C[k];
    return Node{make_float3(a.x, a.y, a.z), make_float3(a.w, b.x, b.y), make_float3(b.z, b.w, c.x),
                make_float3(c.y, c.z, c.w)};
}
__device__ __forceinline__ Node node_pos(const Nodes& S, int k) {
    const float4 a = S.A[k];
    const float2 b = *reinterpret_cast<const float2*>(&S.B[k]);
    Node n = {};
    n.xh = make_float3(a.x, a.y, a.z);
    n.xl = make_float3(a.w, b.x, b.y);
    return n;
}
__device__ __forceinline__ float3 edge(const Node& a, const Node& b) { return (b.xh - a.xh) + (b.xl - a.xl); }
__device__ __forceinline__ float3 ddisp(const Node& a, const Node& b) { return (b.dh - a.dh) + (b.dl - a.dl); }

__device__ __forceinline__ void split(long long v, int sh, float grid, float& hi, float& lo) {
    const int n = (int)((v + (1LL << (sh - 1))) >> sh);
    hi = (float)n * grid;
    lo = (float)(int)(v - ((long long)n << sh)) * FIX_INV_F;
}

// Node k where hi would be rounded (beyond 2^24 grid steps) or the remainder
// is no 32-bit integer (a grid coarser than 2^-8): hi is the value itself
// rounded to 24 bits, lo what that leaves, by 64-bit conversions.  Where the
// kernel has 80 registers the node takes this in place of the ordinary form;
// at 64 a second look at the patch's nodes, when any needs it, keeps the
// ordinary loop as it was (512x256x128, membrane kernel: in place 3.7 % slower,
// second look 1.5 % faster; 256x128x64 with the second look 13 % slower, in
// place no different).
__device__ __forceinline__ void far_node(const Nodes& S, int k, const Q4& q, const Q4& qr, const Fix3& x0) {
    auto put = [](long long v, float& hi, float& lo) {
        hi = __ll2float_rn(v) * FIX_INV_F;
        lo = __ll2float_rn(v - __float2ll_rn(hi * FIX_SCALE_F)) * FIX_INV_F;
    };
    put(q.x - qr.x, S.A[k].x, S.A[k].w);
    put(q.y - qr.y, S.A[k].y, S.B[k].x);
    put(q.z - qr.z, S.A[k].z, S.B[k].y);
    put(q.x - qr.x - x0.x, S.B[k].z, S.C[k].y);
    put(q.y - qr.y - x0.y, S.B[k].w, S.C[k].z);
    put(q.z - qr.z - x0.z, S.C[k].x, S.C[k].w);
}

__device__ __forceinline__ long long to_fixed_f(float u) {   // round(u 2^40), |u| < 2^15
    const float s = u * 65536.0f;
    const float m = rintf(s);
    const float f = (s - m) * 16777216.0f;
    return ((long long)__float2int_rn(m) << 24) + (long long)__float2int_rn(f);
}

__device__ __forceinline__ long long warp_sum_ll(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// One triangle: normal over its squared length (p) with that square, the
// factor of the area direction ((e1 + e2) c at a vertex with edges e1, e2) and
// the local area strain times its modulus; the owner's share of the cell's
// area and volume change (dS, 6 dV).
__device__ __forceinline__ void triangle(const Nodes& S, uint2 t, float S0t, float kal, float4& p, float2& r, long long& s,
                                         long long& v) {
    const Node P0 = node_full(S, t.x & 0xffff), P1 = node_full(S, t.x >> 16), P2 = node_full(S, t.y & 0xffff);
    const float3 e1 = edge(P0, P1), e2 = edge(P0, P2);
    const float3 b1 = ddisp(P0, P1), b2 = ddisp(P0, P2);
    const float3 n = cross(e1, e2);
    // |n|^2 - |n0|^2 = dn.(2 n - dn), dn = n - n0 = (e1 - b1) x b2 + b1 x e2
    const float3 dn = cross(e1 - b1, b2) + cross(b1, e2);
    const float num = dot(dn, 2.0f * n - dn);
    const float nn0 = 2.0f * S0t;
    const float dS = __fdividef(num, 2.0f * (sqrt_fast(nn0 * nn0 + num) + nn0));
    const float n2 = dot(n, n);
    const float in2 = __fdividef(1.0f, n2);
    p = make_float4(n.x * in2, n.y * in2, n.z * in2, n2);
    // a_k = -(2 S / sum |w|^2) w_k with w_k = x_k - centroid = -(e1 + e2) / 3 at
    // vertex 0 and sum |w|^2 = 2/3 (|e1|^2 + |e2|^2 - e1.e2)
    r = make_float2(__fdividef(S0t + dS, dot(e1, e1) + dot(e2, e2) - dot(e1, e2)), __fdividef(kal * dS, S0t));
    if (t.y >> 31) {
        // 6 V of the tetrahedron with the reference node is x0.n (x relative to
        // it): the change x0.n - r0.n0 = d0.n + r0.dn, x0 = r0 + d0
        const float3 d0 = P0.dh + P0.dl, r0 = (P0.xh - P0.dh) + (P0.xl - P0.dl);
        s += to_fixed_f(dS);
        v += to_fixed_f(dot(d0, n) + dot(r0, dn));
    }
}

// One edge (a, b) between the triangles (a, b, c) and (b, a, d): the edge with
// its stretching tension over its length (p); bending coefficient times length
// and 1 / length^2 (r).
//   stretching (neo-Hookean bond): ks kappa (lambda - 1),
//     kappa = lambda^1/2 (lambda^3 + 1) / (lambda^4 + 1);
//   bending: -kb (theta - theta0), theta = atan2((n1 x n2).e / |e|, n1.n2) with
//     n1 = e x ac, n2 = ad x e, where (n1 x n2).e = -|e|^2 n1.ad.
__device__ __forceinline__ void edge_terms(const Nodes& S, uint2 t, float2 rest, float ks, float kb, float4& p, float2& r) {
    const Node A = node_full(S, t.x & 0xffff), B = node_full(S, t.x >> 16);
    const Node Cc = node_pos(S, t.y & 0xffff), D = node_pos(S, t.y >> 16);
    const float3 e = edge(A, B), de = ddisp(A, B);
    const float num = dot(de, 2.0f * e - de);   // |e|^2 - |e0|^2
    const float L0 = rest.x;
    const float L = sqrt_fast(L0 * L0 + num);
    const float lm1 = __fdividef(num, (L + L0) * L0);
    const float lam = 1.0f + lm1;
    const float lam2 = lam * lam;
    const float kappa = __fdividef(sqrt_fast(lam) * (lam2 * lam + 1.0f), lam2 * lam2 + 1.0f);
    const float l2 = dot(e, e);
    const float rl = rsqrtf(l2);
    const float l = l2 * rl;
    const float3 ad = edge(A, D);
    const float3 n1 = cross(e, edge(A, Cc)), n2 = cross(ad, e);
    const float theta = atan2f(-l * dot(n1, ad), dot(n1, n2));
    p = make_float4(e.x, e.y, e.z, ks * kappa * lm1 * rl);
    r = make_float2(-kb * (theta - rest.y) * l, __fdividef(1.0f, l2));
}

template <int MINB>
__global__ void __launch_bounds__(MB, MINB) k_membrane(const __grid_constant__ IbmArgs a) {
    extern __shared__ __align__(16) float4 memb_sm[];
    __shared__ long long red[MB / 32][2];
    const PatchJob J = a.patches[blockIdx.x];
    const PatchTab& tp = J.tab;
    Nodes S;
    S.A = memb_sm;
    S.B = S.A + tp.n_loc;
    S.C = S.B + tp.n_loc;
    float4* edp = S.C + tp.n_loc;
    float4* trp = edp + tp.n_edge;
    float2* edr = reinterpret_cast<float2*>(trp + tp.n_tri);
    float2* trr = edr + tp.n_edge;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint32_t* loc = a.ploc + tp.loc0;
    const uint2* tris = a.ptri + tp.tri0;
    const uint2* edges = a.pedge + tp.edge0;
    const float* rest_tri = a.prest_tri + J.rest_tri;
    const float2* rest_edge = a.prest_edge + J.rest_edge;
    const Fix3* rest_node = a.prest_node + J.rest_node;
    const int tri_end = (tp.n_tri + 31) & ~31;   // a warp has triangles or edges, not both
    // before the previous advance has finished: the tables of this thread's
    // first elements with their rest data, its first node's rest position, its
    // first ring slots
    uint2 it[ROUNDS];
    float2 rs[ROUNDS];
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int k = tid + r * MB, ke = k - tri_end;
        it[r] = make_uint2(0u, 0u);
        rs[r] = make_float2(0.f, 0.f);
        if (k < tp.n_tri) {
            it[r] = tris[k];
            rs[r].x = rest_tri[k];
        } else if (ke >= 0 && ke < tp.n_edge) {
            it[r] = edges[ke];
            rs[r] = rest_edge[ke];
        }
    }
    int id = 0;
    Fix3 x0 = {};
    if (tid < tp.n_loc) {
        id = (int)loc[tid];
        x0 = rest_node[tid];
    }
    const uint2* ring = a.pring + tp.ring0 + tid;
    uint2 sl[RING_ROWS];
#pragma unroll
    for (int j = 0; j < RING_ROWS; ++j)
        sl[j] = tid < 2 * tp.n_own && j <= tp.rows ? ring[j * 2 * tp.n_own] : make_uint2(RING_END, 0u);
    // points with mass moved in the spreading kernel, two kernels back: their
    // membrane forces wait for nothing here and run beside the stream-collide
    // (the wait, which orders everything later, stands at the end).  One-cell
    // channel 57x41x23: 1.5 us per cycle less, filters of eight to ten cells 1.2 us (GB300)
    if (!a.W) pdl_entry();
    const Q4* qc = a.par ? a.qb : a.qa;
    const Q4 qr = qc[J.ref];
    // half of 2^24 grid steps; none for a grid coarser than 2^-8
    const unsigned far_limit = J.grid >= 8 ? 1u << (31 - J.grid) : 0u;
    bool far = false;
    for (int k = tid; k < tp.n_loc; k += MB) {
        if (k != tid) {
            id = (int)loc[k];
            x0 = rest_node[k];
        }
        const Q4 q = qc[J.node0 + id];
        const long long x = q.x - qr.x, y = q.y - qr.y, z = q.z - qr.z;
        // (the upper halves' magnitudes, 2^-8 lu; displacements are within the rest extent of the positions)
        auto is_far = [&] {
            auto mag = [](long long v) { return (unsigned)((int)(v >> 32) ^ (int)(v >> 63)); };
            return (mag(x) | mag(y) | mag(z)) >= far_limit;
        };
        float4 A, B, Cc;
        auto fill = [&](int sh, float grid) {
            split(x, sh, grid, A.x, A.w);
            split(y, sh, grid, A.y, B.x);
            split(z, sh, grid, A.z, B.y);
            split(x - x0.x, sh, grid, B.z, Cc.y);
            split(y - x0.y, sh, grid, B.w, Cc.z);
            split(z - x0.z, sh, grid, Cc.x, Cc.w);
        };
        if constexpr (MINB == 3) {
            if (is_far()) {
                far_node(S, k, q, qr, x0);
                continue;
            }
        }
        if (J.grid == 16) fill(FIX_BITS - 16, 1.0f / 65536.0f);
        else fill(FIX_BITS - J.grid, __int_as_float((127 - J.grid) << 23));
        if constexpr (MINB != 3) far = far || is_far();
        S.A[k] = A;
        S.B[k] = B;
        S.C[k] = Cc;
    }
    if constexpr (MINB == 3) {
        __syncthreads();
    } else if (__syncthreads_or(far)) {
        for (int k = tid; k < tp.n_loc; k += MB) far_node(S, k, qc[J.node0 + (int)loc[k]], qr, rest_node[k]);
        __syncthreads();
    }
    // elements
    long long s = 0, v = 0;
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int k = tid + r * MB, ke = k - tri_end;
        if (k < tp.n_tri) triangle(S, it[r], rs[r].x, J.kal, trp[k], trr[k], s, v);
        else if (ke >= 0 && ke < tp.n_edge) edge_terms(S, it[r], rs[r], J.ks, J.kb, edp[ke], edr[ke]);
    }
    for (int k = tid + ROUNDS * MB; k < tri_end + tp.n_edge; k += MB) {
        const int ke = k - tri_end;
        if (k < tp.n_tri) triangle(S, tris[k], rest_tri[k], J.kal, trp[k], trr[k], s, v);
        else if (ke >= 0) edge_terms(S, edges[ke], rest_edge[ke], J.ks, J.kb, edp[ke], edr[ke]);
    }
    s = warp_sum_ll(s);
    v = warp_sum_ll(v);
    if (lane == 0) { red[wid][0] = s; red[wid][1] = v; }
    __syncthreads();
    // every node's ring: two lanes per node, each half of its slots in order,
    // the edge to the next neighbour carried from slot to slot
    float3 F = make_float3(0.f, 0.f, 0.f), Ad = F, N = F;
    const int own = tid >> 1;
    if (own < tp.n_own) {
        auto edge_from = [&](unsigned k, float3& e, float& tension, float2& r) {   // bit 15: the node is the edge's b
            const float4 p = edp[k & 0x7fffu];
            const float sg = k & 0x8000u ? -1.0f : 1.0f;
            e = make_float3(sg * p.x, sg * p.y, sg * p.z);
            tension = p.w;
            r = edr[k & 0x7fffu];
        };
        float3 e1, e2;
        float t1, t2;
        float2 q1, q2;
        edge_from(sl[0].x, e1, t1, q1);
        auto slot = [&](uint2 t) {
            edge_from(t.x & 0xffffu, e2, t2, q2);
            const float4 p = trp[t.x >> 16];
            const float2 r = trr[t.x >> 16];
            const float d = dot(e1, e2);
            // the triangle's weight in the bending of its three edges
            const float w = q1.x * (1.0f - d * q1.y) + q2.x * (1.0f - d * q2.y) - edr[t.y].x;
            const float3 c = r.x * (e1 + e2);
            const float3 pv = make_float3(p.x, p.y, p.z);
            F = F + (w * pv + (r.y * c + t1 * e1));
            Ad = Ad + c;
            N = N + p.w * pv;
            e1 = e2;
            t1 = t2;
            q1 = q2;
        };
#pragma unroll
        for (int j = 1; j < RING_ROWS; ++j)
            if (sl[j].x != RING_END) slot(sl[j]);
        for (int j = RING_ROWS; j <= tp.rows; ++j) {
            const uint2 t = ring[j * 2 * tp.n_own];
            if (t.x == RING_END) break;
            slot(t);
        }
    }
    auto both = [](float x) { return x + __shfl_xor_sync(0xffffffffu, x, 1); };
    F = make_float3(both(F.x), both(F.y), both(F.z));
    Ad = make_float3(both(Ad.x), both(Ad.y), both(Ad.z));
    N = make_float3(both(N.x), both(N.y), both(N.z));
    if (own < tp.n_own) {
        float4* o = a.acc + 3 * (size_t)(J.node0 + (int)loc[own]);
        if ((tid & 1) == 0) {
            o[0] = make_float4(F.x, F.y, F.z, Ad.x);
            o[1] = make_float4(Ad.y, Ad.z, N.x, N.y);
        } else {
            o[2] = make_float4(N.z, 0.f, 0.f, 0.f);
        }
    }
    // the patch's share of the cell's area and volume change; the last patch of
    // the cell adds the shares (integers: exact, in any order) and forms dS / S0
    // and dV / V0 in FP64 once
    if (wid == MB / 32 - 1) {
        s = warp_sum_ll(lane < MB / 32 ? red[lane][0] : 0);
        v = warp_sum_ll(lane < MB / 32 ? red[lane][1] : 0);
        bool last = false;
        if (lane == 0) {
            a.partials[blockIdx.x] = make_longlong2(s, v);
            __threadfence();
            last = atomicAdd(a.counters + J.cell, 1u) + 1 == (unsigned)J.n_patch;
        }
        if (__shfl_sync(0xffffffffu, (int)last, 0)) {
            __threadfence();
            s = v = 0;
            for (int k = lane; k < J.n_patch; k += 32) {
                const longlong2 pv = __ldcg(a.partials + J.patch0 + k);
                s += pv.x;
                v += pv.y;
            }
            s = warp_sum_ll(s);
            v = warp_sum_ll(v);
            if (lane == 0) {
                const double dS = (double)s * (1.0 / FIX_SCALE), dV = (double)v * (1.0 / (6.0 * FIX_SCALE));
                const CellDev& C = a.cells[J.cell];
                a.cell_sums[J.cell] = make_double2(dS, dV);
                a.cell_rel[J.cell] = make_float2((float)(dS / C.S0), (float)(dV / C.V0));
                a.counters[J.cell] = 0u;
            }
        }
    }
    if (a.W) pdl_entry();
}

// Once, when the context commits: a block per patch.  (Gathered on the host, with
// their upload, the rest data cost the 62-cell filter 0.4 ms of its first step.)
__global__ void __launch_bounds__(MB) k_patch_rest(const PatchRest r) {
    const PatchJob J = r.jobs[blockIdx.x];
    for (int i = threadIdx.x; i < J.tab.n_edge; i += MB) {
        const float4 e = r.edge_rest[J.e0 + r.edge_id[J.tab.edge0 + i]];
        r.rest_edge[J.rest_edge + i] = make_float2(e.x, e.y);
    }
    for (int i = threadIdx.x; i < J.tab.n_tri; i += MB) r.rest_tri[J.rest_tri + i] = r.tri_S0[J.tri0 + r.tri_id[J.tab.tri0 + i]];
    const Q4 ref = r.q0[J.ref];
    for (int i = threadIdx.x; i < J.tab.n_loc; i += MB) {
        const Q4 q = r.q0[J.node0 + (int)r.loc[J.tab.loc0 + i]];
        r.rest_node[J.rest_node + i] = Fix3{q.x - ref.x, q.y - ref.y, q.z - ref.z};
    }
}

// Shared memory of one patch.
size_t patch_bytes(const PatchTab& t) {
    return 48 * (size_t)t.n_loc + 24 * (size_t)(t.n_edge + t.n_tri);
}

// ---- host: patches of one connectivity ----
struct Cutter {
    const MeshTables& m;
    PatchTables& out;
    std::vector<int> nbr;                       // neighbour per ring slot
    std::vector<int> perm, queue, tag;          // nodes in patch order; per node: the subset it is in
    std::vector<int> lnode, ltri, ledge;        // local numbers in the patch being written (-1: none)
    std::vector<int> tris, edges, halo;
    int next_tag = 1;

    Cutter(const MeshTables& mesh, PatchTables& o)
        : m(mesh), out(o), nbr(mesh.ring_off[mesh.n - 1] + mesh.valence[mesh.n - 1]), perm(mesh.n), queue(mesh.n),
          tag(mesh.n, 0), lnode(mesh.n, -1), ltri(mesh.nt, -1), ledge(mesh.n_edges, -1) {
        for (int i = 0; i < m.n; ++i) {
            perm[i] = i;
            for (int s = m.ring_off[i]; s < m.ring_off[i] + m.valence[i]; ++s) {
                const int4 e = m.edges[m.slots[s].y >> 2];
                nbr[s] = e.x == i ? e.y : e.x;
            }
        }
        for (auto* v : {&tris, &edges, &halo}) v->reserve(8 * PATCH_NODES);
    }

    // breadth-first order of perm[b, e) (its nodes carry `from`) into queue, retagged `to`
    void order(int b, int e, int start, int from, int to) {
        int head = 0, tail = 0, scan = b;
        int i = start;
        for (;;) {
            tag[i] = to;
            queue[tail++] = i;
            for (; head < tail; ++head) {
                const int k = queue[head];
                for (int s = m.ring_off[k]; s < m.ring_off[k] + m.valence[k]; ++s)
                    if (tag[nbr[s]] == from) {
                        tag[nbr[s]] = to;
                        queue[tail++] = nbr[s];
                    }
            }
            if (tail == e - b) return;
            while (tag[perm[scan]] != from) ++scan;   // a subset in several pieces
            i = perm[scan];
        }
    }

    // perm[b, e) into k parts: cut the breadth-first order from a far node
    void cut(int b, int e, int k) {
        if (k <= 1 || e - b < 2) {
            emit(b, e);
            return;
        }
        const int t = next_tag;
        next_tag += 3;
        for (int i = b; i < e; ++i) tag[perm[i]] = t;
        order(b, e, perm[b], t, t + 1);
        order(b, e, queue[e - b - 1], t + 1, t + 2);
        std::copy(queue.begin(), queue.begin() + (e - b), perm.begin() + b);
        const int at = b + std::max(1, std::min(e - b - 1, (int)((long long)(e - b) * (k / 2) / k)));
        cut(b, at, k / 2);
        cut(at, e, k - k / 2);
    }

    void emit(int b, int e) {
        std::sort(perm.begin() + b, perm.begin() + e);
        const int* own = perm.data() + b;
        const int n_own = e - b;
        tris.clear();
        edges.clear();
        halo.clear();
        auto take = [](std::vector<int>& num, std::vector<int>& list, int x) {
            if (num[x] < 0) {
                num[x] = (int)list.size();
                list.push_back(x);
            }
        };
        int maxval = 0;
        for (int k = 0; k < n_own; ++k) {
            const int i = own[k];
            maxval = std::max(maxval, m.valence[i]);
            for (int s = m.ring_off[i]; s < m.ring_off[i] + m.valence[i]; ++s) {
                take(ltri, tris, m.slots[s].w);
                take(ledge, edges, m.slots[s].y >> 2);
                take(ledge, edges, m.slots[s].z >> 2);
            }
            lnode[i] = k;
        }
        for (int x : edges)
            for (int v : {m.edges[x].x, m.edges[x].y, m.edges[x].z, m.edges[x].w}) take(lnode, halo, v);
        PatchTab p = {};
        p.n_own = n_own;
        p.n_loc = n_own + (int)halo.size();
        p.n_tri = (int)tris.size();
        p.n_edge = (int)edges.size();
        p.rows = (maxval + 1) / 2;
        const bool fits = patch_bytes(p) <= PATCH_SMEM || n_own == 1;
        if (fits) {
            std::sort(halo.begin(), halo.end());
            for (size_t k = 0; k < halo.size(); ++k) lnode[halo[k]] = n_own + (int)k;
            p.loc0 = (int)out.loc.size();
            p.tri0 = (int)out.tri.size();
            p.edge0 = (int)out.edge.size();
            p.ring0 = (int)out.ring.size();
            out.loc.insert(out.loc.end(), own, own + n_own);
            out.loc.insert(out.loc.end(), halo.begin(), halo.end());
            auto two = [](int x, int y) { return (unsigned)x | ((unsigned)y << 16); };
            for (int t : tris) {
                const int32_t* v = m.tris + 3 * (size_t)t;
                // the patch of a triangle's first vertex adds its share of the cell's sums
                const unsigned owner = lnode[v[0]] < n_own ? 0x80000000u : 0u;
                out.tri.push_back(make_uint2(two(lnode[v[0]], lnode[v[1]]), (unsigned)lnode[v[2]] | owner));
            }
            for (int x : edges) {
                const int4 v = m.edges[x];
                out.edge.push_back(make_uint2(two(lnode[v.x], lnode[v.y]), two(lnode[v.z], lnode[v.w])));
            }
            out.tri_id.insert(out.tri_id.end(), tris.begin(), tris.end());
            out.edge_id.insert(out.edge_id.end(), edges.begin(), edges.end());
            // ring rows: row 0 the first edge of each half, row 1 + j its slot j
            const size_t width = 2 * (size_t)n_own;
            out.ring.resize(out.ring.size() + (size_t)(p.rows + 1) * width, make_uint2(RING_END, 0u));
            for (int k = 0; k < n_own; ++k) {
                const int i = own[k], r0 = m.ring_off[i], n = m.valence[i];
                auto from = [&](int j) {   // the edge to neighbour j, bit 15: i is its b
                    const int x = m.slots[r0 + (j < n ? j : j - n)].y >> 2;
                    return (unsigned)ledge[x] | (m.edges[x].x == i ? 0u : 0x8000u);
                };
                for (int half = 0; half < 2; ++half) {
                    uint2* row = out.ring.data() + p.ring0 + 2 * k + half;
                    const int j0 = half ? (n + 1) / 2 : 0, j1 = half ? n : (n + 1) / 2;
                    row[0] = make_uint2(from(j0), 0u);
                    for (int j = j0; j < j1; ++j)
                        row[(size_t)(1 + j - j0) * width] =
                            make_uint2(from(j + 1) | ((unsigned)ltri[m.slots[r0 + j].w] << 16),
                                       (unsigned)ledge[m.slots[r0 + j].z >> 2]);
                }
            }
            out.tab.push_back(p);
        }
        for (int k = 0; k < n_own; ++k) lnode[own[k]] = -1;
        for (int i : halo) lnode[i] = -1;
        for (int t : tris) ltri[t] = -1;
        for (int x : edges) ledge[x] = -1;
        if (!fits) cut(b, e, 2);
    }
};

}  // namespace

void build_patches(const MeshTables& m, PatchTables& out) {
    Cutter(m, out).cut(0, m.n, (m.n + PATCH_NODES - 1) / PATCH_NODES);
}

size_t patch_smem_bytes(const PatchTab& t) { return patch_bytes(t); }

cudaError_t launch_patch_rest(const PatchRest& r, int n_patches, cudaStream_t s) {
    if (n_patches <= 0) return cudaSuccess;
    k_patch_rest<<<n_patches, MB, 0, s>>>(r);
    return cudaGetLastError();
}

cudaError_t launch_membrane(const IbmArgs& a, cudaStream_t s) {
    if (a.n_patches <= 0) return cudaSuccess;
    // more patches than three blocks per SM hold: four per SM at 64 registers
    // (512x256x128 55.6 -> 51.4 us); fewer wait on each block's latency, which 80
    // registers shorten (256x128x64 cycle 71.1 -> 69.7 us)
    if (a.n_patches > 3 * a.sm_count) return launch_ex(k_membrane<4>, a.n_patches, MB, (size_t)a.patch_smem, s, a.pdl, a);
    return launch_ex(k_membrane<3>, a.n_patches, MB, (size_t)a.patch_smem, s, a.pdl, a);
}

}  // namespace lbibm
