// Geometry of a call on the mesh's static BVH topology, in two launches after
// the morph: pose, vertex normals and the refit of every treelet (a subtree of
// up to TREELET leaves, one block each) in the first, the nodes above the
// treelets in the second.
//
// What bounds it is latency, not bytes (13 MB at 70,789 triangles, 2 us of
// HBM): the form before this one (pose, face normals, vertex normals, then one
// thread per leaf climbing to the root with an atomic per level, then packing,
// then the plane bounds) was eight launches, each a chain of dependent loads
// through L2, 33 us of them the climb.  Here a treelet's triangles sit in shared
// memory, every node reduces its own run of them (its leaves are consecutive
// slots), so there is no order between the nodes and no atomic, and a block
// poses the vertices it needs itself instead of waiting for another launch.
// Measured (morph included, paper-scale face): 0.146 -> 0.067 ms; on the 5,120-triangle
// face 0.097 -> 0.043 ms.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "kernels.h"
#include "refit.cuh"

namespace {

constexpr int TREELET = 256;
// A node of more triangles than this is too curved for a plane bound to cull
// and keeps none (n = 0, h = 1).  Measured on the paper-scale face: with 1,024
// the forward is 0.04 ms slower, with 65,536 as long as with 4,096.
constexpr int PLANE_MAX = 4096;
constexpr int REFIT_THREADS = 256;
// a thread reduces a node of up to this many leaves, a warp together a larger one
constexpr int NODE_THREAD = 8;

struct Tri3 {
    float3 a, b, c;
};

// A treelet's triangles, one column per leaf (conflict-free by leaf), and its
// nodes' results.
struct TreeletShared {
    float v[9][TREELET];
    float leaf_plane[4][TREELET];
    float box[6][TREELET];           // internal node root + j
    float plane[4][TREELET];
};

FR_D Tri3 shared_tri(const TreeletShared& sh, int l) {
    return {f3(sh.v[0][l], sh.v[1][l], sh.v[2][l]), f3(sh.v[3][l], sh.v[4][l], sh.v[5][l]),
            f3(sh.v[6][l], sh.v[7][l], sh.v[8][l])};
}

// Box, area vector, height and magnitude of a run of triangles.
struct Reach {
    Box3 box;
    float3 m;
    FR_D void clear() {
        box.clear();
        m = f3(0.0f, 0.0f, 0.0f);
    }
    FR_D void add(const Tri3& t) {
        box.grow(padded_box(t.a, t.b, t.c));
        m += cross(t.b - t.a, t.c - t.a);
    }
};

FR_D void height_of(const Tri3& t, float3 n, float& h) {
    h = fmaxf(h, fmaxf(dot(n, t.a), fmaxf(dot(n, t.b), dot(n, t.c))));
}

FR_D float warp_min(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
FR_D float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
FR_D float warp_add(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

FR_D void warp_reach(Reach& r) {
    r.box.lo = f3(warp_min(r.box.lo.x), warp_min(r.box.lo.y), warp_min(r.box.lo.z));
    r.box.hi = f3(warp_max(r.box.hi.x), warp_max(r.box.hi.y), warp_max(r.box.hi.z));
    r.m = f3(warp_add(r.m.x), warp_add(r.m.y), warp_add(r.m.z));
}

FR_D void put_node(TreeletShared& sh, int j, const Box3& b, float4 p) {
    sh.box[0][j] = b.lo.x; sh.box[1][j] = b.lo.y; sh.box[2][j] = b.lo.z;
    sh.box[3][j] = b.hi.x; sh.box[4][j] = b.hi.y; sh.box[5][j] = b.hi.z;
    sh.plane[0][j] = p.x; sh.plane[1][j] = p.y; sh.plane[2][j] = p.z; sh.plane[3][j] = p.w;
}

// Box and plane of a child by its code within the treelet (root node, first leaf).
FR_D void get_child(const TreeletShared& sh, int code, int root, int first, Box3& b, float4& p) {
    if (code < 0) {
        const int l = ~code - first;
        const Tri3 t = shared_tri(sh, l);
        b = padded_box(t.a, t.b, t.c);
        p = make_float4(sh.leaf_plane[0][l], sh.leaf_plane[1][l], sh.leaf_plane[2][l], sh.leaf_plane[3][l]);
    } else {
        const int j = code - root;
        b.lo = f3(sh.box[0][j], sh.box[1][j], sh.box[2][j]);
        b.hi = f3(sh.box[3][j], sh.box[4][j], sh.box[5][j]);
        p = make_float4(sh.plane[0][j], sh.plane[1][j], sh.plane[2][j], sh.plane[3][j]);
    }
}

// A child's fields in its parent's record (side 0 or 1).
FR_D void store_child(BvhNode& nd, int side, const Box3& b, float4 p) {
    if (side == 0) {
        nd.a = make_float4(b.lo.x, b.lo.y, b.lo.z, b.hi.x);
        *reinterpret_cast<float2*>(&nd.b) = make_float2(b.hi.y, b.hi.z);
        nd.p0 = p;
    } else {
        *(reinterpret_cast<float2*>(&nd.b) + 1) = make_float2(b.lo.x, b.lo.y);
        nd.c = make_float4(b.lo.z, b.hi.x, b.hi.y, b.hi.z);
        nd.p1 = p;
    }
}

FR_D float3 posed(const float* vm, const float* R, const float* T, int i) {
    return pose_vertex(R, f3(vm[3 * i] - T[0], vm[3 * i + 1] - T[1], vm[3 * i + 2] - T[2]));
}

// Camera-space vertex i and its normal: the sum of its faces' un-normalised
// normals in face order (CSR), each recomputed from the face's posed vertices.
FR_D void vertex_and_normal(const DevItem& it, const float* R, const float* T, const int4* __restrict__ faces,
                            const int* __restrict__ off, const int* __restrict__ idx, int i) {
    const float* vm = it.v_model;
    const float3 p = posed(vm, R, T, i);
    it.v_cam[i] = make_float4(p.x, p.y, p.z, 0.0f);
    float3 m = f3(0.0f, 0.0f, 0.0f);
    const int k1 = off[i + 1];
    for (int k = off[i]; k < k1; ++k) {
        const int4 t = __ldg(&faces[idx[k]]);
        const float3 a = posed(vm, R, T, t.x), b = posed(vm, R, T, t.y), c = posed(vm, R, T, t.z);
        m = add_rn(m, face_normal(a, b, c));
    }
    it.vn[i] = vertex_normal(m);
}

FR_D void refit_treelet(const DevItem& it, TreeletShared& sh, const float* R, const float* T, float reach,
                        const int4* __restrict__ faces, const RefitTopology& topo, int k) {
    const Treelet tl = topo.treelets[k];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int n_nodes = tl.count - 1;
    if (t < tl.count) {
        const int s = tl.first + t, id = it.B.vals[s];
        const int4 fc = __ldg(&faces[id]);
        const Tri3 q = {posed(it.v_model, R, T, fc.x), posed(it.v_model, R, T, fc.y), posed(it.v_model, R, T, fc.z)};
        it.tris[3 * s] = make_float4(q.a.x, q.a.y, q.a.z, __int_as_float(id));
        it.tris[3 * s + 1] = make_float4(q.b.x, q.b.y, q.b.z, 0.0f);
        it.tris[3 * s + 2] = make_float4(q.c.x, q.c.y, q.c.z, 0.0f);
        it.slot_of[id] = s;
        const float w[9] = {q.a.x, q.a.y, q.a.z, q.b.x, q.b.y, q.b.z, q.c.x, q.c.y, q.c.z};
#pragma unroll
        for (int c = 0; c < 9; ++c) sh.v[c][t] = w[c];
        const float3 n = unit_or_zero(cross(q.b - q.a, q.c - q.a));
        float h = -INFINITY;
        height_of(q, n, h);
        const float4 p = plane_record(n, h, reach);
        sh.leaf_plane[0][t] = p.x; sh.leaf_plane[1][t] = p.y; sh.leaf_plane[2][t] = p.z; sh.leaf_plane[3][t] = p.w;
    }
    __syncthreads();
    // lane l of warp w owns node w + 8 l: the large nodes of the pre-order
    // numbering's first chain land in different warps
    {
        const int j = warp + (REFIT_THREADS / 32) * lane;
        int2 run = make_int2(0, 0);
        if (j < n_nodes) run = __ldg(&topo.runs[tl.code + j]);
        run.x -= tl.first;
        if (run.y > 0 && run.y <= NODE_THREAD) {
            Reach r;
            r.clear();
            for (int l = run.x; l < run.x + run.y; ++l) r.add(shared_tri(sh, l));
            const float3 n = unit_or_zero(r.m);
            float h = -INFINITY;
            for (int l = run.x; l < run.x + run.y; ++l) height_of(shared_tri(sh, l), n, h);
            put_node(sh, j, r.box, plane_record(n, h, reach));
        }
        unsigned big = __ballot_sync(0xffffffffu, run.y > NODE_THREAD);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const int f = __shfl_sync(0xffffffffu, run.x, src), c = __shfl_sync(0xffffffffu, run.y, src);
            Reach r;
            r.clear();
            for (int l = f + lane; l < f + c; l += 32) r.add(shared_tri(sh, l));
            warp_reach(r);
            const float3 n = unit_or_zero(r.m);
            float h = -INFINITY;
            for (int l = f + lane; l < f + c; l += 32) height_of(shared_tri(sh, l), n, h);
            h = warp_max(h);
            if (lane == src) {
                put_node(sh, j, r.box, plane_record(n, h, reach));
                if (j == 0) {                     // the treelet's area vector, for the nodes above
                    it.B.treelet_box[3 * k + 2] = make_float4(r.m.x, r.m.y, r.m.z, reach);
                }
            }
        }
        if (j == 0 && run.y <= NODE_THREAD) {     // a treelet of few leaves, or of one
            float3 m = f3(0.0f, 0.0f, 0.0f);
            for (int l = 0; l < tl.count; ++l) {
                const Tri3 q = shared_tri(sh, l);
                m += cross(q.b - q.a, q.c - q.a);
            }
            it.B.treelet_box[3 * k + 2] = make_float4(m.x, m.y, m.z, reach);
        }
    }
    __syncthreads();
    if (t < n_nodes) {
        const int node = tl.code + t;
        const int c0 = it.B.child[2 * node], c1 = it.B.child[2 * node + 1];
        Box3 b0, b1;
        float4 p0, p1;
        get_child(sh, c0, tl.code, tl.first, b0, p0);
        get_child(sh, c1, tl.code, tl.first, b1, p1);
        BvhNode& nd = it.nodes[node];
        nd.a = make_float4(b0.lo.x, b0.lo.y, b0.lo.z, b0.hi.x);
        nd.b = make_float4(b0.hi.y, b0.hi.z, b1.lo.x, b1.lo.y);
        nd.c = make_float4(b1.lo.z, b1.hi.x, b1.hi.y, b1.hi.z);
        nd.d = make_int4(c0, c1, 0, 0);
        nd.p0 = p0;
        nd.p1 = p1;
    }
    if (t == 0) {
        Box3 b;
        float4 p;
        get_child(sh, tl.code, tl.code, tl.first, b, p);
        it.B.treelet_box[3 * k] = make_float4(b.lo.x, b.lo.y, b.lo.z, 0.0f);
        it.B.treelet_box[3 * k + 1] = make_float4(b.hi.x, b.hi.y, b.hi.z, 0.0f);
        if (tl.up >= 0) {
            store_child(it.nodes[tl.up >> 1], tl.up & 1, b, p);
        } else if (tl.code < 0) {                 // the tree is one leaf: a root with it as both children
            // (the second's inverted box is met by every ray, whose slabs it swaps: the leaf is tested twice)
            BvhNode& nd = it.nodes[0];
            nd.a = make_float4(b.lo.x, b.lo.y, b.lo.z, b.hi.x);
            nd.b = make_float4(b.hi.y, b.hi.z, INFINITY, INFINITY);
            nd.c = make_float4(INFINITY, -INFINITY, -INFINITY, -INFINITY);
            nd.d = make_int4(~0, ~0, 0, 0);
            nd.p0 = nd.p1 = make_float4(0.0f, 0.0f, 0.0f, 1.0f);
        }
    }
}

// Bounds the distance of every vertex of the posed mesh from the camera (a whole
// warp calls): the mean's greatest length plus each basis column's times its
// coefficient (1%: the sums' rounding and the BF16 morph's), moved by the
// translation.
FR_D float mesh_reach(const DevItem& it, const float* __restrict__ reach) {
    const int lane = threadIdx.x & 31;
    float r = lane == 0 ? reach[0] : 0.0f;
    for (int k = lane; k < it.S.K; k += 32) r += fabsf(it.P.coef[k]) * reach[1 + k];
    const float* t = it.P.trans;
    return 1.01f * (warp_add(r) + sqrtf(t[0] * t[0] + t[1] * t[1] + t[2] * t[2]));
}

__global__ void __launch_bounds__(REFIT_THREADS) k_pose_refit(const DevItem* items, const int4* __restrict__ faces,
                                                              const int* __restrict__ off, const int* __restrict__ idx,
                                                              RefitTopology topo, int N) {
    __shared__ TreeletShared sh;
    __shared__ float R[9], T[3], reach;
    const DevItem& it = items[blockIdx.y];
    if (threadIdx.x == 0) {
        euler_R(it.P.rot, R);
        T[0] = it.P.trans[0]; T[1] = it.P.trans[1]; T[2] = it.P.trans[2];
    } else if (threadIdx.x >> 5 == 1 && (int)blockIdx.x < topo.n_treelets) {
        const float r = mesh_reach(it, topo.reach);
        if ((threadIdx.x & 31) == 0) reach = r;
    }
    __syncthreads();
    if ((int)blockIdx.x < topo.n_treelets) {
        refit_treelet(it, sh, R, T, reach, faces, topo, blockIdx.x);
    } else {
        const int i = ((int)blockIdx.x - topo.n_treelets) * REFIT_THREADS + threadIdx.x;
        if (i < N) vertex_and_normal(it, R, T, faces, off, idx, i);
    }
}

constexpr int TOP_THREADS = 128;

// One block per node above the treelets: its box and area vector over its run
// of treelets, its height over its triangles' vertices (up to PLANE_MAX
// triangles), into its parent's record.
__global__ void __launch_bounds__(TOP_THREADS) k_refit_top(const DevItem* items, RefitTopology topo) {
    __shared__ float red[TOP_THREADS / 32][9];
    const DevItem& it = items[blockIdx.y];
    const TopNode u = topo.tops[blockIdx.x];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) it.nodes[u.node].d = make_int4(it.B.child[2 * u.node], it.B.child[2 * u.node + 1], 0, 0);
    if (u.up < 0) return;                          // the root: nothing holds its box
    Reach r;
    r.clear();
    for (int k = u.treelet + t; k < u.treelet + u.n_treelets; k += TOP_THREADS) {
        const float4 lo = it.B.treelet_box[3 * k], hi = it.B.treelet_box[3 * k + 1], m = it.B.treelet_box[3 * k + 2];
        r.box.grow({xyz(lo), xyz(hi)});
        r.m += xyz(m);
    }
    warp_reach(r);
    if (lane == 0) {
        const float v[9] = {r.box.lo.x, r.box.lo.y, r.box.lo.z, r.box.hi.x, r.box.hi.y, r.box.hi.z, r.m.x, r.m.y, r.m.z};
        for (int c = 0; c < 9; ++c) red[warp][c] = v[c];
    }
    __syncthreads();
    r.clear();
    for (int w = 0; w < TOP_THREADS / 32; ++w) {
        r.box.grow({f3(red[w][0], red[w][1], red[w][2]), f3(red[w][3], red[w][4], red[w][5])});
        r.m += f3(red[w][6], red[w][7], red[w][8]);
    }
    const bool bound = u.count <= PLANE_MAX;       // block-uniform
    const float3 n = bound ? unit_or_zero(r.m) : f3(0.0f, 0.0f, 0.0f);
    float h = -INFINITY;
    if (bound) {
        for (int s = u.first + t; s < u.first + u.count; s += TOP_THREADS)
            height_of({xyz(it.tris[3 * s]), xyz(it.tris[3 * s + 1]), xyz(it.tris[3 * s + 2])}, n, h);
        h = warp_max(h);
        __syncthreads();                           // red is read above
        if (lane == 0) red[warp][0] = h;
        __syncthreads();
    }
    if (t == 0) {
        if (bound)
            for (int w = 0; w < TOP_THREADS / 32; ++w) h = fmaxf(h, red[w][0]);
        const float reach = it.B.treelet_box[3 * u.treelet + 2].w;
        store_child(it.nodes[u.up >> 1], u.up & 1, r.box, plane_record(n, h, reach));
    }
}

}  // namespace

// Treelets and the nodes above them of a pre-order topology (host).
void build_refit_lists(const BvhTopology& topo, int T, std::vector<int2>& runs, std::vector<Treelet>& treelets,
                       std::vector<TopNode>& tops) {
    runs.assign((size_t)std::max(T - 1, 1), make_int2(0, 1));
    treelets.clear();
    tops.clear();
    if (T == 1) {
        treelets.push_back(Treelet{~0, 0, 1, -1});
        return;
    }
    // children follow their parent in the numbering
    for (int i = T - 2; i >= 0; --i) {
        int first = T, count = 0;
        for (int q = 0; q < 2; ++q) {
            const int c = topo.child[2 * (size_t)i + q];
            first = std::min(first, c < 0 ? ~c : runs[c].x);
            count += c < 0 ? 1 : runs[c].y;
        }
        runs[i] = make_int2(first, count);
    }
    // pre-order walk: treelets come out in slot order, so a node's are consecutive
    struct Visit { int code, up; };
    std::vector<Visit> stack{{0, -1}};
    while (!stack.empty()) {
        const Visit v = stack.back();
        stack.pop_back();
        const int count = v.code < 0 ? 1 : runs[v.code].y, first = v.code < 0 ? ~v.code : runs[v.code].x;
        if (count <= TREELET) {
            treelets.push_back(Treelet{v.code, first, count, v.up});
            continue;
        }
        tops.push_back(TopNode{v.code, v.up, first, count, (int)treelets.size(), 0});
        stack.push_back({topo.child[2 * (size_t)v.code + 1], 2 * v.code + 1});
        stack.push_back({topo.child[2 * (size_t)v.code], 2 * v.code});
    }
    for (TopNode& u : tops) {
        int k = u.treelet;
        while (k < (int)treelets.size() && treelets[k].first < u.first + u.count) ++k;
        u.n_treelets = k - u.treelet;
    }
}

void launch_pose_refit(const DevItem* items, int n, const int4* faces, const int* vf_off, const int* vf_idx,
                       const RefitTopology& topo, int N, cudaStream_t st) {
    const int pose_blocks = (N + REFIT_THREADS - 1) / REFIT_THREADS;
    k_pose_refit<<<dim3(topo.n_treelets + pose_blocks, n), REFIT_THREADS, 0, st>>>(items, faces, vf_off, vf_idx, topo, N);
    fr_count_launches(1);
    if (topo.n_tops > 0) {
        k_refit_top<<<dim3(topo.n_tops, n), TOP_THREADS, 0, st>>>(items, topo);
        fr_count_launches(1);
    }
}
