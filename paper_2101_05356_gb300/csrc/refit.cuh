// Shared by the two ways a call's BVH gets its boxes and plane bounds (the
// static topology's refit.cu, the per-call rebuild's lbvh.cu) and by the pose.
#pragma once
#include "common.cuh"

FR_D unsigned ordered(float f) {
    const unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
FR_D float unordered(unsigned u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// R = Rz(t2) Ry(t1) Rx(t0), row-major
FR_D void euler_R(const float* rot, float R[9]) {
    float sx, cx, sy, cy, sz, cz;
    sincosf(rot[0], &sx, &cx);
    sincosf(rot[1], &sy, &cy);
    sincosf(rot[2], &sz, &cz);
    R[0] = cz * cy; R[1] = cz * sy * sx - sz * cx; R[2] = cz * sy * cx + sz * sx;
    R[3] = sz * cy; R[4] = sz * sy * sx + cz * cx; R[5] = sz * sy * cx - cz * sx;
    R[6] = -sy;     R[7] = cy * sx;                R[8] = cy * cx;
}

// The geometry of a call is computed by different kernels for the static
// topology and for the per-call rebuild, and images are bitwise the same either
// way, so the operations whose fusing the compiler could choose are spelled out.

// a x + b y + c z
FR_D float row_rn(float a, float x, float b, float y, float c, float z) {
    return __fmaf_rn(c, z, __fmaf_rn(a, x, __fmul_rn(b, y)));
}

// v' = R^T w
FR_D float3 pose_vertex(const float* R, float3 w) {
    return f3(row_rn(R[0], w.x, R[3], w.y, R[6], w.z), row_rn(R[1], w.x, R[4], w.y, R[7], w.z),
              row_rn(R[2], w.x, R[5], w.y, R[8], w.z));
}

FR_D float det_rn(float a, float b, float c, float d) { return __fmaf_rn(a, b, -__fmul_rn(c, d)); }

// (b - a) x (c - a)
FR_D float3 face_normal(float3 a, float3 b, float3 c) {
    const float3 u = f3(__fsub_rn(b.x, a.x), __fsub_rn(b.y, a.y), __fsub_rn(b.z, a.z));
    const float3 w = f3(__fsub_rn(c.x, a.x), __fsub_rn(c.y, a.y), __fsub_rn(c.z, a.z));
    return f3(det_rn(u.y, w.z, u.z, w.y), det_rn(u.z, w.x, u.x, w.z), det_rn(u.x, w.y, u.y, w.x));
}

FR_D float3 add_rn(float3 a, float3 b) { return f3(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z)); }

// unit normal of a vertex and the length of the sum m of its faces' normals
FR_D float4 vertex_normal(float3 m) {
    const float len = __fsqrt_rn(__fmaf_rn(m.z, m.z, __fmaf_rn(m.y, m.y, __fmul_rn(m.x, m.x))));
    const float inv = len > 0.0f ? 1.0f / len : 0.0f;
    return make_float4(__fmul_rn(m.x, inv), __fmul_rn(m.y, inv), __fmul_rn(m.z, inv), len);
}

struct Box3 {
    float3 lo, hi;
    FR_D void clear() {
        lo = f3(INFINITY, INFINITY, INFINITY);
        hi = f3(-INFINITY, -INFINITY, -INFINITY);
    }
    FR_D void grow(const Box3& b) {
        lo = f3(fminf(lo.x, b.lo.x), fminf(lo.y, b.lo.y), fminf(lo.z, b.lo.z));
        hi = f3(fmaxf(hi.x, b.hi.x), fmaxf(hi.y, b.hi.y), fmaxf(hi.z, b.hi.z));
    }
};

// A triangle's box, padded so that the FP32 slab test never culls a triangle
// the exact test hits.
FR_D Box3 padded_box(float3 a, float3 b, float3 c) {
    const float3 lo = f3(fminf(a.x, fminf(b.x, c.x)), fminf(a.y, fminf(b.y, c.y)), fminf(a.z, fminf(b.z, c.z)));
    const float3 hi = f3(fmaxf(a.x, fmaxf(b.x, c.x)), fmaxf(a.y, fmaxf(b.y, c.y)), fmaxf(a.z, fmaxf(b.z, c.z)));
    return {f3(lo.x - 1e-5f - 1e-6f * fabsf(lo.x), lo.y - 1e-5f - 1e-6f * fabsf(lo.y), lo.z - 1e-5f - 1e-6f * fabsf(lo.z)),
            f3(hi.x + 1e-5f + 1e-6f * fabsf(hi.x), hi.y + 1e-5f + 1e-6f * fabsf(hi.y), hi.z + 1e-5f + 1e-6f * fabsf(hi.z))};
}

FR_D float3 unit_or_zero(float3 m) {
    const float l = length(m);
    return l > 0.0f && l < INFINITY ? m * (1.0f / l) : f3(0.0f, 0.0f, 0.0f);
}

// The plane bound of a node with unit mean normal n (zero: none) and greatest
// height h = max n . x over its vertices.  The pad covers the rounding of both
// sides of the test, a few 2^-24 of the coordinates' magnitude: not of the
// node's only, since a shadow ray's height is rounded at its origin's, which may
// lie far beyond the node, so `reach` bounds the distance of the whole mesh from
// the camera (17 roundings of it, 1e-6, cover the three products of either dot
// product, the ends' and the sum's).
FR_D float4 plane_record(float3 n, float h, float reach) {
    const bool none = n.x == 0.0f && n.y == 0.0f && n.z == 0.0f;
    return make_float4(n.x, n.y, n.z, none ? 1.0f : h + 1e-5f + 1e-6f * reach);
}
