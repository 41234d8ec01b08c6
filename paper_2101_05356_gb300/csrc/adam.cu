// Fused multi-tensor Adam with the regularisers of the two-stage optimisation
// (Sec. 4, Eq. loss1 and loss3): shape prior, light prior, soft box
// constraints (expression, intensities, light-stage geometry, textures),
// texture symmetry, chromaticity consistency and smoothness.  Two launches
// update every parameter group of a stage: the first adds the regulariser
// gradient (texture stencils read neighbours, so x must not change yet) to the
// render gradient and updates the moments, a thread to a texel or element; the
// second applies the Adam step with per-group learning rate.
//
// Bound by HBM (x, g, m, v and the references read, m, v and x written: 58 MB
// for 512 x 512 textures, 8.5 us) and, in the first launch, by the quotients of
// the chromaticity term.  With one thread per element and the energies in FP64
// that launch took 103 us there, nearly all of it FP64 instructions; measured
// now 22 us, and 8 us the second (13.7 us with one element a thread).
#include <cfloat>

#include "../../include/facert.h"
#include "common.cuh"
#include "kernels.h"

namespace {

constexpr int ADAM_THREADS = 256;

struct GroupTable {
    fr_opt_group g[FR_MAX_OPT_GROUPS];
    int block_start[FR_MAX_OPT_GROUPS + 1];      // first block of each group: moments, update
    int apply_start[FR_MAX_OPT_GROUPS + 1];
    int n_groups;
    float beta1, beta2, eps;
    float bc1[FR_MAX_OPT_GROUPS], bc2[FR_MAX_OPT_GROUPS];   // bias corrections 1 - beta^t per group
};

FR_D float sgnf(float x) { return (float)((x > 0.0f) - (x < 0.0f)); }

// Regulariser gradient and energy contribution of element i of group G (the
// texture groups: texel_grad).
FR_D float reg_grad(const fr_opt_group& G, int i, float x, double* energy) {
    float g = 0.0f;
    double e = 0.0;
    switch (G.kind) {
    case FR_GROUP_COEF: {
        if (i < G.n_prior) {                       // w_i sum (alpha_k / sigma_k)^2, sigma_k = 1
            g += 2.0f * G.w_prior * x;
            e += (double)G.w_prior * x * x;
        } else {                                   // soft box delta in [0, 1]
            const float lo = fminf(x, 0.0f), hi = fmaxf(x - 1.0f, 0.0f);
            g += 2.0f * G.w_box * (lo + hi);
            e += (double)G.w_box * (lo * lo + hi * hi);
        }
        break;
    }
    case FR_GROUP_LIGHT: {                         // w1 sum_j |I_j - m_j|^2, I = scale * i, m = mean(I) fixed
        const int j = i / 3;
        float sc;
        if (G.aux) {
            sc = G.aux[j];
        } else {                                   // scale d^2 / a from the stage geometry [d | a | p]
            const float d = G.aux2[j], a = G.aux2[G.n / 3 + j];
            sc = a > 0.0f ? d * d / a : 0.0f;
        }
        const float* base = G.x + 3 * j;
        const float m = sc * (base[0] + base[1] + base[2]) * (1.0f / 3.0f);
        const float d = sc * x - m;
        g += 2.0f * G.w_prior * d * sc;
        e += (double)G.w_prior * d * d;
        const float lo = fminf(x, 0.0f);          // soft box i > 0
        g += 2.0f * G.w_box * lo;
        e += (double)G.w_box * lo * lo;
        break;
    }
    case FR_GROUP_STAGE: {                         // light geometry [d | a | p0 p1] of N_L lights
        const int NL = G.n / 4;
        const float* X = G.x;
        if (i < 2 * NL) {
            const int j = i < NL ? i : i - NL;
            const float d = X[j], a = X[NL + j];
            float dE_ds = 0.0f;                    // light prior through s = d^2 / a
            if (a > 0.0f) {
                const float s = d * d / a;
                const float* ij = G.aux + 3 * j;
                const float m = s * (ij[0] + ij[1] + ij[2]) * (1.0f / 3.0f);
                for (int c = 0; c < 3; ++c) dE_ds += (s * ij[c] - m) * ij[c];
                dE_ds *= 2.0f * G.w_prior;
            }
            if (i < NL) {                          // d: prior, soft box d >= 0
                if (a > 0.0f) g += dE_ds * 2.0f * d / a;
                const float lo = fminf(d, 0.0f);
                g += 2.0f * G.w_box * lo;
                e += (double)G.w_box * lo * lo;
            } else {                               // a: prior, soft box [0, 1], inside-face term through sqrt(a)
                if (a > 0.0f) g += dE_ds * (-(d * d / a) / a);
                const float lo = fminf(a, 0.0f), hi = fmaxf(a - 1.0f, 0.0f);
                g += 2.0f * G.w_box * (lo + hi);
                e += (double)G.w_box * (lo * lo + hi * hi);
                if (a > 0.0f) {
                    const float ra = sqrtf(a), r = ra * (1.0f / 3.0f);
                    const float p0 = X[2 * NL + 2 * j], p1 = X[2 * NL + 2 * j + 1];
                    const float in = fminf(p0 - r, 0.0f) + fminf(p1 - r, 0.0f) + fminf(1.0f - p0 - p1 - r, 0.0f);
                    g += 2.0f * G.w_box * in * (-1.0f / (6.0f * ra));
                }
            }
        } else {                                   // p_jm: corners inside the homothetic face
            const int q = i - 2 * NL, j = q >> 1, mm = q & 1;
            const float a = X[NL + j];
            const float r = sqrtf(fmaxf(a, 0.0f)) * (1.0f / 3.0f);
            const float p0 = X[2 * NL + 2 * j], p1 = X[2 * NL + 2 * j + 1];
            const float in0 = fminf(p0 - r, 0.0f), in1 = fminf(p1 - r, 0.0f), in2 = fminf(1.0f - p0 - p1 - r, 0.0f);
            g += 2.0f * G.w_box * ((mm == 0 ? in0 : in1) - in2);
            if (mm == 0) e += (double)G.w_box * ((double)in0 * in0 + (double)in1 * in1 + (double)in2 * in2);
        }
        break;
    }
    default:
        break;
    }
    *energy += e;
    return g;
}

// An unevaluated sum hi + mid + lo of three FP32 numbers: the texture energies
// are summed in these instead of in FP64, whose pipe takes 64 cycles per warp
// instruction.  Squares enter exactly (a product with its rounding error, by
// FMA), a weight once per texel, and a sum keeps about 72 bits, more than the 53
// of FP64 (two numbers would keep 48).
struct Triple {
    float hi = 0.0f, mid = 0.0f, lo = 0.0f;
};

FR_D float two_sum(float& s, float x) {            // s += x, returns the rounding error (Knuth)
    const float t = __fadd_rn(s, x), b = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b));
    s = t;
    return e;
}

FR_D void add_mid(Triple& s, float x) { s.lo = __fadd_rn(s.lo, two_sum(s.mid, x)); }
FR_D void add(Triple& s, float x) { add_mid(s, two_sum(s.hi, x)); }

FR_D Triple square(float x) {
    const float q = __fmul_rn(x, x);
    return {q, __fmaf_rn(x, x, -q), 0.0f};
}

FR_D void add_square(Triple& s, float x) {         // s += x^2
    const Triple q = square(x);
    add(s, q.hi);
    add_mid(s, q.mid);
}

FR_D void add_weighted(Triple& s, float w, const Triple& x) {      // s += w x
    const float p = __fmul_rn(w, x.hi), q = __fmul_rn(w, x.mid);
    add(s, p);
    add_mid(s, __fmaf_rn(w, x.hi, -p));
    add_mid(s, q);
    s.lo = __fadd_rn(s.lo, __fmaf_rn(w, x.lo, __fmaf_rn(w, x.mid, -q)));
}

// A texel's energy and the greatest magnitude that entered it.
struct Energy {
    Triple sum;
    float top = 0.0f;
    FR_D void saw(float x) { top = fmaxf(top, fabsf(x)); }
};

// FP32 holds a texel's energy exactly enough unless it is not finite, so large
// that the warp's 32 might overflow together, or so small that the rounding
// errors of its products underflow (below 2^-149: of no account beside 2^-90).
FR_D bool needs_64(const Energy& e) {
    const float a = fabsf(e.sum.hi);
    return !(a < FLT_MAX / 64.0f) || (a < 0x1p-90f && e.top > 0.0f);
}

// A warp's sum: (high 2^-21 + low 2^-42) in units of 2^(exponent - 147).
struct WarpSum {
    long long high;
    int low;
    unsigned exponent;
};

// The sum over the warp's lanes (the whole warp calls; numbers that needs_64
// accepts, so hi is 0 or in [2^-90, 2^122)): integers of three limbs of 21 bits
// below the greatest lane's power of two, added by the warp's integer reduction
// (20 instructions; a butterfly of five Triple additions takes 120).  63 bits
// below the greatest lane; mid is under 2^-20 and lo under 2^-40 of hi (a texel
// has some 20 terms), so 32 lanes' limbs stay below 2^28.
FR_D WarpSum warp_sum(const Triple& x) {
    const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(x.hi)));
    const unsigned exponent = max(top >> 23, 37u);                             // 37 .. 248
    const float limb = 0x1p21f, scale = __uint_as_float((274u - exponent) << 23);   // |hi| scale < 2^21
    float a = x.hi * scale, b = x.mid * scale * limb;
    const int i1 = __float2int_rn(a);
    a = (a - (float)i1) * limb;
    const int i2 = __float2int_rn(a), j2 = __float2int_rn(b);
    a = (a - (float)i2) * limb;
    b = (b - (float)j2) * limb;
    const int i3 = __float2int_rn(a + b + x.lo * scale * limb * limb);
    const long long high = ((long long)__reduce_add_sync(0xffffffffu, i1) << 21) + __reduce_add_sync(0xffffffffu, i2 + j2);
    return {high, __reduce_add_sync(0xffffffffu, i3), exponent};
}

FR_D double value(const WarpSum& s) {
    return ((double)s.high + (double)s.low * 0x1p-21) * (double)__uint_as_float((s.exponent - 20u) << 23) * 0x1p-21;
}

// The energy of texel t in FP64, for the texels of needs_64: the terms of
// texel_grad, each neighbouring pair at its left or upper texel.
__device__ __noinline__ double texel_energy64(const fr_opt_group& G, int C, int t) {
    const int M = G.width;
    const int row = t / M, col = t - row * M;
    const float* X = G.x;
    const float* x = X + (size_t)t * C;
    double e = 0.0;
    for (int c = 0; c < C; ++c) {
        if (G.w_smooth != 0.0f) {
            const int nb[2] = {t + 1, t + M};
            const bool in[2] = {col < M - 1, row < M - 1};
            for (int k = 0; k < 2; ++k)
                if (in[k]) {
                    const double d = x[c] - X[(size_t)nb[k] * C + c];
                    e += 2.0 * (double)G.w_smooth * d * d;
                }
        }
        if (G.w_sym != 0.0f) e += (double)G.w_sym * fabsf(x[c] - X[((size_t)row * M + M - 1 - col) * C + c]);
        if (G.w_box != 0.0f) {
            const double lo = fminf(x[c], 0.0f), hi = fmaxf(x[c] - 1.0f, 0.0f);
            e += (double)G.w_box * (lo * lo + hi * hi);
        }
    }
    if (C == 3 && G.w_chroma != 0.0f && G.aux) {
        const float* q = G.aux + (size_t)t * 3;
        const float S = x[0] + x[1] + x[2] + 1e-6f, S0 = q[0] + q[1] + q[2] + 1e-6f;
        for (int c = 0; c < 3; ++c) e += (double)G.w_chroma * fabsf(x[c] / S - q[c] / S0);
    }
    return e;
}

// Texture regularisers of texel t of a group of C channels: gradients g[C] of
// its channels x[C], energies into e.  One thread takes a whole texel, so the
// chromaticity's sums and quotients are formed once for its channels.  The
// smoothness counts each neighbouring pair twice: its energy is taken once, at
// the left or upper texel, with twice the weight.
template <int C, bool ENERGY>
FR_D void texel_grad(const fr_opt_group& G, int t, const float (&x)[C], float (&g)[C], Energy& e) {
    const int M = G.width;
    const int row = t / M, col = t - row * M;
    const float* X = G.x;
    if (G.w_smooth != 0.0f) {                  // sum_i sum_{j in N4(i)} |X_j - X_i|^2
        Triple sq;
        const int nb[4] = {t - 1, t + 1, t - M, t + M};
        const bool in[4] = {col > 0, col < M - 1, row > 0, row < M - 1};
#pragma unroll
        for (int c = 0; c < C; ++c) {
            float s = 0.0f, d[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                d[k] = in[k] ? x[c] - X[(size_t)nb[k] * C + c] : 0.0f;
                s += d[k];
            }
            g[c] += 4.0f * G.w_smooth * s;
            if (ENERGY) {
                if (c == 0) sq = square(d[1]);
                else add_square(sq, d[1]);
                add_square(sq, d[3]);
                e.saw(d[1]);
                e.saw(d[3]);
            }
        }
        if (ENERGY) add_weighted(e.sum, 2.0f * G.w_smooth, sq);
    }
    if (G.w_sym != 0.0f) {                     // sum |X(x) - X(flip x)|, flip: column -> M - 1 - column
        const int fc = M - 1 - col;
        if (fc != col) {
            Triple ab;
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const float d = x[c] - X[((size_t)row * M + fc) * C + c];
                g[c] += 2.0f * G.w_sym * sgnf(d);
                if (ENERGY) {
                    if (c == 0) ab.hi = fabsf(d);
                    else add(ab, fabsf(d));
                    e.saw(d);
                }
            }
            if (ENERGY) add_weighted(e.sum, G.w_sym, ab);
        }
    }
    if (C == 3 && G.w_chroma != 0.0f && G.aux) {   // sum |kappa(X) - kappa(X0)|, kappa(c) = c / (sum c + 1e-6)
        const float* q = G.aux + (size_t)t * 3;
        const float S = x[0] + x[1] + x[2] + 1e-6f, S0 = q[0] + q[1] + q[2] + 1e-6f;
        float kk[3], sg[3];
        Triple ab;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            kk[k] = x[k] / S;
            const float d = kk[k] - q[k] / S0;
            sg[k] = sgnf(d);
            if (ENERGY) {
                if (k == 0) ab.hi = fabsf(d);
                else add(ab, fabsf(d));
                e.saw(d);
            }
        }
        if (ENERGY) add_weighted(e.sum, G.w_chroma, ab);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float gc = 0.0f;
#pragma unroll
            for (int k = 0; k < 3; ++k) gc += sg[k] * (((k == c) ? 1.0f : 0.0f) - kk[k]) / S;
            g[c] += G.w_chroma * gc;
        }
    }
    if (G.w_box != 0.0f) {                     // soft box [0, 1]
        Triple sq;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const float lo = fminf(x[c], 0.0f), hi = fmaxf(x[c] - 1.0f, 0.0f);
            g[c] += 2.0f * G.w_box * (lo + hi);
            if (ENERGY && (lo != 0.0f || hi != 0.0f)) {     // one of them is 0
                add_square(sq, lo + hi);
                e.saw(lo + hi);
            }
        }
        if (ENERGY) add_weighted(e.sum, G.w_box, sq);
    }
}

FR_D void update_moments(const GroupTable& T, const fr_opt_group& G, size_t i, float g) {
    const float m = T.beta1 * G.m[i] + (1.0f - T.beta1) * g;
    const float v = T.beta2 * G.v[i] + (1.0f - T.beta2) * g * g;
    G.m[i] = m;
    G.v[i] = v;
}

template <int C, bool ENERGY>
FR_D void texel_moments(const GroupTable& T, const fr_opt_group& G, int t, Energy& e) {
    float x[C], g[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
        x[c] = G.x[(size_t)t * C + c];
        g[c] = 0.0f;
    }
    texel_grad<C, ENERGY>(G, t, x, g, e);
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const size_t i = (size_t)t * C + c;
        update_moments(T, G, i, (G.g ? G.g[i] : 0.0f) + g[c]);
    }
}

// Pass 1: gradient (render + regularisers) into m/v, reading x only; pass 2
// applies the parameter update, so stencils read the pre-step values.
FR_D int group_from(const int* start, int n_groups) {
    int lo = 0, hi = n_groups - 1;            // last group whose start <= blockIdx.x
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (start[mid] <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
    }
    return lo;
}

FR_D int group_of_block(const GroupTable& T) { return group_from(T.block_start, T.n_groups); }
FR_D int group_of_apply_block(const GroupTable& T) { return group_from(T.apply_start, T.n_groups); }

// A group's blocks cover its units: the texels of a texture group, the elements
// of any other.
template <bool ENERGY>
__global__ void __launch_bounds__(ADAM_THREADS) k_adam_moments(GroupTable T, double* energy) {
    __shared__ double part[ADAM_THREADS / 32];
    __shared__ WarpSum sums[ADAM_THREADS / 32];
    const int gi = group_of_block(T);
    const fr_opt_group& G = T.g[gi];
    const int i = (blockIdx.x - T.block_start[gi]) * ADAM_THREADS + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool texture = G.kind == FR_GROUP_TEX_RGB || G.kind == FR_GROUP_TEX_MONO;   // block-uniform
    double e = 0.0;
    if (texture) {
        Energy p;
        if (G.kind == FR_GROUP_TEX_RGB) {
            if (i < G.n / 3) texel_moments<3, ENERGY>(T, G, i, p);
        } else if (i < G.n) {
            texel_moments<1, ENERGY>(T, G, i, p);
        }
        if (ENERGY) {
            if (needs_64(p)) {
                e = texel_energy64(G, G.kind == FR_GROUP_TEX_RGB ? 3 : 1, i);
                p.sum = Triple();
            }
            if (__any_sync(0xffffffffu, e != 0.0))
                for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
            const WarpSum sum = warp_sum(p.sum);
            if (lane == 0) sums[warp] = sum;
        }
    } else {
        if (i < G.n) {
            const float x = G.x[i];
            float g = G.g ? G.g[i] : 0.0f;
            g += reg_grad(G, i, x, &e);
            update_moments(T, G, i, g);
        }
        if (ENERGY)
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    }
    if (ENERGY) {
        if (lane == 0) part[warp] = e;
        __syncthreads();
        // one warp turns the warps' sums into FP64, a lane to each: 2 FP64 instructions a warp instead of 9
        // (512 x 512 textures: 21.8 us against 26.7)
        if (warp == 0) {
            e = lane < ADAM_THREADS / 32 ? part[lane] : 0.0;
            if (texture && lane < ADAM_THREADS / 32) e += value(sums[lane]);
            for (int o = ADAM_THREADS / 64; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
            if (lane == 0 && e != 0.0) atomicAdd(energy, e);
        }
    }
}

// One element's update x - lr mh / (sqrt(vh) + eps), clamped.
FR_D float adam_step(const fr_opt_group& G, const GroupTable& T, int gi, float x, float m, float v) {
    const float mh = m / T.bc1[gi], vh = v / T.bc2[gi];
    x = x - G.lr * mh / (sqrtf(vh) + T.eps);
    if (G.clamp_lo < G.clamp_hi) x = fminf(fmaxf(x, G.clamp_lo), G.clamp_hi);
    return x;
}

// Four elements a thread, by 16-byte loads where the group's arrays allow.
__global__ void __launch_bounds__(ADAM_THREADS) k_adam_apply(GroupTable T) {
    const int gi = group_of_apply_block(T);
    const fr_opt_group& G = T.g[gi];
    const long i = ((long)(blockIdx.x - T.apply_start[gi]) * ADAM_THREADS + threadIdx.x) * 4;
    if (i >= G.n) return;
    const bool wide = ((reinterpret_cast<uintptr_t>(G.x) | reinterpret_cast<uintptr_t>(G.m) |
                        reinterpret_cast<uintptr_t>(G.v)) & 15u) == 0;         // group-uniform
    if (wide && i + 4 <= G.n) {
        float4 x = *reinterpret_cast<const float4*>(G.x + i);
        const float4 m = *reinterpret_cast<const float4*>(G.m + i), v = *reinterpret_cast<const float4*>(G.v + i);
        x.x = adam_step(G, T, gi, x.x, m.x, v.x);
        x.y = adam_step(G, T, gi, x.y, m.y, v.y);
        x.z = adam_step(G, T, gi, x.z, m.z, v.z);
        x.w = adam_step(G, T, gi, x.w, m.w, v.w);
        *reinterpret_cast<float4*>(G.x + i) = x;
        return;
    }
    for (long k = i; k < min(i + 4, (long)G.n); ++k) G.x[k] = adam_step(G, T, gi, G.x[k], G.m[k], G.v[k]);
}

}  // namespace

extern "C" fr_status fr_adam(const fr_opt_group* groups, int32_t n_groups, int32_t step, float beta1, float beta2,
                             float eps, double* reg_energy, void* stream) {
    if (!groups || n_groups < 1 || n_groups > FR_MAX_OPT_GROUPS || step < 1) return FR_EINVAL;
    GroupTable T;
    int blocks = 0, apply_blocks = 0;
    for (int k = 0; k < n_groups; ++k) {
        const fr_opt_group& G = groups[k];
        if (!G.x || !G.m || !G.v || G.n < 0) return FR_EINVAL;
        if ((G.kind == FR_GROUP_TEX_RGB || G.kind == FR_GROUP_TEX_MONO) &&
            (G.width < 1 || (long)G.width * G.width * (G.kind == FR_GROUP_TEX_RGB ? 3 : 1) != G.n))
            return FR_EINVAL;
        if (G.kind == FR_GROUP_LIGHT && ((!G.aux && !G.aux2) || G.n % 3 != 0)) return FR_EINVAL;
        if (G.kind == FR_GROUP_STAGE && (!G.aux || G.n % 4 != 0)) return FR_EINVAL;
        T.g[k] = G;
        const int st_k = G.step > 0 ? G.step : step;
        T.bc1[k] = (float)(1.0 - pow((double)beta1, st_k));
        T.bc2[k] = (float)(1.0 - pow((double)beta2, st_k));
        T.block_start[k] = blocks;
        T.apply_start[k] = apply_blocks;
        const int units = G.kind == FR_GROUP_TEX_RGB ? G.n / 3 : G.n;
        blocks += (units + ADAM_THREADS - 1) / ADAM_THREADS;
        apply_blocks += (G.n + 4 * ADAM_THREADS - 1) / (4 * ADAM_THREADS);
    }
    T.block_start[n_groups] = blocks;
    T.apply_start[n_groups] = apply_blocks;
    T.n_groups = n_groups;
    T.beta1 = beta1;
    T.beta2 = beta2;
    T.eps = eps;
    const cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (reg_energy) cudaMemsetAsync(reg_energy, 0, sizeof(double), st);
    if (blocks > 0) {
        if (reg_energy) k_adam_moments<true><<<blocks, ADAM_THREADS, 0, st>>>(T, reg_energy);
        else k_adam_moments<false><<<blocks, ADAM_THREADS, 0, st>>>(T, nullptr);
        k_adam_apply<<<apply_blocks, ADAM_THREADS, 0, st>>>(T);
        fr_count_launches(2);
    }
    return cudaGetLastError() == cudaSuccess ? FR_OK : FR_ECUDA;
}
