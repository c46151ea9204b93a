// k_mlp.cu -- learned curvature on the 5x5x5 fill-level stencil: training
// stencils, the MLP 125 -> 128 -> 128 -> 1 (GELU) with BF16 weights, its FP32
// backward and Adam, and the in-step estimate that keeps the LSQR fit
// (Sec. II.C) as judge and fallback.  Every network evaluation -- the batch
// forward, the training step and the in-step estimate -- runs on the tcgen05
// tensor cores (k_mlp_tc.cu); this file holds the training stencils, the
// gradient reduction with Adam, and the C entry points.
//
// Network (packed parameter block, see include/fsl.h):
//   x = bf16(2 phi - 1) over the canonical stencil (125 values, 3 zero pads)
//   z1 = W1 x + b1, h1 = bf16(gelu(z1)), z2 = W2 h1 + b2, h2 = gelu(z2),
//   y = w3 . h2 + b3 = kappa dx;   gelu(x) = x Phi(x) (erf form)
// Canonical stencil: axes flipped so the Parker-Youngs normal of the middle
// cell has non-negative components, then ordered by decreasing |n_k|.
#include <math.h>

#include <algorithm>

#include "fsl_internal.cuh"
#include "mlp_common.cuh"

namespace fslk {

constexpr int MK = 128;     // padded input width, hidden width
constexpr int MB_BF = 32896;  // bf16 elements of W1 | W2 | w3
constexpr size_t MB_BIAS = (size_t)MB_BF * 2;  // byte offset of the FP32 biases (256-aligned)
// FP32 master / gradient / moment layout
constexpr int M_W1 = 0, M_W2 = 16384, M_W3 = 32768, M_B1 = 32896, M_B2 = 33024, M_B3 = 33152, M_COUNT = 33153;
static_assert(M_W1 == 0 && M_W2 == M_W1 + MK * MK && M_W3 == M_W2 + MK * MK && M_B1 == MB_BF && M_B2 == M_B1 + MK &&
                  M_B3 == M_B2 + MK && M_COUNT == M_B3 + 1,
              "master layout: W1, W2, w3, b1, b2, b3 (the tile partials use the same order)");


// ---- training: gradient reduction and Adam --------------------------------------
// (forward, deltas and the per-tile gradient partials run on the tensor cores
// in k_mlp_train_tile, k_mlp_tc.cu)
// Sum of the per-tile partials of k_mlp_train_tile in tile order into the
// gradient (master layout), and, with master != null, the Adam step on it in
// the same thread (as k_mlp_adam).  Thread 0 also sums the tiles' loss terms.
constexpr int PART_STRIDE = 2 * MK * MK + 4 * MK;  // floats of one tile's partials

__global__ void __launch_bounds__(256) k_mlp_tile_reduce(const float *part, const double *lpart, int ntiles, int n,
                                                         float *grad, float *loss,
                                                         uint8_t *params, float *master, float *m, float *v, float lr,
                                                         float bc1, float bc2) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_enter();
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x < 32 && loss) {  // in the last block, which is half idle
        double l = 0.0;
        for (int t = threadIdx.x; t < ntiles; t += 32) l += lpart[t];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (threadIdx.x == 0) loss[0] = (float)(l / n);
    }
    if (e >= M_COUNT) return;
    // 16 partials in flight: the sum is a chain of adds, the loads need not be
    float acc = 0.f;
    if (e < M_W3) {
        const int mat = e / (MK * MK), k = e % (MK * MK);
        const float *P = part + (size_t)mat * MK * MK + k;
#pragma unroll 16
        for (int t = 0; t < ntiles; ++t) acc += P[(size_t)t * PART_STRIDE];
    } else {
        int vec, c = 0;
        if (e < M_B1) { vec = 2; c = e - M_W3; }
        else if (e < M_B2) { vec = 0; c = e - M_B1; }
        else if (e < M_B3) { vec = 1; c = e - M_B2; }
        else { vec = 3; }
        const float *P = part + (size_t)2 * MK * MK + (size_t)vec * MK + c;
#pragma unroll 16
        for (int t = 0; t < ntiles; ++t) acc += P[(size_t)t * PART_STRIDE];
    }
    if (grad) grad[e] = acc;
    if (master) {
        __nv_bfloat16 *wb = reinterpret_cast<__nv_bfloat16 *>(params);
        float *bias = reinterpret_cast<float *>(params + MB_BIAS);
        const float mm = 0.9f * m[e] + 0.1f * acc, vv = 0.999f * v[e] + 0.001f * acc * acc;
        m[e] = mm;
        v[e] = vv;
        const float w = master[e] - lr * (mm / bc1) / (sqrtf(vv / bc2) + 1e-8f);
        master[e] = w;
        if (e < M_B1) wb[e] = __float2bfloat16_rn(w);
        else bias[e - M_B1] = w;
    }
}

// master parameters -> packed BF16 weights and FP32 biases
__global__ void __launch_bounds__(256) k_mlp_pack(const float *master, uint8_t *params) {
    __nv_bfloat16 *wb = reinterpret_cast<__nv_bfloat16 *>(params);
    float *bias = reinterpret_cast<float *>(params + MB_BIAS);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < M_COUNT; e += gridDim.x * blockDim.x) {
        if (e < M_B1) wb[e] = __float2bfloat16_rn(master[e]);
        else bias[e - M_B1] = master[e];
    }
}

// ---- training stencils ---------------------------------------------------------
__device__ __forceinline__ unsigned long long splitmix64_at(unsigned long long seed, unsigned long long k) {
    unsigned long long z = seed + (k + 1ULL) * 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}
__device__ __forceinline__ double uniform_at(unsigned long long seed, unsigned long long k) {
    return (double)(splitmix64_at(seed, k) >> 11) * (1.0 / 9007199254740992.0);
}

// the multiplier t of the nearest surface point by bisection (see below)
__device__ __noinline__ double nearest_bisect(const double a[3], const double o[3]) {
    double lo = -fmin(a[0] * a[0], fmin(a[1] * a[1], a[2] * a[2])) * (1.0 - 1e-15);
    double hi = fmax(1.0, fmax(fabs(o[0]), fmax(fabs(o[1]), fabs(o[2]))) * fmax(a[0], fmax(a[1], a[2])));
    auto gfun = [&](double t) {
        double s = 0.0;
        for (int k = 0; k < 3; ++k) {
            const double q = a[k] * o[k] / (a[k] * a[k] + t);
            s += q * q;
        }
        return s - 1.0;
    };
    for (int it = 0; it < 64 && gfun(hi) > 0.0; ++it) hi *= 2.0;
    for (int it = 0; it < 100; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (gfun(mid) > 0.0) lo = mid;
        else hi = mid;
    }
    return 0.5 * (lo + hi);
}

// mean curvature at the point of the ellipsoid sum (y/a)^2 = 1 (body frame)
// nearest to o (body frame): x_k = a_k^2 o_k / (a_k^2 + t)
__device__ double nearest_mean_curvature(const double a[3], const double o[3]) {
    // |q(t)| = 1 with q_k = a_k o_k / (a_k^2 + t): Newton's method on 1/|q|, which
    // is nearly linear in t, from the left of the largest root, where no single
    // |q_k| exceeds 1; it converges in four or five steps.  Points it does not
    // settle for (the ellipsoid's centre and focal set) take the bisection.
    double t = -1e300;
    for (int k = 0; k < 3; ++k) t = fmax(t, fabs(a[k] * o[k]) - a[k] * a[k]);
    bool done = false;
    for (int it = 0; it < 12 && !done; ++it) {
        double q2 = 0.0, dq = 0.0;
        for (int k = 0; k < 3; ++k) {
            const double r = 1.0 / (a[k] * a[k] + t), q = a[k] * o[k] * r;
            q2 += q * q;
            dq += q * q * r;
        }
        const double st = q2 / dq * (sqrt(q2) - 1.0);
        done = fabs(st) <= 4e-16 * fmax(fabs(t), a[0] * a[0]);
        t += st;
    }
    if (!done || !(t > -fmin(a[0] * a[0], fmin(a[1] * a[1], a[2] * a[2])) * (1.0 - 1e-15))) t = nearest_bisect(a, o);
    double gr[3], hs[3], gn2 = 0.0, trh = 0.0, ghg = 0.0;
    for (int k = 0; k < 3; ++k) {
        const double x = a[k] * a[k] * o[k] / (a[k] * a[k] + t);
        gr[k] = 2.0 * x / (a[k] * a[k]);
        hs[k] = 2.0 / (a[k] * a[k]);
        gn2 += gr[k] * gr[k];
        trh += hs[k];
        ghg += gr[k] * gr[k] * hs[k];
    }
    const double gn = sqrt(gn2);
    return (gn2 * trh - ghg) / (2.0 * gn2 * gn);
}

// rotation (row-major, FP64) and centre of stencil k's ellipsoid, its surface
// point at `delta` from the middle cell's centre.  Any quaternion is taken as it
// is: the matrix is 1 + 2 w K + 2 K^2 with K the cross product with (x, y, z),
// |(x, y, z)|^2 = s2, a normal matrix of eigenvalues 1 and 1 - 2 s2 +- 2 i w sqrt(s2),
// whose moduli are 1 for a unit quaternion only.  rn: a bound of its norm (1.0001 is
// far above the FP32 rounding).
__device__ __forceinline__ void stencil_frame(long long k, const float *axes, const float *quat, const float *dir,
                                              const float *delta, double R[9], double a[3], double c[3], float &rn) {
    const double w = quat[4 * k], x = quat[4 * k + 1], y = quat[4 * k + 2], z = quat[4 * k + 3];
    const double M[9] = {1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                         2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                         2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)};
    for (int e = 0; e < 9; ++e) R[e] = M[e];
    const float fw = (float)w, s2 = (float)x * (float)x + (float)y * (float)y + (float)z * (float)z, re = 1.0f - 2.0f * s2;
    rn = 1.0001f * sqrtf(fmaxf(1.0f, re * re + 4.0f * fw * fw * s2));
    for (int r = 0; r < 3; ++r) a[r] = axes[3 * k + r];
    const double d[3] = {dir[3 * k], dir[3 * k + 1], dir[3 * k + 2]};
    const double sc = 1.0 / sqrt((d[0] / a[0]) * (d[0] / a[0]) + (d[1] / a[1]) * (d[1] / a[1]) +
                                 (d[2] / a[2]) * (d[2] / a[2]));
    for (int r = 0; r < 3; ++r) c[r] = delta[3 * k + r] - (R[3 * r] * d[0] + R[3 * r + 1] * d[1] + R[3 * r + 2] * d[2]) * sc;
}

// Targets, one thread per stencil: the FP64 rate (2 FMA per clock and SM) bounds
// them, so every lane of a warp has a stencil of its own.
__global__ void __launch_bounds__(128) k_mlp_targets(int n, const float *axes, const float *quat, const float *dir,
                                                     const float *delta, const int *invert, float *target) {
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        double R[9], a[3], c[3], o[3];
        float rn;
        stencil_frame(k, axes, quat, dir, delta, R, a, c, rn);
        for (int r = 0; r < 3; ++r) o[r] = -(R[r] * c[0] + R[3 + r] * c[1] + R[6 + r] * c[2]);  // R^T (0 - C)
        const double H = nearest_mean_curvature(a, o);
        target[k] = (float)(invert[k] ? -H : H);
    }
}

// Stencils, one warp for `per` consecutive ones.  Lane l < per sets up stencil
// l (FP64), then the warp takes them one at a time:
//   cells    the lanes decide the cells the surface |A^-1 R^T (p - C)| = 1 cannot
//            cut, from the value and gradient at the cell's centre; about 45 of
//            125 stay open
//   columns  the same for the sub x sub columns of samples of the open cells
//            (a quarter stays open), queued so that the 32 lanes always sample
//            32 open columns
//   noise    on the partially filled cells, packed onto the lanes (FP64)
// and the canonical BF16 row leaves in one 8-byte store per lane (in 2-byte stores
// where X does not lie on an 8-byte boundary; rows are 256 bytes).  One block of
// 125 sampling threads per stencil, one of which also bisected for the target
// in FP64, took 16 ms for 65536 stencils at sub = 8; this takes 1.55 ms and the
// targets 0.08.
constexpr int ST_WARPS = 4;

struct StWarp {
    float frame[32][17];  // R (9), C (3), semi-axes (3), bound of |A^-1 R^T|, |R|
    float st[128];
    int cnt[128];
    int queue[64];
    uint8_t open[128];
    alignas(16) __nv_bfloat16 row[128];
};

// W warps per stencil: 1, or the ST_WARPS of a block, which share the columns of
// a stencil (each with a queue of its own) and leave the rest to the first warp.
template <int W>
__global__ void __launch_bounds__(32 * ST_WARPS, 5) k_mlp_stencils(int n, int per, const float *axes, const float *quat,
                                                                const float *dir, const float *delta,
                                                                const int *invert, int sub, float noise,
                                                                unsigned long long noise_seed, __nv_bfloat16 *X) {
    __shared__ StWarp smem[ST_WARPS];
    static_assert(W == 1 || W == ST_WARPS, "a warp or a block per stencil");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, part = W == 1 ? 0 : warp;
    StWarp &s = smem[W == 1 ? warp : 0];
    int *queue = smem[warp].queue;
    const unsigned full = 0xffffffffu;
    auto sync = [] {
        if (W == 1) __syncwarp();
        else __syncthreads();
    };
    const long long groups = ((long long)n + per - 1) / per, nw = (long long)gridDim.x * (ST_WARPS / W);
    const int S2 = sub * sub, tot = S2 * sub;
    const int magic = (65536 + sub - 1) / sub;  // c / sub = (c magic) >> 16 for c < 1024, sub <= 32
    const bool wide = (reinterpret_cast<uintptr_t>(X) & 7) == 0;
    const float h = 1.0f / sub, half = 0.5f * (float)(sub - 1) * h + 1e-6f;  // half a column of samples
    for (long long g = W == 1 ? (long long)blockIdx.x * ST_WARPS + warp : blockIdx.x; g < groups; g += nw) {
        const int m = (int)min((long long)per, n - g * per);
        if (lane < m) {
            double R[9], a[3], c[3];
            float rn;
            stencil_frame(g * per + lane, axes, quat, dir, delta, R, a, c, rn);
            float *f = s.frame[lane];
            for (int e = 0; e < 9; ++e) f[e] = (float)R[e];
            for (int r = 0; r < 3; ++r) {
                f[9 + r] = (float)c[r];
                f[12 + r] = (float)a[r];
            }
            f[16] = rn;
            f[15] = f[16] / fminf(fabsf(f[12]), fminf(fabsf(f[13]), fabsf(f[14])));
        }
        sync();
        for (int q = 0; q < m; ++q) {
            const long long k = g * per + q;
            const float *f = s.frame[q];
            float Rm[9], C[3];
#pragma unroll
            for (int e = 0; e < 9; ++e) Rm[e] = f[e];
#pragma unroll
            for (int r = 0; r < 3; ++r) C[r] = f[9 + r];
            const float inv_a0 = 1.0f / f[12], inv_a1 = 1.0f / f[13], inv_a2 = 1.0f / f[14], lip = f[15];
            // r = |A^-1 R^T (p - C)| is a norm of p - C: over a displacement v its change is
            // at most |grad r . v| + (lip |v|)^2 / (2 (r - lip |v|)), and at most lip |v|.
            // reach = |v|, gr = bound of |grad r . v| / |v|.  1: all within the reach
            // inside, 0: none, -1: open.  tol is far above the rounding of the sample test.
            const float tol = 4e-6f * ((fabsf(C[0]) + fabsf(C[1]) + fabsf(C[2]) + 8.0f) * lip + 1.0f);
            auto decide = [&](float px, float py, float pz, float reach, bool along_z) {
                const float y0 = (Rm[0] * px + Rm[3] * py + Rm[6] * pz) * inv_a0;
                const float y1 = (Rm[1] * px + Rm[4] * py + Rm[7] * pz) * inv_a1;
                const float y2 = (Rm[2] * px + Rm[5] * py + Rm[8] * pz) * inv_a2;
                const float r2 = fmaxf(y0 * y0 + y1 * y1 + y2 * y2, 1e-30f), ir = rsqrtf(r2), r = r2 * ir;
                const float v0 = y0 * inv_a0, v1 = y1 * inv_a1, v2 = y2 * inv_a2;
                const float gr = along_z ? fabsf(Rm[6] * v0 + Rm[7] * v1 + Rm[8] * v2) * ir
                                         : f[16] * sqrtf(v0 * v0 + v1 * v1 + v2 * v2) * ir;
                const float lr = lip * reach, rest = r - lr;
                float b = lr;
                if (rest > 0.1f) b = fminf(b, 1.0001f * gr * reach + __fdividef(0.5001f * lr * lr, rest));
                b += tol * (1.0f + r);
                return 1.0f - r > b ? 1 : (r - 1.0f > b ? 0 : -1);
            };
            int nopen = 0;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int e = lane + 32 * t;
                int v = 0;
                if (e < 125)
                    v = decide((float)(e / 25 - 2) - C[0], (float)((e / 5) % 5 - 2) - C[1], (float)(e % 5 - 2) - C[2], 0.8661f,
                               false);
                s.cnt[e] = v == 1 ? tot : 0;
                const unsigned mk = __ballot_sync(full, v < 0);
                if (v < 0) s.open[nopen + __popc(mk & ((1u << lane) - 1u))] = (uint8_t)e;
                nopen += __popc(mk);
            }
            sync();
            // one column of samples: cell e, column (sx, sy)
            auto column = [&](int item) {
                const int slot = item >> 10, col = item & 1023;
                const int e = s.open[slot], sx = (col * magic) >> 16, sy = col - sx * sub;
                const int i = e / 25 - 2, j = (e / 5) % 5 - 2, l = e % 5 - 2;
                const float px = i + (sx + 0.5f) * h - 0.5f - C[0], py = j + (sy + 0.5f) * h - 0.5f - C[1];
                const float b0 = fmaf(Rm[3], py, __fmul_rn(Rm[0], px)), b1 = fmaf(Rm[4], py, __fmul_rn(Rm[1], px)),
                            b2 = fmaf(Rm[5], py, __fmul_rn(Rm[2], px));
                int cnt = 0;
#pragma unroll 4
                for (int sz = 0; sz < sub; ++sz) {
                    const float pz = l + (sz + 0.5f) * h - 0.5f - C[2];
                    const float y0 = fmaf(Rm[6], pz, b0) * inv_a0, y1 = fmaf(Rm[7], pz, b1) * inv_a1,
                                y2 = fmaf(Rm[8], pz, b2) * inv_a2;
                    cnt += (y0 * y0 + y1 * y1 + y2 * y2 <= 1.0f) ? 1 : 0;
                }
                if (cnt) atomicAdd(&s.cnt[e], cnt);
            };
            int queued = 0, slot = 0, col = lane + 32 * part;
            for (int base = 32 * part; base < nopen * S2; base += 32 * W) {  // warp-uniform
                while (col >= S2) {
                    col -= S2;
                    ++slot;
                }
                int v = 0;
                if (slot < nopen) {
                    const int e = s.open[slot], sx = (col * magic) >> 16, sy = col - sx * sub;
                    v = decide((float)(e / 25 - 2) + (sx + 0.5f) * h - 0.5f - C[0],
                               (float)((e / 5) % 5 - 2) + (sy + 0.5f) * h - 0.5f - C[1], (float)(e % 5 - 2) - C[2], half, true);
                    if (v == 1) atomicAdd(&s.cnt[e], sub);
                }
                const unsigned mk = __ballot_sync(full, v < 0);
                if (v < 0) queue[queued + __popc(mk & ((1u << lane) - 1u))] = (slot << 10) | col;
                queued += __popc(mk);
                __syncwarp();
                if (queued >= 32) {
                    queued -= 32;
                    column(queue[queued + lane]);
                    __syncwarp();
                }
                col += 32 * W;
            }
            if (lane < queued) column(queue[lane]);
            sync();
            if (part) {
                sync();  // the first warp is done with the stencil
                continue;
            }
            // fill levels; the partially filled cells (all among the open ones) take the noise
            const bool inv = invert[k] != 0;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int e = lane + 32 * t;
                s.st[e] = (float)(inv ? tot - s.cnt[e] : s.cnt[e]) / (float)tot;
            }
            __syncwarp();
            if (noise > 0.f) {
                int np = 0;
                for (int b = 0; b < nopen; b += 32) {
                    const int e = b + lane < nopen ? s.open[b + lane] : 0;
                    const bool cut = b + lane < nopen && s.st[e] > 0.f && s.st[e] < 1.f;
                    const unsigned mk = __ballot_sync(full, cut);
                    __syncwarp();
                    if (cut) s.open[np + __popc(mk & ((1u << lane) - 1u))] = (uint8_t)e;
                    np += __popc(mk);
                    __syncwarp();
                }
                for (int b = lane; b < np; b += 32) {
                    const int e = s.open[b];
                    const unsigned long long idx = (unsigned long long)k * 125ULL + e;
                    const double u1 = uniform_at(noise_seed, 2 * idx), u2 = uniform_at(noise_seed, 2 * idx + 1);
                    // 1 - u1 is exact (u1 is a multiple of 2^-53)
                    const float nrm = (float)(sqrt(-2.0 * log(1.0 - u1)) * cospi(2.0 * u2));
                    s.st[e] = fminf(fmaxf(s.st[e] + noise * nrm, 0.f), 1.f);
                }
                __syncwarp();
            }
            const Canon cs = canon_of(s.st);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int e = lane + 32 * t;
                s.row[e < 125 ? canon_index(cs, e) : e] = __float2bfloat16_rn(e < 125 ? 2.0f * s.st[e] - 1.0f : 0.f);
            }
            __syncwarp();
            if (wide) {
                reinterpret_cast<uint2 *>(X + k * MK)[lane] = reinterpret_cast<const uint2 *>(s.row)[lane];
            } else {
#pragma unroll
                for (int t = 0; t < 4; ++t) X[k * MK + lane + 32 * t] = s.row[lane + 32 * t];
            }
            sync();
        }
    }
}

// ---- in-step learned curvature (the network on the tensor cores, k_mlp_tc.cu) ----
void launch_mlp_curv(const Dev &d, float *kappa_out, cudaStream_t s) {
    launch_mlp_curv_tc(d, kappa_out, s);
}

}  // namespace fslk

using namespace fslk;

extern "C" {

size_t fsl_mlp_param_bytes(void) { return MB_BIAS + (size_t)(2 * MK + 1) * sizeof(float); }
int fsl_mlp_master_count(void) { return M_COUNT; }

// training workspace (bytes, each part 256-aligned): the gradient (master
// layout), the per-tile partials of the tile kernel and the tiles' loss sums
static size_t up256(size_t v) { return (v + 255) / 256 * 256; }
struct TrainWs {
    size_t grad, part, lpart, total;
};
static TrainWs train_ws(int n) {
    TrainWs w;
    size_t o = 0;
    w.grad = o; o = up256(o + (size_t)M_COUNT * sizeof(float));
    w.part = o; o = up256(o + mlp_tile_partial_floats(n) * sizeof(float));
    w.lpart = o; o = up256(o + (size_t)((n + MK - 1) / MK) * sizeof(double));
    w.total = o;
    return w;
}

size_t fsl_mlp_train_workspace(int n) {
    if (n <= 0) return 0;
    return train_ws(n).total + 1024;
}

int fsl_mlp_stencils(int n, const float *axes, const float *quat, const float *dir, const float *delta,
                     const int32_t *invert, int sub, float noise, uint64_t noise_seed, void *X, float *target,
                     void *stream) {
    if (n < 0 || !axes || !quat || !dir || !delta || !invert || !X || !target || sub < 1 || sub > 32 || noise < 0.f)
        return FSL_EINVAL;
    if (n == 0) return FSL_OK;
    if (reinterpret_cast<uintptr_t>(X) % sizeof(__nv_bfloat16)) return FSL_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    // A few stencils per warp fill the lanes of the FP64 set-up; fewer where that would
    // leave SMs idle.  A block per stencil where the stencils fit one round of resident
    // blocks (5 per SM) and each has columns enough to share: n = 100 at sub = 16 / 32
    // takes 95 / 306 us with a block each and 255 / 1096 with a warp each (204 / 636 with
    // one block of 125 sampling threads each), n = 760 at sub = 8 73 against 97; at
    // sub = 4 760 stencils take 58 either way, at sub = 1 51 against 41, and 2400 at
    // sub = 8 146 against 120.
    const int per = std::min(8, std::max(1, n / (152 * 16 * ST_WARPS)));
    const bool block = n <= 152 * 5 && sub >= 8;
    const long long groups = ((long long)n + per - 1) / per;
    const int grid = block ? n : (int)std::min<long long>((groups + ST_WARPS - 1) / ST_WARPS, 152 * 64);
    k_mlp_targets<<<std::min((n + 127) / 128, 152 * 16), 128, 0, s>>>(n, axes, quat, dir, delta, invert, target);
    (block ? k_mlp_stencils<ST_WARPS> : k_mlp_stencils<1>)<<<grid, 32 * ST_WARPS, 0, s>>>(
        n, per, axes, quat, dir, delta, invert, sub, noise, noise_seed, static_cast<__nv_bfloat16 *>(X));
    return cudaGetLastError() == cudaSuccess ? FSL_OK : FSL_ECUDA;
}

int fsl_mlp_forward(const void *params, const void *X, int n, float *y, float *z1, float *z2, void *stream) {
    if (!params || !X || !y || n < 0 || ((z1 == nullptr) != (z2 == nullptr))) return FSL_EINVAL;
    if (n == 0) return FSL_OK;
    return launch_mlp_forward_tc(static_cast<const uint8_t *>(params), static_cast<const __nv_bfloat16 *>(X), n, y, z1,
                                 z2, (cudaStream_t)stream);
}

int fsl_mlp_status(int reset) { return mlp_tc_status(reset != 0); }

// One training step's gradient (and with master non-null the Adam step): the
// tile kernel over the batch rows perm[row0 .. row0 + n) of X (rows row0 ..
// when perm is null), then the fixed-order reduction of its partials.
static int mlp_step(const void *params, const void *X, const float *target, const int64_t *perm, long long row0, int n,
                    long long n_all, bool follows, float *loss_dev, void *workspace, float *grad_out, void *params_rw,
                    float *master, float *m, float *v, float lr, int step, cudaStream_t s) {
    char *ws = static_cast<char *>(workspace);
    const TrainWs L = train_ws(n);
    float *part = reinterpret_cast<float *>(ws + L.part);
    double *lpart = reinterpret_cast<double *>(ws + L.lpart);
    const int rc = launch_mlp_train_tile(static_cast<const uint8_t *>(params), static_cast<const __nv_bfloat16 *>(X),
                                         target, perm, row0, n, n_all, follows, part, lpart, s);
    if (rc != FSL_OK) return rc;
    const float bc1 = master ? (float)(1.0 - pow(0.9, step)) : 1.f, bc2 = master ? (float)(1.0 - pow(0.999, step)) : 1.f;
    launch_pdl(k_mlp_tile_reduce, (M_COUNT + 255) / 256, 256, s, (const float *)part, (const double *)lpart,
               (n + MK - 1) / MK, n, grad_out, loss_dev, static_cast<uint8_t *>(params_rw), master, m, v, lr, bc1, bc2);
    return cudaGetLastError() == cudaSuccess ? FSL_OK : FSL_ECUDA;
}

int fsl_mlp_gradients(const void *params, const void *X, const float *target, int n, float *grad, float *loss_dev,
                      void *workspace, void *stream) {
    if (!params || !X || !target || !grad || !workspace || n <= 0) return FSL_EINVAL;
    if (reinterpret_cast<uintptr_t>(X) % 16 || reinterpret_cast<uintptr_t>(workspace) % 256) return FSL_EINVAL;
    return mlp_step(params, X, target, nullptr, 0, n, n, false, loss_dev, workspace, grad, nullptr, nullptr, nullptr, nullptr,
                    0.f, 1, (cudaStream_t)stream);
}

int fsl_mlp_train_step(void *params, float *master, float *m, float *v, const void *X, const float *target, int n,
                       float lr, int step, float *loss_dev, void *workspace, void *stream) {
    if (!params || !master || !m || !v || !X || !target || !workspace || n <= 0 || step < 1 || !(lr > 0.f))
        return FSL_EINVAL;
    if (reinterpret_cast<uintptr_t>(X) % 16 || reinterpret_cast<uintptr_t>(workspace) % 256) return FSL_EINVAL;
    return mlp_step(params, X, target, nullptr, 0, n, n, false, loss_dev, workspace, nullptr, params, master, m, v, lr, step,
                    (cudaStream_t)stream);
}

// the epoch loop reads its batches through the permutation inside the tile
// kernel: the epoch workspace is the training workspace of one batch
size_t fsl_mlp_epoch_workspace(int batch) {
    if (batch <= 0) return 0;
    return fsl_mlp_train_workspace(batch);
}

int fsl_mlp_train_epoch(void *params, float *master, float *m, float *v, const void *X, const float *target,
                        const int64_t *perm, int n, int batch, float lr, int step0, float *losses_dev,
                        void *workspace, void *stream) {
    if (!params || !master || !m || !v || !X || !target || !perm || !workspace || batch < 1 || n < batch ||
        step0 < 0 || !(lr > 0.f))
        return FSL_EINVAL;
    if (reinterpret_cast<uintptr_t>(X) % 16 || reinterpret_cast<uintptr_t>(workspace) % 256) return FSL_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int nb = n / batch;
    for (int b = 0; b < nb; ++b) {
        const int rc = mlp_step(params, X, target, perm, (long long)b * batch, batch, n, b > 0,
                                losses_dev ? losses_dev + b : nullptr, workspace, nullptr, params, master, m, v, lr,
                                step0 + b + 1, s);
        if (rc != FSL_OK) return rc;
    }
    return FSL_OK;
}

int fsl_mlp_pack(const float *master, void *params, void *stream) {
    if (!master || !params) return FSL_EINVAL;
    k_mlp_pack<<<(M_COUNT + 255) / 256, 256, 0, (cudaStream_t)stream>>>(master, static_cast<uint8_t *>(params));
    return cudaGetLastError() == cudaSuccess ? FSL_OK : FSL_ECUDA;
}

}  // extern "C"
