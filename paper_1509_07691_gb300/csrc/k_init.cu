// k_init.cu -- initial fill levels by sub-sampling (Sec. III.A), initial cell
// types (Sec. II), refresh of derived data, statistics and the total mass.
#include <math.h>

#include "fsl_internal.cuh"

namespace fslk {

int resident_grid(const void *kernel, int block, size_t smem) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, block, smem);
    return (sms > 0 ? sms : 1) * (per > 0 ? per : 1);
}

int list_blocks(const void *kernel, int block, int per_sm) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int want = (sms > 0 ? sms : 1) * per_sm, cap = resident_grid(kernel, block);
    return want < cap ? want : cap;
}

// ---- fill levels -------------------------------------------------------------
// Inside tests in FP64 with explicitly rounded operations (no contraction),
// evaluated in the same order as the sampling formula states, so that every
// sample point is classified as the definition classifies it.
__device__ __forceinline__ double dsq3(double a, double b, double c) {
    return __dadd_rn(__dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b)), __dmul_rn(c, c));
}

__device__ bool inside(const fsl_geometry &g, double px, double py, double pz) {
    const double dx = __dsub_rn(px, g.c[0]), dy = __dsub_rn(py, g.c[1]), dz = __dsub_rn(pz, g.c[2]);
    const double r2 = dsq3(dx, dy, dz);
    bool in = false;
    switch (g.kind) {
    case 0: in = r2 <= __dmul_rn(g.R, g.R); break;
    case 1: {
        const double r = __dsqrt_rn(r2);
        if (r == 0.0) { in = true; break; }
        const double mu = __ddiv_rn(dz, r);
        const double p2 = __dsub_rn(__dmul_rn(__dmul_rn(1.5, mu), mu), 0.5);
        in = r <= __dmul_rn(g.R, __dadd_rn(1.0, __dmul_rn(g.eps2, p2)));
        break;
    }
    case 2: in = (r2 <= __dmul_rn(g.R, g.R)) && (pz >= g.zw); break;
    case 3: {
        const double ex = __dsub_rn(px, g.c2[0]), ey = __dsub_rn(py, g.c2[1]), ez = __dsub_rn(pz, g.c2[2]);
        in = (r2 <= __dmul_rn(g.R, g.R)) || (dsq3(ex, ey, ez) <= __dmul_rn(g.R2, g.R2));
        break;
    }
    case 4: {
        const double tp = 6.283185307179586;
        const double h = __dadd_rn(g.h0, __dmul_rn(__dmul_rn(g.amp, sin(__ddiv_rn(__dmul_rn(tp, px), g.wavelength))),
                                                   sin(__ddiv_rn(__dmul_rn(tp, py), g.wavelength))));
        in = pz < h;
        break;
    }
    case 5:
        in = __dadd_rn(__dadd_rn(__dmul_rn(g.n[0], px), __dmul_rn(g.n[1], py)), __dmul_rn(g.n[2], pz)) <= g.d;
        break;
    }
    return g.invert ? !in : in;
}

// The same shape as a level function G in FP32, G > 0 inside: an estimate
// that decides most samples without FP64.  Coordinates enter as an integer
// cell offset (exact) plus a fraction, so that their rounding is relative to
// the distance from the shape's centre.
struct Level {
    int kind, sub;
    float sign;              // -1: liquid outside
    int ci[3], ci2[3], zwi;  // centres and wall plane: nearest integer ...
    float cf[3], cf2[3], zwf;  // ... and the rest
    float R, R2, eps2, n[3], nl, d, h0, amp, iw;
};

constexpr float U24 = 5.9604645e-8f;  // half an ulp of 1
constexpr float CELL_HD = 0.8661f;    // half diagonal of a cell

// G at cell (x, y, z) + (ox, oy, oz), |o| <= 1/2.  T bounds the error of G
// against the FP64 test of inside() and L its Lipschitz constant within 0.9
// cells, so that every point within h <= 0.9 of here is inside where
// G > L h + T and outside where G < -(L h + T).  The bounds count each
// rounding: a coordinate difference d is off by at most U24 (2 |d| + 2), a
// radius by U24 (6 r + 10) (approximate rsqrt included), both with room.
// NaN or infinite parameters satisfy neither comparison.
__device__ __forceinline__ float level(const Level &g, int x, int y, int z, float ox, float oy, float oz, float &T,
                                       float &L) {
    float G;
    L = 1.0f;
    if (g.kind <= 3) {
        const float dx = (float)(x - g.ci[0]) + (ox - g.cf[0]), dy = (float)(y - g.ci[1]) + (oy - g.cf[1]),
                    dz = (float)(z - g.ci[2]) + (oz - g.cf[2]);
        const float r2 = fmaxf(dx * dx + dy * dy + dz * dz, 1e-30f), ir = rsqrtf(r2), r = r2 * ir;
        G = g.R - r;
        T = U24 * (16.0f * (r + fabsf(g.R)) + 32.0f);
        if (g.kind == 1) {
            // r <= R (1 + eps P2(mu)): mu^2 is off by at most 32 U24 for r >= 1;
            // |grad of R eps P2| <= 3/2 |R eps| / r
            const float mu = dz * ir, re = g.R * g.eps2;
            G += re * (1.5f * mu * mu - 0.5f);
            T += U24 * 96.0f * fabsf(re);
            L = 1.0f + 1.5f * fabsf(re) / (r - 0.95f);
            if (!(r > 2.0f)) T = INFINITY;
        } else if (g.kind == 2) {
            const float h = (float)(z - g.zwi) + (oz - g.zwf);
            G = fminf(G, h);
            T += U24 * 8.0f * (fabsf(h) + 1.0f);
        } else if (g.kind == 3) {
            const float ex = (float)(x - g.ci2[0]) + (ox - g.cf2[0]), ey = (float)(y - g.ci2[1]) + (oy - g.cf2[1]),
                        ez = (float)(z - g.ci2[2]) + (oz - g.cf2[2]);
            const float q2 = fmaxf(ex * ex + ey * ey + ez * ez, 1e-30f), q = q2 * rsqrtf(q2);
            G = fmaxf(G, g.R2 - q);
            T += U24 * (16.0f * (q + fabsf(g.R2)) + 32.0f);
        }
    } else if (g.kind == 4) {
        // |grad of amp sin sin| <= |amp| k; the phase x / wavelength is off by at most 4 U24 of itself
        const float px = (float)x + ox, py = (float)y + oy, pz = (float)z + oz;
        const float fx = 2.0f * px * g.iw, fy = 2.0f * py * g.iw, am = fabsf(g.amp), k = 6.2832f * fabsf(g.iw);
        G = g.h0 - pz;
        T = U24 * (8.0f * (fabsf(g.h0) + fabsf(pz)) + 32.0f * am + 32.0f * am * (fabsf(fx) + fabsf(fy)) +
                   64.0f * am * fabsf(g.iw) + 4.0f);
        L = 1.0f + am * k;
        if (fabsf(G) <= am + L + T) G += g.amp * sinpif(fx) * sinpif(fy);
        else G += G > 0.f ? -am : am;  // far from the surface: the closest it can be
    } else {
        const float a = g.n[0] * ((float)x + ox), b = g.n[1] * ((float)y + oy), c = g.n[2] * ((float)z + oz);
        G = g.d - (a + b + c);
        T = U24 * 16.0f * (fabsf(g.d) + fabsf(a) + fabsf(b) + fabsf(c) + g.nl);
        L = g.nl;
    }
    return G * g.sign;
}

// Whole cells in FP64 where the level function does not stand for the samples:
// negative radii (inside() squares the radius of kinds 0, 2 and 3) and non-finite
// parameters (a pool of wavelength 0 has no samples inside, and whole cells below
// its crests).  A cell whose centre is more than one cell inside is inside, one
// more than a cell outside is outside, and the rest is sampled: 1, -1, 0.
__device__ int whole_cell(const fsl_geometry &g, double x, double y, double z) {
    const double dx = x - g.c[0], dy = y - g.c[1], dz = z - g.c[2];
    const double ex = x - g.c2[0], ey = y - g.c2[1], ez = z - g.c2[2];
    const double r = sqrt(dx * dx + dy * dy + dz * dz), q = sqrt(ex * ex + ey * ey + ez * ez), e = fabs(g.eps2);
    bool in = r + 1.0 < g.R, out = r - 1.0 > g.R;
    if (g.kind == 1) {
        in = r + 1.0 < g.R * (1.0 - 0.5 * e);
        out = r - 1.0 > g.R * (1.0 + e);
    } else if (g.kind == 2) {
        in = in && z - 1.0 > g.zw;
        out = out || z + 1.0 < g.zw;
    } else if (g.kind == 3) {
        in = in || q + 1.0 < g.R2;
        out = out && q - 1.0 > g.R2;
    } else if (g.kind == 4) {
        in = z + 1.0 < g.h0 - fabs(g.amp);
        out = z - 1.0 > g.h0 + fabs(g.amp);
    }
    const int w = in ? 1 : (out ? -1 : 0);
    return g.invert ? -w : w;
}

// Fill levels: the fraction of the sub^3 sample points of a cell that
// inside() holds for.  Sampling every cell near the surface in FP64 is bound
// by the FP64 rate (2 FMA per clock and SM): one thread per cell took 180 ms
// for the mode-2 droplet of R = 40 in 256^3 at sub = 16; this takes 0.50 ms.  Each thread
// decides its cell from the level function where it can; the block's undecided
// cells (about 1.8 surface layers) are taken by its warps one at a time, first
// in blocks of 4^3 samples (a lane each), then the undecided blocks sample by
// sample, and only samples within T of the surface take the FP64 test.  The
// counts are those of the FP64 test everywhere.
constexpr int FILL_BLOCK = 128;

__device__ __forceinline__ float sample_off(int s, float inv) { return ((float)s + 0.5f) * inv - 0.5f; }

// FP64 test of sample (sx, sy, sz) of a cell, in the arithmetic that defines the
// sample points; out of line, so that none of it is computed ahead of the
// decision (inlined, its divisions ran for every sample and made the kernel
// FP64-bound: 2.3 ms instead of 0.50)
__device__ __noinline__ bool sample_inside(const fsl_geometry &g, int S, int x, int y, int z, int sx, int sy, int sz) {
    const double pz = __dsub_rn(__dadd_rn((double)z, __ddiv_rn(__dadd_rn((double)sz, 0.5), (double)S)), 0.5);
    const double py = __dsub_rn(__dadd_rn((double)y, __ddiv_rn(__dadd_rn((double)sy, 0.5), (double)S)), 0.5);
    const double px = __dsub_rn(__dadd_rn((double)x, __ddiv_rn(__dadd_rn((double)sx, 0.5), (double)S)), 0.5);
    return inside(g, px, py, pz);
}

// 1 or -1: cell (x, y, z) is inside or outside as a whole; 0: open.  WHOLE: as
// whole_cell says, not the level function.
template <bool WHOLE>
__device__ __forceinline__ int decide_cell(const fsl_geometry &g, const Level &lv, int x, int y, int z) {
    if (WHOLE) return whole_cell(g, x, y, z);
    float T, L;
    const float G = level(lv, x, y, z, 0.f, 0.f, 0.f, T, L), B = L * CELL_HD + T;
    return G > B ? 1 : (G < -B ? -1 : 0);
}

template <bool WHOLE>
__global__ void __launch_bounds__(FILL_BLOCK) k_fill(fsl_geometry g, Level lv, int nx, int ny, int nz, float *phi) {
    __shared__ int todo[FILL_BLOCK];
    __shared__ int ntodo;
    const int x = blockIdx.x * FILL_BLOCK + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    const long long row = (long long)nx * ((long long)y + (long long)ny * z);
    if (threadIdx.x == 0) ntodo = 0;
    __syncthreads();
    float T, L;
    if (x < nx) {
        const int w = decide_cell<WHOLE>(g, lv, x, y, z);
        if (w) phi[row + x] = w > 0 ? 1.0f : 0.0f;
        else todo[atomicAdd(&ntodo, 1)] = x;
    }
    __syncthreads();
    const int S = lv.sub, nb = (S + 3) >> 2, lane = threadIdx.x & 31;
    const float inv = 1.0f / (float)S;
    for (int c = threadIdx.x >> 5; c < ntodo; c += FILL_BLOCK / 32) {  // warp-uniform
        const int xc = todo[c];
        int cnt = 0;
        for (int b0 = 0; b0 < nb * nb * nb; b0 += 32) {
            const int b = b0 + lane;
            bool open = false;
            if (b < nb * nb * nb) {
                const int sx = (b % nb) * 4, sy = (b / nb % nb) * 4, sz = (b / (nb * nb)) * 4;
                const int ex = min(S - sx, 4) - 1, ey = min(S - sy, 4) - 1, ez = min(S - sz, 4) - 1;
                const float hx = 0.5f * ex * inv, hy = 0.5f * ey * inv, hz = 0.5f * ez * inv;
                const float G = level(lv, xc, y, z, sample_off(sx, inv) + hx, sample_off(sy, inv) + hy,
                                      sample_off(sz, inv) + hz, T, L);
                const float B = L * (sqrtf(hx * hx + hy * hy + hz * hz) * 1.0001f + 1e-6f) + T;
                if (G > B) cnt += (ex + 1) * (ey + 1) * (ez + 1);
                else open = !(G < -B);
            }
            for (unsigned m = __ballot_sync(0xffffffffu, open); m; m &= m - 1u) {
                const int bb = b0 + __ffs(m) - 1;
                const int sx0 = (bb % nb) * 4, sy0 = (bb / nb % nb) * 4, sz0 = (bb / (nb * nb)) * 4;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int sx = sx0 + (lane & 3), sy = sy0 + ((lane >> 2) & 3), sz = sz0 + (lane >> 4) + 2 * h;
                    if (sx < S && sy < S && sz < S) {
                        const float G = level(lv, xc, y, z, sample_off(sx, inv), sample_off(sy, inv),
                                              sample_off(sz, inv), T, L);
                        const bool in = G > T;
                        cnt += in;
                        if (!in && !(G < -T)) cnt += sample_inside(g, S, xc, y, z, sx, sy, sz) ? 1 : 0;
                    }
                }
            }
        }
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0) phi[row + xc] = (float)((double)cnt / ((double)S * S * S));
    }
}

// The same by a thread per cell: for up to 8 samples, where a warp for each open
// cell leaves most lanes idle, and where the level function bounds nothing and
// every sample of an open cell takes the FP64 test.  (s + 1/2) / sub comes from a
// table, for the divisions are most of that test.  A pool of short waves in
// 256 x 256 x 24 (most cells open) takes 63 / 73 us at sub = 1 / 2, 1440 / 1305
// with a warp per open cell, 294 / 1120 with every open cell's samples in FP64; the
// pool of 256^3 76, 201 and 815 us at sub = 1.  From sub = 3 on k_fill: 1330 us
// against 3178 with FP64 samples, 186 against 2034 on the 256^3 pool.
struct SampleTable {
    double o[64];
};

// out of line for the reason given at sample_inside
__device__ __noinline__ bool table_inside(const fsl_geometry &g, int x, int y, int z, double ox, double oy, double oz) {
    return inside(g, __dsub_rn(__dadd_rn((double)x, ox), 0.5), __dsub_rn(__dadd_rn((double)y, oy), 0.5),
                  __dsub_rn(__dadd_rn((double)z, oz), 0.5));
}

template <bool WHOLE>
__global__ void __launch_bounds__(FILL_BLOCK) k_fill_direct(fsl_geometry g, Level lv, const __grid_constant__ SampleTable tab,
                                                            int nx, int ny, int nz, float *phi) {
    const int x = blockIdx.x * FILL_BLOCK + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    if (x >= nx) return;
    const long long row = (long long)nx * ((long long)y + (long long)ny * z);
    const int w = decide_cell<WHOLE>(g, lv, x, y, z), S = lv.sub;
    if (w) {
        phi[row + x] = w > 0 ? 1.0f : 0.0f;
        return;
    }
    const float inv = 1.0f / (float)S;
    int cnt = 0;
    for (int sz = 0; sz < S; ++sz)
        for (int sy = 0; sy < S; ++sy)
            for (int sx = 0; sx < S; ++sx) {
                float T, L;
                const float G = level(lv, x, y, z, sample_off(sx, inv), sample_off(sy, inv), sample_off(sz, inv), T, L);
                bool in = G > T;
                if (!in && !(G < -T)) in = table_inside(g, x, y, z, tab.o[sx], tab.o[sy], tab.o[sz]);
                cnt += in ? 1 : 0;
            }
    phi[row + x] = (float)((double)cnt / ((double)S * S * S));
}

// integer and fraction of a coordinate; false where it has no int32 part
static bool split(double c, int &i, float &f) {
    if (!(fabs(c) < 1e9)) return false;
    const double r = nearbyint(c);
    i = (int)r;
    f = (float)(c - r);
    return true;
}

void launch_fill_geometry(const fsl_params &p, const fsl_geometry &g, float *phi, cudaStream_t s) {
    dim3 grid((p.nx + FILL_BLOCK - 1) / FILL_BLOCK, p.ny, p.nz);
    Level l = {};
    l.kind = g.kind;
    l.sub = g.sub;
    l.sign = g.invert ? -1.0f : 1.0f;
    bool ok = split(g.zw, l.zwi, l.zwf) || g.kind != 2;
    for (int k = 0; k < 3; ++k) {
        ok = (split(g.c[k], l.ci[k], l.cf[k]) || g.kind > 3) && ok;
        ok = (split(g.c2[k], l.ci2[k], l.cf2[k]) || g.kind != 3) && ok;
    }
    const bool negative = (g.kind <= 3 && g.R < 0.0) || (g.kind == 3 && g.R2 < 0.0);
    l.R = ok ? (float)(g.kind == 1 ? g.R : fabs(g.R)) : NAN;  // NaN: every sample takes the FP64 test
    l.R2 = (float)fabs(g.R2);
    l.eps2 = (float)g.eps2;
    // A half-space by its normal over the largest component: in FP32 a tiny normal is
    // subnormal or zero, and T counts roundings relative to the terms.  Where the FP64
    // products themselves can underflow or overflow, or there is no direction: NaN, and
    // every sample takes the FP64 test.
    const double big = fmax(fabs(g.n[0]), fmax(fabs(g.n[1]), fabs(g.n[2])));
    const double scale = big > 1e-280 && big < 1e280 ? big : NAN;
    for (int k = 0; k < 3; ++k) l.n[k] = (float)(g.n[k] / scale);
    l.d = (float)(g.d / scale);
    l.nl = 1.0001f * sqrtf(l.n[0] * l.n[0] + l.n[1] * l.n[1] + l.n[2] * l.n[2]);
    l.h0 = (float)g.h0;
    l.amp = (float)g.amp;
    l.iw = (float)(1.0 / g.wavelength);
    // no bound at any cell: non-finite parameters, half-spaces without a direction
    const bool blind = g.kind <= 3 ? !isfinite(l.R) || (g.kind == 1 && !isfinite(l.eps2)) || (g.kind == 3 && !isfinite(l.R2))
                       : g.kind == 4 ? !isfinite(l.h0) || !isfinite(l.amp) || !isfinite(l.iw)
                                     : !isfinite(l.nl) || !isfinite(l.d);
    const bool whole = negative || (blind && g.kind != 5);
    if (g.sub <= 2 || blind) {
        SampleTable tab = {};
        for (int k = 0; k < g.sub; ++k) tab.o[k] = ((double)k + 0.5) / (double)g.sub;
        (whole ? k_fill_direct<true> : k_fill_direct<false>)<<<grid, FILL_BLOCK, 0, s>>>(g, l, tab, p.nx, p.ny, p.nz, phi);
    } else {
        (whole ? k_fill<true> : k_fill<false>)<<<grid, FILL_BLOCK, 0, s>>>(g, l, p.nx, p.ny, p.nz, phi);
    }
}

// ---- initial types (Sec. II) -----------------------------------------------
__global__ void __launch_bounds__(256) k_init_types(Dev d, const uint8_t *obstacle, uint8_t *tmp) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= d.N) return;
    const float p = d.phi[i];
    uint8_t t;
    if (obstacle && obstacle[i]) t = T_OBS;
    else if (p <= 0.f) t = T_GAS;
    else if (p >= 1.f) t = T_LIQ;
    else t = T_IF;
    tmp[i] = t;
}

// liquid cells touching gas become interface; phi, m = phi; interface list;
// active segments
__global__ void __launch_bounds__(256) k_init_state(Dev d, const uint8_t *tmp, int walls) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    const bool inb = x < d.nx;
    const int i = inb ? cell_index(d, x, y, z) : 0;
    bool is_if = false, obs_nbr = false;
    if (inb) {
        uint8_t t = tmp[i];
        bool gas_nbr = false;
        // only a liquid cell, or any cell of a domain with obstacles, depends on its
        // neighbours: most cells of a droplet's box are gas (170 us on 256^3 with every cell looking, 81 now)
        if (walls || t == T_LIQ) {
            for (int q = 1; q < Q; ++q) {
                const uint8_t u = tmp[nbr_index(d, x, y, z, cx(q), cy(q), cz(q))];
                gas_nbr |= u == T_GAS;
                obs_nbr |= u == T_OBS;
            }
        }
        if (t == T_LIQ && gas_nbr) t = T_IF;
        float p = d.phi[i];
        if (t == T_OBS || t == T_GAS) p = 0.f;
        if (t == T_LIQ) p = 1.f;
        d.phi[i] = p;
        d.mass[i] = (t & (T_LIQ | T_IF)) ? p : 0.f;
        d.flags[i] = t | (obs_nbr ? B_NEAR : 0);
        is_if = t == T_IF;
        if (t & (T_LIQ | T_IF)) d.seg_active[seg_of(d, i)] = 1;
    }
    if (__any_sync(0xffffffffu, obs_nbr) && (threadIdx.x & 31) == 0) d.counts[C_NEAR] = 1;
    warp_append(d.iflist, d.counts + d.cif, is_if, i);
}

void launch_init_types(const Dev &d, const uint8_t *obstacle, uint8_t *tmp, cudaStream_t s) {
    k_init_types<<<(unsigned)((d.N + 255) / 256), 256, 0, s>>>(d, obstacle, tmp);
}

// f = w_q in both PDF buffers, 16 bytes a store, one direction per grid row.
// Bound by the memory writes: 19 scattered 4-byte stores a thread in
// k_init_state and a copy of the buffer took 0.24 + 0.38 ms on 256^3 in FP32,
// this takes 0.355 (2.55 GB).
template <int S>
__global__ void __launch_bounds__(256) k_init_pdfs(Dev d, void *f2) {
    using T = typename Store<S>::T;
    constexpr int V = 16 / sizeof(T);
    const int q = blockIdx.y;
    alignas(16) T w[V];  // read as one 16-byte word
#pragma unroll
    for (int e = 0; e < V; ++e) {
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < Q; ++k)
            if (k == q) v = wq(k);
        Store<S>::put(w[e], v, v, d);
    }
    const uint4 v = *reinterpret_cast<const uint4 *>(w);
    T *dst[2] = {static_cast<T *>(d.fdst) + (long long)q * d.N, static_cast<T *>(f2) + (long long)q * d.N};
    // whole 16-byte words of the direction's N values, and its ragged ends
    const long long head = min((long long)((V - (long long)q * d.N % V) % V), d.N), words = (d.N - head) / V;
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x, nth = (long long)gridDim.x * blockDim.x;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        uint4 *p = reinterpret_cast<uint4 *>(dst[b] + head);
        for (long long k = tid; k < words; k += nth) p[k] = v;
        if (tid < head) dst[b][tid] = w[0];
        if (tid < d.N - head - words * V) dst[b][head + words * V + tid] = w[0];
    }
}

template <int S>
static void init_state(const Dev &d, void *f2, const uint8_t *tmp, bool walls, cudaStream_t s) {
    dim3 grid((d.nx + 255) / 256, d.ny, d.nz);
    k_init_pdfs<S><<<dim3(152, Q), 256, 0, s>>>(d, f2);
    k_init_state<<<grid, 256, 0, s>>>(d, tmp, walls ? 1 : 0);
}

void launch_init_state(const Dev &d, void *f2, const uint8_t *tmp, bool walls, cudaStream_t s) {
    switch (d.storage) {
    case FSL_F32: init_state<FSL_F32>(d, f2, tmp, walls, s); break;
    case FSL_F16_OFS: init_state<FSL_F16_OFS>(d, f2, tmp, walls, s); break;
    default: init_state<FSL_BF16_OFS>(d, f2, tmp, walls, s); break;
    }
}

// recompute near-obstacle bits, the interface list and the active segments
// after the caller wrote a state (in place: only the near bit changes, and
// readers look at type bits)
__global__ void __launch_bounds__(256) k_refresh(Dev d) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    const bool inb = x < d.nx;
    const int i = inb ? cell_index(d, x, y, z) : 0;
    bool is_if = false, obs_nbr = false;
    if (inb) {
        const uint8_t t = d.flags[i] & T_MASK;
        for (int q = 1; q < Q; ++q) obs_nbr |= (d.flags[nbr_index(d, x, y, z, cx(q), cy(q), cz(q))] & T_OBS) != 0;
        d.flags[i] = t | (obs_nbr ? B_NEAR : 0);
        is_if = t == T_IF;
        if (t & (T_LIQ | T_IF)) d.seg_active[seg_of(d, i)] = 1;
    }
    if (__any_sync(0xffffffffu, obs_nbr) && (threadIdx.x & 31) == 0) d.counts[C_NEAR] = 1;
    warp_append(d.iflist, d.counts + d.cif, is_if, i);
}

void launch_refresh(const Dev &d, cudaStream_t s) {
    dim3 grid((d.nx + 255) / 256, d.ny, d.nz);
    k_refresh<<<grid, 256, 0, s>>>(d);
}

// ---- prescribed flow (the advection test of Sec. III.A) -------------------------
// f' = feq(rho, u) at every liquid and interface cell of the active segments,
// so that the next step carries the fill level along a constant flow by the
// mass exchange alone.  One warp per 32-cell segment.
template <int S>
__global__ void __launch_bounds__(256) k_prescribe(Dev d, float rho, float ux, float uy, float uz) {
    int cnt[1];
    block_counts<1>(d.counts, {C_SEG}, cnt);
    const int nseg = cnt[0];
    const int lane = threadIdx.x & 31;
    const int gw = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nw = (int)((gridDim.x * blockDim.x) >> 5);
    const float uu = 1.5f * (ux * ux + uy * uy + uz * uz);
    for (int k = gw; k < nseg; k += nw) {
        const int s = d.seg_list[k];
        const int row = s / d.nsegx;
        const int x = (s - row * d.nsegx) * SEG + lane;
        if (x >= d.nx) continue;
        const int z = row / d.ny, y = row - z * d.ny;
        const int i = cell_index(d, x, y, z);
        if (!(d.flags[i] & (T_LIQ | T_IF))) continue;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float cu = cx(q) * ux + cy(q) * uy + cz(q) * uz;
            Store<S>::st(d.fdst, (long long)q * d.N + i, q, wq(q) * rho * (1.0f + 3.0f * cu + 4.5f * cu * cu - uu), d);
        }
    }
}

void launch_prescribe(const Dev &d, float rho, float ux, float uy, float uz, cudaStream_t s) {
    static const int g = resident_grid((const void *)k_prescribe<FSL_F32>, 256);
    switch (d.storage) {
    case FSL_F32: k_prescribe<FSL_F32><<<g, 256, 0, s>>>(d, rho, ux, uy, uz); break;
    case FSL_F16_OFS: k_prescribe<FSL_F16_OFS><<<g, 256, 0, s>>>(d, rho, ux, uy, uz); break;
    default: k_prescribe<FSL_BF16_OFS><<<g, 256, 0, s>>>(d, rho, ux, uy, uz); break;
    }
}

// ---- bubble model: liquid cells, non-obstacle cells, fixed-point fill-level sum ----
// of the current state (the entries of the current list parity and [4]; the
// caller zeroes them first).  Block partials, one integer atomic per block and
// quantity, so the totals do not depend on the order of the additions.
__global__ void __launch_bounds__(256) k_bubble_count(Dev d) {
    long long nl = 0, no = 0, sp = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < d.N; i += (long long)gridDim.x * blockDim.x) {
        const uint8_t t = d.flags[i] & T_MASK;
        nl += t == T_LIQ;
        no += t != T_OBS;
        if (t == T_IF) sp += __double2ll_rn((double)d.phi[i] * BUB_FIX);
    }
    __shared__ long long red[3][8];
    for (int o = 16; o > 0; o >>= 1) {
        nl += __shfl_down_sync(0xffffffffu, nl, o);
        no += __shfl_down_sync(0xffffffffu, no, o);
        sp += __shfl_down_sync(0xffffffffu, sp, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = nl;
        red[1][threadIdx.x >> 5] = no;
        red[2][threadIdx.x >> 5] = sp;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        long long t = 0;
        for (int w = 0; w < 8; ++w) t += red[threadIdx.x][w];
        const int par = list_parity(d);
        const int slot = threadIdx.x == 0 ? par : (threadIdx.x == 1 ? 4 : 2 + par);
        if (t) atomicAdd(reinterpret_cast<unsigned long long *>(d.bub_i + slot), (unsigned long long)t);
    }
}

void launch_bubble_count(const Dev &d, cudaStream_t s) {
    static const int g = resident_grid((const void *)k_bubble_count, 256);
    k_bubble_count<<<g, 256, 0, s>>>(d);
}

// ---- statistics ----------------------------------------------------------------
// stats[0..5]: liquid, interface, gas, obstacle, interface without liquid or gas
// neighbour, liquid touching gas.  One atomic per block and counter.
__global__ void __launch_bounds__(256) k_stats(Dev d) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int c[6] = {0, 0, 0, 0, 0, 0};
    if (i < d.N) {
        int x, y, z;
        cell_coords(d, i, x, y, z);
        const uint8_t t = d.flags[i] & T_MASK;
        c[0] = t == T_LIQ;
        c[1] = t == T_IF;
        c[2] = t == T_GAS;
        c[3] = t == T_OBS;
        if (t == T_IF || t == T_LIQ) {
            bool hl = false, hg = false;
            for (int q = 1; q < Q; ++q) {
                const uint8_t u = d.flags[nbr_index(d, x, y, z, cx(q), cy(q), cz(q))] & T_MASK;
                hl |= u == T_LIQ;
                hg |= u == T_GAS;
            }
            c[4] = t == T_IF && (!hl || !hg);
            c[5] = t == T_LIQ && hg;
        }
    }
    __shared__ int red[6][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = 0; k < 6; ++k) {
        int v = c[k];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[k][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        long long s = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[threadIdx.x][w];
        if (s) atomicAdd(reinterpret_cast<unsigned long long *>(d.stats + threadIdx.x), (unsigned long long)s);
    }
}

void launch_stats(const Dev &d, cudaStream_t s) { k_stats<<<(unsigned)((d.N + 255) / 256), 256, 0, s>>>(d); }

// ---- total mass ----------------------------------------------------------------
// sum over interface cells of m plus sum over liquid cells of rho = sum_q f_q.
// Each block writes one FP64 partial; a single block adds the partials in a
// fixed order, so the result does not depend on scheduling.
constexpr int MASS_THREADS = 256;
constexpr int MASS_BLOCKS = 152 * 8;
int max_partials() { return MASS_BLOCKS; }

template <int S>
__global__ void __launch_bounds__(MASS_THREADS) k_mass_partial(Dev d) {
    double acc = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < d.N; i += (long long)gridDim.x * blockDim.x) {
        const uint8_t t = d.flags[i] & T_MASK;
        if (t == T_IF) {
            acc += d.mass[i];
        } else if (t == T_LIQ) {
            float r = 0.f;
#pragma unroll
            for (int q = 0; q < Q; ++q) r += Store<S>::ld(d.fsrc, (long long)q * d.N + i, q, d);
            acc += r;
        }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    __shared__ double red[MASS_THREADS / 32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < MASS_THREADS / 32; ++w) s += red[w];
        d.partial[blockIdx.x] = s;
    }
}

__global__ void __launch_bounds__(MASS_THREADS) k_mass_final(const double *partial, int n, const double *lost, double *out) {
    __shared__ double red[MASS_THREADS];
    double s = 0.0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) s += partial[k];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = MASS_THREADS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = red[0];
        out[1] = *lost;
    }
}

void launch_mass(const Dev &d, double *out, cudaStream_t s) {
    switch (d.storage) {
    case FSL_F32: k_mass_partial<FSL_F32><<<MASS_BLOCKS, MASS_THREADS, 0, s>>>(d); break;
    case FSL_F16_OFS: k_mass_partial<FSL_F16_OFS><<<MASS_BLOCKS, MASS_THREADS, 0, s>>>(d); break;
    default: k_mass_partial<FSL_BF16_OFS><<<MASS_BLOCKS, MASS_THREADS, 0, s>>>(d); break;
    }
    k_mass_final<<<1, MASS_THREADS, 0, s>>>(d.partial, MASS_BLOCKS, d.lost, out);
}

}  // namespace fslk
