// step_common.cuh -- the phases of a time step as device functions over one
// list entry, segment or warp task, for the kernels of k_step.cu and k_curv.cu.
// Internal to libfsl.
#pragma once

#include "collide.cuh"
#include "curv_common.cuh"

namespace fslk {

// index of the source cell x - c_q of every direction
__device__ __forceinline__ void sources(const Dev &d, int x, int y, int z, int src[Q]) {
    const int xs[3] = {x == d.nx - 1 ? 0 : x + 1, x, x == 0 ? d.nx - 1 : x - 1};  // x - c for c = -1, 0, 1
    const int ys[3] = {y == d.ny - 1 ? 0 : y + 1, y, y == 0 ? d.ny - 1 : y - 1};
    const int zs[3] = {z == d.nz - 1 ? 0 : z + 1, z, z == 0 ? d.nz - 1 : z - 1};
#pragma unroll
    for (int q = 0; q < Q; ++q) src[q] = cell_index(d, xs[cx(q) + 1], ys[cy(q) + 1], zs[cz(q) + 1]);
}

// Liquid cells of the active segment s, one lane per cell (see k_sc_bulk).  The
// pass is bound by instruction issue where the cells come from the L2 or take
// 16 bits, so a PDF is addressed by the unsigned 32-bit index of its cell on a base
// that is the same for the whole grid (of its direction): nine row offsets and
// three columns give the 19 sources.  With 64-bit index arithmetic a segment took
// 800 warp instructions, now 470 in FP32 and 550 in 16 bits: 272 -> 260 us a pass in
// FP32 on the 256^3 pool, 265 -> 213 us in FP16 on the 251 x 251 x 256 pool.
template <int S, int COLL>
__device__ __forceinline__ void bulk_segment(const Dev &d, int s, int lane) {
    using St = Store<S>;
    const int row = div_by(s, d.by_nsegx);
    const int x = (s - row * d.nsegx) * SEG + lane;
    const int z = div_by(row, d.by_ny), y = row - z * d.ny;
    const bool inb = x < d.nx;
    const int r0 = row * d.nx, i = r0 + x;
    const uint8_t fl = inb ? d.flags[i] : (uint8_t)T_GAS;
    if (fl & T_LIQ) {
        // offsets of the source rows (z - cz, y - cy) and columns x - cx
        const int dyp = (y == 0 ? d.ny - 1 : -1) * d.nx, dym = (y == d.ny - 1 ? 1 - d.ny : 1) * d.nx;
        const int pl = d.nx * d.ny;
        const int dzp = (z == 0 ? d.nz - 1 : -1) * pl, dzm = (z == d.nz - 1 ? 1 - d.nz : 1) * pl;
        const int xs[3] = {x == d.nx - 1 ? 0 : x + 1, x, x == 0 ? d.nx - 1 : x - 1};
        const int ys[3] = {dym, 0, dyp}, zs[3] = {dzm, 0, dzp};
        unsigned ro[3][3];
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int c = 0; c < 3; ++c) ro[b][c] = (unsigned)(r0 + zs[b] + ys[c]);
        auto off = [&](int q) { return ro[cz(q) + 1][cy(q) + 1] + (unsigned)xs[cx(q) + 1]; };
        float f[Q];
        if (!(fl & B_NEAR)) {
#pragma unroll
            for (int q = 0; q < Q; ++q) f[q] = St::ld_at(d.fsrc, q, off(q), d);
        } else {
            const unsigned own = (unsigned)i;
            f[0] = St::ld_at(d.fsrc, 0, own, d);
#pragma unroll
            for (int q = 1; q < Q; ++q) {
                const bool wall = (d.flags[off(q)] & T_OBS) != 0;
                f[q] = wall ? St::ld_at(d.fsrc, opp(q), own, d) : St::ld_at(d.fsrc, q, off(q), d);
            }
        }
        float rho;
        collide<COLL>(f, d, rho);
        const unsigned own = (unsigned)i;
#pragma unroll
        for (int q = 0; q < Q; ++q) St::st_at(d.fdst, q, own, f[q], d);
    }
    if (!__any_sync(0xffffffffu, (fl & (T_LIQ | T_IF)) != 0) && lane == 0) {
        d.seg_active[s] = 0;
        d.counts[d.cdirty] = 1;
    }
}

// Interface cells (list), one thread per cell.  Each link is resolved by
// the type of its source cell x - c_q:
//   fluid     f_q(x) = f'_q(x - c_q)                        (Eq. lbe1)
//   gas       f_q(x) = feq_q + feq_qbar - f'_qbar(x)         (Eq. reconstruct)
//             with rho_b = 3 p_g + 6 sigma kappa(x), u_b = u(x, t)
//   obstacle  f_q(x) = f'_qbar(x) (bounce-back), or Eq. reconstruct at a
//             contact-line cell when c_qbar . n_t < 0, n_t the interface normal
//             projected into the wall (Fig. inhomo)
// plus the mass exchange of Eqs. (advection1/2) and the conversion test
// (skipped when the types are frozen).  iface_cell reads kappa(x) and, at
// contact-line cells, the PLIC normal of x -- both the cell's own -- so it may
// run right after the curvature of the same cell, in the same kernel.
template <int S, int COLL>
__device__ __forceinline__ void iface_cell(const Dev &d, int i) {
    using St = Store<S>;
    const long long N = d.N;
    int x, y, z;
    cell_coords(d, i, x, y, z);
    int src[Q];
    sources(d, x, y, z, src);
    const uint8_t fl = d.flags[i];
    float fo[Q], f[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) fo[q] = St::ld(d.fsrc, (long long)q * N + i, q, d);
    uint8_t tq[Q];
    bool has_gas = false, has_obs = false;
    float wx = 0.f, wy = 0.f, wz = 0.f;  // sum of vectors x -> obstacle neighbour
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        tq[q] = d.flags[src[q]] & T_MASK;
        has_gas |= (tq[q] & T_GAS) != 0;
        if (tq[q] & T_OBS) {
            has_obs = true;
            wx -= cx(q);
            wy -= cy(q);
            wz -= cz(q);
        }
    }
    // the PDF and fill level of every source cell, loaded unconditionally
    // (in bounds for every cell type; used only on fluid links) so that
    // all of a cell's loads are in flight together
    float fin[Q], phn[Q];
    fin[0] = phn[0] = 0.f;
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        fin[q] = St::ld(d.fsrc, (long long)q * N + src[q], q, d);
        phn[q] = d.phi[src[q]];
    }
    // u_b: velocity of x at time t from its own post-collision PDFs
    float r0 = 0.f, jx = 0.f, jy = 0.f, jz = 0.f;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        r0 += fo[q];
        jx += cx(q) * fo[q];
        jy += cy(q) * fo[q];
        jz += cz(q) * fo[q];
    }
    const float ux = jx / r0, uy = jy / r0, uz = jz / r0;
    const float uu = 1.5f * (ux * ux + uy * uy + uz * uz);
    const float rho_b = gas_density(d) + d.six_sigma * d.kappa[i];
    const bool corner = has_gas && has_obs;
    float ntx = 0.f, nty = 0.f, ntz = 0.f;
    if (corner) {
        const float4 n4 = d.normal[i];
        const float wl = rsqrtf(wx * wx + wy * wy + wz * wz);
        wx *= wl;
        wy *= wl;
        wz *= wl;
        const float wn = n4.x * wx + n4.y * wy + n4.z * wz;
        ntx = n4.x - wn * wx;
        nty = n4.y - wn * wy;
        ntz = n4.z - wn * wz;
    }
    const float phix = d.phi[i];
    float dm = 0.f;
    f[0] = fo[0];
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        const int qb = opp(q);
        const float cu = cx(q) * ux + cy(q) * uy + cz(q) * uz;
        // feq_q + feq_qbar at (rho_b, u_b): the odd terms cancel
        const float recon = 2.0f * wq(q) * rho_b * (1.0f + 4.5f * cu * cu - uu) - fo[qb];
        const bool fluid = (tq[q] & (T_LIQ | T_IF)) != 0;
        const float kq = (tq[q] & T_LIQ) ? 1.0f : 0.5f * (phix + phn[q]);
        const float outdir = -(cx(q) * ntx + cy(q) * nty + cz(q) * ntz);  // c_qbar . n_t
        const float bound = ((tq[q] & T_OBS) && !(corner && outdir < 0.f)) ? fo[qb] : recon;
        f[q] = fluid ? fin[q] : bound;
        dm += fluid ? kq * (fin[q] - fo[qb]) : 0.f;
    }
    float rho;
    collide<COLL>(f, d, rho);
#pragma unroll
    for (int q = 0; q < Q; ++q) St::st(d.fdst, (long long)q * N + i, q, f[q], d);
    const float m = d.mass[i] + dm;
    d.mass[i] = m;
    d.rho[i] = rho;
    if (d.frozen) return;
    if (m > (1.0f + d.eps) * rho) {
        d.flags[i] = fl | B_TOLIQ;
        d.fill[atomicAdd(d.counts + C_FILL, 1)] = i;
    } else if (m < -d.eps * rho) {
        d.flags[i] = fl | B_TOGAS;
        d.empty[atomicAdd(d.counts + C_EMPTY, 1)] = i;
    }
}

// Lattice directions by pair: pair p (0..8) holds q = 2p + 1 with velocity
// c_p and q + 1 with -c_p.  Components packed two bits per pair (1 -> +1,
// 3 -> -1) so that a lane can decode its own pairs without a table.
constexpr unsigned PAIR_CX = 0x1541u;   // p: 0:+1 1:0 2:0 3:+1 4:+1 5:+1 6:+1 7:0 8:0
constexpr unsigned PAIR_CY = 0x14344u;  // p: 0:0 1:+1 2:0 3:+1 4:-1 5:0 6:0 7:+1 8:+1
constexpr unsigned PAIR_CZ = 0x37410u;  // p: 0:0 1:0 2:+1 3:0 4:0 5:+1 6:-1 7:+1 8:-1
__device__ __forceinline__ int pair_c(unsigned packed, int p) {
    const int v = (packed >> (2 * p)) & 3;
    return v == 3 ? -1 : v;
}

// A cell the fast fit deferred: the streaming Givens fit through accessor acc
// (re-solved in FP64 when ill conditioned), then the cell's interface
// stream-collide.
template <int S, int COLL, class Acc>
__device__ __forceinline__ void general_cell(const Dev &d, const Acc &acc, int i) {
    const uint8_t fi = d.flags[i] & (T_MASK | B_NEAR);
    float cond;
    float kap = lsqr_core<float>(acc, fi, cond);
    if (cond * cond > d.fp64_cond) kap = general_fit_fp64(d, acc, fi);
    d.kappa[i] = kap;
    iface_cell<S, COLL>(d, i);
}

// the same, by one thread reading the block from global memory: a cell the fast
// fit deferred in a step of a domain without obstacles (no contact lines: an
// ill-conditioned or degenerate fit, a few per step and more of them in the necks
// of merging droplets); out of line, so that the fused kernel's registers are not
// spent on it
template <int S, int COLL>
__device__ __noinline__ void general_cell_grid(const Dev &d, int i) {
    int x, y, z;
    cell_coords(d, i, x, y, z);
    const GridAcc acc{d, x, y, z};
    general_cell<S, COLL>(d, acc, i);
}

// L lanes per interface cell (a group), rank r = lane % L.  The fit's 27
// block cells are split t = r, r + L, ...; the 9 direction pairs p = r,
// r + L, ...; the rest population goes to rank L - 1.  Partial sums are
// combined over the group by xor-shuffles in a fixed order.
template <int L>
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
    for (int o = 1; o < L; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
template <int L>
__device__ __forceinline__ int group_or(int v) {
#pragma unroll
    for (int o = 1; o < L; o <<= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// lanes per cell of the fused fit + stream-collide, and the blocks per SM its
// register budget is held to (one wave of the list on a 256^3 droplet)
#ifndef FSL_IFACE_LANES
#define FSL_IFACE_LANES 2
#endif
// list position of the j-th cell of warp gw, which takes `cells` consecutive ones of
// every `stride`
__device__ __forceinline__ int own_place(int gw, int cells, int stride, int j) {
    return gw * cells + j / cells * stride + j % cells;
}

// LSQR fit and interface stream-collide of the list cells base .. base + 32/L - 1
// by one warp, L lanes per cell (see k_curv_iface_fast).  A cell whose fit needs
// the general path is left to k_curv_iface_slow (list d.slow), with OWN to this
// warp itself: its later-th such cell is noted in d.slow at the place of the
// later-th list cell the warp has visited (see own_place), so that no other warp
// or counter is involved.  The whole warp must call it.
template <int S, int COLL, int L, bool OWN>
__device__ __forceinline__ void curv_iface_task(const Dev &d, int base, int n, int lane, int gw, int stride, int &later) {
    using St = Store<S>;
    const long long N = d.N;
    constexpr int RS = (27 + L - 1) / L;  // fit rows per lane
    constexpr int PJ = (9 + L - 1) / L;   // direction pairs per lane
    const int r = lane % L;
    const int k = base + lane / L;
    const bool valid = k < n;
    const int i = d.iflist[valid ? k : base];
    int x, y, z;
    cell_coords(d, i, x, y, z);
    // neighbour coordinates (periodic), picked by select: lane-dependent
    // indices into small arrays would put the arrays in local memory
    const int xm = x == 0 ? d.nx - 1 : x - 1, xp = x == d.nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? d.ny - 1 : y - 1, yp = y == d.ny - 1 ? 0 : y + 1;
    const int zm = z == 0 ? d.nz - 1 : z - 1, zp = z == d.nz - 1 ? 0 : z + 1;
    auto px = [&](int o) { return o < 0 ? xm : (o > 0 ? xp : x); };
    auto py = [&](int o) { return o < 0 ? ym : (o > 0 ? yp : y); };
    auto pz = [&](int o) { return o < 0 ? zm : (o > 0 ? zp : z); };
    // ---- LSQR fit (FP32 normal equations), rows split over the group
    const float4 c4 = d.normal[i];
    uint8_t fjs[RS];
    float4 q4s[RS];
#pragma unroll
    for (int s7 = 0; s7 < RS; ++s7) {
        const int t = r + L * s7;
        const int tt = t < 27 ? t : 13;
        const int jj = cell_index(d, px(tt % 3 - 1), py((tt / 3) % 3 - 1), pz(tt / 9 - 1));
        fjs[s7] = d.flags[jj];
        q4s[s7] = d.normal[jj];
    }
    const uint8_t fl = d.flags[i];
    const float phix = d.phi[i];
    // ---- the stream-collide's loads (independent of kappa), issued with the fit's
    float fo[PJ][2], fin[PJ][2], phn[PJ][2];
    uint8_t tq[PJ][2];
    float fo0 = 0.f;
    float r0 = 0.f, jx = 0.f, jy = 0.f, jz = 0.f, wx = 0.f, wy = 0.f, wz = 0.f;
    int gas = 0, obs = 0;
#pragma unroll
    for (int j = 0; j < PJ; ++j) {
        const int p = r + L * j;
        const int pp = p < 9 ? p : 0;
        const int ex = pair_c(PAIR_CX, pp), ey = pair_c(PAIR_CY, pp), ez = pair_c(PAIR_CZ, pp);
        const int q = 2 * pp + 1;
        const int sq = cell_index(d, px(-ex), py(-ey), pz(-ez));  // x - c_q
        const int sb = cell_index(d, px(ex), py(ey), pz(ez));     // x + c_q
        fo[j][0] = St::ld(d.fsrc, (long long)q * N + i, q, d);
        fo[j][1] = St::ld(d.fsrc, (long long)(q + 1) * N + i, q + 1, d);
        tq[j][0] = d.flags[sq] & T_MASK;
        tq[j][1] = d.flags[sb] & T_MASK;
        fin[j][0] = St::ld(d.fsrc, (long long)q * N + sq, q, d);
        fin[j][1] = St::ld(d.fsrc, (long long)(q + 1) * N + sb, q + 1, d);
        phn[j][0] = d.phi[sq];
        phn[j][1] = d.phi[sb];
    }
    if (r == L - 1) fo0 = St::ld(d.fsrc, i, 0, d);
    const bool nozero = !(c4.x == 0.f && c4.y == 0.f && c4.z == 0.f);
    FastFrame F;
    lsqr_fast_frame(nozero ? c4 : make_float4(0.f, 0.f, 1.f, 0.f), F);
    float G[15], rv[5];
#pragma unroll
    for (int t = 0; t < 15; ++t) G[t] = 0.f;
#pragma unroll
    for (int t = 0; t < 5; ++t) rv[t] = 0.f;
    int m = 0;
    bool contact = r == 0 && (fl & B_NEAR) != 0;
#pragma unroll
    for (int s7 = 0; s7 < RS; ++s7) {
        const int t = r + L * s7;
        if (t < 27) lsqr_fast_row(t, fjs[s7], q4s[s7], F, G, rv, m, contact);
    }
#pragma unroll
    for (int t = 0; t < 15; ++t) G[t] = group_sum<L>(G[t]);
#pragma unroll
    for (int t = 0; t < 5; ++t) rv[t] = group_sum<L>(rv[t]);
#pragma unroll
    for (int o = 1; o < L; o <<= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
    contact = group_or<L>(contact ? 1 : 0) != 0;
    float kap = 0.f;
    const bool ok = nozero ? lsqr_fast_solve(G, rv, m, contact, d.fp64_cond, kap) : true;
    if (!nozero) kap = 0.f;
    const bool defer = valid && !ok;
    const bool act = valid && ok;  // group-uniform
    // ---- interface stream-collide of the cell, direction pairs over the group
#pragma unroll
    for (int j = 0; j < PJ; ++j) {
        const int p = r + L * j;
        if (p < 9) {
            const int ex = pair_c(PAIR_CX, p), ey = pair_c(PAIR_CY, p), ez = pair_c(PAIR_CZ, p);
            r0 += fo[j][0] + fo[j][1];
            const float dj = fo[j][0] - fo[j][1];
            jx += ex * dj;
            jy += ey * dj;
            jz += ez * dj;
            gas |= ((tq[j][0] | tq[j][1]) & T_GAS) ? 1 : 0;
            if (tq[j][0] & T_OBS) { obs = 1; wx -= ex; wy -= ey; wz -= ez; }
            if (tq[j][1] & T_OBS) { obs = 1; wx += ex; wy += ey; wz += ez; }
        }
    }
    if (r == L - 1) r0 += fo0;
    r0 = group_sum<L>(r0);
    jx = group_sum<L>(jx);
    jy = group_sum<L>(jy);
    jz = group_sum<L>(jz);
    wx = group_sum<L>(wx);
    wy = group_sum<L>(wy);
    wz = group_sum<L>(wz);
    gas = group_or<L>(gas);
    obs = group_or<L>(obs);
    const float ux = jx / r0, uy = jy / r0, uz = jz / r0;
    const float uu = 1.5f * (ux * ux + uy * uy + uz * uz);
    const float rho_b = gas_density(d) + d.six_sigma * kap;
    const bool corner = gas && obs;
    float ntx = 0.f, nty = 0.f, ntz = 0.f;
    if (corner) {
        const float wl = rsqrtf(wx * wx + wy * wy + wz * wz);
        const float vx = wx * wl, vy = wy * wl, vz = wz * wl;
        const float wn = c4.x * vx + c4.y * vy + c4.z * vz;
        ntx = c4.x - wn * vx;
        nty = c4.y - wn * vy;
        ntz = c4.z - wn * vz;
    }
    float g[PJ][2];
    float dm = 0.f, rg = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll
    for (int j = 0; j < PJ; ++j) {
        const int p = r + L * j;
        const int pp = p < 9 ? p : 0;
        const int ex = pair_c(PAIR_CX, pp), ey = pair_c(PAIR_CY, pp), ez = pair_c(PAIR_CZ, pp);
        const float w = pp < 3 ? 1.0f / 18.0f : 1.0f / 36.0f;
        const float cu = ex * ux + ey * uy + ez * uz;
        const float base2 = 2.0f * w * rho_b * (1.0f + 4.5f * cu * cu - uu);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float sgn = h == 0 ? 1.0f : -1.0f;  // c = sgn c_p
            const float recon = base2 - fo[j][1 - h];
            const bool fluid = (tq[j][h] & (T_LIQ | T_IF)) != 0;
            const float kq = (tq[j][h] & T_LIQ) ? 1.0f : 0.5f * (phix + phn[j][h]);
            const float outdir = -sgn * (ex * ntx + ey * nty + ez * ntz);  // c_qbar . n_t
            const float bound = ((tq[j][h] & T_OBS) && !(corner && outdir < 0.f)) ? fo[j][1 - h] : recon;
            g[j][h] = fluid ? fin[j][h] : bound;
            dm += (fluid && p < 9) ? kq * (fin[j][h] - fo[j][1 - h]) : 0.f;
        }
        if (p < 9) {
            rg += g[j][0] + g[j][1];
            const float dg = g[j][0] - g[j][1];
            gx += ex * dg;
            gy += ey * dg;
            gz += ez * dg;
        }
    }
    if (r == L - 1) rg += fo0;
    rg = group_sum<L>(rg);
    gx = group_sum<L>(gx);
    gy = group_sum<L>(gy);
    gz = group_sum<L>(gz);
    dm = group_sum<L>(dm);
    // collision (Eq. lbe2) of the cell's own pairs
    const float inv = 1.0f / rg;
    const float vx = gx * inv, vy = gy * inv, vz = gz * inv;
    const float vv = 1.5f * (vx * vx + vy * vy + vz * vz);
#pragma unroll
    for (int j = 0; j < PJ; ++j) {
        const int p = r + L * j;
        const int pp = p < 9 ? p : 0;
        const int ex = pair_c(PAIR_CX, pp), ey = pair_c(PAIR_CY, pp), ez = pair_c(PAIR_CZ, pp);
        const float w = pp < 3 ? 1.0f / 18.0f : 1.0f / 36.0f;
        const int q = 2 * pp + 1;
        const float cu = ex * vx + ey * vy + ez * vz;
        float a0, a1;
        if (COLL == FSL_BGK) {
            const float fe0 = w * rg * (1.0f + 3.0f * cu + 4.5f * cu * cu - vv);
            const float fe1 = w * rg * (1.0f - 3.0f * cu + 4.5f * cu * cu - vv);
            a0 = g[j][0] + d.omega_e * (fe0 - g[j][0]);
            a1 = g[j][1] + d.omega_e * (fe1 - g[j][1]);
        } else {
            const float ep = w * rg * (1.0f + 4.5f * cu * cu - vv);
            const float em = w * rg * 3.0f * cu;
            const float fp = 0.5f * (g[j][0] + g[j][1]), fm = 0.5f * (g[j][0] - g[j][1]);
            const float de = d.omega_e * (fp - ep), dd = d.omega_o * (fm - em);
            a0 = g[j][0] - de - dd;
            a1 = g[j][1] - de + dd;
        }
        if (act && p < 9) {
            St::st(d.fdst, (long long)q * N + i, q, a0, d);
            St::st(d.fdst, (long long)(q + 1) * N + i, q + 1, a1, d);
        }
    }
    if (act && r == L - 1) St::st(d.fdst, i, 0, fo0 + d.omega_e * ((1.0f / 3.0f) * rg * (1.0f - vv) - fo0), d);
    if (OWN) {
        const unsigned dm = __ballot_sync(0xffffffffu, defer && r == 0);
        if (defer && r == 0) d.slow[own_place(gw, 32 / L, stride, later + __popc(dm & ((1u << lane) - 1u)))] = i;
        later += __popc(dm);
    } else {
        warp_append(d.slow, d.counts + C_SLOW, defer && r == 0, i);
    }
    if (act && r == 0) {
        d.kappa[i] = kap;
        const float mm = d.mass[i] + dm;
        d.mass[i] = mm;
        d.rho[i] = rg;
        if (!d.frozen) {
            if (mm > (1.0f + d.eps) * rg) {
                d.flags[i] = fl | B_TOLIQ;
                d.fill[atomicAdd(d.counts + C_FILL, 1)] = i;
            } else if (mm < -d.eps * rg) {
                d.flags[i] = fl | B_TOGAS;
                d.empty[atomicAdd(d.counts + C_EMPTY, 1)] = i;
            }
        }
    }
}

// ---- conversion (the paper cites Koerner et al. for it; readings) -------------
//  A  an emptying cell with a filling D3Q19 neighbour stays interface;
//  B  gas neighbours of filling cells and liquid neighbours of emptying cells
//     become interface (deduplicated by an atomic OR on the flag word);
//  C  new cells from gas get f = feq(mean rho, mean u) of their fluid
//     neighbours and m = 0; cells from liquid keep f and get m = rho;
//  D  the excess mass (m - rho of a filled cell, m of an emptied one) is
//     divided equally among the neighbours that are interface after B; the
//     receivers are marked (rmark) and gather it in k_fin_a.  No receiver:
//     added to `lost`.
// convert_mark does A and B of one converted cell, convert_settle C or D of
// one new or converted cell; each is a warp's work, lane q (1..18) for the
// neighbour x + c_q, and all neighbour loads of a cell are in flight together.
//
// A and B, one pass: a warp takes a converted cell (entry k of the filled
// cells, then the emptying ones) and loads its neighbours' types and segment
// flags once.  A needs only the cell's own neighbours' B_TOLIQ bits (set before
// this phase), and B of a cell only its own A decision and its neighbours'
// types, so no barrier separates them; the B_NEW bits B sets on other cells'
// flag words are atomic, and A's clearing of the cell's own B_TOGAS touches
// only its own byte.
__device__ __forceinline__ void convert_mark(const Dev &d, int k, int nfill, int lane) {
    const bool act = lane >= 1 && lane < Q;
    const int q = act ? lane : 1;
    const bool isfill = k < nfill;
    const int i = isfill ? d.fill[k] : d.empty[k - nfill];
    int x, y, z;
    cell_coords(d, i, x, y, z);
    const int j = act ? nbr_index(d, x, y, z, cx(q), cy(q), cz(q)) : i;
    const uint8_t fj = act ? __ldcg(d.flags + j) : (uint8_t)0;
    const int sj = seg_of(d, j);
    const uint8_t sa = (act && isfill) ? d.seg_active[sj] : (uint8_t)1;
    if (!isfill && __any_sync(0xffffffffu, act && (fj & B_TOLIQ))) {  // warp-uniform
        if (lane == 0) d.flags[i] &= (uint8_t)~B_TOGAS;  // A: stays interface
        return;
    }
    if (act && (isfill ? (fj & T_GAS) : (fj & T_LIQ))) {
        unsigned *word = reinterpret_cast<unsigned *>(d.flags + (j & ~3));
        const int sh = (j & 3) * 8;
        const unsigned old = atomicOr(word, (unsigned)B_NEW << sh);
        if (!((old >> sh) & B_NEW)) {
            if (isfill) {
                d.newgas[atomicAdd(d.counts + C_NEWGAS, 1)] = j;
                if (!sa) {
                    d.seg_active[sj] = 1;
                    d.counts[d.cdirty] = 1;
                }
            } else {
                d.liq2if[atomicAdd(d.counts + C_LIQ2IF, 1)] = j;
            }
        }
    }
}

// C (new cells; lane q (1..18) reads neighbour x + c_q) and D (excess of the
// converted cells) touch disjoint cells and read nothing the other writes, so
// they share one phase: item k < ngas + nliq is a new cell, the rest the
// converted cells
template <int S>
__device__ __forceinline__ void convert_settle(const Dev &d, int k, int ngas, int nliq, int nfill, int lane) {
    using St = Store<S>;
    const long long N = d.N;
    const bool act = lane >= 1 && lane < Q;
    const int q = act ? lane : 1;
    if (k >= ngas + nliq) {
        const int kc = k - ngas - nliq;
        const bool isfill = kc < nfill;
        const int i = isfill ? d.fill[kc] : d.empty[kc - nfill];
        int x, y, z;
        cell_coords(d, i, x, y, z);
        const int j = act ? nbr_index(d, x, y, z, cx(q), cy(q), cz(q)) : i;
        const uint8_t fi = isfill ? (uint8_t)0 : __ldcg(d.flags + i);
        const uint8_t fj = act ? __ldcg(d.flags + j) : (uint8_t)0;
        const float4 ni = d.excess_rule ? d.normal[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float m = lane == 0 ? __ldcg(d.mass + i) : 0.f, r = lane == 0 ? __ldcg(d.rho + i) : 0.f;
        if (!isfill && !(fi & B_TOGAS)) return;  // warp-uniform
        bool recv = false;
        float wgt = 0.f;
        if (act) {
            recv = ((fj & T_IF) && !(fj & (B_TOLIQ | B_TOGAS))) || (fj & B_NEW);
            if (recv) d.rmark[j] = 1;
            if (recv && d.excess_rule) wgt = excess_weight(ni, isfill, cx(q), cy(q), cz(q));
        }
        const int n = __popc(__ballot_sync(0xffffffffu, recv));
        float W = wgt;  // sum of the receivers' weights, fixed order
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) W += __shfl_xor_sync(0xffffffffu, W, o);
        if (lane == 0) {
            const float mex = isfill ? m - r : m;
            const bool weighted = d.excess_rule && W > 0.f;
            d.mass[i] = isfill ? r : 0.f;
            d.excess[i] = weighted ? mex / W : (n ? mex / n : 0.f);
            d.exw[i] = weighted ? 1.f : 0.f;
            if (n == 0) atomicAdd(d.lost, (double)mex);
        }
        return;
    }
    if (k < ngas) {
        const int j = d.newgas[k];
        int x, y, z;
        cell_coords(d, j, x, y, z);
        float r = 0.f, ux = 0.f, uy = 0.f, uz = 0.f, c = 0.f;
        if (act) {  // the neighbour's PDFs are loaded with its type (used only if it is fluid)
            const int l = nbr_index(d, x, y, z, cx(q), cy(q), cz(q));
            const uint8_t fl = __ldcg(d.flags + l);
            float v[Q];
#pragma unroll
            for (int p = 0; p < Q; ++p) v[p] = St::ldcg(d.fdst, (long long)p * N + l, p, d);
            if (fl & (T_LIQ | T_IF)) {
                float jx = 0.f, jy = 0.f, jz = 0.f;
#pragma unroll
                for (int p = 0; p < Q; ++p) {
                    r += v[p];
                    jx += cx(p) * v[p];
                    jy += cy(p) * v[p];
                    jz += cz(p) * v[p];
                }
                ux = jx / r;
                uy = jy / r;
                uz = jz / r;
                c = 1.f;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            r += __shfl_xor_sync(0xffffffffu, r, o);
            ux += __shfl_xor_sync(0xffffffffu, ux, o);
            uy += __shfl_xor_sync(0xffffffffu, uy, o);
            uz += __shfl_xor_sync(0xffffffffu, uz, o);
            c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        const float rb = r / c, vx = ux / c, vy = uy / c, vz = uz / c;
        if (lane < Q) {
            const int p = lane;
            const float uu = 1.5f * (vx * vx + vy * vy + vz * vz);
            const float cu = cx(p) * vx + cy(p) * vy + cz(p) * vz;
            St::st(d.fdst, (long long)p * N + j, p, wq(p) * rb * (1.0f + 3.0f * cu + 4.5f * cu * cu - uu), d);
        }
        if (lane == 0) {
            d.mass[j] = 0.f;
            d.rho[j] = rb;
        }
    } else {
        const int j = d.liq2if[k - ngas];
        float r = lane < Q ? St::ldcg(d.fdst, (long long)lane * N + j, lane, d) : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        if (lane == 0) {
            d.mass[j] = r;
            d.rho[j] = r;
        }
    }
}

// ---- final update ------------------------------------------------------------
// A: cells that are interface at t+1 (old interface cells that did not convert,
//    and the new ones) set phi = m / rho and form the interface list of t+1;
//    those k_convert marked as receivers first gather the excess mass of their
//    converted neighbours in fixed q order (and clear the mark).
// excess mass of the converted neighbours of receiver i added to its mass m
// (out of line: few cells per step take it, and the list loop stays short)
// (the 18 neighbours' types are loaded before any is used: one round of loads,
// then the converted neighbours' excess in the order of q)
static __device__ __noinline__ float gather_excess(const Dev &d, int i, float m) {
    d.rmark[i] = 0;
    int x, y, z;
    cell_coords(d, i, x, y, z);
    int js[Q];
    uint8_t fjs[Q];
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        js[q] = nbr_index(d, x, y, z, cx(q), cy(q), cz(q));
        fjs[q] = d.flags[js[q]];
    }
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        const uint8_t fj = fjs[q];
        if (!(fj & (B_TOLIQ | B_TOGAS))) continue;
        const int j = js[q];
        // the share of this cell, at -c_q seen from the converted cell j
        const float w =
            d.exw[j] != 0.f ? excess_weight(d.normal[j], (fj & B_TOLIQ) != 0, -cx(q), -cy(q), -cz(q)) : 1.f;
        m += d.excess[j] * w;
    }
    d.mass[i] = m;
    return m;
}

// entry k of (interface list, new cells from gas, new cells from liquid): phi of
// the next state; true (and the cell in i) if the cell is interface at t+1.
// any: the step converted some cell.
__device__ __forceinline__ bool fin_cell(const Dev &d, int k, bool valid, int nold, int ngas, bool any, int &i,
                                         long long &phisum) {
    bool keep = false;
    i = 0;
    if (valid) {
        i = k < nold ? d.iflist[k] : (k < nold + ngas ? d.newgas[k - nold] : d.liq2if[k - nold - ngas]);
        // the cell's values in one round of loads
        const uint8_t fl = d.flags[i];
        float m = d.mass[i];
        const float rh = d.rho[i];
        const uint8_t rm = any ? d.rmark[i] : (uint8_t)0;
        if (!(k < nold && (fl & (B_TOLIQ | B_TOGAS)))) {
            if (rm) m = gather_excess(d, i, m);  // a converted neighbour shares its excess
            const float ph = m / rh;
            d.phi[i] = ph;
            if (d.bub_i) phisum += __double2ll_rn((double)ph * BUB_FIX);
            keep = true;
        }
    }
    return keep;
}

// fill level (and mass) of entry k of (filled, emptied)
__device__ __forceinline__ void fin_value(const Dev &d, int k, int nfill) {
    if (k < nfill) {
        d.phi[d.fill[k]] = 1.0f;
    } else {
        const int i = d.empty[k - nfill];
        if (d.flags[i] & B_TOGAS) {
            d.phi[i] = 0.0f;
            d.mass[i] = 0.0f;
        }
    }
}

// final type (transient bits cleared) of entry k of (filled, emptied, new from
// gas, new from liquid)
__device__ __forceinline__ void fin_type(const Dev &d, int k, int nfill, int nempty, int ngas) {
    if (k < nfill) {
        const int i = d.fill[k];
        d.flags[i] = T_LIQ | (d.flags[i] & B_NEAR);
    } else if (k < nfill + nempty) {
        const int i = d.empty[k - nfill];
        const uint8_t fl = d.flags[i];
        if (fl & B_TOGAS) d.flags[i] = T_GAS | (fl & B_NEAR);
    } else {
        const int j = k < nfill + nempty + ngas ? d.newgas[k - nfill - nempty] : d.liq2if[k - nfill - nempty - ngas];
        d.flags[j] = T_IF | (d.flags[j] & B_NEAR);
    }
}

// The list of active segments of the next step by the threads tid = 0 .. nth - 1
// (whole warps); its counter is zero before.
__device__ __forceinline__ void seg_rebuild(const Dev &d, int tid, int nth) {
    // the list again: 16 segment flags per thread (one 16-byte load), a warp
    // scan of the counts and one atomic per warp for the warp's place
    const int lane = threadIdx.x & 31, nchunk = (d.nseg + 15) >> 4;
    for (int base = tid - lane; base < nchunk; base += nth) {  // warp-uniform
        const int c = base + lane;
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        if (c < nchunk) {
            if (16 * c + 16 <= d.nseg) {
                const uint4 v = *reinterpret_cast<const uint4 *>(d.seg_active + 16 * c);
                w[0] = v.x;
                w[1] = v.y;
                w[2] = v.z;
                w[3] = v.w;
            } else {
                for (int b = 0; 16 * c + b < d.nseg; ++b)
                    w[b >> 2] |= (uint32_t)(d.seg_active[16 * c + b] != 0) << (8 * (b & 3));
            }
        }
        uint32_t m = 0u;  // bit b: segment 16 c + b is active
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int b = 0; b < 4; ++b) m |= (((w[k] >> (8 * b)) & 0xffu) != 0u ? 1u : 0u) << (4 * k + b);
        const int cntl = __popc(m);
        int incl = cntl;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        int wbase = 0;
        if (lane == 31 && incl) wbase = atomicAdd(d.counts + C_SEG, incl);
        wbase = __shfl_sync(0xffffffffu, wbase, 31);
        int pos = wbase + incl - cntl;
        while (m) {
            const int b = __ffs(m) - 1;
            m &= m - 1u;
            d.seg_list[pos++] = 16 * c + b;
        }
    }
}

}  // namespace fslk
