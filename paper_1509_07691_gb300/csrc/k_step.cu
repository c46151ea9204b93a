// k_step.cu -- the FSLBM time step (Sec. II): fused pull stream-collide with the
// free-boundary condition and mass exchange, conversion of interface cells
// with excess-mass redistribution, and the update of the cell types, of the
// interface list and of the active segments for the next step.
//
// Work decomposition: liquid cells are processed by k_sc_bulk over the active
// x-row segments (coalesced SoA loads, one thread per cell); interface cells
// by k_curv_iface_fast (LSQR model, fit and stream-collide fused) or
// k_sc_iface (other models) over the interface list; everything after the
// collision only touches list entries, so no pass sweeps the whole grid.
#include "step_common.cuh"

namespace fslk {

constexpr int LIST_BLOCK = 128;

// Liquid cells of the active segments: pull stream (Eq. lbe1) and collide.
// One warp per 32-cell x-row segment, one thread per cell (coalesced SoA
// loads and stores).  A liquid cell next to a wall takes bounce-back
// f_q(x) = f'_qbar(x) on its obstacle links.  Interface cells are left to
// k_sc_iface.  A segment without any liquid or interface cell is marked
// inactive.
template <int S, int COLL>
__global__ void __launch_bounds__(256, S == FSL_F32 ? 5 : 4) k_sc_bulk(Dev d) {
    int cnt[1];
    block_counts<1>(d.counts, {C_SEG}, cnt);
    const int nseg = cnt[0];
    const int lane = threadIdx.x & 31;
    const int gw = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nw = (int)((gridDim.x * blockDim.x) >> 5);
    for (int k = gw; k < nseg; k += nw) bulk_segment<S, COLL>(d, d.seg_list[k], lane);
}

template <int S, int COLL>
__global__ void __launch_bounds__(LIST_BLOCK) k_sc_iface(Dev d) {
    pdl_enter();
    int cnt[1];
    block_counts<1>(d.counts, {d.cif}, cnt);
    const int n = cnt[0];
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x)
        iface_cell<S, COLL>(d, d.iflist[k]);
}

// ---- LSQR curvature fused with the interface stream-collide ----------------------
// With the LSQR model the curvature of a cell and its stream-collide run in
// one pass: k_curv_iface_fast fits the cell by the FP32 normal equations
// (as k_lsqr_fast) and, unless the fit defers the cell to the general path,
// goes straight on with the cell's stream-collide, FSL_IFACE_LANES lanes per
// cell; k_curv_iface_slow finishes the deferred cells one warp each (Givens
// fit, FP64 re-solve when ill conditioned, then iface_cell).  In a step of a
// domain without obstacles (no contact lines: a deferral is an ill-conditioned
// or degenerate fit) each warp finishes its own after its share of the list, one
// lane each, and k_curv_iface_slow is not launched: a serial fit then costs its
// own warp only, and many of them (necks of merging droplets, a low
// lsqr_fp64_cond) spread over the GPU.  Ten steps of two touching droplets in
// 128^3: 1.10 ms; 1.49 with the fits in this kernel's last block behind a fence,
// 1.60 in the conversion kernel (one block behind the liquid pass, 64 registers
// a thread), 1.11 with k_curv_iface_slow launched in every step, which costs 2.5 us
// a step where nothing is deferred (32^3 droplet, ten steps: 225, 276, 232 and 256 us).
// iface_cell of one cell changes only that cell's transient flag bits, mass,
// rho and new PDFs, none of which a fit of another cell reads.
constexpr int IFACE_MIN_BLOCKS = 3;

// OWN: a step (types not frozen) of a domain without obstacles
template <int S, int COLL, int L, bool OWN>
__global__ void __launch_bounds__(LIST_BLOCK, IFACE_MIN_BLOCKS) k_curv_iface_fast(const __grid_constant__ Dev d) {
    pdl_enter();
    int cnt[1];
    block_counts<1>(d.counts, {d.cif}, cnt);
    const int n = cnt[0];
    constexpr int CPW = 32 / L;  // cells per warp
    const int lane = threadIdx.x & 31;
    const int gw = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    int later = 0;  // this warp's deferred cells (steps without obstacles)
    for (int base = gw * CPW; base < n; base += nwarps * CPW)
        curv_iface_task<S, COLL, L, OWN>(d, base, n, lane, gw, nwarps * CPW, later);
    if (!OWN) return;
    __syncwarp();
    for (int j = lane; j < later; j += 32) general_cell_grid<S, COLL>(d, d.slow[own_place(gw, CPW, nwarps * CPW, j)]);
}

// General-path cells (contact-line cells, degenerate or ill-conditioned FP32
// fits) of a domain with obstacles or of frozen steps: one warp per cell stages the
// block in shared memory and runs the Givens fit as a pipeline over its lanes
// (general_fit_warp), then one lane the interface stream-collide of the cell.
// PIPE: the fit by lsqr_warp; else lsqr_core by one lane.  The two differ in
// which products are fused (kappa by about 1e-7), and a window's gradients
// magnify the last bits of its states near full and empty cells, so the frozen
// steps of a window keep the one-lane order.
template <int S, int COLL, bool PIPE>
__global__ void __launch_bounds__(LIST_BLOCK) k_curv_iface_slow(const __grid_constant__ Dev d) {
    pdl_enter();
    __shared__ uint8_t sfl[LIST_BLOCK / 32][128];
    __shared__ float4 snm[LIST_BLOCK / 32][27];
    __shared__ FitRows rows[LIST_BLOCK / 32];
    int cnt[1];
    block_counts<1>(d.counts, {C_SLOW}, cnt);
    const int n = cnt[0];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int gw = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nw = (int)((gridDim.x * blockDim.x) >> 5);
    for (int k = gw; k < n; k += nw) {
        const int i = d.slow[k];
        int x, y, z;
        cell_coords(d, i, x, y, z);
        stage_block(d, x, y, z, lane, sfl[w], snm[w]);
        __syncwarp();
        const StagedAcc acc{d, sfl[w], snm[w]};
        if (PIPE) {
            const uint8_t fi = d.flags[i] & (T_MASK | B_NEAR);
            const float kap = general_fit_warp(d, acc, fi, lane, rows[w]);
            if (lane == 0) {
                d.kappa[i] = kap;
                iface_cell<S, COLL>(d, i);
            }
        } else if (lane == 0) {
            general_cell<S, COLL>(d, acc, i);
        }
        __syncwarp();
    }
}

// ---- conversion ------------------------------------------------------------------
// One block of 1024 threads with a block barrier between the two phases, which
// keeps every phase visible to the next: a droplet's step converts a handful of
// cells.  A step of a wide pool converts many, and there this block, behind the
// liquid pass, is 35 us of the step (4 us where nothing converts).
constexpr int CONV_BLOCK = 1024;

template <int S>
__global__ void __launch_bounds__(CONV_BLOCK) k_convert(Dev d) {
    pdl_enter();
    const int nfill = __ldcg(d.counts + C_FILL), nempty = __ldcg(d.counts + C_EMPTY);
    if (nfill + nempty == 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int k = warp; k < nfill + nempty; k += nwarps) convert_mark(d, k, nfill, lane);
    __syncthreads();
    const int ngas = __ldcg(d.counts + C_NEWGAS), nliq = __ldcg(d.counts + C_LIQ2IF);
    for (int k = warp; k < ngas + nliq + nfill + nempty; k += nwarps) convert_settle<S>(d, k, ngas, nliq, nfill, lane);
}

// ---- final update ------------------------------------------------------------
__global__ void __launch_bounds__(LIST_BLOCK) k_fin_a(Dev d) {
    pdl_enter();
    int cnt[6];
    block_counts<6>(d.counts, {d.cif, C_NEWGAS, C_LIQ2IF, C_FILL, C_EMPTY, d.cdirty}, cnt);
    if (blockIdx.x == 0 && threadIdx.x == 0 && cnt[5]) d.counts[C_SEG] = 0;  // filled again by k_fin_b
    const int nold = cnt[0], ngas = cnt[1], nliq = cnt[2];
    const bool any = (cnt[3] + cnt[4]) > 0;
    long long phisum = 0;  // bubble model: fixed-point fill levels of the next interface cells
    warp_uniform_loop(nold + ngas + nliq, [&](int k, bool valid) {
        int i;
        const bool keep = fin_cell(d, k, valid, nold, ngas, any, i, phisum);
        warp_append(d.iflist_next, d.counts + d.cif_next, keep, i);
    });
    if (d.bub_i) {  // block-uniform
        for (int o = 16; o > 0; o >>= 1) phisum += __shfl_down_sync(0xffffffffu, phisum, o);
        __shared__ long long red[LIST_BLOCK / 32];
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = phisum;
        __syncthreads();
        if (threadIdx.x == 0) {
            long long t = 0;
            for (int w = 0; w < LIST_BLOCK / 32; ++w) t += red[w];
            if (t) atomicAdd(reinterpret_cast<unsigned long long *>(d.bub_i + 2 + (list_parity(d) ^ 1)),
                             (unsigned long long)t);
        }
    }
}

// B: final types of the converted cells (transient bits cleared), and the
// list of active segments for the next step (warp-scan compaction),
// rebuilt only when a segment was switched on or off during the step
__global__ void __launch_bounds__(256) k_fin_b(Dev d) {
    pdl_enter();
    int cnt[5];
    block_counts<5>(d.counts, {C_FILL, C_EMPTY, C_NEWGAS, C_LIQ2IF, d.cdirty}, cnt);
    const int nfill = cnt[0], nempty = cnt[1], ngas = cnt[2], nliq = cnt[3];
    const int n = nfill + nempty + ngas + nliq;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    if (d.bub_i && tid == 0) {  // liquid cells of the next state: filled cells join, cells from liquid leave
        const int par = list_parity(d);
        d.bub_i[par ^ 1] = d.bub_i[par] + nfill - nliq;
    }
    for (int k = tid; k < n; k += nth) {
        if (k < nfill + nempty) fin_value(d, k, nfill);
        fin_type(d, k, nfill, nempty, ngas);
    }
    if (!cnt[4]) return;  // the set of active segments did not change (block-uniform)
    seg_rebuild(d, tid, nth);
}

// Final update of a step with frozen types (no conversion, the interface
// list and the active segments stay): phi = m / rho of the interface cells.
__global__ void __launch_bounds__(LIST_BLOCK) k_fin_frozen(Dev d) {
    int cnt[1];
    block_counts<1>(d.counts, {d.cif}, cnt);
    const int n = cnt[0];
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int i = d.iflist[k];
        d.phi[i] = d.mass[i] / d.rho[i];
    }
}

void launch_fin_frozen(const Dev &d, cudaStream_t s) {
    static const int g = list_blocks((const void *)k_fin_frozen, LIST_BLOCK, 4);
    k_fin_frozen<<<g, LIST_BLOCK, 0, s>>>(d);
}

// active segments -> list (warp-ballot compaction); counter zeroed first
__global__ void __launch_bounds__(256) k_seg_compact(Dev d) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const bool act = s < d.nseg && d.seg_active[s];
    warp_append(d.seg_list, d.counts + C_SEG, act, s);
}

void launch_seg_compact(const Dev &d, cudaStream_t s) {
    cudaMemsetAsync(d.counts + C_SEG, 0, sizeof(int), s);
    k_seg_compact<<<(d.nseg + 255) / 256, 256, 0, s>>>(d);
}

template <int S, int COLL>
void launch_bulk(const Dev &d, cudaStream_t s) {
    static const int gb = resident_grid((const void *)k_sc_bulk<S, COLL>, 256);
    k_sc_bulk<S, COLL><<<gb, 256, 0, s>>>(d);
}

template <int S, int COLL>
void launch_iface(const Dev &d, cudaStream_t s) {
    static const int gi = list_blocks((const void *)k_sc_iface<S, COLL>, LIST_BLOCK, 4);
    launch_pdl(k_sc_iface<S, COLL>, gi, LIST_BLOCK, s, d);
}

#define FSL_DISPATCH(FN)                                                                          \
    do {                                                                                          \
        const bool trt = d.collision == FSL_TRT;                                                  \
        switch (d.storage) {                                                                      \
        case FSL_F32: trt ? FN<FSL_F32, FSL_TRT>(d, s) : FN<FSL_F32, FSL_BGK>(d, s); break;        \
        case FSL_F16_OFS: trt ? FN<FSL_F16_OFS, FSL_TRT>(d, s) : FN<FSL_F16_OFS, FSL_BGK>(d, s); break; \
        default: trt ? FN<FSL_BF16_OFS, FSL_TRT>(d, s) : FN<FSL_BF16_OFS, FSL_BGK>(d, s); break;   \
        }                                                                                         \
    } while (0)

template <int S, int COLL>
void launch_ci(const Dev &d, cudaStream_t s) {
    static const int go = list_blocks((const void *)k_curv_iface_fast<S, COLL, FSL_IFACE_LANES, true>, LIST_BLOCK, 4);
    static const int gf = list_blocks((const void *)k_curv_iface_fast<S, COLL, FSL_IFACE_LANES, false>, LIST_BLOCK, 4);
    static const int gs = list_blocks((const void *)k_curv_iface_slow<S, COLL, true>, LIST_BLOCK, 4);
    static const int gz = list_blocks((const void *)k_curv_iface_slow<S, COLL, false>, LIST_BLOCK, 4);
    if (d.inline_general && !d.frozen) {  // the fused kernel finishes its deferred fits itself
        launch_pdl(k_curv_iface_fast<S, COLL, FSL_IFACE_LANES, true>, go, LIST_BLOCK, s, d);
        return;
    }
    launch_pdl(k_curv_iface_fast<S, COLL, FSL_IFACE_LANES, false>, gf, LIST_BLOCK, s, d);
    if (d.frozen) launch_pdl(k_curv_iface_slow<S, COLL, false>, gz, LIST_BLOCK, s, d);
    else launch_pdl(k_curv_iface_slow<S, COLL, true>, gs, LIST_BLOCK, s, d);
}

template <int S, int COLL>
void launch_conv(const Dev &d, cudaStream_t s) {
    launch_pdl(k_convert<S>, 1, CONV_BLOCK, s, d);
}

void launch_sc_bulk(const Dev &d, cudaStream_t s) { FSL_DISPATCH(launch_bulk); }
void launch_convert(const Dev &d, cudaStream_t s) { FSL_DISPATCH(launch_conv); }
void launch_curv_iface(const Dev &d, cudaStream_t s) { FSL_DISPATCH(launch_ci); }
void launch_sc_iface(const Dev &d, cudaStream_t s) { FSL_DISPATCH(launch_iface); }
#undef FSL_DISPATCH

void launch_finalize(const Dev &d, cudaStream_t s) {
    static const int ga = list_blocks((const void *)k_fin_a, LIST_BLOCK, 4);
    static const int gb = list_blocks((const void *)k_fin_b, 256, 4);
    launch_pdl(k_fin_a, ga, LIST_BLOCK, s, d);
    launch_pdl(k_fin_b, gb, 256, s, d);
}

}  // namespace fslk
