// spread_det.cu -- order-deterministic spreading (A2 + A3) of libiblb.
//
// Eq. 8 of the paper, F(x) = sum_j phi_j Delta(q_j - x), written as a gather:
// every cell sums the contributions of the nodes whose stencils cover it in
// a fixed order, so that FP64 runs are bitwise reproducible (the scatter
// with atomics in ib.cu adds in whatever order the hardware serves them).
//
// Per step:
//   0. k_det_clear   the counters (one kernel: a memset node costs a step 3 us,
//                    a kernel 1);
//   1. k_det_bin     per node: the 1D delta weights (as node_lines), the
//                    stencil origin o = floor(q) - 1 per axis, the node's
//                    bin (a tile of DT^D stencil origins), a count per bin,
//                    and the cell tiles its stencil touches (each appended
//                    once to a list of active cell tiles);
//   2. k_det_scan    exclusive prefix sum of the bin counts (one block, 4096
//                    counts at a time);
//   3. k_det_place   node items into their bins' ranges;
//   4. k_det_sort    each bin's items into increasing order;
//   5. k_det_gather  per active cell tile: the bins that can hold a node
//                    covering one of its cells, in a fixed order, and their
//                    nodes in increasing order, staged in shared memory with
//                    their weights at the tile's four coordinates per axis;
//                    every cell sums the nodes that cover it.  F(x) is written
//                    (not added: the band buffer is zero there) and the
//                    cell's band segment flagged.
// The gather used to walk the bins cell by cell, matching every node's stencil
// origin against the cell with a remainder per axis and line: 64 times the
// index work of a node, and most of the step.  10 242 nodes on 96 x 96 x 72 in
// FP64: spread 447 -> 93 us per step (128 before the bins were sorted by warps).
// Only the order of the additions differs from the scatter: the weights are
// the same numbers, formed the same way (3D binary16: to their last bits, see
// delta4_weights).  The same kernels serve the
// single-simulation engine (one slot, node item = node id) and the batched
// engine (items = (slot, node) pairs in slot order, bins and cell tiles
// numbered globally across slots).
#include "ib_core.cuh"
#include "spread_det.cuh"

namespace iblb {
namespace {

constexpr int DT = DET_TILE;     // tile edge in cells (bins and cell tiles)
constexpr int SCAN_BLOCK = 1024;

__device__ __forceinline__ int2 item_of(const int2* __restrict__ items, int it)
{
    return items ? items[it] : make_int2(0, it);
}

__device__ __forceinline__ int wrap(int v, int n)
{
    const int r = v % n;
    return r < 0 ? r + n : r;
}

// Axis k of a slot is periodic unless it is the wall axis with walls.
__device__ __forceinline__ bool periodic_axis(const GridParams& g, int k)
{
    return !(g.walls && k == g.dim - 1);
}

__device__ __forceinline__ int extent(const GridParams& g, int k)
{
    return k == 0 ? g.nx : (k == 1 ? g.ny : g.nz);
}

// Bin coordinate of stencil origin o along axis k: o mod n on periodic axes,
// o + 3 along the wall axis (origins -2 .. n-2 reach a fluid layer, bins
// 1 .. n+1).
__device__ __forceinline__ int bin_coord(const GridParams& g, int k, int o)
{
    return periodic_axis(g, k) ? wrap(o, extent(g, k)) : o + 3;
}

template <int D, typename R, bool KEEP>
__global__ void k_det_bin(const DetSlot* __restrict__ slots, const int2* __restrict__ items,
                          int nitems, int* __restrict__ bin_of, int* __restrict__ org,
                          R* __restrict__ wts, int* __restrict__ cnt, int* __restrict__ active,
                          int2* __restrict__ act_list, int* __restrict__ nact)
{
    const int it = blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= nitems) return;
    const int2 sj = item_of(items, it);
    const DetSlot& d = slots[sj.x];
    const GridParams g = d.g;
    const double* q = d.q + (long long)D * sj.y;
    int o[3] = {0, 0, 0};
    bool ok = true;
    for (int k = 0; k < D; k++) {
        const double qk = q[k];
        if (!(fabs(qk) < 1.0e9)) {  // a diverged node touches nothing
            ok = false;
            break;
        }
        const double fl = floor(qk);
        o[k] = (int)fl - 1;
        const R fr = (R)(qk - fl);  // as node_lines: FP64 split, weights in R
        R w4[4];
        delta4_weights<R, KEEP>(fr, w4);
        for (int s = 0; s < 4; s++) wts[(long long)it * 12 + 4 * k + s] = w4[s];
        org[3 * it + k] = o[k];
    }
    int b[3] = {0, 0, 0};
    if (ok) {
        for (int k = 0; k < D; k++) {
            b[k] = bin_coord(g, k, o[k]);
            if (!periodic_axis(g, k) && (b[k] < 1 || b[k] > extent(g, k) + 1)) ok = false;
        }
    }
    if (!ok) {
        bin_of[it] = -1;
        return;
    }
    const int bin = d.bin_base + b[0] / DT +
                    d.nb[0] * (b[1] / DT + (D == 3 ? d.nb[1] * (b[2] / DT) : 0));
    bin_of[it] = bin;
    atomicAdd(&cnt[bin], 1);
    // cell tiles touched by the stencil lines o .. o+3 (fluid layers only
    // along the wall axis); each is appended to the active list once
    int tl[3][4], nt[3] = {0, 0, 1};
    tl[2][0] = 0;
    for (int k = 0; k < D; k++) {
        const int n = extent(g, k);
        for (int s = 0; s < 4; s++) {
            int c = o[k] + s;
            if (periodic_axis(g, k)) {
                c = wrap(c, n);
            } else if (c < 1 || c > n - 2) {
                continue;
            }
            const int t = c / DT;
            bool seen = false;
            for (int u = 0; u < nt[k]; u++) seen |= (tl[k][u] == t);
            if (!seen) tl[k][nt[k]++] = t;
        }
    }
    for (int a = 0; a < nt[0]; a++)
        for (int c1 = 0; c1 < nt[1]; c1++)
            for (int c2 = 0; c2 < nt[2]; c2++) {
                const int local = tl[0][a] + d.ct[0] * (tl[1][c1] + (D == 3 ? d.ct[1] * tl[2][c2] : 0));
                if (atomicExch(&active[d.cell_base + local], 1) == 0)
                    act_list[atomicAdd(nact, 1)] = make_int2(sj.x, local);
            }
}

__global__ void k_det_clear(int* __restrict__ cnt, int nbins, int* __restrict__ active, int ntiles,
                            int* __restrict__ nact)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    for (int i = t; i < nbins; i += nt) cnt[i] = 0;
    for (int i = t; i < ntiles; i += nt) active[i] = 0;
    if (t == 0) *nact = 0;
}

// Exclusive prefix sum of cnt[0 .. n) into start and cur (one block): 4
// consecutive counts per thread, a scan in each warp and one over the warps.
__global__ void __launch_bounds__(SCAN_BLOCK)
k_det_scan(const int* __restrict__ cnt, int n, int* __restrict__ start, int* __restrict__ cur)
{
    __shared__ int wsum[SCAN_BLOCK / 32];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    int base = 0;
    for (int i0 = 0; i0 < n; i0 += 4 * SCAN_BLOCK) {
        const int i = i0 + 4 * t;
        int c[4], s = 0;
        if (i + 3 < n) {
            const int4 v = *reinterpret_cast<const int4*>(cnt + i);  // i is a multiple of 4
            c[0] = v.x;
            c[1] = v.y;
            c[2] = v.z;
            c[3] = v.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; k++) c[k] = i + k < n ? cnt[i + k] : 0;
        }
        s = c[0] + c[1] + c[2] + c[3];
        int incl = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) wsum[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            int w = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += v;
            }
            wsum[lane] = w;
        }
        __syncthreads();
        int run = base + (wid ? wsum[wid - 1] : 0) + incl - s;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if (i + k < n) {
                start[i + k] = run;
                cur[i + k] = run;
            }
            run += c[k];
        }
        base += wsum[SCAN_BLOCK / 32 - 1];
        __syncthreads();  // wsum is written again in the next round
    }
}

__global__ void k_det_place(const int* __restrict__ bin_of, int nitems, int* __restrict__ cur,
                            int* __restrict__ list)
{
    const int it = blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= nitems) return;
    const int b = bin_of[it];
    if (b >= 0) list[atomicAdd(&cur[b], 1)] = it;
}

// Each bin's range into increasing order, one warp per bin: every lane counts
// the ids below its own (they are distinct), which is its place.  One thread
// per bin inserting in global memory took 47 us where a fine mesh puts some
// 20 nodes into a bin (10 242 nodes of a sphere of radius 24), this 6 us.
__global__ void k_det_sort(const int* __restrict__ cnt, const int* __restrict__ start, int nbins,
                           int* __restrict__ list)
{
    const int b = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (b >= nbins) return;
    const int c = cnt[b];
    if (c < 2) return;
    int* l = list + start[b];
    constexpr int PER = 8;  // ids per lane
    if (c <= 32) {
        const int v = lane < c ? l[lane] : 0x7fffffff;
        int r = 0;
        for (int k = 0; k < c; k++) r += __shfl_sync(0xffffffffu, v, k) < v;
        __syncwarp();
        if (lane < c) l[r] = v;
    } else if (c <= 32 * PER) {
        int v[PER], r[PER];
#pragma unroll
        for (int m = 0; m < PER; m++) {
            v[m] = lane + 32 * m < c ? l[lane + 32 * m] : 0x7fffffff;
            r[m] = 0;
        }
        for (int k = 0; k < c; k++) {
            const int x = l[k];
#pragma unroll
            for (int m = 0; m < PER; m++) r[m] += x < v[m];
        }
        __syncwarp();  // every id is read before the first is written
#pragma unroll
        for (int m = 0; m < PER; m++)
            if (lane + 32 * m < c) l[r[m]] = v[m];
    } else if (lane == 0) {  // nodes heaped on one another
        for (int i = 1; i < c; i++) {
            const int v = l[i];
            int k = i - 1;
            while (k >= 0 && l[k] > v) {
                l[k + 1] = l[k];
                k--;
            }
            l[k + 1] = v;
        }
    }
}

// Cell coordinates of tile tc along axis k that can carry force: [lo, hi].
__device__ __forceinline__ void tile_range(const GridParams& g, int k, int tc, int& lo, int& hi)
{
    const int n = extent(g, k);
    lo = tc * DT;
    hi = min(lo + DT, n) - 1;
    if (!periodic_axis(g, k)) {  // fluid layers only
        lo = max(lo, 1);
        hi = min(hi, n - 2);
    }
}

// Bin tiles along axis k whose origins can cover a cell of [lo, hi], in a
// fixed order (origins hi, hi - 1, .. lo - 3), without repeats: at most 4.
__device__ __forceinline__ int source_bins(const GridParams& g, int k, int lo, int hi, int* out)
{
    int n = 0;
    for (int o = hi; o >= lo - 3; o--) {
        const int b = bin_coord(g, k, o) / DT;
        bool seen = false;
        for (int u = 0; u < n; u++) seen |= (out[u] == b);
        if (!seen) out[n++] = b;
    }
    return n;
}

// 1D weights of a node (origin o, line weights w) on axis k at the DT
// coordinates x0 ..; bit l of the result is set when a stencil line lands on
// x0 + l.  On a periodic axis of fewer than 4 cells several lines land on one
// coordinate and their weights add up.
template <typename R>
__device__ __forceinline__ unsigned axis_weights(const GridParams& g, int k, int o,
                                                 const R* __restrict__ w, int x0, R* out)
{
    const int n = extent(g, k);
    const bool per = periodic_axis(g, k);
    unsigned hits = 0;
    if (per && n < 4) {
        for (int l = 0; l < DT; l++) {
            R s = R(0);
            for (int t = 0; t < 4; t++)
                if (wrap(o + t, n) == x0 + l) {
                    s = (hits >> l) & 1u ? s + w[t] : w[t];
                    hits |= 1u << l;
                }
            out[l] = s;
        }
        return hits;
    }
    int d = per ? wrap(x0 - o, n) : x0 - o;
#pragma unroll
    for (int l = 0; l < DT; l++) {
        const bool h = d >= 0 && d < 4;
        out[l] = h ? w[d] : R(0);
        hits |= h ? 1u << l : 0u;
        d++;
        if (per && d >= n) d -= n;
    }
    return hits;
}

// One block per active cell tile (64 threads and cells in 3D; 32 threads, 16
// of them with a cell, in 2D); every thread stages one node of a batch.
template <int D> constexpr int gather_block() { return D == 3 ? 64 : 32; }

template <int D, typename R>
__global__ void __launch_bounds__(gather_block<D>())
k_det_gather(const DetSlot* __restrict__ slots, const int2* __restrict__ items,
             const int2* __restrict__ act_list, const int* __restrict__ nact,
             const int* __restrict__ cnt, const int* __restrict__ start,
             const int* __restrict__ list, const int* __restrict__ org, const R* __restrict__ wts)
{
    constexpr int B = gather_block<D>();
    constexpr int CELLS = (D == 3) ? DT * DT * DT : DT * DT;
    constexpr int MAXBINS = (D == 3) ? 64 : 16;
    __shared__ int s_bin[3][4], s_ns[3];
    __shared__ int s_first[MAXBINS], s_end[MAXBINS];  // list range start, running total
    __shared__ R s_w[B][3][DT], s_phi[B][3];
    __shared__ unsigned s_hit[B];
    const int t = threadIdx.x;
    const int n_act = *nact;
    for (int a = blockIdx.x; a < n_act; a += gridDim.x) {
        const int2 st = act_list[a];
        const DetSlot& d = slots[st.x];
        const GridParams g = d.g;
        int tc[3];
        tc[0] = st.y % d.ct[0];
        tc[1] = (st.y / d.ct[0]) % d.ct[1];
        tc[2] = (D == 3) ? st.y / (d.ct[0] * d.ct[1]) : 0;
        __syncthreads();  // the last tile's shared arrays are read
        if (t < 3) {
            int nb = 1;
            s_bin[t][0] = 0;
            if (t < D) {
                int lo, hi;
                tile_range(g, t, tc[t], lo, hi);
                nb = source_bins(g, t, lo, hi, s_bin[t]);
            }
            s_ns[t] = nb;
        }
        __syncthreads();
        const int n0 = s_ns[0], n1 = s_ns[1], nbt = n0 * n1 * s_ns[2];
        if (t < nbt) {
            const int i0 = t % n0, i1 = (t / n0) % n1, i2 = t / (n0 * n1);
            const int bin = d.bin_base + s_bin[0][i0] +
                            d.nb[0] * (s_bin[1][i1] + (D == 3 ? d.nb[1] * s_bin[2][i2] : 0));
            s_first[t] = start[bin];
            s_end[t] = cnt[bin];
        }
        __syncthreads();
        if (t == 0)
            for (int b = 1; b < nbt; b++) s_end[b] += s_end[b - 1];
        __syncthreads();
        const int total = nbt > 0 ? s_end[nbt - 1] : 0;
        const int l0 = t % DT, l1 = (t / DT) % DT, l2 = (D == 3) ? t / (DT * DT) : 0;
        const int x[3] = {tc[0] * DT + l0, tc[1] * DT + l1, tc[2] * DT + l2};
        bool inside = t < CELLS;
        for (int k = 0; k < D; k++) {
            int lo, hi;
            tile_range(g, k, tc[k], lo, hi);
            if (x[k] < lo || x[k] > hi) inside = false;
        }
        R acc[3] = {R(0), R(0), R(0)};
        bool touched = false;
        for (int e0 = 0; e0 < total; e0 += B) {
            const int m = min(B, total - e0);
            if (e0) __syncthreads();
            if (t < m) {
                const int e = e0 + t;
                int b = 0;
                while (e >= s_end[b]) b++;
                const int it = list[s_first[b] + e - (b ? s_end[b - 1] : 0)];
                const R* w = wts + (long long)it * 12;
                unsigned hit = 0;
#pragma unroll
                for (int k = 0; k < D; k++)
                    hit |= axis_weights<R>(g, k, org[3 * it + k], w + 4 * k, tc[k] * DT, s_w[t][k]) << (4 * k);
                s_hit[t] = hit;
                const int j = item_of(items, it).y;
                for (int k = 0; k < D; k++) s_phi[t][k] = (R)d.phi[(long long)D * j + k];
            }
            __syncthreads();
            if (inside) {
                for (int i = 0; i < m; i++) {
                    const unsigned hit = s_hit[i];
                    if (!((hit >> l0) & (hit >> (4 + l1)) & (D == 3 ? hit >> (8 + l2) : 1u) & 1u)) continue;
                    const R w01 = s_w[i][0][l0] * s_w[i][1][l1];
                    const R ww = (D == 3) ? w01 * s_w[i][2][l2] : w01;
                    for (int k = 0; k < D; k++) acc[k] += s_phi[i][k] * ww;
                    touched = true;
                }
            }
        }
        if (!touched) continue;
        const long long cell = ((long long)x[2] * g.ny + x[1]) * g.nx + x[0];
        R* F = (R*)d.F;
        if constexpr (sizeof(R) == 4)  // float4 per cell
            reinterpret_cast<float4*>(F)[cell] = make_float4(acc[0], acc[1], D == 3 ? acc[2] : 0.f, 0.f);
        else
            for (int k = 0; k < D; k++) F[(long long)k * g.ncell + cell] = acc[k];
        const long long row = (long long)x[2] * g.ny + x[1];
        d.flags[row * g.nseg_x + (x[0] >> 5)] = 1;
    }
}

template <int D, typename R, bool KEEP>
void launch_det_t(const DetSlot* slots, const int2* items, int nitems, const DetBuffers& b,
                  int nbins, int ncelltiles, int sm_count, cudaStream_t s)
{
    const int nclr = nbins > ncelltiles ? nbins : ncelltiles;
    k_det_clear<<<min((nclr + 255) / 256, 4 * sm_count), 256, 0, s>>>(b.cnt, nbins, b.active,
                                                                      ncelltiles, b.nact);
    const int nb = (nitems + 127) / 128, nb64 = (nitems + 63) / 64;
    k_det_bin<D, R, KEEP><<<nb64, 64, 0, s>>>(slots, items, nitems, b.bin_of, b.org, (R*)b.wts, b.cnt,
                                       b.active, b.act_list, b.nact);
    k_det_scan<<<1, SCAN_BLOCK, 0, s>>>(b.cnt, nbins, b.start, b.cur);
    k_det_place<<<nb, 128, 0, s>>>(b.bin_of, nitems, b.cur, b.list);
    k_det_sort<<<(nbins + 3) / 4, 128, 0, s>>>(b.cnt, b.start, nbins, b.list);
    k_det_gather<D, R><<<sm_count * 16, gather_block<D>(), 0, s>>>(
        slots, items, b.act_list, b.nact, b.cnt, b.start, b.list, b.org, (const R*)b.wts);
}

}  // namespace

void launch_spread_det(int storage, int dim, const DetSlot* slots, const int2* items, int nitems,
                       const DetBuffers& b, int nbins, int ncelltiles, int sm_count,
                       cudaStream_t s)
{
    if (nitems <= 0) return;
    if (storage == ST_FP64) {
        if (dim == 2) launch_det_t<2, double, false>(slots, items, nitems, b, nbins, ncelltiles, sm_count, s);
        else launch_det_t<3, double, false>(slots, items, nitems, b, nbins, ncelltiles, sm_count, s);
    } else {
        if (dim == 2) launch_det_t<2, float, true>(slots, items, nitems, b, nbins, ncelltiles, sm_count, s);
        else if (keep_weights_3d(storage, true)) launch_det_t<3, float, true>(slots, items, nitems, b, nbins, ncelltiles, sm_count, s);
        else launch_det_t<3, float, false>(slots, items, nitems, b, nbins, ncelltiles, sm_count, s);
    }
}

void det_tiles(const GridParams& g, int nb[3], int ct[3])
{
    for (int k = 0; k < 3; k++) {
        nb[k] = 1;
        ct[k] = 1;
    }
    for (int k = 0; k < g.dim; k++) {
        const int n = k == 0 ? g.nx : (k == 1 ? g.ny : g.nz);
        const bool per = !(g.walls && k == g.dim - 1);
        nb[k] = ((per ? n : n + 2) + DT - 1) / DT;
        ct[k] = (n + DT - 1) / DT;
    }
}

}  // namespace iblb
