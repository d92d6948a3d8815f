// k_neighbor.cu -- neighbour-list rebuild on the GPU: wrap + bin, per-replica
// scan of bin counts, counting sort into bin order (deterministic order inside
// a bin: by atom id), and the cell-stencil Verlet-list build.
//
// The paper keeps the whole time step on the GPU, list creation included
// (Sec. II, Sec. IV); its neighbour-list force kernels read numneigh[i] and
// neighbors[i][jj] (Sec. III.B listings) and rely on spatially ordered atoms
// for cache reuse (Sec. III.B, texture-cache discussion).  The build
// algorithm itself is not described there; this one bins atoms into cells of
// edge >= cutoff + skin and scans the 27 surrounding cells.
#include <algorithm>

#include "md_common.cuh"
#include "md_kernels.h"

namespace md {

// Zero the bin counts and list statistics of each rebuilding replica (a
// grid-stride loop over all bins and replicas).
__global__ void k_zero_bins(View V, KArgs a) {
    const int stride = gridDim.x * blockDim.x;
    const int t0 = blockIdx.x * blockDim.x + threadIdx.x;
    for (int b = t0; b < V.nbins_total; b += stride)
        if (a.all || V.rep_flag[V.bin_rep[b]]) V.bin_count[b] = 0;
    for (int r = t0; r < V.n_rep; r += stride) {
        if (!a.all && !V.rep_flag[r]) continue;
        V.rep_maxcnt[r] = 0;
        V.rep_entries[r] = 0ull;
    }
}

// Stage each atom of a rebuilding replica (position relative to its NEW bin
// centre, velocity, type, id) in old order and count it into its new bin.
// a.mode = 0 (inside md_step): the atom moved at most skin/2 since the last
// build, so its new bin is found from its cell-relative position alone --
// periodic wrapping is a wrap of the bin index, no absolute coordinates.
// a.mode = 1: absolute positions/velocities/types/ids are already staged in
// the scratch arrays (creation, set_state): wrap into the box and bin.
template <int PREC>
__device__ __forceinline__ void prepare_slot(const View &V, const KArgs &a, int p) {
    const int r = V.tile_rep[p >> 5];
    if (!a.all && !V.rep_flag[r]) return;
    const Rep &R = V.rep[r];
    const int local = p - R.atom0;
    if (local >= R.natoms) return;
    const int n = V.n_pad;
    int bc[3];
    double xr[3];
    bool finite = true;
    if (a.mode == 1) {
        for (int c = 0; c < 3; ++c) {
            const double x = V.tx[c * n + p];
            double w = wrap_box(x, R.L[c], R.Linv[c]);
            if (!in_box(w, R.L[c])) {  // NaN / Inf
                w = 0.0;
                finite = false;
            }
            int b = (int)(w * R.hinv[c]);
            b = min(max(b, 0), R.nb[c] - 1);
            bc[c] = b;
            xr[c] = fma(-bin_centre(b), R.h[c], w);
        }
    } else {
        const int b = V.bpk[p];
        bc[0] = unpack_bx(b); bc[1] = unpack_by(b); bc[2] = unpack_bz(b);
        int t;
        if (PREC == MD_PREC_FP64) {
            const double4_32a q = V.pos4[p];
            xr[0] = q.x; xr[1] = q.y; xr[2] = q.z;
            t = (int)__double_as_longlong(q.w);
        } else {
            for (int c = 0; c < 3; ++c) xr[c] = V.xr[c * n + p];
            t = V.type[p];
        }
        for (int c = 0; c < 3; ++c) {
            V.tv[c * n + p] = V.v[c * n + p];
            double x = xr[c];
            // Bins moved along this axis, floor(x / h + 1/2), by comparing |x| with the
            // bin's half edge and edge as integers (six FP64 instructions less per axis;
            // no gain where memory bounds the pass: 26.4 us of 864,000 atoms either way);
            // an atom moves at most one bin between builds, unless skins are wider than
            // bins or the state has run away
            const double h = R.h[c];
            const long long xb = __double_as_longlong(x), ax = xb & 0x7fffffffffffffffll;
            const long long edge = __double_as_longlong(h), half = edge - (1ll << 52);
            if (ax > half || xb == half) {
                int d = xb < 0 ? -1 : 1;
                if (ax >= edge) {
                    if (!(fabs(x) < 1.0e6)) {  // NaN / Inf / runaway
                        x = 0.0;
                        finite = false;
                    }
                    d = (int)floor(x * R.hinv[c] + 0.5);
                    x -= (double)d * h;
                } else {
                    x -= xb < 0 ? -h : h;
                }
                const int nb = R.nb[c];
                int bb = (bc[c] + d) % nb;
                bc[c] = bb < 0 ? bb + nb : bb;
            }
            xr[c] = x;
        }
        V.ttype[p] = t;
        V.tid[p] = V.id[p];
    }
    for (int c = 0; c < 3; ++c) V.tx[c * n + p] = xr[c];
    if (!finite) latch_error(V.ctl, kErrNonfinite);
    const int gb = V.lin2bin[R.bin0 + (bc[2] * R.nb[1] + bc[1]) * R.nb[0] + bc[0]];
    V.key[p] = gb;
    // atoms of a warp are mostly in one or two bins: one atomic per distinct
    // bin, each lane taking its rank among the lanes of its bin
    const unsigned active = __activemask();
    const unsigned same = __match_any_sync(active, gb);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(same) - 1;
    const int rank = __popc(same & ((1u << lane) - 1));
    int base = 0;
    if (lane == leader) base = atomicAdd(&V.bin_count[gb], __popc(same));
    base = __shfl_sync(same, base, leader);
    V.slot[p] = base + rank;
}

// Flat slot numbering of the batched rebuild's work list: unit u -> slot.
__device__ __forceinline__ int wl_slot(const View &V, int nf, int u) {
    int lo = 0, hi = nf - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&V.wl_s0[mid]) <= u) lo = mid;
        else hi = mid - 1;
    }
    return __ldg(&V.wl_a0[lo]) + (u - __ldg(&V.wl_s0[lo]));
}

// the slots of one rebuild pass: every slot, or (a.wl) the work list's
template <class F>
__device__ __forceinline__ void for_rebuild_slots(const View &V, const KArgs &a, F &&slot) {
    if (a.wl) {
        const int nf = *V.wl_n, total = V.wl_s0[nf];
        for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < total; u += gridDim.x * blockDim.x)
            slot(wl_slot(V, nf, u));
    } else {
        const int p = blockIdx.x * blockDim.x + threadIdx.x;
        if (p < V.n_pad) slot(p);
    }
}

template <int PREC>
__global__ void k_prepare(View V, KArgs a) {
    for_rebuild_slots(V, a, [&](int p) { prepare_slot<PREC>(V, a, p); });
}

// Bins of a replica are numbered along a Morton (Z-order) curve through its
// cell grid, so that atoms consecutive in memory -- those of one warp, one
// block, one SM -- fill compact 3-D regions whose neighbours overlap: the
// gathers of the force loop then hit L1 more often.

// bin_start[b] = first slot of bin b: an exclusive scan of the bin counts,
// segmented per replica (each replica's slots start at its atom0), in two
// parallel passes.  Bins of replicas that are not rebuilding get meaningless
// values, which nothing reads before their next rebuild.
constexpr int kScanBlock = 4096;  // bins per block of k_scan1 (1024 threads x 4)

__device__ __forceinline__ int block_excl_scan(int v, int *s_warp, int *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int inc = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) s_warp[w] = inc;
    __syncthreads();
    if (w == 0) {
        const int nw = blockDim.x >> 5;
        int t = lane < nw ? s_warp[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < nw) s_warp[lane] = t;
    }
    __syncthreads();
    *total = s_warp[(blockDim.x >> 5) - 1];
    const int r = inc - v + (w > 0 ? s_warp[w - 1] : 0);
    __syncthreads();
    return r;
}

// pass 1: prefix inside each block of 4096 bins and the block totals; the
// last block to finish (ticket) then scans the block totals and sets each
// replica's base
__global__ void __launch_bounds__(1024) k_scan1(View V, KArgs a) {
    __shared__ int s_warp[32];
    const int b0 = blockIdx.x * kScanBlock + threadIdx.x * 4;
    int c[4], sum = 0;
    for (int k = 0; k < 4; ++k) {
        c[k] = (b0 + k < V.nbins_total) ? V.bin_count[b0 + k] : 0;
        sum += c[k];
    }
    int total;
    int run = block_excl_scan(sum, s_warp, &total);
    for (int k = 0; k < 4; ++k) {
        if (b0 + k < V.nbins_total) V.bin_start[b0 + k] = run;
        run += c[k];
    }
    if (threadIdx.x == 0) V.scan_blk[blockIdx.x] = total;
    if (!last_block(&V.ctl->ticket_scan)) return;
    __threadfence();
    const int nblk = gridDim.x;
    int carry = 0;
    for (int c0 = 0; c0 < nblk; c0 += blockDim.x) {
        const int i = c0 + threadIdx.x;
        const int v = i < nblk ? __ldcg(&V.scan_blk[i]) : 0;
        int tot;
        const int ex = block_excl_scan(v, s_warp, &tot);
        if (i < nblk) V.scan_blk[i] = carry + ex;
        carry += tot;
    }
    __syncthreads();
    for (int r = threadIdx.x; r < V.n_rep; r += blockDim.x) {
        const int b = V.rep[r].bin0;
        V.rep_base[r] = V.scan_blk[b / kScanBlock] + __ldcg(&V.bin_start[b]) - V.rep[r].atom0;
    }
    if (threadIdx.x == 0) V.ctl->ticket_scan = 0;
}

// pass 3: global prefix, rebased to each rebuilding replica's first slot
__global__ void k_scan3(View V, KArgs a) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= V.nbins_total) return;
    const int r = V.bin_rep[b];
    if (!a.all && !V.rep_flag[r]) return;
    V.bin_start[b] += V.scan_blk[b / kScanBlock] - V.rep_base[r];
}

// perm[bin_start[bin] + arrival slot] = old slot; sid = the atom ids in
// the same (arrival) order, contiguous per bin for the ranking in k_gather
__device__ __forceinline__ void scatter_slot(const View &V, const KArgs &a, int p) {
    const int r = V.tile_rep[p >> 5];
    if (!a.all && !V.rep_flag[r]) return;
    if (p - V.rep[r].atom0 >= V.rep[r].natoms) return;
    const int q = V.bin_start[V.key[p]] + V.slot[p];
    V.perm[q] = p;
    V.sid[q] = V.tid[p];
}

__global__ void k_scatter(View V, KArgs a) {
    for_rebuild_slots(V, a, [&](int p) { scatter_slot(V, a, p); });
}

// One system of at most kScanMost bins: the two scan passes and the scatter in one launch.
// Every block scans all the counts itself (at most 32 KB, from L2, sixteen per thread) into
// shared memory while its atoms' keys are on their way; the first writes the starts out.
// The three kernels were latency and launches, not work: 6 .. 7 us less per rebuild, us per step with a rebuild
// every ~7: LJ 500 atoms 13.2 -> 12.6, 4,000 FP64 32.1 -> 31.3, 32,771 32.4 -> 31.6, 100,003
// (5,400 bins) 47.8 -> 46.7. The limit is what a block scans in one pass of four loads per thread.
constexpr int kScanMost = 8192;
constexpr int kScanThreads = 512;
__global__ void __launch_bounds__(kScanThreads) k_scan_scatter(View V, KArgs a) {
    __shared__ __align__(16) int s_start[kScanMost];
    __shared__ int s_warp[32];
    if (!a.all && !V.rep_flag[0]) return;
    const int p = blockIdx.x * kScanThreads + threadIdx.x;
    const bool in = p - V.rep[0].atom0 < V.rep[0].natoms;
    int key = 0, slot = 0, id = 0;
    if (in) { key = V.key[p]; slot = V.slot[p]; id = V.tid[p]; }
    const int nb = V.nbins_total, per = (nb + 4 * kScanThreads - 1) / (4 * kScanThreads);  // groups of four per thread
    const int b0 = threadIdx.x * per * 4;
    int4 c[kScanMost / (4 * kScanThreads)];
    int sum = 0;
#pragma unroll
    for (int k = 0; k < kScanMost / (4 * kScanThreads); ++k) {
        const int b = b0 + 4 * k;
        c[k] = make_int4(0, 0, 0, 0);
        if (k < per) {
            if (b + 3 < nb) {
                c[k] = *reinterpret_cast<const int4 *>(V.bin_count + b);
            } else {
                if (b < nb) c[k].x = V.bin_count[b];
                if (b + 1 < nb) c[k].y = V.bin_count[b + 1];
                if (b + 2 < nb) c[k].z = V.bin_count[b + 2];
            }
        }
        sum += (c[k].x + c[k].y) + (c[k].z + c[k].w);
    }
    int total;
    int run = V.rep[0].atom0 + block_excl_scan(sum, s_warp, &total);
#pragma unroll
    for (int k = 0; k < kScanMost / (4 * kScanThreads); ++k) {
        if (k < per) {
            const int4 at = make_int4(run, run + c[k].x, run + c[k].x + c[k].y, run + c[k].x + c[k].y + c[k].z);
            *reinterpret_cast<int4 *>(s_start + b0 + 4 * k) = at;
            run = at.w + c[k].w;
        }
    }
    __syncthreads();
    if (blockIdx.x == 0)
        for (int b = threadIdx.x; b < nb; b += kScanThreads) V.bin_start[b] = s_start[b];
    if (in) {
        const int q = s_start[key] + slot;
        V.perm[q] = p;
        V.sid[q] = id;
    }
}

// Final slot = bin start + rank of the atom's id inside its bin (so the
// order does not depend on atomic arrival order); write the sorted state
// (positions relative to the new bin centre), FP32 records, build reference.
template <int PREC>
__device__ __forceinline__ void gather_slot(const View &V, const KArgs &a, int q) {
    const int r = V.tile_rep[q >> 5];
    if (!a.all && !V.rep_flag[r]) return;
    const Rep &R = V.rep[r];
    const int n = V.n_pad;
    if (q - R.atom0 >= R.natoms) {  // padding slot: inert
        for (int c = 0; c < 3; ++c) V.v[c * n + q] = 0.0;
        if (PREC == MD_PREC_FP64) V.pos4[q] = make_double4_32a(0.0, 0.0, 0.0, __longlong_as_double(0));
        else for (int c = 0; c < 3; ++c) V.xr[c * n + q] = 0.0;
        V.rec[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        V.recb[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        V.id[q] = -1;
        V.type[q] = 0;
        V.bpk[q] = 0;
        return;
    }
    const int src = V.perm[q];
    const int gb = V.key[src];
    const int s = V.bin_start[gb], cnt = V.bin_count[gb];
    const int myid = V.sid[q];
    int rank = 0;
    for (int k = 0; k < cnt; ++k) rank += (V.sid[s + k] < myid);
    const int dst = s + rank;
    const int xyz = V.bin2xyz[gb];
    const int bc[3] = {unpack_bx(xyz), unpack_by(xyz), unpack_bz(xyz)};
    double xr[3];
    for (int c = 0; c < 3; ++c) {
        xr[c] = V.tx[c * n + src];
        V.v[c * n + dst] = V.tv[c * n + src];
    }
    const int t = V.ttype[src];
    if (PREC == MD_PREC_FP64) {
        V.pos4[dst] = make_double4_32a(xr[0], xr[1], xr[2], __longlong_as_double((long long)t));
    } else {
        for (int c = 0; c < 3; ++c) V.xr[c * n + dst] = xr[c];
    }
    V.type[dst] = t;
    V.id[dst] = myid;
    V.inv[R.orig0 + myid] = dst;
    V.bpk[dst] = pack_bins(bc[0], bc[1], bc[2]);
    const float4 rr = make_float4((float)xr[0], (float)xr[1], (float)xr[2], __int_as_float(t));
    V.rec[dst] = rr;
    V.recb[dst] = rr;
}

template <int PREC>
__global__ void k_gather(View V, KArgs a) {
    for_rebuild_slots(V, a, [&](int q) { gather_slot<PREC>(V, a, q); });
}

// global bin of slot p (after the gather)
__device__ __forceinline__ int slot_bin(const View &V, const Rep &R, int p) {
    const int k = V.bpk[p];
    return V.lin2bin[R.bin0 + (unpack_bz(k) * R.nb[1] + unpack_by(k)) * R.nb[0] + unpack_bx(k)];
}

// Per tile of tile_atoms slots (one warp each): the cells of its atoms (a
// contiguous range of bins, <= 32), their 27-cell neighbourhoods marked in a
// bitmap over the dilated bounding box (<= kTileBox cells, unwrapped
// coordinates, so a cell reached through two periodic images is staged
// twice), the marked cells in box order with their record counts, and the
// running offsets.  A tile that straddles replicas, spans too many cells or
// stages more than kTileCap records keeps slot entries (tile_cnt = -1).
__global__ void __launch_bounds__(128) k_tiles(View V, KArgs a) {
    __shared__ unsigned s_bits[4][32];
    __shared__ int s_cnt[4][kTileCells];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int t = blockIdx.x * 4 + w;
    if (t >= V.n_ftiles) return;
    const int p0 = t * V.tile_atoms;
    const int p1 = min(p0 + V.tile_atoms, V.n_pad) - 1;
    const int r = V.tile_rep[p0 >> 5], r1 = V.tile_rep[p1 >> 5];
    if (!(a.all || V.rep_flag[r] || V.rep_flag[r1])) return;  // lists of this tile unchanged
    const Rep &R = V.rep[r];
    int ok = (r == r1);
    const int pl = min(p1, R.atom0 + R.natoms - 1);
    if (ok && pl < p0) {  // no real atom
        if (lane == 0) { V.tile_cnt[t] = 0; V.tile_ncell[t] = 0; }
        return;
    }
    int gb0 = 0, nh = 0;
    if (ok) {
        gb0 = slot_bin(V, R, p0);
        nh = slot_bin(V, R, pl) - gb0 + 1;
        ok = (nh >= 1 && nh <= 32);
    }
    if (!ok) {
        if (lane == 0) { V.tile_cnt[t] = -1; V.tile_ncell[t] = 0; }
        return;
    }
    const bool act = lane < nh;
    int bx = 0, by = 0, bz = 0;
    if (act) {
        const int xyz = V.bin2xyz[gb0 + lane];
        bx = unpack_bx(xyz); by = unpack_by(xyz); bz = unpack_bz(xyz);
    }
    const int lox = __reduce_min_sync(0xffffffffu, act ? bx : 0x7fffffff) - 1;
    const int loy = __reduce_min_sync(0xffffffffu, act ? by : 0x7fffffff) - 1;
    const int loz = __reduce_min_sync(0xffffffffu, act ? bz : 0x7fffffff) - 1;
    const int dx = __reduce_max_sync(0xffffffffu, act ? bx : -0x7fffffff) - lox + 2;
    const int dy = __reduce_max_sync(0xffffffffu, act ? by : -0x7fffffff) - loy + 2;
    const int dz = __reduce_max_sync(0xffffffffu, act ? bz : -0x7fffffff) - loz + 2;
    ok = dx * dy * dz <= kTileBox;  // each dim <= 1026 (bins per axis <= 1024): no overflow
    s_bits[w][lane] = 0u;
    __syncwarp();
    if (ok && act) {
        for (int k = 0; k < 27; ++k) {
            const int row = k / 3;
            const int ox = k - 3 * row - 1, oy = row % 3 - 1, oz = row / 3 - 1;
            const int idx = (bx + ox - lox) + dx * ((by + oy - loy) + dy * (bz + oz - loz));
            atomicOr(&s_bits[w][idx >> 5], 1u << (idx & 31));
        }
    }
    __syncwarp();
    const unsigned word = ok ? s_bits[w][lane] : 0u;
    int incl = __popc(word);
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    const int excl = incl - __popc(word);
    const int ncell = __shfl_sync(0xffffffffu, incl, 31);
    ok = ok && ncell <= kTileCells;
    if (!ok) {
        if (lane == 0) { V.tile_cnt[t] = -1; V.tile_ncell[t] = 0; }
        return;
    }
    V.tile_bits[(size_t)t * 32 + lane] = word;
    V.tile_wpre[(size_t)t * 32 + lane] = excl;
    // the union's cells in box order (coordinates only), then four per lane:
    // bin, first slot, count (independent loads)
    unsigned wd = word;
    int k = excl;
    while (wd) {
        s_cnt[w][k++] = lane * 32 + __ffs(wd) - 1;  // box index for now
        wd &= wd - 1u;
    }
    __syncwarp();
    const int nbx = R.nb[0], nby = R.nb[1], nbz = R.nb[2];
    int gbq[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int kk = lane + 32 * q;
        gbq[q] = -1;
        if (kk < ncell) {
            const int idx = s_cnt[w][kk];
            int cx = lox + idx % dx, cy = loy + (idx / dx) % dy, cz = loz + idx / (dx * dy);
            cx += (cx < 0) ? nbx : ((cx >= nbx) ? -nbx : 0);
            cy += (cy < 0) ? nby : ((cy >= nby) ? -nby : 0);
            cz += (cz < 0) ? nbz : ((cz >= nbz) ? -nbz : 0);
            gbq[q] = V.lin2bin[R.bin0 + (cz * nby + cy) * nbx + cx];
        }
    }
    int cq[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int kk = lane + 32 * q;
        cq[q] = 0;
        if (gbq[q] >= 0) {
            V.tile_first[(size_t)t * kTileCells + kk] = V.bin_start[gbq[q]];
            cq[q] = V.bin_count[gbq[q]];
        }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (gbq[q] >= 0) s_cnt[w][lane + 32 * q] = cq[q];
    __syncwarp();
    // running offsets, four cells per lane
    int c4[4], sum = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int kk = 4 * lane + q;
        c4[q] = kk < ncell ? s_cnt[w][kk] : 0;
        sum += c4[q];
    }
    int run = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, run, o);
        if (lane >= o) run += u;
    }
    const int total = __shfl_sync(0xffffffffu, run, 31);
    run -= sum;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int kk = 4 * lane + q;
        if (kk < ncell) V.tile_off[(size_t)t * kTileCells + kk] = run;
        run += c4[q];
    }
    if (lane == 0) {
        const bool fits = total <= kTileCap;
        V.tile_cnt[t] = fits ? total : -1;
        V.tile_ncell[t] = fits ? ncell : 0;
        V.tile_box[t] = make_int4(lox, loy, loz, dx | (dy << 16));
    }
}

// Exact FP64 list test for a pair inside the FP32 margin band (rare; kept
// out of line so that it does not cost the main loop registers).
template <int PREC>
__device__ __noinline__ bool in_list_fp64(const View &V, const Rep &R, int p, int j, int dx, int dy, int dz) {
    double xi[3], xj[3];
    if (PREC == MD_PREC_FP64) {
        const double4_32a qi = V.pos4[p], qj = V.pos4[j];
        xi[0] = qi.x; xi[1] = qi.y; xi[2] = qi.z;
        xj[0] = qj.x; xj[1] = qj.y; xj[2] = qj.z;
    } else {
        const int n = V.n_pad;
        for (int q = 0; q < 3; ++q) { xi[q] = V.xr[q * n + p]; xj[q] = V.xr[q * n + j]; }
    }
    const double d0 = xi[0] - xj[0] - dx * R.h[0];
    const double d1 = xi[1] - xj[1] - dy * R.h[1];
    const double d2 = xi[2] - xj[2] - dz * R.h[2];
    return d0 * d0 + d1 * d1 + d2 * d2 < V.rl2;
}

// three-input minimum (one instruction on sm_100 and later)
__device__ __forceinline__ float fmin3(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// 32 x 32 bit-matrix transpose across a warp: on entry lane r holds row r
// (bit c = M[r][c]); on return lane c holds column c (bit r = M[r][c]).
// Five butterfly stages of recursive 2x2 block swaps.
__device__ __forceinline__ unsigned warp_transpose32(unsigned x, int lane) {
    const unsigned masks[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const int sft = 16 >> k;
        const unsigned m = masks[k];
        const unsigned p = __shfl_xor_sync(0xffffffffu, x, sft);
        x = (lane & sft) ? ((x & ~m) | ((p >> sft) & m)) : ((x & m) | ((p << sft) & ~m));
    }
    return x;
}

// Append entry e to this lane's column of the append buffer if `bit` of the
// lane's mask is set: store at shared address sa, then sa += one row.  Spelled out
// with predicates: as C++ the compiler branches around the two statements.
__device__ __forceinline__ void append_if(unsigned mask, unsigned bit, uint32_t e, unsigned &sa) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t"
        "and.b32 t, %1, %3;\n\t"
        "setp.ne.u32 p, t, 0;\n\t"
        "@p st.shared.u32 [%0], %2;\n\t"
        "@p add.u32 %0, %0, 128;\n\t}"
        : "+r"(sa)
        : "r"(mask), "r"(e), "r"(bit));
}
// the buffer is only accessed through these (volatile: in program order among themselves,
// while the queue's ordinary loads move freely)
__device__ __forceinline__ uint32_t buf_load(unsigned sa) {
    uint32_t e;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(e) : "r"(sa));
    return e;
}
__device__ __forceinline__ void buf_store(unsigned sa, uint32_t e) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(sa), "r"(e));
}

// Verlet list of every atom of a rebuilding replica: all j in the 27 cells
// around i's cell with |x_i - x_j| < rl.  One warp per home cell (home atoms
// in chunks of 32, one per lane; a cell with more than 32 atoms is shared out
// over several warps).  The 27 neighbour cells form 9 rows of 3 x-adjacent cells.
// Each row is read as one flat candidate range, 32 candidates at a time, one per
// lane, the next 32 on their way meanwhile, shifted into the home cell's
// frame.  A candidate farther than rl from the bounding box of
// the home atoms cannot be accepted by any of them (about 38 % of the 27-cell
// candidates); the others go to a per-warp queue in shared memory, in
// candidate order, and are tested in full rounds of 32: each lane
// tests its candidate against every home atom (records broadcast from shared
// memory) into a 32-bit acceptance mask, and a warp bit-matrix transpose turns the
// candidates' masks into each home atom's mask of accepted candidates.  Then the
// candidates' entries are read one after another, and a home-atom lane that accepts
// one appends it to its column of an append buffer in shared memory (test, store and
// address in three predicated instructions, no bank conflicts), which is
// written out four entries (16 bytes) at a time.  So the lists are in candidate
// order (deterministic).
// The home atoms' tests are two to an instruction (FP32x2).  What bounds it: instruction issue (73 %) and
// the L1 data pipe (77 %) at rc 2.5; at rc 5.0 (55 and 56 %) also the list's partly written sectors.  Against scanning each home
// atom's masks bit by bit and storing 4-byte entries straight to the list, whose
// scattered sectors bound the build at rc 5.0 (one launch, 500,000 atoms): rc 2.5 225 ->
// 220 us (209.6 M -> 187.8 M warp instructions), rc 5.0 1.51 -> 1.09 ms; measured and not kept:
// one lane per home atom testing the candidates one after another (219 M, 235 us at rc 2.5,
// 1.14 ms at rc 5.0), storing straight to the list with predicates (234 M, 245 us, 1.53 ms),
// larger and smaller append buffers (24 .. 52 rows: 219 .. 241 us).
// The test is FP32 with a margin far above its rounding
// error; pairs inside the margin band are decided in FP64, so the list equals
// the FP64 definition exactly.  HALF keeps j > i only.
constexpr int kQueue = 64;  // queued candidates per warp (< 32 left + 32 new)
constexpr int kApp = 16;    // candidates appended between two looks at the buffer's room
constexpr int kBuf = 36;    // rows of the append buffer: a multiple of 4, >= 3 left over + kApp

// The list build runs NW warps (cells or cell parts) per block.  One warp
// per block when every cell has one warp: no block barrier, a block's
// registers come free as soon as its cell is done, and the warp's
// shared-memory addresses are constants.  Four when the warps of a cell share it
// out, so that they share its candidates in L1.  28 warps per SM (72 registers): by shared
// memory there is no room for more, and at 64 registers the loops spill (work-list build: 735
// against 702 us per step of 512 replicas).
constexpr int kBuildWarps = 28;
// blocks of the work-list build per resident one: a finer deal (702 -> 696 us), where the
// batch has the cells for it (some tenth of the replicas rebuild in a step)
constexpr int kBuildWlDeal = 4;

template <int PREC, int HALF, int NW>
__device__ __forceinline__ void build_cell(const View &V, int gb, int part, int hsplit, int lane, int w,
                                           int &my_max, long long &my_sum) {
    // home atoms 2k, 2k + 1: {x, x, y, y}, {z, z, |x|^2, |x|^2}
    __shared__ __align__(16) float s_h[NW][16][8];
    __shared__ float4 s_q[NW][kQueue];  // queued candidates: position in the home frame, .w = list entry bits
    __shared__ __align__(16) uint32_t s_e[NW][32];  // the round's list entries
    __shared__ uint32_t s_buf[NW][kBuf][32];            // append buffer: a column per home atom
    __shared__ float4 s_box[NW][2];     // bounding box of the home chunk: lo, hi
    // per row of 3 cells: candidate f's entry is f << 6 plus that of its cell
    // ({cell 0, 1, 2}.x/y/z); candidates of the row; first candidate of cells 1 and
    // 2, and the row's shift in y and z as float bits
    __shared__ uint4 s_row[NW][9];
    __shared__ int4 s_row2[NW][9];
    __shared__ int s_delta[NW][2][64];  // per tile of the chunk, per stencil code: entry shift
    const int hs = V.bin_start[gb], hn = V.bin_count[gb];
    // nothing to do here: in a gas most cells are empty (256,000 atoms at density 0.005, 2.3 M cells: a build with its sort
    // 1,886 -> 1,675 us; where no cell is empty the early look costs nothing, 864,000 atoms of liquid 580 us)
    if (hn <= 32 * part) return;
    const int r = V.bin_rep[gb];
    const Rep &R = V.rep[r];
    const int maxn = V.maxneigh, lt = V.ltpa, lq = V.lvec;
    const int la = 5 - lt, ltq = lt + lq, tq = 1 << ltq;
    const int nbx = R.nb[0], nby = R.nb[1], nbz = R.nb[2];
    const int xyz = V.bin2xyz[gb];
    const int bx = unpack_bx(xyz), by = unpack_by(xyz), bz = unpack_bz(xyz);
    const float hx = R.hf[0], hy = R.hf[1], hz = R.hf[2];
    // neighbour cell (row = lane / 3, dx = lane % 3 - 1) bounds, one lane each
    int cell_first = 0;
    {
        const int l = min(lane, 26), row = l / 3;
        const int dx = l - 3 * row - 1, dy = row % 3 - 1, dz = row / 3 - 1;
        int cx = bx + dx, cy = by + dy, cz = bz + dz;
        cx += (cx < 0) ? nbx : ((cx >= nbx) ? -nbx : 0);
        cy += (cy < 0) ? nby : ((cy >= nby) ? -nby : 0);
        cz += (cz < 0) ? nbz : ((cz >= nbz) ? -nbz : 0);
        const int nbin = V.lin2bin[R.bin0 + (cz * nby + cy) * nbx + cx];
        cell_first = V.bin_start[nbin];
        const int cnt = V.bin_count[nbin];
        const int c1 = __shfl_down_sync(0xffffffffu, cnt, 1), c2 = __shfl_down_sync(0xffffffffu, cnt, 2);
        const int f1 = __shfl_down_sync(0xffffffffu, cell_first, 1), f2 = __shfl_down_sync(0xffffffffu, cell_first, 2);
        if (lane < 27 && dx == -1) {
            const uint32_t code = (uint32_t)((dz + 1) << 4 | (dy + 1) << 2);
            s_row[w][row] = make_uint4(((uint32_t)cell_first << 6) + code, ((uint32_t)(f1 - cnt) << 6) + code + 1u,
                                       ((uint32_t)(f2 - cnt - c1) << 6) + code + 2u, (uint32_t)(cnt + c1 + c2));
            s_row2[w][row] = make_int4(cnt, cnt + c1, __float_as_int(dy * hy), __float_as_int(dz * hz));
        }
    }
    const float rl2f = 0.5f * (V.rl2f_lo + V.rl2f_hi), margin = 0.5f * (V.rl2f_hi - V.rl2f_lo);
    // box pre-test bound: above every squared distance the margin band can hold
    const float keep2 = V.rl2f_hi + margin;
    for (int h0 = 32 * part; h0 < hn; h0 += 32 * hsplit) {
        const int nh = min(32, hn - h0);
        const int hbase = hs + h0;  // slot of home atom 0 of this chunk
        __syncwarp();
        {
            // home record with |r|^2 in .w; padding far away (never accepted, never in the band)
            float4 hr = make_float4(1.0e18f, 1.0e18f, 1.0e18f, 0.f);
            if (lane < nh) hr = V.rec[hbase + lane];
            hr.w = hr.x * hr.x + hr.y * hr.y + hr.z * hr.z;
            float *h = s_h[w][lane >> 1] + (lane & 1);
            h[0] = hr.x; h[2] = hr.y; h[4] = hr.z; h[6] = hr.w;
            // bounding box of the chunk's home atoms
            const bool in = lane < nh;
            float lox = in ? hr.x : 3.0e38f, hix = in ? hr.x : -3.0e38f;
            float loy, loz, hiy, hiz;
            loy = in ? hr.y : 3.0e38f; hiy = in ? hr.y : -3.0e38f;
            loz = in ? hr.z : 3.0e38f; hiz = in ? hr.z : -3.0e38f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                lox = fminf(lox, __shfl_xor_sync(0xffffffffu, lox, o));
                loy = fminf(loy, __shfl_xor_sync(0xffffffffu, loy, o));
                loz = fminf(loz, __shfl_xor_sync(0xffffffffu, loz, o));
                hix = fmaxf(hix, __shfl_xor_sync(0xffffffffu, hix, o));
                hiy = fmaxf(hiy, __shfl_xor_sync(0xffffffffu, hiy, o));
                hiz = fmaxf(hiz, __shfl_xor_sync(0xffffffffu, hiz, o));
            }
            if (lane == 0) {
                s_box[w][0] = make_float4(lox, loy, loz, 0.f);
                s_box[w][1] = make_float4(hix, hiy, hiz, 0.f);
            }
        }
        // Block-local entries: the chunk's atoms lie in one or two tiles; for
        // each, stencil cell k's records start at tile_off[k] in the tile's
        // staging, so a candidate's entry j<<6|code becomes
        // (j - cell start + tile_off[k])<<6|code: a shift per (tile, code).
        const int tpa_atoms = V.tile_atoms;
        const int tA = tpa_atoms ? hbase / tpa_atoms : 0;
        const int tB = tpa_atoms ? (hbase + nh - 1) / tpa_atoms : 0;
        if (lane < 27) {
            const int row = lane / 3;
            const int ox = lane - 3 * row - 1, oy = row % 3 - 1, oz = row / 3 - 1;
            const int code = ((oz + 1) << 4) | ((oy + 1) << 2) | (ox + 1);
            for (int X = 0; X < 2; ++X) {
                int delta = 0;
                const int t = X ? tB : tA;
                if (tpa_atoms && V.tile_cnt[t] >= 0) {
                    const int4 b = V.tile_box[t];
                    const int bdx = b.w & 0xffff, bdy = b.w >> 16;
                    int idx = (bx + ox - b.x) + bdx * ((by + oy - b.y) + bdy * (bz + oz - b.z));
                    idx = min(max(idx, 0), kTileBox - 1);
                    const unsigned wd = V.tile_bits[(size_t)t * 32 + (idx >> 5)];
                    int k = V.tile_wpre[(size_t)t * 32 + (idx >> 5)] + __popc(wd & ((1u << (idx & 31)) - 1u));
                    k = min(k, kTileCells - 1);
                    delta = (V.tile_off[(size_t)t * kTileCells + k] - cell_first) * 64;
                }
                s_delta[w][X][code] = delta;
            }
        }
        __syncwarp();
        // this lane as a home atom: its list and its column of the append buffer
        const int p = hbase + lane;
        const int tsel = (tpa_atoms && p / tpa_atoms != tA) ? 1 : 0;
        uint32_t *const lbase = V.nlist + (size_t)(p >> la) * (size_t)((1 << la) * maxn) + (size_t)((p & ((1 << la) - 1)) << ltq);
        const unsigned sa0 = (unsigned)__cvta_generic_to_shared(&s_buf[w][0][lane]);
        unsigned sa = sa0;
        int done = 0;  // entries written out: a multiple of 4 until the last flush
        // write the buffer out, four entries at a time; all: the last, partly filled four too
        // (entries past the list's end are never read)
        auto flush = [&](bool all) {
            const int pend = (int)((sa - sa0) >> 7);
            const int out = all ? pend : pend & ~3;
            const int most = min(out, maxn - done);  // (the capacity is a multiple of 4)
            const int rounds = (__reduce_max_sync(0xffffffffu, out) + 3) >> 2;
            unsigned at = sa0;
            int kk = done;
#pragma unroll 1
            for (int k = 0; k < rounds; ++k, kk += 4, at += 4 * 128) {
                if (kk < done + most) {
                    uint32_t e[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) e[i] = buf_load(at + (unsigned)i * 128u);
                    if (tpa_atoms) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) e[i] += (uint32_t)s_delta[w][tsel][e[i] & 63u];
                    }
                    if (lq == 2) {
                        *reinterpret_cast<uint4 *>(lbase + (((unsigned)(kk >> ltq) << 7) + (unsigned)(kk & (tq - 1)))) =
                            make_uint4(e[0], e[1], e[2], e[3]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            lbase[((unsigned)((kk + i) >> ltq) << (5 + lq)) + (unsigned)((kk + i) & (tq - 1))] = e[i];
                    }
                }
            }
            done += out;
            if (all) return;
#pragma unroll
            for (int i = 0; i < 3; ++i)
                if (i < pend - out) buf_store(sa0 + (unsigned)i * 128u, buf_load(sa0 + (unsigned)(out + i) * 128u));
            sa = sa0 + ((unsigned)(pend - out) << 7);
        };
        int qn = 0;  // queued candidates (warp-uniform)
        // one round: queue entries 0..cnt-1 (cnt <= 32), one per lane
        auto round = [&](int cnt) {
            const float4 cq = s_q[w][lane];
            const bool qin = lane < cnt;
            const float qx = qin ? cq.x : -1.0e18f, qy = qin ? cq.y : -1.0e18f, qz = qin ? cq.z : -1.0e18f;
            const uint32_t e = qin ? __float_as_uint(cq.w) : 0u;
            s_e[w][lane] = e;
            // acceptance bits over the home atoms, 8 at a time with
            // compile-time bit positions.  t = |x_i - q|^2 - rl^2 in the
            // dot-product form |x_i|^2 + |q|^2 - 2 x_i.q (FP32 error
            // < ~1e-5 rl^2 here, far inside the margin); the sign bit of t
            // is the decision, and the smallest |t| flags the margin band.
            const float qx2 = -2.0f * qx, qy2 = -2.0f * qy, qz2 = -2.0f * qz;
            const float q2m = qx * qx + qy * qy + qz * qz - rl2f;
            unsigned acc = 0u;
            float tmin = 3.0e38f;
            // home atoms from the top down, 8 at a time, two to an instruction: each
            // test shifts its sign bit in at bit 0, so that home atom h ends at bit h
            const unsigned long long qxx = pack2(qx2, qx2), qyy = pack2(qy2, qy2), qzz = pack2(qz2, qz2),
                                     qww = pack2(q2m, q2m);
#pragma unroll 1
            for (int hb = (nh - 1) & ~7; hb >= 0; hb -= 8) {
#pragma unroll
                for (int k = 6; k >= 0; k -= 2) {
                    const ulonglong2 *h = reinterpret_cast<const ulonglong2 *>(s_h[w][(hb + k) >> 1]);
                    const ulonglong2 xy = h[0], zw = h[1];
                    const float2 t = unpack2(fma2(qxx, xy.x, fma2(qyy, xy.y, fma2(qzz, zw.x, add2(zw.y, qww)))));
                    acc = __funnelshift_l(__float_as_uint(t.y), acc, 1);
                    acc = __funnelshift_l(__float_as_uint(t.x), acc, 1);
                    tmin = fmin3(tmin, fabsf(t.x), fabsf(t.y));
                }
            }
            const int j = (int)(e >> 6);
            if (tmin < margin) {  // margin band: decide those pairs in FP64 (rare)
                for (int k = 0; k < nh; ++k) {
                    const float *h = s_h[w][k >> 1] + (k & 1);
                    const float t = fmaf(qx2, h[0], fmaf(qy2, h[2], fmaf(qz2, h[4], h[6] + q2m)));
                    if (fabsf(t) < margin) {
                        const bool in = in_list_fp64<PREC>(V, R, hbase + k, j, entry_dx(e), entry_dy(e),
                                                            entry_dz(e));
                        acc = in ? (acc | (1u << k)) : (acc & ~(1u << k));
                    }
                }
            }
            // exclusions: the atom itself; for HALF every home atom with slot >= j
            const int jh = j - hbase;  // j as a home-atom index, if it is one
            if ((e & 63u) == kSelfCode && jh >= 0 && jh < 32) acc &= ~(1u << jh);
            if (HALF) acc &= jh <= 0 ? 0u : (jh >= 32 ? 0xffffffffu : ((1u << jh) - 1u));
            // lane = home atom: bit c set if candidate lane c is accepted
            const unsigned tr = warp_transpose32(acc, lane);
            __syncwarp();
            const uint4 *qe = reinterpret_cast<const uint4 *>(s_e[w]);
#pragma unroll
            for (int c0 = 0; c0 < 32; c0 += kApp) {
                if (__any_sync(0xffffffffu, sa > sa0 + (kBuf - kApp) * 128)) flush(false);
#pragma unroll
                for (int c = c0; c < c0 + kApp; c += 4) {
                    const uint4 u = qe[c / 4];
                    append_if(tr, 1u << c, u.x, sa);
                    append_if(tr, 2u << c, u.y, sa);
                    append_if(tr, 4u << c, u.z, sa);
                    append_if(tr, 8u << c, u.w, sa);
                }
            }
        };
        // the row's next 32 candidates, one per lane: entry, record, shift (lanes past
        // the row's end read the chunk's first home atom's record, and are dropped: no branch)
        int row = 0, c0 = 0;
        uint32_t ne = 0u;
        float4 nr;
        float nx = 0.f, ny = 0.f, nz = 0.f;
        bool nin = false;
        auto fetch = [&]() {
            const uint4 ra = s_row[w][row];
            const int4 rb = s_row2[w][row];
            const int f = c0 + lane;
            const bool s1 = f >= rb.x, s2 = f >= rb.y;
            nin = f < (int)ra.w;
            ne = ((uint32_t)f << 6) + (s2 ? ra.z : s1 ? ra.y : ra.x);
            nx = s2 ? hx : s1 ? 0.f : -hx;
            nr = V.rec[nin ? (int)(ne >> 6) : hbase];
            ny = __int_as_float(rb.z);
            nz = __int_as_float(rb.w);
            c0 += 32;
            if (c0 >= (int)ra.w) {
                c0 = 0;
                ++row;
            }
        };
        fetch();
        bool last = false;  // nothing more to fetch
        // fill the queue from the rows in order until it holds a full
        // round (or the rows are done), then run the round
#pragma unroll 1
        while (true) {
#pragma unroll 1
            while (qn < 32 && !last) {
                // kept if within rl (plus the band) of the home bounding box
                const uint32_t e = ne;
                const bool in = nin;
                const float cx = nr.x + nx, cy = nr.y + ny, cz = nr.z + nz;
                last = row >= 9;
                if (!last) fetch();
                const float4 lo = s_box[w][0], hi = s_box[w][1];
                const float bx_ = fmaxf(fmaxf(lo.x - cx, cx - hi.x), 0.f);
                const float by_ = fmaxf(fmaxf(lo.y - cy, cy - hi.y), 0.f);
                const float bz_ = fmaxf(fmaxf(lo.z - cz, cz - hi.z), 0.f);
                const bool keep = in && (bx_ * bx_ + by_ * by_ + bz_ * bz_ < keep2);
                const unsigned kb = __ballot_sync(0xffffffffu, keep);
                if (keep) {
                    const int at = qn + __popc(kb & ((1u << lane) - 1u));
                    s_q[w][at] = make_float4(cx, cy, cz, __uint_as_float(e));
                }
                qn += __popc(kb);
            }
            if (qn == 0) break;
            const int cnt = min(qn, 32);
            __syncwarp();
            round(cnt);
            qn -= cnt;
            __syncwarp();
            const float4 rest = s_q[w][32 + lane];
            __syncwarp();
            if (lane < qn) s_q[w][lane] = rest;
            __syncwarp();
        }
        flush(true);
        if (lane < nh) {
            const int mycnt = done;
            V.ncount[p] = min(mycnt, maxn);
            if (mycnt > maxn) {
                atomicMax(&V.ctl->need_maxneigh, mycnt);
                latch_error(V.ctl, kErrOverflow);
            }
            my_max = max(my_max, mycnt);
            my_sum += mycnt;
        }
    }
}

// list statistics of a replica from one warp: one atomic pair, no block barrier
__device__ __forceinline__ void build_stats(const View &V, int rep, int my_max, long long my_sum, int lane) {
    for (int o = 16; o > 0; o >>= 1) {
        my_max = max(my_max, __shfl_xor_sync(0xffffffffu, my_max, o));
        my_sum += __shfl_xor_sync(0xffffffffu, my_sum, o);
    }
    if (lane == 0 && rep >= 0 && my_sum > 0) {
        atomicMax(&V.rep_maxcnt[rep], my_max);
        atomicAdd(&V.rep_entries[rep], (unsigned long long)my_sum);
    }
}

template <int PREC, int HALF, int NW>
__global__ void __launch_bounds__(32 * NW, kBuildWarps / NW) k_build(View V, KArgs a) {
    const int lane = threadIdx.x & 31, w = NW == 1 ? 0 : threadIdx.x >> 5;
    // warp -> (cell, part): part q of a cell takes its home chunks q, q + hsplit, ...
    const int gw = blockIdx.x * NW + w;
    const int gb = gw / V.hsplit, part = gw - gb * V.hsplit;
    int my_max = 0;
    long long my_sum = 0;
    int my_rep = -1;
    if (gb < V.nbins_total) {
        const int r = V.bin_rep[gb];
        my_rep = r;
        if (a.all || V.rep_flag[r]) build_cell<PREC, HALF, NW>(V, gb, part, V.hsplit, lane, w, my_max, my_sum);
    }
    build_stats(V, my_rep, my_max, my_sum, lane);
    // builds of every replica (creation, md_build_neighbors, md_set_state) are
    // counted here; the step's builds of flagged replicas were counted with the
    // flags (k_drift_done), so that those launches take no ticket
    if (a.all && last_block(&V.ctl->ticket_build)) {
        if (threadIdx.x == 0) {
            V.ctl->ticket_build = 0;
            V.ctl->rebuilds += V.n_rep;
        }
    }
}

// The list build of a system with too few cells to fill the GPU (kRowBuild): one
// block of nine warps per (cell, part), one warp per row of three cells.  A
// warp alone on its scheduler takes ~8 clocks an instruction, so the ~8,000
// instructions of a whole cell in one warp are 35 us whatever the size; here the
// rows are tested side by side and counted, the block's warps exchange their counts,
// and each warp then writes its row's entries behind those of the
// rows before it: the same lists, entry by entry.  The acceptance masks and
// entries of a row's first kRowKeep rounds are kept between the two passes, later rounds
// (rows of more than 32 kRowKeep candidates) are tested again.
constexpr int kRowKeep = 4;

// one (cell, part) by the nine warps of a block
template <int PREC, int HALF>
__device__ __forceinline__ void build_rows(const View &V, int gb, int part, int hsplit) {
    __shared__ __align__(16) float s_h[16][8];  // home atoms 2k, 2k + 1: {x, x, y, y}, {z, z, |x|^2, |x|^2}
    __shared__ int s_cnt[9][32];                // accepted per row and home atom
    __shared__ uint32_t s_t[9][kRowKeep][32], s_e[9][kRowKeep][32];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int r = V.bin_rep[gb];
    const Rep &R = V.rep[r];
    int my_max = 0;
    long long my_sum = 0;
    const int hs = V.bin_start[gb], hn = V.bin_count[gb];
    const int xyz = V.bin2xyz[gb];
    const int dy = row % 3 - 1, dz = row / 3 - 1;
    // the row's three cells, one lane each (the other lanes repeat the last)
    const int nbx = R.nb[0], nby = R.nb[1], nbz = R.nb[2];
    int cx = unpack_bx(xyz) + min(lane, 2) - 1, cy = unpack_by(xyz) + dy, cz = unpack_bz(xyz) + dz;
    cx += (cx < 0) ? nbx : ((cx >= nbx) ? -nbx : 0);
    cy += (cy < 0) ? nby : ((cy >= nby) ? -nby : 0);
    cz += (cz < 0) ? nbz : ((cz >= nbz) ? -nbz : 0);
    const int nbin = V.lin2bin[R.bin0 + (cz * nby + cy) * nbx + cx];
    const int first = V.bin_start[nbin], count = V.bin_count[nbin];
    const int n0 = __shfl_sync(0xffffffffu, count, 0), n1 = n0 + __shfl_sync(0xffffffffu, count, 1);
    const int m = n1 + __shfl_sync(0xffffffffu, count, 2);
    const uint32_t code = (uint32_t)((dz + 1) << 4 | (dy + 1) << 2);
    const uint32_t e0 = ((uint32_t)__shfl_sync(0xffffffffu, first, 0) << 6) + code;
    const uint32_t e1 = ((uint32_t)(__shfl_sync(0xffffffffu, first, 1) - n0) << 6) + code + 1u;
    const uint32_t e2 = ((uint32_t)(__shfl_sync(0xffffffffu, first, 2) - n1) << 6) + code + 2u;
    const float hx = R.hf[0], ys = dy * R.hf[1], zs = dz * R.hf[2];
    const float rl2f = 0.5f * (V.rl2f_lo + V.rl2f_hi), margin = 0.5f * (V.rl2f_hi - V.rl2f_lo);
    const int maxn = V.maxneigh, lt = V.ltpa, lq = V.lvec;
    const int la = 5 - lt, ltq = lt + lq, tq = 1 << ltq;
    for (int h0 = 32 * part; h0 < hn; h0 += 32 * hsplit) {
        const int nh = min(32, hn - h0);
        const int hbase = hs + h0;  // slot of home atom 0 of this chunk
        __syncthreads();
        if (row == 0) {
            // padding far away (never accepted, never in the band)
            float4 hr = make_float4(1.0e18f, 1.0e18f, 1.0e18f, 0.f);
            if (lane < nh) hr = V.rec[hbase + lane];
            float *h = s_h[lane >> 1] + (lane & 1);
            h[0] = hr.x; h[2] = hr.y; h[4] = hr.z;
            h[6] = hr.x * hr.x + hr.y * hr.y + hr.z * hr.z;
        }
        __syncthreads();
        // candidates c0 .. c0 + 31 of the row against the home atoms: this lane's entry,
        // and its home atom's mask of accepted candidates
        auto round = [&](int c0, uint32_t &e) {
            const int f = c0 + lane;
            const bool in = f < m;
            const bool s1 = f >= n0, s2 = f >= n1;
            e = in ? ((uint32_t)f << 6) + (s2 ? e2 : s1 ? e1 : e0) : 0u;
            const int j = (int)(e >> 6);
            const float4 rj = V.rec[in ? j : hbase];
            const float qx = in ? rj.x + (s2 ? hx : s1 ? 0.f : -hx) : -1.0e18f, qy = in ? rj.y + ys : -1.0e18f,
                        qz = in ? rj.z + zs : -1.0e18f;
            const float qx2 = -2.0f * qx, qy2 = -2.0f * qy, qz2 = -2.0f * qz;
            const float q2m = qx * qx + qy * qy + qz * qz - rl2f;
            const unsigned long long qxx = pack2(qx2, qx2), qyy = pack2(qy2, qy2), qzz = pack2(qz2, qz2),
                                     qww = pack2(q2m, q2m);
            unsigned acc = 0u;
            float tmin = 3.0e38f;
#pragma unroll 1
            for (int hb = (nh - 1) & ~7; hb >= 0; hb -= 8) {
#pragma unroll
                for (int k = 6; k >= 0; k -= 2) {
                    const ulonglong2 *h = reinterpret_cast<const ulonglong2 *>(s_h[(hb + k) >> 1]);
                    const ulonglong2 xy = h[0], zw = h[1];
                    const float2 t = unpack2(fma2(qxx, xy.x, fma2(qyy, xy.y, fma2(qzz, zw.x, add2(zw.y, qww)))));
                    acc = __funnelshift_l(__float_as_uint(t.y), acc, 1);
                    acc = __funnelshift_l(__float_as_uint(t.x), acc, 1);
                    tmin = fmin3(tmin, fabsf(t.x), fabsf(t.y));
                }
            }
            if (tmin < margin) {  // margin band: decide those pairs in FP64 (rare)
                for (int k = 0; k < nh; ++k) {
                    const float *h = s_h[k >> 1] + (k & 1);
                    const float t = fmaf(qx2, h[0], fmaf(qy2, h[2], fmaf(qz2, h[4], h[6] + q2m)));
                    if (fabsf(t) < margin) {
                        const bool ok = in_list_fp64<PREC>(V, R, hbase + k, j, entry_dx(e), entry_dy(e), entry_dz(e));
                        acc = ok ? (acc | (1u << k)) : (acc & ~(1u << k));
                    }
                }
            }
            const int jh = j - hbase;
            if ((e & 63u) == kSelfCode && jh >= 0 && jh < 32) acc &= ~(1u << jh);
            if (HALF) acc &= jh <= 0 ? 0u : (jh >= 32 ? 0xffffffffu : ((1u << jh) - 1u));
            return warp_transpose32(acc, lane);
        };
        int cnt = 0;
        for (int c0 = 0, k = 0; c0 < m; c0 += 32, ++k) {
            uint32_t e;
            const unsigned t = round(c0, e);
            cnt += __popc(t);
            if (k < kRowKeep) {
                s_t[row][k][lane] = t;
                s_e[row][k][lane] = e;
            }
        }
        s_cnt[row][lane] = cnt;
        __syncthreads();
        int k0 = 0, total = 0;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int c = s_cnt[q][lane];
            k0 += q < row ? c : 0;
            total += c;
        }
        const int p = hbase + lane;
        uint32_t *const lbase =
            V.nlist + (size_t)(p >> la) * (size_t)((1 << la) * maxn) + (size_t)((p & ((1 << la) - 1)) << ltq);
        for (int c0 = 0, k = 0; c0 < m; c0 += 32, ++k) {
            unsigned t;
            const uint32_t *es;
            __syncwarp();
            if (k < kRowKeep) {
                t = s_t[row][k][lane];
                es = s_e[row][k];
            } else {  // (the last kept round's entries are used up by now)
                uint32_t e;
                t = round(c0, e);
                s_e[row][kRowKeep - 1][lane] = e;
                es = s_e[row][kRowKeep - 1];
                __syncwarp();
            }
            while (__any_sync(0xffffffffu, t != 0u)) {
                if (t) {
                    const uint32_t e = es[__ffs(t) - 1];
                    if (k0 < maxn) lbase[((unsigned)(k0 >> ltq) << (5 + lq)) + (unsigned)(k0 & (tq - 1))] = e;
                    ++k0;
                    t &= t - 1u;
                }
            }
        }
        if (row == 0 && lane < nh) {
            V.ncount[p] = min(total, maxn);
            if (total > maxn) {
                atomicMax(&V.ctl->need_maxneigh, total);
                latch_error(V.ctl, kErrOverflow);
            }
            my_max = max(my_max, total);
            my_sum += total;
        }
    }
    if (row == 0) build_stats(V, r, my_max, my_sum, lane);
}

template <int PREC, int HALF>
__global__ void __launch_bounds__(288) k_build_rows(View V, KArgs a) {
    const int gb = blockIdx.x / V.hsplit, part = blockIdx.x - gb * V.hsplit;
    if (a.all || V.rep_flag[V.bin_rep[gb]]) build_rows<PREC, HALF>(V, gb, part, V.hsplit);
    if (a.all && last_block(&V.ctl->ticket_build)) {
        if (threadIdx.x == 0) {
            V.ctl->ticket_build = 0;
            V.ctl->rebuilds += V.n_rep;
        }
    }
}

// Work list of a batched rebuild: the replicas flagged by the drift, each with
// its first (bin, part) unit and its first slot in flat numberings, its first
// global bin and its first slot.  One block: exclusive scans over the
// replicas, a block's width at a time.
__global__ void __launch_bounds__(1024) k_worklist(View V, KArgs a) {
    __shared__ int s_warp[32];
    int base_u = 0, base_s = 0, base_n = 0;
    for (int q0 = 0; q0 < V.n_rep; q0 += blockDim.x) {
        const int q = q0 + threadIdx.x;
        const bool f = q < V.n_rep && (a.all || V.rep_flag[q]);
        const int units = f ? V.rep[q].nbins * V.rep[q].hsplit : 0;
        const int slots = f ? V.rep[q].ntiles * 32 : 0;
        int tot_u, tot_s, tot_n;
        const int eu = block_excl_scan(units, s_warp, &tot_u);
        const int es = block_excl_scan(slots, s_warp, &tot_s);
        const int en = block_excl_scan(f ? 1 : 0, s_warp, &tot_n);
        if (f) {
            V.wl_u0[base_n + en] = base_u + eu;
            V.wl_bin[base_n + en] = V.rep[q].bin0;
            V.wl_hs[base_n + en] = V.rep[q].hsplit;
            V.wl_s0[base_n + en] = base_s + es;
            V.wl_a0[base_n + en] = V.rep[q].atom0;
        }
        base_u += tot_u;
        base_s += tot_s;
        base_n += tot_n;
    }
    if (threadIdx.x == 0) {
        V.wl_u0[base_n] = base_u;
        V.wl_s0[base_n] = base_s;
        *V.wl_n = base_n;
    }
}

struct Unit {  // a cell and one of the parts it is shared out in
    int gb, part, hsplit;
};

// unit u of the work list: in the last flagged replica f with wl_u0[f] <= u
__device__ __forceinline__ Unit wl_unit(const View &V, int nf, int u) {
    int lo = 0, hi = nf - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&V.wl_u0[mid]) <= u) lo = mid;
        else hi = mid - 1;
    }
    const int local = u - __ldg(&V.wl_u0[lo]), hs = __ldg(&V.wl_hs[lo]);
    return Unit{__ldg(&V.wl_bin[lo]) + local / hs, local % hs, hs};
}

// the work list's units by rows (see build_rows), where there are at most a.aux of them
template <int PREC, int HALF>
__global__ void __launch_bounds__(288, 3) k_build_rows_wl(View V, KArgs a) {
    const int nf = *V.wl_n, total = V.wl_u0[nf];
    if (total > a.aux) return;
    for (int u = blockIdx.x; u < total; u += gridDim.x) {
        const Unit q = wl_unit(V, nf, u);
        build_rows<PREC, HALF>(V, q.gb, q.part, q.hsplit);
    }
}

// Batched rebuild: a fixed grid walks the work list's units (k_worklist), so
// that the bins of replicas keeping their lists cost no block launches.  a.aux: as
// many units or fewer are left to k_build_rows_wl.
template <int PREC, int HALF>
__global__ void __launch_bounds__(32, kBuildWarps) k_build_wl(View V, KArgs a) {
    const int lane = threadIdx.x & 31, w = 0;
    const int nf = *V.wl_n;
    const int total = V.wl_u0[nf];
    if (total <= a.aux) return;
    for (int u = blockIdx.x; u < total; u += gridDim.x) {
        const Unit q = wl_unit(V, nf, u);
        int my_max = 0;
        long long my_sum = 0;
        build_cell<PREC, HALF, 1>(V, q.gb, q.part, q.hsplit, lane, w, my_max, my_sum);
        build_stats(V, V.bin_rep[q.gb], my_max, my_sum, lane);
    }
}

// ------------------------------------------------------------- dispatch ----

// Systems of at most so many (cell, part) units per SM are built by rows.  us per step (a rebuild every
// ~8): LJ 500 atoms 20.7 -> 18.7, 4,000 22.4 -> 20.1, 4,000 FP64 31.6 -> 29.3, 8,000 at rc 4.0 43.8 -> 36.9;
// 32,771 atoms (11 units per SM) 29.3 -> 29.9, 65,536 (21) 38.1 -> 41.8.
constexpr int kRowBuild = 6;
// In a batch the units that count are those of the replicas that rebuild in the step, which only the GPU knows: both
// builds are launched, and one of them returns.  us per step by cells / by rows / so decided: 40 replicas of 8,000
// atoms at rc 5.0 (36 units per SM, one in seven rebuilding) 882 / 902 / 791, all rebuilding together 577 / 865 /
// 522; 4 of 40,000 at rc 2.5 (45) 72 / 82 / 71, together 57 / 70 / 56; 20 of 8,000 at rc 4.0 264 / 257 / 243 (with the
// line at 3 and 12 units per SM 244 and 258).  Batches of at most kRowBuildOnly units per SM in all are built by
// rows only, which saves the second launch (10 replicas of 2,000 atoms at rc 2.5, 8.4 units, 52.7 -> 50.3; at 11.4 of
// denser cells, 8 of 8,000 at rc 5.0 together, it costs 197 -> 238), those of more than kRowBuildWl cells per SM by
// cells only.  In between, the two run side by side in a step's graph where rows are the likely choice (one
// replica in seven rebuilding): 16 replicas of 500 .. 4,000 atoms 68.0 -> 65.2 (64.7 by rows only), 30 of 500 .. 3,000
// 79.3 -> 76.7 (76.2); in larger batches the build by cells loses by it (4 of 60,000 at rc 5.0, 45 units: 430 -> 448).
constexpr int kRowBuildOnly = 9, kRowBuildLikely = 7 * kRowBuild, kRowBuildWl = 64;

// threads per block of the per-slot passes (k_prepare, k_scatter, k_gather), as the drift's: evaluation of 100,003 atoms at
// new coordinates 225 (256) -> 222 us
constexpr int kSortBlock = 64;

void rebuild_sequence(const View &V, bool all, bool staged, std::vector<KCall> &seq) {
    KArgs a{};
    a.all = all ? 1 : 0;
    const bool fp64 = V.prec == MD_PREC_FP64;
    // a batch rebuilding some of its replicas: list them first, then the
    // per-slot and per-bin passes walk the list with fixed grids
    const bool wl = V.n_rep > 1 && !all;
    KArgs as = a;
    as.wl = wl ? 1 : 0;
    const dim3 gs(wl ? (unsigned)(V.n_sm * 2048 / kSortBlock) : (unsigned)((V.n_pad + kSortBlock - 1) / kSortBlock));
    if (wl) seq.push_back(KCall{(const void *)k_worklist, dim3(1), dim3(1024), 0, a});
    const int nzb = (max(V.nbins_total, V.n_rep) + 255) / 256;
    seq.push_back(KCall{(const void *)k_zero_bins, dim3((unsigned)min(nzb, V.n_sm * 8)), dim3(256), 0, a});
    KArgs ap = as;
    ap.mode = staged ? 1 : 0;
    seq.push_back(KCall{fp64 ? (const void *)k_prepare<MD_PREC_FP64> : (const void *)k_prepare<MD_PREC_MIXED>, gs,
                        dim3(kSortBlock), 0, ap});
    if (V.n_rep == 1 && V.nbins_total <= kScanMost) {
        seq.push_back(KCall{(const void *)k_scan_scatter, dim3((V.n_pad + kScanThreads - 1) / kScanThreads),
                            dim3(kScanThreads), 0, a});
    } else {
        const int nblk = (V.nbins_total + kScanBlock - 1) / kScanBlock;
        seq.push_back(KCall{(const void *)k_scan1, dim3(nblk), dim3(1024), 0, a});
        seq.push_back(KCall{(const void *)k_scan3, dim3((V.nbins_total + 255) / 256), dim3(256), 0, a});
        seq.push_back(KCall{(const void *)k_scatter, gs, dim3(kSortBlock), 0, as});
    }
    seq.push_back(KCall{fp64 ? (const void *)k_gather<MD_PREC_FP64> : (const void *)k_gather<MD_PREC_MIXED>, gs,
                        dim3(kSortBlock), 0, as});
    if (V.tile_atoms > 0)
        seq.push_back(KCall{(const void *)k_tiles, dim3((V.n_ftiles + 3) / 4), dim3(128), 0, a});
    list_build_sequence(V, all, seq);
}

void list_build_sequence(const View &V, bool all, std::vector<KCall> &seq) {
    KArgs a{};
    a.all = all ? 1 : 0;
    const bool fp64 = V.prec == MD_PREC_FP64;
    if (V.n_rep > 1 && !all) {
        const bool rows = V.tile_atoms == 0 && V.nbins_total <= V.n_sm * kRowBuildWl;
        const bool only = V.n_units <= V.n_sm * kRowBuildOnly;
        a.aux = !rows ? 0 : only ? V.n_units : V.n_sm * kRowBuild;
        if (rows) {
            const void *kr = fp64 ? (V.half ? (const void *)k_build_rows_wl<MD_PREC_FP64, 1> : (const void *)k_build_rows_wl<MD_PREC_FP64, 0>)
                                  : (V.half ? (const void *)k_build_rows_wl<MD_PREC_MIXED, 1> : (const void *)k_build_rows_wl<MD_PREC_MIXED, 0>);
            seq.push_back(KCall{kr, dim3(std::min(V.n_sm * kRowBuild, V.n_units)), dim3(288), 0, a});
            if (only) return;
        }
        const void *kb = fp64 ? (V.half ? (const void *)k_build_wl<MD_PREC_FP64, 1> : (const void *)k_build_wl<MD_PREC_FP64, 0>)
                              : (V.half ? (const void *)k_build_wl<MD_PREC_MIXED, 1> : (const void *)k_build_wl<MD_PREC_MIXED, 0>);
        const int deal = std::min(kBuildWlDeal, 1 + V.nbins_total / (V.n_sm * kBuildWarps * 4));
        const bool beside = rows && V.n_units <= V.n_sm * kRowBuildLikely;
        seq.push_back(KCall{kb, dim3(V.n_sm * kBuildWarps * deal), dim3(32), 0, a, beside});
        return;
    }
    const void *kb;
    if (V.tile_atoms == 0 && V.nbins_total * V.hsplit <= V.n_sm * kRowBuild) {
        kb = fp64 ? (V.half ? (const void *)k_build_rows<MD_PREC_FP64, 1> : (const void *)k_build_rows<MD_PREC_FP64, 0>)
                  : (V.half ? (const void *)k_build_rows<MD_PREC_MIXED, 1> : (const void *)k_build_rows<MD_PREC_MIXED, 0>);
        seq.push_back(KCall{kb, dim3(V.nbins_total * V.hsplit), dim3(288), 0, a});
        return;
    }
    const int nw = V.hsplit > 1 ? 4 : 1;
    if (nw == 1)
        kb = fp64 ? (V.half ? (const void *)k_build<MD_PREC_FP64, 1, 1> : (const void *)k_build<MD_PREC_FP64, 0, 1>)
                  : (V.half ? (const void *)k_build<MD_PREC_MIXED, 1, 1> : (const void *)k_build<MD_PREC_MIXED, 0, 1>);
    else
        kb = fp64 ? (V.half ? (const void *)k_build<MD_PREC_FP64, 1, 4> : (const void *)k_build<MD_PREC_FP64, 0, 4>)
                  : (V.half ? (const void *)k_build<MD_PREC_MIXED, 1, 4> : (const void *)k_build<MD_PREC_MIXED, 0, 4>);
    seq.push_back(KCall{kb, dim3((V.nbins_total * V.hsplit + nw - 1) / nw), dim3(32 * nw), 0, a});
}

}  // namespace md
