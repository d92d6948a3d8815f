// k_force.cu -- mixed-precision pair-force kernels over the Verlet list (LJ
// full and half list, EAM density and force passes; the FP64 ones are in
// k_fp64.cu), the drift and kick kernels of velocity Verlet, and the md_step
// loop control.
//
// Force loop (paper Sec. III.B): a group of T threads owns atom i
// (T = 1 is the paper's thread-per-atom, T = 32 a warp-per-atom form of its
// block-per-atom); thread `sub` of the group walks list entries sub, sub+T,
// ..., gathers j's record, evaluates the pair term and accumulates; the group
// then reduces its partial sums with warp shuffles (the paper's reduce(ftmp)
// of the block-per-atom listing) and one thread writes atom i.
// Per-type coefficient tables are staged in shared memory; with one atom
// type the two coefficients are held in registers and nothing is staged.
//
// Precision (paper Sec. II, mixed mode: force in single, integration in
// double): MIXED gathers FP32 cell-relative records, does the pair
// arithmetic in FP32, sums each round's (at most Q) pair terms plainly and
// adds the round sum with Kahan compensation (forces, energy and virial
// alike), and folds the compensated sums into FP64 for the group reduction,
// kick and store.
#include <type_traits>

#include <cooperative_groups.h>

#include "md_common.cuh"
#include "md_kernels.h"

namespace md {

// ------------------------------------------------------ FP32 pair helpers --

__device__ __forceinline__ void load_rec(const View &V, int j, float &x, float &y, float &z, int &t) {
    const float4 r = __ldg(&V.rec[j]);
    x = r.x; y = r.y; z = r.z; t = __float_as_int(r.w);
}
// the same by an ordinary load: where the records change during the kernel (k_steps)
__device__ __forceinline__ void load_rec_now(const View &V, int j, float &x, float &y, float &z, int &t) {
    const float4 r = V.rec[j];
    x = r.x; y = r.y; z = r.z; t = __float_as_int(r.w);
}
__device__ __forceinline__ float rcp32(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// List entries, each read once per pass: kept out of L1, which belongs to the records (against evict-first
// loads, .cs: rc 5.0 804 -> 790 us per pass of 864,000 atoms, rc 4.0 77.5 -> 76.5 of 100,000, rc 2.5 the same;
// against ordinary loads 133.5 -> 125.2 of 864,000).
__device__ __forceinline__ uint32_t ld_stream(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.global.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

__device__ __forceinline__ uint4 ld_stream4(const uint32_t *p) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

__device__ __forceinline__ uint2 ld_stream2(const uint32_t *p) {
    uint2 v;
    asm volatile("ld.global.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}

// this thread's Q list entries of one round, one (vector) load
template <int Q>
__device__ __forceinline__ void load_entries(const uint32_t *p, uint32_t (&e)[Q]) {
    if constexpr (Q == 4) {
        const uint4 u = ld_stream4(p);
        e[0] = u.x; e[1] = u.y; e[2] = u.z; e[3] = u.w;
    } else if constexpr (Q == 2) {
        const uint2 u = ld_stream2(p);
        e[0] = u.x; e[1] = u.y;
    } else {
        e[0] = ld_stream(p);
    }
}

// reduce a double over the T consecutive lanes of a group
template <int T>
__device__ __forceinline__ double group_sum(double x) {
    for (int o = T / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// |d|^2 with its operations spelled out (no contraction left to the compiler),
// so that a pair's FP32 r^2 recomputed after the walk is the walk's own
__device__ __forceinline__ float pair_r2(float dx, float dy, float dz) {
    return fmaf(dz, dz, fmaf(dy, dy, dx * dx));
}

// Walk this thread's share of atom i's list: rounds of T*Q entries, the
// thread's Q entries arriving in one (vector) load, the next round's load
// issued before this round's work; the Q records are gathered before any
// arithmetic so that Q gathers are in flight.  For each entry calls
// pair(e, dx, dy, dz, r2, tj) with d = x_i - x_j (periodic image included),
// bracketed per round by pair.round_begin() / pair.round_end(): the pair
// terms of one round (at most Q) are summed plainly and the round's sum is
// added to the running total with compensation (blocked Kahan summation:
// error ~ (Q + 2) u sum |terms| instead of ~n u for n plain additions).
// Pair::kPacked: the x and y components' operations go two to an instruction, and pair gets
// d_x and d_y packed as well: the same values from ~10 % fewer instructions (EAM).
// LOCAL: the entries are block-local and the records come from the block's
// staging in shared memory (srec).
template <int T, int Q, bool LOCAL, class Pair>
__device__ __forceinline__ void walk_list(const View &V, const uint32_t *lp, int sub, int cnt, float xi, float yi,
                                          float zi, float hx, float hy, float hz, const float4 *srec, Pair &pair) {
    constexpr int PER = T * Q;
    const int nr = (cnt + PER - 1) / PER;
    const float hy4 = hy * 0.25f, hz16 = hz * 0.0625f;  // exact: powers of two
    uint32_t cur[Q], nxt[Q];
    if (nr > 0) load_entries<Q>(lp, cur);
    for (int r = 0; r < nr; ++r) {
        if (r + 1 < nr) load_entries<Q>(lp + (size_t)(r + 1) * 32 * Q, nxt);
        const int left = cnt - (r * PER + sub * Q);
        if constexpr (Pair::kPacked) {
            ulonglong2 rj[Q];  // the records: {x, y}, {z, type}
#pragma unroll
            for (int q = 0; q < Q; ++q)
                if (q < left) {
                    const float4 *at = LOCAL ? &srec[entry_j(cur[q]) & (kTileCap - 1)] : &V.rec[entry_j(cur[q])];
                    rj[q] = LOCAL ? *reinterpret_cast<const ulonglong2 *>(at) : __ldg(reinterpret_cast<const ulonglong2 *>(at));
                }
            pair.round_begin();
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                if (q < left) {
                    const uint32_t e = cur[q];
                    // the scalar form's operations (see below), x and y side by side
                    const f32x2 c = add2(pack2(__int_as_float(0x4B400000u | (e & 0x3u)), __int_as_float(0x4B400000u | (e & 0xCu))),
                                         pack2(-12582913.0f, -12582916.0f));
                    const f32x2 dxy = fma2(c, pack2(-hx, -hy4), sub2(pack2(xi, yi), rj[q].x));
                    const float2 zt = unpack2(rj[q].y), d = unpack2(dxy);
                    const float dz = fmaf(-code_z16(e), hz16, zi - zt.x);
                    pair(dxy, d.x, d.y, dz, pair_r2(d.x, d.y, dz), __float_as_int(zt.y));
                }
            }
            pair.round_end();
        } else {
            float xj[Q], yj[Q], zj[Q];
            int tj[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                if (q < left) {
                    if constexpr (LOCAL) {
                        const float4 r4 = srec[entry_j(cur[q]) & (kTileCap - 1)];
                        xj[q] = r4.x; yj[q] = r4.y; zj[q] = r4.z; tj[q] = __float_as_int(r4.w);
                    } else {
                        load_rec(V, entry_j(cur[q]), xj[q], yj[q], zj[q], tj[q]);
                    }
                }
            }
            pair.round_begin();
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                if (q < left) {
                    const uint32_t e = cur[q];
                    const float dx = fmaf(-code_x(e), hx, xi - xj[q]);
                    const float dy = fmaf(-code_y4(e), hy4, yi - yj[q]);
                    const float dz = fmaf(-code_z16(e), hz16, zi - zj[q]);
                    const float r2 = pair_r2(dx, dy, dz);
                    pair(e, dx, dy, dz, r2, tj[q]);
                }
            }
            pair.round_end();
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) cur[q] = nxt[q];
    }
}

// the list walk in this block's tile mode (records staged or gathered)
template <int T, int Q, class Pair>
__device__ __forceinline__ void walk_mode(const View &V, int mode, const uint32_t *lp, int sub, int cnt, float xi,
                                          float yi, float zi, const Rep &R, const float4 *srec, Pair &pair) {
    if (mode == 1)
        walk_list<T, Q, true>(V, lp, sub, cnt, xi, yi, zi, R.hf[0], R.hf[1], R.hf[2], srec, pair);
    else
        walk_list<T, Q, false>(V, lp, sub, cnt, xi, yi, zi, R.hf[0], R.hf[1], R.hf[2], srec, pair);
}

// The same walk for a system too small to fill the GPU with T threads per
// atom, whose rounds would follow one another at the latency of a gather:
// G lanes stand in for each of the T threads, lane g taking rounds g, g + G, ....
// The rounds' sums go to shared memory, and lane g adds term g (g + G, ... ; force
// components, energy and virial terms) of all rounds in the thread's own order: bit for
// bit the sums of walk_list.  What bounds it is the length of a warp's instruction stream at ~9 clocks
// an instruction, so each term is added by one lane (all G lanes adding all terms,
// by shuffles: 1,410 instructions per warp and 11.2 us for 500 atoms).
struct Wide {
    int lt, lg;   // log2 of T and G
    int p;        // this lane's atom
    int sub, g;   // its thread of the atom's T, its lane of that thread's G
};

// lane of the pass's warp number gw
__device__ __forceinline__ Wide wide_lane(const View &V, int lg, int gw) {
    Wide w;
    w.lt = V.ltpa;
    w.lg = lg;
    const int ll = w.lt + lg, lane = threadIdx.x & 31;
    w.p = (gw << (5 - ll)) + (lane >> ll);
    const int i = lane & ((1 << ll) - 1);
    w.sub = i >> lg;
    w.g = i & ((1 << lg) - 1);
    return w;
}

// sum over the T threads of the atom, in group_sum's order
__device__ __forceinline__ double wide_sum(const Wide &w, double x) {
    for (int o = (1 << w.lt) >> 1; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o << w.lg);
    return x;
}

// A wide lane's atom as it is loaded at once, before anything is known about
// it: every dependent load costs a small system ~0.4 us.  (The first list entries lie within
// the list's capacity; past the list's end they are not looked at.)
template <int Q>
struct WideAtom {
    const uint32_t *lp;
    uint32_t cur[Q];
    float x, y, z;
    int t, count;
    unsigned err;
    int remaining;
};

template <int Q>
__device__ __forceinline__ WideAtom<Q> load_wide(const View &V, const Wide &w) {
    WideAtom<Q> a;
    const int la = 5 - w.lt;
    a.lp = V.nlist + (size_t)(w.p >> la) * ((size_t)V.maxneigh << la) +
           (size_t)(((w.p & ((1 << la) - 1)) << w.lt) + w.sub) * Q;
    if (w.g < (V.maxneigh >> w.lt) / Q) load_entries<Q>(a.lp + (size_t)w.g * 32 * Q, a.cur);
    load_rec_now(V, w.p, a.x, a.y, a.z, a.t);
    a.count = V.ncount[w.p];
    a.err = V.ctl->err;
    a.remaining = V.ctl->remaining;
    return a;
}

// NT terms; KT: the most that one lane adds (terms g + k G, k < KT, G >= 2)
template <int Q, int NT, int KT, class Pair>
__device__ __forceinline__ void walk_wide(const View &V, const Wide &w, const Rep &R, int cnt, WideAtom<Q> &at,
                                          float (*s_round)[32], Pair &pair, KahanF (&acc)[KT]) {
    const float hx = R.hf[0], hy4 = R.hf[1] * 0.25f, hz16 = R.hf[2] * 0.0625f;
    const float xi = at.x, yi = at.y, zi = at.z;
    const int lane = threadIdx.x & 31;
    const int per = Q << w.lt, G = 1 << w.lg;
    const int nr = (cnt + per - 1) >> (w.lt + (Q == 4 ? 2 : Q == 2 ? 1 : 0));
    const int most = __reduce_max_sync(0xffffffffu, nr);
    const uint32_t *lp = at.lp;
    const int first = lane - w.g;
    uint32_t (&cur)[Q] = at.cur, nxt[Q];
    for (int r0 = 0; r0 < most; r0 += G) {
        const int r = r0 + w.g;
        if (r + G < nr) load_entries<Q>(lp + (size_t)(r + G) * 32 * Q, nxt);
        const int left = r < nr ? cnt - (r * per + w.sub * Q) : 0;
        float xj[Q], yj[Q], zj[Q];
        int tj[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q)
            if (q < left) load_rec_now(V, entry_j(cur[q]), xj[q], yj[q], zj[q], tj[q]);
        pair.round_begin();
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            if (q < left) {
                const uint32_t e = cur[q];
                const float dx = fmaf(-code_x(e), hx, xi - xj[q]);
                const float dy = fmaf(-code_y4(e), hy4, yi - yj[q]);
                const float dz = fmaf(-code_z16(e), hz16, zi - zj[q]);
                pair(e, dx, dy, dz, pair_r2(dx, dy, dz), tj[q]);
            }
        }
#pragma unroll
        for (int k = 0; k < NT; ++k) s_round[k][lane] = pair.term(k);
        __syncwarp();
        const int n = min(nr - r0, G);  // rounds of this turn
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            const int term = w.g + k * G;
            if (term < NT) {
                const float *s = &s_round[term][first];
#pragma unroll 4
                for (int g = 0; g < n; ++g) acc[k].add(s[g]);
            }
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < Q; ++q) cur[q] = nxt[q];
    }
}

// stage the block's tile when its entries are block-local (before the
// kernel's first block barrier)
__device__ __forceinline__ int begin_tile(const View &V, int T, float4 *srec) {
    const int mode = tile_mode(V, T);
    if (mode == 1) stage_tile(V, blockIdx.x, srec);
    return mode;
}

// Epilogue of atom p (after the group reduction), by the group's lane 0.
//   kModeStoreF: F -> f.   kModeStep: v += c dt a with c = 1 (leapfrog full
//   kick) or 1/2 (last step of the call, F also stored).   kModeEV: F -> f.
__device__ __forceinline__ void epilogue(const View &V, int mode, int rem, int p, int t, double fx, double fy,
                                         double fz, const double *s_ftm) {
    const int n = V.n_pad;
    if (mode == kModeStep || mode == kModeKickDry) {
        const bool last = (mode == kModeStep && rem == 0);
        const double c = (mode == kModeKickDry) ? 0.0 : (last ? 0.5 : 1.0) * V.dt * s_ftm[t];
        V.v[p] += c * fx;
        V.v[n + p] += c * fy;
        V.v[2 * n + p] += c * fz;
        if (last) {
            V.f[p] = fx; V.f[n + p] = fy; V.f[2 * n + p] = fz;
        }
    } else {
        V.f[p] = fx; V.f[n + p] = fy; V.f[2 * n + p] = fz;
    }
}

__device__ __forceinline__ void write_ev(const View &V, int p, int t, double e, const double *w, const double *s_ftm) {
    const int n = V.n_pad;
    V.ev[p] = e;
    write_kinetic(V, p, s_ftm[t]);
    for (int k = 0; k < 6; ++k) V.ev[(2 + k) * n + p] = w[k];
}

// ---------------------------------------------------------------- LJ ----

// The FP64 path's cut-off decision for the pair (p, entry e) of a mixed pass,
// from the FP64 positions with the same formula (rare: only pairs whose FP32
// r^2 lies within rc2f_band of rc^2 -- the unshifted LJ force jumps at rc, so
// there a decision that differs from FP64 would move F_i by ~|f(rc)|).
__device__ __forceinline__ bool in_cut_fp64(const View &V, int p, uint32_t e) {
    const int n = V.n_pad;
    const int j = entry_slot(V, p, e);
    const Rep &R = V.rep[V.tile_rep[p >> 5]];
    const double dx = fma(-(double)entry_dx(e), R.h[0], V.xr[p] - V.xr[j]);
    const double dy = fma(-(double)entry_dy(e), R.h[1], V.xr[n + p] - V.xr[n + j]);
    const double dz = fma(-(double)entry_dz(e), R.h[2], V.xr[2 * n + p] - V.xr[2 * n + j]);
    return dx * dx + dy * dy + dz * dz < V.rc2;
}

// FULL: every neighbour in i's list, F_i only, no atomics.
// HALF: each pair once; F_j -= f_ij by FP64 atomics, F_i += sum by one atomic
//       per component at the end (F zeroed beforehand; kick in k_kick).
template <int MT, int HALF, int EV>
struct LJPair {
    static constexpr bool kPacked = false;
    const View *V;
    const float *lj1, *lj2, *lj3, *lj4, *off;
    float c3, c4, c0;  // one atom type: the energy coefficients and shift, likewise
    float c1, c2;  // one atom type (MT = 0): the coefficients in registers, not
                   // re-read from shared memory for every pair
    float rc2;
    int ti, nt, n;
    float near_min;  // the smallest |r^2 - rc^2| of this thread's pairs
    KahanF ax, ay, az, e;
    KahanF w[6];
    float rx, ry, rz;  // this round's plain partial sums
    float re, rw[6];   // and of the energy and virial terms (EV)
    __device__ __forceinline__ bool in_cut(float r2) {
        const float t = r2 - rc2;  // t < 0 exactly when r2 < rc2
        near_min = fminf(near_min, fabsf(t));
        return t < 0.f;
    }
    __device__ __forceinline__ void round_begin() {
        rx = 0; ry = 0; rz = 0;
        if (EV) {
            re = 0;
            for (int k = 0; k < 6; ++k) rw[k] = 0;
        }
    }
    __device__ __forceinline__ void round_end() {
        ax.add(rx); ay.add(ry); az.add(rz);
        if (EV) {
            e.add(re);
            for (int k = 0; k < 6; ++k) w[k].add(rw[k]);
        }
    }
    // the round's sums, in the order of the wide passes' terms
    __device__ __forceinline__ float term(int k) const {
        return k == 0 ? rx : k == 1 ? ry : k == 2 ? rz : k == 3 ? re : rw[k - 4];
    }
    // energy and virial terms of one pair: summed plainly over the round and
    // added with compensation per round
    __device__ __forceinline__ void add_ev(float ee, float w0, float w1, float w2, float w3, float w4, float w5) {
        re += ee;
        rw[0] += w0; rw[1] += w1; rw[2] += w2; rw[3] += w3; rw[4] += w4; rw[5] += w5;
    }
    __device__ __forceinline__ void operator()(uint32_t ent, float dx, float dy, float dz, float r2, int tj) {
        // full list, forces only: branch-free (the skin entries' terms are
        // computed, finite since r2 >= rc^2 there, and zeroed) -- measured faster
        // than skipping them under a per-lane branch
        if constexpr (!HALF && !EV) {
            const int tp = MT ? ti * nt + tj : 0;
            const float r2i = rcp32(r2);
            const float r6i = r2i * r2i * r2i;
            const float a1 = MT ? lj1[tp] : c1, a2 = MT ? lj2[tp] : c2;
            float fpair = r6i * (a1 * r6i - a2) * r2i;
            fpair = in_cut(r2) ? fpair : 0.f;
            rx += dx * fpair; ry += dy * fpair; rz += dz * fpair;
            return;
        }
        // full list, one atom type, with energy and virial: branch-free
        // as well (a zero force term zeroes the virial terms; the energy term
        // is selected)
        if constexpr (!HALF && EV && !MT) {
            const float r2i = rcp32(r2);
            const float r6i = r2i * r2i * r2i;
            const bool in = in_cut(r2);
            const float fpair = in ? r6i * (c1 * r6i - c2) * r2i : 0.f;
            const float fxp = dx * fpair, fyp = dy * fpair, fzp = dz * fpair;
            rx += fxp; ry += fyp; rz += fzp;
            const float h = 0.5f;
            add_ev(in ? h * (r6i * (c3 * r6i - c4) - c0) : 0.f, h * dx * fxp, h * dy * fyp, h * dz * fzp,
                   h * dx * fyp, h * dx * fzp, h * dy * fzp);
            return;
        }
        if (in_cut(r2)) {
            const int tp = MT ? ti * nt + tj : 0;
            const float r2i = rcp32(r2);
            const float r6i = r2i * r2i * r2i;
            const float a1 = MT ? lj1[tp] : c1, a2 = MT ? lj2[tp] : c2;
            const float fpair = r6i * (a1 * r6i - a2) * r2i;
            const float fxp = dx * fpair, fyp = dy * fpair, fzp = dz * fpair;
            rx += fxp; ry += fyp; rz += fzp;
            if (HALF) {
                const int j = entry_j(ent);
                atomicAdd(&V->f[j], -(double)fxp);
                atomicAdd(&V->f[n + j], -(double)fyp);
                atomicAdd(&V->f[2 * n + j], -(double)fzp);
            }
            if (EV) {
                const float wgt = HALF ? 1.f : 0.5f;
                const float a3 = MT ? lj3[tp] : c3, a4 = MT ? lj4[tp] : c4, a0 = MT ? off[tp] : c0;
                add_ev(wgt * (r6i * (a3 * r6i - a4) - a0), wgt * dx * fxp, wgt * dy * fyp,
                       wgt * dz * fzp, wgt * dx * fyp, wgt * dx * fzp, wgt * dy * fzp);
            }
        }
    }
};

// Mixed: every pair near rc gets the FP64 path's cut-off decision.  A
// thread whose pairs came within rc2f_band of rc^2 (rare) has its atom's list
// walked again by the whole warp, one entry per lane.  Each lane recomputes
// the pair's FP32 r^2 exactly as the walk did (same record, same operations)
// and, for a pair near rc that FP64 decides otherwise, forms the term to take
// out (counted by the walk) or to add (left out by it): force, half-list
// partner, energy and virial alike.  The terms are summed over the warp into
// the atom's first thread.  All 32 lanes call this together.
// T = 0: the wide kernels, whose lanes per atom are a run-time value and whose
// terms go to the lanes (of the atom's first thread) that add them.
template <int T, int Q, int MT, int HALF, int EV, int KT = 1>
__device__ __forceinline__ void fix_near_warp(const View &V, LJPair<MT, HALF, EV> &pr, bool flagged,
                                              int gw, int lane, int tmode, const float4 *srec, const Wide *w = nullptr,
                                              KahanF *acc = nullptr) {
    constexpr bool kWide = T == 0;
    const int L = kWide ? 1 << (w->lt + w->lg) : T;  // lanes per atom
    const int A = 32 / L;
    unsigned m = __ballot_sync(0xffffffffu, flagged);
    while (m) {
        const int a = (__ffs(m) - 1) / L;  // the atom's index in the warp
        m &= (L == 32) ? 0u : ~((((1u << (L & 31)) - 1u)) << (a * L));
        const int p = gw * A + a;
        const Rep &R = V.rep[V.tile_rep[p >> 5]];
        const int cnt = V.ncount[p];
        float xi, yi, zi;
        int ti;
        if constexpr (kWide) load_rec_now(V, p, xi, yi, zi, ti);
        else load_rec(V, p, xi, yi, zi, ti);
        const float hx = R.hf[0], hy4 = R.hf[1] * 0.25f, hz16 = R.hf[2] * 0.0625f;
        const uint32_t *base = V.nlist + (size_t)gw * (size_t)(A * V.maxneigh) + a * L * Q;
        float cx = 0.f, cy = 0.f, cz = 0.f, ce = 0.f, cw[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int k = lane; k < cnt; k += 32) {
            const uint32_t e = kWide ? V.nlist[list_index(p, k, V.ltpa, V.lvec, V.maxneigh)]
                                     : base[(size_t)(k / (L * Q)) * 32 * Q + (k % (L * Q))];
            float xj, yj, zj;
            int tj;
            if (tmode == 1) {
                const float4 r4 = srec[entry_j(e) & (kTileCap - 1)];
                xj = r4.x; yj = r4.y; zj = r4.z; tj = __float_as_int(r4.w);
            } else if constexpr (kWide) {
                load_rec_now(V, entry_j(e), xj, yj, zj, tj);
            } else {
                load_rec(V, entry_j(e), xj, yj, zj, tj);
            }
            const float dx = fmaf(-code_x(e), hx, xi - xj);
            const float dy = fmaf(-code_y4(e), hy4, yi - yj);
            const float dz = fmaf(-code_z16(e), hz16, zi - zj);
            const float r2 = pair_r2(dx, dy, dz);
            const float t = r2 - pr.rc2;
            if (!(fabsf(t) < V.rc2f_band)) continue;
            const bool exact = in_cut_fp64(V, p, e);
            if (exact == (t < 0.f)) continue;
            const float sgn = exact ? 1.f : -1.f;
            const int tp = MT ? ti * pr.nt + tj : 0;
            const float r2i = rcp32(r2);
            const float r6i = r2i * r2i * r2i;
            const float a1 = MT ? pr.lj1[tp] : pr.c1, a2 = MT ? pr.lj2[tp] : pr.c2;
            const float fpair = sgn * r6i * (a1 * r6i - a2) * r2i;
            const float fxp = dx * fpair, fyp = dy * fpair, fzp = dz * fpair;
            cx += fxp; cy += fyp; cz += fzp;
            if (HALF) {
                const int j = entry_j(e);
                atomicAdd(&V.f[j], -(double)fxp);
                atomicAdd(&V.f[pr.n + j], -(double)fyp);
                atomicAdd(&V.f[2 * pr.n + j], -(double)fzp);
            }
            if (EV) {
                const float wgt = HALF ? 1.f : 0.5f;
                const float a3 = MT ? pr.lj3[tp] : pr.c3, a4 = MT ? pr.lj4[tp] : pr.c4, a0 = MT ? pr.off[tp] : pr.c0;
                ce += sgn * wgt * (r6i * (a3 * r6i - a4) - a0);
                cw[0] += wgt * dx * fxp; cw[1] += wgt * dy * fyp; cw[2] += wgt * dz * fzp;
                cw[3] += wgt * dx * fyp; cw[4] += wgt * dx * fzp; cw[5] += wgt * dy * fzp;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            cx += __shfl_xor_sync(0xffffffffu, cx, o);
            cy += __shfl_xor_sync(0xffffffffu, cy, o);
            cz += __shfl_xor_sync(0xffffffffu, cz, o);
            if (EV) {
                ce += __shfl_xor_sync(0xffffffffu, ce, o);
                for (int c = 0; c < 6; ++c) cw[c] += __shfl_xor_sync(0xffffffffu, cw[c], o);
            }
        }
        if constexpr (kWide) {
            const float all[10] = {cx, cy, cz, ce, cw[0], cw[1], cw[2], cw[3], cw[4], cw[5]};
            if (lane / L == a && w->sub == 0) {
#pragma unroll
                for (int k = 0; k < KT; ++k) {
                    const int term = w->g + (k << w->lg);
#pragma unroll
                    for (int q = 0; q < (EV ? 10 : 3); ++q)
                        if (term == q) acc[k].add(all[q]);
                }
            }
        } else if (lane == a * T) {
            pr.ax.add(cx); pr.ay.add(cy); pr.az.add(cz);
            if (EV) {
                pr.e.add(ce);
                for (int c = 0; c < 6; ++c) pr.w[c].add(cw[c]);
            }
        }
    }
}

constexpr int kWideBlock = 64;

// registers per thread allowed to the mixed force-only pass: 56 keeps nine
// 128-thread blocks (36 warps) resident per SM to hide the gather latency;
// groups of 8+ threads and half lists with 4-entry loads take 64 (no spills);
// the full-list energy/virial pass 80 (six blocks instead of five, no
// spills: 0.39 -> 0.37 ms per md_energy_virial on the 864,000-atom liquid);
// the half-list energy pass what it needs
template <int T, int Q, int HALF, int EV>
struct LjRegs {
    static constexpr int value = !EV ? (Q == 4 && (T > 4 || HALF) ? 64 : 56) : (!HALF ? 80 : 255);
};

template <int T, int Q, int HALF, int EV, int MT>
__global__ void __maxnreg__((LjRegs<T, Q, HALF, EV>::value)) k_lj(View V, KArgs a) {
    __shared__ float s_lj1[kMaxTypes * kMaxTypes], s_lj2[kMaxTypes * kMaxTypes];
    __shared__ float s_lj3[kMaxTypes * kMaxTypes], s_lj4[kMaxTypes * kMaxTypes], s_off[kMaxTypes * kMaxTypes];
    __shared__ double s_ftm_sh[kMaxTypes];
    // one atom type: no table to stage, so no block barrier either (unless
    // the block stages records); the coefficients and ftm2v/m are read into
    // registers (-2.1 us per step on the 864,000-atom liquid against staging
    // them)
    constexpr bool kRegOnly = (MT == 0);
    const double *s_ftm = kRegOnly ? V.tab->ftm_m : s_ftm_sh;
    const int np = kRegOnly ? 0 : V.ntypes * V.ntypes;
    for (int k = threadIdx.x; k < np; k += blockDim.x) {
        s_lj1[k] = V.tab->lj1f[k]; s_lj2[k] = V.tab->lj2f[k];
        s_lj3[k] = V.tab->lj3f[k]; s_lj4[k] = V.tab->lj4f[k]; s_off[k] = V.tab->offf[k];
    }
    if (!kRegOnly && threadIdx.x < kMaxTypes) s_ftm_sh[threadIdx.x] = V.tab->ftm_m[threadIdx.x];
    extern __shared__ float4 s_rec[];
    const int tmode = HALF ? 0 : begin_tile(V, T, s_rec);
    if (!kRegOnly || V.tile_atoms != 0) __syncthreads();

    const unsigned err = V.ctl->err;
    const int rem = (a.mode == kModeStep) ? V.ctl->remaining : 0;
    constexpr int A = 32 / T;
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int p = gw * A + lane / T;
    const int sub = lane & (T - 1);
    const bool warp_in = (gw * A < V.n_pad) && err == 0 && tmode >= 0;

    LJPair<MT, HALF, EV> pr;
    pr.V = &V;
    pr.lj1 = s_lj1; pr.lj2 = s_lj2; pr.lj3 = s_lj3; pr.lj4 = s_lj4; pr.off = s_off;
    if (kRegOnly) {
        pr.c1 = V.tab->lj1f[0];
        pr.c2 = V.tab->lj2f[0];
        if (EV) {
            pr.c3 = V.tab->lj3f[0];
            pr.c4 = V.tab->lj4f[0];
            pr.c0 = V.tab->offf[0];
        }
    } else {
        pr.c1 = s_lj1[0]; pr.c2 = s_lj2[0];
    }
    pr.rc2 = V.rc2f;
    pr.nt = V.ntypes;
    pr.n = V.n_pad;
    pr.ti = 0;
    pr.near_min = 3.0e38f;
    pr.ax.zero(); pr.ay.zero(); pr.az.zero(); pr.e.zero();
    for (int k = 0; k < 6; ++k) pr.w[k].zero();
    bool valid = false;
    if (warp_in) {
        const Rep &R = V.rep[V.n_rep == 1 ? 0 : V.tile_rep[p >> 5]];  // one replica: no lookup
        valid = (p - R.atom0) < R.natoms;
        if (valid) {
            const int cnt = V.ncount[p];
            float xi, yi, zi;
            load_rec(V, p, xi, yi, zi, pr.ti);
            const uint32_t *lp = V.nlist + (size_t)gw * (size_t)(A * V.maxneigh) + lane * Q;
            walk_mode<T, Q>(V, tmode, lp, sub, cnt, xi, yi, zi, R, s_rec, pr);
        }
        fix_near_warp<T, Q>(V, pr, pr.near_min < V.rc2f_band, gw, lane, tmode, s_rec);
    }
    const double fx = group_sum<T>(pr.ax.value());
    const double fy = group_sum<T>(pr.ay.value());
    const double fz = group_sum<T>(pr.az.value());
    double e_acc = 0.0, w_acc[6] = {0, 0, 0, 0, 0, 0};
    if (EV) {
        e_acc = group_sum<T>(pr.e.value());
        for (int k = 0; k < 6; ++k) w_acc[k] = group_sum<T>(pr.w[k].value());
    }
    if (valid && sub == 0) {
        if (HALF) {
            const int n = V.n_pad;
            atomicAdd(&V.f[p], fx);
            atomicAdd(&V.f[n + p], fy);
            atomicAdd(&V.f[2 * n + p], fz);
            if (EV) {
                V.ev[p] = e_acc;
                for (int k = 0; k < 6; ++k) V.ev[(2 + k) * n + p] = w_acc[k];
            }
        } else {
            epilogue(V, a.mode, rem, p, pr.ti, fx, fy, fz, s_ftm);
            if (EV) write_ev(V, p, pr.ti, e_acc, w_acc, s_ftm);
        }
    }
}

// Coefficients of an LJ wide pass: the tables of several types in shared memory
template <int MT>
struct WideTab {
    const float *lj1, *lj2, *lj3, *lj4, *off;
    float c1, c2, c3, c4, c0;
};

// stage (several types; ends with a block barrier) or load the coefficients
template <int MT>
__device__ __forceinline__ WideTab<MT> wide_tab(const View &V, float (*s_tab)[kMaxTypes * kMaxTypes]) {
    WideTab<MT> t;
    if (MT) {
        for (int k = threadIdx.x; k < V.ntypes * V.ntypes; k += blockDim.x) {
            s_tab[0][k] = V.tab->lj1f[k]; s_tab[1][k] = V.tab->lj2f[k];
            s_tab[2][k] = V.tab->lj3f[k]; s_tab[3][k] = V.tab->lj4f[k]; s_tab[4][k] = V.tab->offf[k];
        }
        __syncthreads();
        t.lj1 = s_tab[0]; t.lj2 = s_tab[1]; t.lj3 = s_tab[2]; t.lj4 = s_tab[3]; t.off = s_tab[4];
    } else {
        t.c1 = V.tab->lj1f[0]; t.c2 = V.tab->lj2f[0];
        t.c3 = V.tab->lj3f[0]; t.c4 = V.tab->lj4f[0]; t.c0 = V.tab->offf[0];
    }
    return t;
}

// one warp's atoms of the full-list pass (gw: the warp's number); all 32 lanes
template <int Q, int EV, int MT>
__device__ __forceinline__ void lj_wide_warp(const View &V, int mode, int rem, int gw, const Wide &w, WideAtom<Q> &at,
                                             const Rep &R, const WideTab<MT> &tab, float (*s_round)[32]) {
    constexpr int NT = EV ? 10 : 3, KT = (NT + 1) / 2;
    LJPair<MT, 0, EV> pr;
    pr.V = &V;
    pr.lj1 = tab.lj1; pr.lj2 = tab.lj2; pr.lj3 = tab.lj3; pr.lj4 = tab.lj4; pr.off = tab.off;
    pr.c1 = tab.c1; pr.c2 = tab.c2; pr.c3 = tab.c3; pr.c4 = tab.c4; pr.c0 = tab.c0;
    pr.rc2 = V.rc2f;
    pr.nt = V.ntypes;
    pr.n = V.n_pad;
    pr.ti = at.t;
    pr.near_min = 3.0e38f;
    KahanF acc[KT];
    for (int k = 0; k < KT; ++k) acc[k].zero();
    const double ftm = V.tab->ftm_m[MT ? at.t : 0];
    const bool valid = (w.p - R.atom0) < R.natoms;
    walk_wide<Q, NT, KT>(V, w, R, valid ? at.count : 0, at, s_round, pr, acc);
    fix_near_warp<0, Q, MT, 0, EV, KT>(V, pr, pr.near_min < V.rc2f_band, gw, threadIdx.x & 31, 0, nullptr, &w, acc);
#pragma unroll
    for (int k = 0; k < KT; ++k) {
        const int term = w.g + (k << w.lg);
        const double x = wide_sum(w, acc[k].value());
        if (!valid || w.sub != 0) continue;
        if (term < 3) finish_component(V, mode, rem, term, w.p, ftm, x);
        else if (EV && term < NT) V.ev[(size_t)(term == 3 ? 0 : term - 2) * V.n_pad + w.p] = x;
    }
    if (EV && valid && w.sub == 0 && w.g == 0) write_kinetic(V, w.p, ftm);
}

// the full-list pass of a small system (see walk_wide); a.aux = log2 of G
template <int Q, int EV, int MT>
__global__ void __launch_bounds__(kWideBlock) k_lj_wide(View V, KArgs a) {
    __shared__ float s_round[kWideBlock / 32][EV ? 10 : 3][32];
    __shared__ float s_tab[5][kMaxTypes * kMaxTypes];
    const WideTab<MT> tab = wide_tab<MT>(V, s_tab);
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const Wide w = wide_lane(V, a.aux, gw);
    if (w.p >= V.n_pad) return;  // whole warps: n_pad is a multiple of 32
    WideAtom<Q> at = load_wide<Q>(V, w);
    const Rep &R = V.rep[V.n_rep == 1 ? 0 : V.tile_rep[w.p >> 5]];
    if (at.err) return;
    lj_wide_warp<Q, EV, MT>(V, a.mode, at.remaining, gw, w, at, R, tab, s_round[threadIdx.x >> 5]);
}

// Cell-list force pass, no Verlet list (the alternative the paper measures
// against neighbour lists, Sec. III.C): block b stages tile b's cells as the
// block-local lists do, and each atom tests every record of the 27 cells
// around its cell as binned at the last rebuild.  Atoms have moved less than
// skin/2 since then and cells are at least rc + skin wide, so every pair
// within rc is among them.  Lanes of one home cell read the same records in
// the same order (shared-memory broadcasts).  Mixed precision, one thread
// per atom, one 128-atom tile per block; a tile too dense to stage reads the
// cells' records from global memory.  Forces only (no energy/virial).
template <int MT>
__global__ void __launch_bounds__(128) k_lj_cells(View V, KArgs a) {
    __shared__ float s_lj1[kMaxTypes * kMaxTypes], s_lj2[kMaxTypes * kMaxTypes];
    __shared__ double s_ftm[kMaxTypes];
    const int np = V.ntypes * V.ntypes;
    for (int k = threadIdx.x; k < np; k += blockDim.x) { s_lj1[k] = V.tab->lj1f[k]; s_lj2[k] = V.tab->lj2f[k]; }
    if (threadIdx.x < kMaxTypes) s_ftm[threadIdx.x] = V.tab->ftm_m[threadIdx.x];
    extern __shared__ float4 s_rec[];
    const int tmode = begin_tile(V, 1, s_rec);
    __syncthreads();
    const unsigned err = V.ctl->err;
    const int rem = (a.mode == kModeStep) ? V.ctl->remaining : 0;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int t = blockIdx.x;
    LJPair<MT, 0, 0> pr;
    pr.V = &V;
    pr.lj1 = s_lj1; pr.lj2 = s_lj2;
    pr.c1 = s_lj1[0]; pr.c2 = s_lj2[0];
    pr.rc2 = V.rc2f;
    pr.nt = V.ntypes;
    pr.n = V.n_pad;
    pr.ti = 0;
    pr.near_min = 3.0e38f;  // no list entries here: FP32 cut-off decisions
    pr.ax.zero(); pr.ay.zero(); pr.az.zero();
    bool valid = false;
    if (p < V.n_pad && err == 0 && tmode >= 0) {
        const Rep &R = V.rep[V.tile_rep[p >> 5]];
        valid = (p - R.atom0) < R.natoms;
        if (valid) {
            float xi, yi, zi;
            load_rec(V, p, xi, yi, zi, pr.ti);
            const int bk = V.bpk[p];
            const int bx = unpack_bx(bk), by = unpack_by(bk), bz = unpack_bz(bk);
            const int nbx = R.nb[0], nby = R.nb[1], nbz = R.nb[2];
            const float hx = R.hf[0], hy = R.hf[1], hz = R.hf[2];
            const int4 box = V.tile_box[t];
            const int bdx = box.w & 0xffff, bdy = box.w >> 16;
            const int ncell = V.tile_ncell[t], tot = V.tile_cnt[t];
            for (int k = 0; k < 27; ++k) {
                const int row = k / 3;
                const int ox = k - 3 * row - 1, oy = row % 3 - 1, oz = row / 3 - 1;
                // this stencil cell's records: staged (offset, count) or global (first slot, count)
                int first, cnt, base;
                if (tmode == 1) {
                    int idx = (bx + ox - box.x) + bdx * ((by + oy - box.y) + bdy * (bz + oz - box.z));
                    idx = min(max(idx, 0), kTileBox - 1);
                    const unsigned wd = V.tile_bits[(size_t)t * 32 + (idx >> 5)];
                    int kc = V.tile_wpre[(size_t)t * 32 + (idx >> 5)] + __popc(wd & ((1u << (idx & 31)) - 1u));
                    kc = min(kc, ncell - 1);
                    first = V.tile_off[(size_t)t * kTileCells + kc];
                    const int nxt = kc + 1 < ncell ? V.tile_off[(size_t)t * kTileCells + kc + 1] : tot;
                    cnt = min(nxt, kTileCap) - first;
                    base = V.tile_first[(size_t)t * kTileCells + kc];
                } else {
                    int cx = bx + ox, cy = by + oy, cz = bz + oz;
                    cx += (cx < 0) ? nbx : ((cx >= nbx) ? -nbx : 0);
                    cy += (cy < 0) ? nby : ((cy >= nby) ? -nby : 0);
                    cz += (cz < 0) ? nbz : ((cz >= nbz) ? -nbz : 0);
                    const int gb = V.lin2bin[R.bin0 + (cz * nby + cy) * nbx + cx];
                    first = V.bin_start[gb];
                    cnt = V.bin_count[gb];
                    base = first;
                }
                const float sx = ox * hx, sy = oy * hy, sz = oz * hz;
                const int self = (k == 13) ? p - base : -1;  // the atom itself, centre image
                for (int l0 = 0; l0 < cnt; l0 += 4) {
                    pr.round_begin();
                    for (int l = l0; l < l0 + 4 && l < cnt; ++l) {
                        const float4 r4 = (tmode == 1) ? s_rec[(first + l) & (kTileCap - 1)] : V.rec[first + l];
                        if (l == self) continue;
                        const float dx = xi - r4.x - sx, dy = yi - r4.y - sy, dz = zi - r4.z - sz;
                        pr(0u, dx, dy, dz, dx * dx + dy * dy + dz * dz, __float_as_int(r4.w));
                    }
                    pr.round_end();
                }
            }
        }
    }
    if (valid) epilogue(V, a.mode, rem, p, pr.ti, pr.ax.value(), pr.ay.value(), pr.az.value(), s_ftm);
}

void cells_force_sequence(const View &V, int mode, std::vector<KCall> &seq) {
    KArgs a{};
    a.mode = mode;
    const void *fn = V.ntypes > 1 ? (const void *)k_lj_cells<1> : (const void *)k_lj_cells<0>;
    seq.push_back(KCall{fn, dim3((unsigned)V.n_ftiles), dim3(128), kTileSmem, a});
}

// Memory-only twin of the mixed full-list force pass, for measuring the
// ceiling of its access pattern: the same list walk and record gathers, the
// same velocity read/write (with a zero increment), but three additions per
// pair instead of the pair arithmetic and compensated sums.
struct GatherPair {
    static constexpr bool kPacked = false;
    float acc;
    __device__ __forceinline__ void round_begin() {}
    __device__ __forceinline__ void round_end() {}
    __device__ __forceinline__ void operator()(uint32_t, float dx, float dy, float dz, float, int) { acc += dx + dy + dz; }
};

template <int T, int Q>
__global__ void __launch_bounds__(256, 4) k_gather_probe(View V, KArgs a) {
    extern __shared__ float4 s_rec[];
    const int tmode = begin_tile(V, T, s_rec);
    __syncthreads();
    constexpr int A = 32 / T;
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int p = gw * A + lane / T;
    const int sub = lane & (T - 1);
    GatherPair pr;
    pr.acc = 0.f;
    bool valid = false;
    if (gw * A < V.n_pad && tmode >= 0) {
        const Rep &R = V.rep[V.n_rep == 1 ? 0 : V.tile_rep[p >> 5]];  // one replica: no lookup
        valid = (p - R.atom0) < R.natoms;
        if (valid) {
            const int cnt = V.ncount[p];
            float xi, yi, zi;
            int ti;
            load_rec(V, p, xi, yi, zi, ti);
            const uint32_t *lp = V.nlist + (size_t)gw * (size_t)(A * V.maxneigh) + lane * Q;
            walk_mode<T, Q>(V, tmode, lp, sub, cnt, xi, yi, zi, R, s_rec, pr);
        }
    }
    const double sum = group_sum<T>((double)pr.acc);
    if (valid && sub == 0) {
        const int n = V.n_pad;
        const double z = sum * 0.0;  // not foldable: sum may be NaN/Inf only if the state is
        V.v[p] += z;
        V.v[n + p] += z;
        V.v[2 * n + p] += z;
    }
}

template <int Q>
static const void *pick_probe_q(int T) {
    switch (T) {
        case 1: return (const void *)k_gather_probe<1, Q>;
        case 2: return (const void *)k_gather_probe<2, Q>;
        case 4: return (const void *)k_gather_probe<4, Q>;
        case 8: return (const void *)k_gather_probe<8, Q>;
        case 16: return (const void *)k_gather_probe<16, Q>;
        default: return (const void *)k_gather_probe<32, Q>;
    }
}

void gather_probe_sequence(const View &V, int block, std::vector<KCall> &seq) {
    KArgs a{};
    const long long threads = (long long)V.n_pad * V.tpa;
    const void *fn = V.vec == 4 ? pick_probe_q<4>(V.tpa) : (V.vec == 2 ? pick_probe_q<2>(V.tpa) : pick_probe_q<1>(V.tpa));
    const size_t sm = V.tile_atoms > 0 ? kTileSmem : 0;
    seq.push_back(KCall{fn, dim3((unsigned)((threads + block - 1) / block)), dim3(block), sm, a});
}

// zero F before a half-list pass
__global__ void k_zero_f(View V, KArgs a) {
    const int n3 = 3 * V.n_pad;
    if (V.ctl->err) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n3; i += gridDim.x * blockDim.x) V.f[i] = 0.0;
}

// kick after a half-list pass (F complete): mode as in the force epilogue;
// kModeEV adds the kinetic term
__global__ void k_kick(View V, KArgs a) {
    __shared__ double s_ftm[kMaxTypes];
    if (threadIdx.x < kMaxTypes) s_ftm[threadIdx.x] = V.tab->ftm_m[threadIdx.x];
    __syncthreads();
    const unsigned err = V.ctl->err;
    const int rem = (a.mode == kModeStep) ? V.ctl->remaining : 0;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < V.n_pad && err == 0) {
        const Rep &R = V.rep[V.tile_rep[p >> 5]];
        if (p - R.atom0 < R.natoms) {
            const int n = V.n_pad;
            const int t = V.type[p];
            if (a.mode == kModeStep || a.mode == kModeKickDry || a.mode == kModeHalfKick) {
                const double c = (a.mode == kModeKickDry) ? 0.0
                                 : (a.mode == kModeHalfKick || rem == 0 ? 0.5 : 1.0) * V.dt * s_ftm[t];
                V.v[p] += c * V.f[p];
                V.v[n + p] += c * V.f[n + p];
                V.v[2 * n + p] += c * V.f[2 * n + p];
            } else if (a.mode == kModeEV) {
                const double vx = V.v[p], vy = V.v[n + p], vz = V.v[2 * n + p];
                V.ev[n + p] = 0.5 * (vx * vx + vy * vy + vz * vz) / s_ftm[t];
            }
        }
    }
}

// --------------------------------------------------------------- EAM ----
// Finnis-Sinclair analytic EAM (the paper's App. A EAM benchmark; form
// rho = (rc-r)^2, F = -A sqrt(rho), phi = (rc-r)^2 (c0 + c1 r + c2 r^2)).

// pass 1: host density rho_i = sum_j (rc - r)^2 and the embedding derivative
// F'(rho_i) = -A / (2 sqrt(rho_i)) (0 at rho = 0), FP64 per atom
struct RhoPair {
    static constexpr bool kPacked = false;
    KahanF acc;
    float rc, rc2, part;
    __device__ __forceinline__ void round_begin() { part = 0; }
    __device__ __forceinline__ void round_end() { acc.add(part); }
    __device__ __forceinline__ float term(int) const { return part; }
    __device__ __forceinline__ void operator()(uint32_t, float, float, float, float r2, int) {
        const float r = r2 * rsqrtf(r2);  // branch-free: t = 0 beyond rc
        const float t = (r2 < rc2) ? rc - r : 0.f;
        part += t * t;
    }
};
// the same with x and y packed
struct PackedRho : RhoPair {
    static constexpr bool kPacked = true;
    __device__ __forceinline__ void operator()(f32x2, float dx, float dy, float dz, float r2, int t) {
        RhoPair::operator()(0u, dx, dy, dz, r2, t);
    }
};

// F'(rho_i) of atom p, and its embedding energy for an energy pass
__device__ __forceinline__ void finish_rho(const View &V, int mode, int p, double rho) {
    const double Aemb = V.tab->eam[1];
    // single element: the record's type slot is free until the next drift
    // rewrites it, so F'(rho) rides in rec.w and the force pass gathers
    // one 16-byte record per pair instead of two separate loads.  It is
    // stored as FP32, so it is formed in FP32 (one reciprocal square
    // root, a few FP32 ulps) rather than by an FP64 square root and
    // divide on the FP64 pipe for every atom
    const float rf = (float)rho;
    V.rec[p].w = rf > 0.f ? -0.5f * (float)Aemb * rsqrtf(rf) : 0.f;
    if (mode == kModeEV) V.emb[p] = rho > 0.0 ? -Aemb * sqrt(rho) : 0.0;
}

template <int T, int Q, int PACK>
__global__ void __launch_bounds__(256) k_eam_rho(View V, KArgs a) {
    extern __shared__ float4 s_rec[];
    const int tmode = begin_tile(V, T, s_rec);
    if (V.tile_atoms != 0) __syncthreads();  // only a staging block has shared state
    const unsigned err = V.ctl->err;
    constexpr int A = 32 / T;
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int p = gw * A + lane / T;
    const int sub = lane & (T - 1);
    std::conditional_t<PACK, PackedRho, RhoPair> pr;
    pr.acc.zero();
    pr.rc = V.tab->eamf[0];
    pr.rc2 = V.rc2f;
    bool valid = false;
    if (gw * A < V.n_pad && err == 0 && tmode >= 0) {
        const Rep &R = V.rep[V.tile_rep[p >> 5]];
        valid = (p - R.atom0) < R.natoms;
        if (valid) {
            const int cnt = V.ncount[p];
            float xi, yi, zi;
            int ti;
            load_rec(V, p, xi, yi, zi, ti);
            const uint32_t *lp = V.nlist + (size_t)gw * (size_t)(A * V.maxneigh) + lane * Q;
            walk_mode<T, Q>(V, tmode, lp, sub, cnt, xi, yi, zi, R, s_rec, pr);
        }
    }
    const double rho = group_sum<T>(pr.acc.value());
    if (valid && sub == 0) finish_rho(V, a.mode, p, rho);
}

// one warp's atoms of the density pass
template <int Q>
__device__ __forceinline__ void rho_wide_warp(const View &V, int mode, const Wide &w, WideAtom<Q> &at, const Rep &R,
                                              float (*s_round)[32]) {
    RhoPair pr;
    pr.rc = V.tab->eamf[0];
    pr.rc2 = V.rc2f;
    const bool valid = (w.p - R.atom0) < R.natoms;
    KahanF acc[1];
    acc[0].zero();
    walk_wide<Q, 1, 1>(V, w, R, valid ? at.count : 0, at, s_round, pr, acc);
    const double rho = wide_sum(w, acc[0].value());
    if (valid && w.sub == 0 && w.g == 0) finish_rho(V, mode, w.p, rho);
}

// the density pass of a small system (see walk_wide)
template <int Q>
__global__ void __launch_bounds__(kWideBlock) k_eam_rho_wide(View V, KArgs a) {
    __shared__ float s_round[kWideBlock / 32][1][32];
    const Wide w = wide_lane(V, a.aux, (blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (w.p >= V.n_pad) return;
    WideAtom<Q> at = load_wide<Q>(V, w);
    const Rep &R = V.rep[V.n_rep == 1 ? 0 : V.tile_rep[w.p >> 5]];
    if (at.err) return;
    rho_wide_warp<Q>(V, a.mode, w, at, R, s_round[threadIdx.x >> 5]);
}

// pass 2: F_i = -sum_j [phi'(r) + (F'_i + F'_j) rho'(r)] d / r
template <int EV>
struct EamPair {
    static constexpr bool kPacked = false;
    float rc, rc2, c0, c1, c2, fpi;
    KahanF ax, ay, az, e;
    KahanF w[6];
    float rx, ry, rz;  // this round's plain partial sums
    float re, rw[6];   // and of the energy and virial terms (EV)
    __device__ __forceinline__ void round_begin() {
        rx = 0; ry = 0; rz = 0;
        if (EV) {
            re = 0;
            for (int k = 0; k < 6; ++k) rw[k] = 0;
        }
    }
    __device__ __forceinline__ void round_end() {
        ax.add(rx); ay.add(ry); az.add(rz);
        if (EV) {
            e.add(re);
            for (int k = 0; k < 6; ++k) w[k].add(rw[k]);
        }
    }
    // the round's sums, in the order of the wide passes' terms
    __device__ __forceinline__ float term(int k) const {
        return k == 0 ? rx : k == 1 ? ry : k == 2 ? rz : k == 3 ? re : rw[k - 4];
    }
    // -(phi' + (F'_i + F'_j) rho') / r, branch-free: t = 0 beyond rc zeroes the term
    __device__ __forceinline__ float coefficient(float r2, int wj) const {
        const float fpj = __int_as_float(wj);
        const float rinv = rsqrtf(r2);
        const float r = r2 * rinv;
        const float t = (r2 < rc2) ? rc - r : 0.f;
        const float poly = c0 + r * (c1 + r * c2);
        const float dpoly = c1 + 2.f * c2 * r;
        return -t * (-2.f * poly + t * dpoly - 2.f * (fpi + fpj)) * rinv;
    }
    // wj: F'_j, which came with the record (rec.w, set by the density pass)
    __device__ __forceinline__ void operator()(uint32_t, float dx, float dy, float dz, float r2, int wj) {
        if constexpr (!EV) {
            const float coef = coefficient(r2, wj);
            rx += dx * coef; ry += dy * coef; rz += dz * coef;
            return;
        }
        if (r2 < rc2) {
            const float fpj = __int_as_float(wj);
            const float rinv = rsqrtf(r2);
            const float r = r2 * rinv;
            const float t = rc - r;
            const float poly = c0 + r * (c1 + r * c2);
            const float dpoly = c1 + 2.f * c2 * r;
            // -(phi' + (F'_i + F'_j) rho') / r with phi' = -2t poly + t^2 dpoly, rho' = -2t
            const float coef = -t * (-2.f * poly + t * dpoly - 2.f * (fpi + fpj)) * rinv;
            const float fxp = dx * coef, fyp = dy * coef, fzp = dz * coef;
            rx += fxp; ry += fyp; rz += fzp;
            if (EV) {
                const float h = 0.5f;
                re += h * t * t * poly;
                rw[0] += h * dx * fxp; rw[1] += h * dy * fyp; rw[2] += h * dz * fzp;
                rw[3] += h * dx * fyp; rw[4] += h * dx * fzp; rw[5] += h * dy * fzp;
            }
        }
    }
};

// The force-only pass with the x and y components' sums packed; what the
// walk leaves in the wrapped pair are the same sums.  Density and force passes of 80,000 atoms with the force
// pass scalar / packed 33.0 / 32.0 us, 500,000 with both scalar / packed 117.0 / 114.8 us.  (The
// LJ pass, which its gathers bound, is slower packed: 124.8 -> 135.2 us on
// 864,000 atoms, 126.1 .. 132 with only part of it packed or with more registers.)
struct PackedForce {
    using Base = EamPair<0>;
    static constexpr bool kPacked = true;
    Base &b;
    f32x2 rxy;
    KahanF2 axy;
    __device__ __forceinline__ explicit PackedForce(Base &base) : b(base) { axy.zero(); }
    __device__ __forceinline__ void round_begin() {
        rxy = 0ull;
        b.rz = 0.f;
    }
    __device__ __forceinline__ void round_end() {
        axy.add(rxy);
        b.az.add(b.rz);
    }
    __device__ __forceinline__ void operator()(f32x2 dxy, float, float, float dz, float r2, int tj) {
        const float f = b.coefficient(r2, tj);
        rxy = fma2(dxy, pack2(f, f), rxy);
        b.rz = fmaf(dz, f, b.rz);
    }
    __device__ __forceinline__ void finish() {
        b.ax = axy.first();
        b.ay = axy.second();
    }
};

template <int T, int Q, int EV>
__global__ void __launch_bounds__(256) k_eam_force(View V, KArgs a) {
    // single element: ftm2v/m is read where it is used, no table to stage, so
    // no block barrier either unless the block stages records
    const double *s_ftm = V.tab->ftm_m;
    extern __shared__ float4 s_rec[];
    const int tmode = begin_tile(V, T, s_rec);
    if (V.tile_atoms != 0) __syncthreads();
    const unsigned err = V.ctl->err;
    const int rem = (a.mode == kModeStep) ? V.ctl->remaining : 0;
    constexpr int A = 32 / T;
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int p = gw * A + lane / T;
    const int sub = lane & (T - 1);
    EamPair<EV> pr;
    pr.rc = V.tab->eamf[0]; pr.c0 = V.tab->eamf[2]; pr.c1 = V.tab->eamf[3]; pr.c2 = V.tab->eamf[4];
    pr.rc2 = V.rc2f;
    pr.fpi = 0;
    pr.ax.zero(); pr.ay.zero(); pr.az.zero(); pr.e.zero();
    for (int k = 0; k < 6; ++k) pr.w[k].zero();
    bool valid = false;
    int ti = 0;
    if (gw * A < V.n_pad && err == 0 && tmode >= 0) {
        const Rep &R = V.rep[V.tile_rep[p >> 5]];
        valid = (p - R.atom0) < R.natoms;
        if (valid) {
            const int cnt = V.ncount[p];
            float xi, yi, zi;
            load_rec(V, p, xi, yi, zi, ti);
            pr.fpi = __int_as_float(ti);
            const uint32_t *lp = V.nlist + (size_t)gw * (size_t)(A * V.maxneigh) + lane * Q;
            if constexpr (!EV) {
                PackedForce pk(pr);
                walk_mode<T, Q>(V, tmode, lp, sub, cnt, xi, yi, zi, R, s_rec, pk);
                pk.finish();
            } else {
                walk_mode<T, Q>(V, tmode, lp, sub, cnt, xi, yi, zi, R, s_rec, pr);
            }
        }
    }
    const double fx = group_sum<T>(pr.ax.value());
    const double fy = group_sum<T>(pr.ay.value());
    const double fz = group_sum<T>(pr.az.value());
    double e_acc = 0.0, w_acc[6] = {0, 0, 0, 0, 0, 0};
    if (EV) {
        e_acc = group_sum<T>(pr.e.value());
        for (int k = 0; k < 6; ++k) w_acc[k] = group_sum<T>(pr.w[k].value());
    }
    if (valid && sub == 0) {
        // single element (checked at creation): type 0 for the mass; the loaded
        // record's .w holds F'(rho), not a type
        epilogue(V, a.mode, rem, p, 0, fx, fy, fz, s_ftm);
        if (EV) write_ev(V, p, 0, e_acc + V.emb[p], w_acc, s_ftm);
    }
}

// one warp's atoms of the force pass
template <int Q, int EV>
__device__ __forceinline__ void eam_wide_warp(const View &V, int mode, int rem, const Wide &w, WideAtom<Q> &at,
                                              const Rep &R, float (*s_round)[32]) {
    constexpr int NT = EV ? 10 : 3, KT = (NT + 1) / 2;
    EamPair<EV> pr;
    pr.rc = V.tab->eamf[0]; pr.c0 = V.tab->eamf[2]; pr.c1 = V.tab->eamf[3]; pr.c2 = V.tab->eamf[4];
    pr.rc2 = V.rc2f;
    const bool valid = (w.p - R.atom0) < R.natoms;
    const double ftm = V.tab->ftm_m[0];  // single element
    pr.fpi = __int_as_float(at.t);
    KahanF acc[KT];
    for (int k = 0; k < KT; ++k) acc[k].zero();
    walk_wide<Q, NT, KT>(V, w, R, valid ? at.count : 0, at, s_round, pr, acc);
#pragma unroll
    for (int k = 0; k < KT; ++k) {
        const int term = w.g + (k << w.lg);
        const double x = wide_sum(w, acc[k].value());
        if (!valid || w.sub != 0) continue;
        if (term < 3) finish_component(V, mode, rem, term, w.p, ftm, x);
        else if (EV && term == 3) V.ev[w.p] = x + V.emb[w.p];
        else if (EV && term < NT) V.ev[(size_t)(term - 2) * V.n_pad + w.p] = x;
    }
    if (EV && valid && w.sub == 0 && w.g == 0) write_kinetic(V, w.p, ftm);
}

// the force pass of a small system (see walk_wide)
template <int Q, int EV>
__global__ void __launch_bounds__(kWideBlock) k_eam_force_wide(View V, KArgs a) {
    __shared__ float s_round[kWideBlock / 32][EV ? 10 : 3][32];
    const Wide w = wide_lane(V, a.aux, (blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (w.p >= V.n_pad) return;
    WideAtom<Q> at = load_wide<Q>(V, w);
    const Rep &R = V.rep[V.n_rep == 1 ? 0 : V.tile_rep[w.p >> 5]];
    if (at.err) return;
    eam_wide_warp<Q, EV>(V, a.mode, at.remaining, w, at, R, s_round[threadIdx.x >> 5]);
}

// ------------------------------------------------------- drift + control --

// x += dt v (after v += dt/2 a(F) on the first step of an md_step call);
// refresh the FP32 record; per-replica max displacement since the build, which
// k_drift_done turns into rebuild flags.  Mixed precision: two adjacent
// atoms per thread with 16-byte loads and stores (measured faster than one
// atom per thread, and half the blocks' atomics); FP64: one atom per thread.
template <int PREC>
__device__ __forceinline__ float drift_one(const View &V, int p, unsigned err, int first, int &rep) {
    const int n = V.n_pad;
    rep = V.n_rep == 1 ? 0 : V.tile_rep[p >> 5];
    const Rep &R = V.rep[rep];
    const int left = R.natoms - (p - R.atom0);
    double x[3], v[3];  // (loaded before anything is known: the checks' loads would come first otherwise)
    int t;
    if (PREC == MD_PREC_FP64) {
        const double4_32a q = V.pos4[p];
        x[0] = q.x; x[1] = q.y; x[2] = q.z;
        t = (int)__double_as_longlong(q.w);
    } else {
        for (int c = 0; c < 3; ++c) x[c] = V.xr[c * n + p];
        t = V.type[p];
    }
    for (int c = 0; c < 3; ++c) v[c] = V.v[c * n + p];
    const float4 b = V.recb[p];
    if (left <= 0 || err) return 0.f;  // a latched error: leave the state as it is
    if (first) {
        const double hk = 0.5 * V.dt * V.tab->ftm_m[t];
        for (int c = 0; c < 3; ++c) {
            v[c] += hk * V.f[c * n + p];
            V.v[c * n + p] = v[c];
        }
    }
    for (int c = 0; c < 3; ++c) x[c] += V.dt * v[c];
    const float4 nr = make_float4((float)x[0], (float)x[1], (float)x[2], __int_as_float(t));
    if (PREC == MD_PREC_FP64) {
        V.pos4[p] = make_double4_32a(x[0], x[1], x[2], __longlong_as_double((long long)t));
    } else {
        for (int c = 0; c < 3; ++c) V.xr[c * n + p] = x[c];
    }
    V.rec[p] = nr;  // FP64: the records that the force passes test first
    const float ex = nr.x - b.x, ey = nr.y - b.y, ez = nr.z - b.z;
    float d2 = ex * ex + ey * ey + ez * ez;
    if (!(d2 <= 3.0e38f)) d2 = __int_as_float(0x7f800000);  // NaN/Inf -> +Inf
    return d2;
}

// mixed precision: the adjacent atoms p, p+1 (p even, same replica) with
// 16-byte loads and stores of the FP64 arrays; the second atom may be padding,
// which is left untouched.  Returns the larger squared displacement.
__device__ __forceinline__ float drift_pair(const View &V, int p, unsigned err, int first, int &rep) {
    const int n = V.n_pad;
    rep = V.n_rep == 1 ? 0 : V.tile_rep[p >> 5];
    const Rep &R = V.rep[rep];
    const int left = R.natoms - (p - R.atom0);
    const bool two = left > 1;
    double2 x[3], v[3];  // (loaded before anything is known: the checks' loads would come first otherwise)
    for (int c = 0; c < 3; ++c) {
        x[c] = *(const double2 *)&V.xr[c * n + p];
        v[c] = *(const double2 *)&V.v[c * n + p];
    }
    const float4 b0 = V.recb[p], b1 = V.recb[p + 1];
    if (left <= 0 || err) return 0.f;  // a latched error: leave the state as it is
    const int2 t = make_int2(__float_as_int(b0.w), __float_as_int(b1.w));  // the build records hold the types
    if (first) {
        const double hk0 = 0.5 * V.dt * V.tab->ftm_m[t.x], hk1 = two ? 0.5 * V.dt * V.tab->ftm_m[t.y] : 0.0;
        for (int c = 0; c < 3; ++c) {
            const double2 f = *(const double2 *)&V.f[c * n + p];
            v[c].x += hk0 * f.x;
            v[c].y += hk1 * f.y;
            *(double2 *)&V.v[c * n + p] = v[c];
        }
    }
    for (int c = 0; c < 3; ++c) {
        x[c].x += V.dt * v[c].x;
        if (two) x[c].y += V.dt * v[c].y;
        *(double2 *)&V.xr[c * n + p] = x[c];
    }
    const float4 r0 = make_float4((float)x[0].x, (float)x[1].x, (float)x[2].x, __int_as_float(t.x));
    V.rec[p] = r0;
    // NaN/Inf -> +Inf for each atom before the maximum (fmaxf drops a NaN operand)
    float ex = r0.x - b0.x, ey = r0.y - b0.y, ez = r0.z - b0.z;
    float d2 = ex * ex + ey * ey + ez * ez;
    if (!(d2 <= 3.0e38f)) d2 = __int_as_float(0x7f800000);
    if (two) {
        const float4 r1 = make_float4((float)x[0].y, (float)x[1].y, (float)x[2].y, __int_as_float(t.y));
        V.rec[p + 1] = r1;
        ex = r1.x - b1.x; ey = r1.y - b1.y; ez = r1.z - b1.z;
        float d2b = ex * ex + ey * ey + ez * ez;
        if (!(d2b <= 3.0e38f)) d2b = __int_as_float(0x7f800000);
        d2 = fmaxf(d2, d2b);
    }
    return d2;
}

// Small blocks reach more SMs and drain sooner: us per step with 256 / 64 threads (128: as 64), 16,000 atoms 24.66 /
// 24.35, 32,771 28.33 / 28.07, 100,003 43.4 / 42.9, 864,000 209.3 / 208.2.
constexpr int kDriftBlock = 64;

template <int PREC>
__global__ void __launch_bounds__(kDriftBlock) k_drift(View V, KArgs a) {
    const unsigned err = V.ctl->err;
    const int first = V.ctl->first;
    if (blockIdx.x == 0 && threadIdx.x == 0) V.ctl->err_at_drift = err;  // for k_drift_done
    float d2 = 0.f;
    int rep = -1;
    const int t = blockIdx.x * kDriftBlock + threadIdx.x;
    if constexpr (PREC == MD_PREC_MIXED) {
        if (2 * t < V.n_pad) d2 = drift_pair(V, 2 * t, err, first, rep);  // two adjacent atoms per thread
    } else {
        if (t < V.n_pad) d2 = drift_one<PREC>(V, t, err, first, rep);
    }
    note_disp(V.rep_disp, V.skin_half2f, d2, rep);
}

// The step's bookkeeping after the drift, one block: the per-replica maximum
// displacement becomes the rebuild flags (and the count of replica rebuilds),
// the step is counted, the remaining count decremented and the graph's
// conditionals set.  A separate kernel rather than the drift's last block:
// the drift then takes no ticket (a fence and an atomic in each of its
// blocks).  The force pass of the step finds the remaining count already
// decremented (0 on the last step: the closing half kick).  If this step's
// rebuild overflows the list, its force pass skips, the next iteration's
// drift and this kernel see the latched error, change nothing (the rebuild
// flags stay for the host's recovery) and end the loop, and the host
// completes the step after growing the list.
__global__ void __launch_bounds__(256) k_drift_done(View V, KArgs a) {
    // everything thread 0 will need, loaded at once: one memory latency instead of four
    const unsigned err_at_drift = V.ctl->err_at_drift, err = V.ctl->err;
    int rem = V.ctl->remaining;
    const long long steps = V.ctl->steps, rebuilds = V.ctl->rebuilds;
    const unsigned m0 = (int)threadIdx.x < V.n_rep ? V.rep_disp[threadIdx.x] : 0u;
    if (err_at_drift != 0) {
        if (threadIdx.x == 0 && a.in_graph) {
            cudaGraphSetConditional(V.cond_rebuild, 0u);
            cudaGraphSetConditional(V.cond_loop, 0u);
        }
        return;
    }
    int any = 0, nflag = 0;
    bool bad = false;
    for (int q = threadIdx.x; q < V.n_rep; q += blockDim.x) {
        const unsigned m = q == (int)threadIdx.x ? m0 : V.rep_disp[q];
        V.rep_disp[q] = 0u;
        const bool nonfin = m >= 0x7f800000u;
        const int flag = (nonfin || __uint_as_float(m) > V.skin_half2f) ? 1 : 0;
        V.rep_flag[q] = flag;
        any |= flag;
        nflag += flag;
        bad |= nonfin;
    }
    if (bad) latch_error(V.ctl, kErrNonfinite);
    __shared__ int s_n[8];
    for (int o = 16; o > 0; o >>= 1) nflag += __shfl_xor_sync(0xffffffffu, nflag, o);
    if ((threadIdx.x & 31) == 0) s_n[threadIdx.x >> 5] = nflag;
    any = __syncthreads_or(any);
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        int tot = 0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) tot += s_n[k];
        V.ctl->first = 0;
        const bool ok = err == 0 && !bad;
        if (ok) {
            V.ctl->steps = steps + 1;
            V.ctl->rebuilds = rebuilds + tot;  // the builds this step's rebuild conditional runs
            if (rem > 0) V.ctl->remaining = --rem;
        }
        if (a.in_graph) {
            cudaGraphSetConditional(V.cond_rebuild, (any && ok) ? 1u : 0u);
            cudaGraphSetConditional(V.cond_loop, (rem > 0 && ok) ? 1u : 0u);
        }
    }
}

// Whole md_step steps of a small mixed system in one launch: a cluster of
// kStepsCtas blocks drifts, checks the displacements and evaluates forces step after
// step, with the cluster's hardware barrier between the phases, and returns when the
// steps are done or one of them needs a rebuild (which the graph then runs, with that
// step's force pass: the bookkeeping is k_drift_done's).  One step of a few
// thousand atoms in separate launches is four of them, each mostly its own
// start and its first loads.  The phases' arithmetic is k_drift's and
// the wide passes': the same trajectory bit for bit.  The blocks' flags go
// through distributed shared memory; positions, velocities and records are read with
// ordinary loads, ordered by the barriers (release / acquire).
constexpr int kStepsCtas = 16, kStepsThreads = 512;

template <int Q, int EAM, int MT>
__global__ void __cluster_dims__(kStepsCtas, 1, 1) __launch_bounds__(kStepsThreads, 1) k_steps(View V, KArgs a) {
    __shared__ float s_round[kStepsThreads / 32][3][32];
    __shared__ float s_tab[5][kMaxTypes * kMaxTypes];
    __shared__ int s_flag[kStepsCtas];
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const int lane = threadIdx.x & 31, cta = blockIdx.x;
    const unsigned err = V.ctl->err;
    int rem = V.ctl->remaining, first = V.ctl->first;
    if (err != 0) {  // latched before this launch: the same in every block
        if (cta == 0 && threadIdx.x == 0) {
            cudaGraphSetConditional(V.cond_rebuild, 0u);
            cudaGraphSetConditional(V.cond_loop, 0u);
        }
        return;
    }
    WideTab<MT> tab;
    if (!EAM) tab = wide_tab<MT>(V, s_tab);
    const Rep &R = V.rep[0];
    const int gtid = cta * kStepsThreads + threadIdx.x, gw0 = gtid >> 5;
    const int warps = (int)(((long long)V.n_pad << (V.ltpa + a.aux)) >> 5);
    constexpr int kThreads = kStepsCtas * kStepsThreads;
    cluster.sync();  // every block runs before its shared memory is written
    int done = 0, flags = 0;
    while (true) {
        float d2 = 0.f;
        for (int p = 2 * gtid; p < V.n_pad; p += 2 * kThreads) {
            int rep;
            d2 = fmaxf(d2, drift_pair(V, p, 0u, first, rep));
        }
        first = 0;
        // 1: an atom beyond skin/2, 2: a non-finite one (d2 = +Inf)
        int f = __syncthreads_or(d2 > V.skin_half2f) ? 1 : 0;
        if (f) f |= __syncthreads_or(__float_as_uint(d2) >= 0x7f800000u) ? 2 : 0;
        if (threadIdx.x < kStepsCtas) *cluster.map_shared_rank(&s_flag[cta], threadIdx.x) = f;
        cluster.sync();
        flags = __reduce_or_sync(0xffffffffu, lane < kStepsCtas ? s_flag[lane] : 0);
        if (flags) break;
        ++done;
        --rem;
        if constexpr (EAM) {
            for (int gw = gw0; gw < warps; gw += kThreads / 32) {
                const Wide w = wide_lane(V, a.aux, gw);
                WideAtom<Q> at = load_wide<Q>(V, w);
                rho_wide_warp<Q>(V, kModeStep, w, at, R, s_round[threadIdx.x >> 5]);
            }
            cluster.sync();
        }
        for (int gw = gw0; gw < warps; gw += kThreads / 32) {
            const Wide w = wide_lane(V, a.aux, gw);
            WideAtom<Q> at = load_wide<Q>(V, w);
            if constexpr (EAM) eam_wide_warp<Q, 0>(V, kModeStep, rem, w, at, R, s_round[threadIdx.x >> 5]);
            else lj_wide_warp<Q, 0, MT>(V, kModeStep, rem, gw, w, at, R, tab, s_round[threadIdx.x >> 5]);
        }
        cluster.sync();
        if (rem <= 0) break;
    }
    if (cta == 0 && threadIdx.x == 0) {
        const bool bad = flags & 2, rebuild = (flags & 1) && !bad;
        if (rebuild) {  // this step is counted; its rebuild and force pass follow
            ++done;
            --rem;
            V.ctl->rebuilds += 1;
        }
        if (bad) latch_error(V.ctl, kErrNonfinite);
        V.rep_flag[0] = flags ? 1 : 0;
        V.rep_disp[0] = 0u;
        V.ctl->first = 0;
        V.ctl->steps += done;
        V.ctl->remaining = rem;
        cudaGraphSetConditional(V.cond_rebuild, rebuild ? 1u : 0u);
        cudaGraphSetConditional(V.cond_loop, (rem > 0 && !bad) ? 1u : 0u);
    }
}

// before the WHILE node: loop while steps remain and no error is latched
__global__ void k_loop_init(View V, KArgs a) {
    if (threadIdx.x == 0 && blockIdx.x == 0)
        cudaGraphSetConditional(V.cond_loop, (V.ctl->remaining > 0 && V.ctl->err == 0) ? 1u : 0u);
}

// ------------------------------------------------------------- dispatch ----

template <int Q, int HALF, int EV, int MT>
static const void *pick_lj_t(int T) {
    switch (T) {
        case 1: return (const void *)k_lj<1, Q, HALF, EV, MT>;
        case 2: return (const void *)k_lj<2, Q, HALF, EV, MT>;
        case 4: return (const void *)k_lj<4, Q, HALF, EV, MT>;
        case 8: return (const void *)k_lj<8, Q, HALF, EV, MT>;
        case 16: return (const void *)k_lj<16, Q, HALF, EV, MT>;
        default: return (const void *)k_lj<32, Q, HALF, EV, MT>;
    }
}

template <int Q>
static const void *pick_lj_q(int T, int half, int ev, int mt) {
    if (half) {
        if (ev) return mt ? pick_lj_t<Q, 1, 1, 1>(T) : pick_lj_t<Q, 1, 1, 0>(T);
        return mt ? pick_lj_t<Q, 1, 0, 1>(T) : pick_lj_t<Q, 1, 0, 0>(T);
    }
    if (ev) return mt ? pick_lj_t<Q, 0, 1, 1>(T) : pick_lj_t<Q, 0, 1, 0>(T);
    return mt ? pick_lj_t<Q, 0, 0, 1>(T) : pick_lj_t<Q, 0, 0, 0>(T);
}

static const void *pick_lj(int T, int Q, int half, int ev, int mt) {
    if (Q == 4) return pick_lj_q<4>(T, half, ev, mt);
    if (Q == 2) return pick_lj_q<2>(T, half, ev, mt);
    return pick_lj_q<1>(T, half, ev, mt);
}

template <int Q, int PACK>
static const void *pick_rho_q(int T) {
    switch (T) {
        case 1: return (const void *)k_eam_rho<1, Q, PACK>;
        case 2: return (const void *)k_eam_rho<2, Q, PACK>;
        case 4: return (const void *)k_eam_rho<4, Q, PACK>;
        case 8: return (const void *)k_eam_rho<8, Q, PACK>;
        case 16: return (const void *)k_eam_rho<16, Q, PACK>;
        default: return (const void *)k_eam_rho<32, Q, PACK>;
    }
}

// The density pass with x and y packed has fewer instructions in a longer chain: from this many threads per SM
// (about the resident ones). Density plus force pass, scalar -> packed: 60,000 atoms 29.5 -> 30.4 us, 80,000 32.0 ->
// 33.2, 108,000 36.8 -> 36.8 (a step 46.0 -> 46.4), 150,000 62.7 -> 62.2 per step, 256,000 69.4 -> 67.7,
// 500,000 117.0 -> 115.0.
constexpr int kPackThreads = 900;

static const void *pick_rho(int T, int Q, bool pack) {
    if (Q == 4) return pack ? pick_rho_q<4, 1>(T) : pick_rho_q<4, 0>(T);
    if (Q == 2) return pack ? pick_rho_q<2, 1>(T) : pick_rho_q<2, 0>(T);
    return pack ? pick_rho_q<1, 1>(T) : pick_rho_q<1, 0>(T);
}

template <int Q, int EV>
static const void *pick_eamf_q(int T) {
    switch (T) {
        case 1: return (const void *)k_eam_force<1, Q, EV>;
        case 2: return (const void *)k_eam_force<2, Q, EV>;
        case 4: return (const void *)k_eam_force<4, Q, EV>;
        case 8: return (const void *)k_eam_force<8, Q, EV>;
        case 16: return (const void *)k_eam_force<16, Q, EV>;
        default: return (const void *)k_eam_force<32, Q, EV>;
    }
}

static const void *pick_eamf(int T, int Q, int ev) {
    if (Q == 4) return ev ? pick_eamf_q<4, 1>(T) : pick_eamf_q<4, 0>(T);
    if (Q == 2) return ev ? pick_eamf_q<2, 1>(T) : pick_eamf_q<2, 0>(T);
    return ev ? pick_eamf_q<1, 1>(T) : pick_eamf_q<1, 0>(T);
}

// log2 of the lanes that stand in for one thread of the list layout (walk_wide): as
// many as keep the whole system within kWideThreads threads per SM, at most
// sixteen.  us per step at 512 / 640 / 880-1024 / 2048 threads per SM: 4,000
// atoms 26.2 (8 lanes) / 26.0 (16), 16,000 atoms 28.9 (4) / 29.4 (8), 32,771 atoms 34.6 (2) / 32.5 (4) / 36
// (8); one lane: 31 .. 33.  32 lanes for the smallest systems measured the same as 16.
// Two lanes pay up to 640 threads per SM only (60,000 atoms: 36.9 us with one, 38.0 with two).
// Lanes beyond the rounds of the longest list only stand by and add to the terms' sums: none where there are as
// many lanes as rounds, and up to kWideIdle threads per SM where there would be more (EAM 4,000 atoms with 8 threads per
// atom, two or three rounds, 4 lanes / 2: 25.2 / 21.8 us per step, LJ 4,096 with 4 at rc 1.12, one round, 8 / 1: 22.8 / 20.3;
// but 5,000 atoms with lists of five rounds, 4 lanes / 8 21.0 / 19.9).
constexpr int kWideThreads = 880, kWideThreads2 = 640, kWideIdle = 300, kWideMost = 4;

int wide_lanes(const View &V) {
    if (V.prec != MD_PREC_MIXED || V.half || V.tile_atoms > 0) return 0;
    const int rounds = (V.list_most + (V.vec << V.ltpa) - 1) >> (V.ltpa + V.lvec);
    int lg = 0;
    while (lg < kWideMost && V.ltpa + lg < 5 && (1 << lg) < rounds &&
           ((long long)V.n_pad << (V.ltpa + lg + 1)) <= (long long)V.n_sm * ((2 << lg) <= rounds ? kWideThreads : kWideIdle))
        ++lg;
    if (lg == 1 && ((long long)V.n_pad << (V.ltpa + 1)) > (long long)V.n_sm * kWideThreads2) lg = 0;
    return lg;
}

#define PICK_WIDE(K, ...) \
    (V.vec == 4 ? (const void *)K<4, ##__VA_ARGS__> : V.vec == 2 ? (const void *)K<2, ##__VA_ARGS__> : (const void *)K<1, ##__VA_ARGS__>)

// the mixed pair passes: [LJ pass], or [density, force] for EAM
static void mixed_force_sequence(const View &V, int mode, int block, KArgs a, std::vector<KCall> &seq) {
    const int T = V.tpa;
    const int ev = (mode == kModeEV) ? 1 : 0;
    const int lg = wide_lanes(V);
    if (lg > 0) {
        a.aux = lg;
        const dim3 grid((unsigned)((((long long)V.n_pad << (V.ltpa + lg)) + kWideBlock - 1) / kWideBlock));
        if (V.pot == MD_POT_LJ) {
            const void *fn = V.ntypes > 1 ? (ev ? PICK_WIDE(k_lj_wide, 1, 1) : PICK_WIDE(k_lj_wide, 0, 1))
                                          : (ev ? PICK_WIDE(k_lj_wide, 1, 0) : PICK_WIDE(k_lj_wide, 0, 0));
            seq.push_back(KCall{fn, grid, dim3(kWideBlock), 0, a});
        } else {
            KArgs ar = a;
            ar.in_graph = 0;
            seq.push_back(KCall{PICK_WIDE(k_eam_rho_wide), grid, dim3(kWideBlock), 0, ar});
            seq.push_back(KCall{ev ? PICK_WIDE(k_eam_force_wide, 1) : PICK_WIDE(k_eam_force_wide, 0), grid,
                                dim3(kWideBlock), 0, a});
        }
        return;
    }
    const long long threads = (long long)V.n_pad * T;
    const dim3 grid((unsigned)((threads + block - 1) / block));
    const size_t sm = V.tile_atoms > 0 ? kTileSmem : 0;
    if (V.pot == MD_POT_LJ) {
        seq.push_back(KCall{pick_lj(T, V.vec, V.half, ev, V.ntypes > 1 ? 1 : 0), grid, dim3(block), sm, a});
    } else {
        KArgs ar = a;
        ar.in_graph = 0;
        seq.push_back(KCall{pick_rho(T, V.vec, threads >= (long long)V.n_sm * kPackThreads), grid, dim3(block), sm, ar});
        seq.push_back(KCall{pick_eamf(T, V.vec, ev), grid, dim3(block), sm, a});
    }
}

void force_sequence(const View &V, int mode, int block, bool in_graph, std::vector<KCall> &seq) {
    KArgs a{};
    a.mode = mode;
    a.in_graph = in_graph ? 1 : 0;
    KArgs af = a;
    if (V.half) {  // the kick and the closing store follow in k_kick, once F is complete
        seq.push_back(KCall{(const void *)k_zero_f, dim3((3 * V.n_pad + 255) / 256), dim3(256), 0, a});
        af.mode = kModeStoreF;
        af.in_graph = 0;
    }
    if (V.prec == MD_PREC_FP64) fp64_force_sequence(V, mode, af, seq);
    else mixed_force_sequence(V, mode, block, af, seq);
    if (V.half) seq.push_back(KCall{(const void *)k_kick, dim3((V.n_pad + 255) / 256), dim3(256), 0, a});
}

void drift_sequence(const View &V, bool in_graph, std::vector<KCall> &seq) {
    KArgs a{};
    a.in_graph = in_graph ? 1 : 0;
    if (V.prec == MD_PREC_FP64)
        seq.push_back(KCall{(const void *)k_drift<MD_PREC_FP64>,
                            dim3((V.n_pad + kDriftBlock - 1) / kDriftBlock), dim3(kDriftBlock), 0, a});
    else  // two atoms per thread
        seq.push_back(KCall{(const void *)k_drift<MD_PREC_MIXED>, dim3((V.n_pad / 2 + kDriftBlock - 1) / kDriftBlock),
                            dim3(kDriftBlock), 0, a});
    seq.push_back(KCall{(const void *)k_drift_done, dim3(1), dim3(256), 0, a});
}

// Which systems run their steps in k_steps.  Two things decide, since the rest of the chip stands idle meanwhile:
//   * the turns that the cluster's 8,192 threads take through a pass, at two lanes or more per thread of the list
//     layout: at most two.  us per step in separate launches / in k_steps (a rebuild every ~8), LJ at rc 2.5, one
//     turn: 500 atoms 20.4 / 12.5, 4,096 22.8 / 20.3; two: 2,000 atoms with 4 threads per atom 21.1 / 18.2, 4,096
//     with 2 23.3 / 21.7, 1,000 with 8 21.4 / 18.7 (rc 4.0 30.4 / 30.2); three: 1,500 with 8 21.2 / 21.6 (rc 3.2
//     25.1 / 26.1), 3,000 with 4 22.8 / 23.0; four: 4,096 with 4 24.0 / 26.3; 4,096 with 16 24.5 / 60.7;
//   * the list slots of all its passes, two for EAM (the list's capacity is 128 per atom at rc 2.5): with more of them
//     the lanes left per thread get few and walk longer lists.  EAM 2,048 atoms 19.6 / 15.5, with 4 threads per atom
//     21.1 / 19.7, 2,916 20.0 / 21.5, 4,000 21.1 / 21.6; LJ 5,000 atoms 23.5 / 28.1.
// Clusters of eight blocks: LJ 500, 4,000 and 5,000 atoms 13.5, 19.2 and 28.6.
constexpr int kStepsMost = 4096 * 128, kStepsTurns = 2;

bool steps_sequence(const View &V, std::vector<KCall> &seq) {
    // (at least two lanes per thread of the list layout)
    const int passes = V.pot == MD_POT_EAM_FS ? 2 : 1;
    if (V.prec != MD_PREC_MIXED || V.n_rep != 1 || V.half || V.tile_atoms > 0 || V.ltpa >= 5 ||
        (long long)V.n_pad * V.maxneigh * passes > kStepsMost ||
        ((long long)V.n_pad << (V.ltpa + 1)) > (long long)kStepsTurns * kStepsCtas * kStepsThreads)
        return false;
    KArgs a{};
    a.in_graph = 1;
    a.aux = 1;
    while (a.aux < kWideMost && V.ltpa + a.aux < 5 &&
           ((long long)V.n_pad << (V.ltpa + a.aux + 1)) <= kStepsCtas * kStepsThreads)
        ++a.aux;
    const void *fn = V.pot == MD_POT_EAM_FS ? PICK_WIDE(k_steps, 1, 0)
                     : V.ntypes > 1         ? PICK_WIDE(k_steps, 0, 1)
                                            : PICK_WIDE(k_steps, 0, 0);
    // a cluster of 16 needs the function's consent and a GPU that can place it
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kStepsCtas);
    cfg.blockDim = dim3(kStepsThreads);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kStepsCtas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) != cudaSuccess || clusters < 1) {
        cudaGetLastError();
        return false;
    }
    seq.push_back(KCall{fn, dim3(kStepsCtas), dim3(kStepsThreads), 0, a});
    return true;
}

void kick_sequence(const View &V, int mode, std::vector<KCall> &seq) {
    KArgs a{};
    a.mode = mode;
    seq.push_back(KCall{(const void *)k_kick, dim3((V.n_pad + 255) / 256), dim3(256), 0, a});
}

void loop_init_sequence(const View &V, std::vector<KCall> &seq) {
    KArgs a{};
    a.in_graph = 1;
    seq.push_back(KCall{(const void *)k_loop_init, dim3(1), dim3(32), 0, a});
}

}  // namespace md
