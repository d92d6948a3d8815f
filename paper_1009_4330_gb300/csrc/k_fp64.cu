// k_fp64.cu -- the passes over the Verlet list whose pair terms are double
// precision: the forces of the plain FP64 mode (LJ full and half list, EAM
// density and force) and, in both precision modes, the force-matching
// backward passes (LJ, EAM).
//
// GB300 issues 2 FP64 lanes per clock and SM, 1/64 of its FP32 rate: one warp
// FP64 instruction (conversions between double and float or int included)
// holds the pipe for 16 clocks, in which the SM could issue 64 others.  So
// these passes are bound by the number of FP64 instructions, and everything
// that can be done in FP32 or integers is:
//   * a list entry is first tested in FP32 on the 16-byte records (cut-off
//     plus a margin far above the FP32 error).  Only the entries that pass, ~70 % (the
//     list reaches rc + skin), are queued in shared memory and evaluated in FP64, eight
//     lanes to an atom (short lists: all of a warp's in one queue), so that the FP64
//     instructions run with full warps;
//   * x_i plus the stencil cell's shift is formed once per atom (3 values per
//     axis, in shared memory), which leaves one FP64 subtraction per
//     component of d;
//   * the FP64 <-> FP32 moves around the reciprocal (square root) seeds and
//     the exact cut-off comparison are integer operations on the words of the
//     double.
// 17 FP64 instructions per evaluated LJ pair instead of 28 per list entry, with the
// FP64 pipe 79-86 % busy.  Against one pass of FP64 arithmetic over every
// entry (time per pass): LJ 256,000 atoms, half list 994 -> 443 us; LJ 4,000
// atoms 30.6 -> 19 us; EAM 108,000 atoms (density + force) 863 -> 366 us; backward
// LJ 32,768 atoms, two types 534 -> 195 us, EAM 108,000 atoms 1,337 -> 728 us.
//
// The atoms are dealt out evenly, in units of four, to one wave of one-warp
// blocks (at most 20 per SM): a second, partly filled wave cost up to 30 % of
// a pass.  A warp works through its range in batches of at most 32 atoms, in four
// groups of eight lanes; a group takes the batch's next atom as soon as it is
// done with one and does not wait for the others (its lanes' partial sums go
// to shared memory), so that lists of different lengths even out.  The k-th
// accepted entry of an atom's list is always summed by lane k mod 8, in list order, and the
// eight partial sums are added in one fixed tree: the result does not depend
// on how the atoms are dealt out, on the list layout (threads per atom, vector width)
// or on the other atoms.
#include <algorithm>
#include <type_traits>

#include "md_common.cuh"
#include "md_kernels.h"

namespace md {

constexpr int kGrp = 8;       // lanes per atom
constexpr int kGroups = 4;    // groups per warp
constexpr int kRing = 64;     // queued entries per group: < 32 left + one fill of at most 32
constexpr int kBatchAtoms = 32;
constexpr int kSumStride = kBatchAtoms + 1;
constexpr int kUnit = 4;      // atoms per dealt unit
constexpr unsigned kFull = 0xffffffffu;
constexpr float kScreen = 1.0009765625f;  // entries are screened at 2^-10 above rc^2: far beyond the FP32 error of r^2
// Warps per SM of the one wave: 20 (at most 96 registers) for the LJ and EAM
// density passes without energies, 16 for the others.  32,000 / 256,000-atom LJ pass: 84.4 /
// 523 us with 16, 74.4 / 515 with 20, 91.0 / 596 with 12 (EAM backward: 844, 863, 818).
// Systems of U = 4 fill at most 16 warps per SM and are compiled for as many: with more than 128 registers a
// part of them made a second wave (LJ backward, two types, 9,700 atoms 92 -> 69 us).
constexpr int kWarpsMany = 20, kWarpsFew = 16;

// shared memory of a warp with NS sums per lane:
//   uint32 ring[4][64]; double xs[32][9]; double sums[NS * 8][33]
constexpr size_t kSumsAt = (size_t)kGroups * kRing * 4 + (size_t)kBatchAtoms * 9 * 8;
constexpr size_t fp64_smem(int NS) { return kSumsAt + (size_t)NS * kGrp * kSumStride * 8; }

// where the FP64 positions come from: the FP64 mode's pos4, or the backward
// passes' packed records (64 bytes per atom: x, y, z, a | gx, gy, gz, b)
struct SrcPos4 {
    static constexpr bool packed = false;
};
struct SrcPack {
    static constexpr bool packed = true;
};

template <class Src>
__device__ __forceinline__ double4_32a load_pos(const View &V, int j) {
    if constexpr (Src::packed) return V.bpack[2 * (size_t)j];
    else return V.pos4[j];
}

// Q consecutive list entries (streamed: each is read once per pass)
template <int Q>
__device__ __forceinline__ void load_chunk(const uint32_t *p, uint32_t (&e)[Q]) {
    if constexpr (Q == 4) {
        const uint4 u = __ldcs(reinterpret_cast<const uint4 *>(p));
        e[0] = u.x; e[1] = u.y; e[2] = u.z; e[3] = u.w;
    } else if constexpr (Q == 2) {
        const uint2 u = __ldcs(reinterpret_cast<const uint2 *>(p));
        e[0] = u.x; e[1] = u.y;
    } else {
        e[0] = __ldcs(p);
    }
}

__device__ __forceinline__ bool below(double r2, double rc2) {
    // r2 >= 0 (or NaN, whose bits are above every number's): the order of the bits
    return (unsigned long long)__double_as_longlong(r2) < (unsigned long long)__double_as_longlong(rc2);
}

// first entry of slot p's list
__device__ __forceinline__ const uint32_t *list_of(const View &V, int p, int Q) {
    const int la = 5 - V.ltpa;
    return V.nlist + (size_t)(p >> la) * ((size_t)V.maxneigh << la) + (size_t)((p & ((1 << la) - 1)) << V.ltpa) * Q;
}

// The walk of a batch with short lists (a gas): at most eight entries an atom, kShortPairs in all.  Each lane tests its own atom's
// entries, all atoms' accepted ones share one queue, and the warp evaluates it 32 pairs at a time.  As pair k of an
// atom is the only one of its partial sum k, each is stored as it comes: the same bits as the groups' walk below, which such
// lists leave mostly idle (eight lanes for one or two pairs, ~75 instructions an atom).  us per LJ pass of 256,000 atoms at
// density 0.005 / 0.02 / 0.05 (full list) groups 30.3 / 63.5 / 95.8, so 24.6 /
// 36.8 / 71.7.  The backward passes keep to the groups: the second walk cost them registers (EAM 6,912 atoms 80 -> 95
// us), and so do systems small enough for U = 4.
constexpr int kShortPairs = kGroups * kRing / 2;
template <class Src, int Q, class Pair>
__device__ __forceinline__ void short_walk(const View &V, const Rep &R, int p0, int cnt, int most, char *smem, Pair &pair) {
    const int lane = threadIdx.x;
    uint2 *const queue = reinterpret_cast<uint2 *>(smem);  // entry; atom of the batch and index among its accepted
    const double *const xs = reinterpret_cast<const double *>(smem + kGroups * kRing * 4);
    double *const sums = reinterpret_cast<double *>(smem + kSumsAt);
#pragma unroll
    for (int k = 0; k < Pair::kSums * kGrp; ++k) sums[k * kSumStride + lane] = 0.0;
    const float hx = R.hf[0], hy4 = R.hf[1] * 0.25f, hz16 = R.hf[2] * 0.0625f;
    const float keep2 = V.rc2f * kScreen;
    const int p = p0 + lane, lt = V.ltpa;
    const uint32_t *const lp = list_of(V, p, Q);
    float4 ri = make_float4(0.f, 0.f, 0.f, 0.f);
    if (cnt > 0) ri = V.rec[p];
    int mine = 0, total = 0;
    for (int k0 = 0; k0 < most; k0 += Q) {
        uint32_t e[Q];
        float4 rj[Q];
        const int left = cnt - k0;
        if (left > 0) {
            const int c = k0 / Q;
            load_chunk<Q>(lp + (size_t)(c >> lt) * (32 * Q) + (c & ((1 << lt) - 1)) * Q, e);
#pragma unroll
            for (int q = 0; q < Q; ++q)
                if (q < left) {
                    if (V.tile_atoms) e[q] = ((uint32_t)entry_slot(V, p, e[q]) << 6) | (e[q] & 63u);
                    rj[q] = __ldg(&V.rec[entry_j(e[q])]);
                }
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            bool acc = false;
            if (q < left) {
                const float dx = fmaf(-code_x(e[q]), hx, ri.x - rj[q].x);
                const float dy = fmaf(-code_y4(e[q]), hy4, ri.y - rj[q].y);
                const float dz = fmaf(-code_z16(e[q]), hz16, ri.z - rj[q].z);
                acc = fmaf(dz, dz, fmaf(dy, dy, dx * dx)) < keep2;
            }
            const unsigned b = __ballot_sync(kFull, acc);
            if (acc) {
                queue[total + __popc(b & ((1u << lane) - 1u))] = make_uint2(e[q], (unsigned)(mine << 5 | lane));
                ++mine;
            }
            total += __popc(b);
        }
    }
    __syncwarp();
    for (int i = lane; i - lane < total; i += 32) {
        const bool on = i < total;
        const uint2 q = on ? queue[i] : make_uint2(((uint32_t)p0 << 6) | kSelfCode, 0u);
        const int a = q.y & 31u;
        pair.begin(V, p0 + a);
        const double4_32a xj = load_pos<Src>(V, entry_j(q.x));
        const double *const x = xs + a * 9;
        const double dx = x[q.x & 3u] - xj.x, dy = x[3 + ((q.x >> 2) & 3u)] - xj.y, dz = x[6 + ((q.x >> 4) & 3u)] - xj.z;
        pair(V, q.x, on, dx, dy, dz, fma(dz, dz, fma(dy, dy, dx * dx)), xj.w);
        if (on) pair.store(sums + a, (int)(q.y >> 5));
    }
    __syncwarp();
}

// The walk over the lists of a batch: atoms p0 .. p0 + nb - 1 (nb <= 32, one replica).
// U: pairs in flight per lane.  A lane's FP64 chain is ~13 dependent
// instructions; with 16 warps per SM other warps fill the pipe (U = 1), a system
// too small for that evaluates up to four pairs per lane at once.
// Pair, zero-initialised (a group that gets no atom evaluates its lanes' idle pairs all the same), supplies
//   kSums                                  sums per lane
//   begin(V, p)                            per-atom values of slot p, sums zeroed
//   operator()(V, e, on, dx, dy, dz, r2, w)   one pair per lane (on: this lane has one)
//   store(sums, cls)                       this lane's partial sums -> shared memory
template <class Src, int Q, int U, class Pair>
__device__ __forceinline__ void fp64_walk(const View &V, const Rep &R, int p0, int nb, char *smem, Pair &pair) {
    const int lane = threadIdx.x, grp = lane >> 3, cls = lane & 7;
    uint32_t *const ring = reinterpret_cast<uint32_t *>(smem) + grp * kRing;
    double *const xs = reinterpret_cast<double *>(smem + kGroups * kRing * 4);
    double *const sums = reinterpret_cast<double *>(smem + kSumsAt);
    constexpr bool kShort = !Src::packed && U == 1;  // batches of short lists are walked by short_walk
    int count = 0;  // (loaded with the positions)
    if (kShort && lane < nb) count = V.ncount[p0 + lane];
    // x_i shifted into the frames of the neighbouring cells: dx = -1, 0, 1 -> x_i + h, x_i, x_i - h
    for (int k = lane; k < 3 * nb; k += 32) {
        const int i = k / 3, c = k - 3 * i;
        const double x = reinterpret_cast<const double *>(Src::packed ? &V.bpack[2 * (size_t)(p0 + i)] : &V.pos4[p0 + i])[c];
        xs[3 * k] = x + R.h[c];
        xs[3 * k + 1] = x;
        xs[3 * k + 2] = x - R.h[c];
    }
    __syncwarp();
    if constexpr (kShort) {
        const int most = __reduce_max_sync(kFull, count);
        if (most <= kGrp && __reduce_add_sync(kFull, count) <= kShortPairs) {
            short_walk<Src, Q>(V, R, p0, count, most, smem, pair);
            return;
        }
    }
    const float hx = R.hf[0], hy4 = R.hf[1] * 0.25f, hz16 = R.hf[2] * 0.0625f;
    const float keep2 = V.rc2f * kScreen;
    const int lt = V.ltpa;
    const unsigned gmask = 0xffu << (grp * kGrp), lower = (1u << cls) - 1u;

    int a = grp, next = kGroups;  // this group's atom; the first atom not taken yet
    bool active = a < nb;
    int p = p0 + a, cnt = 0, k0 = 0, head = 0, fill = 0;
    const uint32_t *lp = V.nlist;
    float xi = 0.f, yi = 0.f, zi = 0.f;
    uint32_t nxt[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) nxt[q] = 0u;

    // this lane's chunk of the next fill (entries k0 + cls Q ...)
    auto prefetch = [&]() {
        const int k = k0 + cls * Q;
        if (k < cnt) {
            const int c = k / Q;  // Q is a power of two
            load_chunk<Q>(lp + (size_t)(c >> lt) * (32 * Q) + (c & ((1 << lt) - 1)) * Q, nxt);
        }
    };
    auto start = [&]() {  // the group's next atom
        p = p0 + a;
        cnt = V.ncount[p];
        const float4 r = V.rec[p];
        xi = r.x; yi = r.y; zi = r.z;
        lp = list_of(V, p, Q);
        k0 = 0;
        head = 0;
        fill = 0;
        pair.begin(V, p);
        prefetch();
    };
    if (active) start();

    while (true) {
        // fill: one chunk per lane until every group has U entries per lane or its list is used up;
        // groups that have room for a chunk join in, and so fill less often on their own (LJ, 32,000
        // / 256,000 atoms, half list: 81.7 -> 77.6 / 464.7 -> 456.5 us)
        bool need = active && k0 < cnt && fill - head < kGrp * U;
        while (__any_sync(kFull, need)) {
            need = active && k0 < cnt && fill - head <= kRing - kGrp * Q;
            const int left = need ? cnt - (k0 + cls * Q) : 0;
            uint32_t e[Q];
            float4 rj[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                e[q] = nxt[q];
                if (q < left) {
                    if (V.tile_atoms) e[q] = ((uint32_t)entry_slot(V, p, e[q]) << 6) | (e[q] & 63u);
                    rj[q] = __ldg(&V.rec[entry_j(e[q])]);
                }
            }
            if (need) {
                k0 += kGrp * Q;
                prefetch();
            }
            unsigned acc = 0u;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                if (q < left) {
                    const float dx = fmaf(-code_x(e[q]), hx, xi - rj[q].x);
                    const float dy = fmaf(-code_y4(e[q]), hy4, yi - rj[q].y);
                    const float dz = fmaf(-code_z16(e[q]), hz16, zi - rj[q].z);
                    if (fmaf(dz, dz, fmaf(dy, dy, dx * dx)) < keep2) acc |= 1u << q;
                }
            }
            // list order: the lower lanes' accepted entries, then this lane's own
            int before = 0, total = 0;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const unsigned b = (__ballot_sync(kFull, (acc >> q) & 1u) & gmask) >> (grp * kGrp);
                before += __popc(b & lower);
                total += __popc(b);
            }
            int at = fill + before;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                if ((acc >> q) & 1u) {
                    ring[at & (kRing - 1)] = e[q];
                    ++at;
                }
            }
            fill += total;
            need = active && k0 < cnt && fill - head < kGrp * U;
        }
        __syncwarp();
        if (!__any_sync(kFull, active)) break;
        const int mine = active ? fill - head - cls : 0;  // this lane has pairs u with 8 u < mine
        // an idle lane evaluates its atom with itself (and drops it)
        const uint32_t self = ((uint32_t)(active ? p : p0) << 6) | kSelfCode;
        const double *const x = xs + (active ? a : 0) * 9;
        auto run = [&](auto count) {
            constexpr int C = decltype(count)::value;
            uint32_t e[C];
            double4_32a q[C];
#pragma unroll
            for (int u = 0; u < C; ++u) {
                e[u] = u * kGrp < mine ? ring[(head + u * kGrp + cls) & (kRing - 1)] : self;
                q[u] = load_pos<Src>(V, entry_j(e[u]));
            }
#pragma unroll
            for (int u = 0; u < C; ++u) {
                const bool on = u * kGrp < mine;
                const double dx = x[e[u] & 3u] - q[u].x;
                const double dy = x[3 + ((e[u] >> 2) & 3u)] - q[u].y;
                const double dz = x[6 + ((e[u] >> 4) & 3u)] - q[u].z;
                pair(V, e[u], on, dx, dy, dz, fma(dz, dz, fma(dy, dy, dx * dx)), q[u].w);
            }
        };
        if (U == 4 && __any_sync(kFull, mine > 2 * kGrp)) run(std::integral_constant<int, U>());
        else if (U == 4 && __any_sync(kFull, mine > kGrp)) run(std::integral_constant<int, U == 4 ? 2 : 1>());
        else if (__any_sync(kFull, mine > 0)) run(std::integral_constant<int, 1>());
        head += kGrp * U;
        // groups whose atom is done take the batch's next ones
        const bool done = active && k0 >= cnt && head >= fill;
        const unsigned m = __ballot_sync(kFull, done);
        if (done) {
            pair.store(sums + a, cls);
            a = next + __popc(m & ((1u << (grp * kGrp)) - 1u)) / kGrp;
            active = a < nb;
            if (active) start();
        }
        next += __popc(m) / kGrp;
        __syncwarp();
    }
}

// the eight lanes' partial sums of sum s of the batch's atom a, in one fixed tree
__device__ __forceinline__ double lane_total(const char *smem, int s, int a) {
    const double *sums = reinterpret_cast<const double *>(smem + kSumsAt) + s * kGrp * kSumStride + a;
    double c[kGrp];
#pragma unroll
    for (int k = 0; k < kGrp; ++k) c[k] = sums[k * kSumStride];
    return ((c[0] + c[4]) + (c[2] + c[6])) + ((c[1] + c[5]) + (c[3] + c[7]));
}

// f(first slot, valid atoms, replica) for every batch of this warp's range
template <class F>
__device__ __forceinline__ void for_batches(const View &V, F &&f) {
    const long long units = V.n_pad / kUnit;
    const int end = (int)(units * (blockIdx.x + 1) / gridDim.x) * kUnit;
    for (int p = (int)(units * blockIdx.x / gridDim.x) * kUnit; p < end;) {
        const int pe = min(end, (p | (kBatchAtoms - 1)) + 1);  // aligned slots of one 32-atom tile, so of one replica
        const Rep &R = V.rep[V.n_rep == 1 ? 0 : V.tile_rep[p >> 5]];
        const int nb = min(max(R.natoms - (p - R.atom0), 0), pe - p);
        if (nb > 0) f(p, nb, R);
        p = pe;
        __syncwarp();
    }
}

// f(sum, atom) over a batch's ns x nb results, spread over the lanes
template <class F>
__device__ __forceinline__ void for_sums(int ns, int nb, F &&f) {
    const int lg = nb > 1 ? 32 - __clz(nb - 1) : 0;
    for (int k = threadIdx.x; k < ns << lg; k += 32) {
        const int a = k & ((1 << lg) - 1);
        if (a < nb) f(k >> lg, a);
    }
}

// -------------------------------------------------------------------- LJ --

template <int HALF, int EV, int MT>
struct Lj64 {
    static constexpr int kSums = EV ? 10 : 3;
    double ax, ay, az, e, w[6];
    double c1, c2, c3, c4, c0, rc2;
    int ti;
    __device__ __forceinline__ void begin(const View &V, int p) {
        ax = 0.0; ay = 0.0; az = 0.0;
        if (EV) {
            e = 0.0;
#pragma unroll
            for (int k = 0; k < 6; ++k) w[k] = 0.0;
        }
        if (MT) ti = V.type[p] * V.ntypes;
    }
    __device__ __forceinline__ void operator()(const View &V, uint32_t ent, bool on, double dx, double dy, double dz,
                                               double r2, double wj) {
        const bool in = on && below(r2, rc2);
        if (MT) {
            const int tp = ti + (in ? (int)__double_as_longlong(wj) : 0);
            c1 = V.tab->lj1[tp]; c2 = V.tab->lj2[tp];
            if (EV) { c3 = V.tab->lj3[tp]; c4 = V.tab->lj4[tp]; c0 = V.tab->off[tp]; }
        }
        const double r2i = rcp64(r2);
        const double r6i = r2i * r2i * r2i;
        const double fpair = in ? r6i * (c1 * r6i - c2) * r2i : 0.0;
        if (!EV && !HALF) {
            ax = fma(dx, fpair, ax); ay = fma(dy, fpair, ay); az = fma(dz, fpair, az);
            return;
        }
        const double fx = dx * fpair, fy = dy * fpair, fz = dz * fpair;
        ax += fx; ay += fy; az += fz;
        if (HALF && in) {
            const int j = entry_j(ent), n = V.n_pad;
            atomicAdd(&V.f[j], -fx);
            atomicAdd(&V.f[n + j], -fy);
            atomicAdd(&V.f[2 * n + j], -fz);
        }
        if (EV) {  // a full list's terms are halved at the atom's end
            e += in ? r6i * (c3 * r6i - c4) - c0 : 0.0;
            w[0] = fma(dx, fx, w[0]); w[1] = fma(dy, fy, w[1]); w[2] = fma(dz, fz, w[2]);
            w[3] = fma(dx, fy, w[3]); w[4] = fma(dx, fz, w[4]); w[5] = fma(dy, fz, w[5]);
        }
    }
    __device__ __forceinline__ void store(double *s, int cls) {
        s[cls * kSumStride] = ax; s[(kGrp + cls) * kSumStride] = ay; s[(2 * kGrp + cls) * kSumStride] = az;
        if (EV) {
            s[(3 * kGrp + cls) * kSumStride] = e;
#pragma unroll
            for (int k = 0; k < 6; ++k) s[((4 + k) * kGrp + cls) * kSumStride] = w[k];
        }
    }
};

template <int Q, int U, int HALF, int EV, int MT>
__global__ void __launch_bounds__(32, U == 4 || EV ? kWarpsFew : kWarpsMany) k64_lj(View V, KArgs a) {
    extern __shared__ char smem[];
    if (V.ctl->err) return;
    const int rem = (a.mode == kModeStep) ? V.ctl->remaining : 0;
    Lj64<HALF, EV, MT> pr{};
    pr.rc2 = V.rc2;
    if (!MT) {
        pr.c1 = V.tab->lj1[0]; pr.c2 = V.tab->lj2[0];
        if (EV) { pr.c3 = V.tab->lj3[0]; pr.c4 = V.tab->lj4[0]; pr.c0 = V.tab->off[0]; }
    }
    for_batches(V, [&](int p0, int nb, const Rep &R) {
        fp64_walk<SrcPos4, Q, U>(V, R, p0, nb, smem, pr);
        for_sums(EV ? 10 : 3, nb, [&](int s, int i) {
            const double x = lane_total(smem, s, i);
            const int p = p0 + i;
            if (s >= 3) V.ev[(size_t)(s == 3 ? 0 : s - 2) * V.n_pad + p] = (HALF ? 1.0 : 0.5) * x;
            else if (HALF) atomicAdd(&V.f[(size_t)s * V.n_pad + p], x);
            else finish_component(V, a.mode, rem, s, p, V.tab->ftm_m[MT ? V.type[p] : 0], x);
        });
        // (half lists: the kinetic term follows in k_kick)
        if (EV && !HALF && (int)threadIdx.x < nb)
            write_kinetic(V, p0 + threadIdx.x, V.tab->ftm_m[MT ? V.type[p0 + threadIdx.x] : 0]);
    });
}

// ------------------------------------------------------------------- EAM --

struct Rho64 {
    static constexpr int kSums = 1;
    double rho, rc, rc2;
    __device__ __forceinline__ void begin(const View &, int) { rho = 0.0; }
    __device__ __forceinline__ void operator()(const View &, uint32_t, bool on, double, double, double, double r2,
                                               double) {
        const double t = rc - r2 * rsqrt64(r2);
        const double u = on && below(r2, rc2) ? t : 0.0;
        rho = fma(u, u, rho);
    }
    __device__ __forceinline__ void store(double *s, int cls) { s[cls * kSumStride] = rho; }
};

template <int Q, int U>
__global__ void __launch_bounds__(32, U == 4 ? kWarpsFew : kWarpsMany) k64_eam_rho(View V, KArgs a) {
    extern __shared__ char smem[];
    if (V.ctl->err) return;
    Rho64 pr{};
    pr.rc = V.tab->eam[0];
    pr.rc2 = V.rc2;
    const double Aemb = V.tab->eam[1];
    for_batches(V, [&](int p0, int nb, const Rep &R) {
        fp64_walk<SrcPos4, Q, U>(V, R, p0, nb, smem, pr);
        for_sums(1, nb, [&](int, int i) {
            const double rho = lane_total(smem, 0, i);
            const double sr = sqrt(rho);
            V.fp64[p0 + i] = rho > 0.0 ? -0.5 * Aemb / sr : 0.0;
            if (a.mode == kModeEV) V.emb[p0 + i] = rho > 0.0 ? -Aemb * sr : 0.0;
        });
    });
}

// The pair function about its own cut-off: with t = rc - r, phi = t^2 (p0 + p1 t + p2 t^2),
//   phi' = -t (2 p0 + 3 p1 t + 4 p2 t^2),  phi'' = 2 (p0 + 3 p1 t + 6 p2 t^2),
// two FP64 instructions each instead of five for phi' and eight for both from the
// polynomial in r and its derivative.
struct EamPoly {
    double p0, p1, p2;
    __device__ __forceinline__ explicit EamPoly(const PairTab *tab) {
        const double rc = tab->eam[0], c0 = tab->eam[2], c1 = tab->eam[3], c2 = tab->eam[4];
        p0 = fma(rc, fma(rc, c2, c1), c0);
        p1 = -fma(2.0 * rc, c2, c1);
        p2 = c2;
    }
};

template <int EV>
struct Eam64 {
    static constexpr int kSums = EV ? 10 : 3;
    double ax, ay, az, e, w[6];
    double rc, rc2, p0, p1, p2, d0, d1, d2, fpi;  // d: 2 p0, 3 p1, 4 p2
    __device__ __forceinline__ void begin(const View &V, int p) {
        ax = 0.0; ay = 0.0; az = 0.0;
        if (EV) {
            e = 0.0;
#pragma unroll
            for (int k = 0; k < 6; ++k) w[k] = 0.0;
        }
        fpi = V.fp64[p];
    }
    __device__ __forceinline__ void operator()(const View &V, uint32_t ent, bool on, double dx, double dy, double dz,
                                               double r2, double) {
        const bool in = on && below(r2, rc2);
        const double fpj = V.fp64[entry_j(ent)];
        const double rinv = rsqrt64(r2);
        const double r = r2 * rinv;
        const double t = rc - r;
        // -(phi' + (F'_i + F'_j) rho') / r with rho' = -2t
        double coef = t * fma(2.0, fpi + fpj, fma(t, fma(t, d2, d1), d0)) * rinv;
        coef = in ? coef : 0.0;
        if (!EV) {
            ax = fma(dx, coef, ax); ay = fma(dy, coef, ay); az = fma(dz, coef, az);
            return;
        }
        const double fx = dx * coef, fy = dy * coef, fz = dz * coef;
        ax += fx; ay += fy; az += fz;
        e += in ? t * t * fma(t, fma(t, p2, p1), p0) : 0.0;
        w[0] = fma(dx, fx, w[0]); w[1] = fma(dy, fy, w[1]); w[2] = fma(dz, fz, w[2]);
        w[3] = fma(dx, fy, w[3]); w[4] = fma(dx, fz, w[4]); w[5] = fma(dy, fz, w[5]);
    }
    __device__ __forceinline__ void store(double *s, int cls) {
        s[cls * kSumStride] = ax; s[(kGrp + cls) * kSumStride] = ay; s[(2 * kGrp + cls) * kSumStride] = az;
        if (EV) {
            s[(3 * kGrp + cls) * kSumStride] = e;
#pragma unroll
            for (int k = 0; k < 6; ++k) s[((4 + k) * kGrp + cls) * kSumStride] = w[k];
        }
    }
};

template <int Q, int U, int EV>
__global__ void __launch_bounds__(32, kWarpsFew) k64_eam_force(View V, KArgs a) {
    extern __shared__ char smem[];
    if (V.ctl->err) return;
    const int rem = (a.mode == kModeStep) ? V.ctl->remaining : 0;
    Eam64<EV> pr{};
    pr.rc = V.tab->eam[0];
    pr.rc2 = V.rc2;
    const EamPoly poly(V.tab);
    pr.p0 = poly.p0; pr.p1 = poly.p1; pr.p2 = poly.p2;
    pr.d0 = 2.0 * poly.p0; pr.d1 = 3.0 * poly.p1; pr.d2 = 4.0 * poly.p2;
    const double ftm = V.tab->ftm_m[0];  // single element
    for_batches(V, [&](int p0, int nb, const Rep &R) {
        fp64_walk<SrcPos4, Q, U>(V, R, p0, nb, smem, pr);
        for_sums(EV ? 10 : 3, nb, [&](int s, int i) {
            const double x = lane_total(smem, s, i);
            const int p = p0 + i;
            if (s < 3) finish_component(V, a.mode, rem, s, p, ftm, x);
            else if (s == 3) V.ev[p] = 0.5 * x + V.emb[p];
            else V.ev[(size_t)(s - 2) * V.n_pad + p] = 0.5 * x;
        });
        if (EV && (int)threadIdx.x < nb) write_kinetic(V, p0 + threadIdx.x, ftm);
    });
}

// -------------------------------------------------------------- backward --
// The force-matching backward passes, g = dL/dF.  k_bwd_pack writes one
// 64-byte record per atom (two sectors): its FP64 position and its g, so that a pair's
// gather is two 32-byte loads instead of seven 8-byte ones.

// sum += a b where `in`.  A lane without a pair within rc (an entry between rc and the margin, or an idle
// lane, which evaluates its own atom) adds nothing: a factor of zero instead would let a NaN or an infinity in g
// through.  Predicated, since a branch around the sums keeps a lane's pairs from overlapping: EAM backward of 6,912
// atoms 80.5 us with zero factors, 95.0 with a branch, 80.5 so.
__device__ __forceinline__ void add_if(bool in, double a, double b, double &sum) {
    asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p fma.rn.f64 %0, %1, %2, %0;\n\t}"
        : "+d"(sum)
        : "d"(a), "d"(b), "r"((unsigned)in));
}

template <int PREC>
__global__ void k_bwd_pack(View V, const double *grad_f) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= V.n_pad) return;
    const Rep &R = V.rep[V.tile_rep[p >> 5]];
    const int n = V.n_pad;
    double4_32a x = make_double4_32a(0.0, 0.0, 0.0, __longlong_as_double(0)), g = make_double4_32a(0.0, 0.0, 0.0, 0.0);
    if (p - R.atom0 < R.natoms) {
        const long long o = R.orig0 + V.id[p];
        if (PREC == MD_PREC_FP64) {
            x = V.pos4[p];
        } else {
            x.x = V.xr[p]; x.y = V.xr[n + p]; x.z = V.xr[2 * n + p];
            x.w = __longlong_as_double((long long)V.type[p]);
        }
        g.x = grad_f[3 * o]; g.y = grad_f[3 * o + 1]; g.z = grad_f[3 * o + 2];
    }
    V.bpack[2 * (size_t)p] = x;
    V.bpack[2 * (size_t)p + 1] = g;
}

// dL/dx of a batch's atoms, straight to the caller's order
__device__ __forceinline__ void grad_out(const View &V, const Rep &R, int p0, int nb, const char *smem,
                                         double *grad_x, double sign = 1.0) {
    if (!grad_x) return;
    for_sums(3, nb, [&](int s, int i) { grad_x[3 * (R.orig0 + V.id[p0 + i]) + s] = sign * lane_total(smem, s, i); });
}

// LJ.  dL/dx_i = sum_j M_ij (g_i - g_j),  M = s(r) I + (s'(r)/r) d d^T, s = -U'(r)/r.
// Parameters: dL/dtheta = sum_i g_i . sum_j (ds/dtheta) d; over the two orders
// of a pair g_i . d sums to (g_i - g_j) . d, so each ordered pair contributes
// half of that, which the position gradient needs anyway.  Per unordered type
// pair two sums: S = sum s (g_i - g_j).d and S12 = sum r^-14 (g_i - g_j).d, then
//   dL/deps = S / (2 eps),  dL/dsig = 6 (lj1 S12 + S) / (2 sig)
// (ds/dsig = (12 lj1 r^-14 - 6 lj2 r^-8) / sig = 6 (lj1 r^-14 + s) / sig).
// One type: the two sums in registers; several: in shared memory, per lane.
__device__ __forceinline__ int pair_index(int ta, int tb, int nt) {  // upper triangle, row-major
    const int lo = min(ta, tb), hi = max(ta, tb);
    return lo * nt - lo * (lo - 1) / 2 + (hi - lo);
}

template <int MT>
struct LjBwd64 {
    double gx, gy, gz, gix, giy, giz, S, S12;
    double c1, c2, rc2;
    double *par;  // MT: [pair][2][32]
    int ti, nt;
    __device__ __forceinline__ void begin(const View &V, int p) {
        gx = 0.0; gy = 0.0; gz = 0.0;
        const double4_32a g = V.bpack[2 * (size_t)p + 1];
        gix = g.x; giy = g.y; giz = g.z;
        if (MT) ti = V.type[p];
    }
    __device__ __forceinline__ void operator()(const View &V, uint32_t ent, bool on, double dx, double dy, double dz,
                                               double r2, double wj) {
        const bool in = on && below(r2, rc2);
        const double4_32a gj = V.bpack[2 * (size_t)entry_j(ent) + 1];
        const int tj = MT && in ? (int)__double_as_longlong(wj) : 0;
        if (MT) {
            c1 = V.tab->lj1[ti * nt + tj];
            c2 = V.tab->lj2[ti * nt + tj];
        }
        const double r2i = rcp64(r2);
        const double r6i = r2i * r2i * r2i, r8i = r6i * r2i;
        const double c1r6 = c1 * r6i;
        const double s = r8i * (c1r6 - c2);
        const double spr = r8i * r2i * fma(-14.0, c1r6, 8.0 * c2);
        const double dgx = gix - gj.x, dgy = giy - gj.y, dgz = giz - gj.z;
        const double ddg = fma(dz, dgz, fma(dy, dgy, dx * dgx));
        const double t = spr * ddg;
        add_if(in, s, dgx, gx); add_if(in, t, dx, gx);
        add_if(in, s, dgy, gy); add_if(in, t, dy, gy);
        add_if(in, s, dgz, gz); add_if(in, t, dz, gz);
        if (MT) {
            double *q = par + pair_index(ti, tj, nt) * 64 + (threadIdx.x & 31);
            if (in) {
                q[0] = fma(ddg, s, q[0]);
                q[32] = fma(ddg * r8i, r6i, q[32]);
            }
        } else {
            add_if(in, ddg, s, S);
            add_if(in, ddg * r8i, r6i, S12);
        }
    }
    __device__ __forceinline__ void store(double *s, int cls) {
        s[cls * kSumStride] = gx; s[(kGrp + cls) * kSumStride] = gy; s[(2 * kGrp + cls) * kSumStride] = gz;
    }
};

// gp_part: [block][2 per unordered type pair]
template <int Q, int U, int MT>
__global__ void __launch_bounds__(32, kWarpsFew) k64_lj_bwd(View V, KArgs, double *grad_x) {
    extern __shared__ char smem[];
    const int nt = V.ntypes, npar = nt * (nt + 1);
    const int lane = threadIdx.x;
    LjBwd64<MT> pr{};
    pr.rc2 = V.rc2;
    pr.nt = nt;
    pr.par = reinterpret_cast<double *>(smem + fp64_smem(3));
    if (MT) {
        for (int k = 0; k < npar; ++k) pr.par[k * 32 + lane] = 0.0;
    } else {
        pr.c1 = V.tab->lj1[0];
        pr.c2 = V.tab->lj2[0];
    }
    for_batches(V, [&](int p0, int nb, const Rep &R) {
        fp64_walk<SrcPack, Q, U>(V, R, p0, nb, smem, pr);
        grad_out(V, R, p0, nb, smem, grad_x);
    });
    double *part = V.gp_part + (size_t)blockIdx.x * npar;
    if (MT) {
        for (int k = 0; k < npar; ++k) {
            const double x = warp_sum(pr.par[k * 32 + lane]);
            if (lane == 0) part[k] = x;
        }
    } else {
        const double x = warp_sum(pr.S), y = warp_sum(pr.S12);
        if (lane == 0) { part[0] = x; part[1] = y; }
    }
}

// block u: the two sums of unordered type pair u over the blocks' partials in
// a fixed order, and its (eps, sig) gradients in both places
__global__ void __launch_bounds__(512) k_gp_reduce(View V, int nblocks, double *grad_params) {
    __shared__ double s_w[16];
    const int nt = V.ntypes, npar = nt * (nt + 1), u = blockIdx.x;
    double s = 0.0, s12 = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
        s += V.gp_part[(size_t)b * npar + 2 * u];
        s12 += V.gp_part[(size_t)b * npar + 2 * u + 1];
    }
    s = block_sum(s, s_w);
    s12 = block_sum(s12, s_w);
    if (threadIdx.x != 0) return;
    int ta = 0, left = u;
    while (left >= nt - ta) left -= nt - ta++;
    const int tb = ta + left, q = ta * nt + tb, qt = tb * nt + ta;
    const double ge = 0.5 * s * V.tab->inv_eps[q];
    const double gs = 3.0 * fma(V.tab->lj1[q], s12, s) * V.tab->inv_sig[q];
    grad_params[q] = ge;
    grad_params[qt] = ge;
    grad_params[nt * nt + q] = gs;
    grad_params[nt * nt + qt] = gs;
}

// EAM: the vector-Jacobian product of the Finnis-Sinclair forces (App. A EAM
// form) for L = sum_i g_i.F_i, in two passes over the full list.  With d = x_i - x_j,
// r = |d|, u = d/r, G = g_i - g_j, w = G.u, s = phi' + (F'_i + F'_j) rho' and
// k = phi'' + (F'_i + F'_j) rho'':
//   pass 1: rho_i and lambda_i = sum_j w rho'(r); then F'_i, mu_i = lambda_i F''(rho_i)
//           (kept as -2 mu_i) and the atom's share -lambda_i dF'_i/dA of dL/dA;
//   pass 2: dL/dx_i = -sum_j [(s/r) G + (w (k - s/r) + (mu_i + mu_j) rho') u]
//           and dL/dc_q = -sum_j (g_i.u) dphi'/dc_q, where (as for LJ) half of w
//           stands for g_i.u over the two orders of a pair.
struct EamBwd1 {
    double rho, lam, gix, giy, giz, rc, rc2;
    __device__ __forceinline__ void begin(const View &V, int p) {
        rho = 0.0;
        lam = 0.0;
        const double4_32a g = V.bpack[2 * (size_t)p + 1];
        gix = g.x; giy = g.y; giz = g.z;
    }
    __device__ __forceinline__ void operator()(const View &V, uint32_t ent, bool on, double dx, double dy, double dz,
                                               double r2, double) {
        const bool in = on && below(r2, rc2);
        const double4_32a gj = V.bpack[2 * (size_t)entry_j(ent) + 1];
        const double ir = rsqrt64(r2), r = r2 * ir;
        const double t = rc - r, tir = t * ir;
        // w rho'(r) with w = (g_i - g_j).d / r and rho' = -2 (rc - r); the -2 at the atom's end
        const double Gd = fma(giz - gj.z, dz, fma(giy - gj.y, dy, (gix - gj.x) * dx));
        add_if(in, t, t, rho);
        add_if(in, tir, Gd, lam);
    }
    __device__ __forceinline__ void store(double *s, int cls) {
        s[cls * kSumStride] = rho;
        s[(kGrp + cls) * kSumStride] = lam;
    }
};

template <int Q, int U>
__global__ void __launch_bounds__(32, kWarpsFew) k64_eam_bwd1(View V, KArgs) {
    extern __shared__ char smem[];
    EamBwd1 pr{};
    pr.rc = V.tab->eam[0];
    pr.rc2 = pr.rc * pr.rc;
    const double Aem = V.tab->eam[1];
    double partA = 0.0;
    for_batches(V, [&](int p0, int nb, const Rep &R) {
        fp64_walk<SrcPack, Q, U>(V, R, p0, nb, smem, pr);
        if ((int)threadIdx.x < nb) {
            const int p = p0 + threadIdx.x, n = V.n_pad;
            const double rho = lane_total(smem, 0, threadIdx.x), lam = -2.0 * lane_total(smem, 1, threadIdx.x);
            const double sq = rho > 0.0 ? sqrt(rho) : 0.0;
            V.bw[p] = rho > 0.0 ? -0.5 * Aem / sq : 0.0;
            V.bw[n + p] = rho > 0.0 ? -2.0 * lam * (0.25 * Aem / (rho * sq)) : 0.0;
            partA += rho > 0.0 ? lam * (0.5 / sq) : 0.0;
        }
    });
    partA = warp_sum(partA);
    if (threadIdx.x == 0) V.gp_part[(size_t)blockIdx.x * 4] = partA;
}

struct EamBwd2 {
    double gx, gy, gz, g0, g1, g2;
    double gix, giy, giz, fpi, mui;
    double rc, rc2, d0, d1, d2, q0, q1, q2;  // d: 2 p0, 3 p1, 4 p2 (phi'); q: 2 p0, 6 p1, 12 p2 (phi'')
    __device__ __forceinline__ void begin(const View &V, int p) {
        gx = 0.0; gy = 0.0; gz = 0.0;
        const double4_32a g = V.bpack[2 * (size_t)p + 1];
        gix = g.x; giy = g.y; giz = g.z;
        fpi = V.bw[p];
        mui = V.bw[V.n_pad + p];
    }
    __device__ __forceinline__ void operator()(const View &V, uint32_t ent, bool on, double dx, double dy, double dz,
                                               double r2, double) {
        const bool in = on && below(r2, rc2);
        const int j = entry_j(ent);
        const double4_32a gj = V.bpack[2 * (size_t)j + 1];
        const double fpj = V.bw[j], muj = V.bw[V.n_pad + j];
        const double ir = rsqrt64(r2), r = r2 * ir;
        const double t = rc - r;
        const double Gx = gix - gj.x, Gy = giy - gj.y, Gz = giz - gj.z;
        const double w = fma(Gz, dz, fma(Gy, dy, Gx * dx)) * ir;  // G.u
        const double m = fma(t, fma(t, d2, d1), d0);      // phi' = -t m
        const double d2phi = fma(t, fma(t, q2, q1), q0);
        const double fs = fpi + fpj;
        const double tir = t * ir;
        const double sir = -tir * fma(2.0, fs, m);       // s / r
        const double kv = fma(2.0, fs, d2phi);
        // (w (k - s/r) + (mu_i + mu_j) rho') / r with rho' = -2t; the pass before left -2 mu
        const double b = fma(w, kv - sir, t * (mui + muj)) * ir;
        // dphi'/dc = (-2t, t (t - 2r), 2 r t (t - r)), with t = rc - r
        const double wt = w * t;
        add_if(in, b, dx, gx); add_if(in, sir, Gx, gx);
        add_if(in, b, dy, gy); add_if(in, sir, Gy, gy);
        add_if(in, b, dz, gz); add_if(in, sir, Gz, gz);
        add_if(in, wt, 1.0, g0);
        add_if(in, wt, fma(-3.0, r, rc), g1);
        add_if(in, wt * r, fma(-2.0, r, rc), g2);
    }
    __device__ __forceinline__ void store(double *s, int cls) {
        s[cls * kSumStride] = gx; s[(kGrp + cls) * kSumStride] = gy; s[(2 * kGrp + cls) * kSumStride] = gz;
    }
};

template <int Q, int U>
__global__ void __launch_bounds__(32, kWarpsFew) k64_eam_bwd2(View V, KArgs, double *grad_x) {
    extern __shared__ char smem[];
    EamBwd2 pr{};
    pr.rc = V.tab->eam[0];
    pr.rc2 = pr.rc * pr.rc;
    const EamPoly poly(V.tab);
    pr.d0 = 2.0 * poly.p0; pr.d1 = 3.0 * poly.p1; pr.d2 = 4.0 * poly.p2;
    pr.q0 = 2.0 * poly.p0; pr.q1 = 6.0 * poly.p1; pr.q2 = 12.0 * poly.p2;
    for_batches(V, [&](int p0, int nb, const Rep &R) {
        fp64_walk<SrcPack, Q, U>(V, R, p0, nb, smem, pr);
        grad_out(V, R, p0, nb, smem, grad_x, -1.0);
    });
    const double g0 = warp_sum(pr.g0), g1 = warp_sum(-0.5 * pr.g1), g2 = warp_sum(-pr.g2);
    if (threadIdx.x == 0) {
        double *part = V.gp_part + (size_t)blockIdx.x * 4;
        part[1] = g0;
        part[2] = g1;
        part[3] = g2;
    }
}

// block t: parameter t over the blocks' partials in a fixed order -> grad_params
// {0 (the cut-off), A, c0, c1, c2}
__global__ void __launch_bounds__(512) k_eam_gp_reduce(View V, int nblocks, double *grad_params) {
    __shared__ double s_w[16];
    const int t = blockIdx.x;
    double s = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) s += V.gp_part[(size_t)b * 4 + t];
    s = block_sum(s, s_w);
    if (threadIdx.x != 0) return;
    grad_params[1 + t] = s;
    if (t == 0) grad_params[0] = 0.0;
}

// -------------------------------------------------------------- dispatch --

// One wave of warps (fewer than `per_sm` where their shared memory does not
// fit), or one per unit of four atoms in a system smaller than that, which then
// keeps several pairs in flight per lane instead (U = 4).
constexpr size_t kSmemPerSm = 200 * 1024;

static int wave_warps(const View &V, size_t smem, int per_sm) {
    const int fit = (int)(kSmemPerSm / (smem + 1024));  // 1 KB reserved per block
    return std::min(V.n_pad / kUnit, V.n_sm * std::min(per_sm, fit));
}

static bool small64(const View &V) { return V.n_pad / kUnit <= V.n_sm * kWarpsFew; }

static KCall fp64_call(const View &V, const void *fn, size_t smem, int per_sm, const KArgs &a) {
    return KCall{fn, dim3((unsigned)wave_warps(V, smem, per_sm)), dim3(32), smem, a};
}

// kernel K<Q, U, ...> for the list's vector width and the system's size
#define PICK64_U(K, Q, ...) (small64(V) ? (const void *)K<Q, 4, ##__VA_ARGS__> : (const void *)K<Q, 1, ##__VA_ARGS__>)
#define PICK64(K, ...)                                  \
    (V.vec == 4   ? PICK64_U(K, 4, ##__VA_ARGS__)       \
     : V.vec == 2 ? PICK64_U(K, 2, ##__VA_ARGS__)       \
                  : PICK64_U(K, 1, ##__VA_ARGS__))

void fp64_force_sequence(const View &V, int mode, KArgs a, std::vector<KCall> &seq) {
    const bool ev = mode == kModeEV, mt = V.ntypes > 1;
    const size_t sm = fp64_smem(ev ? 10 : 3);
    if (V.pot == MD_POT_LJ) {
        const void *fn;
        if (V.half)
            fn = ev ? (mt ? PICK64(k64_lj, 1, 1, 1) : PICK64(k64_lj, 1, 1, 0))
                    : (mt ? PICK64(k64_lj, 1, 0, 1) : PICK64(k64_lj, 1, 0, 0));
        else
            fn = ev ? (mt ? PICK64(k64_lj, 0, 1, 1) : PICK64(k64_lj, 0, 1, 0))
                    : (mt ? PICK64(k64_lj, 0, 0, 1) : PICK64(k64_lj, 0, 0, 0));
        seq.push_back(fp64_call(V, fn, sm, ev ? kWarpsFew : kWarpsMany, a));
    } else {
        KArgs ar = a;
        ar.in_graph = 0;
        seq.push_back(fp64_call(V, PICK64(k64_eam_rho), fp64_smem(1), kWarpsMany, ar));
        seq.push_back(
            fp64_call(V, ev ? PICK64(k64_eam_force, 1) : PICK64(k64_eam_force, 0), sm, kWarpsFew, a));
    }
}

int backward_partials_per_block(const View &V) { return V.pot == MD_POT_LJ ? V.ntypes * (V.ntypes + 1) : 4; }

// both EAM passes share one grid: their partials lie in one row per block
static size_t backward_smem(const View &V) {
    size_t sm = fp64_smem(3);
    if (V.pot == MD_POT_LJ && V.ntypes > 1) sm += (size_t)backward_partials_per_block(V) * 32 * sizeof(double);
    return sm;
}

int backward_partial_blocks(const View &V) { return wave_warps(V, backward_smem(V), kWarpsFew); }

static cudaError_t launch_pack(const View &V, const double *grad_f, cudaStream_t s) {
    const dim3 g((unsigned)((V.n_pad + 255) / 256));
    if (V.prec == MD_PREC_FP64) k_bwd_pack<MD_PREC_FP64><<<g, 256, 0, s>>>(V, grad_f);
    else k_bwd_pack<MD_PREC_MIXED><<<g, 256, 0, s>>>(V, grad_f);
    return cudaGetLastError();
}

// (the density pass takes no grad_x and leaves the third argument alone)
static cudaError_t launch64(const View &V, const KCall &k, double *grad_x, cudaStream_t s) {
    View Vc = V;
    KArgs a = k.args;
    void *args[3] = {(void *)&Vc, (void *)&a, (void *)&grad_x};
    return cudaLaunchKernel(k.fn, k.grid, k.block, args, k.smem, s);
}

cudaError_t launch_backward(const View &V, const double *grad_f, double *grad_x, double *grad_params, cudaStream_t s) {
    cudaError_t e = launch_pack(V, grad_f, s);
    if (e != cudaSuccess) return e;
    const void *fn = V.ntypes > 1 ? PICK64(k64_lj_bwd, 1) : PICK64(k64_lj_bwd, 0);
    e = launch64(V, fp64_call(V, fn, backward_smem(V), kWarpsFew, KArgs{}), grad_x, s);
    if (e != cudaSuccess) return e;
    if (grad_params)
        k_gp_reduce<<<V.ntypes * (V.ntypes + 1) / 2, 512, 0, s>>>(V, backward_partial_blocks(V), grad_params);
    return cudaGetLastError();
}

cudaError_t launch_eam_backward(const View &V, const double *grad_f, double *grad_x, double *grad_params,
                                cudaStream_t s) {
    cudaError_t e = launch_pack(V, grad_f, s);
    if (e != cudaSuccess) return e;
    e = launch64(V, fp64_call(V, PICK64(k64_eam_bwd1), backward_smem(V), kWarpsFew, KArgs{}), grad_x, s);
    if (e != cudaSuccess) return e;
    e = launch64(V, fp64_call(V, PICK64(k64_eam_bwd2), backward_smem(V), kWarpsFew, KArgs{}), grad_x, s);
    if (e != cudaSuccess) return e;
    if (grad_params) k_eam_gp_reduce<<<4, 512, 0, s>>>(V, backward_partial_blocks(V), grad_params);
    return cudaGetLastError();
}

}  // namespace md
