// k_misc.cu -- moving state between the caller's original order and the
// library's cell-sorted order, deterministic energy/virial reduction, list export
// and the halo buffers of a spatial decomposition.
#include <algorithm>

#include "md_common.cuh"
#include "md_kernels.h"

namespace md {

// ------------------------------------------------------------------ I/O ----

// Stage replica r's caller arrays (x, v, type of that replica alone, original
// order) into the rebuild scratch: atom `local` goes to slot atom0 + local.
__global__ void k_stage_in(View V, int r, const double *x, const double *v, const int *type) {
    const int local = blockIdx.x * blockDim.x + threadIdx.x;
    const Rep &R = V.rep[r];
    if (local >= R.natoms) return;
    const int p = R.atom0 + local;
    const int n = V.n_pad;
    for (int c = 0; c < 3; ++c) {
        V.tx[c * n + p] = x[3 * (size_t)local + c];
        V.tv[c * n + p] = v[3 * (size_t)local + c];
    }
    V.ttype[p] = type[local];
    V.tid[p] = local;
}

// absolute position of sorted slot p from its cell-relative coordinates
template <int PREC>
__device__ __forceinline__ void abs_pos(const View &V, const Rep &R, int p, double x[3]) {
    const int b = V.bpk[p];
    const int bc[3] = {unpack_bx(b), unpack_by(b), unpack_bz(b)};
    if (PREC == MD_PREC_FP64) {
        const double4_32a q = V.pos4[p];
        x[0] = q.x; x[1] = q.y; x[2] = q.z;
    } else {
        for (int c = 0; c < 3; ++c) x[c] = V.xr[c * V.n_pad + p];
    }
    for (int c = 0; c < 3; ++c) x[c] = fma(bin_centre(bc[c]), R.h[c], x[c]);
}

// Stage new positions and/or velocities (original order; NULL keeps the
// current value) together with the current types and ids, for a full rebuild.
template <int PREC>
__global__ void k_restage(View V, const double *x, const double *v) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= V.n_pad) return;
    const Rep &R = V.rep[V.tile_rep[p >> 5]];
    if (p - R.atom0 >= R.natoms) return;
    const int n = V.n_pad;
    const int id = V.id[p];
    const int d = R.atom0 + id;
    const long long o = R.orig0 + id;
    double xa[3];
    abs_pos<PREC>(V, R, p, xa);
    for (int c = 0; c < 3; ++c) {
        V.tx[c * n + d] = x ? x[3 * o + c] : xa[c];
        V.tv[c * n + d] = v ? v[3 * o + c] : V.v[c * n + p];
    }
    V.ttype[d] = V.type[p];
    V.tid[d] = id;
}

template <int PREC>
__global__ void k_state_out(View V, double *x, double *v, double *f) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= V.n_pad) return;
    const Rep &R = V.rep[V.tile_rep[p >> 5]];
    if (p - R.atom0 >= R.natoms) return;
    const int n = V.n_pad;
    const long long o = R.orig0 + V.id[p];
    if (x) {
        double xa[3];
        abs_pos<PREC>(V, R, p, xa);
        for (int c = 0; c < 3; ++c) {
            x[3 * o + c] = wrap_box(xa[c], R.L[c], R.Linv[c]);
        }
    }
    if (v) for (int c = 0; c < 3; ++c) v[3 * o + c] = V.v[c * n + p];
    if (f) for (int c = 0; c < 3; ++c) f[3 * o + c] = V.f[c * n + p];
}

// ------------------------------------------------------ energy / virial ----

// Fixed-order stages: per 32-atom tile (one warp each), per segment of a
// replica's tiles (one block each), and, where a replica has several
// segments, over these in the last block.  The FP64 adds bound it (2 lanes per clock
// and SM): a warp's eight sums are reduced by halves (lanes exchange the half they do
// not keep: 9 adds instead of 8 trees of 5), and the tiles of a few
// large systems are spread over several blocks each.
constexpr int kEvSegment = 256;  // tiles per block

__device__ __forceinline__ double ev_fold(double keep, double send, int o) {
    return keep + __shfl_xor_sync(0xffffffffu, send, o);
}

__global__ void k_ev_tiles(View V) {
    const int lane = threadIdx.x & 31;
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= V.n_tiles) return;
    const int p = t * 32 + lane;
    const Rep &R = V.rep[V.tile_rep[t]];
    const bool ok = (p - R.atom0) < R.natoms;
    double x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = ok ? V.ev[(size_t)k * V.n_pad + p] : 0.0;
    // lane bit 4 keeps terms 0..3 or 4..7, bit 3 two of these, bit 2 one
    const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
    double y[4], z[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) y[k] = ev_fold(h4 ? x[k + 4] : x[k], h4 ? x[k] : x[k + 4], 16);
#pragma unroll
    for (int k = 0; k < 2; ++k) z[k] = ev_fold(h3 ? y[k + 2] : y[k], h3 ? y[k] : y[k + 2], 8);
    double u = ev_fold(h2 ? z[1] : z[0], h2 ? z[0] : z[1], 4);
    u = ev_fold(u, u, 2);
    u = ev_fold(u, u, 1);
    if ((lane & 3) == 0) V.ev_tile[(size_t)t * 8 + (lane >> 2)] = u;
}

// nseg blocks per replica, 256 threads: thread = (slot, term)
__global__ void __launch_bounds__(256) k_ev_reduce(View V, int nseg, double *out) {
    __shared__ double s_w[8][8];
    const int r = blockIdx.x / nseg, seg = blockIdx.x - r * nseg;
    const Rep &R = V.rep[r];
    const int term = threadIdx.x & 7, slot = threadIdx.x >> 3, w = threadIdx.x >> 5;
    auto sum = [&](const double *rows, int n) {  // sum of n rows of eight terms; thread < 8 gets its term
        double acc = 0.0;
#pragma unroll 4
        for (int t = slot; t < n; t += 32) acc += __ldcg(&rows[(size_t)t * 8 + term]);
        acc += __shfl_xor_sync(0xffffffffu, acc, 8);
        acc += __shfl_xor_sync(0xffffffffu, acc, 16);
        __syncthreads();
        if ((threadIdx.x & 31) < 8) s_w[w][term] = acc;
        __syncthreads();
        double tot = 0.0;
        if (threadIdx.x < 8)
            for (int k = 0; k < 8; ++k) tot += s_w[k][term];
        return tot;
    };
    const int t0 = R.tile0 + (int)((long long)R.ntiles * seg / nseg);
    const int t1 = R.tile0 + (int)((long long)R.ntiles * (seg + 1) / nseg);
    const double part = sum(V.ev_tile + (size_t)t0 * 8, t1 - t0);
    if (nseg == 1) {
        if (threadIdx.x < 8) out[8 * r + term] = part;
        return;
    }
    if (threadIdx.x < 8) V.ev_seg[(size_t)blockIdx.x * 8 + term] = part;
    if (!last_block(&V.ctl->ticket_ev)) return;
    __threadfence();
    for (int q = 0; q < V.n_rep; ++q) {
        const double tot = sum(V.ev_seg + (size_t)q * nseg * 8, nseg);
        if (threadIdx.x < 8) out[8 * q + term] = tot;
    }
    if (threadIdx.x == 0) V.ctl->ticket_ev = 0;
}

// ------------------------------------------------------------ list out ----

__global__ void k_neighbors_out(View V, int *counts, int *nbr, int cap) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= V.n_pad) return;
    const Rep &R = V.rep[V.tile_rep[p >> 5]];
    if (p - R.atom0 >= R.natoms) return;
    const long long o = R.orig0 + V.id[p];
    const int c = V.ncount[p];
    counts[o] = c;
    for (int k = 0; k < c && k < cap; ++k) {
        const uint32_t e = V.nlist[list_index(p, k, V.ltpa, V.lvec, V.maxneigh)];
        nbr[o * cap + k] = V.id[entry_slot(V, p, e)];
    }
}


// ------------------------------------------------------------------ halo ----
// Device-side communication buffers of a spatial decomposition (paper
// Sec. V: the buffers are built on the GPU and only opened there): rows of
// the selected per-atom quantities of the atoms named by the caller's
// indices, gathered from (pack) or scattered into (unpack) the cell-sorted
// state through the inverse map of the last build.
constexpr int kHaloX = 1, kHaloV = 2, kHaloF = 4, kHaloFP = 8, kHaloEV = 16;

__device__ __forceinline__ int halo_slot(const View &V, const int *idx, long long k, long long n_real) {
    const long long o = idx[k];
    if (o < 0 || o >= n_real) {
        latch_error(V.ctl, kErrConfig);
        return -1;
    }
    return V.inv[o];
}

template <int PREC>
__global__ void k_halo_pack(View V, const int *idx, long long m, int what, int width, double sx, double sy, double sz,
                            long long n_real, double *buf) {
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < m; k += (long long)gridDim.x * blockDim.x) {
        double *row = buf + k * width;
        const int p = halo_slot(V, idx, k, n_real);
        if (p < 0) {
            for (int c = 0; c < width; ++c) row[c] = __longlong_as_double(0x7ff8000000000000ll);  // NaN
            continue;
        }
        const Rep &R = V.rep[V.tile_rep[p >> 5]];
        const int n = V.n_pad;
        int c = 0;
        if (what & kHaloX) {
            double xa[3];
            abs_pos<PREC>(V, R, p, xa);
            const double sh[3] = {sx, sy, sz};
            for (int a = 0; a < 3; ++a) {
                row[c++] = wrap_box(xa[a], R.L[a], R.Linv[a]) + sh[a];
            }
        }
        if (what & kHaloV) for (int a = 0; a < 3; ++a) row[c++] = V.v[a * n + p];
        if (what & kHaloF) for (int a = 0; a < 3; ++a) row[c++] = V.f[a * n + p];
        if (what & kHaloFP) row[c++] = PREC == MD_PREC_FP64 ? V.fp64[p] : (double)V.rec[p].w;
        if (what & kHaloEV) for (int q = 0; q < 8; ++q) row[c++] = V.ev[(size_t)q * n + p];
    }
}

template <int PREC>
__global__ void k_halo_unpack(View V, const int *idx, long long m, int what, int width, int accumulate,
                              long long n_real, const double *buf) {
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < m; k += (long long)gridDim.x * blockDim.x) {
        const int p = halo_slot(V, idx, k, n_real);
        if (p < 0) continue;
        const Rep &R = V.rep[V.tile_rep[p >> 5]];
        const int n = V.n_pad;
        const double *row = buf + k * width;
        int c = 0;
        if (what & kHaloX) {
            // position relative to the centre of the atom's cell at the last
            // build, nearest periodic image (the atom keeps its cell and list)
            const int b = V.bpk[p];
            const int bc[3] = {unpack_bx(b), unpack_by(b), unpack_bz(b)};
            double d[3];
            for (int a = 0; a < 3; ++a) {
                double t = fma(-bin_centre(bc[a]), R.h[a], row[c++]);
                t -= R.L[a] * rint(t * R.Linv[a]);
                d[a] = t;
            }
            if (PREC == MD_PREC_FP64) {
                const double4_32a q = V.pos4[p];
                V.pos4[p] = make_double4_32a(d[0], d[1], d[2], q.w);
            } else {
                for (int a = 0; a < 3; ++a) V.xr[a * n + p] = d[a];
            }
            const float4 r = V.rec[p];
            V.rec[p] = make_float4((float)d[0], (float)d[1], (float)d[2], r.w);
        }
        if (what & kHaloV) for (int a = 0; a < 3; ++a) V.v[a * n + p] = row[c++];
        if (what & kHaloF)
            for (int a = 0; a < 3; ++a) {
                const double f = row[c++];
                V.f[a * n + p] = accumulate ? V.f[a * n + p] + f : f;
            }
        if (what & kHaloFP) {
            if (PREC == MD_PREC_FP64) V.fp64[p] = row[c++];
            else V.rec[p].w = (float)row[c++];
        }
    }
}

// largest squared displacement of any atom since the last build (the
// rebuild criterion of a decomposed step, taken after the ghosts' update)
template <int PREC>
__global__ void k_disp_max(View V) {
    float d2 = 0.f;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < V.n_pad; p += gridDim.x * blockDim.x) {
        const Rep &R = V.rep[V.tile_rep[p >> 5]];
        if (p - R.atom0 >= R.natoms) continue;
        double x[3];
        if (PREC == MD_PREC_FP64) {
            const double4_32a q = V.pos4[p];
            x[0] = q.x; x[1] = q.y; x[2] = q.z;
        } else {
            for (int a = 0; a < 3; ++a) x[a] = V.xr[a * V.n_pad + p];
        }
        const float4 b = V.recb[p];
        const double ex = x[0] - b.x, ey = x[1] - b.y, ez = x[2] - b.z;
        float e = (float)(ex * ex + ey * ey + ez * ez);
        if (!(e <= 3.0e38f)) e = __int_as_float(0x7f800000);
        d2 = fmaxf(d2, e);
    }
    for (int o = 16; o > 0; o >>= 1) d2 = fmaxf(d2, __shfl_xor_sync(0xffffffffu, d2, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&V.ctl->disp_max, __float_as_uint(d2));
}

// ------------------------------------------------------------ launchers ----

static dim3 grid_of(int n, int b) { return dim3((unsigned)((n + b - 1) / b)); }

cudaError_t launch_stage_in(const View &V, int r, int natoms, const double *x, const double *v, const int *type,
                            cudaStream_t s) {
    k_stage_in<<<grid_of(natoms, 256), 256, 0, s>>>(V, r, x, v, type);
    return cudaGetLastError();
}

cudaError_t launch_restage(const View &V, const double *x, const double *v, cudaStream_t s) {
    if (V.prec == MD_PREC_FP64) k_restage<MD_PREC_FP64><<<grid_of(V.n_pad, 256), 256, 0, s>>>(V, x, v);
    else k_restage<MD_PREC_MIXED><<<grid_of(V.n_pad, 256), 256, 0, s>>>(V, x, v);
    return cudaGetLastError();
}

cudaError_t launch_state_out(const View &V, double *x, double *v, double *f, cudaStream_t s) {
    if (V.prec == MD_PREC_FP64) k_state_out<MD_PREC_FP64><<<grid_of(V.n_pad, 256), 256, 0, s>>>(V, x, v, f);
    else k_state_out<MD_PREC_MIXED><<<grid_of(V.n_pad, 256), 256, 0, s>>>(V, x, v, f);
    return cudaGetLastError();
}

cudaError_t launch_ev_reduce(const View &V, double *out, cudaStream_t s) {
    k_ev_tiles<<<grid_of(V.n_tiles * 32, 256), 256, 0, s>>>(V);
    // segments of about kEvSegment tiles, at most kEvSegments in all
    const int per = (V.n_tiles / V.n_rep + kEvSegment - 1) / kEvSegment;
    const int nseg = std::max(1, std::min(per, kEvSegments / V.n_rep));
    k_ev_reduce<<<V.n_rep * nseg, 256, 0, s>>>(V, nseg, out);
    return cudaGetLastError();
}

cudaError_t launch_neighbors_out(const View &V, int *counts, int *nbr, int cap, cudaStream_t s) {
    k_neighbors_out<<<grid_of(V.n_pad, 256), 256, 0, s>>>(V, counts, nbr, cap);
    return cudaGetLastError();
}


cudaError_t launch_halo_pack(const View &V, const int *idx, long long m, int what, int width, const double shift[3],
                             long long n_real, double *buf, cudaStream_t s) {
    if (m <= 0) return cudaSuccess;
    const dim3 g((unsigned)std::min<long long>((m + 255) / 256, 8192));
    if (V.prec == MD_PREC_FP64)
        k_halo_pack<MD_PREC_FP64><<<g, 256, 0, s>>>(V, idx, m, what, width, shift[0], shift[1], shift[2], n_real, buf);
    else
        k_halo_pack<MD_PREC_MIXED><<<g, 256, 0, s>>>(V, idx, m, what, width, shift[0], shift[1], shift[2], n_real, buf);
    return cudaGetLastError();
}

cudaError_t launch_halo_unpack(const View &V, const int *idx, long long m, int what, int width, int accumulate,
                               long long n_real, const double *buf, cudaStream_t s) {
    if (m <= 0) return cudaSuccess;
    const dim3 g((unsigned)std::min<long long>((m + 255) / 256, 8192));
    if (V.prec == MD_PREC_FP64)
        k_halo_unpack<MD_PREC_FP64><<<g, 256, 0, s>>>(V, idx, m, what, width, accumulate, n_real, buf);
    else
        k_halo_unpack<MD_PREC_MIXED><<<g, 256, 0, s>>>(V, idx, m, what, width, accumulate, n_real, buf);
    return cudaGetLastError();
}

cudaError_t launch_disp_max(const View &V, cudaStream_t s) {
    const dim3 g((unsigned)std::min(std::max(1, (V.n_pad + 255) / 256), V.n_sm * 8));
    if (V.prec == MD_PREC_FP64) k_disp_max<MD_PREC_FP64><<<g, 256, 0, s>>>(V);
    else k_disp_max<MD_PREC_MIXED><<<g, 256, 0, s>>>(V);
    return cudaGetLastError();
}

}  // namespace md
