// Near-body band sweeps of the preconditioner: damped Jacobi sweeps of the
// full ghost-cell operator on the ghost cells and the fluid cells near them,
// after the ghost rows are set from the V-cycle's output.
//
// A sweep of a few thousand cells is bound by the latency of its gathers, in
// FP64 by the pipe (operations of one block: 2 per clock). So all sweeps run
// in one launch: every row of the band is read once into registers (up to
// eight coefficients and the band positions of its neighbours, tabulated per
// classification), and a sweep is the neighbours' reads, the row's arithmetic
// and one barrier. A band that one block can own is kept in its shared memory;
// a larger one in two alternating L2-resident vectors of a thread-block
// cluster; a band too large for that takes one launch per sweep on the whole
// device.
//
// Before, one block of 1024 threads swept bands up to 8192 cells through
// global memory (12 us for 8 sweeps of a 2D band, 73 us for one of the 96^3
// sphere cases, 430 us in FP64 at 129x85x77) and two launches per sweep the
// larger ones.
#pragma once

#include <cooperative_groups.h>

namespace ibm {

constexpr int BAND_THREADS = 512, BAND_MAX_CTAS = 16;
// rows a thread of one block may own (their coefficients and neighbours take 20
// registers each, 30 in FP64)
template <typename T> struct BandRows { enum { MAX = sizeof(T) == 4 ? 4 : 1 }; };

// nbr[m nb + q]: band position of neighbour m of band cell q (FLUID: -x, +x,
// -y, +y, -z, +z, itself where there is no cell; GHOST: its eight stencil
// cells), or -1 outside the band, whose values the sweeps do not change
struct BandDev {
    int nb;
    const int64_t *cell, *gpos;
    const int *nbr;
};

// cell of neighbour m of the FLUID cell c at (i, j, k)
__device__ __forceinline__ int64_t band_face_cell(const GridDev &g, int64_t c, int i, int j, int k, int m) {
    const int64_t st = m < 2 ? 1 : (m < 4 ? (int64_t)g.nx : (int64_t)g.nx * g.ny);
    const int p = m < 2 ? i : (m < 4 ? j : k), n = m < 2 ? g.nx : (m < 4 ? g.ny : g.nz);
    if (m & 1) return p < n - 1 ? c + st : c;
    return p > 0 ? c - st : c;
}

__global__ void k_band_nbr(GridDev g, GhostDev gh, int nb, const int64_t *band, const int64_t *gpos, int *nbr) {
    grid_begin();
    const int t = blockIdx.x * blockDim.x + threadIdx.x, m = blockIdx.y;
    if (t >= nb) return;
    const int64_t c = band[t], gq = gpos[t];
    int64_t n = c;
    if (gq >= 0) {
        n = gh.sidx[8 * gq + m];
    } else if (m < 6) {
        int i, j, k;
        split3(g, (uint32_t)c, i, j, k);
        n = band_face_cell(g, c, i, j, k, m);
    }
    int lo = 0, hi = nb;   // the band is ascending
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (band[mid] < n) lo = mid + 1;
        else hi = mid;
    }
    nbr[band_slot(nb, m, t)] = lo < nb && band[lo] == n ? lo : -1;
}

// one row of the band: v - (A z) and the damped inverse diagonal
template <typename T>
struct BandRow {
    T k[8], v, wd, dg, zc;
    int idx[8];
    bool ghost;

    // row of band cell q; zh[m nb + q] takes the values outside the band (their
    // entries in idx serve the sweeps of one launch, whose bands are small)
    __device__ __forceinline__ void load(const GridDev &g, const GhostDev &gh, const OpT<T> &o, const BandDev &b,
                                         const uint8_t *type, const T *vv, const T *z, T omega, int q, T *zh) {
        const int64_t c = b.cell[q], gq = b.gpos[q];
        int64_t n[8];
        ghost = gq >= 0;
        v = vv[c];
        dg = T(0);
#pragma unroll
        for (int m = 0; m < 8; ++m) idx[m] = b.nbr[band_slot(b.nb, m, q)];
        if (ghost) {
            // the ghost row solved for its value from the FLUID corners
            zc = v;
            wd = omega;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                n[m] = gh.sidx[8 * gq + m];
                k[m] = o.wp[8 * gq + m];
                if (type[n[m]] == FLUID) zc += k[m] * z[n[m]];
            }
        } else {
            int i, j, l;
            split3(g, (uint32_t)c, i, j, l);
            zc = z[c];
#pragma unroll
            for (int m = 0; m < 8; ++m) n[m] = m < 6 ? band_face_cell(g, c, i, j, l, m) : c;
            k[0] = o.cxm[i];
            k[1] = o.cxp[i];
            k[2] = o.cym[j];
            k[3] = o.cyp[j];
            k[4] = g.ndim == 3 ? o.czm[l] : T(0);
            k[5] = g.ndim == 3 ? o.czp[l] : T(0);
            k[6] = k[7] = T(0);
            if constexpr (sizeof(T) == 8) dg = o.dg[c];
            else dg = o.cxs[i] + o.cys[j] + (g.ndim == 3 ? o.czs[l] : T(0));
            wd = -omega / dg;
        }
#pragma unroll
        for (int m = 0; m < 8; ++m)
            if (idx[m] < 0) {
                const size_t h = band_slot(b.nb, m, q);
                zh[h] = z[n[m]];
                idx[m] = -1 - (int)h;
            }
    }

    template <bool LOCAL>
    __device__ __forceinline__ void sweep(const T *cur, const T *zh) {
        T x[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const T *p = idx[m] >= 0 ? cur + idx[m] : zh + (-1 - idx[m]);
            x[m] = LOCAL ? *p : __ldcg(p);   // (other blocks write cur: read it from L2)
        }
        T s;
        if (ghost) {
            s = zc;
#pragma unroll
            for (int m = 0; m < 8; ++m) s -= k[m] * x[m];
        } else if (sizeof(T) == 4) {
            // FP32: difference form, so constants are annihilated exactly
            s = k[0] * (x[0] - zc) + k[1] * (x[1] - zc) + k[2] * (x[2] - zc) + k[3] * (x[3] - zc);
            s += k[4] * (x[4] - zc) + k[5] * (x[5] - zc);
        } else {
            s = k[0] * x[0] + k[1] * x[1] + k[2] * x[2] + k[3] * x[3];
            s += k[4] * x[4] + k[5] * x[5];
            s -= dg * zc;
        }
        zc += wd * (v - s);
    }
};

// all sweeps in one launch of one cluster (LOCAL: one block, the vectors in
// shared memory; else buf, 10 nb entries: two vectors and the outside values)
template <typename T, int IT, bool LOCAL>
__global__ void __launch_bounds__(BAND_THREADS, 1)
    k_band_sweeps(GridDev g, GhostDev gh, OpT<T> o, BandDev b, const uint8_t *type, const T *v, T *z, T omega, int sweeps,
                  T *buf, int ncta) {
    extern __shared__ double band_smem[];
    grid_begin();
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    T *w = LOCAL ? reinterpret_cast<T *>(band_smem) : buf;
    T *cur = w, *nxt = w + b.nb, *zh = w + 2 * (size_t)b.nb;
    const int nt = ncta * BAND_THREADS, q0 = blockIdx.x * BAND_THREADS + threadIdx.x;
    BandRow<T> row[IT];
#pragma unroll
    for (int u = 0; u < IT; ++u) {
        const int q = q0 + u * nt;
        if (q < b.nb) {
            row[u].load(g, gh, o, b, type, v, z, omega, q, zh);
            cur[q] = row[u].zc;
        }
    }
    for (int s = 0; s < sweeps; ++s) {
        if (LOCAL) __syncthreads();
        else cl.sync();
#pragma unroll
        for (int u = 0; u < IT; ++u) {
            const int q = q0 + u * nt;
            if (q < b.nb) {
                row[u].template sweep<LOCAL>(cur, zh);
                nxt[q] = row[u].zc;
            }
        }
        T *t = cur;
        cur = nxt;
        nxt = t;
    }
#pragma unroll
    for (int u = 0; u < IT; ++u) {
        const int q = q0 + u * nt;
        if (q < b.nb) z[b.cell[q]] = row[u].zc;
    }
}

// one sweep per launch: the band's start values and the outside values
template <typename T>
__global__ void k_band_start(GridDev g, GhostDev gh, OpT<T> o, BandDev b, const uint8_t *type, const T *v, const T *z,
                             T omega, T *cur, T *zh) {
    grid_begin();
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= b.nb) return;
    BandRow<T> r;
    r.load(g, gh, o, b, type, v, z, omega, q, zh);
    cur[q] = r.zc;
}

// a sweep (from cur to nxt; out not null: into out at the band's cells)
template <typename T>
__global__ void k_band_sweep(GridDev g, GhostDev gh, OpT<T> o, BandDev b, const T *v, T omega, const T *cur,
                             const T *zh, T *nxt, T *out) {
    grid_begin();
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= b.nb) return;
    const int64_t c = b.cell[q], gq = b.gpos[q];
    T x[8];
    const T zc = cur[q];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        const size_t h = band_slot(b.nb, m, q);
        const int n = b.nbr[h];
        x[m] = n >= 0 ? cur[n] : zh[h];
    }
    T s, wd;
    if (gq >= 0) {
        s = zc;
        wd = omega;
#pragma unroll
        for (int m = 0; m < 8; ++m) s -= o.wp[8 * gq + m] * x[m];
    } else {
        int i, j, k;
        split3(g, (uint32_t)c, i, j, k);
        const T czm = g.ndim == 3 ? o.czm[k] : T(0), czp = g.ndim == 3 ? o.czp[k] : T(0);
        if constexpr (sizeof(T) == 4) {
            s = o.cxm[i] * (x[0] - zc) + o.cxp[i] * (x[1] - zc) + o.cym[j] * (x[2] - zc) + o.cyp[j] * (x[3] - zc);
            s += czm * (x[4] - zc) + czp * (x[5] - zc);
            wd = -omega / (o.cxs[i] + o.cys[j] + (g.ndim == 3 ? o.czs[k] : T(0)));
        } else {
            const T dg = o.dg[c];
            s = o.cxm[i] * x[0] + o.cxp[i] * x[1] + o.cym[j] * x[2] + o.cyp[j] * x[3];
            s += czm * x[4] + czp * x[5];
            s -= dg * zc;
            wd = -omega / dg;
        }
    }
    const T r = zc + wd * (v[c] - s);
    if (out) out[c] = r;
    else nxt[q] = r;
}

}  // namespace ibm
