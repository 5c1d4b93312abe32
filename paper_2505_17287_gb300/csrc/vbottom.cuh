// The bottom of the V-cycle in one launch: the coarse levels held in the
// shared memory of one thread-block cluster.
//
// Below some ten thousand cells a multigrid pass launched on its own is bound
// by the launch and by one or two L2 round trips (1.6-2.5 us and a 1-2 us gap,
// whatever its size; a level takes 16 of them per cycle). Here a level's
// coefficients, right-hand side and correction live in the shared memory of
// up to 16 blocks, so that a colour pass costs its shared-memory loads and
// one barrier. (k_vtail, whose passes go through L2, showed that the launch
// alone is not the cost: its passes were no faster than launches.)
//
// Layout: a level's planes along its outer axis (z in 3D, y in 2D) are dealt
// to the blocks in consecutive runs of B; every array is kept per red-black
// colour, each row's cells of a colour packed (h = i >> 1), so that a pass
// reads shared memory without bank conflicts. Each row ends in one zero pad
// entry and the corrections carry a halo plane on either side, so no access
// needs a bound: a face outside the grid has coefficient 0. A thread owns up
// to IT pairs of cells of a level (one of each colour) and keeps their
// coefficients in registers over the level's sweeps. A block pushes the cells
// of its first and last plane into its neighbours' halos as it writes them
// (distributed shared memory), and the transfers read the neighbours' rows
// the same way.
//
// What does not change between cycles (coefficients, transfer tables, the
// coarsest solution operator) is packed once per classification into one image
// per block (k_bottom_image), which a launch copies in with 16-byte
// asynchronous copies: gathering it from the level arrays took 7-17 us of a
// launch, the copy of 150 KB takes about 2.
//
// A cluster barrier costs about 1000 cycles and a block barrier about 40, so
// the levels that one block can take in less than that (BotPar::single on)
// belong to block 0 alone; the other blocks wait for the way back up.
//
// Every cell evaluates the expression of the per-level kernels in their
// order, so the cycle's values are the same bits.
#pragma once

#include <cooperative_groups.h>

namespace ibm {

namespace cg = cooperative_groups;

constexpr int BOT_THREADS = 512, BOT_MAX_LV = 12, BOT_MAX_CTAS = 16;
constexpr int BOT_SMEM = 226 * 1024;   // dynamic shared memory a block may use
// pairs of cells a thread may own: their coefficients take 14 registers each
// in 3D, twice that in FP64, of the 128 that 512 threads leave a thread
template <typename T> struct BotItems { enum { MAX = sizeof(T) == 4 ? 4 : 2 }; };
// levels of at most this many cells are taken by one block: FP32 passes by
// their instruction issue (about 120 cycles per 512 pairs), FP64 passes by
// the block's FP64 pipe (112 cycles per warp of pairs)
template <typename T> struct BotSingle { enum { CELLS = sizeof(T) == 4 ? 4096 : 768 }; };

// gather (restriction) and scatter (prolongation) tables of one axis in
// shared memory: offsets in ints / T entries
struct BotAxis {
    int gi, gw, I, J, w, v;
};

template <typename T>
struct BotLv {
    int nx, ny, nz;
    int nh, rs;         // cells of one colour per row, and the row stride (nh + 1)
    int P, hr, B;       // planes along the outer axis, rows per plane, planes per block
    int it;             // pairs per thread (1, 2 or 4)
    FastDiv fnh, fhr, fnx, fB;
    // offsets (in T) of colour 0 in shared memory and the distance to colour 1:
    // x (with halo planes), f / dinv / tx / pn (rows of the block), ti (one row
    // more), to (one plane more); d and the residual r of colour 0
    int ox, sx, of, od, ot, opn, sc, oi, si, oo, so, odd, orr;
    const T *tx, *ti, *to;       // low-side coefficients (ti: y in 3D; to: outer axis)
    const T *d, *dinv, *pn;
    const T *f;                  // first level: right-hand side in
    T *x;                        // first level: correction out
    BotAxis ax[3];               // to the next level
};

template <typename T>
struct BotPar {
    BotLv<T> lv[BOT_MAX_LV];
    Xfer<T> X[BOT_MAX_LV];       // transfer tables of level l to l + 1 (global)
    int nl, single, nu1, nu2, ncta;
    int nc;                      // cells of the coarsest level
    const T *cm;                 // its solution operator, nc x nc
    int otmp, ocf, ocx, ocm;     // transfer scratch; coarsest f and x, cell-ordered; cm's copy
    int oint;                    // T entry at which the integer tables start
    int sbytes, bytes;           // shared memory: the image's part (first), all of it
    const uint4 *image;          // ncta images of sbytes bytes
    T w;
};

// y = M f with M n x n, one warp per row (the sum's order does not depend on
// the number of warps)
template <typename T>
__device__ __forceinline__ void coarse_apply_dev(int n, const T *M, const T *f, T *x) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int row = threadIdx.x >> 5; row < n; row += nw) {
        T s = T(0);
        for (int q = lane; q < n; q += 32) s += M[row * n + q] * f[q];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) x[row] = s;
    }
}

// planes [p0, p0 + np) of level v in block r
template <typename T>
__device__ __forceinline__ void bot_planes(const BotLv<T> &v, int r, int &p0, int &np) {
    p0 = r * v.B;
    np = max(0, min(v.B, v.P - p0));
}

// parity (j + k) & 1 of local row `row`, and its plane
template <typename T, bool D3>
__device__ __forceinline__ int bot_row(const BotLv<T> &v, int row, int p0, int &lp) {
    if (D3) {
        lp = (int)v.fhr.div((uint32_t)row);
        return (row - lp * v.hr + p0 + lp) & 1;
    }
    lp = row;
    return (p0 + row) & 1;
}

// x entry xi of colour q and its copies in the neighbours' halos (dn, up:
// the neighbours' shared memory; fl bit 1 first plane, bit 2 last plane)
template <typename T>
__device__ __forceinline__ void bot_put(const BotLv<T> &v, T *sm, T *dn, T *up, int q, int xi, int fl, int np, T val) {
    const int o = v.ox + q * v.sx + xi, ps = v.hr * v.rs;
    sm[o] = val;
    if ((fl & 2) && dn) dn[o + v.B * ps] = val;
    if ((fl & 4) && up) up[o - np * ps] = val;
}

// the pairs of cells a thread owns on a level: coefficients of the faces in
// the order x-, x+, (y-, y+,) outer-, outer+ and the inverse diagonal of
// either colour (0: no such cell or inactive), x entry, row parity and
// first / last plane flags
template <typename T, bool D3, int IT>
struct BotOwn {
    static constexpr int NF = D3 ? 6 : 4;
    T k[IT][2][NF], di[IT][2];
    int xi[IT], fl[IT];

    __device__ __forceinline__ void load(const BotLv<T> &v, const T *sm, int p0, int np) {
        const int items = np * v.hr * v.nh, ps = v.hr * v.rs;
#pragma unroll
        for (int u = 0; u < IT; ++u) {
            const int t = (int)threadIdx.x + u * BOT_THREADS;
            di[u][0] = di[u][1] = T(0);
            xi[u] = ps;
            fl[u] = 8;   // no pair
            if (t >= items) continue;
            const int row = (int)v.fnh.div((uint32_t)t), idx = t + row;   // row rs + h
            int lp;
            const int par = bot_row<T, D3>(v, row, p0, lp);
            xi[u] = idx + ps;
            fl[u] = par | (lp == 0 ? 2 : 0) | (lp == np - 1 ? 4 : 0);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int pc = (q + par) & 1, o = 1 - q;
                di[u][q] = sm[v.od + q * v.sc + idx];
                k[u][q][0] = sm[v.ot + q * v.sc + idx];
                k[u][q][1] = sm[v.ot + o * v.sc + idx + pc];
                if (D3) {
                    k[u][q][2] = sm[v.oi + q * v.si + idx];
                    k[u][q][3] = sm[v.oi + o * v.si + idx + v.rs];
                }
                k[u][q][NF - 2] = sm[v.oo + q * v.so + idx];
                k[u][q][NF - 1] = sm[v.oo + o * v.so + idx + ps];
            }
        }
    }

    // f + sum over the faces of T_f x_nb (the order of k_offdiag<T, false>)
    __device__ __forceinline__ T sum(const BotLv<T> &v, const T *sm, int u, int q) const {
        const int ps = v.hr * v.rs, pc = (q + fl[u]) & 1;
        const T *xo = sm + v.ox + (1 - q) * v.sx + xi[u];
        T s = sm[v.of + q * v.sc + xi[u] - ps];
        s += k[u][q][0] * xo[pc - 1];
        s += k[u][q][1] * xo[pc];
        if (D3) {
            s += k[u][q][2] * xo[-v.rs];
            s += k[u][q][3] * xo[v.rs];
        }
        s += k[u][q][NF - 2] * xo[-ps];
        s += k[u][q][NF - 1] * xo[ps];
        return s;
    }

    template <bool OMEGA>
    __device__ __forceinline__ void colour(const BotLv<T> &v, T *sm, T *dn, T *up, int q, bool first, T w, int np) {
        const int ps = v.hr * v.rs;
#pragma unroll
        for (int u = 0; u < IT; ++u) {
            if (!pos(di[u][q])) continue;
            T val;
            if (first) {
                const T f = sm[v.of + q * v.sc + xi[u] - ps];
                val = OMEGA ? w * (f * di[u][q]) : f * di[u][q];
            } else {
                const T s = sum(v, sm, u, q);
                val = OMEGA ? relax(sm[v.ox + q * v.sx + xi[u]], s * di[u][q], w) : s * di[u][q];
            }
            bot_put(v, sm, dn, up, q, xi[u], fl[u], np, val);
        }
    }

    // pn times the residual of colour 0 (colour 1, relaxed last, has none)
    __device__ __forceinline__ void resid(const BotLv<T> &v, T *sm) const {
        const int ps = v.hr * v.rs;
#pragma unroll
        for (int u = 0; u < IT; ++u) {
            if (fl[u] & 8) continue;
            const int idx = xi[u] - ps;
            const T p = sm[v.opn + idx];
            T val = T(0);
            if (pos(p)) {
                const T s = sum(v, sm, u, 0);
                val = p * (s - sm[v.odd + idx] * sm[v.ox + xi[u]]);
            }
            sm[v.orr + idx] = val;
        }
    }
};

struct BotCtx {
    cg::cluster_group cl;
    bool wide;   // the level's barrier is the cluster's
    __device__ __forceinline__ void sync() const {
        if (wide) cl.sync();
        else __syncthreads();
    }
};

// sweeps before the coarse-grid correction and the residual restricted along x
template <typename T, bool OMEGA, bool D3, int IT>
__device__ __forceinline__ void bot_down(const BotPar<T> &P, const BotLv<T> &v, const BotCtx &C, T *sm, const int *si,
                                         T *dn, T *up, int p0, int np, int cnx, FastDiv fcx) {
    BotOwn<T, D3, IT> own;
    own.load(v, sm, p0, np);
    for (int s = 0; s < P.nu1; ++s) {
        own.template colour<OMEGA>(v, sm, dn, up, 0, s == 0, P.w, np);
        C.sync();
        own.template colour<OMEGA>(v, sm, dn, up, 1, false, P.w, np);
        C.sync();
    }
    own.resid(v, sm);
    __syncthreads();
    T *tmp = sm + P.otmp;
    const int *gi = si + v.ax[0].gi;
    const T *gw = sm + v.ax[0].gw, *R = sm + v.orr;
    const int items = np * v.hr * cnx;
    for (int t = threadIdx.x; t < items; t += BOT_THREADS) {
        const int row = (int)fcx.div((uint32_t)t), I = t - row * cnx;
        int lp;
        const int par = bot_row<T, D3>(v, row, p0, lp);
        // (a missing entry has weight 0; its index is clamped)
        T val[4], acc = T(0);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const int i = max(gi[4 * I + s], 0);
            val[s] = ((i + par) & 1) == 0 ? R[row * v.rs + (i >> 1)] : T(0);
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) acc += gw[4 * I + s] * val[s];
        tmp[t] = acc;
    }
}

// sweeps after the coarse-grid correction
template <typename T, bool OMEGA, bool D3, int IT>
__device__ __forceinline__ void bot_up(const BotPar<T> &P, const BotLv<T> &v, const BotCtx &C, T *sm, T *dn, T *up,
                                       int p0, int np) {
    BotOwn<T, D3, IT> own;
    own.load(v, sm, p0, np);
    for (int s = 0; s < P.nu2; ++s) {
        own.template colour<OMEGA>(v, sm, dn, up, 1, false, P.w, np);
        C.sync();
        own.template colour<OMEGA>(v, sm, dn, up, 0, false, P.w, np);
        C.sync();
    }
}

// the images of k_vbottom's blocks (cleared beforehand), one block each
template <typename T, bool D3>
__global__ void __launch_bounds__(BOT_THREADS) k_bottom_image(const __grid_constant__ BotPar<T> P, uint4 *image) {
    grid_begin();
    const int r = blockIdx.x, tid = threadIdx.x;
    T *sm = reinterpret_cast<T *>(reinterpret_cast<char *>(image) + (size_t)r * P.sbytes);
    int *si = reinterpret_cast<int *>(sm + P.oint);
    for (int l = 0; l + 1 < P.nl; ++l) {
        const BotLv<T> &v = P.lv[l], &c = P.lv[l + 1];
        int p0, np;
        bot_planes(v, r, p0, np);
        const int rows = np * v.hr, halo = p0 + np < v.P ? v.hr : 0;
        const int n = np > 0 ? (rows + halo) * v.nx : 0;
        const int64_t g0 = (int64_t)p0 * v.hr * v.nx;
        for (int t = tid; t < n; t += BOT_THREADS) {
            const int row = (int)v.fnx.div((uint32_t)t), i = t - row * v.nx;
            int lp;
            const int q = (i + bot_row<T, D3>(v, row, p0, lp)) & 1, idx = row * v.rs + (i >> 1);
            sm[v.oo + q * v.so + idx] = v.to[g0 + t];
            if (row >= rows) continue;
            sm[v.ot + q * v.sc + idx] = v.tx[g0 + t];
            sm[v.od + q * v.sc + idx] = v.dinv[g0 + t];
            sm[v.opn + q * v.sc + idx] = v.pn[g0 + t];
            if (D3) sm[v.oi + q * v.si + idx] = v.ti[g0 + t];
            if (q == 0) sm[v.odd + idx] = v.d[g0 + t];
        }
        const Xfer<T> &X = P.X[l];
        auto axis = [&](const BotAxis &a, int nf, int nc, const int *G, const T *gw, const int *I, const int *J,
                        const T *w, const T *vv) {
            for (int q = tid; q < 4 * nc; q += BOT_THREADS) {
                si[a.gi + q] = G[q];
                sm[a.gw + q] = gw[q];
            }
            for (int q = tid; q < nf; q += BOT_THREADS) {
                si[a.I + q] = I[q];
                si[a.J + q] = J[q];
                sm[a.w + q] = w[q];
                sm[a.v + q] = vv[q];
            }
        };
        axis(v.ax[0], v.nx, c.nx, X.Gx, X.gwx, X.Ix, X.Jx, X.wx, X.vx);
        axis(v.ax[1], v.ny, c.ny, X.Gy, X.gwy, X.Iy, X.Jy, X.wy, X.vy);
        axis(v.ax[2], v.nz, c.nz, X.Gz, X.gwz, X.Iz, X.Jz, X.wz, X.vz);
    }
    for (int q = tid; q < P.nc * P.nc; q += BOT_THREADS) sm[P.ocm + q] = P.cm[q];
}

template <typename T, bool OMEGA, bool D3>
__global__ void __launch_bounds__(BOT_THREADS, 1) k_vbottom(const __grid_constant__ BotPar<T> P) {
    extern __shared__ double bot_smem[];
    T *sm = reinterpret_cast<T *>(bot_smem);
    const int *si = reinterpret_cast<const int *>(sm + P.oint);
    grid_release();
    BotCtx C{cg::this_cluster(), false};
    const int r = P.ncta > 1 ? (int)C.cl.block_rank() : 0, tid = threadIdx.x;
    {
        const char *src = reinterpret_cast<const char *>(P.image) + (size_t)r * P.sbytes;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(sm);
        for (int q = 16 * tid; q < P.sbytes; q += 16 * BOT_THREADS)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + q), "l"(src + q) : "memory");
        // the corrections start at zero, their halos and pads included
        for (int l = 0; l + 1 < P.nl; ++l) {
            const BotLv<T> &v = P.lv[l];
            if (r * v.B < v.P)
                for (int q = tid; q < 2 * v.sx; q += BOT_THREADS) sm[v.ox + q] = T(0);
        }
    }
    // (the image is older than the previous kernel: it is written while the
    // stream is idle or before a copy that every kernel after it waits for)
    grid_wait();
    {
        const BotLv<T> &v = P.lv[0];
        int p0, np;
        bot_planes(v, r, p0, np);
        const int n = np * v.hr * v.nx;
        const int64_t g0 = (int64_t)p0 * v.hr * v.nx;
#pragma unroll 4
        for (int t = tid; t < n; t += BOT_THREADS) {
            const int row = (int)v.fnx.div((uint32_t)t), i = t - row * v.nx;
            int lp;
            const int q = (i + bot_row<T, D3>(v, row, p0, lp)) & 1;
            sm[v.of + q * v.sc + row * v.rs + (i >> 1)] = v.f[g0 + t];
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    // (every block's halos are cleared before a neighbour writes into them)
    C.wide = P.ncta > 1;
    C.sync();
    T *tmp = sm + P.otmp;
    // the transfer scratch of the block that holds plane pl of level v
    auto scratch = [&](const BotLv<T> &v, int pl, int &lrow) -> const T * {
        const int o = (int)v.fB.div((uint32_t)pl);
        lrow = (pl - o * v.B) * v.hr;
        return C.wide ? C.cl.map_shared_rank(tmp, o) : tmp;
    };
    const int lend = r == 0 ? P.nl - 1 : P.single;   // levels this block takes part in
    for (int l = 0; l < lend; ++l) {
        const BotLv<T> &v = P.lv[l], &c = P.lv[l + 1];
        int p0, np, c0, cnp;
        bot_planes(v, r, p0, np);
        bot_planes(c, r, c0, cnp);
        C.wide = l < P.single;
        T *dn = C.wide && r > 0 && np > 0 ? C.cl.map_shared_rank(sm, r - 1) : nullptr;
        T *up = C.wide && np > 0 && p0 + np < v.P ? C.cl.map_shared_rank(sm, r + 1) : nullptr;
        if (v.it == 1) bot_down<T, OMEGA, D3, 1>(P, v, C, sm, si, dn, up, p0, np, c.nx, c.fnx);
        else if (v.it == 2) bot_down<T, OMEGA, D3, 2>(P, v, C, sm, si, dn, up, p0, np, c.nx, c.fnx);
        else bot_down<T, OMEGA, D3, BotItems<T>::MAX>(P, v, C, sm, si, dn, up, p0, np, c.nx, c.fnx);
        C.sync();
        // along y and z into level l + 1
        const bool last = l + 2 == P.nl;
        const int items = cnp * c.hr * c.nx;
        for (int t = tid; t < items; t += BOT_THREADS) {
            const int row = (int)c.fnx.div((uint32_t)t), I = t - row * c.nx;
            int lp;
            const int par = bot_row<T, D3>(c, row, c0, lp), q = (I + par) & 1;
            const int J = D3 ? row - lp * c.hr : c0 + row, K = D3 ? c0 + lp : 0;
            const int idx = row * c.rs + (I >> 1);
            T acc = T(0);
            if (last || pos(sm[c.od + q * c.sc + idx])) {
                // all reads (from up to 16 rows, some in other blocks) are
                // issued before the sums; a missing entry has weight 0
                T val[4][4];
#pragma unroll
                for (int s3 = 0; s3 < (D3 ? 4 : 1); ++s3) {
                    const int k = max(si[v.ax[2].gi + 4 * K + s3], 0);
#pragma unroll
                    for (int s2 = 0; s2 < 4; ++s2) {
                        const int j = max(si[v.ax[1].gi + 4 * J + s2], 0);
                        int lrow;
                        const T *src = scratch(v, D3 ? k : j, lrow);
                        val[s3][s2] = src[(lrow + (D3 ? j : 0)) * c.nx + I];
                    }
                }
#pragma unroll
                for (int s3 = 0; s3 < (D3 ? 4 : 1); ++s3) {
                    T a2 = T(0);
#pragma unroll
                    for (int s2 = 0; s2 < 4; ++s2) a2 += sm[v.ax[1].gw + 4 * J + s2] * val[s3][s2];
                    acc += sm[v.ax[2].gw + 4 * K + s3] * a2;
                }
            }
            // (inactive cells of the coarsest level have zero rows and columns in cm)
            if (last) sm[P.ocf + t] = acc;
            else sm[c.of + q * c.sc + idx] = acc;
        }
        __syncthreads();
    }
    if (r == 0) {
        coarse_apply_dev<T>(P.nc, sm + P.ocm, sm + P.ocf, sm + P.ocx);
        __syncthreads();
    }
    for (int l = lend - 1; l >= 0; --l) {
        const BotLv<T> &v = P.lv[l], &c = P.lv[l + 1];
        int p0, np, c0, cnp;
        bot_planes(v, r, p0, np);
        bot_planes(c, r, c0, cnp);
        C.wide = l < P.single;
        T *dn = C.wide && r > 0 && np > 0 ? C.cl.map_shared_rank(sm, r - 1) : nullptr;
        T *up = C.wide && np > 0 && p0 + np < v.P ? C.cl.map_shared_rank(sm, r + 1) : nullptr;
        const bool last = l + 2 == P.nl;
        const int cps = c.hr * c.rs, ps = v.hr * v.rs;
        // prolongation along x of the block's coarse rows
        {
            const int items = cnp * c.hr * v.nx;
            for (int t = tid; t < items; t += BOT_THREADS) {
                const int row = (int)v.fnx.div((uint32_t)t), i = t - row * v.nx;
                int lp;
                const int par = bot_row<T, D3>(c, row, c0, lp);
                auto cx = [&](int I) -> T {
                    return last ? sm[P.ocx + row * c.nx + I]
                                : sm[c.ox + ((I + par) & 1) * c.sx + cps + row * c.rs + (I >> 1)];
                };
                const int J2 = si[v.ax[0].J + i];
                T val = sm[v.ax[0].w + i] * cx(si[v.ax[0].I + i]);
                if (J2 >= 0) val += sm[v.ax[0].v + i] * cx(J2);
                tmp[t] = val;
            }
        }
        C.sync();
        // along y and z, and the correction
        const int items = np * v.hr * v.nx;
        for (int t = tid; t < items; t += BOT_THREADS) {
            const int row = (int)v.fnx.div((uint32_t)t), i = t - row * v.nx;
            int lp;
            const int par = bot_row<T, D3>(v, row, p0, lp), q = (i + par) & 1, idx = row * v.rs + (i >> 1);
            const T p = sm[v.opn + q * v.sc + idx];
            if (!pos(p)) continue;
            const int j = D3 ? row - lp * v.hr : p0 + row, k = D3 ? p0 + lp : 0;
            // (no second coarse index: weight 0, the first one's value read again)
            T val[2][2];
            int lrow;
#pragma unroll
            for (int q3 = 0; q3 < (D3 ? 2 : 1); ++q3) {
                const int kc = D3 && q3 && si[v.ax[2].J + k] >= 0 ? si[v.ax[2].J + k] : si[v.ax[2].I + k];
#pragma unroll
                for (int q2 = 0; q2 < 2; ++q2) {
                    const int jc = q2 && si[v.ax[1].J + j] >= 0 ? si[v.ax[1].J + j] : si[v.ax[1].I + j];
                    const T *src = scratch(c, D3 ? kc : jc, lrow);
                    val[q3][q2] = src[(lrow + (D3 ? jc : 0)) * v.nx + i];
                }
            }
            T acc = T(0);
#pragma unroll
            for (int q3 = 0; q3 < (D3 ? 2 : 1); ++q3) {
                T a2 = T(0);
                a2 += sm[v.ax[1].w + j] * val[q3][0];
                a2 += sm[v.ax[1].v + j] * val[q3][1];
                acc += sm[(q3 ? v.ax[2].v : v.ax[2].w) + k] * a2;
            }
            const int fl = (lp == 0 ? 2 : 0) | (lp == np - 1 ? 4 : 0);
            bot_put(v, sm, dn, up, q, idx + ps, fl, np, sm[v.ox + q * v.sx + idx + ps] + acc * p);
        }
        C.sync();
        if (v.it == 1) bot_up<T, OMEGA, D3, 1>(P, v, C, sm, dn, up, p0, np);
        else if (v.it == 2) bot_up<T, OMEGA, D3, 2>(P, v, C, sm, dn, up, p0, np);
        else bot_up<T, OMEGA, D3, BotItems<T>::MAX>(P, v, C, sm, dn, up, p0, np);
    }
    {
        const BotLv<T> &v = P.lv[0];
        int p0, np;
        bot_planes(v, r, p0, np);
        const int n = np * v.hr * v.nx;
        const int64_t g0 = (int64_t)p0 * v.hr * v.nx;
        for (int t = tid; t < n; t += BOT_THREADS) {
            const int row = (int)v.fnx.div((uint32_t)t), i = t - row * v.nx;
            int lp;
            const int q = (i + bot_row<T, D3>(v, row, p0, lp)) & 1;
            v.x[g0 + t] = sm[v.ox + q * v.sx + v.hr * v.rs + row * v.rs + (i >> 1)];
        }
    }
}

}  // namespace ibm
