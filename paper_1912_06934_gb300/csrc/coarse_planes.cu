// Coarse solver M_c^-1 = A_c^-1 (Alg. 2 and Alg. 3 of arXiv 1912.06934) in
// FP64, built on the 3^d stencil of the Galerkin operator.
//
// A_c couples a coarse node only with the coarse nodes at most one coarse
// step away on every axis (Eq. 3 with the support regions of Sec. 2.1).
// Numbered plane by plane along the last grid axis (z in 3D, y in 2D), A_c is
// block tridiagonal: D_k on the diagonal (the couplings inside plane k),
// L_k = A_c[k][k-1] and U_k = A_c[k][k+1]. It is factorised from both ends
// towards the middle plane h = np / 2 (a twisted block factorisation), the
// two ends concurrently on two thread-block clusters:
//   planes k < h:  S_k = D_k - L_k G_{k-1},  G_k = S_k^-1 U_k;
//   planes k > h:  S_k = D_k - U_k G_{k+1},  G_k = S_k^-1 L_k;
//   plane h:       S_h = D_h - L_h G_{h-1} - U_h G_{h+1},
// which needs only the inverse of each plane's dense Schur complement S_k
// (m x m, m = nodes per plane x block size): np m^3 multiply-adds instead of
// the (np m)^3 of a dense inverse, along a dependent chain of about np / 2
// planes instead of np. A_c^-1 v is then
//   y_k = S_k^-1 (v_k - L_k y_{k-1}) (k < h),  y_k = S_k^-1 (v_k - U_k y_{k+1}) (k > h),
//   w_h = S_h^-1 (v_h - L_h y_{h-1} - U_h y_{h+1}),
//   w_k = y_k - G_k w_{k+1} (k < h),  w_k = y_k - G_k w_{k-1} (k > h).
//
// Every S_k is inverted by Gauss-Jordan elimination with partial pivoting
// inside the plane (ties to the lowest row; magnitudes compared through the
// integer order of their FP64 bit patterns). Both the factorisation and the
// application run as thread-block clusters (up to 16 CTAs on 16 SMs) whose
// CTAs own columns (factorisation, dealt out in turn) or contiguous rows
// (application, see there) and exchange pivot columns and partial vectors through
// distributed shared memory, with hardware cluster barriers between steps (no
// spin waits).
#include "common.cuh"
#include <cooperative_groups.h>
#include <initializer_list>
#include <mutex>

namespace cg = cooperative_groups;

namespace msrsb {

// Offsets and sizes of the plane structure. Node J of the coarse grid
// (x fastest) lies in plane k = J / PN at in-plane index u = J % PN; dof
// J * bd + l of A_c is row u * bd + l of plane k. Stencil entry q of a node
// couples it with the node at offset (q%3 - 1, (q/3)%3 - 1, q/9 - 1); with NI
// in-plane offsets a (9 in 3D, 3 in 2D) and plane offset o in {-1, 0, 1},
// q = a + NI * (o + 1).
struct PlaneGeom {
    int dim, nb0, nb1, bd;
    int np;   // planes
    int PN;   // coarse nodes per plane
    int m;    // rows of a plane = PN * bd
    int NI;   // in-plane stencil offsets
    int nq;   // stencil entries per node (3^dim)
};

// In-plane neighbour of local node u at in-plane offset a, or -1.
__device__ __forceinline__ int plane_nbr(const PlaneGeom &G, int u, int a) {
    if (G.dim == 3) {
        const int u0 = u % G.nb0 + a % 3 - 1, u1 = u / G.nb0 + a / 3 - 1;
        return (u0 < 0 || u0 >= G.nb0 || u1 < 0 || u1 >= G.nb1) ? -1 : u0 + G.nb0 * u1;
    }
    const int u0 = u + a - 1;
    return (u0 < 0 || u0 >= G.nb0) ? -1 : u0;
}

// In-plane offset index a with node v = plane_nbr(u, a), or -1 if v is not
// adjacent to u.
__device__ __forceinline__ int plane_offset(const PlaneGeom &G, int u, int v) {
    if (G.dim == 3) {
        const int d0 = v % G.nb0 - u % G.nb0, d1 = v / G.nb0 - u / G.nb0;
        return (d0 < -1 || d0 > 1 || d1 < -1 || d1 > 1) ? -1 : (d0 + 1) + 3 * (d1 + 1);
    }
    const int d0 = v - u;
    return (d0 < -1 || d0 > 1) ? -1 : d0 + 1;
}

// Stencil value: row (node J, component l), stencil entry q, column component c.
__device__ __forceinline__ double st_val(const double *__restrict__ Acs, const PlaneGeom &G, int J, int q, int l,
                                         int c) {
    return Acs[(((long)J * G.nq + q) * G.bd + l) * G.bd + c];
}

// v - sum over in-plane neighbours b and components c of the coupling of
// (node J, component l) with plane p's node (stencil entries from `base`)
// times vec[(neighbour * bd + c) * stride] (vec points at the column or row
// of plane p wanted)
__device__ __forceinline__ double sub_coupling(double v, const PlaneGeom &G, const double *__restrict__ Acs, int J,
                                               int u, int l, int base, const double *vec, long stride) {
    for (int b = 0; b < G.NI; ++b) {
        const int tn = plane_nbr(G, u, b);
        if (tn < 0) continue;
        for (int c = 0; c < G.bd; ++c) v = fma(-st_val(Acs, G, J, b + base, l, c), vec[(tn * G.bd + c) * stride], v);
    }
    return v;
}

constexpr int kPlaneThreads = 256;
constexpr int kPlaneMaxCols = 128;  // columns of a plane one CTA of the factorisation owns
constexpr int kPlaneMaxRows = 768;  // rows of a plane the factorisation takes
constexpr int kPlaneMaxCluster = 16;
constexpr int kFactorThreads = kPlaneThreads + 32;  // a warp of its own for the pivot's reciprocal

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// shared-memory address of p in CTA `rank` of the cluster
__device__ __forceinline__ unsigned map_rank(const void *p, int rank) {
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void st_rank(unsigned a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void st_rank(unsigned a, int v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ double ld_rank(unsigned a) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}

// The lane (as a mask of one bit) with the largest key, ties to the lowest row;
// 0 when every key is negative. Keys are magnitudes as 63-bit integers: the
// high words decide unless they tie.
__device__ __forceinline__ unsigned plane_top(long long key, int row) {
    const unsigned hi = key < 0 ? 0u : (unsigned)(key >> 32) + 1u, mh = __reduce_max_sync(0xffffffffu, hi);
    if (!mh) return 0u;
    unsigned who = __ballot_sync(0xffffffffu, hi == mh);
    if (who & (who - 1u)) {
        const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)key : 0u);
        const bool top = hi == mh && (unsigned)key == ml;
        const unsigned r = __reduce_min_sync(0xffffffffu, top ? (unsigned)row : 0xffffffffu);
        who = __ballot_sync(0xffffffffu, top && (unsigned)row == r);
    }
    return who;
}

// Factorisation. With middle = 0 the grid holds one cluster per side (side 0:
// planes 0 .. h-1 upwards, side 1: planes np-1 .. h+1 downwards); with
// middle = 1 one cluster takes plane h. Outputs (row-major m x m per plane):
// X_k with S_k^-1 = X_k Pi_k (Pi_k the row interchanges of the elimination,
// kept as the gather pi_k: (Pi_k v)[i] = v[pi_k[i]]), and G_k for k != h.
// status[0] = 1 + (global row) on a zero pivot. keep: a CTA's columns of the
// last G_k stay in shared memory, where its columns of the next S_k need them.
//
// The elimination is a chain of m pivot steps per plane. A step's update (m^2
// FMAs over the cluster) keeps the FP64 pipes of 16 SMs busy for 1.4 us at m =
// 256 (measured: an SM starts a warp's FP64 FMA every 19 cycles); the pivot
// search, the exchange of the pivot column and the cluster barrier are latency,
// and took 3 us when they followed it. They now run beside it, and are short:
//  - columns are dealt out in turn (column j to CTA j mod nct), so the owner of
//    the next pivot column changes at every step;
//  - at step kk the owner of column kk + 1 brings that column up to date first,
//    finds its pivot, and stores the column into every CTA's shared memory
//    before it arrives at the barrier; the others arrive at once. All then
//    update their own columns, and wait for the barrier only at the start of
//    step kk + 1;
//  - the pivot's reciprocal (a chain of FP64 operations as long as the column's
//    exchange) is taken by a warp of its own beside that exchange;
//  - a warp updates whole columns, the pivot column's rows of a lane in RPL
//    registers, so that row interchange, pivot-row entry and update need no
//    CTA barrier and read no pivot column twice;
//  - a thread's row of S_k takes its couplings from registers, and the columns of
//    X_k that G_k combines are listed once per plane, so that their loads from
//    other CTAs are independent of one another.
// Three pivot-column buffers: a CTA arrives for column kk + 1 when it has done
// with step kk - 1, so the column that a passed barrier lets the next owner
// overwrite is two steps old. Every arrive releases, the readers' too: what orders
// their reads before that store is the barrier (a relaxed arrive of the CTAs that
// only read gave the same times). The arithmetic and its order are those of the
// plain elimination. Measured, both factorisation launches: 128^3 (9 dependent
// planes of 256) 11.2 -> 4.9 ms, 48^3 elasticity (5 of 243) 5.6 -> 2.7 ms, 64^3 (5
// of 64, with the explicit inverse) 0.79 -> 0.61 ms; of a step's 4,200 cycles at
// m = 256 the update takes 2,790, the owner's column, search, exchange and
// release 4,000 beside it.
template <int RPL>
__global__ void __launch_bounds__(kFactorThreads, 1) plane_factor_kernel(PlaneGeom G, int h, int middle, int keep,
                                                                      const double *__restrict__ Acs,
                                                                      double *__restrict__ X,
                                                                      double *__restrict__ Gm, int *__restrict__ pi,
                                                                      int *__restrict__ status) {
    constexpr int RPT = (32 * RPL + kPlaneThreads - 1) / kPlaneThreads;  // rows per thread
    constexpr int kWarps = kPlaneThreads / 32;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), nct = (int)cluster.num_blocks();
    // side 0: planes 0 .. h-1 upwards; side 1: planes np-1 .. h+1 downwards;
    // middle: plane h with the Schur complements from both sides
    const int side = middle ? 0 : (int)(blockIdx.x / nct);
    const int nplanes = middle ? 1 : (side == 0 ? h : G.np - 1 - h);
    const int m = G.m, bd = G.bd, NI = G.NI;
    const int cw = (m + nct - 1) / nct;
    const int ncol = rank < m ? (m - rank + nct - 1) / nct : 0;  // own columns: rank, rank + nct, ...
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool worker = tid < kPlaneThreads;
    extern __shared__ double sm[];
    double *Sown = sm;                     // own columns of S_k, column-major [cw][m]
    double *pcol = Sown + (long)cw * m;    // pivot columns [3][m], written by their owners
    int *pil = (int *)(pcol + 3 * m);      // gather pi [m]
    int *pinv = pil + m;                   // inverse of pi [m]
    double *Gown = (double *)(pinv + m);   // own columns of the last G_k [cw][m] (keep)
    __shared__ double s_inv[3], s_best[kWarps], s_top;
    __shared__ int s_p[3], s_bad[3], s_idx[kWarps];
    __shared__ double s_gval[kWarps][27];    // one column's list of a warp: value, address of X's column
    __shared__ unsigned s_gcol[kWarps][27];
    unsigned rcol[kPlaneMaxCluster];  // the pivot buffers of every CTA
#pragma unroll
    for (int r = 0; r < kPlaneMaxCluster; ++r) rcol[r] = map_rank(pcol, r < nct ? r : 0);

    // Column kk (local index jl) is up to date through step kk - 1 and its rows
    // v[] (row tid + 256 t) are in this CTA's registers: find the pivot among
    // rows kk .. m-1 (largest magnitude, ties to the lowest row), store the
    // column with rows kk and pivot interchanged here and in every CTA's pivot
    // buffer, with 1 / pivot.
    auto publish = [&](int kk, int jl, const double (&v)[RPT]) {
        if (worker) {
            long long best = -1;
            int bi = m;
            double bv = 0.0;
#pragma unroll
            for (int t = 0; t < RPT; ++t) {
                const int i = tid + t * kPlaneThreads;
                if (i >= kk && i < m) {
                    const long long a = __double_as_longlong(v[t]) & 0x7fffffffffffffffLL;
                    if (a > best) {
                        best = a;
                        bi = i;
                        bv = v[t];
                    }
                }
                if (i == kk) s_top = v[t];
            }
            const unsigned who = plane_top(best, bi);
            if (who ? who >> lane & 1u : lane == 0) {
                s_idx[warp] = who ? bi : m;
                s_best[warp] = who ? bv : 0.0;
            }
        }
        __syncthreads();
        int bi;
        double pv;
        {  // the warps' candidates, one per lane
            const int w = lane & (kWarps - 1);
            const int i2 = s_idx[w];
            const double v2 = s_best[w];
            const long long best = __double_as_longlong(v2) & 0x7fffffffffffffffLL;
            const unsigned who = plane_top(i2 < m && lane < kWarps ? best : -1, i2);
            const int src = who ? __ffs(who) - 1 : 0;
            bi = who ? __shfl_sync(0xffffffffu, i2, src) : m;
            pv = __shfl_sync(0xffffffffu, v2, src);
        }
        // zero, infinite or NaN, by the bits
        const long long pb = __double_as_longlong(pv) & 0x7fffffffffffffffLL;
        const bool bad = bi >= m || pb == 0 || pb >= 0x7ff0000000000000LL;
        const int p = bi < m ? bi : kk, buf = kk % 3;
        if (!worker) {  // the pivot's row and reciprocal, one destination a lane
            if (lane < nct) {
                st_rank(map_rank(s_p + buf, lane), p);
                st_rank(map_rank(s_bad + buf, lane), bad ? 1 : 0);
                st_rank(map_rank(s_inv + buf, lane), bad ? 0.0 : 1.0 / pv);
            }
            return;
        }
        const double vt = s_top;
        double *col = Sown + (long)jl * m;
#pragma unroll
        for (int t = 0; t < RPT; ++t) {
            const int i = tid + t * kPlaneThreads;
            if (i < m) {
                const double x = bad ? v[t] : (i == kk ? pv : (i == p ? vt : v[t]));
                const unsigned at = (unsigned)(buf * m + i) * 8u;
                col[i] = x;
#pragma unroll
                for (int r = 0; r < kPlaneMaxCluster; ++r)
                    if (r < nct) st_rank(rcol[r] + at, x);
            }
        }
    };

    cluster.sync();  // every CTA runs before another stores into its shared memory
    for (int st = 0; st < nplanes; ++st) {
        const int k = middle ? h : (side == 0 ? st : G.np - 1 - st);
        // ---- S_k = D_k - C_{k,p} G_p over the planes p finished before it, own columns ----
        // (C_{k,p}: the couplings of plane k with plane p = k -+ 1, stencil entries from base 0 / 2 NI)
        const int Jbase = k * G.PN;
        int pa = -1, pb = -1;  // planes p (their G_p) and stencil bases
        int ba = 0, bb = 0;
        if (middle) {
            if (h > 0) pa = h - 1, ba = 0;
            if (h + 1 < G.np) pb = h + 1, bb = 2 * NI;
        } else if (st > 0) {
            pa = side == 0 ? k - 1 : k + 1;
            ba = side == 0 ? 0 : 2 * NI;
        }
        if (worker)
            for (int i = tid; i < m; i += kPlaneThreads) {  // a thread's row, all own columns
                const int ui = i / bd, l = i - ui * bd;
                int nbr[9];  // dof 0 of the row's in-plane neighbours, -1 off the grid
#pragma unroll
                for (int a = 0; a < 9; ++a) {
                    nbr[a] = a < NI ? plane_nbr(G, ui, a) : -1;
                    if (nbr[a] >= 0) nbr[a] *= bd;
                }
                for (int jl = 0; jl < ncol; ++jl) {
                    const int j = rank + jl * nct, uj = j / bd, a = plane_offset(G, ui, uj);
                    Sown[(long)jl * m + i] = a >= 0 ? st_val(Acs, G, Jbase + ui, a + NI, l, j - uj * bd) : 0.0;
                }
                for (int side2 = 0; side2 < 2; ++side2) {
                    const int pl = side2 ? pb : pa, base = side2 ? bb : ba;
                    if (pl < 0) continue;
                    const bool own = keep && !middle;
#pragma unroll
                    for (int a0 = 0; a0 < 9; a0 += 3) {  // three neighbours at a time, in order
                        double cf[9];
#pragma unroll
                        for (int a = 0; a < 3; ++a)
#pragma unroll
                            for (int c = 0; c < 3; ++c)
                                cf[a * 3 + c] = nbr[a0 + a] >= 0 && c < bd
                                                    ? -st_val(Acs, G, Jbase + ui, a0 + a + base, l, c) : 0.0;
#pragma unroll 2
                        for (int jl = 0; jl < ncol; ++jl) {
                            const double *vec = own ? Gown + (long)jl * m : Gm + (long)pl * m * m + rank + jl * nct;
                            const long sd = own ? 1 : m;
                            double v = Sown[(long)jl * m + i];
#pragma unroll
                            for (int a = 0; a < 3; ++a)
#pragma unroll
                                for (int c = 0; c < 3; ++c)
                                    if (nbr[a0 + a] >= 0 && c < bd)
                                        v = fma(cf[a * 3 + c], vec[(nbr[a0 + a] + c) * sd], v);
                            Sown[(long)jl * m + i] = v;
                        }
                    }
                }
                pil[i] = i;
            }
        __syncthreads();
        // ---- Gauss-Jordan with partial pivoting, one pivot per step ----
        if (rank == 0) {
            double v[RPT];
#pragma unroll
            for (int t = 0; t < RPT; ++t) {
                const int i = tid + t * kPlaneThreads;
                v[t] = worker && i < m ? Sown[i] : 0.0;
            }
            publish(0, 0, v);
        }
        cluster_arrive();
        for (int kk = 0; kk < m; ++kk) {
            cluster_wait();  // pivot column kk is in every CTA's buffer
            const int buf = kk % 3, p = s_p[buf];
            const double inv = s_inv[buf];
            const double *f = pcol + buf * m;
            if (s_bad[buf]) {  // uniform over the cluster
                if (rank == 0 && tid == 0) *status = 1 + k * m + kk;
                cluster.sync();  // no CTA leaves while another may still write its shared memory
                return;
            }
            const bool next = kk + 1 < m && rank == (kk + 1) % nct;
            if (next) {  // column kk + 1 first, and its pivot
                const int jl = (kk + 1) / nct;
                const double *cj = Sown + (long)jl * m;
                __syncthreads();  // the column's step kk - 1 is done (by the warp it belongs to)
                const double ck = cj[kk], x = cj[p] * inv;
                double v[RPT];
#pragma unroll
                for (int t = 0; t < RPT; ++t) {
                    const int i = tid + t * kPlaneThreads;
                    v[t] = 0.0;
                    if (worker && i < m) v[t] = i == kk ? x : fma(-f[i], x, i == p ? ck : cj[i]);
                }
                publish(kk + 1, jl, v);
            }
            // releases the owner's stores, and every thread's reads of step kk - 1 before another
            // CTA's store into that buffer two barriers on
            if (kk + 1 < m) cluster_arrive();
            if (!worker) {
                if (lane == 0 && p != kk) {
                    const int t = pil[kk];
                    pil[kk] = pil[p];
                    pil[p] = t;
                }
                continue;
            }
            double fr[RPL];
#pragma unroll
            for (int t = 0; t < RPL; ++t) fr[t] = f[min(lane + 32 * t, m - 1)];
            // two columns of the warp side by side; the pivot column itself is 0 - f / pivot
            for (int jl0 = warp; jl0 < ncol; jl0 += 2 * kWarps) {
                double c[2][RPL], ck[2], x[2];
                double *cj[2];
                bool put[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int jl = jl0 + u * kWarps, j = rank + jl * nct;
                    put[u] = jl < ncol && !(next && j == kk + 1);
                    cj[u] = Sown + (long)(put[u] ? jl : jl0) * m;
                    ck[u] = j == kk ? 0.0 : cj[u][kk];
                    x[u] = cj[u][p];
#pragma unroll
                    for (int t = 0; t < RPL; ++t) c[u][t] = j == kk ? 0.0 : cj[u][min(lane + 32 * t, m - 1)];
                    const double xi = x[u] * inv;
                    x[u] = j == kk ? inv : xi;
                }
                __syncwarp();
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (!put[u]) continue;  // uniform over the warp
#pragma unroll
                    for (int t = 0; t < RPL; ++t) {
                        const int i = lane + 32 * t;
                        const double r = fma(fr[t], -x[u], i == p ? ck[u] : c[u][t]);  // no branch around the FMA
                        c[u][t] = i == kk ? x[u] : r;
                    }
#pragma unroll
                    for (int t = 0; t < RPL; ++t)
                        if (lane + 32 * t < m) cj[u][lane + 32 * t] = c[u][t];
                }
                __syncwarp();
            }
        }
        __syncthreads();
        for (int i = tid; i < m; i += kFactorThreads) pinv[pil[i]] = i;
        // ---- X_k (own columns, row-major in global) and pi_k ----
        double *Xk = X + (long)k * m * m;
        for (int idx = tid; idx < ncol * m; idx += kFactorThreads) {
            const int i = idx / ncol, jl = idx - i * ncol;
            Xk[(long)i * m + rank + jl * nct] = Sown[(long)jl * m + i];
        }
        if (rank == 0)
            for (int i = tid; i < m; i += kFactorThreads) pi[(long)k * m + i] = pil[i];
        cluster.sync();  // every CTA's X_k columns are final
        // ---- G_k = X_k Pi_k C_{k,q}, q the plane after k on this side (k+1 on
        // side 0, k-1 on side 1), own columns j (rows of plane q): a warp per column ----
        if (!middle && worker) {
            double *Gk = Gm + (long)k * m * m;
            const int qb = side == 0 ? 2 * NI : 0;  // stencil entries towards plane q
            for (int jl = warp; jl < ncol; jl += kWarps) {
                const int j = rank + jl * nct, uj = j / bd, mj = j - uj * bd;
                // rows s of plane k with C_{k,q}[s][j] != 0: the in-plane neighbours of uj
                if (lane < NI * bd) {
                    const int a = lane / bd, ls = lane - a * bd, us = plane_nbr(G, uj, a);
                    double u = 0.0;
                    unsigned at = ~0u;
                    if (us >= 0) {
                        const int cc = pinv[us * bd + ls];
                        u = st_val(Acs, G, Jbase + us, plane_offset(G, us, uj) + qb, ls, mj);
                        at = map_rank(Sown + (long)(cc / nct) * m, cc % nct);
                    }
                    s_gval[warp][lane] = u;
                    s_gcol[warp][lane] = at;  // ~0: no such row
                }
                __syncwarp();
                for (int i = lane; i < m; i += 32) {
                    double v = 0.0;
                    for (int e0 = 0; e0 < NI * bd; e0 += 9) {
                        double x[9];
#pragma unroll
                        for (int e = 0; e < 9; ++e) {
                            const unsigned at = e0 + e < NI * bd ? s_gcol[warp][e0 + e] : ~0u;
                            x[e] = at != ~0u ? ld_rank(at + 8u * i) : 0.0;
                        }
#pragma unroll
                        for (int e = 0; e < 9; ++e)
                            if (e0 + e < NI * bd && s_gcol[warp][e0 + e] != ~0u) v = fma(x[e], s_gval[warp][e0 + e], v);
                    }
                    if (keep) Gown[(long)jl * m + i] = v;
                    Gk[(long)i * m + j] = v;
                }
                __syncwarp();
            }
        }
        cluster.sync();  // remote reads of this plane's X columns are done before they are overwritten
    }
}

using PlaneFactorFn = void (*)(PlaneGeom, int, int, int, const double *, double *, double *, int *, int *);
// the instance whose lanes hold a column of m rows
static PlaneFactorFn plane_factor_fn(int m) {
    return m <= 64 ? plane_factor_kernel<2> : m <= 128 ? plane_factor_kernel<4> : m <= 256 ? plane_factor_kernel<8>
           : m <= 384 ? plane_factor_kernel<12> : plane_factor_kernel<24>;
}

// ---- application w = A_c^-1 v --------------------------------------------------------
//
// With H_k = X_k Pi_k C_{k,p} (p the plane before k on its side; the middle plane
// has one towards each side) beside G_k = X_k Pi_k C_{k,q},
//   u_k = X_k Pi_k v_k                              all planes at once,
//   y_k = u_k - H_k y_p                             outwards in, one cluster a side,
//   w_h = u_h - H_h0 y_{h-1} - H_h1 y_{h+1}         the middle plane,
//   w_k = y_k - G_k w_q                             inwards out, one cluster a side.
// The chain's step is then one dense product of a plane. (Applying C to y_p and X_k
// Pi_k to the result at every step put the couplings, formed by every CTA of the
// cluster, and the permutation on the chain: 100 us an application at 128^3, 82 at
// 48^3 elasticity; a solve took 27.3 and 13.0 ms, now 26.0 and 11.2.) What is left
// of a step is bound by the FP64 pipes of the cluster's 16 SMs, m^2 / 16 FMAs each
// at one warp's FMA in 19 cycles, beside the row sums and the cluster barrier. A half-warp takes a row: its 16 lanes sum in four
// steps and store the result into the 16 CTAs, one each.

// pinv[pi_k[i]] = i into shared memory
__device__ __forceinline__ void plane_pinv(const int *__restrict__ pk, int m, int *pinv) {
    for (int i = threadIdx.x; i < m; i += blockDim.x) pinv[pk[i]] = i;
}

constexpr int kPlaneHRows = 16;

// H_k, kPlaneHRows rows a CTA: blockIdx.y = plane, blockIdx.z = 0: the side's H_k
// (the middle plane: towards h - 1), 1: the middle plane towards h + 1 (plane np of H).
// A thread's column lists its at most 9 bd entries of C once for all the rows.
__global__ void __launch_bounds__(256) plane_h_kernel(PlaneGeom G, int h, const double *__restrict__ Acs,
                                                      const double *__restrict__ X, const int *__restrict__ pi,
                                                      double *__restrict__ H) {
    const int m = G.m, bd = G.bd, NI = G.NI, np = G.np, k = blockIdx.y;
    const int to_prev = blockIdx.z ? 0 : (k <= h);  // couplings towards plane k - 1, else k + 1
    if (blockIdx.z && k != h) return;
    const int p = to_prev ? k - 1 : k + 1;
    if (p < 0 || p >= np) return;
    const int r0 = blockIdx.x * kPlaneHRows, nr = min(kPlaneHRows, m - r0);
    extern __shared__ double sm[];
    double *xs = sm;                                // the CTA's rows of X_k
    int *pinv = (int *)(xs + (long)kPlaneHRows * m);
    const double *Xk = X + (long)k * m * m + (long)r0 * m;
    for (int t = threadIdx.x; t < nr * m; t += blockDim.x) xs[t] = Xk[t];
    plane_pinv(pi + (long)k * m, m, pinv);
    __syncthreads();
    double *Hk = H + (long)(blockIdx.z ? np : k) * m * m + (long)r0 * m;
    const int qb = to_prev ? 0 : 2 * NI, Jbase = k * G.PN;
    for (int j = threadIdx.x; j < m; j += blockDim.x) {
        const int uj = j / bd, mj = j - uj * bd;
        double acc[kPlaneHRows];
#pragma unroll
        for (int r = 0; r < kPlaneHRows; ++r) acc[r] = 0.0;
        for (int a = 0; a < NI; ++a) {  // rows s of plane k that couple with column j: the neighbours of uj
            const int us = plane_nbr(G, uj, a);
            if (us < 0) continue;
            const int qq = plane_offset(G, us, uj) + qb;
            for (int ls = 0; ls < bd; ++ls) {
                const double c = st_val(Acs, G, Jbase + us, qq, ls, mj);
                const double *x = xs + pinv[us * bd + ls];
#pragma unroll
                for (int r = 0; r < kPlaneHRows; ++r)
                    if (r < nr) acc[r] = fma(x[(long)r * m], c, acc[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < kPlaneHRows; ++r)
            if (r < nr) Hk[(long)r * m + j] = acc[r];
    }
}

// sum over a half-warp (16 lanes a row), in every lane
__device__ __forceinline__ double half_sum(double a) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}

constexpr int kPlaneURows = kPlaneThreads / 16;  // rows a CTA of the launches without a chain
constexpr int kPlaneUPre = 16;   // entries of a row per lane read ahead

// wc_k = u_k = X_k Pi_k v_k; the head of X's rows and pi are loaded before the wait
__global__ void __launch_bounds__(kPlaneThreads) plane_u_kernel(int m, const double *__restrict__ X,
                                                                const int *__restrict__ pi,
                                                                const double *__restrict__ vc,
                                                                double *__restrict__ wc) {
    extern __shared__ double sm[];  // Pi_k v_k
    const int k = blockIdx.y, hl = threadIdx.x & 15, i = blockIdx.x * kPlaneURows + (threadIdx.x >> 4);
    const double *x = X + (long)k * m * m + (long)min(i, m - 1) * m;
    double a[kPlaneUPre];
#pragma unroll
    for (int t = 0; t < kPlaneUPre; ++t) a[t] = __ldg(x + min(hl + 16 * t, m - 1));
    const int j0 = threadIdx.x, p0 = j0 < m ? __ldg(pi + (long)k * m + j0) : 0;
    pdl_prologue();
    if (j0 < m) sm[j0] = vc[(long)k * m + p0];
    for (int j = j0 + kPlaneThreads; j < m; j += kPlaneThreads) sm[j] = vc[(long)k * m + pi[(long)k * m + j]];
    __syncthreads();
    double s = 0.0;
#pragma unroll
    for (int t = 0; t < kPlaneUPre; ++t)
        if (hl + 16 * t < m) s = fma(a[t], sm[hl + 16 * t], s);
    for (int j = hl + 16 * kPlaneUPre; j < m; j += 16) s = fma(x[j], sm[j], s);
    s = half_sum(s);
    if (hl == 0 && i < m) wc[(long)k * m + i] = s;
}

// w_h = u_h - H_h0 y_{h-1} - H_h1 y_{h+1}
__global__ void __launch_bounds__(kPlaneThreads) plane_middle_kernel(int m, int np, int h,
                                                                     const double *__restrict__ H, double *wc,
                                                                     float *__restrict__ wc32) {
    const int hl = threadIdx.x & 15, i = blockIdx.x * kPlaneURows + (threadIdx.x >> 4);
    const long row = (long)min(i, m - 1) * m;
    const double *m0 = H + (long)h * m * m + row, *m1 = H + (long)np * m * m + row;
    double a[kPlaneUPre], b[kPlaneUPre];
#pragma unroll
    for (int t = 0; t < kPlaneUPre; ++t) {
        a[t] = h > 0 ? __ldg(m0 + min(hl + 16 * t, m - 1)) : 0.0;
        b[t] = h + 1 < np ? __ldg(m1 + min(hl + 16 * t, m - 1)) : 0.0;
    }
    pdl_prologue();
    double s = 0.0;
    const double *y0 = wc + (long)max(h - 1, 0) * m, *y1 = wc + (long)min(h + 1, np - 1) * m;
#pragma unroll
    for (int t = 0; t < kPlaneUPre; ++t) {
        const int j = hl + 16 * t;
        if (j < m && h > 0) s = fma(a[t], y0[j], s);
        if (j < m && h + 1 < np) s = fma(b[t], y1[j], s);
    }
#pragma unroll 4
    for (int j = hl + 16 * kPlaneUPre; j < m; j += 16) {
        if (h > 0) s = fma(m0[j], y0[j], s);
        if (h + 1 < np) s = fma(m1[j], y1[j], s);
    }
    s = half_sum(s);
    if (hl == 0 && i < m) {
        const double w = wc[(long)h * m + i] - s;
        wc[(long)h * m + i] = w;
        if (wc32) wc32[(long)h * m + i] = (float)w;
    }
}

// One cluster a side. forward: y_k = u_k - H_k y_p over the side's planes after its
// first (whose y is u); backward: w_k = y_k - G_k w_q from the middle outwards. u, y
// and w share wc; wc32 (nullable) gets an FP32 copy of w. A CTA owns rw rows of every
// plane; with `stage` its rows of a step's matrix are copied to shared memory two
// steps ahead (they do not depend on the chain), so that a step waits only for the
// cluster barrier and its own products.
__global__ void __launch_bounds__(kPlaneThreads, 1) plane_chain_kernel(int m, int np, int h, int forward, int stage,
                                                                     const double *__restrict__ M, double *wc,
                                                                     float *__restrict__ wc32) {
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), nct = (int)cluster.num_blocks();
    const int rw = (m + nct - 1) / nct, r0 = rank * rw, nr = max(0, min(m, r0 + rw) - r0);
    const int tid = threadIdx.x, hl = tid & 15, warp = tid >> 5, sub = (tid >> 4) & 1;
    const int side = (int)(blockIdx.x / nct);
    // planes k0, k0 + dk, ... (nsteps of them), after plane k0 - dk
    const int dk = (side == 0) == (forward != 0) ? 1 : -1;
    const int k0 = forward ? (side == 0 ? 1 : np - 2) : (side == 0 ? h - 1 : h + 1);
    const int nsteps = forward ? (side == 0 ? h - 1 : np - 2 - h) : (side == 0 ? h : np - 1 - h);
    extern __shared__ __align__(16) double sm[];
    const int ms = (m + 1) & ~1;
    double *prev = sm;               // the plane before, double buffered [2][ms] (written by every CTA)
    double *mat = prev + 2 * ms;     // staged rows [2][rw * m], on a 16-byte boundary
    const bool wide = (m & 1) == 0;  // rows of whole 16-byte vectors
    auto issue = [&](int st) {
        if (stage && st < nsteps) {
            const double *src = M + (long)(k0 + st * dk) * m * m + (long)r0 * m;
            double *dst = mat + (long)(st & 1) * rw * m;
            if (wide)
                for (int q = tid; q < nr * m / 2; q += kPlaneThreads) cp_async16(dst + 2 * q, src + 2 * q);
            else
                for (int q = tid; q < nr * m; q += kPlaneThreads) cp_async8(dst + q, src + q);
        }
        cp_async_commit();  // one group per step, empty or not
    };
    issue(0);
    issue(1);
    pdl_prologue();
    if (nsteps > 0)
        for (int j = tid; j < m; j += kPlaneThreads) prev[j] = wc[(long)(k0 - dk) * m + j];
    cluster.sync();  // every CTA runs before another stores into its shared memory
    const int i0 = 2 * warp + sub;  // this half-warp's first row of the CTA's
    double head = nsteps > 0 && i0 < nr ? wc[(long)k0 * m + r0 + i0] : 0.0;  // its u or y, one step ahead
    for (int st = 0; st < nsteps; ++st) {
        const int buf = st & 1, k = k0 + st * dk;
        const double *y = prev + buf * ms, *rows = stage ? mat + (long)buf * rw * m : M + (long)k * m * m + (long)r0 * m;
        const double next = st + 1 < nsteps && i0 < nr ? wc[(long)(k + dk) * m + r0 + i0] : 0.0;
        cp_async_wait<1>();
        __syncthreads();
        for (int q = i0; q - sub < nr; q += 2 * (kPlaneThreads / 32)) {
            const bool has = q < nr;
            const double base = q == i0 ? head : has ? wc[(long)k * m + r0 + q] : 0.0;
            const double *row = rows + (long)min(q, nr - 1) * m;
            double s = 0.0;
#pragma unroll 4
            for (int j = hl; j < m; j += 16) s = fma(row[j], y[j], s);
            const double w = base - half_sum(s);
            if (has) {  // 16 lanes a row, a destination each
                if (hl < nct) st_rank(map_rank(prev + (buf ^ 1) * ms + r0 + q, hl), w);
                if (hl == 0) {
                    wc[(long)k * m + r0 + q] = w;
                    if (wc32 && !forward) wc32[(long)k * m + r0 + q] = (float)w;
                }
            }
        }
        head = next;
        __syncthreads();  // this step's staged rows are no longer read
        issue(st + 2);
        cluster.sync();
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// The explicit inverse A_c^-1 (row-major n_C x n_C) from the plane factors,
// for coarse systems small enough that one dense product per application
// beats the dependent plane steps: CTA b builds the columns
// kInvCols*b .. kInvCols*b + kInvCols-1, the same recurrences as
// the factored application on identity columns, independent across CTAs.
constexpr int kInvCols = 4;

// W_k = X_k Pi_k (e_k - C_{k,pa} W_pa - C_{k,pb} W_pb) for the CTA's columns
// (planes pa / pb with stencil bases ba / bb; -1: none)
__device__ __forceinline__ void inv_fwd_plane(const PlaneGeom &G, const double *__restrict__ Acs,
                                              const double *__restrict__ X, const int *__restrict__ pi, double *Wc,
                                              double *t, double *tp, int c0, int k, int pa, int ba, int pb, int bb) {
    const int m = G.m, bd = G.bd, tid = threadIdx.x, Jbase = k * G.PN;
    for (int idx = tid; idx < m * kInvCols; idx += kPlaneThreads) {
        const int j = idx / kInvCols, q = idx - j * kInvCols;
        const int uj = j / bd, l = j - uj * bd;
        double v = (c0 + q == k * m + j) ? 1.0 : 0.0;
        if (pa >= 0) v = sub_coupling(v, G, Acs, Jbase + uj, uj, l, ba, Wc + (long)pa * m * kInvCols + q, kInvCols);
        if (pb >= 0) v = sub_coupling(v, G, Acs, Jbase + uj, uj, l, bb, Wc + (long)pb * m * kInvCols + q, kInvCols);
        t[idx] = v;
    }
    __syncthreads();
    const int *pk = pi + (long)k * m;
    for (int idx = tid; idx < m * kInvCols; idx += kPlaneThreads) {
        const int j = idx / kInvCols, q = idx - j * kInvCols;
        tp[idx] = t[pk[j] * kInvCols + q];
    }
    __syncthreads();
    const double *Xk = X + (long)k * m * m;
    for (int idx = tid; idx < m * kInvCols; idx += kPlaneThreads) {
        const int i = idx / kInvCols, q = idx - i * kInvCols;
        const double *xr = Xk + (long)i * m;
        double s = 0.0;
        for (int j = 0; j < m; ++j) s = fma(__ldg(xr + j), tp[j * kInvCols + q], s);
        Wc[((long)k * m + i) * kInvCols + q] = s;
    }
    __syncthreads();
}

// W_k -= G_k W_kq for the CTA's columns
__device__ __forceinline__ void inv_back_plane(const PlaneGeom &G, const double *__restrict__ Gm, double *Wc, int k,
                                               int kq) {
    const int m = G.m, tid = threadIdx.x;
    const double *Gk = Gm + (long)k * m * m;
    for (int idx = tid; idx < m * kInvCols; idx += kPlaneThreads) {
        const int i = idx / kInvCols, q = idx - i * kInvCols;
        const double *gr = Gk + (long)i * m;
        double s = 0.0;
        for (int j = 0; j < m; ++j) s = fma(__ldg(gr + j), Wc[((long)kq * m + j) * kInvCols + q], s);
        Wc[((long)k * m + i) * kInvCols + q] -= s;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kPlaneThreads) plane_inverse_kernel(PlaneGeom G, int h,
                                                                      const double *__restrict__ Acs,
                                                                      const double *__restrict__ X,
                                                                      const double *__restrict__ Gm,
                                                                      const int *__restrict__ pi,
                                                                      double *__restrict__ Ainv) {
    const int m = G.m, NI = G.NI, np = G.np, nC = np * m;
    const int c0 = blockIdx.x * kInvCols, ncols = min(kInvCols, nC - c0);
    const int tid = threadIdx.x;
    extern __shared__ double sm[];
    double *Wc = sm;                           // the columns being built, [nC][kInvCols]
    double *t = Wc + (long)nC * kInvCols;      // [m][kInvCols]
    double *tp = t + (long)m * kInvCols;       // [m][kInvCols]
    for (int k = 0; k < h; ++k) inv_fwd_plane(G, Acs, X, pi, Wc, t, tp, c0, k, k - 1, 0, -1, 0);
    for (int k = np - 1; k > h; --k) inv_fwd_plane(G, Acs, X, pi, Wc, t, tp, c0, k, k + 1 < np ? k + 1 : -1, 2 * NI, -1, 0);
    inv_fwd_plane(G, Acs, X, pi, Wc, t, tp, c0, h, h - 1, 0, h + 1 < np ? h + 1 : -1, 2 * NI);
    for (int k = h - 1; k >= 0; --k) inv_back_plane(G, Gm, Wc, k, k + 1);
    for (int k = h + 1; k < np; ++k) inv_back_plane(G, Gm, Wc, k, k - 1);
    for (int idx = tid; idx < nC * ncols; idx += kPlaneThreads) {
        const int row = idx / ncols, q = idx - row * ncols;
        Ainv[(long)row * nC + c0 + q] = Wc[(long)row * kInvCols + q];
    }
}

// ---- host side ----------------------------------------------------------------------

static size_t factor_smem(int m, int nct, bool keep) {
    const size_t cols = (size_t)((m + nct - 1) / nct) * m * sizeof(double);
    return (keep ? 2 : 1) * cols + 3 * (size_t)m * sizeof(double) + 3 * (size_t)m * sizeof(int);
}
static size_t solve_smem(int m) { return 2 * (size_t)(m + 1) * sizeof(double); }
// with the staged rows (see plane_chain_kernel)
static size_t solve_smem_staged(int m, int nct) {
    const int rw = (m + nct - 1) / nct;
    return solve_smem(m) + 2 * (size_t)rw * m * sizeof(double);
}

constexpr size_t kPlaneSmemMax = 220 * 1024;

static cudaLaunchConfig_t cluster_cfg(cudaLaunchAttribute *attr, int nct, size_t smem, cudaStream_t s, bool pdl,
                                      int threads = kPlaneThreads) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = nct;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nct);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 2 : 1;
    return cfg;
}

// Cluster size for planes of m rows: the largest of 16 (where the device
// allows non-portable clusters), 8, 4, 2, 1, not above m, whose shared memory
// fits and which the device can schedule; 0 if none.
static int plane_cluster(int m) {
    static int cap = 0;  // set once per process; the attributes are per function
    static std::once_flag once;
    std::call_once(once, [] {
        bool wide = true;  // non-portable cluster sizes
        for (int rows : {64, 128, 256, 384, kPlaneMaxRows}) {
            wide = cudaFuncSetAttribute(plane_factor_fn(rows), cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
                       cudaSuccess && wide;
            cudaFuncSetAttribute(plane_factor_fn(rows), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kPlaneSmemMax);
        }
        wide = cudaFuncSetAttribute(plane_chain_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
                   cudaSuccess && wide;
        cap = wide ? kPlaneMaxCluster : 8;
        cudaFuncSetAttribute(plane_chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPlaneSmemMax);
        cudaFuncSetAttribute(plane_h_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPlaneSmemMax);
        cudaGetLastError();
    });
    if (m < 1 || solve_smem(m) > kPlaneSmemMax) return 0;
    for (int nct = cap; nct >= 1; nct >>= 1) {
        if (nct > m) continue;
        const int cw = (m + nct - 1) / nct;
        const size_t sf = factor_smem(m, nct, false);
        if (cw > kPlaneMaxCols || m > kPlaneMaxRows || sf > kPlaneSmemMax) return 0;  // smaller clusters need more per CTA
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cf = cluster_cfg(attr, nct, sf, nullptr, false, kFactorThreads);
        cudaLaunchConfig_t cs = cluster_cfg(attr, nct, solve_smem(m), nullptr, false);
        int nf = 0, ns = 0;
        if (cudaOccupancyMaxActiveClusters(&nf, plane_factor_fn(m), &cf) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&ns, plane_chain_kernel, &cs) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        if (nf > 0 && ns > 0) return nct;
    }
    return 0;
}

static void plane_geom(int dim, const int nb[3], int bd, PlaneGeom *G) {
    G->dim = dim;
    G->nb0 = nb[0];
    G->nb1 = dim == 3 ? nb[1] : 1;
    G->bd = bd;
    G->np = dim == 3 ? nb[2] : nb[1];
    G->PN = dim == 3 ? nb[0] * nb[1] : nb[0];
    G->m = G->PN * bd;
    G->NI = dim == 3 ? 9 : 3;
    G->nq = dim == 3 ? 27 : 9;
}

// Whether the plane factorisation serves this coarse grid (one cluster holds
// a plane); otherwise the caller uses the dense inverse.
bool planes_fit(int dim, const int nb[3], int bd) {
    PlaneGeom G;
    plane_geom(dim, nb, bd, &G);
    return plane_cluster(G.m) > 0;
}

msrsb_status plane_factor(int dim, const int nb[3], int bd, const double *Acs, CoarsePlanes *cp, cudaStream_t s) {
    PlaneGeom G;
    plane_geom(dim, nb, bd, &G);
    const int nct = plane_cluster(G.m);
    if (!nct) return fail(MSRSB_ESHAPE, "coarse planes of %d unknowns do not fit one thread-block cluster", G.m);
    cp->m = G.m;
    cp->np = G.np;
    cp->nct = nct;
    cp->stage = 0;
    {  // staged application where its shared memory fits and the cluster can be scheduled with it
        const size_t ss = solve_smem_staged(G.m, nct);
        if (ss <= kPlaneSmemMax) {
            cudaLaunchAttribute a2[2];
            cudaLaunchConfig_t cs = cluster_cfg(a2, nct, ss, nullptr, false);
            int ns = 0;
            if (cudaOccupancyMaxActiveClusters(&ns, plane_chain_kernel, &cs) == cudaSuccess && ns > 0) cp->stage = 1;
            cudaGetLastError();
        }
    }
    const long mm = (long)G.m * G.m;
    const int h = G.np / 2;  // side 0: planes 0 .. h-1, side 1: np-1 .. h+1 (never longer than side 0)
    cp->h = h;
    MSRSB_TRY(dalloc(&cp->X, (size_t)G.np * mm, s));
    MSRSB_TRY(dalloc(&cp->G, (size_t)G.np * mm, s));
    MSRSB_TRY(dalloc(&cp->pi, (size_t)G.np * G.m, s));
    int *status = nullptr;
    MSRSB_TRY(dalloc(&status, 1, s));
    MSRSB_CUDA(cudaMemsetAsync(status, 0, sizeof(int), s));
    int keep = 0;  // the sides keep their last G_k's columns where shared memory allows it
    {
        cudaLaunchAttribute a2[2];
        const size_t sk = factor_smem(G.m, nct, true);
        cudaLaunchConfig_t ck = cluster_cfg(a2, nct, sk, nullptr, false, kFactorThreads);
        int nk = 0;
        if (sk <= kPlaneSmemMax && cudaOccupancyMaxActiveClusters(&nk, plane_factor_fn(G.m), &ck) == cudaSuccess && nk > 0)
            keep = 1;
        cudaGetLastError();
    }
    const size_t sf = factor_smem(G.m, nct, keep), sfm = factor_smem(G.m, nct, false);
    if (h > 0) {  // the two sides, one cluster each, concurrently
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = cluster_cfg(attr, nct, sf, s, false, kFactorThreads);
        cfg.gridDim = dim3((G.np - 1 - h > 0 ? 2 : 1) * nct);
        count_launch();
        MSRSB_CUDA(cudaLaunchKernelEx(&cfg, plane_factor_fn(G.m), G, h, 0, keep, Acs, cp->X, cp->G, cp->pi, status));
    }
    {  // the middle plane
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = cluster_cfg(attr, nct, sfm, s, false, kFactorThreads);
        count_launch();
        MSRSB_CUDA(cudaLaunchKernelEx(&cfg, plane_factor_fn(G.m), G, h, 1, 0, Acs, cp->X, cp->G, cp->pi, status));
    }
    int bad = 0;
    MSRSB_TRY(read_back(&bad, status, sizeof(int), s));
    dfree(status, s);
    if (bad) return fail(MSRSB_EBREAKDOWN, "coarse operator is singular (zero pivot at coarse row %d)", bad - 1);
    return MSRSB_OK;
}

// The couplings H_k that the application needs (not the explicit inverse).
msrsb_status plane_couplings(int dim, const int nb[3], int bd, const double *Acs, CoarsePlanes *cp, cudaStream_t s) {
    PlaneGeom G;
    plane_geom(dim, nb, bd, &G);
    MSRSB_TRY(dalloc(&cp->H, (size_t)(G.np + 1) * G.m * G.m, s));
    if (G.np == 1) return MSRSB_OK;
    const size_t smem = (size_t)kPlaneHRows * G.m * sizeof(double) + (size_t)G.m * sizeof(int);
    plane_h_kernel<<<dim3(ceil_div(G.m, kPlaneHRows), G.np, 2), 256, smem, s>>>(G, cp->h, Acs, cp->X, cp->pi, cp->H);
    MSRSB_LAUNCHED("plane_h_kernel");
    return MSRSB_OK;
}

msrsb_status plane_solve(const CoarsePlanes *cp, const double *vc, double *wc, float *wc32, cudaStream_t s) {
    const int m = cp->m, np = cp->np, h = cp->h;
    auto chain = [&](int forward) -> msrsb_status {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = cluster_cfg(attr, cp->nct, cp->stage ? solve_smem_staged(m, cp->nct) : solve_smem(m), s,
                                             true);
        const int other = forward ? np - 2 - h : np - 1 - h;  // steps of side 1
        cfg.gridDim = dim3((other > 0 ? 2 : 1) * cp->nct);
        const double *M = forward ? cp->H : cp->G;
        count_launch();
        cudaError_t e = cudaLaunchKernelEx(&cfg, plane_chain_kernel, m, np, h, forward, cp->stage, M, wc, wc32);
        if (e == cudaErrorNotSupported || e == cudaErrorInvalidValue) {  // programmatic serialisation refused
            cudaGetLastError();
            cfg.numAttrs = 1;
            e = cudaLaunchKernelEx(&cfg, plane_chain_kernel, m, np, h, forward, cp->stage, M, wc, wc32);
        }
        MSRSB_CUDA(e);
        return MSRSB_OK;
    };
    const int tiles = ceil_div(m, kPlaneURows);
    MSRSB_PDL((plane_u_kernel), dim3(tiles, np), kPlaneThreads, (size_t)m * sizeof(double), s, m, (const double *)cp->X,
              (const int *)cp->pi, vc, wc);
    if (h > 1) MSRSB_TRY(chain(1));  // side 0 is never the shorter one
    MSRSB_PDL((plane_middle_kernel), tiles, kPlaneThreads, 0, s, m, np, h, (const double *)cp->H, wc, wc32);
    if (h > 0) MSRSB_TRY(chain(0));
    return MSRSB_OK;
}

// Ainv (n_C x n_C row-major) = A_c^-1 from the plane factors.
msrsb_status plane_inverse(int dim, const int nb[3], int bd, const double *Acs, const CoarsePlanes *cp, double *Ainv,
                           cudaStream_t s) {
    PlaneGeom G;
    plane_geom(dim, nb, bd, &G);
    const long nC = (long)G.np * G.m;
    const size_t smem = ((size_t)nC + 2 * G.m) * kInvCols * sizeof(double);
    if (smem > kPlaneSmemMax) return fail(MSRSB_ESHAPE, "explicit coarse inverse too large (n_C = %ld)", nC);
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(plane_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPlaneSmemMax);
        cudaGetLastError();
    });
    plane_inverse_kernel<<<ceil_div(nC, kInvCols), kPlaneThreads, smem, s>>>(G, cp->h, Acs, cp->X, cp->G, cp->pi,
                                                                             Ainv);
    MSRSB_LAUNCHED("plane_inverse_kernel");
    return MSRSB_OK;
}

void plane_free(CoarsePlanes *cp, cudaStream_t s) {
    dfree(cp->X, s);
    dfree(cp->G, s);
    dfree(cp->H, s);
    dfree(cp->pi, s);
}

}  // namespace msrsb
