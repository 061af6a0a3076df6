// Block (3x3) Gauss-Seidel, the pre- and post-smoother of the mechanics
// configuration (Sec. 4.2-4.3, Alg. 4 of arXiv 1912.06934), in the node colour
// order (colours of coordinate parity; nodes of one colour never share a 3^dim
// stencil): one launch per colour and direction.
//
// A sweep's work is reading A's blocks once; with one thread per node on the
// caller's block rows (36-byte records, an index and a colour looked up per
// block, half of the blocks skipped) a colour's launch took 21 us at 48^3, of
// which the blocks' bytes account for 1 to 2.5. Here every colour's rows keep
// their blocks in the order the sweeps use them: those towards earlier colours,
// then those towards later ones, then the diagonal, in groups of kGsBlocks
// blocks (9 vectors of 16 bytes), zero where the pattern has none. Up to eight
// lanes share a row, a group each (a colour of 48^3 has 14,700 rows, 0.8 warps a
// scheduler with one thread a row), vector t of all of a row's groups side by
// side so that its lanes read whole lines. The blocks and columns do not depend
// on the previous kernel and are loaded before griddepcontrol.wait; one round
// of gathers follows it, of 16-byte records (the vectors the sweeps read are
// kept padded to four components a node).
//
// Three uses of the same storage:
//  forward from zero: e_i = D_i^-1 (v_i - sum_{earlier} A_ik e_k);
//  the residual after it: v - A e = -U e, since (D + L) e = v: the blocks towards
//    later colours alone;
//  backward on z: with r = v - A z, e_i = D_i^-1 (r_i - sum_{later} A_ik e_k) and
//    z_i += e_i is, colour by colour, z_i += D_i^-1 (v_i - sum_k A_ik z_k) with
//    the z of the moment: the residual needs no pass of its own.
// Measured inside a 48^3 mixed PCG solve (352,947 unknowns): 16 sweep launches and
// two residuals of an iteration 398 -> 147 us, a colour's launch 21 -> 7.5 us (16.5
// MB of blocks backward, 2.5 us at the copy rate), the solve 25.2 -> 14.4 ms.
#include "common.cuh"
#include <cstring>
#include <type_traits>

namespace msrsb {

template <typename T>
using GsVec = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
template <typename T>
constexpr int kGsBlocks = 16 / (int)sizeof(T);  // blocks a group; 9 vectors hold them
constexpr int kGsThreads = 128;  // a sweep's CTA; 7 of them fit an SM (FP32), so that 48^3's 920 are resident at once

// blocks towards earlier (dir 0) or later (1) colours of a row of colour c: a
// neighbour at offset o has colour c xor f, f the odd axes of o, 2^popc(f) offsets each
static int gs_count(int dim, int c, int dir) {
    int n = 0;
    for (int f = 1; f < 1 << dim; ++f)
        if (((c ^ f) > c) == (dir == 1)) n += 1 << __builtin_popcount(f);
    return n;
}

// one thread per (row of the colour, group)
template <typename T>
__global__ void __launch_bounds__(256) gs_fill_kernel(int cnt, int c, int ge, int ng,
                                                      const int32_t *__restrict__ rows,
                                                      const int32_t *__restrict__ rowptr,
                                                      const int32_t *__restrict__ colidx,
                                                      const uint8_t *__restrict__ colour,
                                                      const double *__restrict__ val, T *__restrict__ out,
                                                      int32_t *__restrict__ col) {
    constexpr int GB = kGsBlocks<T>;
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= (long)cnt * ng) return;
    const int r = (int)(t / ng), g = (int)(t - (long)r * ng);
    const int i = rows[r];
    int k[GB], ent[GB];  // the group's columns, and their entries of A (-1: none)
#pragma unroll
    for (int u = 0; u < GB; ++u) {
        k[u] = i;  // no block: zero times the row's own value
        ent[u] = -1;
    }
    int n[2] = {0, 0};
    for (int e = rowptr[i]; e < rowptr[i + 1]; ++e) {
        const int j = colidx[e], cj = colour[j];
        const int at = j == i ? ng * GB - 1 : (cj < c ? n[0]++ : ge * GB + n[1]++);
#pragma unroll
        for (int u = 0; u < GB; ++u)
            if (at == g * GB + u) {
                k[u] = j;
                ent[u] = e;
            }
    }
    T b[9 * GB];
#pragma unroll
    for (int u = 0; u < GB; ++u)
#pragma unroll
        for (int q = 0; q < 9; ++q) b[9 * u + q] = ent[u] >= 0 ? T(val[(long)ent[u] * 9 + q]) : T(0);
    GsVec<T> *o = reinterpret_cast<GsVec<T> *>(out);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        GsVec<T> v;
        memcpy(&v, b + q * GB, 16);
        o[((long)r * 9 + q) * ng + g] = v;
    }
#pragma unroll
    for (int u = 0; u < GB; ++u) col[((long)r * ng + g) * GB + u] = k[u];
}

template <typename T>
msrsb_status gs_setup(msrsb_handle *h, cudaStream_t s) {
    const msrsb_mat &A = h->A;
    GsEll &E = h->gs;
    constexpr int GB = kGsBlocks<T>;
    E.ncol = h->ncolours;
    long tot = 0;
    for (int c = 0; c < E.ncol; ++c) {
        E.ge[c] = ceil_div(gs_count(h->grid.dim, c, 0), GB);
        E.ng[c] = E.ge[c] + ceil_div(gs_count(h->grid.dim, c, 1) + 1, GB);
        E.base[c] = tot;
        tot += (long)(h->colour_ptr_h[c + 1] - h->colour_ptr_h[c]) * E.ng[c];
    }
    T *v = nullptr;
    MSRSB_TRY(dalloc(&v, (size_t)tot * 9 * GB, s));
    E.val = v;
    MSRSB_TRY(dalloc(&E.col, (size_t)tot * GB, s));
    for (int c = 0; c < E.ncol; ++c) {
        const int cnt = h->colour_ptr_h[c + 1] - h->colour_ptr_h[c];
        if (!cnt) continue;
        gs_fill_kernel<T><<<ceil_div((long)cnt * E.ng[c], 256), 256, 0, s>>>(
            cnt, c, E.ge[c], E.ng[c], h->colour_rows + h->colour_ptr_h[c], A.rowptr, A.colidx, h->colour, A.val,
            v + E.base[c] * 9 * GB, E.col + E.base[c] * GB);
        MSRSB_LAUNCHED("gs_fill_kernel");
    }
    return MSRSB_OK;
}
template msrsb_status gs_setup<float>(msrsb_handle *, cudaStream_t);
template msrsb_status gs_setup<double>(msrsb_handle *, cudaStream_t);

// one group's blocks and columns
template <typename T>
struct GsGroup {
    T b[9 * kGsBlocks<T>];
    int k[kGsBlocks<T>];
};
template <typename T>
__device__ __forceinline__ void gs_load(GsGroup<T> &G, const T *__restrict__ val, const int32_t *__restrict__ col,
                                        int r, int ng, int g) {
    constexpr int GB = kGsBlocks<T>;
    const GsVec<T> *p = reinterpret_cast<const GsVec<T> *>(val) + (long)r * 9 * ng + g;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const GsVec<T> v = __ldg(p + q * ng);
        memcpy(G.b + q * GB, &v, 16);
    }
    if constexpr (GB == 4) {
        const int4 k = __ldg(reinterpret_cast<const int4 *>(col) + (long)r * ng + g);
        G.k[0] = k.x, G.k[1] = k.y, G.k[2] = k.z, G.k[3] = k.w;
    } else {
        const int2 k = __ldg(reinterpret_cast<const int2 *>(col) + (long)r * ng + g);
        G.k[0] = k.x, G.k[1] = k.y;
    }
}
// the padded vector's record of node k
template <typename T>
__device__ __forceinline__ void gs_node(const T *x4, int k, T (&x)[4]) {
    const GsVec<T> *p = reinterpret_cast<const GsVec<T> *>(x4 + 4 * (long)k);
#pragma unroll
    for (int q = 0; q < (int)sizeof(T) / 4; ++q) {
        const GsVec<T> v = p[q];
        memcpy(reinterpret_cast<char *>(x) + 16 * q, &v, 16);
    }
}
// s += the group's blocks times x4 (skip: except the block of column `skip`)
template <typename T>
__device__ __forceinline__ void gs_accumulate(const GsGroup<T> &G, const T *x4, int skip, T (&s)[3]) {
    constexpr int GB = kGsBlocks<T>;
    T x[GB][4];
#pragma unroll
    for (int u = 0; u < GB; ++u) gs_node<T>(x4, G.k[u], x[u]);
#pragma unroll
    for (int u = 0; u < GB; ++u)
        if (G.k[u] != skip) {
#pragma unroll
            for (int l = 0; l < 3; ++l)
#pragma unroll
                for (int m = 0; m < 3; ++m) s[l] = fma(G.b[9 * u + 3 * l + m], x[u][m], s[l]);
        }
}
template <typename T, int L>
__device__ __forceinline__ void gs_row_sum(T (&s)[3]) {  // over a row's L lanes, to all of them
    const unsigned mask = L == 32 ? 0xffffffffu : ((1u << L) - 1u) << (threadIdx.x & 31 & ~(L - 1));
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1)
#pragma unroll
        for (int l = 0; l < 3; ++l) s[l] += __shfl_xor_sync(mask, s[l], o, L);
}

// One colour of a sweep, L lanes a row over the groups 0 .. ng1 - 1 of each row:
// e_i = D_i^-1 (v_i - sum A_ik x_k), x the padded vector; then x_i = e_i
// (forward: from zero) and z_i = e_i where z is given, or z_i += e_i and x_i = z_i
// (backward).
template <typename T, typename TV, typename TZ, int L>
__global__ void __launch_bounds__(kGsThreads, sizeof(T) == 4 ? 7 : 4) gs_sweep_kernel(int cnt, int forward, const int32_t *__restrict__ rows, int ng,
                                                       int ng1, const T *__restrict__ val,
                                                       const int32_t *__restrict__ col, const T *__restrict__ dinv,
                                                       const TV *__restrict__ v, T *x4, TZ *z) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x, r = t / L, g = t & (L - 1);
    const bool on = r < cnt;
    GsGroup<T> G;
    // rows of four lanes and more: lane l finishes component l; else lane 0 does all
    constexpr int NC = L >= 4 ? 1 : 3;
    const int l0 = NC == 1 ? g : 0;
    const bool fin = NC == 1 ? g < 3 : g == 0;
    T d[3 * NC];
    int i = 0;
    if (on) {
        if (g < ng1) gs_load<T>(G, val, col, r, ng, g);
        i = __ldg(rows + r);
        if (fin)
#pragma unroll
            for (int q = 0; q < 3 * NC; ++q) d[q] = __ldg(dinv + (long)i * 9 + 3 * l0 + q);
    }
    pdl_prologue();
    if (!on) return;  // whole rows leave together
    T a[NC];
    TZ zo[NC];
#pragma unroll
    for (int l = 0; l < NC; ++l) {
        a[l] = fin ? T(v[3 * (long)i + l0 + l]) : T(0);
        zo[l] = fin && !forward ? z[3 * (long)i + l0 + l] : TZ(0);
    }
    T s[3] = {T(0), T(0), T(0)};
    // forward, the row's own record (where padding points) holds an older vector
    const int skip = forward ? i : -1;
    if (g < ng1) gs_accumulate<T>(G, x4, skip, s);
    for (int q = g + L; q < ng1; q += L) {
        gs_load<T>(G, val, col, r, ng, q);
        gs_accumulate<T>(G, x4, skip, s);
    }
    gs_row_sum<T, L>(s);
    T b[3];  // v - sum, all components
    if constexpr (NC == 1) {
        const unsigned mask = ((1u << L) - 1u) << (threadIdx.x & 31 & ~(L - 1));
#pragma unroll
        for (int l = 0; l < 3; ++l) b[l] = __shfl_sync(mask, a[0], l, L) - s[l];
    } else {
#pragma unroll
        for (int l = 0; l < 3; ++l) b[l] = a[l] - s[l];
    }
    if (!fin) return;
#pragma unroll
    for (int l = 0; l < NC; ++l) {
        T e = d[3 * l] * b[0] + d[3 * l + 1] * b[1] + d[3 * l + 2] * b[2];
        const long o = 3 * (long)i + l0 + l;
        if (forward) {
            if (z) z[o] = to_prec<TZ>(e);
        } else {
            const TZ zn = TZ(zo[l] + to_prec<TZ>(e));
            z[o] = zn;
            e = to_prec<T>(zn);
        }
        x4[4 * (long)i + l0 + l] = e;
    }
}

// the colours of one residual launch
struct GsColours {
    int cnt[8], ge[8], ng[8], row0[8];
    long base[8];
};

// r = -U e (the residual after a forward sweep from zero), eight lanes a row,
// colour blockIdx.y
template <typename T>
__global__ void __launch_bounds__(256) gs_resid_kernel(const __grid_constant__ GsColours C,
                                                       const int32_t *__restrict__ rows, const T *__restrict__ val,
                                                       const int32_t *__restrict__ col, const T *x4,
                                                       T *__restrict__ out) {
    constexpr int L = 8, GB = kGsBlocks<T>;
    const int c = blockIdx.y, cnt = C.cnt[c], ge = C.ge[c], ng = C.ng[c];
    const int t = blockIdx.x * blockDim.x + threadIdx.x, r = t / L, g = t & (L - 1);
    const bool on = r < cnt;
    val += C.base[c] * 9 * GB;
    col += C.base[c] * GB;
    GsGroup<T> G;
    int i = 0;
    if (on) {
        if (ge + g < ng) gs_load<T>(G, val, col, r, ng, ge + g);
        i = __ldg(rows + C.row0[c] + r);
    }
    pdl_prologue();
    if (!on) return;
    T s[3] = {T(0), T(0), T(0)};
    if (ge + g < ng) gs_accumulate<T>(G, x4, i, s);
    for (int q = ge + g + L; q < ng; q += L) {
        gs_load<T>(G, val, col, r, ng, q);
        gs_accumulate<T>(G, x4, i, s);
    }
    gs_row_sum<T, L>(s);
    if (g == 0)
#pragma unroll
        for (int l = 0; l < 3; ++l) out[3 * (long)i + l] = -s[l];
}

template <typename T, typename TV, typename TZ, int L>
static msrsb_status gs_colour(const msrsb_handle *h, int c, int forward, int ng1, const TV *v, T *x4, TZ *z,
                              cudaStream_t s) {
    constexpr int GB = kGsBlocks<T>;
    const GsEll &E = h->gs;
    const int r0 = h->colour_ptr_h[c], cnt = h->colour_ptr_h[c + 1] - r0;
    MSRSB_PDL((gs_sweep_kernel<T, TV, TZ, L>), ceil_div((long)cnt * L, kGsThreads), kGsThreads, 0, s, cnt, forward,
              h->colour_rows + r0, E.ng[c], ng1, (const T *)E.val + E.base[c] * 9 * GB, E.col + E.base[c] * GB,
              (const T *)h->dinv, v, x4, z);
    return MSRSB_OK;
}

// A sweep over all colours. Forward: x4 = (D + L)^-1 v (padded), z = the same
// where given. Backward: z += (D + U)^-1 (v - A z) with x4 = z (padded, in T) on
// entry. Lanes a row: the power of two that gives each lane of a row one group,
// at most eight.
template <typename T, typename TV, typename TZ>
msrsb_status gs_sweep(const msrsb_handle *h, int forward, const TV *v, T *x4, TZ *z, cudaStream_t s) {
    const GsEll &E = h->gs;
    for (int q = 0; q < E.ncol; ++q) {
        const int c = forward ? q : E.ncol - 1 - q;
        if (h->colour_ptr_h[c + 1] == h->colour_ptr_h[c]) continue;
        const int n1 = forward ? E.ge[c] : E.ng[c];
        if (n1 <= 1) MSRSB_TRY((gs_colour<T, TV, TZ, 1>(h, c, forward, n1, v, x4, z, s)));
        else if (n1 <= 2) MSRSB_TRY((gs_colour<T, TV, TZ, 2>(h, c, forward, n1, v, x4, z, s)));
        else if (n1 <= 4) MSRSB_TRY((gs_colour<T, TV, TZ, 4>(h, c, forward, n1, v, x4, z, s)));
        else MSRSB_TRY((gs_colour<T, TV, TZ, 8>(h, c, forward, n1, v, x4, z, s)));
    }
    return MSRSB_OK;
}
template msrsb_status gs_sweep<double, double, double>(const msrsb_handle *, int, const double *, double *, double *,
                                                       cudaStream_t);
template msrsb_status gs_sweep<float, double, double>(const msrsb_handle *, int, const double *, float *, double *,
                                                      cudaStream_t);
template msrsb_status gs_sweep<float, float, double>(const msrsb_handle *, int, const float *, float *, double *,
                                                     cudaStream_t);

template <typename T>
msrsb_status gs_resid(const msrsb_handle *h, const T *x4, T *r, cudaStream_t s) {
    const GsEll &E = h->gs;
    GsColours C{};
    int most = 0;
    for (int c = 0; c < E.ncol; ++c) {
        C.row0[c] = h->colour_ptr_h[c];
        C.cnt[c] = h->colour_ptr_h[c + 1] - h->colour_ptr_h[c];
        C.ge[c] = E.ge[c];
        C.ng[c] = E.ng[c];
        C.base[c] = E.base[c];
        most = C.cnt[c] > most ? C.cnt[c] : most;
    }
    MSRSB_PDL((gs_resid_kernel<T>), dim3(ceil_div((long)most * 8, 256), E.ncol), 256, 0, s, C, h->colour_rows,
              (const T *)E.val, E.col, x4, r);
    return MSRSB_OK;
}
template msrsb_status gs_resid<double>(const msrsb_handle *, const double *, double *, cudaStream_t);
template msrsb_status gs_resid<float>(const msrsb_handle *, const float *, float *, cudaStream_t);

}  // namespace msrsb
