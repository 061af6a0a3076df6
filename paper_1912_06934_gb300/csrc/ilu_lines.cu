// ILU(0) smoother (second stage of Alg. 4) in a line-block elimination order.
//
// The grid is cut into blocks of whole x-lines, 2 lines high in y (and 2 deep
// in z in 3D). Blocks are coloured by the parity of their y (and z) block
// index, 2 colours in 2D and 4 in 3D, so two blocks of one colour never share
// a 3^dim stencil. The order is colour, then block, then the natural order
// inside the block (x fastest): each block keeps the natural order of the
// paper's MATLAB setting over its 2 (or 4) lines, and the strong couplings
// along x stay inside the sequential chains. Compared with a pointwise parity
// colouring this is a much stronger smoother on anisotropic and stretched
// grids, with fewer launches per application (2 C - 1 for C colours).
//
// Inside a block, the earlier neighbours of point (x, q) (q its line inside
// the block) are the previous point (x-1, q) of its own line and points of the
// block's earlier lines. A triangular sweep therefore takes the lines of a
// block in turn: every other contribution is gathered in parallel, and what
// remains is the first-order recurrence y_x = s_x - l_x y_{x-1} along the
// line, solved by a warp scan of affine maps. The factorisation runs one CTA
// per block, one warp per line, on a wavefront: line q trails line q-1 by two
// points, since (x, q) needs (x+1, q-1).
#include "common.cuh"
#include "lines.cuh"
#include <climits>
#include <cstring>
#include <type_traits>
#include <vector>
#include <cub/device/device_radix_sort.cuh>

namespace msrsb {


void diag_pos_launch(int n, const int32_t *rowptr, const int32_t *colidx, int32_t *dpos, int *status, cudaStream_t s);

// sort key of every row: colour, block, line inside the block, x
__global__ void line_key_kernel(int n, int dim, int nx, int ny, int nz, uint32_t *__restrict__ key,
                                int32_t *__restrict__ idx) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int x = i % nx, y = (i / nx) % ny, z = dim == 3 ? i / (nx * ny) : 0;
    const int by = y >> 1, bz = z >> 1, nby = (ny + 1) >> 1, nbz = dim == 3 ? (nz + 1) >> 1 : 1;
    const int c = (by & 1) | (dim == 3 ? ((bz & 1) << 1) : 0);
    const int sub = (y & 1) | (dim == 3 ? ((z & 1) << 1) : 0);
    const long blk = (long)by + (long)nby * bz;
    key[i] = (uint32_t)((((long)c * nby * nbz + blk) * 4 + sub) * nx + x);
    idx[i] = i;
}

// pos[rows[p]] = p; and every row's stencil-offset mask: bit
// (dx + 1) + 3 (dy + 1) + 9 (dz + 1) for each of its columns (the pattern
// lies in the 3^dim neighbourhood with ascending columns, so entry e of a row
// is the e-th set bit of its mask)
__global__ void lines_pos_kernel(int n, int dim, int nx, int ny, const int32_t *__restrict__ rows,
                                 const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                                 int32_t *__restrict__ pos, uint32_t *__restrict__ rmask) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int i = rows[p];
    pos[i] = p;
    const int xi = i % nx, yi = (i / nx) % ny, zi = dim == 3 ? i / (nx * ny) : 0;
    uint32_t m = 0;
    for (int e = rowptr[i]; e < rowptr[i + 1]; ++e) {
        const int j = colidx[e];
        const int xj = j % nx, yj = (j / nx) % ny, zj = dim == 3 ? j / (nx * ny) : 0;
        m |= 1u << ((xj - xi + 1) + 3 * (yj - yi + 1) + 9 * (zj - zi + 1));
    }
    rmask[i] = m;
}

// ---- factorisation --------------------------------------------------------------------

constexpr int kOffChunk = 4;

// Phase 1 of one colour, every row at once (one warp per row, lane e holding
// entry e): the earlier entries of earlier colours (positions below c0, all
// final) come first in the order, so they are eliminated in parallel before
// the in-block ones, in position order: l_ik = a_ik / u_kk (as a product with
// the stored 1 / u_kk), then every later entry (i, j) that row k also holds
// gets a_ij -= l_ik u_kj. Entry (k, j) is found from row k's stencil-offset
// mask (lines_pos_kernel): a popcount gives its place in row k, read straight
// from global memory, the chunk's reads issued together.
template <typename TF>
__global__ void __launch_bounds__(128) lines_factor_off_kernel(int c0, int cnt, int dim, int nx, int ny,
                                                               const int32_t *__restrict__ rows,
                                                               const int32_t *__restrict__ rowptr,
                                                               const int32_t *__restrict__ colidx,
                                                               const int32_t *__restrict__ pos,
                                                               const uint32_t *__restrict__ rmask,
                                                               TF *__restrict__ lu, const TF *__restrict__ rdiag) {
    const int w = (int)(((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (w >= cnt) return;  // whole warps leave together
    const int i = rows[c0 + w];
    const int b = rowptr[i], len = rowptr[i + 1] - b;  // len <= 32 (set-up checks it)
    const bool mine = lane < len;
    const int j = mine ? colidx[b + lane] : 0;
    const int pj = mine ? pos[j] : INT_MAX;
    TF a = mine ? lu[b + lane] : TF(0);
    const int xi = i % nx, yi = (i / nx) % ny, zi = dim == 3 ? i / (nx * ny) : 0;
    int ox = 1, oy = 1, oz = 1;  // this entry's offset from row i, zero-based per axis
    if (mine) {
        ox = j % nx - xi + 1;
        oy = (j / nx) % ny - yi + 1;
        oz = dim == 3 ? j / (nx * ny) - zi + 1 : 1;
    }
    const bool lower = mine && pj < c0;
    int kb = 0;
    uint32_t km = 0;
    TF rd = TF(0);
    if (lower) {  // the pivot row's start, mask and 1 / u_kk
        kb = rowptr[j];
        km = rmask[j];
        rd = rdiag[j];
    }
    const unsigned lm = __ballot_sync(0xffffffffu, lower);
    const int nlow = __popc(lm);
    int rank = 0;  // place of this pivot in the position order
    for (unsigned mm = lm; mm; mm &= mm - 1) {
        const int po = __shfl_sync(0xffffffffu, pj, __ffs(mm) - 1);
        rank += (lower && po < pj) ? 1 : 0;
    }
    for (int t0 = 0; t0 < nlow; t0 += kOffChunk) {
        TF u[kOffChunk], rk[kOffChunk];
        int ql[kOffChunk];
#pragma unroll
        for (int t = 0; t < kOffChunk; ++t) {
            const bool on = t0 + t < nlow;  // uniform
            const unsigned bm = __ballot_sync(0xffffffffu, lower && rank == t0 + t);
            const int qq = on ? __ffs(bm) - 1 : 0;
            ql[t] = on ? qq : -1;
            const int pk = __shfl_sync(0xffffffffu, pj, qq);
            const int kx = __shfl_sync(0xffffffffu, ox, qq), ky = __shfl_sync(0xffffffffu, oy, qq),
                      kz = __shfl_sync(0xffffffffu, oz, qq);
            const int kbt = __shfl_sync(0xffffffffu, kb, qq);
            const uint32_t kmt = __shfl_sync(0xffffffffu, km, qq);
            rk[t] = __shfl_sync(0xffffffffu, rd, qq);
            const int dx = ox - kx + 1, dy = oy - ky + 1, dz = oz - kz + 1;  // j's offset from k
            const bool near = dx >= 0 && dx <= 2 && dy >= 0 && dy <= 2 && dz >= 0 && dz <= 2;
            const int o = near ? dx + 3 * dy + 9 * dz : 0;
            const bool hit = on && mine && pj > pk && near && ((kmt >> o) & 1u);
            u[t] = hit ? lu[kbt + __popc(kmt & ((1u << o) - 1u))] : TF(0);
        }
#pragma unroll
        for (int t = 0; t < kOffChunk; ++t) {
            const TF lik = __shfl_sync(0xffffffffu, a, ql[t] < 0 ? 0 : ql[t]) * rk[t];
            if (ql[t] >= 0) {  // uniform
                if (lane == ql[t]) a = lik;
                else a = a - lik * u[t];
            }
        }
    }
    if (mine) lu[b + lane] = a;
}

// Phase 2 of one colour: the in-block earlier entries. CTA b0 + blockIdx.x
// handles one block, warp q its line q; at time step T warp q finishes point
// x = T - 2 q of its line. With couplings reaching at most one point along x,
// point (q, x) needs the points (q', x - 1 .. x + 1) of the lines q' < q
// (finished at steps up to T - 1) and (q, x - 1). A point's row is final
// once finished and is then needed for at most 2 nsub more steps, so each
// line keeps its last kRing rows in shared memory: a row is copied in
// (cp.async) kAhead steps before its turn and written through to global
// memory when finished. In-block tests come from the grid position of the
// columns (the order's key), so no position gather sits on the critical path.
// A row's entries lie at distinct offsets of the 3^dim stencil, in column
// order, so a finished row also keeps the mask of its offsets (bit
// (dx + 1) + 3 (dy + 1) + 9 (dz + 1)): entry (k, j) of a pivot row k is then
// found by a popcount of the mask below j's offset from k.
constexpr int kRing = 16, kAhead = 4, kPivChunk = 4, kLinesMaxNx = 256;

template <typename TF>
__global__ void __launch_bounds__(128) lines_factor_ring_kernel(
    int c, int b0, const int32_t *__restrict__ blk_start, const int32_t *__restrict__ blk_nsub, int dim, int nx,
    int ny, const int32_t *__restrict__ rows, const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
    TF *__restrict__ lu, TF *__restrict__ rdiag, int *__restrict__ status) {
    __shared__ TF s_val[4][kRing][32];
    __shared__ int32_t s_col[4][kRing][32];
    __shared__ TF s_rd[4][kRing];
    __shared__ unsigned s_mask[4][kRing];
    __shared__ int32_t s_ri[4][kLinesMaxNx], s_rb[4][kLinesMaxNx], s_rl[4][kLinesMaxNx];
    const int b = b0 + blockIdx.x, q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int st = blk_start[b], nsub = blk_nsub[b];
    for (int t = threadIdx.x; t < nsub * nx; t += blockDim.x) {
        const int i = rows[st + t], rb = rowptr[i];
        s_ri[t / nx][t % nx] = i;
        s_rb[t / nx][t % nx] = rb;
        s_rl[t / nx][t % nx] = rowptr[i + 1] - rb;
    }
    __syncthreads();
    const int y0 = ((s_ri[0][0] / nx) % ny) & ~1;
    const int nyb = min(2, ny - y0);  // lines of the block along y
    int yq = 0, zq = 0;
    if (q < nsub) {
        const int r = s_ri[q][0] / nx;
        yq = r % ny;
        zq = dim == 3 ? r / ny : 0;
    }
    const int kin_base = ((yq & 1) | ((zq & 1) << 1)) * nx;  // in-block order key of (q, 0)
    const int steps = nx + 2 * (nsub - 1);
    for (int T = -kAhead; T < steps; ++T) {
        if (q < nsub) {
            const int xl = T - 2 * q + kAhead;
            if (xl >= 0 && xl < nx && lane < s_rl[q][xl]) {
                const int e = s_rb[q][xl] + lane;
                cp_async4(&s_col[q][xl & (kRing - 1)][lane], colidx + e);
                cp_async_val(&s_val[q][xl & (kRing - 1)][lane], lu + e);
            }
        }
        cp_async_commit();
        if (T < 0) continue;  // uniform over the CTA
        cp_async_wait<kAhead>();
        const int x = T - 2 * q;
        if (q < nsub && x >= 0 && x < nx) {
            const int slot = x & (kRing - 1);
            const int i = s_ri[q][x], len = s_rl[q][x];
            const bool mine = lane < len;
            const int j = mine ? s_col[q][slot][lane] : -1;
            TF a = mine ? s_val[q][slot][lane] : TF(0);
            int xj = 0, yj = 0, zj = 0;
            if (mine) {
                xj = j % nx;
                const int r = j / nx;
                yj = r % ny;
                zj = dim == 3 ? r / ny : 0;
            }
            // this entry's stencil offset from row i (zero-based per axis)
            const int ox = xj - x + 1, oy = yj - yq + 1, oz = zj - zq + 1;
            const unsigned mask_i = __reduce_or_sync(0xffffffffu, mine ? 1u << (ox + 3 * oy + 9 * oz) : 0u);
            const bool inb = mine && (yj >> 1) == (yq >> 1) && (zj >> 1) == (zq >> 1);
            const int kin_j = ((yj & 1) | ((zj & 1) << 1)) * nx + xj;
            const int colj = ((yj >> 1) & 1) | (dim == 3 ? (((zj >> 1) & 1) << 1) : 0);
            const bool piv = inb && kin_j < kin_base + x;
            // Inside one block the key (z & 1, y & 1, x) orders the points as
            // their indices do, so the pivots come in lane (column) order.
            const bool later_in = inb;  // in-block: later than pivot k when kin_j > kin_k
            const bool later_off = mine && !inb && colj > c;
            unsigned rest = __ballot_sync(0xffffffffu, piv);
            while (rest) {  // uniform
                // every match of the chunk first (the pivot rows are final), then
                // the eliminations in order
                TF u[kPivChunk], rk[kPivChunk];
                int ql[kPivChunk];
#pragma unroll
                for (int t = 0; t < kPivChunk; ++t) {
                    const bool on = rest != 0;  // uniform
                    const int qq = on ? __ffs(rest) - 1 : 0;
                    rest &= rest - 1;
                    ql[t] = on ? qq : -1;
                    // pivot k: its offset from row i, hence its grid position
                    const int kx = __shfl_sync(0xffffffffu, ox, qq), ky = __shfl_sync(0xffffffffu, oy, qq),
                              kz = __shfl_sync(0xffffffffu, oz, qq);
                    const int xk = x + kx - 1, yk = yq + ky - 1, zk = zq + kz - 1;
                    const int kin_k = ((yk & 1) | ((zk & 1) << 1)) * nx + xk;
                    const int lk = on ? (yk & 1) + (zk & 1) * nyb : q, sk = on ? xk & (kRing - 1) : slot;
                    rk[t] = on ? s_rd[lk][sk] : TF(0);
                    const unsigned mk = on ? s_mask[lk][sk] : 0u;
                    // j's offset from k
                    const int dx = ox - kx + 1, dy = oy - ky + 1, dz = oz - kz + 1;
                    const bool near = dx >= 0 && dx <= 2 && dy >= 0 && dy <= 2 && dz >= 0 && dz <= 2;
                    const int o = near ? dx + 3 * dy + 9 * dz : 0;
                    const bool hit = on && near && (later_off || (later_in && kin_j > kin_k)) && ((mk >> o) & 1u);
                    u[t] = hit ? s_val[lk][sk][__popc(mk & ((1u << o) - 1u))] : TF(0);
                }
#pragma unroll
                for (int t = 0; t < kPivChunk; ++t) {
                    const TF lik = __shfl_sync(0xffffffffu, a, ql[t] < 0 ? 0 : ql[t]) * rk[t];
                    if (ql[t] >= 0) {  // uniform
                        if (lane == ql[t]) a = lik;
                        else a = a - lik * u[t];
                    }
                }
            }
            if (mine) {
                s_val[q][slot][lane] = a;
                lu[s_rb[q][x] + lane] = a;
            }
            const unsigned dm = __ballot_sync(0xffffffffu, mine && j == i);
            const TF uii = __shfl_sync(0xffffffffu, a, dm ? __ffs(dm) - 1 : 0);
            if (lane == 0) {
                const bool bad = !dm || uii == TF(0) || !isfinite((double)uii);
                if (bad) atomicCAS(status, 0, 1 + i);
                const TF rd = bad ? TF(0) : TF(1) / uii;
                s_rd[q][slot] = rd;
                s_mask[q][slot] = mask_i;
                rdiag[i] = rd;
            }
        }
        __syncthreads();  // the step's rows are final before the next step reads them
    }
    cp_async_wait<0>();
}

// ---- factors for the sweeps -------------------------------------------------------------
//
// A's pattern lies in the 3^dim neighbourhood, so a point's entries fall on at
// most 8 neighbour lines of 3 points each and on its own line, and the line
// (the same for every point of a line) says which block it belongs to. The
// factors are therefore stored by neighbour line and x offset, zeros where the
// pattern has no entry, without column indices: half the bytes of column and
// value pairs, read as 16-byte vectors.
//  - off-block: up to 5 neighbour lines lie in other blocks (per axis one of
//    the two neighbours); by the colours' order, colour c has noff[0][c]
//    lines of earlier and noff[1][c] of later colours. nbr[dir][line][5] holds
//    the first position of each (ascending in z, then y); off[dir] their
//    coefficients.
//  - in-block: the block's other lines; in[0] of a point of line q holds
//    (l to x-1 on its own line, then 3 per earlier line of the block), in[1]
//    (u to x+1, 1 / u_pp, then 3 per later line).
// Group g (kLineGroup<T> values, 16 bytes) of point x of a line sits at
// (line * groups + g) * nx + x, so a warp reads consecutive vectors. Every
// line keeps room for its widest in-block record; groups past a line's own
// count are never read.
// nbr[dir][line][5] (dir 0: lines of earlier colours, 1: of later ones), the
// line's own first position where there is no such line
__global__ void lines_nbr_kernel(int nlines, int dim, int nx, int ny, int nz, const int32_t *__restrict__ rows,
                                 const int32_t *__restrict__ pos, int32_t *__restrict__ nbr) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nlines) return;
    const int i = rows[l * nx], y = (i / nx) % ny, z = dim == 3 ? i / (nx * ny) : 0;
    const int c = ((y >> 1) & 1) | (dim == 3 ? ((z >> 1) & 1) << 1 : 0);
    int cnt[2] = {0, 0};
    for (int dz = dim == 3 ? -1 : 0; dz <= (dim == 3 ? 1 : 0); ++dz)
        for (int dy = -1; dy <= 1; ++dy) {
            const int yk = y + dy, zk = z + dz;
            if (yk < 0 || yk >= ny || zk < 0 || zk >= nz) continue;
            if ((yk >> 1) == (y >> 1) && (zk >> 1) == (z >> 1)) continue;
            const int ck = ((yk >> 1) & 1) | (dim == 3 ? ((zk >> 1) & 1) << 1 : 0);
            const int d = ck < c ? 0 : 1;  // blocks of one colour are not neighbours
            nbr[((long)d * nlines + l) * kLineNbr + cnt[d]++] = pos[nx * (yk + (long)ny * zk)];
        }
    for (int d = 0; d < 2; ++d)
        for (int k = cnt[d]; k < kLineNbr; ++k) nbr[((long)d * nlines + l) * kLineNbr + k] = l * nx;
}

template <typename T>
__global__ void __launch_bounds__(128) lines_fill_kernel(int n, int dim, int nx, int ny, int nz,
                                                         const int32_t *__restrict__ rowptr,
                                                         const uint32_t *__restrict__ rmask,
                                                         const T *__restrict__ lu, const int32_t *__restrict__ rows,
                                                         const IluLines L, T *__restrict__ offl, T *__restrict__ offu,
                                                         T *__restrict__ inl, T *__restrict__ inu) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int i = rows[p], x = i % nx, y = (i / nx) % ny, z = dim == 3 ? i / (nx * ny) : 0;
    const int c = ((y >> 1) & 1) | (dim == 3 ? ((z >> 1) & 1) << 1 : 0);
    const int sy = min(2, ny - (y & ~1)), q = (y & 1) + (z & 1) * sy;
    T off[2][kLineOff], in[2][kLineIn];
#pragma unroll
    for (int k = 0; k < kLineOff; ++k) off[0][k] = off[1][k] = T(0);
#pragma unroll
    for (int k = 0; k < kLineIn; ++k) in[0][k] = in[1][k] = T(0);
    const uint32_t mask = rmask[i];
    int e = rowptr[i], cnt[2] = {0, 0};
    for (int o = 0; o < (dim == 3 ? 27 : 18); o += 3) {  // entries in column order, three x offsets at a time
        const int dy = (o / 3) % 3 - 1, dz = dim == 3 ? o / 9 - 1 : 0;
        if (dim != 3 && o < 9) continue;  // 2D rows use the bits of dz = 0
        const uint32_t m3 = (mask >> o) & 7u;
        const int yk = y + dy, zk = z + dz;
        if (yk < 0 || yk >= ny || zk < 0 || zk >= nz) continue;
        T v[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) v[d] = (m3 >> d) & 1u ? lu[e + __popc(m3 & ((1u << d) - 1u))] : T(0);
        e += __popc(m3);
        if (dy == 0 && dz == 0) {
            in[0][0] = v[0];
            in[1][0] = v[2];
            in[1][1] = T(1) / v[1];
        } else if ((yk >> 1) == (y >> 1) && (zk >> 1) == (z >> 1)) {
            const int qk = (yk & 1) + (zk & 1) * sy;
            T *dst = qk < q ? in[0] + 1 + 3 * qk : in[1] + 2 + 3 * (qk - q - 1);
#pragma unroll
            for (int d = 0; d < 3; ++d) dst[d] = v[d];
        } else {
            const int ck = ((yk >> 1) & 1) | (dim == 3 ? ((zk >> 1) & 1) << 1 : 0);
            const int dir = ck < c ? 0 : 1;
            T *dst = off[dir] + 3 * cnt[dir]++;
#pragma unroll
            for (int d = 0; d < 3; ++d) dst[d] = v[d];
        }
    }
    constexpr int G = kLineGroup<T>;
    const long line = p / nx, lc = line - L.cptr[c] / nx;  // the line, and its place in the colour
    using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    auto put = [&](T *dst, long at, const T *src) {
        V v;
        memcpy(&v, src, 16);
        reinterpret_cast<V *>(dst)[at] = v;
    };
    for (int d = 0; d < 2; ++d) {
        const int ng = line_groups<T>(3 * L.noff[d][c]);
        T *o = (d == 0 ? offl : offu) + L.obase[d][c];
        for (int g = 0; g < ng; ++g) put(o, (lc * ng + g) * nx + x, off[d] + g * G);
        constexpr int NI = line_groups<T>(kLineIn);
        for (int g = 0; g < NI; ++g) put(d == 0 ? inl : inu, (line * NI + g) * nx + x, in[d] + g * G);
    }
}

// ---- host side ---------------------------------------------------------------------------------

bool lines_fit(const msrsb_grid *g) { return g->nx >= 1 && g->nx <= kLinesMaxNx && (g->dim == 2 || g->dim == 3); }

// Order, block table and ILU(0) factors of a scalar operator in the
// line-block order; lu holds A's values (TF) on entry and is overwritten.
// A's pattern lies within every point's 3^dim neighbourhood (stencil_check):
// blocks of one colour are then uncoupled and a point couples to its line
// neighbours x - 1, x + 1 only.
template <typename TF>
msrsb_status lines_setup(msrsb_handle *h, TF *lu, cudaStream_t s) {
    const msrsb_mat &A = h->A;
    const msrsb_grid &g = h->grid;
    const int n = h->n, dim = g.dim, nx = g.nx, ny = g.ny, nz = dim == 3 ? g.nz : 1;
    IluLines &L = h->lines;
    L.nx = nx;
    L.ncol = dim == 3 ? 4 : 2;
    // ---- the order: sort rows by (colour, block, line, x) ----
    uint32_t *key = nullptr, *key2 = nullptr;
    int32_t *idx = nullptr;
    MSRSB_TRY(dalloc(&key, n, s));
    MSRSB_TRY(dalloc(&key2, n, s));
    MSRSB_TRY(dalloc(&idx, n, s));
    MSRSB_TRY(dalloc(&L.rows, n, s));
    MSRSB_TRY(dalloc(&h->pos_of, n, s));
    line_key_kernel<<<ceil_div(n, 256), 256, 0, s>>>(n, dim, nx, ny, nz, key, idx);
    MSRSB_LAUNCHED("line_key_kernel");
    size_t tmp = 0;
    MSRSB_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, tmp, key, key2, idx, L.rows, n, 0, 32, s));
    char *tb = nullptr;
    MSRSB_TRY(dalloc(&tb, tmp, s));
    MSRSB_CUDA(cub::DeviceRadixSort::SortPairs(tb, tmp, key, key2, idx, L.rows, n, 0, 32, s));
    dfree(tb, s);
    dfree(key, s);
    dfree(key2, s);
    dfree(idx, s);
    uint32_t *rmask = nullptr;
    MSRSB_TRY(dalloc(&rmask, n, s));
    lines_pos_kernel<<<ceil_div(n, 256), 256, 0, s>>>(n, dim, nx, ny, L.rows, A.rowptr, A.colidx, h->pos_of, rmask);
    MSRSB_LAUNCHED("lines_pos_kernel");
    // ---- block table (host): blocks of each colour in block order ----
    const int nby = (ny + 1) / 2, nbz = dim == 3 ? (nz + 1) / 2 : 1;
    std::vector<int32_t> bline, bstart, bnsub;
    int run = 0;
    for (int c = 0; c < L.ncol; ++c) {
        L.cptr[c] = run;
        L.bptr[c] = (int)bstart.size();
        for (int bz = 0; bz < nbz; ++bz)
            for (int by = 0; by < nby; ++by) {
                const int cc = (by & 1) | (dim == 3 ? ((bz & 1) << 1) : 0);
                if (cc != c) continue;
                const int sy = ny - 2 * by < 2 ? 1 : 2, sz = dim == 3 ? (nz - 2 * bz < 2 ? 1 : 2) : 1;
                bline.push_back(run / nx);
                bstart.push_back(run);
                bnsub.push_back(sy * sz);
                run += sy * sz * nx;
            }
    }
    L.cptr[L.ncol] = run;
    L.bptr[L.ncol] = (int)bstart.size();
    if (run != n) return fail(MSRSB_ESHAPE, "line blocks cover %d of %d rows", run, n);
    const int nblk = (int)bstart.size();
    int32_t *blk_start = nullptr;
    MSRSB_TRY(dalloc(&blk_start, nblk, s));
    MSRSB_TRY(dalloc(&L.blk_line, nblk, s));
    MSRSB_TRY(dalloc(&L.blk_nsub, nblk, s));
    MSRSB_TRY(upload(L.blk_line, bline.data(), nblk * sizeof(int32_t), s));
    MSRSB_TRY(upload(blk_start, bstart.data(), nblk * sizeof(int32_t), s));
    MSRSB_TRY(upload(L.blk_nsub, bnsub.data(), nblk * sizeof(int32_t), s));
    // ---- factorisation, colour by colour ----
    int *status = nullptr;
    TF *rdiag = nullptr;
    int32_t *dpos = nullptr;
    MSRSB_TRY(dalloc(&status, 1, s));
    MSRSB_TRY(dalloc(&rdiag, n, s));
    MSRSB_TRY(dalloc(&dpos, n, s));
    MSRSB_CUDA(cudaMemsetAsync(status, 0, sizeof(int), s));
    diag_pos_launch(n, A.rowptr, A.colidx, dpos, status, s);
    MSRSB_LAUNCHED("diag_pos_kernel");
    for (int c = 0; c < L.ncol; ++c) {
        const int nb = L.bptr[c + 1] - L.bptr[c];
        if (!nb) continue;
        const int cnt = L.cptr[c + 1] - L.cptr[c];
        if (c > 0) {
            lines_factor_off_kernel<TF><<<ceil_div((long)cnt * 32, 128), 128, 0, s>>>(
                L.cptr[c], cnt, dim, nx, ny, L.rows, A.rowptr, A.colidx, h->pos_of, rmask, lu, rdiag);
            MSRSB_LAUNCHED("lines_factor_off_kernel");
        }
        lines_factor_ring_kernel<TF><<<nb, 128, 0, s>>>(c, L.bptr[c], blk_start, L.blk_nsub, dim, nx, ny, L.rows,
                                                        A.rowptr, A.colidx, lu, rdiag, status);
        MSRSB_LAUNCHED("lines_factor_ring_kernel");
    }
    // ---- the sweeps' coefficients by neighbour line, and the lines' neighbours ----
    const int nlines = n / nx;
    long ot[2] = {0, 0};
    for (int c = 0; c < L.ncol; ++c) {
        const int flips = dim == 3 ? 3 : 1;  // neighbour blocks' colours: c with y's and z's parity flipped
        L.noff[0][c] = L.noff[1][c] = 0;
        for (int f = 1; f <= flips; ++f) L.noff[(c ^ f) < c ? 0 : 1][c] += f == 3 || dim == 2 ? 1 : 2;
        for (int d = 0; d < 2; ++d) {
            L.obase[d][c] = ot[d];
            ot[d] += (long)(L.cptr[c + 1] - L.cptr[c]) * line_groups<TF>(3 * L.noff[d][c]) * kLineGroup<TF>;
        }
    }
    TF *offl = nullptr, *offu = nullptr, *inl = nullptr, *inu = nullptr;
    MSRSB_TRY(dalloc(&offl, ot[0], s));
    L.off[0] = offl;
    MSRSB_TRY(dalloc(&offu, ot[1], s));
    L.off[1] = offu;
    MSRSB_TRY(dalloc(&inl, (size_t)n * kLineIn, s));
    L.in[0] = inl;
    MSRSB_TRY(dalloc(&inu, (size_t)n * kLineIn, s));
    L.in[1] = inu;
    MSRSB_TRY(dalloc(&L.nbr, (size_t)2 * nlines * kLineNbr, s));
    lines_nbr_kernel<<<ceil_div(nlines, 128), 128, 0, s>>>(nlines, dim, nx, ny, nz, L.rows, h->pos_of, L.nbr);
    MSRSB_LAUNCHED("lines_nbr_kernel");
    lines_fill_kernel<TF><<<ceil_div(n, 128), 128, 0, s>>>(n, dim, nx, ny, nz, A.rowptr, rmask, lu, L.rows, L, offl,
                                                           offu, inl, inu);
    MSRSB_LAUNCHED("lines_fill_kernel");
    int hs = 0;
    MSRSB_TRY(read_back(&hs, status, sizeof(int), s));
    dfree(rdiag, s);
    dfree(rmask, s);
    dfree(status, s);
    dfree(dpos, s);
    dfree(blk_start, s);
    if (hs < 0) return fail(MSRSB_EINVAL, "ILU(0): row %d has more than 32 entries", -hs - 1);
    if (hs) return fail(MSRSB_EBREAKDOWN, "ILU(0): zero pivot at row %d", hs - 1);
    return MSRSB_OK;
}
template msrsb_status lines_setup<double>(msrsb_handle *, double *, cudaStream_t);
template msrsb_status lines_setup<float>(msrsb_handle *, float *, cudaStream_t);

void lines_free(IluLines *L, cudaStream_t s) {
    dfree(L->rows, s);
    dfree(L->blk_line, s);
    dfree(L->blk_nsub, s);
    dfree(L->nbr, s);
    for (int d = 0; d < 2; ++d) {
        dfree(L->off[d], s);
        dfree(L->in[d], s);
    }
}

}  // namespace msrsb
