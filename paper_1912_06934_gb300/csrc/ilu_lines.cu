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

namespace msrsb {


// ---- the order ------------------------------------------------------------------------
//
// Colour c's lines start at line cl[c] (a line has nx positions); its blocks follow
// row of blocks by row of blocks, and only the last block along y or z is thinner than
// two lines, so a line's place in the order is arithmetic.
struct LineGrid {
    int dim, nx, ny, nz;
    int cl[5];  // first line of each colour (+ end)
    int Ly[2];  // lines along y in blocks of even and of odd index
};

__device__ __forceinline__ int line_at(const LineGrid &G, int y, int z) {
    const int by = y >> 1, bz = z >> 1, sy = min(2, G.ny - 2 * by), sz = min(2, G.nz - 2 * bz);
    return G.cl[(by & 1) | ((bz & 1) << 1)] + (bz >> 1) * 2 * G.Ly[by & 1] + (by >> 1) * 2 * sz + (y & 1) +
           (z & 1) * sy;
}

// the grid position of line l of colour c
__device__ __forceinline__ void line_yz(const LineGrid &G, int c, int l, int &y, int &z) {
    const int r = l - G.cl[c], row = 2 * G.Ly[c & 1], bz = 2 * (r / row) + (c >> 1), sz = min(2, G.nz - 2 * bz);
    const int r2 = r % row, by = 2 * (r2 / (2 * sz)) + (c & 1), sy = min(2, G.ny - 2 * by), sub = r2 % (2 * sz);
    y = 2 * by + sub % sy;
    z = 2 * bz + sub / sy;
}

// A point's offsets in the 3^dim stencil: o = (dx + 1) + 3 (dy + 1) + 9 (dz + 1), dz = 0
// in 2D. The factorisation works on rows of kLineRow values by offset, in the order, with
// zeros where the pattern has no entry: an entry's place in any row is then known
// without a search, and a warp (lane o = offset o) reads and writes rows as they lie.
constexpr int kLineRow = 27;
constexpr int kLineDiag = 13;

// rows[p] and pos[i], every row's values D[p][o] in the factorisation's precision and
// its pattern rmask[p] (bit o). A warp a row; the pattern lies in the 3^dim neighbourhood
// with strictly ascending columns (stencil_check), so entry e of a row is the e-th set
// bit of its mask. 2^21 rows of 27 beside the coarse factorisation: 0.57 ms. (Sorting
// the rows by a key, converting the values, forming masks and finding diagonals: 0.80.)
template <typename TF>
__global__ void __launch_bounds__(256) lines_gather_kernel(int n, const LineGrid G, const int32_t *__restrict__ rowptr,
                                                           const int32_t *__restrict__ colidx,
                                                           const double *__restrict__ val, int32_t *__restrict__ rows,
                                                           int32_t *__restrict__ pos, uint32_t *__restrict__ rmask,
                                                           TF *__restrict__ D) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= n) return;  // whole warps leave together
    const int x = i % G.nx, r = i / G.nx, y = r % G.ny, z = r / G.ny;
    const int b = rowptr[i], len = rowptr[i + 1] - b;
    const bool mine = lane < len;
    int o = 0;
    TF v = TF(0);
    if (mine) {
        const int j = colidx[b + lane];
        v = TF(val[b + lane]);
        if (G.nx >= 3 && G.ny >= 3) {  // offsets as the digits of j - i in the strides
            const int nxy = G.nx * G.ny;
            int t = j - i + nxy + G.nx + 1;
            const int oz = (t >= nxy) + (t >= 2 * nxy);
            t -= oz * nxy;
            const int oy = (t >= G.nx) + (t >= 2 * G.nx);
            o = t - oy * G.nx + 3 * oy + 9 * oz;
        } else {
            const int rj = j / G.nx;
            o = (j % G.nx - x + 1) + 3 * (rj % G.ny - y + 1) + 9 * (rj / G.ny - z + 1);
        }
    }
    const uint32_t m = __reduce_or_sync(0xffffffffu, mine ? 1u << o : 0u);
    const TF w = __shfl_sync(0xffffffffu, v, __popc(m & ((1u << lane) - 1u)) & 31);
    const int p = line_at(G, y, z) * G.nx + x;
    if (lane < kLineRow) D[p * kLineRow + lane] = (m >> lane) & 1u ? w : TF(0);
    if (lane == 0) {
        rows[p] = i;
        pos[i] = p;
        rmask[p] = m;
    }
}

// ---- factorisation --------------------------------------------------------------------
//
// Row by row in the order (IKJ): for every earlier entry k of row i, in position order,
// l_ik = a_ik / u_kk (as a product with the stored 1 / u_kk), then every later entry
// (i, j) that row k also holds gets a_ij -= l_ik u_kj. With rows by offset, row k's entry
// towards j sits at offset o_j - o_k + 13, the same for every point of a line: which
// lanes a pivot updates and where their operands lie is worked out once per line.

// The lane's neighbour line (its first position; -1 outside the grid or no offset)
__device__ __forceinline__ int lane_line(const LineGrid &G, int lane, int y, int z) {
    const int yj = y + (lane / 3) % 3 - 1, zj = z + lane / 9 - 1;
    if (lane >= kLineRow || yj < 0 || yj >= G.ny || zj < 0 || zj >= G.nz) return -1;
    return line_at(G, yj, zj) * G.nx;
}

// whether pivot offset ok, on the line at kp, updates the lane's entry (line at pl): near
// row k, and later than it
__device__ __forceinline__ bool pivot_hits(int lane, int pl, int ok, int kp) {
    const int dx = lane % 3 - ok % 3, dy = (lane / 3) % 3 - (ok / 3) % 3, dz = lane / 9 - ok / 9;
    return pl >= 0 && abs(dx) <= 1 && abs(dy) <= 1 && abs(dz) <= 1 && (pl > kp || (pl == kp && dx > 0));
}

// Phase 1 of one colour: the pivots of earlier colours (all final) on up to kLineNbr
// neighbour lines, which come first in the order. A warp takes every fourth point of a
// piece of a line; a point's operands are loaded together. 2^19 rows: 0.42 to
// 0.59 ms with searches for the operands, now 0.25 to 0.31.
constexpr int kOffPoints = 32;

template <typename TF>
__global__ void __launch_bounds__(128) lines_factor_off_kernel(const LineGrid G, int c,
                                                               const uint32_t *__restrict__ rmask, TF *D,
                                                               const TF *__restrict__ rdiag) {
    const int lane = threadIdx.x & 31, pieces = (G.nx + kOffPoints - 1) / kOffPoints;
    const int l = G.cl[c] + blockIdx.x / pieces, x0 = (blockIdx.x % pieces) * kOffPoints;
    int y, z;
    line_yz(G, c, l, y, z);
    const int pl = lane_line(G, lane, y, z), c0 = G.cl[c] * G.nx;
    int kp[kLineNbr], ko[kLineNbr], last = -1;  // the pivots' lines in position order, offset towards x - 1
    unsigned hits = 0;
#pragma unroll
    for (int t = 0; t < kLineNbr; ++t) {
        const int key = pl > last && pl < c0 && lane % 3 == 1 ? pl : INT_MAX;
        const int first = __reduce_min_sync(0xffffffffu, key);
        const unsigned who = __ballot_sync(0xffffffffu, key == first);
        kp[t] = first == INT_MAX ? -1 : first;
        ko[t] = first == INT_MAX ? 0 : __ffs(who) - 2;
        if (first == INT_MAX) continue;
        last = first;
#pragma unroll
        for (int d = 0; d < 3; ++d) hits |= pivot_hits(lane, pl, ko[t] + d, first) ? 1u << (3 * t + d) : 0u;
    }
    const int x1 = min(x0 + kOffPoints, G.nx);
    for (int x = x0 + (int)(threadIdx.x >> 5); x < x1; x += 4) {
        const int p = l * G.nx + x;
        const uint32_t m = rmask[p];
        const unsigned h = (m >> lane) & 1u ? hits : 0u;  // only entries of the pattern change
        TF a = lane < kLineRow ? D[p * kLineRow + lane] : TF(0);
        TF u[3 * kLineNbr], rk[3 * kLineNbr];
#pragma unroll
        for (int t = 0; t < kLineNbr; ++t)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int ok = ko[t] + d, pk = kp[t] + x + d - 1;
                const bool on = kp[t] >= 0 && ((m >> ok) & 1u);  // uniform
                u[3 * t + d] = on && ((h >> (3 * t + d)) & 1u) ? D[pk * kLineRow + lane - ok + kLineDiag] : TF(0);
                rk[3 * t + d] = on ? rdiag[pk] : TF(0);
            }
#pragma unroll
        for (int t = 0; t < kLineNbr; ++t)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int ok = ko[t] + d;
                if (kp[t] < 0 || !((m >> ok) & 1u)) continue;  // uniform
                const TF lik = __shfl_sync(0xffffffffu, a, ok) * rk[3 * t + d];
                if (lane == ok) a = lik;
                else a = a - lik * u[3 * t + d];
            }
        if (lane < kLineRow) D[p * kLineRow + lane] = a;
    }
}

// Phase 2 of one colour: the pivots inside the block. CTA b0 + blockIdx.x handles one
// block, warp q its line q; at time step T warp q finishes point x = T - 2 q of its
// line. With couplings reaching at most one point along x, point (q, x) needs the points
// (q', x - 1 .. x + 1) of the lines q' < q (finished at steps up to T - 1) and (q, x - 1).
// A point's row is final once finished and is then needed for at most 2 nsub more steps,
// so each line keeps its last kRing rows in shared memory: a row is copied in (cp.async)
// kAhead steps before its turn and written through to global memory when finished. The
// chain of steps bounds it: a step's operands are all read first, then every pivot costs
// a shuffle, a product and an update. (Searching for the operands by columns and masks put
// about 650 instructions on a step: 0.76 ms a colour of 2^19 rows, now 0.25; 2^16 rows
// 0.18, now 0.06.)
constexpr int kRing = 16, kAhead = 4, kLinesMaxNx = 256;
constexpr int kBlkPiv = 10;  // three earlier lines of the block, then the line's point before

template <typename TF>
__global__ void __launch_bounds__(128) lines_factor_ring_kernel(const LineGrid G, int c, int b0,
                                                                const int32_t *__restrict__ blk_line,
                                                                const int32_t *__restrict__ blk_nsub,
                                                                const int32_t *__restrict__ rows,
                                                                const uint32_t *__restrict__ rmask,
                                                                TF *__restrict__ D, TF *__restrict__ rdiag,
                                                                int *__restrict__ status) {
    __shared__ TF s_val[4][kRing][32];
    __shared__ TF s_rd[4][kRing];
    __shared__ uint32_t s_mask[4][kLinesMaxNx];
    const int b = b0 + blockIdx.x, q = threadIdx.x >> 5, lane = threadIdx.x & 31, nx = G.nx;
    const int lb = blk_line[b], nsub = blk_nsub[b];
    for (int t = threadIdx.x; t < nsub * nx; t += blockDim.x) s_mask[t / nx][t % nx] = rmask[lb * nx + t];
    int ok0[3] = {0, 0, 0};  // offset towards x - 1 on the block's line t
    unsigned hits = 0;
    if (q < nsub) {
        int y, z;
        line_yz(G, c, lb + q, y, z);
        const int pl = lane_line(G, lane, y, z);
        for (int t = 0; t < 3; ++t) {
            if (t >= q) break;
            int yt, zt;
            line_yz(G, c, lb + t, yt, zt);
            ok0[t] = 3 * (yt - y + 1) + 9 * (zt - z + 1);
#pragma unroll
            for (int d = 0; d < 3; ++d)
                hits |= pivot_hits(lane, pl, ok0[t] + d, (lb + t) * nx) ? 1u << (3 * t + d) : 0u;
        }
        hits |= pivot_hits(lane, pl, kLineDiag - 1, (lb + q) * nx) ? 1u << 9 : 0u;
    }
    __syncthreads();
    const int p0 = (lb + q) * nx;
    const int steps = nx + 2 * (nsub - 1);
    for (int T = -kAhead; T < steps; ++T) {
        if (q < nsub) {
            const int xl = T - 2 * q + kAhead;
            if (xl >= 0 && xl < nx && lane < kLineRow)
                cp_async_val(&s_val[q][xl & (kRing - 1)][lane], D + (p0 + xl) * kLineRow + lane);
        }
        cp_async_commit();
        if (T < 0) continue;  // uniform over the CTA
        cp_async_wait<kAhead>();
        __syncwarp();
        const int x = T - 2 * q;
        if (q < nsub && x >= 0 && x < nx) {
            const int slot = x & (kRing - 1);
            const uint32_t m = s_mask[q][x];
            const unsigned h = (m >> lane) & 1u ? hits : 0u;
            TF a = lane < kLineRow ? s_val[q][slot][lane] : TF(0);
            TF u[kBlkPiv], rk[kBlkPiv];
#pragma unroll
            for (int t = 0; t < kBlkPiv; ++t) {
                const int ok = t < 9 ? ok0[t / 3] + t % 3 : kLineDiag - 1;
                const int ql = t < 9 ? t / 3 : q, sk = (x + (t < 9 ? t % 3 - 1 : -1)) & (kRing - 1);
                const bool on = (t == 9 || t / 3 < q) && ((m >> ok) & 1u);  // uniform
                u[t] = on && ((h >> t) & 1u) ? s_val[ql][sk][lane - ok + kLineDiag] : TF(0);
                rk[t] = on ? s_rd[ql][sk] : TF(0);
            }
#pragma unroll
            for (int t = 0; t < kBlkPiv; ++t) {
                const int ok = t < 9 ? ok0[t / 3] + t % 3 : kLineDiag - 1;
                if ((t < 9 && t / 3 >= q) || !((m >> ok) & 1u)) continue;  // uniform
                const TF lik = __shfl_sync(0xffffffffu, a, ok) * rk[t];
                if (lane == ok) a = lik;
                else a = a - lik * u[t];
            }
            if (lane < kLineRow) {
                s_val[q][slot][lane] = a;
                D[(p0 + x) * kLineRow + lane] = a;
            }
            const TF uii = __shfl_sync(0xffffffffu, a, kLineDiag);
            if (lane == 0) {
                const bool bad = !((m >> kLineDiag) & 1u) || uii == TF(0) || !isfinite(uii);
                if (bad) atomicCAS(status, 0, 1 + rows[p0 + x]);
                const TF rd = bad ? TF(0) : TF(1) / uii;
                s_rd[q][slot] = rd;
                rdiag[p0 + x] = rd;
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
__global__ void __launch_bounds__(128) lines_fill_kernel(int n, const LineGrid H, const T *__restrict__ D,
                                                         const IluLines L, T *__restrict__ offl, T *__restrict__ offu,
                                                         T *__restrict__ inl, T *__restrict__ inu) {
    __shared__ T s_row[128 * kLineRow];  // the CTA's rows; a thread's row starts at an odd multiple of the banks
    const int p0 = blockIdx.x * 128, cnt = min(128, n - p0);
    for (int t = threadIdx.x; t < cnt * kLineRow; t += 128) s_row[t] = D[p0 * kLineRow + t];
    __syncthreads();
    const int p = p0 + threadIdx.x, nx = H.nx;
    if (p >= n) return;
    int c = 0, y, z;
    while (p >= H.cl[c + 1] * nx) ++c;
    const int x = p % nx;
    line_yz(H, c, p / nx, y, z);
    const int sy = min(2, H.ny - (y & ~1)), q = (y & 1) + (z & 1) * sy;
    T off[2][kLineOff], in[2][kLineIn];
#pragma unroll
    for (int k = 0; k < kLineOff; ++k) off[0][k] = off[1][k] = T(0);
#pragma unroll
    for (int k = 0; k < kLineIn; ++k) in[0][k] = in[1][k] = T(0);
    int cnts[2] = {0, 0};
    for (int o = 0; o < kLineRow; o += 3) {  // neighbour lines ascending in z, then y
        const int dy = (o / 3) % 3 - 1, dz = o / 9 - 1;
        const int yk = y + dy, zk = z + dz;
        if (yk < 0 || yk >= H.ny || zk < 0 || zk >= H.nz) continue;
        const T *v = s_row + threadIdx.x * kLineRow + o;
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
            const int ck = ((yk >> 1) & 1) | (((zk >> 1) & 1) << 1);
            const int dir = ck < c ? 0 : 1;
            T *dst = off[dir] + 3 * cnts[dir]++;
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

// Order, block table and ILU(0) factors (in precision TF) of a scalar operator in the
// line-block order. A's pattern lies within every point's 3^dim neighbourhood
// (stencil_check): blocks of one colour are then uncoupled and a point couples to its
// line neighbours x - 1, x + 1 only.
template <typename TF>
msrsb_status lines_setup(msrsb_handle *h, cudaStream_t s) {
    const msrsb_mat &A = h->A;
    const msrsb_grid &g = h->grid;
    const int n = h->n, dim = g.dim, nx = g.nx, ny = g.ny, nz = dim == 3 ? g.nz : 1;
    IluLines &L = h->lines;
    L.nx = nx;
    L.ncol = dim == 3 ? 4 : 2;
    // ---- block table (host): blocks of each colour in block order ----
    const int nby = (ny + 1) / 2, nbz = dim == 3 ? (nz + 1) / 2 : 1;
    std::vector<int32_t> bline, bnsub;
    int run = 0;
    for (int c = 0; c < L.ncol; ++c) {
        L.cptr[c] = run;
        L.bptr[c] = (int)bline.size();
        for (int bz = 0; bz < nbz; ++bz)
            for (int by = 0; by < nby; ++by) {
                const int cc = (by & 1) | (dim == 3 ? ((bz & 1) << 1) : 0);
                if (cc != c) continue;
                const int sy = ny - 2 * by < 2 ? 1 : 2, sz = dim == 3 ? (nz - 2 * bz < 2 ? 1 : 2) : 1;
                bline.push_back(run / nx);
                bnsub.push_back(sy * sz);
                run += sy * sz * nx;
            }
    }
    L.cptr[L.ncol] = run;
    L.bptr[L.ncol] = (int)bline.size();
    if (run != n) return fail(MSRSB_ESHAPE, "line blocks cover %d of %d rows", run, n);
    const int nblk = (int)bline.size();
    MSRSB_TRY(dalloc(&L.blk_line, nblk, s));
    MSRSB_TRY(dalloc(&L.blk_nsub, nblk, s));
    MSRSB_TRY(upload(L.blk_line, bline.data(), nblk * sizeof(int32_t), s));
    MSRSB_TRY(upload(L.blk_nsub, bnsub.data(), nblk * sizeof(int32_t), s));
    LineGrid G{dim, nx, ny, nz, {0, 0, 0, 0, 0}, {0, 0}};
    for (int c = 0; c < 5; ++c) G.cl[c] = L.cptr[c < L.ncol ? c : L.ncol] / nx;
    for (int y = 0; y < ny; ++y) ++G.Ly[(y >> 1) & 1];
    MSRSB_TRY(dalloc(&L.rows, n, s));
    MSRSB_TRY(dalloc(&h->pos_of, n, s));
    uint32_t *rmask = nullptr;
    TF *D = nullptr, *rdiag = nullptr;
    int *status = nullptr;
    MSRSB_TRY(dalloc(&rmask, n, s));
    MSRSB_TRY(dalloc(&D, (size_t)n * kLineRow, s));
    MSRSB_TRY(dalloc(&rdiag, n, s));
    MSRSB_TRY(dalloc(&status, 1, s));
    MSRSB_CUDA(cudaMemsetAsync(status, 0, sizeof(int), s));
    lines_gather_kernel<TF><<<ceil_div(n, 8), 256, 0, s>>>(n, G, A.rowptr, A.colidx, A.val, L.rows, h->pos_of, rmask, D);
    MSRSB_LAUNCHED("lines_gather_kernel");
    // ---- factorisation, colour by colour ----
    for (int c = 0; c < L.ncol; ++c) {
        const int nb = L.bptr[c + 1] - L.bptr[c];
        if (!nb) continue;
        if (c > 0) {
            lines_factor_off_kernel<TF><<<(G.cl[c + 1] - G.cl[c]) * ceil_div(nx, kOffPoints), 128, 0, s>>>(G, c, rmask,
                                                                                                          D, rdiag);
            MSRSB_LAUNCHED("lines_factor_off_kernel");
        }
        lines_factor_ring_kernel<TF><<<nb, 128, 0, s>>>(G, c, L.bptr[c], L.blk_line, L.blk_nsub, L.rows, rmask, D,
                                                        rdiag, status);
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
    lines_fill_kernel<TF><<<ceil_div(n, 128), 128, 0, s>>>(n, G, D, L, offl, offu, inl, inu);
    MSRSB_LAUNCHED("lines_fill_kernel");
    int hs = 0;
    MSRSB_TRY(read_back(&hs, status, sizeof(int), s));
    dfree(rdiag, s);
    dfree(rmask, s);
    dfree(status, s);
    dfree(D, s);
    if (hs) return fail(MSRSB_EBREAKDOWN, "ILU(0): zero pivot at row %d", hs - 1);
    return MSRSB_OK;
}
template msrsb_status lines_setup<double>(msrsb_handle *, cudaStream_t);
template msrsb_status lines_setup<float>(msrsb_handle *, cudaStream_t);

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
