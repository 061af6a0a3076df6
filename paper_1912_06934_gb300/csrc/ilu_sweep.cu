// Application z += U^-1 L^-1 r of the line-block ILU(0) smoother (ilu_lines.cu
// holds the order, the factorisation and the coefficients' layout).
//
// One launch per colour and direction, one CTA per line block. A launch is a
// short chain of dependent steps: one gather of the other blocks' values, then
// the block's lines in turn, each a first-order recurrence along x. It is bound
// by that chain on small grids, by instruction issue and the coefficients'
// bytes on large ones. What follows from it:
//  - the coefficients do not depend on the previous kernel: every lane copies
//    those of its own points to shared memory asynchronously before
//    griddepcontrol.wait (no registers held, no column indices to load, see
//    lines.cuh), and the recurrence's coefficients are composed there too, so
//    that only the values' half of the scan is left for after the wait;
//  - z is read with the gather and added to at the end, so that no line waits
//    for global memory;
//  - only the warps of a line run its scan, and only they meet inside it.
// FP32: one warp a line, a lane holding the points lane + 32 s; the segments of
// 32 are scanned side by side, with no barrier inside a line. FP64: a warp's
// FMA occupies its scheduler's FP64 unit for some 60 cycles, so the segments
// lie in warps of their own (up to 4 a line, on as many schedulers), and the
// lines still to come take each finished line's contributions at once instead
// of all of them at their turn.
// Measured against one thread per point with column indices beside the values
// and every warp of the CTA in every scan, the rest of the solve as it was then
// (whole calls): solves of 64^3 in FP64 10.6 -> 6.9 ms, of 128^3 in FP32 33.3 ->
// 27.2, 8 lockstep right-hand sides of 80^3 in FP32 46.2 -> 36.3. A launch inside a
// solve now takes 4.9 us at 64^3 (FP32), 8.2
// (FP64), 19.4 at 128^3 (FP32; 36 MB of coefficients, 5.4 us at the copy rate).
#include "common.cuh"
#include "lines.cuh"
#include <atomic>
#include <cstring>
#include <type_traits>

namespace msrsb {

template <typename T>
using LineVec = typename std::conditional<sizeof(T) == 4, float4, double2>::type;

// groups 0 .. ng-1 of a record (`stride` vectors apart) into registers, zeros after
template <typename T, int N>
__device__ __forceinline__ void line_load(T (&v)[N], int ng, const LineVec<T> *p, int stride) {
    constexpr int G = kLineGroup<T>;
#pragma unroll
    for (int g = 0; g < N / G; ++g) {
        LineVec<T> t;
        memset(&t, 0, sizeof(t));
        if (g < ng) t = p[g * stride];
        memcpy(v + g * G, &t, 16);
    }
}

// The recurrence v_k = a_k + b_k v_{k-1}, v_-1 = 0, along a line, by WPL warps
// of S segments of 32 points. `prepare` composes the coefficients alone (the
// steps of an affine scan whose maps are kept before each step), `solve` runs
// the values of NV vectors through them: every segment's scan, then the
// carries, segment by segment and warp by warp.
template <typename T, int S, int WPL>
struct LineScan {
    T st[5][S], b[S];
    // wB: the warps' composed coefficients, read after the CTA's first barrier
    __device__ __forceinline__ void prepare(const T (&bb)[S], int lane, T *wB) {
#pragma unroll
        for (int s = 0; s < S; ++s) b[s] = bb[s];
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int s = 0; s < S; ++s) {
                st[i][s] = b[s];
                const T bp = __shfl_up_sync(0xffffffffu, b[s], 1 << i);
                if (lane >= 1 << i) b[s] = b[s] * bp;
            }
        if constexpr (WPL > 1) {
            if (lane == 31) {
                T t = b[0];
#pragma unroll
                for (int s = 1; s < S; ++s) t = t * b[s];
                wB[threadIdx.x >> 5] = t;
            }
        }
    }
    // wl: this warp's place in its line; wA [NV][32]: the warps' composed values
    template <int NV>
    __device__ __forceinline__ void solve(T (&a)[NV][S], int lane, int wl, T *wA, const T *wB) const {
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int c = 0; c < NV; ++c) {
                    const T ap = __shfl_up_sync(0xffffffffu, a[c][s], 1 << i);
                    if (lane >= 1 << i) a[c][s] = fma(st[i][s], ap, a[c][s]);
                }
        if constexpr (S * WPL > 1) {
            T carry[NV], al[NV][S], bl[S];
#pragma unroll
            for (int s = 0; s < S; ++s) {
                bl[s] = __shfl_sync(0xffffffffu, b[s], 31);
#pragma unroll
                for (int c = 0; c < NV; ++c) al[c][s] = __shfl_sync(0xffffffffu, a[c][s], 31);
            }
#pragma unroll
            for (int c = 0; c < NV; ++c) carry[c] = T(0);
            if constexpr (WPL > 1) {
                const int w = threadIdx.x >> 5;
#pragma unroll
                for (int c = 0; c < NV; ++c) {
                    T t = al[c][0];
#pragma unroll
                    for (int s = 1; s < S; ++s) t = fma(bl[s], t, al[c][s]);
                    if (lane == 0) wA[c * 32 + w] = t;
                }
                asm volatile("bar.sync 1, %0;" ::"n"(32 * WPL) : "memory");  // one line at a time
                for (int u = w - wl; u < w; ++u) {
                    const T bu = wB[u];
#pragma unroll
                    for (int c = 0; c < NV; ++c) carry[c] = fma(bu, carry[c], wA[c * 32 + u]);
                }
            }
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int c = 0; c < NV; ++c) {
                    if (s > 0 || WPL > 1) a[c][s] = fma(b[s], carry[c], a[c][s]);
                    carry[c] = fma(bl[s], carry[c], al[c][s]);
                }
        }
    }
};

// One colour's part of the factors (see IluLines) and its blocks.
template <typename T>
struct LinesColour {
    int b0, l0;           // first block, first line
    int noff[2], ng[2];   // neighbour lines of earlier / later colours, groups of their coefficients
    int room;             // groups per point reserved in shared memory for the off-block part
    int stage;            // the off-block part goes through shared memory
    const T *off[2];
};

// groups of the in-block record of line q of nsub
template <typename T>
__host__ __device__ __forceinline__ int in_groups(int dir, int q, int nsub) {
    return line_groups<T>(dir ? 2 + 3 * (nsub - 1 - q) : 1 + 3 * q);
}

// mode 0: forward over the block's lines; 1: backward; 2: forward then
// backward (the last colour, which has no later one). CTA (b, g): block b,
// vectors g NV .. of k (several right-hand sides: every coefficient serves NV
// vectors and their scans interleave). Shared memory: the off-block
// coefficients [lines][room][nx], the in-block ones packed by line, the
// block's values [NV][lines][nx + 2] with a zero beyond each end of a line.
template <typename T, typename TZ, int S, int WPL, int NV>
__global__ void __launch_bounds__(128 * WPL, 1) lines_sweep_kernel(
    int mode, int k, int nx, int nlines, const int32_t *__restrict__ blk_line, const int32_t *__restrict__ blk_nsub,
    const __grid_constant__ LinesColour<T> C, const int32_t *__restrict__ nbr, const T *__restrict__ inl,
    const T *__restrict__ inu, const int32_t *__restrict__ rows, const __grid_constant__ Cols<T> ys,
    const __grid_constant__ Cols<TZ> zs) {
    using V = LineVec<T>;
    extern __shared__ __align__(16) unsigned char s_raw[];
    constexpr int NI = line_groups<T>(kLineIn), G = kLineGroup<T>;
    constexpr bool eager = sizeof(T) == 8;
    const int wl = (threadIdx.x >> 5) % WPL;  // this warp's place in its line
    const int q = (threadIdx.x >> 5) / WPL, lane = threadIdx.x & 31, nlin = blockDim.x / (32 * WPL);
    const int x0 = lane + 32 * S * wl;  // the lane's points are x0 + 32 s in processing order
    const int nxs = nx + 2, dir = mode == 1;
    const int b = C.b0 + blockIdx.x, v0 = blockIdx.y * NV;
    const int nsub = __ldg(blk_nsub + b), line = __ldg(blk_line + b) + (q < nsub ? q : 0);
    const int st = line * nx, noff = C.noff[dir], ng = C.ng[dir];
    int ib = 0, itot = 0;  // this line's place among the packed in-block records
    for (int t = 0; t < nlin; ++t) {
        const int g = in_groups<T>(dir, t, nlin);  // blocks of fewer lines need no more
        if (t < q) ib += g;
        itot += g;
    }
    V *s_off = reinterpret_cast<V *>(s_raw) + (long)q * C.room * nx;
    V *s_in = reinterpret_cast<V *>(s_raw) + (long)(nlin * C.room + ib) * nx;
    T *sm = reinterpret_cast<T *>(reinterpret_cast<V *>(s_raw) + (long)(nlin * C.room + itot) * nx) + 1;
    T *wA = sm - 1 + NV * nlin * nxs, *wB = wA + NV * 32;  // composed maps of the warps (WPL > 1; wB [2 sweeps][32])
    const bool live = q < nsub;  // whole warps
    const int nin = in_groups<T>(dir, q, nsub), nbk = in_groups<T>(1, q, nsub);
    const V *goff = reinterpret_cast<const V *>(C.off[dir]) + (long)(line - C.l0) * ng * nx;
    const V *gin = reinterpret_cast<const V *>(dir ? inu : inl) + (long)line * NI * nx;
    const V *ginu = reinterpret_cast<const V *>(inu) + (long)line * NI * nx;
    int nb[kLineNbr], row[S];
    LineScan<T, S, WPL> scan;
    // the recurrence's coefficients, from the staged records of direction d
    auto scan_prepare = [&](int d) {
        T bb[S];
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int xx = x0 + 32 * s, x = d ? nx - 1 - xx : xx;
            bb[s] = T(1);
            if (xx < nx) {
                const T *r = reinterpret_cast<const T *>(s_in + x);
                bb[s] = d ? -r[1] * r[0] : -r[0];
            }
        }
        scan.prepare(bb, lane, wB + 32 * d);
    };
    if (live) {
        if (C.stage)
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const int xx = x0 + 32 * s, x = mode == 1 ? nx - 1 - xx : xx;
                if (xx < nx)
                    for (int g = 0; g < ng; ++g) cp_async16(s_off + g * nx + x, goff + g * nx + x);
            }
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int xx = x0 + 32 * s, x = mode == 1 ? nx - 1 - xx : xx;
            if (xx < nx)
                for (int g = 0; g < nin; ++g) cp_async16(s_in + g * nx + x, gin + g * nx + x);
        }
        cp_async_commit();
#pragma unroll
        for (int l = 0; l < kLineNbr; ++l)
            nb[l] = l < noff ? __ldg(nbr + ((long)dir * nlines + line) * kLineNbr + l) : 0;
        if (mode != 0)
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const int x = nx - 1 - x0 - 32 * s;
                row[s] = x >= 0 ? __ldg(rows + st + x) : 0;
            }
        if (lane < 2 * NV && wl == 0) sm[((lane >> 1) * nlin + q) * nxs + (lane & 1 ? nx : -1)] = T(0);
        cp_async_wait<0>();
        scan_prepare(dir);
    }
    pdl_prologue();
    T a[NV][S];
    TZ zv[NV][S];
    if (live) {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int xx = x0 + 32 * s;
            if (xx >= nx) continue;
            const int x = mode == 1 ? nx - 1 - xx : xx;
            const int xm = max(x - 1, 0), xp = min(x + 1, nx - 1);
            T g[NV][3 * kLineNbr], own[NV], off[kLineOff];
#pragma unroll
            for (int c = 0; c < NV; ++c) {
                const int v = NV == 1 || v0 + c < k ? v0 + c : v0;
                const T *y = ys.p[v];
#pragma unroll
                for (int l = 0; l < kLineNbr; ++l)
                    if (l < noff) {
                        const T *yl = y + nb[l];
                        g[c][3 * l] = yl[xm];
                        g[c][3 * l + 1] = yl[x];
                        g[c][3 * l + 2] = yl[xp];
                    }
                own[c] = y[st + x];
                if (mode != 0) zv[c][s] = zs.p[v][row[s]];
            }
            if (C.stage) line_load<T>(off, ng, s_off + x, nx);
            else line_load<T>(off, ng, goff + x, nx);
#pragma unroll
            for (int c = 0; c < NV; ++c) {
                T acc = T(0);
#pragma unroll
                for (int l = 0; l < kLineNbr; ++l)
                    if (l < noff) {
#pragma unroll
                        for (int d = 0; d < 3; ++d) acc = fma(off[3 * l + d], g[c][3 * l + d], acc);
                    }
                a[c][s] = own[c] - acc;
            }
        }
    }
    // the warps' composed coefficients are there, every off-block part has been read
    if (WPL > 1) __syncthreads();
    else __syncwarp();
    if (mode == 2 && live) {  // the backward record takes the place of the off-block one
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int x = nx - 1 - x0 - 32 * s;  // the point this lane takes backwards
            if (x >= 0)
                for (int g = 0; g < nbk; ++g) cp_async16(s_off + g * nx + x, ginu + g * nx + x);
        }
        cp_async_commit();
    }
    // own value of every slot into a (the values of the direction's points)
    auto own_values = [&](int d) {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int xx = x0 + 32 * s, x = d ? nx - 1 - xx : xx;
            if (xx < nx)
#pragma unroll
                for (int c = 0; c < NV; ++c) a[c][s] = sm[(c * nlin + q) * nxs + x];
        }
    };
    // a -= the contributions of the block's line l, entry `first` of the record on
    auto take_line = [&](int d, int l, int first) {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int xx = x0 + 32 * s, x = d ? nx - 1 - xx : xx;
            if (xx < nx)
#pragma unroll
                for (int e = 0; e < 3; ++e) {
                    const int i = first + e;
                    const T cf = reinterpret_cast<const T *>(s_in + (i / G) * nx + x)[i % G];
#pragma unroll
                    for (int c = 0; c < NV; ++c) a[c][s] = fma(-cf, sm[(c * nlin + l) * nxs + x + e - 1], a[c][s]);
                }
        }
    };
    // solve this warp's line from a and publish it
    auto finish_line = [&](int d) {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int xx = x0 + 32 * s, x = d ? nx - 1 - xx : xx;
            if (xx < nx) {
                if (d) {
                    const T di = reinterpret_cast<const T *>(s_in + x)[1];
#pragma unroll
                    for (int c = 0; c < NV; ++c) a[c][s] = di * a[c][s];
                }
            } else {
#pragma unroll
                for (int c = 0; c < NV; ++c) a[c][s] = T(0);
            }
        }
        scan.solve(a, lane, wl, wA, wB + 32 * d);
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int xx = x0 + 32 * s, x = d ? nx - 1 - xx : xx;
            if (xx < nx)
#pragma unroll
                for (int c = 0; c < NV; ++c) {
                    sm[(c * nlin + q) * nxs + x] = a[c][s];
                    if (NV == 1 || v0 + c < k) {
                        if (d || mode == 0) ys.p[v0 + c][st + x] = a[c][s];
                        if (d) {
                            TZ *zp = zs.p[v0 + c] + row[s];
                            *zp = TZ(zv[c][s] + to_prec<TZ>(a[c][s]));
                        }
                    }
                }
        }
    };
    if (mode != 1) {
        for (int qq = 0; qq < nsub; ++qq) {
            if (q == qq) {  // whole warps
                if (!eager)
                    for (int l = 0; l < q; ++l) take_line(0, l, 1 + 3 * l);
                finish_line(0);
                if (mode == 2) {  // the backward coefficients while the later lines are at work
                    cp_async_wait<0>();
                    s_in = s_off;
                    scan_prepare(1);
                }
            }
            if (mode == 2 || qq + 1 < nsub) __syncthreads();
            if (eager && q > qq && live) take_line(0, qq, 1 + 3 * qq);
        }
        if (mode == 0) return;
        if (live) own_values(1);
    }
    for (int qq = nsub - 1; qq >= 0; --qq) {
        // the lines from the last, each from its end: e_x = udinv_x ((t_x - sum_in U e) - urec_x e_{x+1})
        if (q == qq) {
            if (!eager)
                for (int l = q + 1; l < nsub; ++l) take_line(1, l, 2 + 3 * (l - q - 1));
            finish_line(1);
        }
        if (qq > 0) __syncthreads();
        if (eager && q < qq) take_line(1, qq, 2 + 3 * (qq - q - 1));
    }
}

// ---- host side ---------------------------------------------------------------------------------

constexpr size_t kSweepSmemMax = 220 * 1024;
constexpr int kSweepStageCtas = 304;  // two per SM

// z_c += U^-1 L^-1 r_c for c < k, r_c given in the line-block order in ry_c
// (overwritten): 2 C - 1 launches for C colours
template <typename T, typename TZ, int S, int WPL, int NV>
static msrsb_status lines_sweeps(const msrsb_handle *h, int k, const Cols<T> &ry, const Cols<TZ> &z, cudaStream_t s) {
    const IluLines &L = h->lines;
    const int last = L.ncol - 1, nlin = L.ncol == 4 ? 4 : 2;
    {  // more than 48 KB of shared memory has to be asked for, once per device
        static std::atomic<unsigned long long> asked{0};
        int dev = 0;
        MSRSB_CUDA(cudaGetDevice(&dev));
        const unsigned long long bit = 1ull << (dev & 63);
        if (!(asked.load(std::memory_order_relaxed) & bit)) {
            MSRSB_CUDA(cudaFuncSetAttribute(lines_sweep_kernel<T, TZ, S, WPL, NV>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSweepSmemMax));
            asked.fetch_or(bit, std::memory_order_relaxed);
        }
    }
    auto launch = [&](int mode, int c) -> msrsb_status {
        const int nb = L.bptr[c + 1] - L.bptr[c];
        if (!nb) return MSRSB_OK;
        LinesColour<T> C;
        C.b0 = L.bptr[c];
        C.l0 = L.cptr[c] / L.nx;
        for (int d = 0; d < 2; ++d) {
            C.noff[d] = L.noff[d][c];
            C.ng[d] = line_groups<T>(3 * L.noff[d][c]);
            C.off[d] = (const T *)L.off[d] + L.obase[d][c];
        }
        const int dir = mode == 1, back = mode == 2 ? in_groups<T>(1, 0, nlin) : 0;
        int gin = 0;
        for (int t = 0; t < nlin; ++t) gin += in_groups<T>(dir, t, nlin);
        const size_t vals = ((size_t)NV * nlin * (L.nx + 2) + (WPL > 1 ? (NV + 2) * 32 : 0)) * sizeof(T);
        // Up to two CTAs per SM the off-block part is staged ahead of the
        // wait. Beyond, a launch has several waves, only the first of which
        // gains by that, and the shared memory costs CTAs in flight: read
        // where it is used (128^3 FP32 solve, whole call: 24.5 ms with it staged,
        // 22.5 without; 64^3 FP32, one wave: 1 % less with it). So it is on FP64
        // lines too wide for the shared memory.
        C.stage = nb * ceil_div(k, NV) <= kSweepStageCtas && (size_t)(nlin * (C.ng[dir] > back ? C.ng[dir] : back) + gin) * L.nx * 16 + vals <= kSweepSmemMax;
        C.room = C.stage && C.ng[dir] > back ? C.ng[dir] : back;
        const size_t smem = (size_t)(nlin * C.room + gin) * L.nx * 16 + vals;
        MSRSB_PDL((lines_sweep_kernel<T, TZ, S, WPL, NV>), dim3(nb, ceil_div(k, NV)), 32 * WPL * nlin, smem, s, mode, k, L.nx,
                  h->n / L.nx, L.blk_line, L.blk_nsub, C, L.nbr, (const T *)L.in[0], (const T *)L.in[1], L.rows, ry, z);
        return MSRSB_OK;
    };
    for (int c = 0; c < last; ++c) MSRSB_TRY(launch(0, c));
    MSRSB_TRY(launch(2, last));
    for (int c = last - 1; c >= 0; --c) MSRSB_TRY(launch(1, c));
    return MSRSB_OK;
}

template <typename T, typename TZ, int NV>
static msrsb_status lines_sweeps_nv(const msrsb_handle *h, int k, const Cols<T> &ry, const Cols<TZ> &z,
                                    cudaStream_t s) {
    const int seg = ceil_div(h->lines.nx, 32);  // nx <= 256
    if constexpr (sizeof(T) == 8) {
        if (seg <= 1) return lines_sweeps<T, TZ, 1, 1, NV>(h, k, ry, z, s);
        if (seg <= 2) return lines_sweeps<T, TZ, 1, 2, NV>(h, k, ry, z, s);
        if (seg <= 3) return lines_sweeps<T, TZ, 1, 3, NV>(h, k, ry, z, s);
        if (seg <= 4) return lines_sweeps<T, TZ, 1, 4, NV>(h, k, ry, z, s);
        if constexpr (NV == 1) return lines_sweeps<T, TZ, 2, 4, NV>(h, k, ry, z, s);
    } else {
        if (seg <= 1) return lines_sweeps<T, TZ, 1, 1, NV>(h, k, ry, z, s);
        if (seg <= 2) return lines_sweeps<T, TZ, 2, 1, NV>(h, k, ry, z, s);
        if (seg <= 3) return lines_sweeps<T, TZ, 3, 1, NV>(h, k, ry, z, s);
        if (seg <= 4) return lines_sweeps<T, TZ, 4, 1, NV>(h, k, ry, z, s);
        if constexpr (NV == 1) {
            if (seg <= 6) return lines_sweeps<T, TZ, 6, 1, NV>(h, k, ry, z, s);
            return lines_sweeps<T, TZ, 8, 1, NV>(h, k, ry, z, s);
        }
    }
    return fail(MSRSB_EINVAL, "line sweeps take lines of at most %d points", NV == 1 ? 256 : 128);
}

template <typename T, typename TZ>
msrsb_status lines_apply(const msrsb_handle *h, T *ry, TZ *z, cudaStream_t s) {
    Cols<T> r{};
    Cols<TZ> zc{};
    r.p[0] = ry;
    zc.p[0] = z;
    return lines_sweeps_nv<T, TZ, 1>(h, 1, r, zc, s);
}
template msrsb_status lines_apply<double, double>(const msrsb_handle *, double *, double *, cudaStream_t);
template msrsb_status lines_apply<float, double>(const msrsb_handle *, float *, double *, cudaStream_t);
template msrsb_status lines_apply<float, float>(const msrsb_handle *, float *, float *, cudaStream_t);

// The lockstep solves serve lines of up to 128 points in 3D, 256 in 2D.
bool lines_multi_fit(const msrsb_handle *h) {
    const IluLines &L = h->lines;
    return L.nx <= (L.ncol == 4 ? 128 : 256);
}

// lines_apply for k right-hand sides
template <typename T, typename TZ>
msrsb_status lines_apply_multi(const msrsb_handle *h, int k, Cols<T> ry, Cols<TZ> z, cudaStream_t s) {
    if (!lines_multi_fit(h) || k < 1 || k > kMaxRhs) return fail(MSRSB_EINVAL, "multi-vector sweep shape");
    if (k == 1 || h->lines.nx > 128) return lines_sweeps_nv<T, TZ, 1>(h, k, ry, z, s);
    return lines_sweeps_nv<T, TZ, 2>(h, k, ry, z, s);
}
template msrsb_status lines_apply_multi<double, double>(const msrsb_handle *, int, Cols<double>, Cols<double>,
                                                        cudaStream_t);
template msrsb_status lines_apply_multi<float, double>(const msrsb_handle *, int, Cols<float>, Cols<double>,
                                                       cudaStream_t);

}  // namespace msrsb
