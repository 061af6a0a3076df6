// Arnoldi orthogonalisation of the GMRES solver (Alg. 3's outer Krylov
// method, Sec. 2.3): classical Gram-Schmidt with the reorthogonalisation
// delayed by one step (DCGS2: Swirydowicz, Langou, Ananthan, Yang and Thomas,
// Numer. Linear Algebra Appl. 28 (2021); Bielich et al., Parallel Comput. 112
// (2022)), which reads the Krylov basis twice per step instead of four times.
//
// Step j holds the orthonormal v_0 .. v_{j-1} and p, the Krylov vector of the
// previous step projected once (p = w_{j-1} - V h). It
//   1. applies the preconditioner and the operator to p itself:
//      zhat = M^-1 p, what = A zhat;
//   2. forms s = V^T p, t = V^T what, rho = p.p, sigma = p.what in one pass;
//   3. finishes v_j: alpha^2 = rho - s.s, v_j = (p - V s) / alpha, which
//      completes Hessenberg column j-1 (+= s, subdiagonal alpha);
//   4. gets w_j = A M^-1 v_j without another product: p = alpha v_j + V s, so
//      what = alpha w_j + A Z s = alpha w_j + V_j (H s) (the Arnoldi relation),
//      and V_j^T w_j follows from s, t, rho, sigma and H s alone;
//   5. writes v_j and the next p = w_j - V_j (V_j^T w_j) in a second pass.
// zhat = alpha z_j + Z s, i.e. Zhat = Z R with R upper triangular
// (R[:, j] = (s, alpha)), so the update x += Z y becomes x += Zhat R^-1 y.
// Step 0 starts from the unit v_0 (alpha = 1, no s); a cycle that ends after
// m steps finishes column m-1 with steps 2-3 alone.
#include "common.cuh"
#include "df.cuh"

namespace msrsb {

static_assert(kArnBlocks % 4 == 0, "the step's scalars sum the chunks in four fixed quarters");

// ---- pass 1: dot products ------------------------------------------------------------------

template <int W>
__device__ __forceinline__ void ld_df(const float *h, const float *l, long i, float (&vh)[W], float (&vl)[W]) {
    if constexpr (W == 4) {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(h) + i);
        const float4 b = __ldg(reinterpret_cast<const float4 *>(l) + i);
        vh[0] = a.x, vh[1] = a.y, vh[2] = a.z, vh[3] = a.w;
        vl[0] = b.x, vl[1] = b.y, vl[2] = b.z, vl[3] = b.w;
    } else {
        vh[0] = __ldg(h + i);
        vl[0] = __ldg(l + i);
    }
}

// Block (b, g): rows of chunk b and the vectors q = QB g .. QB g + QB - 1. q < nv:
// V_q . p -> partial row 2q, V_q . w -> row 2q + 1; q = nv: p . p -> row 2 nv, p . w
// -> row 2 nv + 1 (w null: the products with w are 0). Double-float planes of
// W-element groups, FP32 arithmetic with error-free transformations up to the per-warp
// sums; the two products of an element run as one packed pair, two vectors a CTA so
// that p and what are read half as often, three CTAs an SM (4, 6 or 8 vectors a CTA: 2
// to 5% more time a solve of 80^3 .. 128^3 unknowns, the registers leave too few warps).
// Right-hand sides solved together share the launches (blockIdx.z). 2^21 unknowns, 16
// vectors on average: 87 us, now 73; 8 times 80^3: 8 x 25 us, now 115.
constexpr int kDotsVecs = 2;

template <int W>
__global__ void __launch_bounds__(256, 3) dcgs2_dots_df_kernel(long NW, int nv, long ldv,
                                                                  const __grid_constant__ ArnBatch<float> B,
                                                                  long pstride, double *__restrict__ partial) {
    const ArnRhs<float> &A = B.r[blockIdx.z];
    const float *Vh = A.Vh, *Vl = A.Vl, *Ph = A.Ph, *Pl = A.Pl, *Wh = A.Wh, *Wl = A.Wl;
    partial += blockIdx.z * pstride;
    pdl_prologue();
    constexpr int QB = kDotsVecs;
    __shared__ double red[2 * QB][8];
    const int q0 = blockIdx.y * QB;
    const long chunk = (NW + gridDim.x - 1) / gridDim.x;
    const long b0 = blockIdx.x * chunk, b1 = b0 + chunk < NW ? b0 + chunk : NW;
    const float *ah[QB], *al[QB];
#pragma unroll
    for (int t = 0; t < QB; ++t) {  // beyond nv: p again, not stored
        ah[t] = q0 + t < nv ? Vh + (q0 + t) * ldv : Ph;
        al[t] = q0 + t < nv ? Vl + (q0 + t) * ldv : Pl;
    }
    const bool hw = Wh != nullptr;
    DF2 sa[QB];
#pragma unroll
    for (int t = 0; t < QB; ++t) sa[t] = DF2{0ull, 0ull};
    for (long i = b0 + threadIdx.x; i < b1; i += blockDim.x) {
        float ph[W], pl[W], wh[W], wl[W], vh[QB][W], vl[QB][W];
        ld_df<W>(Ph, Pl, i, ph, pl);
        if (hw) ld_df<W>(Wh, Wl, i, wh, wl);
#pragma unroll
        for (int t = 0; t < QB; ++t)
            if (q0 + t <= nv) ld_df<W>(ah[t], al[t], i, vh[t], vl[t]);
#pragma unroll
        for (int e = 0; e < W; ++e) {
            const float w = hw ? wh[e] : 0.f;
            const unsigned long long bh = pk2(ph[e], w), bl = pk2(pl[e], hw ? wl[e] : 0.f), nbh = pk2(-ph[e], -w);
#pragma unroll
            for (int t = 0; t < QB; ++t)
                if (q0 + t <= nv) df2_fma_acc(sa[t], pk2(vh[t][e], vh[t][e]), pk2(vl[t][e], vl[t][e]), bh, bl, nbh);
        }
    }
#pragma unroll
    for (int t = 0; t < QB; ++t) {
        if (q0 + t > nv) break;
        DF sp, sw;
        unpk2(sa[t].hi, sp.hi, sw.hi);
        unpk2(sa[t].lo, sp.lo, sw.lo);
        for (int o = 16; o > 0; o >>= 1) {
            sp = df_add(sp, df_shfl_down(sp, o));
            sw = df_add(sw, df_shfl_down(sw, o));
        }
        if ((threadIdx.x & 31) == 0) {
            red[2 * t][threadIdx.x >> 5] = (double)sp.hi + (double)sp.lo;
            red[2 * t + 1][threadIdx.x >> 5] = hw ? (double)sw.hi + (double)sw.lo : 0.0;
        }
    }
    __syncthreads();
    // eight lanes a row sum the warps' parts
    const int row = threadIdx.x >> 3, sub = threadIdx.x & 7;
    static_assert(2 * QB * 8 % 32 == 0 && 2 * QB * 8 <= 256, "whole warps");
    if (threadIdx.x < 2 * QB * 8) {
        double a = q0 + (row >> 1) <= nv ? red[row][sub] : 0.0;
        for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (sub == 0 && q0 + (row >> 1) <= nv)
            partial[(long)(2 * q0 + row) * gridDim.x + blockIdx.x] = a;
    }
}

// The same in FP64 (the FP64 form's basis), a vector a CTA: the FP64 pipe bounds it, and
// several vectors a CTA (2: 5.81 ms, 4: 6.03 ms a solve of 64^3 unknowns against 5.51)
// leave it fewer warps.
__global__ void __launch_bounds__(256) dcgs2_dots_kernel(long N, int nv, long ldv,
                                                         const __grid_constant__ ArnBatch<double> B, long pstride,
                                                         double *__restrict__ partial) {
    const double *V = B.r[blockIdx.z].Vh, *P = B.r[blockIdx.z].Ph, *Wv = B.r[blockIdx.z].Wh;
    partial += blockIdx.z * pstride;
    pdl_prologue();
    __shared__ double red[2][8];
    const int q = blockIdx.y;
    const long chunk = (N + gridDim.x - 1) / gridDim.x;
    const long b0 = blockIdx.x * chunk, b1 = b0 + chunk < N ? b0 + chunk : N;
    const double *a = q < nv ? V + q * ldv : P;
    double sp = 0.0, sw = 0.0;
#pragma unroll 4
    for (long i = b0 + threadIdx.x; i < b1; i += blockDim.x) {
        const double v = __ldg(a + i);
        sp = fma(v, __ldg(P + i), sp);
        if (Wv) sw = fma(v, __ldg(Wv + i), sw);
    }
    sp = warp_sum(sp);
    sw = warp_sum(sw);
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = sp;
        red[1][threadIdx.x >> 5] = sw;
    }
    __syncthreads();
    const int row = threadIdx.x >> 3, sub = threadIdx.x & 7;
    if (threadIdx.x < 32) {
        double x = row < 2 ? red[row][sub] : 0.0;
        for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (sub == 0 && row < 2) partial[(long)(2 * q + row) * gridDim.x + blockIdx.x] = x;
    }
}

// ---- the step's scalars (one CTA a right-hand side) ----------------------------------------------------------
//
// Sums the dot products' row-chunk partials (d = (s_0, t_0, s_1, t_1, ...,
// rho, sigma), one warp per product, fixed order) and finishes column j-1 of
// Hu (+= s, Hu[j][j-1] = alpha), copied to H for the Givens rotation; with
// `full` (what given) also R[:, j] = (s, alpha), the provisional column j of Hu
// (V_j^T w_j) and the update coefficients cv = s / alpha (for v_j),
// cp = H s / alpha + Hu[:, j] (for the next p), scal[0] = 1 / alpha.
template <typename T>
__global__ void __launch_bounds__(256) dcgs2_scalar_kernel(int m, int j, const __grid_constant__ ArnBatch<T> B,
                                                           long pstride, const double *__restrict__ partial) {
    double *__restrict__ kh = B.r[blockIdx.x].kh;
    const bool full = B.r[blockIdx.x].Wh != nullptr;
    partial += blockIdx.x * pstride;
    pdl_prologue();
    const KhLayout L(m);
    double *H = kh + L.H, *Hu = kh + L.Hu, *R = kh + L.R;
    double *cv = kh + L.cv, *cp = kh + L.cp, *sc = kh + L.scal;
    __shared__ double s_d[2 * 513], s_hs[513];
    __shared__ double s_ss, s_st;
    const int tid = threadIdx.x;
    {  // four lanes per product, each a fixed quarter of the chunks, loads issued together
        const int sub = tid & 3, nrows = 2 * (j + 1);
        for (int row0 = 0; row0 < nrows; row0 += 64) {
            const int row = row0 + (tid >> 2);
            double a = 0.0;
            if (row < nrows) {
#pragma unroll
                for (int k = 0; k < kArnBlocks / 4; ++k) a += partial[(long)row * kArnBlocks + sub + 4 * k];
            }
            a += __shfl_xor_sync(0xffffffffu, a, 1);
            a += __shfl_xor_sync(0xffffffffu, a, 2);
            if (sub == 0 && row < nrows) s_d[row] = a;
        }
    }
    __syncthreads();
    const double *s_s = s_d;  // s_q = s_d[2q], t_q = s_d[2q + 1]
    if (tid < 32) {
        double a = 0.0, b = 0.0;
        for (int q = tid; q < j; q += 32) {
            a = fma(s_d[2 * q], s_d[2 * q], a);
            b = fma(s_d[2 * q], s_d[2 * q + 1], b);
        }
        a = warp_sum(a);
        b = warp_sum(b);
        if (tid == 0) {
            s_ss = a;
            s_st = b;
        }
    }
    __syncthreads();
    const double rho = s_d[2 * j], sig = s_d[2 * j + 1];
    double alpha = 1.0;  // v_0 is a unit vector already
    if (j > 0) {
        const double a2 = rho - s_ss;
        alpha = a2 > 0.0 ? sqrt(a2) : 0.0;  // 0: breakdown, the Krylov space is invariant
        double *hu = Hu + (long)(j - 1) * (m + 1), *hc = H + (long)(j - 1) * (m + 1);
        for (int q = tid; q <= j; q += blockDim.x) {
            const double v = q < j ? hu[q] + s_s[2 * q] : alpha;
            hu[q] = v;
            hc[q] = v;
        }
    }
    if (!full) return;
    const double inva = alpha > 0.0 ? 1.0 / alpha : 0.0;
    double *rc = R + (long)j * m;
    for (int q = tid; q <= j; q += blockDim.x) rc[q] = q < j ? s_s[2 * q] : alpha;
    __syncthreads();  // column j-1 of Hu is complete
    // H s over the finished columns 0 .. j-1 (Hu[r][c] != 0 only for r <= c + 1),
    // eight independent loads in flight per thread
    for (int r = tid; r <= j; r += blockDim.x) {
        double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        int c = r > 0 ? r - 1 : 0;
        for (; c + 8 <= j; c += 8) {
#pragma unroll
            for (int u = 0; u < 8; ++u) acc[u] = fma(Hu[(long)(c + u) * (m + 1) + r], s_s[2 * (c + u)], acc[u]);
        }
        for (; c < j; ++c) acc[0] = fma(Hu[(long)c * (m + 1) + r], s_s[2 * c], acc[0]);
        s_hs[r] = ((acc[0] + acc[1]) + (acc[2] + acc[3])) + ((acc[4] + acc[5]) + (acc[6] + acc[7]));
    }
    __syncthreads();
    double *hn = Hu + (long)j * (m + 1);
    for (int q = tid; q < j; q += blockDim.x) {
        const double h = (s_d[2 * q + 1] - s_hs[q]) * inva;
        hn[q] = h;
        cp[q] = fma(s_hs[q], inva, h);
        cv[q] = s_d[2 * q] * inva;
    }
    if (tid == 0) {
        const double h = ((sig - s_st) * inva - s_hs[j]) * inva;
        hn[j] = h;
        cp[j] = fma(s_hs[j], inva, h);
        sc[0] = inva;
    }
}

// ---- pass 2: v_j and the next p -------------------------------------------------------------
//
// v_j = p / alpha - sum_q cv_q V_q (written over p) and
// p' = what / alpha - sum_q cp_q V_q - cp_j v_j (written to O), q < nv = j:
// both combinations read each V_q once and run as one packed pair. Three CTAs an SM:
// with the registers of one or two, 128^3 unknowns took 98 us a step instead of 58 (63
// as scalars); 8 times 80^3: 8 x 17 us, now 85.
template <int W>
__global__ void __launch_bounds__(256, 3) dcgs2_update_df_kernel(long NW, int nv, int m, long ldv,
                                                                    const __grid_constant__ ArnBatch<float> B) {
    const ArnRhs<float> &A = B.r[blockIdx.y];
    if (!A.Wh) return;  // this right-hand side's cycle ends here
    const float *Vh = A.Vh, *Vl = A.Vl, *Wh = A.Wh, *Wl = A.Wl;
    float *Ph = A.Ph, *Pl = A.Pl, *Oh = A.Oh, *Ol = A.Ol;
    const KhLayout L(m);
    const double *kv = A.kh + L.cv, *kp = A.kh + L.cp, *ksc = A.kh + L.scal;
    pdl_prologue();
    __shared__ ulonglong2 ch[512];  // -(cv, cp): high words and their negatives, low words
    __shared__ unsigned long long cw[512];
    __shared__ DF s_inva, s_cn;
    for (int q = threadIdx.x; q <= nv; q += blockDim.x) {
        const DF b = df_from(-kp[q]);
        if (q < nv) {
            const DF a = df_from(-kv[q]);
            ch[q] = make_ulonglong2(pk2(a.hi, b.hi), pk2(-a.hi, -b.hi));
            cw[q] = pk2(a.lo, b.lo);
        } else {
            s_cn = b;
        }
    }
    if (threadIdx.x == 0) s_inva = df_from(ksc[0]);
    __syncthreads();
    const DF ia = s_inva;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < NW; i += (long)gridDim.x * blockDim.x) {
        float ph[W], pl[W], wh[W], wl[W];
        ld_df<W>(Ph, Pl, i, ph, pl);
        ld_df<W>(Wh, Wl, i, wh, wl);
        DF2 ac[W];  // (v_j, p') of an element as one packed pair
#pragma unroll
        for (int e = 0; e < W; ++e) {
            const DF a = df_mul(DF{ph[e], pl[e]}, ia), b = df_mul(DF{wh[e], wl[e]}, ia);
            ac[e] = DF2{pk2(a.hi, b.hi), pk2(a.lo, b.lo)};
        }
#pragma unroll 2
        for (int q = 0; q < nv; ++q) {
            float vh[W], vl[W];
            ld_df<W>(Vh + q * ldv, Vl + q * ldv, i, vh, vl);
            const ulonglong2 c = ch[q];
            const unsigned long long cl = cw[q];
#pragma unroll
            for (int e = 0; e < W; ++e)
                df2_fma_acc(ac[e], pk2(vh[e], vh[e]), pk2(vl[e], vl[e]), c.x, cl, c.y);
        }
        float vh[W], vl[W], oh[W], ol[W];
#pragma unroll
        for (int e = 0; e < W; ++e) {
            DF a, b;
            unpk2(ac[e].hi, a.hi, b.hi);
            unpk2(ac[e].lo, a.lo, b.lo);
            const DF v = two_sum(a.hi, a.lo);
            df_fma_acc(b, v.hi, v.lo, s_cn.hi, s_cn.lo);
            const DF o = two_sum(b.hi, b.lo);
            vh[e] = v.hi, vl[e] = v.lo, oh[e] = o.hi, ol[e] = o.lo;
        }
        if constexpr (W == 4) {
            reinterpret_cast<float4 *>(Ph)[i] = make_float4(vh[0], vh[1], vh[2], vh[3]);
            reinterpret_cast<float4 *>(Pl)[i] = make_float4(vl[0], vl[1], vl[2], vl[3]);
            reinterpret_cast<float4 *>(Oh)[i] = make_float4(oh[0], oh[1], oh[2], oh[3]);
            reinterpret_cast<float4 *>(Ol)[i] = make_float4(ol[0], ol[1], ol[2], ol[3]);
        } else {
            Ph[i] = vh[0], Pl[i] = vl[0], Oh[i] = oh[0], Ol[i] = ol[0];
        }
    }
}

// The same in FP64; Wv and O may be the same vector (read before written,
// element by element).
__global__ void __launch_bounds__(256) dcgs2_update_kernel(long N, int nv, int m, long ldv,
                                                           const __grid_constant__ ArnBatch<double> B) {
    const ArnRhs<double> &A = B.r[blockIdx.y];
    if (!A.Wh) return;  // this right-hand side's cycle ends here
    const double *V = A.Vh, *Wv = A.Wh;
    double *P = A.Ph, *O = A.Oh;
    const KhLayout L(m);
    const double *kv = A.kh + L.cv, *kp = A.kh + L.cp, *ksc = A.kh + L.scal;
    pdl_prologue();
    __shared__ double cvs[512], cps[513];
    for (int q = threadIdx.x; q <= nv; q += blockDim.x) {
        if (q < nv) cvs[q] = kv[q];
        cps[q] = kp[q];
    }
    __syncthreads();
    const double ia = ksc[0];
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
        double av = P[i] * ia, ap = Wv[i] * ia;
#pragma unroll 4
        for (int q = 0; q < nv; ++q) {
            const double v = __ldg(V + q * ldv + i);
            av = fma(-cvs[q], v, av);
            ap = fma(-cps[q], v, ap);
        }
        P[i] = av;
        O[i] = fma(-cps[nv], av, ap);
    }
}

// ---- host side ------------------------------------------------------------------------------

static bool al16(const void *p) { return ((uintptr_t)p & 15) == 0; }

static bool al16(const ArnRhs<float> &A) {
    return al16(A.Vh) && al16(A.Vl) && al16(A.Ph) && al16(A.Pl) && al16(A.Wh) && al16(A.Wl) && al16(A.Oh) && al16(A.Ol);
}
static bool al16(int k, const ArnBatch<float> &B) {
    for (int c = 0; c < k; ++c)
        if (!al16(B.r[c])) return false;
    return true;
}

// Step j of k right-hand sides (the vectors before v_j: nv = j of N, stride N) in three
// launches: dots, scalars, update. partial: k * arn_partial(m) doubles.
msrsb_status arnoldi_step(long N, int j, int m, int k, const ArnBatch<float> &B, double *partial, cudaStream_t s) {
    if (m > 512 || j > m) return fail(MSRSB_EINVAL, "Arnoldi step %d of %d", j, m);
    const long ps = (long)arn_partial(m);
    const bool v4 = N % 4 == 0 && al16(k, B);
    const long NW = v4 ? N / 4 : N;
    const dim3 gd(kArnBlocks, ceil_div(j + 1, kDotsVecs), k);
    if (v4)
        MSRSB_PDL((dcgs2_dots_df_kernel<4>), gd, 256, 0, s, NW, j, N, B, ps, partial);
    else
        MSRSB_PDL((dcgs2_dots_df_kernel<1>), gd, 256, 0, s, NW, j, N, B, ps, partial);
    MSRSB_PDL((dcgs2_scalar_kernel<float>), k, 256, 0, s, m, j, B, ps, (const double *)partial);
    bool any = false;
    for (int c = 0; c < k; ++c) any = any || B.r[c].Wh;
    if (!any) return MSRSB_OK;
    const dim3 gu(ceil_div(NW, 256) < 2048 ? (unsigned)ceil_div(NW, 256) : 2048u, k);
    if (v4)
        MSRSB_PDL((dcgs2_update_df_kernel<4>), gu, 256, 0, s, NW, j, m, N, B);
    else
        MSRSB_PDL((dcgs2_update_df_kernel<1>), gu, 256, 0, s, NW, j, m, N, B);
    return MSRSB_OK;
}

msrsb_status arnoldi_step(long N, int j, int m, int k, const ArnBatch<double> &B, double *partial, cudaStream_t s) {
    if (m > 512 || j > m) return fail(MSRSB_EINVAL, "Arnoldi step %d of %d", j, m);
    const long ps = (long)arn_partial(m);
    MSRSB_PDL((dcgs2_dots_kernel), dim3(kArnBlocks, j + 1, k), 256, 0, s, N, j, N, B, ps,
              partial);
    MSRSB_PDL((dcgs2_scalar_kernel<double>), k, 256, 0, s, m, j, B, ps, (const double *)partial);
    bool any = false;
    for (int c = 0; c < k; ++c) any = any || B.r[c].Wh;
    if (!any) return MSRSB_OK;
    const unsigned g = ceil_div(N, 256) < 2048 ? (unsigned)ceil_div(N, 256) : 2048u;
    MSRSB_PDL((dcgs2_update_kernel), dim3(g, k), 256, 0, s, N, j, m, N, B);
    return MSRSB_OK;
}

}  // namespace msrsb
