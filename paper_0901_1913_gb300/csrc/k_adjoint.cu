// k_adjoint.cu -- exact gradients and Newton refinement at peaks.
//
// Sec. 3e: near the best and the nearly-as-good frequencies the search should
// be refined "using the ungridded data".  For each requested peak (curve c,
// bin j) one CTA works straight from the samples, in double:
//   * chi^2(A, f) = sum_i w_i (x'_i - sum_l A_l M_l(f, tau_i))^2 (Sec. 2, Eq.
//     "eqchigen" with the Eq. "eqtrunc" basis, x' = x - xbar), minimised over A
//     by the normal equations (Eq. "eqchix");
//   * gradients of Delta = chi2_0 - chi2_min at the bin frequency by the
//     envelope theorem (the minimisers xbar and A need not be differentiated):
//       dDelta/dx_i     = 2 w_i (m_i - xbar)
//       dDelta/dsigma_i = -2 sigma_i^-3 [(x_i - xbar)^2 - (x_i - m_i)^2]
//       dDelta/df       = 2 sum_i w_i r_i m_f,i,  r = x' - m', m_f = d m'/df;
//   * Newton steps on f with the exact second derivative of chi2_min(f),
//       d2 chi2_min/df2 = 2 sum w (m_f^2 - r m_ff) - 2 V^T alpha^-1 V,
//       V_l = sum w (M_l m_f - r dM_l/df)  (Schur complement of the joint
//     Hessian in (A, f)), safeguarded to stay within one bin of the start and
//     to increase Delta.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "fc2_common.cuh"
#include "fc2_df.cuh"
#include "fc2_internal.h"
#include "fc2_solve.cuh"

namespace fc2 {

// Bound by the double pipe: a warp's double instruction holds its SM
// sub-partition for 64 clocks however many lanes work, so the sample passes
// count double operations (per sample and Newton step about 73 for the sums
// and 95 for the derivatives at H = 4) and nothing runs on one lane:
//   * phasors from the exact fixed-point phase through two 256-entry tables
//     and a short Taylor series (d_phasor; 13 operations where sincospi takes
//     about 35);
//   * the block sums exchange halves of the value list at each butterfly step
//     (about one addition per value where a butterfly per value takes five);
//   * one factorisation L D L^T per trial frequency, by a warp in shared
//     memory with the trailing elements spread over the lanes, serves Delta, the
//     coefficients and the second derivative (two single-lane solves of the
//     padded 17-square system took longer than the sums);
//   * the derivative pass reads back the phasors of the first 2048 samples
//     from shared memory (45 KB a CTA, three CTAs an SM);
//   * 128 threads per entry and one CTA per entry: while one entry's warp
//     solves, the SM's other entries keep the pipe busy.
// 1024 entries of n = 2000, H = 4: 7436 -> 2515 us (2962 us without the kept
// phasors), near the double pipe's time for about five Newton steps; eight
// entries of n = 400, H = 3: about 700 -> 162 us.
constexpr int AD_NT = 128;
constexpr int AD_NW = AD_NT / 32;
constexpr int AD_HM = 8;
constexpr int AD_NQ = 6 * AD_HM;       // most values of one block sum
constexpr int AD_M = 2 * AD_HM + 1;
constexpr int AD_ZC = 2048;            // samples whose phasors are kept from pass A to pass B

struct AdjShared {
    double2 tab[512];                  // phasor tables (d_phasor)
    double2 z[AD_ZC];                  // phasors of the first samples (each read back by its writer)
    double red[AD_NW][AD_NQ];
    double tot[AD_NQ];
    // lower triangle: the Schur complements u; above the diagonal, mat[k][l] =
    // L[l][k]; column m: the right-hand side y = L^-1 beta
    double mat[AD_M][AD_M + 1];
    double diag[AD_M];                 // alpha'_ll
    double rd[AD_M];                   // 1 / d_k, 0 for a dropped column
    double coef[AD_M];                 // coefficients (tau frame, absolute units)
    double f, fbest, dbest, step;
    int state;                         // 0 continue, 1 backtracked, 2 done
};

// Warp sums of NV values: at each of the five butterfly steps a lane keeps one
// half of its list and adds the partner's copy of it.  Lane results go to
// row[index].
template <int NV>
FC2_D void warp_scatter_sum(double* v, double* row) {
    const int lane = threadIdx.x & 31;
    int base = 0, len = NV;
    auto step = [&](auto n_tag, int o) {
        constexpr int n = decltype(n_tag)::value;
        constexpr int h = (n + 1) / 2;
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double hi = (h + i < n) ? v[h + i] : 0.0;
            const double send = up ? v[i] : hi;
            const double keep = up ? hi : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        base += up ? h : 0;
        len = up ? len - h : (len < h ? len : h);
    };
    constexpr int n1 = (NV + 1) / 2, n2 = (n1 + 1) / 2, n3 = (n2 + 1) / 2, n4 = (n3 + 1) / 2;
    constexpr int n5 = (n4 + 1) / 2;
    step(std::integral_constant<int, NV>{}, 16);
    step(std::integral_constant<int, n1>{}, 8);
    step(std::integral_constant<int, n2>{}, 4);
    step(std::integral_constant<int, n3>{}, 2);
    step(std::integral_constant<int, n4>{}, 1);
#pragma unroll
    for (int i = 0; i < n5; ++i)
        if (i < len) row[base + i] = v[i];
}

// Block sums of NV values into sh.tot, valid on all threads after the call.
template <int NV>
FC2_D void block_sum(double* v, AdjShared& sh) {
    static_assert(NV <= AD_NQ, "reduction buffer too small");
    warp_scatter_sum<NV>(v, sh.red[threadIdx.x >> 5]);
    __syncthreads();
    if (threadIdx.x < NV) {
        double y = sh.red[0][threadIdx.x];
#pragma unroll
        for (int q = 1; q < AD_NW; ++q) y += sh.red[q][threadIdx.x];
        sh.tot[threadIdx.x] = y;
    }
    __syncthreads();
}

FC2_D double warp_total(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Factor the normalised system of the sums in sh.tot (Q_1..Q_2H, P_1..P_H as
// re, im pairs) by one warp; returns Delta' = sum_{l >= 1} y_l^2 / d_l.  A
// column whose relative pivot is at most 1e-13 is dropped.
template <int H>
FC2_D double adj_factor(AdjShared& sh, double iw, double sp, double s1) {
    constexpr int m = 2 * H + 1, W = m + 1;
    const int lane = threadIdx.x & 31;
    for (int q = lane; q < 6 * H; q += 32) sh.tot[q] *= (q < 4 * H) ? iw : sp;
    __syncwarp();
    auto qr = [&](int k) { return k == 0 ? 1.0 : sh.tot[2 * k - 2]; };
    auto qi = [&](int k) { return k == 0 ? 0.0 : sh.tot[2 * k - 1]; };
    for (int idx = lane; idx < m * W; idx += 32) {
        const int l = idx / W, k = idx - l * W;
        if (k > l && k < m) continue;
        const int hl = (l + 1) >> 1, hk = (k + 1) >> 1;
        double v;
        if (k == m) {  // beta_l
            v = l == 0 ? s1 * sp : sh.tot[4 * H + 2 * hl - ((l & 1) ? 1 : 2)];
        } else if (k == 0) {
            v = l == 0 ? 1.0 : ((l & 1) ? qi(hl) : qr(hl));
        } else {
            const int d = hl - hk, s = hl + hk;
            if (((l ^ k) & 1) == 0) v = 0.5 * (qr(d) + ((l & 1) ? -qr(s) : qr(s)));
            else v = 0.5 * (qi(s) + ((l & 1) ? qi(d) : -qi(d)));  // sin cos, cos sin
        }
        sh.mat[l][k] = v;
        if (k == l) sh.diag[l] = v;
    }
    __syncwarp();
#pragma unroll 1
    for (int k = 0; k < m; ++k) {
        const double d = sh.mat[k][k], all = sh.diag[k];
        const double r = (all > 0.0 && d > 1e-13 * all) ? 1.0 / d : 0.0;
        const int l = k + 1 + lane;
        if (l < m) sh.mat[k][l] = sh.mat[l][k] * r;
        if (lane == 0) sh.rd[k] = r;
        __syncwarp();
        for (int idx = lane; idx < (m - 1 - k) * W; idx += 32) {
            const int row = k + 1 + idx / W, j = idx % W;
            if (j == m || (j > k && j <= row))
                sh.mat[row][j] = fma(-sh.mat[k][row], j == m ? sh.mat[k][m] : sh.mat[j][k],
                                     sh.mat[row][j]);
        }
        __syncwarp();
    }
    const double y = lane < m ? sh.mat[lane][m] : 0.0;
    return warp_total(lane > 0 && lane < m ? y * y * sh.rd[lane] : 0.0);
}

// Coefficients of the factored system (times unit) into sh.coef: L^T A = D^-1 y.
template <int H>
FC2_D void adj_coef(AdjShared& sh, double unit) {
    constexpr int m = 2 * H + 1;
    const int lane = threadIdx.x & 31;
    double a = lane < m ? sh.mat[lane][m] * sh.rd[lane] : 0.0;
#pragma unroll 1
    for (int k = m - 1; k > 0; --k) {
        const double ak = __shfl_sync(0xffffffffu, a, k);
        if (lane < k) a = fma(-sh.mat[lane][k], ak, a);
    }
    if (lane < m) sh.coef[lane] = a * unit;
}

// V^T alpha'^-1 V of the factored system, lane l holding V_l.
template <int H>
FC2_D double adj_quad(const AdjShared& sh, double v) {
    constexpr int m = 2 * H + 1;
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int k = 0; k + 1 < m; ++k) {
        const double vk = __shfl_sync(0xffffffffu, v, k);
        if (lane > k && lane < m) v = fma(-sh.mat[k][lane], vk, v);
    }
    return warp_total(lane < m ? v * v * sh.rd[lane] : 0.0);
}

template <int H>
FC2_D void backward_entry(const AdjTab& tb, int64_t e, const AdjOut& out, AdjShared& sh) {
    constexpr int m = 2 * H + 1;
    constexpr int NB = 2 + m;  // S1, S2, V_0..V_2H
    const int c = (int)(tb.ent[e] >> 32);
    const int64_t j = tb.ent[e] & 0xffffffffll;
    const double* sc = tb.scal + (int64_t)c * SC_COUNT;
    const double W = sc[SC_W], chi0 = sc[SC_CHI0];
    const double iw = 1.0 / W, sp = (chi0 > 0.0) ? rsqrt(W * chi0) : 0.0;
    const int64_t a0 = tb.off[c], a1 = tb.off[c + 1], n = a1 - a0;
    const double g_up = tb.gout ? tb.gout[e] : 1.0;
    const double df = tb.df[c];
    const double f0 = tb.fmin[c] + (double)j * df;
    const double lo = f0 - df, hi = f0 + df;
    const int r_in = (int)(e % (tb.K > 0 ? tb.K : 1));
    const double2* t1 = sh.tab;
    const double2* t2 = sh.tab + 256;
    if (threadIdx.x == 0) { sh.f = f0; sh.fbest = f0; sh.dbest = -INFINITY; sh.step = 0.0; sh.state = 0; }
    __syncthreads();
#pragma unroll 1
    for (int it = 0; it <= tb.max_iter; ++it) {
        const double f = sh.f;
        // ---- pass A: trigonometric sums at f (Eq. "eqPQ") and the solve
        {
            double acc[6 * H];
#pragma unroll
            for (int q = 0; q < 6 * H; ++q) acc[q] = 0.0;
#pragma unroll 1
            for (int64_t i = a0 + threadIdx.x; i < a1; i += AD_NT) {
                const double2 z1 = d_phasor(frac_fx(f, tb.tau[i]), t1, t2);
                if (i - a0 < AD_ZC) sh.z[i - a0] = z1;
                const double a = tb.wq[i], b = tb.wp[i];
                double cr = z1.x, ci = z1.y;
#pragma unroll
                for (int k = 0; k < 2 * H; ++k) {
                    acc[2 * k] = fma(a, cr, acc[2 * k]);
                    acc[2 * k + 1] = fma(a, ci, acc[2 * k + 1]);
                    if (k < H) {
                        acc[4 * H + 2 * k] = fma(b, cr, acc[4 * H + 2 * k]);
                        acc[4 * H + 2 * k + 1] = fma(b, ci, acc[4 * H + 2 * k + 1]);
                    }
                    if (k + 1 < 2 * H) {
                        const double nr = cr * z1.x - ci * z1.y, ni = cr * z1.y + ci * z1.x;
                        cr = nr;
                        ci = ni;
                    }
                }
            }
            block_sum<6 * H>(acc, sh);
        }
        if (threadIdx.x < 32) {
            const double dv = adj_factor<H>(sh, iw, sp, sc[SC_S1]) * chi0;
            const bool lower = it > 0 && dv < sh.dbest;
            __syncwarp();
            if (!lower) adj_coef<H>(sh, (W > 0.0) ? sqrt(chi0 / W) : 0.0);
            if (threadIdx.x == 0) {
                if (lower) {
                    // the step lowered Delta: halve it from the best point
                    sh.step *= 0.5;
                    sh.f = sh.fbest + sh.step;
                    sh.state = (fabs(sh.step) < tb.tol) ? 2 : 1;
                } else {
                    sh.fbest = f;
                    sh.dbest = dv;
                    sh.state = 0;
                }
            }
        }
        __syncthreads();
        if (sh.state == 2 || it == tb.max_iter) break;
        if (sh.state == 1) continue;
        // ---- pass B: model, residual and f-derivatives at the best f
        {
            double bs[NB], cf[m];
#pragma unroll
            for (int q = 0; q < NB; ++q) bs[q] = 0.0;
#pragma unroll
            for (int q = 0; q < m; ++q) cf[q] = sh.coef[q];
#pragma unroll 1
            for (int64_t i = a0 + threadIdx.x; i < a1; i += AD_NT) {
                const double ta = tb.tau[i];
                const double2 z1 = i - a0 < AD_ZC ? sh.z[i - a0]
                                                  : d_phasor(frac_fx(f, ta), t1, t2);
                const double w = tb.wq[i], wx = tb.wp[i];  // w, w (x - xbar)
                // model, and its f-derivatives in units of om = 2 pi tau
                double zr[H], zi[H], mv = cf[0], s1 = 0.0, s2 = 0.0;
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    if (h == 0) { zr[0] = z1.x; zi[0] = z1.y; }
                    else {
                        zr[h] = zr[h - 1] * z1.x - zi[h - 1] * z1.y;
                        zi[h] = zr[h - 1] * z1.y + zi[h - 1] * z1.x;
                    }
                    const double as = cf[2 * h + 1], ac = cf[2 * h + 2];
                    const double g1 = as * zi[h] + ac * zr[h];
                    const double g2 = as * zr[h] - ac * zi[h];
                    mv += g1;
                    s1 = fma((double)(h + 1), g2, s1);
                    s2 = fma((double)((h + 1) * (h + 1)), g1, s2);
                }
                const double om = 2.0 * M_PI * ta;
                const double mf = om * s1, mff = -(om * om) * s2;
                const double wr = fma(-w, mv, wx), wm = w * mf, wo = wr * om;
                bs[0] = fma(wr, mf, bs[0]);
                bs[1] = fma(-wr, mff, fma(wm, mf, bs[1]));
                bs[2] += wm;
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    const double wh = (double)(h + 1) * wo;
                    bs[3 + 2 * h] = fma(-wh, zr[h], fma(wm, zi[h], bs[3 + 2 * h]));
                    bs[4 + 2 * h] = fma(wh, zi[h], fma(wm, zr[h], bs[4 + 2 * h]));
                }
                if (it == 0) {
                    // gradients at the bin frequency, in the caller's sample order
                    const double xp = wx / w, r = xp - mv;  // x - xbar
                    const int64_t src = tb.perm ? (int64_t)tb.perm[i] : i;
                    const int64_t o = (int64_t)tb.K * a0 + (int64_t)r_in * n + (src - a0);
                    if (out.d_dx) out.d_dx[o] = g_up * 2.0 * w * mv;
                    if (out.d_dsig) out.d_dsig[o] = g_up * (-2.0 * w * sqrt(w)) * (xp * xp - r * r);
                }
            }
            block_sum<NB>(bs, sh);
        }
        if (threadIdx.x < 32) {
            // V^T alpha^-1 V = W (V / W)^T alpha'^-1 (V / W)
            const double q = adj_quad<H>(sh, threadIdx.x < m ? sh.tot[2 + threadIdx.x] * iw : 0.0);
            if (threadIdx.x == 0) {
                const double S1 = sh.tot[0], S2 = sh.tot[1];
                const double g = 2.0 * S1;  // dDelta/df
                if (it == 0 && out.d_df) out.d_df[e] = g_up * g;
                const double gpp = -(2.0 * S2 - 2.0 * W * q);  // d2 Delta / df2
                double step;
                if (gpp < 0.0) step = -g / gpp;
                else step = (g >= 0.0 ? 0.25 : -0.25) * df;  // not concave: move uphill
                if (step > 0.5 * df) step = 0.5 * df;
                if (step < -0.5 * df) step = -0.5 * df;
                double fn = f + step;
                if (fn < lo) fn = lo;
                if (fn > hi) fn = hi;
                sh.step = fn - f;
                if (fabs(sh.step) < tb.tol) {
                    sh.fbest = fn;  // converged: the last Newton update
                    sh.state = 2;
                } else {
                    sh.f = fn;
                    sh.state = 0;
                }
            }
        }
        __syncthreads();
        if (sh.state == 2) break;
    }
    if (threadIdx.x == 0) {
        if (out.f_ref) out.f_ref[e] = sh.fbest;
        if (out.d_ref) out.d_ref[e] = sh.dbest;
    }
}

__global__ void __launch_bounds__(AD_NT, 3) k_backward(AdjTab tb, int64_t E, AdjOut out) {
    __shared__ AdjShared sh;
    for (int i = threadIdx.x; i < 512; i += AD_NT) sh.tab[i] = tb.phasors[i];
    for (int64_t e = blockIdx.x; e < E; e += gridDim.x) {
        switch (tb.H[(int)(tb.ent[e] >> 32)]) {
            case 1: backward_entry<1>(tb, e, out, sh); break;
            case 2: backward_entry<2>(tb, e, out, sh); break;
            case 3: backward_entry<3>(tb, e, out, sh); break;
            case 4: backward_entry<4>(tb, e, out, sh); break;
            case 5: backward_entry<5>(tb, e, out, sh); break;
            case 6: backward_entry<6>(tb, e, out, sh); break;
            case 7: backward_entry<7>(tb, e, out, sh); break;
            default: backward_entry<8>(tb, e, out, sh); break;
        }
        __syncthreads();
    }
}

cudaError_t launch_backward_tab(const AdjTab& tb, int64_t E, const AdjOut& out, cudaStream_t s) {
    const unsigned blocks = (unsigned)std::min<int64_t>(E, INT32_MAX);
    k_backward<<<blocks, AD_NT, 0, s>>>(tb, E, out);
    return cudaGetLastError();
}

}  // namespace fc2

namespace fc2 {

// Host side of fc2_backward for one plan: entries (0 << 32 | j), outputs to
// the caller's buffers (device in place, host through staging).
fc2_status plan_backward(fc2_plan_s* p, int K, const int64_t* peak_j, const double* grad_out,
                         double* f_ref, double* d_ref, double* d_df, double* d_dx,
                         double* d_dsig) {
    if (!p || K < 1 || !peak_j) return FC2_ERR_INVALID_ARG;
    if (p->H > AD_HM) return FC2_ERR_UNSUPPORTED;
    for (int k = 0; k < K; ++k)
        if (peak_j[k] < 0 || peak_j[k] >= p->N) return FC2_ERR_INVALID_ARG;
    if (cudaSetDevice(p->device) != cudaSuccess) return FC2_ERR_CUDA;
    cudaStream_t s = p->stream;
    const int64_t n = p->n;
    auto is_dev = [&](const void* q) {
        cudaPointerAttributes at;
        bool d = q && cudaPointerGetAttributes(&at, q) == cudaSuccess && at.type == cudaMemoryTypeDevice;
        cudaGetLastError();
        return d;
    };
    const bool dx_dev = is_dev(d_dx), ds_dev = is_dev(d_dsig);
    int64_t* d_off = nullptr; int* d_H = nullptr; double *d_fmin = nullptr, *d_df_c = nullptr;
    int64_t* d_ent = nullptr; double* d_g = nullptr;
    double *o_f = nullptr, *o_d = nullptr, *o_df = nullptr, *o_dx = nullptr, *o_ds = nullptr;
    cudaError_t e = cudaSuccess;
    auto ok = [&](cudaError_t r) { if (e == cudaSuccess) e = r; return e == cudaSuccess; };
    ok(pool_alloc((void**)&d_off, 16, s)) && ok(pool_alloc((void**)&d_H, 4, s)) &&
        ok(pool_alloc((void**)&d_fmin, 8, s)) && ok(pool_alloc((void**)&d_df_c, 8, s)) &&
        ok(pool_alloc((void**)&d_ent, K * 8, s)) && ok(pool_alloc((void**)&o_f, K * 8, s)) &&
        ok(pool_alloc((void**)&o_d, K * 8, s)) && ok(pool_alloc((void**)&o_df, K * 8, s));
    if (grad_out) ok(pool_alloc((void**)&d_g, K * 8, s));
    if (d_dx && !dx_dev) ok(pool_alloc((void**)&o_dx, (size_t)K * n * 8, s));
    if (d_dsig && !ds_dev) ok(pool_alloc((void**)&o_ds, (size_t)K * n * 8, s));
    std::vector<int64_t> ent(K);
    for (int k = 0; k < K; ++k) ent[k] = peak_j[k];
    const int64_t offh[2] = {0, n};
    if (e == cudaSuccess) {
        ok(cudaMemcpyAsync(d_off, offh, 16, cudaMemcpyHostToDevice, s));
        ok(cudaMemcpyAsync(d_H, &p->H, 4, cudaMemcpyHostToDevice, s));
        ok(cudaMemcpyAsync(d_fmin, &p->f_min, 8, cudaMemcpyHostToDevice, s));
        ok(cudaMemcpyAsync(d_df_c, &p->df, 8, cudaMemcpyHostToDevice, s));
        ok(cudaMemcpyAsync(d_ent, ent.data(), K * 8, cudaMemcpyHostToDevice, s));
        if (grad_out) ok(cudaMemcpyAsync(d_g, grad_out, K * 8, cudaMemcpyDefault, s));
        AdjTab tb{d_off, d_H, d_fmin, d_df_c, p->d_scal, p->d_tau, p->d_wq, p->d_wp,
                  p->has_perm ? p->d_perm : nullptr, d_ent, d_g,
                  reinterpret_cast<const double2*>(p->d_dftab) + 512, K, 1e-10, 40};
        AdjOut out{o_f, o_d, o_df, dx_dev ? d_dx : o_dx, ds_dev ? d_dsig : o_ds};
        if (!d_dx) out.d_dx = nullptr;
        if (!d_dsig) out.d_dsig = nullptr;
        ok(launch_backward_tab(tb, K, out, s));
        std::vector<double> hf(K), hd(K), hg(K);
        ok(cudaMemcpyAsync(hf.data(), o_f, K * 8, cudaMemcpyDeviceToHost, s));
        ok(cudaMemcpyAsync(hd.data(), o_d, K * 8, cudaMemcpyDeviceToHost, s));
        ok(cudaMemcpyAsync(hg.data(), o_df, K * 8, cudaMemcpyDeviceToHost, s));
        if (d_dx && !dx_dev) ok(cudaMemcpyAsync(d_dx, o_dx, (size_t)K * n * 8, cudaMemcpyDeviceToHost, s));
        if (d_dsig && !ds_dev) ok(cudaMemcpyAsync(d_dsig, o_ds, (size_t)K * n * 8, cudaMemcpyDeviceToHost, s));
        ok(cudaStreamSynchronize(s));
        if (e == cudaSuccess) {
            for (int k = 0; k < K; ++k) {
                if (f_ref) f_ref[k] = hf[k];
                if (d_ref) d_ref[k] = hd[k];
                if (d_df) d_df[k] = hg[k];
            }
        }
    }
    for (void* q : {(void*)d_off, (void*)d_H, (void*)d_fmin, (void*)d_df_c, (void*)d_ent, (void*)d_g,
                    (void*)o_f, (void*)o_d, (void*)o_df, (void*)o_dx, (void*)o_ds})
        if (q) cudaFreeAsync(q, s);
    cudaStreamSynchronize(s);
    if (e == cudaErrorMemoryAllocation) return FC2_ERR_OOM;
    return e == cudaSuccess ? FC2_OK : FC2_ERR_CUDA;
}

}  // namespace fc2
