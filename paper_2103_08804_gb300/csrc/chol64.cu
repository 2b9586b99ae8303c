// Cholesky factor and triangular solves in float64 (CR_FP64 contexts).
//
// This GPU's float64 pipe does two multiply-adds per SM and cycle, so what
// counts here is that no lane multiplies padding and that every SM gets a
// share: panels of 16 columns, 16 x 16 tiles.  A (lower triangle, a copy of
// S) is factored in place below the diagonal blocks; the factors of the 16 x
// 16 diagonal blocks go to D.  Per panel J:
//   chol64_panel_kernel   every CTA factors A_JJ for itself (a few
//                         microseconds, one launch less than a separate
//                         kernel), then solves its rows of L_IJ
//   chol64_trail_kernel   A_IK -= L_IJ L_KJ^dag, one 16 x 16 tile per CTA
// The triangular solves take 128 rows at a time: one CTA holds the 128 x 128
// diagonal triangle in shared memory, then all rows beside it are updated.
#include "common.cuh"

namespace {

using zd = cpx<double>;
constexpr int NP = 16;            // panel width
constexpr int TR = 128;           // rows of a solve step
constexpr int PANEL_ROWS = 32;    // rows of L_IJ per CTA

CR_D zd shfl16(zd v, int src) {
    return {__shfl_sync(0xffffffffu, v.x, src, 16), __shfl_sync(0xffffffffu, v.y, src, 16)};
}

__global__ void __launch_bounds__(128) chol64_panel_kernel(double* __restrict__ A_, int P, int J,
                                                           double* __restrict__ D_,
                                                           int* __restrict__ status) {
    __shared__ zd l[NP][NP + 1];
    __shared__ zd col[2][NP];
    __shared__ double dinv[NP];
    zd* A = (zd*)A_;
    zd* D = (zd*)D_ + (size_t)J * NP * NP;
    const int base = J * NP, n = min(NP, P - base), t = threadIdx.x, k = t & 15, ti = t >> 4;
    // entries (ti, k) and (ti + 8, k) of the diagonal block, identity past P
    zd a[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int i = ti + 8 * q;
        a[q] = (i < n && k <= i) ? A[(size_t)(base + i) * P + base + k]
                                 : zd{i == k ? 1.0 : 0.0, 0.0};
    }
    bool bad = false;
    for (int j = 0; j < NP; ++j) {
        if (k == j) {
            col[j & 1][ti] = a[0];
            col[j & 1][ti + 8] = a[1];
        }
        __syncthreads();
        const zd* cj = col[j & 1];
        double d = cj[j].x;
        if (!(d > 0.0)) {
            bad = true;
            d = 1.0;
        }
        const double piv = sqrt(d), ip = 1.0 / piv;
        if (t == 0) dinv[j] = ip;
        const zd lk = conj(ip * cj[k]);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = ti + 8 * q;
            if (i > j && k >= j) {
                const zd li = ip * cj[i];
                if (k == j) a[q] = li;
                else if (k <= i) a[q] = a[q] - li * lk;
            } else if (i == j && k == j) {
                a[q] = {piv, 0.0};
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int i = ti + 8 * q;
        const zd v = k <= i ? a[q] : zd{0.0, 0.0};
        l[i][k] = v;
        if (blockIdx.x == 0) D[i * NP + k] = v;
    }
    if (blockIdx.x == 0 && t == 0 && bad) set_status(status, CR_ESINGULAR);
    __syncthreads();
    // rows below: x L_JJ^dag = a, column by column, 16 lanes (columns) a row
    const int r0 = base + NP + blockIdx.x * PANEL_ROWS;
#pragma unroll
    for (int p = 0; p < PANEL_ROWS / 8; ++p) {
        const int row = r0 + 8 * p + ti;
        zd v = row < P ? A[(size_t)row * P + base + k] : zd{0.0, 0.0};
#pragma unroll
        for (int c = 0; c < NP; ++c) {
            const zd x = dinv[c] * shfl16(v, c);
            if (k == c) v = x;
            else if (k > c) v = v - x * conj(l[k][c]);
        }
        if (row < P) A[(size_t)row * P + base + k] = v;
    }
}

// Tiles (a, b), b <= a, of the trailing matrix; 64 threads, 2 x 2 outputs.
__global__ void __launch_bounds__(64) chol64_trail_kernel(double* __restrict__ A_, int P, int J) {
    __shared__ zd li[NP][NP + 1], lk[NP][NP + 1];
    zd* A = (zd*)A_;
    const long long idx = blockIdx.x;
    int a = (int)((sqrt(8.0 * (double)idx + 1.0) - 1.0) * 0.5);
    while ((long long)a * (a + 1) / 2 > idx) --a;
    while ((long long)(a + 1) * (a + 2) / 2 <= idx) ++a;
    const int b = (int)(idx - (long long)a * (a + 1) / 2);
    const int c0 = J * NP, i0 = c0 + NP + a * NP, k0 = c0 + NP + b * NP;
    const int t = threadIdx.x, tx = t & 7, ty = t >> 3;
    for (int e = t; e < NP * NP; e += 64) {
        const int r = e / NP, c = e % NP;
        li[r][c] = i0 + r < P ? A[(size_t)(i0 + r) * P + c0 + c] : zd{0.0, 0.0};
        lk[r][c] = k0 + r < P ? A[(size_t)(k0 + r) * P + c0 + c] : zd{0.0, 0.0};
    }
    zd acc[2][2];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = i0 + ty + 8 * p, k = k0 + tx + 8 * q;
            acc[p][q] = i < P && k < P ? A[(size_t)i * P + k] : zd{0.0, 0.0};
        }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NP; ++c) {
        const zd x0 = li[ty][c], x1 = li[ty + 8][c], y0 = conj(lk[tx][c]), y1 = conj(lk[tx + 8][c]);
        acc[0][0] = acc[0][0] - x0 * y0;
        acc[0][1] = acc[0][1] - x0 * y1;
        acc[1][0] = acc[1][0] - x1 * y0;
        acc[1][1] = acc[1][1] - x1 * y1;
    }
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = i0 + ty + 8 * p, k = k0 + tx + 8 * q;
            if (i < P && k < P) A[(size_t)i * P + k] = acc[p][q];
        }
}

// Entry (i, c), c <= i, of L: the diagonal 16-blocks are in D.
CR_D zd l_entry(const zd* A, const zd* D, int P, int i, int c) {
    return i / NP == c / NP ? D[(size_t)(i / NP) * NP * NP + (i % NP) * NP + c % NP]
                            : A[(size_t)i * P + c];
}

CR_HD int tri(int i, int j) { return i * (i + 1) / 2 + j; }
constexpr size_t DIAG_SMEM = (size_t)TR * (TR + 1) / 2 * sizeof(zd) + TR * (sizeof(zd) + sizeof(double));

// Solve with the diagonal block of step b: out = L_bb^-1 v (or L_bb^-dag v
// when BWD), one CTA of 256.  16 unknowns at a time: one warp solves them
// (lanes = unknowns), then all threads update the rest of the block.
template <bool BWD>
__global__ void __launch_bounds__(256) trsv64_diag_kernel(const double* __restrict__ A_,
                                                          const double* __restrict__ D_, int P,
                                                          int b, const double* __restrict__ in_,
                                                          double* __restrict__ out_,
                                                          const double* __restrict__ skip) {
    if (skip && *skip != 0.0) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    zd* l = (zd*)smem_raw;                       // packed lower triangle
    zd* v = l + TR * (TR + 1) / 2;               // [TR]
    double* dinv = (double*)(v + TR);            // [TR]
    const zd* A = (const zd*)A_;
    const zd* D = (const zd*)D_;
    const int base = b * TR, n = min(TR, P - base), t = threadIdx.x, lane = t & 31;
    for (int e = t; e < n * TR; e += 256) {
        const int i = e / TR, c = e % TR;
        if (c <= i) l[tri(i, c)] = l_entry(A, D, P, base + i, base + c);
    }
    if (t < n) {
        v[t] = ((const zd*)in_)[base + t];
        dinv[t] = 1.0 / l_entry(A, D, P, base + t, base + t).x;
    }
    __syncthreads();
    const int nblk = (n + NP - 1) / NP;
    for (int s = 0; s < nblk; ++s) {
        const int o = (BWD ? nblk - 1 - s : s) * NP, m = min(NP, n - o);
        if (t < 32) {
            const int k = lane & 15;
            zd x = k < m ? v[o + k] : zd{0.0, 0.0};
            for (int q = 0; q < m; ++q) {
                const int c = BWD ? m - 1 - q : q;
                const zd xc = dinv[o + c] * shfl16(x, c);
                if (k == c) x = xc;
                else if (BWD ? k < c : (k > c && k < m))
                    x = x - (BWD ? conj(l[tri(o + c, o + k)]) : l[tri(o + k, o + c)]) * xc;
            }
            if (lane < m) v[o + lane] = x;
        }
        __syncthreads();
        if (BWD ? t < o : (t >= o + NP && t < n)) {
            zd acc = v[t];
            for (int c = 0; c < m; ++c)
                acc = acc - (BWD ? conj(l[tri(o + c, t)]) : l[tri(t, o + c)]) * v[o + c];
            v[t] = acc;
        }
        __syncthreads();
    }
    if (t < n) ((zd*)out_)[base + t] = v[t];
}

// v_i -= sum_c L_ic x_c over the columns c of step b, for the rows below it
// (one warp a row), or v_i -= sum_c conj(L_ci) x_c for the rows above (BWD;
// lanes along i, warps along c).
template <bool BWD>
__global__ void __launch_bounds__(256) trsv64_rest_kernel(const double* __restrict__ A_, int P, int b,
                                                          const double* __restrict__ x_,
                                                          double* __restrict__ v_,
                                                          const double* __restrict__ skip) {
    if (skip && *skip != 0.0) return;
    __shared__ zd x[TR];
    __shared__ zd part[8][32];
    const zd* A = (const zd*)A_;
    zd* v = (zd*)v_;
    const int base = b * TR, n = min(TR, P - base), t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t < n) x[t] = ((const zd*)x_)[base + t];
    __syncthreads();
    if (!BWD) {
        const int row = base + n + blockIdx.x * 8 + warp;
        if (row >= P) return;
        zd s = {0.0, 0.0};
        for (int c = lane; c < n; c += 32) s = s + A[(size_t)row * P + base + c] * x[c];
        s = warp_sum(s);
        if (lane == 0) v[row] = v[row] - s;
    } else {
        const int i = blockIdx.x * 32 + lane;
        zd s = {0.0, 0.0};
        if (i < base)
#pragma unroll 4
            for (int c = warp; c < n; c += 8) s = s + conj(A[(size_t)(base + c) * P + i]) * x[c];
        part[warp][lane] = s;
        __syncthreads();
        if (warp == 0 && i < base) {
            zd tot = part[0][lane];
            for (int w = 1; w < 8; ++w) tot = tot + part[w][lane];
            v[i] = v[i] - tot;
        }
    }
}

}  // namespace

size_t chol64_diag_bytes(int P) { return (size_t)((P + NP - 1) / NP) * NP * NP * sizeof(zd); }

cr_status chol64_prepare(cr_ctx* c) {
    cudaError_t e = cudaFuncSetAttribute(trsv64_diag_kernel<false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DIAG_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(trsv64_diag_kernel<true>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DIAG_SMEM);
    return e == cudaSuccess ? CR_OK : cr_fail(c, CR_ECUDA, "chol64_prepare: %s", cudaGetErrorString(e));
}

// A = S copied, factored in place (D: the diagonal blocks' factors).
cr_status chol64_factor(cr_ctx* c, double* A, double* D) {
    const int P = c->P, nb = (P + NP - 1) / NP;
    cudaError_t e = cudaMemcpyAsync(A, c->S, (size_t)P * P * sizeof(zd), cudaMemcpyDeviceToDevice,
                                    c->stream);
    if (e != cudaSuccess) return cr_fail(c, CR_ECUDA, "chol64: %s", cudaGetErrorString(e));
    for (int J = 0; J < nb; ++J) {
        const int rows = P - (J + 1) * NP;
        const int g = rows > 0 ? (rows + PANEL_ROWS - 1) / PANEL_ROWS : 1;
        CR_LAUNCH(c, CR_KERNEL_CHOL,
                  chol64_panel_kernel<<<g, 128, 0, c->stream>>>(A, P, J, D, c->d_status));
        if (rows <= 0) break;
        const long long T = nb - J - 1;
        CR_LAUNCH(c, CR_KERNEL_CHOL, chol64_trail_kernel<<<(unsigned)(T * (T + 1) / 2), 64, 0, c->stream>>>(
                                         A, P, J));
    }
    return cr_check_launch(c, "float64 Cholesky");
}

// d = L^{-dag} L^{-1} r (r and y are scratch)
void chol64_solve(cr_ctx* c, const double* A, const double* D, double* r, double* y, double* d,
                  const double* skip) {
    const int P = c->P, nt = (P + TR - 1) / TR;
    for (int b = 0; b < nt; ++b) {
        const int rows = P - (b + 1) * TR;
        CR_LAUNCH(c, CR_KERNEL_TRSV, trsv64_diag_kernel<false><<<1, 256, DIAG_SMEM, c->stream>>>(
                                         A, D, P, b, r, y, skip));
        if (rows > 0)
            CR_LAUNCH(c, CR_KERNEL_TRSV, trsv64_rest_kernel<false><<<(rows + 7) / 8, 256, 0, c->stream>>>(
                                             A, P, b, y, r, skip));
    }
    for (int b = nt - 1; b >= 0; --b) {
        CR_LAUNCH(c, CR_KERNEL_TRSV, trsv64_diag_kernel<true><<<1, 256, DIAG_SMEM, c->stream>>>(
                                         A, D, P, b, y, d, skip));
        if (b > 0)
            CR_LAUNCH(c, CR_KERNEL_TRSV,
                      trsv64_rest_kernel<true><<<(b * TR + 31) / 32, 256, 0, c->stream>>>(A, P, b, d, y, skip));
    }
}
