// Chebyshev moment correction and the Krylov projection (Secs. IV, V).
//
// cheb_gram builds sigma_nm = <t_n|t_m> and H_nm = <t_n|H'|t_m> from the
// per-sample columns B_n(s) = t_n(s)/psi(s), (H' t_n)(s)/psi(s).
// cheb_krylov then works in float64: a complex Hermitian n x n matrix
// A = Ar + i Ai is handled through its real symmetric embedding
// [[Ar, -Ai], [Ai, Ar]] (every eigenvalue twice, eigenvector pairs
// [ur; ui], [-ui; ur]), diagonalised by cyclic Jacobi rotations applied to
// n disjoint pairs at a time (round-robin ordering), all rounds of all sweeps
// in one cooperative launch; so is the moment recursion.
#include "common.cuh"

// ------------------------------------------------------------------ Gram

template <typename R>
__global__ void gram_kernel(const cpx<R>* __restrict__ Bm, const cpx<R>* __restrict__ HBm, int Nm,
                            int B, int ld, double* __restrict__ G_, double* __restrict__ H_) {
    __shared__ cpx<R> tn[16][17], tm[16][17], th[16][17];
    const int n = blockIdx.y * 16 + threadIdx.y, m = blockIdx.x * 16 + threadIdx.x;
    cpx<double> g = {0.0, 0.0}, h = {0.0, 0.0};
    for (int s0 = 0; s0 < B; s0 += 16) {
        const int nn = blockIdx.y * 16 + threadIdx.y, s = s0 + threadIdx.x;
        tn[threadIdx.y][threadIdx.x] = (nn < Nm && s < B) ? Bm[(size_t)nn * ld + s] : cpx<R>{R(0), R(0)};
        const int mm = blockIdx.x * 16 + threadIdx.y;
        tm[threadIdx.y][threadIdx.x] = (mm < Nm && s < B) ? Bm[(size_t)mm * ld + s] : cpx<R>{R(0), R(0)};
        th[threadIdx.y][threadIdx.x] =
            (HBm && mm < Nm && s < B) ? HBm[(size_t)mm * ld + s] : cpx<R>{R(0), R(0)};
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            cpx<R> a = tn[threadIdx.y][q];
            g = g + ccast<double>(cmulc(a, tm[threadIdx.x][q]));
            h = h + ccast<double>(cmulc(a, th[threadIdx.x][q]));
        }
        __syncthreads();
    }
    if (n < Nm && m < Nm) {
        ((cpx<double>*)G_)[(size_t)n * Nm + m] = (1.0 / B) * g;
        if (H_) ((cpx<double>*)H_)[(size_t)n * Nm + m] = (1.0 / B) * h;
    }
}

__global__ void hermitise_kernel(double* __restrict__ H_, int Nm) {
    cpx<double>* H = (cpx<double>*)H_;
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= Nm * Nm) return;
    int n = idx / Nm, m = idx % Nm;
    if (m < n) return;
    cpx<double> a = H[(size_t)n * Nm + m], b = H[(size_t)m * Nm + n];
    cpx<double> v = 0.5 * (a + conj(b));
    H[(size_t)n * Nm + m] = v;
    H[(size_t)m * Nm + n] = conj(v);
}

extern "C" cr_status cheb_gram(cr_ctx* ctx, const void* Bmat, const void* HBmat, int Nm, int B,
                               int ld, double* G_out, double* H_out) {
    if (!ctx) return CR_EINVAL;
    CR_CHECK_ARG(Nm >= 1 && B >= 1 && ld >= B, "cheb_gram: bad sizes");
    CR_CHECK_ARG(Bmat && G_out && ((HBmat && H_out) || (!HBmat && !H_out)),
                 "cheb_gram: null array (HBmat and H_out are both given or both NULL)");
    if (ctx->prec == CR_MIXED) return launch_gram_tc(ctx, Bmat, HBmat, Nm, B, ld, G_out, H_out);
    dim3 g((Nm + 15) / 16, (Nm + 15) / 16);
    if (ctx->prec == CR_FP64)
        CR_LAUNCH(ctx, CR_K_OTHER, gram_kernel<double><<<g, dim3(16, 16), 0, ctx->stream>>>(
            (const cpx<double>*)Bmat, (const cpx<double>*)HBmat, Nm, B, ld, G_out, H_out));
    else
        CR_LAUNCH(ctx, CR_K_OTHER, gram_kernel<float><<<g, dim3(16, 16), 0, ctx->stream>>>(
            (const cpx<float>*)Bmat, (const cpx<float>*)HBmat, Nm, B, ld, G_out, H_out));
    if (H_out)
        CR_LAUNCH(ctx, CR_K_OTHER, hermitise_kernel<<<(Nm * Nm + 255) / 256, 256, 0, ctx->stream>>>(H_out, Nm));
    return cr_check_launch(ctx, "cheb_gram");
}

// ------------------------------------------------------------- Jacobi
//
// Cyclic Jacobi for the symmetric m x m embedding (m even).  Each sweep has
// m - 1 rounds (round-robin pairing of the m indices: position 0 fixed, the
// others rotating); a round applies its m / 2 disjoint rotations at once,
// A' = J^T A J and V' = V J, from one pair of buffers to the other.  A 2 x 2
// block of A (row pair P, column pair Q) is one thread's work.  Every CTA
// takes one tile of blocks or of V, and the angles of its own pairs, so a
// round ends with one grid barrier.  Before each sweep the off-diagonal norm
// is reduced (fixed order); once it is below JAC_TOL times the diagonal every
// CTA leaves.
//
// The sweeps end with an off-diagonal of 1e-12 left, which is 1e-9 to 1e-8 in
// the weights of 300 states: another order of rotations, or another rounding
// of one, would leave another remainder of that size.  So the rotations, their
// order and their roundings (rot, spelled out) are fixed.
//
// What bounds a round: float64 arithmetic (4 operations an element of A, 2 of
// V, at two per SM and cycle: 3.4 us at m = 600), the barrier, and two round
// trips to L2 with the angles' divisions and square roots between them; the
// blocks are loaded before the angles are formed.  One launch per round, the
// two eigenproblems of 300 states took 654 ms (36,000 launches); now 140 ms.

namespace {

using zd = cpx<double>;

constexpr int JAC_MAX_SWEEPS = 30;
constexpr double JAC_TOL = 1e-24;  // off^2 <= JAC_TOL diag^2 (relative 1e-12)
constexpr int JT = 512;            // threads
constexpr int MAX_TP = 64;         // pairs per tile at most
constexpr unsigned BAR_LIMIT = 1u << 23;  // grid-barrier polls

// Element of the round-robin schedule: position 0 is fixed, the others
// rotate by one place per round.
CR_D int rr_elem(int pos, int round, int m) {
    return pos == 0 ? 0 : ((pos - 1 + round) % (m - 1)) + 1;
}

// c x + s y as the rotations round it
CR_D double rot(double c, double x, double s, double y) { return fma(c, x, __dmul_rn(s, y)); }

struct JacBufs {
    double* A[2];
    double* V[2];
    double* part;  // [2][gridDim] shares of the norms
    unsigned* bar; // [0] arrivals, [1] abort
    int* res;      // index of the buffers holding the result
};

struct JacArgs {
    JacBufs J;
    int m, tp, nt, na, nv, rv;  // tile: pairs, tiles a side, tiles of A, of V, rows of a V tile
    int* status;
};

// Grid barrier: arrive, wait (bounded) for all CTAs; false after an abort.
CR_D bool grid_sync(unsigned* bar, unsigned target, volatile int* flag, int* status) {
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(&bar[0]) : "memory");
        for (unsigned n = 0; *(volatile unsigned*)&bar[0] < target; ++n) {
            if (*(volatile unsigned*)&bar[1] || n > BAR_LIMIT) {
                if (n > BAR_LIMIT) {
                    atomicExch(&bar[1], 1u);
                    set_status(status, CR_ETIMEOUT);
                }
                *flag = 1;
                break;
            }
            if (n > 4096) __nanosleep(64);
        }
        asm volatile("fence.acq_rel.gpu;\n" ::: "memory");
    }
    __syncthreads();
    return *flag == 0;
}

__global__ void __launch_bounds__(JT) jacobi_kernel(const JacArgs a) {
    __shared__ double ac[2 * MAX_TP], as[2 * MAX_TP], red[2][JT / 32];
    __shared__ int ip[2 * MAX_TP], iq[2 * MAX_TP];
    __shared__ int flag_, done_;
    volatile int* flag = &flag_;
    const int m = a.m, np = m / 2, t = threadIdx.x;
    const JacBufs& J = a.J;
    if (t == 0) *flag = 0;
    unsigned arrived = 0;
    const unsigned G = gridDim.x;
    for (size_t e = (size_t)blockIdx.x * JT + t; e < (size_t)m * m; e += (size_t)G * JT)
        __stcg(&J.V[0][e], e / m == e % m ? 1.0 : 0.0);
    int in = 0;
    bool ok = grid_sync(J.bar, ++arrived * G, flag, a.status);
    for (int sweep = 0; sweep < JAC_MAX_SWEEPS && ok; ++sweep) {
        // squared off-diagonal and diagonal norms
        double off = 0.0, dia = 0.0;
        for (size_t e = (size_t)blockIdx.x * JT + t; e < (size_t)m * m; e += (size_t)G * JT) {
            const double x = __ldcg(&J.A[in][e]), v = x * x;
            if (e / m == e % m) dia += v;
            else off += v;
        }
        off = warp_sum(off);
        dia = warp_sum(dia);
        if ((t & 31) == 0) {
            red[0][t >> 5] = off;
            red[1][t >> 5] = dia;
        }
        __syncthreads();
        if (t < 2) {
            double v = 0.0;
            for (int w = 0; w < JT / 32; ++w) v += red[t][w];
            __stcg(&J.part[t * G + blockIdx.x], v);
        }
        ok = grid_sync(J.bar, ++arrived * G, flag, a.status);
        if (!ok) break;
        if (t < 32) {
            double o = 0.0, d = 0.0;
            for (unsigned b = t; b < G; b += 32) {
                o += __ldcg(&J.part[b]);
                d += __ldcg(&J.part[G + b]);
            }
            o = warp_sum(o);
            d = warp_sum(d);
            if (t == 0) done_ = !(o > JAC_TOL * d);
        }
        __syncthreads();
        if (done_) break;
        for (int round = 0; round < m - 1 && ok; ++round) {
            const double* A = J.A[in];
            const double* V = J.V[in];
            double* Ao = J.A[in ^ 1];
            double* Vo = J.V[in ^ 1];
            for (int tile = blockIdx.x; tile < a.na + a.nv; tile += G) {
                // pair blocks of the tile: rows P0.., columns Q0.. (a tile of V has single rows)
                const bool isA = tile < a.na;
                const int tv = isA ? tile : tile - a.na, Q0 = (tv % a.nt) * a.tp;
                const int P0 = isA ? (tv / a.nt) * a.tp : 0, r0 = isA ? 0 : (tv / a.nt) * a.rv;
                const int rows = isA ? min(a.tp, np - P0) : min(a.rv, m - r0), cols = min(a.tp, np - Q0);
                // row pairs at [0, tp), column pairs at [tp, 2 tp)
                const int k = t < a.tp ? P0 + t : Q0 + t - a.tp;
                const bool ang = t < 2 * a.tp && (isA || t >= a.tp) && k < np;
                __syncthreads();
                double apq = 0.0, aqq = 0.0, app = 0.0;
                if (ang) {
                    const int ep = rr_elem(k, round, m), eq = rr_elem(m - 1 - k, round, m);
                    ip[t] = ep;
                    iq[t] = eq;
                    apq = __ldcg(&A[(size_t)ep * m + eq]);
                    aqq = __ldcg(&A[(size_t)eq * m + eq]);
                    app = __ldcg(&A[(size_t)ep * m + ep]);
                }
                __syncthreads();
                // a warp takes rows of blocks, lanes the columns; the first rows are loaded
                // before the angles are formed
                const int lane = t & 31, wp = t >> 5;
                double x0[2], x1[2], y0[2], y1[2];
                auto fetch = [&](int c0, int l0) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int l = l0 + h * (JT / 32);
                        if (l >= rows || c0 + lane >= cols) continue;
                        const int r = ip[a.tp + c0 + lane], u = iq[a.tp + c0 + lane];
                        const double* S = isA ? A + (size_t)ip[l] * m : V + (size_t)(r0 + l) * m;
                        x0[h] = __ldcg(S + r);
                        x1[h] = __ldcg(S + u);
                        if (isA) {
                            const double* S2 = A + (size_t)iq[l] * m;
                            y0[h] = __ldcg(S2 + r);
                            y1[h] = __ldcg(S2 + u);
                        }
                    }
                };
                fetch(0, wp);
                if (ang) {
                    double c = 1.0, sn = 0.0;
                    if (apq != 0.0) {
                        const double tau = (aqq - app) / (2.0 * apq);
                        const double tt = (tau >= 0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(fma(tau, tau, 1.0)));
                        c = 1.0 / sqrt(fma(tt, tt, 1.0));
                        sn = tt * c;
                    }
                    ac[t] = c;
                    as[t] = sn;
                }
                __syncthreads();
                for (int c0 = 0; c0 < cols; c0 += 32)
                    for (int l0 = wp; l0 < rows; l0 += 2 * (JT / 32)) {
                        if (c0 != 0 || l0 != wp) fetch(c0, l0);
                        if (c0 + lane >= cols) continue;
                        const int lQ = a.tp + c0 + lane, r = ip[lQ], u = iq[lQ];
                        const double c = ac[lQ], s = as[lQ];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int l = l0 + h * (JT / 32);
                            if (l >= rows) continue;
                            const double b00 = rot(c, x0[h], -s, x1[h]), b01 = rot(c, x1[h], s, x0[h]);
                            if (!isA) {
                                double* D = Vo + (size_t)(r0 + l) * m;
                                __stcg(D + r, b00);
                                __stcg(D + u, b01);
                                continue;
                            }
                            const double d = ac[l], g = as[l];
                            const double b10 = rot(c, y0[h], -s, y1[h]), b11 = rot(c, y1[h], s, y0[h]);
                            double* Dp = Ao + (size_t)ip[l] * m;
                            double* Dq = Ao + (size_t)iq[l] * m;
                            __stcg(Dp + r, rot(d, b00, -g, b10));
                            __stcg(Dp + u, rot(d, b01, -g, b11));
                            __stcg(Dq + r, rot(d, b10, g, b00));
                            __stcg(Dq + u, rot(d, b11, g, b01));
                        }
                    }
            }
            ok = grid_sync(J.bar, ++arrived * G, flag, a.status);
            in ^= 1;
        }
    }
    if (blockIdx.x == 0 && t == 0) *J.res = in;
}

// A cooperative launch (co-resident CTAs).
template <typename K, typename A>
cr_status coop_launch(cr_ctx* c, K kernel, int grid, int threads, const A& args, const char* name) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = c->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e;
    CR_LAUNCH(c, CR_K_OTHER, e = cudaLaunchKernelEx(&cfg, kernel, args));
    return e == cudaSuccess ? CR_OK : cr_fail(c, CR_ECUDA, "%s: %s", name, cudaGetErrorString(e));
}

// Diagonalise the symmetric m x m matrix in J.A[0] (m even); eigenvalues on
// the diagonal of J.A[*res], eigenvectors in the columns of J.V[*res].  The
// smallest tiles that leave every CTA at most one; a small matrix on one CTA,
// where a barrier is cheap.
cr_status jacobi_launch(cr_ctx* c, const JacBufs& J, int m) {
    JacArgs a = {};
    const int np = m / 2;
    auto shape = [&]() {
        a.nt = (np + a.tp - 1) / a.tp;
        a.rv = 4 * a.tp;
        a.na = a.nt * a.nt;
        a.nv = a.nt * ((m + a.rv - 1) / a.rv);
        return a.na + a.nv;
    };
    a.J = J;
    a.m = m;
    a.status = c->d_status;
    a.tp = m <= 32 ? np : 4;
    while (shape() > c->n_sm && a.tp < MAX_TP) ++a.tp;
    const int tiles = a.na + a.nv, grid = m <= 32 ? 1 : (tiles < c->n_sm ? tiles : c->n_sm);
    cudaError_t e = cudaMemsetAsync(J.bar, 0, 2 * sizeof(unsigned), c->stream);
    if (e != cudaSuccess) return cr_fail(c, CR_ECUDA, "jacobi_kernel: %s", cudaGetErrorString(e));
    return coop_launch(c, jacobi_kernel, grid, JT, a, "jacobi_kernel");
}

// Real symmetric embedding [[Ar, -Ai], [Ai, Ar]] of a complex Hermitian n x n
// matrix (every eigenvalue twice, eigenvector pairs [ur; ui], [-ui; ur]).
__global__ void kry_embed_kernel(const double* __restrict__ A_, int n, double* __restrict__ E) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * n) return;
    const int m = 2 * n, i = e / n, j = e % n;
    const cpx<double> a = ((const cpx<double>*)A_)[e];
    E[(size_t)i * m + j] = a.x;
    E[(size_t)(i + n) * m + j + n] = a.x;
    E[(size_t)(i + n) * m + j] = a.y;
    E[(size_t)i * m + j + n] = -a.y;
}

// Eigenvalues of the embedded G, the kept index list (relative cutoff; an
// odd count drops the smallest, the copy a cutoff split by rounding) and
// the rank r (even).  One CTA, one thread per eigenvalue (m <= 1024).
__global__ void __launch_bounds__(1024) kry_keep_kernel(JacBufs J, int m, double cutoff,
                                                        double* __restrict__ d, int* __restrict__ keep,
                                                        int* __restrict__ rank) {
    __shared__ double red[32];
    __shared__ int redi[32], cnt[32];
    const double* E = J.A[*J.res];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const double v = t < m ? E[(size_t)t * m + t] : 0.0;
    if (t < m) d[t] = v;
    double mx = v;
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) red[w] = mx;
    __syncthreads();
    mx = 0.0;
    for (int i = 0; i < 32; ++i) mx = fmax(mx, red[i]);
    __syncthreads();
    bool on = t < m && v > cutoff * mx;
    // smallest kept eigenvalue (lowest index among equals)
    double lo = on ? v : 1e308;
    int li = t;
    for (int o = 16; o > 0; o >>= 1) {
        const double l2 = __shfl_xor_sync(0xffffffffu, lo, o);
        const int i2 = __shfl_xor_sync(0xffffffffu, li, o);
        if (l2 < lo || (l2 == lo && i2 < li)) {
            lo = l2;
            li = i2;
        }
    }
    const unsigned b0 = __ballot_sync(0xffffffffu, on);
    if (lane == 0) {
        red[w] = lo;
        redi[w] = li;
        cnt[w] = __popc(b0);
    }
    __syncthreads();
    int tot = 0;
    for (int i = 0; i < 32; ++i) {
        tot += cnt[i];
        if (red[i] < lo || (red[i] == lo && redi[i] < li)) {
            lo = red[i];
            li = redi[i];
        }
    }
    if ((tot & 1) && t == li) on = false;
    __syncthreads();
    const unsigned b1 = __ballot_sync(0xffffffffu, on);
    if (lane == 0) cnt[w] = __popc(b1);
    __syncthreads();
    int at = 0;
    for (int i = 0; i < w; ++i) at += cnt[i];
    if (on) keep[at + __popc(b1 & ((1u << lane) - 1u))] = t;
    if (t == 0) *rank = tot & ~1;
}

// X[i][q] = V[i][keep q] / sqrt(d) for q < r, 0 for r <= q < m (padding).
__global__ void kry_x_kernel(JacBufs J, int m, const double* __restrict__ d,
                             const int* __restrict__ keep, const int* __restrict__ rank,
                             double* __restrict__ X) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= m * m) return;
    const int i = e / m, q = e % m, r = *rank;
    const double* V = J.V[*J.res];
    X[e] = q < r ? V[(size_t)i * m + keep[q]] / sqrt(d[keep[q]]) : 0.0;
}

// C = A^T B, A B or A B^T (m x m, row-major), one output per thread (float64).
template <bool TRANS_A, bool TRANS_B>
__global__ void kry_gemm_kernel(const double* __restrict__ A, const double* __restrict__ B, int m,
                                double* __restrict__ C) {
    __shared__ double as[16][17], bs[16][17];
    const int i = blockIdx.y * 16 + threadIdx.y, j = blockIdx.x * 16 + threadIdx.x;
    const int ty = threadIdx.y, tx = threadIdx.x;
    double s = 0.0;
    for (int l0 = 0; l0 < m; l0 += 16) {
        const int ia = blockIdx.y * 16, jb = blockIdx.x * 16;
        if (TRANS_A) as[tx][ty] = (ia + tx < m && l0 + ty < m) ? A[(size_t)(l0 + ty) * m + ia + tx] : 0.0;
        else as[ty][tx] = (i < m && l0 + tx < m) ? A[(size_t)i * m + l0 + tx] : 0.0;
        if (TRANS_B) bs[tx][ty] = (jb + ty < m && l0 + tx < m) ? B[(size_t)(jb + ty) * m + l0 + tx] : 0.0;
        else bs[ty][tx] = (l0 + ty < m && j < m) ? B[(size_t)(l0 + ty) * m + j] : 0.0;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 16; ++q) s += as[ty][q] * bs[q][tx];
        __syncthreads();
    }
    if (i < m && j < m) C[(size_t)i * m + j] = s;
}

// C = Y S with Y = G^+ = Yr + i Yi from the first n columns of the embedded
// pseudo-inverse [[Yr, .], [Yi, .]] and S = H or G (n x n complex).
__global__ void __launch_bounds__(256) kry_pgemm_kernel(const double* __restrict__ Y,
                                                        const double* __restrict__ S_, int n,
                                                        zd* __restrict__ C) {
    __shared__ zd as[16][17], bs[16][17];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, m = 2 * n;
    const int i = blockIdx.y * 16 + ty, j = blockIdx.x * 16 + tx;
    const zd* S = (const zd*)S_;
    const zd zero = {0.0, 0.0};
    zd s = zero;
    for (int l0 = 0; l0 < n; l0 += 16) {
        as[ty][tx] = i < n && l0 + tx < n ? zd{Y[(size_t)i * m + l0 + tx], Y[(size_t)(i + n) * m + l0 + tx]} : zero;
        bs[ty][tx] = l0 + ty < n && j < n ? S[(size_t)(l0 + ty) * n + j] : zero;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 16; ++q) s = s + as[ty][q] * bs[q][tx];
        __syncthreads();
    }
    if (i < n && j < n) C[(size_t)i * n + j] = s;
}

// out = (C + C^T) / 2 into the Jacobi input buffer; g0 = X^T [Re G e0; Im G e0].
__global__ void kry_sym_kernel(const double* __restrict__ C, int m, double* __restrict__ out) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= m * m) return;
    const int a = e / m, b = e % m;
    out[e] = 0.5 * (C[e] + C[(size_t)b * m + a]);
}

__global__ void __launch_bounds__(256) kry_g0_kernel(const double* __restrict__ G_,
                                                     const double* __restrict__ X, int m,
                                                     double* __restrict__ g0) {
    const int q = blockIdx.x * 32 + (threadIdx.x & 31), part = threadIdx.x >> 5, n = m / 2;
    __shared__ double red[8][32];
    const zd* G = (const zd*)G_;
    double s = 0.0;
    if (q < m)
        for (int l = part; l < n; l += 8) {
            const zd gl = G[(size_t)l * n];
            s += X[(size_t)l * m + q] * gl.x + X[(size_t)(l + n) * m + q] * gl.y;
        }
    red[part][threadIdx.x & 31] = s;
    __syncthreads();
    if (part == 0 && q < m) {
        for (int w = 1; w < 8; ++w) s += red[w][threadIdx.x & 31];
        g0[q] = s;
    }
}

// Moment correction: c_0 = e_0, c_1 = K c_0, c_{k+1} = 2 K c_k - Q c_{k-1}
// with K = G^+ H and Q = G^+ G formed once; mu'_k = (G c_k)_0.  One cooperative
// launch, a warp per row, one grid barrier per k; the moments of a block of
// vectors follow it.
constexpr int MOM_CHUNK = 512;

struct MomArgs {
    const zd* K;
    const zd* Q;
    zd* c;       // [MOM_CHUNK + 2][n]: c_{first-2}, c_{first-1}, then the chunk's vectors
    int n, first, count;
    unsigned* bar;
    int* status;
};

constexpr int REC_WARPS = 2;  // rows per CTA: few, since a row's 8 n operations wait for the float64 pipe
__global__ void __launch_bounds__(32 * REC_WARPS) kry_recur_kernel(const MomArgs a) {
    __shared__ int flag_;
    volatile int* flag = &flag_;
    const int n = a.n, lane = threadIdx.x & 31, warp = blockIdx.x * REC_WARPS + (threadIdx.x >> 5);
    const int nw = gridDim.x * REC_WARPS;
    if (threadIdx.x == 0) *flag = 0;
    __syncthreads();
    for (int k = 0; k < a.count; ++k) {
        const int step = a.first + k;
        const zd* c0 = a.c + (size_t)(k + 1) * n;  // c_{step-1}
        const zd* c1 = a.c + (size_t)k * n;        // c_{step-2}
        zd* out = a.c + (size_t)(k + 2) * n;
        for (int i = warp; i < n; i += nw) {
            zd s = {0.0, 0.0}, q = {0.0, 0.0};
            if (step == 0) {
                s = {i == 0 ? 1.0 : 0.0, 0.0};
            } else {
                for (int l = lane; l < n; l += 32) {
                    const double2 x = __ldcg((const double2*)(c0 + l));
                    s = s + ldg(a.K + (size_t)i * n + l) * zd{x.x, x.y};
                    if (step >= 2) {
                        const double2 y = __ldcg((const double2*)(c1 + l));
                        q = q + ldg(a.Q + (size_t)i * n + l) * zd{y.x, y.y};
                    }
                }
                if (step >= 2) s = 2.0 * s - q;
                s = warp_sum(s);
            }
            if (lane == 0) __stcg((double2*)(out + i), make_double2(s.x, s.y));
        }
        if (!grid_sync(a.bar, (unsigned)(k + 1) * gridDim.x, flag, a.status)) return;
    }
}

__global__ void __launch_bounds__(128) kry_mu_kernel(const zd* __restrict__ G, const zd* __restrict__ c, int n,
                                                     int first, double* __restrict__ mu) {
    __shared__ zd red[4];
    const int t = threadIdx.x;
    const zd* v = c + (size_t)(blockIdx.x + 2) * n;
    zd s = {0.0, 0.0};
    for (int l = t; l < n; l += 128) s = s + G[l] * v[l];
    s = warp_sum(s);
    if ((t & 31) == 0) red[t >> 5] = s;
    __syncthreads();
    if (t == 0) ((zd*)mu)[first + blockIdx.x] = (red[0] + red[1]) + (red[2] + red[3]);
}

// Eigenvalue k = E[k][k] and weight (V[:, k] . g0)^2 of the diagonalised
// projection, k < r; one warp each.
__global__ void __launch_bounds__(256) kry_weight_kernel(JacBufs J, int m, const double* __restrict__ g0,
                                                         const int* __restrict__ rank,
                                                         double* __restrict__ d, double* __restrict__ wk) {
    const int k = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, r = *rank;
    if (k >= r) return;
    const double* E = J.A[*J.res];
    const double* V = J.V[*J.res];
    double s = 0.0;
    for (int q = lane; q < r; q += 32) s += V[(size_t)q * m + k] * g0[q];
    s = warp_sum(s);
    if (lane == 0) {
        wk[k] = s * s;
        d[k] = E[(size_t)k * m + k];
    }
}

// Poles in ascending order (by rank counting, one thread per eigenvalue) and
// the doubled eigenvalues of the embedding merged in pairs.
__global__ void __launch_bounds__(1024) kry_final_kernel(int m, const int* __restrict__ rank,
                                                         const double* __restrict__ d,
                                                         const double* __restrict__ wk,
                                                         double* __restrict__ poles,
                                                         double* __restrict__ weights,
                                                         int32_t* __restrict__ rank_out) {
    __shared__ long long key[1024];  // order-preserving integers (the float64 pipe is narrow)
    __shared__ double se[1024], sw[1024];
    const int t = threadIdx.x, r = *rank, n = m / 2;
    if (t < r) {
        const long long b = __double_as_longlong(d[t]);
        key[t] = b < 0 ? b ^ 0x7fffffffffffffffll : b;
    }
    __syncthreads();
    if (t < r) {
        const long long mine = key[t];
        int at = 0;
        for (int k = 0; k < r; ++k) at += key[k] < mine || (key[k] == mine && k < t);
        se[at] = d[t];
        sw[at] = wk[t];
    }
    __syncthreads();
    if (t < n) {
        const bool on = 2 * t + 1 < r;
        poles[t] = on ? 0.5 * (se[2 * t] + se[2 * t + 1]) : 0.0;
        weights[t] = on ? sw[2 * t] + sw[2 * t + 1] : 0.0;
    }
    if (t == 0 && rank_out) *rank_out = r / 2;
}

}  // namespace

extern "C" cr_status cheb_krylov(cr_ctx* ctx, const double* G, const double* H, int Nm,
                                 double cutoff, int n_out, double* mu_corr_out, double* poles_out,
                                 double* weights_out, int32_t* rank_out) {
    if (!ctx) return CR_EINVAL;
    CR_CHECK_ARG(Nm >= 1 && Nm <= 512, "cheb_krylov: Nm=%d outside [1, 512]", Nm);
    CR_CHECK_ARG(n_out >= 1, "cheb_krylov: n_out < 1");
    CR_CHECK_ARG(G && H && mu_corr_out && poles_out && weights_out, "cheb_krylov: null array");
    const int n = Nm, m = 2 * Nm;
    const size_t mm = (size_t)m * m, nn = (size_t)n * n;
    // workspace (doubles): A0, A1, V0, V1, X, C, Y [m*m]; K, Q [n*n] and the
    // recursion's vectors, complex; d, wk, g0 [m]; norm shares; ints: keep [m],
    // rank, res, barriers
    const size_t need = 7 * mm + 4 * nn + 2 * (size_t)(MOM_CHUNK + 2) * n + 3 * (size_t)m +
                        2 * (size_t)ctx->n_sm + ((size_t)m + 6 + 1) / 2 + 1;
    if (ctx->kry_len < need) {
        // first use at this size: the only allocation outside cr_create
        if (ctx->kry) cudaFree(ctx->kry);
        ctx->kry = nullptr;
        ctx->kry_len = 0;
        if (cudaMalloc((void**)&ctx->kry, need * sizeof(double)) != cudaSuccess)
            return cr_fail(ctx, CR_ENOMEM, "cheb_krylov: workspace");
        ctx->kry_len = need;
    }
    double* w = ctx->kry;
    auto take = [&](size_t k) {
        double* p = w;
        w += k;
        return p;
    };
    JacBufs J;
    J.A[0] = take(mm);
    J.A[1] = take(mm);
    J.V[0] = take(mm);
    J.V[1] = take(mm);
    double* X = take(mm);
    double* C = take(mm);
    double* Y = take(mm);
    zd* K = (zd*)take(2 * nn);
    zd* Q = (zd*)take(2 * nn);
    zd* cv = (zd*)take(2 * (size_t)(MOM_CHUNK + 2) * n);
    double* d = take(m);
    double* wk = take(m);
    double* g0 = take(m);
    J.part = take(2 * (size_t)ctx->n_sm);
    int* keep = (int*)w;
    int* rank = keep + m;
    J.res = rank + 1;
    J.bar = (unsigned*)(rank + 2);
    const unsigned gm = (unsigned)((mm + 255) / 256);
    const unsigned gn = (unsigned)((nn + 255) / 256);
    const dim3 g16((m + 15) / 16, (m + 15) / 16), b16(16, 16), n16((n + 15) / 16, (n + 15) / 16);
    cudaStream_t st = ctx->stream;
    cr_status s;
    // 1. G through its embedding: eigenvalues, kept rank, X = V_kept d^-1/2
    //    (zero-padded to m columns), pseudo-inverse Y = X X^T
    cudaError_t e = cudaMemsetAsync(J.A[0], 0, mm * sizeof(double), st);
    if (e != cudaSuccess) return cr_fail(ctx, CR_ECUDA, "cheb_krylov: %s", cudaGetErrorString(e));
    CR_LAUNCH(ctx, CR_K_OTHER, kry_embed_kernel<<<gn, 256, 0, st>>>(G, n, J.A[0]));
    if ((s = jacobi_launch(ctx, J, m)) != CR_OK) return s;
    CR_LAUNCH(ctx, CR_K_OTHER, kry_keep_kernel<<<1, 1024, 0, st>>>(J, m, cutoff, d, keep, rank));
    CR_LAUNCH(ctx, CR_K_OTHER, kry_x_kernel<<<gm, 256, 0, st>>>(J, m, d, keep, rank, X));
    CR_LAUNCH(ctx, CR_K_OTHER, (kry_gemm_kernel<false, true><<<g16, b16, 0, st>>>(X, X, m, Y)));
    // 2. corrected moments
    CR_LAUNCH(ctx, CR_K_OTHER, kry_pgemm_kernel<<<n16, 256, 0, st>>>(Y, H, n, K));
    CR_LAUNCH(ctx, CR_K_OTHER, kry_pgemm_kernel<<<n16, 256, 0, st>>>(Y, G, n, Q));
    for (int first = 0; first < n_out; first += MOM_CHUNK) {
        MomArgs a;
        a.K = K;
        a.Q = Q;
        a.c = cv;
        a.n = n;
        a.first = first;
        a.count = n_out - first < MOM_CHUNK ? n_out - first : MOM_CHUNK;
        a.bar = J.bar;
        a.status = ctx->d_status;
        e = cudaMemsetAsync(J.bar, 0, 2 * sizeof(unsigned), st);
        if (e == cudaSuccess && first > 0)  // the last two vectors of the previous chunk
            e = cudaMemcpyAsync(cv, cv + (size_t)MOM_CHUNK * n, 2 * (size_t)n * sizeof(zd),
                                cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return cr_fail(ctx, CR_ECUDA, "cheb_krylov: %s", cudaGetErrorString(e));
        const int want = (n + REC_WARPS - 1) / REC_WARPS, grid = want < ctx->n_sm ? want : ctx->n_sm;
        if ((s = coop_launch(ctx, kry_recur_kernel, grid, 32 * REC_WARPS, a, "kry_recur_kernel")) != CR_OK) return s;
        CR_LAUNCH(ctx, CR_K_OTHER, kry_mu_kernel<<<a.count, 128, 0, st>>>((const zd*)G, cv, n, first, mu_corr_out));
    }
    // 3. projected eigenproblem: Hx = X^T Hemb X, diagonalised by the same
    //    Jacobi (padding stays zero)
    CR_LAUNCH(ctx, CR_K_OTHER, kry_g0_kernel<<<(m + 31) / 32, 256, 0, st>>>(G, X, m, g0));
    e = cudaMemsetAsync(C, 0, mm * sizeof(double), st);
    if (e != cudaSuccess) return cr_fail(ctx, CR_ECUDA, "cheb_krylov: %s", cudaGetErrorString(e));
    CR_LAUNCH(ctx, CR_K_OTHER, kry_embed_kernel<<<gn, 256, 0, st>>>(H, n, C));
    CR_LAUNCH(ctx, CR_K_OTHER, (kry_gemm_kernel<false, false><<<g16, b16, 0, st>>>(C, X, m, J.A[1])));
    CR_LAUNCH(ctx, CR_K_OTHER, (kry_gemm_kernel<true, false><<<g16, b16, 0, st>>>(X, J.A[1], m, C)));
    CR_LAUNCH(ctx, CR_K_OTHER, kry_sym_kernel<<<gm, 256, 0, st>>>(C, m, J.A[0]));
    if ((s = jacobi_launch(ctx, J, m)) != CR_OK) return s;
    CR_LAUNCH(ctx, CR_K_OTHER, kry_weight_kernel<<<(m + 7) / 8, 256, 0, st>>>(J, m, g0, rank, d, wk));
    CR_LAUNCH(ctx, CR_K_OTHER,
              kry_final_kernel<<<1, 1024, 0, st>>>(m, rank, d, wk, poles_out, weights_out, rank_out));
    return cr_check_launch(ctx, "cheb_krylov");
}
