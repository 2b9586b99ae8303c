// The RBM ansatz of Sec. I: theta = b + sigma W, log psi, bond-ratio tables,
// and the explicit log-derivatives of Sec. III.
#include "common.cuh"

// ------------------------------------------------------------------ tables
//
// Exchanging the antiparallel spins of bond (i, i') with s = sigma_i changes
// theta_m by -s D_m, D_m = 2 (W_im - W_i'm), so
//   cosh(theta_m - s D_m) / cosh(theta_m) = cosh D_m - s tanh(theta_m) sinh D_m
// and the visible factor by exp(-s 2 (a_i - a_i')).  The tables hold D, cosh D,
// sinh D per (bond, hidden unit), padded to Mp columns with the neutral
// values (0, 1, 0), and exp(-/+ 2 (a_i - a_i')) per bond: cosh and sinh
// interleaved, or in a row each (planar), for the sampler (slot 0), transposed
// for the float64 local target (slot 1).
template <typename R>
__global__ void tables_kernel(const cpx<R>* __restrict__ prm, const int2* __restrict__ bonds, int N,
                              int M, int Mp, int Nb, cpx<R>* D, cpx<R>* CS, cpx<R>* ChT, cpx<R>* ShT,
                              cpx<R>* ea, int planar) {
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= Nb * Mp) return;
    int b = idx / Mp, m = idx % Mp;
    int2 bd = bonds[b];
    cpx<R> d = {R(0), R(0)}, ch = {R(1), R(0)}, sh = {R(0), R(0)};
    if (m < M) {
        const cpx<R>* W = prm + N + M;
        cpx<R> wi = W[(size_t)bd.x * M + m], wj = W[(size_t)bd.y * M + m];
        d = R(2) * (wi - wj);
        ccoshsinh_(d, &ch, &sh);
    }
    if (CS) {
        D[idx] = d;
        const size_t at = planar ? (size_t)2 * Mp * b + m : 2 * (size_t)idx;
        CS[at] = ch;
        CS[at + (planar ? Mp : 1)] = sh;
    } else {
        ChT[(size_t)m * Nb + b] = ch;
        ShT[(size_t)m * Nb + b] = sh;
    }
    if (m == 0) {
        cpx<R> da = R(2) * (prm[bd.x] - prm[bd.y]);
        ea[2 * b] = cexp_(-da);
        ea[2 * b + 1] = cexp_(da);
    }
}

template <typename R>
static cr_status build_tables_t(cr_ctx* c, const void* params, int slot, int planar) {
    const cr_tables& t = c->tab[slot];
    int n = c->Nb * c->Mp;
    CR_LAUNCH(c, CR_K_OTHER, tables_kernel<R><<<(n + 255) / 256, 256, 0, c->stream>>>(
        (const cpx<R>*)params, c->d_bonds, c->N, c->M, c->Mp, c->Nb, (cpx<R>*)t.D, (cpx<R>*)t.CS,
        (cpx<R>*)t.ChT, (cpx<R>*)t.ShT, (cpx<R>*)t.ea, planar));
    return cr_check_launch(c, "tables_kernel");
}

cr_status build_tables(cr_ctx* c, const void* params, int slot, int planar) {
    return c->prec == CR_FP64 ? build_tables_t<double>(c, params, slot, planar)
                              : build_tables_t<float>(c, params, slot, planar);
}

// ------------------------------------------------------ theta and log psi
//
// theta = b + sigma W for a block of walkers, then per walker
//   MODE_LOGPSI: theta_out = theta, out = a.sigma + sum_j log 2cosh theta_j
//   MODE_MATVEC: out = v_a.sigma + sum_j T_j (v_b + sigma V_W)_j, i.e. O v
//                with O_a = sigma, O_b = T, O_W = sigma (x) T (Sec. III).
//
// A warp takes TH_W walkers (per group of LJ lanes) and all their hidden units,
// JW per lane, so the sums over hidden units end in a few shuffles; M > LJ JW
// takes several passes.  Sites come 16 at a time through shared memory (W
// rows by cp.async, signs converted once), double-buffered: per site a lane
// reads TH_W signs (a broadcast) and JW weights for 2 TH_W JW multiply-adds.
// JW and LJ are the smallest that hold M, so few lanes multiply padding; TH_W
// is 1 to 8 by the number of walkers (launch_theta_t).
//
// Bound by the FMA pipe and, for log psi, by the exponential, sine and cosine
// of every theta; log(2 cosh) of two units shares one logarithm and one
// angle.  16 x 16 lattice, 65536 walkers: 547 -> 490 us (one block of 128
// threads per 16 walkers before, weights read from L2 by every block); M = 72:
// 921 -> 530 us; float64 at N = M = 12: 130 -> 15 us.  Packed pairs of
// multiply-adds did not help (527 us).
//
// The sum over units is of log cosh; M log 2, which would be most of it where
// theta is small, comes in with the last level, whose rounding errors are kept.
// With log 2cosh summed plainly the error depends on where the layout's partial
// sums pass powers of two.  Error of float32 against 64 bits, |theta| < 0.1, 48
// sites with 96 units: 3.2e-6 with a sum of 128 threads, 3.5e-6 with this layout
// and plain sums, 2.3e-6 so (the rounding of the result alone 2.2e-6); 64 sites
// with 128 units 4.2e-6, 3.6e-6, 2.3e-6.  16 x 16 lattice, 65536 walkers: 486 us
// with plain sums, 490 so.
enum { MODE_LOGPSI = 0, MODE_MATVEC = 1 };

namespace {

constexpr int TH_KC = 16;  // sites per stage
constexpr int TH_WARPS = 8;

CR_D void cp_async8(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
CR_D void cp_async_all() { asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory"); }

// Unit q of a lane: pairs of neighbours first (one 16-byte access of a float
// row), a single unit last when JW is odd.
template <int LJ, int JW> CR_D int unit_of(int l, int q) {
    return q < (JW & ~1) ? 2 * l + (q & 1) + 2 * LJ * (q >> 1) : LJ * (JW - 1) + l;
}

// near_node_terms as a call: inlined, its rare branch makes theta_kernel spill.
template <typename R> __device__ __noinline__ NearNode<R> near_node_call(R ax, R y, R e) {
    return near_node_terms(ax, y, e);
}

// log(cosh z) summed over the lane's units: s z and (1 + w) / 2 of each (|w| <=
// 1, so two arguments add up without a branch cut), the logarithm of two units'
// product at once.
template <typename R> CR_D void lncosh_parts(cpx<R> z, cpx<R>* lin, cpx<R>* half) {
    const R sg = z.x < R(0) ? R(-1) : R(1);
    const R e = m_exp(R(-2) * sg * z.x), h = R(0.5) * e;
    R s, c;
    m_sincos(R(-2) * sg * z.y, &s, &c);
    *lin = *lin + sg * z;
    *half = {R(0.5) + h * c, h * s};
    if (abs2(*half) < R(0.015625 / 4)) {  // near_node of twice that
        const NearNode<R> n = near_node_call(sg * z.x, z.y, e);
        *half = {R(0.5) * n.om + e * n.c * n.c, -sg * e * n.s * n.c};
    }
}

// s + v, its rounding error added to *e (Knuth's two-sum, TAOCP 2, 4.2.2).
template <typename R> CR_D R add_exact(R s, R v, R* e) {
    const R t = s + v, b = t - s;
    *e += (s - (t - b)) + (v - b);
    return t;
}

}  // namespace

template <typename R, int LJ, int JW, int TH_W, int MODE>
__global__ void __launch_bounds__(32 * TH_WARPS, 2) theta_kernel(const cpx<R>* __restrict__ prm,
                                                              const int8_t* __restrict__ spins, int B,
                                                              int N, int M, cpx<R>* __restrict__ theta_out,
                                                              cpx<R>* __restrict__ out,
                                                              const cpx<R>* __restrict__ T,
                                                              const double* __restrict__ skip,
                                                              R ln2_hi, R ln2_lo) {
    if (skip && *skip != 0.0) return;  // converged CG: nothing left to do
    constexpr int NG = 32 / LJ, WB = TH_W * NG * TH_WARPS, JB = LJ * JW, NT = 32 * TH_WARPS;
    __shared__ __align__(16) R sg[2][TH_KC][WB];
    __shared__ __align__(16) cpx<R> wv[2][TH_KC][JB];
    const int t = threadIdx.x, lane = t & 31, l = lane & (LJ - 1);
    const int wl = ((t >> 5) * NG + lane / LJ) * TH_W;  // first walker of the group in the block
    const int w0 = blockIdx.x * WB;
    const cpx<R>* a = prm;
    const cpx<R>* b = prm + N;
    const cpx<R>* W = prm + N + M;
    cpx<R> part[TH_W];
#pragma unroll
    for (int w = 0; w < TH_W; ++w) part[w] = {R(0), R(0)};
    // 4 signs of a walker are one aligned word (spins may start at any byte)
    const bool quad = (N & 3) == 0 && ((uintptr_t)spins & 3) == 0;
    for (int jb = 0; jb < M; jb += JB) {
        cpx<R> acc[TH_W][JW];
#pragma unroll
        for (int q = 0; q < JW; ++q) {
            const int j = jb + unit_of<LJ, JW>(l, q);
            const cpx<R> bj = j < M ? b[j] : cpx<R>{R(0), R(0)};
#pragma unroll
            for (int w = 0; w < TH_W; ++w) acc[w][q] = bj;
        }
        // stage of sites i0 .. i0 + 15 into buffer s: weights, then signs
        auto fetch = [&](int i0, int s) {
            for (int e = t; e < TH_KC * JB; e += NT) {
                const int k = e / JB, j = e % JB;
                cpx<R>* dst = &wv[s][k][j];
                if (i0 + k < N && jb + j < M) {
                    const cpx<R>* src = W + (size_t)(i0 + k) * M + jb + j;
                    cp_async8(dst, src);
                    if (sizeof(R) == 8) cp_async8((char*)dst + 8, (const char*)src + 8);
                } else {
                    *dst = {R(0), R(0)};
                }
            }
            for (int e = t; e < WB * (TH_KC / 4); e += NT) {
                const int w = e % WB, k = 4 * (e / WB);
                const int8_t* src = spins + (size_t)(w0 + w) * N + i0 + k;
                char4 v = make_char4(0, 0, 0, 0);
                if (w0 + w < B) {
                    if (quad) {
                        if (i0 + k < N) v = *reinterpret_cast<const char4*>(src);
                    } else {
                        if (i0 + k < N) v.x = src[0];
                        if (i0 + k + 1 < N) v.y = src[1];
                        if (i0 + k + 2 < N) v.z = src[2];
                        if (i0 + k + 3 < N) v.w = src[3];
                    }
                }
                sg[s][k][w] = R(v.x);
                sg[s][k + 1][w] = R(v.y);
                sg[s][k + 2][w] = R(v.z);
                sg[s][k + 3][w] = R(v.w);
            }
        };
        __syncthreads();
        fetch(0, 0);
        cp_async_all();
        __syncthreads();
        for (int i0 = 0, s = 0; i0 < N; i0 += TH_KC, s ^= 1) {
            if (i0 + TH_KC < N) fetch(i0 + TH_KC, s ^ 1);
            const int kn = min(TH_KC, N - i0);
#pragma unroll 4
            for (int k = 0; k < kn; ++k) {
                R sv[TH_W];
                cpx<R> wk[JW];
#pragma unroll
                for (int w = 0; w < TH_W; ++w) sv[w] = sg[s][k][wl + w];
#pragma unroll
                for (int q = 0; q < JW; ++q) wk[q] = wv[s][k][unit_of<LJ, JW>(l, q)];
#pragma unroll
                for (int w = 0; w < TH_W; ++w)
#pragma unroll
                    for (int q = 0; q < JW; ++q) {
                        acc[w][q].x = fma(sv[w], wk[q].x, acc[w][q].x);
                        acc[w][q].y = fma(sv[w], wk[q].y, acc[w][q].y);
                    }
            }
            if (jb == 0 && l < kn) {  // a.sigma: a lane per site of the stage
                const cpx<R> ai = a[i0 + l];
#pragma unroll
                for (int w = 0; w < TH_W; ++w) part[w] = part[w] + sg[s][l][wl + w] * ai;
            }
            cp_async_all();
            __syncthreads();
        }
#pragma unroll
        for (int w = 0; w < TH_W; ++w) {
            const int ww = w0 + wl + w;
            if (ww >= B) break;
            cpx<R>* to = MODE == MODE_LOGPSI && theta_out ? theta_out + (size_t)ww * M : nullptr;
            cpx<R> one[2];
#pragma unroll
            for (int q = 0; q < JW; ++q) {
                const int j = jb + unit_of<LJ, JW>(l, q);
                const cpx<R> th = acc[w][q];
                if (MODE == MODE_MATVEC) {
                    if (j < M) part[w] = part[w] + T[(size_t)ww * M + j] * th;
                    continue;
                }
                one[q & 1] = {R(1), R(0)};
                if (j < M) {
                    if (to) to[j] = th;
                    lncosh_parts(th, &part[w], &one[q & 1]);
                }
                if ((q & 1) || q == JW - 1) {
                    const cpx<R> p = (q & 1) ? one[0] * one[1] : one[0];
                    part[w] = part[w] + cpx<R>{R(0.5) * m_log(abs2(p)), m_atan2(p.y, p.x)};
                }
            }
        }
    }
#pragma unroll
    for (int w = 0; w < TH_W; ++w) {
        cpx<R> v = part[w];
#pragma unroll
        for (int o = LJ / 2; o > 1; o >>= 1)
            v = v + cpx<R>{__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o)};
        const cpx<R> v2 = {__shfl_xor_sync(0xffffffffu, v.x, 1), __shfl_xor_sync(0xffffffffu, v.y, 1)};
        part[w] = v + v2;
        if (MODE == MODE_LOGPSI) {
            R e = ln2_lo;
            const R t = add_exact(add_exact(v.x, v2.x, &e), ln2_hi, &e);
            part[w].x = isfinite(e) ? t + e : t;  // an infinite sum has no remainder
        }
    }
#pragma unroll
    for (int w = 0; w < TH_W; ++w)
        if (l == 0 && w0 + wl + w < B) out[w0 + wl + w] = part[w];
}

template <typename R, int TW, int MODE>
static cr_status launch_theta_w(cr_ctx* c, const void* params, const int8_t* spins, int B,
                                void* theta, void* out, const void* T, const double* skip) {
#define LAUNCH(LJ, JW)                                                                           \
    {                                                                                            \
        constexpr int WB = TW * (32 / LJ) * TH_WARPS;                                            \
        CR_LAUNCH(c, (MODE == MODE_LOGPSI ? CR_KERNEL_THETA : CR_KERNEL_OV),                     \
                  (theta_kernel<R, LJ, JW, TW, MODE>                                             \
                   <<<(B + WB - 1) / WB, 32 * TH_WARPS, 0, c->stream>>>(                         \
                       (const cpx<R>*)params, spins, B, c->N, c->M, (cpx<R>*)theta,              \
                       (cpx<R>*)out, (const cpx<R>*)T, skip, hi, lo)));                          \
    }
    // units per lane and pass: the fewest padded units (float64: registers for two)
    const int M = c->M;
    // M log 2 as two words; log 2 in two doubles
    const double L = 0.6931471805599453, ln2 = M * L, rest = std::fma((double)M, L, -ln2) + M * 2.3190468138462996e-17;
    const R hi = (R)ln2, lo = (R)(ln2 - (double)hi + rest);
    if (M <= 16) LAUNCH(16, 1)
    else if (M <= 32) LAUNCH(32, 1)
    else if (M <= 64 || sizeof(R) == 8) LAUNCH(32, 2)
    else {
        const int passes = (M + 127) / 128, per = (M + passes - 1) / passes;
        if (per <= 96) LAUNCH(32, (sizeof(R) == 8 ? 2 : 3))
        else LAUNCH(32, (sizeof(R) == 8 ? 2 : 4))
    }
#undef LAUNCH
    return cr_check_launch(c, "theta_kernel");
}

// Walkers per group (TH_W) of a launch over B walkers.  A block is one unit of
// time on its SM, two share one: with nb blocks for the fullest SM the launch
// takes nb / 2 pairs and perhaps a single, and the TH_W with the least total is
// taken.  The two tables are a block's time alone and a pair's, us at N = M =
// 256; they keep their order at other sizes (N = 64 with 33 and 128 units, N =
// 100 with 100, N = 36 with 72).  B = 3000 at N = M = 256: 97 us with the
// smallest count that gave every SM a block, now 56; 10000: 133, now 107; the
// values do not depend on the choice.  Float64 is bound by its pipe: one walker
// a group is the best or equal up to 8192 walkers (64 sites, 33 units: 224 us,
// four 254), and the weights it reads again are hidden.
template <typename R, int MODE>
static cr_status launch_theta_t(cr_ctx* c, const void* params, const int8_t* spins, int B,
                                void* theta, void* out, const void* T, const double* skip) {
    if (B == 0) return CR_OK;
    if constexpr (sizeof(R) == 8) return launch_theta_w<R, 1, MODE>(c, params, spins, B, theta, out, T, skip);
    static const struct { int tw, single, pair; } shapes[] = {{1, 42, 64},  {2, 43, 66},  {4, 56, 84},
                                                              {5, 63, 107}, {6, 70, 110}, {8, 90, 144}};
    const int groups = TH_WARPS * (c->M <= 16 ? 2 : 1);
    int tw = 1;
    long long best = -1;
    for (const auto& q : shapes) {
        const long long blocks = ((long long)B + q.tw * groups - 1) / (q.tw * groups);
        const long long nb = (blocks + c->n_sm - 1) / c->n_sm;
        const long long cost = nb / 2 * q.pair + (nb & 1) * q.single;
        if (best < 0 || cost < best) {
            best = cost;
            tw = q.tw;
        }
    }
#define TW(K) return launch_theta_w<R, K, MODE>(c, params, spins, B, theta, out, T, skip)
    switch (tw) {
        case 1: TW(1);
        case 2: TW(2);
        case 4: TW(4);
        case 5: TW(5);
        case 6: TW(6);
        default: TW(8);
    }
#undef TW
}

cr_status launch_logpsi(cr_ctx* c, const void* params, const int8_t* spins, int B, void* theta,
                        void* logpsi) {
    return c->prec == CR_FP64
               ? launch_theta_t<double, MODE_LOGPSI>(c, params, spins, B, theta, logpsi, nullptr,
                                                     nullptr)
               : launch_theta_t<float, MODE_LOGPSI>(c, params, spins, B, theta, logpsi, nullptr,
                                                    nullptr);
}

// u_s = sum_k O_k(s) v_k for the structured O of Sec. III.
cr_status launch_ov(cr_ctx* c, const void* v, const int8_t* spins, int B, const void* T, void* u,
                    const double* skip) {
    return c->prec == CR_FP64
               ? launch_theta_t<double, MODE_MATVEC>(c, v, spins, B, nullptr, u, T, skip)
               : launch_theta_t<float, MODE_MATVEC>(c, v, spins, B, nullptr, u, T, skip);
}

// ------------------------------------------------------------- logderiv

template <typename R>
__global__ void tanh_kernel(const cpx<R>* __restrict__ theta, size_t n, cpx<R>* __restrict__ out) {
    size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < n) out[idx] = ctanh_(theta[idx]);
}

template <typename R>
__global__ void o_explicit_kernel(const int8_t* __restrict__ spins, const cpx<R>* __restrict__ theta,
                                  int B, int N, int M, int P, cpx<R>* __restrict__ O) {
    size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)B * P) return;
    int s = (int)(idx / P), k = (int)(idx % P);
    cpx<R> v;
    if (k < N) {
        v = {R(spins[(size_t)s * N + k]), R(0)};
    } else if (k < N + M) {
        v = ctanh_(theta[(size_t)s * M + (k - N)]);
    } else {
        int i = (k - N - M) / M, j = (k - N - M) % M;
        v = R(spins[(size_t)s * N + i]) * ctanh_(theta[(size_t)s * M + j]);
    }
    O[idx] = v;
}

template <typename R>
static cr_status logderiv_t(cr_ctx* ctx, const int8_t* spins, const void* theta, int B,
                            void* tanh_out, void* O_out) {
    if (tanh_out) {
        size_t n = (size_t)B * ctx->M;
        CR_LAUNCH(ctx, CR_K_OTHER, tanh_kernel<R><<<(unsigned)((n + 255) / 256), 256, 0, ctx->stream>>>(
            (const cpx<R>*)theta, n, (cpx<R>*)tanh_out));
    }
    if (O_out) {
        size_t n = (size_t)B * ctx->P;
        CR_LAUNCH(ctx, CR_K_OTHER, o_explicit_kernel<R><<<(unsigned)((n + 255) / 256), 256, 0, ctx->stream>>>(
            spins, (const cpx<R>*)theta, B, ctx->N, ctx->M, ctx->P, (cpx<R>*)O_out));
    }
    return cr_check_launch(ctx, "logderiv");
}

cr_status logderiv_impl(cr_ctx* ctx, const int8_t* spins, const void* theta, int B, void* tanh_out,
                        void* O_out) {
    return ctx->prec == CR_FP64 ? logderiv_t<double>(ctx, spins, theta, B, tanh_out, O_out)
                                : logderiv_t<float>(ctx, spins, theta, B, tanh_out, O_out);
}

// --------------------------------------------------------------- C ABI

extern "C" cr_status rbm_logpsi(cr_ctx* ctx, const cr_state* st, const int8_t* spins, int B,
                                void* theta_out, void* logpsi_out) {
    if (!ctx) return CR_EINVAL;
    CR_CHECK_ARG(st && st->params, "rbm_logpsi: null state");
    CR_CHECK_ARG(B >= 0 && B <= ctx->max_walkers, "rbm_logpsi: B=%d outside [0, %d]", B,
                 ctx->max_walkers);
    if (B == 0) return CR_OK;
    CR_CHECK_ARG(spins && logpsi_out, "rbm_logpsi: null spins or output");
    return launch_logpsi(ctx, st->params, spins, B, theta_out, logpsi_out);
}

extern "C" cr_status logderiv(cr_ctx* ctx, const cr_state* st, const int8_t* spins,
                              const void* theta, int B, void* tanh_out, void* O_out) {
    if (!ctx) return CR_EINVAL;
    CR_CHECK_ARG(st && st->params, "logderiv: null state");
    CR_CHECK_ARG(B >= 0 && B <= ctx->max_walkers, "logderiv: B=%d outside [0, %d]", B,
                 ctx->max_walkers);
    if (B == 0) return CR_OK;
    CR_CHECK_ARG(spins && theta, "logderiv: null spins or theta");
    return logderiv_impl(ctx, spins, theta, B, tanh_out, O_out);
}

// ------------------------------------------------- start of projection step n
//
// The recursion of Sec. III fits RBM_n from a starting point the paper leaves
// open.  RBM_1 starts from psi with a_0 += i pi/2: e^{i pi sigma_0 / 2} =
// i sigma_0, so that RBM equals 2i S^z_0 psi exactly, a state with weight on
// H' S^z_q psi; RBM_n (n >= 2) starts from RBM_{n-1} (warm start).
template <typename R>
__global__ void init_params_kernel(const cpx<R>* __restrict__ src, int P, int shift_a0,
                                   cpx<R>* __restrict__ out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= P) return;
    cpx<R> v = src[k];
    if (shift_a0 && k == 0) v.y += R(1.5707963267948966);  // + i pi/2
    out[k] = v;
}

extern "C" cr_status cheb_init_params(cr_ctx* ctx, int n, const void* psi, const void* prev,
                                      void* out) {
    if (!ctx) return CR_EINVAL;
    CR_CHECK_ARG(n >= 1, "cheb_init_params: n must be >= 1");
    CR_CHECK_ARG(out && (n == 1 ? psi != nullptr : prev != nullptr),
                 "cheb_init_params: null parameter vector");
    const void* src = n == 1 ? psi : prev;
    const int P = ctx->P, g = (P + 255) / 256;
    if (ctx->prec == CR_FP64)
        CR_LAUNCH(ctx, CR_K_OTHER, init_params_kernel<double><<<g, 256, 0, ctx->stream>>>(
                                       (const cpx<double>*)src, P, n == 1, (cpx<double>*)out));
    else
        CR_LAUNCH(ctx, CR_K_OTHER, init_params_kernel<float><<<g, 256, 0, ctx->stream>>>(
                                       (const cpx<float>*)src, P, n == 1, (cpx<float>*)out));
    return cr_check_launch(ctx, "init_params_kernel");
}
