// Shared device helpers and the context structure of libchebrbm.
//
// Complex numbers are stored interleaved (re, im); cpx<R> is layout-identical
// to float2 / double2 so that every complex load is one vector load.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <vector>

#include "chebrbm.h"

#define CR_HD __host__ __device__ __forceinline__
#define CR_D __device__ __forceinline__

template <typename R>
struct alignas(2 * sizeof(R)) cpx {
    R x, y;
};

template <typename R> CR_HD cpx<R> mk(R x, R y) { return cpx<R>{x, y}; }
template <typename R> CR_HD cpx<R> operator+(cpx<R> a, cpx<R> b) { return {a.x + b.x, a.y + b.y}; }
template <typename R> CR_HD cpx<R> operator-(cpx<R> a, cpx<R> b) { return {a.x - b.x, a.y - b.y}; }
template <typename R> CR_HD cpx<R> operator-(cpx<R> a) { return {-a.x, -a.y}; }
template <typename R> CR_HD cpx<R> operator*(cpx<R> a, cpx<R> b) {
    return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename R> CR_HD cpx<R> operator*(R s, cpx<R> a) { return {s * a.x, s * a.y}; }
template <typename R> CR_HD cpx<R> conj(cpx<R> a) { return {a.x, -a.y}; }
template <typename R> CR_HD R abs2(cpx<R> a) { return a.x * a.x + a.y * a.y; }
// conj(a) * b
template <typename R> CR_HD cpx<R> cmulc(cpx<R> a, cpx<R> b) {
    return {a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x};
}
template <typename R> CR_HD cpx<R> cdiv(cpx<R> a, cpx<R> b) {
    R d = R(1) / abs2(b);
    return {(a.x * b.x + a.y * b.y) * d, (a.y * b.x - a.x * b.y) * d};
}
template <typename D, typename S> CR_HD cpx<D> ccast(cpx<S> a) { return {(D)a.x, (D)a.y}; }

// Read-only cached complex loads.
CR_D cpx<float> ldg(const cpx<float>* p) {
    float2 v = __ldg((const float2*)p);
    return {v.x, v.y};
}
CR_D cpx<double> ldg(const cpx<double>* p) {
    double2 v = __ldg((const double2*)p);
    return {v.x, v.y};
}

// Math wrappers (CUDA's own functions for each precision).
CR_D float m_exp(float x) { return expf(x); }
CR_D double m_exp(double x) { return exp(x); }
CR_D float m_log(float x) { return logf(x); }
CR_D double m_log(double x) { return log(x); }
CR_D float m_expm1(float x) { return expm1f(x); }
CR_D double m_expm1(double x) { return expm1(x); }
CR_D float m_log1p(float x) { return log1pf(x); }
CR_D double m_log1p(double x) { return log1p(x); }
CR_D float m_atan2(float y, float x) { return atan2f(y, x); }
CR_D double m_atan2(double y, double x) { return atan2(y, x); }
CR_D void m_sincos(float x, float* s, float* c) { sincosf(x, s, c); }
CR_D void m_sincos(double x, double* s, double* c) { sincos(x, s, c); }
CR_D float m_rsqrt(float x) { return rsqrtf(x); }
CR_D double m_rsqrt(double x) { return rsqrt(x); }
CR_D float m_sqrt(float x) { return sqrtf(x); }
CR_D double m_sqrt(double x) { return sqrt(x); }
CR_D float m_cosh(float x) { return coshf(x); }
CR_D double m_cosh(double x) { return cosh(x); }
CR_D float m_sinh(float x) { return sinhf(x); }
CR_D double m_sinh(double x) { return sinh(x); }

template <typename R> CR_D cpx<R> cexp_(cpx<R> z) {
    R e = m_exp(z.x), s, c;
    m_sincos(z.y, &s, &c);
    return {e * c, e * s};
}

// With e = exp(-2|x|) and w = exp(-2 sign(x) z), z = x + iy,
//   |1 + w|^2 = 1 + e^2 + 2 e cos 2y = (1 - e)^2 + 4 e cos^2 y,
// the denominator of tanh z and, under a logarithm, |2 cosh z|^2 e^{-2|x|}.  The
// first sum cancels next to a zero of cosh z: within 3e-4 of one, float32 can
// leave nothing or less than nothing, and an infinite or NaN tanh stops its
// walker and every sum it enters.  The second sum does not cancel (1 - e from
// expm1, cos y itself); it is taken where the first has lost six bits, so that
// values away from a zero keep the bits they had.
template <typename R> struct NearNode {
    R d, om, s, c;  // |1 + w|^2, 1 - e, sin y, cos y
};
template <typename R> CR_D NearNode<R> near_node_terms(R ax, R y, R e) {
    NearNode<R> n;
    n.om = -m_expm1(R(-2) * ax);
    m_sincos(y, &n.s, &n.c);
    n.d = n.om * n.om + R(4) * e * n.c * n.c;
    return n;
}
template <typename R> CR_D bool near_node(R d) { return d < R(0.015625); }

// tanh(x + iy) = (sign(x)(1 - e^2) + 2 i e sin 2y) / (1 + e^2 + 2 e cos 2y),
// e = exp(-2|x|): the identity tanh z = sinh 2z-ish form rescaled by e so
// that nothing overflows for large |x|.  *d: the denominator.
template <typename R> CR_D cpx<R> ctanh_far(cpx<R> z, R* d) {
    R ax = z.x < R(0) ? -z.x : z.x;
    R e = m_exp(R(-2) * ax);
    R e2 = e * e, s, c;
    m_sincos(R(2) * z.y, &s, &c);
    *d = R(1) + e2 + R(2) * e * c;
    R inv = R(1) / *d;
    R re = (R(1) - e2) * inv;
    return {z.x < R(0) ? -re : re, R(2) * e * s * inv};
}
template <typename R> CR_D cpx<R> ctanh_near(cpx<R> z) {
    const R ax = z.x < R(0) ? -z.x : z.x, e = m_exp(R(-2) * ax);
    const NearNode<R> n = near_node_terms(ax, z.y, e);
    const R inv = R(1) / n.d, re = n.om * (R(1) + e) * inv;
    return {z.x < R(0) ? -re : re, R(4) * e * n.s * n.c * inv};
}
template <typename R> CR_D cpx<R> ctanh_(cpx<R> z) {
    R d;
    const cpx<R> t = ctanh_far(z, &d);
    return near_node(d) ? ctanh_near(z) : t;
}

// log(2 cosh z) = s z + log(1 + w), s = sign(Re z), w = exp(-2 s z), |w| <= 1.
// *d: |1 + w|^2.
template <typename R> CR_D cpx<R> clncosh2_far(cpx<R> z, R* d) {
    R sg = z.x < R(0) ? R(-1) : R(1);
    R e = m_exp(R(-2) * sg * z.x), s, c;
    m_sincos(R(-2) * sg * z.y, &s, &c);
    R wr = e * c, wi = e * s;
    const R q = R(2) * wr + e * e;
    *d = R(1) + q;
    return {sg * z.x + R(0.5) * m_log1p(q), sg * z.y + m_atan2(wi, R(1) + wr)};
}
template <typename R> CR_D cpx<R> clncosh2_near(cpx<R> z) {
    const R sg = z.x < R(0) ? R(-1) : R(1), e = m_exp(R(-2) * sg * z.x);
    const NearNode<R> n = near_node_terms(sg * z.x, z.y, e);
    return {sg * z.x + R(0.5) * m_log(n.d),
            sg * z.y + m_atan2(R(-2) * sg * e * n.s * n.c, n.om + R(2) * e * n.c * n.c)};
}

// cosh and sinh of a complex number.
template <typename R> CR_D void ccoshsinh_(cpx<R> z, cpx<R>* ch, cpx<R>* sh) {
    R chx = m_cosh(z.x), shx = m_sinh(z.x), s, c;
    m_sincos(z.y, &s, &c);
    *ch = {chx * c, shx * s};
    *sh = {shx * c, chx * s};
}

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of
// (c0,c1,c2,c3) -> (hi(M1 c2)^c1^k0, lo(M1 c2), hi(M0 c0)^c3^k1, lo(M0 c0)),
// key bumped by the Weyl constants between rounds.
CR_D uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

// Warp reductions.
template <typename R> CR_D R warp_sum(R v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
template <typename R> CR_D cpx<R> warp_sum(cpx<R> v) {
    return {warp_sum(v.x), warp_sum(v.y)};
}
template <typename R> CR_D cpx<R> warp_prod(cpx<R> v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cpx<R> w = {__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o)};
        v = v * w;
    }
    return v;
}

// Device status codes are cr_status values; the first error wins.
CR_D void set_status(int* st, int code) { atomicCAS(st, 0, code); }

// ------------------------------------------------------------ context

// Bond-ratio tables of one RBM (see rbm.cu, build_tables):
//   D[b][j]  = 2 (W_ij - W_jj')         (b = (i, j'), padded columns 0)
//   CS[b][j] = (cosh D, sinh D)          (padded columns 1 and 0)
//   ChT/ShT  = cosh D, sinh D transposed, [Mp][Nb]
//   ea[b][0] = exp(-2 (a_i - a_j')), ea[b][1] = exp(+2 (a_i - a_j'))
struct cr_tables {
    void* D;    // slot 0
    void* CS;   // slot 0
    void* ChT;  // slot 1
    void* ShT;  // slot 1
    void* ea;
};

struct cr_ktimer {
    int kid;                 // armed kernel family, -1 when off
    int cap, count;
    cudaEvent_t* ev;         // [2 * cap]: start, stop pairs
};

struct cr_ctx {
    int Lx, Ly, N, M, Mp, Nb, P;
    double J;
    cr_prec prec;
    int max_walkers, flags;
    int n_chunks;            // walker chunks of the reductions (<= max_chunks)
    int red_rows;            // chunk rows allocated (>= max_chunks), used while !chunks_set
    bool chunks_set;         // n_chunks was asked for
    int max_chunks;          // chunks the partial-row workspace holds
    int n_sm;                // multiprocessors of the device
    cudaStream_t stream;
    char err[512];

    int* d_status;           // device status word
    int2* d_bonds;           // [Nb]
    cr_tables tab[2];        // 0: sampler, 1: local target (float64 contexts)
    uint16_t* sw_list;       // accepted moves of a sweep launch [maxB][sweep_list_cap], or null
    int* sw_count;           // their number [maxB], or null
    void* xtab;              // exchange table (float32 contexts)
    void* xout;              // xsum_out [maxB] (float32 contexts)
    void* theta_tmp;         // [maxB][M]
    void* lp_tmp;            // [2][maxB]
    void* u_tmp;             // [maxB]
    double* partial;         // [red_rows][P + 2 + M] complex, context precision
    double* red;             // [3][P + 2 + M] complex128 reduced sums
    double* F;               // [P] complex128
    double* cg;              // x, r, p, Ap, 1 / diag: [5][P] complex128
    void* p_lo;              // [P] context precision
    double* cgpart;          // per-CTA dot products of a CG step: p.Ap [ceil(P/32)],
                             // r.r and r.z [2][ceil(P/64)]
    double* scal;            // scalars [64]
    double* S;               // [P][P] complex128 (explicit S only)
    double* kry;             // Krylov workspace
    size_t kry_len;
    void* Lf;                // Cholesky factor, factor precision, padded (explicit S only)
    void* chol_x;            // inverses of its 512 x 512 diagonal blocks
    unsigned char* chol_pl;  // bf16 operands of the trailing update (mixed only)
    unsigned char* Xt;       // bf16 operands of the explicit S (mixed explicit S only)
    float* spair_g;          // its pair sums (float32 in mixed contexts, else float64)
    // Krylov Gram on the tensor cores (mixed): sized on first use
    unsigned char* gram_x;   // bf16 planes of the B and HB columns
    size_t gram_x_cap;
    double* gram_part;       // per-segment sums
    size_t gram_part_cap;
    int2* gram_tiles;
    size_t gram_tiles_cap;
    int gram_key;            // 2 Nm + (H wanted) of the tile list held, 0 if none
    // estimator sums on the tensor cores (mixed contexts; allocated at creation)
    unsigned char* ored_x;   // bf16 planes of Y0, Y1 and A = sigma
    double* ored_part;       // per-segment sums, border sums per 512 walkers
    int2* ored_tiles;
    int ored;                // 1 when the path is set up
    void* lp_work;           // linear-prediction scratch (sized on first use)
    size_t lp_work_cap;
    long long n_launches;    // kernels launched so far
    cr_ktimer kt;
    // fused CG solve (cg_fused.cu; mixed contexts with N, M <= 256)
    int fcg;                 // 1 when the fused solve covers this context
    unsigned char* fcg_a1;   // sigma operand tiles of the O v contraction
    unsigned char* fcg_b2;   // sigma^T operand chunks of the O^dag w contraction
    unsigned char* fcg_v2;   // bf16 planes of the W part of p
    size_t fcg_v2plane;
    void* fcg_vab;           // float32 a- and b-parts of p [N + M]
    void* fcg_part;          // partial rows, complex float32 [n_sm][P]
    double* fcg_psc;         // scalar partials [n_sm][8]
    unsigned* fcg_bar;       // grid-barrier counter and abort flag
    int fcg_ctas;            // CTAs of the fused CG (0: one per SM)
    cudaEvent_t ev_fork, ev_join;  // batched runs: fork from / join into the caller's stream
};

// What xsum_kernel (exchange.cu) leaves per configuration: with
// lam = base + ex ln 2, the exchanged amplitudes of the antiparallel bonds sum to
// e^lam (off + slow), and weighted with s_i d_b of the probe to
// e^lam (offd + slow_d).  float4: (re hi, re lo, im hi, im lo).
struct alignas(16) xsum_out {
    float4 off, offd, base;
    int nanti, ex, pad[2];
    cpx<double> slow, slow_d;
};

static inline int rsize(const cr_ctx* c) { return c->prec == CR_FP64 ? 8 : 4; }

cr_status cr_fail(cr_ctx* c, cr_status s, const char* fmt, ...);
bool cr_kt_begin(cr_ctx* c, int kid);
void cr_kt_end(cr_ctx* c);

// Launch a kernel through the context: counts it and, when its family is
// armed for timing, brackets it with CUDA events on the context stream.
#define CR_LAUNCH(c, kid, ...)                    \
    do {                                          \
        const bool cr_kt_on_ = cr_kt_begin(c, kid); \
        __VA_ARGS__;                              \
        if (cr_kt_on_) cr_kt_end(c);              \
        ++(c)->n_launches;                        \
    } while (0)
#define CR_K_OTHER (-2)
cr_status cr_check_launch(cr_ctx* c, const char* what);

// Explicit S and the direct solve (spair.cu, chol.cu).  Float64 contexts up
// to CHOL_SMALL_P parameters solve once in float64; every other explicit-S
// context refines the solution.
#define CHOL_SMALL_P 2048
bool chol_refined(const cr_ctx* c);
void chol_sizes(const cr_ctx* c, size_t* factor, size_t* inverses, size_t* planes);
size_t chol_cgpart_len(const cr_ctx* c);
cr_status chol_prepare(cr_ctx* c);
cr_status chol_factor(cr_ctx* c);
cr_status chol_refine_solve(cr_ctx* c, const double* F, int maxit);
cr_status chol_plain_solve(cr_ctx* c, const double* F);
size_t chol64_diag_bytes(int P);
cr_status chol64_prepare(cr_ctx* c);
cr_status chol64_factor(cr_ctx* c, double* A, double* D);
void chol64_solve(cr_ctx* c, const double* A, const double* D, double* r, double* y, double* d,
                  const double* skip);
// Device scratch that grows on demand (once-per-sequence calls only): frees
// and reallocates *p when cap < need; CR_ENOMEM with the caller's name.
cr_status cr_grow(cr_ctx* c, void** p, size_t* cap, size_t need, const char* who);
void ored_sizes(const cr_ctx* c, size_t* x_bytes, size_t* part_bytes, std::vector<int2>* tiles);
cr_status launch_oreduce_tc(cr_ctx* c, const int8_t* spins, const void* T, const void* g, int B,
                            double* redR, double* redO);
cr_status launch_gram_tc(cr_ctx* c, const void* Bm, const void* HBm, int Nm, int B, int ld,
                         double* G, double* H);
cr_status launch_sbuild(cr_ctx* c, const int8_t* spins, const void* T, int B, const double* redO,
                        double shift);

// Fused CG solve (cg_fused.cu).
bool fcg_supported(const cr_ctx* c);
void fcg_sizes(const cr_ctx* c, size_t* a1, size_t* b2, size_t* v2plane, size_t* part);
cr_status fcg_prepare(cr_ctx* c);
cr_status launch_cg_fused(cr_ctx* c, const int8_t* spins, const void* T, int B, const double* redO,
                          double shift, double tol, int maxit, int precond, int apply_only,
                          const double* v_in, void* u_out);

int sweep_list_cap(const cr_ctx* c);
bool sweep_takes_lists(const cr_ctx* c);  // for any number of walkers and proposals
cr_status sweep_prepare(cr_ctx* c);

// Sums over exchanged amplitudes in float32 (exchange.cu).
size_t xsum_table_bytes(const cr_ctx* c);
cr_status xsum_prepare(cr_ctx* c);
cr_status launch_xsum(cr_ctx* c, const void* params, const int8_t* spins, const void* theta, int n,
                      int probe, double qx, double qy, xsum_out* out);

// Tables for a state (rbm.cu); planar: CS as [b][cosh row, sinh row].
cr_status build_tables(cr_ctx* c, const void* params, int slot, int planar = 0);
// theta / log psi of an RBM at a walker batch (rbm.cu).
cr_status launch_logpsi(cr_ctx* c, const void* params, const int8_t* spins, int B, void* theta,
                        void* logpsi);

#define CR_CHECK_ARG(cond, ...)                                  \
    do {                                                         \
        if (!(cond)) return cr_fail(ctx, CR_EINVAL, __VA_ARGS__); \
    } while (0)
