// The whole matrix-free CG solve of the natural-gradient update (Sec. III),
//   (S + lambda I) x = F,   S v = (1/B) sum_s conj(O_s) ((O_s - Obar) . v),
// in ONE persistent kernel for CR_MIXED contexts: one CTA per SM, a bounded
// grid barrier between phases, the two O-contractions on the tensor cores
// (tcgen05, bf16 splits, float32 accumulation in TMEM) and the CG vectors in
// float64.
//
// With O_s = [sigma_s | T_s | sigma_s (x) T_s] (T = tanh theta) and
// v = [va | vb | V]:
//   u_s  = (O_s . v) = sigma_s . va + sum_j T_sj (vb_j + (sigma V)_sj)
//   w_s  = u_s - ubar,   ubar = Obar . v = mean_s u_s
//   S v  = (1/B) [ sum_s sigma_s w_s | sum_s conj(T_s) w_s |
//                  sum_s sigma_s (x) conj(T_s) w_s ]
// Centering u with ubar (known from Obar . p, a P-dot product of the
// previous phase) makes O^dag w the covariance form directly: no
// cancellation between O^dag u / B and Obar^* ubar, and
//   p^dag (S + lambda I) p = (1/B) sum_s |w_s|^2 + lambda |p|^2
// comes from the walker phase, which saves the grid barrier of a separate
// p . Ap reduction.  The CG is Hestenes-Stiefel from x = 0, optionally with
// the Jacobi preconditioner diag(S) + lambda, stopping at |r| <= tol |F|.
//
// The CG is the Chronopoulos-Gear form of Hestenes-Stiefel CG (Chronopoulos
// and Gear, J. Comput. Appl. Math. 25, 1989): with u = M^-1 r and w = A u,
//   gamma = (r, u), delta = (u, A u), beta = gamma / gamma_prev,
//   alpha = gamma / (delta - beta gamma / alpha_prev),
//   p = u + beta p, s = w + beta s (s = A p), x += alpha p, r -= alpha s,
// the same iterates as the textbook recursion in exact arithmetic, with both
// inner products of an iteration formed together: delta comes out of the
// walker phase (the centred form above) and gamma from the slice phase, so
// an iteration needs two grid barriers.  Should the recurrence's (p, A p)
// lose positivity to rounding, the iteration restarts (beta = 0).
//
// Per CG iteration:
//   W   walker phase (each CTA its walker range), the product A u:
//       W1: D1 = sigma V on the tensor cores (A = sigma tile [128 walkers x
//           32 sites] exact in bf16, B = three bf16 planes of V [128 columns
//           (Re/Im of 64 hidden units) x 32 sites], streamed by bulk copies
//           through a 4-stage ring; two walker tiles share a stage of V where
//           a CTA has them), then u_s from D1 (TMEM) and T (global);
//       W2: D2^T = Y^T sigma on the tensor cores (A = three bf16 planes of
//           Y_sn = (conj(T_sj) w_s).{re,im} [128 columns x 32 walkers],
//           formed by the compute warps, B = sigma^T [sites x 32 walkers]),
//           accumulated over the CTA's walkers, then written as the CTA's
//           partial row; the a- and b-sums on the CUDA cores.
//   |   grid barrier
//   S   each CTA its slice of P: A u from the partial rows (Kahan-compensated
//       float32 sums in a fixed order), alpha, beta, the updates of p, s, x,
//       r, the new u and its bf16 planes, the partial inner products.
//   |   grid barrier
// The convergence test |r| <= tol |F| opens each walker phase; the operand
// copies of that phase start before it, the MMAs after it.
//
// Warp 0 (one thread) issues the MMAs, warp 17 (one thread) the bulk copies,
// warps 1-16 ("compute warps") do everything else.  Every wait is bounded: a
// wait that gives up sets CR_ETIMEOUT and a global abort flag, after which
// all CTAs leave the solve at their next grid barrier.
//
// What bounds it (16 x 16 lattice, alpha = 1, 65536 walkers; us per CG
// iteration from %globaltimer): W1 73 and W2 72 wait on latency -- the ring
// of V and the read of T in W1, the read of T and the stores of Y to shared
// memory in W2 --, the slice phase 22 moves the partial rows (2 x 80 MB)
// through L2, a- and b-sums 10, barriers 11.  With one thread for copies and
// MMAs, which divided for its ring positions and built every descriptor
// anew, W1 took 133 whatever was taken out of it (T, copies, MMAs): the
// issuing thread was the bound, so copies and MMAs have a thread each and
// advance by constants.  A float64 warp instruction takes the SM 16 cycles
// however many lanes need it, so the slice phase packs its float64 work into
// full warps, the scalars of an iteration are one thread's work, and sums of
// several scalars split their slots over the lanes.  With 8 compute warps,
// one walker tile per stage of V, one issuing thread and float64 scalars in
// every warp an iteration took 248 (W1 105, W2 84, slice 35), now 188; a
// chain of 64 sites (alpha = 2, 16384 walkers) 46 (slice 12), now 37 (8).
#include <cuda_bf16.h>

#include "common.cuh"
#include "tc.cuh"

namespace {

constexpr int NCW = 16;                         // compute warps
constexpr int NCT = 32 * NCW;                   // compute threads
constexpr int FC_THREADS = NCT + 64;            // warp 0 issues MMAs, the last warp copies
constexpr int NS1 = 4;                          // W1 operand stages
constexpr int W1_A = 128 * 32 * 2;              // sigma tile of one K-chunk
constexpr int W1_W = 128;                       // columns of a W1 pass
constexpr int W1_B_PLANE = W1_W * 32 * 2;       // one bf16 plane of V
constexpr int W1_STAGE = 2 * W1_A + 3 * W1_B_PLANE; // 40 KB
constexpr int Y_BLK = 128 * 32 * 2;             // one plane of one 128-column n-block
constexpr uint32_t WAIT_LIMIT = 1u << 26;       // mbarrier polls
constexpr unsigned BAR_LIMIT = 1u << 23;        // grid-barrier polls (~1 s with the sleeps)
constexpr int MAX_WPC = 512;                    // walkers per CTA
constexpr int KS_MAX = 512;                     // parameters per CTA (its CG slice in smem)

struct Geo {
    int N, M, P, B;
    int G;       // CTAs
    int wpc;     // walkers per CTA (the last CTA may have fewer)
    int tpu;     // W1 walker tiles per unit (a pair shares the stages of V): 1 or 2
    int ntpc;    // W1 walker tiles per CTA (a multiple of tpu)
    int trows;   // rows per W1 tile (<= 128)
    int Kp;      // sites padded to a multiple of 32 (W1 contraction length)
    int nkc1;    // W1 K-chunks of 32 sites
    int npass1;  // W1 column passes of 128 (the last one wlast1 wide)
    int wlast1;
    int Np;      // sites padded to a multiple of 16 (W2 MMA N)
    int nb2;     // W2 n-blocks of 128 columns of Y
    int nbp;     // n-blocks per W2 pass (<= 2)
    int npass2;
    int nwc;     // W2 walker chunks of 32 per CTA
    int kslice;  // parameters per CTA in phases C and P
    size_t ring; // bytes of the operand ring (W1 and W2 share it)
    size_t smem; // dynamic shared memory
};

struct Args {
    Geo g;
    const int8_t* spins;
    const cpx<float>* T;
    const cpx<double>* F;
    const cpx<double>* sO;    // sums over walkers: sum O_k [P], then sum |T_j|^2 at P + 2 + j
    double shift, tol;
    int maxit, precond, apply_only;
    const cpx<double>* v_in;  // apply_only: the vector v
    cpx<float>* u_out;        // apply_only: u = O v [B] (or NULL)
    double* cg;               // complex128 x, r, p, Ap, d [5][P]
    unsigned char* a1;        // sigma tiles of W1, per CTA
    unsigned char* b2;        // sigma^T chunks of W2, per CTA
    unsigned char* v2;        // three bf16 planes of the W part of p
    size_t v2_plane;
    cpx<float>* vab;          // float32 a- and b-parts of p [N + M]
    float* part;              // partial rows, complex float32 [G][P]
    double* psc;              // scalar partials [G][8]
    unsigned* bar;            // [0] grid-barrier counter, [1] abort flag
    double* scal;             // [1] F.F, [2] done, [3] iterations, [4] r.r
    int* status;
};

// scalar partial slots, one value per CTA: psc[cta * 8 + slot]
enum { S_WW = 0, S_RR = 1, S_GAM = 2, S_FF = 3, S_OUR = 4, S_OUI = 5, S_UU = 6 };

CR_D void split3(float x, __nv_bfloat16* hi, __nv_bfloat16* mid, __nv_bfloat16* lo) {
    *hi = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(*hi);
    *mid = __float2bfloat16_rn(r1);
    *lo = __float2bfloat16_rn(r1 - __bfloat162float(*mid));
}

CR_D __nv_bfloat16 split_term(float x, int pl) {
    __nv_bfloat16 h, m, l;
    split3(x, &h, &m, &l);
    return pl == 0 ? h : (pl == 1 ? m : l);
}

CR_D uint4 pack8(const __nv_bfloat16* v) {
    uint4 r;
    uint32_t* w = reinterpret_cast<uint32_t*>(&r);
#pragma unroll
    for (int q = 0; q < 4; ++q)
        w[q] = (uint32_t)__bfloat16_as_ushort(v[2 * q]) |
               ((uint32_t)__bfloat16_as_ushort(v[2 * q + 1]) << 16);
    return r;
}

// 32 aligned bytes
CR_D void ldg32(const void* p, float4* a, float4* b) {
    asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(a->x), "=f"(a->y), "=f"(a->z), "=f"(a->w), "=f"(b->x), "=f"(b->y), "=f"(b->z), "=f"(b->w)
                 : "l"(p));
}

CR_D void kadd(float& s, float& c, float v) {
    const float y = v - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
}

// generic-proxy global writes -> visible to later bulk copies (async proxy)
CR_D void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;\n" ::: "memory"); }

// barrier among the compute threads (warps 1-16)
CR_D void compute_sync() { asm volatile("bar.sync 1, %0;\n" ::"n"(NCT) : "memory"); }

CR_D void mbar_arrive(uint64_t* mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(tc::smem_u32(mbar)) : "memory");
}

// byte offset of element (row, k) in a 32-column K-major tile
CR_D uint32_t koff(int row, int k) { return tc::kmajor_offset(row, k, 32); }

// offset (bytes, within one plane) of element (column n, site i) of the W1
// operand of V: blocks [pass of 128 columns][K-chunk of 32 sites]
CR_HD size_t v2_offset(const Geo& g, int n, int i) {
    const int ps = n / W1_W, nl = n % W1_W, kc = i >> 5, il = i & 31;
    const int width = ps < g.npass1 - 1 ? W1_W : g.wlast1;
    return ((size_t)W1_W * ps * g.Kp + (size_t)width * 32 * kc) * 2 +
           tc::kmajor_offset(nl, il, 32);
}

struct Smem {
    unsigned char* ring;
    // the CTA's slice of the CG vectors, resident for the whole solve
    cpx<double>* x;     // [KS_MAX]
    cpx<double>* r;
    cpx<double>* p;
    cpx<double>* sv;    // s = A p
    cpx<double>* ob;    // Obar_k = (sum_s O_sk) / B
    double* d;          // inverse of the Jacobi diagonal (1 without preconditioning)
    cpx<double>* tot;   // [NCT] row sums of the row groups
    cpx<float>* wbuf;   // [wpc] centred u of the CTA's walkers
    cpx<float>* va;     // [N]
    cpx<float>* vb;     // [M]
    cpx<float>* xch;    // [NCT] exchange
    double* red;        // [8 NCW]
    uint64_t* mb;       // mbarriers
    uint32_t* slot;     // TMEM address
    int* flag;          // [0] CTA abort, [1] done
    double* bc;         // [10] broadcast scalars
};

// mbarrier indices
enum { FULL1 = 0, EMPTY1 = NS1, D1FULL = 2 * NS1, D1EMPTY = D1FULL + 2, FULL2 = D1EMPTY + 2,
       EMPTY2 = FULL2 + 2, D2FULL = EMPTY2 + 2, GO, NMB };

CR_D Smem carve(unsigned char* sm, const Geo& g) {
    Smem s;
    s.ring = sm;
    unsigned char* p = sm + g.ring;
    s.x = (cpx<double>*)p;
    p += KS_MAX * 16;
    s.r = (cpx<double>*)p;
    p += KS_MAX * 16;
    s.p = (cpx<double>*)p;
    p += KS_MAX * 16;
    s.sv = (cpx<double>*)p;
    p += KS_MAX * 16;
    s.ob = (cpx<double>*)p;
    p += KS_MAX * 16;
    s.d = (double*)p;
    p += KS_MAX * 8;
    s.tot = (cpx<double>*)p;
    p += NCT * 16;
    s.wbuf = (cpx<float>*)p;
    p += (size_t)MAX_WPC * 8;
    s.va = (cpx<float>*)p;
    p += 256 * 8;
    s.vb = (cpx<float>*)p;
    p += 256 * 8;
    s.xch = (cpx<float>*)p;
    p += NCT * 8;
    s.red = (double*)p;
    p += 8 * NCW * 8;
    s.bc = (double*)p;
    p += 10 * 8;
    s.mb = (uint64_t*)p;
    p += NMB * 8;
    s.slot = (uint32_t*)p;
    p += 16;
    s.flag = (int*)p;
    return s;
}

// Bounded mbarrier wait; gives up at once after a CTA abort.
CR_D bool wait_mb(uint64_t* mb, uint32_t parity, volatile int* flag, unsigned* bar, int* status) {
    if (flag[0]) return false;
    for (int rep = 0; rep < 64; ++rep) {
        if (tc::mbar_wait(mb, parity, WAIT_LIMIT >> 6)) return true;
        if (flag[0] || *(volatile unsigned*)&bar[1]) {
            flag[0] = 1;
            return false;
        }
    }
    flag[0] = 1;
    atomicExch(&bar[1], 1u);
    set_status(status, CR_ETIMEOUT);
    return false;
}

// Grid barrier (all threads of every CTA): arrive on the counter, wait
// (bounded) until all G CTAs of this round arrived.  Returns false after an
// abort anywhere.
CR_D bool grid_sync(unsigned* bar, unsigned target, volatile int* flag, int* status) {
    tc::fence_before_sync();
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(&bar[0]) : "memory");
        unsigned n = 0;
        for (;;) {
            if (*(volatile unsigned*)&bar[0] >= target) break;
            if (*(volatile unsigned*)&bar[1]) {
                flag[0] = 1;
                break;
            }
            if (++n > BAR_LIMIT) {
                flag[0] = 1;
                atomicExch(&bar[1], 1u);
                set_status(status, CR_ETIMEOUT);
                break;
            }
            if (n > 4096) __nanosleep(64);  // spin first: most waits are a few microseconds
        }
        asm volatile("fence.acq_rel.gpu;\n" ::: "memory");  // acquire what the others released
    }
    __syncthreads();
    tc::fence_after_sync();
    return flag[0] == 0;
}

// Warp sums of NV <= 8 values in 9 float64 additions, not 5 NV: the lanes split
// the slots among them.  Lane l ends with the sum of slot l / 4.
template <int NV>
CR_D double warp_sums(const double (&v)[NV]) {
    const int lane = threadIdx.x & 31;
    double x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = q < NV ? v[q < NV ? q : 0] : 0.0;
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1) {
        const bool up = lane & (4 * h);
#pragma unroll
        for (int q = 0; q < h; ++q) {
            const double give = up ? x[q] : x[q + h], keep = up ? x[q + h] : x[q];
            x[q] = keep + __shfl_xor_sync(0xffffffffu, give, 4 * h);
        }
    }
    x[0] += __shfl_xor_sync(0xffffffffu, x[0], 2);
    return x[0] + __shfl_xor_sync(0xffffffffu, x[0], 1);
}

// The CTA's partials of NV scalar slots (compute threads only): warp sums,
// then one barrier, then the warp values of each slot added in a fixed tree
// order and written to psc[cta * 8 + slot].
template <int NV>
CR_D void put_psc(double* psc, int cta, const double (&v)[NV], const int (&sl)[NV], double* red,
                  bool live = true) {
    const int cw = (threadIdx.x >> 5) - 1, lane = threadIdx.x & 31;
    if (!live) {  // a warp of zeros
        if (lane < 8) red[cw * 8 + lane] = 0.0;
    } else if (NV == 1) {
        const double w = warp_sum(v[0]);
        if (lane == 0) red[cw * 8] = w;
    } else {
        const double x = warp_sums<NV>(v);
        if ((lane & 3) == 0) red[cw * 8 + (lane >> 2)] = x;
    }
    compute_sync();
    const int ct = threadIdx.x - 32;
    if (ct < NV) {
        const double* r = red + ct;
        double tot = 0.0;
#pragma unroll
        for (int w = 0; w < NCW; w += 4)
            tot += (r[8 * w] + r[8 * w + 8]) + (r[8 * w + 16] + r[8 * w + 24]);
        psc[(size_t)cta * 8 + sl[ct]] = tot;
    }
}

// Sums over all CTAs of NV slots, by one warp, all loads in flight at once,
// in a fixed order (the same values in every lane and every CTA).
template <int NV>
CR_D void sum_psc(const double* psc, int G, const int (&sl)[NV], double (&out)[NV]) {
    const int lane = threadIdx.x & 31;
    double v[NV][5], s[NV];
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        const int cc = lane + 32 * m;
#pragma unroll
        for (int q = 0; q < NV; ++q) v[q][m] = cc < G ? psc[(size_t)cc * 8 + sl[q]] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        double x = (v[q][0] + v[q][1]) + (v[q][2] + v[q][3]);
        for (int cc = lane + 160; cc < G; cc += 32) x += psc[(size_t)cc * 8 + sl[q]];
        s[q] = x + v[q][4];
    }
    if (NV == 1) {
        out[0] = warp_sum(s[0]);
    } else {
        const double tot = warp_sums<NV>(s);
#pragma unroll
        for (int q = 0; q < NV; ++q) out[q] = __shfl_sync(0xffffffffu, tot, 4 * q);
    }
}

// The operands of entry k (value pk) of the vector the walker phase
// multiplies: float32 a- and b-parts, three bf16 planes of the W part.
CR_D void emit_p(const Args& a, int k, cpx<double> pk) {
    const Geo& g = a.g;
    const int N = g.N, M = g.M;
    if (k < N + M) {
        a.vab[k] = ccast<float>(pk);
        return;
    }
    const int i = (k - N - M) / M, j = (k - N - M) % M;
    const float re = (float)pk.x, im = (float)pk.y;
#pragma unroll
    for (int pl = 0; pl < 3; ++pl) {
        __nv_bfloat16* base = (__nv_bfloat16*)(a.v2 + pl * a.v2_plane);
        base[v2_offset(g, 2 * j, i) / 2] = split_term(re, pl);
        base[v2_offset(g, 2 * j + 1, i) / 2] = split_term(im, pl);
    }
}

}  // namespace

__global__ void __launch_bounds__(FC_THREADS, 1) cg_fused_kernel(const __grid_constant__ Args a) {
    extern __shared__ __align__(1024) unsigned char sm_raw[];
    const Geo& g = a.g;
    const int N = g.N, M = g.M, P = g.P, B = g.B, G = g.G;
    const int c = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int ct = t >= 32 && t < 32 + NCT ? t - 32 : -1;  // compute-thread index (warps 1-16)
    const bool copier = t == 32 + NCT;
    Smem s = carve(sm_raw, g);
    volatile int* flag = s.flag;  // [0] CTA abort, [1] solve finished
    const int s0 = c * g.wpc, s1 = min(B, s0 + g.wpc), nw = max(0, s1 - s0);
    const int k0 = min(P, c * g.kslice), k1 = min(P, k0 + g.kslice);
    cpx<double>* X = (cpx<double>*)a.cg;
    cpx<double>* Ap = X + 3 * P;
    const double invB = 1.0 / B;
    const bool vecS = (N & 15) == 0 && ((uintptr_t)a.spins & 15) == 0;  // 16-byte loads of spins

    if (t == 0) {
        for (int i = 0; i < NMB; ++i) {
            uint32_t cnt = 1;
            if (i == D1EMPTY || i == D1EMPTY + 1) cnt = NCT;
            if (i == FULL2 || i == FULL2 + 1) cnt = 1 + NCT;
            tc::mbar_init(&s.mb[i], cnt);
        }
        tc::fence_mbar_init();
        flag[0] = 0;
        flag[1] = 0;
    }
    if (warp == 0) {
        tc::tmem_alloc(s.slot, 512u);
        tc::tmem_relinquish();
    }

    // ---------------------------------------------------------- prologue
    // the spin operands of this CTA's walkers: W1 sigma tiles and W2 sigma^T
    // chunks (zero outside the walker range and past the last site)
    if (ct >= 0) {
        const int n1 = g.ntpc * g.nkc1 * 128 * 4;
        for (int e = ct; e < n1; e += NCT) {
            const int q8 = e & 3, r = (e >> 2) & 127, blk = e >> 9;
            const int tt = blk / g.nkc1, kc = blk % g.nkc1;
            const int sl = tt * g.trows + r, sw = s0 + sl;
            __nv_bfloat16 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int i = kc * 32 + q8 * 8 + q;
                const bool ok = r < g.trows && sl < nw && i < N;
                v[q] = __float2bfloat16_rn(ok ? (float)a.spins[(size_t)sw * N + i] : 0.f);
            }
            *reinterpret_cast<uint4*>(a.a1 + ((size_t)(c * g.ntpc + tt) * g.nkc1 + kc) * W1_A +
                                      koff(r, q8 * 8)) = pack8(v);
        }
        const int n2 = g.nwc * g.Np * 4;
        for (int e = ct; e < n2; e += NCT) {
            const int q8 = e & 3, i = (e >> 2) % g.Np, wc = (e >> 2) / g.Np;
            __nv_bfloat16 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int sl = wc * 32 + q8 * 8 + q;
                const bool ok = sl < nw && i < N;
                v[q] = __float2bfloat16_rn(ok ? (float)a.spins[(size_t)(s0 + sl) * N + i] : 0.f);
            }
            *reinterpret_cast<uint4*>(a.b2 + ((size_t)c * g.nwc + wc) * g.Np * 64 + koff(i, q8 * 8)) =
                pack8(v);
        }
        // this CTA's slice: x = 0, r = F, p = s = 0, u = r / d (apply_only:
        // u = v), the operands of u and the partial inner products
        double ff = 0.0, gam = 0.0, our = 0.0, oui = 0.0, uu = 0.0;
        for (int k = k0 + ct; k < k1; k += NCT) {
            const int kl = k - k0;
            const cpx<double> obk = invB * a.sO[k];
            s.ob[kl] = obk;
            cpx<double> uk;
            if (a.apply_only) {
                uk = a.v_in[k];
                s.r[kl] = uk;
                s.d[kl] = 1.0;
            } else {
                double d = 1.0;
                if (a.precond) {
                    const double o2 = k < N ? 1.0
                                            : invB * a.sO[P + 2 + (k < N + M ? k - N : (k - N - M) % M)].x;
                    d = o2 - abs2(obk) + a.shift;
                }
                const cpx<double> f = a.F[k];
                uk = (1.0 / d) * f;
                s.x[kl] = {0.0, 0.0};
                s.r[kl] = f;
                s.d[kl] = 1.0 / d;
                ff += abs2(f);
                gam += cmulc(f, uk).x;
            }
            s.p[kl] = {0.0, 0.0};
            s.sv[kl] = {0.0, 0.0};
            emit_p(a, k, uk);
            const cpx<double> ou = obk * uk;
            our += ou.x;
            oui += ou.y;
            uu += abs2(uk);
        }
        fence_proxy_async_global();
        const double pv[6] = {ff, ff, gam, our, oui, uu};
        const int ps[6] = {S_FF, S_RR, S_GAM, S_OUR, S_OUI, S_UU};
        put_psc<6>(a.psc, c, pv, ps, s.red);
    }
    unsigned round = 1;
    bool ok = grid_sync(a.bar, round++ * G, flag, a.status);
    const uint32_t taddr = *s.slot;

    int its = 0, done = 0;
    double ff = 0.0, rr = 0.0, gam = 0.0, gam_prev = 1.0, alpha_prev = 1.0;
    // pipeline counters (identical in every role of the CTA)
    uint32_t g1 = 0, u1 = 0, g2 = 0, u2 = 0;
    // last copy issued into each stage (copy thread) and last MMA commit (MMA
    // thread), so that an abort can wait (bounded) for what is still in flight
    int last1[NS1] = {-1, -1, -1, -1}, last2[2] = {-1, -1}, lastm1 = -1, lastm2 = -1;
    // a unit: tpu walker tiles x one column pass, D1 in TMEM columns [256 h, +128 tpu)
    const int units = g.ntpc / g.tpu * g.npass1;
    const int total1 = units * g.nkc1;
    auto width_of = [&](int ps) { return ps < g.npass1 - 1 ? W1_W : g.wlast1; };

    while (ok) {
        // ======================================================= walker phase
        // producer: W1 operand copies start at once (their data was released
        // before the barrier); the MMAs wait for the convergence decision
        int cq = 0, ckc = 0, cps = 0, ct0 = 0;  // copy cursor: stage, K-chunk, column pass, first tile
        auto load1 = [&]() {
            const uint32_t gq = g1 + cq, b = gq & (NS1 - 1);
            if (gq >= NS1 && !wait_mb(&s.mb[EMPTY1 + b], ((gq / NS1) - 1) & 1, flag, a.bar, a.status))
                return;
            const int w = width_of(cps);
            unsigned char* st = s.ring + (size_t)b * W1_STAGE;
            tc::mbar_expect_tx(&s.mb[FULL1 + b], (uint32_t)(g.tpu * W1_A + 3 * w * 64));
            const unsigned char* va = a.v2 + ((size_t)W1_W * cps * g.Kp + (size_t)w * 32 * ckc) * 2;
            for (int pl = 0; pl < 3; ++pl, va += a.v2_plane)
                tc::bulk_g2s(st + 2 * W1_A + pl * W1_B_PLANE, va, (uint32_t)(w * 64), &s.mb[FULL1 + b]);
            const unsigned char* sa = a.a1 + ((size_t)(c * g.ntpc + ct0) * g.nkc1 + ckc) * W1_A;
            tc::bulk_g2s(st, sa, W1_A, &s.mb[FULL1 + b]);
            if (g.tpu == 2) tc::bulk_g2s(st + W1_A, sa + (size_t)g.nkc1 * W1_A, W1_A, &s.mb[FULL1 + b]);
            last1[b] = (int)gq;
            ++cq;
            if (++ckc == g.nkc1) {
                ckc = 0;
                if (++cps == g.npass1) {
                    cps = 0;
                    ct0 += g.tpu;
                }
            }
        };
        const int npre = NS1 - 1 < total1 ? NS1 - 1 : total1;
        if (copier)
            for (int q = 0; q < npre; ++q) load1();
        if (warp == 1) {
            // the inner products of the current r and u, and the decision
            const int sl6[6] = {S_RR, S_GAM, S_OUR, S_OUI, S_UU, S_FF};
            double v6[6];
            sum_psc<6>(a.psc, G, sl6, v6);
            const double r2 = v6[0], gm = v6[1], our = v6[2], oui = v6[3], uu = v6[4], f2 = v6[5];
            if (lane == 0) {
                if (its == 0) s.bc[0] = f2;
                const double fnorm2 = s.bc[0];
                const int conv = !a.apply_only && !(r2 > a.tol * a.tol * fnorm2);
                // the decision of the whole CTA: converged, out of iterations, or aborted
                const int fin = conv || (!a.apply_only && its >= a.maxit) || flag[0];
                s.bc[7] = conv;
                s.bc[1] = r2;
                s.bc[2] = our;  // ubar = Obar . u
                s.bc[3] = oui;
                s.bc[4] = uu;
                s.bc[6] = gm;
                flag[1] = fin;
                mbar_arrive(&s.mb[GO]);
            }
        }
        if (ct >= 0) {
            for (int i = ct; i < N; i += NCT) s.va[i] = a.vab[i];
            for (int j = ct; j < M; j += NCT) s.vb[j] = a.vab[N + j];
        }
        // the decision reaches warps 0 and 17 through GO, the compute warps
        // through their barrier; flag[1], written once before either, is uniform
        if (ct < 0) wait_mb(&s.mb[GO], (uint32_t)its & 1, flag, a.bar, a.status);
        if (ct >= 0) compute_sync();
        ff = s.bc[0];
        rr = s.bc[1];
        gam = s.bc[6];
        if (flag[1]) {
            // finished: let the copies issued above land, then leave
            if (copier)
                for (int q = 0; q < npre; ++q) {
                    const uint32_t gq = g1 + q;
                    tc::mbar_wait(&s.mb[FULL1 + gq % NS1], (gq / NS1) & 1, WAIT_LIMIT);
                }
            done = s.bc[7] != 0.0;
            __syncthreads();
            break;
        }
        const cpx<double> ubar = {s.bc[2], s.bc[3]};
        const cpx<float> ubar32 = ccast<float>(ubar);
        const double uu = s.bc[4];
        double ww = 0.0;  // sum |w_s|^2 of this thread's walkers
        if (warp == 0) {
            if (lane == 0) {
                // ------------------------------------------------- W1 MMAs
                const uint64_t d0 = tc::make_desc(tc::smem_u32(s.ring), 128, 512);
                uint32_t gq = g1, uu1 = u1;
                for (int un = 0; un < units; un += g.npass1)
                    for (int ps = 0; ps < g.npass1; ++ps, ++uu1) {
                        const uint32_t h = uu1 & 1, idesc = tc::make_idesc_bf16(128, width_of(ps));
                        if (uu1 >= 2)
                            wait_mb(&s.mb[D1EMPTY + h], ((uu1 >> 1) - 1) & 1, flag, a.bar, a.status);
                        for (int kc = 0; kc < g.nkc1; ++kc, ++gq) {
                            const uint32_t b = gq & (NS1 - 1);
                            wait_mb(&s.mb[FULL1 + b], (gq / NS1) & 1, flag, a.bar, a.status);
                            tc::fence_after_sync();
                            uint64_t ad = d0 + b * (W1_STAGE >> 4);
                            const uint64_t bd = ad + (2 * W1_A >> 4);
                            uint32_t dt = taddr + 256 * h;
                            for (int i = 0; i < g.tpu; ++i, ad += W1_A >> 4, dt += W1_W) {
                                // small terms first: they are added to a small accumulator
#pragma unroll
                                for (int pl = 2; pl >= 0; --pl)
#pragma unroll
                                    for (int ks = 0; ks < 2; ++ks)
                                        tc::mma_bf16(dt, ad + ks * 16, bd + ((pl * W1_B_PLANE + ks * 256) >> 4),
                                                     idesc, kc != 0 || pl != 2 || ks != 0);
                            }
                            tc::commit(&s.mb[EMPTY1 + b]);
                        }
                        tc::commit(&s.mb[D1FULL + h]);
                    }
                lastm1 = (int)gq - 1;
            }
            __syncwarp();
        } else if (ct < 0) {
            if (copier)
                while (cq < total1 && !flag[0]) load1();
            __syncwarp();
        } else {
            // --------------------------------------------- W1 compute warps
            // a TMEM lane block is read by four warps: two tiles x two column
            // splits, or four splits of one tile; each thread sums its walker's
            // u over its 16-column groups (8 hidden units)
            const int lb = warp & 3, qd = (warp - 1) >> 2, row = 32 * lb + lane;
            const int nsp = 4 / g.tpu, ti = qd / nsp, sp = qd % nsp;
            // whole 32-byte sectors per lane: rows are M apart, and next to the
            // operand ring there is no L1 to keep the other half of one
            const bool vecT = (M & 3) == 0 && ((uintptr_t)a.T & 31) == 0;
            cpx<float> uacc = {0.f, 0.f};
            for (int unit = 0; unit < units; ++unit) {
                const int tt = unit / g.npass1 * g.tpu + ti, ps = unit % g.npass1;
                const uint32_t uu1 = u1 + unit, h = uu1 & 1;
                const int sl = tt * g.trows + row;
                const bool valid = row < g.trows && sl < nw;
                const int sw = s0 + sl;
                const cpx<float>* Tr = a.T + (size_t)sw * M;
                const int w = width_of(ps), ngr = w / 16;
                // T of a group as four 16-byte loads, fetched a group ahead of its use
                auto fetchT = [&](int grp, float4* tv) {
                    const int j0 = W1_W / 2 * ps + 8 * grp;
                    if (grp >= ngr || !valid) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) tv[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                    } else if (vecT && j0 + 8 <= M) {
                        ldg32(Tr + j0, &tv[0], &tv[1]);
                        ldg32(Tr + j0 + 4, &tv[2], &tv[3]);
                    } else {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int j = j0 + 2 * q;
                            const cpx<float> t0 = j < M ? ldg(Tr + j) : cpx<float>{0.f, 0.f};
                            const cpx<float> t1 = j + 1 < M ? ldg(Tr + j + 1) : cpx<float>{0.f, 0.f};
                            tv[q] = make_float4(t0.x, t0.y, t1.x, t1.y);
                        }
                    }
                };
                float4 tc0[4], tc1[4];
                fetchT(sp, tc0);
                if (ps == 0) {
                    // sigma . va: the threads of a row take 16-site blocks in turn
                    // (16-byte loads when N % 16 == 0 and the spins are aligned)
                    uacc = {0.f, 0.f};
                    if (valid) {
                        const int8_t* sr = a.spins + (size_t)sw * N;
                        if (vecS) {
                            for (int b16 = sp; b16 < N / 16; b16 += nsp) {
                                const int4 raw = __ldg(reinterpret_cast<const int4*>(sr) + b16);
                                const int8_t* sv = reinterpret_cast<const int8_t*>(&raw);
#pragma unroll
                                for (int q = 0; q < 16; ++q)
                                    uacc = uacc + (float)sv[q] * s.va[16 * b16 + q];
                            }
                        } else if ((N & 15) == 0) {  // unaligned: the same order, byte by byte
#pragma unroll 1
                            for (int b16 = sp; b16 < N / 16; b16 += nsp)
#pragma unroll 1
                                for (int i = 16 * b16; i < 16 * b16 + 16; ++i)
                                    uacc = uacc + (float)sr[i] * s.va[i];
                        } else {
                            for (int i = sp; i < N; i += nsp) uacc = uacc + (float)sr[i] * s.va[i];
                        }
                    }
                }
                wait_mb(&s.mb[D1FULL + h], (uu1 >> 1) & 1, flag, a.bar, a.status);
                tc::fence_after_sync();
                for (int grp = sp; grp < ngr; grp += nsp) {
                    fetchT(grp + nsp, tc1);
                    float d[16];
                    tc::tmem_ld16(taddr + ((uint32_t)(32 * lb) << 16) + 256 * h + W1_W * ti + 16 * grp, d);
                    const int j0 = W1_W / 2 * ps + 8 * grp;
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int j = j0 + q;
                        const int jv = j < M ? j : 0;
                        const float4 tq = tc0[q >> 1];
                        const cpx<float> tj = (q & 1) ? cpx<float>{tq.z, tq.w} : cpx<float>{tq.x, tq.y};
                        const cpx<float> x = {d[2 * q] + s.vb[jv].x, d[2 * q + 1] + s.vb[jv].y};
                        uacc = uacc + tj * x;  // tj = 0 past M and on invalid rows
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) tc0[q] = tc1[q];
                }
                tc::fence_before_sync();
                mbar_arrive(&s.mb[D1EMPTY + h]);
                if (ps == g.npass1 - 1) {
                    // u of the tile's rows: the splits meet
                    if (sp > 0) s.xch[(ti * nsp + sp) * 128 + row] = uacc;
                    compute_sync();
                    if (sp == 0 && row < g.trows && sl < g.wpc) {
                        cpx<float> wv = {0.f, 0.f};
                        if (valid) {
                            cpx<float> u = uacc;
                            for (int r = 1; r < nsp; ++r) u = u + s.xch[(ti * nsp + r) * 128 + row];
                            if (a.u_out) a.u_out[sw] = u;
                            wv = u - ubar32;
                            ww += (double)abs2(wv);
                        }
                        s.wbuf[sl] = wv;
                    }
                    compute_sync();
                }
            }
        }
        g1 += total1;
        u1 += units;
        // TMEM: every D1 read is done before the W2 MMAs reuse the columns
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();

        // a-sums: sum_s sigma_si w_s per site.  Thread (block b16 of 16 sites,
        // walker subset sub) sums its walkers from 16-byte spin loads, eight
        // walkers' loads in flight; each site's nsub partial sums are then
        // added in a fixed order, through the operand ring (idle here).
        if (ct >= 0) {
            const int NG = (N + 15) / 16, nsub = min(NCT / NG, 32);
            const int b16 = ct % NG, sub = ct / NG;
            cpx<float>* xa = (cpx<float>*)s.ring;  // [nsub][NG * 16]
            if (sub < nsub) {
                float ax[16], ay[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) ax[q] = ay[q] = 0.f;
                for (int sl0 = sub; sl0 < nw; sl0 += 8 * nsub) {
                    int4 raw[8];
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        const int sl = sl0 + m * nsub;
                        const int8_t* sr = a.spins + (size_t)(s0 + (sl < nw ? sl : 0)) * N;
                        if (sl >= nw) {
                            raw[m] = make_int4(0, 0, 0, 0);
                        } else if (vecS) {
                            raw[m] = __ldg(reinterpret_cast<const int4*>(sr) + b16);
                        } else {
                            int8_t sv[16];
#pragma unroll
                            for (int q = 0; q < 16; ++q) sv[q] = 16 * b16 + q < N ? sr[16 * b16 + q] : (int8_t)0;
                            memcpy(&raw[m], sv, 16);
                        }
                    }
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        const int sl = sl0 + m * nsub;
                        const cpx<float> wv = sl < nw ? s.wbuf[sl] : cpx<float>{0.f, 0.f};
                        const int8_t* sv = reinterpret_cast<const int8_t*>(&raw[m]);
#pragma unroll
                        for (int q = 0; q < 16; ++q) {
                            ax[q] = fmaf((float)sv[q], wv.x, ax[q]);
                            ay[q] = fmaf((float)sv[q], wv.y, ay[q]);
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < 16; ++q) xa[sub * NG * 16 + 16 * b16 + q] = {ax[q], ay[q]};
            }
            compute_sync();
            for (int i = ct; i < N; i += NCT) {
                float sx = 0.f, sy = 0.f, cx = 0.f, cy = 0.f;
                for (int r = 0; r < nsub; ++r) {
                    const cpx<float> v = xa[r * NG * 16 + i];
                    kadd(sx, cx, v.x);
                    kadd(sy, cy, v.y);
                }
                a.part[2 * ((size_t)c * P + i)] = sx - cx;
                a.part[2 * ((size_t)c * P + i) + 1] = sy - cy;
            }
        }
        tc::fence_before_sync();
        __syncthreads();  // the ring is W2's from here
        tc::fence_after_sync();

        for (int ps2 = 0; ps2 < g.npass2; ++ps2) {
            const int nbq = min(g.nbp, g.nb2 - ps2 * g.nbp);
            const int jp0 = 64 * g.nbp * ps2, Jp = 64 * nbq;
            const size_t stage2 = (size_t)g.nbp * 3 * Y_BLK + (size_t)g.Np * 64;
            if (warp == 0) {
                if (lane == 0) {
                    // --------------------------------------------- W2 MMAs
                    const uint32_t idesc = tc::make_idesc_bf16(128, g.Np);
                    const uint64_t d0 = tc::make_desc(tc::smem_u32(s.ring), 128, 512);
                    const uint64_t so = (uint64_t)(g.nbp * 3 * Y_BLK) >> 4, po = (uint64_t)(g.nbp * Y_BLK) >> 4;
                    for (int wc = 0; wc < g.nwc; ++wc) {
                        const uint32_t gq = g2 + wc, b = gq & 1;
                        wait_mb(&s.mb[FULL2 + b], (gq >> 1) & 1, flag, a.bar, a.status);
                        tc::fence_after_sync();
                        const uint64_t yd = d0 + b * (stage2 >> 4), sd = yd + so;
                        for (int nb = 0; nb < nbq; ++nb)
#pragma unroll
                            for (int pl = 2; pl >= 0; --pl)
#pragma unroll
                                for (int ks = 0; ks < 2; ++ks)
                                    tc::mma_bf16(taddr + nb * g.Np, yd + pl * po + nb * (Y_BLK >> 4) + ks * 16,
                                                 sd + ks * 16, idesc, wc != 0 || pl != 2 || ks != 0);
                        tc::commit(&s.mb[EMPTY2 + b]);
                        lastm2 = (int)gq;
                    }
                    tc::commit(&s.mb[D2FULL]);
                }
                __syncwarp();
            } else if (ct < 0) {
                if (copier) {
                    const unsigned char* src = a.b2 + (size_t)c * g.nwc * g.Np * 64;
                    for (int wc = 0; wc < g.nwc && !flag[0]; ++wc, src += (size_t)g.Np * 64) {
                        const uint32_t gq = g2 + wc, b = gq & 1;
                        if (gq >= 2 && !wait_mb(&s.mb[EMPTY2 + b], ((gq >> 1) - 1) & 1, flag, a.bar, a.status))
                            break;
                        tc::mbar_expect_tx(&s.mb[FULL2 + b], (uint32_t)(g.Np * 64));
                        tc::bulk_g2s(s.ring + b * stage2 + (size_t)g.nbp * 3 * Y_BLK, src,
                                     (uint32_t)(g.Np * 64), &s.mb[FULL2 + b]);
                        last2[b] = (int)gq;
                    }
                }
                __syncwarp();
            } else {
                // ---------------------------------------- W2 compute warps
                const int tpj = NCT / Jp;  // threads per hidden unit: 4 or 8
                const int j = jp0 + ct % Jp, grp = ct / Jp;
                const bool live = grp < 4;  // a chunk has four groups of 8 walkers
                float bsx = 0.f, bsy = 0.f, bcx = 0.f, bcy = 0.f;
                // T of this thread's walkers of a chunk, fetched one chunk ahead
                // (compile-time indices throughout, so the buffers stay in registers)
                cpx<float> tcur[8], tnxt[8];
                const bool mine = live && j < M;
                const cpx<float>* Tj = a.T + (size_t)(s0 + grp * 8) * M + j;
#define FCG_FETCH_T(WC, TV)                                                                       \
    _Pragma("unroll") for (int q = 0; q < 8; ++q) {                                               \
        const int sl = (WC) * 32 + grp * 8 + q;                                                   \
        TV[q] = (mine && sl < nw) ? ldg(Tj + (size_t)((WC) * 32 + q) * M) : cpx<float>{0.f, 0.f}; \
    }
                FCG_FETCH_T(0, tcur)
                for (int wc = 0; wc < g.nwc; ++wc) {
                    const uint32_t gq = g2 + wc, b = gq & 1;
                    if (wc + 1 < g.nwc) {
                        FCG_FETCH_T(wc + 1, tnxt)
                    }
                    if (gq >= 2) wait_mb(&s.mb[EMPTY2 + b], ((gq >> 1) - 1) & 1, flag, a.bar, a.status);
                    tc::fence_after_sync();
                    unsigned char* sy = s.ring + b * stage2;
                    if (live) {
                        __nv_bfloat16 h[2][8], m[2][8], l[2][8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const int sl = wc * 32 + grp * 8 + q;
                            // walkers past the CTA's range contribute exact zeros (their
                            // slots of wbuf are never written)
                            const cpx<float> y = sl < nw ? conj(tcur[q]) * s.wbuf[sl] : cpx<float>{0.f, 0.f};
                            kadd(bsx, bcx, y.x);
                            kadd(bsy, bcy, y.y);
                            split3(y.x, &h[0][q], &m[0][q], &l[0][q]);
                            split3(y.y, &h[1][q], &m[1][q], &l[1][q]);
                        }
                        const int nl = 2 * (j - jp0), nb = nl >> 7, r0 = nl & 127;
#pragma unroll
                        for (int cmp = 0; cmp < 2; ++cmp) {
                            const uint32_t o = koff(r0 + cmp, grp * 8);
                            *reinterpret_cast<uint4*>(sy + (0 * g.nbp + nb) * Y_BLK + o) = pack8(h[cmp]);
                            *reinterpret_cast<uint4*>(sy + (1 * g.nbp + nb) * Y_BLK + o) = pack8(m[cmp]);
                            *reinterpret_cast<uint4*>(sy + (2 * g.nbp + nb) * Y_BLK + o) = pack8(l[cmp]);
                        }
                    }
                    tc::fence_proxy_async();
                    mbar_arrive(&s.mb[FULL2 + b]);
#pragma unroll
                    for (int q = 0; q < 8; ++q) tcur[q] = tnxt[q];
                }
#undef FCG_FETCH_T
                // the pass's D2^T rows -> partial row (W part); b-sums
                wait_mb(&s.mb[D2FULL], u2 & 1, flag, a.bar, a.status);
                tc::fence_after_sync();
                const int lb = warp & 3, qd = (warp - 1) >> 2, row = 32 * lb + lane;
                for (int nb = 0; nb < nbq; ++nb) {
                    const int nl = 128 * nb + row, jj = jp0 + (nl >> 1), cmp = nl & 1;
                    for (int grp = qd; grp < g.Np / 16; grp += 4) {
                        float d[16];
                        tc::tmem_ld16(taddr + ((uint32_t)(32 * lb) << 16) + nb * g.Np + 16 * grp, d);
                        if (jj < M)
#pragma unroll
                            for (int q = 0; q < 16; ++q) {
                                const int i = 16 * grp + q;
                                if (i < N) a.part[2 * ((size_t)c * P + N + M + (size_t)i * M + jj) + cmp] = d[q];
                            }
                    }
                }
                s.xch[ct] = {bsx - bcx, bsy - bcy};
                compute_sync();
                if (ct < Jp && j < M) {
                    cpx<float> tot = s.xch[ct];
                    for (int r = 1; r < tpj; ++r) tot = tot + s.xch[ct + r * Jp];
                    a.part[2 * ((size_t)c * P + N + j)] = tot.x;
                    a.part[2 * ((size_t)c * P + N + j) + 1] = tot.y;
                }
                compute_sync();
            }
            g2 += g.nwc;
            u2 += 1;
            tc::fence_before_sync();
            __syncthreads();
            tc::fence_after_sync();
        }
        if (ct >= 0) {
            const double pv[1] = {ww};
            const int ps[1] = {S_WW};
            put_psc<1>(a.psc, c, pv, ps, s.red);
        }
        ok = grid_sync(a.bar, round++ * G, flag, a.status);
        if (!ok) break;

        // ================================================= slice phase
        if (warp == 1) {
            const int sl1[1] = {S_WW};
            double v1[1];
            sum_psc<1>(a.psc, G, sl1, v1);
            // delta = (u, A u) = (1/B) sum_s |w_s|^2 + lambda |u|^2; one thread
            // does the scalars (float64 divisions of all warps queue up)
            const double delta = v1[0] * invB + a.shift * uu;
            // (p, A p) by the recurrence, delta - beta^2 (p_prev, A p_prev); it holds
            // while the directions stay A-conjugate.  When rounding has eroded that
            // (float32-accurate products at a large condition number) it can come
            // out tiny or negative: then the recurrence restarts with beta = 0
            // (p = u, s = A u, a steepest-descent step, whose denominator delta
            // is a sum of squares).
            if (lane == 0) {
                const double beta0 = its == 0 ? 0.0 : gam / gam_prev;
                const double den = its == 0 ? delta : delta - beta0 * gam / alpha_prev;
                const bool restart = its == 0 || !(den > 1e-6 * delta);
                s.bc[5] = restart ? 0.0 : beta0;
                s.bc[8] = gam / (restart ? delta : den);
            }
        }
        __syncthreads();
        const double beta = s.bc[5], alpha = s.bc[8];
        if (ct >= 0) {
            double r2 = 0.0, gm = 0.0, our = 0.0, oui = 0.0, u2s = 0.0;
            // Row sums: a warp takes 32 neighbouring parameters and every
            // ng-th partial row, as many row groups as there are warps for.
            // Float64 work (a warp instruction takes the SM 16 cycles,
            // however many lanes are live) is then left to full warps.
            const int L = k1 - k0, cw = ct >> 5, nlw = (L + 31) >> 5, ng = nlw ? NCW / nlw : 1;
            const int rg = nlw ? cw / nlw : 0, kk = nlw ? 32 * (cw % nlw) + lane : 0, k = k0 + kk;
            const cpx<double> du = ubar - ccast<double>(ubar32);
            constexpr int BATCH = 19;
            double tx = 0.0, ty = 0.0;
            if (rg < ng && kk < L) {
                float sx = 0.f, sy = 0.f, cx = 0.f, cy = 0.f;
                // rows rg, rg + ng, ... with BATCH loads in flight
                for (int cb = rg; cb < G; cb += BATCH * ng) {
                    float2 v[BATCH];
#pragma unroll
                    for (int q = 0; q < BATCH; ++q) {
                        const int cc = cb + q * ng;
                        v[q] = cc < G ? *reinterpret_cast<const float2*>(a.part + 2 * ((size_t)cc * P + k))
                                      : make_float2(0.f, 0.f);
                    }
#pragma unroll
                    for (int q = 0; q < BATCH; ++q) {
                        kadd(sx, cx, v[q].x);
                        kadd(sy, cy, v[q].y);
                    }
                }
                tx = (double)sx - (double)cx;
                ty = (double)sy - (double)cy;
            }
            if (ng > 1) {
                s.tot[ct] = {tx, ty};
                compute_sync();
            }
            if (rg == 0 && kk < L) {
                // the row groups in a fixed order
                for (int r = 1; r < ng; ++r) {
                    tx += s.tot[ct + 32 * nlw * r].x;
                    ty += s.tot[ct + 32 * nlw * r].y;
                }
                const cpx<double> uk = s.d[kk] * s.r[kk];
                // (A u)_k = (S + lambda) u: the centred O^dag w with the
                // rounding of ubar put back
                const cpx<double> auk =
                    invB * cpx<double>{tx, ty} - conj(s.ob[kk]) * du + a.shift * uk;
                if (a.apply_only) {
                    Ap[k] = auk;
                } else {
                    const cpx<double> pk = uk + beta * s.p[kk];
                    const cpx<double> sk = auk + beta * s.sv[kk];
                    s.p[kk] = pk;
                    s.sv[kk] = sk;
                    s.x[kk] = s.x[kk] + alpha * pk;
                    const cpx<double> rk = s.r[kk] - alpha * sk;
                    s.r[kk] = rk;
                    const cpx<double> un = s.d[kk] * rk;
                    emit_p(a, k, un);
                    r2 += abs2(rk);
                    gm += cmulc(rk, un).x;
                    const cpx<double> ou = s.ob[kk] * un;
                    our += ou.x;
                    oui += ou.y;
                    u2s += abs2(un);
                }
            }
            if (!a.apply_only) {
                fence_proxy_async_global();
                const double pv[5] = {r2, gm, our, oui, u2s};
                const int ps[5] = {S_RR, S_GAM, S_OUR, S_OUI, S_UU};
                put_psc<5>(a.psc, c, pv, ps, s.red, rg == 0);
            }
        }
        gam_prev = gam;
        alpha_prev = alpha;
        ++its;
        if (a.apply_only) break;
        ok = grid_sync(a.bar, round++ * G, flag, a.status);
    }

    if (!a.apply_only && ct >= 0)
        for (int k = k0 + ct; k < k1; k += NCT) X[k] = s.x[k - k0];
    if (c == 0 && t == 32 && !a.apply_only) {
        a.scal[1] = ff;
        a.scal[2] = done ? 1.0 : 0.0;
        a.scal[3] = (double)its;
        a.scal[4] = rr;
    }
    // nothing of this CTA is in flight past here on the normal path; after an
    // abort, wait (bounded) for the copies it issued to land and for its last
    // MMA commits, before the shared memory and TMEM are released
    if (flag[0] && copier) {
        for (int b = 0; b < NS1; ++b)
            if (last1[b] >= 0) tc::mbar_wait(&s.mb[FULL1 + b], (last1[b] / NS1) & 1, WAIT_LIMIT);
        for (int b = 0; b < 2; ++b)
            if (last2[b] >= 0) tc::mbar_wait(&s.mb[FULL2 + b], (last2[b] >> 1) & 1, WAIT_LIMIT);
    }
    if (flag[0] && t == 0) {
        if (lastm1 >= 0)
            tc::mbar_wait(&s.mb[EMPTY1 + lastm1 % NS1], (lastm1 / NS1) & 1, WAIT_LIMIT);
        if (lastm2 >= 0) tc::mbar_wait(&s.mb[EMPTY2 + (lastm2 & 1)], (lastm2 >> 1) & 1, WAIT_LIMIT);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(taddr, 512u);
}

// ------------------------------------------------------------------ host

// W1 walker tiles of a CTA with wpc walkers: one, or pairs.
static int w1_tiles(int wpc) { return wpc > 128 ? 2 * ((wpc + 255) / 256) : 1; }

static bool fcg_geometry(const cr_ctx* c, int B, Geo* g) {
    const int N = c->N, M = c->M;
    if (c->prec != CR_MIXED || N > 256 || M > 256 || B < 1) return false;
    g->N = N;
    g->M = M;
    g->P = c->P;
    g->B = B;
    int G = (B + 31) / 32;
    if (c->fcg_ctas > 0 && c->fcg_ctas < G) G = c->fcg_ctas;  // the walker-block shape chosen
    const int Gp = (c->P + KS_MAX - 1) / KS_MAX;  // every CTA's CG slice fits in shared memory
    const int Gw = (B + MAX_WPC - 1) / MAX_WPC;   // and its walkers
    if (G < Gp) G = Gp;
    if (G < Gw) G = Gw;
    if (G > c->n_sm) G = c->n_sm;
    g->G = G;
    g->wpc = (B + G - 1) / G;
    if (g->wpc > MAX_WPC) return false;
    g->tpu = g->wpc > 128 ? 2 : 1;
    g->ntpc = w1_tiles(g->wpc);
    g->trows = (g->wpc + g->ntpc - 1) / g->ntpc;
    g->Kp = ((N + 31) / 32) * 32;
    g->nkc1 = g->Kp / 32;
    const int nc1 = ((2 * M + 15) / 16) * 16;
    g->npass1 = (nc1 + W1_W - 1) / W1_W;
    g->wlast1 = nc1 - W1_W * (g->npass1 - 1);
    g->Np = ((N + 15) / 16) * 16;
    g->nb2 = (2 * M + 127) / 128;
    g->nbp = g->nb2 < 2 ? g->nb2 : 2;
    g->npass2 = (g->nb2 + g->nbp - 1) / g->nbp;
    g->nwc = (g->wpc + 31) / 32;
    g->kslice = (g->P + G - 1) / G;
    if (g->kslice > KS_MAX) return false;
    const size_t r1 = (size_t)NS1 * W1_STAGE;
    const size_t r2 = 2 * ((size_t)g->nbp * 3 * Y_BLK + (size_t)g->Np * 64);
    g->ring = r1 > r2 ? r1 : r2;
    g->smem = g->ring + (size_t)KS_MAX * 88 + (size_t)MAX_WPC * 8 + 2 * 256 * 8 + NCT * 24 +
              8 * NCW * 8 + 10 * 8 + NMB * 8 + 16 + 16;
    return g->smem <= 227 * 1024;
}

// Workspace of the fused solve for up to max_walkers walkers (bytes per
// buffer), or false if the context is not covered.
bool fcg_supported(const cr_ctx* c) {
    Geo g;
    return fcg_geometry(c, c->max_walkers, &g);
}

void fcg_sizes(const cr_ctx* c, size_t* a1, size_t* b2, size_t* v2plane, size_t* part) {
    Geo g;
    fcg_geometry(c, c->max_walkers, &g);
    // the largest tile / chunk counts over walker counts up to max_walkers:
    // every CTA count G <= n_sm with wpc = ceil(B / G) <= ceil(max_walkers / G)
    size_t nt = 0, nc = 0;
    for (int G = 1; G <= c->n_sm; ++G) {
        const int wpc = (c->max_walkers + G - 1) / G;
        if (wpc > MAX_WPC) continue;
        const size_t t1 = (size_t)G * w1_tiles(wpc), t2 = (size_t)G * ((wpc + 31) / 32);
        if (t1 > nt) nt = t1;
        if (t2 > nc) nc = t2;
    }
    *a1 = nt * g.nkc1 * W1_A;
    *b2 = nc * (size_t)g.Np * 64;
    *v2plane = (size_t)W1_W * g.npass1 * g.Kp * 2;
    *part = (size_t)c->n_sm * c->P * 8;
}

cr_status fcg_prepare(cr_ctx* c) {
    cudaError_t e = cudaFuncSetAttribute(cg_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         227 * 1024);
    return e == cudaSuccess ? CR_OK : cr_fail(c, CR_ECUDA, "fcg_prepare: %s", cudaGetErrorString(e));
}

// One fused solve (apply_only = 0) or one product (S + shift I) v into
// cg[3P] (apply_only = 1).  redO: walker sums of O and |T|^2.
cr_status launch_cg_fused(cr_ctx* c, const int8_t* spins, const void* T, int B, const double* redO,
                          double shift, double tol, int maxit, int precond, int apply_only,
                          const double* v_in, void* u_out) {
    Args a;
    if (!fcg_geometry(c, B, &a.g)) return cr_fail(c, CR_EINVAL, "fused CG: unsupported shape");
    a.spins = spins;
    a.T = (const cpx<float>*)T;
    a.F = (const cpx<double>*)c->F;
    a.sO = (const cpx<double>*)redO;
    a.shift = shift;
    a.tol = tol;
    a.maxit = maxit;
    a.precond = precond;
    a.apply_only = apply_only;
    a.v_in = (const cpx<double>*)v_in;
    a.u_out = (cpx<float>*)u_out;
    a.cg = c->cg;
    a.a1 = c->fcg_a1;
    a.b2 = c->fcg_b2;
    a.v2 = c->fcg_v2;
    a.v2_plane = c->fcg_v2plane;
    a.vab = (cpx<float>*)c->fcg_vab;
    a.part = (float*)c->fcg_part;
    a.psc = c->fcg_psc;
    a.bar = c->fcg_bar;
    a.scal = c->scal;
    a.status = c->d_status;
    cudaError_t e = cudaMemsetAsync(c->fcg_bar, 0, 2 * sizeof(unsigned), c->stream);
    if (e != cudaSuccess) return cr_fail(c, CR_ECUDA, "fused CG: %s", cudaGetErrorString(e));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.g.G);
    cfg.blockDim = dim3(FC_THREADS);
    cfg.dynamicSmemBytes = a.g.smem;
    cfg.stream = c->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    CR_LAUNCH(c, CR_KERNEL_FCG, e = cudaLaunchKernelEx(&cfg, cg_fused_kernel, a));
    if (e != cudaSuccess) return cr_fail(c, CR_ECUDA, "cg_fused_kernel: %s", cudaGetErrorString(e));
    return cr_check_launch(c, "cg_fused_kernel");
}
