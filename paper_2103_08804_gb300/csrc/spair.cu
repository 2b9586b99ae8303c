// Explicit S of the natural-gradient update (Sec. III).
//
// With sigma_0 = t_0 = 1 in front of the spins and of T_j = tanh theta_j,
// every log-derivative is O_k = sigma_i t_j for one (i, j) other than (0, 0),
// so
//   sum_s conj(O_k) O_l = sum_s (sigma_i sigma_i') (conj(t_j) t_j')
// depends on the unordered spin pair {i, i'} (sigma^2 = 1: the pairs i = i'
// are all the row of ones) and on the pair (j, j') up to conjugation.  The
// P x P matrix of complex sums is therefore one real product
//   G[y][r] = sum_s Y_y(s) A_r(s),
//   A: 1 + N (N + 1) / 2 spin products, +-1, exact in one bf16 plane,
//   Y: (M + 1)^2 real columns, Re and Im of conj(t_j) t_j' (j < j') and
//      |t_j|^2, float32 values split into NPL bf16 terms,
// about P^2 / 2 x NPL multiply-adds per walker where the Gram matrix of
// [Re O | Im O] takes 2 P^2 x 6 (both of its operands need the split):
// eight times fewer for NPL = 3.  NPL = 3 holds all 24 bits of a float32;
// NPL = 2 (CR_CTX_S_BF16X3) is good to about 2^-17 per product.  That is the
// form of CR_MIXED contexts; the others form the same sums on the FMA pipes
// (spair_fma_kernel), an eighth of the additions of the P x P sums: float64
// in CR_FP64, two float32 words in CR_FP32 (products rounded to float32 as
// before; error-free additions, so that the two words hold the sum to about
// 2^-46; the float64 pipe does 1/64 of the float32 rate here).  Against 64 bits
// the float32 form's S has the error of float64 sums of the same products,
// 8.6e-9 of its norm (12 to 48 sites, 1024 to 32768 walkers); a Kahan sum,
// which rounds each corrected term, had 1.16e-8.
//
// TMEM accumulates in float32 with an error that grows with the number of
// MMAs added into one accumulator (measured: relative ~1e-8 each), so a
// tile is accumulated over chunks of 256 walkers (48 MMAs) in one TMEM half
// while the other half is added into float32 registers of the drain warps.
//
//   spair_a_kernel, spair_y_kernel   the operands, tiles of 32 walkers in the
//                                    K-major core-matrix layout
//   spair_tc_kernel                  G, tiles of 128 Y columns x 256 pairs
//   spair_mean_kernel                Obar = (sum_s O) / B
//   spair_expand_kernel              S = G / B - conj(Obar) Obar^T + shift I
//
// The MMA's M side takes Y (three planes) and its N side the pairs (one
// plane): 40 KB of operands per 32 walkers and tile; the other way round it
// would be 56 KB, and L2 already delivers 14 TB/s of them.  At N = M = 100 and 32768 walkers the whole explicit-S solve went from
// 203.4 to 102.7 ms with this in place of the Gram matrix of [Re O | Im O]
// (111 ms), the error of the update from 3.6e-7 to 3.0e-7.
#include <cuda_bf16.h>

#include "common.cuh"
#include "tc.cuh"

namespace {

constexpr uint32_t WAIT_LIMIT = 1u << 26;  // bounded mbarrier polls
constexpr int KC = 32;                      // walkers per operand tile
constexpr int CHUNK = 8;                    // operand tiles per TMEM accumulation
constexpr int YT = 128, AT = 256;           // tile of G: Y columns x pairs
constexpr int Y_TILE = YT * KC * 2;         // bytes of one plane
constexpr int A_TILE = AT * KC * 2;
constexpr int SP_THREADS = 320;             // warp 0 issues MMAs, 1-8 drain, 9 copies
constexpr size_t OPERAND_BUDGET = (size_t)3 << 30;  // bytes of operands held at once

template <int NPL> struct Ring {
    static constexpr int STAGE = NPL * Y_TILE + A_TILE;
    static constexpr int NSTG = 5;
    static constexpr size_t SMEM = (size_t)NSTG * STAGE + 256;
};

CR_D void split3(float x, __nv_bfloat16* hi, __nv_bfloat16* mid, __nv_bfloat16* lo) {
    *hi = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(*hi);
    *mid = __float2bfloat16_rn(r1);
    *lo = __float2bfloat16_rn(r1 - __bfloat162float(*mid));
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

// Pairs a < b numbered b (b - 1) / 2 + a.
CR_HD int pair_index(int a, int b) { return b * (b - 1) / 2 + a; }
CR_D void pair_of(int p, int* a, int* b) {
    int y = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)p)) * 0.5f);
    while (y * (y - 1) / 2 > p) --y;
    while ((y + 1) * y / 2 <= p) ++y;
    *b = y;
    *a = p - y * (y - 1) / 2;
}

struct PairGeo {
    int nA, nY;          // rows of A (pairs and the ones), columns of Y
    int nab, nyb;        // blocks of 256 and 128
    int ntiles, nseg;    // tiles of G, K segments
    int slab;            // walkers per pass over the operands (a multiple of 256)
    size_t a_bytes, y_bytes, g_elems;  // operands of a slab; elements of one G
};

int npl_of(const cr_ctx* c) { return (c->flags & CR_CTX_S_BF16X3) ? 2 : 3; }

PairGeo pair_geometry(const cr_ctx* c) {
    PairGeo g;
    g.nA = 1 + c->N * (c->N + 1) / 2;
    g.nY = (c->M + 1) * (c->M + 1);
    g.nab = (g.nA + AT - 1) / AT;
    g.nyb = (g.nY + YT - 1) / YT;
    g.ntiles = g.nab * g.nyb;
    constexpr int CW = KC * CHUNK;
    const size_t per = 2 * ((size_t)g.nab * AT + (size_t)npl_of(c) * g.nyb * YT);  // bytes a walker
    const int nch = (c->max_walkers + CW - 1) / CW;
    size_t fit = OPERAND_BUDGET / (per * CW);
    if (fit < 1) fit = 1;
    const int chunks = (size_t)nch < fit ? nch : (int)fit;
    g.slab = chunks * CW;
    // few tiles: split the walkers so that every SM has an item, a chunk at least each
    g.nseg = c->n_sm / g.ntiles;
    if (g.nseg > chunks) g.nseg = chunks;
    if (g.nseg < 1) g.nseg = 1;
    g.a_bytes = (size_t)g.nab * AT * g.slab * 2;
    g.y_bytes = (size_t)npl_of(c) * g.nyb * YT * g.slab * 2;
    g.g_elems = (size_t)g.nab * AT * g.nyb * YT;
    return g;
}

// A tiles: [block of 256 pairs][32 walkers], pair r < N (N + 1) / 2 is
// (i, i') of the extended spins, the last one is the row of ones; zero past
// the walkers and the pairs.  Grid (walker tile, pair block); the walkers'
// spins are staged once, extended by sigma_0 = 1.
__global__ void __launch_bounds__(256) spair_a_kernel(const int8_t* __restrict__ spins, int s0,
                                                      int B, int N, int nA, int nkc,
                                                      unsigned char* __restrict__ A) {
    extern __shared__ __align__(1024) unsigned char sm[];
    int8_t* sg = (int8_t*)sm;  // [N + 1][KC]
    const int kc = blockIdx.x, ab = blockIdx.y, t = threadIdx.x;
    for (int e = t; e < KC * (N + 1); e += blockDim.x) {
        const int w = e / (N + 1), i = e % (N + 1), s = s0 + kc * KC + w;
        sg[i * KC + w] = s < B ? (i == 0 ? (int8_t)1 : spins[(size_t)s * N + i - 1]) : (int8_t)0;
    }
    __syncthreads();
    unsigned char* out = A + ((size_t)ab * nkc + kc) * A_TILE;
    for (int e = t; e < AT * (KC / 8); e += blockDim.x) {
        const int r = e % AT, grp = e / AT, p = ab * AT + r;
        int a = 0, b = 0;
        if (p < nA - 1) pair_of(p, &a, &b);
        __nv_bfloat16 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int x = sg[a * KC + grp * 8 + q] * sg[b * KC + grp * 8 + q];  // (0, 0): ones
            v[q] = __float2bfloat16_rn(p < nA ? (float)x : 0.f);
        }
        *reinterpret_cast<uint4*>(out + tc::kmajor_offset(r, grp * 8, KC)) = pack8(v);
    }
}

// Y tiles: [block of 128 columns][32 walkers][plane].  Columns 2 p and 2 p + 1
// are Re and Im of conj(t_j) t_j' of pair p = (j, j') of the extended hidden
// units; the M + 1 columns from M (M + 1) on are |t_j|^2.  A thread forms two
// adjacent columns of 8 walkers.  Grid (walker tile, column block).
template <int NPL>
__global__ void __launch_bounds__(256) spair_y_kernel(const cpx<float>* __restrict__ T, int s0,
                                                      int B, int M, int nY, int nkc,
                                                      unsigned char* __restrict__ Y) {
    const int kc = blockIdx.x, yb = blockIdx.y, t = threadIdx.x;
    const int c2 = t & 63, grp = t >> 6;  // column pair of the block, 8 walkers
    const int y = yb * YT + 2 * c2, nOff = M * (M + 1);
    int j[2] = {0, 0}, jp[2] = {0, 0};
    const bool off = y < nOff;
    if (off) {
        pair_of(y >> 1, &j[0], &jp[0]);
    } else {
        j[0] = jp[0] = y - nOff;  // nOff is even: both columns are |t|^2
        j[1] = jp[1] = y + 1 - nOff;
    }
    __nv_bfloat16 h[2][8], m[2][8], l[2][8];
    const cpx<float> one = {1.f, 0.f}, zero = {0.f, 0.f};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int s = s0 + kc * KC + grp * 8 + q;
        const cpx<float>* Ts = T + (size_t)s * M - 1;  // t_j = Ts[j], j >= 1
        float x0 = 0.f, x1 = 0.f;
        if (s < B && y < nY) {
            if (off) {
                const cpx<float> a = j[0] ? ldg(Ts + j[0]) : one, b = ldg(Ts + jp[0]);
                const cpx<float> v = cmulc(a, b);
                x0 = v.x;
                x1 = v.y;
            } else {
                x0 = j[0] ? abs2(ldg(Ts + j[0])) : 1.f;
                const cpx<float> b = y + 1 < nY ? ldg(Ts + j[1]) : zero;
                x1 = abs2(b);
            }
        }
        split3(x0, &h[0][q], &m[0][q], &l[0][q]);
        split3(x1, &h[1][q], &m[1][q], &l[1][q]);
    }
    unsigned char* out = Y + ((size_t)yb * nkc + kc) * NPL * Y_TILE;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const uint32_t o = tc::kmajor_offset(2 * c2 + k, grp * 8, KC);
        *reinterpret_cast<uint4*>(out + o) = pack8(h[k]);
        *reinterpret_cast<uint4*>(out + Y_TILE + o) = pack8(m[k]);
        if (NPL == 3) *reinterpret_cast<uint4*>(out + 2 * Y_TILE + o) = pack8(l[k]);
    }
}

struct PairArgs {
    const unsigned char* A;
    const unsigned char* Y;
    int nkc;           // walker tiles of the operands
    int kseg, nseg;    // walker tiles per item (the last segment may have fewer), segments
    int nab, nyb;
    float* G;          // [nseg][pair][Y column]
    int add;           // a later slab: add to G
    int* status;
};

// Persistent, one CTA per SM; an item is one tile of G over one K segment,
// items segment-major and pair blocks fastest, so that the CTAs running
// together read few Y blocks.  Warp 9 (one thread) copies an operand stage
// with two bulk copies, running ahead across items; warp 0 (one thread)
// issues the MMAs, chunk c to TMEM columns [256 (c % 2), +256); warps 1-8
// drain.  Bound by the MMAs (six of 128 x 256 x 16 a stage).  While one thread
// did copies and MMAs, dividing for its cursor and ring positions, that thread
// was the bound: 10 x 10 lattice, alpha = 1, 32768 walkers 10.3 ms, now 5.1.
template <int NPL>
__global__ void __launch_bounds__(SP_THREADS, 1) spair_tc_kernel(const PairArgs a) {
    using RG = Ring<NPL>;
    constexpr int NSTG = RG::NSTG;
    extern __shared__ __align__(1024) unsigned char sm[];
    uint64_t* full = (uint64_t*)(sm + NSTG * RG::STAGE);
    uint64_t* empty = full + NSTG;      // [NSTG] MMAs reading a stage done
    uint64_t* cdone = full + 2 * NSTG;  // [2] MMAs of a chunk done (per TMEM half)
    uint64_t* drained = cdone + 2;      // [2] TMEM half read by the 256 drain threads
    uint32_t* slot = (uint32_t*)(drained + 2);
    volatile int* abort = (volatile int*)(slot + 1);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) {
        for (int i = 0; i < 2 * NSTG + 2; ++i) tc::mbar_init(&full[i], 1);
        tc::mbar_init(&drained[0], 256);
        tc::mbar_init(&drained[1], 256);
        tc::fence_mbar_init();
        *abort = 0;
    }
    if (warp == 0) {
        tc::tmem_alloc(slot, 512u);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t taddr = *slot;
    const int ntiles = a.nab * a.nyb, nitems = ntiles * a.nseg;
    auto wait = [&](uint64_t* bar, uint32_t par) {
        for (int i = 0; i < 64; ++i) {
            if (tc::mbar_wait(bar, par, WAIT_LIMIT >> 6)) return true;
            if (*abort) return false;
        }
        *abort = 1;
        return false;
    };
    // walker tiles [k0, k1) of an item
    auto krange = [&](int item, int* k0, int* k1) {
        *k0 = (item / ntiles) * a.kseg;
        *k1 = min(a.nkc, *k0 + a.kseg);
    };
    if (warp == 0) {
        if (lane == 0) {
            const uint32_t idesc = tc::make_idesc_bf16(YT, AT);
            const uint64_t d0 = tc::make_desc(tc::smem_u32(sm), 128, 16 * KC);
            uint32_t b = 0, ph = 0, gc = 0;
            int last = -1, lastph = 0;  // stage of the last commit
            bool ok = true;
            for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
                int k0, k1;
                krange(item, &k0, &k1);
                for (int kc = k0; kc < k1 && ok; kc += CHUNK, ++gc) {
                    const uint32_t h = gc & 1, dt = taddr + h * 256;
                    // the TMEM half of chunk gc was last used by chunk gc - 2
                    if (gc >= 2 && !wait(&drained[h], ((gc >> 1) - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    const int n = min(CHUNK, k1 - kc);
                    for (int k = 0; k < n; ++k) {
                        if (!wait(&full[b], ph)) {
                            ok = false;
                            break;
                        }
                        tc::fence_after_sync();
                        const uint64_t yd = d0 + b * (uint32_t)(RG::STAGE >> 4);
                        const uint64_t ad = yd + (NPL * Y_TILE >> 4);
#pragma unroll
                        for (int ks = 0; ks < KC / 16; ++ks)
#pragma unroll
                            for (int pl = 0; pl < NPL; ++pl)
                                tc::mma_bf16(dt, yd + (pl * (Y_TILE >> 4) + ks * 16), ad + ks * 16, idesc,
                                             k != 0 || ks != 0 || pl != 0);
                        tc::commit(&empty[b]);
                        last = (int)b;
                        lastph = (int)ph;
                        if (++b == NSTG) {
                            b = 0;
                            ph ^= 1;
                        }
                    }
                    if (ok) tc::commit(&cdone[h]);
                }
            }
            if (!ok) {
                *abort = 1;
                set_status(a.status, CR_ETIMEOUT);
                // let issued MMAs finish (bounded)
                if (last >= 0) tc::mbar_wait(&empty[last], (uint32_t)lastph, WAIT_LIMIT);
            }
        }
        __syncwarp();
    } else if (warp == SP_THREADS / 32 - 1) {
        if (lane == 0) {
            uint32_t b = 0, ph = 0, g = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
                int k0, k1;
                krange(item, &k0, &k1);
                const int tile = item % ntiles, ab = tile % a.nab, yb = tile / a.nab;
                const unsigned char* ys = a.Y + ((size_t)yb * a.nkc + k0) * NPL * Y_TILE;
                const unsigned char* as = a.A + ((size_t)ab * a.nkc + k0) * A_TILE;
                for (int kc = k0; kc < k1; ++kc, ++g, ys += NPL * Y_TILE, as += A_TILE) {
                    if (g >= NSTG && !wait(&empty[b], ph ^ 1)) {
                        ok = false;
                        break;
                    }
                    unsigned char* st = sm + (size_t)b * RG::STAGE;
                    tc::mbar_expect_tx(&full[b], (uint32_t)RG::STAGE);
                    tc::bulk_g2s(st, ys, NPL * Y_TILE, &full[b]);
                    tc::bulk_g2s(st + NPL * Y_TILE, as, A_TILE, &full[b]);
                    if (++b == NSTG) {
                        b = 0;
                        ph ^= 1;
                    }
                }
            }
            // every copy lands before the CTA leaves (bounded): the last NSTG
            // stages; where MMAs consumed them all this does not wait
            for (uint32_t q = 0; q < NSTG && q < g; ++q) {
                if (b == 0) ph ^= 1;
                b = b == 0 ? NSTG - 1 : b - 1;
                tc::mbar_wait(&full[b], ph, WAIT_LIMIT);
            }
        }
        __syncwarp();
    } else {
        // drain: warp w reads TMEM lanes 32 (w % 4) .. + 31 (Y columns) and
        // the 128 pairs from 128 c2 on, c2 = (w - 1) / 4
        const int lb = warp & 3, c2 = (warp - 1) >> 2;
        const size_t ldg_ = (size_t)a.nyb * YT;
        bool ok = true;
        int gc = 0;
        for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
            int k0, k1;
            krange(item, &k0, &k1);
            const int tile = item % ntiles, ab = tile % a.nab, yb = tile / a.nab;
            float acc[128];
#pragma unroll
            for (int q = 0; q < 128; ++q) acc[q] = 0.f;
            for (int kc = k0; kc < k1; kc += CHUNK, ++gc) {
                const uint32_t h = gc & 1;
                // warp-uniform outcome: tcgen05.ld below is a warp-wide instruction
                if (!__all_sync(0xffffffffu, wait(&cdone[h], (gc >> 1) & 1))) {
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
#pragma unroll
                for (int ch = 0; ch < 8; ++ch) {
                    float v[16];
                    tc::tmem_ld16(taddr + ((uint32_t)(32 * lb) << 16) + h * 256 + 128 * c2 + 16 * ch, v);
#pragma unroll
                    for (int q = 0; q < 16; ++q) acc[16 * ch + q] = __fadd_rn(acc[16 * ch + q], v[q]);
                }
                tc::fence_before_sync();
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(
                                 tc::smem_u32(&drained[h]))
                             : "memory");
            }
            if (!ok) break;
            // lanes hold consecutive Y columns: coalesced rows of G
            float* out = a.G + (size_t)(item / ntiles) * a.nab * AT * ldg_ +
                         ((size_t)ab * AT + 128 * c2) * ldg_ + (size_t)yb * YT + 32 * lb + lane;
            if (a.add) {
#pragma unroll
                for (int q = 0; q < 128; ++q) out[q * ldg_] = __fadd_rn(out[q * ldg_], acc[q]);
            } else {
#pragma unroll
                for (int q = 0; q < 128; ++q) out[q * ldg_] = acc[q];
            }
        }
        if (!ok && t == 32) set_status(a.status, CR_ETIMEOUT);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(taddr, 512u);
}

// extended (i, j) of parameter k
CR_D void param_of(int k, int N, int M, int* i, int* j) {
    if (k < N) {
        *i = k + 1;
        *j = 0;
    } else if (k < N + M) {
        *i = 0;
        *j = k - N + 1;
    } else {
        *i = (k - N - M) / M + 1;
        *j = (k - N - M) % M + 1;
    }
}

// Obar in float64, formed once: the float64 pipe is what the expansion waits
// for.
__global__ void spair_mean_kernel(const double* __restrict__ redO, int P, int B, double* __restrict__ ob) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < P) ((cpx<double>*)ob)[k] = (1.0 / B) * ((const cpx<double>*)redO)[k];
}

// S of the 32 x 32 tile (by, bx), bx <= by, and its mirror image: S_kl of
// the lower triangle from the segments' sums (float64, in segment order),
// the upper triangle its exact conjugate.
template <typename T>
__global__ void __launch_bounds__(256) spair_expand_kernel(const T* __restrict__ G, int nseg,
                                                           size_t seg_stride, size_t ld, int N,
                                                           int M, int P, int B,
                                                           const double* __restrict__ ob_,
                                                           double shift, double* __restrict__ S_) {
    const int bx = blockIdx.x, by = blockIdx.y;
    if (bx > by) return;
    __shared__ cpx<double> tl[32][33];
    const cpx<double>* ob = (const cpx<double>*)ob_;
    cpx<double>* S = (cpx<double>*)S_;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const double inv = 1.0 / B;
    const int l = bx * 32 + tx, nA = 1 + N * (N + 1) / 2, nOff = M * (M + 1);
    int il = 0, jl = 0;
    cpx<double> ol = {0.0, 0.0};
    if (l < P) {
        param_of(l, N, M, &il, &jl);
        ol = ob[l];
    }
    for (int q = ty; q < 32; q += 8) {
        const int k = by * 32 + q;
        if (k >= P || l >= P) continue;
        int ik, jk;
        param_of(k, N, M, &ik, &jk);
        const int row = ik == il ? nA - 1 : pair_index(min(ik, il), max(ik, il));
        const T* g = G + (size_t)row * ld;
        cpx<double> v = {0.0, 0.0};
        if (jk == jl) {
            v.x = (double)g[nOff + jk];
            for (int sg = 1; sg < nseg; ++sg) v.x += (double)g[sg * seg_stride + nOff + jk];
        } else {
            const int y = 2 * pair_index(min(jk, jl), max(jk, jl));
            v = ccast<double>(*reinterpret_cast<const cpx<T>*>(g + y));
            for (int sg = 1; sg < nseg; ++sg)
                v = v + ccast<double>(*reinterpret_cast<const cpx<T>*>(g + sg * seg_stride + y));
            if (jk > jl) v = conj(v);  // the sum held is that of conj(t_jl) t_jk
        }
        const cpx<double> m = cmulc(ob[k], ol);
        v = {fma(inv, v.x, -m.x), fma(inv, v.y, -m.y)};
        if (k == l) v = {v.x + shift, 0.0};
        tl[q][tx] = v;
        if (l <= k) S[(size_t)k * P + l] = v;
    }
    __syncthreads();
    for (int q = ty; q < 32; q += 8) {
        const int r = bx * 32 + q, c = by * 32 + tx;  // mirror: row r, column c, r < c
        if (r < P && c < P && r < c) S[(size_t)r * P + c] = conj(tl[tx][q]);
    }
}

// The pair sums on the FMA pipes: a tile of 8 Q pairs x 16 Q columns of Y per
// CTA and K segment, 8 x 16 threads with Q x Q sums each.  32 walkers at a
// time, their spin products and tanh products formed in shared memory.
// Float32: products rounded to float32, sums s + c by two-sum (Knuth, The Art
// of Computer Programming vol. 2, 4.2.2); float64: plain sums, Q = 2, so that
// small systems still spread over the SMs.
template <typename R> struct FmaTile { static constexpr int Q = sizeof(R) == 4 ? 4 : 2; };
constexpr int FMA_W = 32;

template <typename R>
__global__ void __launch_bounds__(128) spair_fma_kernel(const int8_t* __restrict__ spins,
                                                        const cpx<R>* __restrict__ T, int B, int N,
                                                        int M, int nA, int nY, int seg_walkers,
                                                        double* __restrict__ G, size_t seg_stride) {
    constexpr int Q = FmaTile<R>::Q, TI = 8 * Q, TJ = 16 * Q;
    __shared__ R as[FMA_W][TI];
    __shared__ __align__(16) R ys[FMA_W][TJ];
    __shared__ int2 pa[TI], py[TJ / 2];
    const int y0 = blockIdx.x * TJ, a0 = blockIdx.y * TI, seg = blockIdx.z;
    const int s0 = seg * seg_walkers, s1 = min(B, s0 + seg_walkers);
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4, nOff = M * (M + 1);
    if (t < TI) {
        int a = 0, b = 0;
        if (a0 + t < nA - 1) pair_of(a0 + t, &a, &b);
        pa[t] = make_int2(a, b);
    }
    for (int e = t; e < TJ / 2; e += 128) {
        const int y = y0 + 2 * e;
        int a, b;
        if (y < nOff) pair_of(y >> 1, &a, &b);
        else { a = y - nOff; b = a + 1; }  // two squares |t_a|^2, |t_b|^2
        py[e] = make_int2(a, b);
    }
    R acc[Q][Q], cmp[Q][Q];
#pragma unroll
    for (int p = 0; p < Q; ++p)
#pragma unroll
        for (int q = 0; q < Q; ++q) acc[p][q] = cmp[p][q] = R(0);
    const cpx<R> one = {R(1), R(0)}, zero = {R(0), R(0)};
    for (int sb = s0; sb < s1; sb += FMA_W) {
        __syncthreads();
        for (int e = t; e < FMA_W * TI; e += 128) {
            const int w = e / TI, r = e % TI, s = sb + w;
            R v = R(0);
            if (s < s1 && a0 + r < nA) {
                const int2 p = pa[r];
                const int8_t* sp = spins + (size_t)s * N - 1;
                v = R((p.x ? sp[p.x] : 1) * (p.y ? sp[p.y] : 1));
            }
            as[w][r] = v;
        }
        for (int e = t; e < FMA_W * TJ / 2; e += 128) {
            const int w = e / (TJ / 2), c = e % (TJ / 2), s = sb + w, y = y0 + 2 * c;
            cpx<R> v = zero;
            if (s < s1 && y < nY) {
                const int2 p = py[c];
                const cpx<R>* ts = T + (size_t)s * M - 1;
                const cpx<R> a = p.x ? ldg(ts + p.x) : one;
                const cpx<R> b = y < nOff || y + 1 < nY ? ldg(ts + p.y) : zero;
                v = y < nOff ? cmulc(a, b) : cpx<R>{abs2(a), abs2(b)};
            }
            ys[w][2 * c] = v.x;
            ys[w][2 * c + 1] = v.y;
        }
        __syncthreads();
        const int nw = min(FMA_W, s1 - sb);
#pragma unroll 4
        for (int w = 0; w < nw; ++w) {
            R av[Q], yv[Q];
#pragma unroll
            for (int p = 0; p < Q; ++p) av[p] = as[w][ty + 8 * p];
#pragma unroll
            for (int q = 0; q < Q; ++q) yv[q] = ys[w][Q * tx + q];
#pragma unroll
            for (int p = 0; p < Q; ++p)
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    if constexpr (sizeof(R) == 8) {
                        acc[p][q] = fma(av[p], yv[q], acc[p][q]);
                    } else {
                        // (av = +-1: the product is exact)
                        const R x = __fmul_rn(av[p], yv[q]), u = __fadd_rn(acc[p][q], x);
                        const R z = __fsub_rn(u, acc[p][q]);
                        cmp[p][q] = __fadd_rn(cmp[p][q], __fadd_rn(__fsub_rn(acc[p][q], __fsub_rn(u, z)),
                                                                   __fsub_rn(x, z)));
                        acc[p][q] = u;
                    }
                }
        }
    }
    double* out = G + seg * seg_stride;
#pragma unroll
    for (int p = 0; p < Q; ++p)
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int r = a0 + ty + 8 * p, y = y0 + Q * tx + q;
            if (r < nA && y < nY) out[(size_t)r * (nY + (nY & 1)) + y] = (double)acc[p][q] + (double)cmp[p][q];
        }
}

// Grid of the FMA form: segments of whole 32-walker stages, about four CTAs
// per SM, their sums held at once.
struct FmaGeo {
    int nA, nY, ga, gy, nseg, seg_walkers;
    size_t ld, seg_stride;
};

FmaGeo fma_geometry(const cr_ctx* c) {
    FmaGeo g;
    const int Q = c->prec == CR_FP64 ? FmaTile<double>::Q : FmaTile<float>::Q;
    g.nA = 1 + c->N * (c->N + 1) / 2;
    g.nY = (c->M + 1) * (c->M + 1);
    g.ga = (g.nA + 8 * Q - 1) / (8 * Q);
    g.gy = (g.nY + 16 * Q - 1) / (16 * Q);
    const long long tiles = (long long)g.ga * g.gy;
    const int stages = (c->max_walkers + FMA_W - 1) / FMA_W;
    long long ns = (4LL * c->n_sm + tiles - 1) / tiles;
    if (ns > stages) ns = stages;
    const int per = (int)((stages + ns - 1) / ns);
    g.nseg = (stages + per - 1) / per;
    g.seg_walkers = per * FMA_W;
    g.ld = g.nY + (g.nY & 1);
    g.seg_stride = (size_t)g.nA * g.ld;
    return g;
}

template <typename T>
cr_status expand(cr_ctx* c, const T* G, int nseg, size_t seg_stride, size_t ld, int B,
                 const double* redO, double shift) {
    const int P = c->P, nt = (P + 31) / 32;
    double* ob = c->cg;  // the solution vectors are not in use yet
    CR_LAUNCH(c, CR_K_OTHER, spair_mean_kernel<<<(P + 255) / 256, 256, 0, c->stream>>>(redO, P, B, ob));
    CR_LAUNCH(c, CR_K_OTHER, spair_expand_kernel<T><<<dim3(nt, nt), 256, 0, c->stream>>>(
                                 G, nseg, seg_stride, ld, c->N, c->M, P, B, ob, shift, c->S));
    return cr_check_launch(c, "explicit S");
}

template <typename R>
cr_status spair_fma_t(cr_ctx* c, const int8_t* spins, const void* T, int B, const double* redO,
                      double shift) {
    const FmaGeo g = fma_geometry(c);
    const int nseg = (B + g.seg_walkers - 1) / g.seg_walkers;
    double* G = (double*)c->spair_g;
    CR_LAUNCH(c, CR_KERNEL_SBUILD, spair_fma_kernel<R><<<dim3(g.gy, g.ga, nseg), 128, 0, c->stream>>>(
                                       spins, (const cpx<R>*)T, B, c->N, c->M, g.nA, g.nY,
                                       g.seg_walkers, G, g.seg_stride));
    return expand<double>(c, G, nseg, g.seg_stride, g.ld, B, redO, shift);
}

template <int NPL>
cr_status spair_t(cr_ctx* c, const int8_t* spins, const void* T, int B, const double* redO,
                  double shift) {
    const PairGeo g = pair_geometry(c);
    const int N = c->N, M = c->M;
    constexpr int CW = KC * CHUNK;
    int nseg = 0, cps = 0;  // segments and chunks per segment of the first slab
    for (int s0 = 0; s0 < B; s0 += g.slab) {
        const int nw = B - s0 < g.slab ? B - s0 : g.slab;
        const int nch = (nw + CW - 1) / CW, nkc = nch * CHUNK;
        if (s0 == 0) {
            nseg = g.nseg < nch ? g.nseg : nch;
            cps = (nch + nseg - 1) / nseg;
            nseg = (nch + cps - 1) / cps;
        }
        // later slabs keep the first one's segment length: never more segments
        const int sg = (nch + cps - 1) / cps;
        CR_LAUNCH(c, CR_K_OTHER,
                  spair_a_kernel<<<dim3(nkc, g.nab), 256, KC * (N + 1), c->stream>>>(
                      spins, s0, B, N, g.nA, nkc, c->Xt));
        CR_LAUNCH(c, CR_K_OTHER,
                  spair_y_kernel<NPL><<<dim3(nkc, g.nyb), 256, 0, c->stream>>>(
                      (const cpx<float>*)T, s0, B, M, g.nY, nkc, c->Xt + g.a_bytes));
        PairArgs a;
        a.A = c->Xt;
        a.Y = c->Xt + g.a_bytes;
        a.nkc = nkc;
        a.kseg = cps * CHUNK;
        a.nseg = sg;
        a.nab = g.nab;
        a.nyb = g.nyb;
        a.G = c->spair_g;
        a.add = s0 > 0;
        a.status = c->d_status;
        const int items = g.ntiles * sg, grid = items < c->n_sm ? items : c->n_sm;
        CR_LAUNCH(c, CR_KERNEL_SBUILD,
                  spair_tc_kernel<NPL><<<grid, SP_THREADS, Ring<NPL>::SMEM, c->stream>>>(a));
    }
    return expand<float>(c, c->spair_g, nseg, g.g_elems, (size_t)g.nyb * YT, B, redO, shift);
}

}  // namespace

void spair_sizes(const cr_ctx* c, size_t* x_bytes, size_t* g_bytes) {
    if (c->prec != CR_MIXED) {
        const FmaGeo g = fma_geometry(c);
        *x_bytes = 0;
        *g_bytes = (size_t)g.nseg * g.seg_stride * sizeof(double);
        return;
    }
    const PairGeo g = pair_geometry(c);
    *x_bytes = g.a_bytes + g.y_bytes;
    *g_bytes = (size_t)g.nseg * g.g_elems * sizeof(float);
}

cr_status spair_prepare(cr_ctx* c) {
    cudaError_t e = cudaFuncSetAttribute(spair_tc_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Ring<2>::SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(spair_tc_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)Ring<3>::SMEM);
    return e == cudaSuccess ? CR_OK : cr_fail(c, CR_ECUDA, "spair_prepare: %s", cudaGetErrorString(e));
}

// S + shift I into c->S (full Hermitian, float64).
cr_status launch_sbuild(cr_ctx* c, const int8_t* spins, const void* T, int B, const double* redO,
                        double shift) {
    if (c->prec == CR_FP64) return spair_fma_t<double>(c, spins, T, B, redO, shift);
    if (c->prec == CR_FP32) return spair_fma_t<float>(c, spins, T, B, redO, shift);
    return npl_of(c) == 2 ? spair_t<2>(c, spins, T, B, redO, shift)
                          : spair_t<3>(c, spins, T, B, redO, shift);
}
