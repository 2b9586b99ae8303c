// Direct shifted solve (S + lambda I) x = F of the natural-gradient update
// (Sec. III): blocked right-looking Cholesky S = L L^dag on many CTAs, then
// iterative refinement in float64.
//
// S (float64, full Hermitian, shift on its diagonal) stays untouched; its
// lower triangle is copied into the factor buffer and factored in place.
// Float64 contexts factor in float64 (chol64.cu).  The others factor in
// float32, in 64-column panels.  Per panel J:
//   potrf_inv_kernel  L_JJ = chol(A_JJ) and X_JJ = L_JJ^-1   (one CTA, registers)
//   trsm_kernel       L_IJ = A_IJ X_JJ^dag, I > J             (64 x 64 tiles)
//   syrk_tc_kernel    A_IK -= L_IJ L_KJ^dag, J < K <= I       (mixed: tcgen05)
//   syrk_kernel       the same on the FMA pipes               (float32)
// (mixed: the first panel of a pair updates the second's columns only, and
// the rest of A is read and written once per pair)
// The inverses X_JJ turn the panel's triangular solve into a product, and,
// merged pairwise into the inverses of 512 x 512 diagonal blocks, the
// triangular solves of the refinement into two products per 512 rows.
//
// The solve with a float32 factor (and float32 arithmetic in the triangular
// solves) is accurate to about kappa * 2^-24, so it is refined in float64
// (Wilkinson's iterative refinement; the residual is formed in float64):
//   x = 0, r = F;  repeat { d = L^{-dag} L^{-1} r;  x += d;  r = F - S x }
// until |r| <= REFINE_TOL |F|, the residual stops shrinking (by 2x), or
// REFINE_MAXIT steps.  Float64 contexts up to CHOL_SMALL_P parameters take
// the float64 solve without refinement.  Every later launch of a refinement
// step returns at once when the done flag is set, so the launch sequence is
// fixed (graph-capturable).
#include <cuda_bf16.h>

#include "common.cuh"
#include "tc.cuh"

namespace {

using cf = cpx<float>;

constexpr int NB = 64;
constexpr int SB = 512;                     // rows of a merged diagonal inverse
constexpr int REFINE_MAXIT = 10;
constexpr double REFINE_TOL = 1e-12;
constexpr int RES_ROWS = 2;    // rows of S a warp of the residual kernel reads at once

// L is held as [lrows(P)][lcols(P)], rows and columns past P zero, so that
// the tensor-core update needs no masks and every row starts on 128 bytes.
CR_HD int lcols(int P) { return (P + NB - 1) / NB * NB; }
CR_HD int lrows(int P) { return lcols(P) + 256; }  // a 256-row tile may start at any 64

// L <- S in float32 (only the lower triangle is used).
__global__ void chol_copy_kernel(const double* __restrict__ S_, int P, cf* __restrict__ L) {
    // (rows on the grid's x axis: there may be more than its y axis holds)
    const int k = blockIdx.y * blockDim.x + threadIdx.x, i = blockIdx.x, ld = lcols(P);
    if (k >= ld) return;
    L[(size_t)i * ld + k] = i < P && k < P ? ccast<float>(((const cpx<double>*)S_)[(size_t)i * P + k])
                                           : cf{0.f, 0.f};
}

// Merged inverses: X holds one [SB][SB] block per SB rows of L.
CR_D cf* xblock(cf* X, int row) {
    return X + (size_t)(row / SB) * SB * SB + (size_t)(row % SB) * SB + row % SB;
}

// Factor the diagonal block J and invert the factor, 16 x 16 threads with 4
// x 4 entries each (rows ty + 16 a, columns tx + 16 b) in registers.  At
// column j the entries of columns k > j belong to the block still to be
// factored and those of columns k <= j to the inverse that grows in their
// place (column j of L itself is stored when it is formed), so one 64 x 64
// array and one rank-1 update per column serve both.  Row and column j go
// through shared memory, double-buffered: one barrier per column.  A
// non-positive pivot sets CR_ESINGULAR and is replaced by 1 so the
// factorisation runs to the end.  Bound by the 64 dependent column steps
// (barrier, square root, divide, update).
__global__ void __launch_bounds__(256) potrf_inv_kernel(cf* __restrict__ L, int P, int J,
                                                        cf* __restrict__ X, int* __restrict__ status) {
    __shared__ cf col[2][NB], xrow[2][NB];
    const int base = J * NB, n = min(NB, P - base), ld = lcols(P);
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    cf a[4][4];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = ty + 16 * p, k = tx + 16 * q;
            a[p][q] = (i < n && k <= i) ? L[(size_t)(base + i) * ld + base + k]
                                        : cf{i == k ? 1.f : 0.f, 0.f};
        }
    bool bad = false;
#pragma unroll
    for (int jb = 0; jb < 4; ++jb)
        for (int jj = 0; jj < 16; ++jj) {
            const int j = 16 * jb + jj, buf = j & 1;
            if (tx == jj)
#pragma unroll
                for (int p = 0; p < 4; ++p) col[buf][ty + 16 * p] = a[p][jb];
            if (ty == jj)
#pragma unroll
                for (int q = 0; q < 4; ++q) xrow[buf][tx + 16 * q] = a[jb][q];
            __syncthreads();
            float d = col[buf][j].x;
            if (!(d > 0.f)) {
                bad = true;
                d = 1.f;
            }
            const float piv = m_sqrt(d), ip = 1.f / piv;
            // row factors: conj(l_k) of the block to the right of column j, the
            // inverse's row j (scaled) to the left of it
            cf rk[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = tx + 16 * q;
                rk[q] = k > j ? conj(ip * col[buf][k]) : ip * xrow[buf][k];
                if (k == j) rk[q] = {ip, 0.f};
            }
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int i = ty + 16 * p;
                if (i > j) {
                    const cf li = ip * col[buf][i];
                    if (tx == jj) {
                        if (i < n) L[(size_t)(base + i) * ld + base + j] = li;
                        a[p][jb] = {0.f, 0.f};  // the unit matrix's entry, updated below
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) a[p][q] = a[p][q] - li * rk[q];
                } else if (i == j) {
                    if (tx == jj && j < n) L[(size_t)(base + j) * ld + base + j] = {piv, 0.f};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (tx + 16 * q <= j) a[p][q] = rk[q];
                }
            }
        }
    cf* Xb = xblock(X, base);
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = ty + 16 * p, k = tx + 16 * q;
            Xb[(size_t)i * SB + k] = k <= i ? a[p][q] : cf{0.f, 0.f};
        }
    if (t == 0 && bad) set_status(status, CR_ESINGULAR);
}

// One 32-deep step of a 64 x 64 tile product, 16 x 16 threads, 4 x 4 outputs
// each (rows ty + 16 q, columns 4 tx + q).
constexpr int KT = 32;
constexpr int BP = NB + 2;  // rows of Bs start on 16 bytes
CR_D void tile_step(const cf (*As)[NB + 1], const cf (*Bs)[BP], int tx, int ty, cf (&acc)[4][4]) {
#pragma unroll
    for (int c = 0; c < KT; ++c) {
        cf av[4], bv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) av[q] = As[c][ty + 16 * q];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float4 v = *reinterpret_cast<const float4*>(&Bs[c][4 * tx + 2 * q]);
            bv[2 * q] = {v.x, v.y};
            bv[2 * q + 1] = {v.z, v.w};
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int q2 = 0; q2 < 4; ++q2) acc[q][q2] = acc[q][q2] + av[q] * bv[q2];
    }
}

// ------------------------------------------- trailing update, tensor cores
//
// A_IK -= L_IJ L_KJ^dag with the panel's float32 values split into three
// bf16 terms (six products, all 24 bits, float32 accumulation).  With K real
// index 2 c + part,
//   rows   N side, row i:                [Re L_ic, Im L_ic]
//   cols   M side, row 2k: [Re, Im] of L_kc; row 2k + 1: [-Im, Re]
// so that D[2k + part][i] = (Re, Im)(L_i . conj(L_k)): lanes (D rows) hold
// consecutive floats of a row of A, and a tile's 256 rows x 64 columns are
// read and written coalesced.  A panel is 128 real deep.  An MMA's addition
// truncates 2^-24 or so of its accumulator, so its error grows with the number
// of them that meet a large one: the eight MMAs of the first panel's leading
// products have an accumulator of their own; the small products of both
// panels, 2^-8 of those, go into another, and the second panel's leading ones
// into that after them, from a second copy of their operands.  Then one float32
// addition and subtraction for the pair.
constexpr uint32_t WAIT_LIMIT = 1u << 26;  // bounded mbarrier polls
constexpr int TC_ROWS = 256, TC_COLS = 64;  // tile of A
constexpr int TC_KC = 32, TC_NKC = 2 * NB / TC_KC;  // K tiles of a panel; operands hold two panels
constexpr int N_TILE = TC_ROWS * TC_KC * 2, M_TILE = 2 * TC_COLS * TC_KC * 2;  // bytes, one plane
constexpr int TC_STAGE = 3 * (N_TILE + M_TILE);
constexpr int TC_NSTG = 3;
constexpr size_t TC_SMEM = (size_t)TC_NSTG * TC_STAGE + 256;
constexpr int TC_DRAIN = 512;                 // 16 drain warps
constexpr int TC_THREADS = TC_DRAIN + 64;

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

// the three terms of 8 consecutive K values of one operand row
CR_D void put_row(unsigned char* tile, int plane, int row, int kk, const float* x) {
    __nv_bfloat16 h[8], m[8], l[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) split3(x[q], &h[q], &m[q], &l[q]);
    const uint32_t o = tc::kmajor_offset(row, kk, TC_KC);
    *reinterpret_cast<uint4*>(tile + o) = pack8(h);
    *reinterpret_cast<uint4*>(tile + plane + o) = pack8(m);
    *reinterpret_cast<uint4*>(tile + 2 * plane + o) = pack8(l);
}

// L_IJ = A_IJ X_JJ^dag for one 64-row block below block J (full here: it is
// not the last block).  planes: also the bf16 operands of the trailing
// update (rows past P are zero there; rows count from the first row below
// the pair's first panel, second: the pair's second panel); a thread's
// outputs are 4 adjacent columns, so it forms 16-byte operand groups from its
// own registers.
__global__ void __launch_bounds__(256) trsm_kernel(cf* __restrict__ L, int P, int J, cf* __restrict__ X,
                                                   unsigned char* __restrict__ planes, size_t m_off,
                                                   int second) {
    __shared__ __align__(16) cf As[KT][NB + 1];
    __shared__ __align__(16) cf Bs[KT][BP];
    const int base = J * NB, r0 = base + NB, i0 = r0 + blockIdx.x * NB, ld = lcols(P);
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    const cf* Xb = xblock(X, base);
    cf acc[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) acc[q][q2] = {0.f, 0.f};
    for (int cc = 0; cc < NB; cc += KT) {
#pragma unroll
        for (int e = t; e < NB * KT; e += 256) {
            const int r = e / KT, c = e % KT;
            As[c][r] = i0 + r < P ? L[(size_t)(i0 + r) * ld + base + cc + c] : cf{0.f, 0.f};
            Bs[c][r] = conj(Xb[(size_t)r * SB + cc + c]);
        }
        __syncthreads();
        tile_step(As, Bs, tx, ty, acc);
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int r = ty + 16 * q;
        float re[8], im[8];
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) {
            re[2 * q2] = acc[q][q2].x;
            re[2 * q2 + 1] = acc[q][q2].y;
            im[2 * q2] = -acc[q][q2].y;
            im[2 * q2 + 1] = acc[q][q2].x;
        }
        if (i0 + r < P) {
            float4* out = reinterpret_cast<float4*>(L + (size_t)(i0 + r) * ld + base + 4 * tx);
            out[0] = make_float4(re[0], re[1], re[2], re[3]);
            out[1] = make_float4(re[4], re[5], re[6], re[7]);
        }
        if (!planes) continue;
        const int row = i0 - r0 + second * NB + r, k = 8 * tx, kc = second * TC_NKC + k / TC_KC, kk = k % TC_KC;
        put_row(planes + ((size_t)(row / TC_ROWS) * 2 * TC_NKC + kc) * 3 * N_TILE, N_TILE, row % TC_ROWS, kk, re);
        unsigned char* mt = planes + m_off + ((size_t)(row / TC_COLS) * 2 * TC_NKC + kc) * 3 * M_TILE;
        put_row(mt, M_TILE, 2 * (row % TC_COLS), kk, re);
        put_row(mt, M_TILE, 2 * (row % TC_COLS) + 1, kk, im);
    }
}

// Tiles of the matrix below the pair's first panel (from row r0), 256 rows x
// 64 columns.  npan = 1, after the first panel: the tiles of column block 0,
// the second panel's.  npan = 2, after the second: row block rb takes the
// column blocks 1 <= cb <= 4 rb + 3 that exist (tile index 2 rb^2 + rb + cb -
// 1), one subtraction for both panels, but not the first 64 rows, which are
// done.
//
// Bound: 16 bytes of A per entry and update against 1.5 KB of MMA operands,
// which L2 serves.  A panel at a time (10 x 10 lattice, alpha = 1: P = 10200)
// the kernel moved A at 3.9 TB/s, waiting for the loads of 8 drain warps: 159
// launches, 11.4 ms.  In pairs, with 16 drain warps that have a whole tile of
// A in flight while its MMAs run: 8.0 ms, with 48 MMAs a panel into one
// accumulator, two of which alternate; 8.7 now, with both held for a tile.  That
// buys the factor's accuracy: the residual that one correction leaves, over P =
// 168 ... 10200, went from 2.15 times that of a factor by float32 multiply-adds
// and substitution to 1.11 (1.12 on the FMA pipes here, the inverses' share),
// the corrections needed from 3.03 to 2.62 on average (2.71).  A drain after each
// panel gave 1.15 and 10.2 ms, both panels' leading products in one accumulator
// 1.27 and 8.2.
//
// Persistent: warp 0 (one thread) issues a tile's MMAs into TMEM columns [0,
// 256) and [256, 512), warps 1-16 drain (warp w: lanes 32 (w % 4), rows 64 ((w -
// 1) / 4)), warp 17 (one thread) copies operand stages.
__global__ void __launch_bounds__(TC_THREADS, 1) syrk_tc_kernel(float* __restrict__ Lf, int P, int r0,
                                                                int npan, int ntiles,
                                                                const unsigned char* __restrict__ planes,
                                                                size_t m_off, int* __restrict__ status) {
    extern __shared__ __align__(1024) unsigned char sm[];
    uint64_t* full = (uint64_t*)(sm + TC_NSTG * TC_STAGE);
    uint64_t* empty = full + TC_NSTG;
    uint64_t* dfull = empty + TC_NSTG;  // MMAs of a tile done
    uint64_t* dempty = dfull + 1;       // both accumulators read by the drain threads
    uint32_t* slot = (uint32_t*)(dempty + 1);
    volatile int* abort = (volatile int*)(slot + 1);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) {
        for (int i = 0; i < 2 * TC_NSTG + 1; ++i) tc::mbar_init(&full[i], 1);
        tc::mbar_init(dempty, TC_DRAIN);
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
    auto wait = [&](uint64_t* bar, uint32_t par) {
        for (int i = 0; i < 64; ++i) {
            if (tc::mbar_wait(bar, par, WAIT_LIMIT >> 6)) return true;
            if (*abort) return false;
        }
        *abort = 1;
        return false;
    };
    auto tile_of = [&](int idx, int* rb, int* cb) {
        if (npan == 1) {
            *rb = idx;
            *cb = 0;
            return;
        }
        int r = (int)((sqrtf(1.0f + 8.0f * (float)idx) - 1.0f) * 0.25f);
        while (2 * r * r + r > idx) --r;
        while (2 * (r + 1) * (r + 1) + r + 1 <= idx) ++r;
        *rb = r;
        *cb = idx - (2 * r * r + r) + 1;
    };
    const int nmine = ntiles > (int)blockIdx.x ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int nst = npan == 1 ? TC_NKC : 3 * TC_NKC;  // operand stages of a tile
    if (warp == 0) {
        if (lane == 0) {
            constexpr int PA[6] = {0, 0, 1, 0, 1, 2}, PB[6] = {0, 1, 0, 2, 1, 0};
            const uint32_t idesc = tc::make_idesc_bf16(2 * TC_COLS, TC_ROWS);
            const uint64_t d0 = tc::make_desc(tc::smem_u32(sm), 128, 16 * TC_KC);
            uint32_t b = 0, ph = 0;
            int last = -1, lastph = 0;  // stage of the last commit
            bool ok = true;
            for (int ti = 0; ti < nmine && ok; ++ti) {
                if (ti >= 1 && !wait(dempty, (ti - 1) & 1)) {
                    ok = false;
                    break;
                }
                for (int kc = 0; kc < nst; ++kc) {
                    if (!wait(&full[b], ph)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after_sync();
                    const uint64_t nd = d0 + b * (uint32_t)(TC_STAGE >> 4);
                    const uint64_t md = nd + (3 * N_TILE >> 4);
                    // first panel: leading products to [0, 256), small ones to [256, 512);
                    // second: its small ones there too, its leading ones last
                    const bool lead = kc < TC_NKC || kc >= 2 * TC_NKC, small = kc < 2 * TC_NKC;
#pragma unroll
                    for (int ks = 0; ks < TC_KC / 16; ++ks) {
                        if (lead)
                            tc::mma_bf16(taddr + (small ? 0 : 256), md + ks * 16, nd + ks * 16, idesc,
                                         kc != 0 || ks != 0);
                        if (small)
#pragma unroll
                            for (int pr = 1; pr < 6; ++pr)
                                tc::mma_bf16(taddr + 256, md + (PA[pr] * (M_TILE >> 4) + ks * 16),
                                             nd + (PB[pr] * (N_TILE >> 4) + ks * 16), idesc,
                                             kc != 0 || ks != 0 || pr > 1);
                    }
                    tc::commit(&empty[b]);
                    last = (int)b;
                    lastph = (int)ph;
                    if (++b == TC_NSTG) {
                        b = 0;
                        ph ^= 1;
                    }
                }
                if (ok) tc::commit(dfull);
            }
            if (!ok) {
                *abort = 1;
                set_status(status, CR_ETIMEOUT);
                // let issued MMAs finish (bounded)
                if (last >= 0) tc::mbar_wait(&empty[last], (uint32_t)lastph, WAIT_LIMIT);
            }
        }
        __syncwarp();
    } else if (warp == TC_THREADS / 32 - 1) {
        if (lane == 0) {
            uint32_t b = 0, ph = 0, g = 0;
            bool ok = true;
            for (int ti = 0; ti < nmine && ok; ++ti) {
                int rb, cb;
                tile_of(blockIdx.x + ti * gridDim.x, &rb, &cb);
                const unsigned char* ns = planes + (size_t)rb * 2 * TC_NKC * 3 * N_TILE;
                const unsigned char* ms = planes + m_off + (size_t)cb * 2 * TC_NKC * 3 * M_TILE;
                for (int kc = 0; kc < nst; ++kc, ++g) {
                    if (g >= TC_NSTG && !wait(&empty[b], ph ^ 1)) {
                        ok = false;
                        break;
                    }
                    unsigned char* st = sm + (size_t)b * TC_STAGE;
                    // the second panel's leading terms come a second time, alone
                    const bool again = kc >= 2 * TC_NKC;
                    const int k = again ? kc - TC_NKC : kc, np = again ? 1 : 3;
                    tc::mbar_expect_tx(&full[b], (uint32_t)(np * (N_TILE + M_TILE)));
                    tc::bulk_g2s(st, ns + (size_t)k * 3 * N_TILE, np * N_TILE, &full[b]);
                    tc::bulk_g2s(st + 3 * N_TILE, ms + (size_t)k * 3 * M_TILE, np * M_TILE, &full[b]);
                    if (++b == TC_NSTG) {
                        b = 0;
                        ph ^= 1;
                    }
                }
            }
            // every copy lands before the CTA leaves (bounded): the last
            // stages; where MMAs consumed them all this does not wait
            for (uint32_t q = 0; q < TC_NSTG && q < g; ++q) {
                if (b == 0) ph ^= 1;
                b = b == 0 ? TC_NSTG - 1 : b - 1;
                tc::mbar_wait(&full[b], ph, WAIT_LIMIT);
            }
        }
        __syncwarp();
    } else {
        const int lb = warp & 3, c4 = (warp - 1) >> 2;
        const size_t ld = 2 * (size_t)lcols(P);
        bool ok = true;
        for (int ti = 0; ti < nmine && ok; ++ti) {
            int rb, cb;
            tile_of(blockIdx.x + ti * gridDim.x, &rb, &cb);
            float* Af = Lf + ((size_t)r0 + rb * TC_ROWS + 64 * c4) * ld + 2 * (r0 + cb * TC_COLS) +
                        32 * lb + lane;
            const bool live = npan == 1 || rb > 0 || c4 > 0;  // warp-uniform
            float c[64];
#pragma unroll
            for (int q = 0; q < 64; ++q) c[q] = live ? Af[q * ld] : 0.f;
            ok = __all_sync(0xffffffffu, wait(dfull, ti & 1));
            if (!ok) break;
            tc::fence_after_sync();
#pragma unroll
            for (int ch = 0; ch < 8; ++ch) {
                float v[8], w[8];
                const uint32_t at = taddr + ((uint32_t)(32 * lb) << 16) + 64 * c4 + 8 * ch;
                tc::tmem_ld8x2(at, at + 256, v, w);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    c[8 * ch + q] = __fsub_rn(c[8 * ch + q], __fadd_rn(v[q], w[q]));
            }
            tc::fence_before_sync();
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(tc::smem_u32(dempty)) : "memory");
            if (live)
#pragma unroll
                for (int q = 0; q < 64; ++q) Af[q * ld] = c[q];
        }
        if (!ok && t == 32) set_status(status, CR_ETIMEOUT);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(taddr, 512u);
}

// Trailing update of the lower block pairs (I, K), J < K <= I, one CTA per
// pair (linear index -> row a = I - J - 1, column b = K - J - 1 with b <= a).
__global__ void __launch_bounds__(256) syrk_kernel(cf* __restrict__ L, int P, int J) {
    __shared__ __align__(16) cf As[KT][NB + 1];
    __shared__ __align__(16) cf Bs[KT][BP];
    const long long idx = blockIdx.x;
    int a = (int)((sqrt(8.0 * (double)idx + 1.0) - 1.0) * 0.5);
    while ((long long)a * (a + 1) / 2 > idx) --a;
    while ((long long)(a + 1) * (a + 2) / 2 <= idx) ++a;
    const int b = (int)(idx - (long long)a * (a + 1) / 2);
    const int i0 = (J + 1 + a) * NB, k0 = (J + 1 + b) * NB, c0 = J * NB, ld = lcols(P);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    cf acc[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) acc[q][q2] = {0.f, 0.f};
    for (int cc = 0; cc < NB; cc += KT) {
        for (int e = threadIdx.x; e < NB * KT; e += 256) {
            const int r = e / KT, c = e % KT, gi = i0 + r, gk = k0 + r;
            As[c][r] = gi < P ? L[(size_t)gi * ld + c0 + cc + c] : cf{0.f, 0.f};
            Bs[c][r] = gk < P ? conj(L[(size_t)gk * ld + c0 + cc + c]) : cf{0.f, 0.f};
        }
        __syncthreads();
        tile_step(As, Bs, tx, ty, acc);
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) {
            const int i = i0 + ty + 16 * q, k = k0 + 4 * tx + q2;
            if (i < P && k < P) {
                cf* p = L + (size_t)i * ld + k;
                *p = *p - acc[q][q2];
            }
        }
}

// Inverse of a lower-triangular [[L11, 0], [L21, L22]] from X11 and X22 of
// size s: X21 = -X22 (L21 X11), one 64 x 64 tile per CTA.  Pass 0 writes W =
// L21 X11 into the unused upper block (rows of X11, columns of X22), pass 1
// writes X21.  Grid (s / 64, s / 64, pairs of all SB blocks); pairs whose
// lower part lies past P do not exist.
__global__ void __launch_bounds__(256) xmerge_kernel(const cf* __restrict__ L, int P, int s, int pass,
                                                     cf* __restrict__ X) {
    __shared__ __align__(16) cf As[KT][NB + 1];
    __shared__ __align__(16) cf Bs[KT][BP];
    const int ppb = SB / (2 * s), sb = blockIdx.z / ppb, pr = blockIdx.z % ppb;
    const int o1 = pr * 2 * s, o2 = o1 + s, base = sb * SB, ld = lcols(P);
    if (base + o2 >= P) return;
    const int ib = blockIdx.y, jb = blockIdx.x;  // 64-blocks of the s x s result
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    cf* Xs = X + (size_t)sb * SB * SB;
    cf acc[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) acc[q][q2] = {0.f, 0.f};
    // X11 is lower triangular (rows k >= column j), so is X22 (k <= i)
    const int kb = pass == 0 ? jb * NB : 0, ke = pass == 0 ? s : (ib + 1) * NB;
    for (int cc = kb; cc < ke; cc += KT) {
        for (int e = t; e < NB * KT; e += 256) {
            const int r = e / KT, c = e % KT, i = ib * NB + r, gi = base + o2 + i;
            As[c][r] = pass == 0 ? (gi < P ? L[(size_t)gi * ld + base + o1 + cc + c] : cf{0.f, 0.f})
                                 : Xs[(size_t)(o2 + i) * SB + o2 + cc + c];
            const int k = e / NB, j = e % NB;
            Bs[k][j] = pass == 0 ? Xs[(size_t)(o1 + cc + k) * SB + o1 + jb * NB + j]
                                 : Xs[(size_t)(o1 + cc + k) * SB + o2 + jb * NB + j];
        }
        __syncthreads();
        tile_step(As, Bs, tx, ty, acc);
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) {
            const int i = ib * NB + ty + 16 * q, j = jb * NB + 4 * tx + q2;
            if (pass == 0) Xs[(size_t)(o1 + i) * SB + o2 + j] = acc[q][q2];
            else Xs[(size_t)(o2 + i) * SB + o1 + j] = -acc[q][q2];
        }
}

// Triangular solves by 512-row blocks b.  Forward, L y = r:
//   y_b = X_b r_b (diag), then r_i -= L_ib y_b below (rest; r is scratch);
// one warp per row.  Backward, L^dag x = y:
//   x_b = X_b^dag y_b (diag), then y_i -= sum_c conj(L_ci) x_c above (rest; y
// is scratch); a CTA takes 32 rows i (lanes), its warps share the c.  The
// products run in float32, the vectors are float64.  Bound by
// reading L once per direction.
__global__ void __launch_bounds__(256) trsv_fwd_kernel(const cf* __restrict__ L, int P, int b,
                                                       const cf* __restrict__ X, int rest,
                                                       double* __restrict__ r_,
                                                       double* __restrict__ y_,
                                                       const double* __restrict__ skip) {
    if (skip && *skip != 0.0) return;
    __shared__ cf v[SB];
    cpx<double>* r = (cpx<double>*)r_;
    cpx<double>* y = (cpx<double>*)y_;
    const int base = b * SB, n = min(SB, P - base), t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const cpx<double>* src = (rest ? y : r) + base;
    for (int e = t; e < SB; e += 256) v[e] = e < n ? ccast<float>(src[e]) : cf{0.f, 0.f};
    __syncthreads();
    const int i = blockIdx.x * 8 + warp;  // row of the block, or below it
    if (rest) {
        const int row = base + n + i;
        if (row >= P) return;
        const cf* Lr = L + (size_t)row * lcols(P) + base;  // n = SB: not the last block
        cf s = {0.f, 0.f};
#pragma unroll
        for (int c = 0; c < SB; c += 32) s = s + Lr[c + lane] * v[c + lane];
        s = warp_sum(s);
        if (lane == 0) r[row] = r[row] - ccast<double>(s);
    } else if (i < n) {
        const cf* Xr = X + (size_t)b * SB * SB + (size_t)i * SB;
        cf s = {0.f, 0.f};
        for (int c = 0; c <= i; c += 32)
            if (c + lane <= i) s = s + Xr[c + lane] * v[c + lane];
        s = warp_sum(s);
        if (lane == 0) y[base + i] = ccast<double>(s);
    }
}

__global__ void __launch_bounds__(256) trsv_bwd_kernel(const cf* __restrict__ L, int P, int b,
                                                       const cf* __restrict__ X, int rest,
                                                       double* __restrict__ y_,
                                                       double* __restrict__ x_,
                                                       const double* __restrict__ skip) {
    if (skip && *skip != 0.0) return;
    __shared__ cf v[SB];
    __shared__ cf part[8][32];
    cpx<double>* y = (cpx<double>*)y_;
    cpx<double>* x = (cpx<double>*)x_;
    const int base = b * SB, n = min(SB, P - base), t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const cpx<double>* src = (rest ? x : y) + base;
    for (int e = t; e < SB; e += 256) v[e] = e < n ? ccast<float>(src[e]) : cf{0.f, 0.f};
    __syncthreads();
    const int i = blockIdx.x * 32 + lane, lim = rest ? base : n;
    const size_t ld = rest ? (size_t)lcols(P) : (size_t)SB;
    const cf* A = rest ? L + (size_t)base * ld : X + (size_t)b * SB * SB;
    cf s = {0.f, 0.f};
    if (i < lim) {
        // warp w takes the columns c in [64 w, 64 w + 64), sixteen loads in flight;
        // in the diagonal block, entries above the diagonal of a 64-block are
        // zero and the 64-blocks above it are left out
        const int c1 = min(n, 64 * warp + 64);
        int c = 64 * warp;
        if (rest || c + 63 >= blockIdx.x * 32)
            for (; c < c1; c += 16) {
                cf a[16];
#pragma unroll
                for (int q = 0; q < 16; ++q)
                    a[q] = c + q < c1 ? A[(size_t)(c + q) * ld + i] : cf{0.f, 0.f};
#pragma unroll
                for (int q = 0; q < 16; ++q) s = s + conj(a[q]) * v[c + q];
            }
    }
    part[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && i < lim) {
        cf tot = part[0][lane];
        for (int w = 1; w < 8; ++w) tot = tot + part[w][lane];
        if (rest) y[i] = y[i] - ccast<double>(tot);
        else x[base + i] = ccast<double>(tot);
    }
}

// x = 0, r = F, flags cleared; scal[1] = F.F (float64, one CTA).
__global__ void __launch_bounds__(1024) refine_init_kernel(const double* __restrict__ F_, int P,
                                                           double* __restrict__ x_,
                                                           double* __restrict__ r_,
                                                           double* __restrict__ scal) {
    __shared__ double red[32];
    const cpx<double>* F = (const cpx<double>*)F_;
    cpx<double>* x = (cpx<double>*)x_;
    cpx<double>* r = (cpx<double>*)r_;
    double s = 0.0;
    for (int k = threadIdx.x; k < P; k += blockDim.x) {
        x[k] = {0.0, 0.0};
        r[k] = F[k];
        s += abs2(F[k]);
    }
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 32; ++w) t += red[w];
        scal[1] = t;
        scal[2] = t > 0.0 ? 0.0 : 1.0;  // F = 0: x = 0 is exact
        scal[3] = 0.0;
        scal[4] = t;
        scal[8] = t;
    }
}

// r = F - S (x + d), RES_ROWS rows of S per warp (they share the reads of x
// and d); per-CTA partial sums of |r|^2.
__global__ void __launch_bounds__(256) refine_resid_kernel(const double* __restrict__ S_, int P,
                                                           const double* __restrict__ F_,
                                                           const double* __restrict__ x_,
                                                           const double* __restrict__ d_,
                                                           double* __restrict__ r_,
                                                           double* __restrict__ part,
                                                           const double* __restrict__ skip) {
    if (*skip != 0.0) return;
    __shared__ double red[8];
    const cpx<double>* S = (const cpx<double>*)S_;
    const cpx<double>* x = (const cpx<double>*)x_;
    const cpx<double>* d = (const cpx<double>*)d_;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double acc = 0.0;
    const int row = (blockIdx.x * 8 + warp) * RES_ROWS;
    if (row < P) {
        cpx<double> s[RES_ROWS];
        const cpx<double>* Sr[RES_ROWS];
#pragma unroll
        for (int q = 0; q < RES_ROWS; ++q) {
            s[q] = {0.0, 0.0};
            Sr[q] = S + (size_t)min(row + q, P - 1) * P;
        }
#pragma unroll 4
        for (int l = lane; l < P; l += 32) {
            const cpx<double> v = x[l] + d[l];
#pragma unroll
            for (int q = 0; q < RES_ROWS; ++q) s[q] = s[q] + Sr[q][l] * v;
        }
#pragma unroll
        for (int q = 0; q < RES_ROWS; ++q) {
            s[q] = warp_sum(s[q]);
            if (lane == 0 && row + q < P) {
                const cpx<double> rv = ((const cpx<double>*)F_)[row + q] - s[q];
                ((cpx<double>*)r_)[row + q] = rv;
                acc += abs2(rv);
            }
        }
    }
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

// x += d; |r|^2 from the partial sums in a fixed order; stop on
// convergence or stagnation.
__global__ void __launch_bounds__(1024) refine_check_kernel(int P, double* __restrict__ x_,
                                                            const double* __restrict__ d_,
                                                            const double* __restrict__ part,
                                                            int npart, double tol,
                                                            double* __restrict__ scal) {
    // every thread has read the flag before thread 0 sets it below: a warp that
    // saw it set would leave its part of the last correction out
    const bool done = scal[2] != 0.0;
    __syncthreads();
    if (done) return;
    cpx<double>* x = (cpx<double>*)x_;
    const cpx<double>* d = (const cpx<double>*)d_;
    for (int k = threadIdx.x; k < P; k += blockDim.x) x[k] = x[k] + d[k];
    if (threadIdx.x < 32) {
        double rr = 0.0;
        for (int b = threadIdx.x; b < npart; b += 32) rr += part[b];
        rr = warp_sum(rr);
        if (threadIdx.x != 0) return;
        const double prev = scal[8];
        scal[3] += 1.0;
        scal[4] = rr;
        scal[8] = rr;
        if (!(rr > tol * tol * scal[1]) || rr > 0.25 * prev) scal[2] = 1.0;
    }
}

// Bytes of the trailing update's operands: the N side (rows in blocks of
// 256), then the M side (two real rows per column).
size_t n_plane_bytes(int P) { return (size_t)((P + TC_ROWS - 1) / TC_ROWS) * 2 * TC_NKC * 3 * N_TILE; }
size_t m_plane_bytes(int P) {
    return (size_t)((P + TC_ROWS - 1) / TC_ROWS) * (TC_ROWS / TC_COLS) * 2 * TC_NKC * 3 * M_TILE;
}

cr_status factor32(cr_ctx* c) {
    const int P = c->P, nb = (P + NB - 1) / NB;
    cf* L = (cf*)c->Lf;
    cf* X = (cf*)c->chol_x;
    const bool tcu = c->prec == CR_MIXED;
    const size_t m_off = n_plane_bytes(P);
    CR_LAUNCH(c, CR_K_OTHER,
              chol_copy_kernel<<<dim3(lrows(P), (lcols(P) + 255) / 256), 256, 0, c->stream>>>(c->S, P, L));
    for (int J = 0; J < nb; ++J) {
        CR_LAUNCH(c, CR_KERNEL_CHOL, potrf_inv_kernel<<<1, 256, 0, c->stream>>>(L, P, J, X, c->d_status));
        const int rows = P - (J + 1) * NB;
        if (rows <= 0) break;
        // mixed: rows below the first panel of the pair (J - second, + 1), in
        // blocks of 256, zero past P
        const int second = tcu ? J & 1 : 0, r0 = (J + 1 - second) * NB;
        const int nrb = (P - r0 + TC_ROWS - 1) / TC_ROWS, ncb = (P - r0 + NB - 1) / NB;
        CR_LAUNCH(c, CR_KERNEL_CHOL,
                  trsm_kernel<<<tcu ? 4 * nrb - second : ncb, 256, 0, c->stream>>>(
                      L, P, J, X, tcu ? c->chol_pl : nullptr, m_off, second));
        if (tcu) {
            const int nt = second ? 2 * (nrb - 1) * (nrb - 1) + (nrb - 1) + ncb - 1 : nrb;
            CR_LAUNCH(c, CR_KERNEL_CHOL,
                      syrk_tc_kernel<<<nt < c->n_sm ? nt : c->n_sm, TC_THREADS, TC_SMEM, c->stream>>>(
                          (float*)c->Lf, P, r0, 1 + second, nt, c->chol_pl, m_off, c->d_status));
        } else {
            const long long T = nb - J - 1;
            CR_LAUNCH(c, CR_KERNEL_CHOL,
                      syrk_kernel<<<(unsigned)(T * (T + 1) / 2), 256, 0, c->stream>>>(L, P, J));
        }
    }
    // merge the 64-row inverses up to SB rows (or all of a smaller matrix)
    const int nsb = (P + SB - 1) / SB;
    for (int s = NB; s < SB && s < P; s *= 2)
        for (int pass = 0; pass < 2; ++pass)
            CR_LAUNCH(c, CR_KERNEL_CHOL,
                      xmerge_kernel<<<dim3(s / NB, s / NB, nsb * (SB / (2 * s))), 256, 0, c->stream>>>(
                          L, P, s, pass, X));
    return cr_check_launch(c, "blocked Cholesky");
}

// d = L^{-dag} L^{-1} r (r and y are scratch)
void solve32(cr_ctx* c, double* r, double* y, double* d, const double* done) {
    const int P = c->P, nsb = (P + SB - 1) / SB;
    const cf* L = (const cf*)c->Lf;
    const cf* X = (const cf*)c->chol_x;
    for (int b = 0; b < nsb; ++b) {
        const int n = P - b * SB < SB ? P - b * SB : SB, rows = P - b * SB - n;
        CR_LAUNCH(c, CR_KERNEL_TRSV,
                  trsv_fwd_kernel<<<(n + 7) / 8, 256, 0, c->stream>>>(L, P, b, X, 0, r, y, done));
        if (rows > 0)
            CR_LAUNCH(c, CR_KERNEL_TRSV,
                      trsv_fwd_kernel<<<(rows + 7) / 8, 256, 0, c->stream>>>(L, P, b, X, 1, r, y, done));
    }
    for (int b = nsb - 1; b >= 0; --b) {
        const int n = P - b * SB < SB ? P - b * SB : SB, rows = b * SB;
        CR_LAUNCH(c, CR_KERNEL_TRSV,
                  trsv_bwd_kernel<<<(n + 31) / 32, 256, 0, c->stream>>>(L, P, b, X, 0, y, d, done));
        if (rows > 0)
            CR_LAUNCH(c, CR_KERNEL_TRSV,
                      trsv_bwd_kernel<<<(rows + 31) / 32, 256, 0, c->stream>>>(L, P, b, X, 1, y, d, done));
    }
}

int resid_grid(int P) { return (P + 8 * RES_ROWS - 1) / (8 * RES_ROWS); }

}  // namespace

bool chol_refined(const cr_ctx* c) {
    return (c->flags & CR_CTX_EXPLICIT_S) && (c->prec != CR_FP64 || c->P > CHOL_SMALL_P);
}

void chol_sizes(const cr_ctx* c, size_t* factor, size_t* inverses, size_t* planes) {
    const size_t P = c->P;
    if (c->prec == CR_FP64) {
        *factor = P * P * 16;
        *inverses = chol64_diag_bytes(c->P);
        *planes = 0;
        return;
    }
    *factor = (size_t)lrows(c->P) * lcols(c->P) * sizeof(cf);
    *inverses = ((P + SB - 1) / SB) * (size_t)SB * SB * sizeof(cf);
    *planes = c->prec == CR_MIXED ? n_plane_bytes(c->P) + m_plane_bytes(c->P) : 0;
}

size_t chol_cgpart_len(const cr_ctx* c) { return resid_grid(c->P); }

cr_status chol_prepare(cr_ctx* c) {
    if (c->prec == CR_FP64) return chol64_prepare(c);
    cudaError_t e = cudaFuncSetAttribute(syrk_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)TC_SMEM);
    return e == cudaSuccess ? CR_OK : cr_fail(c, CR_ECUDA, "chol_prepare: %s", cudaGetErrorString(e));
}

cr_status chol_factor(cr_ctx* c) {
    return c->prec == CR_FP64 ? chol64_factor(c, (double*)c->Lf, (double*)c->chol_x) : factor32(c);
}

// The iterates above into cg[0 .. P); scal[3] steps, scal[4] |r|^2.
cr_status chol_refine_solve(cr_ctx* c, const double* F, int maxit) {
    if (maxit > REFINE_MAXIT) maxit = REFINE_MAXIT;
    if (maxit < 1) maxit = 1;
    const int P = c->P, grid = resid_grid(P);
    double* x = c->cg;
    double* r = c->cg + 2 * (size_t)P;
    double* y = c->cg + 4 * (size_t)P;
    double* d = c->cg + 6 * (size_t)P;
    const double* done = c->scal + 2;
    CR_LAUNCH(c, CR_K_OTHER, refine_init_kernel<<<1, 1024, 0, c->stream>>>(F, P, x, r, c->scal));
    for (int it = 0; it < maxit; ++it) {
        if (c->prec == CR_FP64) chol64_solve(c, (double*)c->Lf, (double*)c->chol_x, r, y, d, done);
        else solve32(c, r, y, d, done);
        CR_LAUNCH(c, CR_K_OTHER, refine_resid_kernel<<<grid, 256, 0, c->stream>>>(
                                     c->S, P, F, x, d, r, c->cgpart, done));
        CR_LAUNCH(c, CR_K_OTHER, refine_check_kernel<<<1, 1024, 0, c->stream>>>(
                                     P, x, d, c->cgpart, grid, REFINE_TOL, c->scal));
    }
    return cr_check_launch(c, "refined solve");
}

// x = (L L^dag)^-1 F in float64, no refinement (small float64 contexts):
// scal[1] = F.F on the way.
cr_status chol_plain_solve(cr_ctx* c, const double* F) {
    const size_t P = c->P;
    double* x = c->cg;
    double* r = c->cg + 2 * P;
    CR_LAUNCH(c, CR_K_OTHER, refine_init_kernel<<<1, 1024, 0, c->stream>>>(F, c->P, x, r, c->scal));
    chol64_solve(c, (double*)c->Lf, (double*)c->chol_x, r, c->cg + 4 * P, x, nullptr);
    return cr_check_launch(c, "direct solve");
}
