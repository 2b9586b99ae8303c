// Sums over the antiparallel bonds of exchanged amplitudes, in float32: the
// off-diagonal part of (H' v)(s) for the local target, the Krylov columns
// (target.cu) and the symmetry projection (symmetry.cu).
//
// Exchanging the antiparallel spins of bond b = (i, i') takes theta_m to
// theta_m - s D_bm, s = sigma_i, D_bm = 2 (W_im - W_i'm).  With x_m = Re
// theta_m, y_m = Im theta_m, a_m = e^{-2 max(0, -x_m)} and
// z_m = e^{-2 theta_m} a_m (both of modulus <= 1),
//   2 cosh(theta_m - s D_bm) = e^{|x_m| + i y_m} e^{-s D_bm} (a_m + z_m q_bm^s),
//   q_bm^s = e^{2 s D_bm},
// so that v(s^{ij}) = e^{a.s + sum_m (|x_m| + i y_m)} e_b^s prod_m (a_m + z_m q_bm^s)
// with the bond constant e_b^s = exp(-s [2 (a_i - a_i') + sum_m D_bm]).  A factor
// is one complex multiply-add and one complex multiply (13 flops in 8 operations
// of the FMA pipe, against 14 operations for cosh theta cosh D - s sinh theta
// sinh D) and takes one table value; no factor divides, so a sample may sit at
// a node of v.
//
// The products run over hidden units spread across lanes: G lanes hold the
// whole hidden layer of a walker, 2 KP units each, in registers, so a warp
// evaluates 32 / G bonds at a time and reads table rows from shared memory
// without conflicts.  The table [bond][s][units] streams through shared
// memory in tiles of bonds, double-buffered by bulk copies (or stays, when it
// fits); a CTA keeps WPW walkers per warp while a tile passes.  Four bonds'
// lane products are multiplied together in one transposed butterfly.  The
// previous form had lanes over bonds, gathering two table values per factor
// from L2, and spent a further millisecond in float64 exponentials of one
// lane per warp; what is left of those is in the callers, one thread per
// walker.
//
// The lanes' products of the unexchanged factors set a power-of-two scale
// per lane, so the exchanged products stay near 1.  One that leaves
// [1e-30, 1e30] all the same (theta or D of order 40, a node of v where the
// scale was taken) is formed again by slow_product, cosh and sinh with a
// running exponent.
#include "common.cuh"
#include "tc.cuh"

namespace {

using cf = cpx<float>;
using zd = cpx<double>;
typedef unsigned long long u64;

constexpr int XW = 16;                        // warps per CTA
constexpr int MAX_TILE = 64;                  // bonds per tile
constexpr int TILE_BYTES = 84 * 1024;         // bytes of one tile at most
constexpr uint32_t WAIT_LIMIT = 1u << 26;     // bounded mbarrier polls

CR_D u64 pk(float a, float b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
CR_D void upk(u64 v, float* a, float* b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(*a), "=f"(*b) : "l"(v)); }
CR_D u64 fma2(u64 a, u64 b, u64 c) {
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
CR_D u64 mul2(u64 a, u64 b) {
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
CR_D u64 neg2(u64 a) { return a ^ 0x8000000080000000ull; }

// Sums carried as an unevaluated pair hi + lo (error-free two-term additions,
// Knuth, The Art of Computer Programming vol. 2, 4.2.2).  The terms are float32,
// so a pair keeps what a float64 sum of them would to 2^-46: against 64 bits
// the target has 0.85 to 0.89 (14 draws, 12 to 256 sites) and the symmetry
// projection 0.97 (5 draws) of the error of the form with float64 sums.
struct ff { float hi, lo; };
CR_D void ff_add(ff& s, float v) {
    const float t = __fadd_rn(s.hi, v), z = __fsub_rn(t, s.hi);
    s.lo = __fadd_rn(s.lo, __fadd_rn(__fsub_rn(s.hi, __fsub_rn(t, z)), __fsub_rn(v, z)));
    s.hi = t;
}
CR_D ff ff_warp_sum(ff s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h = __shfl_xor_sync(0xffffffffu, s.hi, o), l = __shfl_xor_sync(0xffffffffu, s.lo, o);
        ff_add(s, h);
        s.lo = __fadd_rn(s.lo, l);
    }
    return s;
}

// ------------------------------------------------------------------ table
//
// Row (b, s): rowf4 - 1 float4 of two units each (q re, re, im, im), then
// (e_b^s, d_b) with d_b = e^{-iq.r_i'} - e^{-iq.r_i} of the probe.  One warp
// per bond.
__global__ void __launch_bounds__(128) xtable_kernel(const cf* __restrict__ prm,
                                                     const int2* __restrict__ bonds, int N, int M,
                                                     int Nb, int rowf4, int Lx, int probe, double qx,
                                                     double qy, float4* __restrict__ tab) {
    const int b = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= Nb) return;
    const int2 bd = bonds[b];
    const cf* W = prm + N + M;
    const cf* wi = W + (size_t)bd.x * M;
    const cf* wj = W + (size_t)bd.y * M;
    float4* row = tab + (size_t)b * 2 * rowf4;
    zd sum = {0.0, 0.0};
    for (int p = lane; p < rowf4 - 1; p += 32) {
        cf q[2][2];  // [sign][unit]
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int m = 2 * p + u;
            q[0][u] = q[1][u] = {1.f, 0.f};  // padding units: z = 0
            if (m < M) {
                const cf d = 2.f * (wi[m] - wj[m]);
                sum = sum + ccast<double>(d);
                float sn, cs;
                m_sincos(2.f * d.y, &sn, &cs);
                const float ep = m_exp(2.f * d.x), em = m_exp(-2.f * d.x);
                q[0][u] = {ep * cs, ep * sn};
                q[1][u] = {em * cs, -em * sn};
            }
        }
#pragma unroll
        for (int s = 0; s < 2; ++s)
            row[(size_t)s * rowf4 + p] = make_float4(q[s][0].x, q[s][1].x, q[s][0].y, q[s][1].y);
    }
    sum = warp_sum(sum);
    if (lane < 2) {
        const zd da = 2.0 * (ccast<double>(prm[bd.x]) - ccast<double>(prm[bd.y]));
        const zd e = cexp_((lane ? 1.0 : -1.0) * (da + sum));
        cf d = {0.f, 0.f};
        if (probe) {
            float s0, c0, s1, c1;
            m_sincos((float)(qx * (bd.x % Lx) + qy * (bd.x / Lx)), &s0, &c0);
            m_sincos((float)(qx * (bd.y % Lx) + qy * (bd.y / Lx)), &s1, &c1);
            d = {c1 - c0, s0 - s1};
        }
        row[(size_t)lane * rowf4 + rowf4 - 1] = make_float4((float)e.x, (float)e.y, d.x, d.y);
    }
}

struct XArgs {
    const int8_t* spins;  // [n][N]
    const cf* th;         // [n][M]
    const cf* prm;
    const float4* tab;
    const int2* bonds;
    int n, N, M, Nb, rowf4;
    int nbt, ntiles;      // bonds per tile, tiles
    int probe;
    xsum_out* out;        // [n]
    int* status;
};

// e_b^s prod_m (a_m + z_m q_bm^s) of one bond by the whole warp, from cosh and
// sinh with a running exponent, scaled by 2^-ex0.
__device__ __noinline__ zd slow_product(const XArgs& A, int w, int b, int s, int ex0) {
    const int lane = threadIdx.x & 31;
    const int2 bd = A.bonds[b];
    const cf* W = A.prm + A.N + A.M;
    cf pr = {1.f, 0.f};
    int ex = 0;
    double ysum = 0.0;  // sum_m y_m, the phase that the common factor carries
    for (int m = lane; m < A.M; m += 32) {
        const cf th = A.th[(size_t)w * A.M + m];
        ysum += (double)th.y;
        const cf d = 2.f * (W[(size_t)bd.x * A.M + m] - W[(size_t)bd.y * A.M + m]);
        cf ch, sh;
        ccoshsinh_(d, &ch, &sh);
        const float ax = fabsf(th.x), sg = th.x < 0.f ? -1.f : 1.f, e = m_exp(-2.f * ax);
        float sn, cs;
        m_sincos(th.y, &sn, &cs);
        const float p = 0.5f * (1.f + e), q = 0.5f * sg * (1.f - e);
        const cf x = cf{p * cs, q * sn} * ch, y = (float)s * (cf{q * cs, p * sn} * sh);
        pr = pr * (x - y);
        int ee;
        frexpf(fmaxf(fabsf(pr.x), fabsf(pr.y)), &ee);
        pr = {ldexpf(pr.x, -ee), ldexpf(pr.y, -ee)};
        ex += ee;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const cf v = {__shfl_xor_sync(0xffffffffu, pr.x, o), __shfl_xor_sync(0xffffffffu, pr.y, o)};
        ex += __shfl_xor_sync(0xffffffffu, ex, o);
        pr = pr * v;
        int ee;
        frexpf(fmaxf(fabsf(pr.x), fabsf(pr.y)), &ee);
        pr = {ldexpf(pr.x, -ee), ldexpf(pr.y, -ee)};
        ex += ee;
    }
    pr = {__shfl_sync(0xffffffffu, pr.x, 0), __shfl_sync(0xffffffffu, pr.y, 0)};
    const zd da = 2.0 * (ccast<double>(A.prm[bd.x]) - ccast<double>(A.prm[bd.y]));
    const zd e = cexp_((s > 0 ? -1.0 : 1.0) * da);
    const zd v = e * (cexp_(zd{0.0, -warp_sum(ysum)}) * ccast<double>(pr));
    return {ldexp(v.x, ex + A.M - ex0), ldexp(v.y, ex + A.M - ex0)};
}

CR_D cf cshfl(cf v, int o) {
    return {__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o)};
}

// prod over the lane's units of (a + z q) for two table rows, in step (packed
// float32 pairs: the scalar form took 4052 us where this takes 3959 on the 16 x 16
// lattice's target, 65536 walkers).
template <int G, int KP>
CR_D void products(const float4* const (&row)[2], const u64 (&zr)[KP], const u64 (&zi)[KP],
                   const u64 (&av)[KP], cf* pr) {
    u64 pre[2], pim[2];
#pragma unroll
    for (int k = 0; k < KP; ++k) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(row[h] + k * G);
            const u64 x = fma2(zr[k], q.x, fma2(neg2(zi[k]), q.y, av[k]));
            const u64 y = fma2(zr[k], q.y, mul2(zi[k], q.x));
            if (k == 0) {
                pre[h] = x;
                pim[h] = y;
            } else {
                const u64 nr = fma2(pre[h], x, neg2(mul2(pim[h], y)));
                pim[h] = fma2(pre[h], y, mul2(pim[h], x));
                pre[h] = nr;
            }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float r0, r1, i0, i1;
        upk(pre[h], &r0, &r1);
        upk(pim[h], &i0, &i1);
        pr[h] = cf{r0, i0} * cf{r1, i1};
    }
}

template <int G, int KP, int WPW>
__global__ void __launch_bounds__(32 * XW, 1) xsum_kernel(const __grid_constant__ XArgs A) {
    constexpr int NG = 32 / G;          // bonds at a time
    extern __shared__ __align__(1024) unsigned char sm[];
    const int rowf4 = A.rowf4, Nb = A.Nb, N = A.N, M = A.M, nmw = (Nb + 31) / 32;
    const size_t tile_bytes = (size_t)A.nbt * 2 * rowf4 * 16;
    unsigned char* p = sm + 2 * tile_bytes;
    uint64_t* full = (uint64_t*)p;      // [2]
    uint64_t* empty = full + 2;         // [2]
    int2* bonds = (int2*)(empty + 2);   // [Nb]
    uint32_t* masks = (uint32_t*)(bonds + Nb);                     // [XW][WPW][2][nmw]: antiparallel, sigma_i > 0
    uint16_t* lists = (uint16_t*)(masks + (size_t)XW * WPW * 2 * nmw);  // [XW][MAX_TILE]
    int8_t* sgs = (int8_t*)(lists + XW * MAX_TILE);                // [XW][N]
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31, gl = lane & (G - 1), gi = lane / G;
    if (t == 0) {
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&full[i], 1);
            tc::mbar_init(&empty[i], XW);
        }
        tc::fence_mbar_init();
    }
    for (int e = t; e < Nb; e += 32 * XW) bonds[e] = A.bonds[e];
    __syncthreads();
    const int per = XW * WPW, nblk = (A.n + per - 1) / per;
    const int nmine = nblk > (int)blockIdx.x ? (nblk - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const bool resident = A.ntiles <= 2;          // the table stays in the two buffers
    const int nloads = resident ? A.ntiles : nmine * A.ntiles;
    int issued = 0;
    auto load = [&]() {  // thread 0
        const int tl = issued % A.ntiles, b0 = tl * A.nbt, nb = min(A.nbt, Nb - b0), buf = issued & 1;
        const uint32_t bytes = (uint32_t)(nb * 2 * rowf4 * 16);
        tc::mbar_expect_tx(&full[buf], bytes);
        tc::bulk_g2s(sm + buf * tile_bytes, A.tab + (size_t)b0 * 2 * rowf4, bytes, &full[buf]);
        ++issued;
    };
    if (t == 0)
        while (issued < 2 && issued < nloads) load();
    uint32_t* mk = masks + (size_t)warp * WPW * 2 * nmw;
    uint16_t* lst = lists + warp * MAX_TILE;
    int8_t* sg = sgs + (size_t)warp * N;
    bool ok = true;
    int step = 0;  // tiles consumed
    for (int blk = 0; blk < nmine && ok; ++blk) {
        const int w0 = (blockIdx.x + blk * gridDim.x) * per + warp * WPW;
        u64 zr[WPW][KP], zi[WPW][KP], av[WPW][KP];
        ff sx[WPW], sy[WPW], dx[WPW], dy[WPW];
        int ex[WPW];
        // ------------------------------------------------ the warp's walkers
#pragma unroll
        for (int u = 0; u < WPW; ++u) {
            const int w = w0 + u;
            sx[u] = sy[u] = dx[u] = dy[u] = ff{0.f, 0.f};
            ex[u] = 0;
            const bool live = w < A.n;
            __syncwarp();
            if (live)
                for (int i = lane; i < N; i += 32) sg[i] = A.spins[(size_t)w * N + i];
            __syncwarp();
            int nanti = 0;
            for (int q = 0; q < nmw; ++q) {
                const int b = 32 * q + lane;
                bool anti = false, up = false;
                if (live && b < Nb) {
                    const int2 bd = bonds[b];
                    up = sg[bd.x] > 0;
                    anti = sg[bd.x] != sg[bd.y];
                }
                const uint32_t ma = __ballot_sync(0xffffffffu, anti), mu = __ballot_sync(0xffffffffu, up);
                if (lane == 0) {
                    mk[(2 * u) * nmw + q] = ma;
                    mk[(2 * u + 1) * nmw + q] = mu;
                }
                nanti += __popc(ma);
            }
            // a.s + sum_m |x_m| + i y_m, and the factors' operands (scaled so that
            // the lane's product of a + z is in [0.5, 1))
            ff br = {0.f, 0.f}, bi = {0.f, 0.f}, ys = {0.f, 0.f};
            if (live)
                for (int i = lane; i < N; i += 32) {
                    const cf a = A.prm[i];
                    const float s = (float)sg[i];
                    ff_add(br, s * a.x);
                    ff_add(bi, s * a.y);
                }
            cf lp = {1.f, 0.f};
            int le = 0;
#pragma unroll
            for (int k = 0; k < KP; ++k) {
                float r[2], i[2], a[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int m = 2 * (k * G + gl) + h;
                    r[h] = i[h] = 0.f;
                    a[h] = 1.f;
                    if (live && m < M) {
                        const cf th = A.th[(size_t)w * M + m];
                        const float e = m_exp(-2.f * fabsf(th.x));
                        float sn, cs;
                        m_sincos(-2.f * th.y, &sn, &cs);
                        const float mag = th.x < 0.f ? 1.f : e;
                        a[h] = th.x < 0.f ? e : 1.f;
                        r[h] = mag * cs;
                        i[h] = mag * sn;
                        if (gi == 0) {  // the groups hold copies
                            ff_add(br, fabsf(th.x));
                            ff_add(ys, th.y);
                        }
                    }
                    const cf f = {a[h] + r[h], i[h]};
                    lp = lp * f;
                }
                zr[u][k] = pk(r[0], r[1]);
                zi[u][k] = pk(i[0], i[1]);
                av[u][k] = pk(a[0], a[1]);
                const float mx = fmaxf(fabsf(lp.x), fabsf(lp.y));
                const int e = mx > 1e-30f ? ilogbf(mx) + 1 : 0;
                lp = {ldexpf(lp.x, -e), ldexpf(lp.y, -e)};
                le += e;
            }
            const u64 sc = pk(ldexpf(1.f, -le), 1.f);  // one factor of the lane carries its scale
            zr[u][0] = mul2(zr[u][0], sc);
            zi[u][0] = mul2(zi[u][0], sc);
            av[u][0] = mul2(av[u][0], sc);
            int et = le;
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) et += __shfl_xor_sync(0xffffffffu, et, o);
            ex[u] = et;
            ys = ff_warp_sum(ys);
            br = ff_warp_sum(br);
            bi = ff_warp_sum(bi);
            ff_add(bi, ys.hi);
            bi.lo += ys.lo;
            if (live && lane == 0) {
                A.out[w].base = make_float4(br.hi, br.lo, bi.hi, bi.lo);
                A.out[w].nanti = nanti;
                A.out[w].ex = et;
                A.out[w].slow = {0.0, 0.0};
                A.out[w].slow_d = {0.0, 0.0};
            }
        }
        // ------------------------------------------------- the table's tiles
        for (int tl = 0; tl < A.ntiles; ++tl, ++step) {
            const int buf = resident ? tl : step & 1;
            // (the outcome is uniform in the warp: shuffles follow)
            if (!__all_sync(0xffffffffu, tc::mbar_wait(&full[buf], resident ? 0 : (step >> 1) & 1, WAIT_LIMIT))) {
                ok = false;
                break;
            }
            const float4* tile = (const float4*)(sm + buf * tile_bytes);
            const int b0 = tl * A.nbt, nb = min(A.nbt, Nb - b0);
#pragma unroll
            for (int u = 0; u < WPW; ++u) {
                const uint32_t* ma = mk + (2 * u) * nmw;
                const uint32_t* mu = ma + nmw;
                // the tile's antiparallel bonds, bit 15: sigma_i = -1
                int cnt = 0;
                __syncwarp();
                for (int q = 0; q < nb; q += 32) {
                    const int l = q + lane, b = b0 + l;
                    const bool on = l < nb && ((ma[b >> 5] >> (b & 31)) & 1u);
                    const uint32_t bal = __ballot_sync(0xffffffffu, on);
                    if (on)
                        lst[cnt + __popc(bal & ((1u << lane) - 1u))] =
                            (uint16_t)(l | (((mu[b >> 5] >> (b & 31)) & 1u) ? 0 : 0x8000));
                    cnt += __popc(bal);
                }
                __syncwarp();
                for (int base = 0; base < cnt; base += 4 * NG) {
                    // two bonds at a time, in step (a bond past the list repeats its first)
                    cf pr[4];
#pragma unroll
                    for (int v = 0; v < 4; v += 2) {
                        if (v > 0 && base + v * NG >= cnt) {
                            pr[v] = pr[v + 1] = {1.f, 0.f};
                            continue;
                        }
                        const float4* row[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int idx = base + (v + h) * NG + gi, e = lst[idx < cnt ? idx : 0];
                            row[h] = tile + (2 * (e & 0x7fff) + (e >> 15)) * rowf4 + gl;
                        }
                        products<G, KP>(row, zr[u], zi[u], av[u], &pr[v]);
                    }
                    // transposed butterfly: after the two halvings a lane holds the
                    // product of bond v = 2 (gl / (G/2)) + (gl / (G/4)) % 2
                    const bool h1 = gl & (G / 2), h2 = gl & (G / 4);
                    cf k0 = h1 ? pr[2] : pr[0], k1 = h1 ? pr[3] : pr[1];
                    k0 = k0 * cshfl(h1 ? pr[0] : pr[2], G / 2);
                    k1 = k1 * cshfl(h1 ? pr[1] : pr[3], G / 2);
                    cf k = h2 ? k1 : k0;
                    k = k * cshfl(h2 ? k0 : k1, G / 4);
#pragma unroll
                    for (int o = G / 8; o > 0; o >>= 1) k = k * cshfl(k, o);
                    const int v = (h1 ? 2 : 0) + (h2 ? 1 : 0), idx = base + v * NG + gi;
                    const bool mine = idx < cnt && (gl & (G / 4 - 1)) == 0;
                    bool bad = false;
                    if (mine) {
                        const int e = lst[idx];
                        const float4 c = tile[(size_t)(2 * (e & 0x7fff) + (e >> 15)) * rowf4 + rowf4 - 1];
                        const cf term = cf{c.x, c.y} * k;
                        const float mag = fmaxf(fabsf(term.x), fabsf(term.y));
                        const float mk_ = fmaxf(fabsf(k.x), fabsf(k.y));
                        bad = !(mag < 1e30f && mag > 1e-30f && mk_ < 1e30f && mk_ > 1e-30f);
                        if (!bad) {
                            ff_add(sx[u], term.x);
                            ff_add(sy[u], term.y);
                            if (A.probe) {
                                const cf td = (e >> 15 ? -1.f : 1.f) * (cf{c.z, c.w} * term);
                                ff_add(dx[u], td.x);
                                ff_add(dy[u], td.y);
                            }
                        }
                    }
                    uint32_t bm = __ballot_sync(0xffffffffu, bad);
                    while (bm) {
                        const int src = __ffs(bm) - 1;
                        bm &= bm - 1;
                        const int e = lst[__shfl_sync(0xffffffffu, idx, src)];
                        const int s = e >> 15 ? -1 : 1, b = b0 + (e & 0x7fff);
                        const zd term = slow_product(A, w0 + u, b, s, ex[u]);
                        if (lane == 0) {
                            const float4 c = tile[(size_t)(2 * (e & 0x7fff) + (e >> 15)) * rowf4 + rowf4 - 1];
                            A.out[w0 + u].slow = A.out[w0 + u].slow + term;
                            A.out[w0 + u].slow_d =
                                A.out[w0 + u].slow_d + (double)s * (zd{(double)c.z, (double)c.w} * term);
                        }
                    }
                }
            }
            __syncwarp();
            if (!resident) {
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(tc::smem_u32(&empty[buf]))
                                 : "memory");
                // the next tile of this buffer, once every warp has left it
                if (t == 0 && issued < nloads) {
                    if (tc::mbar_wait(&empty[buf], (step >> 1) & 1, WAIT_LIMIT)) load();
                    else ok = false;
                }
                if (warp == 0) ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
            }
        }
        if (!ok) break;
#pragma unroll
        for (int u = 0; u < WPW; ++u) {
            const ff x = ff_warp_sum(sx[u]), y = ff_warp_sum(sy[u]);
            ff p = {0.f, 0.f}, q = {0.f, 0.f};
            if (A.probe) {
                p = ff_warp_sum(dx[u]);
                q = ff_warp_sum(dy[u]);
            }
            if (lane == 0 && w0 + u < A.n) {
                A.out[w0 + u].off = make_float4(x.hi, x.lo, y.hi, y.lo);
                A.out[w0 + u].offd = make_float4(p.hi, p.lo, q.hi, q.lo);
            }
        }
    }
    if (!ok) {
        if (lane == 0) set_status(A.status, CR_ETIMEOUT);
        // copies in flight land before the shared memory is released (bounded)
        if (t == 0)
            for (int q = issued > 2 ? issued - 2 : 0; q < issued; ++q)
                tc::mbar_wait(&full[q & 1], (q >> 1) & 1, WAIT_LIMIT);
    }
}

// Lanes per hidden layer and unit pairs per lane for M hidden units: the
// fewest padded units, as many units per lane as registers allow (fewer
// lanes per bond then share a warp).
struct Shape { int G, KP; };
Shape shape_of(int M) {
    static const Shape s[] = {{8, 1}, {8, 2}, {8, 3}, {8, 4}, {16, 3}, {16, 4}, {32, 3}, {32, 4}, {32, 6}, {32, 8}};
    for (const Shape& q : s)
        if (M <= 2 * q.G * q.KP) return q;
    return s[9];
}
int row_f4(int M) {
    const Shape s = shape_of(M);
    return s.G * s.KP + 1;
}
int wpw_of(int M) { return shape_of(M).KP <= 4 ? 2 : 1; }

size_t xsum_smem(const cr_ctx* c, int nbt) {
    const int wpw = wpw_of(c->M), nmw = (c->Nb + 31) / 32;
    return 2 * (size_t)nbt * 2 * row_f4(c->M) * 16 + 32 + (size_t)c->Nb * 8 +
           (size_t)XW * wpw * 2 * nmw * 4 + XW * MAX_TILE * 2 + (size_t)XW * c->N;
}

// Bonds per tile: whole tables of at most two tiles stay in shared memory.
int tile_bonds(const cr_ctx* c) {
    int nbt = TILE_BYTES / (2 * row_f4(c->M) * 16);
    if (nbt > MAX_TILE) nbt = MAX_TILE;
    if (nbt > c->Nb) nbt = c->Nb;
    while (nbt > 1 && xsum_smem(c, nbt) > 227 * 1024) --nbt;
    const int nt = (c->Nb + nbt - 1) / nbt;
    return (c->Nb + nt - 1) / nt;  // tiles of equal size
}

template <int G, int KP>
cr_status xsum_t(cr_ctx* c, const XArgs* a) {
    constexpr int WPW = KP <= 4 ? 2 : 1;
    if (!a) {
        cudaError_t e = cudaFuncSetAttribute(xsum_kernel<G, KP, WPW>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        return e == cudaSuccess ? CR_OK : cr_fail(c, CR_ECUDA, "xsum: %s", cudaGetErrorString(e));
    }
    const int per = XW * WPW, nblk = (a->n + per - 1) / per;
    CR_LAUNCH(c, CR_KERNEL_TARGET,
              xsum_kernel<G, KP, WPW><<<nblk < c->n_sm ? nblk : c->n_sm, 32 * XW, xsum_smem(c, a->nbt),
                                        c->stream>>>(*a));
    return cr_check_launch(c, "xsum_kernel");
}

cr_status xsum_dispatch(cr_ctx* c, const XArgs* a) {
    const Shape s = shape_of(c->M);
    switch (s.G * 16 + s.KP) {
        case 8 * 16 + 1: return xsum_t<8, 1>(c, a);
        case 8 * 16 + 2: return xsum_t<8, 2>(c, a);
        case 8 * 16 + 3: return xsum_t<8, 3>(c, a);
        case 8 * 16 + 4: return xsum_t<8, 4>(c, a);
        case 16 * 16 + 3: return xsum_t<16, 3>(c, a);
        case 16 * 16 + 4: return xsum_t<16, 4>(c, a);
        case 32 * 16 + 3: return xsum_t<32, 3>(c, a);
        case 32 * 16 + 4: return xsum_t<32, 4>(c, a);
        case 32 * 16 + 6: return xsum_t<32, 6>(c, a);
        default: return xsum_t<32, 8>(c, a);
    }
}

}  // namespace

size_t xsum_table_bytes(const cr_ctx* c) { return (size_t)c->Nb * 2 * row_f4(c->M) * 16; }

cr_status xsum_prepare(cr_ctx* c) { return xsum_dispatch(c, nullptr); }

cr_status launch_xsum(cr_ctx* c, const void* params, const int8_t* spins, const void* theta, int n,
                      int probe, double qx, double qy, xsum_out* out) {
    const int rf = row_f4(c->M);
    CR_LAUNCH(c, CR_K_OTHER,
              xtable_kernel<<<(c->Nb + 3) / 4, 128, 0, c->stream>>>((const cf*)params, c->d_bonds, c->N, c->M,
                                                                    c->Nb, rf, c->Lx, probe, qx, qy,
                                                                    (float4*)c->xtab));
    XArgs a;
    a.spins = spins;
    a.th = (const cf*)theta;
    a.prm = (const cf*)params;
    a.tab = (const float4*)c->xtab;
    a.bonds = c->d_bonds;
    a.n = n;
    a.N = c->N;
    a.M = c->M;
    a.Nb = c->Nb;
    a.rowf4 = rf;
    a.nbt = tile_bonds(c);
    a.ntiles = (c->Nb + a.nbt - 1) / a.nbt;
    a.probe = probe;
    a.out = out;
    a.status = c->d_status;
    return xsum_dispatch(c, &a);
}
