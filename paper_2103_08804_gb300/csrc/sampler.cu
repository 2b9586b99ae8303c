// Metropolis sampling of |psi_s|^2 (Sec. III) with S^z-conserving exchange
// moves on nearest-neighbour bonds.
//
// sweep_kernel: one warp per walker.  Lane l owns the KPL hidden units j =
// 32 k + l (k < KPL) of the padded width Mp = 32 KPL and keeps tanh(theta) for
// them in registers.  The amplitude ratio of a proposal is the product over
// hidden units of (cosh D - s tanh(theta) sinh D) from the bond tables, so
// the inner loop is complex FMA only; accepted moves update tanh(theta) by the
// same addition formula.  Proposals on parallel bonds are no-ops (rejected):
// the 64 proposals of a Philox block are tested at once, two per lane, and
// after an accepted move only the bonds that share one site with it change
// sides.
//
// sweep_l1_kernel takes smaller tables, which stay in L1 (sweep_in_l1 has the
// rule and both sides' times); what follows is the form for large ones.
//
// What bounds it: a proposal is a chain of a table read (4 KB from L2 at 256
// hidden units), the product across the warp, the accept test and, mostly,
// the update.  The rows of the next proposal that can be evaluated are
// therefore copied into the warp's shared memory (cp.async, every lane its own
// 16 bytes) while the present one is computed, and theta, which only the
// output needs, is left out of the chain: accepted moves go to a list, and
// replay_slice_kernel or finish_kernel applies them in order afterwards (the
// same subtractions in the same order, independent loads, a table too large
// for L1 taken in slices of its units that fit in shared memory).  16 x 16
// lattice, 65536 walkers: 8.0 -> 5.5 ms, of which the sweep
// kernel 4.8; it issues on 65% of its cycles, 480 instructions per evaluated
// proposal, at 27% of the L2 rate.
#include "common.cuh"

namespace {

// 16 bytes global -> shared, asynchronous, visible to the issuing thread after
// its wait_group
CR_D void cp16(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
CR_D void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> CR_D void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// First proposal after pos (proposals 2 l in e, 2 l + 1 in o), 64 if none.
CR_D int next_after(uint32_t e, uint32_t o, int pos) {
    const int le = (pos + 2) >> 1, lo = (pos + 1) >> 1;
    const uint32_t es = le < 32 ? e >> le : 0u, os = lo < 32 ? o >> lo : 0u;
    const int pe = es ? 2 * (le + __ffs(es) - 1) : 64, po = os ? 2 * (lo + __ffs(os) - 1) + 1 : 64;
    return min(pe, po);
}

// Complex arithmetic of the accept test with its float32 roundings spelled
// out: a decision u < ratio is a float32 comparison, so a walker's trajectory
// depends on the last bit of every step, and the compiler's choice of which
// product of a sum it fuses changes with the code around it.  YX: the y part
// fuses a.y b.x (else a.x b.y).
template <bool YX> CR_D cpx<float> cmul_rn(cpx<float> a, cpx<float> b) {
    return {__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)),
            YX ? __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)) : __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x))};
}
template <bool YX> CR_D cpx<double> cmul_rn(cpx<double> a, cpx<double> b) { return a * b; }
// |a|^2; YY: fuses y^2
template <bool YY> CR_D float abs2_rn(cpx<float> a) {
    return YY ? __fmaf_rn(a.y, a.y, __fmul_rn(a.x, a.x)) : __fmaf_rn(a.x, a.x, __fmul_rn(a.y, a.y));
}
template <bool YY> CR_D double abs2_rn(cpx<double> a) { return abs2(a); }
template <bool YY> CR_D cpx<float> cdiv_rn(cpx<float> a, cpx<float> b) {
    const float d = __frcp_rn(abs2_rn<YY>(b));
    return {__fmul_rn(__fmaf_rn(a.x, b.x, __fmul_rn(a.y, b.y)), d),
            __fmul_rn(__fmaf_rn(a.y, b.x, -__fmul_rn(a.x, b.y)), d)};
}
template <bool YY> CR_D cpx<double> cdiv_rn(cpx<double> a, cpx<double> b) { return cdiv(a, b); }

// the same product in every lane (one value for the whole warp)
template <typename R> CR_D cpx<R> warp_prod_rn(cpx<R> v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v = cmul_rn<true>(v, cpx<R>{__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o)});
    return {__shfl_sync(0xffffffffu, v.x, 0), __shfl_sync(0xffffffffu, v.y, 0)};
}

// tanh of a lane's units 32 k + lane < M (0 past M).  Next to a node, which is
// rare, the lane's values are formed again behind one branch: a branch per unit
// would keep the units' chains of exponentials and sines from running side by
// side.
template <typename R, int KPL>
CR_D void tanh_units(const cpx<R> (&th)[KPL], int M, int lane, cpx<R> (&T)[KPL]) {
    bool near = false;
#pragma unroll
    for (int k = 0; k < KPL; ++k) {
        R d = R(1);
        T[k] = {R(0), R(0)};
        if (32 * k + lane < M) T[k] = ctanh_far(th[k], &d);
        near = near || near_node(d);
    }
    if (near)
#pragma unroll
        for (int k = 0; k < KPL; ++k)
            if (32 * k + lane < M) T[k] = ctanh_(th[k]);
}

// theta (theta_out may be null: in place already), tanh theta and log psi of
// walker w, whose units 32 k + lane are th[k].
template <typename R, int KPL>
CR_D void walker_outputs(const cpx<R> (&th)[KPL], int lane, int w, int M, int N, const cpx<R>* prm,
                         const int8_t* sg, cpx<R>* theta_out, cpx<R>* logpsi_out, cpx<R>* tanh_out) {
    cpx<R> lp = {R(0), R(0)};
    bool near = false;
#pragma unroll
    for (int k = 0; k < KPL; ++k) {
        const int j = 32 * k + lane;
        if (j < M) {
            R d, dt = R(1);
            if (theta_out) theta_out[(size_t)w * M + j] = th[k];
            lp = lp + clncosh2_far(th[k], &d);
            if (tanh_out) tanh_out[(size_t)w * M + j] = ctanh_far(th[k], &dt);
            near = near || near_node(d) || near_node(dt);
        }
    }
    if (near) {
        lp = {R(0), R(0)};
#pragma unroll
        for (int k = 0; k < KPL; ++k) {
            const int j = 32 * k + lane;
            if (j < M) {
                R d;
                const cpx<R> v = clncosh2_far(th[k], &d);
                lp = lp + (near_node(d) ? clncosh2_near(th[k]) : v);
                if (tanh_out) tanh_out[(size_t)w * M + j] = ctanh_(th[k]);
            }
        }
    }
    if (!logpsi_out) return;
    for (int i = lane; i < N; i += 32) lp = lp + R(sg[i]) * prm[i];
    lp = warp_sum(lp);
    if (lane == 0) logpsi_out[w] = lp;
}

constexpr int LIST_NEG = 0x8000;  // list entry: bond, this bit for s = -1

}  // namespace

template <typename R, int KPL>
__global__ void __launch_bounds__(128) sweep_kernel(
    int8_t* __restrict__ spins, const cpx<R>* __restrict__ theta, cpx<R>* __restrict__ Tws, int B,
    int N, int M, int Nb, const int2* __restrict__ bonds_g, const cpx<R>* __restrict__ CS,
    const cpx<R>* __restrict__ ea, int p_base, int n_prop, int more, uint32_t k0, uint32_t k1,
    unsigned long long counter, const unsigned long long* __restrict__ dcounter,
    uint16_t* __restrict__ list, int cap, int* __restrict__ count) {
    if (dcounter) counter = *dcounter;  // stream position kept on the device
    constexpr int Mp = 32 * KPL, ROW = 2 * Mp;       // (ch, sh) pairs of a bond
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    cpx<R>* buf = (cpx<R>*)smem_raw + wid * 2 * ROW;  // [4][2][ROW]
    uint32_t* bonds = (uint32_t*)((cpx<R>*)smem_raw + 8 * ROW);  // [Nb], sites packed 16 + 16
    int8_t* sg = (int8_t*)(bonds + Nb) + wid * N;     // [4][N]
    for (int e = threadIdx.x; e < Nb; e += blockDim.x) {
        const int2 bd = bonds_g[e];
        bonds[e] = (uint32_t)bd.x | ((uint32_t)bd.y << 16);
    }
    const int w = blockIdx.x * 4 + wid;
    if (w < B)
        for (int i = lane; i < N; i += 32) sg[i] = spins[(size_t)w * N + i];
    __syncthreads();
    if (w >= B) return;

    cpx<R> T[KPL];
#pragma unroll
    for (int k = 0; k < KPL; ++k) {
        const int j = 32 * k + lane;
        T[k] = j < M ? (p_base ? Tws : theta)[(size_t)w * M + j] : cpx<R>{R(0), R(0)};
    }
    if (!p_base) {
        cpx<R> t[KPL];
        tanh_units(T, M, lane, t);
#pragma unroll
        for (int k = 0; k < KPL; ++k) T[k] = t[k];
    }
    // copy the rows of bond b into buffer q: every lane the pairs it will read
    auto fetch = [&](int b, int q) {
        const unsigned char* src = (const unsigned char*)(CS + (size_t)b * ROW);
        unsigned char* dst = (unsigned char*)(buf + q * ROW);
#pragma unroll
        for (int k = 0; k < KPL; ++k) {
            const int o = (32 * k + lane) * 2 * (int)sizeof(cpx<R>);
#pragma unroll
            for (int c = 0; c < 2 * (int)sizeof(cpx<R>); c += 16) cp16(dst + o + c, src + o + c);
        }
    };
    int nacc = 0, q = 0;
    uint32_t ent = 0;
    uint16_t* lst = list + (size_t)w * cap;
    for (int p0 = 0; p0 < n_prop; p0 += 64) {
        const unsigned long long step = counter + (unsigned long long)((p_base + p0) >> 1) + lane;
        const uint4 rnd = philox4x32_10(
            make_uint4((uint32_t)w, (uint32_t)step, (uint32_t)(step >> 32), 0u), k0, k1);
        // this lane's two proposals
        const int b0 = (int)__umulhi(rnd.x, (uint32_t)Nb), b1 = (int)__umulhi(rnd.z, (uint32_t)Nb);
        const uint32_t s0 = bonds[b0], s1 = bonds[b1];
        const bool v0 = p0 + 2 * lane < n_prop, v1 = p0 + 2 * lane + 1 < n_prop;
        // proposals on antiparallel bonds
        uint32_t A0 = __ballot_sync(0xffffffffu, v0 && sg[s0 & 0xffff] != sg[s0 >> 16]);
        uint32_t A1 = __ballot_sync(0xffffffffu, v1 && sg[s1 & 0xffff] != sg[s1 >> 16]);
        int cur = next_after(A0, A1, -1);
        if (cur < 64) {
            fetch(__shfl_sync(0xffffffffu, (cur & 1) ? b1 : b0, cur >> 1), q);
            cp_commit();
        }
        while (cur < 64) {
            const int src = cur >> 1;
            const int b = __shfl_sync(0xffffffffu, (cur & 1) ? b1 : b0, src);
            const uint32_t bs = __shfl_sync(0xffffffffu, (cur & 1) ? s1 : s0, src);
            const uint32_t ua = __shfl_sync(0xffffffffu, (cur & 1) ? rnd.w : rnd.y, src);
            const uint32_t bx = bs & 0xffff, by = bs >> 16;
            // proposals whose bond shares one site with this one: an accepted move
            // takes them to the other side
            const uint32_t x0 = s0 & 0xffff, y0 = s0 >> 16, x1 = s1 & 0xffff, y1 = s1 >> 16;
            const uint32_t O0 = __ballot_sync(0xffffffffu, v0 && ((x0 == bx || x0 == by) != (y0 == bx || y0 == by)));
            const uint32_t O1 = __ballot_sync(0xffffffffu, v1 && ((x1 == bx || x1 == by) != (y1 == bx || y1 == by)));
            int nxt = next_after(A0 | O0, A1 | O1, cur);
            if (nxt < 64) fetch(__shfl_sync(0xffffffffu, (nxt & 1) ? b1 : b0, nxt >> 1), q ^ 1);
            cp_commit();
            const int si = sg[bx];
            const cpx<R> e = ea[2 * b + (si > 0 ? 0 : 1)];
            const R s = R(si);
            cp_wait<1>();
            const cpx<R>* row = buf + q * ROW + 2 * lane;
            cpx<R> f[KPL];
            cpx<R> pl = {R(1), R(0)};
#pragma unroll
            for (int k = 0; k < KPL; ++k) {
                const cpx<R> ch = row[64 * k], sh = row[64 * k + 1];
                cpx<R> ts = cmul_rn<false>(T[k], sh);
                f[k] = {ch.x - s * ts.x, ch.y - s * ts.y};
                pl = cmul_rn<false>(pl, f[k]);
            }
            const cpx<R> pw = warp_prod_rn(pl);
            const R ratio2 = abs2_rn<false>(e) * abs2_rn<false>(pw);
            const R u = (R(ua >> 9) + R(0.5)) * R(1.1920928955078125e-07);
            if (u < ratio2) {
#pragma unroll
                for (int k = 0; k < KPL; ++k) {
                    const cpx<R> ch = row[64 * k], sh = row[64 * k + 1];
                    cpx<R> tc = cmul_rn<(KPL > 1)>(T[k], ch);
                    T[k] = cdiv_rn<KPL == 1>(cpx<R>{tc.x - s * sh.x, tc.y - s * sh.y}, f[k]);
                }
                __syncwarp();
                if (lane == 0) {
                    sg[bx] = (int8_t)(-si);
                    sg[by] = (int8_t)si;
                }
                __syncwarp();
                A0 ^= O0;
                A1 ^= O1;
                if (lane == (nacc & 31)) ent = (uint32_t)b | (si > 0 ? 0u : (uint32_t)LIST_NEG);
                ++nacc;
                if ((nacc & 31) == 0) lst[nacc - 32 + lane] = (uint16_t)ent;
            }
            if (nxt < 64 && !((((nxt & 1) ? A1 : A0) >> (nxt >> 1)) & 1u)) {
                // the prefetched proposal turned parallel: take the one after it.  Its
                // copy lands first, also where none follows in this block: copies have no
                // order among themselves, and the next block's first rows go to the
                // same buffer
                nxt = next_after(A0, A1, nxt);
                cp_wait<0>();
                if (nxt < 64) {
                    fetch(__shfl_sync(0xffffffffu, (nxt & 1) ? b1 : b0, nxt >> 1), q ^ 1);
                    cp_commit();
                }
            }
            cur = nxt;
            q ^= 1;
        }
    }
    cp_wait<0>();
    if (lane < (nacc & 31)) lst[(nacc & ~31) + lane] = (uint16_t)ent;
    __syncwarp();
    for (int i = lane; i < N; i += 32) spins[(size_t)w * N + i] = sg[i];
    if (more)
#pragma unroll
        for (int k = 0; k < KPL; ++k)
            if (32 * k + lane < M) Tws[(size_t)w * M + 32 * k + lane] = T[k];
    if (lane == 0) count[w] = nacc;
}

// The same sweep where the tables stay in L1: the rows are read as they are
// needed (cosh and sinh in rows of their own) and theta is carried along, so
// that neither a list nor a second pass over it is needed.  The same operations
// in the same order on every value.
template <typename R, int KPL>
__global__ void __launch_bounds__(128) sweep_l1_kernel(
    const cpx<R>* __restrict__ prm, int8_t* __restrict__ spins, cpx<R>* __restrict__ theta, int B, int N,
    int M, int Nb, const int2* __restrict__ bonds_g, const cpx<R>* __restrict__ Dt,
    const cpx<R>* __restrict__ CS, const cpx<R>* __restrict__ ea, int n_prop, uint32_t k0, uint32_t k1,
    unsigned long long counter, const unsigned long long* __restrict__ dcounter,
    cpx<R>* __restrict__ logpsi_out, cpx<R>* __restrict__ tanh_out, int32_t* __restrict__ n_acc) {
    if (dcounter) counter = *dcounter;  // stream position kept on the device
    constexpr int Mp = 32 * KPL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int2* bonds = (int2*)smem_raw;                       // [Nb]
    int8_t* sg_all = (int8_t*)(bonds + Nb);              // [4][N]
    for (int e = threadIdx.x; e < Nb; e += blockDim.x) bonds[e] = bonds_g[e];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int w = blockIdx.x * 4 + wid;
    int8_t* sg = sg_all + wid * N;
    if (w < B)
        for (int i = lane; i < N; i += 32) sg[i] = spins[(size_t)w * N + i];
    __syncthreads();
    if (w >= B) return;

    cpx<R> th[KPL], T[KPL];
#pragma unroll
    for (int k = 0; k < KPL; ++k) {
        const int j = 32 * k + lane;
        th[k] = j < M ? theta[(size_t)w * M + j] : cpx<R>{R(0), R(0)};
    }
    tanh_units(th, M, lane, T);
    int nacc = 0;
    uint4 rnd = make_uint4(0, 0, 0, 0);
    for (int p = 0; p < n_prop; ++p) {
        if ((p & 63) == 0) {
            const unsigned long long step = counter + (unsigned long long)(p >> 1) + lane;
            rnd = philox4x32_10(make_uint4((uint32_t)w, (uint32_t)step, (uint32_t)(step >> 32), 0u), k0, k1);
        }
        const int src = (p >> 1) & 31;
        const uint32_t ub = __shfl_sync(0xffffffffu, (p & 1) ? rnd.z : rnd.x, src);
        const uint32_t ua = __shfl_sync(0xffffffffu, (p & 1) ? rnd.w : rnd.y, src);
        const int b = (int)__umulhi(ub, (uint32_t)Nb);
        const int2 bd = bonds[b];
        const int si = sg[bd.x];
        if (si == sg[bd.y]) continue;  // parallel: no-op, counts as rejected
        const R s = R(si);
        const cpx<R>* row = CS + 2 * (size_t)b * Mp + lane;
        cpx<R> ch[KPL], sh[KPL], f[KPL];
        cpx<R> pl = {R(1), R(0)};
#pragma unroll
        for (int k = 0; k < KPL; ++k) {
            ch[k] = ldg(row + 32 * k);
            sh[k] = ldg(row + Mp + 32 * k);
            const cpx<R> ts = cmul_rn<false>(T[k], sh[k]);
            f[k] = {ch[k].x - s * ts.x, ch[k].y - s * ts.y};
            pl = cmul_rn<false>(pl, f[k]);
        }
        const cpx<R> pw = warp_prod_rn(pl);
        const cpx<R> e = ea[2 * b + (si > 0 ? 0 : 1)];
        const R ratio2 = abs2_rn<false>(e) * abs2_rn<false>(pw);
        const R u = (R(ua >> 9) + R(0.5)) * R(1.1920928955078125e-07);
        if (u < ratio2) {
            const cpx<R>* dr = Dt + (size_t)b * Mp + lane;
#pragma unroll
            for (int k = 0; k < KPL; ++k) {
                const cpx<R> d = ldg(dr + 32 * k);
                th[k] = {th[k].x - s * d.x, th[k].y - s * d.y};
                const cpx<R> tc = cmul_rn<(KPL > 1)>(T[k], ch[k]);
                T[k] = cdiv_rn<KPL == 1>(cpx<R>{tc.x - s * sh[k].x, tc.y - s * sh[k].y}, f[k]);
            }
            __syncwarp();
            if (lane == 0) {
                sg[bd.x] = (int8_t)(-si);
                sg[bd.y] = (int8_t)si;
            }
            __syncwarp();
            ++nacc;
        }
    }
    __syncwarp();
    for (int i = lane; i < N; i += 32) spins[(size_t)w * N + i] = sg[i];
    if (lane == 0 && n_acc) n_acc[w] = nacc;
    walker_outputs<R, KPL>(th, lane, w, M, N, prm, sg, theta, logpsi_out, tanh_out);
}

// theta -> theta - sum of the listed moves' s D, in the list's order, for one
// unit j of walker w (lane's unit; entries broadcast from the lanes that read
// them).
template <typename R, int KPL>
CR_D void replay_list(const uint16_t* __restrict__ lst, int n, const cpx<R>* __restrict__ Dt, int Mp,
                      int lane, cpx<R> (&th)[KPL]) {
    for (int e0 = 0; e0 < n; e0 += 32) {
        const int mine = e0 + lane < n ? lst[e0 + lane] : 0;
        const int m = min(32, n - e0);
        for (int c = 0; c < m; c += 4) {
            cpx<R> d[4][KPL];
            R s[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int e = __shfl_sync(0xffffffffu, mine, c + v);  // c + v < 32
                s[v] = c + v < m ? (e & LIST_NEG ? R(-1) : R(1)) : R(0);
                const cpx<R>* dr = Dt + (size_t)(e & (LIST_NEG - 1)) * Mp;
#pragma unroll
                for (int k = 0; k < KPL; ++k) d[v][k] = ldg(dr + 32 * k);
            }
#pragma unroll
            for (int v = 0; v < 4; ++v)
                if (c + v < m)
#pragma unroll
                    for (int k = 0; k < KPL; ++k)
                        th[k] = {th[k].x - s[v] * d[v][k].x, th[k].y - s[v] * d[v][k].y};
        }
    }
}

// 16 aligned bytes: two units in float32, one in float64
CR_D void lds16(const unsigned char* p, cpx<float> (&d)[2]) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    d[0] = {v.x, v.y};
    d[1] = {v.z, v.w};
}
CR_D void lds16(const unsigned char* p, cpx<double> (&d)[1]) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    d[0] = {v.x, v.y};
}

// The same for a table that does not fit in L1: a CTA holds a slice of the
// units of all bonds in shared memory (LPW pieces of 16 bytes per bond) and
// takes every ncta-th group of walkers, LPW lanes to a walker.  Bound by
// shared memory, 8 bytes per move and unit (16 x 16 lattice, alpha = 1, 65536
// walkers: 0.60 ms; through L1, a warp to a walker and one unit to a lane,
// 1.17).
template <typename R, int LPW>
__global__ void __launch_bounds__(1024, 1) replay_slice_kernel(cpx<R>* __restrict__ theta, int B, int M,
                                                               int Mp, int Nb, int ncta,
                                                               const cpx<R>* __restrict__ Dt,
                                                               const uint16_t* __restrict__ list, int cap,
                                                               const int* __restrict__ count) {
    constexpr int U = 16 / sizeof(cpx<R>), JW = LPW * U, GPW = 32 / LPW;
    extern __shared__ __align__(16) unsigned char sm_rp[];
    const int slice = blockIdx.x / ncta, part = blockIdx.x % ncta;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31, grp = lane / LPW, li = lane % LPW;
    for (int e = t; e < Nb * LPW; e += 1024)
        cp16(sm_rp + (size_t)e * 16, Dt + (size_t)(e / LPW) * Mp + slice * JW + (e % LPW) * U);
    cp_commit();
    cp_wait<0>();
    __syncthreads();
    const unsigned char* Ds = sm_rp + li * 16;
    const int j = slice * JW + li * U;
    for (int wb = (part * 32 + warp) * GPW; wb < B; wb += ncta * 32 * GPW) {
        const int w = wb + grp;
        const int n = w < B ? count[w] : 0;
        const int nmax = __reduce_max_sync(0xffffffffu, n);
        const uint16_t* lst = list + (size_t)(w < B ? w : 0) * cap;
        cpx<R> th[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            th[u] = w < B && j + u < M ? theta[(size_t)w * M + j + u] : cpx<R>{R(0), R(0)};
        for (int e0 = 0; e0 < nmax; e0 += 4 * LPW) {
            // four entries a lane (lists start on 8 bytes)
            uint2 mine = make_uint2(0u, 0u);
            if (e0 + 4 * li < n) mine = *reinterpret_cast<const uint2*>(lst + e0 + 4 * li);
            const int m = min(4 * LPW, nmax - e0);
            for (int c = 0; c < m; c += 4) {
                const uint32_t x = __shfl_sync(0xffffffffu, mine.x, c >> 2, LPW);
                const uint32_t y = __shfl_sync(0xffffffffu, mine.y, c >> 2, LPW);
                cpx<R> d[4][U];
                R s[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const uint32_t q = v < 2 ? x : y, ent = (v & 1) ? q >> 16 : q & 0xffffu;
                    const bool in = e0 + c + v < n;
                    s[v] = ent & LIST_NEG ? R(-1) : R(1);
                    const unsigned char* row = Ds + (in ? ent & (LIST_NEG - 1) : 0u) * (LPW * 16);
                    lds16(row, d[v]);
                }
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    if (e0 + c + v < n)
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            th[u] = {th[u].x - s[v] * d[v][u].x, th[u].y - s[v] * d[v][u].y};
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (w < B && j + u < M) theta[(size_t)w * M + j + u] = th[u];
    }
}

// One warp per walker: the listed moves (list may be null: none left), then
// theta, tanh theta and log psi of the walker.
template <typename R, int KPL>
__global__ void __launch_bounds__(128) finish_kernel(
    const cpx<R>* __restrict__ prm, const int8_t* __restrict__ spins, cpx<R>* __restrict__ theta, int B,
    int N, int M, const cpx<R>* __restrict__ Dt, const uint16_t* __restrict__ list, int cap,
    const int* __restrict__ count, int last, int first, cpx<R>* __restrict__ logpsi_out,
    cpx<R>* __restrict__ tanh_out, int32_t* __restrict__ n_acc) {
    const int lane = threadIdx.x & 31, w = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (w >= B) return;
    cpx<R> th[KPL];
#pragma unroll
    for (int k = 0; k < KPL; ++k) {
        const int j = 32 * k + lane;
        th[k] = j < M ? theta[(size_t)w * M + j] : cpx<R>{R(0), R(0)};
    }
    const int n = count ? count[w] : 0;
    if (list) {
        replay_list<R, KPL>(list + (size_t)w * cap, n, Dt + lane, 32 * KPL, lane, th);
#pragma unroll
        for (int k = 0; k < KPL; ++k)
            if (32 * k + lane < M) theta[(size_t)w * M + 32 * k + lane] = th[k];
    }
    if (lane == 0 && n_acc) n_acc[w] = (first ? 0 : n_acc[w]) + n;
    if (!last) return;
    walker_outputs<R, KPL>(th, lane, w, M, N, prm, spins + (size_t)w * N, (cpx<R>*)nullptr, logpsi_out,
                           tanh_out);
}

// Advance a device-resident stream position (after the sweep that used it).
__global__ void advance_counter_kernel(unsigned long long* ctr, unsigned long long calls) {
    *ctr += calls;
}

// Whether a sweep reads its tables through L1 (sweep_l1_kernel) or prefetches
// rows and replays lists (sweep_kernel).  The first has no second pass and no
// list, but every evaluated proposal waits for its rows; warps hide that where
// there are many of them with few units each, or where the tables (cosh, sinh
// and D, 24 or 48 bytes a bond and unit) stay in L1.  Times of four sweeps, us,
// lists / L1, one GB300 (152 SMs):
//   units, table             walkers: 608      1400     3001     6001     20005
//   15 x 6 lattice, 40, 270 KB     146/151  165/158  214/179  390/333 1087/890
//   14 x 9, 48, 378 KB             195/221  220/230  288/258  529/487 1489/1291
//   16 x 16, 64, 768 KB            418/489  470/507  598/552 1087/1055 3035/2764
//   90 sites, 128, 270 KB          181/185  211/203  275/235  511/447 1529/1410
//   8 x 8, 128, 384 KB             132/159  153/167  200/189  368/354 1102/1126
//   10 x 8, 128, 480 KB            164/203  191/216  257/240  466/452 1395/1447
//   10 x 10, 100, 600 KB           197/261  231/275  315/303  570/576 1721/1855
//   12 x 12, 128, 864 KB           289/385     -     456/443  819/851 2462/2782
//   24 sites, 250, 144 KB (a sweep) 40/41    44/41    69/65   101/97   267/279
// With 128 units an SM holds five blocks of four walkers, and L1 is as fast as
// the lists or faster where its last wave is full (3001 and 6001 walkers; 3648:
// 8 x 8 282/317), the more so beside lists that have just begun another block
// per SM (from 2433 walkers).  With 8 units a lane the few warps hide little.
// Float64: the pipe is the bound, L1 is 1 to 10% ahead up to 4 units a lane and
// 5 to 15% behind above.
static size_t sweep_table_bytes(const cr_ctx* c) { return (size_t)c->Nb * c->Mp * 24; }  // float32
bool sweep_takes_lists(const cr_ctx* c) {
    return c->Mp > 128 || (c->prec != CR_FP64 && sweep_table_bytes(c) > 256 * 1024);
}
static bool sweep_in_l1(const cr_ctx* c, int B, int n_prop) {
    if (!sweep_takes_lists(c)) return true;
    if (c->prec == CR_FP64) return false;
    const int kpl = c->Mp / 32;
    const size_t kb = sweep_table_bytes(c) / 1024;
    const int sm = (B - 1) / c->n_sm;  // walkers of the fullest SM, less one
    if (kpl <= 2) return sm >= (int)(kb < 600 ? kb / 50 : 12);
    if (kpl == 4) {
        if (kb <= 300) return sm >= 6;
        return kb <= 448 ? sm % 20 >= 12 : kb <= 640 && sm < 40 && sm % 20 >= 16;
    }
    return kpl == 8 && kb <= 160 && (n_prop >= 48 || (sm >= 8 && sm < 48));
}

// Proposals per sweep launch: its list of accepted moves per walker.
int sweep_list_cap(const cr_ctx* c) { return c->N > 512 ? (c->N + 63) / 64 * 64 : 512; }

template <typename R, int KPL>
static size_t sweep_smem(const cr_ctx* c) {
    return (size_t)8 * 2 * 32 * KPL * sizeof(cpx<R>) + (size_t)c->Nb * 4 + 4 * (size_t)c->N;
}

// Lanes per walker of the sliced replay: the widest slice whose table of all
// bonds fits in shared memory.
constexpr int REPLAY_SMEM = 224 * 1024;
static int replay_lanes(const cr_ctx* c, int lanes) {
    while ((size_t)c->Nb * lanes * 16 > REPLAY_SMEM) lanes /= 2;
    return lanes;
}

template <typename R, int LPW>
static void launch_replay(cr_ctx* c, cpx<R>* th, int B, const cpx<R>* D, int cap) {
    constexpr int JW = LPW * 16 / (int)sizeof(cpx<R>), walkers = 32 * (32 / LPW);
    const int ns = (c->M + JW - 1) / JW, most = (B + walkers - 1) / walkers;
    int ncta = c->n_sm / ns > 1 ? c->n_sm / ns : 1;
    if (ncta > most) ncta = most;
    CR_LAUNCH(c, CR_K_OTHER,
              (replay_slice_kernel<R, LPW><<<ns * ncta, 1024, (size_t)c->Nb * LPW * 16, c->stream>>>(
                  th, B, c->M, c->Mp, c->Nb, ncta, D, c->sw_list, cap, c->sw_count)));
}

template <typename R>
static void launch_replay_slices(cr_ctx* c, cpx<R>* th, int B, const cpx<R>* D, int cap) {
    switch (replay_lanes(c, sizeof(R) == 4 ? 16 : 32)) {
        case 32: launch_replay<R, 32>(c, th, B, D, cap); break;
        case 16: launch_replay<R, 16>(c, th, B, D, cap); break;
        case 8: launch_replay<R, 8>(c, th, B, D, cap); break;
        default: launch_replay<R, 4>(c, th, B, D, cap); break;
    }
}

template <typename R, int KPL>
static cr_status sweep_k(cr_ctx* c, const void* params, int8_t* spins, void* theta, int B, int n_prop,
                         uint64_t seed, uint64_t counter, const uint64_t* dcounter, void* logpsi_out,
                         void* tanh_out, int32_t* n_acc) {
    const cr_tables& t = c->tab[0];
    cpx<R>* th = (cpx<R>*)theta;
    if (sweep_in_l1(c, B, n_prop)) {
        CR_LAUNCH(c, CR_KERNEL_SWEEP,
                  (sweep_l1_kernel<R, KPL><<<(B + 3) / 4, 128, c->Nb * sizeof(int2) + 4 * c->N, c->stream>>>(
                      (const cpx<R>*)params, spins, th, B, c->N, c->M, c->Nb, c->d_bonds, (const cpx<R>*)t.D,
                      (const cpx<R>*)t.CS, (const cpx<R>*)t.ea, n_prop, (uint32_t)seed,
                      (uint32_t)(seed >> 32), (unsigned long long)counter,
                      (const unsigned long long*)dcounter, (cpx<R>*)logpsi_out, (cpx<R>*)tanh_out, n_acc)));
        return cr_check_launch(c, "mc_sweep");
    }
    const cpx<R>* D = (const cpx<R>*)t.D;
    const int cap = sweep_list_cap(c), grid = (B + 3) / 4;
    // a table that fits in L1 beside the loads in flight is replayed whole, by the finishing warps;
    // a larger one in slices of units that fit in shared memory
    const bool slices = (size_t)c->Nb * c->Mp * sizeof(cpx<R>) > 128 * 1024 && KPL > 1;
    int p = 0;
    do {
        const int np = n_prop - p < cap ? n_prop - p : cap;
        const bool last = p + np >= n_prop;
        if (np > 0)
            CR_LAUNCH(c, CR_KERNEL_SWEEP,
                      (sweep_kernel<R, KPL><<<grid, 128, sweep_smem<R, KPL>(c), c->stream>>>(
                          spins, th, (cpx<R>*)c->theta_tmp, B, c->N, c->M, c->Nb, c->d_bonds,
                          (const cpx<R>*)t.CS, (const cpx<R>*)t.ea, p, np, !last, (uint32_t)seed,
                          (uint32_t)(seed >> 32), (unsigned long long)counter,
                          (const unsigned long long*)dcounter, c->sw_list, cap, c->sw_count)));
        if (np > 0 && slices) launch_replay_slices<R>(c, th, B, D, cap);
        CR_LAUNCH(c, CR_K_OTHER,
                  (finish_kernel<R, KPL><<<grid, 128, 0, c->stream>>>(
                      (const cpx<R>*)params, spins, th, B, c->N, c->M, D,
                      np > 0 && !slices ? c->sw_list : nullptr, cap, np > 0 ? c->sw_count : nullptr, last,
                      p == 0, (cpx<R>*)logpsi_out, (cpx<R>*)tanh_out, n_acc)));
        p += np;
    } while (p < n_prop);
    return cr_check_launch(c, "mc_sweep");
}

template <typename R>
static cr_status sweep_t(cr_ctx* c, const void* params, int8_t* spins, void* theta, int B,
                         int n_prop, uint64_t seed, uint64_t counter, const uint64_t* dcounter,
                         void* logpsi_out, void* tanh_out, int32_t* n_acc) {
#define SWEEP(K) \
    sweep_k<R, K>(c, params, spins, theta, B, n_prop, seed, counter, dcounter, logpsi_out, tanh_out, n_acc)
    switch (c->Mp / 32) {
        case 1: return SWEEP(1);
        case 2: return SWEEP(2);
        case 4: return SWEEP(4);
        case 8: return SWEEP(8);
        default: return SWEEP(16);
    }
#undef SWEEP
}

// Opt the sweep of this context's width into the shared memory it needs
// (once per context; the bound covers every context of that width).
template <typename R>
static cr_status sweep_prepare_t(cr_ctx* c) {
    cudaError_t e = cudaSuccess;
#define OPT(K)                                                                                        \
    case K:                                                                                           \
        e = cudaFuncSetAttribute(sweep_kernel<R, K>, cudaFuncAttributeMaxDynamicSharedMemorySize,     \
                                 (int)(8 * 2 * 32 * K * sizeof(cpx<R>) + 2048 * 4 + 4 * 1024));       \
        break;
    switch (c->Mp / 32) {
        OPT(1) OPT(2) OPT(4) OPT(8) OPT(16)
    }
#undef OPT
    const auto opt = [&](const void* f) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, REPLAY_SMEM);
    };
    opt((const void*)replay_slice_kernel<R, 32>);
    opt((const void*)replay_slice_kernel<R, 16>);
    opt((const void*)replay_slice_kernel<R, 8>);
    opt((const void*)replay_slice_kernel<R, 4>);
    return e == cudaSuccess ? CR_OK : cr_fail(c, CR_ECUDA, "sweep_prepare: %s", cudaGetErrorString(e));
}

cr_status sweep_prepare(cr_ctx* c) {
    return c->prec == CR_FP64 ? sweep_prepare_t<double>(c) : sweep_prepare_t<float>(c);
}

extern "C" cr_status mc_sweep(cr_ctx* ctx, const cr_state* st, int8_t* spins, void* theta, int B,
                              int n_sweeps, cr_philox* rng, void* logpsi_out, void* tanh_out,
                              int32_t* n_accepted) {
    if (!ctx) return CR_EINVAL;
    CR_CHECK_ARG(st && st->params, "mc_sweep: null state");
    CR_CHECK_ARG(!st->probe, "mc_sweep: the sampled state must be a plain RBM");
    CR_CHECK_ARG(B >= 0 && B <= ctx->max_walkers, "mc_sweep: B=%d outside [0, %d]", B,
                 ctx->max_walkers);
    CR_CHECK_ARG(n_sweeps >= 0, "mc_sweep: n_sweeps < 0");
    CR_CHECK_ARG(rng, "mc_sweep: null rng");
    CR_CHECK_ARG(ctx->Mp <= 512, "mc_sweep: M > 512 not supported");
    const int n_prop = n_sweeps * ctx->N;
    const uint64_t calls = (uint64_t)(n_prop + 1) / 2;
    if (B > 0) {
        CR_CHECK_ARG(spins && theta, "mc_sweep: null spins or theta");
        cr_status s = build_tables(ctx, st->params, 0, sweep_in_l1(ctx, B, n_prop));
        if (s != CR_OK) return s;
        s = ctx->prec == CR_FP64
                ? sweep_t<double>(ctx, st->params, spins, theta, B, n_prop, rng->seed,
                                  rng->counter, rng->device_counter, logpsi_out, tanh_out,
                                  n_accepted)
                : sweep_t<float>(ctx, st->params, spins, theta, B, n_prop, rng->seed,
                                 rng->counter, rng->device_counter, logpsi_out, tanh_out,
                                 n_accepted);
        if (s != CR_OK) return s;
    }
    if (rng->device_counter) {
        CR_LAUNCH(ctx, CR_K_OTHER, advance_counter_kernel<<<1, 1, 0, ctx->stream>>>(
                                       (unsigned long long*)rng->device_counter, calls));
        return cr_check_launch(ctx, "advance_counter_kernel");
    }
    rng->counter += calls;
    return CR_OK;
}
