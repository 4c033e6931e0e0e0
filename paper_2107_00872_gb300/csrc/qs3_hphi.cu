// qs3_hphi.cu -- the matrix-free product psi = H phi (Alg. 9 of the paper,
// with the readings: norm ratio sqrt(N_a'/N_a) of Eq. (hak2), pull-form phase
// e^{+ik.l} with T^l a' = a'_rep, hop amplitude Jxy/2 of Eq. (1)).
//
// GPU design: one thread per row (consecutive threads own consecutive ranks,
// so in the colex order the gathers phi[a'] of one hop class land close
// together), a persistent grid striding over 256-row tiles of all sectors of
// a basis, the binomial table and the site-coordinate table staged in shared
// memory, and no atomics.  Per row:
//   - unrank (Alg. 1) the row's rank, or the representative's rank sigma[row];
//   - diagonal: sum_b Jz_b/4 - (1/2) sum_{i in a} s_i + (down-down Jz) + field,
//     with s_i = sum_j Jz_ij folded into the per-site constant u_i;
//   - for each down spin i and each bond (i, j) with j empty: the hop target
//     is the sorted list with i replaced by j (Alg. 3); its rank (U(1)), or
//     its representative and stabiliser via the pruned translation search and
//     the two-level index over sigma (k-sectors, Alg. 7-9);
//   - accumulate in the vector's precision (fp32 or fp64), write psi once.
#include <algorithm>
#include <atomic>

#include "qs3_fixed.cuh"
#include "qs3_hphi_common.cuh"

namespace qs3 {


// TB (k-sectors): representative and row from the representative table
// (LatView::orb, SecView::t2) instead of the search and sigma lookup
template <int ND, typename VT, bool KS, bool TB = false>
__global__ void __launch_bounds__(NTHREADS, (KS && TB && sizeof(VT) == 16) ? 4 : 3) k_hphi(LatView L, const SecView *__restrict__ secs,
                                                   const int *__restrict__ tile0, int S, int ntiles,
                                                   const VT *__restrict__ phi, VT *__restrict__ psi,
                                                   const int *__restrict__ active) {
    using R = typename VTr<VT>::R;
    using CT = typename VTr<VT>::C;
    extern __shared__ __align__(16) unsigned char smem[];
    SmemLayout sm = carve(L, smem);
    stage_tables(L, sm.sC, KS ? sm.sxyz : nullptr);
    R *snorm = (R *)sm.snorm;
    if (threadIdx.x < 9) {
        snorm[threadIdx.x] = (R)sqrt((double)threadIdx.x);
        snorm[9 + threadIdx.x] = threadIdx.x ? (R)(1.0 / sqrt((double)threadIdx.x)) : (R)0;
    }
    const R *jxy = jxy_table<VT>(L);
    __syncthreads();
    // persistent grid striding over the tiles of all sectors (better balanced
    // than contiguous per-block ranges, measured); a block restages the phase
    // table of its tile's sector when the sector changes
    CT *ph = (CT *)sm.sph;
    int cur = -1;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int s = (S == 1) ? 0 : sector_of_tile(tile0, S, t);
        if (active && !active[s]) continue;
        const SecView sv = secs[s];
        if (KS && s != cur) {
            __syncthreads();
            const CT *g = phase_table<CT>(sv);
            for (int i = threadIdx.x; i < L.N; i += blockDim.x) ph[i] = g[i];
            __syncthreads();
            cur = s;
        }
        const uint64_t row = (uint64_t)(t - sv.tile0) * TILE + threadIdx.x;
        if (row >= sv.dim) continue;
        const uint64_t rank = KS ? __ldg(sv.sigma + row) : row;
        int c[ND];
        unrank(rank, sm.sC, L.np1, c);
        const VT *ph_in = phi + sv.off;
        const VT x0 = ph_in[row];
        R rs = 0;
        int st_row = 1;
        if constexpr (KS) {
            st_row = sv.stab[row];
            rs = snorm[9 + st_row];
        }
        // diagonal in the vector precision: fp32 kernels keep off the fp64 unit
        R e = diag_c0<R>(L), dd = 0;
        CT acc;
        acc.x = 0; acc.y = 0;
        // k-sectors with one hop amplitude on every bond: sum phase x phi over
        // the hops and multiply by the amplitude once (two fp64 multiplies
        // fewer per hop)
        const R juni = (R)L.jh_uniform;
        const bool uni = KS && juni != (R)0;
        CT acch;
        acch.x = 0; acch.y = 0;
        // U(1), fp32, N_down <= 4: per occupied site, the ranks of its first
        // DEGB hop targets are formed first and their gathers then issue
        // together, so a thread keeps several independent loads in flight
        // (measured: 5% faster for fp32; the fp64 kernels run slower this way)
        constexpr bool BATCH = !KS && ND <= 4 && sizeof(R) == 4;
        constexpr int DEGB = 6;
        if constexpr (BATCH) {
#pragma unroll
            for (int m = 0; m < ND; ++m) {
                const int i = c[m];
                e += diag_u<R>(L, i);
                const int e0 = __ldg(L.adj_ptr + i), e1 = __ldg(L.adj_ptr + i + 1);
                uint64_t r2b[DEGB];
                R cfb[DEGB];
#pragma unroll
                for (int b = 0; b < DEGB; ++b) {
                    const int q = e0 + b;
                    cfb[b] = 0;
                    r2b[b] = 0;
                    if (q < e1) {
                        const int j = __ldg(L.adj_nbr + q);
                        bool occ = false;
#pragma unroll
                        for (int k = 0; k < ND; ++k) occ |= (c[k] == j);
                        if (occ) {
                            dd += diag_jz<R>(L, q);
                        } else {
                            const bool inplace = (m == 0 || j > c[m > 0 ? m - 1 : 0]) &&
                                                 (m == ND - 1 || j < c[m + 1 < ND ? m + 1 : m]);
                            if (inplace) {
                                r2b[b] = rank - sm.sC[(m + 1) * L.np1 + c[m]] + sm.sC[(m + 1) * L.np1 + j];
                            } else {
                                int tt[ND];
#pragma unroll
                                for (int k = 0; k < ND; ++k) tt[k] = (k == m) ? j : c[k];
                                sort_net(tt);
                                r2b[b] = rank_of(tt, sm.sC, L.np1);
                            }
                            cfb[b] = __ldg(jxy + q);
                        }
                    }
                }
                VT vb[DEGB];
#pragma unroll
                for (int b = 0; b < DEGB; ++b)
                    if (cfb[b] != (R)0) vb[b] = ph_in[r2b[b]];
#pragma unroll
                for (int b = 0; b < DEGB; ++b)
                    if (cfb[b] != (R)0) madd_r(acc, cfb[b], vb[b]);
                // sites with more than DEGB neighbours: the rest one at a time
                for (int q = e0 + DEGB; q < e1; ++q) {
                    const int j = __ldg(L.adj_nbr + q);
                    bool occ = false;
#pragma unroll
                    for (int k = 0; k < ND; ++k) occ |= (c[k] == j);
                    if (occ) {
                        dd += diag_jz<R>(L, q);
                        continue;
                    }
                    int tt[ND];
#pragma unroll
                    for (int k = 0; k < ND; ++k) tt[k] = (k == m) ? j : c[k];
                    sort_net(tt);
                    madd_r(acc, __ldg(jxy + q), ph_in[rank_of(tt, sm.sC, L.np1)]);
                }
            }
        }
        // the k-sector hop body (with the representative search) stays rolled:
        // unrolled N_down times it overflows the instruction cache (measured)
        constexpr int UNR = KS ? 1 : ND;
#pragma unroll UNR
        for (int m = 0; m < (BATCH ? 0 : ND); ++m) {
            const int i = pick(c, m);
            e += diag_u<R>(L, i);
            const int e0 = __ldg(L.adj_ptr + i), e1 = __ldg(L.adj_ptr + i + 1);
            // a hop to c_{m-1} < j < c_{m+1} keeps its place in the sorted list
            // (and lands on an empty site): its rank changes in the m-th term only
            const int lo = m > 0 ? pick(c, m > 0 ? m - 1 : 0) : -1;
            const int hi = m < ND - 1 ? pick(c, m < ND - 1 ? m + 1 : m) : L.np1;
            const uint64_t base = rank - sm.sC[(m + 1) * L.np1 + i];
            for (int q = e0; q < e1; ++q) {
                const int j = __ldg(L.adj_nbr + q);
                const bool inpl = j > lo && j < hi;
                if (!inpl) {
                    bool occ = false;
#pragma unroll
                    for (int k = 0; k < ND; ++k) occ |= (c[k] == j);
                    if (occ) {
                        dd += diag_jz<R>(L, q);
                        continue;
                    }
                }
                int tt[ND];
#pragma unroll
                for (int k = 0; k < ND; ++k) tt[k] = (k == m) ? j : c[k];
                const R jh = __ldg(jxy + q);
                if constexpr (!KS) {
                    // j keeps position m when it stays between the neighbours of
                    // c_m: only the m-th term of the rank changes
                    const bool inplace = (m == 0 || j > c[m > 0 ? m - 1 : 0]) && (m == ND - 1 || j < c[m + 1 < ND ? m + 1 : m]);
                    uint64_t r2;
                    if (inplace) {
                        r2 = rank - sm.sC[(m + 1) * L.np1 + c[m]] + sm.sC[(m + 1) * L.np1 + j];
                    } else {
                        sort_net(tt);
                        r2 = rank_of(tt, sm.sC, L.np1);
                    }
                    madd_r(acc, jh, ph_in[r2]);
                } else {
                    uint32_t idx;
                    int u;
                    if constexpr (TB) {
                        uint64_t r2;
                        if (inpl) {
                            r2 = base + sm.sC[(m + 1) * L.np1 + j];
                        } else {
                            sort_net(tt);
                            r2 = rank_of(tt, sm.sC, L.np1);
                        }
                        const uint32_t e = __ldg(L.orb + r2);
                        if ((e >> 12) >= L.n_orb) continue;     // never for a complete table
                        const int32_t row2 = __ldg(sv.t2 + (e >> 12));
                        if (row2 < 0) continue;
                        idx = (uint32_t)row2;
                        u = (int)(e & 4095u);
                    } else {
                        int rep[ND];
                        int ax, by, cz;
                        const uint64_t r2 = canon(tt, L, sm.sxyz, sm.sC, rep, ax, by, cz);
                        if (!sigma_find(sv, rep, sm.sC, L.np1, r2, idx)) continue;
                        u = ax + L.L[0] * (by + L.L[1] * cz);
                    }
                    CT p = ph[u];   // generic load (L1-cached)
                    const int st = __ldg(sv.stab + idx);
                    if (uni) {
                        // uniform J^xy: the amplitude is applied once per row below
                        if (st != st_row) {
                            const R f = snorm[st] * rs;
                            p.x *= f;
                            p.y *= f;
                        }
                        acc_add(acch, p, ph_in[idx]);
                    } else {
                        const R w = (st == st_row) ? jh : jh * snorm[st] * rs;
                        p.x *= w;
                        p.y *= w;
                        acc_add(acc, p, ph_in[idx]);
                    }
                }
            }
        }
        if (KS && uni) madd_r(acc, juni, acch);
        madd_r(acc, e + (R)0.5 * dd, x0);
        store(psi + sv.off + row, acc);
    }
}

// H Phi of the binary64 engine on the integer units: k-sectors with the
// representative table and one hop amplitude J/2 on every bond.  phi comes
// twice (HxVec): as binary64 (the diagonal term) and as its gather image
// (hd_pack).  Each hop's product
// phase x phi is formed exactly on the images (the phases on the grid 2^-52,
// staged per sector as digits) with mad.wide.s32, folded at weight 2^52
// (rounded to nearest) and added to the row sum (RowAcc); terms whose target
// stabiliser differs from the row's (norm ratio != 1, rare) are summed in
// binary64 as in k_hphi.  The row sum is rounded to binary64 once, then
// psi = J/2 sum + diag phi in binary64.
// the row sum of the integer H Phi: (re, im) 2^(r - 1075), r the group
// exponent of the largest term so far; a term T 2^(em - 1075) (|T| <= 2^53.5:
// a phase of modulus 2^52 times two components of at most 2^53, over 2^52) is
// rounded to nearest onto that grid, and a term of a coarser group first moves
// the sum to its grid.  ROW_TERMS of them stay below 2^62, which rshift_round
// needs and one more term keeps; rows of more terms are folded into binary64
// (RowAcc::fold) every ROW_TERMS.  The error of a fold is at most (terms +
// moves) / 2 units of its grid, i.e. about 2^-54 of the largest term each
// (binary64 accumulation: 2^-53 of each partial sum).
constexpr int ROW_TERMS = 256;
struct RowAcc {
    long long re = 0, im = 0;
    int r = -100000;
    __device__ __forceinline__ double2 value() const {
        return make_double2(i128_ldexp(re, r - 1075), i128_ldexp(im, r - 1075));
    }
    __device__ __forceinline__ void fold(double2 &sum) {
        const double2 v = value();
        sum.x += v.x;
        sum.y += v.y;
        re = im = 0;
        r = -100000;
    }
};
// x 2^-d rounded to nearest, 0 <= d <= 63, |x| < 2^62 (0 for d = 63)
__device__ __forceinline__ long long rshift_round(long long x, int d) {
    return (x + (long long)((1ull << d) >> 1)) >> d;
}
__device__ __forceinline__ void row_add(RowAcc &a, long long tr, long long ti, int em) {
    if (em > a.r) {
        const int d = min(em - a.r, 63);
        a.re = rshift_round(a.re, d);
        a.im = rshift_round(a.im, d);
        a.r = em;
    }
    const int d = min(a.r - em, 63);
    a.re += rshift_round(tr, d);
    a.im += rshift_round(ti, d);
}
// the term phase x phi on the digits: (pr + i pi)(fr + i fi), folded at
// weight 2^52 (rounded to nearest): units 2^(em - 1075) for phi on the grid
// of em and the phase on 2^-52
__device__ __forceinline__ void term_x(int4 p, int2 f1, int2 f0, long long &tr, long long &ti) {
    const long long hr = mad_w(p.x, f1.x, 0), hn = mad_w(p.z, f1.y, 0);
    const long long mr = mad_w(p.x, f0.x, mad_w(p.y, f1.x, 0));
    const long long mn = mad_w(p.z, f0.y, mad_w(p.w, f1.y, 0));
    const long long hi = mad_w(p.x, f1.y, mad_w(p.z, f1.x, 0));
    const long long mi = mad_w(p.x, f0.y, mad_w(p.y, f1.y, mad_w(p.z, f0.x, mad_w(p.w, f1.x, 0))));
    tr = (hr - hn) + ((mr - mn + (1ll << 25)) >> 26);
    ti = hi + ((mi + (1ll << 25)) >> 26);
}

template <int ND>
__global__ void __launch_bounds__(NTHREADS, 4) k_hphi_x(LatView L, const SecView *__restrict__ secs,
                                                       const int *__restrict__ tile0, int S, int ntiles,
                                                       HxVec hv, double2 *__restrict__ psi,
                                                       const int *__restrict__ active) {
    extern __shared__ __align__(16) unsigned char smem[];
    SmemLayout sm = carve(L, smem);
    stage_tables(L, sm.sC, sm.sxyz);
    double *snorm = (double *)sm.snorm;
    if (threadIdx.x < 9) {
        snorm[threadIdx.x] = sqrt((double)threadIdx.x);
        snorm[9 + threadIdx.x] = threadIdx.x ? 1.0 / sqrt((double)threadIdx.x) : 0.0;
    }
    hv.at_slot();
    const double juni = L.jh_uniform;
    __syncthreads();
    int4 *pd = (int4 *)sm.sph;          // the current sector's phases: (re.P1, re.P0, im.P1, im.P0) on 2^-52
    int cur = -1;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int s = (S == 1) ? 0 : sector_of_tile(tile0, S, t);
        if (active && !active[s]) continue;
        const SecView sv = secs[s];
        if (s != cur) {
            __syncthreads();
            for (int i = threadIdx.x; i < L.N; i += blockDim.x) {
                const double2 p = sv.ph64[i];
                int a1, a0, b1, b0;
                fx_digits((uint32_t)__double2hiint(p.x), (uint32_t)__double2loint(p.x), 1023, a1, a0);
                fx_digits((uint32_t)__double2hiint(p.y), (uint32_t)__double2loint(p.y), 1023, b1, b0);
                pd[i] = make_int4(a1, a0, b1, b0);
            }
            __syncthreads();
            cur = s;
        }
        const uint64_t row = (uint64_t)(t - sv.tile0) * TILE + threadIdx.x;
        if (row >= sv.dim) continue;
        const uint64_t rank = __ldg(sv.sigma + row);
        int c[ND];
        unrank(rank, sm.sC, L.np1, c);
        const double2 x0 = hv.value(sv.off + row);
        const int st_row = sv.stab[row];
        const double rs = snorm[9 + st_row];
        double e = L.c0, dd = 0.0;
        RowAcc acc;
        int nt = 0;
        double2 acc64 = make_double2(0.0, 0.0);
#pragma unroll 1
        for (int m = 0; m < ND; ++m) {
            const int i = pick(c, m);
            e += diag_u<double>(L, i);
            const int e0 = __ldg(L.adj_ptr + i), e1 = __ldg(L.adj_ptr + i + 1);
            // a hop to c_{m-1} < j < c_{m+1} keeps its place in the sorted list
            const int lo = m > 0 ? pick(c, m > 0 ? m - 1 : 0) : -1;
            const int hi = m < ND - 1 ? pick(c, m < ND - 1 ? m + 1 : m) : L.np1;
            const uint64_t base = rank - sm.sC[(m + 1) * L.np1 + i];
            for (int q = e0; q < e1; ++q) {
                const int j = __ldg(L.adj_nbr + q);
                const bool inpl = j > lo && j < hi;
                if (!inpl) {
                    bool occ = false;
#pragma unroll
                    for (int k = 0; k < ND; ++k) occ |= (c[k] == j);
                    if (occ) {
                        dd += diag_jz<double>(L, q);
                        continue;
                    }
                }
                uint64_t r2;
                if (inpl) {
                    r2 = base + sm.sC[(m + 1) * L.np1 + j];
                } else {
                    int tt[ND];
#pragma unroll
                    for (int k = 0; k < ND; ++k) tt[k] = (k == m) ? j : c[k];
                    sort_net(tt);
                    r2 = rank_of(tt, sm.sC, L.np1);
                }
                const uint32_t ee = __ldg(L.orb + r2);
                if ((ee >> 12) >= L.n_orb) continue;     // never for a complete table
                const int32_t row2 = __ldg(sv.t2 + (ee >> 12));
                if (row2 < 0) continue;
                const uint32_t idx = (uint32_t)row2;
                const int u = (int)(ee & 4095u);
                const int st = __ldg(sv.stab + idx);
                if (st == st_row) {
                    int2 f1, f0;
                    int em;
                    hd_unpack(__ldg(hv.hd + sv.off + idx), f1, f0, em);
                    long long tr, ti;
                    term_x(pd[u], f1, f0, tr, ti);
                    if (++nt > ROW_TERMS) {
                        acc.fold(acc64);
                        nt = 1;
                    }
                    row_add(acc, tr, ti, em);
                } else {
                    double2 p = sv.ph64[u];
                    const double f = snorm[st] * rs;
                    p.x *= f;
                    p.y *= f;
                    acc_add(acc64, p, hv.value(sv.off + idx));
                }
            }
        }
        double2 acch = acc.value();
        acch.x += acc64.x;
        acch.y += acc64.y;
        const double ed = e + 0.5 * dd;
        double2 out;
        out.x = fma(ed, x0.x, juni * acch.x);
        out.y = fma(ed, x0.y, juni * acch.y);
        psi[sv.off + row] = out;
    }
}

// The hops of the representative c (rank0 `rank`) of an orbit, in the order
// the row kernels visit them: targets g2 << 12 | u at my[h stride], their
// |Stab| at mys[h stride]; returns their number, and in e, dd the diagonal's
// site part and the J^z of its down-spin pairs (each met twice).
template <int ND, typename R>
__device__ __forceinline__ int orbit_hops(const LatView &L, uint32_t rank, const int (&c)[ND],
                                          const uint32_t *__restrict__ sC, const uint8_t *__restrict__ ostab,
                                          uint32_t *my, uint8_t *mys, size_t stride, R &e, R &dd) {
    e = diag_row<R>(L);
    dd = 0;
    int nh = 0, npair = 0;
#pragma unroll 1
    for (int m = 0; m < ND; ++m) {
        const int i = pick(c, m);
        if (!L.diag_uniform) e += diag_u<R>(L, i);
        const int e0 = __ldg(L.adj_ptr + i), e1 = __ldg(L.adj_ptr + i + 1);
        const int lo = m > 0 ? pick(c, m > 0 ? m - 1 : 0) : -1;
        const int hi = m < ND - 1 ? pick(c, m < ND - 1 ? m + 1 : m) : L.np1;
        const uint32_t base = rank - sC[(m + 1) * L.np1 + i];
        for (int q = e0; q < e1; ++q) {
            const int j = __ldg(L.adj_nbr + q);
            const bool inpl = j > lo && j < hi;
            if (!inpl) {
                bool occ = false;
#pragma unroll
                for (int k = 0; k < ND; ++k) occ |= (c[k] == j);
                if (occ) {
                    if (L.diag_uniform) ++npair;
                    else dd += diag_jz<R>(L, q);
                    continue;
                }
            }
            uint32_t r2;
            if (inpl) {
                r2 = base + sC[(m + 1) * L.np1 + j];
            } else {
                int tt[ND];
#pragma unroll
                for (int k = 0; k < ND; ++k) tt[k] = (k == m) ? j : c[k];
                sort_net(tt);
                r2 = rank_of32(tt, sC, L.np1);
            }
            const uint32_t ee = __ldg(L.orb + r2);
            if ((ee >> 12) >= L.n_orb) continue;                 // never for a complete table
            my[nh * stride] = ee;
            mys[nh * stride] = __ldg(ostab + (ee >> 12));
            ++nh;
        }
    }
    if (L.diag_uniform) dd = diag_pairs<R>(L, npair);
    return nh;
}

// H Phi batched over sectors (all momenta of one basis share the orbits and
// their hops; only the phases and the rows differ): one thread per (orbit g,
// group of osg sectors) unranks g's representative once, lists its hop
// targets (orbit, translation, |Stab|) and its diagonal once in shared
// memory (maxh entries per thread), then forms g's row in each sector of the
// group from them (osg from orb_group).
// A table has fewer than 2^32 states, so ranks and binomials (rows 0 .. N_down)
// are 32-bit words: 16 KB instead of 48 KB staged per block at N = 1000, and four
// resident blocks instead of three (10x10x10, N_down = 3, 28 sectors: integer 674
// -> 498 us, c128 720 -> 630, c64 406 -> 233, with the group rule's staging term).
constexpr int OSG = 8;

// the binary64 engine's product on the integer units: per term one row
// lookup, the digits of the target and its group exponent, the exact product
// with the sector's phase digits and the row sum, as in k_hphi_x (whose
// output it reproduces bit for bit: the terms come in the same order)
template <int ND>
__global__ void __launch_bounds__(NTHREADS, 4) k_hphi_o(LatView L, const SecView *__restrict__ secs, int S,
                                                   const uint64_t *__restrict__ oreps,
                                                   const uint8_t *__restrict__ ostab, uint32_t n_orb, int ngrp, int osg,
                                                   const int4 *__restrict__ phdig, HxVec hv,
                                                   double2 *__restrict__ psi, const int *__restrict__ active,
                                                   int maxh) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *sC = (uint32_t *)smem;                             // binomial rows 0 .. N_down
    double *snorm = (double *)(sC + (((ND + 1) * L.np1 + 1) & ~1));
    uint32_t *hl = (uint32_t *)(snorm + 18);                     // hop targets g2 << 12 | u
    uint8_t *hs = (uint8_t *)(hl + (size_t)maxh * blockDim.x);     // their |Stab|
    for (int i = threadIdx.x; i < (ND + 1) * L.np1; i += blockDim.x) sC[i] = (uint32_t)L.binom[i];
    if (threadIdx.x < 9) {
        snorm[threadIdx.x] = sqrt((double)threadIdx.x);
        snorm[9 + threadIdx.x] = threadIdx.x ? 1.0 / sqrt((double)threadIdx.x) : 0.0;
    }
    hv.at_slot();
    __syncthreads();
    const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= (uint64_t)n_orb * ngrp) return;
    const uint32_t g = (uint32_t)(tid % n_orb);
    const int grp = (int)(tid / n_orb);
    const int s_lo = grp * osg, s_hi = min(S, s_lo + osg);
    bool any = false;
    for (int s = s_lo; s < s_hi; ++s) any |= (!active || active[s]) && __ldg(secs[s].t2 + g) >= 0;
    if (!any) return;
    uint32_t *my = hl + threadIdx.x;                             // entry h at my[h * blockDim.x]
    uint8_t *mys = hs + threadIdx.x;
    const uint32_t rank = (uint32_t)__ldg(oreps + g);            // a table has fewer than 2^32 states
    int c[ND];
    unrank32(rank, sC, L.np1, c);
    const int st_row = __ldg(ostab + g);
    double e, dd;
    const int nh = orbit_hops<ND, double>(L, rank, c, sC, ostab, my, mys, blockDim.x, e, dd);
    const double ed = e + 0.5 * dd;
    const double juni = L.jh_uniform;
    for (int s = s_lo; s < s_hi; ++s) {
        if (active && !active[s]) continue;
        const int32_t *t2 = secs[s].t2;
        const int32_t row = __ldg(t2 + g);
        if (row < 0) continue;
        const uint64_t off = secs[s].off;
        const int4 *pds = phdig + (size_t)s * L.N;
        RowAcc acc;
        double2 acc64 = make_double2(0.0, 0.0);
        // four terms at a time: their row lookups, then their digit gathers,
        // are in flight together; the terms are added in list order
        for (int h0 = 0; h0 < nh; h0 += 4) {
            int us[4];                                           // u | |Stab| << 12
            int32_t r2[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const bool in = h0 + b < nh;
                const uint32_t ee = in ? my[(size_t)(h0 + b) * blockDim.x] : 0u;
                us[b] = (int)(ee & 4095u) | (in ? (int)mys[(size_t)(h0 + b) * blockDim.x] << 12 : 0);
                r2[b] = in ? __ldg(t2 + (ee >> 12)) : -1;
            }
            int4 q[4];
#pragma unroll
            for (int b = 0; b < 4; ++b)
                q[b] = r2[b] >= 0 && us[b] >> 12 == st_row ? __ldg(hv.hd + off + (uint32_t)r2[b]) : make_int4(0, 0, 0, 0);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                if (r2[b] < 0) continue;
                const int u = us[b] & 4095;
                if (us[b] >> 12 == st_row) {
                    int2 f1, f0;
                    int em;
                    hd_unpack(q[b], f1, f0, em);
                    long long tr, ti;
                    term_x(__ldg(pds + u), f1, f0, tr, ti);
                    row_add(acc, tr, ti, em);
                } else {
                    double2 p = secs[s].ph64[u];
                    const double f = snorm[us[b] >> 12] * snorm[9 + st_row];
                    p.x *= f;
                    p.y *= f;
                    acc_add(acc64, p, hv.value(off + (uint32_t)r2[b]));
                }
            }
        }
        double2 acch = acc.value();
        acch.x += acc64.x;
        acch.y += acc64.y;
        const double2 x0 = hv.value(off + (uint32_t)row);
        double2 out;
        out.x = fma(ed, x0.x, juni * acch.x);
        out.y = fma(ed, x0.y, juni * acch.y);
        psi[off + (uint32_t)row] = out;
    }
}

// the same batching in the vector's own arithmetic (complex128 / complex64
// FMAs; one hop amplitude on every bond): output identical bit for bit to
// k_hphi.  Bound by the four fp64 FMAs of a term in complex128; against
// k_hphi the hop list, the ranks, the site part of the diagonal and its
// occupied pairs (fp64 additions that any lane made the whole warp take) are
// paid once per group of sectors instead of per row.  10x10, N_down = 4, all
// 100 momenta: 510 us at four resident blocks (64 registers), 877 us at three,
// 525 at five, against 1099 us of k_hphi; the terms' 4 FMAs alone take 490 us
// of the fp64 pipe.
template <int ND, typename VT>
__global__ void __launch_bounds__(NTHREADS, 4) k_hphi_of(LatView L, const SecView *__restrict__ secs, int S,
                                                    const uint64_t *__restrict__ oreps,
                                                    const uint8_t *__restrict__ ostab, uint32_t n_orb, int ngrp,
                                                    int osg, const VT *__restrict__ phi, VT *__restrict__ psi,
                                                    const int *__restrict__ active, int maxh) {
    using R = typename VTr<VT>::R;
    using CT = typename VTr<VT>::C;
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *sC = (uint32_t *)smem;                             // binomial rows 0 .. N_down
    R *snorm = (R *)(sC + (((ND + 1) * L.np1 + 1) & ~1));         // 18 of R in the room of 18 doubles
    uint32_t *hl = (uint32_t *)((double *)snorm + 18);
    uint8_t *hs = (uint8_t *)(hl + (size_t)maxh * blockDim.x);
    for (int i = threadIdx.x; i < (ND + 1) * L.np1; i += blockDim.x) sC[i] = (uint32_t)L.binom[i];
    if (threadIdx.x < 9) {
        snorm[threadIdx.x] = (R)sqrt((double)threadIdx.x);
        snorm[9 + threadIdx.x] = threadIdx.x ? (R)(1.0 / sqrt((double)threadIdx.x)) : (R)0;
    }
    __syncthreads();
    const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= (uint64_t)n_orb * ngrp) return;
    const uint32_t g = (uint32_t)(tid % n_orb);
    const int s_lo = (int)(tid / n_orb) * osg, s_hi = min(S, s_lo + osg);
    bool any = false;
    for (int s = s_lo; s < s_hi; ++s) any |= (!active || active[s]) && __ldg(secs[s].t2 + g) >= 0;
    if (!any) return;
    uint32_t *my = hl + threadIdx.x;
    uint8_t *mys = hs + threadIdx.x;
    const uint32_t rank = (uint32_t)__ldg(oreps + g);            // a table has fewer than 2^32 states
    int c[ND];
    unrank32(rank, sC, L.np1, c);
    const int st_row = __ldg(ostab + g);
    const R rs = snorm[9 + st_row];
    R e, dd;
    const int nh = orbit_hops<ND, R>(L, rank, c, sC, ostab, my, mys, blockDim.x, e, dd);
    const R ed = e + (R)0.5 * dd, juni = (R)L.jh_uniform;
    for (int s = s_lo; s < s_hi; ++s) {
        if (active && !active[s]) continue;
        const int32_t *t2 = secs[s].t2;
        const int32_t row = __ldg(t2 + g);
        if (row < 0) continue;
        const VT *__restrict__ ph_in = phi + secs[s].off;
        const CT *__restrict__ ph = phase_table<CT>(secs[s]);
        CT acch;
        acch.x = 0; acch.y = 0;
        // four terms at a time: their row lookups, then their gathers, are in
        // flight together; the terms are added in list order
        for (int h0 = 0; h0 < nh; h0 += 4) {
            uint32_t ee[4];
            int32_t r2[4];
            VT v[4];
            CT p[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const bool in = h0 + b < nh;
                ee[b] = in ? my[(size_t)(h0 + b) * blockDim.x] : 0u;
                r2[b] = in ? __ldg(t2 + (ee[b] >> 12)) : -1;
            }
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if (r2[b] >= 0) {
                    v[b] = ph_in[r2[b]];
                    p[b] = ph[ee[b] & 4095u];
                }
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                if (r2[b] < 0) continue;
                const int st = mys[(size_t)(h0 + b) * blockDim.x];
                if (st != st_row) {
                    const R f = snorm[st] * rs;
                    p[b].x *= f;
                    p[b].y *= f;
                }
                acc_add(acch, p[b], v[b]);
            }
        }
        CT acc;
        acc.x = 0; acc.y = 0;
        madd_r(acc, juni, acch);
        madd_r(acc, ed, ph_in[row]);
        store(psi + secs[s].off + row, acc);
    }
}

// nnz count per sector: the diagonal plus every hop that lands on a member of the sector
template <int ND, bool KS>
__global__ void __launch_bounds__(NTHREADS) k_count(LatView L, const SecView *__restrict__ secs,
                                                    const int *__restrict__ tile0, int S, int ntiles,
                                                    unsigned long long *out) {
    extern __shared__ __align__(16) unsigned char smem[];
    SmemLayout sm = carve(L, smem);
    stage_tables(L, sm.sC, KS ? sm.sxyz : nullptr);
    __syncthreads();
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int s = (S == 1) ? 0 : sector_of_tile(tile0, S, t);
        const SecView sv = secs[s];
        const uint64_t row = (uint64_t)(t - sv.tile0) * TILE + threadIdx.x;
        unsigned long long cnt = 0;
        if (row < sv.dim) {
            const uint64_t rank = KS ? sv.sigma[row] : row;
            int c[ND];
            unrank(rank, sm.sC, L.np1, c);
            cnt = 1;
#pragma unroll
            for (int m = 0; m < ND; ++m) {
                const int i = c[m];
                for (int q = L.adj_ptr[i]; q < L.adj_ptr[i + 1]; ++q) {
                    const int j = L.adj_nbr[q];
                    bool occ = false;
#pragma unroll
                    for (int k = 0; k < ND; ++k) occ |= (c[k] == j);
                    if (occ) continue;
                    if constexpr (!KS) {
                        ++cnt;
                    } else {
                        int tt[ND];
#pragma unroll
                        for (int k = 0; k < ND; ++k) tt[k] = (k == m) ? j : c[k];
                        int rep[ND];
                        int ax, by, cz;
                        const uint64_t r2 = canon(tt, L, sm.sxyz, sm.sC, rep, ax, by, cz);
                        uint32_t idx;
                        if (sigma_find(sv, rep, sm.sC, L.np1, r2, idx)) ++cnt;
                    }
                }
            }
        }
        for (int o = 16; o; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(out + s, cnt);
    }
}

// N_down = 0: H is the constant c0 on the single vacuum state of each sector
template <typename VT>
__global__ void k_diag0(double c0, uint64_t n, const VT *__restrict__ phi, VT *__restrict__ psi) {
    using R = typename VTr<VT>::R;
    using CT = typename VTr<VT>::C;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        CT acc; acc.x = 0; acc.y = 0;
        madd_r(acc, (R)c0, phi[i]);
        store(psi + i, acc);
    }
}


template <typename VT> struct DtIdx;
template <> struct DtIdx<float> { static constexpr int v = QS3_F32; };
template <> struct DtIdx<double> { static constexpr int v = QS3_F64; };
template <> struct DtIdx<float2> { static constexpr int v = QS3_C64; };
template <> struct DtIdx<double2> { static constexpr int v = QS3_C128; };

template <typename VT, typename KF>
static int tune_grid(KF kern, Basis &B, int occ, cudaStream_t st, const VT *phi, VT *psi, const int *active,
                     int &best_bps, size_t smem = (size_t)-1) {
    if (smem == (size_t)-1) smem = B.smem_bytes;
    return tune_blocks(B, occ, st, best_bps, [&](int grid) {
        kern<<<grid, NTHREADS, smem, st>>>(B.lv, B.d_secs.as<SecView>(), B.tile0_d, B.S, B.ntiles, phi, psi,
                                           active);
    });
}

template <int ND, typename VT, bool KS, bool TB>
static int hphi_ndt(Basis &B, const void *phi, void *psi, cudaStream_t st, const int *active) {
    static std::atomic<unsigned long long> cache{0};
    int grid = 1, occ = 1;
    QS3_TRY(launch_rows(k_hphi<ND, VT, KS, TB>, B, B.smem_bytes, cache, &grid, &occ));
    if (B.ntiles == 0) return QS3_OK;
    int &bps = B.tune_hphi[DtIdx<VT>::v];
    if (bps == 0) {
        cudaStreamCaptureStatus cst = cudaStreamCaptureStatusNone;
        QS3_CUDA(cudaStreamIsCapturing(st, &cst));
        if (cst == cudaStreamCaptureStatusNone) {
            int b = occ;
            QS3_TRY(tune_grid(k_hphi<ND, VT, KS, TB>, B, occ, st, (const VT *)phi, (VT *)psi, active, b));
            bps = b;
        }
    }
    if (bps > 0) grid = std::max(1, std::min(B.ntiles, std::min(bps, occ) * num_sms()));
    k_hphi<ND, VT, KS, TB><<<grid, NTHREADS, B.smem_bytes, st>>>(B.lv, B.d_secs.as<SecView>(), B.tile0_d,
                                                                  B.S, B.ntiles, (const VT *)phi, (VT *)psi, active);
    QS3_LAUNCHED();
    return QS3_OK;
}

template <int ND, typename VT, bool KS>
static int hphi_nd(Basis &B, const void *phi, void *psi, cudaStream_t st, const int *active) {
    if constexpr (KS) {
        if (B.lv.orb) return hphi_ndt<ND, VT, true, true>(B, phi, psi, st, active);
    }
    return hphi_ndt<ND, VT, KS, false>(B, phi, psi, st, active);
}

template <typename VT, bool KS>
static int hphi_vt(Basis &B, const void *phi, void *psi, cudaStream_t st, const int *a) {
    switch (B.nd) {
        case 1: return hphi_nd<1, VT, KS>(B, phi, psi, st, a);
        case 2: return hphi_nd<2, VT, KS>(B, phi, psi, st, a);
        case 3: return hphi_nd<3, VT, KS>(B, phi, psi, st, a);
        case 4: return hphi_nd<4, VT, KS>(B, phi, psi, st, a);
        case 5: return hphi_nd<5, VT, KS>(B, phi, psi, st, a);
        case 6: return hphi_nd<6, VT, KS>(B, phi, psi, st, a);
        case 7: return hphi_nd<7, VT, KS>(B, phi, psi, st, a);
        case 8: return hphi_nd<8, VT, KS>(B, phi, psi, st, a);
        default: return set_err(QS3_ERR_INVALID_ARG, "n_down %d", B.nd);
    }
}

template <int ND>
static int hphix_nd(Basis &B, const HxVec &hv, double2 *psi, cudaStream_t st, const int *active) {
    static std::atomic<unsigned long long> cache{0};
    int grid = 1, occ = 1;
    QS3_TRY(launch_rows(k_hphi_x<ND>, B, B.smem_bytes, cache, &grid, &occ));
    if (B.ntiles == 0) return QS3_OK;
    auto launch = [&](int g) {
        k_hphi_x<ND><<<g, NTHREADS, B.smem_bytes, st>>>(B.lv, B.d_secs.as<SecView>(), B.tile0_d, B.S,
                                                         B.ntiles, hv, psi, active);
    };
    int &bps = B.tune_hphix;
    if (bps == 0) {
        cudaStreamCaptureStatus cst = cudaStreamCaptureStatusNone;
        QS3_CUDA(cudaStreamIsCapturing(st, &cst));
        if (cst == cudaStreamCaptureStatusNone && !hv.dx) {
            int b = occ;
            QS3_TRY(tune_blocks(B, occ, st, b, launch));
            bps = b;
        }
    }
    if (bps > 0) grid = std::max(1, std::min(B.ntiles, std::min(bps, occ) * num_sms()));
    launch(grid);
    QS3_LAUNCHED();
    return QS3_OK;
}

// sectors per thread of the orbit-batched kernels: the power of two g up to
// OSG that makes (waves of resident blocks + 1/2 for the last one) times
// (setting a thread up + g sectors) smallest.  Listing an orbit's hops costs
// about as much as one sector in fp32, half of one in binary64 and on the
// integer units, staging the binomials half of one per four loads a thread.
// 10x10, N_down = 4, 20 sectors, 1 / 2 / 4 per thread: c64 83 / 57 / 57 us,
// c128 146 / 128 / 135, integer 146 / 114 / 120; all 100, 4 / 8 per thread: c64
// 188 / 169, c128 507 / 519, integer 417 / 410; 10x10x10, N_down = 3 (16 loads a
// thread), 28 sectors, 2 / 4 / 8: c64 347 / 268 / 233, integer 594 / 520 / 491 (one run).
static int orb_group(const Basis &B, bool fp32) {
    const uint64_t wave = 4ull * NTHREADS * (uint64_t)num_sms();
    const int setup = (fp32 ? 2 : 1) + (B.nd + 1) * (B.N + 1) / (4 * NTHREADS);     // in half sectors
    uint64_t least = ~0ull;
    int best = 1;
    for (int g = 1; g <= OSG; g *= 2) {
        const uint64_t c = (2 * B.n_orb * (uint64_t)((B.S + g - 1) / g) + wave) * (uint64_t)(2 * g + setup);
        if (c < least) { least = c; best = g; }
    }
    return best;
}
// shared memory of the 32-bit binomials and the hop lists; 0: too many hops per row
static size_t orb_smem(const Basis &B) {
    const size_t maxh = (size_t)std::max(1, B.nd * B.max_degree);
    const size_t smem = (((size_t)(B.nd + 1) * (B.N + 1) + 1) & ~(size_t)1) * 4 + 18 * 8 + maxh * NTHREADS * 5;
    static_assert(MAX_DYN_SMEM / (NTHREADS * 5) < ROW_TERMS, "k_hphi_o sums a list without folds");
    return smem <= (size_t)MAX_DYN_SMEM ? smem : 0;
}

// what the orbit-batched kernels have of an SM: resident blocks, and the shared
// memory that those use in KB
struct OrbRoom {
    size_t blocks, used;
};
static OrbRoom orb_room(const Basis &B) {
    const size_t per = orb_smem(B) / 1024 + 2;                   // 1 KB of each block is the system's
    const size_t blocks = std::min<size_t>(4, 228 / per);
    return {blocks, blocks * per};
}
// rows that put one block on every SM
static uint64_t one_wave() { return NTHREADS * (uint64_t)num_sms(); }

template <int ND>
static int hphio_nd(Basis &B, const HxVec &hv, double2 *psi, cudaStream_t st, const int *active) {
    const int maxh = std::max(1, B.nd * B.max_degree);
    const size_t smem = orb_smem(B);
    static std::atomic<int> attr{0};
    if (attr.load(std::memory_order_acquire) == 0) {
        QS3_CUDA(cudaFuncSetAttribute(k_hphi_o<ND>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_DYN_SMEM));
        attr.store(1, std::memory_order_release);
    }
    const int osg = orb_group(B, false), ngrp = (B.S + osg - 1) / osg;
    const uint64_t nthr = B.n_orb * (uint64_t)ngrp;
    if (nthr == 0) return QS3_OK;
    const int grid = (int)((nthr + NTHREADS - 1) / NTHREADS);
    k_hphi_o<ND><<<grid, NTHREADS, smem, st>>>(B.lv, B.d_secs.as<SecView>(), B.S, B.d_oreps.as<uint64_t>(),
                                                B.d_ostab.as<uint8_t>(), (uint32_t)B.n_orb, ngrp, osg,
                                                B.d_phdig.as<int4>(), hv, psi, active, maxh);
    QS3_LAUNCHED();
    return QS3_OK;
}

// the orbit-batched FMA kernel serves bases with the representative table and
// one hop amplitude, of one sector too (c128 k_hphi / k_hphi_of: 10x10, N_down =
// 4 31 / 27 us a call, 12x12 53 / 37, 10x10x10, N_down = 3 71 / 54; c64 21 / 18, 23
// / 21, 44 / 38), as far as its hop lists leave room: k_hphi lists nothing and
// keeps its blocks and its L1 cache, unless its 64-bit tables are large too.  With
// three or four blocks resident that leave the L1 60 KB (complex64: 80 KB) the
// orbits are faster everywhere, but for complex64 with one sector to share a list
// over more than one wave.  Fewer blocks, or less L1, cost more than the sharing
// of few sectors gives, so the rows must fill the chip (one block on every SM) as
// many times as `waves` says, and the sectors be `share` at least.  Square
// lattices of degree 8 to 48, k_hphi / k_hphi_of in us, c128 and c64:
//   tables of 109 KB: 40x40, N_down = 3, 28 bonds a site (one block), one sector
//     1325 / 940 and 1185 / 753
//   four blocks, little L1: 10x10, N_down = 3, 14 bonds, one sector 41 / 41 and 27
//     / 31, 100 sectors 137 / 102 and 49 / 45; 14x14, 196 sectors 863 / 412 and 246
//     / 147
//   three or four blocks: 16x16, N_down = 4, one sector, 4 bonds 201 / 131 and 74 /
//     80, 12 bonds 547 / 379 and 203 / 253, two sectors 1086 / 580 and 371 / 337
//   two blocks: 10x10, N_down = 4, 20 bonds, 2 sectors 160 / 150 and 68 / 109, 16
//     832 / 565 and 309 / 293; 14x14, N_down = 3, 28 bonds, 4 sectors 76 / 90 and
//     51 / 65, 196 1671 / 1059 and 484 / 424; 16x16, N_down = 4, 16 bonds, 2 sectors
//     1439 / 920 and 500 / 533, 4 2785 / 1545 and 950 / 767
//   one block: 10x10, N_down = 4, 36 bonds, 4 sectors 437 / 509 and 210 / 297, 8
//     815 / 755 and 327 / 483, 100 8901 / 6480 and 2966 / 3111; 16x16, 24 bonds, one
//     sector 1070 / 1361 in c128
constexpr size_t HEAVY_TABLES = 64 * 1024;
static bool hphi_of_ok(const Basis &B, bool fp32) {
    if (!(B.has_k && B.lv.orb && B.d_oreps.p && B.lv.jh_uniform != 0.0) || !orb_smem(B)) return false;
    if (B.smem_bytes > HEAVY_TABLES) return true;
    const auto [blocks, used] = orb_room(B);
    uint64_t waves;
    int share = 1;
    if (blocks >= 3) {
        waves = fp32 ? (used > 196 ? 16 : used > 176 ? 4 : 0) : (used > 196 ? 1 : 0);
    } else if (blocks == 2) {
        waves = fp32 ? (used > 196 ? 24 : 16) : (used > 196 ? 4 : 0);
        share = fp32 ? 4 : 1;
    } else {
        if (fp32) return false;
        waves = 8;
        share = OSG;
    }
    if (fp32 && B.S == 1 && B.n_orb > blocks * one_wave()) return false;
    return B.S >= share && B.n_orb * (uint64_t)B.S >= waves * one_wave();
}

template <int ND, typename VT>
static int hphiof_nd(Basis &B, const void *phi, void *psi, cudaStream_t st, const int *active, int dt) {
    static std::atomic<unsigned long long> cache{0};
    const int maxh = std::max(1, B.nd * B.max_degree);
    const size_t smem = orb_smem(B);
    int grid = 1, occ = 1;
    QS3_TRY(launch_rows(k_hphi_of<ND, VT>, B, smem, cache, &grid, &occ));
    if (B.tune_hphi[dt] == 0) B.tune_hphi[dt] = occ;             // the grid covers all orbits: nothing to tune
    const int osg = orb_group(B, sizeof(VT) == 8), ngrp = (B.S + osg - 1) / osg;
    const uint64_t nthr = B.n_orb * (uint64_t)ngrp;
    if (nthr == 0) return QS3_OK;
    k_hphi_of<ND, VT><<<(int)((nthr + NTHREADS - 1) / NTHREADS), NTHREADS, smem, st>>>(
        B.lv, B.d_secs.as<SecView>(), B.S, B.d_oreps.as<uint64_t>(), B.d_ostab.as<uint8_t>(), (uint32_t)B.n_orb, ngrp,
        osg, (const VT *)phi, (VT *)psi, active, maxh);
    QS3_LAUNCHED();
    return QS3_OK;
}

template <typename VT>
static int hphiof_vt(Basis &B, const void *phi, void *psi, cudaStream_t st, const int *a, int dt) {
    switch (B.nd) {
        case 1: return hphiof_nd<1, VT>(B, phi, psi, st, a, dt);
        case 2: return hphiof_nd<2, VT>(B, phi, psi, st, a, dt);
        case 3: return hphiof_nd<3, VT>(B, phi, psi, st, a, dt);
        case 4: return hphiof_nd<4, VT>(B, phi, psi, st, a, dt);
        case 5: return hphiof_nd<5, VT>(B, phi, psi, st, a, dt);
        case 6: return hphiof_nd<6, VT>(B, phi, psi, st, a, dt);
        case 7: return hphiof_nd<7, VT>(B, phi, psi, st, a, dt);
        case 8: return hphiof_nd<8, VT>(B, phi, psi, st, a, dt);
        default: return set_err(QS3_ERR_INVALID_ARG, "n_down %d", B.nd);
    }
}

bool hphi_x_ok(const Basis &B) {
    return B.has_k && B.lv.orb && B.lv.jh_uniform != 0.0 && B.nd > 0 && !B.stored_terms && B.total > 0;
}

// the orbit-batched kernel, unless its hop lists do not fit.  One sector shares
// no lists: there k_hphi_o gains what unranking and the lookups in flight give,
// as long as four blocks are resident or the orbits are one wave of fewer, and
// the L1 keeps 60 KB; a last wave that is nearly empty, or fewer warps over
// several waves, cost more.  k_hphi_x / k_hphi_o in us a call: 4 bonds a site,
// 10x10, N_down = 4 37 / 33, 12x12 40 / 39, 10x10x10, N_down = 3 61 / 51; 12
// bonds (three blocks) 10x10 75 / 69, 12x12 86 / 108; 20 bonds (two) 116 / 115, 133
// / 191; 28 bonds (one) 161 / 190, 183 / 347, 8x8 130 / 121
static bool hphi_o_ok(const Basis &B) {
    if (!B.d_oreps.p || !orb_smem(B)) return false;
    if (B.S >= 2) return true;
    const auto [blocks, used] = orb_room(B);
    return used <= 196 && (blocks == 4 || B.n_orb <= blocks * one_wave());
}

int hphi_x_launch(Basis &B, const HxVec &hv, void *psi, cudaStream_t st, const int *active) {
    if (!hphi_x_ok(B)) return set_err(QS3_ERR_STATE, "the integer H Phi needs a k-sector basis with the "
                                                     "representative table and one hop amplitude");
    double2 *o = (double2 *)psi;
    if (hphi_o_ok(B)) {
        switch (B.nd) {
            case 1: return hphio_nd<1>(B, hv, o, st, active);
            case 2: return hphio_nd<2>(B, hv, o, st, active);
            case 3: return hphio_nd<3>(B, hv, o, st, active);
            case 4: return hphio_nd<4>(B, hv, o, st, active);
            case 5: return hphio_nd<5>(B, hv, o, st, active);
            case 6: return hphio_nd<6>(B, hv, o, st, active);
            case 7: return hphio_nd<7>(B, hv, o, st, active);
            case 8: return hphio_nd<8>(B, hv, o, st, active);
            default: return set_err(QS3_ERR_INVALID_ARG, "n_down %d", B.nd);
        }
    }
    switch (B.nd) {
        case 1: return hphix_nd<1>(B, hv, o, st, active);
        case 2: return hphix_nd<2>(B, hv, o, st, active);
        case 3: return hphix_nd<3>(B, hv, o, st, active);
        case 4: return hphix_nd<4>(B, hv, o, st, active);
        case 5: return hphix_nd<5>(B, hv, o, st, active);
        case 6: return hphix_nd<6>(B, hv, o, st, active);
        case 7: return hphix_nd<7>(B, hv, o, st, active);
        case 8: return hphix_nd<8>(B, hv, o, st, active);
        default: return set_err(QS3_ERR_INVALID_ARG, "n_down %d", B.nd);
    }
}

int hphi_launch(Basis &B, qs3_dtype dt, const void *phi, void *psi, cudaStream_t st, const int *active) {
    if (!phi || !psi) return set_err(QS3_ERR_INVALID_ARG, "NULL vector");
    if (phi == psi) return set_err(QS3_ERR_INVALID_ARG, "phi and psi alias");
    if (dt == QS3_C128DF) return hphi_df_launch(B, phi, nullptr, 0, psi, st, active);
    if (dt == QS3_C128X) return hphi_x_binary64(B, phi, psi, st);
    if (B.has_k && (dt == QS3_F32 || dt == QS3_F64))
        return set_err(QS3_ERR_STATE, "k-sector bases need complex vectors (C64/C128)");
    if (B.total == 0) return QS3_OK;
    if (B.nd == 0) {
        const int grid = (int)std::min<uint64_t>((B.total + 255) / 256, 1024);
        switch (dt) {
            case QS3_F32: k_diag0<float><<<grid, 256, 0, st>>>(B.lv.c0, B.total, (const float *)phi, (float *)psi); break;
            case QS3_F64: k_diag0<double><<<grid, 256, 0, st>>>(B.lv.c0, B.total, (const double *)phi, (double *)psi); break;
            case QS3_C64: k_diag0<float2><<<grid, 256, 0, st>>>(B.lv.c0, B.total, (const float2 *)phi, (float2 *)psi); break;
            case QS3_C128: k_diag0<double2><<<grid, 256, 0, st>>>(B.lv.c0, B.total, (const double2 *)phi, (double2 *)psi); break;
            default: return set_err(QS3_ERR_INVALID_ARG, "dtype %d", (int)dt);
        }
        QS3_LAUNCHED();
        return QS3_OK;
    }
    if (B.has_k) {
        if (B.stored_terms && (dt == QS3_C64 || dt == QS3_C128)) return hphi_stored_launch(B, dt, phi, psi, st, active);
        if (!B.lv.orb && B.d_orec.p && (dt == QS3_C64 || dt == QS3_C128))
            return hphi_forms_launch(B, dt, phi, psi, st, active);
        if ((dt == QS3_C64 || dt == QS3_C128) && hphi_of_ok(B, dt == QS3_C64)) {
            if (dt == QS3_C64) return hphiof_vt<float2>(B, phi, psi, st, active, dt);
            return hphiof_vt<double2>(B, phi, psi, st, active, dt);
        }
        if (dt == QS3_C64) return hphi_vt<float2, true>(B, phi, psi, st, active);
        if (dt == QS3_C128) return hphi_vt<double2, true>(B, phi, psi, st, active);
    } else {
        bool done = false;
        QS3_TRY(hphi_u1_launch(B, dt, phi, psi, st, active, &done));
        if (done) return QS3_OK;
        if (dt == QS3_F32) return hphi_vt<float, false>(B, phi, psi, st, active);
        if (dt == QS3_F64) return hphi_vt<double, false>(B, phi, psi, st, active);
        if (dt == QS3_C64) return hphi_vt<float2, false>(B, phi, psi, st, active);
        if (dt == QS3_C128) return hphi_vt<double2, false>(B, phi, psi, st, active);
    }
    return set_err(QS3_ERR_INVALID_ARG, "dtype %d", (int)dt);
}

template <int ND, bool KS>
static int count_nd(Basis &B, unsigned long long *d_out) {
    static std::atomic<unsigned long long> cache{0};
    int grid = 1;
    QS3_TRY(launch_rows(k_count<ND, KS>, B, B.smem_bytes, cache, &grid));
    k_count<ND, KS><<<grid, NTHREADS, B.smem_bytes>>>(B.lv, B.d_secs.as<SecView>(), B.tile0_d, B.S,
                                                       B.ntiles, d_out);
    QS3_LAUNCHED();
    return QS3_OK;
}

template <bool KS>
static int count_ks(Basis &B, unsigned long long *d_out) {
    switch (B.nd) {
        case 1: return count_nd<1, KS>(B, d_out);
        case 2: return count_nd<2, KS>(B, d_out);
        case 3: return count_nd<3, KS>(B, d_out);
        case 4: return count_nd<4, KS>(B, d_out);
        case 5: return count_nd<5, KS>(B, d_out);
        case 6: return count_nd<6, KS>(B, d_out);
        case 7: return count_nd<7, KS>(B, d_out);
        case 8: return count_nd<8, KS>(B, d_out);
        default: return set_err(QS3_ERR_INVALID_ARG, "n_down %d", B.nd);
    }
}

int count_nnz(Basis &B, uint64_t *nnz) {
    if (!B.nnz_valid) {
        B.nnz_sec.assign(B.S, 0);
        if (B.nd == 0 || B.total == 0) {
            for (int s = 0; s < B.S; ++s) B.nnz_sec[s] = B.dims[s];
        } else {
            DevBuf d;
            QS3_TRY(d.alloc(8 * (size_t)B.S));
            QS3_CUDA(cudaMemset(d.p, 0, 8 * (size_t)B.S));
            QS3_TRY(B.has_k ? count_ks<true>(B, d.as<unsigned long long>())
                            : count_ks<false>(B, d.as<unsigned long long>()));
            QS3_CUDA(cudaMemcpy(B.nnz_sec.data(), d.p, 8 * (size_t)B.S, cudaMemcpyDeviceToHost));
        }
        B.nnz = 0;
        for (uint64_t v : B.nnz_sec) B.nnz += v;
        B.nnz_valid = true;
    }
    *nnz = B.nnz;
    return QS3_OK;
}

}  // namespace qs3

extern "C" int qs3_hphi(qs3_basis_t b, qs3_dtype dtype, const void *phi, void *psi, void *stream) {
    qs3::clear_err();
    if (!b) return qs3::set_err(QS3_ERR_INVALID_ARG, "basis is NULL");
    return qs3::hphi_launch(b->B, dtype, phi, psi, (cudaStream_t)stream);
}
