// qs3_hphi_u1.cu -- the product psi = H phi of U(1)-only bases whose ranks
// fit 32 bits (C(N, N_down) < 2^32): Alg. 4 applied matrix-free, pull form,
// no atomics, real or complex vectors in fp32 or fp64.
//
// k_hphi_u1s, the kernel of long segments.  The rows that share their upper
// spins U = (c_2 < ... < c_Nd) are consecutive: rank0 = B(U) + c_1 with
// B(U) = sum_{m >= 2} C(c_m, m) and c_1 = 0 .. c_2 - 1.  A warp takes runs of
// such segments.  What depends on U alone is formed once per segment, one
// lane per hop of an upper spin c_m -> j: whether j is occupied (then J^z
// goes to the segment's diagonal), else the ranks of its targets.  With
// U' = U - c_m + j the target of the row c_1 is B(U') + c_1 for c_1 < j, a
// load at consecutive addresses across the warp; a row with c_1 = j cannot
// take the hop (the pair adds its J^z), and for c_1 > j, where j becomes the
// lowest site, the target is B(U') - C(j, 2) + j + C(c_1, 2).  A hop of c_1
// itself to j < c_2 stays in the segment.  So no row is unranked and no
// target rank is formed per row except where c_1 hops past c_2.
//
// k_hphi_u1n, the kernel of short segments: one thread per row, 32-bit
// unranking, the hop of c_m to j in place when c_{m-1} < j < c_{m+1} (one
// table read), else re-sorted; the neighbour and the amplitude come in one
// load.  In fp64 it takes 1068 us on the open 24x24 lattice, N_down = 3
// (31,628,736 rows), where the general row kernel with its 64-bit ranks and
// rolled adjacency took 1272; the hops' FMAs and the diagonal are 18 fp64
// operations per row, 1083 us at the measured rate of the pipe.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "qs3_hphi_common.cuh"

namespace qs3 {

// what these kernels read of the lattice (LatView is four times as large, and
// the smallest products are bound by their launch)
struct U1View {
    int N, np1;
    const uint64_t *binom;
    double c0;
    float c0f;
    const double *u;
    const float *u_f;
    const int2 *adj_pad, *adjt;
    const int4 *adj_pad64;
    const float *adj_jz_pad, *adjt_jz;
    const double *adj_jz_pad64;
};
static U1View u1_view(const LatView &L) {
    return {L.N, L.np1, L.binom, L.c0, L.c0f, L.u, L.u_f, L.adj_pad, L.adjt, L.adj_pad64, L.adj_jz_pad, L.adjt_jz, L.adj_jz_pad64};
}
template <typename R> __device__ __forceinline__ R diag_c0(const U1View &L);
template <> __device__ __forceinline__ double diag_c0<double>(const U1View &L) { return L.c0; }
template <> __device__ __forceinline__ float diag_c0<float>(const U1View &L) { return L.c0f; }
template <typename R> __device__ __forceinline__ R diag_u(const U1View &L, int i);
template <> __device__ __forceinline__ double diag_u<double>(const U1View &L, int i) { return __ldg(L.u + i); }
template <> __device__ __forceinline__ float diag_u<float>(const U1View &L, int i) { return __ldg(L.u_f + i); }

// entry b of site i's fixed-width adjacency (one load): the neighbour and the
// hop amplitude, padded with the site itself and amplitude 0
template <typename R> struct Nbr {
    int j;
    R cf;
};
__device__ __forceinline__ Nbr<float> nbr_at(const int2 *__restrict__ t, int at) {
    const int2 v = __ldg(t + at);
    return {v.x, __int_as_float(v.y)};
}
__device__ __forceinline__ Nbr<double> nbr_at(const int4 *__restrict__ t, int at) {
    const int4 v = __ldg(t + at);
    return {v.x, __hiloint2double(v.w, v.z)};
}
__device__ __forceinline__ const int2 *pad_table(const U1View &L, float) { return L.adj_pad; }
__device__ __forceinline__ const int4 *pad_table(const U1View &L, double) { return L.adj_pad64; }
__device__ __forceinline__ float pad_jz(const U1View &L, int at, float) { return __ldg(L.adj_jz_pad + at); }
__device__ __forceinline__ double pad_jz(const U1View &L, int at, double) { return __ldg(L.adj_jz_pad64 + at); }

// one hop of an upper spin of a segment: the rank of the target of c_1 = 0
// (B(U')), the site j, the hop amplitude and J^z
struct SegHop {
    uint32_t base;
    int j;
    float cf, jz;
};

constexpr int SEG_WARPS = NTHREADS / 32;
constexpr int SEG_RUN = 4;                 // consecutive segments per run of a warp
// k_hphi_u1s serves real fp32 vectors of N_down = 3 (more spins with such segments
// exceed 32-bit ranks; with N_down = 2 they are few: N = 1024 81 us, k_hphi_u1n 17)
// on lattices of up to four neighbours, where the segments are long and few
// hops of c_1 leave them: a lane whose hop passes c_2 sends its whole pass the
// slow way.  N >= SEG_N (four neighbours: SEG_N_4) where every bond is at most N
// / SEG_REACH sites long, or, with one longer bond, the closing one of a ring, N
// >= SEG_N_RING.  k_hphi_u1n / k_hphi_u1s in us:
//   rings 483 172 / 212, 600 321 / 325, 700 500 / 451, 1000 1550 / 1204, 1600 6680 /
//   4377; open chains 483 170 / 156, 1000 1539 / 1019; open L x L 22 (bonds of N /
//   22) 246 / 270, 23 315 / 324, 24 401 / 399, 28 1006 / 971, 32 2233 / 2106, 40 9025 /
//   8232; open 8 x 64 281 / 270, 2 x 300 435 / 336; bonds of N / 8 (open 128 x 8) 2528 /
//   2799; periodic 32 x 32 2293 / 2676, 3 x 200 446 / 466; six neighbours, open
//   10x10x10 3046 / 3532; complex64, open 32 x 32 3295 / 3817 and ring 1000 1503 / 1870
// Four resident blocks (open 32 x 32, 3: 2269, 5: 2237), runs of four segments (1:
// 2208, 8: 2368).  fp64 stays with k_hphi_u1n: the fp64 pipe bounds both (1176 / 1068
// us at L = 24).
constexpr int SEG_N = 483, SEG_N_4 = 512, SEG_N_RING = 700;      // SEG_REACH: qs3_internal.cuh
static bool segments_pay(const Basis &B) {
    if (B.nd != 3 || B.lv.pad_w > 4) return false;
    if (B.n_long_bonds) return B.n_long_bonds == 1 && B.N >= SEG_N_RING;
    return B.N >= (B.lv.pad_w == 2 ? SEG_N : SEG_N_4);
}
constexpr int SEG_ROWS = 4;                // rows per lane and pass

// a segment as its rows see it
template <int ND> struct Seg {
    int U[ND - 1], dC[ND - 1];             // c_2 .. c_Nd; what the rank gains when U[k] moves one place down
    uint32_t base;                         // B(U)
    float e;                               // the diagonal's part of the upper spins
    int nhi, nh;                           // hops: [0, nhi) to j >= c_2, [nhi, nh) below
};

// the rows c_1 = x + lane + 32 r of a segment (FULL: all of them exist)
template <int ND, int DEG, int RL, bool FULL>
__device__ __forceinline__ void seg_rows(const U1View &L, const uint32_t *sC, const SegHop *hop,
                                         const Seg<ND> &sg, int x, int lane,
                                         const float *__restrict__ phi, float *__restrict__ psi) {
    using VT = float;
    using R = float;
    using CT = typename VTr<VT>::C;
    constexpr int NU = ND - 1;
    const int np1 = L.np1, N = L.N, len = sg.U[0];
    const int c0 = x + lane;
    const VT *__restrict__ own = phi + sg.base;
    CT acc[RL];
    R er[RL];
    bool in[RL];
    Nbr<R> n1[DEG][RL];
    int far = -1;
#pragma unroll
    for (int r = 0; r < RL; ++r) {
        acc[r].x = 0;
        acc[r].y = 0;
        in[r] = FULL || c0 + 32 * r < len;
#pragma unroll
        for (int b = 0; b < DEG; ++b) {
            n1[b][r].j = -1;
            n1[b][r].cf = 0;
            if (in[r]) n1[b][r] = nbr_at(L.adjt, b * N + c0 + 32 * r);
        }
        er[r] = in[r] ? sg.e + diag_u<R>(L, c0 + 32 * r) : (R)0;
    }
    // hops of the upper spins above every c_1: consecutive addresses
#pragma unroll 4
    for (int q = 0; q < sg.nhi; ++q) {
        const VT *__restrict__ p = phi + (hop[q].base + (uint32_t)c0);
        const R cf = hop[q].cf;
#pragma unroll
        for (int r = 0; r < RL; ++r)
            if (in[r]) madd_r(acc[r], cf, p[32 * r]);
    }
    // hops of c_1
#pragma unroll
    for (int b = 0; b < DEG; ++b)
#pragma unroll
        for (int r = 0; r < RL; ++r) far = max(far, n1[b][r].j);
    if (__any_sync(0xffffffffu, far >= len)) {
        // some hop passes c_2 (an occupied j is counted from the upper spin's side)
#pragma unroll
        for (int b = 0; b < DEG; ++b)
#pragma unroll
            for (int r = 0; r < RL; ++r) {
                const int j = n1[b][r].j;
                uint32_t at = sg.base + (uint32_t)j;
                bool ok = in[r] && j >= 0;
                if (ok && j >= len) {
                    at = sg.base;
                    int p = 1;
#pragma unroll
                    for (int k = 0; k < NU; ++k) {
                        ok &= sg.U[k] != j;
                        if (sg.U[k] < j) {
                            at += (uint32_t)sg.dC[k];
                            ++p;
                        }
                    }
                    if (ok) at += sC[p * np1 + j];
                }
                if (ok) madd_r(acc[r], n1[b][r].cf, phi[at]);
            }
    } else {
#pragma unroll
        for (int b = 0; b < DEG; ++b)
#pragma unroll
            for (int r = 0; r < RL; ++r)
                if (FULL || in[r]) madd_r(acc[r], n1[b][r].cf, own[n1[b][r].j]);
    }
    // hops of the upper spins to j < c_2
    for (int q = sg.nhi; q < sg.nh; ++q) {
        const SegHop h = hop[q];
        if (h.j >= x + 32 * RL) {
            const VT *__restrict__ p = phi + (h.base + (uint32_t)c0);
#pragma unroll
            for (int r = 0; r < RL; ++r)
                if (in[r]) madd_r(acc[r], h.cf, p[32 * r]);
        } else {
            const uint32_t b1 = h.base - sC[2 * np1 + h.j] + (uint32_t)h.j;
#pragma unroll
            for (int r = 0; r < RL; ++r) {
                const int c = c0 + 32 * r;
                if (in[r]) {
                    if (c == h.j) er[r] += h.jz;
                    else madd_r(acc[r], h.cf, phi[c < h.j ? h.base + (uint32_t)c : b1 + sC[2 * np1 + c]]);
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < RL; ++r)
        if (in[r]) {
            madd_r(acc[r], er[r], own[c0 + 32 * r]);
            store(psi + sg.base + c0 + 32 * r, acc[r]);
        }
}

template <int ND, int DEG>
__global__ void __launch_bounds__(NTHREADS, 4) k_hphi_u1s(U1View L, uint32_t nseg, const float *__restrict__ phi,
                                                          float *__restrict__ psi, const int *__restrict__ active) {
    using R = float;
    constexpr int NU = ND - 1, H = NU * DEG, RL = SEG_ROWS;
    static_assert(H <= 32, "one lane per hop of the upper spins");
    extern __shared__ __align__(16) unsigned char smem[];
    if (active && !active[0]) return;
    const int np1 = L.np1, N = L.N;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // this warp's hop list, then the binomial rows 0 .. N_down
    SegHop *hop = (SegHop *)smem + (size_t)warp * H;
    uint32_t *sC = (uint32_t *)((SegHop *)smem + (size_t)SEG_WARPS * H);
    for (int i = threadIdx.x; i < (ND + 1) * np1; i += blockDim.x) sC[i] = (uint32_t)L.binom[i];
    __syncthreads();
    const int hm = lane / DEG, hb = lane - hm * DEG;
    const uint32_t nrun = (nseg + SEG_RUN - 1) / SEG_RUN;
    for (uint32_t run = blockIdx.x * SEG_WARPS + warp; run < nrun; run += gridDim.x * SEG_WARPS) {
        Seg<ND> sg;
        unrank32(run * SEG_RUN, sC, np1, sg.U);
        const uint32_t s1 = min(nseg, (run + 1) * SEG_RUN);
        for (uint32_t s = run * SEG_RUN;;) {
            const int len = sg.U[0];
            sg.base = 0;
            sg.e = diag_c0<R>(L);
#pragma unroll
            for (int k = 0; k < NU; ++k) {
                const uint32_t hi = sC[(k + 2) * np1 + sg.U[k]];
                sg.base += hi;
                sg.dC[k] = (int)(sC[(k + 1) * np1 + sg.U[k]] - hi);
                sg.e += diag_u<R>(L, sg.U[k]);
            }
            // the hops of the upper spins, one per lane: those to j >= c_2, then the others
            int j = -1;
            R dz = 0;
            SegHop h;
            if (lane < H) {
                const int i = pick(sg.U, hm), at = hb * N + i;
                const Nbr<float> nb = nbr_at(L.adjt, at);
                j = nb.j == i ? -1 : nb.j;
                if (j >= 0) {
                    h.cf = nb.cf;
                    h.jz = __ldg(L.adjt_jz + at);
                    bool occ = false;
                    int u[NU];
#pragma unroll
                    for (int k = 0; k < NU; ++k) {
                        occ |= sg.U[k] == j;
                        u[k] = (k == hm) ? j : sg.U[k];
                    }
                    sort_net(u);
                    h.base = 0;
#pragma unroll
                    for (int k = 0; k < NU; ++k) h.base += sC[(k + 2) * np1 + u[k]];
                    h.j = j;
                    if (occ) {
                        dz = h.jz;
                        j = -1;
                    }
                }
            }
            const unsigned hi = __ballot_sync(0xffffffffu, j >= len), lt = (1u << lane) - 1u;
            const unsigned lo = __ballot_sync(0xffffffffu, j >= 0 && j < len);
            sg.nhi = __popc(hi);
            sg.nh = sg.nhi + __popc(lo);
            __syncwarp();
            if (j >= 0) hop[j >= len ? __popc(hi & lt) : sg.nhi + __popc(lo & lt)] = h;
            if (__any_sync(0xffffffffu, dz != (R)0)) {
                // each pair of upper neighbours was met from both ends
#pragma unroll
                for (int o = 16; o; o >>= 1) dz += __shfl_xor_sync(0xffffffffu, dz, o);
                sg.e += (R)0.5 * dz;
            }
            __syncwarp();
            int x = 0;
            for (; x + 32 * RL <= len; x += 32 * RL) seg_rows<ND, DEG, RL, true>(L, sC, hop, sg, x, lane, phi, psi);
            for (; x < len; x += 32) seg_rows<ND, DEG, 1, false>(L, sC, hop, sg, x, lane, phi, psi);
            if (++s >= s1) break;
            // the next list of upper spins
            bool carry = true;
#pragma unroll
            for (int k = 0; k < NU; ++k) {
                if (carry) {
                    if (k + 1 < NU && sg.U[k] + 1 == sg.U[k + 1 < NU ? k + 1 : k]) {
                        sg.U[k] = k;
                    } else {
                        ++sg.U[k];
                        carry = false;
                    }
                }
            }
        }
    }
}

template <int ND, typename VT, int DEGB>
__global__ void __launch_bounds__(NTHREADS, sizeof(typename VTr<VT>::R) == 8 || DEGB > 4 ? 4 : 6) k_hphi_u1n(U1View L, uint32_t dim,
                                                                         const VT *__restrict__ phi,
                                                                         VT *__restrict__ psi,
                                                                         const int *__restrict__ active) {
    using R = typename VTr<VT>::R;
    using CT = typename VTr<VT>::C;
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *sC = (uint32_t *)smem;
    const int np1 = L.np1;
    for (int i = threadIdx.x; i < (ND + 1) * np1; i += blockDim.x) sC[i] = (uint32_t)L.binom[i];
    __syncthreads();
    if (active && !active[0]) return;
    const auto *__restrict__ tab = pad_table(L, (R)0);
    for (uint64_t rw = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; rw < dim; rw += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t row = (uint32_t)rw;
        int c[ND];
        unrank32(row, sC, np1, c);
        const VT x0 = phi[row];
        R e = diag_c0<R>(L), dd = 0;
        CT acc;
        acc.x = 0; acc.y = 0;
#pragma unroll
        for (int m = 0; m < ND; ++m) {
            const int i = c[m];
            e += diag_u<R>(L, i);
            const int lo = m > 0 ? c[m > 0 ? m - 1 : 0] : -1;
            const int hi = m < ND - 1 ? c[m < ND - 1 ? m + 1 : m] : np1;
            const uint32_t *col = sC + (m + 1) * np1;
            const uint32_t base = row - col[i];
            uint32_t r2b[DEGB];
            R cfb[DEGB];
            bool ok[DEGB];
#pragma unroll
            for (int b = 0; b < DEGB; ++b) {
                const Nbr<R> nb = nbr_at(tab, i * DEGB + b);
                const int j = nb.j;
                r2b[b] = base + col[j];
                cfb[b] = nb.cf;
                // fp64: a padded entry (j = c_m) adds nothing, not 0 times phi
                ok[b] = sizeof(R) == 4 || j != i;
                if (!(j > lo && j < hi)) {
                    // occupied, or passing another down spin
                    bool occ = false;
#pragma unroll
                    for (int k = 0; k < ND; ++k) occ |= (c[k] == j);
                    if (occ) {
                        dd += pad_jz(L, i * DEGB + b, (R)0);
                        cfb[b] = 0;
                        ok[b] = sizeof(R) == 4;
                        r2b[b] = row;
                    } else {
                        int tt[ND];
#pragma unroll
                        for (int k = 0; k < ND; ++k) tt[k] = (k == m) ? j : c[k];
                        sort_net(tt);
                        r2b[b] = rank_of32(tt, sC, np1);
                    }
                }
            }
            VT vb[DEGB];
#pragma unroll
            for (int b = 0; b < DEGB; ++b) vb[b] = phi[r2b[b]];
#pragma unroll
            for (int b = 0; b < DEGB; ++b)
                if (ok[b]) madd_r(acc, cfb[b], vb[b]);
        }
        madd_r(acc, e + (R)0.5 * dd, x0);
        store(psi + row, acc);
    }
}

// k_hphi_u1n in fp64: the rank and the load of every padded entry, and in
// complex128 at N_down = 4 the registers of four spins' hops, cost what its 32-bit
// ranks gain over the general kernel unless most entries are real.  General kernel
// / k_hphi_u1n in us, fp64 and complex128 of N_down = 3: open 32 x 32 8968 / 5889 and
// 12043 / 10440, ring 1000 4898 / 3493 and 6200 / 5735; five sixths real (open 6x6x6)
// 96 / 95 and 143 / 148; three quarters (open 2 x 300) 1159 / 1132 and 1748 / 1983,
// (honeycomb of 288 sites) 139 / 149 and 205 / 207.  N_down = 4: open 12 x 12 783 /
// 771 and 1204 / 1287, ring 150 592 / 577 and 874 / 914, open 4x4x4 (three quarters) 51
// / 53 and 72 / 80
static bool fp64_rows_pay(const Basis &B, bool cplx) {
    return (!cplx || B.nd <= 3) && 2.0 * B.nb >= (cplx ? 0.85 : 0.8) * (double)B.N * B.lv.pad_w;
}

// the persistent launch of kern (grid in blocks, at most `blocks`): every
// resident block in fp32, four per SM in fp64, or as many as qs3_basis_tuning
// imposed.  fp64, open lattices, blocks per SM 3 / 4 / 5 / 6: L = 16 110 / 108 /
// 113 / 111 us, L = 24 1101 / 1070 / 1138 / 1184, L = 12 with N_down = 4 796 / 774
// / 819 / 853 (warps beyond those that keep the fp64 pipe busy only evict each
// other's lines); fp32 is best at the most blocks everywhere.  So no trial
// launches: twelve of them made the first product on a basis 15 times a later
// one.
template <typename KF, typename VT>
static int u1_run(KF kern, Basis &B, size_t smem, uint64_t blocks, uint32_t n, const VT *phi, VT *psi, cudaStream_t st,
                  const int *active, int dt, std::atomic<unsigned long long> &cache) {
    int grid = 1, occ = 1;
    QS3_TRY(launch_rows(kern, B, smem, cache, &grid, &occ));
    auto launch = [&](int g) {
        kern<<<std::max(1, (int)std::min<uint64_t>(blocks, (uint64_t)g)), NTHREADS, smem, st>>>(u1_view(B.lv), n, phi, psi,
                                                                                              active);
    };
    int &bps = B.tune_hphi[dt];
    if (bps == 0) bps = sizeof(typename VTr<VT>::R) == 8 ? std::min(occ, 4) : occ;
    launch((bps > 0 ? std::min(bps, occ) : occ) * num_sms());
    QS3_LAUNCHED();
    return QS3_OK;
}

template <int ND, typename VT>
static int u1_nd(Basis &B, const void *phi, void *psi, cudaStream_t st, const int *active, int dt, bool *done) {
    const int N = B.N;
    const VT *p = (const VT *)phi;
    VT *q = (VT *)psi;
    const size_t tab = (size_t)(ND + 1) * (N + 1) * sizeof(uint32_t);
    if constexpr (ND == 3 && std::is_same_v<VT, float>) {
        const int dw = B.lv.pad_w;
        const size_t smem = tab + (size_t)SEG_WARPS * (ND - 1) * dw * sizeof(SegHop);
        if (segments_pay(B) && smem <= (size_t)MAX_DYN_SMEM) {
            const uint64_t nseg = (uint64_t)N * (N - 1) / 2;                 // C(N, N_down - 1)
            const uint64_t blocks = (nseg + SEG_WARPS * SEG_RUN - 1) / (SEG_WARPS * SEG_RUN);
            *done = true;
            static std::atomic<unsigned long long> s2{0}, s4{0};
            if (dw == 2) return u1_run(k_hphi_u1s<ND, 2>, B, smem, blocks, (uint32_t)nseg, p, q, st, active, dt, s2);
            return u1_run(k_hphi_u1s<ND, 4>, B, smem, blocks, (uint32_t)nseg, p, q, st, active, dt, s4);
        }
    }
    if constexpr (sizeof(typename VTr<VT>::R) == 8)
        if (!fp64_rows_pay(B, std::is_same_v<VT, double2>)) return QS3_OK;
    if constexpr (ND <= 4) {
        const uint64_t blocks = (B.total + NTHREADS - 1) / NTHREADS;
        *done = true;
        static std::atomic<unsigned long long> c2{0}, c4{0}, c6{0};
        if (B.lv.pad_w == 2) return u1_run(k_hphi_u1n<ND, VT, 2>, B, tab, blocks, (uint32_t)B.total, p, q, st, active, dt, c2);
        if (B.lv.pad_w == 4) return u1_run(k_hphi_u1n<ND, VT, 4>, B, tab, blocks, (uint32_t)B.total, p, q, st, active, dt, c4);
        return u1_run(k_hphi_u1n<ND, VT, 6>, B, tab, blocks, (uint32_t)B.total, p, q, st, active, dt, c6);
    }
    return QS3_OK;
}

template <typename VT>
static int u1_vt(Basis &B, const void *phi, void *psi, cudaStream_t st, const int *a, int dt, bool *done) {
    switch (B.nd) {
        case 1: return u1_nd<1, VT>(B, phi, psi, st, a, dt, done);
        case 2: return u1_nd<2, VT>(B, phi, psi, st, a, dt, done);
        case 3: return u1_nd<3, VT>(B, phi, psi, st, a, dt, done);
        case 4: return u1_nd<4, VT>(B, phi, psi, st, a, dt, done);
        default: return QS3_OK;
    }
}

int hphi_u1_launch(Basis &B, qs3_dtype dt, const void *phi, void *psi, cudaStream_t st, const int *active, bool *done) {
    *done = false;
    if (!B.narrow_ranks || !B.lv.pad_w || B.total == 0) return QS3_OK;
    switch (dt) {
        case QS3_F32: return u1_vt<float>(B, phi, psi, st, active, dt, done);
        case QS3_F64: return u1_vt<double>(B, phi, psi, st, active, dt, done);
        case QS3_C64: return u1_vt<float2>(B, phi, psi, st, active, dt, done);
        case QS3_C128: return u1_vt<double2>(B, phi, psi, st, active, dt, done);
        default: return QS3_OK;
    }
}

}  // namespace qs3
