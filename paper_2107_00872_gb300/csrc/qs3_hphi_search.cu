// qs3_hphi_search.cu -- psi = H phi on momentum sectors without a
// representative table (lattices whose C(N, N_down) states do not fit one),
// complex64 / complex128, by origin forms.
//
// The representative of Alg. 7 is the minimum of a state over all
// translations; finding it for every hop target is a search whose ties every
// lane of a warp pays for (about 1900 instructions per warp and hop on the
// 6x6x6 cube, 18.8 ms for 17,313,563 rows).  But a hop does not need the
// representative itself, only the row and the translation, and any invariant
// of the orbit finds them.  The origin form of a state is the smallest of its
// N_down translates that move one of its spins to site 0, written as the
// sorted list of the other spins (packed, the largest site highest): N_down
// candidates, no ties to follow, and for a hop c_m -> j the candidate of a
// spin c_k, k != m, is the sorted list of the unmoved spins' differences to
// c_k, formed once per row and m, with one more difference inserted.
//
// The rows' origin forms are sorted once per basis: orec[i] = (packed form,
// row, w | (|Stab| - 1) << 28) with w the cell of the representative's spin
// that the form has at the origin.  A form is found through its largest site
// (finfo, staged in shared memory) and the rank of its other sites, which give
// a bucket of about one record.  With origin o of the target's form (the spin
// moved there), T_u rep = target for u = o - w.  So a hop costs three
// dependent loads, each a sector per lane: bucket, record, phi.
// 6x6x6, N_down = 5, k = 0, complex128: 12.0 ms (18.8 with the search on
// occupation masks; 13.2 with two-site prefixes, separate key and value lists
// and the diagonal's fp64 additions per row); 8x8x8, N_down = 4, complex64:
// 1.81 ms (3.45, 2.06).  About 480 instructions per warp and hop, half of the
// issue slots; the loads' latency at 45 % occupancy is the rest.  At its bound of 64
// registers the complex128 kernel spills (N_down = 5: 184 bytes stored and 260
// loaded a thread, N_down = 4 116 / 136), the complex64 one from N_down = 6 on.
#include <cub/cub.cuh>

#include <algorithm>
#include <atomic>

#include "qs3_hphi_common.cuh"

namespace qs3 {

// coordinates x, y, z of a cell in one word (LatView::xyz)
__device__ __forceinline__ int px(uint32_t p) { return (int)(p & 2047u); }
__device__ __forceinline__ int py(uint32_t p) { return (int)((p >> 11) & 2047u); }
__device__ __forceinline__ int pz(uint32_t p) { return (int)(p >> 22); }
__device__ __forceinline__ int wrap(int d, int L) { return d + ((d >> 31) & L); }

// the site of the difference a - b
__device__ __forceinline__ int site_diff(int ax, int ay, int az, int bx, int by, int bz, int Lx, int Ly, int Lz) {
    return wrap(ax - bx, Lx) + Lx * (wrap(ay - by, Ly) + Ly * wrap(az - bz, Lz));
}
// the packed key of an ascending list (base = 2^bits per site)
template <int M, typename KT>
__device__ __forceinline__ KT pack_list(const int (&l)[M], KT base) {
    KT k = (KT)l[M - 1];
#pragma unroll
    for (int i = M - 2; i >= 0; --i) k = k * base + (KT)l[i];
    return k;
}
template <int M, typename KT>
__device__ __forceinline__ void unpack_list(KT k, int bits, int (&l)[M]) {
    const uint32_t mask = (1u << bits) - 1u;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        l[i] = (int)((uint32_t)k & mask);
        k >>= bits;
    }
}

// the origin form of the list c: key, and the spin (its coordinates) at the origin
template <int ND, typename KT>
__device__ __forceinline__ KT origin_form(const int (&c)[ND], const LatView &L, const uint32_t *__restrict__ sxyz,
                                          KT base, uint32_t &at) {
    const int Lx = L.L[0], Ly = L.L[1], Lz = L.L[2];
    int X[ND], Y[ND], Z[ND];
#pragma unroll
    for (int k = 0; k < ND; ++k) {
        const uint32_t p = sxyz[c[k]];
        X[k] = px(p);
        Y[k] = py(p);
        Z[k] = pz(p);
    }
    KT best = (KT)~(KT)0;
    at = 0;
#pragma unroll
    for (int k = 0; k < ND; ++k) {
        int l[ND - 1];
#pragma unroll
        for (int i = 0; i < ND - 1; ++i) {
            const int o = i < k ? i : i + 1;
            l[i] = site_diff(X[o], Y[o], Z[o], X[k], Y[k], Z[k], Lx, Ly, Lz);
        }
        sort_net(l);
        const KT key = pack_list<ND - 1, KT>(l, base);
        if (key < best || k == 0) {
            best = key;
            at = sxyz[c[k]];
        }
    }
    return best;
}

// p f out of line, so that the multiplications of the rare targets whose
// |Stab| differs are a branch and not predicated fp64 instructions that every
// hop issues
template <typename CT, typename R> __device__ __noinline__ CT scaled(CT p, R f) {
    p.x *= f;
    p.y *= f;
    return p;
}
template <typename KT> __device__ __forceinline__ KT rec_key(uint4 r);
template <> __device__ __forceinline__ uint32_t rec_key<uint32_t>(uint4 r) { return r.x; }
template <> __device__ __forceinline__ unsigned long long rec_key<unsigned long long>(uint4 r) {
    return ((unsigned long long)r.y << 32) | r.x;
}

// hops in flight together: 2 hops at 4 (complex128) or 3 resident blocks per SM
// took 13.1 / 2.06 ms on the two cubes, 3 hops 13.5 / 2.12, 1 hop 14.6 / 2.10
constexpr int SH_HB = 2;

template <int ND, typename VT, typename KT>
__global__ void __launch_bounds__(NTHREADS, sizeof(VT) == 16 ? 4 : 3) k_hphi_f(LatView L, const SecView *__restrict__ secs,
                                                        const int *__restrict__ tile0, int S, int ntiles,
                                                        const VT *__restrict__ phi, VT *__restrict__ psi,
                                                        const int *__restrict__ active, unsigned fi_off) {
    using R = typename VTr<VT>::R;
    using CT = typename VTr<VT>::C;
    constexpr int NO = ND - 1;             // unmoved spins; sites of an origin form
    extern __shared__ __align__(16) unsigned char smem[];
    SmemLayout sm = carve(L, smem);
    stage_tables(L, sm.sC, sm.sxyz);
    R *snorm = (R *)sm.snorm;
    if (threadIdx.x < 9) {
        snorm[threadIdx.x] = (R)sqrt((double)threadIdx.x);
        snorm[9 + threadIdx.x] = threadIdx.x ? (R)(1.0 / sqrt((double)threadIdx.x)) : (R)0;
    }
    const R *jxy = jxy_table<VT>(L);
    const R juni = (R)L.jh_uniform;
    const bool uni = juni != (R)0;
    const int np1 = L.np1, Lx = L.L[0], Ly = L.L[1], Lz = L.L[2], bits = L.form_bits;
    const KT kbase = (KT)1 << bits;
    __syncthreads();
    CT *ph = (CT *)sm.sph;
    uint2 *sfi = (uint2 *)(smem + fi_off);
    int cur = -1;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int s = (S == 1) ? 0 : sector_of_tile(tile0, S, t);
        if (active && !active[s]) continue;
        const SecView &sv = secs[s];
        if (s != cur) {
            __syncthreads();
            const CT *g = phase_table<CT>(sv);
            for (int i = threadIdx.x; i < L.N; i += blockDim.x) {
                ph[i] = g[i];
                sfi[i] = sv.finfo[i];
            }
            __syncthreads();
            cur = s;
        }
        const uint64_t row = (uint64_t)(t - sv.tile0) * TILE + threadIdx.x;
        if (row >= sv.dim) continue;
        int c[ND];
        unrank(__ldg(sv.sigma + row), sm.sC, np1, c);
        const VT *__restrict__ ph_in = phi + sv.off;
        const uint4 *__restrict__ orec = sv.orec;
        const uint32_t *__restrict__ fsub = sv.fsub;
        const int st_row = sv.stab[row];
        const R rs = snorm[9 + st_row];
        R e = diag_row<R>(L), dd = 0;
        int npair = 0;
        CT acc, acch;
        acc.x = 0; acc.y = 0;
        acch.x = 0; acch.y = 0;
#pragma unroll 1
        for (int m = 0; m < ND; ++m) {
            const int i = pick(c, m);
            if (!L.diag_uniform) e += diag_u<R>(L, i);
            const int e0 = __ldg(L.adj_ptr + i), e1 = __ldg(L.adj_ptr + i + 1);
            // the unmoved spins and, for each, the sorted differences of the others to it
            int oX[NO], oY[NO], oZ[NO], E[NO][NO > 1 ? NO - 1 : 1];
            uint32_t oP[NO];
#pragma unroll
            for (int k = 0; k < NO; ++k) {
                oP[k] = sm.sxyz[k < m ? c[k] : c[k + 1]];
                oX[k] = px(oP[k]);
                oY[k] = py(oP[k]);
                oZ[k] = pz(oP[k]);
            }
            if constexpr (NO > 1) {
#pragma unroll
                for (int k = 0; k < NO; ++k) {
#pragma unroll
                    for (int q = 0; q < NO - 1; ++q) {
                        const int o = q < k ? q : q + 1;
                        E[k][q] = site_diff(oX[o], oY[o], oZ[o], oX[k], oY[k], oZ[k], Lx, Ly, Lz);
                    }
                    sort_net(E[k]);
                }
            }
#pragma unroll 1
            for (int q0 = e0; q0 < e1; q0 += SH_HB) {
                KT key[SH_HB];
                uint32_t org[SH_HB];
                bool go[SH_HB];
#pragma unroll
                for (int h = 0; h < SH_HB; ++h) {
                    key[h] = (KT)~(KT)0;
                    org[h] = 0;
                    go[h] = q0 + h < e1;
                    if (!go[h]) continue;
                    const int j = __ldg(L.adj_nbr + q0 + h);
#pragma unroll
                    for (int k = 0; k < ND; ++k) go[h] &= c[k] != j;
                    if (!go[h]) {
                        if (L.diag_uniform) ++npair;
                        else dd += diag_jz<R>(L, q0 + h);
                        continue;
                    }
                    const uint32_t pj = sm.sxyz[j];
                    const int jx = px(pj), jy = py(pj), jz = pz(pj);
                    // the moved spin at the origin
                    int l[NO];
#pragma unroll
                    for (int k = 0; k < NO; ++k) l[k] = site_diff(oX[k], oY[k], oZ[k], jx, jy, jz, Lx, Ly, Lz);
                    sort_net(l);
                    key[h] = pack_list<NO, KT>(l, kbase);
                    org[h] = pj;
                    // an unmoved spin at the origin
#pragma unroll
                    for (int k = 0; k < NO; ++k) {
                        int v = site_diff(jx, jy, jz, oX[k], oY[k], oZ[k], Lx, Ly, Lz);
                        int f[NO];
#pragma unroll
                        for (int x = 0; x < NO - 1; ++x) {
                            f[x] = min(E[k][x], v);
                            v = max(E[k][x], v);
                        }
                        f[NO - 1] = v;
                        const KT kk = pack_list<NO, KT>(f, kbase);
                        if (kk < key[h]) {
                            key[h] = kk;
                            org[h] = oP[k];
                        }
                    }
                }
                // the forms' rows: bucket, record, phi -- each stage's loads together
                uint32_t lo[SH_HB], hi[SH_HB];
#pragma unroll
                for (int h = 0; h < SH_HB; ++h) {
                    lo[h] = hi[h] = 0u;
                    if (go[h]) {
                        int f[NO];
                        unpack_list<NO, KT>(key[h], bits, f);
                        uint64_t low;
                        const uint2 fi = sfi[prefix_of(f, sm.sC, np1, 0, low)];
                        const uint32_t *b = fsub + fi.x + (uint32_t)(low >> fi.y);
                        lo[h] = __ldg(b);
                        hi[h] = __ldg(b + 1);
                    }
                }
                uint32_t val[SH_HB], wst[SH_HB];
#pragma unroll
                for (int h = 0; h < SH_HB; ++h) {
                    while (hi[h] - lo[h] > 4u) {
                        const uint32_t mid = (lo[h] + hi[h]) >> 1;
                        if (rec_key<KT>(__ldg(orec + mid)) <= key[h]) lo[h] = mid; else hi[h] = mid;
                    }
                }
                uint4 rec[SH_HB];
#pragma unroll
                for (int h = 0; h < SH_HB; ++h)
                    if (lo[h] < hi[h]) rec[h] = __ldg(orec + lo[h]);
#pragma unroll
                for (int h = 0; h < SH_HB; ++h) {
                    bool found = lo[h] < hi[h] && rec_key<KT>(rec[h]) == key[h];
                    while (!found && ++lo[h] < hi[h]) {
                        rec[h] = __ldg(orec + lo[h]);
                        found = rec_key<KT>(rec[h]) == key[h];
                    }
                    go[h] = go[h] && found;
                    val[h] = rec[h].z;
                    wst[h] = rec[h].w;
                }
                VT xv[SH_HB];
#pragma unroll
                for (int h = 0; h < SH_HB; ++h)
                    if (go[h]) xv[h] = ph_in[val[h]];
#pragma unroll
                for (int h = 0; h < SH_HB; ++h) {
                    if (!go[h]) continue;
                    const int st = (int)(wst[h] >> 28) + 1;
                    const uint32_t wp = sm.sxyz[wst[h] & 0xfffffffu];
                    const int u = site_diff(px(org[h]), py(org[h]), pz(org[h]), px(wp), py(wp), pz(wp), Lx, Ly, Lz);
                    CT p = ph[u];
                    if (uni) {
                        // uniform J^xy: the amplitude is applied once per row below
                        if (st != st_row) p = scaled(p, snorm[st] * rs);
                        acc_add(acch, p, xv[h]);
                    } else {
                        const R jh = __ldg(jxy + q0 + h);
                        const R wgt = (st == st_row) ? jh : jh * snorm[st] * rs;
                        p.x *= wgt;
                        p.y *= wgt;
                        acc_add(acc, p, xv[h]);
                    }
                }
            }
        }
        if (uni) madd_r(acc, juni, acch);
        if (L.diag_uniform) dd = diag_pairs<R>(L, npair);
        madd_r(acc, e + (R)0.5 * dd, ph_in[row]);
        store(psi + sv.off + row, acc);
    }
}

// the origin forms of a sector's rows
template <int ND, typename KT>
__global__ void __launch_bounds__(NTHREADS) k_forms(LatView L, SecView sv, KT *__restrict__ key,
                                                    uint2 *__restrict__ val) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *sC = (uint64_t *)smem;
    uint32_t *sxyz = (uint32_t *)(sC + (L.nd + 3) * L.np1);
    stage_tables(L, sC, sxyz);
    __syncthreads();
    for (uint64_t row = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; row < sv.dim;
         row += (uint64_t)gridDim.x * blockDim.x) {
        int c[ND];
        unrank(__ldg(sv.sigma + row), sC, L.np1, c);
        uint32_t at;
        key[row] = origin_form<ND, KT>(c, L, sxyz, (KT)1 << L.form_bits, at);
        const uint32_t w = (uint32_t)(px(at) + L.L[0] * (py(at) + L.L[1] * pz(at)));
        val[row] = make_uint2((uint32_t)row, w | ((uint32_t)(sv.stab[row] - 1) << 28));
    }
}

// the records in order: (form, row, w | (|Stab| - 1) << 28)
template <typename KT>
__global__ void k_form_recs(const KT *__restrict__ key, const uint2 *__restrict__ val, uint64_t d, uint4 *__restrict__ rec) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < d; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t k = key[i];
        rec[i] = make_uint4((uint32_t)k, (uint32_t)(k >> 32), val[i].x, val[i].y);
    }
}
// per largest site P <= N: the first form with one >= P
template <typename KT>
__global__ void k_form_first(const KT *__restrict__ key, uint64_t d, int bits, int no, uint32_t np,
                             uint32_t *__restrict__ first) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= np; i += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t lo = 0, hi = d;
        const uint64_t k = (uint64_t)i << (bits * (no - 1));
        while (lo < hi && i < np) {
            const uint64_t mid = (lo + hi) >> 1;
            if ((uint64_t)key[mid] < k) lo = mid + 1; else hi = mid;
        }
        first[i] = (uint32_t)(i < np ? lo : d);
    }
}
template <int NO, typename KT>
__global__ void __launch_bounds__(NTHREADS) k_form_fill(LatView L, const KT *__restrict__ key, uint64_t d,
                                                        const uint32_t *__restrict__ first,
                                                        const uint2 *__restrict__ info, uint32_t *__restrict__ sub) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *sC = (uint64_t *)smem;
    stage_tables(L, sC, nullptr);
    __syncthreads();
    for (uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; r < d; r += (uint64_t)gridDim.x * blockDim.x) {
        int f[NO];
        uint64_t low, lowp;
        unpack_list<NO, KT>(key[r], L.form_bits, f);
        const uint32_t P = prefix_of(f, sC, L.np1, 0, low);
        const uint2 pi = info[P];
        uint32_t *e = sub + pi.x;
        const uint32_t q = (uint32_t)(low >> pi.y);
        uint32_t q0 = 0;
        if (r > first[P]) {
            unpack_list<NO, KT>(key[r - 1], L.form_bits, f);
            prefix_of(f, sC, L.np1, 0, lowp);
            q0 = (uint32_t)(lowp >> pi.y) + 1;
        }
        for (uint32_t k = q0; k <= q; ++k) e[k] = (uint32_t)r;
        if (r + 1 == first[P + 1]) {
            uint32_t nq;
            bucket_shift(P, first[P + 1] - first[P], NO, 0, L.binom, L.np1, nq);
            for (uint32_t k = q + 1; k <= nq; ++k) e[k] = (uint32_t)(r + 1);
        }
    }
}
// whether the origin forms of a basis exist, and the bytes they hold
static bool forms_apply(const Basis &B) {
    int bits = 1;
    while ((1 << bits) < B.N) ++bits;
    return B.has_k && B.nd >= 2 && B.nsub == 1 && B.total > 0 && (B.nd - 1) * bits <= 64;
}

// shared memory of k_hphi_f: the row kernels' tables, then the index of the largest site
static size_t forms_off(const Basis &B) { return (B.smem_bytes + 15) & ~(size_t)15; }
static size_t forms_smem(const Basis &B) { return forms_off(B) + (size_t)B.N * sizeof(uint2); }

template <int ND, typename KT>
static int build_forms_nd(Basis &B) {
    constexpr int NO = ND - 1;
    const int S = B.S, bits = B.lv.form_bits;
    const uint32_t np = (uint32_t)B.N;
    uint64_t dmax = 0;
    for (uint64_t d : B.dims) dmax = std::max(dmax, d);
    // per sector at most a bucket per row or site, and an end per site
    DevBuf rec, info, sub;
    QS3_TRY(rec.alloc(B.total * sizeof(uint4)));
    QS3_TRY(info.alloc((uint64_t)S * np * sizeof(uint2)));
    QS3_TRY(sub.alloc((B.total + 2 * (uint64_t)S * np) * 4));
    const cudaStream_t s0 = 0;
    DevBuf kin, vin, key, val, first, size, off, tmp;
    QS3_TRY(kin.alloc(dmax * sizeof(KT), s0));
    QS3_TRY(vin.alloc(dmax * sizeof(uint2), s0));
    QS3_TRY(key.alloc(dmax * sizeof(KT), s0));
    QS3_TRY(val.alloc(dmax * sizeof(uint2), s0));
    QS3_TRY(first.alloc(((uint64_t)np + 1) * 4, s0));
    QS3_TRY(size.alloc(((uint64_t)np + 1) * 4, s0));
    QS3_TRY(off.alloc(((uint64_t)np + 1) * 4, s0));
    size_t tb = 0, tb2 = 0;
    using U64 = unsigned long long;
    QS3_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, tb, kin.as<KT>(), key.as<KT>(), vin.as<U64>(), val.as<U64>(),
                                             (int64_t)dmax, 0, bits * NO));
    QS3_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tb2, size.as<uint32_t>(), off.as<uint32_t>(), (int64_t)np + 1));
    tb = std::max(tb, tb2);
    QS3_TRY(tmp.alloc(tb, s0));
    const size_t smem = (size_t)(B.nd + 3) * (B.N + 1) * 8 + (size_t)B.N * 4;
    QS3_CUDA(cudaFuncSetAttribute(k_forms<ND, KT>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_DYN_SMEM));
    QS3_CUDA(cudaFuncSetAttribute(k_form_fill<NO, KT>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_DYN_SMEM));
    const uint64_t *bin = B.lv.binom;
    const int gp = (int)((np + 256) / 256);
    uint64_t base = 0;
    for (int s = 0; s < S; ++s) {
        const uint64_t d = B.dims[s];
        SecView &v = B.secs[s];
        uint2 *is = info.as<uint2>() + (uint64_t)s * np;
        uint32_t *ss = sub.as<uint32_t>() + base;
        const int g = (int)std::max<uint64_t>(1, std::min<uint64_t>((d + NTHREADS - 1) / NTHREADS, 8192));
        if (d > 0) {
            k_forms<ND, KT><<<g, NTHREADS, smem>>>(B.lv, v, kin.as<KT>(), vin.as<uint2>());
            QS3_LAUNCHED();
            size_t t2 = tb;
            QS3_CUDA(cub::DeviceRadixSort::SortPairs(tmp.p, t2, kin.as<KT>(), key.as<KT>(), vin.as<U64>(), val.as<U64>(),
                                                     (int64_t)d, 0, bits * NO));
            k_form_recs<KT><<<g, NTHREADS>>>(key.as<KT>(), val.as<uint2>(), d, rec.as<uint4>() + B.offs[s]);
            QS3_LAUNCHED();
        }
        k_form_first<KT><<<gp, 256>>>(key.as<KT>(), d, bits, NO, np, first.as<uint32_t>());
        QS3_LAUNCHED();
        QS3_CUDA(cudaMemsetAsync(size.as<uint32_t>() + np, 0, 4));
        k_bucket_size<false><<<gp, 256>>>(NO, B.N + 1, 0, bin, 1, np, 0, first.as<uint32_t>(), size.as<uint32_t>());
        QS3_LAUNCHED();
        size_t t2 = tb;
        QS3_CUDA(cub::DeviceScan::ExclusiveSum(tmp.p, t2, size.as<uint32_t>(), off.as<uint32_t>(), (int64_t)np + 1));
        k_bucket_info<false><<<gp, 256>>>(NO, B.N + 1, 0, bin, 1, np, 0, first.as<uint32_t>(), off.as<uint32_t>(), is, ss);
        QS3_LAUNCHED();
        if (d > 0) {
            k_form_fill<NO, KT><<<g, NTHREADS, smem>>>(B.lv, key.as<KT>(), d, first.as<uint32_t>(), is, ss);
            QS3_LAUNCHED();
        }
        v.orec = rec.as<uint4>() + B.offs[s];
        v.finfo = is;
        v.fsub = ss;
        base += d + 2 * (uint64_t)np;
    }
    QS3_CUDA(cudaDeviceSynchronize());
    B.d_orec = std::move(rec);
    B.d_finfo = std::move(info);
    B.d_fsub = std::move(sub);
    QS3_CUDA(cudaMemcpy(B.d_secs.p, B.secs.data(), B.secs.size() * sizeof(SecView), cudaMemcpyHostToDevice));
    return QS3_OK;
}

template <int ND>
static int build_forms_k(Basis &B) {
    return (ND - 1) * B.lv.form_bits <= 32 ? build_forms_nd<ND, uint32_t>(B) : build_forms_nd<ND, unsigned long long>(B);
}

int build_forms(Basis &B, size_t max_bytes) {
    if (!forms_apply(B)) return set_err(QS3_ERR_STATE, "no origin forms for this basis");
    int bits = 1;
    while ((1 << bits) < B.N) ++bits;
    if (forms_smem(B) > (size_t)MAX_DYN_SMEM) return set_err(QS3_ERR_OVERFLOW, "origin forms need more shared memory");
    // the records and their index, and the sort's buffers
    if (B.total * (16 + 4 + 3 * 16) > max_bytes) return set_err(QS3_ERR_OOM, "origin forms exceed the limit");
    B.lv.form_bits = bits;
    switch (B.nd) {
        case 2: return build_forms_k<2>(B);
        case 3: return build_forms_k<3>(B);
        case 4: return build_forms_k<4>(B);
        case 5: return build_forms_k<5>(B);
        case 6: return build_forms_k<6>(B);
        case 7: return build_forms_k<7>(B);
        case 8: return build_forms_k<8>(B);
        default: return set_err(QS3_ERR_INVALID_ARG, "n_down %d", B.nd);
    }
}

template <int ND, typename VT, typename KT>
static int forms_run(Basis &B, const void *phi, void *psi, cudaStream_t st, const int *active, int dt) {
    static std::atomic<unsigned long long> cache{0};
    int grid = 1, occ = 1;
    const size_t smem = forms_smem(B);
    QS3_TRY(launch_rows(k_hphi_f<ND, VT, KT>, B, smem, cache, &grid, &occ));
    if (B.ntiles == 0) return QS3_OK;
    k_hphi_f<ND, VT, KT><<<grid, NTHREADS, smem, st>>>(B.lv, B.d_secs.as<SecView>(), B.tile0_d, B.S, B.ntiles,
                                                       (const VT *)phi, (VT *)psi, active, (unsigned)forms_off(B));
    QS3_LAUNCHED();
    if (B.tune_hphi[dt] == 0) B.tune_hphi[dt] = occ;             // always the whole occupancy
    return QS3_OK;
}

template <typename VT>
static int forms_vt(Basis &B, const void *phi, void *psi, cudaStream_t st, const int *a, int dt) {
#define QS3_F(n)                                                                                          \
    ((n - 1) * B.lv.form_bits <= 32 ? forms_run<n, VT, uint32_t>(B, phi, psi, st, a, dt)                  \
                                    : forms_run<n, VT, unsigned long long>(B, phi, psi, st, a, dt))
    switch (B.nd) {
        case 2: return QS3_F(2);
        case 3: return QS3_F(3);
        case 4: return QS3_F(4);
        case 5: return QS3_F(5);
        case 6: return QS3_F(6);
        case 7: return QS3_F(7);
        case 8: return QS3_F(8);
        default: return set_err(QS3_ERR_INVALID_ARG, "n_down %d", B.nd);
    }
#undef QS3_F
}

int hphi_forms_launch(Basis &B, qs3_dtype dt, const void *phi, void *psi, cudaStream_t st, const int *active) {
    if (dt == QS3_C64) return forms_vt<float2>(B, phi, psi, st, active, dt);
    if (dt == QS3_C128) return forms_vt<double2>(B, phi, psi, st, active, dt);
    return set_err(QS3_ERR_INVALID_ARG, "dtype %d", (int)dt);
}

}  // namespace qs3
