// qs3_internal.cuh -- host structures and device helpers shared by the
// libqs3 translation units (GPU path only).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "qs3.h"

namespace qs3 {

constexpr int MAXND = QS3_MAX_NDOWN;
constexpr int TILE = 256;          // rows per tile (one thread per row)
constexpr int NTHREADS = 256;
constexpr int BROWS = 2048;        // rows per chunk of the vector kernels (8 per thread)
// every kernel with dynamic shared memory gets this one limit (bases larger
// than it are rejected at creation), so concurrent host threads setting the
// attribute never disagree
constexpr int MAX_DYN_SMEM = 200 * 1024;

// ------------------------------------------------------------------ errors
int set_err(int code, const char *fmt, ...);
void clear_err();
const char *last_err();

#define QS3_CUDA(call)                                                                             \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess)                                                                     \
            return ::qs3::set_err(e_ == cudaErrorMemoryAllocation ? QS3_ERR_OOM : QS3_ERR_CUDA,   \
                                  "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__,       \
                                  __LINE__);                                                       \
    } while (0)

// every kernel launch of the library is followed by QS3_LAUNCHED(): it counts
// the launch (qs3_kernel_launches) and turns a launch error into a status
void count_launch(long long n = 1);   // n < 0 takes back launches that were only captured
#define QS3_LAUNCHED()                                                                             \
    do {                                                                                           \
        ::qs3::count_launch();                                                                     \
        QS3_CUDA(cudaGetLastError());                                                              \
    } while (0)

#define QS3_TRY(expr)                                                                              \
    do {                                                                                           \
        int s_ = (expr);                                                                           \
        if (s_ != QS3_OK) return s_;                                                               \
    } while (0)

// owning device buffer.  alloc(bytes) is a cudaMalloc, for what a handle
// keeps; alloc(bytes, st) takes the memory from the device's pool in the order
// of stream st, and the release returns it in that order: for the scratch of
// one call, all of whose uses are on st (or were waited for).  A cudaMalloc /
// cudaFree pair of such scratch cost up to 0.4 ms per call and made every
// other stream wait.  The pool keeps at most POOL_KEEP_BYTES unused; requests
// above POOL_MAX_BYTES are a cudaMalloc all the same, because what the pool
// does not keep it maps at 2.0 ms per GB against 0.55 (a 250-vector Krylov
// basis of 31 GB: 232 ms a solve against 186).
struct DevBuf {
    void *p = nullptr;
    size_t n = 0;
    bool pooled = false;
    cudaStream_t st = nullptr;
    DevBuf() = default;
    DevBuf(const DevBuf &) = delete;
    DevBuf &operator=(const DevBuf &) = delete;
    DevBuf(DevBuf &&o) noexcept : p(o.p), n(o.n), pooled(o.pooled), st(o.st) { o.p = nullptr; o.n = 0; }
    DevBuf &operator=(DevBuf &&o) noexcept {
        if (this != &o) { release(); p = o.p; n = o.n; pooled = o.pooled; st = o.st; o.p = nullptr; o.n = 0; }
        return *this;
    }
    ~DevBuf() { release(); }
    void release();
    int alloc(size_t bytes);                      // QS3_ERR_OOM on failure
    int alloc(size_t bytes, cudaStream_t st);
    int upload(const void *src, size_t bytes);    // alloc + H2D copy
    int upload(const void *src, size_t bytes, cudaStream_t st);
    template <class T> T *as() const { return (T *)p; }
};

constexpr size_t POOL_KEEP_BYTES = (size_t)512 << 20, POOL_MAX_BYTES = (size_t)256 << 20;
// the current device's unused pool memory goes back, but for `keep` bytes.
// A basis that is destroyed leaves POOL_IDLE_BYTES, the pool's smallest unit:
// with none left, the next small basis mapped it again and its destruction
// unmapped it (one sector of 5x5: destruction 175 us, now 94).
void pool_trim(size_t keep);
constexpr size_t POOL_IDLE_BYTES = (size_t)32 << 20;

// ------------------------------------------------------- device-side views

// Lattice data needed by every kernel.  binom rows m = 0..nd+2, each of
// np1 = N + 1 entries: binom[m * np1 + c] = C(c, m).
struct LatView {
    int N, nd, np1;
    int L[3];
    int has_k;
    int key_bits;                 // bits per site of a packed key, 0 -> compare ranks
    int form_bits;                // bits per site of a packed origin form (0: none built)
    int mask_ok;                  // canon_mask applies: L <= 32 along each axis, keys fit 64 bits
    const uint64_t *binom;
    const int *adj_ptr;           // N + 1
    const int *adj_nbr;           // 2 n_bonds
    const double *adj_jxy;        // 2 n_bonds: hop amplitude J^xy / 2 of the bond
    const double *adj_jz;         // 2 n_bonds
    const float *adj_jxy_f;       // fp32 copy of adj_jxy
    const double *u;              // N: -(1/2) sum_j Jz_ij + h_i
    double c0;                    // sum_b Jz_b / 4 - (1/2) sum_i h_i
    const float *u_f;             // fp32 copies of u, c0 and adj_jz for the fp32 kernels
    float c0f;
    const float *adj_jz_f;
    // the fp32 remainders v - fl32(v) of adj_jxy, u, adj_jz and c0: with the
    // fp32 copies they are the double-float constants of the C128DF product
    const float *adj_jxy_lo;
    const float *u_lo;
    const float *adj_jz_lo;
    float c0lo;
    const uint32_t *xyz;          // N: the site's cell coordinates x | y << 11 | z << 22
    int nsub;                     // spins per unit cell: site r is spin r % nsub of cell r / nsub
    int ncell;                    // cells, the order of the translation group
    // representative table (k-sectors, optional): for every state a, by its
    // rank0, orb[rank0] = g << 12 | u, where the orbit's representative is the
    // g-th of the sorted list of all representatives and a = T_u (rep): the
    // translation by -u (u the flat site index) takes a to its representative
    const uint32_t *orb;
    uint32_t n_orb;               // orbits in the table (entries >= n_orb << 12 are invalid)
    // diagonal constants of lattices with one J^z and the same u on every site
    // (diag_uniform): c0 plus N_down times u, and the sums of 0, 1, ... J^z, all
    // added one by one as the row kernels do
    int diag_uniform;
    double e_row;
    float e_row_f;
    const double *pair_sum;
    const float *pair_sum_f;
    double jh_uniform;            // the hop amplitude J^xy / 2 when every bond has the same one, else 0
    // U(1)-only bases of largest degree <= 6: fixed-width adjacency, pad_w
    // entries per site, (neighbour, hop amplitude) in one load: fp32 in 8 bytes,
    // fp64 in 16 (neighbour, -, amplitude); a site with fewer neighbours is
    // padded with itself and zero couplings.  adjt: the fp32 entries transposed
    // (entry b of site i at b N + i), so that threads of consecutive
    // sites read consecutive words
    int pad_w;                    // 2, 4 or 6; 0 when the tables are not built
    const int2 *adj_pad, *adjt;
    const int4 *adj_pad64;
    const float *adj_jz_pad, *adjt_jz;
    const double *adj_jz_pad64;
};

constexpr uint32_t ONE_BUCKET = 0x80u;    // beyond every shift

struct SecView {
    const uint64_t *sigma;        // sorted rank0 of the representatives (NULL: U(1))
    const uint8_t *stab;          // |Stab| of each representative
    // index over sigma: the rows whose representatives share their two largest
    // sites (pre2; else the largest one), prefix P, are split by the rank of
    // their other sites into buckets of a few rows: pinfo[P] = (first entry o,
    // shift), rows of bucket q = low rank >> shift are sub[o + q] .. sub[o + q
    // + 1] - 1.  With N_down <= 3, where most prefixes have a row or two, a prefix
    // of one bucket (up to three rows) has no entries but pinfo[P] = (first row,
    // ONE_BUCKET | rows << 8), one dependent load less
    const uint2 *pinfo;
    const uint32_t *sub;
    int pre2;
    // origin forms of the rows (qs3_hphi_search.cu), when built: the sorted
    // records (form, row, w | (|Stab| - 1) << 28), and their index by the
    // largest site
    const uint4 *orec;
    const uint2 *finfo;
    const uint32_t *fsub;
    uint64_t dim;
    uint64_t off;                 // offset of the sector in a concatenated vector
    int K[3];
    int tile0;                    // first tile of the sector
    const double2 *ph64;          // k-sectors: per-site phases e^{-2 pi i K.r/L} (fp64) ...
    const float2 *ph32;           // ... and their fp32 copy; NULL for U(1)
    const float4 *phdf;           // ... and their double-float split (re.hi, re.lo, im.hi, im.lo)
    const int32_t *t2;            // with the representative table: orbit g -> row of this sector, -1 if absent
};

// ---------------------------------------------------------- host basis
constexpr int SEG_REACH = 24;

struct Basis {
    int N = 0, nd = 0, nb = 0;
    int L[3] = {0, 0, 0};
    int nsub = 1, ncell = 0;                // spins per cell, cells (the group order)
    bool has_k = false;
    int S = 0;                              // sectors
    std::vector<int> K;                     // 3 S
    std::vector<uint64_t> dims, offs;       // S, S + 1
    uint64_t total = 0;
    std::vector<int> tile0;                 // S + 1
    int ntiles = 0;
    std::vector<int> chunk0;                // S + 1, chunks of BROWS rows (vector kernels)
    int nchunks = 0;
    // host copies of the model
    std::vector<int> bi, bj;
    std::vector<double> jxy, jz, h, pos;
    std::vector<uint64_t> binom;            // host copy of the binomial rows 0 .. nd + 2
    bool has_h = false;
    int n_long_bonds = 0;                   // bonds of more than N / SEG_REACH sites' distance in the numbering
    // device data
    DevBuf d_tab;                           // the tables that lv points to, tile0, chunk0 and K
    const int *tile0_d = nullptr, *chunk0_d = nullptr, *K_d = nullptr;
    DevBuf d_sigma, d_stab, d_pinfo, d_sub;  // every sector's lists, one after another
    DevBuf d_orec, d_finfo, d_fsub;          // origin forms and their index (without a representative table)
    DevBuf d_ph;                            // S x N per-site phase tables and the roots (k-sectors)
    const double2 *roots_d = nullptr;       // e^{-2 pi i n / ncell}, n < ncell
    DevBuf d_secs;
    LatView lv{};
    std::vector<SecView> secs;
    uint64_t nnz = 0;                       // structural non-zeros (count_nnz), total and per sector
    std::vector<uint64_t> nnz_sec;
    bool nnz_valid = false;
    size_t smem_bytes = 0;                  // dynamic shared memory of the row kernels
    DevBuf d_orb, d_t2;                     // representative table (LatView::orb, SecView::t2)
    uint64_t n_orb = 0;                     // orbits (all representatives) when the table exists
    DevBuf d_oreps, d_ostab;                // with the table: each orbit's representative (rank0) and |Stab|
    DevBuf d_phdig;                         // with the table: S x N phases as digits on 2^-52 (int4)
    // autotuned launch choices, 0 = not yet tuned: resident H Phi blocks per
    // SM per vector dtype (the persistent grid, i.e. rows in flight per SM),
    // and basis vectors per pass of the double-float dot products
    int tune_hphi[5] = {0, 0, 0, 0, 0};     // indexed by qs3_dtype
    int tune_hphix = 0;                     // the same for the binary64 engine's integer H Phi
    int tune_nv = 0;
    int tune_nv64 = 0;                      // the same for the binary64 dot products (IEEE engine)
    bool narrow_ranks = false;              // U(1) with C(N, N_down) < 2^32: 32-bit rank kernels apply
    // stored terms of the k-sector H Phi (opt-in): row pointers, target rows,
    // codes (u | st << 12 | q << 16) and per-row diagonals
    DevBuf d_trp, d_tcol, d_tcode, d_tdiag;
    uint64_t n_terms = 0;
    bool stored_terms = false;
    int max_degree = 0;                     // largest number of adjacency entries of a site
};

// sector of tile t (binary search over tile0[0..S])
__device__ __forceinline__ int sector_of_tile(const int *tile0, int S, int t) {
    int lo = 0, hi = S - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (tile0[mid] <= t) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// --------------------------------------------------- combinatorial helpers

// ascending bubble network on registers (static indexing only)
template <int ND>
__device__ __forceinline__ void sort_net(int (&a)[ND]) {
#pragma unroll
    for (int i = 0; i < ND; ++i) {
#pragma unroll
        for (int j = 0; j < ND - 1 - i; ++j) {
            int lo = min(a[j], a[j + 1]);
            int hi = max(a[j], a[j + 1]);
            a[j] = lo;
            a[j + 1] = hi;
        }
    }
}

// rank0 = sum_m C(c_m, m + 1) of an ascending list (Eq. a_of_n, 0-based)
template <int ND>
__device__ __forceinline__ uint64_t rank_of(const int (&c)[ND], const uint64_t *__restrict__ sC, int np1) {
    uint64_t r = 0;
#pragma unroll
    for (int m = 0; m < ND; ++m) r += sC[(m + 1) * np1 + c[m]];
    return r;
}

// largest x in [m-1, hi] with C(x, m) <= r (col = column m of the table).
// C(x, m) ~ (x - (m-1)/2)^m / m! gives a float estimate of x; the exact table
// values then correct it by a step or two, with a binary search as fallback,
// so the result is exact for every r.
__device__ __forceinline__ int col_search(const uint64_t *__restrict__ col, int m, int hi, uint64_t r) {
    // log2(m!) for m = 0..8
    constexpr float lf[9] = {0.f, 0.f, 1.f, 2.5849625f, 4.5849625f, 6.9068906f, 9.4918531f, 12.299208f, 15.299208f};
    int x = m - 1;
    if (r > 0) {
        // uint64 -> float through two 32-bit halves (a 64-bit conversion would use the fp64 unit)
        const float rf = (float)(uint32_t)(r >> 32) * 4294967296.f + (float)(uint32_t)r;
        const float e = exp2f((__log2f(rf) + lf[m]) / (float)m) + 0.5f * (float)(m - 1);
        x = (int)e;
    }
    x = max(m - 1, min(x, hi));
#pragma unroll 1
    for (int it = 0; it < 3 && x < hi && col[x + 1] <= r; ++it) ++x;
#pragma unroll 1
    for (int it = 0; it < 3 && col[x] > r; ++it) --x;
    if (col[x] > r || (x < hi && col[x + 1] <= r)) {
        int lo = m - 1, h = hi;
        while (lo < h) {
            const int mid = (lo + h + 1) >> 1;
            if (col[mid] <= r) lo = mid; else h = mid - 1;
        }
        x = lo;
    }
    return x;
}

// inverse of rank_of (Alg. 1): greedy largest-first column search
template <int ND>
__device__ __forceinline__ void unrank(uint64_t r, const uint64_t *__restrict__ sC, int np1, int (&c)[ND]) {
    int hi = np1 - 2;
#pragma unroll
    for (int m = ND; m >= 2; --m) {
        const uint64_t *col = sC + m * np1;
        const int x = col_search(col, m, hi, r);
        c[m - 1] = x;
        r -= col[x];
        hi = x - 1;
    }
    if (ND >= 1) c[0] = (int)r;
}

// 32-bit forms for state spaces with C(N, N_down) < 2^32: every binomial a
// rank needs (rows 0..N_down) then fits 32 bits
template <int ND>
__device__ __forceinline__ uint32_t rank_of32(const int (&c)[ND], const uint32_t *__restrict__ sC, int np1) {
    uint32_t r = 0;
#pragma unroll
    for (int m = 0; m < ND; ++m) r += sC[(m + 1) * np1 + c[m]];
    return r;
}

__device__ __forceinline__ int col_search32(const uint32_t *__restrict__ col, int m, int hi, uint32_t r) {
    constexpr float lf[9] = {0.f, 0.f, 1.f, 2.5849625f, 4.5849625f, 6.9068906f, 9.4918531f, 12.299208f, 15.299208f};
    int x = m - 1;
    if (r > 0) x = (int)(exp2f((__log2f((float)r) + lf[m]) / (float)m) + 0.5f * (float)(m - 1));
    x = max(m - 1, min(x, hi));
#pragma unroll 1
    for (int it = 0; it < 3 && x < hi && col[x + 1] <= r; ++it) ++x;
#pragma unroll 1
    for (int it = 0; it < 3 && col[x] > r; ++it) --x;
    if (col[x] > r || (x < hi && col[x + 1] <= r)) {
        int lo = m - 1, h = hi;
        while (lo < h) {
            const int mid = (lo + h + 1) >> 1;
            if (col[mid] <= r) lo = mid; else h = mid - 1;
        }
        x = lo;
    }
    return x;
}

template <int ND>
__device__ __forceinline__ void unrank32(uint32_t r, const uint32_t *__restrict__ sC, int np1, int (&c)[ND]) {
    int hi = np1 - 2;
#pragma unroll
    for (int m = ND; m >= 2; --m) {
        const uint32_t *col = sC + m * np1;
        const int x = col_search32(col, m, hi, r);
        c[m - 1] = x;
        r -= col[x];
        hi = x - 1;
    }
    if (ND >= 1) c[0] = (int)r;
}

// select a[i] for a runtime i without dynamic register indexing
template <int ND>
__device__ __forceinline__ int pick(const int (&a)[ND], int i) {
    int v = a[0];
#pragma unroll
    for (int m = 1; m < ND; ++m) v = (i == m) ? a[m] : v;
    return v;
}

// Minimum-rank translate of the site list t (the representative of its
// orbit, Alg. 7), found without trying every translation.  Translations move
// unit cells; a site is spin sb of cell (x, y, z), index sb + nsub (x + Lx
// (y + Ly z)), so the order of sites follows their cells first.
//
// The rank order is the lexicographic order of the descending list of site
// indices r = x + Lx (y + Ly z), so a representative first minimises its
// largest site, which is the (z, y, x)-largest spin.  Hence, exactly:
//  - a representative has a spin at x = 0, one at y = 0 and one at z = 0
//    (otherwise a -1 shift along that axis lowers every site index), so the
//    shifts along each axis are taken from the spins' coordinates;
//  - level z: keep the z-shifts that minimise max z' over all spins;
//  - level y: for those, keep the y-shifts that minimise max y' over the
//    spins at the top z';
//  - level x: likewise max x' over the spins at the top (z', y').
// Every surviving translation gives the same largest site; the full keys
// (sorted lists) of the survivors -- usually one -- decide.  On return rep
// holds the sorted representative, (ax, by, cz) the coordinates moved to the
// origin (T^t a' = rep with t = -(ax, by, cz)), and the function returns its
// rank0.
template <int ND>
__device__ __forceinline__ uint64_t canon_gen(const int (&t)[ND], const LatView &L, const uint32_t *__restrict__ sxyz,
                                          const uint64_t *__restrict__ sC, int (&rep)[ND], int &ax, int &by,
                                          int &cz) {
    int X[ND], Y[ND], Z[ND], SB[ND];
#pragma unroll
    for (int m = 0; m < ND; ++m) {
        uint32_t p = sxyz[t[m]];
        X[m] = p & 2047u;
        Y[m] = (p >> 11) & 2047u;
        Z[m] = p >> 22;
        SB[m] = L.nsub > 1 ? t[m] % L.nsub : 0;     // the spin's place in its cell
    }
    const int Lx = L.L[0], Ly = L.L[1], Lz = L.L[2];
    const int kb = L.key_bits;
    // level z
    uint32_t mz = 1u;
    int bz = 0;
    if (Lz > 1) {
        bz = 0x7fffffff;
        mz = 0u;
#pragma unroll
        for (int c = 0; c < ND; ++c) {
            bool dup = false;
#pragma unroll
            for (int k = 0; k < c; ++k) dup |= (Z[k] == Z[c]);
            int mx = 0;
#pragma unroll
            for (int m = 0; m < ND; ++m) {
                int d = Z[m] - Z[c];
                d += (d < 0) ? Lz : 0;
                mx = max(mx, d);
            }
            if (!dup) {
                if (mx < bz) { bz = mx; mz = 1u << c; }
                else if (mx == bz) mz |= 1u << c;
            }
        }
    }
    uint64_t best = ~0ull;
    int bc = 0, bb = 0, ba = 0;
    for (uint32_t m1 = mz; m1; m1 &= m1 - 1) {
        const int c = __ffs(m1) - 1;
        const int zc = pick(Z, c);
        int zz[ND];
        uint32_t tz = 0u;
#pragma unroll
        for (int m = 0; m < ND; ++m) {
            int d = Z[m] - zc;
            d += (d < 0) ? Lz : 0;
            zz[m] = d;
            tz |= (d == bz ? 1u : 0u) << m;
        }
        // level y over the top-z spins
        uint32_t my = 1u;
        int byv = 0;
        if (Ly > 1) {
            byv = 0x7fffffff;
            my = 0u;
#pragma unroll
            for (int b = 0; b < ND; ++b) {
                bool dup = false;
#pragma unroll
                for (int k = 0; k < b; ++k) dup |= (Y[k] == Y[b]);
                int mx = -1;
#pragma unroll
                for (int m = 0; m < ND; ++m) {
                    int d = Y[m] - Y[b];
                    d += (d < 0) ? Ly : 0;
                    mx = ((tz >> m) & 1u) ? max(mx, d) : mx;
                }
                if (!dup) {
                    if (mx < byv) { byv = mx; my = 1u << b; }
                    else if (mx == byv) my |= 1u << b;
                }
            }
        }
        for (uint32_t m2 = my; m2; m2 &= m2 - 1) {
            const int b = __ffs(m2) - 1;
            const int yb = pick(Y, b);
            int yy[ND];
            uint32_t ty = 0u;
#pragma unroll
            for (int m = 0; m < ND; ++m) {
                int d = Y[m] - yb;
                d += (d < 0) ? Ly : 0;
                yy[m] = d;
                ty |= (((tz >> m) & 1u) && d == byv ? 1u : 0u) << m;
            }
            // level x over the top-(z, y) spins
            uint32_t mx3 = 1u;
            if (Lx > 1) {
                int bxv = 0x7fffffff;
                mx3 = 0u;
#pragma unroll
                for (int a = 0; a < ND; ++a) {
                    bool dup = false;
#pragma unroll
                    for (int k = 0; k < a; ++k) dup |= (X[k] == X[a]);
                    int mx = -1;
#pragma unroll
                    for (int m = 0; m < ND; ++m) {
                        int d = X[m] - X[a];
                        d += (d < 0) ? Lx : 0;
                        mx = ((ty >> m) & 1u) ? max(mx, d) : mx;
                    }
                    if (!dup) {
                        if (mx < bxv) { bxv = mx; mx3 = 1u << a; }
                        else if (mx == bxv) mx3 |= 1u << a;
                    }
                }
            }
            for (uint32_t m3 = mx3; m3; m3 &= m3 - 1) {
                const int a = __ffs(m3) - 1;
                const int xa = pick(X, a);
                int s[ND];
#pragma unroll
                for (int m = 0; m < ND; ++m) {
                    int d = X[m] - xa;
                    d += (d < 0) ? Lx : 0;
                    s[m] = SB[m] + L.nsub * (d + Lx * (yy[m] + Ly * zz[m]));
                }
                sort_net(s);
                uint64_t key;
                if (kb) {
                    key = 0;
#pragma unroll
                    for (int m = ND - 1; m >= 0; --m) key = (key << kb) | (uint64_t)s[m];
                } else {
                    key = rank_of(s, sC, L.np1);
                }
                if (key < best) {
                    best = key;
                    bc = c; bb = b; ba = a;
#pragma unroll
                    for (int m = 0; m < ND; ++m) rep[m] = s[m];
                }
            }
        }
    }
    ax = pick(X, ba);
    by = pick(Y, bb);
    cz = pick(Z, bc);
    return kb ? rank_of(rep, sC, L.np1) : best;
}

// the highest set bit of the L-bit word m (held twice in a row in mm, L <= 32)
// rotated right by c
__device__ __forceinline__ int rot_top(uint64_t mm, uint32_t full, int c) {
    return 31 - __clz((int)((uint32_t)(mm >> c) & full));
}
__device__ __forceinline__ uint64_t twice(uint32_t m, int L) { return (uint64_t)m | ((uint64_t)m << L); }
__device__ __forceinline__ uint32_t low_ones(int L) { return 0xffffffffu >> (32 - L); }

// the same minimum by occupation masks (LatView::mask_ok: L <= 32 along each
// axis and packed keys of 64 bits).  Along an axis the spins' coordinates
// form an L-bit word; the largest coordinate after moving c to 0 is the
// highest set bit of the word rotated by c, so a level costs a few integer
// instructions per candidate instead of a pass over all spins (ND^2
// subtract / wrap / max steps in canon_gen), and the spins at the top are
// those with one coordinate value.  A candidate whose top (y, x) exceeds the
// smallest met so far cannot win.  X, Y, Z, SB: the spins' cell coordinates
// and places in the cell, in any order; best: the packed sorted list of the
// representative (kb bits per site, the largest site highest).
template <int ND>
__device__ __forceinline__ void canon_mask(const int (&X)[ND], const int (&Y)[ND], const int (&Z)[ND],
                                           const int (&SB)[ND], const LatView &L, uint64_t &best, int &ax, int &by,
                                           int &cz) {
    const int Lx = L.L[0], Ly = L.L[1], Lz = L.L[2];
    const int kb = L.key_bits;
    // level z
    uint32_t mz = 1u;
    int bz = 0;
    if (Lz > 1) {
        uint32_t m = 0;
#pragma unroll
        for (int k = 0; k < ND; ++k) m |= 1u << Z[k];
        const uint64_t mm = twice(m, Lz);
        const uint32_t full = low_ones(Lz);
        bz = 32;
#pragma unroll
        for (int k = 0; k < ND; ++k) {
            const int t = rot_top(mm, full, Z[k]);
            mz = t < bz ? 0u : mz;
            bz = min(bz, t);
            mz |= t == bz ? 1u << Z[k] : 0u;
        }
    }
    best = ~0ull;
    int gy = 32, gx = 32;                  // the smallest top (y, x) so far
    ax = by = cz = 0;
    while (mz) {
        const int zc = __ffs(mz) - 1;
        mz &= mz - 1;
        int zt = zc + bz;                  // the z of the top spins
        zt -= zt >= Lz ? Lz : 0;
        // level y over the top-z spins
        uint32_t my = 1u;
        int byv = 0;
        if (Ly > 1) {
            uint32_t m = 0;
#pragma unroll
            for (int k = 0; k < ND; ++k) m |= Z[k] == zt ? 1u << Y[k] : 0u;
            const uint64_t mm = twice(m, Ly);
            const uint32_t full = low_ones(Ly);
            byv = 32;
#pragma unroll
            for (int k = 0; k < ND; ++k) {
                const int t = rot_top(mm, full, Y[k]);
                my = t < byv ? 0u : my;
                byv = min(byv, t);
                my |= t == byv ? 1u << Y[k] : 0u;
            }
        }
        if (byv > gy) continue;
        if (byv < gy) {
            gy = byv;
            gx = 32;
        }
        while (my) {
            const int yc = __ffs(my) - 1;
            my &= my - 1;
            int yt = yc + byv;
            yt -= yt >= Ly ? Ly : 0;
            // level x over the top-(z, y) spins
            uint32_t mx = 1u;
            int bxv = 0;
            if (Lx > 1) {
                uint32_t m = 0;
#pragma unroll
                for (int k = 0; k < ND; ++k) m |= (Z[k] == zt && Y[k] == yt) ? 1u << X[k] : 0u;
                const uint64_t mm = twice(m, Lx);
                const uint32_t full = low_ones(Lx);
                bxv = 32;
#pragma unroll
                for (int k = 0; k < ND; ++k) {
                    const int t = rot_top(mm, full, X[k]);
                    mx = t < bxv ? 0u : mx;
                    bxv = min(bxv, t);
                    mx |= t == bxv ? 1u << X[k] : 0u;
                }
            }
            if (bxv > gx) continue;
            if (bxv < gx) {
                gx = bxv;
                best = ~0ull;
            }
            while (mx) {
                const int xc = __ffs(mx) - 1;
                mx &= mx - 1;
                int s[ND];
#pragma unroll
                for (int k = 0; k < ND; ++k) {
                    int dx = X[k] - xc, dy = Y[k] - yc, dz = Z[k] - zc;
                    dx += dx < 0 ? Lx : 0;
                    dy += dy < 0 ? Ly : 0;
                    dz += dz < 0 ? Lz : 0;
                    s[k] = SB[k] + L.nsub * (dx + Lx * (dy + Ly * dz));
                }
                sort_net(s);
                uint64_t key = 0;
#pragma unroll
                for (int k = ND - 1; k >= 0; --k) key = (key << kb) | (uint64_t)s[k];
                if (key < best) {
                    best = key;
                    ax = xc;
                    by = yc;
                    cz = zc;
                }
            }
        }
    }
}

// the sorted list of a packed key
template <int ND>
__device__ __forceinline__ void unpack_key(uint64_t key, int kb, int (&rep)[ND]) {
    const uint32_t mask = (1u << kb) - 1u;
#pragma unroll
    for (int k = 0; k < ND; ++k) {
        rep[k] = (int)((uint32_t)key & mask);
        key >>= kb;
    }
}

// the representative of the site list t, by whichever search applies: two spins
// have nothing to gain from the masks (31x32, S^+_q from N_down = 2 without the
// table 1483 us by canon_gen, 1620 by masks)
template <int ND>
__device__ __forceinline__ uint64_t canon(const int (&t)[ND], const LatView &L, const uint32_t *__restrict__ sxyz,
                                          const uint64_t *__restrict__ sC, int (&rep)[ND], int &ax, int &by,
                                          int &cz) {
    if (ND <= 2 || !L.mask_ok) return canon_gen(t, L, sxyz, sC, rep, ax, by, cz);
    int X[ND], Y[ND], Z[ND], SB[ND];
#pragma unroll
    for (int m = 0; m < ND; ++m) {
        const uint32_t p = sxyz[t[m]];
        X[m] = p & 2047u;
        Y[m] = (p >> 11) & 2047u;
        Z[m] = p >> 22;
        SB[m] = L.nsub > 1 ? t[m] % L.nsub : 0;
    }
    uint64_t key;
    canon_mask(X, Y, Z, SB, L, key, ax, by, cz);
    unpack_key(key, L.key_bits, rep);
    return rank_of(rep, sC, L.np1);
}

// prefix of a sorted list used by the index over sigma -- the colex rank of
// its two largest sites (pre2), or its largest site -- and the rank of the
// other sites
template <int ND>
__device__ __forceinline__ uint32_t prefix_of(const int (&c)[ND], const uint64_t *__restrict__ sC, int np1, int pre2,
                                              uint64_t &low) {
    low = 0;
    if constexpr (ND >= 2) {
#pragma unroll
        for (int m = 0; m + 2 < ND; ++m) low += sC[(m + 1) * np1 + c[m]];
        if (pre2) return (uint32_t)(sC[2 * np1 + c[ND - 1]] + (uint64_t)c[ND - 2]);
        low += sC[(ND - 1) * np1 + c[ND - 2]];
    }
    return (uint32_t)c[ND - 1];
}

// the row of rank r among rows lo .. hi - 1 of a sector (a bucket of the
// index): buckets of up to four rows -- nearly all -- are read at once
__device__ __forceinline__ bool bucket_find(const uint64_t *__restrict__ sigma, uint32_t lo, uint32_t hi, uint64_t r,
                                            uint32_t &idx) {
    while (hi - lo > 4u) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__ldg(sigma + mid) <= r) lo = mid; else hi = mid;
    }
    uint64_t v[4];
#pragma unroll
    for (uint32_t i = 0; i < 4; ++i) v[i] = lo + i < hi ? __ldg(sigma + lo + i) : ~0ull;
    bool found = false;
#pragma unroll
    for (uint32_t i = 0; i < 4; ++i)
        if (v[i] == r) {
            found = true;
            idx = lo + i;
        }
    return found;
}

// the largest x with C(x, 2) <= P
__device__ __forceinline__ int tri_root(uint32_t P) {
    int x = (int)(0.5f + sqrtf(0.25f + 2.0f * (float)P));
    while ((uint64_t)x * (x - 1) / 2 > P) --x;
    while ((uint64_t)x * (x + 1) / 2 <= P) ++x;
    return x;
}

// the buckets of prefix P (SecView::pinfo): nq of them, 2^shift low ranks
// each, at most `most`
__device__ __forceinline__ int bucket_shift(uint32_t P, uint32_t most, int nd, int pre2,
                                            const uint64_t *__restrict__ binom, int np1, uint32_t &nq) {
    uint64_t w;                            // low ranks
    if (pre2) {
        const int x = tri_root(P);
        w = binom[(size_t)(nd - 2) * np1 + (P - (uint64_t)x * (x - 1) / 2)];
    } else {
        w = binom[(size_t)(nd - 1) * np1 + P];
    }
    most = most > 1 ? most : 1;
    int sh = 0;
    while (w && ((w - 1) >> sh) + 1 > most) ++sh;
    nq = w ? (uint32_t)(((w - 1) >> sh) + 1) : 1u;
    return sh;
}

// position of the representative c, of rank r, in sector sv
template <int ND>
__device__ __forceinline__ bool sigma_find(const SecView &sv, const int (&c)[ND], const uint64_t *__restrict__ sC,
                                           int np1, uint64_t r, uint32_t &idx) {
    uint64_t low;
    const uint2 pi = __ldg(sv.pinfo + prefix_of(c, sC, np1, sv.pre2, low));
    uint32_t lo = pi.x, hi = pi.x + (pi.y >> 8);
    if (ND > 3 || !(pi.y & ONE_BUCKET)) {
        const uint32_t *e = sv.sub + pi.x + (uint32_t)(low >> pi.y);
        lo = __ldg(e);
        hi = __ldg(e + 1);
    }
    return bucket_find(sv.sigma, lo, hi, r, idx);
}

// stage the binomial table (rows 0..nd+2) and the coordinate table in smem
__device__ __forceinline__ void stage_tables(const LatView &L, uint64_t *sC, uint32_t *sxyz) {
    const int nC = (L.nd + 3) * L.np1;
    for (int i = threadIdx.x; i < nC; i += blockDim.x) sC[i] = L.binom[i];
    if (sxyz)
        for (int i = threadIdx.x; i < L.N; i += blockDim.x) sxyz[i] = L.xyz[i];
}

// entries of every (sector, prefix): its buckets plus the end (ONE: none for one
// bucket, whose rows are in its pinfo)
template <bool ONE>
static __global__ void k_bucket_size(int nd, int np1, int pre2, const uint64_t *__restrict__ binom, int S, uint32_t np,
                              int half, const uint32_t *__restrict__ first, uint32_t *__restrict__ size) {
    const uint64_t cnt = (uint64_t)S * np;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t s = i / np;
        const uint32_t P = (uint32_t)(i - s * np);
        const uint32_t *f = first + s * (np + 1) + P;
        uint32_t nq;
        bucket_shift(P, (f[1] - f[0]) >> half, nd, pre2, binom, np1, nq);
        size[i] = ONE && nq == 1 ? 0 : nq + 1;
    }
}
template <bool ONE>
static __global__ void k_bucket_info(int nd, int np1, int pre2, const uint64_t *__restrict__ binom, int S, uint32_t np,
                              int half, const uint32_t *__restrict__ first, const uint32_t *__restrict__ off,
                              uint2 *__restrict__ pinfo, uint32_t *__restrict__ sub) {
    const uint64_t cnt = (uint64_t)S * np;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t s = i / np;
        const uint32_t P = (uint32_t)(i - s * np);
        const uint32_t *f = first + s * (np + 1) + P;
        uint32_t nq;
        const int sh = bucket_shift(P, (f[1] - f[0]) >> half, nd, pre2, binom, np1, nq);
        if (ONE && nq == 1) {
            pinfo[i] = make_uint2(f[0], ONE_BUCKET | (f[1] - f[0]) << 8);
            continue;
        }
        pinfo[i] = make_uint2(off[i], (uint32_t)sh);
        // an empty prefix: one empty bucket
        if (f[0] == f[1])
            for (uint32_t q = 0; q <= nq; ++q) sub[(uint64_t)off[i] + q] = f[0];
    }
}

size_t row_kernel_smem(const Basis &B, int extra_nd);

// -------------------------------------------------------------- entry points
// implemented in qs3_hphi.cu
int hphi_launch(Basis &B, qs3_dtype dt, const void *phi, void *psi, cudaStream_t st,
                const int *active = nullptr);
// C128DF product: phi in double-float form (float4 per element), or phi +
// (*dx) ld when dx (device) is given; psi complex128, or double-float when out_df
int hphi_df_launch(Basis &B, const void *phi, const int *dx, uint64_t ld, void *psi, cudaStream_t st,
                   const int *active = nullptr, bool out_df = false);
// H Phi of a U(1)-only basis with 32-bit ranks (qs3_hphi_u1.cu); *done = false
// when no kernel there takes it (the caller then runs the general one)
int hphi_u1_launch(Basis &B, qs3_dtype dt, const void *phi, void *psi, cudaStream_t st, const int *active, bool *done);
// the same on momentum sectors by origin forms (qs3_hphi_search.cu), built at
// creation of a basis without a representative table
int build_forms(Basis &B, size_t max_bytes);
int hphi_forms_launch(Basis &B, qs3_dtype dt, const void *phi, void *psi, cudaStream_t st, const int *active);
int count_nnz(Basis &B, uint64_t *nnz);
// the binary64 engine's H Phi on the integer units (qs3_hphi.cu, k_hphi_x and the
// orbit-batched k_hphi_o).  Its input: the gather image hd (hd_pack) and the
// binary64 values, interleaved (phi) or the engine's word-planar slot (plane, D
// elements per word plane; slot *dx of a store when dx is given)
struct HxVec {
    const int4 *hd;
    const double2 *phi;
    const uint2 *plane;
    uint64_t D;
    const int *dx;
#ifdef __CUDACC__
    __device__ __forceinline__ void at_slot() {
        if (dx) plane += (uint64_t)(*dx) * 2 * D;
    }
    __device__ __forceinline__ double2 value(uint64_t i) const {
        if (phi) return phi[i];
        const uint2 h = plane[i], l = plane[D + i];
        return make_double2(__hiloint2double((int)h.x, (int)l.x), __hiloint2double((int)h.y, (int)l.y));
    }
#endif
};
bool hphi_x_ok(const Basis &B);
int hphi_x_launch(Basis &B, const HxVec &hv, void *psi, cudaStream_t st, const int *active = nullptr);
// qs3_hphi with QS3_C128X: phi's image in scratch, then hphi_x_launch
// (qs3_solver.cu, where the digit kernels live); asynchronous on st
int hphi_x_binary64(Basis &B, const void *phi, void *psi, cudaStream_t st);
// representative table: build (QS3_OK, or an error when it cannot be built) / release
int build_rep_table(Basis &B, size_t max_bytes);
// stored-term H Phi of k-sector bases: build (QS3_OK or an error) / release / apply
int build_terms(Basis &B, size_t max_bytes);
void drop_terms(Basis &B);
int hphi_stored_launch(Basis &B, qs3_dtype dt, const void *phi, void *psi, cudaStream_t st, const int *active);
constexpr size_t REP_TABLE_AUTO_BYTES = (size_t)1 << 30;   // built at basis creation up to this size
void drop_rep_table(Basis &B);
// implemented in qs3_obs.cu
int sq_launch(int op, Basis &src, int s_src, const void *phi, Basis &dst, int s_dst, const int *Q, void *psi,
              cudaStream_t st);
int smq_launch(Basis &src, int s_src, const void *phi, Basis &dst, int s_dst, const int *Q, void *psi,
               cudaStream_t st);

}  // namespace qs3

struct qs3_basis_s {
    qs3::Basis B;
};
