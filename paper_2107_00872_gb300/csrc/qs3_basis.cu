// qs3_basis.cu -- lattice ingest and symmetry-adapted basis construction on
// the device (Sec. "Representative states and Hamiltonian matrix elements in
// symmetry-adapted basis sets", Alg. 5-6 of the paper, re-designed).
//
// Instead of testing all C(N, N_down) states with all N translations
// (Alg. 5/6), the device enumerates the C(N-1, N_down-1) states that have a
// down spin at site 0.  Every translation orbit contains such states: the
// translates T^{-pos(c_m)} c that move one of its spins to the origin.  A
// state c emits its orbit's representative exactly once, when c has the
// smallest rank among those origin-containing translates.  The stabiliser
// of c is the set of pos(c_m) whose translate reproduces c, which gives
// |Stab| and the compatibility test e^{ik.t} = 1 on it (N_{a,k} > 0 in
// Alg. 5).  The representatives are sorted by rank (CUB radix sort, a
// library primitive) once for all sectors; each sector takes the compatible
// ones in order.  The rows of every sector are indexed by their largest sites
// and buckets of the rank of the others (SecView::pinfo).
#include <cub/cub.cuh>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <utility>

#include "qs3_internal.cuh"
#include "qs3_fixed.cuh"

namespace qs3 {

// ------------------------------------------------------------ error state
static thread_local char g_err[1024];

int set_err(int code, const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return code;
}

void clear_err() { g_err[0] = 0; }

static std::atomic<unsigned long long> g_launches{0};
void count_launch(long long n) { g_launches.fetch_add((unsigned long long)n, std::memory_order_relaxed); }

const char *last_err() { return g_err; }

void DevBuf::release() {
    if (p) {
        if (pooled) cudaFreeAsync(p, st); else cudaFree(p);
    }
    p = nullptr;
    n = 0;
}

// the pool of the current device (created at its first use, kept by the
// process), nullptr where the device has none
static std::mutex g_pool_mu;
static cudaMemPool_t g_pool[64];
static bool g_pool_tried[64];
static cudaMemPool_t device_pool(bool create) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (!g_pool_tried[dev] && create) {
        g_pool_tried[dev] = true;
        cudaMemPoolProps pr = {};
        pr.allocType = cudaMemAllocationTypePinned;
        pr.location.type = cudaMemLocationTypeDevice;
        pr.location.id = dev;
        cudaMemPool_t mp = nullptr;
        if (cudaMemPoolCreate(&mp, &pr) == cudaSuccess) {
            uint64_t keep = POOL_KEEP_BYTES;
            cudaMemPoolSetAttribute(mp, cudaMemPoolAttrReleaseThreshold, &keep);
            g_pool[dev] = mp;
        }
        cudaGetLastError();
    }
    return g_pool[dev];
}
void pool_trim(size_t keep) {
    if (cudaMemPool_t mp = device_pool(false)) cudaMemPoolTrimTo(mp, keep);
    cudaGetLastError();
}

// allocation fault injection (qs3_inject_alloc_failure): the number of
// allocations still allowed to succeed, or -1 when off
static std::atomic<long long> g_alloc_budget{-1};
static std::atomic<int> g_wait_starve{0};
int take_wait_injection() {
    for (int n = g_wait_starve.load(); n > 0;)
        if (g_wait_starve.compare_exchange_weak(n, n - 1)) return 1;
    return 0;
}

// one allocation against the injected budget (true: refused)
static bool refuse_alloc() {
    for (long long v = g_alloc_budget.load(); v >= 0;) {
        if (v == 0) return true;
        if (g_alloc_budget.compare_exchange_weak(v, v - 1)) break;
    }
    return false;
}

int DevBuf::alloc(size_t bytes) {
    release();
    pooled = false;
    if (bytes == 0) bytes = 16;
    if (refuse_alloc()) return set_err(QS3_ERR_OOM, "device allocation of %zu bytes refused (injected failure)", bytes);
    cudaError_t e = cudaMalloc(&p, bytes);
    if (e == cudaErrorMemoryAllocation) {
        // what the pool holds unused goes back first
        cudaGetLastError();
        pool_trim(0);
        e = cudaMalloc(&p, bytes);
    }
    if (e != cudaSuccess) {
        p = nullptr;
        cudaGetLastError();
        return set_err(e == cudaErrorMemoryAllocation ? QS3_ERR_OOM : QS3_ERR_CUDA, "cudaMalloc(%zu): %s", bytes,
                       cudaGetErrorString(e));
    }
    n = bytes;
    return QS3_OK;
}

int DevBuf::alloc(size_t bytes, cudaStream_t stream) {
    cudaMemPool_t mp = bytes <= POOL_MAX_BYTES ? device_pool(true) : nullptr;
    if (!mp) return alloc(bytes);
    release();
    if (bytes == 0) bytes = 16;
    if (refuse_alloc()) return set_err(QS3_ERR_OOM, "device allocation of %zu bytes refused (injected failure)", bytes);
    cudaError_t e = cudaMallocFromPoolAsync(&p, bytes, mp, stream);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        cudaStreamSynchronize(stream);
        pool_trim(0);
        e = cudaMallocFromPoolAsync(&p, bytes, mp, stream);
    }
    if (e != cudaSuccess) {
        p = nullptr;
        cudaGetLastError();
        return set_err(e == cudaErrorMemoryAllocation ? QS3_ERR_OOM : QS3_ERR_CUDA, "cudaMallocFromPoolAsync(%zu): %s",
                       bytes, cudaGetErrorString(e));
    }
    n = bytes;
    pooled = true;
    st = stream;
    return QS3_OK;
}

int DevBuf::upload(const void *src, size_t bytes) {
    QS3_TRY(alloc(bytes));
    if (bytes) QS3_CUDA(cudaMemcpy(p, src, bytes, cudaMemcpyHostToDevice));
    return QS3_OK;
}

int DevBuf::upload(const void *src, size_t bytes, cudaStream_t stream) {
    QS3_TRY(alloc(bytes, stream));
    // src is pageable: the call returns when it has been read
    if (bytes) QS3_CUDA(cudaMemcpyAsync(p, src, bytes, cudaMemcpyHostToDevice, stream));
    return QS3_OK;
}

// must match carve() in qs3_hphi.cu: binomial rows 0..nd+2, coordinates (k
// only), sqrt table (18 doubles), the current sector's phases (k only)
size_t row_kernel_smem(const Basis &B, int /*extra_nd*/) {
    size_t s = (size_t)(B.nd + 3) * (B.N + 1) * sizeof(uint64_t);
    if (B.has_k) s += (size_t)B.N * sizeof(uint32_t);
    s = (s + 15) & ~(size_t)15;
    s += 18 * sizeof(double);
    s = (s + 15) & ~(size_t)15;
    if (B.has_k) s += (size_t)B.N * 2 * sizeof(double);
    return s;
}

// ------------------------------------------------------ enumeration kernel

// Candidates: the states with a spin at site (cell 0, place s0) and none on
// places below s0 (s0 = the lowest place of the cell that the state
// occupies; with one spin per cell s0 = 0): the other N_down - 1 spins are
// an (N_down - 1)-subset of the M - 1 sites after it in the list of sites
// with place >= s0 (index q -> place s0 + q % w, cell q / w, w = nsub - s0).
// Every orbit has such members (move any spin on place s0 to cell 0); a
// candidate is designated when it has the smallest rank of them, so each
// orbit is taken once, from its designated member, with |Stab| (the moves
// that give the candidate back) and the compatibility of those moves with K.
template <int ND>
__global__ void __launch_bounds__(NTHREADS) k_enum_reps(LatView L, int s0, uint64_t ncand, uint64_t cap,
                                                        unsigned long long *counter, uint64_t *out_rank,
                                                        uint8_t *out_stab) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *sC = (uint64_t *)smem;
    uint32_t *sxyz = (uint32_t *)(sC + (L.nd + 3) * L.np1);
    const int nC = (L.nd + 3) * L.np1;
    for (int i = threadIdx.x; i < nC; i += blockDim.x) sC[i] = L.binom[i];
    for (int i = threadIdx.x; i < L.N; i += blockDim.x) sxyz[i] = L.xyz[i];
    __syncthreads();
    const int Lx = L.L[0], Ly = L.L[1], Lz = L.L[2];
    const int ns = L.nsub, w = ns - s0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t base = (uint64_t)blockIdx.x * blockDim.x; base < ncand; base += stride) {
        const uint64_t j = base + threadIdx.x;
        bool take = false;
        uint64_t rep_rank = 0;
        int st = 0;
        if (j < ncand) {
            int c[ND];
            c[0] = s0;
            if (ND >= 2) {
                constexpr int NM1 = (ND > 1) ? ND - 1 : 1;
                int cc[NM1];
                unrank<NM1>(j, sC, L.np1, cc);
#pragma unroll
                for (int m = 0; m + 1 < ND; ++m) {
                    const int q = cc[m] + 1;
                    c[m + 1] = (w == 1) ? s0 + ns * q : s0 + q % w + ns * (q / w);
                }
            }
            const uint64_t rc = rank_of(c, sC, L.np1);
            int X[ND], Y[ND], Z[ND], SB[ND];
#pragma unroll
            for (int m = 0; m < ND; ++m) {
                uint32_t p = sxyz[c[m]];
                X[m] = p & 2047u;
                Y[m] = (p >> 11) & 2047u;
                Z[m] = p >> 22;
                SB[m] = ns > 1 ? c[m] % ns : 0;
            }
            bool designated = true;
#pragma unroll
            for (int m = 0; m < ND; ++m) {
                if (SB[m] != s0) continue;
                int sl[ND];
#pragma unroll
                for (int q = 0; q < ND; ++q) {
                    int xx = X[q] - X[m]; xx += (xx < 0) ? Lx : 0;
                    int yy = Y[q] - Y[m]; yy += (yy < 0) ? Ly : 0;
                    int zz = Z[q] - Z[m]; zz += (zz < 0) ? Lz : 0;
                    sl[q] = SB[q] + ns * (xx + Lx * (yy + Ly * zz));
                }
                sort_net(sl);
                const uint64_t rm = rank_of(sl, sC, L.np1);
                designated &= (rm >= rc);
                st += rm == rc;
            }
            take = designated;
            if (take) {
                int rep[ND];
                int ax, by, cz;
                rep_rank = canon(c, L, sxyz, sC, rep, ax, by, cz);
            }
        }
        // warp-aggregated slot allocation
        const unsigned mask = __ballot_sync(0xffffffffu, take);
        const int lane = threadIdx.x & 31;
        unsigned long long basepos = 0;
        if (lane == 0 && mask) basepos = atomicAdd(counter, (unsigned long long)__popc(mask));
        basepos = __shfl_sync(0xffffffffu, basepos, 0);
        const unsigned long long pos = basepos + __popc(mask & ((1u << lane) - 1u));
        if (take && pos < cap) {
            out_rank[pos] = rep_rank;
            out_stab[pos] = (uint8_t)st;
        }
    }
}

static int gcd_of(int a, int b) {
    while (b) {
        const int t = a % b;
        a = b;
        b = t;
    }
    return a;
}

// The rows of the sector of momentum K, exactly: the orbits on whose
// stabiliser e^{ik.t} = 1, which by the character sum are (1 / G) sum_t
// e^{ik.t} Fix(t) (for K = 0 Burnside's count of all orbits).  A translation of
// order o moves the sites in cycles of o and fixes C(N / o, N_down / o)
// subsets when o divides N_down, none otherwise.  The translations with o t =
// 0 are the multiples of L_a / g_a along each axis, g_a = gcd(o, L_a), so e^{ik.t}
// sums over them to prod g_a when every g_a divides K_a and to 0 otherwise;
// Moebius inversion over the divisors of o leaves those of order o.
static uint64_t sector_dim(const Basis &B, const int *K) {
    auto moebius = [](int n) {
        int m = 1;
        for (int p = 2; p <= n; ++p) {
            if (n % p) continue;
            n /= p;
            if (n % p == 0) return 0;
            m = -m;
        }
        return m;
    };
    auto killed_by = [&](int o) {
        long long f = 1;
        for (int a = 0; a < 3; ++a) {
            const int g = gcd_of(o, B.L[a]);
            f *= K[a] % g == 0 ? g : 0;
        }
        return f;
    };
    __int128 sum = 0;
    for (int o = 1; o <= B.nd; ++o) {
        if (B.nd % o) continue;
        long long e = 0;
        for (int d = 1; d <= o; ++d)
            if (o % d == 0) e += moebius(o / d) * killed_by(d);
        if (e) sum += (__int128)e * B.binom[(size_t)(B.nd / o) * (B.N + 1) + B.N / o];
    }
    return (uint64_t)(sum / B.ncell);
}
static uint64_t count_orbits(const Basis &B) {
    const int K0[3] = {0, 0, 0};
    return sector_dim(B, K0);
}

// the representatives of all orbits, sorted by rank0, with |Stab|: n of them
template <int ND>
static int enum_orbits(Basis &B, DevBuf &kout, DevBuf &vout, uint64_t &n) {
    const std::vector<uint64_t> &hb = B.binom;
    const size_t smem = (size_t)(B.nd + 3) * (B.N + 1) * 8 + (size_t)B.N * 4;
    QS3_CUDA(cudaFuncSetAttribute(k_enum_reps<ND>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_DYN_SMEM));
    int dev = 0, nsm = 0;
    QS3_CUDA(cudaGetDevice(&dev));
    QS3_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    n = count_orbits(B);
    DevBuf cnt, kin, vin;
    QS3_TRY(cnt.alloc(sizeof(unsigned long long), (cudaStream_t)0));
    QS3_CUDA(cudaMemset(cnt.p, 0, sizeof(unsigned long long)));
    QS3_TRY(kin.alloc(n * 8, (cudaStream_t)0));
    QS3_TRY(vin.alloc(n, (cudaStream_t)0));
    // per lowest occupied place s0 of the cell: C(M - 1, ND - 1) candidates,
    // M = (cells) (nsub - s0); one spin per cell: C(N - 1, ND - 1)
    for (int s0 = 0; s0 < B.nsub; ++s0) {
        const uint64_t M = (uint64_t)B.ncell * (B.nsub - s0);
        const uint64_t nc = (M >= 1 && M - 1 >= (uint64_t)(ND - 1)) ? hb[(size_t)(ND - 1) * (B.N + 1) + (M - 1)] : 0;
        if (!nc) continue;
        const int grid = (int)std::min<uint64_t>((nc + NTHREADS - 1) / NTHREADS, (uint64_t)nsm * 8);
        k_enum_reps<ND><<<grid, NTHREADS, smem>>>(B.lv, s0, nc, n, cnt.as<unsigned long long>(), kin.as<uint64_t>(),
                                                  vin.as<uint8_t>());
        QS3_LAUNCHED();
    }
    QS3_TRY(kout.alloc(n * 8));
    QS3_TRY(vout.alloc(n));
    // ranks are below C(N, N_down): only those bits are sorted
    int bits = 1;
    while (bits < 64 && (hb[(size_t)ND * (B.N + 1) + B.N] >> bits)) ++bits;
    size_t tb = 0;
    QS3_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, tb, kin.as<unsigned long long>(), kout.as<unsigned long long>(),
                                             vin.as<uint8_t>(), vout.as<uint8_t>(), (int64_t)n, 0, bits));
    DevBuf tmp;
    QS3_TRY(tmp.alloc(tb, (cudaStream_t)0));
    QS3_CUDA(cub::DeviceRadixSort::SortPairs(tmp.p, tb, kin.as<unsigned long long>(), kout.as<unsigned long long>(),
                                             vin.as<uint8_t>(), vout.as<uint8_t>(), (int64_t)n, 0, bits));
    uint64_t got = 0;
    QS3_CUDA(cudaMemcpy(&got, cnt.p, sizeof(got), cudaMemcpyDeviceToHost));
    if (got != n)
        return set_err(QS3_ERR_CUDA, "enumerated %llu orbits, %llu expected", (unsigned long long)got,
                       (unsigned long long)n);
    return QS3_OK;
}

// flag[i n + g] = 1 when orbit g belongs to the sector of momentum K[i], i <
// ns: e^{ik.t} = 1 on its stabiliser (N_{a,k} > 0 in Alg. 5).  An orbit with
// a trivial stabiliser belongs to every sector; the others' stabilisers are
// among the moves of one spin onto the spins of its place in the cell.
template <int ND>
__global__ void __launch_bounds__(NTHREADS) k_members(LatView L, const uint64_t *__restrict__ reps,
                                                      const uint8_t *__restrict__ stab, uint64_t n, int ns,
                                                      const int *__restrict__ K, uint32_t *__restrict__ flag) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *sC = (uint64_t *)smem;
    uint32_t *sxyz = (uint32_t *)(sC + (L.nd + 3) * L.np1);
    stage_tables(L, sC, sxyz);
    __syncthreads();
    const int Lx = L.L[0], Ly = L.L[1], Lz = L.L[2], G = L.ncell;
    for (uint64_t g = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; g < n; g += (uint64_t)gridDim.x * blockDim.x) {
        if (__ldg(stab + g) == 1) {
            for (int i = 0; i < ns; ++i) flag[(uint64_t)i * n + g] = 1u;
            continue;
        }
        int c[ND], X[ND], Y[ND], Z[ND], SB[ND];
        unrank(__ldg(reps + g), sC, L.np1, c);
#pragma unroll
        for (int m = 0; m < ND; ++m) {
            const uint32_t p = sxyz[c[m]];
            X[m] = p & 2047u;
            Y[m] = (p >> 11) & 2047u;
            Z[m] = p >> 22;
            SB[m] = L.nsub > 1 ? c[m] % L.nsub : 0;
        }
        // the stabiliser's translations, bit m: the move of spin m onto spin 0
        uint32_t fix = 0;
#pragma unroll
        for (int m = 1; m < ND; ++m) {
            int sl[ND];
            bool same = SB[m] == SB[0];
#pragma unroll
            for (int q = 0; q < ND; ++q) {
                int x = X[q] + X[0] - X[m], y = Y[q] + Y[0] - Y[m], z = Z[q] + Z[0] - Z[m];
                x += x < 0 ? Lx : 0; x -= x >= Lx ? Lx : 0;
                y += y < 0 ? Ly : 0; y -= y >= Ly ? Ly : 0;
                z += z < 0 ? Lz : 0; z -= z >= Lz ? Lz : 0;
                sl[q] = SB[q] + L.nsub * (x + Lx * (y + Ly * z));
            }
            sort_net(sl);
#pragma unroll
            for (int q = 0; q < ND; ++q) same &= sl[q] == c[q];
            fix |= same ? 1u << m : 0u;
        }
        for (int i = 0; i < ns; ++i) {
            const long long Kx = K[3 * i], Ky = K[3 * i + 1], Kz = K[3 * i + 2];
            bool ok = true;
#pragma unroll
            for (int m = 1; m < ND; ++m) {
                const long long num = Kx * (X[m] - X[0]) * (G / Lx) + Ky * (Y[m] - Y[0]) * (G / Ly) +
                                      Kz * (Z[m] - Z[0]) * (G / Lz);
                ok &= !((fix >> m) & 1u) || num % G == 0;
            }
            flag[(uint64_t)i * n + g] = ok ? 1u : 0u;
        }
    }
}

// rows of ns sectors from the scanned flags (pos: ns n + 1 entries): the
// representatives and |Stab| of the members, one sector after another (room
// for cap of them)
__global__ void k_take(const uint32_t *__restrict__ pos, const uint64_t *__restrict__ reps,
                       const uint8_t *__restrict__ stab, uint64_t n, uint64_t cnt, uint64_t cap,
                       uint64_t *__restrict__ sigma, uint8_t *__restrict__ sst) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t p = pos[i];
        if (pos[i + 1] == p || p >= cap) continue;
        const uint64_t g = i % n;
        sigma[p] = reps[g];
        sst[p] = stab[g];
    }
}

// per sector s and prefix P: the first row with a prefix >= P, by a binary
// search over the sector's rows (first[s (np + 1) + P], P <= np)
__global__ void k_first(int nd, int np1, int pre2, const SecView *__restrict__ secs, int S, uint32_t np,
                        const uint64_t *__restrict__ binom, uint32_t *__restrict__ first) {
    const uint64_t cnt = (uint64_t)S * (np + 1);
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += (uint64_t)gridDim.x * blockDim.x) {
        const int s = (int)(i / (np + 1));
        const uint32_t P = (uint32_t)(i - (uint64_t)s * (np + 1));
        const uint64_t *sig = secs[s].sigma;
        uint64_t lo = 0, hi = secs[s].dim;
        if (P == np) {
            lo = hi;
        } else {
            // the smallest rank with prefix P
            uint64_t r;
            if (pre2) {
                const int x = tri_root(P);
                r = binom[(size_t)nd * np1 + x] + binom[(size_t)(nd - 1) * np1 + (P - (uint64_t)x * (x - 1) / 2)];
            } else {
                r = binom[(size_t)nd * np1 + P];
            }
            while (lo < hi) {
                const uint64_t mid = (lo + hi) >> 1;
                if (sig[mid] < r) lo = mid + 1; else hi = mid;
            }
        }
        first[i] = (uint32_t)lo;
    }
}

// the entries of each prefix from its rows: row i writes the buckets that
// start at it (those after its predecessor's up to its own), the last row of
// a prefix also the ones after
template <int ND>
__global__ void __launch_bounds__(NTHREADS) k_bucket_fill(LatView L, const SecView *__restrict__ secs,
                                                          const int *__restrict__ tile0, int S, int t0, int t1,
                                                          uint32_t np, const uint32_t *__restrict__ first,
                                                          const uint2 *__restrict__ pinfo, uint32_t *__restrict__ sub) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *sC = (uint64_t *)smem;
    stage_tables(L, sC, nullptr);
    __syncthreads();
    for (int64_t t = (int64_t)t0 + blockIdx.x; t < t1; t += gridDim.x) {
        const int s = S == 1 ? 0 : sector_of_tile(tile0, S, (int)t);
        const uint64_t row = (uint64_t)(t - secs[s].tile0) * TILE + threadIdx.x;
        if (row >= secs[s].dim) continue;
        const uint64_t *sig = secs[s].sigma;
        int c[ND];
        unrank(sig[row], sC, L.np1, c);
        uint64_t low;
        const uint32_t P = prefix_of(c, sC, L.np1, secs[s].pre2, low);
        const uint32_t *f = first + (uint64_t)s * (np + 1) + P;
        const uint2 pi = pinfo[(uint64_t)s * np + P];
        if (ND <= 3 && (pi.y & ONE_BUCKET)) continue;
        uint32_t *e = sub + pi.x;
        const uint32_t q = (uint32_t)(low >> pi.y);
        uint32_t q0 = 0;
        if (row > f[0]) q0 = (uint32_t)((low - (sig[row] - sig[row - 1])) >> pi.y) + 1;
        for (uint32_t k = q0; k <= q; ++k) e[k] = (uint32_t)row;
        if (row + 1 == f[1]) {
            uint32_t nq;
            bucket_shift(P, (f[1] - f[0]) >> 1, L.nd, secs[s].pre2, L.binom, L.np1, nq);
            for (uint32_t k = q + 1; k <= nq; ++k) e[k] = (uint32_t)(row + 1);
        }
    }
}

// The sectors of a k-sector basis (B.dims set, each below 2^32): the orbits
// are enumerated and sorted once, and each sector takes the compatible ones in
// order (a flag per orbit and sector, scanned), as many sectors at a time as
// 2^27 flags hold and at least one, whose rows 32-bit positions number.
// keep_reps / keep_stab receive the orbits' list for the representative table.
template <int ND>
static int build_sectors_nd(Basis &B, DevBuf &keep_reps, DevBuf &keep_stab, uint64_t &n) {
    QS3_TRY(enum_orbits<ND>(B, keep_reps, keep_stab, n));
    const int S = B.S;
    if (S == 1 && B.dims[0] == n) {
        // every orbit; the table's copy is made when there may be one
        if (n < (1ull << 20)) {
            QS3_TRY(B.d_sigma.alloc(n * 8));
            QS3_TRY(B.d_stab.alloc(n));
            QS3_CUDA(cudaMemcpyAsync(B.d_sigma.p, keep_reps.p, n * 8, cudaMemcpyDeviceToDevice));
            QS3_CUDA(cudaMemcpyAsync(B.d_stab.p, keep_stab.p, n, cudaMemcpyDeviceToDevice));
        } else {
            B.d_sigma = std::move(keep_reps);
            B.d_stab = std::move(keep_stab);
        }
        return QS3_OK;
    }
    const size_t smem = (size_t)(B.nd + 3) * (B.N + 1) * 8 + (size_t)B.N * 4;
    QS3_CUDA(cudaFuncSetAttribute(k_members<ND>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_DYN_SMEM));
    uint64_t total = 0;
    for (uint64_t d : B.dims) total += d;
    QS3_TRY(B.d_sigma.alloc(total * 8));
    QS3_TRY(B.d_stab.alloc(total));
    DevBuf pos, tmp;
    const int grp = (int)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)S, (1ull << 27) / std::max<uint64_t>(n, 1)));
    QS3_TRY(pos.alloc(((uint64_t)grp * n + 1) * 4, (cudaStream_t)0));
    size_t tb = 0;
    QS3_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tb, pos.as<uint32_t>(), pos.as<uint32_t>(), (int64_t)((uint64_t)grp * n + 1)));
    QS3_TRY(tmp.alloc(tb, (cudaStream_t)0));
    uint64_t off = 0;
    for (int s0 = 0; s0 < S; s0 += grp) {
        const int ns = std::min(grp, S - s0);
        const uint64_t cnt = (uint64_t)ns * n;
        uint64_t rows = 0;
        for (int s = s0; s < s0 + ns; ++s) rows += B.dims[s];
        const int g1 = (int)std::max<uint64_t>(1, std::min<uint64_t>((n + NTHREADS - 1) / NTHREADS, 4096));
        QS3_CUDA(cudaMemsetAsync(pos.as<uint32_t>() + cnt, 0, 4));
        k_members<ND><<<g1, NTHREADS, smem>>>(B.lv, keep_reps.as<uint64_t>(), keep_stab.as<uint8_t>(), n, ns,
                                              B.K_d + 3 * s0, pos.as<uint32_t>());
        QS3_LAUNCHED();
        size_t t2 = tb;
        QS3_CUDA(cub::DeviceScan::ExclusiveSum(tmp.p, t2, pos.as<uint32_t>(), pos.as<uint32_t>(), (int64_t)(cnt + 1)));
        const int g2 = (int)std::max<uint64_t>(1, std::min<uint64_t>((cnt + 255) / 256, 16384));
        k_take<<<g2, 256>>>(pos.as<uint32_t>(), keep_reps.as<uint64_t>(), keep_stab.as<uint8_t>(), n, cnt, rows,
                            B.d_sigma.as<uint64_t>() + off, B.d_stab.as<uint8_t>() + off);
        QS3_LAUNCHED();
        uint32_t end = 0;
        QS3_CUDA(cudaMemcpy(&end, pos.as<uint32_t>() + cnt, 4, cudaMemcpyDeviceToHost));
        if (end != rows)
            return set_err(QS3_ERR_CUDA, "%u rows of sectors %d .. %d, %llu expected", end, s0, s0 + ns - 1,
                           (unsigned long long)rows);
        off += rows;
    }
    return QS3_OK;
}

// the sectors' views as the kernels read them
static int put_secs(Basis &B) {
    QS3_CUDA(cudaMemcpy(B.d_secs.p, B.secs.data(), B.secs.size() * sizeof(SecView), cudaMemcpyHostToDevice));
    return QS3_OK;
}

// the index over every sector's rows (SecView::pinfo, sub), as many sectors at
// a time as INDEX_GROUP entries hold and at least one: the offsets in a group
// are 32 bits (a sector of fewer than 2^32 rows has fewer than 3 2^30 + 2 np
// entries), the groups' places in d_sub 64
constexpr uint64_t INDEX_GROUP = (uint64_t)1 << 22;
template <int ND>
static int build_index_nd(Basis &B) {
    const int S = B.S;
    // two-site prefixes unless that makes many more prefixes than rows
    const uint64_t np2 = (uint64_t)B.N * (B.N - 1) / 2;
    const int pre2 = ND >= 2 && (uint64_t)S * np2 / 8 <= B.total ? 1 : 0;
    const uint32_t np = pre2 ? (uint32_t)np2 : (uint32_t)B.N;
    for (auto &v : B.secs) v.pre2 = pre2;
    QS3_TRY(put_secs(B));
    // at most rows / 2 buckets and the end for a prefix of four rows or more, two
    // entries for the others (ONE: none)
    constexpr bool ONE = ND <= 3;
    auto entries = [&](int s) { return B.dims[s] / 4 * 3 + 4 + (ONE ? 0 : 2 * (uint64_t)np); };
    std::vector<int> g0{0};
    uint64_t most = 0, in_group = 0, cnt_max = 0;
    for (int s = 0; s < S; ++s) {
        if (s > g0.back() && in_group + entries(s) > INDEX_GROUP) {
            g0.push_back(s);
            in_group = 0;
        }
        in_group += entries(s);
        most += entries(s);
        cnt_max = std::max(cnt_max, (uint64_t)(s + 1 - g0.back()) * np);
    }
    g0.push_back(S);
    QS3_TRY(B.d_pinfo.alloc(std::max<uint64_t>((uint64_t)S * np, 1) * sizeof(uint2)));
    QS3_TRY(B.d_sub.alloc(std::max<uint64_t>(most, 1) * 4));
    DevBuf first, size, off, tmp;
    QS3_TRY(first.alloc((cnt_max + S) * 4, (cudaStream_t)0));
    QS3_TRY(size.alloc((cnt_max + 1) * 4, (cudaStream_t)0));
    QS3_TRY(off.alloc((cnt_max + 1) * 4, (cudaStream_t)0));
    size_t tb = 0;
    QS3_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tb, size.as<uint32_t>(), off.as<uint32_t>(), (int64_t)(cnt_max + 1)));
    QS3_TRY(tmp.alloc(tb, (cudaStream_t)0));
    const size_t smem = (size_t)(B.nd + 3) * (B.N + 1) * 8;
    QS3_CUDA(cudaFuncSetAttribute(k_bucket_fill<ND>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_DYN_SMEM));
    const uint64_t *bin = B.lv.binom;
    uint64_t base = 0;
    for (size_t g = 0; g + 1 < g0.size(); ++g) {
        const int s0 = g0[g], ns = g0[g + 1] - s0;
        const uint64_t cnt = (uint64_t)ns * np;
        const int g1 = (int)std::max<uint64_t>(1, std::min<uint64_t>((cnt + ns + 255) / 256, 16384));
        const SecView *secs = B.d_secs.as<SecView>() + s0;
        uint2 *pinfo = B.d_pinfo.as<uint2>() + (uint64_t)s0 * np;
        uint32_t *sub = B.d_sub.as<uint32_t>() + base;
        k_first<<<g1, 256>>>(B.nd, B.N + 1, pre2, secs, ns, np, bin, first.as<uint32_t>());
        QS3_LAUNCHED();
        QS3_CUDA(cudaMemsetAsync(size.as<uint32_t>() + cnt, 0, 4));
        k_bucket_size<ONE><<<g1, 256>>>(B.nd, B.N + 1, pre2, bin, ns, np, 1, first.as<uint32_t>(), size.as<uint32_t>());
        QS3_LAUNCHED();
        size_t t2 = tb;
        QS3_CUDA(cub::DeviceScan::ExclusiveSum(tmp.p, t2, size.as<uint32_t>(), off.as<uint32_t>(), (int64_t)(cnt + 1)));
        k_bucket_info<ONE><<<g1, 256>>>(B.nd, B.N + 1, pre2, bin, ns, np, 1, first.as<uint32_t>(), off.as<uint32_t>(), pinfo, sub);
        QS3_LAUNCHED();
        const int t0 = B.tile0[s0], t1 = B.tile0[s0 + ns];
        if (t1 > t0) {
            k_bucket_fill<ND><<<std::min(t1 - t0, 8192), NTHREADS, smem>>>(B.lv, secs, B.tile0_d + s0, ns, t0, t1,
                                                                           np, first.as<uint32_t>(), pinfo, sub);
            QS3_LAUNCHED();
        }
        for (int s = s0; s < s0 + ns; ++s) {
            B.secs[s].pinfo = B.d_pinfo.as<uint2>() + (uint64_t)s * np;
            B.secs[s].sub = sub;
            base += entries(s);
        }
    }
    return QS3_OK;
}

#define QS3_ND_CALL(nd, CALL)                                            \
    switch (nd) {                                                        \
        case 1: return CALL(1);                                          \
        case 2: return CALL(2);                                          \
        case 3: return CALL(3);                                          \
        case 4: return CALL(4);                                          \
        case 5: return CALL(5);                                          \
        case 6: return CALL(6);                                          \
        case 7: return CALL(7);                                          \
        case 8: return CALL(8);                                          \
        default: return set_err(QS3_ERR_INVALID_ARG, "n_down %d", (nd)); \
    }

static int build_sectors(Basis &B, DevBuf &reps, DevBuf &stab, uint64_t &n) {
#define QS3_CALL(k) build_sectors_nd<k>(B, reps, stab, n)
    QS3_ND_CALL(B.nd, QS3_CALL)
#undef QS3_CALL
}

static int build_index(Basis &B) {
#define QS3_CALL(k) build_index_nd<k>(B)
    QS3_ND_CALL(B.nd, QS3_CALL)
#undef QS3_CALL
}

// ---------------------------------------------------- representative table
// For lattices whose C(N, N_down) states fit a 4-byte-per-state table, the
// result of the representative search of Alg. 7 for every state is tabulated
// once: orb[rank0(a)] = g << 12 | u with a = T_u (rep_g).  A hop target then
// costs one rank and two table loads instead of the search and the binary
// search in sigma.  It is the same function: where several translations reach
// the representative (a non-trivial stabiliser) they differ by a stabiliser
// element, whose phase is 1 on every sector that holds the representative.

// orb[rank0(T_u rep_g)] = g << 12 | u for every orbit g and translation u
template <int ND>
__global__ void __launch_bounds__(NTHREADS) k_orbit_fill(LatView L, const uint64_t *__restrict__ reps, uint64_t n,
                                                         uint32_t *__restrict__ orb) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *sC = (uint64_t *)smem;
    uint32_t *sxyz = (uint32_t *)(sC + (L.nd + 3) * L.np1);
    const int nC = (L.nd + 3) * L.np1;
    for (int i = threadIdx.x; i < nC; i += blockDim.x) sC[i] = L.binom[i];
    for (int i = threadIdx.x; i < L.N; i += blockDim.x) sxyz[i] = L.xyz[i];
    __syncthreads();
    const int Lx = L.L[0], Ly = L.L[1], Lz = L.L[2], G = L.ncell, ns = L.nsub;
    const uint64_t total = n * (uint64_t)G;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t g = i / (uint64_t)G;
        const int u = (int)(i - g * (uint64_t)G);         // cell translation
        int c[ND];
        unrank(reps[g], sC, L.np1, c);
        const uint32_t pu = sxyz[u * ns];                  // the coordinates of cell u
        const int ux = pu & 2047u, uy = (pu >> 11) & 2047u, uz = pu >> 22;
        int t[ND];
#pragma unroll
        for (int m = 0; m < ND; ++m) {
            const uint32_t p = sxyz[c[m]];
            int x = (int)(p & 2047u) + ux, y = (int)((p >> 11) & 2047u) + uy, z = (int)(p >> 22) + uz;
            x -= (x >= Lx) ? Lx : 0;
            y -= (y >= Ly) ? Ly : 0;
            z -= (z >= Lz) ? Lz : 0;
            t[m] = c[m] % ns + ns * (x + Lx * (y + Ly * z));
        }
        sort_net(t);
        orb[rank_of(t, sC, L.np1)] = ((uint32_t)g << 12) | (uint32_t)u;
    }
}

// t2[s n + g] = row of representative g in sector s, -1 if the sector lacks it
__global__ void k_orbit_rows(const SecView *__restrict__ secs, int S, const uint64_t *__restrict__ reps, uint64_t n,
                             int32_t *__restrict__ t2) {
    const uint64_t total = n * (uint64_t)S;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const int s = (int)(i / n);
        const uint64_t g = i - (uint64_t)s * n;
        const uint64_t r = reps[g];
        const uint64_t *sig = secs[s].sigma;
        uint64_t lo = 0, hi = secs[s].dim;
        while (lo < hi) {
            const uint64_t mid = (lo + hi) >> 1;
            if (sig[mid] < r) lo = mid + 1; else hi = mid;
        }
        t2[i] = (lo < secs[s].dim && sig[lo] == r) ? (int32_t)lo : -1;
    }
}

// the per-site phases of every sector as fixed-point digits on the grid
// 2^-52 (re.P1, re.P0, im.P1, im.P0), for the integer H Phi
__global__ void k_phase_digits(const double2 *__restrict__ ph64, uint64_t n, int4 *__restrict__ out) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const double2 p = ph64[i];
        int a1, a0, b1, b0;
        fx_digits((uint32_t)__double2hiint(p.x), (uint32_t)__double2loint(p.x), 1023, a1, a0);
        fx_digits((uint32_t)__double2hiint(p.y), (uint32_t)__double2loint(p.y), 1023, b1, b0);
        out[i] = make_int4(a1, a0, b1, b0);
    }
}

// reps / stab: the orbits' list when the caller has it (n of them; taken over), else empty
template <int ND>
static int build_table_nd(Basis &B, size_t max_bytes, DevBuf &reps, DevBuf &stab, uint64_t n) {
    const uint64_t ns = B.binom[(size_t)ND * (B.N + 1) + B.N];     // C(N, N_down)
    if (ns >= (1ull << 32)) return set_err(QS3_ERR_OVERFLOW, "C(N, N_down) = %llu states: no table", (unsigned long long)ns);
    const uint64_t n_est = ns / (uint64_t)B.ncell + 1;             // orbits, about C(N, N_down) / (cells)
    if (ns * 4 + n_est * 4 * (uint64_t)B.S > max_bytes)
        return set_err(QS3_ERR_OOM, "representative table of ~%llu bytes exceeds the limit",
                       (unsigned long long)(ns * 4 + n_est * 4 * (uint64_t)B.S));
    if (!reps.p) {
        n = count_orbits(B);
        if (n < (1ull << 20)) QS3_TRY(enum_orbits<ND>(B, reps, stab, n));
    }
    int dev = 0, nsm = 0;
    QS3_CUDA(cudaGetDevice(&dev));
    QS3_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    if (n >= (1ull << 20)) return set_err(QS3_ERR_OVERFLOW, "%llu orbits exceed the table's 20-bit index", (unsigned long long)n);
    if (ns * 4 + n * 4 * (uint64_t)B.S > max_bytes)
        return set_err(QS3_ERR_OOM, "representative table exceeds the limit");
    DevBuf orb, t2;
    QS3_TRY(orb.alloc(ns * 4));
    QS3_TRY(t2.alloc(n * 4 * (uint64_t)B.S));
    QS3_CUDA(cudaMemset(orb.p, 0xff, ns * 4));
    const size_t smem = (size_t)(B.nd + 3) * (B.N + 1) * 8 + (size_t)B.N * 4;
    QS3_CUDA(cudaFuncSetAttribute(k_orbit_fill<ND>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_DYN_SMEM));
    const uint64_t tot = n * (uint64_t)B.ncell;
    int grid = (int)std::min<uint64_t>((tot + NTHREADS - 1) / NTHREADS, (uint64_t)nsm * 8);
    k_orbit_fill<ND><<<std::max(grid, 1), NTHREADS, smem>>>(B.lv, reps.as<uint64_t>(), n, orb.as<uint32_t>());
    QS3_LAUNCHED();
    const uint64_t tot2 = n * (uint64_t)B.S;
    int grid2 = (int)std::min<uint64_t>((tot2 + 255) / 256, (uint64_t)nsm * 8);
    k_orbit_rows<<<std::max(grid2, 1), 256>>>(B.d_secs.as<SecView>(), B.S, reps.as<uint64_t>(), n, t2.as<int32_t>());
    QS3_LAUNCHED();
    DevBuf phd;
    const uint64_t nph = (uint64_t)B.S * B.N;
    QS3_TRY(phd.alloc(nph * sizeof(int4)));
    k_phase_digits<<<(int)std::min<uint64_t>((nph + 255) / 256, 4096), 256>>>(B.secs[0].ph64, nph, phd.as<int4>());
    QS3_LAUNCHED();
    QS3_CUDA(cudaDeviceSynchronize());
    B.d_orb = std::move(orb);
    B.d_t2 = std::move(t2);
    B.d_oreps = std::move(reps);
    B.d_ostab = std::move(stab);
    B.d_phdig = std::move(phd);
    B.n_orb = n;
    B.lv.orb = B.d_orb.as<uint32_t>();
    B.lv.n_orb = (uint32_t)n;
    for (int s = 0; s < B.S; ++s) B.secs[s].t2 = B.d_t2.as<int32_t>() + (size_t)s * n;
    return put_secs(B);                      // after the wait: no kernel reads the old views
}

static int build_rep_table(Basis &B, size_t max_bytes, DevBuf &reps, DevBuf &stab, uint64_t n) {
    if (!B.has_k || B.nd == 0 || B.total == 0) return set_err(QS3_ERR_STATE, "the table serves k-sector bases only");
    if (B.N > 4096) return set_err(QS3_ERR_OVERFLOW, "N > 4096");
    if (B.lv.orb) return QS3_OK;
#define QS3_CALL(k) build_table_nd<k>(B, max_bytes, reps, stab, n)
    QS3_ND_CALL(B.nd, QS3_CALL)
#undef QS3_CALL
}

int build_rep_table(Basis &B, size_t max_bytes) {
    DevBuf reps, stab;
    return build_rep_table(B, max_bytes, reps, stab, 0);
}

void drop_rep_table(Basis &B) {
    B.lv.orb = nullptr;
    B.lv.n_orb = 0;
    for (auto &v : B.secs) v.t2 = nullptr;
    B.d_orb.release();
    B.d_t2.release();
    B.d_oreps.release();
    B.d_ostab.release();
    B.d_phdig.release();
    B.n_orb = 0;
    if (!B.secs.empty()) B.d_secs.upload(B.secs.data(), B.secs.size() * sizeof(SecView));
}

// the origin forms (qs3_hphi_search.cu); drop_rep_table then puts the views
static void drop_forms(Basis &B) {
    for (auto &v : B.secs) {
        v.orec = nullptr;
        v.finfo = nullptr;
        v.fsub = nullptr;
    }
    B.d_orec.release();
    B.d_finfo.release();
    B.d_fsub.release();
}

// per-sector phase tables ph[s N + r] = exp(-2 pi i sum_alpha K_alpha r_alpha / L_alpha):
// the phase e^{ik.t} of the translation t = -(r_x, r_y, r_z) that moves site r
// to the origin; the angle is reduced exactly in integers
// per sector s and cell translation u (u < G = Lx Ly Lz; rows of N entries,
// the entries past G repeat the table): e^{-2 pi i K.t_u / L} with the angle
// reduced exactly in integers
__global__ void k_phase_tables(int S, int N, int G, int Lx, int Ly, int Lz, const int *__restrict__ K,
                               double2 *__restrict__ ph64, float2 *__restrict__ ph32, float4 *__restrict__ phdf) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= S * N) return;
    const int s = i / N, r = (i % N) % G;
    const long long x = r % Lx, y = (r / Lx) % Ly, z = r / (Lx * Ly);
    const long long num =
        ((long long)K[3 * s] * x * (G / Lx) + (long long)K[3 * s + 1] * y * (G / Ly) + (long long)K[3 * s + 2] * z * (G / Lz)) % G;
    double sn, cs;
    sincospi(-2.0 * (double)num / (double)G, &sn, &cs);
    ph64[i] = make_double2(cs, sn);
    ph32[i] = make_float2((float)cs, (float)sn);
    const float ch = __double2float_rn(cs), sh = __double2float_rn(sn);
    phdf[i] = make_float4(ch, __double2float_rn(cs - (double)ch), sh, __double2float_rn(sn - (double)sh));
}

__global__ void k_roots(int G, double2 *__restrict__ w) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= G) return;
    double sn, cs;
    sincospi(-2.0 * (double)n / (double)G, &sn, &cs);
    w[n] = make_double2(cs, sn);
}

// ---------------------------------------------------------------- host side

// tables laid out one after another, each on a 16-byte boundary
struct TableImage {
    std::vector<unsigned char> data;
    template <class T> size_t add(const std::vector<T> &v) {
        const size_t at = data.size();
        data.resize((at + v.size() * sizeof(T) + 15) & ~(size_t)15);
        if (!v.empty()) std::memcpy(data.data() + at, v.data(), v.size() * sizeof(T));
        return at;
    }
};

static bool binom_table(int N, int rows, std::vector<uint64_t> &t, uint64_t *cnd, int nd) {
    // t[m * (N+1) + c] = C(c, m), saturated at UINT64_MAX; returns false if C(N, nd) >= 2^63
    t.assign((size_t)rows * (N + 1), 0);
    for (int c = 0; c <= N; ++c) t[c] = 1;
    const uint64_t SAT = ~0ull;
    for (int m = 1; m < rows; ++m)
        for (int c = 1; c <= N; ++c) {
            uint64_t a = t[(size_t)(m - 1) * (N + 1) + c - 1], b = t[(size_t)m * (N + 1) + c - 1];
            uint64_t s = (a == SAT || b == SAT || a + b < a) ? SAT : a + b;
            t[(size_t)m * (N + 1) + c] = s;
        }
    *cnd = t[(size_t)nd * (N + 1) + N];
    return *cnd < (1ull << 63);
}

static int check_translation(const Basis &B) {
    // bonds as an unordered-pair multiset with summed couplings
    std::map<std::pair<int, int>, std::pair<double, double>> bonds;
    for (int b = 0; b < B.nb; ++b) {
        int i = std::min(B.bi[b], B.bj[b]), j = std::max(B.bi[b], B.bj[b]);
        auto &v = bonds[{i, j}];
        v.first += B.jxy[b];
        v.second += B.jz[b];
    }
    const int Lx = B.L[0], Ly = B.L[1], ns = B.nsub;
    // site r = spin r % ns of cell r / ns; the shift moves the cell by one along axis a
    auto shift = [&](int r, int a) {
        const int sb = r % ns, q = r / ns;
        int x = q % Lx, y = (q / Lx) % Ly, z = q / (Lx * Ly);
        if (a == 0) x = (x + 1) % Lx;
        if (a == 1) y = (y + 1) % Ly;
        if (a == 2) z = (z + 1) % B.L[2];
        return sb + ns * (x + Lx * (y + Ly * z));
    };
    for (int a = 0; a < 3; ++a) {
        if (B.L[a] == 1) continue;
        for (auto &kv : bonds) {
            int i = shift(kv.first.first, a), j = shift(kv.first.second, a);
            auto it = bonds.find({std::min(i, j), std::max(i, j)});
            if (it == bonds.end() || std::fabs(it->second.first - kv.second.first) > 1e-12 ||
                std::fabs(it->second.second - kv.second.second) > 1e-12)
                return set_err(QS3_ERR_SYMMETRY, "bond (%d,%d) is not invariant under the translation along axis %d",
                               kv.first.first, kv.first.second, a);
        }
    }
    // the field must be the same on every copy of a spin of the unit cell
    if (B.has_h)
        for (int i = 1; i < B.N; ++i)
            if (B.h[i] != B.h[i % ns]) return set_err(QS3_ERR_SYMMETRY, "site field is not translation invariant (site %d)", i);
    return QS3_OK;
}

static int basis_create(const qs3_lattice *lat, int nd, int nsec, const int32_t *K, Basis &B) {
    if (!lat) return set_err(QS3_ERR_INVALID_ARG, "lattice is NULL");
    const int N = lat->n_sites, nb = lat->n_bonds;
    if (N < 1 || N > QS3_MAX_SITES) return set_err(QS3_ERR_OVERFLOW, "n_sites %d outside [1, %d]", N, QS3_MAX_SITES);
    if (nd < 0 || nd > QS3_MAX_NDOWN || nd > N)
        return set_err(nd > QS3_MAX_NDOWN ? QS3_ERR_OVERFLOW : QS3_ERR_INVALID_ARG, "n_down %d", nd);
    if (nb < 0 || (nb > 0 && (!lat->bi || !lat->bj || !lat->jxy || !lat->jz)))
        return set_err(QS3_ERR_INVALID_ARG, "bond arrays");
    if (nsec < 1) return set_err(QS3_ERR_INVALID_ARG, "n_sectors %d", nsec);
    if (!K && nsec != 1) return set_err(QS3_ERR_INVALID_ARG, "a U(1)-only basis has exactly one sector");
    B.N = N;
    B.nd = nd;
    B.nb = nb;
    B.bi.assign(lat->bi, lat->bi + nb);
    B.bj.assign(lat->bj, lat->bj + nb);
    B.jxy.assign(lat->jxy, lat->jxy + nb);
    B.jz.assign(lat->jz, lat->jz + nb);
    for (int b = 0; b < nb; ++b) {
        if (B.bi[b] < 0 || B.bi[b] >= N || B.bj[b] < 0 || B.bj[b] >= N || B.bi[b] == B.bj[b])
            return set_err(QS3_ERR_INVALID_ARG, "bond %d joins (%d, %d)", b, B.bi[b], B.bj[b]);
        if (!std::isfinite(B.jxy[b]) || !std::isfinite(B.jz[b]))
            return set_err(QS3_ERR_INVALID_ARG, "bond %d has a non-finite coupling", b);
    }
    B.has_h = lat->h != nullptr;
    if (B.has_h) B.h.assign(lat->h, lat->h + N);
    for (int a = 0; a < 3; ++a) B.L[a] = lat->L[a];
    const bool haveL = B.L[0] > 0 || B.L[1] > 0 || B.L[2] > 0;
    B.nsub = lat->n_sub > 0 ? lat->n_sub : 1;
    if (haveL) {
        for (int a = 0; a < 3; ++a)
            if (B.L[a] < 1 || B.L[a] > (a == 2 ? 1023 : 2047))
                return set_err(QS3_ERR_INVALID_ARG, "L[%d] = %d outside the coordinate range", a, B.L[a]);
        if ((long long)B.nsub * B.L[0] * B.L[1] * B.L[2] != N)
            return set_err(QS3_ERR_INVALID_ARG, "n_sub*Lx*Ly*Lz = %lld != n_sites %d",
                           (long long)B.nsub * B.L[0] * B.L[1] * B.L[2], N);
    } else {
        if (B.nsub != 1) return set_err(QS3_ERR_INVALID_ARG, "n_sub %d without a translation group", B.nsub);
        if (N > 2047 && K) return set_err(QS3_ERR_INVALID_ARG, "translation group needed");
    }
    B.has_k = K != nullptr;
    B.S = nsec;
    if (B.has_k) {
        if (!haveL) return set_err(QS3_ERR_SYMMETRY, "momentum sectors need a translation group L");
        B.K.assign(K, K + 3 * nsec);
        for (int s = 0; s < nsec; ++s)
            for (int a = 0; a < 3; ++a)
                if (B.K[3 * s + a] < 0 || B.K[3 * s + a] >= B.L[a])
                    return set_err(QS3_ERR_SYMMETRY, "K[%d][%d] = %d outside [0, %d)", s, a, B.K[3 * s + a], B.L[a]);
        QS3_TRY(check_translation(B));
    } else {
        B.K.assign(3, 0);
    }
    if (!haveL) { B.L[0] = N; B.L[1] = 1; B.L[2] = 1; }
    B.ncell = B.L[0] * B.L[1] * B.L[2];
    if (lat->pos) B.pos.assign(lat->pos, lat->pos + 3 * (size_t)N);

    // binomial rows 0..nd+2
    std::vector<uint64_t> tb;
    uint64_t cnd = 0;
    if (!binom_table(N, nd + 3, tb, &cnd, nd))
        return set_err(QS3_ERR_OVERFLOW, "C(%d, %d) does not fit in 63 bits", N, nd);
    B.binom = std::move(tb);

    // the sectors' rows, and what they are limited to, before anything is allocated
    B.dims.assign(nsec, 0);
    B.offs.assign(nsec + 1, 0);
    B.tile0.assign(nsec + 1, 0);
    B.chunk0.assign(nsec + 1, 0);
    for (int s = 0; s < nsec; ++s) {
        const int *k = &B.K[3 * s];
        if (!B.has_k) B.dims[s] = cnd;
        else if (nd == 0) B.dims[s] = k[0] == 0 && k[1] == 0 && k[2] == 0 ? 1 : 0;   // the vacuum
        else B.dims[s] = sector_dim(B, k);
        if (B.has_k && B.dims[s] >= (1ull << 32))
            return set_err(QS3_ERR_OVERFLOW, "sector dimension %llu exceeds 2^32", (unsigned long long)B.dims[s]);
        B.offs[s + 1] = B.offs[s] + B.dims[s];
        const uint64_t nt = (B.dims[s] + TILE - 1) / TILE;
        if ((uint64_t)B.tile0[s] + nt > (1ull << 31) - 1) return set_err(QS3_ERR_OVERFLOW, "too many rows");
        B.tile0[s + 1] = B.tile0[s] + (int)nt;
        B.chunk0[s + 1] = B.chunk0[s] + (int)((B.dims[s] + BROWS - 1) / BROWS);
    }
    B.total = B.offs[nsec];
    B.ntiles = B.tile0[nsec];
    B.nchunks = B.chunk0[nsec];

    // every table of the lattice and of the sectors in one device image (one
    // allocation and one copy: a basis of few rows is bound by those)
    TableImage img;
    const size_t o_binom = img.add(B.binom);

    // adjacency (CSR, both directions), diagonal constants
    std::vector<int> deg(N + 1, 0);
    for (int b = 0; b < nb; ++b) { deg[B.bi[b] + 1]++; deg[B.bj[b] + 1]++; }
    B.max_degree = 0;
    for (int i = 0; i < N; ++i) B.max_degree = std::max(B.max_degree, deg[i + 1]);
    for (int i = 0; i < N; ++i) deg[i + 1] += deg[i];
    std::vector<int> nbr(2 * (size_t)nb), fill(deg.begin(), deg.end() - 1);
    std::vector<double> ajxy(2 * (size_t)nb), ajz(2 * (size_t)nb), u(N, 0.0);
    std::vector<float> ajxyf(2 * (size_t)nb);
    double c0 = 0.0;
    for (int b = 0; b < nb; ++b) {
        int i = B.bi[b], j = B.bj[b];
        int p = fill[i]++, q = fill[j]++;
        nbr[p] = j; nbr[q] = i;
        ajxy[p] = ajxy[q] = 0.5 * B.jxy[b];            // hop amplitude J^xy / 2 of Eq. (1)
        ajz[p] = ajz[q] = B.jz[b];
        ajxyf[p] = ajxyf[q] = (float)(0.5 * B.jxy[b]);
        u[i] -= 0.5 * B.jz[b];
        u[j] -= 0.5 * B.jz[b];
        c0 += 0.25 * B.jz[b];
    }
    if (B.has_h)
        for (int i = 0; i < N; ++i) { u[i] += B.h[i]; c0 -= 0.5 * B.h[i]; }
    const std::vector<float> uf(u.begin(), u.end()), ajzf(ajz.begin(), ajz.end());
    // double-float remainders (v - fl32(v), rounded to fp32)
    auto rem = [](const std::vector<double> &v, const std::vector<float> &h) {
        std::vector<float> r(v.size());
        for (size_t i = 0; i < v.size(); ++i) r[i] = (float)(v[i] - (double)h[i]);
        return r;
    };
    const size_t o_ptr = img.add(deg), o_nbr = img.add(nbr), o_jxy = img.add(ajxy), o_jz = img.add(ajz),
                 o_jxyf = img.add(ajxyf), o_u = img.add(u), o_uf = img.add(uf), o_jzf = img.add(ajzf),
                 o_jxyl = img.add(rem(ajxy, ajxyf)), o_ul = img.add(rem(u, uf)), o_jzl = img.add(rem(ajz, ajzf));
    for (int b = 0; b < nb; ++b) B.n_long_bonds += std::abs(B.bi[b] - B.bj[b]) * SEG_REACH > N;
    // fixed-width copies of the adjacency for the U(1) kernels
    const int padw = K ? 0 : B.max_degree <= 2 ? 2 : B.max_degree <= 4 ? 4 : (B.max_degree <= 6 ? 6 : 0);
    const size_t np = (size_t)N * padw;
    size_t o_pad = 0;
    if (padw) {
        // int4 | fp64 J^z | int2 | int2 transposed | fp32 J^z | fp32 J^z transposed
        std::vector<int4> pad(np * 3);
        int4 *p64 = pad.data();
        double *z64 = (double *)(p64 + np);
        int2 *p32 = (int2 *)(z64 + np), *t32 = p32 + np;
        float *z32 = (float *)(t32 + np), *zt = z32 + np;
        for (int i = 0; i < N; ++i)
            for (int e = 0; e < padw; ++e) {
                const size_t a = (size_t)i * padw + e, t = (size_t)e * N + i;
                const int q = deg[i] + e;
                const bool real = q < deg[i + 1];
                const float jf = real ? ajxyf[q] : 0.f;
                const double jd = real ? ajxy[q] : 0.0;
                int bf, bd[2];
                std::memcpy(&bf, &jf, 4);
                std::memcpy(bd, &jd, 8);
                const int j = real ? nbr[q] : i;
                p64[a] = make_int4(j, 0, bd[0], bd[1]);
                z64[a] = real ? ajz[q] : 0.0;
                p32[a] = t32[t] = make_int2(j, bf);
                z32[a] = zt[t] = real ? ajzf[q] : 0.f;
            }
        o_pad = img.add(pad);
    }
    std::vector<uint32_t> xyz(N);
    for (int r = 0; r < N; ++r) {
        // the coordinates of the site's cell
        const int q = r / B.nsub;
        int x = q % B.L[0], y = (q / B.L[0]) % B.L[1], z = q / (B.L[0] * B.L[1]);
        // coordinates are only used with a translation group (x, y < 2048, z < 1024)
        xyz[r] = haveL ? ((uint32_t)x | ((uint32_t)y << 11) | ((uint32_t)z << 22)) : 0u;
    }
    const size_t o_xyz = img.add(xyz), o_tile = img.add(B.tile0), o_chunk = img.add(B.chunk0), o_K = img.add(B.K);

    int bits = 1;
    while ((1 << bits) < N) ++bits;
    LatView &L = B.lv;
    L.N = N;
    L.nd = nd;
    L.np1 = N + 1;
    for (int a = 0; a < 3; ++a) L.L[a] = B.L[a];
    L.has_k = B.has_k;
    L.key_bits = (bits * nd <= 64) ? bits : 0;
    L.mask_ok = L.key_bits > 0 && L.L[0] <= 32 && L.L[1] <= 32 && L.L[2] <= 32;
    L.c0 = c0;
    L.c0f = (float)c0;
    L.c0lo = (float)(c0 - (double)(float)c0);
    L.nsub = B.nsub;
    L.ncell = B.ncell;
    L.pad_w = padw;
    L.jh_uniform = 0.0;
    if (nb > 0) {
        bool same = true;
        for (int b = 1; b < nb; ++b) same &= B.jxy[b] == B.jxy[0];
        if (same) L.jh_uniform = 0.5 * B.jxy[0];
    }

    L.diag_uniform = 0;
    size_t o_pair = 0, npair = 0;
    if (B.has_k && nb > 0 && nd > 0) {
        bool same = true;
        for (int i = 1; i < N; ++i) same &= u[i] == u[0];
        for (size_t q = 1; q < ajz.size(); ++q) same &= ajz[q] == ajz[0];
        if (same) {
            npair = (size_t)nd * B.max_degree + 1;
            std::vector<double> sums(npair + (npair + 1) / 2, 0.0);
            float *pf = (float *)(sums.data() + npair);
            for (size_t n = 1; n < npair; ++n) {
                sums[n] = sums[n - 1] + ajz[0];
                pf[n] = pf[n - 1] + ajzf[0];
            }
            o_pair = img.add(sums);
            L.e_row = c0;
            L.e_row_f = L.c0f;
            for (int k = 0; k < nd; ++k) {
                L.e_row += u[0];
                L.e_row_f += uf[0];
            }
            L.diag_uniform = 1;
        }
    }

    QS3_TRY(B.d_tab.upload(img.data.data(), img.data.size()));
    {
        const unsigned char *t = B.d_tab.as<unsigned char>();
        L.binom = (const uint64_t *)(t + o_binom);
        L.adj_ptr = (const int *)(t + o_ptr);
        L.adj_nbr = (const int *)(t + o_nbr);
        L.adj_jxy = (const double *)(t + o_jxy);
        L.adj_jz = (const double *)(t + o_jz);
        L.adj_jxy_f = (const float *)(t + o_jxyf);
        L.u = (const double *)(t + o_u);
        L.u_f = (const float *)(t + o_uf);
        L.adj_jz_f = (const float *)(t + o_jzf);
        L.adj_jxy_lo = (const float *)(t + o_jxyl);
        L.u_lo = (const float *)(t + o_ul);
        L.adj_jz_lo = (const float *)(t + o_jzl);
        L.xyz = (const uint32_t *)(t + o_xyz);
        if (padw) {
            L.adj_pad64 = (const int4 *)(t + o_pad);
            L.adj_jz_pad64 = (const double *)(L.adj_pad64 + np);
            L.adj_pad = (const int2 *)(L.adj_jz_pad64 + np);
            L.adjt = L.adj_pad + np;
            L.adj_jz_pad = (const float *)(L.adjt + np);
            L.adjt_jz = L.adj_jz_pad + np;
        }
        if (npair) {
            L.pair_sum = (const double *)(t + o_pair);
            L.pair_sum_f = (const float *)(L.pair_sum + npair);
        }
        B.tile0_d = (const int *)(t + o_tile);
        B.chunk0_d = (const int *)(t + o_chunk);
        B.K_d = (const int *)(t + o_K);
    }

    // sectors
    DevBuf oreps, ostab;
    uint64_t n_orb = 0;
    if (B.has_k && nd == 0) {
        std::vector<uint64_t> zero(nsec, 0);
        std::vector<uint8_t> one(nsec, 1);
        QS3_TRY(B.d_sigma.upload(zero.data(), zero.size() * 8));
        QS3_TRY(B.d_stab.upload(one.data(), one.size()));
    } else if (B.has_k) {
        QS3_TRY(build_sectors(B, oreps, ostab, n_orb));
    }
    B.secs.resize(nsec);
    const size_t nph = B.has_k ? (size_t)nsec * N : 0;
    if (B.has_k) {
        // double-float and complex128 phases, the roots of unity, complex64 phases
        QS3_TRY(B.d_ph.alloc(nph * (sizeof(float4) + sizeof(double2) + sizeof(float2)) + (size_t)B.ncell * sizeof(double2)));
        float4 *pdf = B.d_ph.as<float4>();
        double2 *p64 = (double2 *)(pdf + nph), *rt = p64 + nph;
        const int tot = nsec * N;
        k_phase_tables<<<(tot + 255) / 256, 256>>>(nsec, N, B.ncell, B.L[0], B.L[1], B.L[2], B.K_d, p64,
                                                   (float2 *)(rt + B.ncell), pdf);
        QS3_LAUNCHED();
        k_roots<<<(B.ncell + 255) / 256, 256>>>(B.ncell, rt);
        QS3_LAUNCHED();
        B.roots_d = rt;
    }
    for (int s = 0; s < nsec; ++s) {
        SecView &v = B.secs[s];
        v.sigma = B.has_k ? B.d_sigma.as<uint64_t>() + B.offs[s] : nullptr;
        v.stab = B.has_k ? B.d_stab.as<uint8_t>() + B.offs[s] : nullptr;
        v.dim = B.dims[s];
        v.off = B.offs[s];
        for (int a = 0; a < 3; ++a) v.K[a] = B.K[3 * s + a];
        v.tile0 = B.tile0[s];
        v.phdf = B.has_k ? B.d_ph.as<float4>() + (size_t)s * N : nullptr;
        v.ph64 = B.has_k ? (const double2 *)(B.d_ph.as<float4>() + nph) + (size_t)s * N : nullptr;
        v.ph32 = B.has_k ? (const float2 *)(B.roots_d + B.ncell) + (size_t)s * N : nullptr;
    }
    QS3_TRY(B.d_secs.alloc(B.secs.size() * sizeof(SecView)));
    if (B.has_k && nd > 0) QS3_TRY(build_index(B));
    QS3_TRY(put_secs(B));
    B.smem_bytes = row_kernel_smem(B, 0);
    if (B.smem_bytes > 200 * 1024)
        return set_err(QS3_ERR_OVERFLOW, "lattice tables need %zu bytes of shared memory", B.smem_bytes);
    B.narrow_ranks = !B.has_k && nd >= 1 && B.total > 0 && B.total < (1ull << 32);
    // the representative table when it is small (a bounded fraction of the
    // device memory); otherwise H Phi runs the representative search
    if (B.has_k && nd > 0 && B.total > 0 && N <= 4096) {
        size_t fr = 0, tt = 0;
        QS3_CUDA(cudaMemGetInfo(&fr, &tt));
        const size_t lim = std::min<size_t>(REP_TABLE_AUTO_BYTES, fr / 8);
        if (build_rep_table(B, lim, oreps, ostab, n_orb) != QS3_OK) {
            drop_rep_table(B);
            clear_err();
            // without it, the origin forms of the rows
            oreps.release();
            ostab.release();
            QS3_CUDA(cudaMemGetInfo(&fr, &tt));
            if (build_forms(B, fr / 8) != QS3_OK) {
                if (cudaPeekAtLastError() != cudaSuccess) return QS3_ERR_CUDA;
                clear_err();
            }
        }
    }
    QS3_CUDA(cudaDeviceSynchronize());       // the handle may be used on any stream
    return QS3_OK;
}

}  // namespace qs3

using namespace qs3;

extern "C" {

int qs3_basis_create(const qs3_lattice *lat, int32_t n_down, int32_t n_sectors, const int32_t *K, qs3_basis_t *out) {
    clear_err();
    if (!out) return set_err(QS3_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    qs3_basis_s *h = new (std::nothrow) qs3_basis_s();
    if (!h) return set_err(QS3_ERR_OOM, "host allocation");
    int st = basis_create(lat, n_down, n_sectors, K, h->B);
    if (st != QS3_OK) {
        delete h;
        return st;
    }
    *out = h;
    return QS3_OK;
}

int qs3_basis_destroy(qs3_basis_t b) {
    clear_err();
    delete b;
    pool_trim(POOL_IDLE_BYTES);
    return QS3_OK;
}

int qs3_basis_info(qs3_basis_t b, int32_t *n_sectors, uint64_t *total_dim) {
    clear_err();
    if (!b) return set_err(QS3_ERR_INVALID_ARG, "basis is NULL");
    if (n_sectors) *n_sectors = b->B.S;
    if (total_dim) *total_dim = b->B.total;
    return QS3_OK;
}

int qs3_basis_dims(qs3_basis_t b, uint64_t *dims) {
    clear_err();
    if (!b || !dims) return set_err(QS3_ERR_INVALID_ARG, "NULL argument");
    for (int s = 0; s < b->B.S; ++s) dims[s] = b->B.dims[s];
    return QS3_OK;
}

int qs3_basis_ranks(qs3_basis_t b, int32_t s, uint64_t *ranks, uint8_t *stab) {
    clear_err();
    if (!b || !ranks) return set_err(QS3_ERR_INVALID_ARG, "NULL argument");
    Basis &B = b->B;
    if (s < 0 || s >= B.S) return set_err(QS3_ERR_INVALID_ARG, "sector %d", s);
    if (!B.has_k) return set_err(QS3_ERR_INVALID_ARG, "a U(1)-only sector has ranks 0..dim-1");
    if (B.dims[s]) {
        QS3_CUDA(cudaMemcpy(ranks, B.secs[s].sigma, B.dims[s] * 8, cudaMemcpyDeviceToHost));
        if (stab) QS3_CUDA(cudaMemcpy(stab, B.secs[s].stab, B.dims[s], cudaMemcpyDeviceToHost));
    }
    return QS3_OK;
}

int qs3_basis_nnz(qs3_basis_t b, uint64_t *nnz) {
    clear_err();
    if (!b || !nnz) return set_err(QS3_ERR_INVALID_ARG, "NULL argument");
    QS3_TRY(count_nnz(b->B, nnz));
    return QS3_OK;
}

int qs3_basis_rep_table(qs3_basis_t b, int32_t mode, int32_t *active) {
    clear_err();
    if (!b) return set_err(QS3_ERR_INVALID_ARG, "basis is NULL");
    if (mode < -1 || mode > 1) return set_err(QS3_ERR_INVALID_ARG, "mode %d", mode);
    int st = QS3_OK;
    if (mode == 0) {
        drop_forms(b->B);
        drop_rep_table(b->B);
    } else if (mode == 1) {
        size_t fr = 0, tt = 0;
        QS3_CUDA(cudaMemGetInfo(&fr, &tt));
        st = build_rep_table(b->B, fr - fr / 16);
        if (st != QS3_OK) {
            std::string msg = last_err();
            drop_rep_table(b->B);
            set_err(st, "%s", msg.c_str());
        }
    }
    if (active) *active = b->B.lv.orb ? 1 : 0;
    return st;
}

int qs3_basis_tuning(qs3_basis_t b, int32_t set, int32_t *hphi_blocks_per_sm, int32_t *dot_vectors,
                     int32_t *dot_vectors64) {
    clear_err();
    if (!b) return set_err(QS3_ERR_INVALID_ARG, "basis is NULL");
    Basis &B = b->B;
    auto nv_ok = [](const int32_t *v) { return !v || *v == 0 || *v == 1 || *v == 2 || *v == 4; };
    auto nv64_ok = [&](const int32_t *v) { return nv_ok(v) || *v == 8; };
    if (set) {
        if (hphi_blocks_per_sm)
            for (int i = 0; i < 5; ++i)
                if (hphi_blocks_per_sm[i] < 0) return set_err(QS3_ERR_INVALID_ARG, "blocks per SM %d", hphi_blocks_per_sm[i]);
        if (!nv_ok(dot_vectors)) return set_err(QS3_ERR_INVALID_ARG, "dot vectors per pass %d", *dot_vectors);
        if (!nv64_ok(dot_vectors64)) return set_err(QS3_ERR_INVALID_ARG, "dot vectors per pass %d", *dot_vectors64);
        if (hphi_blocks_per_sm)
            for (int i = 0; i < 5; ++i) B.tune_hphi[i] = hphi_blocks_per_sm[i];
        if (dot_vectors) B.tune_nv = *dot_vectors;
        if (dot_vectors64) B.tune_nv64 = *dot_vectors64;
    } else {
        if (hphi_blocks_per_sm)
            for (int i = 0; i < 5; ++i) hphi_blocks_per_sm[i] = B.tune_hphi[i];
        if (dot_vectors) *dot_vectors = B.tune_nv;
        if (dot_vectors64) *dot_vectors64 = B.tune_nv64;
    }
    return QS3_OK;
}

int64_t qs3_inject_alloc_failure(int64_t after) {
    return (int64_t)qs3::g_alloc_budget.exchange(after < 0 ? -1 : (long long)after);
}

int32_t qs3_inject_wait_timeout(int32_t n) { return qs3::g_wait_starve.exchange(n > 0 ? n : 0); }

const char *qs3_last_error(void) { return qs3::last_err(); }

const char *qs3_strerror(int status) {
    switch (status) {
        case QS3_OK: return "ok";
        case QS3_ERR_INVALID_ARG: return "invalid argument";
        case QS3_ERR_OVERFLOW: return "size overflow";
        case QS3_ERR_SYMMETRY: return "symmetry violated";
        case QS3_ERR_OOM: return "out of device memory";
        case QS3_ERR_CUDA: return "CUDA error";
        case QS3_ERR_NOT_CONVERGED: return "not converged";
        case QS3_ERR_TIMEOUT: return "device wait timed out";
        case QS3_ERR_STATE: return "invalid state";
        default: return "unknown status";
    }
}

const char *qs3_version(void) { return "qs3-gb300 0.1 (sm_103a)"; }

uint64_t qs3_kernel_launches(void) { return qs3::g_launches.load(); }

}  // extern "C"
