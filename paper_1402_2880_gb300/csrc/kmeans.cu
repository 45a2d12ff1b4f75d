// Constrained k-means grouping of molecules into MO groups (Section "Defining
// neighbouring lists of atoms and MOs").
//
// Centres start on a grid spread over the bounding box of the molecules; each
// iteration links every molecule to a centre with at most n_link molecules per
// centre, then moves every centre to the centroid of its molecules, until the
// average move falls below tol or max_iter iterations ran.
//
// The paper links atoms in list order (one OpenMP lock per centre) and evens
// out the order dependence by shuffling the centres at every iteration. Here
// the link step is the molecule-proposing deferred-acceptance matching: an
// unlinked molecule proposes to its next centre in increasing (distance^2,
// centre index); a centre keeps the n_link proposers with the smallest
// (distance^2, molecule index), and one it rejects or displaces proposes on.
// The matching that comes out does not depend on the order of the proposals
// (preferences are strict), so warps make them concurrently, one molecule and
// the chain of molecules it displaces per warp, with a lock per centre. Squared
// distances are (dx*dx + dy*dy) + dz*dz with explicitly rounded operations (no
// fused multiply-add).
#include <algorithm>
#include <cmath>
#include <vector>

#include "sscf_internal.h"

namespace sscf {
namespace {

__device__ __forceinline__ double d2_rn(const double* a, const double* b) {
    const double dx = __dsub_rn(b[0], a[0]), dy = __dsub_rn(b[1], a[1]), dz = __dsub_rn(b[2], a[2]);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// Squared distances are compared as their bits (they are not negative): a CTA's
// warps share one FP64 pipe of two lanes per clock.
__device__ __forceinline__ long long key(double d) { return __double_as_longlong(d); }
// (d, i) < (e, j) lexicographically
__device__ __forceinline__ bool lex_less(long long d, int i, long long e, int j) { return d < e || (d == e && i < j); }

// Squared distances of all (molecule, centre) pairs, molecule-major.
__global__ void k_km_dist(int n, int nc, const double* __restrict__ pos, const double* __restrict__ cen,
                          double* __restrict__ D) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= (long long)n * nc) return;
    const int m = (int)(i / nc), c = (int)(i - (long long)m * nc);
    D[i] = d2_rn(pos + 3 * (size_t)m, cen + 3 * (size_t)c);
}

// What a centre holds: its members sorted by (distance^2 as a key, molecule).
// full: the last member's key with the sign bit set once there are n_link, else 0.
struct KmCentre {
    long long d[kMaxMolPerGroup];
    long long full;
    int m[kMaxMolPerGroup];
    int n, lock;
};
constexpr long long kKeyBits = 0x7fffffffffffffffll;
constexpr int kKmLoads = 8;   // distances in flight per lane
constexpr int kKmSpin = 1 << 22;   // polls of a centre's lock before a warp gives up

// The matching. A warp takes an unlinked molecule, finds its next centre (lanes
// over the centres, a lexicographic minimum), and inserts it under the centre's
// lock, a lane per member; a displaced molecule is the warp's next one and goes on
// after the centre that let it go, so that nothing but the centres' lists is kept.
// A full centre's last member only ever comes closer, so a centre whose last
// member is closer already would reject the molecule and is passed over without
// a proposal. A step is a row of distances and a few hundred clocks in a list, and
// chains of steps are serial: the lists sit in shared memory where they fit
// one CTA (IN_SMEM), in global memory with many CTAs else. D = NULL: distances
// from the positions (more pairs than are worth storing). No warp waits while it
// holds a lock.
// 1000 molecules, 150 centres, 101 matchings: 7 ms (34 with the distances compared
// in FP64, whose two lanes per clock a CTA's warps shared, rejections proposed one by
// one and one CTA for every size); with a pair of launches and a host round trip per
// round of proposals, each centre scanning all molecules, 219-318 ms.
template <bool IN_SMEM>
__global__ void __launch_bounds__(1024) k_km_match(int n, int nc, int n_link, const double* __restrict__ pos,
                                                   const double* __restrict__ cen, const double* __restrict__ D,
                                                   KmCentre* __restrict__ lists, int* __restrict__ next,
                                                   int* __restrict__ failed) {
    extern __shared__ __align__(16) unsigned char kmraw[];
    KmCentre* const L = IN_SMEM ? (KmCentre*)kmraw : lists;
    if (IN_SMEM) {
        for (int c = threadIdx.x; c < nc; c += blockDim.x) {
            L[c].n = L[c].lock = 0;
            L[c].full = 0;
        }
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    auto fence = [] {
        if (IN_SMEM) __threadfence_block();
        else __threadfence();
    };
    const int per = (n + 31) / 32;
    for (;;) {
        // (molecules that warps take at the same time lie far apart, or they would queue for one centre)
        int t = 0;
        if (lane == 0) t = atomicAdd(next, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= 32 * per) break;
        int m = (t & 31) * per + (t >> 5);
        if (m >= n) continue;
        long long ld = -1;   // the last proposal of m: everything after (ld, lc) is open
        int lc = -1;
        while (m >= 0) {
            long long bd = 0x7fffffffffffffffll;
            int bc = 0x7fffffff;
            for (int c0 = lane; c0 < nc; c0 += 32 * kKmLoads) {
                long long dv[kKmLoads];
#pragma unroll
                for (int u = 0; u < kKmLoads; ++u) {
                    const int c = min(c0 + 32 * u, nc - 1);
                    dv[u] = key(D ? D[(size_t)m * nc + c] : d2_rn(pos + 3 * (size_t)m, cen + 3 * (size_t)c));
                }
#pragma unroll
                for (int u = 0; u < kKmLoads; ++u) {
                    const int c = c0 + 32 * u;
                    if (c >= nc) break;
                    const long long d = dv[u], full = *(volatile long long*)&L[c].full;
                    if ((full == 0 || d <= (full & kKeyBits)) && lex_less(ld, lc, d, c) && lex_less(d, c, bd, bc)) {
                        bd = d;
                        bc = c;
                    }
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const long long od = __shfl_xor_sync(0xffffffffu, bd, o);
                const int oc = __shfl_xor_sync(0xffffffffu, bc, o);
                if (lex_less(od, oc, bd, bc)) {
                    bd = od;
                    bc = oc;
                }
            }
            int ok = 0;
            if (lane == 0) {
                int spins = kKmSpin + 1;
                if (bc < nc)   // (no centre left: cannot happen while there is room for every molecule)
                    for (spins = 0; spins <= kKmSpin && atomicCAS(&L[bc].lock, 0, 1) != 0;) ++spins;
                ok = spins <= kKmSpin;
                if (!ok) atomicExch(failed, 1);
            }
            if (!__shfl_sync(0xffffffffu, ok, 0)) break;
            __syncwarp();
            fence();
            // the centre's members, one per lane; those before m; the worst of n_link + 1 goes on
            volatile KmCentre& k = L[bc];
            const int held = k.n;
            const bool mine = lane < held;
            const long long qd = mine ? k.d[lane] : 0;
            const int qm = mine ? k.m[lane] : 0;
            const int p = __popc(__ballot_sync(0xffffffffu, mine && lex_less(qd, qm, bd, m)));
            int out = -1;   // the molecule to go on with, and its last proposal's distance
            long long out_d = 0;
            if (held == n_link) {
                out = __shfl_sync(0xffffffffu, qm, held - 1);
                out_d = __shfl_sync(0xffffffffu, qd, held - 1);
            }
            if (p == n_link) {   // m is rejected
                out = m;
                out_d = bd;
            } else {
                if (mine && lane >= p && lane + 1 < n_link) {
                    k.d[lane + 1] = qd;
                    k.m[lane + 1] = qm;
                }
                if (lane == 0) {
                    k.d[p] = bd;
                    k.m[p] = m;
                    if (held < n_link) k.n = held + 1;
                }
                const long long last = __shfl_sync(0xffffffffu, qd, max(n_link - 2, 0));
                if (lane == 0 && held >= n_link - 1) k.full = (p == n_link - 1 ? bd : last) | ~kKeyBits;
            }
            fence();
            __syncwarp();
            if (lane == 0) atomicExch(&L[bc].lock, 0);
            m = out;
            ld = out_d;
            lc = bc;
        }
    }
    if (IN_SMEM) {
        __syncthreads();
        for (int c = threadIdx.x; c < nc; c += blockDim.x) lists[c] = L[c];
    }
}

// Every centre's members as holders, and the centroid of the members summed in
// increasing molecule index; a centre without members keeps its place.
__global__ void k_km_centroids(int nc, const double* __restrict__ pos, const KmCentre* __restrict__ lists,
                               const double* __restrict__ cen, const int* __restrict__ failed,
                               double* __restrict__ cen_new, int* __restrict__ holder) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c == 0) cen_new[3 * (size_t)nc] = (double)*failed;   // to be read with the centres
    if (c >= nc) return;
    const int k = lists[c].n;
    int m[kMaxMolPerGroup];
    double x[kMaxMolPerGroup][3];
#pragma unroll
    for (int i = 0; i < kMaxMolPerGroup; ++i) m[i] = i < k ? lists[c].m[i] : 0x7fffffff;
#pragma unroll
    for (int i = 1; i < kMaxMolPerGroup; ++i)   // by index
#pragma unroll
        for (int j = i; j > 0; --j) {
            const int a = min(m[j - 1], m[j]), b = max(m[j - 1], m[j]);
            m[j - 1] = a;
            m[j] = b;
        }
#pragma unroll
    for (int i = 0; i < kMaxMolPerGroup; ++i)
#pragma unroll
        for (int d = 0; d < 3; ++d) x[i][d] = i < k ? pos[3 * (size_t)m[i] + d] : 0.0;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
#pragma unroll
    for (int i = 0; i < kMaxMolPerGroup; ++i) {
        if (i >= k) break;
        holder[m[i]] = c;
        s0 = __dadd_rn(s0, x[i][0]);
        s1 = __dadd_rn(s1, x[i][1]);
        s2 = __dadd_rn(s2, x[i][2]);
    }
    cen_new[3 * c] = k == 0 ? cen[3 * c] : __ddiv_rn(s0, (double)k);
    cen_new[3 * c + 1] = k == 0 ? cen[3 * c + 1] : __ddiv_rn(s1, (double)k);
    cen_new[3 * c + 2] = k == 0 ? cen[3 * c + 2] : __ddiv_rn(s2, (double)k);
}

struct Buf {
    std::vector<void*> ptrs;
    ~Buf() {
        for (void* p : ptrs) raw_free(p);
    }
    template <typename T>
    T* get(size_t n) {
        void* p = raw_alloc(n * sizeof(T));
        if (p) ptrs.push_back(p);
        return (T*)p;
    }
};

#define KM_CK(call)                                 \
    do {                                            \
        if ((call) != cudaSuccess) {                \
            cudaGetLastError();                     \
            return SSCF_ERR_CUDA;                   \
        }                                           \
    } while (0)

struct KmState {
    int n, nc, n_link;
    double *pos, *D;
    KmCentre* lists;
    int *holder, *next;   // next: [0] first molecule not taken, [1] a warp gave up
};
constexpr long long kKmMaxPairs = 1ll << 27;           // distances stored up to here (1 GB)
constexpr size_t kKmMaxSmem = 200 * 1024;
// Molecules up to which one CTA with the lists in shared memory matches faster than
// 128 with them in global memory (us per iteration, host included: 125 molecules 46
// against 64, 343 87 against 98, 1000 116 against 79, 4096 832 against 175).
constexpr int kKmOneCta = 512;

// The links of the centres `cen` (in st.lists) and the centroids they give.
int link_all(cudaStream_t s, const KmState& st, const double* cen, double* cen_new) {
    const int th = 256;
    const size_t list_bytes = (size_t)st.nc * sizeof(KmCentre);
    KM_CK(cudaMemsetAsync(st.lists, 0, list_bytes + 8, s));   // and next, which follows them
    if (st.D) {
        const long long pairs = (long long)st.n * st.nc;
        k_km_dist<<<(unsigned)((pairs + th - 1) / th), th, 0, s>>>(st.n, st.nc, st.pos, cen, st.D);
    }
    if (st.n <= kKmOneCta && list_bytes <= kKmMaxSmem) {
        KM_CK(allow_dynamic_smem<k_km_match<true>>());
        k_km_match<true><<<1, 1024, list_bytes, s>>>(st.n, st.nc, st.n_link, st.pos, cen, st.D, st.lists, st.next,
                                                     st.next + 1);
    } else {
        k_km_match<false><<<128, th, 0, s>>>(st.n, st.nc, st.n_link, st.pos, cen, st.D, st.lists, st.next,
                                             st.next + 1);
    }
    k_km_centroids<<<(st.nc + 31) / 32, 32, 0, s>>>(st.nc, st.pos, st.lists, cen, st.next + 1, cen_new, st.holder);
    KM_CK(cudaGetLastError());
    return SSCF_OK;
}

}  // namespace
}  // namespace sscf

using namespace sscf;

extern "C" int sscf_group_molecules(int n_atoms, const double* xyz, int n_link, int max_iter, double tol,
                                    void* cuda_stream, int* group_of_mol, int* n_groups_out, int* iters_out) {
    if (n_atoms <= 0 || n_atoms % 3 != 0 || !xyz || !group_of_mol) return SSCF_ERR_INVALID_ARG;
    if (n_link < 1 || n_link > kMaxMolPerGroup || max_iter < 0 || !(tol >= 0.0)) return SSCF_ERR_INVALID_ARG;
    const int n = n_atoms / 3;
    std::vector<double> pos(3 * (size_t)n);
    for (int m = 0; m < n; ++m)
        for (int d = 0; d < 3; ++d) {
            pos[3 * (size_t)m + d] = xyz[9 * (size_t)m + d];   // the molecule's first (oxygen) atom
            if (!std::isfinite(pos[3 * (size_t)m + d])) return SSCF_ERR_NONFINITE;
        }
    // centres: a grid over the bounding box, refined along the axis with the
    // largest spacing (lowest axis on ties) until it has ceil(n / n_link) points
    double lo[3], L[3];
    for (int d = 0; d < 3; ++d) {
        double a = pos[d], b = pos[d];
        for (int m = 1; m < n; ++m) {
            a = std::min(a, pos[3 * (size_t)m + d]);
            b = std::max(b, pos[3 * (size_t)m + d]);
        }
        lo[d] = a;
        L[d] = std::max(b - a, 1.0);
    }
    const long long need = ((long long)n + n_link - 1) / n_link;
    long long g[3] = {1, 1, 1};
    while (g[0] * g[1] * g[2] < need) {
        int best = 0;
        for (int d = 1; d < 3; ++d)
            if (L[d] / (double)g[d] > L[best] / (double)g[best]) best = d;
        g[best]++;
    }
    const int nc = (int)(g[0] * g[1] * g[2]);
    std::vector<double> cen(3 * (size_t)nc + 1), cen_new(3 * (size_t)nc + 1);   // and whether a warp gave up
    {
        size_t c = 0;
        for (long long k = 0; k < g[2]; ++k)
            for (long long j = 0; j < g[1]; ++j)
                for (long long i = 0; i < g[0]; ++i, ++c) {
                    const long long idx[3] = {i, j, k};
                    for (int d = 0; d < 3; ++d)
                        cen[3 * c + d] = lo[d] + ((double)(2 * idx[d] + 1) * L[d]) / (double)(2 * g[d]);
                }
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    Buf buf;
    KmState km;
    km.n = n;
    km.nc = nc;
    km.n_link = n_link;
    km.pos = buf.get<double>(3 * (size_t)n);
    double* d_cen = buf.get<double>(cen.size());
    double* d_cen_new = buf.get<double>(cen.size());
    km.lists = buf.get<KmCentre>((size_t)nc + 1);
    km.holder = buf.get<int>(n);
    km.next = (int*)(km.lists + nc);
    if (!km.pos || !d_cen || !d_cen_new || !km.lists || !km.holder) return SSCF_ERR_OOM;
    // (without room for the distances the matching computes them as it goes)
    km.D = (long long)n * nc <= kKmMaxPairs ? buf.get<double>((size_t)n * nc) : nullptr;
    KM_CK(cudaMemcpyAsync(km.pos, pos.data(), pos.size() * 8, cudaMemcpyHostToDevice, st));
    KM_CK(cudaMemcpyAsync(d_cen, cen.data(), cen.size() * 8, cudaMemcpyHostToDevice, st));
    int s = link_all(st, km, d_cen, d_cen_new);
    if (s != SSCF_OK) return s;
    int it = 0;
    for (it = 1; it <= max_iter; ++it) {
        KM_CK(cudaMemcpyAsync(cen_new.data(), d_cen_new, cen_new.size() * 8, cudaMemcpyDeviceToHost, st));
        KM_CK(cudaStreamSynchronize(st));
        if (cen_new[3 * (size_t)nc] != 0.0) return SSCF_ERR_TIMEOUT;
        std::swap(d_cen, d_cen_new);   // the links are due whether or not the centres have settled
        s = link_all(st, km, d_cen, d_cen_new);
        if (s != SSCF_OK) return s;
        double moved = 0.0;
        for (int c = 0; c < nc; ++c) {
            const double dx = cen_new[3 * c] - cen[3 * c], dy = cen_new[3 * c + 1] - cen[3 * c + 1],
                         dz = cen_new[3 * c + 2] - cen[3 * c + 2];
            const double xx = dx * dx, yy = dy * dy, zz = dz * dz;
            const double t = xx + yy;
            moved += std::sqrt(t + zz);
        }
        std::swap(cen, cen_new);
        if (moved / nc < tol) break;
    }
    if (it > max_iter) it = max_iter;
    std::vector<int> holder(n);
    KM_CK(cudaMemcpyAsync(holder.data(), km.holder, (size_t)n * 4, cudaMemcpyDeviceToHost, st));
    KM_CK(cudaMemcpyAsync(cen_new.data(), d_cen_new, cen_new.size() * 8, cudaMemcpyDeviceToHost, st));
    KM_CK(cudaStreamSynchronize(st));
    if (cen_new[3 * (size_t)nc] != 0.0) return SSCF_ERR_TIMEOUT;
    std::vector<int> remap(nc, -1);
    for (int m = 0; m < n; ++m) {
        if (holder[m] < 0 || holder[m] >= nc) return SSCF_ERR_STATE;
        remap[holder[m]] = 0;
    }
    int G = 0;
    for (int c = 0; c < nc; ++c)
        if (remap[c] == 0) remap[c] = G++;
    for (int m = 0; m < n; ++m) group_of_mol[m] = remap[holder[m]];
    if (n_groups_out) *n_groups_out = G;
    if (iters_out) *iters_out = it;
    return SSCF_OK;
}
