// Pair selection, block schedules and the row-local sweep (Section "Partial
// diagonalization" and Section "Orthonormalization", step d).
//
// The paper applies pair updates block-parallel: blocks of one label
// (Figure "jacobi") touch disjoint MOs and run concurrently, labels run one
// after the other. Here the labels are the colours of a greedy edge colouring
// of the MO-group graph, and inside a block pairs go by the in-block colour
// (i_loc + j_loc) mod n. Every 2x2 update uses coefficients fixed at the start
// of the sweep, so the whole sweep acts on each AO row of C independently. A
// colour is one launch: every block's rows with work are shared by its CTAs, which
// read and write the tiles of the block's two sides in place.
#include <math.h>

#include <algorithm>
#include <vector>

#include "block_scan.h"
#include "sscf_internal.h"

#include <type_traits>

namespace sscf {

namespace {

__device__ __forceinline__ unsigned long long dkey(double v) { return (unsigned long long)__double_as_longlong(v); }

__device__ __forceinline__ void atomic_max_pos(double* addr, double v) {
    atomicMax((unsigned long long*)addr, dkey(v));
}

// local MO index -> (side tile position, column) for a group side made of
// `no` occupied MOs (tiles first) and then virtual MOs
__device__ __forceinline__ void side_pos(int loc, int no, int not_, int& tpos, int& col) {
    if (loc < no) {
        tpos = loc >> 4;
        col = loc & 15;
    } else {
        int v = loc - no;
        tpos = not_ + (v >> 4);
        col = v & 15;
    }
}

// --------------------------------------------------------------------------
// rotation candidates: count |F_ij| >= tau (F_ij != 0) per cluster and the
// largest |F|. The cap of rot_cap_factor * N_occ is a per-cluster rule: every
// cluster of a batch selects exactly as it would alone.
// --------------------------------------------------------------------------
struct ClSel {
    unsigned long long cand, prefix, mask, rank, thr, kmax;
};

template <typename T>
__global__ void k_rot_stats(int n_gnb, const int* __restrict__ gnb_row, const int* __restrict__ gnb_col,
                            const int* __restrict__ group_nmol, const int* __restrict__ group_nvt,
                            const int* __restrict__ group_cl, const int* __restrict__ blk_tp0,
                            const T* __restrict__ F, double tau, DeviceScalars* sc, ClSel* cl) {
    const int e = blockIdx.x;
    const int A = gnb_row[e], B = gnb_col[e];
    const int no = 4 * group_nmol[A], nv = 2 * group_nmol[B], nvt = group_nvt[B];
    unsigned cnt = 0;
    double mx = 0.0;
    for (int p = threadIdx.x; p < no * nv; p += blockDim.x) {
        const int i = p / nv, j = p % nv;
        const int tp = blk_tp0[e] + (i >> 4) * nvt + (j >> 4);
        const double f = fabs((double)F[(size_t)tp * 256 + (i & 15) * 16 + (j & 15)]);
        mx = fmax(mx, f);
        if (f >= tau && f > 0.0) ++cnt;
    }
    for (int off = 16; off > 0; off >>= 1) {
        cnt += __shfl_xor_sync(0xffffffffu, cnt, off);
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    }
    if ((threadIdx.x & 31) == 0) {
        if (cnt) atomicAdd(&cl[group_cl[A]].cand, (unsigned long long)cnt);
        atomic_max_pos(&sc->max_fov, mx);
    }
}

// one radix-select pass over the candidate keys (8 bits, most significant
// first) of every cluster whose candidates exceed its cap. A CTA takes a
// contiguous range of blocks (clusters are contiguous in block order) and
// counts in shared memory, adding its nonzero bins to the cluster's global
// histogram when the cluster changes and at the end: the early passes put
// most keys in a few bins, which global atomics per key would serialise on.
template <typename T>
__global__ void __launch_bounds__(256) k_rot_hist(int shift, int n_gnb, const int* __restrict__ gnb_row,
                                                  const int* __restrict__ gnb_col,
                                                  const int* __restrict__ group_nmol, const int* __restrict__ group_nvt,
                                                  const int* __restrict__ group_cl, const int* __restrict__ blk_tp0,
                                                  const T* __restrict__ F, double tau,
                                                  const ClSel* __restrict__ cl, unsigned long long* __restrict__ hist) {
    __shared__ unsigned s_h[256];
    const int per = (n_gnb + gridDim.x - 1) / gridDim.x;
    const int e_lo = blockIdx.x * per, e_hi = min(n_gnb, e_lo + per);
    for (int i = threadIdx.x; i < 256; i += blockDim.x) s_h[i] = 0u;
    int cur = -1;   // cluster whose counts s_h holds (the same in every thread)
    auto flush = [&]() {
        __syncthreads();
        for (int i = threadIdx.x; i < 256; i += blockDim.x)
            if (s_h[i]) {
                atomicAdd(&hist[(size_t)cur * 256 + i], (unsigned long long)s_h[i]);
                s_h[i] = 0u;
            }
        __syncthreads();
    };
    __syncthreads();
    for (int e = e_lo; e < e_hi; ++e) {
        const int A = gnb_row[e], B = gnb_col[e];
        const int c = group_cl[A];
        if (c != cur) {
            if (cur >= 0) flush();
            cur = c;
        }
        const ClSel s = cl[c];
        if (s.cand <= s.kmax) continue;
        const int no = 4 * group_nmol[A], nv = 2 * group_nmol[B], nvt = group_nvt[B];
        for (int p = threadIdx.x; p < no * nv; p += blockDim.x) {
            const int i = p / nv, j = p % nv;
            const int tp = blk_tp0[e] + (i >> 4) * nvt + (j >> 4);
            const double f = fabs((double)F[(size_t)tp * 256 + (i & 15) * 16 + (j & 15)]);
            if (!(f >= tau && f > 0.0)) continue;
            const unsigned long long k = dkey(f);
            if ((k & s.mask) != s.prefix) continue;
            atomicAdd(&s_h[(k >> shift) & 255ull], 1u);
        }
    }
    if (cur >= 0) flush();
}

// one warp per cluster: pick the bin holding the kmax-th largest key (last_shift:
// the final pass; keys below it are zero for every candidate). Lane l holds bins
// 255 - 8 l and the seven below it, so that a scan over the lanes counts from the
// largest keys down (one thread reading 256 bins one after the other: 16-20 us a
// pass; now 3).
__global__ void k_rot_pick(int shift, int last_shift, int n_clusters, ClSel* cl, unsigned long long* hist) {
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c >= n_clusters) return;
    ClSel s = cl[c];
    unsigned long long* h = hist + (size_t)c * 256;
    if (s.cand > s.kmax) {
        if (shift == 56) s.rank = s.kmax;
        unsigned long long v[8], sum = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            v[i] = h[255 - 8 * lane - i];
            h[255 - 8 * lane - i] = 0ull;
            sum += v[i];
        }
        unsigned long long cum = sum;   // keys in this lane's bins and all above
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long u = __shfl_up_sync(0xffffffffu, cum, o);
            if (lane >= o) cum += u;
        }
        // the first lane that reaches the rank, and its bin (bin 0 takes what is left)
        const unsigned reach = __ballot_sync(0xffffffffu, cum >= s.rank);
        const int at = reach ? __ffs(reach) - 1 : 31;
        unsigned long long above = cum - sum;   // keys above the bin
        int b = 255 - 8 * lane;
        bool found = false;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            found = found || b == 0 || above + v[i] >= s.rank;
            if (!found) {
                above += v[i];
                --b;
            }
        }
        b = __shfl_sync(0xffffffffu, b, at);
        above = __shfl_sync(0xffffffffu, above, at);
        s.prefix |= (unsigned long long)b << shift;
        s.mask |= 255ull << shift;
        s.rank -= above;
    }
    if (shift == last_shift) s.thr = s.cand > s.kmax ? s.prefix : 0ull;
    if (lane == 0) cl[c] = s;
}

// The whole selection (k_rot_stats, the radix passes) in one CTA, for a single
// cluster of few blocks (kSelSmallBlocks): the launches between the passes cost
// more than the passes (11 of them, 17 in FP64, ~4 us each), until one CTA has too
// many keys to read. With the pair lists, without and with more candidates than the
// cap, us in one CTA against the launches: FP32 at 16 blocks 22 and 37 against 52 and
// 72, at 64 (45 and 64 molecules) 28 and 62 against 54 and 66, 36 and 80 against 58 and
// 68, at 308 191 to 279 against 76 to 81; FP64 at 64 30 and 91 against 76 and 95, 32 and
// 116 against 80 and 102, at 308 291 to 433 against 107.
constexpr int kSelSmallBlocks = 64;
template <typename T>
__global__ void __launch_bounds__(1024) k_rot_select_small(int last_shift, int n_gnb, const int* __restrict__ gnb_row,
                                                           const int* __restrict__ gnb_col,
                                                           const int* __restrict__ group_nmol,
                                                           const int* __restrict__ group_nvt,
                                                           const int* __restrict__ blk_tp0, const T* __restrict__ F,
                                                           double tau, unsigned long long kmax, DeviceScalars* sc,
                                                           ClSel* cl) {
    __shared__ unsigned s_h[256];
    __shared__ unsigned s_cnt, s_bin, s_above;
    __shared__ unsigned long long s_max;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        s_cnt = 0u;
        s_max = 0ull;
    }
    for (int i = threadIdx.x; i < 256; i += blockDim.x) s_h[i] = 0u;
    __syncthreads();
    // tau <= |F| and 0 < |F|, compared as keys (64 clocks of an SM quarter for an FP64 compare)
    const unsigned long long k_inf = dkey(INFINITY), k_tau = tau > 0.0 ? dkey(tau) : 1ull;
    // every candidate key, a block per warp or, of fewer blocks than warps, several warps per block
    const int w_per = n_gnb < 32 ? 32 / n_gnb : 1, sub = warp % w_per;
    auto each = [&](auto f) {
        for (int e = warp / w_per; e < n_gnb; e += 32 / w_per) {
            const int no = 4 * group_nmol[gnb_row[e]], B = gnb_col[e], nv = 2 * group_nmol[B], nvt = group_nvt[B];
            const T* fe = F + (size_t)blk_tp0[e] * 256;
#pragma unroll 4
            for (int p = lane + 32 * sub; p < no * 16; p += 32 * w_per) {
                const int i = p >> 4, j = p & 15;   // a block has one virtual tile: nvt = 1, nv <= 16
                if (j >= nv) continue;
                const unsigned long long k = dkey(fabs((double)fe[(size_t)(i >> 4) * nvt * 256 + (i & 15) * 16 + j]));
                f(k, k >= k_tau && k <= k_inf);
            }
        }
    };
    unsigned cnt = 0;
    unsigned long long mx = 0ull;
    each([&](unsigned long long k, bool in) {
        if (k > mx && k <= k_inf) mx = k;
        cnt += in;
    });
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long u = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = u > mx ? u : mx;
    }
    if (lane == 0) {
        atomicAdd(&s_cnt, cnt);
        atomicMax(&s_max, mx);
    }
    __syncthreads();
    unsigned long long prefix = 0ull, mask = 0ull, rank = kmax;
    if (s_cnt > kmax) {
        for (int shift = 56; shift >= last_shift; shift -= 8) {
            each([&](unsigned long long k, bool in) {
                if (in && (k & mask) == prefix) atomicAdd(&s_h[k >> shift & 255ull], 1u);
            });
            __syncthreads();
            if (warp == 0) {   // the bin of the rank-th largest key (k_rot_pick)
                unsigned h[8], sum = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    h[i] = s_h[255 - 8 * lane - i];
                    s_h[255 - 8 * lane - i] = 0u;
                    sum += h[i];
                }
                unsigned cum = sum;
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned u = __shfl_up_sync(0xffffffffu, cum, o);
                    if (lane >= o) cum += u;
                }
                const unsigned reach = __ballot_sync(0xffffffffu, (unsigned long long)cum >= rank);
                const int at = reach ? __ffs(reach) - 1 : 31;
                unsigned above = cum - sum;
                int b = 255 - 8 * lane;
                bool found = false;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    found = found || b == 0 || (unsigned long long)(above + h[i]) >= rank;
                    if (!found) {
                        above += h[i];
                        --b;
                    }
                }
                if (lane == at) {
                    s_bin = (unsigned)b;
                    s_above = above;
                }
            }
            __syncthreads();
            prefix |= (unsigned long long)s_bin << shift;
            mask |= 255ull << shift;
            rank -= s_above;
        }
    }
    if (threadIdx.x == 0) {
        atomicMax((unsigned long long*)&sc->max_fov, s_max);
        cl->cand = s_cnt;
        cl->kmax = kmax;
        cl->thr = s_cnt > kmax ? prefix : 0ull;
    }
}

// per block: kept pairs sorted by (in-block colour, i_loc) with Jacobi angles
// p = (F_ii - F_jj) / (2 F_ij), t = 1/(p + sgn(p) sqrt(1 + p^2)),
// c = 1/sqrt(1 + t^2), s = t c in FP64 (sgn(0) = +1)
constexpr int kListThreads = 128;
template <typename T>
__global__ void __launch_bounds__(kListThreads) k_rot_lists(int n_gnb, const int* __restrict__ gnb_row, const int* __restrict__ gnb_col,
                            const int* __restrict__ group_nmol, const int* __restrict__ group_nvt,
                            const int* __restrict__ group_occ0_mo, const int* __restrict__ group_virt0_mo,
                            const int* __restrict__ group_cl, const int* __restrict__ blk_tp0,
                            const T* __restrict__ F, const double* __restrict__ Fd, double tau, DeviceScalars* sc,
                            const ClSel* __restrict__ cl, int* __restrict__ pr_n,
                            int* __restrict__ pr_lvl, uint16_t* __restrict__ pr_ij, T* __restrict__ pr_cs,
                            int* __restrict__ pr_touch) {
    // kept pairs per level, as a bit per i: a pair's place in the list is its level's start plus the
    // kept i below its own, so that every pair is placed, and its angle computed, on its own (one
    // thread per level walked its pairs one after the other: 54 us at 8 molecules; now 14)
    __shared__ unsigned s_lv[kMaxSub];
    __shared__ int s_lvl[kMaxSub + 1];
    const int e = blockIdx.x;
    const int A = gnb_row[e], B = gnb_col[e];
    const int no = 4 * group_nmol[A], nv = 2 * group_nmol[B], nvt = group_nvt[B];
    const int nsub = max(no, nv);
    const unsigned long long thr = cl[group_cl[A]].thr;
    __shared__ int s_touch;
    if (threadIdx.x == 0) s_touch = 0;
    for (int s = threadIdx.x; s < kMaxSub; s += blockDim.x) s_lv[s] = 0u;
    __syncthreads();
    constexpr int kPer = 32 * 16 / kListThreads;
    T val[kPer];   // F_ij of the kept pairs of this thread
    unsigned kept = 0;
    int touch_t = 0;   // side tiles this thread's kept pairs touch: bits 0-2 side A, 3-5 side B
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int p = threadIdx.x + u * kListThreads, i = p >> 4, j = p & 15;
        val[u] = (T)0;
        if (i < no && j < nv) {
            const int tp = blk_tp0[e] + (i >> 4) * nvt + (j >> 4);
            val[u] = F[(size_t)tp * 256 + (i & 15) * 16 + (j & 15)];
            const double f = fabs((double)val[u]);
            if (f >= tau && f > 0.0 && dkey(f) >= thr) {
                kept |= 1u << u;
                touch_t |= (1 << (i >> 4)) | (1 << (3 + (j >> 4)));
                const int s = i + j;
                atomicOr(&s_lv[s >= nsub ? s - nsub : s], 1u << i);
            }
        }
    }
    if (touch_t) atomicOr(&s_touch, touch_t);
    __syncthreads();
    if (threadIdx.x < 32) {   // level starts: two levels per lane, 64 >= kMaxSub + 1
        const int a0 = 2 * threadIdx.x, c0 = a0 < kMaxSub ? __popc(s_lv[a0]) : 0, c1 = a0 + 1 < kMaxSub ? __popc(s_lv[a0 + 1]) : 0;
        int inc = c0 + c1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if ((int)threadIdx.x >= o) inc += v;
        }
        if (a0 <= kMaxSub) s_lvl[a0] = inc - c0 - c1;
        if (a0 + 1 <= kMaxSub) s_lvl[a0 + 1] = inc - c1;
    }
    __syncthreads();
    for (int s = threadIdx.x; s <= kMaxSub; s += blockDim.x) pr_lvl[(size_t)e * (kMaxSub + 1) + s] = s_lvl[s];
    if (threadIdx.x == 0) {
        const int run = s_lvl[kMaxSub];
        pr_n[e] = run;
        if (run) atomicAdd(&sc->n_rot, (unsigned long long)run);
        pr_touch[e] = s_touch;
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        if (!(kept >> u & 1)) continue;
        const int p0 = threadIdx.x + u * kListThreads, i = p0 >> 4, j = p0 & 15;
        const int s = i + j >= nsub ? i + j - nsub : i + j;
        const int pos = s_lvl[s] + __popc(s_lv[s] & ((1u << i) - 1u));
        const double fij = (double)val[u];
        const double fii = Fd[group_occ0_mo[A] + i], fjj = Fd[group_virt0_mo[B] + j];
        const double p = __ddiv_rn(__dsub_rn(fii, fjj), __dmul_rn(2.0, fij));
        const double sg = p >= 0.0 ? 1.0 : -1.0;
        const double t = __ddiv_rn(1.0, __dadd_rn(p, __dmul_rn(sg, sqrt(__dadd_rn(1.0, __dmul_rn(p, p))))));
        const double cc = __ddiv_rn(1.0, sqrt(__dadd_rn(1.0, __dmul_rn(t, t))));
        const double ss = __dmul_rn(t, cc);
        const size_t q = (size_t)e * kOrthoCap + pos;
        pr_ij[q] = (uint16_t)(i | (j << 8));
        pr_cs[2 * q] = (T)cc;
        pr_cs[2 * q + 1] = (T)ss;
    }
}

// --------------------------------------------------------------------------
// orthonormalisation: d_i = sqrt(sigma_ii), eta, pair lists
// --------------------------------------------------------------------------
template <typename T>
__global__ void k_ortho_scale(int w, int t_lo, int t_hi, const int* __restrict__ tile_group,
                              const int* __restrict__ tile_kind, const int* __restrict__ tile_nmo,
                              const int* __restrict__ tile_mo0, const int* __restrict__ group_ot0,
                              const int* __restrict__ group_not, const int* __restrict__ group_vt0,
                              const int* __restrict__ self_blk, const int* __restrict__ blk_tp,
                              const T* __restrict__ sig, double* __restrict__ dsc, unsigned* err) {
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    int t = t_lo + (idx >> 4), c = idx & 15;
    if (t >= t_hi) return;
    if (c >= tile_nmo[t]) return;
    const int g = tile_group[t];
    const int pos = tile_kind[t] == 0 ? t - group_ot0[g] : group_not[g] + (t - group_vt0[g]);
    const int tp = blk_tp[self_blk[g] * 9 + pos * 3 + pos];
    double s = (double)sig[(size_t)tp * 256 + c * 17];
    if (!(s > 0.0) || !isfinite(s)) {
        atomicOr(err, kErrNonFinite);
        s = 1.0;
    }
    dsc[tile_mo0[t] + c] = sqrt(s);
}

template <typename T>
__device__ __forceinline__ double sig_hat(const T* sig, const int* blk_tp, int e, bool same, int ia, int ib, int ci,
                                          int cj, double di, double dj) {
    int tp;
    double v;
    if (same && ib < ia) {
        tp = blk_tp[e * 9 + ib * 3 + ia];
        v = (double)sig[(size_t)tp * 256 + cj * 16 + ci];
    } else {
        tp = blk_tp[e * 9 + ia * 3 + ib];
        v = (double)sig[(size_t)tp * 256 + ci * 16 + cj];
    }
    return __ddiv_rn(v, __dmul_rn(di, dj));
}

// MO of local index `loc` in group g for the pass (occupied first)
__device__ __forceinline__ int pass_mo(int loc, int no, const int* occ0, const int* virt0, int g) {
    return loc < no ? occ0[g] + loc : virt0[g] + (loc - no);
}

template <typename T>
__global__ void k_ortho_eta(int w, const int* __restrict__ oblk, int n_oblk, const int* __restrict__ gnb_row,
                            const int* __restrict__ gnb_col, const int* __restrict__ group_nmol,
                            const int* __restrict__ group_not, const int* __restrict__ occ0,
                            const int* __restrict__ virt0, const int* __restrict__ blk_tp,
                            const T* __restrict__ sig, const double* __restrict__ dsc, DeviceScalars* sc,
                            const int* __restrict__ group_cl, double* __restrict__ cl_eta) {
    const int e = oblk[blockIdx.x];
    const int A = gnb_row[e], B = gnb_col[e];
    const int noA = 4 * group_nmol[A], noB = 4 * group_nmol[B];
    const int nA = w == 1 ? noA : 6 * group_nmol[A], nB = w == 1 ? noB : 6 * group_nmol[B];
    const bool same = A == B;
    double mx = 0.0;
    for (int p = threadIdx.x; p < nA * nB; p += blockDim.x) {
        const int i = p / nB, j = p % nB;
        if (same && j <= i) continue;
        int ia, ci, ib, cj;
        side_pos(i, noA, group_not[A], ia, ci);
        side_pos(j, noB, group_not[B], ib, cj);
        const double di = dsc[pass_mo(i, noA, occ0, virt0, A)], dj = dsc[pass_mo(j, noB, occ0, virt0, B)];
        mx = fmax(mx, fabs(sig_hat(sig, blk_tp, e, same, ia, ib, ci, cj, di, dj)));
    }
    for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if ((threadIdx.x & 31) == 0) {
        atomic_max_pos(&sc->eta, mx);
        atomic_max_pos(&cl_eta[group_cl[A]], mx);
    }
}

template <typename T>
__global__ void __launch_bounds__(kListThreads) k_ortho_lists(int w, double tol, const int* __restrict__ oblk, const int* __restrict__ gnb_row,
                              const int* __restrict__ gnb_col, const int* __restrict__ group_nmol,
                              const int* __restrict__ group_not, const int* __restrict__ occ0,
                              const int* __restrict__ virt0, const int* __restrict__ blk_tp,
                              const T* __restrict__ sig, const double* __restrict__ dsc, DeviceScalars* sc,
                              const int* __restrict__ group_cl, const double* __restrict__ cl_eta,
                              int* __restrict__ pr_n, int* __restrict__ pr_lvl, uint16_t* __restrict__ pr_ij,
                              T* __restrict__ pr_cs, int* __restrict__ pr_touch) {
    // as k_rot_lists: kept pairs per level as a bit per i
    __shared__ unsigned long long s_lv[kMaxSub];
    __shared__ int s_lvl[kMaxSub + 1];
    const int e = oblk[blockIdx.x];
    const int A = gnb_row[e], B = gnb_col[e];
    const int noA = 4 * group_nmol[A], noB = 4 * group_nmol[B];
    const int nA = w == 1 ? noA : 6 * group_nmol[A], nB = w == 1 ? noB : 6 * group_nmol[B];
    const bool same = A == B;
    const int nsub = max(nA, nB);
    const double eta = cl_eta[group_cl[A]];   // threshold of the block's own cluster
    const bool active = !(eta < tol);
    const double cut = 1e-3 * eta;
    __shared__ int s_touch;
    if (threadIdx.x == 0) s_touch = 0;
    for (int s = threadIdx.x; s < kMaxSub; s += blockDim.x) s_lv[s] = 0ull;
    __syncthreads();
    constexpr int kPer = 48 * 48 / kListThreads;
    T half[kPer];   // half the normalised overlap of the kept pairs of this thread
    unsigned kept = 0;
    int touch_t = 0;   // side tiles this thread's kept pairs touch: bits 0-2 side A, 3-5 side B
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int p = threadIdx.x + u * kListThreads, i = p / 48, j = p - 48 * i;
        half[u] = (T)0;
        if (active && i < nA && j < nB && !(same && j <= i)) {
            int ia, ci, ib, cj;
            side_pos(i, noA, group_not[A], ia, ci);
            side_pos(j, noB, group_not[B], ib, cj);
            const double di = dsc[pass_mo(i, noA, occ0, virt0, A)], dj = dsc[pass_mo(j, noB, occ0, virt0, B)];
            const double sh = sig_hat(sig, blk_tp, e, same, ia, ib, ci, cj, di, dj);
            if (fabs(sh) >= cut) {
                kept |= 1u << u;
                touch_t |= (1 << ia) | (1 << (3 + ib));
                half[u] = (T)__dmul_rn(0.5, sh);
                const int s = i + j;
                atomicOr(&s_lv[s >= nsub ? s - nsub : s], 1ull << i);
            }
        }
    }
    if (touch_t) atomicOr(&s_touch, touch_t);
    __syncthreads();
    if (threadIdx.x < 32) {   // level starts: two levels per lane, 64 >= kMaxSub + 1
        const int a0 = 2 * threadIdx.x, c0 = a0 < kMaxSub ? __popcll(s_lv[a0]) : 0,
                  c1 = a0 + 1 < kMaxSub ? __popcll(s_lv[a0 + 1]) : 0;
        int inc = c0 + c1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if ((int)threadIdx.x >= o) inc += v;
        }
        if (a0 <= kMaxSub) s_lvl[a0] = inc - c0 - c1;
        if (a0 + 1 <= kMaxSub) s_lvl[a0 + 1] = inc - c1;
    }
    __syncthreads();
    for (int s = threadIdx.x; s <= kMaxSub; s += blockDim.x) pr_lvl[(size_t)e * (kMaxSub + 1) + s] = s_lvl[s];
    if (threadIdx.x == 0) {
        const int run = s_lvl[kMaxSub];
        pr_n[e] = run;
        if (run) atomicAdd(&sc->n_combo, (unsigned long long)run);
        pr_touch[e] = s_touch;
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        if (!(kept >> u & 1)) continue;
        const int p = threadIdx.x + u * kListThreads, i = p / 48, j = p - 48 * i;
        const int s = i + j >= nsub ? i + j - nsub : i + j;
        const size_t q = (size_t)e * kOrthoCap + s_lvl[s] + __popcll(s_lv[s] & ((1ull << i) - 1ull));
        pr_ij[q] = (uint16_t)(i | (j << 8));
        pr_cs[2 * q] = half[u];
        pr_cs[2 * q + 1] = (T)0;
    }
}

// --------------------------------------------------------------------------
// Structural fill of a sweep (value-independent), then block-major apply.
//
// A unit is the set of tiles a block side touches: (group, occupied) and
// (group, virtual) for rotations and occupied passes, the whole group for
// passes over all MOs. A 2x2 update of an active block (one with pairs) can
// fill one side from the other, so before the sweep every row block is
// closed under "a block with pairs has both of its sides or neither"; all
// tiles of the units it holds are inserted as zero tiles. After that no
// update creates a tile: the sweep runs colour by colour, block-major, in
// place, and a final compaction drops the tiles left all-zero.
// --------------------------------------------------------------------------
struct SweepArgs {
    int mode;        // 0 rotations (A occupied | B virtual), 1 combinations
    int which;       // combinations: 0 all MOs, 1 occupied MOs
    int n_tiles, n_occ_tiles, n_groups, cap, n_blk, max_cl_groups, n_clusters;
    double trunc;
    float trunc_f;   // smallest float >= trunc: |x| < trunc <=> |x| < trunc_f for every float x
    const int* blk;          // blocks of the pass by colour
    const int* mol_cluster;  // closure: cluster of every row block
    const int* cl_g0;        // closure: first group, occupied tile and virtual tile of every cluster
    const int* cl_ot0;
    const int* cl_vt0;
    const int* clblk_ptr;    // closure: blocks of the pass by cluster
    const int* clblk;
    const int* unit_lab;     // closure: component label of every unit (2 per group), cluster-local
    int* lab_start;          // closure: per label, first entry of its members in lab_mem, and their count
    int* lab_cnt;
    int* lab_mem;            // closure: the units of every component, in increasing order
    const int* gnb_colour;   // closure: colour of every block ...
    int col_lo, col_hi;      // ... only blocks of colours [col_lo, col_hi) link units
    const int* gnb_row;
    const int* gnb_col;
    const int* group_nmol;
    const int* group_ot0;
    const int* group_not;
    const int* group_vt0;
    const int* group_nvt;
    const int* tile_group;
    const int* tile_kind;
    const int* tile_mo0;
    const int* tile_nmo;
    const int* pr_n;
    const int* pr_lvl;
    const int* pr_touch;     // tiles of each side a block's pairs touch: bits 0-2 side A, 3-5 side B
    const uint16_t* pr_ij;
    const void* pr_cs;
    const double* dsc;       // combinations: divide the pass's MOs by d_i first ...
    const double* cl_eta;    // ... in clusters whose eta is not below the pass's target
    double tol;              // (below it the pass has converged and changes nothing)
    unsigned long long* upd; // counter of 2x2 row updates
    const int* cci_ptr;
    const int* cci_row;
    const int* cci_slot;
    const int* in_nt;
    const int* in_tile;
    const void* in_val;
    int* out_nt;
    int* out_tile;
    void* out_val;
    unsigned char* out_nz;   // flags of out: 0 = the tile is all zero (written by the closure, kept by the sweep)
    unsigned char* col_nz;   // sweeps: the same flags in column-index order (flag_base)
    void* blk_info;          // a BlockInfo per block in colour order
    const unsigned char* in_nz;   // closure: flags of the input (NULL: every listed tile may be nonzero)
    int normalise_pass;      // closure in mode 1: divide by d_i (the first closure of a pass)
    unsigned* err;
};


// truncation test |x| < threshold, decided exactly in the storage precision;
// FP64 on the bit patterns (those of non-negative doubles order as the values
// do, and a NaN is above any threshold, as it is not below in the comparison of
// values): the FP64 pipe has two lanes per clock and SM, and a comparison there
// costs as much as the update it follows
__device__ __forceinline__ bool below(double x, const SweepArgs& a) {
    return ((unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull) <
           (unsigned long long)__double_as_longlong(a.trunc);
}
__device__ __forceinline__ bool below(float x, const SweepArgs& a) { return fabsf(x) < a.trunc_f; }
// x != 0 without the FP64 pipe
__device__ __forceinline__ bool nonzero(double x) { return (__double_as_longlong(x) << 1) != 0; }
__device__ __forceinline__ bool nonzero(float x) { return x != 0.f; }

// Connected components of a pass's units (the occupied or the virtual tiles
// of one group) under its active blocks, one CTA per cluster. The closure of a
// row is then the set of units whose component holds a unit the row has:
// "a block with pairs has both of its sides or neither", applied until nothing
// changes, is exactly that. Unit u of a cluster with ng groups: occupied
// tiles of local group u (u < ng), virtual tiles of local group u - ng.
// Hook-and-compress: roots are linked to the smaller root across every active
// block, then every label is replaced by its root, until no block links two
// roots. A label only ever points to a smaller unit of the same component.
__global__ void __launch_bounds__(1024) k_closure_labels(SweepArgs a, int* __restrict__ unit_lab) {
    extern __shared__ int slab[];   // 2 ng labels
    const int k = blockIdx.x;
    const int g0 = a.cl_g0[k], ng = a.cl_g0[k + 1] - g0, nu = 2 * ng;
    const int jb0 = a.clblk_ptr[k], jb1 = a.clblk_ptr[k + 1];
    const bool groups = a.mode == 1 && a.which == 0;   // occupied and virtual tiles of a group move together
    for (int u = threadIdx.x; u < nu; u += blockDim.x) slab[u] = u;
    __syncthreads();
    auto find = [&](int u) {
        int v = slab[u];
        while (v != u) {
            u = v;
            v = slab[u];
        }
        return u;
    };
    // every round that links at least one pair of roots removes a root, so at
    // most nu rounds can change anything
    for (int it = 0; it <= nu; ++it) {
        int changed = 0;
        const int n_edges = (jb1 - jb0) + (groups ? ng : 0);
        for (int j = threadIdx.x; j < n_edges; j += blockDim.x) {
            int u, v;
            if (j < jb1 - jb0) {
                const int e = a.clblk[jb0 + j];
                if (a.pr_n[e] == 0) continue;
                const int col = a.gnb_colour[e];
                if (col < a.col_lo || col >= a.col_hi) continue;
                u = a.gnb_row[e] - g0;
                v = a.mode == 0 ? ng + (a.gnb_col[e] - g0) : a.gnb_col[e] - g0;
            } else {
                u = j - (jb1 - jb0);
                v = ng + u;
            }
            const int ru = find(u), rv = find(v);
            if (ru != rv) {
                atomicMin(&slab[max(ru, rv)], min(ru, rv));
                changed = 1;
            }
        }
        const int any = __syncthreads_or(changed);
        for (int u = threadIdx.x; u < nu; u += blockDim.x) slab[u] = find(u);
        __syncthreads();
        if (!any) break;
    }
    for (int u = threadIdx.x; u < nu; u += blockDim.x) unit_lab[2 * g0 + u] = slab[u];
    // The members of every component in increasing unit order (CSR by label):
    // counts, an exclusive scan, then one warp places the units in order, the
    // lanes of a group of 32 with equal labels taking consecutive entries.
    int* cnt = slab + nu;
    for (int u = threadIdx.x; u < nu; u += blockDim.x) cnt[u] = 0;
    __syncthreads();
    for (int u = threadIdx.x; u < nu; u += blockDim.x) atomicAdd(&cnt[slab[u]], 1);
    __syncthreads();
    __shared__ int part[33];
    const int per = (nu + blockDim.x - 1) / blockDim.x;
    const int lo = threadIdx.x * per, hi = min(nu, lo + per);
    int sum = 0;
    for (int i = lo; i < hi; ++i) sum += cnt[i];
    int run = block_scan(sum, part);
    for (int i = lo; i < hi; ++i) {
        const int c = cnt[i];
        a.lab_start[2 * g0 + i] = run;
        a.lab_cnt[2 * g0 + i] = c;
        cnt[i] = run;   // from here on: the next free entry of label i
        run += c;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        for (int base = 0; base < nu; base += 32) {
            const int u = base + lane;
            const unsigned act = __ballot_sync(0xffffffffu, u < nu);
            if (u < nu) {
                const int l = slab[u];
                const unsigned peers = __match_any_sync(act, l);
                a.lab_mem[2 * g0 + cnt[l] + __popc(peers & ((1u << lane) - 1u))] = u;
                __syncwarp(act);   // every peer has read cnt[l] before its first lane moves it
                if (lane == __ffs(peers) - 1) cnt[l] += __popc(peers);
            }
            __syncwarp();
        }
    }
}

// Components with more members than this are marked by a whole warp.
constexpr int kSmallComp = 8;
constexpr int kBigMax = 64;   // large components listed per row (more: marked by their claimant)
template <typename T>
__global__ void __launch_bounds__(256) k_closure(SweepArgs a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    if (*a.err & (kErrCapacity | kErrSortSize)) return;   // an earlier kernel of the step overflowed
    // everything a row block touches belongs to its own cluster: units and
    // labels are indexed inside the cluster's ranges
    const int r = blockIdx.x;
    const int k = a.mol_cluster[r];
    const int g0 = a.cl_g0[k], ng = a.cl_g0[k + 1] - g0, nu = 2 * ng;
    const int uw = (2 * a.max_cl_groups + 31) >> 5;   // words of a bitset over a cluster's units
    const int nw = (nu + 31) >> 5;
    unsigned* present = (unsigned*)smraw;      // by label: components holding a nonzero tile of the row
    unsigned* onu = present + uw;              // by unit: units of the new row
    int* wpos = (int*)(onu + uw);              // per word of onu: its tile count, then its first slot
    int* oldt = wpos + uw;                     // the row's tile ids (sorted)
    short* oslot = (short*)(oldt + a.cap);     // per new slot: its slot in the row, or -1
    __shared__ int s_big[kBigMax];
    __shared__ int s_nbig;
    __shared__ int part[33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int* lab = a.unit_lab + 2 * g0;
    const int* lstart = a.lab_start + 2 * g0;
    const int* lcnt = a.lab_cnt + 2 * g0;
    const int* lmem = a.lab_mem + 2 * g0;
    for (int i = threadIdx.x; i < nw; i += blockDim.x) present[i] = onu[i] = 0u;
    if (threadIdx.x == 0) s_nbig = 0;
    const int n0 = a.in_nt[r];
    for (int s = threadIdx.x; s < n0; s += blockDim.x) oldt[s] = a.in_tile[(size_t)r * a.cap + s];
    __syncthreads();
    auto mark = [&](int l, int j0, int dj) {
        const int m0 = lstart[l], mn = lcnt[l];
        for (int j = j0; j < mn; j += dj) {
            const int m = lmem[m0 + j];
            atomicOr(&onu[m >> 5], 1u << (m & 31));
        }
    };
    // The row keeps every unit of every component that holds one of its
    // nonzero tiles: a tile flagged all-zero keeps nothing and creates no fill.
    // The first thread to claim a component marks its members (a large one is
    // listed for a warp instead).
    for (int s = threadIdx.x; s < n0; s += blockDim.x) {
        if (a.in_nz && !a.in_nz[(size_t)r * a.cap + s]) continue;
        const int t = oldt[s];
        const int g = a.tile_group[t] - g0;
        const int u = ((a.mode == 1 && a.which == 0) || a.tile_kind[t] == 0) ? g : ng + g;
        const int l = lab[u];
        const unsigned bit = 1u << (l & 31);
        if (atomicOr(&present[l >> 5], bit) & bit) continue;
        if (lcnt[l] > kSmallComp) {
            const int i = atomicAdd(&s_nbig, 1);
            if (i < kBigMax) {
                s_big[i] = l;
                continue;
            }
        }
        mark(l, 0, 1);
    }
    __syncthreads();
    const int nbig = min(s_nbig, kBigMax);
    for (int b = warp; b < nbig; b += nwarps) mark(s_big[b], lane, 32);
    __syncthreads();
    // tiles per word of the new unit set, then their first slots (units in
    // order: occupied units by group, then virtual ones, i.e. tile ids ascending)
    auto ntiles = [&](int u) { return u < ng ? a.group_not[g0 + u] : a.group_nvt[g0 + u - ng]; };
    for (int w = threadIdx.x; w < nw; w += blockDim.x) {
        unsigned b = onu[w];
        int c = 0;
        while (b) {
            c += ntiles(32 * w + __ffs(b) - 1);
            b &= b - 1;
        }
        wpos[w] = c;
    }
    __syncthreads();
    const int per = (nw + blockDim.x - 1) / blockDim.x;
    const int w0 = threadIdx.x * per, w1 = min(nw, w0 + per);
    int cnt = 0;
    for (int w = w0; w < w1; ++w) cnt += wpos[w];
    int run = block_scan(cnt, part);
    const int n1 = part[32];
    if (n1 > a.cap) {
        if (threadIdx.x == 0) atomicOr(a.err, kErrCapacity);
        return;
    }
    for (int w = w0; w < w1; ++w) {
        const int c = wpos[w];
        wpos[w] = run;
        run += c;
    }
    __syncthreads();
    // the new row: tile ids, the slot each had in the row (binary search of the
    // sorted old list), flags: tiles that were in the row survived the last
    // compaction (or come from the guess or a restart) and may be nonzero;
    // inserted tiles are zero
    for (int w = threadIdx.x; w < nw; w += blockDim.x) {
        unsigned b = onu[w];
        int pos = wpos[w];
        while (b) {
            const int u = 32 * w + __ffs(b) - 1;
            b &= b - 1;
            const int g = u < ng ? u : u - ng;
            const int t0 = u < ng ? a.group_ot0[g0 + g] : a.group_vt0[g0 + g];
            const int nt = ntiles(u);
            for (int i = 0; i < nt; ++i, ++pos) {
                const int t = t0 + i;
                int lo = 0, hi = n0;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (oldt[mid] < t) lo = mid + 1;
                    else hi = mid;
                }
                const int os = lo < n0 && oldt[lo] == t ? lo : -1;
                a.out_tile[(size_t)r * a.cap + pos] = t;
                oslot[pos] = (short)os;
                a.out_nz[(size_t)r * a.cap + pos] = os < 0 ? 0 : (a.in_nz ? a.in_nz[(size_t)r * a.cap + os] : 1);
            }
        }
    }
    if (threadIdx.x == 0) a.out_nt[r] = n1;
    __syncthreads();
    // values, 16 bytes at a time
    using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    constexpr int kVec = 16 / (int)sizeof(T);
    constexpr int kPer = kTileVals / kVec;   // 16-byte pieces per tile
    const V* inv = (const V*)a.in_val + (size_t)r * a.cap * kPer;
    V* outv = (V*)a.out_val + (size_t)r * a.cap * kPer;
    const bool normalise = a.mode == 1 && a.normalise_pass && !(a.cl_eta[k] < a.tol);
    for (int idx = threadIdx.x; idx < n1 * kPer; idx += blockDim.x) {
        const int s = idx / kPer, piece = idx - s * kPer;
        const int os = oslot[s];
        V v;
        if (os >= 0) {
            v = inv[(size_t)os * kPer + piece];
            const int t = a.out_tile[(size_t)r * a.cap + s];
            if (normalise && (a.which == 0 || a.tile_kind[t] == 0)) {
                T* e = (T*)&v;
                const int nmo = a.tile_nmo[t], mo0 = a.tile_mo0[t];
#pragma unroll
                for (int q = 0; q < kVec; ++q) {
                    const int col = (piece * kVec + q) & 15;
                    if (col < nmo) e[q] = e[q] / (T)a.dsc[mo0 + col];
                }
            }
        } else {
            T* e = (T*)&v;
#pragma unroll
            for (int q = 0; q < kVec; ++q) e[q] = (T)0;
        }
        outv[(size_t)s * kPer + piece] = v;
    }
}


// The tile flags of the sweep's input in column-index order: entry k of tile
// t's list (row cci_row[p], slot cci_slot[p], p = cci_ptr[t] + k) gets the flag
// of that tile in that row, so that the sweep kernels test a block's rows for
// work with contiguous reads, and raise both copies of a flag together. Every
// tile's flags start on a 16-byte boundary and are zero up to the next one.
__host__ __device__ constexpr size_t flag_bytes(size_t entries, size_t n_tiles) { return entries + 16 * n_tiles + 32; }
__device__ __forceinline__ int flag_base(int tile, int ptr) { return ((ptr + 15) & ~15) + 16 * tile; }

// One CTA per tile.
__global__ void __launch_bounds__(256) k_flags_by_column(int cap, const int* __restrict__ cci_ptr,
                                                         const int* __restrict__ cci_row,
                                                         const int* __restrict__ cci_slot,
                                                         const unsigned char* __restrict__ nz,
                                                         unsigned char* __restrict__ col_nz) {
    const int t = blockIdx.x;
    const int lo = cci_ptr[t], n = cci_ptr[t + 1] - lo;
    unsigned char* f = col_nz + flag_base(t, lo);
    for (int k = threadIdx.x; k < ((n + 15) & ~15); k += blockDim.x)
        f[k] = k < n ? nz[(size_t)cci_row[lo + k] * cap + cci_slot[lo + k]] : 0;
}

// side tiles of a block: up to 3 per side, as (first tile of a run, offset)
struct Side {
    int n;           // tiles on the side
    int run0;        // first tile of the occupied (or only) run
    int nrun0;       // tiles in that run
    int run1;        // first tile of the virtual run (all-MO passes) or -1
};

__device__ __forceinline__ Side side_of(const SweepArgs& a, int g, bool virt_only, bool with_virt) {
    Side s;
    if (virt_only) {
        s.run0 = a.group_vt0[g];
        s.nrun0 = a.group_nvt[g];
        s.run1 = -1;
        s.n = s.nrun0;
    } else {
        s.run0 = a.group_ot0[g];
        s.nrun0 = a.group_not[g];
        s.run1 = with_virt ? a.group_vt0[g] : -1;
        s.n = s.nrun0 + (with_virt ? a.group_nvt[g] : 0);
    }
    return s;
}

constexpr int kUnroll = 1;                 // pairs of one level in flight per thread (measured best)
constexpr int kSegUnroll = 4;              // panel segments in flight per thread

template <typename T> struct Vec;
template <> struct Vec<float> {
    using type = float4;
    static constexpr int n = 4;
    __device__ static float4 zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
};
template <> struct Vec<double> {
    using type = double2;
    static constexpr int n = 2;
    __device__ static double2 zero() { return make_double2(0.0, 0.0); }
};

// Rows per thread and row blocks per CTA: FP32 panels are processed two
// adjacent AO rows per thread with packed f32x2 arithmetic; FP64 one row.
template <typename T> struct ApplyShape;
template <> struct ApplyShape<float> {
    static constexpr int rows = 2, chunk = 64;
};
template <> struct ApplyShape<double> {
    static constexpr int rows = 1, chunk = 32;
};
template <typename T> __host__ __device__ constexpr int apply_nr() { return ApplyShape<T>::chunk * kAoPerMol; }
// even, bank-spread panel stride
template <typename T> __host__ __device__ constexpr int apply_nrp() { return apply_nr<T>() + 2; }
template <typename T> __host__ __device__ constexpr int apply_threads() { return apply_nr<T>() / ApplyShape<T>::rows; }

__device__ __forceinline__ float2 trunc2(float2 v, float t) {
    v.x = fabsf(v.x) < t ? 0.f : v.x;
    v.y = fabsf(v.y) < t ? 0.f : v.y;
    return v;
}

// One CTA = one active block of the colour x a chunk of row blocks. The
// block's side tiles of those rows are staged in shared memory as a
// [tile][column][row] panel; every thread owns one (FP64) or two adjacent
// (FP32) AO rows and applies the block's pairs to them in schedule order,
// level by level. Rows are independent, so no barrier is needed between
// levels; pairs of one level touch disjoint MOs, so kUnroll of them are
// loaded, updated and stored together.
template <typename T, int MODE, int NT, int PCAP>
__global__ void __launch_bounds__(apply_threads<T>()) k_apply_colour(SweepArgs a, int p0) {
    constexpr int CH = ApplyShape<T>::chunk, NRP = apply_nrp<T>();
    extern __shared__ __align__(16) unsigned char smraw[];
    T* panel = (T*)smraw;                                    // [NT tiles][16][NRP]
    T* pcs = panel + NT * 16 * NRP;                          // np * 2 coefficients
    unsigned* poff = (unsigned*)(pcs + 2 * PCAP);            // np packed panel offsets
    __shared__ int s_lvl[kMaxSub + 1];
    __shared__ int s_row[CH];
    __shared__ int s_slot[CH][NT];
    __shared__ int s_cp[NT];   // start of each panel tile's flags (-1: not held)
    // side A occupies panel tiles [0, kSideA), side B [kSideA, NT)
    constexpr int kSideA = MODE == 0 ? 2 : NT / 2;
    if (*a.err & (kErrCapacity | kErrSortSize)) return;
    const int e = a.blk[p0 + blockIdx.y];
    const int np = a.pr_n[e];
    if (np == 0) return;
    const int A = a.gnb_row[e], B = a.gnb_col[e];
    const bool with_virt = MODE == 1 && a.which == 0;
    const Side sa = side_of(a, A, false, with_virt);
    const Side sb = side_of(a, B, MODE == 0, with_virt);
    const int pa = a.cci_ptr[sa.run0], n_rows = a.cci_ptr[sa.run0 + 1] - pa;
    const int pb = a.cci_ptr[sb.run0];
    const int k0 = blockIdx.x * CH;
    if (k0 >= n_rows) return;
    if (a.cci_ptr[sb.run0 + 1] - pb != n_rows) {
        if (threadIdx.x == 0) atomicOr(a.err, kErrCapacity);
        return;
    }
    const int nk = min(CH, n_rows - k0);
    if (threadIdx.x == 0) atomicAdd(a.upd, (unsigned long long)np * (unsigned long long)(nk * 6));
    // a combination block inside one group: both sides are the same tiles, held once
    const bool same = MODE == 1 && A == B;
    const int pav = sa.run1 >= 0 ? a.cci_ptr[sa.run1] : 0;
    const int pbv = sb.run1 >= 0 ? a.cci_ptr[sb.run1] : 0;
    for (int t = threadIdx.x; t < nk; t += blockDim.x) {
        const int k = k0 + t;
        s_row[t] = a.cci_row[pa + k];
        const int so = a.cci_slot[pa + k];
        const int sv = sa.run1 >= 0 ? a.cci_slot[pav + k] : 0;
        const int bo = a.cci_slot[pb + k];
        const int bv = sb.run1 >= 0 ? a.cci_slot[pbv + k] : 0;
        for (int i = 0; i < NT / 2 + (NT & 1); ++i) {
            if (i < kSideA) s_slot[t][i] = i < sa.nrun0 ? so + i : (i < sa.n ? sv + (i - sa.nrun0) : -1);
            if (i < NT - kSideA)
                s_slot[t][kSideA + i] = same ? -1 : (i < sb.nrun0 ? bo + i : (i < sb.n ? bv + (i - sb.nrun0) : -1));
        }
    }
    if (threadIdx.x < NT) {
        const int p = threadIdx.x;
        int tile = -1;
        if (p < kSideA) {
            if (p < sa.nrun0) tile = sa.run0 + p;
            else if (p < sa.n) tile = sa.run1 + (p - sa.nrun0);
        } else if (!same) {
            const int i = p - kSideA;
            if (i < sb.nrun0) tile = sb.run0 + i;
            else if (i < sb.n) tile = sb.run1 + (i - sb.nrun0);
        }
        s_cp[p] = tile >= 0 ? flag_base(tile, a.cci_ptr[tile]) : -1;
    }
    __syncthreads();
    // a chunk whose held tiles are all flagged zero in all its rows stays as it
    // is (the updates of zeros are zeros): nothing to load, update or store
    bool work = false;
    for (int t = threadIdx.x; t < nk; t += blockDim.x)
        for (int p = 0; p < NT; ++p) work |= s_cp[p] >= 0 && a.col_nz[s_cp[p] + k0 + t];
    if (!__syncthreads_or(work)) return;
    const int* lvl = a.pr_lvl + (size_t)e * (kMaxSub + 1);
    for (int i = threadIdx.x; i <= kMaxSub; i += blockDim.x) s_lvl[i] = lvl[i];
    const T* cs = (const T*)a.pr_cs + (size_t)e * kOrthoCap * 2;
    const uint16_t* ij = a.pr_ij + (size_t)e * kOrthoCap;
    const int noA = 4 * a.group_nmol[A], noB = 4 * a.group_nmol[B];
    for (int q = threadIdx.x; q < np; q += blockDim.x) {
        const unsigned w = ij[q];
        const int il = w & 255, jl = w >> 8;
        int ta, ca, tb, cb;
        if (MODE == 0) {
            ta = il >> 4;
            ca = il & 15;
            tb = kSideA + (jl >> 4);
            cb = jl & 15;
        } else {
            side_pos(il, noA, sa.nrun0, ta, ca);
            side_pos(jl, noB, sb.nrun0, tb, cb);
            if (!same) tb += kSideA;
        }
        poff[q] = (unsigned)((ta * 16 + ca) * NRP) | ((unsigned)((tb * 16 + cb) * NRP) << 16);
        pcs[2 * q] = cs[2 * q];
        pcs[2 * q + 1] = cs[2 * q + 1];
    }
    __syncthreads();
    T* val = (T*)a.out_val;   // in place
    // panel load: one 16-value AO-row segment (rb, p, k) per item, vector loads,
    // kSegUnroll segments in flight per thread, transposed into the panel
    using V = typename Vec<T>::type;
    constexpr int kVPer = 16 / Vec<T>::n;   // vector loads per segment
    const int nseg = nk * 6 * NT;
    for (int s0 = threadIdx.x; s0 < nseg; s0 += blockDim.x * kSegUnroll) {
        V buf[kSegUnroll][kVPer];
#pragma unroll
        for (int u = 0; u < kSegUnroll; ++u) {
            const int sg = s0 + u * blockDim.x;
            if (sg < nseg) {
                const int rb = sg / (6 * NT), rem = sg - rb * (6 * NT), p = rem / 6, kr = rem - p * 6;
                const int sl = s_slot[rb][p];
                if (sl >= 0) {
                    const V* src = (const V*)(val + ((size_t)s_row[rb] * a.cap + sl) * kTileVals + kr * 16);
#pragma unroll
                    for (int v = 0; v < kVPer; ++v) buf[u][v] = src[v];
                } else {
#pragma unroll
                    for (int v = 0; v < kVPer; ++v) buf[u][v] = Vec<T>::zero();
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kSegUnroll; ++u) {
            const int sg = s0 + u * blockDim.x;
            if (sg < nseg) {
                const int rb = sg / (6 * NT), rem = sg - rb * (6 * NT), p = rem / 6, kr = rem - p * 6;
                const T* e2 = (const T*)buf[u];
                T* dst = panel + (p * 16) * NRP + rb * 6 + kr;
#pragma unroll
                for (int col = 0; col < 16; ++col) dst[col * NRP] = e2[col];
            }
        }
    }
    __syncthreads();
    constexpr int R = ApplyShape<T>::rows;
    const int row = threadIdx.x * R;
    // a warp whose rows hold only zeros in the block's tiles has nothing to update
    bool nzrow = false;
    if (row < nk * 6)
        for (int cidx = 0; cidx < NT * 16 && !nzrow; ++cidx)
#pragma unroll
            for (int r2 = 0; r2 < R; ++r2) nzrow |= nonzero(panel[cidx * NRP + row + r2]);
    const bool warp_busy = __any_sync(0xffffffffu, nzrow);
    if (row < nk * 6 && warp_busy) {
        T* pr = panel + row;
        for (int sub = 0; sub < kMaxSub; ++sub) {
            const int q1 = s_lvl[sub + 1];
            int q = s_lvl[sub];
            if (q == np) break;
            for (; q < q1; q += kUnroll) {
                if constexpr (R == 2) {
                    unsigned off[kUnroll];
                    float2 x[kUnroll], y[kUnroll];
                    float c0[kUnroll], c1[kUnroll];
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u) {
                        if (q + u < q1) {
                            off[u] = poff[q + u];
                            c0[u] = pcs[2 * (q + u)];
                            c1[u] = pcs[2 * (q + u) + 1];
                            x[u] = *(const float2*)(pr + (off[u] & 0xffffu));
                            y[u] = *(const float2*)(pr + (off[u] >> 16));
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u) {
                        if (q + u < q1) {
                            float2 xn, yn;
                            if (MODE == 0) {
                                const float2 cc = make_float2(c0[u], c0[u]);
                                xn = __ffma2_rn(cc, x[u], __fmul2_rn(make_float2(c1[u], c1[u]), y[u]));
                                yn = __ffma2_rn(cc, y[u], __fmul2_rn(make_float2(-c1[u], -c1[u]), x[u]));
                            } else {
                                const float2 nh = make_float2(-c0[u], -c0[u]);
                                xn = __ffma2_rn(nh, y[u], x[u]);
                                yn = __ffma2_rn(nh, x[u], y[u]);
                            }
                            *(float2*)(pr + (off[u] & 0xffffu)) = trunc2(xn, a.trunc_f);
                            *(float2*)(pr + (off[u] >> 16)) = trunc2(yn, a.trunc_f);
                        }
                    }
                } else {
                    unsigned off[kUnroll];
                    T x[kUnroll], y[kUnroll], c0[kUnroll], c1[kUnroll];
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u) {
                        if (q + u < q1) {
                            off[u] = poff[q + u];
                            c0[u] = pcs[2 * (q + u)];
                            c1[u] = pcs[2 * (q + u) + 1];
                            x[u] = pr[off[u] & 0xffffu];
                            y[u] = pr[off[u] >> 16];
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u) {
                        if (q + u < q1) {
                            T xn, yn;
                            if (MODE == 0) {
                                xn = c0[u] * x[u] + c1[u] * y[u];
                                yn = c0[u] * y[u] - c1[u] * x[u];
                            } else {
                                xn = x[u] - c0[u] * y[u];
                                yn = y[u] - c0[u] * x[u];
                            }
                            pr[off[u] & 0xffffu] = below(xn, a) ? (T)0 : xn;
                            pr[off[u] >> 16] = below(yn, a) ? (T)0 : yn;
                        }
                    }
                }
            }
        }
    }
    __syncthreads();
    for (int sg = threadIdx.x; sg < nseg; sg += blockDim.x) {
        const int rb = sg / (6 * NT), rem = sg - rb * (6 * NT), p = rem / 6, kr = rem - p * 6;
        const int sl = s_slot[rb][p];
        if (sl < 0) continue;
        V out[kVPer];
        T* e2 = (T*)out;
        const T* srcp = panel + (p * 16) * NRP + rb * 6 + kr;
        bool any = false;
#pragma unroll
        for (int col = 0; col < 16; ++col) {
            e2[col] = srcp[col * NRP];
            any |= nonzero(e2[col]);
        }
        if (any) {   // the tile may be nonzero now
            a.out_nz[(size_t)s_row[rb] * a.cap + sl] = 1;
            a.col_nz[s_cp[p] + k0 + rb] = 1;
        }
        V* dst = (V*)(val + ((size_t)s_row[rb] * a.cap + sl) * kTileVals + kr * 16);
#pragma unroll
        for (int v = 0; v < kVPer; ++v) dst[v] = out[v];
    }
}

// Sweeps, one warp at a time. Same updates, order and truncation as
// k_apply_colour; what differs is where the values sit and who waits for whom.
//
// A CTA serves a block (A, B) of the colour. It reads the tile flags of all the
// block's rows: one bit per row block with work (where every touched tile is
// flagged all-zero, the updates would leave the zeros as they are). The AO rows
// of the row blocks with work, six each, are the block's work, in runs of 32
// entries; CTA s of the block takes the s-th share of the runs, and its warps
// take run after run from it and work on them alone, so only a block's last run
// is not full. (A warp that listed its own chunk of the rows ran half-empty:
// 68.9 -> 45.8 ms for an occupied pass at 4096 molecules. CTAs that stay and
// take runs of other blocks when theirs are done were slower: 55 ms.)
//
// Two ways to run the updates of a block, by its number of pairs:
//   dense   both sides of an entry's AO rows in registers (two adjacent rows
//           packed in occupied passes, one in passes over all MOs). At level l
//           slot i pairs x_i with y_((l - i) mod n); y is held in slot order and
//           the value slot i has updated is the partner of slot i + 1 at the next
//           level, so writing it to register i + 1 rotates y without a move. A
//           slot without a pair has (c, t) = (0, 0), which leaves both values as
//           they are. Per slot two FMAs, a compare and a multiply per value, and
//           half a coefficient load: 7.6 clocks of an SM quarter per slot and row
//           packed, 8.2 unpacked, in a loop of its own; the FMA and ALU pipes
//           would take 4, the operand reads of the register file bound it. (In passes over
//           all MOs one warp per quarter of an SM waits for instructions of the unrolled
//           loops, results and barriers instead: 15 to 27 % of the issue slots used.)
//   list    the block's pairs one after the other in schedule order, both sides
//           in a shared-memory panel [column][lane], one AO row per lane, up to
//           four pairs of a level in flight. Self blocks, rotations, combination
//           blocks with few pairs, and everything in FP64 storage, where the FP64
//           pipe (two lanes per clock and SM) is the bound and slots without a
//           pair are not to cost anything: there a CTA's warps share the panel
//           and each level's pairs.
// n = max(MOs of A, MOs of B) is the modulus of the in-block colour; the dense
// loop exists for every n a pair of groups can have, so blocks of partly filled
// groups run it as well (their missing MOs are zero columns without pairs).
// Measured (one pass or sweep, FP32; before: full groups in a kernel with one
// side in registers, the others staged for the generic kernel): occupied pass
// at 4096 molecules 68.9 -> 41.9 ms, at 997 9.9 -> 5.3; four passes over all
// MOs at 512 18.6 -> 5.2; rotations at 4096 14.8 -> 9.6, at 997 3.2 -> 1.7.
// FP64 at 343 molecules: occupied pass 14.5 -> 10.4, rotations 2.3 -> 1.5.
constexpr int kFullCH = 32;                  // row blocks per word of the bits of rows with work
constexpr int kFullBatch = 8;                // 16-byte pieces of a tile per lane and run of 32 row pairs, all in flight
// runs a CTA takes at least: one per warp, or two where a launch could have more than kWsManyRuns
// runs per CTA that its registers leave room for (at 4096 molecules most shares are empty, and fewer of
// them are launched: 43.0 -> 41.9 ms; at 997 one per warp spreads better, 5.8 -> 5.3; passes over all MOs
// at 700, where the line lies near 900 molecules, 7.6 ms against 8.3 with two)
constexpr int kWsManyRuns = 32;
// rotations: CTAs of a launch as a multiple of the resident ones (2, 4, 8, 16: 13.8, 10.8, 9.6, 9.5 ms
// at 4096 molecules, 1.91, 1.88, 1.74, 1.74 at 997)
constexpr int kWsRotWaves = 8;
// combinations: the same limit. Without one a colour's CTAs grow with the square of the cluster (12,288 at
// 4096 molecules, 3.1 million at 65,536), nearly all without a row of work, and each reads its block's flags
// to find that out. Occupied pass, limits 2, 4, 8, 16, 32 and none: 41.8, 38.8, 38.0, 37.1, 37.1, 37.1 ms at
// 4096 molecules; 135, 123, 119, 120, 122, 127 at 8192; 357, 349, 342, 340, 347, 502 at 32,768; 750, 750, 745,
// 741, 744, 1503 at 65,536; FP64 at 1000 108, 98.4, 95.0, 93.0, 93.1, 93.1. Four passes over all MOs, limits 4, 8,
// 16, 32, 64 and none: 43.2, 42.9, 41.9, 43.8, 51.7, 68.0 at 4096; 714, 714, 714, 741, 771, 10593 at 65,536.
constexpr int kWsCombWaves = 16;
constexpr int kWsPad = 34;                   // floats per panel column: 16-byte pieces scatter over all banks
// pairs from which a combination block runs dense, as a divisor of n^2: the dense loop costs
// ~8 n^2 clocks per row whatever the number of pairs, the list ~15 per pair with more latency (3, 4,
// 8: 5.7, 5.35, 5.2 ms for the passes over all MOs at 512 molecules; few blocks lie in between later)
constexpr int kWsDenseDiv = 8;
// MODE 0 rotations, MODE 1 combinations of occupied MOs (ALL = false) or of all MOs
template <typename T, int MODE, bool ALL> struct WarpShape {
    static constexpr bool f32 = std::is_same<T, float>::value;
    static constexpr int nta = ALL ? 3 : 2;                    // side tiles
    static constexpr int ntb = MODE == 0 ? 1 : nta;
    static constexpr int nmax = ALL ? 48 : 32;                 // largest modulus
    static constexpr int gstep = ALL ? 6 : 4;                  // MOs per molecule and side
    // warps that share a run: FP32 one; FP64 all four of the CTA, each a quarter of a level's pairs (a
    // quarter of an SM starts one FP64 instruction of a warp every 64 clocks, busy or not; with a run
    // per warp a colour of few blocks left most quarters idle: occupied pass at 343 molecules 12.7 ms,
    // now 10.4; a step's sweeps at 32 0.44 ms, now 0.19)
    static constexpr int warps = 4, threads = 32 * warps;
    static constexpr int team = f32 ? 1 : warps, runs = warps / team;   // runs a CTA has in hand
    // order of the CTAs: all shares of a block, then the next block (the long blocks first: the short
    // ones even out the end; FP64 occupied pass at 343 molecules 15.9 -> 12.7 ms, rotations at 4096
    // 9.7 -> 9.2), or the first share of all blocks, then the second (FP32 combinations, whose later
    // shares are the empty ones: 5.2 against 5.6 ms at 512 molecules)
    static constexpr bool by_block = !f32 || MODE == 0;
    static constexpr int halves = f32 && MODE == 1 && !ALL ? 2 : 1;   // AO rows of an entry in the dense loop
    // bytes of the block's coefficients or pairs, with four entries ending the list. FP32: at most
    // kRotCap rotations of 16; a dense table of n^2 (c, t), or 8-byte combinations (fewer than
    // n^2 / kWsDenseDiv, or n (n - 1) / 2 of a self block). FP64: coefficients, then the 4-byte words.
    static constexpr int cap = (MODE == 0 ? kRotCap : nmax * nmax) + 4;
    static constexpr int table = f32 ? (MODE == 0 ? cap * 16 : nmax * nmax * 8) : cap * (MODE == 0 ? 20 : 12);
    static_assert(MODE == 0 || (nmax * (nmax - 1) / 2 + 4) * 8 <= nmax * nmax * 8, "");
    static_assert(table % 16 == 0, "");
    // bytes per warp: the list's panel; the dense loop's: one side of 32 row pairs (occupied passes),
    // or a run's tiles as they lie in memory and the next run's (passes over all MOs)
    static constexpr int raw = f32 && ALL ? (nta + ntb) * 32 * 64 : 0;
    static constexpr int panel = (nta + ntb) * 16 * kWsPad * (int)sizeof(T);
    static constexpr int per_warp = 2 * raw > panel ? 2 * raw : panel;
    static_assert(MODE == 0 || ALL || per_warp >= nta * 16 * 64 * 4, "");
    static constexpr size_t smem = (size_t)table + (size_t)runs * per_warp;   // + row bits
    // CTAs per SM the register budget is cut for: the dense loop holds 2 n values per row; FP64 runs as
    // many as its panels leave room for
    static constexpr int min_ctas = f32 ? (MODE == 0 ? 6 : (ALL ? 2 : 3)) : (MODE == 0 ? 6 : (ALL ? 3 : 5));
    // resident CTAs: as many, but in FP32 passes over all MOs, whose 117 KB leave room for one (four
    // warps, one per quarter of an SM)
    static constexpr int fit = kSmSmem / ((int)smem + 1024), resident = fit < min_ctas ? fit : min_ctas;
    static constexpr int many_runs = kWsManyRuns * min_ctas / resident;
};

// 1.0 where |v| >= t, 0.0 below (and for NaN): one compare that writes the
// factor itself
__device__ __forceinline__ float ge_abs_factor(float v, float t) {
    float k;
    asm("set.ge.f32.f32 %0, %1, %2;" : "=f"(k) : "f"(fabsf(v)), "f"(t));
    return k;
}

// v with a value below t in magnitude set to zero, as a product with a 0/1
// factor: a compare on the ALU pipe and a multiply on the FMA pipe instead of a
// compare and a select on the ALU pipe, which has half the rate (a value set to
// zero may come out as -0, which every later test treats as zero)
__device__ __forceinline__ float trunc_mul(float v, float t) { return __fmul_rn(v, ge_abs_factor(v, t)); }
__device__ __forceinline__ float fma_s(float c, float a, float b) { return __fmaf_rn(c, a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

__device__ __forceinline__ float2 trunc_mul(float2 v, float t) {
    return __fmul2_rn(v, make_float2(ge_abs_factor(v.x, t), ge_abs_factor(v.y, t)));
}
__device__ __forceinline__ float2 fma_s(float c, float2 a, float2 b) { return __ffma2_rn(make_float2(c, c), a, b); }

// The NS levels of a block on a lane's AO rows (V: one, or two packed). Slots
// run downwards: the updated partner of slot i goes to register i + 1, whose old
// value slot i + 1 has already used; slot NS - 1's goes to register 0 at the end
// of the level.
template <int NS, typename V>
__device__ __forceinline__ void dense_levels(V (&x)[NS], V (&ys)[NS], const float2* coef) {
    static_assert(NS % 2 == 0, "");
#pragma unroll 1
    for (int lv = 0; lv < NS; ++lv) {
        const float4* c4 = (const float4*)(coef + lv * NS);
        V carry;
#pragma unroll
        for (int h = NS / 2 - 1; h >= 0; --h) {
            const float4 q = c4[h];
#pragma unroll
            for (int u = 1; u >= 0; --u) {
                const int i = 2 * h + u;
                const float c = u ? q.z : q.x, t = u ? q.w : q.y;
                const V xn = fma_s(c, ys[i], x[i]);
                const V yn = fma_s(c, x[i], ys[i]);
                x[i] = trunc_mul(xn, t);
                const V yt = trunc_mul(yn, t);
                if (i == NS - 1) carry = yt;
                else ys[i + 1] = yt;
            }
        }
        ys[0] = carry;
    }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool in) {   // zeros where !in
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = in ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

// What a CTA of k_apply_warp needs to start on block q of the pass (colour
// order), gathered once per sweep so that it costs one load instead of a chain
// of dependent ones: (block, pairs, touched tiles, rows), (column lists of the
// sides' first tiles, rows of B, molecules of A and of B), (column lists of the
// sides' virtual tiles in passes over all MOs), (flags of each side's tiles).
struct BlockInfo {
    int4 i0, i1, i2;
    int flagA[3], flagB[3];
};
template <int MODE, bool ALL>
__global__ void k_block_info(SweepArgs a, int n, BlockInfo* __restrict__ info) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const int e = a.blk[q];
    const int A = a.gnb_row[e], B = a.gnb_col[e];
    const int ta0 = a.group_ot0[A], tb0 = MODE == 0 ? a.group_vt0[B] : a.group_ot0[B];
    const int pa = a.cci_ptr[ta0], pb = a.cci_ptr[tb0];
    int touch = a.pr_touch[e];
    const bool same = MODE == 1 && A == B;
    if (same) touch |= touch >> 3;   // one set of tiles, held as side A
    BlockInfo b;
    b.i0 = make_int4(e, a.pr_n[e], touch, a.cci_ptr[ta0 + 1] - pa);
    b.i1 = make_int4(pa, pb, a.cci_ptr[tb0 + 1] - pb, a.group_nmol[A] | (a.group_nmol[B] << 8) | ((int)same << 16));
    b.i2 = make_int4(ALL ? a.cci_ptr[a.group_vt0[A]] : 0, ALL ? a.cci_ptr[a.group_vt0[B]] : 0, 0, 0);
    for (int t = 0; t < 3; ++t) {
        const int ta = t < a.group_not[A] ? ta0 + t : a.group_vt0[A];
        const int tb = MODE == 0 ? tb0 : (t < a.group_not[B] ? tb0 + t : a.group_vt0[B]);
        b.flagA[t] = flag_base(ta, a.cci_ptr[ta]);
        b.flagB[t] = flag_base(tb, a.cci_ptr[tb]);
    }
    info[q] = b;
    // the 2x2 row updates the algorithm defines, rows proven unchanged and skipped included
    const int col = a.gnb_colour[e];
    if (b.i0.y && col >= a.col_lo && col < a.col_hi)
        atomicAdd(a.upd, (unsigned long long)b.i0.y * (unsigned long long)(b.i0.w * kAoPerMol));
}

template <typename T, int MODE, bool ALL>
__global__ void __launch_bounds__((WarpShape<T, MODE, ALL>::threads), (WarpShape<T, MODE, ALL>::min_ctas))
k_apply_warp(SweepArgs a, int p0, int nb, int min_runs) {
    using Sh = WarpShape<T, MODE, ALL>;
    constexpr bool F32 = Sh::f32;
    constexpr int kWsWarps = Sh::warps, kWsThreads = Sh::threads;
    constexpr int NTA = Sh::nta, NTB = Sh::ntb;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int s_wsum[kWsWarps], s_next, s_lvl[Sh::team > 1 ? kMaxSub + 1 : 1];
    // The next colour's CTAs may start once all of these have, and wait below for these to end: what a
    // CTA reads before that was written before the sweep's first colour.
    asm volatile("griddepcontrol.launch_dependents;");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const BlockInfo& info = ((const BlockInfo*)a.blk_info)[p0 + (Sh::by_block ? blockIdx.x / (gridDim.x / nb) : blockIdx.x % nb)];
    const int4 i0 = info.i0, i1 = info.i1, i2 = info.i2;
    const int e = i0.x, np = i0.y, touch = i0.z, n_rows = i0.w;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (np == 0 || (*a.err & (kErrCapacity | kErrSortSize))) return;
    const int pa = i1.x, pb = i1.y;
    if (i1.z != n_rows) {
        if (threadIdx.x == 0) atomicOr(a.err, kErrCapacity);
        return;
    }
    const int mA = i1.w & 255, mB = (i1.w >> 8) & 255;
    const bool same = (i1.w >> 16) & 1;
    // occupied MOs and tiles of both sides, MOs of the pass on each side
    const int noA = 4 * mA, noB = MODE == 0 ? 0 : 4 * mB;
    const int otA = (noA + 15) >> 4, otB = MODE == 0 ? 0 : (noB + 15) >> 4;
    const int nA = MODE == 0 ? noA : Sh::gstep * mA, nB = MODE == 0 ? 2 * mB : Sh::gstep * mB;
    const int n = max(nA, nB);
    // bits of the row blocks with work, 16 flags per load (a tile's flags start on 16 bytes and are
    // zero past its last row), then the bits before each word
    unsigned* bits = (unsigned*)(smraw + Sh::smem);
    const int nw = (n_rows + kFullCH - 1) / kFullCH;
    int* wpre = (int*)(bits + nw);
    for (int hw = threadIdx.x; hw < 2 * nw; hw += kWsThreads) {
        uint4 f = make_uint4(0u, 0u, 0u, 0u);
        if (16 * hw < n_rows) {
#pragma unroll
            for (int t = 0; t < NTA + NTB; ++t) {
                const bool sideB = t >= NTA;
                const int tt = sideB ? t - NTA : t;
                if (!(touch >> (sideB ? 3 + tt : tt) & 1)) continue;
                const uint4 v = *(const uint4*)(a.col_nz + (sideB ? info.flagB[tt] : info.flagA[tt]) + 16 * (size_t)hw);
                f.x |= v.x;
                f.y |= v.y;
                f.z |= v.z;
                f.w |= v.w;
            }
        }
        // four 0/1 bytes of a word to four bits: byte i lands on bit 24 + i
        constexpr unsigned kGather = 0x01020408u;
        ((unsigned short*)bits)[hw] = (unsigned short)((f.x * kGather >> 24 & 15u) | (f.y * kGather >> 24 & 15u) << 4 |
                                                       (f.z * kGather >> 24 & 15u) << 8 | (f.w * kGather >> 24 & 15u) << 12);
    }
    __syncthreads();
    const int wper = (nw + kWsThreads - 1) / kWsThreads;
    const int wlo = min(nw, (int)threadIdx.x * wper), whi = min(nw, wlo + wper);
    int cnt = 0;
    for (int w = wlo; w < whi; ++w) cnt += __popc(bits[w]);
    int inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) s_wsum[warp] = inc;
    __syncthreads();
    int n_work = 0, before = inc - cnt;
#pragma unroll
    for (int w = 0; w < kWsWarps; ++w) {
        before += w < warp ? s_wsum[w] : 0;
        n_work += s_wsum[w];
    }
    const bool dense = F32 && MODE == 1 && !same && np * kWsDenseDiv >= n * n;
    const int hh = dense ? Sh::halves : 1;   // AO rows of a lane's entry (adjacent ones)
    const int n_ent = kAoPerMol / hh * n_work, n_run = (n_ent + 31) / 32;
    const int shares = gridDim.x / nb, share = Sh::by_block ? blockIdx.x % shares : blockIdx.x / nb;
    const int per = max(min_runs, (n_run + shares - 1) / shares);
    const int run_lo = share * per, run_hi = min(n_run, run_lo + per);
    if (run_lo >= run_hi) return;
    if (threadIdx.x == 0) s_next = run_lo;
    if constexpr (Sh::team > 1)
        for (int l = threadIdx.x; l <= kMaxSub; l += kWsThreads) s_lvl[l] = a.pr_lvl[(size_t)e * (kMaxSub + 1) + l];
    for (int w = wlo; w < whi; ++w) {
        wpre[w] = before;
        before += __popc(bits[w]);
    }
    // panel column of a side's local MO: occupied MOs from column 0, virtual ones (passes over
    // all MOs) from the tile after the occupied ones
    auto colA = [&](int i) { return MODE == 0 || !ALL || i < noA ? i : 16 * otA + i - noA; };
    auto colB = [&](int j) { return MODE == 0 || !ALL || j < noB ? j : 16 * otB + j - noB; };
    // table (dense) or list of the block's pairs
    const T* cs = (const T*)a.pr_cs + (size_t)e * kOrthoCap * 2;
    const uint16_t* ij = a.pr_ij + (size_t)e * kOrthoCap;
    float2* table = (float2*)smraw;
    float2* pair2 = (float2*)smraw;
    float4* pair4 = (float4*)smraw;
    double* coef64 = (double*)smraw;                                                     // FP64: c, or c and s
    unsigned* word64 = (unsigned*)(coef64 + (size_t)Sh::cap * (MODE == 0 ? 2 : 1));
    if (dense) {
        for (int i = threadIdx.x; i < n * n; i += kWsThreads) table[i] = make_float2(0.f, 0.f);
        __syncthreads();
    }
    for (int q = threadIdx.x; q < np; q += kWsThreads) {
        const int w = ij[q], il = w & 255, jl = w >> 8;
        const int s = il + jl, lv = s >= n ? s - n : s;
        // list: panel offsets of both sides (12 bits each) and, between them, the level
        const unsigned off = (unsigned)(colA(il) * kWsPad) | (unsigned)lv << 12 |
                             ((unsigned)(((same ? 0 : 16 * NTA) + colB(jl)) * kWsPad) << 18);
        if constexpr (F32) {
            const float2 c = ((const float2*)cs)[q];
            if constexpr (MODE == 0) pair4[q] = make_float4(__uint_as_float(off), c.x, c.y, 0.f);
            else if (dense) table[lv * n + il] = make_float2(-c.x, a.trunc_f);
            else pair2[q] = make_float2(__uint_as_float(off), -c.x);
        } else {
            if constexpr (MODE == 0) {
                coef64[2 * q] = cs[2 * q];
                coef64[2 * q + 1] = cs[2 * q + 1];
            } else {
                coef64[q] = -cs[2 * q];
            }
            word64[q] = off;
        }
    }
    if (!dense && threadIdx.x < 4) {   // ends the list: a level of its own
        const int q = np + threadIdx.x;
        if constexpr (!F32) word64[q] = 63u << 12;
        else if constexpr (MODE == 0) pair4[q] = make_float4(__uint_as_float(63u << 12), 0.f, 0.f, 0.f);
        else pair2[q] = make_float2(__uint_as_float(63u << 12), 0.f);
    }
    __syncthreads();
    T* const mem = (T*)(smraw + Sh::table + (size_t)(warp / Sh::team) * Sh::per_warp);   // the run's
    T* const val = (T*)a.out_val;                                           // in place
    // the block's pairs on the panel, in schedule order (lanes hold different rows)
    auto run_list = [&](bool active) {
        // pairs of one level touch different columns: up to four of them in flight
        {
            auto upd = [&](int q, auto width) {
                constexpr int N = decltype(width)::value;
                T *px[N], *py[N], xv[N], yv[N], c0[N], c1[N];
#pragma unroll
                for (int u = 0; u < N; ++u) {
                    unsigned off;
                    if constexpr (!F32) {
                        off = word64[q + u];
                        c0[u] = coef64[MODE == 0 ? 2 * (q + u) : q + u];
                        c1[u] = MODE == 0 ? coef64[2 * (q + u) + 1] : 0.0;
                    } else if constexpr (MODE == 0) {
                        const float4 c = pair4[q + u];
                        off = __float_as_uint(c.x);
                        c0[u] = c.y;
                        c1[u] = c.z;
                    } else {
                        const float2 c = pair2[q + u];
                        off = __float_as_uint(c.x);
                        c0[u] = c.y;
                        c1[u] = 0.f;
                    }
                    px[u] = mem + (off & 0xfffu) + lane;
                    py[u] = mem + (off >> 18) + lane;
                    xv[u] = *px[u];
                    yv[u] = *py[u];
                }
#pragma unroll
                for (int u = 0; u < N; ++u) {
                    T xn, yn;
                    if constexpr (MODE == 0) {
                        xn = fma(c0[u], xv[u], mul_rn(c1[u], yv[u]));
                        yn = fma(c0[u], yv[u], mul_rn(-c1[u], xv[u]));
                    } else {
                        xn = fma(c0[u], yv[u], xv[u]);
                        yn = fma(c0[u], xv[u], yv[u]);
                    }
                    *px[u] = below(xn, a) ? (T)0 : xn;
                    *py[u] = below(yn, a) ? (T)0 : yn;
                }
            };
            auto level = [&](int q) {
                unsigned off;
                if constexpr (!F32) off = word64[q];
                else if constexpr (MODE == 0) off = __float_as_uint(pair4[q].x);
                else off = __float_as_uint(pair2[q].x);
                return off >> 12 & 63u;
            };
            if constexpr (Sh::team > 1) {   // a level's pairs, a warp's share each
                for (int l = 0; l < kMaxSub; ++l) {
                    const int q0 = s_lvl[l], q1 = s_lvl[l + 1], part = (q1 - q0 + Sh::team - 1) / Sh::team;
                    const int end = min(q1, q0 + (warp + 1) * part);
                    if (active)
                        for (int q = q0 + warp * part; q < end;) {
                            if (q + 4 <= end) {
                                upd(q, std::integral_constant<int, 4>());
                                q += 4;
                            } else if (q + 2 <= end) {
                                upd(q, std::integral_constant<int, 2>());
                                q += 2;
                            } else {
                                upd(q, std::integral_constant<int, 1>());
                                q += 1;
                            }
                        }
                    if (q1 > q0) __syncthreads();
                }
                return;
            }
            if (!active) return;
            for (int q = 0; q < np;) {
                const unsigned l = level(q);
                if (level(q + 3) == l) {
                    upd(q, std::integral_constant<int, 4>());
                    q += 4;
                } else if (level(q + 1) == l) {
                    upd(q, std::integral_constant<int, 2>());
                    q += 2;
                } else {
                    upd(q, std::integral_constant<int, 1>());
                    q += 1;
                }
            }
        }
    };
    // 16-byte pieces of an AO row of a tile, rows a warp moves at a time, and a lane's row and piece
    using V = typename std::conditional<F32, float4, double2>::type;
    constexpr int kV = 16 / (int)sizeof(T), kPieces = 16 / kV, kAt = 32 / kPieces, kTimes = 32 / kAt;
    const int qe = lane / kPieces, qp = lane % kPieces;
    // an AO row of a run: the tiles (row block * cap + slot) its first occupied tile and its virtual
    // one have on either side, and 8 * position in the block's row list + AO row of the row block
    struct Row {
        unsigned a, b, av, bv;
        int k;
    };
    auto look_up = [&](int run) {
        Row r{0, 0, 0, 0, 0};
        const int idx = 32 * run + lane, per_mol = kAoPerMol / hh;
        if (idx >= n_ent) return r;
        const int rank = hh == 2 ? idx / 3 : idx / kAoPerMol;   // its row block is the rank-th set bit
        int lo = 0, hi = nw;                // last word with wpre <= rank
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (wpre[mid] <= rank) lo = mid;
            else hi = mid;
        }
        unsigned w = bits[lo];
        int left = rank - wpre[lo], pos = 0;
#pragma unroll
        for (int half = 16; half > 0; half >>= 1) {
            const unsigned low = w & ((1u << half) - 1u);
            const int c = __popc(low);
            if (left >= c) {
                left -= c;
                pos += half;
                w >>= half;
            } else {
                w = low;
            }
        }
        const int k = 32 * lo + pos;
        const unsigned row0 = (unsigned)a.cci_row[pa + k] * (unsigned)a.cap;
        r.a = row0 + (unsigned)a.cci_slot[pa + k];
        r.b = row0 + (unsigned)a.cci_slot[pb + k];
        if constexpr (ALL) {
            r.av = row0 + (unsigned)a.cci_slot[i2.x + k];
            r.bv = row0 + (unsigned)a.cci_slot[i2.y + k];
        }
        r.k = 8 * k + (idx - per_mol * rank) * hh;
        return r;
    };
    auto touched = [&](int t) { return (touch >> (t >= NTA ? 3 + t - NTA : t) & 1) && !(t >= NTA && same); };
    // panel tile t of a row, and the row's 16 values there
    auto tile_of = [&](const Row& r, int t) {
        const bool sideB = t >= NTA;
        const int tt = sideB ? t - NTA : t;
        if (ALL && tt >= (sideB ? otB : otA)) return sideB ? r.bv : r.av;
        return (sideB ? r.b : r.a) + (unsigned)tt;
    };
    auto values = [&](const Row& r, unsigned tile) { return val + (size_t)tile * kTileVals + (r.k & 7) * kTileW; };
    // of a value written nonzero: the tile's flags (1 only means "may be nonzero")
    auto raise = [&](const Row& r, int t, unsigned tile) {
        a.out_nz[tile] = 1;
        a.col_nz[(t >= NTA ? info.flagB[t - NTA] : info.flagA[t]) + (r.k >> 3)] = 1;
    };
    auto row_from = [&](const Row& r, int src) {   // lane src's row
        Row o{0, 0, 0, 0, 0};
        o.a = __shfl_sync(0xffffffffu, r.a, src);
        o.b = __shfl_sync(0xffffffffu, r.b, src);
        if constexpr (ALL) {
            o.av = __shfl_sync(0xffffffffu, r.av, src);
            o.bv = __shfl_sync(0xffffffffu, r.bv, src);
        }
        o.k = __shfl_sync(0xffffffffu, r.k, src);
        return o;
    };
    auto grab = [&]() { return lane == 0 ? atomicAdd(&s_next, 1) : 0; };
    int run = run_lo;
    if constexpr (Sh::team == 1) run = __shfl_sync(0xffffffffu, grab(), 0);
    if (run >= run_hi) return;
    if (MODE == 0 || !dense) {
        T* const pq = mem + kV * qp * kWsPad + qe;
        // tiles in flight; a team's warps move different tiles
        constexpr int kTiles = F32 ? NTA + NTB : 1;
        const int t_lo = Sh::team > 1 ? warp : 0;
        auto all_wait = [] {
            if constexpr (Sh::team > 1) __syncthreads();
            else __syncwarp();
        };
        while (run < run_hi) {
            const Row r = look_up(run);
            int grabbed = run + 1;
            if constexpr (Sh::team == 1) grabbed = grab();
            const int take = min(32, n_ent - 32 * run);
#pragma unroll
            for (int t0 = t_lo; t0 < NTA + NTB; t0 += kTiles * Sh::team) {
                V v[kTiles][kTimes];
#pragma unroll
                for (int u = 0; u < kTimes; ++u) {
                    const Row o = row_from(r, kAt * u + qe);
#pragma unroll
                    for (int t = 0; t < kTiles; ++t) {
                        v[t][u] = V{};
                        if (t0 + t < NTA + NTB && kAt * u + qe < take && touched(t0 + t))
                            v[t][u] = *((const V*)values(o, tile_of(o, t0 + t)) + qp);
                    }
                }
#pragma unroll
                for (int t = 0; t < kTiles && t0 + t < NTA + NTB; ++t)
#pragma unroll
                    for (int u = 0; u < kTimes; ++u)
#pragma unroll
                        for (int w = 0; w < kV; ++w)
                            pq[((t0 + t) * 16 + w) * kWsPad + kAt * u] = ((const T*)&v[t][u])[w];
            }
            all_wait();
            run_list(lane < take);
            all_wait();
#pragma unroll
            for (int u = 0; u < kTimes; ++u) {
                const Row o = row_from(r, kAt * u + qe);
                if (kAt * u + qe >= take) continue;
#pragma unroll
                for (int t = t_lo; t < NTA + NTB; t += Sh::team) {
                    if (!touched(t)) continue;
                    V f;
                    bool nz = false;
#pragma unroll
                    for (int w = 0; w < kV; ++w) {
                        const T x = pq[(t * 16 + w) * kWsPad + kAt * u];
                        ((T*)&f)[w] = x;
                        nz |= nonzero(x);
                    }
                    const unsigned tile = tile_of(o, t);
                    *((V*)values(o, tile) + qp) = f;
                    if (nz) raise(o, t, tile);
                }
            }
            all_wait();
            run = Sh::team > 1 ? grabbed : __shfl_sync(0xffffffffu, grabbed, 0);
        }
        return;
    }
    // an occupied pass: 32 row pairs per run. Eight lanes move one contiguous 128-byte row pair of a
    // tile; a per-warp panel [column][lane] of packed rows, one side at a time, turns it around.
    if constexpr (F32 && MODE == 1 && !ALL) {
        float2* const panel = (float2*)mem;
        const int le = lane >> 3, lp = lane & 7;            // entry (mod 4) and 16-byte piece a lane moves
        const int prow = lp >> 2, pcol = 4 * (lp & 3);      // the piece's row of the pair and first column
        // a column's entries are rotated by its quarter of the tile: the pieces of eight lanes, and a
        // column of all lanes, hit all banks
        auto at = [&](int col) { return panel + col * 32 + ((lane + (col & 12)) & 31); };
        auto part = [&](int t, int u) {
            return (float*)panel + ((16 * t + pcol) * 32 + ((4 * u + le + pcol) & 31)) * 2 + prow;
        };
        auto one_run = [&](auto ns) {
            constexpr int NS = decltype(ns)::value;
            const int take = n_ent - 32 * run;
            const Row r = look_up(run);
            float4 v[NTA + NTB][kFullBatch];
#pragma unroll
            for (int u = 0; u < kFullBatch; ++u) {
                const Row o = row_from(r, 4 * u + le);
#pragma unroll
                for (int t = 0; t < NTA + NTB; ++t) {
                    v[t][u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (4 * u + le < take && touched(t)) v[t][u] = *((const float4*)values(o, tile_of(o, t)) + lp);
                }
            }
            auto put = [&](int t0) {
#pragma unroll
                for (int t = 0; t < NTA; ++t)
#pragma unroll
                    for (int u = 0; u < kFullBatch; ++u) {
                        float* d = part(t, u);
                        d[0] = v[t0 + t][u].x;
                        d[64] = v[t0 + t][u].y;
                        d[128] = v[t0 + t][u].z;
                        d[192] = v[t0 + t][u].w;
                    }
                __syncwarp();
            };
            // y in slot order: level 0 pairs slot i with y_(-i mod n), and after n levels the order is
            // the same again
            float2 x[NS], ys[NS];
            put(0);
#pragma unroll
            for (int i = 0; i < NS; ++i) x[i] = i < nA ? *at(i) : make_float2(0.f, 0.f);
            __syncwarp();
            put(NTA);
#pragma unroll
            for (int i = 0; i < NS; ++i) ys[i] = (NS - i) % NS < nB ? *at((NS - i) % NS) : make_float2(0.f, 0.f);
            dense_levels<NS>(x, ys, table);
            // panel -> tiles, up to the side's last MO (four per molecule: a piece is never cut)
            auto store = [&](bool sideB) {
                __syncwarp();
#pragma unroll
                for (int u = 0; u < kFullBatch; ++u) {
                    const Row o = row_from(r, 4 * u + le);
                    if (4 * u + le >= take) continue;
#pragma unroll
                    for (int t = 0; t < NTA; ++t) {
                        const int pt = sideB ? NTA + t : t;
                        if (!touched(pt) || 16 * t + pcol >= (sideB ? noB : noA)) continue;
                        const float* d = part(t, u);
                        const float4 f = make_float4(d[0], d[64], d[128], d[192]);
                        const unsigned tile = tile_of(o, pt);
                        *((float4*)values(o, tile) + lp) = f;
                        if (f.x != 0.f || f.y != 0.f || f.z != 0.f || f.w != 0.f) raise(o, pt, tile);
                    }
                }
                __syncwarp();
            };
            __syncwarp();
#pragma unroll
            for (int i = 0; i < NS; ++i)
                if ((NS - i) % NS < nB) *at((NS - i) % NS) = ys[i];
            store(true);
#pragma unroll
            for (int i = 0; i < NS; ++i)
                if (i < nA) *at(i) = x[i];
            store(false);
        };
        while (run < run_hi) {
            switch (n / Sh::gstep) {
                case 1: one_run(std::integral_constant<int, 1 * Sh::gstep>()); break;
                case 2: one_run(std::integral_constant<int, 2 * Sh::gstep>()); break;
                case 3: one_run(std::integral_constant<int, 3 * Sh::gstep>()); break;
                case 4: one_run(std::integral_constant<int, 4 * Sh::gstep>()); break;
                case 5: one_run(std::integral_constant<int, 5 * Sh::gstep>()); break;
                case 6: one_run(std::integral_constant<int, 6 * Sh::gstep>()); break;
                case 7: one_run(std::integral_constant<int, 7 * Sh::gstep>()); break;
                default: one_run(std::integral_constant<int, 8 * Sh::gstep>()); break;
            }
            run = __shfl_sync(0xffffffffu, grab(), 0);
        }
    }
    // a pass over all MOs: 32 AO rows per run, whose tiles come in by cp.async while the run before
    // computes
    if constexpr (F32 && MODE == 1 && ALL) {
        // where piece p (columns 4p .. 4p + 3) of panel tile t of the run's row e lies: eight lanes
        // reading the same piece of consecutive rows hit all banks
        auto at = [&](int buf, int t, int e, int p) {
            return mem + buf * (Sh::raw / 4) + ((t * 32 + e) * 16 + 4 * (p ^ ((e >> 1) & 3)));
        };
        auto fetch = [&](int buf, int run_) {
            const int take = n_ent - 32 * run_;
            const Row r = look_up(run_);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const Row o = row_from(r, 8 * u + qe);
                const int e = 8 * u + qe;
#pragma unroll
                for (int t = 0; t < NTA + NTB; ++t)
                    cp_async16(at(buf, t, e, qp), values(o, tile_of(o, t)) + 4 * qp, e < take && touched(t));
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        fetch(0, run);
        int run2 = __shfl_sync(0xffffffffu, grab(), 0);
        int buf = 0;
        auto one_run = [&](auto ns) {
            constexpr int NS = decltype(ns)::value;
            const int take = n_ent - 32 * run;
            float x[NS], ys[NS];
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
            // column of a panel side in a lane's own row (scalar accesses: virtual MOs may follow a
            // partly filled occupied tile)
            auto column = [&](int t0, int col) {
                return at(buf, t0 + (col >> 4), lane, (col >> 2) & 3) + (col & 3);
            };
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                x[i] = i < nA ? *column(0, colA(i)) : 0.f;
                ys[i] = (NS - i) % NS < nB ? *column(NTA, colB((NS - i) % NS)) : 0.f;
            }
            if (run2 < run_hi) fetch(1 - buf, run2);
            dense_levels<NS>(x, ys, table);
            // back to the run's buffer (columns without an MO still hold what they held), then four
            // lanes per 64-byte row
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                if (i < nA) *column(0, colA(i)) = x[i];
                if ((NS - i) % NS < nB) *column(NTA, colB((NS - i) % NS)) = ys[i];
            }
            const Row r = look_up(run);
            __syncwarp();
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const Row o = row_from(r, 8 * u + qe);
                if (8 * u + qe >= take) continue;
#pragma unroll
                for (int t = 0; t < NTA + NTB; ++t) {
                    if (!touched(t)) continue;
                    const float4 f = *(const float4*)at(buf, t, 8 * u + qe, qp);
                    const unsigned tile = tile_of(o, t);
                    *((float4*)values(o, tile) + qp) = f;
                    if (f.x != 0.f || f.y != 0.f || f.z != 0.f || f.w != 0.f) raise(o, t, tile);
                }
            }
            __syncwarp();
        };
        while (run < run_hi) {
            const int grabbed = grab();   // the run after the next one
            switch (n / Sh::gstep) {
                case 1: one_run(std::integral_constant<int, 1 * Sh::gstep>()); break;
                case 2: one_run(std::integral_constant<int, 2 * Sh::gstep>()); break;
                case 3: one_run(std::integral_constant<int, 3 * Sh::gstep>()); break;
                case 4: one_run(std::integral_constant<int, 4 * Sh::gstep>()); break;
                case 5: one_run(std::integral_constant<int, 5 * Sh::gstep>()); break;
                case 6: one_run(std::integral_constant<int, 6 * Sh::gstep>()); break;
                case 7: one_run(std::integral_constant<int, 7 * Sh::gstep>()); break;
                default: one_run(std::integral_constant<int, 8 * Sh::gstep>()); break;
            }
            buf ^= 1;
            run = run2;
            run2 = __shfl_sync(0xffffffffu, grabbed, 0);
        }
    }
}

// drop tiles whose 6x16 values are all zero; in -> out
// (skipped entirely when an earlier kernel of the pass set the error word:
// `out` is then the pass's untouched input and stays as it was).
// One CTA per row block: a warp per tile marks the nonzero tiles in a shared
// bitmask, one thread turns the mask into word offsets, and the warps copy the
// nonzero tiles to their compacted slots (order kept); three barriers per row.
constexpr int kCompactMaxWords = 1024;   // 32768 slots (the 16-bit slot limit)
template <typename T>
__global__ void __launch_bounds__(256) k_compact(int cap, const int* __restrict__ in_nt,
                                                 const int* __restrict__ in_tile, const T* __restrict__ in_val,
                                                 int* __restrict__ out_nt, int* __restrict__ out_tile,
                                                 T* __restrict__ out_val, const unsigned* __restrict__ err) {
    __shared__ unsigned s_bits[kCompactMaxWords];
    __shared__ int s_pre[kCompactMaxWords];
    if (*err & (kErrCapacity | kErrSortSize)) return;
    const int r = blockIdx.x;
    const int n = in_nt[r];
    const int nw = (n + 31) >> 5;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    using VT = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    constexpr int kPer = kTileVals * (int)sizeof(T) / 16;   // 16-byte pieces per tile (24 or 48)
    for (int i = threadIdx.x; i < nw; i += blockDim.x) s_bits[i] = 0u;
    __syncthreads();
    for (int s = warp; s < n; s += nwarps) {
        const VT* v = (const VT*)(in_val + ((size_t)r * cap + s) * kTileVals);
        bool nz = false;
        for (int i = lane; i < kPer; i += 32) {
            const VT x = v[i];
            if constexpr (sizeof(T) == 4)
                nz |= x.x != 0.f || x.y != 0.f || x.z != 0.f || x.w != 0.f;
            else
                nz |= nonzero(x.x) || nonzero(x.y);
        }
        if (__any_sync(0xffffffffu, nz) && lane == 0) atomicOr(&s_bits[s >> 5], 1u << (s & 31));
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int run = 0;
        for (int w = 0; w < nw; ++w) {
            s_pre[w] = run;
            run += __popc(s_bits[w]);
        }
        out_nt[r] = run;
    }
    __syncthreads();
    for (int s = warp; s < n; s += nwarps) {
        const unsigned w = s_bits[s >> 5];
        if (!(w >> (s & 31) & 1u)) continue;
        const int pos = s_pre[s >> 5] + __popc(w & ((1u << (s & 31)) - 1u));
        const VT* v = (const VT*)(in_val + ((size_t)r * cap + s) * kTileVals);
        VT* o = (VT*)(out_val + ((size_t)r * cap + pos) * kTileVals);
        for (int i = lane; i < kPer; i += 32) o[i] = v[i];
        if (lane == 0) out_tile[(size_t)r * cap + pos] = in_tile[(size_t)r * cap + s];
    }
}

}  // namespace

size_t sweep_flag_bytes(const Ctx* c) { return flag_bytes((size_t)c->n_mol * c->cap, c->n_tiles); }
size_t sweep_info_bytes(const Ctx* c) { return (size_t)std::max(c->n_gnb, 1) * sizeof(BlockInfo); }

size_t closure_smem_bytes(const Ctx* c) {
    const size_t uw = (size_t)(2 * c->max_cl_groups + 31) / 32;
    return 3 * uw * 4 + (size_t)c->cap * 4 + (size_t)((c->cap + 1) & ~1) * 2 + 16;
}

size_t closure_labels_smem_bytes(const Ctx* c) { return (size_t)4 * c->max_cl_groups * 4; }

// --------------------------------------------------------------------------
// launchers
// --------------------------------------------------------------------------
template <typename T>
static cudaError_t select_rot_t(Ctx* c) {
    const double tau = c->prm.eps;
    ClSel* cl = (ClSel*)c->d_cl_sel;
    // the keys are the bit patterns of |F| as doubles; a float widened to double
    // has its 29 lowest mantissa bits zero, so for FP32 storage the radix passes
    // below bit 24 would only ever pick bin 0 and are left out
    const int last = std::is_same<T, float>::value ? 24 : 0;
    if (c->n_clusters == 1 && c->n_gnb <= kSelSmallBlocks) {
        k_rot_select_small<T><<<1, 1024, 0, c->stream>>>(last, c->n_gnb, c->d_gnb_row, c->d_gnb_col, c->d_group_nmol,
                                                         c->d_group_nvt, c->d_rot_blk_tp0, (const T*)c->d_F, tau,
                                                         c->h_cl_sel_init[5], c->d_sc, cl);
        c->n_launch += 1;
    } else {
        // per-cluster state: counts and prefixes zero, kmax = rot_cap_factor * N_occ(cluster)
        cudaError_t e = cudaMemcpyAsync(c->d_cl_sel, c->d_cl_sel_init, c->h_cl_sel_init.size() * 8,
                                        cudaMemcpyDeviceToDevice, c->stream);
        if (e != cudaSuccess) return e;
        k_rot_stats<T><<<c->n_gnb, 256, 0, c->stream>>>(c->n_gnb, c->d_gnb_row, c->d_gnb_col, c->d_group_nmol,
                                                        c->d_group_nvt, c->d_group_cl, c->d_rot_blk_tp0,
                                                        (const T*)c->d_F, tau, c->d_sc, cl);
        const int hb = std::min(c->n_gnb, 1024);
        for (int shift = 56; shift >= last; shift -= 8) {
            k_rot_hist<T><<<hb, 256, 0, c->stream>>>(shift, c->n_gnb, c->d_gnb_row, c->d_gnb_col, c->d_group_nmol,
                                                     c->d_group_nvt, c->d_group_cl, c->d_rot_blk_tp0, (const T*)c->d_F,
                                                     tau, cl, c->d_cl_hist);
            k_rot_pick<<<(c->n_clusters + 3) / 4, 128, 0, c->stream>>>(shift, last, c->n_clusters, cl, c->d_cl_hist);
        }
        c->n_launch += std::is_same<T, double>::value ? 1 + 2 * 8 : 1 + 2 * 5;
    }
    c->n_launch += 1;
    k_rot_lists<T><<<c->n_gnb, kListThreads, 0, c->stream>>>(
        c->n_gnb, c->d_gnb_row, c->d_gnb_col, c->d_group_nmol, c->d_group_nvt, c->d_group_occ0_mo,
        c->d_group_virt0_mo, c->d_group_cl, c->d_rot_blk_tp0, (const T*)c->d_F, c->d_Fd, tau, c->d_sc, cl, c->d_pr_n,
        c->d_pr_lvl, c->d_pr_ij, (T*)c->d_pr_cs, c->d_pr_touch);
    return cudaGetLastError();
}

cudaError_t launch_select_rot(Ctx* c) {
    return c->prec == SSCF_FP64 ? select_rot_t<double>(c) : select_rot_t<float>(c);
}

template <typename T>
static cudaError_t ortho_prepare_t(Ctx* c, int w, double tol) {
    const int t_hi = w == 1 ? c->n_occ_tiles : c->n_tiles;
    k_ortho_scale<T><<<(t_hi * 16 + 255) / 256, 256, 0, c->stream>>>(
        w, 0, t_hi, c->d_tile_group, c->d_tile_kind, c->d_tile_nmo, c->d_tile_mo0, c->d_group_ot0, c->d_group_not,
        c->d_group_vt0, c->d_self_blk, c->d_ort_blk_tp[w], (const T*)c->d_sig, c->d_scale, &c->d_sc->err);
    const int nob = (int)c->h_ocolour_blk.size();
    cudaError_t e = cudaMemsetAsync(c->d_cl_eta, 0, (size_t)c->n_clusters * 8, c->stream);
    if (e != cudaSuccess) return e;
    k_ortho_eta<T><<<nob, 256, 0, c->stream>>>(w, c->d_ocolour_blk, nob, c->d_gnb_row, c->d_gnb_col,
                                              c->d_group_nmol, c->d_group_not, c->d_group_occ0_mo,
                                              c->d_group_virt0_mo, c->d_ort_blk_tp[w], (const T*)c->d_sig,
                                              c->d_scale, c->d_sc, c->d_group_cl, c->d_cl_eta);
    k_ortho_lists<T><<<nob, kListThreads, 0, c->stream>>>(w, tol, c->d_ocolour_blk, c->d_gnb_row, c->d_gnb_col,
                                                c->d_group_nmol, c->d_group_not, c->d_group_occ0_mo,
                                                c->d_group_virt0_mo, c->d_ort_blk_tp[w], (const T*)c->d_sig,
                                                c->d_scale, c->d_sc, c->d_group_cl, c->d_cl_eta, c->d_pr_n,
                                                c->d_pr_lvl, c->d_pr_ij,
                                                (T*)c->d_pr_cs, c->d_pr_touch);
    return cudaGetLastError();
}

cudaError_t launch_ortho_prepare(Ctx* c, int w, double tol) {
    c->n_launch += 3;
    return c->prec == SSCF_FP64 ? ortho_prepare_t<double>(c, w, tol) : ortho_prepare_t<float>(c, w, tol);
}

template <typename T>
static void fill_args(Ctx* c, SweepArgs& a, int mode, int which) {
    a.mode = mode;
    a.which = which;
    a.n_tiles = c->n_tiles;
    a.n_occ_tiles = c->n_occ_tiles;
    a.n_groups = c->n_groups;
    a.max_cl_groups = c->max_cl_groups;
    a.n_clusters = c->n_clusters;
    a.in_nz = nullptr;
    a.normalise_pass = 1;
    a.gnb_colour = c->d_gnb_colour;
    a.col_lo = 0;
    a.col_hi = c->n_colours;
    a.mol_cluster = c->d_mol_cluster;
    a.cl_g0 = c->d_cl_g0;
    a.cl_ot0 = c->d_cl_ot0;
    a.cl_vt0 = c->d_cl_vt0;
    a.clblk_ptr = c->d_clblk_ptr[mode == 0 ? 0 : 1];
    a.clblk = c->d_clblk[mode == 0 ? 0 : 1];
    a.cap = c->cap;
    a.n_blk = mode == 0 ? c->n_gnb : (int)c->h_ocolour_blk.size();
    a.trunc = mode == 0 ? c->prm.eps : 1e-3 * c->prm.eps;
    a.trunc_f = (float)a.trunc;
    if ((double)a.trunc_f < a.trunc) a.trunc_f = nextafterf(a.trunc_f, INFINITY);
    a.blk = mode == 0 ? c->d_colour_blk : c->d_ocolour_blk;
    a.gnb_row = c->d_gnb_row;
    a.gnb_col = c->d_gnb_col;
    a.group_nmol = c->d_group_nmol;
    a.group_ot0 = c->d_group_ot0;
    a.group_not = c->d_group_not;
    a.group_vt0 = c->d_group_vt0;
    a.group_nvt = c->d_group_nvt;
    a.tile_group = c->d_tile_group;
    a.tile_kind = c->d_tile_kind;
    a.tile_mo0 = c->d_tile_mo0;
    a.tile_nmo = c->d_tile_nmo;
    a.pr_n = c->d_pr_n;
    a.pr_lvl = c->d_pr_lvl;
    a.pr_touch = c->d_pr_touch;
    a.pr_ij = c->d_pr_ij;
    a.pr_cs = c->d_pr_cs;
    a.dsc = c->d_scale;
    a.cl_eta = c->d_cl_eta;
    a.tol = c->ortho_tol;
    a.upd = &c->d_sc->upd[mode == 0 ? 0 : 1];
    a.cci_ptr = c->d_cci_ptr;
    a.cci_row = c->d_cci_row;
    a.cci_slot = c->d_cci_slot;
    a.err = &c->d_sc->err;
}

// The closure of the sweep's colours [col_lo, col_hi) (components over the
// active blocks of those colours); unless it is the first of the pass, a unit
// whose tiles in a row are all flagged zero does not count as held there.
template <typename T>
static cudaError_t closure_t(Ctx* c, int mode, int which, int col_lo, int col_hi, bool first) {
    SweepArgs a;
    fill_args<T>(c, a, mode, which);
    const int in = c->cur, out = 1 - c->cur;
    a.in_nt = c->d_c_nt[in];
    a.in_tile = c->d_c_tile[in];
    a.in_val = c->d_c_val[in];
    a.out_nt = c->d_c_nt[out];
    a.out_tile = c->d_c_tile[out];
    a.out_val = c->d_c_val[out];
    a.out_nz = c->d_c_nz[out];
    a.unit_lab = c->d_unit_lab;
    a.in_nz = first ? nullptr : c->d_c_nz[in];
    a.normalise_pass = first ? 1 : 0;
    a.col_lo = col_lo;
    a.col_hi = col_hi;
    const size_t smem = closure_smem_bytes(c);
    if (smem > (size_t)kMaxDynSmem) return cudaErrorInvalidValue;
    cudaError_t e = allow_dynamic_smem<k_closure<T>>();
    if (e != cudaSuccess) return e;
    a.lab_start = c->d_lab_start;
    a.lab_cnt = c->d_lab_cnt;
    a.lab_mem = c->d_lab_mem;
    const size_t lsmem = closure_labels_smem_bytes(c);
    if (lsmem > (size_t)kMaxDynSmem) return cudaErrorInvalidValue;
    e = allow_dynamic_smem<k_closure_labels>();
    if (e != cudaSuccess) return e;
    k_closure_labels<<<c->n_clusters, 1024, lsmem, c->stream>>>(a, c->d_unit_lab);
    k_closure<T><<<c->n_mol, 256, smem, c->stream>>>(a);
    c->cur = out;
    return cudaGetLastError();
}

// The generic kernel for every block, on request (apply_variant 1).
template <typename T, int MODE, int NT, int PCAP>
static cudaError_t apply_generic_t(Ctx* c, const SweepArgs& a, int col_lo, int col_hi) {
    const size_t smem = (size_t)NT * 16 * apply_nrp<T>() * sizeof(T) + (size_t)2 * PCAP * sizeof(T) + (size_t)PCAP * 4;
    cudaError_t e = allow_dynamic_smem<k_apply_colour<T, MODE, NT, PCAP>>();
    if (e != cudaSuccess) return e;
    const std::vector<int>& ptr = MODE == 0 ? c->h_colour_ptr : c->h_ocolour_ptr;
    constexpr int CH = ApplyShape<T>::chunk;
    const int gx = (c->n_mol + CH - 1) / CH;
    for (int col = col_lo; col < col_hi; ++col) {
        const int nb = ptr[col + 1] - ptr[col];
        if (nb == 0) continue;
        k_apply_colour<T, MODE, NT, PCAP><<<dim3(gx, nb), apply_threads<T>(), smem, c->stream>>>(a, ptr[col]);
        c->n_launch += 1;
    }
    return cudaGetLastError();
}

// The warp-at-a-time kernel, one launch per colour.
template <typename T, int MODE, bool ALL>
static cudaError_t apply_warp_t(Ctx* c, SweepArgs& a, int col_lo, int col_hi) {
    using Sh = WarpShape<T, MODE, ALL>;
    // the bits of a block's rows (a cluster's at most) and the counts before each word
    const int chunks = (c->n_mol + kFullCH - 1) / kFullCH;
    const size_t smem = Sh::smem + (size_t)std::min(chunks, (c->max_cl_mol + kFullCH - 1) / kFullCH) * 8;
    if (smem > (size_t)kMaxDynSmem) return cudaErrorInvalidValue;
    cudaError_t e = allow_dynamic_smem<k_apply_warp<T, MODE, ALL>>();
    if (e != cudaSuccess) return e;
    if (a.n_blk == 0) return cudaSuccess;
    a.blk_info = c->d_blk_info;
    k_block_info<MODE, ALL><<<(a.n_blk + 127) / 128, 128, 0, c->stream>>>(a, a.n_blk, (BlockInfo*)c->d_blk_info);
    c->n_launch += 1;
    const std::vector<int>& ptr = MODE == 0 ? c->h_colour_ptr : c->h_ocolour_ptr;
    // CTAs per block: sweep_shape, for as many runs as the largest cluster's rows can give (variant 2: one CTA
    // takes all runs of its block; same results)
    const int full = c->n_sm * Sh::resident;
    // A colour's CTAs start while the last of the one before run, so that the end of one launch hides the
    // start of the next: rotations at 997 molecules 1.74 -> 1.50 ms, at 4096 9.3 -> 9.0, FP64 at 343 1.52 ->
    // 1.40; FP32 combinations 5.28 -> 5.20 and 42.2 -> 42.0. Not FP64 combinations, whose long blocks come
    // first and would gather on the SMs that end early (343: 10.4 -> 11.9), and not inside a captured graph, where
    // it has not been tried.
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing(c->stream, &capture);
    if (e != cudaSuccess) return e;
    const bool overlap = (Sh::f32 || MODE == 0) && capture == cudaStreamCaptureStatusNone;
    bool after_colour = false;
    for (int col = col_lo; col < col_hi; ++col) {
        const int nb = ptr[col + 1] - ptr[col];
        if (nb == 0) continue;
        const int runs = (kAoPerMol / Sh::halves * c->max_cl_mol + 31) / 32;   // at most, of a block
        const SweepShape shape = sweep_shape(nb, runs, Sh::runs, full, MODE == 0 ? kWsRotWaves : kWsCombWaves,
                                             MODE == 0 ? 0 : Sh::many_runs);
        const int gx = c->apply_variant == 2 ? 1 : shape.shares;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(nb * gx);
        cfg.blockDim = dim3(Sh::threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = c->stream;
        cudaLaunchAttribute early = {};
        early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        early.val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = &early;
        cfg.numAttrs = overlap && after_colour ? 1 : 0;
        e = cudaLaunchKernelEx(&cfg, k_apply_warp<T, MODE, ALL>, a, ptr[col], nb, shape.min_runs);
        if (e != cudaSuccess) return e;
        after_colour = true;
        c->n_launch += 1;
    }
    return cudaGetLastError();
}

template <typename T, int MODE, int NT, int PCAP>
static cudaError_t apply_mode_t(Ctx* c, int which, int col_lo, int col_hi) {
    SweepArgs a;
    fill_args<T>(c, a, MODE, which);
    a.in_nt = a.out_nt = c->d_c_nt[c->cur];
    a.in_tile = a.out_tile = c->d_c_tile[c->cur];
    a.in_val = a.out_val = c->d_c_val[c->cur];
    a.out_nz = c->d_c_nz[c->cur];
    a.col_nz = c->d_c_cnz;
    a.col_lo = col_lo;
    a.col_hi = col_hi;
    k_flags_by_column<<<c->n_tiles, 256, 0, c->stream>>>(c->cap, c->d_cci_ptr, c->d_cci_row, c->d_cci_slot,
                                                         a.out_nz, a.col_nz);
    c->n_launch += 1;
    if (c->apply_variant != 1) return apply_warp_t<T, MODE, NT == 6>(c, a, col_lo, col_hi);
    return apply_generic_t<T, MODE, NT, PCAP>(c, a, col_lo, col_hi);
}

// side tiles and pair capacity per pass: rotations 2 occupied + 1 virtual
// tiles, 32 x 16 pairs; occupied passes 2 + 2 tiles, 32 x 32 pairs; passes over
// all MOs 3 + 3 tiles, 48 x 48 pairs
template <typename T>
static cudaError_t apply_t(Ctx* c, int mode, int which, int col_lo, int col_hi) {
    if (mode == 0) return apply_mode_t<T, 0, 3, kRotCap>(c, which, col_lo, col_hi);
    if (which == 1) return apply_mode_t<T, 1, 4, 32 * 32>(c, which, col_lo, col_hi);
    return apply_mode_t<T, 1, 6, kOrthoCap>(c, which, col_lo, col_hi);
}

cudaError_t launch_closure(Ctx* c, int mode, int which, int col_lo, int col_hi, bool first) {
    c->n_launch += 2;
    if (col_hi < 0) col_hi = c->n_colours;
    return c->prec == SSCF_FP64 ? closure_t<double>(c, mode, which, col_lo, col_hi, first)
                                : closure_t<float>(c, mode, which, col_lo, col_hi, first);
}

cudaError_t launch_apply(Ctx* c, int mode, int which, int col_lo, int col_hi) {
    if (col_hi < 0) col_hi = c->n_colours;
    return c->prec == SSCF_FP64 ? apply_t<double>(c, mode, which, col_lo, col_hi)
                                : apply_t<float>(c, mode, which, col_lo, col_hi);
}

cudaError_t launch_compact(Ctx* c) {
    c->n_launch += 1;
    const int in = c->cur, out = 1 - c->cur;
    if (c->prec == SSCF_FP64)
        k_compact<double><<<c->n_mol, 256, 0, c->stream>>>(c->cap, c->d_c_nt[in], c->d_c_tile[in],
                                                           (const double*)c->d_c_val[in], c->d_c_nt[out],
                                                           c->d_c_tile[out], (double*)c->d_c_val[out], &c->d_sc->err);
    else
        k_compact<float><<<c->n_mol, 256, 0, c->stream>>>(c->cap, c->d_c_nt[in], c->d_c_tile[in],
                                                          (const float*)c->d_c_val[in], c->d_c_nt[out],
                                                          c->d_c_tile[out], (float*)c->d_c_val[out], &c->d_sc->err);
    c->cur = out;
    return cudaGetLastError();
}

}  // namespace sscf
