// Adjoint of the SCC energy at the current (converged) MOs: forces and the
// gradients with respect to the eight Slater-Koster prefactors.
//
//   dE = sum P * dH0 + sum (P (Q_a + Q_b) / 2 - W) * dS + dq^T dgamma dq / 2,
//   W  = P H P / 2 = 2 C_o F_oo C_o^T,   F_oo = C_o^T H C_o,
//
// the first-order change of E = sum P H0 + dq^T gamma dq / 2 (Eq. H_dftb,
// Eq. pop) under the orthonormality constraint C^T S C = I with F_ov = 0.
// F_oo is formed on the occupied blocks of neighbouring groups (the same
// tile-pair transform as C^T S C), Z = C_o F_oo row by row, then P_mn and
// W_mn on the molecule-pair pattern are contracted with the analytic
// derivatives of the Slater-Koster blocks.
#include <math.h>

#include <algorithm>

#include <type_traits>

#include "block_scan.h"
#include "shares.h"
#include "sscf_internal.h"
#include "sum3.h"

namespace sscf {

namespace {

// Z = C_o F_oo, row-major like C: row block r gets the occupied tiles of every
// group adjacent (or equal) to a group whose occupied tiles it holds.
//
// k_zlists writes the rows' tile lists; k_zmul the values.
__global__ void __launch_bounds__(256) k_zlists(int n_occ_tiles, int n_groups, int cap, const int* __restrict__ c_nt,
                                                const int* __restrict__ c_tile, const int* __restrict__ tile_group,
                                                const int* __restrict__ group_ot0, const int* __restrict__ group_not,
                                                const int* __restrict__ gnb_ptr, const int* __restrict__ gnb_col,
                                                int* __restrict__ z_nt, int* __restrict__ z_tile,
                                                unsigned* __restrict__ err) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int gw = (n_groups + 31) >> 5;
    unsigned* pres = (unsigned*)smraw;          // gw: groups with occupied tiles in row r
    unsigned* outg = pres + gw;                 // gw: groups of Z's tiles
    __shared__ int part[33];
    const int r = blockIdx.x;
    for (int i = threadIdx.x; i < gw; i += blockDim.x) pres[i] = outg[i] = 0u;
    __syncthreads();
    const int n0 = c_nt[r];
    for (int s = threadIdx.x; s < n0; s += blockDim.x) {
        const int t = c_tile[(size_t)r * cap + s];
        if (t >= n_occ_tiles) continue;
        const int g = tile_group[t];
        atomicOr(&pres[g >> 5], 1u << (g & 31));
    }
    __syncthreads();
    for (int g = threadIdx.x; g < n_groups; g += blockDim.x) {
        if (!((pres[g >> 5] >> (g & 31)) & 1)) continue;
        for (int e = gnb_ptr[g]; e < gnb_ptr[g + 1]; ++e) {
            const int B = gnb_col[e];
            atomicOr(&outg[B >> 5], 1u << (B & 31));
        }
    }
    __syncthreads();
    // sorted output tile list (occupied tiles, group order)
    const int per = (n_groups + blockDim.x - 1) / blockDim.x;
    const int g0 = threadIdx.x * per, g1 = min(n_groups, g0 + per);
    int cnt = 0;
    for (int g = g0; g < g1; ++g)
        if ((outg[g >> 5] >> (g & 31)) & 1) cnt += group_not[g];
    int pos = block_scan(cnt, part);
    const int n_out = part[32];
    if (n_out > cap) {
        if (threadIdx.x == 0) {
            atomicOr(err, kErrCapacity);
            z_nt[r] = 0;
        }
        return;
    }
    for (int g = g0; g < g1; ++g)
        if ((outg[g >> 5] >> (g & 31)) & 1)
            for (int i = 0; i < group_not[g]; ++i) z_tile[(size_t)r * cap + pos++] = group_ot0[g] + i;
    if (threadIdx.x == 0) z_nt[r] = n_out;
}

// first position of the sorted list with a tile >= t
__device__ __forceinline__ int first_at(const int* __restrict__ list, int n, int t) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (list[mid] < t) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// What the kernels below start with, for one MO group's molecules (rows) and one out
// group A: the rows, their first slot of A's tiles in Z (-1: none), and for up to
// max_nb neighbours B of A the slots of B's two tiles in the rows (or -1) and whether
// any row holds one. False if no row has tiles of A.
template <int THREADS>
__device__ __forceinline__ bool z_lookup(int m0, int nm, int otA, int e0, int nb, int cap,
                                         const int* __restrict__ grp_mol, const int* __restrict__ c_nt,
                                         const int* __restrict__ c_tile, const int* __restrict__ group_ot0,
                                         const int* __restrict__ group_not, const int* __restrict__ gnb_col,
                                         const int* __restrict__ z_nt, const int* __restrict__ z_tile, int* s_mol,
                                         int* s_z, int2* slot, int* any) {
    bool mine = false;
    if ((int)threadIdx.x < nm) {
        const int r = grp_mol[m0 + threadIdx.x];
        const int n = z_nt[r];
        const int* zt = z_tile + (size_t)r * cap;
        const int p = first_at(zt, n, otA);
        mine = p < n && zt[p] == otA;
        s_mol[threadIdx.x] = r;
        s_z[threadIdx.x] = mine ? p : -1;
    }
    if (!__syncthreads_or(mine)) return false;
    for (int i = threadIdx.x; i < nb; i += THREADS) any[i] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < nb * nm; i += THREADS) {
        const int k = i / nm, q = i - k * nm;
        const int B = gnb_col[e0 + k], t = group_ot0[B];
        const int* ct = c_tile + (size_t)s_mol[q] * cap;
        const int n = c_nt[s_mol[q]];
        const int p = first_at(ct, n, t);
        int2 s = make_int2(-1, -1);
        if (p < n && ct[p] == t) {
            s.x = p;
            if (group_not[B] > 1 && p + 1 < n && ct[p + 1] == t + 1) s.y = p + 1;
        } else if (group_not[B] > 1 && p < n && ct[p] == t + 1) {
            s.y = p;
        }
        slot[k * kMaxMolPerGroup + q] = s;
        if (s.x >= 0 || s.y >= 0) any[k] = 1;
    }
    __syncthreads();
    return true;
}

// Z's values in FP32 storage. A CTA makes the 48 x 32 outputs of one MO group's molecules (48 AO
// rows) and one out group A (two tiles), over the in groups B adjacent to A that
// any of the rows holds: per B it stages the rows' 48 x 32 values and the 32 x 32
// block F[B, A] (loading the next B's meanwhile), so that a block of F is read once per group of molecules, and
// each of 96 threads keeps 4 x 4 outputs. Terms are added in the order of the
// row's tiles and of the MOs inside a tile, one product at a time; a tile that a
// row does not hold contributes zeros. (One warp per row and out tile read a
// block of F for six rows of work and looked it up by a binary search:
// 27.6 ms at 2000 molecules; 6.6 with scalar multiply-adds, F staged value by
// value and loads not overlapped; now 5.4, with the registers cut for seven CTAs per
// SM; 5.7 cut for six.)
constexpr int kZThreads = 96;
constexpr int kZRows = kMaxMolPerGroup * kAoPerMol;   // 48
constexpr int kZStride = kZRows + 4;                  // values per staged MO (16-byte aligned, bank-spread)
constexpr int kFStride = 36;                          // values per staged MO of B
// Neighbours of A in one launch, whose slots are in shared memory. Where a group has more (MANY), the
// neighbours from nb_lo on are taken and the sums go on from where the launch before left them. (One
// kernel for both was slower: 5.9 ms instead of 5.6 at 2000 molecules.)
constexpr int kZNb = 128;
__host__ __device__ constexpr size_t z_lookup_smem(int max_nb) {
    return (size_t)max_nb * (kMaxMolPerGroup * sizeof(int2) + sizeof(int));
}
constexpr size_t kZmulSmem = (size_t)32 * (kZStride + kFStride) * sizeof(float);   // and z_lookup_smem
template <bool MANY>
__global__ void __launch_bounds__(kZThreads, 7)
k_zmul(int g_lo, int nb_lo, int max_nb, int cap, const int* __restrict__ group_cl, const int* __restrict__ cl_g0,
       const int* __restrict__ grp_mol_ptr, const int* __restrict__ grp_mol,
       const int* __restrict__ c_nt, const int* __restrict__ c_tile, const float* __restrict__ c_val,
       const int* __restrict__ group_ot0, const int* __restrict__ group_not, const int* __restrict__ gnb_ptr,
       const int* __restrict__ gnb_col, const int* __restrict__ blk_tp, const int* __restrict__ gnb_rev,
       const float* __restrict__ F, const int* __restrict__ z_nt, const int* __restrict__ z_tile, float* __restrict__ z_val) {
    extern __shared__ __align__(16) unsigned char smraw[];
    float* sc = (float*)smraw;                                // [32 MOs of B][kZStride]: the rows' values
    float* sf = sc + 32 * kZStride;                       // [32 MOs of B][kFStride]: F[B, A], 32 MOs of A
    int2* slot = (int2*)(sf + 32 * kFStride);         // [neighbour of A][molecule]: slots of B's two tiles, or -1
    int* any = (int*)(slot + (size_t)max_nb * kMaxMolPerGroup);   // [neighbour of A]: some row holds a tile of B
    __shared__ int s_mol[kMaxMolPerGroup], s_z[kMaxMolPerGroup];
    const int G = g_lo + blockIdx.y, cl = group_cl[G], A = cl_g0[cl] + blockIdx.x;
    if (A >= cl_g0[cl + 1]) return;
    const int m0 = grp_mol_ptr[G], nm = grp_mol_ptr[G + 1] - m0;
    const int e0 = gnb_ptr[A] + (MANY ? nb_lo : 0), nb = MANY ? min(max_nb, gnb_ptr[A + 1] - e0) : gnb_ptr[A + 1] - e0;
    if (MANY && nb <= 0) return;
    const int otA = group_ot0[A], ntA = group_not[A];
    if (!z_lookup<kZThreads>(m0, nm, otA, e0, nb, cap, grp_mol, c_nt, c_tile, group_ot0, group_not, gnb_col, z_nt, z_tile,
                             s_mol, s_z, slot, any))
        return;
    const int ti = threadIdx.x >> 3, tj = threadIdx.x & 7;   // rows 4 ti .. 4 ti + 3, MOs 4 tj .. 4 tj + 3 of A
    float acc[4][4];
    // output row i of the thread: where its four values go (NULL: nowhere)
    auto out = [&](int i) -> float* {
        const int row = 4 * ti + i, q = row / kAoPerMol;
        if (q >= nm || s_z[q] < 0 || (tj >> 2) >= ntA) return nullptr;
        return z_val + ((size_t)s_mol[q] * cap + s_z[q] + (tj >> 2)) * kTileVals + (row - q * kAoPerMol) * kTileW +
               4 * (tj & 3);
    };
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    if (MANY && nb_lo > 0)
        for (int i = 0; i < 4; ++i)
            if (const float* z = out(i))
                for (int j = 0; j < 4; ++j) acc[i][j] = z[j];
    // 16-byte pieces: of the rows along the MOs, turned to [MO][row], and of F[B, A], whose tile pairs
    // are stored for blocks (lower group, upper group), inside a group for positions a <= b; turned
    // when stored the other way. The next neighbour's are loaded during this one's products.
    using V = float4;
    constexpr int kV = 4, kPer = 16 / kV;   // values of a piece, pieces per tile row
    constexpr int kC = kZRows * 2 * kPer / kZThreads, kF = (4 * 16 * kPer + kZThreads - 1) / kZThreads;
    static_assert(kC * kZThreads == kZRows * 2 * kPer, "");
    V vc[kC], vf[kF];
    int turned = 0;   // bit pB * 2 + pA: the tile pair is stored as [A][B]
    auto load = [&](int k) {
        const int e = e0 + k, B = gnb_col[e], eb = B <= A ? gnb_rev[e] : e;   // entry (min, max)
        const int ntB = group_not[B];
        turned = B < A ? 0 : B == A ? 4 : 15;   // (inside a group [pB][pA] is stored for pB <= pA)
#pragma unroll
        for (int h = 0; h < kC; ++h) {
            const int i = threadIdx.x + h * kZThreads;
            const int row = i / (2 * kPer), rem = i - row * (2 * kPer), t = rem / kPer, p = rem - t * kPer;
            const int q = row / kAoPerMol;
            const int s = q < nm ? (t ? slot[k * kMaxMolPerGroup + q].y : slot[k * kMaxMolPerGroup + q].x) : -1;
            vc[h] = V{};
            if (s >= 0)
                vc[h] = *(const V*)(c_val + ((size_t)s_mol[q] * cap + s) * kTileVals + (row - q * kAoPerMol) * kTileW +
                                    p * kV);
        }
#pragma unroll
        for (int h = 0; h < kF; ++h) {
            const int i = threadIdx.x + h * kZThreads, t = i / (16 * kPer), piece = i - t * (16 * kPer);
            const int pB = t >> 1, pA = t & 1;
            vf[h] = V{};
            if (t < 4 && pB < ntB && pA < ntA) {
                const int tp = blk_tp[(size_t)eb * 9 + ((turned >> (pB * 2 + pA)) & 1 ? pA * 3 + pB : pB * 3 + pA)];
                vf[h] = *((const V*)(F + (size_t)tp * 256) + piece);
            }
        }
    };
    auto next = [&](int k) {
        while (k < nb && !any[k]) ++k;
        return k;
    };
    int k = next(0);
    if (k < nb) load(k);
    while (k < nb) {
        __syncthreads();   // the buffers are free
#pragma unroll
        for (int h = 0; h < kC; ++h) {
            const int i = threadIdx.x + h * kZThreads;
            const int row = i / (2 * kPer), rem = i - row * (2 * kPer), t = rem / kPer, p = rem - t * kPer;
#pragma unroll
            for (int u = 0; u < kV; ++u) sc[(t * 16 + p * kV + u) * kZStride + row] = ((const float*)&vc[h])[u];
        }
#pragma unroll
        for (int h = 0; h < kF; ++h) {
            const int i = threadIdx.x + h * kZThreads, t = i / (16 * kPer), piece = i - t * (16 * kPer);
            const int r = piece / kPer, c = (piece - r * kPer) * kV, pB = t >> 1, pA = t & 1;
            if (t >= 4) continue;
            if ((turned >> t) & 1) {
#pragma unroll
                for (int u = 0; u < kV; ++u)
                    sf[(pB * 16 + c + u) * kFStride + pA * 16 + r] = ((const float*)&vf[h])[u];
            } else {
                *(V*)(sf + (pB * 16 + r) * kFStride + pA * 16 + c) = vf[h];
            }
        }
        __syncthreads();
        k = next(k + 1);
        if (k < nb) load(k);
#pragma unroll 8
        for (int q = 0; q < 32; ++q) {
            float c[4], f[4];
            *(V*)c = *(const V*)(sc + q * kZStride + 4 * ti);
            *(V*)f = *(const V*)(sf + q * kFStride + 4 * tj);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
#pragma unroll
                for (int j = 0; j < 4; j += 2) {
                    const float2 v = __ffma2_rn(make_float2(c[i], c[i]), make_float2(f[j], f[j + 1]),
                                                make_float2(acc[i][j], acc[i][j + 1]));
                    acc[i][j] = v.x;
                    acc[i][j + 1] = v.y;
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (float* z = out(i)) *(V*)z = *(const V*)acc[i];
    }
}

// The same in FP64 storage, whose pipe (two lanes per clock and SM) bounds it: no product may be
// spent on a tile that a row does not hold, and those are many in a large cluster (in the kernel
// above 1.3 times the products that are there at 1000 molecules, 1.8 at 2000). A CTA takes the
// same rows and out group, a warp one molecule, and walks the tiles that its own row holds; a
// lane keeps rows kh, kh + 2, kh + 4 of column j of A's tiles. Terms in the same
// order. (With absent tiles as zeros 40.4 ms at 1000 molecules, one warp per row and
// out tile 37.9; now 30.9, of which the products take 29.9. The adjoint at 2000:
// 178, 139, now 106 ms.)
constexpr int kZ64Threads = 32 * kMaxMolPerGroup;
constexpr int kF64Stride = 34;   // values per staged MO of B (16-byte aligned)
constexpr size_t kZmul64Smem =
    (size_t)2 * (32 * kF64Stride + kMaxMolPerGroup * 2 * kTileVals) * sizeof(double);   // and z_lookup_smem
template <bool MANY>
__global__ void __launch_bounds__(kZ64Threads)
k_zmul64(int g_lo, int nb_lo, int max_nb, int cap, const int* __restrict__ group_cl, const int* __restrict__ cl_g0,
         const int* __restrict__ grp_mol_ptr, const int* __restrict__ grp_mol,
         const int* __restrict__ c_nt, const int* __restrict__ c_tile, const double* __restrict__ c_val,
         const int* __restrict__ group_ot0, const int* __restrict__ group_not, const int* __restrict__ gnb_ptr,
         const int* __restrict__ gnb_col, const int* __restrict__ blk_tp, const int* __restrict__ gnb_rev,
         const double* __restrict__ F, const int* __restrict__ z_nt, const int* __restrict__ z_tile,
         double* __restrict__ z_val) {
    extern __shared__ __align__(16) unsigned char smraw[];
    double* sf = (double*)smraw;                      // two buffers: [32 MOs of B][kF64Stride]: F[B, A]
    double* sc = sf + 2 * 32 * kF64Stride;            // two buffers: [molecule][B's two tiles]
    int2* slot = (int2*)(sc + 2 * kMaxMolPerGroup * 2 * kTileVals);   // as above
    int* any = (int*)(slot + (size_t)max_nb * kMaxMolPerGroup);
    __shared__ int s_mol[kMaxMolPerGroup], s_z[kMaxMolPerGroup];
    const int G = g_lo + blockIdx.y, cl = group_cl[G], A = cl_g0[cl] + blockIdx.x;
    if (A >= cl_g0[cl + 1]) return;
    const int m0 = grp_mol_ptr[G], nm = grp_mol_ptr[G + 1] - m0;
    const int e0 = gnb_ptr[A] + (MANY ? nb_lo : 0), nb = MANY ? min(max_nb, gnb_ptr[A + 1] - e0) : gnb_ptr[A + 1] - e0;
    if (MANY && nb <= 0) return;
    const int otA = group_ot0[A], ntA = group_not[A];
    if (!z_lookup<kZ64Threads>(m0, nm, otA, e0, nb, cap, grp_mol, c_nt, c_tile, group_ot0, group_not, gnb_col, z_nt,
                               z_tile, s_mol, s_z, slot, any))
        return;
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;   // q: the warp's molecule
    const int j = lane & 15, kh = lane >> 4;
    const bool mine = q < nm && s_z[q] >= 0;
    // row kh of the warp's first tile of A in Z (only where mine)
    double* const z = z_val + (mine ? ((size_t)s_mol[q] * cap + s_z[q]) * kTileVals + kh * kTileW + j : 0);
    double acc[2][3];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int u = 0; u < 3; ++u)
            acc[a][u] = MANY && nb_lo > 0 && mine && a < ntA ? z[a * kTileVals + 2 * u * kTileW] : 0.0;
    double2 vc[3] = {}, vf[2] = {};
    int turned = 0;   // as above
    auto load = [&](int k) {
        const int e = e0 + k, B = gnb_col[e], eb = B <= A ? gnb_rev[e] : e;   // entry (min, max)
        const int ntB = group_not[B];
        turned = B < A ? 0 : B == A ? 4 : 15;
#pragma unroll
        for (int h = 0; h < 3; ++h) {
            const int i = lane + 32 * h, t = i / (kTileVals / 2), p = i - t * (kTileVals / 2);
            const int s = q < nm ? (t ? slot[k * kMaxMolPerGroup + q].y : slot[k * kMaxMolPerGroup + q].x) : -1;
            if (s >= 0) vc[h] = *((const double2*)(c_val + ((size_t)s_mol[q] * cap + s) * kTileVals) + p);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = threadIdx.x + h * kZ64Threads, t = i >> 7, pB = t >> 1, pA = t & 1;
            if (pB < ntB && pA < ntA) {
                const int tp = blk_tp[(size_t)eb * 9 + ((turned >> t) & 1 ? pA * 3 + pB : pB * 3 + pA)];
                vf[h] = *((const double2*)(F + (size_t)tp * 256) + (i & 127));
            }
        }
    };
    auto next = [&](int k) {
        while (k < nb && !any[k]) ++k;
        return k;
    };
    int phase = 0, k = next(0);
    if (k < nb) load(k);
    while (k < nb) {
        // (a buffer is written again after the barrier that all threads reach past its products)
        double* const f = sf + phase * 32 * kF64Stride;
        double* const c = sc + (phase * kMaxMolPerGroup + q) * 2 * kTileVals;
        phase ^= 1;
#pragma unroll
        for (int h = 0; h < 3; ++h) ((double2*)c)[lane + 32 * h] = vc[h];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = threadIdx.x + h * kZ64Threads, t = i >> 7, pB = t >> 1, pA = t & 1;
            const int r = (i & 127) >> 3, col = 2 * (i & 7);
            if ((turned >> t) & 1) {
                f[(pB * 16 + col) * kF64Stride + pA * 16 + r] = vf[h].x;
                f[(pB * 16 + col + 1) * kF64Stride + pA * 16 + r] = vf[h].y;
            } else {
                *(double2*)(f + (pB * 16 + r) * kF64Stride + pA * 16 + col) = vf[h];
            }
        }
        __syncthreads();
        const int2 held = q < nm ? slot[k * kMaxMolPerGroup + q] : make_int2(-1, -1);
        k = next(k + 1);
        if (k < nb) load(k);
        auto products = [&](auto two) {
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                if ((t ? held.y : held.x) < 0) continue;
                const double *ct = c + t * kTileVals + kh * kTileW, *ft = f + t * 16 * kF64Stride + j;
#pragma unroll 4
                for (int i = 0; i < 16; i += 2) {
                    double2 x[3];
#pragma unroll
                    for (int u = 0; u < 3; ++u) x[u] = *(const double2*)(ct + 2 * u * kTileW + i);
#pragma unroll
                    for (int a = 0; a < (decltype(two)::value ? 2 : 1); ++a) {
                        const double f0 = ft[i * kF64Stride + 16 * a], f1 = ft[(i + 1) * kF64Stride + 16 * a];
#pragma unroll
                        for (int u = 0; u < 3; ++u) {
                            acc[a][u] += x[u].x * f0;
                            acc[a][u] += x[u].y * f1;
                        }
                    }
                }
            }
        };
        if (ntA > 1) products(std::true_type());
        else products(std::false_type());
    }
    if (mine)
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int u = 0; u < 3; ++u)
                if (a < ntA) z[a * kTileVals + 2 * u * kTileW] = acc[a][u];
}

struct SKd {
    double V0[4], S0[4];
    double r_decay, rc2;
};

__device__ __forceinline__ double dist2_rn(const double* a, const double* b) {
    double dx = __dsub_rn(b[0], a[0]);
    double dy = __dsub_rn(b[1], a[1]);
    double dz = __dsub_rn(b[2], a[2]);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

__device__ __forceinline__ int ao_off(int k) { return k == 0 ? 0 : 3 + k; }

// Contribution of the ordered atom pair (a in m, b in n) to dE: the force on
// atom a (-2 g, g = sum P dH/dR + GS dS/dR, R = x_b - x_a; the pair (b, a)
// gives the same on a) and the parameter partials sum P H0^(k) and GS S^(k).
__device__ __forceinline__ void pair_terms(const SKd& P, const double* xa, const double* xb, int na, int nb,
                                           const double* Pm, const double* GS, double* fa, double* dpar) {
    double d2 = dist2_rn(xa, xb);
    if (!(d2 <= P.rc2)) return;
    const double r = sqrt(d2);
    double e[3], R[3];
    for (int d = 0; d < 3; ++d) {
        R[d] = xb[d] - xa[d];
        e[d] = R[d] / r;
    }
    const double decay = exp(-r / P.r_decay);
    for (int tab = 0; tab < 2; ++tab) {
        const double* V0 = tab == 0 ? P.V0 : P.S0;
        const double* Wt = tab == 0 ? Pm : GS;
        double V[4], dV[4];
        for (int q = 0; q < 4; ++q) {
            V[q] = V0[q] * decay;
            dV[q] = -V[q] / P.r_decay;
        }
        double g[3] = {0, 0, 0};
        double par[4] = {0, 0, 0, 0};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                if (i >= na || jj >= nb) continue;
                const double w = Wt[i * 4 + jj];
                if (w == 0.0) continue;
                for (int k = 0; k < 3; ++k) {
                    double v;
                    if (i == 0 && jj == 0) {
                        v = dV[0] * e[k];
                    } else if (i == 0 || jj == 0) {
                        const int c = i == 0 ? jj - 1 : i - 1;
                        const double dec = ((c == k ? 1.0 : 0.0) - e[c] * e[k]) / r;
                        v = dec * V[1] + e[c] * dV[1] * e[k];
                        if (jj == 0) v = -v;
                    } else {
                        const int ci = i - 1, cj = jj - 1;
                        const double dei = ((ci == k ? 1.0 : 0.0) - e[ci] * e[k]) / r;
                        const double dej = ((cj == k ? 1.0 : 0.0) - e[cj] * e[k]) / r;
                        v = (dei * e[cj] + e[ci] * dej) * (V[2] - V[3]) + e[ci] * e[cj] * (dV[2] - dV[3]) * e[k] +
                            (ci == cj ? dV[3] * e[k] : 0.0);
                    }
                    g[k] += w * v;
                }
                // parameter partials: the block is linear in the prefactors
                if (i == 0 && jj == 0) {
                    par[0] += w * decay;
                } else if (i == 0 || jj == 0) {
                    const int c = i == 0 ? jj - 1 : i - 1;
                    par[1] += w * (jj == 0 ? -e[c] : e[c]) * decay;
                } else {
                    const int ci = i - 1, cj = jj - 1;
                    par[2] += w * e[ci] * e[cj] * decay;
                    par[3] += w * ((ci == cj ? 1.0 : 0.0) - e[ci] * e[cj]) * decay;
                }
            }
        for (int k = 0; k < 3; ++k) fa[k] += -2.0 * g[k];
        for (int q = 0; q < 4; ++q) dpar[tab * 4 + q] += par[q];
    }
}

// One CTA per row block m, one warp per pattern neighbour n: P_mn (n >= m only,
// P_nm = P_mn^T) and W_mn = 2 sum_t C[m,t] Z[n,t]^T on the tiles both rows hold,
// written as 6 x 6 blocks. Products of FP32 values are rounded to FP32 and added
// up without further error worth the name: in FP64 in FP64 storage, in three
// floats (no less than FP64 carries) in FP32 storage, where FP64 additions
// bounded the kernel (two lanes per clock and SM; 72 of them per shared tile
// and lane): 34.2 ms at 2000 molecules with the pair terms; now 3.2, and 0.33 for
// those. (Two floats, 48 bits: 2.5.)
constexpr int kGradWarps = 8;
template <typename T> struct SumOf;
template <> struct SumOf<double> {
    double v;
    __device__ __forceinline__ void add(const SumOf& o) { v += o.v; }
    __device__ __forceinline__ double value() const { return v; }
};
template <> struct SumOf<float> {
    Sum3 v;
    __device__ __forceinline__ void add(const SumOf& o) { v.add(o.v); }
    __device__ __forceinline__ double value() const { return v.value(); }
};
// two sums of products
template <typename T> struct SumsOf;
template <> struct SumsOf<double> {
    double v[2];
    __device__ __forceinline__ void zero() { v[0] = v[1] = 0.0; }
    __device__ __forceinline__ void add_products(double a, double b0, double b1) {
        v[0] += a * b0;
        v[1] += a * b1;
    }
    __device__ __forceinline__ SumOf<double> get(int i) const { return {v[i]}; }
};
template <> struct SumsOf<float> {
    Sum3x2 v;
    __device__ __forceinline__ void zero() { v.h = v.l = v.m = make_float2(0.f, 0.f); }
    __device__ __forceinline__ void add_products(float a, float b0, float b1) {
        v.add(make_float2(__fmul_rn(a, b0), __fmul_rn(a, b1)));
    }
    __device__ __forceinline__ SumOf<float> get(int i) const {
        return {i ? Sum3{v.h.y, v.l.y, v.m.y} : Sum3{v.h.x, v.l.x, v.m.x}};
    }
};
// What a lane of a tile's 16 columns sums: FP64 all 36 products, the halves of the
// warp on two tiles; FP32, whose sums are three registers, 18 (three AO rows of m per
// half), both halves on one tile. (FP32 sums one by one instead of in pairs: 4.0 ms;
// the next tile's values loaded ahead, or three CTAs per SM: spills, 3.6 and 3.2.)
template <typename T> struct GradShape;
template <> struct GradShape<double> { static constexpr int tiles = 2; };
template <> struct GradShape<float> { static constexpr int tiles = 1; };
// the lanes' sums of one product, and the padding that spreads them over the banks
template <typename T> __host__ __device__ constexpr int grad_lanes() { return 16 * GradShape<T>::tiles; }
template <typename T> __host__ __device__ constexpr size_t grad_smem(int map_n) {
    return (size_t)((map_n + 3) & ~3) * 4 + (size_t)kGradWarps * 36 * (grad_lanes<T>() + 1) * sizeof(SumOf<T>);
}
template <typename T>
__global__ void __launch_bounds__(kGradWarps * 32, 2)
k_grad_blocks(int n_occ_tiles, int map_n, const int* __restrict__ mol_ot0, int cap, const int* __restrict__ c_nt,
              const int* __restrict__ c_tile, const T* __restrict__ c_val, const int* __restrict__ z_nt,
              const int* __restrict__ z_tile, const T* __restrict__ z_val, const int* __restrict__ mp_ptr,
              const int* __restrict__ mp_col, const int* __restrict__ mp_rev, double* __restrict__ Pb,
              double* __restrict__ Wb) {
    extern __shared__ __align__(16) int smap[];   // map_n: slot in C row m of each occupied tile of m's cluster, or -1
    constexpr int kTiles = GradShape<T>::tiles, kRows = 3 * kTiles;   // tiles at a time, AO rows of m per lane
    constexpr int kLanes = grad_lanes<T>(), kPad = kLanes + 1;
    SumOf<T>* sums = (SumOf<T>*)(smap + ((map_n + 3) & ~3));   // [warp][36][kPad]: the lanes' sums
    const int m = blockIdx.x;
    const int t0 = mol_ot0[m];
    for (int i = threadIdx.x; i < map_n; i += blockDim.x) smap[i] = -1;
    __syncthreads();
    const int ntm = c_nt[m];
    for (int s = threadIdx.x; s < ntm; s += blockDim.x) {
        const int t = c_tile[(size_t)m * cap + s];
        if (t < n_occ_tiles) smap[t - t0] = s;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int e0 = mp_ptr[m], ne = mp_ptr[m + 1] - e0;
    const int col = lane & 15, half = lane >> 4;
    const int row0 = kTiles == 2 ? 0 : kRows * half;   // the lane's first AO row of m
    SumOf<T>* mys = sums + (size_t)warp * 36 * kPad;
    // 2 sum_t C[m,t] B[n,t]^T over the occupied tiles of row n's list that row m holds
    auto block = [&](int n, const int* __restrict__ b_nt, const int* __restrict__ b_tile, const T* __restrict__ b_val,
                     double* out, double* out_t) {
        SumsOf<T> acc[kRows * 3];
#pragma unroll
        for (int u = 0; u < kRows * 3; ++u) acc[u].zero();
        const int nt = b_nt[n];
        const T* cm0 = c_val + (size_t)m * cap * kTileVals + row0 * kTileW + col;
        const T* bn0 = b_val + (size_t)n * cap * kTileVals + col;
        // 32 of n's tiles at a time, the shared ones found with one ballot
        for (int base = 0; base < nt; base += 32) {
            const int s = base + lane;
            const int t = s < nt ? b_tile[(size_t)n * cap + s] : n_occ_tiles;
            const int sm_ = t < n_occ_tiles ? smap[t - t0] : -1;
            unsigned mm = __ballot_sync(0xffffffffu, sm_ >= 0);
            const bool past = __any_sync(0xffffffffu, s < nt && t >= n_occ_tiles);
            while (mm) {
                int src = __ffs(mm) - 1;
                mm &= mm - 1;
                if (kTiles == 2) {   // the second half takes the next one
                    const int b1 = __ffs(mm) - 1;
                    mm &= mm - 1;
                    if (half) src = b1;
                }
                const int sl = __shfl_sync(0xffffffffu, sm_, src < 0 ? 0 : src);
                if (src < 0) continue;
                const T* cm = cm0 + sl * kTileVals;
                const T* bn = bn0 + (base + src) * kTileVals;
                T a6[kRows], b6[6];
#pragma unroll
                for (int k = 0; k < kRows; ++k) a6[k] = cm[k * kTileW];
#pragma unroll
                for (int k = 0; k < 6; ++k) b6[k] = bn[k * kTileW];
#pragma unroll
                for (int k = 0; k < kRows; ++k)
#pragma unroll
                    for (int l = 0; l < 3; ++l) acc[k * 3 + l].add_products(a6[k], b6[2 * l], b6[2 * l + 1]);
            }
            if (past) break;   // tiles are sorted: occupied tiles first
        }
#pragma unroll
        for (int u = 0; u < kRows * 6; ++u) mys[(row0 * 6 + u) * kPad + (kTiles == 2 ? lane : col)] = acc[u / 2].get(u & 1);
        __syncwarp();
        for (int u = lane; u < 36; u += 32) {
            SumOf<T> v = mys[u * kPad];
            for (int j = 1; j < kLanes; ++j) v.add(mys[u * kPad + j]);
            const double x = 2.0 * v.value();
            out[u] = x;
            if (out_t) out_t[(u % 6) * 6 + u / 6] = x;
        }
        __syncwarp();
    };
    for (int w = warp; w < ne; w += kGradWarps) {
        const int e = e0 + w, n = mp_col[e];
        if (n >= m)
            block(n, c_nt, c_tile, c_val, Pb + (size_t)e * 36, n > m ? Pb + (size_t)mp_rev[e] * 36 : nullptr);
        block(n, z_nt, z_tile, z_val, Wb + (size_t)e * 36, nullptr);
    }
}

// The pair terms of the molecule pairs: one thread per ordered atom pair (kind k
// of the nine: O-O first, then the pairs of O and H, then H-H, each for all
// molecule pairs, so that the threads of a warp run the same loops). Nine
// threads per warp did them at the end of each pair's block before, and the FP64
// pipe spends the same time on nine lanes as on 32.
constexpr int kPairOut = 11;   // force on a, parameter partials
__global__ void __launch_bounds__(128) k_pair_terms(int n_mp, const int* __restrict__ mp_row,
                                                    const int* __restrict__ mp_col, const double* __restrict__ xyz,
                                                    const double* __restrict__ Q, SKd P, const double* __restrict__ Pb,
                                                    const double* __restrict__ Wb, double* __restrict__ out) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n_mp) return;
    const int ia = blockIdx.y / 3, ib = blockIdx.y % 3;
    const int m = mp_row[e], n = mp_col[e];
    const int a = 3 * m + ia, b = 3 * n + ib;
    double fa[3] = {0, 0, 0}, dp[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (a != b) {
        const int na = ia == 0 ? 4 : 1, nb = ib == 0 ? 4 : 1, oa = ao_off(ia), ob = ao_off(ib);
        const double h = 0.5 * (Q[a] + Q[b]);
        double Pm[16], GS[16];   // the atom pair's na x nb values
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const bool in = i < na && j < nb;
                const size_t u = (size_t)e * 36 + (in ? (oa + i) * 6 + ob + j : 0);
                Pm[i * 4 + j] = in ? Pb[u] : 0.0;
                GS[i * 4 + j] = in ? h * Pb[u] - Wb[u] : 0.0;
            }
        pair_terms(P, xyz + 3 * a, xyz + 3 * b, na, nb, Pm, GS, fa, dp);
    }
    double* o = out + (size_t)blockIdx.y * kPairOut * n_mp + e;
#pragma unroll
    for (int k = 0; k < 3; ++k) o[(size_t)k * n_mp] = fa[k];
#pragma unroll
    for (int q = 0; q < 8; ++q) o[(size_t)(3 + q) * n_mp] = dp[q];
}

// Per molecule, in neighbour order: the forces on its atoms and the parameter
// partials of its pairs. One thread per molecule and output.
__global__ void k_pair_sum(int n_mol, int n_mp, const int* __restrict__ mp_ptr, const double* __restrict__ pt,
                           double* __restrict__ gmol, double* __restrict__ pmol) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 17 * n_mol) return;
    const int m = i / 17, u = i - 17 * m;
    double s = 0.0;
    for (int e = mp_ptr[m]; e < mp_ptr[m + 1]; ++e) {
        if (u < 9) {   // atom u / 3, component u % 3
            for (int ib = 0; ib < 3; ++ib) s += pt[((size_t)(u / 3 * 3 + ib) * kPairOut + u % 3) * n_mp + e];
        } else {
            for (int k = 0; k < 9; ++k) s += pt[((size_t)k * kPairOut + 3 + u - 9) * n_mp + e];
        }
    }
    if (u < 9) gmol[(size_t)m * 9 + u] = s;
    else pmol[(size_t)m * 8 + u - 9] = s;
}

// dE/dx_a of dq^T gamma dq / 2: -dq_a sum_b dq_b gamma_ab^3 (x_a - x_b), one
// warp per 32 atoms a and share of the atoms b (the FP64 pipe bounds it: one
// thread per atom over all b kept a third of the SMs busy, 7.3 ms at 6000
// atoms; now 1.3). rsqrt is nearer to the exact value than a division by a square
// root: 1.01 and 1.50 units of 2^-53 at most over 4 million arguments from 0.01 to
// 10^6, 0.36 and 0.50 on average.
__global__ void __launch_bounds__(32) k_gamma_force(int n, const double* __restrict__ xyz,
                                                    const int* __restrict__ species, const int* __restrict__ atom_lo,
                                                    const int* __restrict__ atom_hi, const double* __restrict__ dq,
                                                    double invU0, double invU1, double* __restrict__ part) {
    const int a0 = blockIdx.x * 32, a = min(a0 + (int)threadIdx.x, n - 1);
    const int lo = atom_lo[a], hi = atom_hi[a];   // gamma couples atoms of one cluster only
    const double xa = xyz[3 * a], ya = xyz[3 * a + 1], za = xyz[3 * a + 2];
    const double ia = species[a] == 0 ? invU0 : invU1;
    int b0, b1;
    share_range(atom_lo[a0], atom_hi[min(a0 + 31, n - 1)], b0, b1);
    double f[3] = {0, 0, 0};
    for (int b = b0; b < b1; ++b) {
        const double dx = xa - xyz[3 * b], dy = ya - xyz[3 * b + 1], dz = za - xyz[3 * b + 2];
        const double h = 0.5 * (ia + (species[b] == 0 ? invU0 : invU1));
        const double g = rsqrt(dx * dx + dy * dy + dz * dz + h * h);
        const double w = b != a && b >= lo && b < hi ? dq[b] * g * g * g : 0.0;
        f[0] += w * dx;
        f[1] += w * dy;
        f[2] += w * dz;
    }
    if (a0 + (int)threadIdx.x >= n) return;
    for (int d = 0; d < 3; ++d) part[(size_t)blockIdx.y * 3 * n + 3 * a + d] = f[d];
}

// dE/dxyz: the gamma forces' shares and the molecules' pair forces
__global__ void k_grad_finish(int n_atoms, int n_shares, const double* __restrict__ part,
                              const double* __restrict__ dq, const double* __restrict__ gmol,
                              double* __restrict__ grad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 3 * n_atoms) return;
    double s = 0.0;
    for (int y = 0; y < n_shares; ++y) s += part[(size_t)y * 3 * n_atoms + i];
    grad[i] = gmol[i] - dq[i / 3] * s;
}

// parameter gradients: one warp per parameter
__global__ void k_par_finish(int n_mol, const double* __restrict__ pmol, double* __restrict__ dpar) {
    const int lane = threadIdx.x & 31, p = threadIdx.x >> 5;
    double s = 0.0;
    for (int m = lane; m < n_mol; m += 32) s += pmol[(size_t)m * 8 + p];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) dpar[p] = s;
}

}  // namespace

template <typename T>
static cudaError_t adjoint_t(Ctx* c, double* d_grad, double* d_par, double* d_gmol, double* d_pmol) {
    const int in = c->cur, zb = 1 - c->cur;
    const int gw = (c->n_groups + 31) / 32;
    const size_t smem_l = (size_t)2 * gw * 4;
    int max_nb = 1;
    for (int g = 0; g < c->n_groups; ++g) max_nb = std::max(max_nb, c->h_gnb_ptr[g + 1] - c->h_gnb_ptr[g]);
    const int per = std::min(max_nb, kZNb);
    constexpr bool kFP64 = std::is_same<T, double>::value;
    const size_t smem_z = (kFP64 ? kZmul64Smem : kZmulSmem) + z_lookup_smem(per), smem_g = grad_smem<T>(c->max_cl_otiles);
    if (smem_l > (size_t)kMaxDynSmem || smem_g > (size_t)kMaxDynSmem) return cudaErrorInvalidValue;
    cudaError_t e = allow_dynamic_smem<k_zlists>();
    if (e != cudaSuccess) return e;
    k_zlists<<<c->n_mol, 256, smem_l, c->stream>>>(
        c->n_occ_tiles, c->n_groups, c->cap, c->d_c_nt[in], c->d_c_tile[in], c->d_tile_group, c->d_group_ot0,
        c->d_group_not, c->d_gnb_ptr, c->d_gnb_col, c->d_c_nt[zb], c->d_c_tile[zb], &c->d_sc->err);
    const bool many = max_nb > kZNb;
    auto zmul = [&] {
        if constexpr (kFP64) {
            e = many ? allow_dynamic_smem<k_zmul64<true>>() : allow_dynamic_smem<k_zmul64<false>>();
            return many ? k_zmul64<true> : k_zmul64<false>;
        } else {
            e = many ? allow_dynamic_smem<k_zmul<true>>() : allow_dynamic_smem<k_zmul<false>>();
            return many ? k_zmul<true> : k_zmul<false>;
        }
    }();
    if (e != cudaSuccess) return e;
    // groups of molecules on grid y (65535 at most), out groups of their cluster on grid x
    for (int nb_lo = 0; nb_lo < max_nb; nb_lo += per)
        for (int g0 = 0; g0 < c->n_groups; g0 += 65535) {
            const int ng = std::min(65535, c->n_groups - g0);
            zmul<<<dim3(c->max_cl_groups, ng), kFP64 ? kZ64Threads : kZThreads, smem_z, c->stream>>>(
                g0, nb_lo, per, c->cap, c->d_group_cl, c->d_cl_g0, c->d_grp_mol_ptr, c->d_grp_mol, c->d_c_nt[in], c->d_c_tile[in],
                (const T*)c->d_c_val[in], c->d_group_ot0, c->d_group_not, c->d_gnb_ptr, c->d_gnb_col, c->d_ort_blk_tp[1],
                c->d_gnb_rev, (const T*)c->d_sig, c->d_c_nt[zb], c->d_c_tile[zb], (T*)c->d_c_val[zb]);
            c->n_launch += 1;
        }
    SKd P;
    for (int i = 0; i < 4; ++i) {
        P.V0[i] = c->prm.V0[i];
        P.S0[i] = c->prm.S0[i];
    }
    P.r_decay = c->prm.r_decay;
    P.rc2 = c->prm.r_cut * c->prm.r_cut;
    double* Pb = c->d_adj;
    double* Wb = Pb + (size_t)c->n_mp * 36;
    double* pt = Wb + (size_t)c->n_mp * 36;
    e = allow_dynamic_smem<k_grad_blocks<T>>();
    if (e != cudaSuccess) return e;
    k_grad_blocks<T><<<c->n_mol, kGradWarps * 32, smem_g, c->stream>>>(
        c->n_occ_tiles, c->max_cl_otiles, c->d_mol_ot0, c->cap, c->d_c_nt[in], c->d_c_tile[in],
        (const T*)c->d_c_val[in], c->d_c_nt[zb], c->d_c_tile[zb], (const T*)c->d_c_val[zb], c->d_mp_ptr, c->d_mp_col,
        c->d_mp_rev, Pb, Wb);
    k_pair_terms<<<dim3((c->n_mp + 127) / 128, 9), 128, 0, c->stream>>>(c->n_mp, c->d_mp_row, c->d_mp_col, c->d_xyz,
                                                                       c->d_Q, P, Pb, Wb, pt);
    k_pair_sum<<<(17 * c->n_mol + 127) / 128, 128, 0, c->stream>>>(c->n_mol, c->n_mp, c->d_mp_ptr, pt, d_gmol, d_pmol);
    k_gamma_force<<<dim3((c->n_atoms + 31) / 32, c->n_shares), 32, 0, c->stream>>>(
        c->n_atoms, c->d_xyz, c->d_species, c->d_atom_lo, c->d_atom_hi, c->d_dq, 1.0 / c->prm.U[0],
        1.0 / c->prm.U[1], c->d_share);
    k_grad_finish<<<(3 * c->n_atoms + 127) / 128, 128, 0, c->stream>>>(c->n_atoms, c->n_shares, c->d_share, c->d_dq,
                                                                      d_gmol, d_grad);
    k_par_finish<<<1, 8 * 32, 0, c->stream>>>(c->n_mol, d_pmol, d_par);
    c->n_launch += 7;
    return cudaGetLastError();
}

size_t adjoint_scratch_values(const Ctx* c) { return (size_t)c->n_mp * (36 + 36 + 9 * kPairOut); }

cudaError_t launch_adjoint(Ctx* c, double* d_grad, double* d_par, double* d_gmol, double* d_pmol) {
    return c->prec == SSCF_FP64 ? adjoint_t<double>(c, d_grad, d_par, d_gmol, d_pmol)
                                : adjoint_t<float>(c, d_grad, d_par, d_gmol, d_pmol);
}

}  // namespace sscf
