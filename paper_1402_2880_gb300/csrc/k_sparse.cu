// Sparse products of the C^T X C kernel (Section "Computation kernel for the
// matrix products C^T X C") and the density / Mulliken charges (Eq. pop).
//
// The paper builds C^T X C from 16-column strips of X C computed with dense
// 16x16 blocks. Here the 16-column strip is a tile: Y = X C is formed per
// tile column (column-major, only the row blocks reachable through X), and
// every kept block of C^T X C is one output-stationary 16x16 tile pair
// reduced over the row blocks the two columns share.
#include <cuda_bf16.h>

#include "block_scan.h"
#include "sscf_internal.h"
#include "sum3.h"

#include <algorithm>
#include <type_traits>

namespace sscf {

namespace {

template <typename T> struct Acc;
template <> struct Acc<double> { using type = double; };
template <> struct Acc<float> { using type = float; };

// ---------------------------------------------------------------------------
// Column index of C: per tile, the (row block, slot) pairs sorted by row.
// ---------------------------------------------------------------------------
__global__ void k_ci_count(int n_mol, int cap, const int* __restrict__ c_nt, const int* __restrict__ c_tile,
                           int* __restrict__ cnt) {
    int r = blockIdx.x;
    for (int s = threadIdx.x; s < c_nt[r]; s += blockDim.x) atomicAdd(&cnt[c_tile[(size_t)r * cap + s]], 1);
}

// exclusive scan of n counts into ptr (n + 1 entries); one CTA of 1024 threads
__global__ void k_scan(int n, const int* __restrict__ cnt, int* __restrict__ ptr) {
    __shared__ int part[33];
    const int per = (n + blockDim.x - 1) / blockDim.x;
    const int lo = threadIdx.x * per, hi = min(n, lo + per);
    int s = 0;
    for (int i = lo; i < hi; ++i) s += cnt[i];
    int run = block_scan(s, part);
    if (threadIdx.x == 0) ptr[n] = part[32];
    for (int i = lo; i < hi; ++i) {
        ptr[i] = run;
        run += cnt[i];
    }
}

__global__ void k_ci_fill(int n_mol, int cap, const int* __restrict__ c_nt, const int* __restrict__ c_tile,
                          const int* __restrict__ ptr, int* __restrict__ cursor, int* __restrict__ row,
                          int* __restrict__ slot) {
    int r = blockIdx.x;
    for (int s = threadIdx.x; s < c_nt[r]; s += blockDim.x) {
        int t = c_tile[(size_t)r * cap + s];
        int pos = ptr[t] + atomicAdd(&cursor[t], 1);
        row[pos] = r;
        slot[pos] = s;
    }
}

// Sort every tile's segment by row. The rows of one tile are distinct and lie
// in its cluster, so a bitmap over the cluster's rows orders them: an entry
// moves to the number of set bits below its row. One CTA per tile.
constexpr int kSortMax = 8192;          // entries per tile (16 per thread)
constexpr int kSortThreads = 512;
__global__ void __launch_bounds__(kSortThreads) k_ci_sort(const int* __restrict__ ptr, int* __restrict__ row,
                                                          int* __restrict__ slot, const int* __restrict__ tile_row0,
                                                          int n_rows, unsigned* __restrict__ err) {
    extern __shared__ unsigned sbits[];               // n_rows bits, then the set bits before each word
    const int nw = (n_rows + 31) >> 5;
    int* wpre = (int*)(sbits + nw);
    __shared__ int part[33];
    const int t = blockIdx.x;
    const int lo = ptr[t], n = ptr[t + 1] - lo;
    if (n <= 1) return;
    if (n > kSortMax) {
        if (threadIdx.x == 0) atomicOr(err, kErrSortSize);
        return;
    }
    const int r0 = tile_row0[t];
    for (int w = threadIdx.x; w < nw; w += blockDim.x) sbits[w] = 0u;
    __syncthreads();
    constexpr int kPer = kSortMax / kSortThreads;
    int rv[kPer], sv[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int i = threadIdx.x + j * kSortThreads;
        if (i < n) {
            rv[j] = row[lo + i];
            sv[j] = slot[lo + i];
            const int rr = rv[j] - r0;
            atomicOr(&sbits[rr >> 5], 1u << (rr & 31));
        }
    }
    __syncthreads();
    const int per = (nw + blockDim.x - 1) / blockDim.x;
    const int w0 = threadIdx.x * per, w1 = min(nw, w0 + per);
    int c = 0;
    for (int w = w0; w < w1; ++w) c += __popc(sbits[w]);
    int run = block_scan(c, part);
    for (int w = w0; w < w1; ++w) {
        wpre[w] = run;
        run += __popc(sbits[w]);
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int i = threadIdx.x + j * kSortThreads;
        if (i < n) {
            const int rr = rv[j] - r0;
            const int pos = wpre[rr >> 5] + __popc(sbits[rr >> 5] & ((1u << (rr & 31)) - 1u));
            row[lo + pos] = rv[j];
            slot[lo + pos] = sv[j];
        }
    }
}

// The whole column index in one CTA, for small systems (kCiSmallEntries): a bit
// per (tile, row block) in shared memory; the set bits before a row are its
// place in the tile's list, so that nothing is sorted. Four launches and two
// memsets of a few microseconds each otherwise: 20 us of kernels and the gaps
// between them a call at 8 molecules, now 4.6; at 343 (54,880 entries) one CTA
// took 65 us, the launches 32.
constexpr long long kCiSmallEntries = 12288;      // rows x capacity
constexpr size_t kCiSmallSmem = 96 * 1024;
__global__ void __launch_bounds__(1024) k_ci_small(int n_mol, int n_tiles, int cap, const int* __restrict__ c_nt,
                                                   const int* __restrict__ c_tile, int* __restrict__ ptr,
                                                   int* __restrict__ row, int* __restrict__ slot) {
    extern __shared__ unsigned cbits[];               // [n_tiles][words], then the tiles' starts
    const int words = (n_mol + 31) >> 5;
    int* start = (int*)(cbits + (size_t)n_tiles * words);
    __shared__ int s_w[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < n_tiles * words; i += blockDim.x) cbits[i] = 0u;
    __syncthreads();
    for (int r = warp; r < n_mol; r += 32)
        for (int s = lane; s < c_nt[r]; s += 32)
            atomicOr(&cbits[(size_t)c_tile[(size_t)r * cap + s] * words + (r >> 5)], 1u << (r & 31));
    __syncthreads();
    int base = 0;   // entries of the tiles before this round's 1024
    for (int t0 = 0; t0 < n_tiles; t0 += 1024) {
        const int t = t0 + threadIdx.x;
        int cnt = 0;
        if (t < n_tiles)
            for (int w = 0; w < words; ++w) cnt += __popc(cbits[(size_t)t * words + w]);
        int inc = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) s_w[warp] = inc;
        __syncthreads();
        int before = base, total = base;
        for (int w = 0; w < 32; ++w) {
            before += w < warp ? s_w[w] : 0;
            total += s_w[w];
        }
        if (t < n_tiles) start[t] = ptr[t] = before + inc - cnt;
        base = total;
        __syncthreads();
    }
    if (threadIdx.x == 0) ptr[n_tiles] = base;
    for (int r = warp; r < n_mol; r += 32)
        for (int s = lane; s < c_nt[r]; s += 32) {
            const int t = c_tile[(size_t)r * cap + s];
            const unsigned* b = cbits + (size_t)t * words;
            int pos = start[t] + __popc(b[r >> 5] & ((1u << (r & 31)) - 1u));
            for (int w = 0; w < (r >> 5); ++w) pos += __popc(b[w]);
            row[pos] = r;
            slot[pos] = s;
        }
}

// ---------------------------------------------------------------------------
// Y[:, t] = X C[:, t] for tiles t in [tile_lo, tile_hi), column-major output.
// One CTA per tile: mark the row blocks reachable from the tile's rows
// through the molecule-pair pattern (tiles below own_below: the tile's own
// rows only; n_share CTAs per tile do that each and share the rows, so that a
// few tiles fill the GPU), then one warp per output row block sums X[r, n] (6x6)
// C[n, t] (6x16) over the pattern neighbours n holding t.
// ---------------------------------------------------------------------------
// CTAs per SM that a launch aims at (FP32, one CTA per tile: 4.4 ms at 4096 molecules, 1.18 at 997;
// 8: 4.4 and 0.73; 32: 3.7 and 0.68; FP64 at 343: 1.86 -> 0.99)
// clusters of a few rows in a batch, H and S, us, so many CTAs against four rows per warp: 1000 of 3
// molecules, FP32 56 + 49, 28 + 25, FP64 59 + 51, 45 + 29; 300 of 30, FP32 264 + 229, 210 + 162, FP64
// 1475 + 984, 1417 + 963
constexpr int kXcCtas = 32;
constexpr int kXcBatch = 4;   // matched neighbours whose loads are in flight together
template <typename T>
__global__ void k_xc(int tile_lo, int n_t, int n_share, int n_rows, int own_below, int cap, int capY, const int* __restrict__ tile_row0,
                     const int* __restrict__ cci_ptr, const int* __restrict__ cci_row,
                     const int* __restrict__ cci_slot, const T* __restrict__ c_val, const int* __restrict__ mp_ptr,
                     const int* __restrict__ mp_col, const T* __restrict__ Xb, int* __restrict__ y_n,
                     int* __restrict__ y_row, T* __restrict__ y_val, unsigned* __restrict__ err) {
    // row maps are local to the tile's cluster: row r -> r - r0, n_rows = largest cluster
    extern __shared__ int sm[];
    const int nw = (n_rows + 31) / 32;
    unsigned* bits = (unsigned*)sm;               // n_rows bits
    int* wpre = (int*)(bits + nw);                // prefix of popcounts per word
    short* rowpos = (short*)(wpre + nw);          // n_rows: index into the tile's column list or -1
    __shared__ int part[33];
    // tiles from own_below on (the longer ones: every reachable row) first
    const int t = tile_lo + (int)((blockIdx.x / n_share + (unsigned)max(own_below - tile_lo, 0)) % n_t);
    const int share = blockIdx.x % n_share;   // of the tile's rows of Y
    const int r0 = tile_row0[t];
    const int lo = cci_ptr[t], nc = cci_ptr[t + 1] - lo;
    if (nc > 32767) {   // the 16-bit row map cannot index this column
        if (threadIdx.x == 0) {
            atomicOr(err, kErrCapacity);
            y_n[t] = 0;
        }
        return;
    }
    for (int i = threadIdx.x; i < n_rows; i += blockDim.x) rowpos[i] = -1;
    for (int i = threadIdx.x; i < nw; i += blockDim.x) bits[i] = 0u;
    __syncthreads();
    for (int k = threadIdx.x; k < nc; k += blockDim.x) rowpos[cci_row[lo + k] - r0] = (short)k;
    for (int k = threadIdx.x; k < nc; k += blockDim.x) {
        int r = cci_row[lo + k];
        if (t < own_below) {   // Y only where C[:, t] has rows: enough for C[:, t]^T Y[:, t]
            const int n = r - r0;
            atomicOr(&bits[n >> 5], 1u << (n & 31));
            continue;
        }
        for (int e = mp_ptr[r]; e < mp_ptr[r + 1]; ++e) {
            int n = mp_col[e] - r0;
            atomicOr(&bits[n >> 5], 1u << (n & 31));
        }
    }
    __syncthreads();
    const int w_per = (nw + blockDim.x - 1) / blockDim.x;
    const int w0 = threadIdx.x * w_per, w1 = min(nw, w0 + w_per);
    int n_set = 0;
    for (int w = w0; w < w1; ++w) n_set += __popc(bits[w]);
    int before = block_scan(n_set, part);
    for (int w = w0; w < w1; ++w) {
        wpre[w] = before;
        before += __popc(bits[w]);
    }
    __syncthreads();
    const int ny = part[32];
    if (ny > capY) {
        if (threadIdx.x == 0) {
            atomicOr(err, kErrCapacity);
            y_n[t] = 0;
        }
        return;
    }
    if (threadIdx.x == 0 && share == 0) y_n[t] = ny;
    // write sorted row list (every share writes the same and reads its own rows)
    for (int w = threadIdx.x; w < nw; w += blockDim.x) {
        unsigned b = bits[w];
        int p = wpre[w];
        while (b) {
            int i = __ffs(b) - 1;
            b &= b - 1;
            y_row[(size_t)t * capY + p++] = r0 + w * 32 + i;
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    // A lane's outputs: FP64 three AO rows of one column; FP32 two AO rows of two columns, which
    // takes 6 loads of C and 3 of X a neighbour where the other needs 6 and 9 (and leaves a quarter of
    // the lanes idle): the loads bound the FP32 kernel (4096 molecules, H and S: 3.7 + 2.7 ms, now 3.5 + 2.4)
    constexpr bool kWide = std::is_same<T, float>::value;
    const int col = kWide ? 2 * (lane & 7) : lane & 15;
    const int q0 = kWide ? 2 * min(lane >> 3, 2) : lane >> 4;   // FP64: AO rows q0, q0 + 2, q0 + 4
    const bool idle = kWide && lane >= 24;
    for (int k = share * nwarps + warp; k < ny; k += n_share * nwarps) {
        const int r = y_row[(size_t)t * capY + k];
        T acc0 = 0, acc1 = 0, acc2 = 0;
        float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        // 32 pattern neighbours at a time: their ids, positions and slots are
        // looked up in parallel, one per lane; the matched ones are then summed
        // in pattern order with their data broadcast from the owning lane
        const int e_lo = mp_ptr[r], e_hi = mp_ptr[r + 1];
        for (int eb = e_lo; eb < e_hi; eb += 32) {
            const int e = eb + lane;
            int sl = -1, nl = 0;
            if (e < e_hi) {
                nl = mp_col[e];
                const int j = rowpos[nl - r0];
                if (j >= 0) sl = cci_slot[lo + j];
            }
            unsigned mm = __ballot_sync(0xffffffffu, sl >= 0);
            while (mm) {
                // kXcBatch matched neighbours per round: their loads in flight together, sums in order
                int src[kXcBatch];
#pragma unroll
                for (int u = 0; u < kXcBatch; ++u) {
                    src[u] = mm ? __ffs(mm) - 1 : -1;
                    if (mm) mm &= mm - 1;
                }
                if constexpr (kWide) {
                    float2 c6[kXcBatch][6];
                    float x[kXcBatch][12];   // AO rows q0, q0 + 1 of the 6x6 block
#pragma unroll
                    for (int u = 0; u < kXcBatch; ++u) {
                        const int sv = src[u] < 0 ? 0 : src[u];
                        const int n = __shfl_sync(0xffffffffu, nl, sv);
                        const int ss = __shfl_sync(0xffffffffu, sl, sv);
                        if (src[u] >= 0) {
                            const T* cv = c_val + ((size_t)n * cap + ss) * kTileVals + col;
                            const float4* xb = (const float4*)(Xb + (size_t)(eb + sv) * 36 + q0 * 6);
#pragma unroll
                            for (int q = 0; q < 6; ++q) c6[u][q] = *(const float2*)(cv + q * kTileW);
#pragma unroll
                            for (int h = 0; h < 3; ++h) *(float4*)&x[u][4 * h] = xb[h];
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kXcBatch; ++u) {
                        if (src[u] < 0) continue;
#pragma unroll
                        for (int q = 0; q < 6; ++q) {
                            acc[0] = __ffma2_rn(make_float2(x[u][q], x[u][q]), c6[u][q], acc[0]);
                            acc[1] = __ffma2_rn(make_float2(x[u][6 + q], x[u][6 + q]), c6[u][q], acc[1]);
                        }
                    }
                } else {
                    T c6[kXcBatch][6];
                    const T* xb[kXcBatch];
#pragma unroll
                    for (int u = 0; u < kXcBatch; ++u) {
                        const int sv = src[u] < 0 ? 0 : src[u];
                        const int n = __shfl_sync(0xffffffffu, nl, sv);
                        const int ss = __shfl_sync(0xffffffffu, sl, sv);
                        xb[u] = Xb + (size_t)(eb + sv) * 36;
                        if (src[u] >= 0) {
                            const T* cv = c_val + ((size_t)n * cap + ss) * kTileVals + col;
#pragma unroll
                            for (int q = 0; q < 6; ++q) c6[u][q] = cv[q * kTileW];
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kXcBatch; ++u) {
                        if (src[u] < 0) continue;
                        // the lane's three rows of the 6x6 block, two values per load
                        double xr[3][6];
#pragma unroll
                        for (int rr = 0; rr < 3; ++rr) {
                            const double2* x2 = (const double2*)(xb[u] + (q0 + 2 * rr) * 6);
#pragma unroll
                            for (int h = 0; h < 3; ++h) {
                                const double2 v = x2[h];
                                xr[rr][2 * h] = v.x;
                                xr[rr][2 * h + 1] = v.y;
                            }
                        }
#pragma unroll
                        for (int q = 0; q < 6; ++q) {
                            acc0 += xr[0][q] * c6[u][q];
                            acc1 += xr[1][q] * c6[u][q];
                            acc2 += xr[2][q] * c6[u][q];
                        }
                    }
                }
            }
        }
        T* yv = y_val + ((size_t)t * capY + k) * kTileVals;
        if constexpr (kWide) {
            if (!idle) {
                *(float2*)(yv + q0 * kTileW + col) = acc[0];
                *(float2*)(yv + (q0 + 1) * kTileW + col) = acc[1];
            }
        } else {
            yv[(q0)*kTileW + col] = acc0;
            yv[(q0 + 2) * kTileW + col] = acc1;
            yv[(q0 + 4) * kTileW + col] = acc2;
        }
    }
}

// ---------------------------------------------------------------------------
// Tile-pair transform: out[p] (16x16) = C[:, a]^T Y[:, b] for every listed
// pair (a, b). CTAs (a, split) share tile a's pairs, each with a map row block ->
// slot of a in shared memory. Rows are summed in ascending order (fixed order),
// 32 of b's rows at a time. FP64 storage here; FP32 storage: k_transform_tc.
//
// A quarter of an SM starts one FP64 instruction of a warp every 64 clocks, busy
// or not, so a CTA's four warps work on one pair, four columns of b each; with a
// pair per warp, a system with fewer pairs than four per SM waited for three
// quarters idle (32 molecules 89 us a launch, now 29; 343 3.8 + 2.1 ms, now 3.2 + 1.9). They walk b's rows (sorted) and stage the 6x16 tiles
// C[r, a] and Y[r, b] of the rows present in a, kStage row blocks at a time, into
// one of two buffers while the loads of the next ones are in flight; a lane
// owns 2x1 of the result and takes a 16-byte and an 8-byte shared load for two FMAs.
// ---------------------------------------------------------------------------
constexpr int kTfWarps = 4;
constexpr int kStage = 4;   // row blocks staged at a time
constexpr int kTfStageVals = kStage * 2 * kTileVals;   // values of a buffer: [kStage][2][96]

__global__ void __launch_bounds__(kTfWarps * 32)
k_transform(int n_split, int n_rows, const int* __restrict__ tile_row0, int cap, int capY, const int* __restrict__ tp_ptr,
            const int* __restrict__ tp_b, const int* __restrict__ tp_out, const int* __restrict__ cci_ptr,
            const int* __restrict__ cci_row, const int* __restrict__ cci_slot, const double* __restrict__ c_val,
            const int* __restrict__ y_n, const int* __restrict__ y_row, const double* __restrict__ y_val,
            double* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char sraw[];
    double2* stage = (double2*)sraw;                                 // two buffers
    short* slot_of = (short*)((double*)sraw + 2 * kTfStageVals);     // n_rows (cluster-local)
    // CTA (a, s) takes the pairs of tile a with index = s (mod n_split)
    const int a = blockIdx.x / n_split, split = blockIdx.x % n_split;
    const int p0 = tp_ptr[a], p1 = tp_ptr[a + 1];
    if (p0 + split >= p1) return;
    const int r0 = tile_row0[a];
    const int lo = cci_ptr[a], nc = cci_ptr[a + 1] - lo;
    for (int i = threadIdx.x; i < n_rows; i += blockDim.x) slot_of[i] = -1;
    __syncthreads();
    for (int k = threadIdx.x; k < nc; k += blockDim.x) slot_of[cci_row[lo + k] - r0] = (short)cci_slot[lo + k];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i0 = 2 * (lane >> 2), j0 = 4 * warp + (lane & 3);
    constexpr int kHalf = kTileVals / 2, kLoads = kStage * 2 * kHalf / (kTfWarps * 32);   // 16-byte pieces
    static_assert(kLoads * kTfWarps * 32 == kStage * 2 * kHalf, "");
    int phase = 0;
    for (int p = p0 + split; p < p1; p += n_split) {
        const int b = tp_b[p];
        const int nb = y_n[b];
        const int* yr = y_row + (size_t)b * capY;
        int k0 = -32, at = -1;   // the 32 rows being staged; a lane's tile C[r, a] among them
        unsigned m = 0;          // those not staged yet
        // the next up to kStage matched row blocks: their number (0: none left), and this thread's pieces
        double2 v[kLoads];
        auto next = [&] {
            while (!m) {
                k0 += 32;
                if (k0 >= nb) return 0;
                at = -1;
                if (k0 + lane < nb) {
                    const int r = yr[k0 + lane], sl = slot_of[r - r0];
                    if (sl >= 0) at = r * cap + sl;
                }
                m = __ballot_sync(0xffffffffu, at >= 0);
            }
            int n = 0, tile[kStage], row[kStage];
#pragma unroll
            for (int g = 0; g < kStage; ++g) {
                const int src = m ? __ffs(m) - 1 : 0;
                n += m != 0;
                m &= m - 1;
                tile[g] = __shfl_sync(0xffffffffu, at, src);
                row[g] = k0 + src;
            }
#pragma unroll
            for (int j = 0; j < kLoads; ++j) {
                const int piece = threadIdx.x + j * kTfWarps * 32, g = piece / (2 * kHalf), q = piece % (2 * kHalf);
                int t = tile[0], k = row[0];
#pragma unroll
                for (int h = 1; h < kStage; ++h)
                    if (g == h) {
                        t = tile[h];
                        k = row[h];
                    }
                if (g < n)
                    v[j] = q < kHalf ? *((const double2*)(c_val + (size_t)t * kTileVals) + q)
                                     : *((const double2*)(y_val + ((size_t)b * capY + k) * kTileVals) + q - kHalf);
            }
            return n;
        };
        double sum0 = 0.0, sum1 = 0.0, acc0 = 0.0, acc1 = 0.0;
        int n = next();
        while (n) {
            double2* buf = stage + phase * (kTfStageVals / 2);
            phase ^= 1;
#pragma unroll
            for (int j = 0; j < kLoads; ++j) {
                const int piece = threadIdx.x + j * kTfWarps * 32;
                if (piece < n * 2 * kHalf) buf[piece] = v[j];
            }
            __syncthreads();   // (the other buffer's readers are past it before anyone writes there again)
            const bool last = m == 0;   // of these 32 rows
            const int staged = n;
            n = next();
            for (int g = 0; g < staged; ++g) {
                const double* bc = (const double*)(buf + (size_t)g * 2 * kHalf);
                const double* by = bc + kTileVals;
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    const double2 c = *(const double2*)(bc + q * 16 + i0);
                    const double y = by[q * 16 + j0];
                    acc0 += c.x * y;
                    acc1 += c.y * y;
                }
            }
            if (last) {
                sum0 += acc0;
                sum1 += acc1;
                acc0 = acc1 = 0.0;
            }
        }
        double* o = out + (size_t)tp_out[p] * 256;
        o[i0 * 16 + j0] = sum0;
        o[(i0 + 1) * 16 + j0] = sum1;
    }
}

// x = hi + lo with hi, lo in TF32 (10 explicit mantissa bits each): hi by
// round-to-nearest, ties away, lo the rounded remainder, so hi + lo carries ~21
// bits. Rounded in the bits, as cvt.rna.tf32 rounds (the kernel ran 5 % longer
// with that instruction). The last step keeps a NaN, which the bits would lose;
// an infinite x has a NaN remainder.
__device__ __forceinline__ uint32_t round_tf32(float x) { return (__float_as_uint(x) + 0x1000u) & 0xffffe000u; }
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
    hi = round_tf32(x);
    const float r = x - __uint_as_float(hi);
    lo = __float_as_uint(__fmaf_rn(r, 0.f, __uint_as_float(round_tf32(r))));
}

// D (16x8, FP32) += A (16x8, TF32, row-major) x B (8x8, TF32, column-major)
__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// FP32 storage: the 16x16 block of a pair as two m16n8 tensor-core tiles, K = the
// AO rows of up to four matched row blocks (24 rows, 3 k-steps of 8) at a time.
// Each product is split into TF32 hi + lo parts and summed as hi*hi + hi*lo +
// lo*hi (the lo*lo term is below FP32 rounding), into FP32 fragments that are
// added up in FP64 every 32 of b's rows (one alone, in a small system, is taken as it is: 2 us of a launch's 19).
// A row of a 6x16 tile is 64 bytes, so a warp reads a fragment's four rows of two
// columns per lane straight from memory: no staging, no shared-memory traffic, and
// a's tiles are found in L1 by the CTA's other warps (b's pass it by). Bound by the
// splits (48 of ~75 instructions a k-step) and the L2 latency that three CTAs'
// 80-register warps leave uncovered (issue slots 55 % used); four CTAs spill, two
// are 20 % slower. Staged through shared memory, with cvt.rna.tf32: 6.45 + 3.95 ms
// for the two transforms of an early iteration at 4096 molecules, now 5.27 + 3.17; at
// 997 1.50 + 1.21, now 1.18 + 0.81. (The sums in two floats, 48 bits: 5.06 + 2.97
// and 1.13 + 0.78, but they are to carry no less than FP64 does.)
constexpr int kTcWarps = 8, kTcCtas = 3;
__device__ __forceinline__ float2 load_stream(const float* p) {
    float2 v;
    asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__global__ void __launch_bounds__(kTcWarps * 32, kTcCtas)
k_transform_tc(int n_split, int n_rows, const int* __restrict__ tile_row0, int cap, int capY,
               const int* __restrict__ tp_ptr, const int* __restrict__ tp_b, const int* __restrict__ tp_out,
               const int* __restrict__ cci_ptr, const int* __restrict__ cci_row, const int* __restrict__ cci_slot,
               const float* __restrict__ c_val, const int* __restrict__ y_n, const int* __restrict__ y_row,
               const float* __restrict__ y_val, float* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char sraw[];
    int2* lists = (int2*)sraw;                       // [warps][32]: matched row blocks (tile of C, b's position)
    short* slot_of = (short*)(lists + kTcWarps * 32);   // n_rows (cluster-local)
    // CTA (a, s) takes the pairs of tile a with index = s (mod n_split)
    const int a = blockIdx.x / n_split, split = blockIdx.x % n_split;
    const int p0 = tp_ptr[a], p1 = tp_ptr[a + 1];
    if (p0 + split >= p1) return;
    const int r0 = tile_row0[a];
    const int lo = cci_ptr[a], nc = cci_ptr[a + 1] - lo;
    for (int i = threadIdx.x; i < n_rows; i += blockDim.x) slot_of[i] = -1;
    __syncthreads();
    for (int k = threadIdx.x; k < nc; k += blockDim.x) slot_of[cci_row[lo + k] - r0] = (short)cci_slot[lo + k];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int2* list = lists + warp * 32;
    const int gq = lane >> 2, tq = lane & 3;
    // A k-step's fragments are rows tq and tq + 4 of its eight. Over the 24 rows of four blocks these are
    // rows tq | lowhi, tq+2, tq | lowhi, tq+2 of blocks 0, 0|1, 1, 2, 2|3, 3, where lowhi is row tq + 4 of the
    // one block or row tq - 2 of the next. A fragment's columns gq and gq + 8 are columns 2gq and 2gq + 1.
    const bool early = tq < 2;
    const int o0 = tq * 16 + 2 * gq, o1 = (early ? tq + 4 : tq - 2) * 16 + 2 * gq, o2 = (tq + 2) * 16 + 2 * gq;
    // the next pair's tile, row count and first rows, and the next 32 rows of this one, are read ahead
    const int step = kTcWarps * n_split;
    int p = p0 + split + warp * n_split;
    int b = p < p1 ? tp_b[p] : 0, nb = p < p1 ? y_n[b] : 0;
    int r = lane < nb ? y_row[(size_t)b * capY + lane] : -1;
    int b_next = p + step < p1 ? tp_b[p + step] : 0;
    for (; p < p1; p += step) {
        const int nb_next = p + step < p1 ? y_n[b_next] : 0;
        const int b_after = p + 2 * step < p1 ? tp_b[p + 2 * step] : 0;
        const int* yr = y_row + (size_t)b * capY;
        const float* yb = y_val + (size_t)b * capY * kTileVals;
        float acc[2][4];
        double sum[2][4];
        bool added = false;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[h][q] = 0.f;
        for (int k0 = 0; k0 < nb; k0 += 32) {
            const int k = k0 + lane;
            int at = -1;   // index of the tile C[r, a]
            if (r >= 0) {
                const int sl = slot_of[r - r0];
                if (sl >= 0) at = r * cap + sl;
            }
            if (k0 + 32 < nb)
                r = k + 32 < nb ? yr[k + 32] : -1;
            else
                r = lane < nb_next ? y_row[(size_t)b_next * capY + lane] : -1;
            const unsigned m = __ballot_sync(0xffffffffu, at >= 0);
            if (!m) continue;   // nothing to add, nothing to flush
            if (at >= 0) list[__popc(m & ((1u << lane) - 1u))] = make_int2(at, k);
            __syncwarp();
            const int n = __popc(m);
            for (int g = 0; g < n; g += kStage) {
                const int rows = min(n - g, kStage) * kAoPerMol;
                float2 cv[6], yv[6];
#pragma unroll
                for (int u = 0; u < 6; ++u) {
                    // blocks 0, 0|1, 1, 2, 2|3, 3
                    const int blk = u == 0 ? 0 : u == 1 ? (early ? 0 : 1) : u == 2 ? 1 : u == 3 ? 2 : u == 4 ? (early ? 2 : 3) : 3;
                    const int off = u % 3 == 0 ? o0 : u % 3 == 1 ? o1 : o2;
                    cv[u] = yv[u] = make_float2(0.f, 0.f);
                    if (4 * u + tq < rows) {
                        const int2 e = list[g + blk];
                        cv[u] = *(const float2*)(c_val + (size_t)e.x * kTileVals + off);
                        yv[u] = load_stream(yb + (size_t)e.y * kTileVals + off);
                    }
                }
#pragma unroll
                for (int u = 0; u < 3; ++u) {
                    if (8 * u >= rows) break;
                    uint32_t ah[4], al[4];
                    split_tf32(cv[2 * u].x, ah[0], al[0]);
                    split_tf32(cv[2 * u].y, ah[1], al[1]);
                    split_tf32(cv[2 * u + 1].x, ah[2], al[2]);
                    split_tf32(cv[2 * u + 1].y, ah[3], al[3]);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        uint32_t bh[2], bl[2];
                        split_tf32(h ? yv[2 * u].y : yv[2 * u].x, bh[0], bl[0]);
                        split_tf32(h ? yv[2 * u + 1].y : yv[2 * u + 1].x, bh[1], bl[1]);
                        mma_tf32(acc[h], al, bh);
                        mma_tf32(acc[h], ah, bl);
                        mma_tf32(acc[h], ah, bh);
                    }
                }
            }
            __syncwarp();
            if (!added && k0 + 32 >= nb) break;   // the only partial sums: as they are
            if (added) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int q = 0; q < 4; ++q) sum[h][q] += (double)acc[h][q];
            } else {
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int q = 0; q < 4; ++q) sum[h][q] = (double)acc[h][q];
            }
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[h][q] = 0.f;
            added = true;
        }
        if (added)
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[h][q] = (float)sum[h][q];
        // rows 2gq and 2gq + 1 of the block, columns 4tq to 4tq + 3
        float4* o = (float4*)(out + (size_t)tp_out[p] * 256) + 8 * gq + tq;
        o[0] = make_float4(acc[0][0], acc[1][0], acc[0][1], acc[1][1]);
        o[4] = make_float4(acc[0][2], acc[1][2], acc[0][3], acc[1][3]);
        if (nb == 0) r = lane < nb_next ? y_row[(size_t)b_next * capY + lane] : -1;
        b = b_next;
        nb = nb_next;
        b_next = b_after;
    }
}

// diag(F) per MO from the diagonal tile pairs
template <typename T>
__global__ void k_extract_diag(int n_tiles, const int* __restrict__ tile_mo0, const int* __restrict__ tile_nmo,
                               const T* __restrict__ Ft, double* __restrict__ Fd) {
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n_tiles * 16) return;
    int t = idx >> 4, c = idx & 15;
    if (c < tile_nmo[t]) Fd[tile_mo0[t] + c] = (double)Ft[(size_t)t * 256 + c * 17];
}

// ---------------------------------------------------------------------------
// Density: P_mn = 2 sum_{occ tiles t in rows m and n} C[m,t] C[n,t]^T on the
// molecule-pair pattern; q_a += sum_{mu in a} sum_nu P_mu,nu S_mu,nu and the
// band energy sum P*H0 per molecule (Eq. pop). One CTA per row block m, one
// warp per neighbour n >= m (P_nm = P_mn^T): each pair's shares of q and of
// the band energy are written for both rows, and k_density_sum adds them per
// molecule in neighbour order.
// ---------------------------------------------------------------------------
constexpr int kDensWarps = 8;
constexpr int kDensFlush = 32;  // tiles per lane in one FP32 sum
constexpr int kDensUnroll = 1;  // shared tiles per half-warp and round (2 measured no faster)
constexpr int kDensMinBlocks = 2;   // resident CTAs per SM the register budget aims at
// FP32 storage adds its partial sums of 32 products in three floats (Sum3; FP64
// before): the FP64 pipe, two lanes per clock and SM, was two thirds busy with
// them and with the sums over a warp (density at 997 and 4096 molecules 0.55 and
// 3.60 ms, now 0.43 and 2.83). A lane keeps two floats in shared memory and the
// third, 2^-48 of the sum, as eight bits of bf16 in a register (as floats: 0.47 and
// 3.14 ms): 56 bits where FP64 carried 53.

// s += v; lost: what the two floats of s drop of it
__device__ __forceinline__ void sum_add(float2& s, float v, float& lost) {
    float h, l, e;
    two_sum(s.x, v, h, e);
    two_sum(s.y, e, l, lost);
    s = make_float2(h, l);
}

// The sums of a pair's 36 products over its 32 lanes: lane u sums product u (32
// entries, from entry u on around: no bank conflicts) and four entries of one of
// the last four products, which the eight lanes that share it then add up.
__device__ __forceinline__ void pair_sums(const float2* acc, int lane, double& p0, double& p1) {
    const float2 *row0 = acc + lane * 32, *row1 = acc + (32 + (lane >> 3)) * 32 + 4 * (lane & 7);
    Sum3 s0 = {0.f, 0.f, 0.f}, s1 = {0.f, 0.f, 0.f};
    for (int j = 0; j < 32; ++j) s0.add(row0[(j + lane) & 31]);
    for (int j = 0; j < 4; ++j) s1.add(row1[(j + (lane >> 3)) & 3]);
    p0 = s0.value();
    p1 = s1.value();
}

template <typename T>
__global__ void __launch_bounds__(kDensWarps * 32, kDensMinBlocks)
k_density(int n_occ_tiles, int map_n, const int* __restrict__ mol_ot0, int cap, const int* __restrict__ c_nt,
          const int* __restrict__ c_tile, const T* __restrict__ c_val, const int* __restrict__ mp_ptr,
          const int* __restrict__ mp_col, const double* __restrict__ H0b, const double* __restrict__ Sb,
          const int* __restrict__ mp_rev, double2* __restrict__ dpart, double* __restrict__ P_out) {
    // slot of every occupied tile of m's cluster in row m, or -1 (map_n = largest cluster);
    // then the sums of each lane's 36 products (in mixed precision of FP32 sums of
    // kDensFlush tiles each), kept in shared memory to save registers
    extern __shared__ int smap[];
    constexpr bool kSplit = !std::is_same<typename Acc<T>::type, double>::value;   // FP32 storage
    double* sacc = (double*)(smap + ((map_n + 1) & ~1));   // [warp][36][32]: the lanes' sums
    const int m = blockIdx.x;
    const int t0 = mol_ot0[m];
    // P_nm = P_mn^T: this CTA takes the pairs with n >= m (neighbour lists are
    // sorted) and hands each pair's share of the charges and of the band
    // energy to both rows
    __shared__ int s_jlo;
    if (threadIdx.x == 0) s_jlo = 0;
    for (int i = threadIdx.x; i < map_n; i += blockDim.x) smap[i] = -1;
    __syncthreads();
    for (int w = threadIdx.x; w < mp_ptr[m + 1] - mp_ptr[m]; w += blockDim.x)
        if (mp_col[mp_ptr[m] + w] < m) atomicAdd(&s_jlo, 1);
    const int ntm = c_nt[m];
    for (int s = threadIdx.x; s < ntm; s += blockDim.x) {
        int t = c_tile[(size_t)m * cap + s];
        if (t < n_occ_tiles) smap[t - t0] = s;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int e0 = mp_ptr[m], ne = mp_ptr[m + 1] - e0;
    using A = typename Acc<T>::type;
    const int col = lane & 15, half = lane >> 4;
    double* wsum = sacc + (size_t)warp * 36 * 32;
    using L = typename std::conditional<kSplit, float2, double>::type;
    __nv_bfloat162 low[18];
    // a lane's next partial sums
    auto flush = [&](A* acc, int part) {
        L* d = (L*)wsum + lane;
#pragma unroll
        for (int u = 0; u < 36; u += 2) {
            if constexpr (kSplit) {
                if (part == 0) {
                    d[u * 32] = make_float2(acc[u], 0.f);
                    d[u * 32 + 32] = make_float2(acc[u + 1], 0.f);
                } else {
                    float l0, l1;
                    sum_add(d[u * 32], acc[u], l0);
                    sum_add(d[u * 32 + 32], acc[u + 1], l1);
                    low[u / 2] = __hadd2(low[u / 2], __floats2bfloat162_rn(l0, l1));
                }
            } else {
                d[u * 32] = acc[u];
                d[u * 32 + 32] = acc[u + 1];
            }
            acc[u] = acc[u + 1] = 0;
        }
    };
    // sum_id: atoms of m, atoms of n, energy; take: which of its nine products the lane adds
    const int sum_id = lane >> 2;
    unsigned take = 0;
    for (int j = 0; j < 9; ++j) {
        const int u = 9 * (lane & 3) + j, ao = sum_id < 3 ? u / 6 : u % 6, atom = max(ao - 3, 0);
        if (sum_id == 6 || atom == sum_id % 3) take |= 1u << j;
    }
    for (int w = s_jlo + warp; w < ne; w += kDensWarps) {
        const int e = e0 + w;
        const int n = mp_col[e];
        A acc[36];
        int n_part = 0;   // partial sums of this lane so far
        if constexpr (kSplit)
#pragma unroll
            for (int u = 0; u < 18; ++u) low[u] = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 36; ++u) acc[u] = 0;
        const int ntn = c_nt[n];
        int since = 0;
        // 32 of n's tiles at a time: one coalesced load of their ids, the shared
        // ones found with one ballot; then each half-warp takes kDensUnroll shared
        // tiles per round, so their loads are in flight together
        for (int base = 0; base < ntn; base += 32) {
            const int s = base + lane;
            const int t = s < ntn ? c_tile[(size_t)n * cap + s] : n_occ_tiles;
            const int sm_ = t < n_occ_tiles ? smap[t - t0] : -1;
            unsigned mm = __ballot_sync(0xffffffffu, sm_ >= 0);
            const bool virt_seen = __any_sync(0xffffffffu, s < ntn && t >= n_occ_tiles);
            while (mm) {
                int src[kDensUnroll];
#pragma unroll
                for (int u = 0; u < kDensUnroll; ++u) {
                    // bits in order: half 0 takes the 1st, 3rd, ..., half 1 the 2nd, 4th, ...
                    int b0 = -1, b1 = -1;
                    if (mm) {
                        b0 = __ffs(mm) - 1;
                        mm &= mm - 1;
                    }
                    if (mm) {
                        b1 = __ffs(mm) - 1;
                        mm &= mm - 1;
                    }
                    src[u] = half ? b1 : b0;
                }
                A a6[kDensUnroll][6], b6[kDensUnroll][6];
#pragma unroll
                for (int u = 0; u < kDensUnroll; ++u) {
                    const int ss = __shfl_sync(0xffffffffu, s, src[u] < 0 ? 0 : src[u]);
                    const int sm2 = __shfl_sync(0xffffffffu, sm_, src[u] < 0 ? 0 : src[u]);
                    if (src[u] >= 0) {
                        const T* cm = c_val + ((size_t)m * cap + sm2) * kTileVals + col;
                        const T* cn = c_val + ((size_t)n * cap + ss) * kTileVals + col;
#pragma unroll
                        for (int k = 0; k < 6; ++k) {
                            a6[u][k] = (A)cm[k * kTileW];
                            b6[u][k] = (A)cn[k * kTileW];
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < kDensUnroll; ++u) {
                    if (src[u] < 0) continue;
#pragma unroll
                    for (int k = 0; k < 6; ++k)
#pragma unroll
                        for (int l = 0; l < 6; ++l) acc[k * 6 + l] += a6[u][k] * b6[u][l];
                    if constexpr (kSplit) {
                        if (++since == kDensFlush) {
                            since = 0;
                            flush(acc, n_part++);
                        }
                    }
                }
            }
            if (virt_seen) break;   // tiles are sorted: occupied tiles first
        }
        flush(acc, n_part++);
        __syncwarp();
        if constexpr (!kSplit) {
            // lane u < 36 adds up product u over the 32 lanes (rotated start: no bank conflicts) and
            // weights it by S and H0; then row sums of P o S by the atoms of m, column sums by the atoms
            // of n (AOs: O s, p, p, p, then H1 s, H2 s), and sum P o H0 (in FP64 storage the order of the
            // sums is kept: an SCF that does not settle turns a last bit into another result)
            const bool self = n == m;
            const int er = self ? e : mp_rev[e];
            double qr[3] = {0, 0, 0}, qc[3] = {0, 0, 0}, eb = 0.0;
            for (int u = lane; u < 36; u += 32) {
                const double* row = wsum + u * 32;
                double v = 0.0;
                for (int j = 0; j < 32; ++j) v += row[(j + lane) & 31];
                const double P = 2.0 * v;
                const int k = u / 6, l = u - 6 * k;   // AO of m, AO of n
                if (P_out) {
                    P_out[(size_t)e * 36 + u] = P;
                    if (!self) P_out[(size_t)er * 36 + l * 6 + k] = P;
                }
                const double pq = P * Sb[(size_t)e * 36 + u];
                qr[0] += k < 4 ? pq : 0.0;
                qr[1] += k == 4 ? pq : 0.0;
                qr[2] += k == 5 ? pq : 0.0;
                qc[0] += l < 4 ? pq : 0.0;
                qc[1] += l == 4 ? pq : 0.0;
                qc[2] += l == 5 ? pq : 0.0;
                eb += P * H0b[(size_t)e * 36 + u];
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    qr[i] += __shfl_xor_sync(0xffffffffu, qr[i], off);
                    qc[i] += __shfl_xor_sync(0xffffffffu, qc[i], off);
                }
                eb += __shfl_xor_sync(0xffffffffu, eb, off);
            }
            __syncwarp();
            if (lane == 0) {
                dpart[2 * (size_t)e] = make_double2(qr[0], qr[1]);
                dpart[2 * (size_t)e + 1] = make_double2(qr[2], eb);
                if (!self) {
                    dpart[2 * (size_t)er] = make_double2(qc[0], qc[1]);
                    dpart[2 * (size_t)er + 1] = make_double2(qc[2], eb);
                }
            }
            continue;
        } else {
            double p[2];
            pair_sums((const float2*)wsum, lane, p[0], p[1]);
            {
                unsigned any = 0;
#pragma unroll
                for (int u = 0; u < 18; ++u) any |= *(const unsigned*)&low[u] & 0x7fff7fffu;
                if (__any_sync(0xffffffffu, any != 0)) {   // the third parts, in the same way
                    __syncwarp();
                    float2* f = (float2*)wsum + lane;
#pragma unroll
                    for (int u = 0; u < 36; ++u)
                        f[u * 32] = make_float2(u & 1 ? __high2float(low[u / 2]) : __low2float(low[u / 2]), 0.f);
                    __syncwarp();
                    double l0, l1;
                    pair_sums((const float2*)wsum, lane, l0, l1);
                    p[0] += l0;
                    p[1] += l1;
                }
            }
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) p[1] += __shfl_xor_sync(0xffffffffu, p[1], off);
            __syncwarp();
            // the products weighted by S (36) and by H0 (36) back to shared memory, then four lanes
            // each for the sums of P o S over the atoms of m and of n (AOs: O s, p, p, p, then H1 s,
            // H2 s) and of P o H0
            const bool self = n == m;
            const int er = self ? e : mp_rev[e];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                if (i && (lane & 7)) break;
                const int u = i ? 32 + (lane >> 3) : lane;
                const double P = 2.0 * p[i];
                if (P_out) {
                    P_out[(size_t)e * 36 + u] = P;
                    const int k = u / 6, l = u - 6 * k;   // AO of m, AO of n
                    if (!self) P_out[(size_t)er * 36 + l * 6 + k] = P;
                }
                wsum[u] = P * Sb[(size_t)e * 36 + u];
                wsum[36 + u] = P * H0b[(size_t)e * 36 + u];
            }
            __syncwarp();
            if (lane < 28) {
                const double* w9 = wsum + (sum_id == 6 ? 36 : 0) + 9 * (lane & 3);
                double v = 0.0;
#pragma unroll
                for (int j = 0; j < 9; ++j) v += (take >> j) & 1 ? w9[j] : 0.0;
                v += __shfl_xor_sync(0x0fffffffu, v, 1);
                v += __shfl_xor_sync(0x0fffffffu, v, 2);
                if ((lane & 3) == 0) {
                    double* out = (double*)dpart;   // per entry: atoms O, H1, H2 and the energy
                    if (sum_id < 3 || sum_id == 6) out[4 * (size_t)e + min(sum_id, 3)] = v;
                    if (sum_id >= 3 && !self) out[4 * (size_t)er + sum_id - 3] = v;
                }
            }
            __syncwarp();
        }
    }
}

// q and the band energy of every molecule: its pairs' shares summed in
// neighbour order
__global__ void k_density_sum(int n_mol, const int* __restrict__ mp_ptr, const double2* __restrict__ dpart,
                              double* __restrict__ q, double* __restrict__ e_mol) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= n_mol) return;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    for (int e = mp_ptr[m]; e < mp_ptr[m + 1]; ++e) {
        const double2 a = dpart[2 * (size_t)e], b = dpart[2 * (size_t)e + 1];
        s0 += a.x;
        s1 += a.y;
        s2 += b.x;
        s3 += b.y;
    }
    q[3 * m] = s0;
    q[3 * m + 1] = s1;
    q[3 * m + 2] = s2;
    e_mol[m] = s3;
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static cudaError_t ensure_attrs();

cudaError_t launch_colindex(Ctx* c) {
    cudaError_t ea = ensure_attrs();
    if (ea != cudaSuccess) return ea;
    const int b = c->cur;
    const size_t small = (size_t)c->n_tiles * ((c->n_mol + 31) / 32 + 1) * 4;
    if ((long long)c->n_mol * c->cap <= kCiSmallEntries && small <= kCiSmallSmem) {
        c->n_launch += 1;
        k_ci_small<<<1, 1024, small, c->stream>>>(c->n_mol, c->n_tiles, c->cap, c->d_c_nt[b], c->d_c_tile[b],
                                                  c->d_cci_ptr, c->d_cci_row, c->d_cci_slot);
        return cudaGetLastError();
    }
    c->n_launch += 4;
    cudaMemsetAsync(c->d_cci_cnt, 0, (size_t)c->n_tiles * 4, c->stream);
    k_ci_count<<<c->n_mol, 128, 0, c->stream>>>(c->n_mol, c->cap, c->d_c_nt[b], c->d_c_tile[b], c->d_cci_cnt);
    k_scan<<<1, 1024, 0, c->stream>>>(c->n_tiles, c->d_cci_cnt, c->d_cci_ptr);
    cudaMemsetAsync(c->d_cci_cnt, 0, (size_t)c->n_tiles * 4, c->stream);
    k_ci_fill<<<c->n_mol, 128, 0, c->stream>>>(c->n_mol, c->cap, c->d_c_nt[b], c->d_c_tile[b], c->d_cci_ptr,
                                               c->d_cci_cnt, c->d_cci_row, c->d_cci_slot);
    const size_t ssmem = (size_t)2 * ((c->max_cl_mol + 31) / 32) * 4;
    k_ci_sort<<<c->n_tiles, kSortThreads, ssmem, c->stream>>>(c->d_cci_ptr, c->d_cci_row, c->d_cci_slot,
                                                              c->d_tile_row0, c->max_cl_mol, &c->d_sc->err);
    return cudaGetLastError();
}

static bool g_attr_done[64] = {false};   // per device: function attributes are set per device

template <typename T>
static cudaError_t set_attrs() {
    cudaError_t e;
    e = cudaFuncSetAttribute(k_xc<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_density<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    return e;
}

static cudaError_t ensure_attrs() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64 && g_attr_done[dev]) return cudaSuccess;
    e = cudaFuncSetAttribute(k_ci_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCiSmallSmem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_transform, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_transform_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    e = set_attrs<double>();
    if (e != cudaSuccess) return e;
    e = set_attrs<float>();
    if (e == cudaSuccess && dev >= 0 && dev < 64) g_attr_done[dev] = true;
    return e;
}

cudaError_t launch_xc(Ctx* c, bool use_h, int tile_lo, int tile_hi, int own_below) {
    c->n_launch += 1;
    cudaError_t e = ensure_attrs();
    if (e != cudaSuccess) return e;
    const int b = c->cur;
    const int n = tile_hi - tile_lo;
    if (n <= 0) return cudaSuccess;
    const int nr = c->max_cl_mol;
    const size_t smem = (size_t)((nr + 31) / 32) * 8 + (size_t)nr * 2 + 64;
    if (smem > 200 * 1024) return cudaErrorInvalidValue;
    // CTAs per tile: enough for kXcCtas per SM, but a warp gets four rows unless that leaves the SMs with
    // fewer than eight (each CTA of a tile builds the tile's maps anew)
    const int fill = (8 * c->n_sm + n - 1) / n, most = (kXcCtas * c->n_sm + n - 1) / n;
    const int sh = std::min({8, most, std::max(fill, (nr + 31) / 32)});
    if (c->prec == SSCF_FP64)
        k_xc<double><<<n * sh, 256, smem, c->stream>>>(tile_lo, n, sh, nr, own_below, c->cap, c->capY, c->d_tile_row0, c->d_cci_ptr, c->d_cci_row,
                                                  c->d_cci_slot, (const double*)c->d_c_val[b], c->d_mp_ptr,
                                                  c->d_mp_col, (const double*)(use_h ? c->d_Hb : c->d_Sbt),
                                                  c->d_y_n, c->d_y_row, (double*)c->d_y_val, &c->d_sc->err);
    else
        k_xc<float><<<n * sh, 256, smem, c->stream>>>(tile_lo, n, sh, nr, own_below, c->cap, c->capY, c->d_tile_row0, c->d_cci_ptr, c->d_cci_row,
                                                 c->d_cci_slot, (const float*)c->d_c_val[b], c->d_mp_ptr,
                                                 c->d_mp_col, (const float*)(use_h ? c->d_Hb : c->d_Sbt),
                                                 c->d_y_n, c->d_y_row, (float*)c->d_y_val, &c->d_sc->err);
    return cudaGetLastError();
}

cudaError_t launch_xc_rot(Ctx* c) {
    // the occupied tiles enter the rotation transform only through their
    // diagonal tile pairs C[:, a]^T H C[:, a], whose sum runs over a's rows
    // (one launch for all tiles keeps the CTAs of both kinds in one grid)
    return launch_xc(c, true, 0, c->n_tiles, c->n_occ_tiles);
}

template <typename T>
static cudaError_t transform_t(Ctx* c, const int* ptr, const int* bl, const int* outl, void* out) {
    constexpr bool kFP64 = std::is_same<T, double>::value;
    const int split = transform_split(c);
    const int grid = c->n_tiles * split;
    if constexpr (kFP64) {
        const size_t smem = (size_t)2 * kTfStageVals * sizeof(T) + (size_t)c->max_cl_mol * 2;
        k_transform<<<grid, kTfWarps * 32, smem, c->stream>>>(
            split, c->max_cl_mol, c->d_tile_row0, c->cap, c->capY, ptr, bl, outl, c->d_cci_ptr, c->d_cci_row,
            c->d_cci_slot, (const T*)c->d_c_val[c->cur], c->d_y_n, c->d_y_row, (const T*)c->d_y_val, (T*)out);
    } else {
        const size_t smem = (size_t)kTcWarps * 32 * sizeof(int2) + (size_t)c->max_cl_mol * 2;
        k_transform_tc<<<grid, kTcWarps * 32, smem, c->stream>>>(
            split, c->max_cl_mol, c->d_tile_row0, c->cap, c->capY, ptr, bl, outl, c->d_cci_ptr, c->d_cci_row,
            c->d_cci_slot, (const T*)c->d_c_val[c->cur], c->d_y_n, c->d_y_row, (const T*)c->d_y_val, (T*)out);
    }
    return cudaGetLastError();
}

cudaError_t launch_transform_rot(Ctx* c) {
    c->n_launch += 3;
    cudaError_t e = ensure_attrs();
    if (e != cudaSuccess) return e;
    if ((size_t)2 * kTfStageVals * 8 + (size_t)c->max_cl_mol * 2 > 200 * 1024) return cudaErrorInvalidValue;
    if (c->prec == SSCF_FP64) {
        e = transform_t<double>(c, c->d_rot_tp_ptr, c->d_rot_tp_b, c->d_rot_tp_out, c->d_F);
        if (e == cudaSuccess)
            e = transform_t<double>(c, c->d_diag_tp_ptr, c->d_diag_tp_b, c->d_diag_tp_out, c->d_Fdiag_tiles);
        if (e == cudaSuccess)
            k_extract_diag<double><<<(c->n_tiles * 16 + 255) / 256, 256, 0, c->stream>>>(
                c->n_tiles, c->d_tile_mo0, c->d_tile_nmo, (const double*)c->d_Fdiag_tiles, c->d_Fd);
    } else {
        e = transform_t<float>(c, c->d_rot_tp_ptr, c->d_rot_tp_b, c->d_rot_tp_out, c->d_F);
        if (e == cudaSuccess)
            e = transform_t<float>(c, c->d_diag_tp_ptr, c->d_diag_tp_b, c->d_diag_tp_out, c->d_Fdiag_tiles);
        if (e == cudaSuccess)
            k_extract_diag<float><<<(c->n_tiles * 16 + 255) / 256, 256, 0, c->stream>>>(
                c->n_tiles, c->d_tile_mo0, c->d_tile_nmo, (const float*)c->d_Fdiag_tiles, c->d_Fd);
    }
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t launch_transform_ortho(Ctx* c, int w) {
    c->n_launch += 1;
    cudaError_t e = ensure_attrs();
    if (e != cudaSuccess) return e;
    if (c->prec == SSCF_FP64)
        return transform_t<double>(c, c->d_ort_tp_ptr[w], c->d_ort_tp_b[w], c->d_ort_tp_out[w], c->d_sig);
    return transform_t<float>(c, c->d_ort_tp_ptr[w], c->d_ort_tp_b[w], c->d_ort_tp_out[w], c->d_sig);
}

cudaError_t launch_density(Ctx* c, double* P_out) {
    c->n_launch += 2;
    cudaError_t e = ensure_attrs();
    if (e != cudaSuccess) return e;
    const size_t smem = (size_t)((c->max_cl_otiles + 1) & ~1) * 4 + (size_t)kDensWarps * 36 * 32 * 8;
    if (smem > 200 * 1024) return cudaErrorInvalidValue;
    const int b = c->cur;
    double2* dpart = (double2*)c->d_dens_part;
    if (c->prec == SSCF_FP64)
        k_density<double><<<c->n_mol, kDensWarps * 32, smem, c->stream>>>(
            c->n_occ_tiles, c->max_cl_otiles, c->d_mol_ot0, c->cap, c->d_c_nt[b], c->d_c_tile[b],
            (const double*)c->d_c_val[b], c->d_mp_ptr, c->d_mp_col, c->d_H0b, c->d_Sb, c->d_mp_rev, dpart, P_out);
    else
        k_density<float><<<c->n_mol, kDensWarps * 32, smem, c->stream>>>(
            c->n_occ_tiles, c->max_cl_otiles, c->d_mol_ot0, c->cap, c->d_c_nt[b], c->d_c_tile[b],
            (const float*)c->d_c_val[b], c->d_mp_ptr, c->d_mp_col, c->d_H0b, c->d_Sb, c->d_mp_rev, dpart, P_out);
    k_density_sum<<<(c->n_mol + 127) / 128, 128, 0, c->stream>>>(c->n_mol, c->d_mp_ptr, dpart, c->d_q, c->d_e_mol);
    return cudaGetLastError();
}

}  // namespace sscf
