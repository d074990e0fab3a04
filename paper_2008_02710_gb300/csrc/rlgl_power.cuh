// The persistent all-green sweep (power iteration, Sec. 2.3.1): the moves
// of a single-chain all-green solve in one cooperative kernel, one pass over
// the in-links and two grid barriers a move.
//
// With G_t = [N] a move is M_t = C_t, H <- H + C_t, C_{t+1} = M_t P (Eqs.
// recursion_M, recursion_H, recursion_C; every node's cash leaves it). The
// general sweep makes it in three phases (statistics, select, pull) with
// three barriers. Here the select's work is folded into the pull's row
// epilogue: once the in-link sum of row j is complete, one thread reads
// C_t,j, adds it to H_j, stores C_{t+1},j = the sum and the next move's
// moved cash per weight m~_j = C_{t+1},j s_j, and sums the statistics of
// C_{t+1} and of M_t. A move is
//   pull    : merge-path tiles over the in-links, one warp per tile (the
//             warp's lanes meet only at __syncwarp, never at a block-wide
//             barrier), gathering m~ of the current move; the next tile's
//             bounds and in-link sources are loaded while the warp works on
//             the current one. A row that ends in the tile where it began
//             goes through the epilogue with the tile. A row whose in-links
//             cross tile boundaries adds one piece per tile it spans into a
//             zero-at-rest accumulator.
//   barrier
//   split   : each row that crossed a tile boundary (one per tile whose
//             first row ends in it but began in an earlier tile) takes its
//             sum from the accumulator and goes through the epilogue.
//   barrier ; every block takes the same decisions (stop test of Alg. 1,
//             re-derivation triggers) from the same totals.
// Measured on R-MAT 20 and symmetrised R-MAT 22 (all-green to a fixed move
// count; 8.60 ms and 91.9 ms with the pieces counted as they arrived and the
// row finished by its last piece, within the pull, one fence per piece):
// finishing the split rows after a barrier instead, 7.40 / 79.6 ms; loading
// the next tile's bounds and sources ahead, at three blocks an SM (the
// registers it needs), 7.03 / 77.5 ms; warp tiles of 384 rather than 256
// items (FP32), 6.99 / 72.7 ms. Gathering m~ into shared memory with
// cp.async (two tiles ahead, the warp's operands staged in dynamic shared
// memory) was slower than loading it: 10.9 ms on R-MAT 20.
// What bounds a move is the gathers of m~ (a random 4-byte load from L2
// moves a 32-byte sector: 313 G/s over the GPU whatever the array's size, so
// 60 us for R-MAT 20's 18.9 M in-links) and the instructions of the merge.
// Measured then, us a move on R-MAT 20 / symmetrised R-MAT 24:
//   three blocks of 256 threads an SM, no hot sources        105 / 3126
//   one block of 768, the 14336 sources with the most out-links in shared
//   memory (half and a third of the gathers), merge steps without branches,
//   one load of row ends a lane, no merge for tiles inside a row  85 / 2775
//   and the links' loads not kept in L1 and first to leave L2     71 / 2557
//   no register spilled, two sums a node instead of four          71 / 2295
//   tiles from a counter of the block, not of the GPU             71 / 2136
// More hot sources are slower: what shared memory takes is taken from L1,
// which the loads in flight need (36864: 170 / 6690 us with the same merge as
// the first row). A spilled register in the tile loop costs more than a larger
// tile gives: 1024 threads at 64 registers 120 / 3880 us. A load from L2 into
// a register that a shared-memory load also writes waits for it: the hot
// values are read first.
// The moved cash alternates between two buffers (mt and the residual
// source hsrc, free while no re-derivation runs). The per-move totals
// rotate over three slots: the decision of move t reads slot q, move t adds
// into slot q + 1, and slot q + 2 (read one decision ago) is cleared by
// block 0 at the decision; no block can reach slot q + 2 again before
// block 0 has arrived at the next barrier.
// The moves and their floating-point sums are those of the general sweep's
// all-green moves up to the order of the in-link sums: m~ = C s rounded to
// the cash type, in-link sums in the cash type in merge-path order over warp
// tiles (a split row's pieces added in arrival order), H accumulated in
// FP64.
#pragma once

#include "rlgl_sweep.cuh"

namespace rlgl {

constexpr int kWarpsPerBlock = kThreads / 32;
constexpr int kPowerMinBlocks = 3;  // k_rederive_pull: blocks per SM (launch bounds: up to 85 registers a thread)
// The all-green sweep: one block of 768 threads an SM, so that the warps
// share one copy of the hot sources and a thread has 80 registers.
constexpr int kPowThreads = 768;
constexpr int kPowWarps = kPowThreads / 32;

// Merge-path items per lane of a warp tile: 12 for FP32 cash (384-item
// tiles), 8 for FP64 (256-item tiles). A tile's joins and epilogue are FP64
// additions, so that fewer items a tile cost more of them: 6 a lane, R-MAT of
// 1.5 M nodes, 100 moves 14.8 -> 16.9 ms, of 20000 nodes 4.8 -> 5.25 ms.
__host__ __device__ constexpr int power_ipt(int cash_bytes) { return cash_bytes == 4 ? 12 : 8; }

// Shared memory of one warp of the power sweep: its merge-path tile (the
// gathered in-link values, the row ends) and each row's in-link sum (local
// row index). With FP32 cash the bits of a sum take the place of the row's
// end: that is last read before the sum is there (see power_tiles).
template <typename T>
struct PowWarp {
    static constexpr int kItems = 32 * power_ipt((int)sizeof(T));
    T val[kItems];
    int ends[kItems + 1];
    T sums[kItems];
    __device__ __forceinline__ T sum(int k) const { return sums[k]; }
    __device__ __forceinline__ void set_sum(int k, T v) { sums[k] = v; }
};
template <>
struct PowWarp<float> {
    static constexpr int kItems = 32 * power_ipt((int)sizeof(float));
    float val[kItems];
    int ends[kItems + 1];
    __device__ __forceinline__ float sum(int k) const { return __int_as_float(ends[k]); }
    __device__ __forceinline__ void set_sum(int k, float v) { ends[k] = __float_as_int(v); }
};

// Hot sources kept in shared memory, and the block's dynamic shared memory.
__host__ __device__ constexpr int hot_cap(int cash_bytes) { return cash_bytes == 4 ? 14336 : 4096; }
template <typename T>
struct PowSmem {
    alignas(16) T hot[hot_cap((int)sizeof(T))];
    PowWarp<T> warp[kPowWarps];
    int next;  // the block's next tile to hand out
};

// Per-thread sums of a move: ||C_{t+1}||_1, sum C_{t+1} (in the cash type,
// combined per block and then in FP64). Sum M_t and sum |M_t| are the same
// two sums of the move before, for M_t = C_t.
template <typename T>
struct PowAcc {
    T a, s;
};

// Row epilogue of an all-green move: row r's in-link sum v is C_{t+1},r;
// old = C_t,r and sc = s_r.
template <typename T>
__device__ __forceinline__ void power_row_with(const SweepArgs<T>& A, T* __restrict__ mt_next, int r, T v,
                                               T old, T sc, PowAcc<T>& acc) {
    A.c[r] = v;
    mt_next[source_of(A.rank, r)] = v * sc;
    red_add(A.H + r, widen(old));  // M_t,r joins the history (no load: the L2 adds)
    acc.a += fabs(v);
    acc.s += v;
}

template <typename T>
__device__ __forceinline__ void power_row(const SweepArgs<T>& A, T* __restrict__ mt_next, int r, T v,
                                          PowAcc<T>& acc) {
    const T old = __ldcg(A.c + r);  // C_t,r (this kernel stored it one move ago)
    const T sc = __ldg(row_scale(A.sf, A.s, T(0)) + r);
    power_row_with<T>(A, mt_next, r, v, old, sc, acc);
}

// Bounds of tile b: first row, first in-link, rows ending in it, in-links.
struct TileB {
    long long e0;
    int r0, nr, ne;
};

__device__ __forceinline__ TileB tile_bounds(const long long* __restrict__ tile_r,
                                             const long long* __restrict__ tile_e, long long b) {
    TileB t;
    t.r0 = (int)__ldg(tile_r + b);
    t.e0 = __ldg(tile_e + b);
    t.nr = (int)(__ldg(tile_r + b + 1) - t.r0);
    t.ne = (int)(__ldg(tile_e + b + 1) - t.e0);
    return t;
}

// Segmented inclusive scan over the lanes of a warp: the running sum of val
// restarts wherever key changes (keys >= 0 form contiguous runs).
template <typename T, typename K>
__device__ __forceinline__ T warp_segscan(K key, T val) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, val, o);
        const K ky = __shfl_up_sync(0xffffffffu, key, o);
        const bool add = lane >= o && ky == key && key >= 0;
        // (no run reaches this far, nor further; an FP64 addition holds the
        // SM's FP64 pipe for 16 cycles)
        if (sizeof(T) == 8 && !__any_sync(0xffffffffu, add)) break;
        if (add) val += y;
    }
    return val;
}

// The hot front of the moved cash (written by all blocks one move ago: from
// L2) into shared memory; returns its length.
template <typename T>
__device__ __forceinline__ int load_hot(const SweepArgs<T>& A, const T* __restrict__ mt, PowSmem<T>& sm) {
    const int n_hot = A.n_hot ? __ldg(A.n_hot) : 0;
    if (threadIdx.x == 0) sm.next = kPowWarps;  // (every warp's first is its own)
    constexpr int kPer = 16 / (int)sizeof(T);
    const int nv = n_hot / kPer;
    const float4* src = reinterpret_cast<const float4*>(mt);
    float4* dst = reinterpret_cast<float4*>(sm.hot);
    for (int k = threadIdx.x; k < nv; k += 4 * kPowThreads) {
        float4 x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (k + q * kPowThreads < nv) x[q] = __ldcg(src + k + q * kPowThreads);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (k + q * kPowThreads < nv) dst[k + q * kPowThreads] = x[q];
    }
    for (int k = nv * kPer + (int)threadIdx.x; k < n_hot; k += kPowThreads) sm.hot[k] = __ldcg(mt + k);
    __syncthreads();
    return n_hot;
}

// v = *p (from L2) where pred, else unchanged, in place.
__device__ __forceinline__ void ld_over(float& v, const float* p, bool pred) {
    asm volatile("{ .reg .pred q; setp.ne.s32 q, %2, 0; @q ld.global.cg.f32 %0, [%1]; }"
                 : "+f"(v)
                 : "l"(p), "r"((int)pred));
}
__device__ __forceinline__ void ld_over(double& v, const double* p, bool pred) {
    asm volatile("{ .reg .pred q; setp.ne.s32 q, %2, 0; @q ld.global.cg.f64 %0, [%1]; }"
                 : "+d"(v)
                 : "l"(p), "r"((int)pred));
}

// One move's pull with the row epilogue, a warp per merge-path tile: block k
// of G takes the tiles k, k + G, k + 2G, ..., its warps one after another
// from a counter in shared memory (lane 0 asks one turn ahead). Tiles are of
// one size, so that the blocks end together. With the last two rounds handed
// out one at a time from a counter of the whole GPU, which 3648 warps asked:
// symmetrised R-MAT 24, 60 moves, 137.7 ms against 128.1; weighted R-MAT of
// 2 M nodes, 20 moves, 4.06 against 3.89; R-MAT 20 4.32 against 4.34.
// While a warp sums a tile, the next tile's bounds and in-link sources are in
// flight. No block-wide barrier: a warp's lanes meet only at __syncwarp. The
// pieces of rows that cross tile boundaries go into facc.
template <typename T, bool kHasW>
__device__ __forceinline__ void power_tiles(const SweepArgs<T>& A, const T* __restrict__ mt_cur,
                                            PowSmem<T>& sm, int n_hot, PowAcc<T>& acc) {
    constexpr int kPowIpt = power_ipt((int)sizeof(T));
    const int lane = threadIdx.x & 31;
    PowWarp<T>& ws = sm.warp[threadIdx.x >> 5];
    const unsigned long long pol = stream_policy();
    // (tiles: at most 2^38 / 256, an int; rows: below 2^27)
    const int ntiles = (int)A.nwtiles;
    int b = (int)(threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x;
    const T* __restrict__ scale = row_scale(A.sf, A.s, T(0));
    int grab = 0;
    if (lane == 0) grab = atomicAdd(&sm.next, 1);  // for the turn after
    TileB t{0, 0, 0, 0};
    int sidx[kPowIpt];
    if (b < ntiles) t = tile_bounds(A.wtile_r, A.wtile_e, b);
#pragma unroll
    for (int q = 0; q < kPowIpt; ++q) {
        const int k = lane + q * 32;
        sidx[q] = (b < ntiles && k < t.ne) ? ld_stream(A.t_src + t.e0 + k, pol) : -1;
    }
    while (b < ntiles) {
        T oldv = T(0), scv = T(0);
        int start0;
        TileB tn{0, 0, 0, 0};
        int bn;
        {
            // m~ of this move was written by other warps one move ago: L2
            T v[kPowIpt];
#pragma unroll
            for (int q = 0; q < kPowIpt; ++q)
                v[q] = (unsigned int)sidx[q] < (unsigned int)n_hot ? sm.hot[sidx[q]] : T(0);
            // the others over them, where the value is a global load's: the
            // shared loads come first, because a load into a register waits
            // for an earlier one into it, and those are short
#pragma unroll
            for (int q = 0; q < kPowIpt; ++q) ld_over(v[q], mt_cur + sidx[q], sidx[q] >= n_hot);
#pragma unroll
            for (int q = 0; q < kPowIpt; ++q) {
                const int k = lane + q * 32;
                if (kHasW && k < t.ne) asm volatile("prefetch.global.L1 [%0];" ::"l"(A.t_w + t.e0 + k));
            }
            // the next tile's bounds and sources, in flight over this tile
            bn = __shfl_sync(0xffffffffu, grab, 0) * (int)gridDim.x + (int)blockIdx.x;
            if (bn < ntiles && lane == 0) grab = atomicAdd(&sm.next, 1);
            if (bn < ntiles) tn = tile_bounds(A.wtile_r, A.wtile_e, bn);
#pragma unroll
            for (int q = 0; q < kPowIpt; ++q) {
                const int k = lane + q * 32;
                sidx[q] = (bn < ntiles && k < tn.ne) ? ld_stream(A.t_src + tn.e0 + k, pol) : -1;
            }
            if (t.nr == 0) {
                // every item a link of one row that goes on: no merge
                T sum = T(0);
#pragma unroll
                for (int q = 0; q < kPowIpt; ++q) {
                    const int k = lane + q * 32;
                    sum += (kHasW && k < t.ne) ? v[q] * (T)__ldg(A.t_w + t.e0 + k) : v[q];
                }
                sum = warp_sum(sum);
                if (lane == 0) atomicAdd(A.facc + t.r0, sum);
                b = bn;
                t = tn;
                continue;
            }
            // (a tile seldom holds more than 32 rows)
            int re = 0;
            if (lane < t.nr) re = (int)(__ldg(A.t_ptr + t.r0 + 1 + lane) - t.e0);
            start0 = (int)(__ldg(A.t_ptr + t.r0) - t.e0);
            // the epilogue's first row of this lane, read with the gathers
            if (lane < t.nr) {
                oldv = __ldcg(A.c + t.r0 + lane);
                scv = __ldg(scale + t.r0 + lane);
            }
#pragma unroll
            for (int q = 0; q < kPowIpt; ++q) {
                const int k = lane + q * 32;
                if (k < t.ne) ws.val[k] = kHasW ? v[q] * (T)__ldg(A.t_w + t.e0 + k) : v[q];
            }
            if (lane < t.nr) ws.ends[lane] = re;
            for (int k = lane + 32; k < t.nr; k += 32) ws.ends[k] = (int)(__ldg(A.t_ptr + t.r0 + 1 + k) - t.e0);
        }
        if (lane == 0) ws.ends[t.nr] = 0x7fffffff;
        __syncwarp();
        const int total = t.nr + t.ne;
        int d = lane * kPowIpt;
        int rowA = -1, rowB = -1;  // local rows
        T accA = T(0), accB = T(0);
        int i = 0, j = 0, row_start = 0;
        if (d < total) {
            int lo = max(0, d - t.ne), hi = min(d, t.nr);
            while (lo < hi) {
                int mid = (lo + hi) >> 1;
                if (ws.ends[mid] >= d - mid) hi = mid; else lo = mid + 1;
            }
            i = lo;
            j = d - lo;
            row_start = (i == 0) ? start0 : ws.ends[i - 1];
        }
        // From here on a lane reads only the ends of rows of which it holds an
        // item, and writes in this loop only sums of rows that lie in it
        // whole: no other lane holds an item of those. Every other sum is
        // written once all lanes have left the loop.
        __syncwarp();
        if (d < total) {
            bool whole = (j == row_start);  // no in-link of row i before this lane
            T sum = T(0);
            int end = ws.ends[i], j0 = j;   // the row's end; the lane's first in-link of the row
#pragma unroll
            for (int q = 0; q < kPowIpt; ++q) {
                if (d + q < total) {
                    const bool link = j < end;
                    if (link) sum += ws.val[j];
                    if (!link && whole) ws.set_sum(i, sum);  // a row with no in-link sums to zero
                    if (!link && !whole) {
                        rowA = i;
                        accA = sum;
                    }
                    if (!link) {
                        sum = T(0);
                        j0 = j;
                        ++i;
                        // (the next item's row, or past the last of the tile, which none writes)
                        if (q + 1 < kPowIpt) end = ws.ends[i];
                        whole = true;
                    }
                    j += link ? 1 : 0;
                }
            }
            if (j > j0 || !whole) {
                rowB = i;
                accB = sum;
            }
        }
        __syncwarp();
        const T run = warp_segscan<T>(rowB, accB);
        const int pkey = __shfl_up_sync(0xffffffffu, rowB, 1);
        const T pval = __shfl_up_sync(0xffffffffu, run, 1);
        const bool first_split = start0 < 0;  // the tile's first row began in an earlier tile
        if (rowA >= 0) {
            T sum = accA;
            if (lane > 0 && pkey == rowA) sum += pval;
            if (rowA == 0 && first_split)
                atomicAdd(A.facc + t.r0, sum);  // finished after the barrier
            else
                ws.set_sum(rowA, sum);
        }
        const int last = (total - 1) / kPowIpt;
        if (lane == last && rowB >= 0) atomicAdd(A.facc + t.r0 + rowB, run);
        __syncwarp();
        // the rows that end in this tile and began in it (the next move's
        // buffer is taken here: held over the tile it would be a spill)
        T* __restrict__ mt_next = mt_cur == A.mt ? A.mt2 : A.mt;
        for (int k = lane; k < t.nr; k += 32) {
            if (k == 0 && first_split) continue;
            if (k == lane)
                power_row_with<T>(A, mt_next, t.r0 + k, ws.sum(k), oldv, scv, acc);
            else
                power_row<T>(A, mt_next, t.r0 + k, ws.sum(k), acc);
        }
        __syncwarp();  // the warp's shared memory is rewritten next
        b = bn;
        t = tn;
    }
}

// The rows whose in-links cross warp tiles, once every piece is in facc
// (after the move's first grid barrier): the row that ends in tile b began
// in an earlier tile when t_ptr[r0] < e0. Each such row ends in one tile.
template <typename T>
__device__ __forceinline__ void power_split_rows(const SweepArgs<T>& A, T* __restrict__ mt_next, PowAcc<T>& acc) {
    // (32 tiles a warp, neighbouring warps' on different SMs: with a block's
    // warps on neighbouring tiles one SM had all of a small chain's split
    // rows; 50000 nodes, 100 moves, 3.04 -> 2.83 ms, FP64 4.28 -> 4.00)
    for (long long b = ((long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
         b < A.nwtiles; b += (long long)gridDim.x * blockDim.x) {
        const long long r0 = __ldg(A.wtile_r + b);
        if (__ldg(A.wtile_r + b + 1) == r0 || __ldg(A.t_ptr + r0) >= __ldg(A.wtile_e + b)) continue;
        const T v = __ldcg(A.facc + r0);
        A.facc[r0] = T(0);
        power_row<T>(A, mt_next, (int)r0, v, acc);
    }
}

// The FP64 residual pull of a re-derivation (Eq. recursion_H_res), y_j +=
// sum over the in-links e of row j of hsrc[t_src[e]] (* t_w[e]), over the
// same warp tiles as the all-green sweep (kIpt items a lane: the tiles'
// size for the context's cash type) and with the same load order: the next
// tile's bounds and sources are in flight while a warp sums the current
// one. A row's sum goes into y with one reduction where it ends in the tile
// and began in it; a row that crosses a lane or tile boundary adds a piece
// per tile (lanes joined by a segmented scan), so y (zero at rest) holds
// every row's sum once the kernel has ended. Same guard as the block-tile
// pull of kind 1.
template <bool kHasW, int kIpt>
struct RederiveWarp {
    double val[32 * kIpt];
    int end[32 * kIpt + 1];
};

template <bool kHasW, int kIpt>
__global__ void __launch_bounds__(kThreads, kPowerMinBlocks)
    k_rederive_pull(double* __restrict__ y, const double* __restrict__ hsrc, const long long* __restrict__ t_ptr,
                    const int* __restrict__ t_src, const float* __restrict__ t_w,
                    const long long* __restrict__ wtile_r, const long long* __restrict__ wtile_e, long long ntiles,
                    const DevState* st) {
    if (!(st->force_refresh || (st->want_refresh && !st->done))) return;
    __shared__ RederiveWarp<kHasW, kIpt> sm[kWarpsPerBlock];
    RederiveWarp<kHasW, kIpt>& ws = sm[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const unsigned long long pol = stream_policy();
    const long long nw = (long long)gridDim.x * kWarpsPerBlock;
    long long b = (long long)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
    TileB t{0, 0, 0, 0};
    int sidx[kIpt];
    if (b < ntiles) t = tile_bounds(wtile_r, wtile_e, b);
#pragma unroll
    for (int q = 0; q < kIpt; ++q) {
        const int k = lane + q * 32;
        sidx[q] = (b < ntiles && k < t.ne) ? ld_stream(t_src + t.e0 + k, pol) : -1;
    }
    while (b < ntiles) {
        const long long bn = b + nw;
        TileB tn{0, 0, 0, 0};
        int start0;
        {
            double v[kIpt];
#pragma unroll
            for (int q = 0; q < kIpt; ++q) v[q] = (sidx[q] >= 0) ? __ldcg(hsrc + sidx[q]) : 0.0;
            // the next tile's bounds and sources, in flight over this tile
            if (bn < ntiles) tn = tile_bounds(wtile_r, wtile_e, bn);
#pragma unroll
            for (int q = 0; q < kIpt; ++q) {
                const int k = lane + q * 32;
                sidx[q] = (bn < ntiles && k < tn.ne) ? ld_stream(t_src + tn.e0 + k, pol) : -1;
            }
            if (t.nr == 0) {
                // every item a link of one row that goes on: no merge
                double sum = 0.0;
#pragma unroll
                for (int q = 0; q < kIpt; ++q) {
                    const int k = lane + q * 32;
                    sum += (kHasW && k < t.ne) ? v[q] * (double)__ldg(t_w + t.e0 + k) : v[q];
                }
                sum = warp_sum(sum);
                if (lane == 0) red_add(y + t.r0, sum);
                b = bn;
                t = tn;
                continue;
            }
            // (a tile seldom holds more than 32 rows)
            int re = 0;
            if (lane < t.nr) re = (int)(__ldg(t_ptr + t.r0 + 1 + lane) - t.e0);
            start0 = (int)(__ldg(t_ptr + t.r0) - t.e0);
#pragma unroll
            for (int q = 0; q < kIpt; ++q) {
                const int k = lane + q * 32;
                if (k < t.ne) ws.val[k] = kHasW ? v[q] * (double)__ldg(t_w + t.e0 + k) : v[q];
            }
            if (lane < t.nr) ws.end[lane] = re;
            for (int k = lane + 32; k < t.nr; k += 32) ws.end[k] = (int)(__ldg(t_ptr + t.r0 + 1 + k) - t.e0);
        }
        if (lane == 0) ws.end[t.nr] = 0x7fffffff;
        __syncwarp();
        const int total = t.nr + t.ne;
        int d = lane * kIpt;
        long long rowA = -1, rowB = -1;
        double accA = 0.0, accB = 0.0;
        if (d < total) {
            int lo = max(0, d - t.ne), hi = min(d, t.nr);
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (ws.end[mid] >= d - mid) hi = mid; else lo = mid + 1;
            }
            int i = lo, j = d - lo;
            const int row_start = (i == 0) ? start0 : ws.end[i - 1];
            bool whole = (j == row_start);  // no in-link of row i before this lane
            double sum = 0.0;
            int end = ws.end[i], j0 = j;  // the row's end; the lane's first in-link of the row
#pragma unroll
            for (int q = 0; q < kIpt; ++q) {
                if (d + q < total) {
                    const bool link = j < end;
                    if (link) sum += ws.val[j];
                    if (!link && whole && j > j0) red_add(y + (t.r0 + i), sum);
                    if (!link && !whole) {
                        rowA = t.r0 + i;
                        accA = sum;
                    }
                    if (!link) {
                        sum = 0.0;
                        j0 = j;
                        ++i;
                        end = ws.end[i];
                        whole = true;
                    }
                    j += link ? 1 : 0;
                }
            }
            if (j > j0 || !whole) {
                rowB = t.r0 + i;
                accB = sum;
            }
        }
        const double run = warp_segscan<double>(rowB, accB);
        const long long pkey = __shfl_up_sync(0xffffffffu, rowB, 1);
        const double pval = __shfl_up_sync(0xffffffffu, run, 1);
        if (rowA >= 0) red_add(y + rowA, accA + ((lane > 0 && pkey == rowA) ? pval : 0.0));
        const int last = (total - 1) / kIpt;
        if (lane == last && rowB >= 0) red_add(y + rowB, run);
        __syncwarp();  // the warp's shared memory is rewritten next
        b = bn;
        t = tn;
    }
}

// Block sums of the per-thread move sums into the slot: in the cash type up
// to three warps, in FP64 beyond (a block holds 24).
template <typename T>
__device__ __forceinline__ void power_publish(PowAcc<T>& acc, SweepSlot* sl, T (&scratch)[2][kPowWarps]) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const T a = warp_sum(acc.a), s = warp_sum(acc.s);
    if (lane == 0) {
        scratch[0][wid] = a;
        scratch[1][wid] = s;
    }
    __syncthreads();
    if (wid < 2) {
        T v = lane < kPowWarps ? scratch[wid][lane] : T(0);
        v += __shfl_down_sync(0xffffffffu, v, 16);
        v += __shfl_down_sync(0xffffffffu, v, 8);
        double x = v;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0 && x != 0.0) atomicAdd(wid == 0 ? &sl->a : &sl->s, x);
    }
    if (threadIdx.x == 0 && blockIdx.x == 0) sl->tstamp = globaltimer();
    acc.a = acc.s = T(0);
}

template <typename T, bool kHasW>
__global__ void __launch_bounds__(kPowThreads, 1) k_power(SweepArgs<T> A) {
    DevState* st = A.st;
    SweepState* sw = A.sw;
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    if (st->done) {
        if (A.use_cond && lead) cudaGraphSetConditional(A.cond_loop, 0u);
        return;
    }
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    PowSmem<T>& sm = *reinterpret_cast<PowSmem<T>*>(dyn_smem);
    __shared__ T tscratch[2][kPowWarps];
    __shared__ SweepCtl sc;
    __shared__ Control ctl;
    __shared__ double s_l1_refresh;
    {
        const unsigned int* src = reinterpret_cast<const unsigned int*>(&st->ctl);
        unsigned int* dst = reinterpret_cast<unsigned int*>(&ctl);
        for (int k = threadIdx.x; k < (int)(sizeof(Control) / 4); k += blockDim.x) dst[k] = src[k];
        if (threadIdx.x == 0) s_l1_refresh = st->l1_refresh;
    }
    const int n = A.n;
    if (threadIdx.x == 0) {
        sc.moves = st->moves;
        sc.solve_moves = st->solve_moves;
        sc.iters = st->iters;
        sc.tot_green = st->tot_green;
        sc.tot_edges = st->tot_edges;
        sc.push_moves = st->push_moves;
        sc.pull_moves = st->pull_moves;
        sc.hsum = st->hsum;
        sc.habs = st->habs;
        sc.t_start = st->t_start;
        sc.fresh = st->fresh;
        sc.stall_mark = st->stall_mark;
        sc.stall_count = st->stall_count;
        const unsigned long long arr = ld_acquire_u64(&sw->bar.arrived);
        sc.target = arr - arr % gridDim.x;
        sc.p = (int)(sw->bar.parity % 3u);  // the slot the first decision reads (clear)
        sc.want_refresh = 0;
        sc.have_lag = 0;
        sc.mm = make_double2(0.0, 0.0);
    }
    __syncthreads();
    if (ctl.test_skip_barrier && blockIdx.x == gridDim.x - 1 && gridDim.x > 1) return;
    // the moved cash of the current move; the next one's goes to the other
    // of the two buffers
    T* mt_cur = A.mt;
    PowAcc<T> acc{T(0), T(0)};

    // ------------------------------------------------------- prologue
    // m~ = C s for the first move, the split rows' accumulators cleared, and
    // the statistics of the cash for the first stop test.
    {
        const T* scale = row_scale(A.sf, A.s, T(0));
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
             i += (long long)gridDim.x * blockDim.x) {
            const T v = A.c[i];
            A.mt[source_of(A.rank, (int)i)] = v * __ldg(scale + i);
            A.facc[i] = T(0);
            acc.a += fabs(v);
            acc.s += v;
        }
        power_publish<T>(acc, &sw->slot[sc.p], tscratch);
    }
    if (!grid_barrier(&sw->bar, sc.target, ctl.barrier_limit_ns)) goto aborted;

    for (;;) {
        // ------------------------------------------------------ decide
        // (thread 0 of every block, from the same totals)
        if (threadIdx.x == 0) {
            SweepSlot* sl = &sw->slot[sc.p];
            if (blockIdx.x == 0) clear_slot(&sw->slot[rot3(rot3(sc.p))]);  // read one decision ago
            const double2 as = ldcg_pair(&sl->a);         // ||C||_1 (and pr, unused)
            const double2 rts = ldcg_pair(&sl->reserve);  // block 0's timer in .y
            const double sum = __ldcg(&sl->s);
            const double l1 = as.x;
            const unsigned long long now = (unsigned long long)__double_as_longlong(rts.y);
            sc.hsum += sc.mm.x;  // the last move's sum M and sum |M|
            sc.habs += sc.mm.y;
            sc.mm = make_double2(sum, l1);  // and this move's, should it be made
            sc.l1 = l1;
            int stop = -1;
            bool skip = false, want_refresh = false;
            if (sc.want_refresh) {
                // the last move was to be followed by a re-derivation
                skip = true;
                want_refresh = true;
            } else {
                if (sc.iters == 0) sc.t_start = now;
                sc.iters++;
                const bool degenerate = !(fabs(sc.hsum) > 1e-12 * sc.habs) || sc.habs == 0.0;
                const bool converged = sc.moves >= 1 && l1 / fabs(sc.hsum) < ctl.tol;
                if (degenerate) {
                    stop = ST_DEGENERATE;
                } else if (converged) {
                    if (ctl.mixed && !sc.fresh) {
                        want_refresh = true;
                        skip = true;
                    } else {
                        stop = ST_OK;
                    }
                } else if (sc.solve_moves >= ctl.max_steps) {
                    stop = ST_NOCONV;
                } else if ((double)(now - sc.t_start) > ctl.time_limit_ns || sc.iters > ctl.max_iters) {
                    stop = ST_TIMEOUT;
                }
                if (stop < 0 && !skip && ctl.mixed &&
                    ((ctl.refresh_factor > 0.0 && l1 < ctl.refresh_factor * s_l1_refresh) ||
                     cash_stalled(l1, sc.stall_mark, sc.stall_count, ctl.stall_moves)))
                    want_refresh = true;  // after this move
            }
            sc.leave = (stop >= 0 || skip) ? 1 : 0;
            sc.want_refresh = want_refresh ? 1 : 0;
            if (blockIdx.x == 0) {
                st->l1 = l1;
                st->sum = sum;
                st->sumr = l1;
                st->theta = 0.0;
                st->theta_f = 0.0f;
                st->hsum = sc.hsum;
                st->habs = sc.habs;
                st->iters = sc.iters;
                st->t_start = sc.t_start;
                st->stall_mark = sc.stall_mark;
                st->stall_count = sc.stall_count;
                if (sc.have_lag) {
                    // the last move's record: H 1 after it
                    MoveRecord* rec = A.log + ((sc.moves - 1) % kLogCap);
                    rec->hsum = sc.hsum;
                }
                if (sc.leave) {
                    st->mode = MODE_NONE;
                    sw->bar.parity = (unsigned int)rot3(sc.p);  // clear (cleared one decision ago)
                    if (stop >= 0) {
                        st->done = 1;
                        st->status = stop;
                    } else {
                        st->want_refresh = 1;
                        st->skip_move = 1;
                    }
                    if (A.use_cond) {
                        if (stop >= 0) cudaGraphSetConditional(A.cond_loop, 0u);
                        if (ctl.mixed) cudaGraphSetConditional(A.cond_refresh, stop >= 0 ? 0u : 1u);
                    }
                } else {
                    // the move is made: green = every node, every in-link pulled
                    st->green = n;
                    st->edges = ctl.nnz;
                    st->mode = MODE_PULL;
                    st->moves = sc.moves + 1;
                    st->solve_moves = sc.solve_moves + 1;
                    st->tot_green = sc.tot_green + n;
                    st->tot_edges = sc.tot_edges + ctl.nnz;
                    st->pull_moves = sc.pull_moves + 1;
                    st->fresh = 0;
                    st->skip_move = 0;
                    MoveRecord rec;
                    rec.move = sc.moves;
                    rec.green = n;
                    rec.edges = ctl.nnz;
                    rec.mode = MODE_PULL;
                    rec.pad = 0;
                    rec.theta = 0.0;
                    rec.l1 = l1;
                    rec.hsum = sc.hsum;  // completed at the next decision
                    for (int q = 0; q < 6; ++q) rec.phase_us[q] = 0.f;
                    A.log[sc.moves % kLogCap] = rec;
                }
            }
            if (!sc.leave) {
                sc.have_lag = 1;  // (here: a move of this launch has a record to complete)
                sc.moves++;
                sc.solve_moves++;
                sc.tot_green += n;
                sc.tot_edges += ctl.nnz;
                sc.pull_moves++;
                sc.fresh = 0;
            }
        }
        __syncthreads();
        if (sc.leave) return;

        // ----------------------------------------------------------- move
        SweepSlot* nsl = &sw->slot[rot3(sc.p)];  // this move's sums
        if (lead) sc.ts[0][0] = globaltimer();
        const int n_hot = load_hot<T>(A, mt_cur, sm);
        power_tiles<T, kHasW>(A, mt_cur, sm, n_hot, acc);
        if (!grid_barrier(&sw->bar, sc.target, ctl.barrier_limit_ns, blockIdx.x == 0 ? sc.ts[0] + 1 : nullptr))
            break;
        power_split_rows<T>(A, mt_cur == A.mt ? A.mt2 : A.mt, acc);
        power_publish<T>(acc, nsl, tscratch);
        if (!grid_barrier(&sw->bar, sc.target, ctl.barrier_limit_ns, blockIdx.x == 0 ? sc.ts[0] + 3 : nullptr))
            break;
        if (lead) {
            MoveRecord* rec = A.log + ((sc.moves - 1) % kLogCap);
            // the move's work (pull, then the split rows) and the waits at its
            // two barriers (slots 4 and 5)
            rec->phase_us[4] = (float)((sc.ts[0][1] - sc.ts[0][0]) + (sc.ts[0][3] - sc.ts[0][2])) * 1e-3f;
            rec->phase_us[5] = (float)((sc.ts[0][2] - sc.ts[0][1]) + (sc.ts[0][4] - sc.ts[0][3])) * 1e-3f;
        }
        mt_cur = mt_cur == A.mt ? A.mt2 : A.mt;
        if (threadIdx.x == 0) sc.p = rot3(sc.p);
        __syncthreads();
    }
aborted:
    // A barrier wait gave up: end the solve with an error status.
    if (threadIdx.x == 0) {
        st->done = 1;
        st->status = ST_BARRIER;
        if (A.use_cond) {
            cudaGraphSetConditional(A.cond_loop, 0u);
            if (ctl.mixed) cudaGraphSetConditional(A.cond_refresh, 0u);
        }
    }
}

}  // namespace rlgl
