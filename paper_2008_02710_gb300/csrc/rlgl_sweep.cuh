// The persistent sweep: the moves of a single-chain solve (the loop of
// Alg. 1 with its stop test) in one cooperative kernel, so that a move
// costs three grid barriers (two with the stale threshold) instead of three
// to four kernel launches, their drain and their serial last-block tails.
//
// One block of 1024 threads an SM owns every G-th group of nodes; a move is
//   stats   : the statistics of its nodes' cash; block sums go to one FP64
//             atomic per statistic in the move's slot;
//   barrier ; every block reads the totals and takes the same decisions
//             (stop, re-derivation, theta) from the same numbers;
//   [top-k] : TOPFRAC only: the radix passes of the exact k-th largest |C|,
//             each a count over the block's nodes and a barrier;
//   select  : its green nodes give up their cash and are listed;
//   barrier ; every block reads the move's links and picks push or pull;
//   push    : its own green rows, and a share of the pieces of the longest
//             rows of all blocks, or
//   pull    : its share of the merge-path tiles;
//   barrier ; while it waits, a block does the move's bookkeeping.
// Measured against the same moves with four blocks of 256 threads an SM, a
// frontier compacted across the GPU (a reservation per block, 20 bytes a row
// written and read again, row offsets and dense moved cash for every node)
// and pushed in chunks of 1024 links: R-MAT 20, per-link threshold, a move
// 34.5 -> 31.3 us (select 9.4 + 3.8 wait -> 8.4 + 2.3; push 20.4 -> 20.5, of
// which 2.67 M scattered additions take about 18 however they are issued:
// 23 us as a kernel of their own on the same links); PageRank of an R-MAT
// graph of 500000 nodes 63 -> 48 us; symmetrised R-MAT 24, a move 317 -> 293
// us, and 234 us with what a move touches once a node or link first to leave
// L2 and no degree loaded beside 1/d (select 156 -> 78, push 161 -> 156); 239
// in the order of the nodes (see push_rows).
// With the stale threshold (Control::theta_lag) a move after the first of a
// launch has no stats phase and no first barrier: its select gathers the
// statistics of the cash it reads, and the next move's threshold and
// decisions come from them, taken while the block waits at the last
// barrier.
// The kernel returns when the solve stops (it then ends the graph's loop) or
// when the FP32 cash of the MIXED path must be re-derived in FP64 (the
// graph's re-derivation runs and the loop launches the sweep again).
//
// Co-residency: the kernel is launched cooperatively with at most as many
// blocks as fit on the GPU at once. Every barrier wait is bounded in time;
// a wait that gives up raises an abort flag on which every block leaves,
// and the solve ends with the status ST_BARRIER.
#pragma once
#include <cstddef>

#include "rlgl_kernels.cuh"

namespace rlgl {

// The sweep runs one block of 1024 threads per SM. Against four of 256 a
// grid barrier with four FP64 totals takes 1.4 us instead of 3.0 (measured:
// the arrivals queue on one counter), and the block's warps can share out
// its nodes through shared memory.
constexpr int kSweepThreads = 1024;
constexpr int kSweepWarps = kSweepThreads / 32;
constexpr int ST_BARRIER = 9;

// Per-move accumulators, zero at rest. Three slots rotate: the slot of
// move t is cleared by block 0 during move t + 1, after its first barrier,
// when every block has finished reading it.
// Every group of fields that all blocks update or read at one time sits on
// its own 128-byte line, and so does the barrier: the blocks' atomics on one
// line do not queue behind those on another or behind the barrier's polls,
// and the fields read together after a barrier are pairs in 16 bytes (one
// request per pair, the pairs in parallel).
// (An alignment specifier applies to every declarator of its declaration:
// one field per declaration here.)
struct SweepSlot {
    alignas(128) double a;       // ||C||_1 of the cash
    double pr;                   // sum v^r of the cash
    alignas(128) double msum;    // sum m_i of the moved cash
    double mabs;                 // sum |m_i|
    alignas(128) unsigned long long reserve;  // packed frontier reservation
    unsigned long long tstamp;   // block 0's timer at the end of its stats (or select)
    alignas(128) double s;       // sum C (the all-green sweep)
    unsigned long long chunk_next;  // next pull tile to hand out
    unsigned long long pieces;   // pieces of long green rows
};
static_assert(offsetof(SweepSlot, pr) == offsetof(SweepSlot, a) + 8 && offsetof(SweepSlot, a) % 16 == 0,
              "a, pr: one 16-byte pair");
static_assert(offsetof(SweepSlot, mabs) == offsetof(SweepSlot, msum) + 8 && offsetof(SweepSlot, msum) % 16 == 0,
              "msum, mabs: one 16-byte pair");
static_assert(offsetof(SweepSlot, tstamp) == offsetof(SweepSlot, reserve) + 8 &&
                  offsetof(SweepSlot, reserve) % 16 == 0,
              "reserve, tstamp: one 16-byte pair");

struct alignas(128) GridBar {
    unsigned long long arrived;  // arrivals since the solve began (grid size per barrier)
    unsigned int abort;          // a wait gave up: every block leaves
    unsigned int parity;         // slot of the next move (kept across launches)
    unsigned int tk_pass;        // top-k radix passes made so far (kept across launches)
};

// The two 8-byte fields at p (16-byte aligned), read from L2 in one request.
__device__ __forceinline__ double2 ldcg_pair(const void* p) {
    return __ldcg(reinterpret_cast<const double2*>(p));
}

struct SweepState {
    GridBar bar;
    SweepSlot slot[3];  // in rotation
    // TOPFRAC: the radix passes' digit histograms (zero at rest), three in
    // rotation: pass q adds into q mod 3, every block reads it after the
    // pass's barrier, and block 0 then clears (q + 2) mod 3, which every
    // block read before that barrier and pass q + 2 will fill after the next.
    unsigned int tk_hist[3][kRadixBins];
};

__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Thread 0: the arrival half of a grid barrier. Makes the block's writes
// visible (fence) and adds one to the arrival count (no value returned);
// target grows by the grid size, the count once every block has arrived.
__device__ __forceinline__ void bar_arrive(GridBar* bar, unsigned long long& target) {
    target += gridDim.x;
    __threadfence();
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], 1;" ::"l"(&bar->arrived) : "memory");
}

// Thread 0: the waiting half of a grid barrier. Polls the arrival count
// until it reaches target, at most limit_ns; a wait that runs out raises the
// abort flag, and a raised flag ends every other wait. Returns 0 when the
// sweep must stop.
__device__ __forceinline__ int bar_wait(GridBar* bar, unsigned long long target,
                                        unsigned long long limit_ns) {
    int ok = 1;
    const unsigned long long t0 = globaltimer();
    unsigned int spins = 0;
    while (ld_acquire_u64(&bar->arrived) < target) {
        if ((++spins & 15u) == 0u) {
            if (ld_acquire_u32(&bar->abort)) {
                ok = 0;
                break;
            }
            if (globaltimer() - t0 > limit_ns) {
                atomicExch(&bar->abort, 1u);
                ok = 0;
                break;
            }
        }
        __nanosleep(32);
    }
    return ok;
}

// Grid-wide barrier of a cooperative launch: the count only grows, so no
// block has to reset or release anything. `target` is the block's expected
// arrival count (kept by thread 0). `before` runs in thread 0 between its
// arrival and its wait (off the critical path unless this block arrives
// last), `after` in every lane of warp 0 once the wait is over, before the
// rest of the block goes on (the block meets twice in all). The wait is
// bounded by limit_ns; returns false (in every thread of the block) when the
// sweep must stop. When ts is given, thread 0 stores its arrival and release
// times in ts[0], ts[1].
template <typename F, typename G>
__device__ __forceinline__ bool grid_barrier_with(GridBar* bar, unsigned long long& target,
                                                  unsigned long long limit_ns, unsigned long long* ts,
                                                  F&& before, G&& after) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x < 32) {
        int ok = 1;
        if (threadIdx.x == 0) {
            if (ts) ts[0] = globaltimer();
            bar_arrive(bar, target);
            before();
            ok = bar_wait(bar, target, limit_ns);
            if (ts) ts[1] = globaltimer();
            s_ok = ok;
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        __syncwarp();
        if (ok) after();
    }
    __syncthreads();
    return s_ok != 0;
}

__device__ __forceinline__ bool grid_barrier(GridBar* bar, unsigned long long& target,
                                             unsigned long long limit_ns,
                                             unsigned long long* ts = nullptr) {
    return grid_barrier_with(bar, target, limit_ns, ts, []() {}, []() {});
}

// A green row: its node and the moved cash per weight.
template <typename T>
struct alignas(2 * sizeof(T)) Green {
    int id;
    T m;
};

// A piece of a long green row: links [pos, pos + len), moved cash per weight m.
template <typename T>
struct Piece {
    long long pos;
    int len;
    T m;
};

template <typename T>
struct SweepArgs {
    T* c;
    double* H;
    const double* s;
    const float* sf;
    const long long* row_ptr;
    const T* ideg;
    const unsigned char* masks;
    const int* deg;     // links of each row
    Green<T>* list;     // the sweep's green rows, each block's in its own part
    Piece<T>* pieces;   // pieces of its long green rows
    int n_hubs;  // hub targets of the push, and the only one when there is one
    int hub1;
    const int* rank;  // source order of mt and mt2 (see source_of)
    const int* n_hot;  // length of its hot front
    T* mt;
    T* mt2;      // power sweep: the moved cash of every other move
    T* facc;     // power sweep: sums of rows split across tiles (zero at rest)
    const int* col;
    const float* w;
    const long long* t_ptr;
    const int* t_src;
    const float* t_w;
    const long long* tile_r;
    const long long* tile_e;
    long long ntiles;
    const long long* wtile_r;  // power sweep: merge-path tiles of a warp
    const long long* wtile_e;
    long long nwtiles;
    DevState* st;
    SweepState* sw;
    MoveRecord* log;
    unsigned long long cond_loop;
    unsigned long long cond_refresh;
    int use_cond;
    int n;
    const int* hubs;  // hub table of the push (nullptr: none)
};

// s_i in the cash type: FP32 on the MIXED path, FP64 on the FP64 path.
__device__ __forceinline__ const float* row_scale(const float* sf, const double*, float) { return sf; }
__device__ __forceinline__ const double* row_scale(const float*, const double* s, double) { return s; }

// x^r for the rare exponents r > 2, out of line so that the node loops do
// not carry pow's registers.
template <typename T>
__device__ __noinline__ T pow_r(T x, int r) {
    return pow(x, (T)r);
}

// ------------------------------------------------------- the node passes
//
// A block owns its groups of nodes (OwnNodes) and selects, lists and pushes its
// own green rows; only rows of more than kHubRow links are cut into pieces
// that all blocks share. So a row's entry is written and read on the same SM,
// no space has to be reserved across the GPU, and nothing of a red node is
// read but its cash (and its 1/degree for the per-link test).
//
// What bounds it: on an L2-resident chain the push's scattered additions
// (about 210 G/s over the whole GPU, measured), beyond L2 the bytes of the
// cash, the row offsets and the links; the rest is the instructions spent on
// a node and the latency of a phase.

// Nodes a lane handles per group: node g0 + 32 q + lane for q < kV, so that
// every access of a warp is to consecutive addresses.
template <typename T>
struct NodeVec {
    static constexpr int kV = sizeof(T) == 4 ? 4 : 2;
};

// (double)v without the FP64 pipe, which takes 16 cycles an SM and warp for
// an addition or a conversion: a normal number's exponent and fraction moved
// to their places; zeros, subnormals, infinities and NaN by the conversion.
__device__ __forceinline__ double widen(float v) {
    const unsigned int u = __float_as_uint(v), e = (u >> 23) & 255u;
    if (e == 0u || e == 255u) return (double)v;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }

// v >= th for th >= 0, v = |x|: the FP64 comparison as one of the bit
// patterns (their order is that of the values; NaN compares false).
__device__ __forceinline__ bool at_least(float v, float th) { return v >= th; }
__device__ __forceinline__ bool at_least(double v, double th) {
    const unsigned long long a = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    return a >= (unsigned long long)__double_as_longlong(th) && a <= 0x7ff0000000000000ull;
}

// The out-degree of a node from its 1/d: FP32's 1/d is within 2^-24 of the
// quotient and the reciprocal taken here within 2^-23, so that for d < 2^20
// the result is within 2^-2 of d; beyond (and in FP64, where a division costs
// more than the load) it is loaded. Beyond L2 the load is a sector a green
// node.
__device__ __forceinline__ int degree_of(float idg, const int* deg) {
    float d;
    asm("rcp.approx.f32 %0, %1;" : "=f"(d) : "f"(idg));  // (within 2^-23)
    return idg > 0x1p-20f ? __float2int_rn(d) : __ldg(deg);
}
__device__ __forceinline__ int degree_of(double, const int* deg) { return __ldg(deg); }

// A block's hub targets (see kHubSlots) and their sums of the move.
template <typename T>
struct HotSmem {
    int hub[kHubSlots];
    double hot[kHubSlots];  // zero at rest
    // with a single hub: the threads' sums, zero at rest. (In shared memory:
    // few chains have a hub, and the node loops need their registers. As a
    // pair of FP32 numbers with the roundings carried along, PageRank of
    // 500000 nodes takes as long: 3301 and 3300 us.)
    double one[kSweepThreads];
};

// Rows of kShortRow < links <= kHubRow met by the block's push, left for
// whichever warp is free at the end: a warp with several of them would
// otherwise keep the GPU waiting.
template <typename T>
struct MidRows {
    static constexpr int kCap = 1024;
    long long base[kCap];
    T m[kCap];
    int len[kCap];
};

// The dynamic shared memory of the sweep.
template <typename T>
struct SweepSmem {
    union {
        MidRows<T> mid;
        PullSmem<T> pull[kSweepThreads / kThreads];
        unsigned int hist[kRadixBins];  // TOPFRAC: the block's digit histogram
    };
    HotSmem<T> hot;
    int next_group;  // node group to hand out next within the block
    int n_list;      // green rows listed
    int next_list;   // green row to push next
    int n_mid;       // rows in mid
    int next_mid;
    int next_piece[kSweepWarps];  // piece of a long row that a warp pushes next
};

// What a node pass needs to know of the move.
template <typename T>
struct MoveView {
    const unsigned char* mask;
    unsigned long long* n_pieces;  // the move's count of pieces of long rows
    T th;
    int sched, r;
    bool link;    // statistics of v_i = |C_i| / d_i
    bool acc;     // gather the statistics of the cash
    bool dense;   // write the dense moved cash mt too (the move may pull)
};

// A thread's sums over a pass.
template <typename T>
struct NodeAcc {
    T a, pr, m, ma;
    unsigned long long edges;
};
template <typename T>
constexpr NodeAcc<T> kNoAcc = {T(0), T(0), T(0), T(0), 0ull};

// The additions of kU edges a lane (target j, -1: none; amount v) to the
// cash. Targets in the hub table (PageRank's auxiliary node, which
// every node feeds) are summed apart: one of them by thread, several by warp
// in shared memory.
template <typename T, int kU>
__device__ __forceinline__ void add_edges(T* __restrict__ c, int (&j)[kU], const T (&v)[kU], int n_hubs, int hub1,
                                          HotSmem<T>& hot) {
    if (n_hubs == 0) {
#pragma unroll
        for (int q = 0; q < kU; ++q)
            if (j[q] >= 0) red_add(c + j[q], v[q]);
    } else if (n_hubs == 1) {
#pragma unroll
        for (int q = 0; q < kU; ++q) {
            if (j[q] == hub1) hot.one[threadIdx.x] += (double)v[q];
            else if (j[q] >= 0) red_add(c + j[q], v[q]);
        }
    } else {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int q = 0; q < kU; ++q) {
            int slot = -1;
            if (j[q] >= 0) {
                const int t = hub_slot(j[q]);
                if (hot.hub[t] == j[q]) slot = t;
                else red_add(c + j[q], v[q]);
            }
            unsigned int m = __ballot_sync(0xffffffffu, slot >= 0);
            while (m) {
                const int t = __shfl_sync(0xffffffffu, slot, __ffs(m) - 1);
                const bool mine = slot == t;
                const double x = warp_sum(mine ? (double)v[q] : 0.0);
                if (lane == 0) atomicAdd(&hot.hot[t], x);
                m &= ~__ballot_sync(0xffffffffu, mine);
            }
        }
    }
}

// Pushes the links [pos, pos + len) of one row by the whole warp, four
// links a lane in flight.
template <typename T, bool kHasW, bool kFar>
__device__ __forceinline__ void push_row(const SweepArgs<T>& A, long long pos, int len, T m, HotSmem<T>& hot) {
    const int lane = threadIdx.x & 31;
    const unsigned long long pol = stream_policy();
    for (int o = 0; o < len; o += 128) {
        int j[4];
        T v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = o + q * 32 + lane;
            j[q] = e < len ? ld_run<kFar>(A.col + pos + e, pol) : -1;
            v[q] = m;
            if (kHasW && e < len) v[q] = m * (T)ld_run<kFar>(A.w + pos + e, pol);
        }
        add_edges<T, 4>(A.c, j, v, A.n_hubs, A.hub1, hot);
    }
}

// The block's hub sums of the move into the cash, one addition per hub.
template <typename T>
__device__ __forceinline__ void flush_hubs(const SweepArgs<T>& A, HotSmem<T>& hot) {
    if (A.n_hubs == 1) {
        const double x = warp_sum(hot.one[threadIdx.x]);
        if ((threadIdx.x & 31) == 0 && x != 0.0) atomicAdd(&hot.hot[hub_slot(A.hub1)], x);
        hot.one[threadIdx.x] = 0.0;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < kHubSlots; t += blockDim.x)
        if (hot.hot[t] != 0.0) {
            red_add(A.c + hot.hub[t], (T)hot.hot[t]);
            hot.hot[t] = 0.0;
        }
}

// The nodes of a block: every gridDim.x-th group of consecutive nodes, from
// group blockIdx.x on, so that nodes near one another (the green range of a
// block-round-robin move, a host's pages, the long rows of ids sorted by
// degree) fall to all blocks alike. A group is what a warp takes at a time:
// 128 nodes where every warp gets several of them, down to 32 where they
// would not otherwise all get one.
// Measured against one contiguous span a block, R-MAT 20, 40 moves of eight
// blocks in turn: 3562 -> 1858 us, FP64 3782 -> 1994; ids sorted by degree,
// per-link threshold, 60 moves: 11476 -> 7705 us, FP64 10717 -> 6609; ids at
// random: 2699 -> 2706 us, FP64 3298 -> 3268.
template <typename T>
struct OwnNodes {
    int shift;  // log2 of a group's nodes
    __device__ __forceinline__ explicit OwnNodes(int n) {
        const int mean = (n + (int)gridDim.x - 1) / (int)gridDim.x;  // nodes a block
        shift = mean >= 128 * 2 * kSweepWarps ? 7 : (mean >= 64 * kSweepWarps ? 6 : 5);
        static_assert(NodeVec<T>::kV == 2 || NodeVec<T>::kV == 4, "a group is at most 64 or 128 nodes");
        if (NodeVec<T>::kV == 2 && shift > 6) shift = 6;
    }
    __device__ __forceinline__ int group() const { return 1 << shift; }
    // The first node of the block's group j (n or more: it has no such
    // group). (n < 2^27, and a warp asks for one group beyond the block's last
    // at most: below 2^31)
    __device__ __forceinline__ int first(int j) const { return (j * (int)gridDim.x + (int)blockIdx.x) << shift; }
    // The block's node k, counted over its groups. Only the chain's last
    // group may hold fewer nodes, and it is the last of its block: of a block
    // with m nodes, nodes 0 to m - 1 are in range.
    __device__ __forceinline__ int node(int k) const { return first(k >> shift) + (k & ((1 << shift) - 1)); }
};

// The passes over the nodes. STATS: the statistics of the cash. SELECT: the
// green nodes give up their cash (m_i = C_i, C_i <- 0, H_i += m_i) and are
// listed for the push. ALL: every node does, for a pull (dense moved cash m~
// in mt, no list).
enum Pass : int { PASS_STATS, PASS_SELECT, PASS_ALL };

// With FP32 cash, and for the statistics, warp w of a block takes its groups
// of nodes w, w + 32, ..., so that one cash has one sum, and one threshold
// from it, in every run. (From a counter, as the warps became free, sum v of
// the same cash differed by up to 1e-8 of itself from run to run, and with it
// two or three of symmetrised R-MAT 24's green nodes.) An FP64 selection,
// whose sums differ by 1e-16 whatever their order, takes its groups from a
// counter in shared memory (zero at the start of a pass; warp w starts with
// group w): weighted R-MAT 22, 12 moves, 2788 -> 2766 us. The next group's
// cash is loaded before the current one is listed.
template <typename T, bool kHasW, bool kFar, int kPass>
__device__ __forceinline__ void node_pass(const SweepArgs<T>& A, const MoveView<T>& mv, const SchedAux& ax,
                                          SweepSmem<T>& sm, NodeAcc<T>& acc) {
    constexpr int kV = NodeVec<T>::kV;
    const int lane = threadIdx.x & 31;
    const OwnNodes<T> own(A.n);
    const int n = A.n, group = own.group();
    const bool need_idg = mv.link && (kPass == PASS_STATS || mv.acc || mv.sched == SCHED_LINK);
    const bool scale_is_idg = !kHasW && need_idg;  // unit weights: s_i = 1/d_i
    const T* scale = row_scale(A.sf, A.s, T(0));
    const T th = mv.th;
    T C[kV], idg[kV];
    auto load = [&](int g) {
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            const int i = g + q * 32 + lane;
            C[q] = idg[q] = T(0);
            if (q * 32 < group && i < n) {
                C[q] = __ldcg(A.c + i);
                if (need_idg) idg[q] = kFar ? ld_stream(A.ideg + i, stream_policy()) : __ldg(A.ideg + i);
            }
        }
    };
    int g0 = own.first((int)(threadIdx.x >> 5));
    load(g0);
    while (g0 < n) {
        const int g = g0 + lane;
        if constexpr (kPass == PASS_STATS || sizeof(T) == 4) {
            g0 += (int)gridDim.x * kSweepWarps << own.shift;
        } else {
            int nxt = 0;
            if (lane == 0) nxt = atomicAdd(&sm.next_group, 1);
            g0 = own.first(kSweepWarps + __shfl_sync(0xffffffffu, nxt, 0));
        }
        unsigned int gm = 0u;  // green nodes of this lane
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            const int i = g + q * 32;
            if (q * 32 >= group || i >= n) continue;
            const T av = fabs(C[q]);
            const T tv = mv.link ? av * idg[q] : av;
            if (kPass == PASS_STATS || mv.acc) {
                acc.a += av;
                if (mv.link && mv.r == 1) acc.pr += tv;
                else if (mv.r == 2) acc.pr += tv * tv;
            }
            bool green = kPass == PASS_ALL;
            if (kPass == PASS_SELECT) {
                // (the |C| and |C| / d tests of green_test_v)
                if (mv.sched == SCHED_LINK || mv.sched == SCHED_THRESHOLD || mv.sched == SCHED_TOPFRAC)
                    green = C[q] != T(0) && at_least(tv, th);
                else
                    green = green_test_v<T>(mv.sched, C[q], idg[q], i, th, mv.mask, ax);
            }
            if (green) gm |= 1u << q;
        }
        if (kPass == PASS_STATS) {
            load(g0);
            continue;
        }
        // green rows of the group, by node, and their place in the list
        int k = 0;
        if constexpr (kPass == PASS_SELECT) {
#pragma unroll
            for (int q = 0; q < kV; ++q) {
                k += __popc(__ballot_sync(0xffffffffu, (gm >> q & 1u) != 0u));
            }
            if (lane == 0 && k > 0) k = atomicAdd(&sm.n_list, k);
            k = __shfl_sync(0xffffffffu, k, 0);
        }
        T m[kV];  // moved cash per weight
        int deg[kV];
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            const int i = g + q * 32;
            m[q] = T(0);
            deg[q] = 0;
            if (gm >> q & 1u) {
                m[q] = C[q] * (scale_is_idg ? idg[q] : __ldg(scale + i));
                // (unit weights: see push_rows)
                if (kPass == PASS_SELECT)
                    deg[q] = (kFar ? need_idg : scale_is_idg) ? degree_of(idg[q], A.deg + i) : __ldg(A.deg + i);
            }
        }
#pragma unroll
        for (int q = 0; q < kV; ++q) {
            const int i = g + q * 32;
            if (!(gm >> q & 1u)) continue;
            acc.m += C[q];
            acc.ma += fabs(C[q]);
            A.c[i] = T(0);
            red_add<kFar>(A.H + i, widen(C[q]), stream_policy());  // no load: the L2 adds
        }
        if (kPass == PASS_ALL || mv.dense) {
#pragma unroll
            for (int q = 0; q < kV; ++q)
                if (q * 32 < group && g + q * 32 < n) A.mt[source_of(A.rank, g + q * 32)] = m[q];
        }
        if constexpr (kPass == PASS_ALL) load(g0);
        if constexpr (kPass == PASS_SELECT) {
            int longest = 0;
#pragma unroll
            for (int q = 0; q < kV; ++q) {
                const unsigned int bal = __ballot_sync(0xffffffffu, (gm >> q & 1u) != 0u);
                if (gm >> q & 1u) {
                    Green<T> e;
                    e.id = g + q * 32;
                    e.m = m[q];
                    A.list[own.node(k + __popc(bal & ((1u << lane) - 1u)))] = e;
                }
                k += __popc(bal);
                acc.edges += (unsigned int)deg[q];
                longest = max(longest, deg[q]);
            }
            load(g0);
            if (__any_sync(0xffffffffu, longest > kHubRow)) {
                // long rows: their pieces by the whole warp
#pragma unroll
                for (int q = 0; q < kV; ++q) {
                    unsigned int b = __ballot_sync(0xffffffffu, deg[q] > kHubRow);
                    while (b) {
                        const int l = __ffs(b) - 1;
                        b &= b - 1u;
                        const int len = __shfl_sync(0xffffffffu, deg[q], l);
                        const int np = (len + kHubRow - 1) / kHubRow;
                        long long z = 0;
                        if (lane == 0) z = (long long)atomicAdd(mv.n_pieces, (unsigned long long)np);
                        z = __shfl_sync(0xffffffffu, z, 0);
                        Piece<T> pc;
                        pc.m = __shfl_sync(0xffffffffu, m[q], l);
                        const long long pos = __ldg(A.row_ptr + (g - lane + q * 32 + l));
                        for (int t = lane; t < np; t += 32) {
                            pc.pos = pos + (long long)t * kHubRow;
                            pc.len = min(kHubRow, len - t * kHubRow);
                            A.pieces[z + t] = pc;
                        }
                    }
                }
            }
        }
    }
}

// A thread's share of sum v^r over the block's nodes for r > 2 (ideg: 1/d
// for the per-link v, else NULL), out of line: rare, and a call to pow inside
// the node passes would cost them registers.
template <typename T>
__device__ __noinline__ T pow_sum(const T* c, const T* ideg, int n, int r) {
    T sum = T(0);
    const OwnNodes<T> own(n);
    for (int k = threadIdx.x; own.node(k) < n; k += kSweepThreads) {
        const int i = own.node(k);
        const T av = fabs(__ldcg(c + i));
        sum += (T)pow(ideg ? av * __ldg(ideg + i) : av, (T)r);
    }
    return sum;
}

// The push of the green rows: the GPU's pieces of long rows (warp w takes
// every W-th of them, neighbours on different SMs) and the block's listed
// rows 32 at a time, lane k holding row k: the links of the 32 rows are taken
// together in windows of 32, and lane e finds its row in a window as the
// number of rows that begin at or before it (one warp-wide or and a bit
// count). Four windows are in flight.
// On a chain that fits the L2 the pieces come first and the block's rows of
// more than kShortRow links last, one warp each, so that all warps end
// together (all rows in the order of the list instead: R-MAT 20 2728 -> 3000
// us, PageRank of 500000 nodes 3221 -> 4003).
// Beyond L2, where a warp has many batches, an FP32 chain's rows are pushed
// in the order of the list whatever their length, and the pieces spread over
// it: about the order of the nodes, in which a frontier compacted over the GPU
// was pushed. The order of the additions decides how an FP32 cash is rounded,
// and a chain that mixes slowly stops where ||C||_1 crosses the tolerance:
// symmetrised R-MAT 24 loses 1.6 % of it a move, and long rows first moved it
// by 1e-3, so that 4 of 40 chains stopped one move apart from what they did
// before, in every run. In this order all 40 stop as they did, but for the 3
// that differ from run to run by themselves; 85.2 -> 86.8 ms.
template <typename T, bool kHasW, bool kFar>
__device__ __forceinline__ void push_rows(const SweepArgs<T>& A, SweepSmem<T>& sm, int np) {
    const int lane = threadIdx.x & 31;
    const unsigned int upto = 0xffffffffu >> (31 - lane);
    constexpr bool kInOrder = kFar && sizeof(T) == 4;
    int& next = sm.next_piece[threadIdx.x >> 5];  // (not a register held over the loop)
    if (lane == 0) next = (int)((threadIdx.x >> 5) * gridDim.x + blockIdx.x);
    auto pieces = [&](int end) {
        __syncwarp();
        int p = next;
        __syncwarp();
        for (; p < end; p += (int)gridDim.x * kSweepWarps) {
            // (written by other blocks during this kernel: from L2)
            const long long pos = __ldcg(&A.pieces[p].pos);
            const int len = __ldcg(&A.pieces[p].len);
            const T m = __ldcg(&A.pieces[p].m);
            push_row<T, kHasW, kFar>(A, pos, len, m, sm.hot);
        }
        if (lane == 0) next = p;
    };
    if (!kInOrder) pieces(np);
    const unsigned long long pol = stream_policy();
    const int nl = sm.n_list;
    const OwnNodes<T> own(A.n);
    for (;;) {
        int z = 0;
        if (lane == 0) z = atomicAdd(&sm.next_list, 32);
        z = __shfl_sync(0xffffffffu, z, 0);
        if (kInOrder) pieces(z >= nl ? np : (int)((long long)np * z / nl));
        if (z >= nl) break;
        int len = 0;
        long long base = 0;
        T m = T(0);
        if (z + lane < nl) {
            const Green<T>* e = A.list + own.node(z + lane);
            const int id = __ldcg(&e->id);
            m = __ldcg(&e->m);
            base = __ldg(A.row_ptr + id);
            // (from both offsets where the selection took the degree from
            // 1/d; else the degree is in L1 since)
            len = kFar || (sizeof(T) == 4 && !kHasW) ? (int)(__ldg(A.row_ptr + id + 1) - base) : __ldg(A.deg + id);
            if (len > kHubRow) len = 0;  // in pieces
        }
        const unsigned int mid = __ballot_sync(0xffffffffu, len > kShortRow);
        if (!kInOrder && mid) {
            int k = 0;
            if (lane == 0) k = atomicAdd(&sm.n_mid, __popc(mid));
            k = __shfl_sync(0xffffffffu, k, 0) + __popc(mid & (upto >> 1));
            if (len > kShortRow && k < MidRows<T>::kCap) {
                sm.mid.base[k] = base;
                sm.mid.m[k] = m;
                sm.mid.len[k] = len;
                len = 0;
            }
        }
        int end = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += y;
        }
        const int E = __shfl_sync(0xffffffffu, end, 31);
        const int start = end - len;
        const unsigned int bit = len > 0 ? 1u << (start & 31) : 0u;
        const int win = start >> 5;
        // the rows with links, in order: row r of them is lane rank[r]
        const unsigned int some = __ballot_sync(0xffffffffu, len > 0);
        if (some != 0xffffffffu) {
            // (the last rows, or long ones among them: close the gaps)
            const int src = (int)__fns(some, 0, lane + 1);
            base = __shfl_sync(0xffffffffu, base - start, src & 31);
            m = __shfl_sync(0xffffffffu, m, src & 31);
        } else {
            base -= start;  // base + e: the link of edge e of the 32 rows
        }
        int rows = -1;  // the last row that began before the window
        for (int w0 = 0; w0 * 32 < E; w0 += 4) {
            int j[4];
            T v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                j[q] = -1;
                v[q] = T(0);
                if ((w0 + q) * 32 >= E) continue;
                const unsigned int word = __reduce_or_sync(0xffffffffu, win == w0 + q ? bit : 0u);
                const int k = rows + __popc(word & upto);
                rows += __popc(word);
                const int e = (w0 + q) * 32 + lane;
                const long long pos = __shfl_sync(0xffffffffu, base, k) + e;
                v[q] = __shfl_sync(0xffffffffu, m, k);
                if (e < E) {
                    j[q] = ld_run<kFar>(A.col + pos, pol);
                    if (kHasW) v[q] *= (T)ld_run<kFar>(A.w + pos, pol);
                }
            }
            add_edges<T, 4>(A.c, j, v, A.n_hubs, A.hub1, sm.hot);
        }
    }
    __syncthreads();
    const int nm = min(sm.n_mid, MidRows<T>::kCap);
    for (;;) {
        int z = 0;
        if (lane == 0) z = atomicAdd(&sm.next_mid, 1);
        z = __shfl_sync(0xffffffffu, z, 0);
        if (z >= nm) break;
        push_row<T, kHasW, kFar>(A, sm.mid.base[z], sm.mid.len[z], sm.mid.m[z], sm.hot);
    }
}

// The dense moved cash of a move that pulls though it was not expected to:
// cleared, then set from the block's list (a grid barrier follows: the pull
// reads all of it).
template <typename T>
__device__ __forceinline__ void dense_from_lists(const SweepArgs<T>& A, SweepSmem<T>& sm) {
    const OwnNodes<T> own(A.n);
    for (int k = threadIdx.x; own.node(k) < A.n; k += kSweepThreads) A.mt[source_of(A.rank, own.node(k))] = T(0);
    __syncthreads();
    for (int k = threadIdx.x; k < sm.n_list; k += kSweepThreads) {
        const Green<T>* e = A.list + own.node(k);
        A.mt[source_of(A.rank, __ldcg(&e->id))] = __ldcg(&e->m);
    }
}

// TOPFRAC inside the sweep: one pass of the exact k-th largest |C| by radix
// select over the IEEE bit patterns of |C| (the phase form is k_radix_pass).
// The block counts the digit at `shift` (`width` bits) of the keys that
// match `prefix` above it, over its grid-stride share of the nodes (equal
// digits of a warp merged with __match_any_sync, one shared-memory add per
// distinct digit), and adds its nonzero counts to the pass's histogram.
template <typename T>
__device__ __forceinline__ void sweep_radix_count(const T* c, int n, unsigned int* ghist,
                                                  unsigned long long prefix, int shift, int width, unsigned int* h) {
    const int nbins = 1 << width;
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) h[b] = 0u;
    __syncthreads();
    const int hi_shift = shift + width;
    const unsigned long long mask = (unsigned long long)(nbins - 1);
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long base = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        const long long i = base + lane;
        int digit = -1;
        if (i < n) {
            // the cash other blocks moved last move: from L2
            const unsigned long long k = (unsigned long long)KeyOf<T>::key(__ldcg(c + i));
            const bool match = (hi_shift >= KeyOf<T>::bits) || ((k >> hi_shift) == (prefix >> hi_shift));
            if (match) digit = (int)((k >> shift) & mask);
        }
        const unsigned int peers = __match_any_sync(0xffffffffu, digit);
        if (digit >= 0 && lane == __ffs(peers) - 1) atomicAdd(&h[digit], (unsigned int)__popc(peers));
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nbins; b += blockDim.x)
        if (h[b]) atomicAdd(&ghist[b], h[b]);
}

// After the pass's barrier: the bucket of the remaining k-th largest key,
// the same in every block (the same counts, the same scan). Thread t owns 2
// bins counted from the top; thread 0 gets the new prefix and remainder.
__device__ __forceinline__ void sweep_radix_pick(const unsigned int* ghist, int shift, int width,
                                                 unsigned long long& prefix, long long& remain) {
    __shared__ int found;
    __shared__ long long above_found;
    if (threadIdx.x == 0) found = -1;
    constexpr int per = kRadixBins / kSweepThreads;  // 2
    const int nbins = 1 << width;
    const int top = nbins - 1 - (int)threadIdx.x * per;
    unsigned long long mine = 0;
    unsigned int hb[per];
#pragma unroll
    for (int q = 0; q < per; ++q) {
        const int b = top - q;
        hb[q] = (b >= 0) ? __ldcg(&ghist[b]) : 0u;
        mine += hb[q];
    }
    unsigned long long total;
    const unsigned long long above = block_exscan<kSweepThreads>(mine, &total);
    const long long rem = remain;
    if ((long long)above < rem && (long long)(above + mine) >= rem) {
        long long cum = (long long)above;
#pragma unroll
        for (int q = 0; q < per; ++q) {
            const int b = top - q;
            if (b >= 0 && cum + (long long)hb[q] >= rem) {
                found = b;
                above_found = cum;
                break;
            }
            cum += hb[q];
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int digit = found >= 0 ? found : 0;
        const long long cum = found >= 0 ? above_found : 0;
        prefix |= (unsigned long long)digit << shift;
        remain = rem - cum;
    }
}

// The evolving scalars of the solve, one copy per block in shared memory,
// kept by the block's thread 0. Every block's copy goes through the same
// updates from the same values read after the barriers, so all copies stay
// identical and every block takes the same decisions.
struct SweepCtl {
    long long moves, solve_moves, iters, mask_cursor;
    long long tot_green, tot_edges, push_moves, pull_moves;
    long long green, edges;
    double hsum, habs, theta, l1, sumr, mabs;
    double stall_mark;
    long long stall_count;
    unsigned long long t_start;
    float theta_f;
    int fresh, sched, mode;
    int leave;         // 1: return now (stop, or re-derive before testing again)
    int want_refresh;  // return after this move for a re-derivation
    int p;             // slot of the move
    unsigned long long target;  // expected arrival count at the next barrier
    unsigned long long ts[2][7];  // block 0: move start, then arrival / release at each barrier
    int tb;            // ts of the move (its predecessor's are still to be logged)
    SchedAux ax;       // this move's block-round-robin range and PC constants
    int have_lag;      // stale threshold: a move of this launch has set the statistics
    int stop;          // status to stop with now or after this move (-1: none)
    int owed;          // block 0: the last move's state and log entry are still to be written
    MoveRecord rec;    // block 0: that entry (its times are in ts)
    double limit;      // links from which a move pulls
    int all;           // this move is all-green
    double2 mm, apr;   // this move's totals: sum m, sum |m|; ||C||_1, sum v^r
    unsigned long long rsv;  // its links and green nodes, packed
    long long n_pieces;  // its pieces of long rows
    double mean;       // sum v^r / N of the cash the statistics were taken of
    unsigned long long now;  // block 0's timer when they were taken
    // TOPFRAC: this move's radix select
    unsigned long long tk_prefix;
    long long tk_remain;
    unsigned int tk_pass;  // passes made by the solve so far (histogram rotation)
};

// A move whose predecessor used at least this share of the links from which
// a move pulls writes its dense moved cash while it selects; one that pulls
// without having done so sets it from the lists (two passes more, once: its
// successor is expected to pull).
constexpr double kDenseShare = 0.5;

// x / y and u / v in the time of one FP64 division (0.3 us): the even lanes
// of warp 0 take the first, the odd ones the second. Every lane of warp 0
// calls it; all of them get both.
__device__ __forceinline__ double2 two_ratios(double x, double y, double u, double v) {
    const bool odd = (threadIdx.x & 1u) != 0u;
    const double q = (odd ? u : x) / (odd ? v : y);
    return make_double2(__shfl_sync(0xffffffffu, q, 0), __shfl_sync(0xffffffffu, q, 1));
}

// mean^(1/r) for r >= 2, out of line (rare; pow is large).
__device__ __noinline__ double root_r(double mean, int r) { return pow(mean, 1.0 / r); }

// What thread 0 decides for the next move from the statistics of a cash
// (l1 = ||C||_1, mean = sum v^r / N): its schedule, threshold and schedule
// constants, and how it will be made.
template <typename T>
__device__ __forceinline__ void set_move(SweepCtl& sc, const Control& ctl, MoveView<T>& mv, SweepSmem<T>& sm,
                                         const unsigned char* masks, int n, double l1, double mean) {
    const int r = ctl.r;
    int sched = ctl.sched;
    if (ctl.safety_every > 0 && ((sc.solve_moves + 1) % ctl.safety_every) == 0) sched = SCHED_ALL_GREEN;
    double theta = 0.0;
    if (sched == SCHED_THRESHOLD || sched == SCHED_LINK)
        theta = ctl.theta_arg > 0.0 ? ctl.theta_arg : ctl.theta_scale * (r == 1 ? mean : root_r(mean, r));
    sc.sched = sched;
    sc.theta = theta;
    sc.theta_f = (sched == SCHED_LINK) ? __double2float_rn(theta) : __double2float_ru(theta);
    if (sched == SCHED_BLOCK_RR || sched == SCHED_PC) sc.ax = sched_aux(ctl, n, sc.moves, l1, sched);
    mv.sched = sched;
    mv.th = std::is_same<T, float>::value ? (T)sc.theta_f : (T)sc.theta;
    mv.mask = (sched == SCHED_MASK) ? masks + (sc.mask_cursor % ctl.n_masks) * (long long)n : nullptr;
    mv.acc = ctl.theta_lag && sc.have_lag;
    sc.all = sched == SCHED_ALL_GREEN ? 1 : 0;
    mv.dense = sc.all || (double)sc.edges >= kDenseShare * sc.limit;
    sm.next_group = sm.n_list = sm.next_list = sm.n_mid = sm.next_mid = 0;
}

// Block 0, thread 0: what other kernels and the host read of the last move.
// Written while the block waits at the next barrier or before it returns.
__device__ __forceinline__ void write_owed(SweepCtl& sc, DevState* st, MoveRecord* log) {
    if (!sc.owed) return;
    sc.owed = 0;
    st->theta = sc.rec.theta;
    st->green = sc.rec.green;
    st->edges = sc.rec.edges;
    st->hsum = sc.hsum;
    st->habs = sc.habs;
    st->last_mabs = sc.mabs;
    st->moves = sc.moves;
    st->solve_moves = sc.solve_moves;
    st->tot_green = sc.tot_green;
    st->tot_edges = sc.tot_edges;
    st->push_moves = sc.push_moves;
    st->pull_moves = sc.pull_moves;
    st->fresh = 0;
    st->skip_move = 0;
    st->mask_cursor = sc.mask_cursor;
    st->mode = sc.rec.mode;
    const unsigned long long* ts = sc.ts[sc.tb ^ 1];
    for (int q = 0; q < 6; ++q) sc.rec.phase_us[q] = (float)(ts[q + 1] - ts[q]) * 1e-3f;
    log[sc.rec.move % kLogCap] = sc.rec;
}

__device__ __forceinline__ void clear_slot(SweepSlot* o) {
    o->a = 0.0;
    o->s = 0.0;
    o->pr = 0.0;
    o->msum = 0.0;
    o->mabs = 0.0;
    o->reserve = 0ull;
    o->chunk_next = 0ull;
    o->pieces = 0ull;
}

__device__ __forceinline__ int rot3(int q) { return q == 2 ? 0 : q + 1; }

// Sums of four values a lane over the warp: the total of v[k] ends in lanes
// 8 k to 8 k + 7. Six additions in a row of five steps, where four sums one
// by one take twenty (an FP64 addition holds the SM's FP64 pipe for 16
// cycles). The first two steps are in T, the last three (eight partial sums)
// in R.
template <typename R, typename T>
__device__ __forceinline__ R warp_sum4(const T (&v)[4]) {
    const int lane = threadIdx.x & 31;
    const bool hi = (lane & 16) != 0, hh = (lane & 8) != 0;
    T a = hi ? v[2] : v[0], b = hi ? v[3] : v[1];
    a += __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[2], 16);
    b += __shfl_xor_sync(0xffffffffu, hi ? v[1] : v[3], 16);
    T half = hh ? b : a;
    half += __shfl_xor_sync(0xffffffffu, hh ? a : b, 8);
    R x = half;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// The block's sums of a pass into the move's slot: sum m, sum |m|, ||C||_1,
// sum v^r in the cash type up to four warps, in FP64 beyond, the links and
// green nodes packed (green: the block's count of them, NULL for none); one
// FP64 (or 64-bit) addition per total that is not zero. A grid barrier
// follows every call, so the scratch is free again.
template <typename T>
struct PubSmem {
    T v[4][kSweepWarps];
    unsigned long long r[kSweepWarps];
};
template <typename T>
__device__ __forceinline__ void publish(const NodeAcc<T>& acc, SweepSlot* sl, PubSmem<T>& ps, bool stamp,
                                        const int* green = nullptr) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    {
        const T v[4] = {acc.m, acc.ma, acc.a, acc.pr};
        const T x = warp_sum4<T>(v);
        const unsigned long long r = warp_sum(acc.edges);
        if ((lane & 7) == 0) ps.v[lane >> 3][wid] = x;
        if (lane == 0) ps.r[wid] = r;
    }
    __syncthreads();
    if (wid == 0) {
        const T v[4] = {ps.v[0][lane], ps.v[1][lane], ps.v[2][lane], ps.v[3][lane]};
        const double x = warp_sum4<double>(v);
        double* out = lane < 8 ? &sl->msum : (lane < 16 ? &sl->mabs : (lane < 24 ? &sl->a : &sl->pr));
        if ((lane & 7) == 0 && x != 0.0) atomicAdd(out, x);
        if (lane == 0 && blockIdx.x == 0 && stamp) sl->tstamp = globaltimer();
    } else if (wid == 1) {
        const unsigned long long r = (warp_sum(ps.r[lane]) << kCountBits) + (green ? (unsigned int)*green : 0u);
        if (lane == 0 && r) atomicAdd(&sl->reserve, r);
    }
}

template <typename T, bool kHasW, bool kFar>
__device__ __forceinline__ void sweep_moves(const SweepArgs<T>& A) {
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    if (A.st->done) {
        if (A.use_cond && lead) cudaGraphSetConditional(A.cond_loop, 0u);
        return;
    }
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    SweepSmem<T>& sm = *reinterpret_cast<SweepSmem<T>*>(dyn_smem);
    __shared__ PubSmem<T> ps;
    __shared__ SweepCtl sc;
    __shared__ MoveView<T> mv;
    // The solve's parameters, copied once: after every barrier a global read
    // would go to L2 again.
    __shared__ Control ctl;
    __shared__ double s_l1_refresh;
    __shared__ unsigned long long s_limit_ns;  // the solve's time limit
    {
        const unsigned int* src = reinterpret_cast<const unsigned int*>(&A.st->ctl);
        unsigned int* dst = reinterpret_cast<unsigned int*>(&ctl);
        for (int k = threadIdx.x; k < (int)(sizeof(Control) / 4); k += blockDim.x) dst[k] = src[k];
        for (int k = threadIdx.x; k < kHubSlots; k += blockDim.x) {
            sm.hot.hub[k] = A.n_hubs ? __ldg(A.hubs + k) : -1;
            sm.hot.hot[k] = 0.0;
        }
        sm.hot.one[threadIdx.x] = 0.0;
    }
    __syncthreads();
    const int n = A.n;
    if (threadIdx.x == 0) {
        s_l1_refresh = A.st->l1_refresh;
        // an integer number of ns exceeds the limit when it exceeds its floor
        s_limit_ns = ctl.time_limit_ns < 9e18 ? (unsigned long long)ctl.time_limit_ns : ~0ull;
        sc.moves = A.st->moves;
        sc.solve_moves = A.st->solve_moves;
        sc.iters = A.st->iters;
        sc.mask_cursor = A.st->mask_cursor;
        sc.tot_green = A.st->tot_green;
        sc.tot_edges = A.st->tot_edges;
        sc.push_moves = A.st->push_moves;
        sc.pull_moves = A.st->pull_moves;
        sc.edges = A.st->edges;  // the last move's (0 at the start of a solve)
        sc.hsum = A.st->hsum;
        sc.habs = A.st->habs;
        sc.t_start = A.st->t_start;
        sc.fresh = A.st->fresh;
        sc.stall_mark = A.st->stall_mark;
        sc.stall_count = A.st->stall_count;
        // Every barrier adds exactly the grid size, and no barrier can
        // complete before this block arrives: rounding down what has arrived
        // gives the count at the start of this launch.
        const unsigned long long arr = ld_acquire_u64(&A.sw->bar.arrived);
        sc.target = arr - arr % gridDim.x;
        sc.p = (int)(A.sw->bar.parity % 3u);
        sc.tk_pass = A.sw->bar.tk_pass;
        sc.limit = ctl.pull_crossover * (double)ctl.nnz;
        sc.l1 = sc.sumr = sc.mean = 0.0;
        sc.have_lag = sc.leave = sc.owed = sc.want_refresh = sc.tb = 0;
        sc.stop = -1;
        sc.ts[0][0] = globaltimer();
        mv.mask = nullptr;
        mv.th = T(0);
        mv.sched = ctl.sched;
        mv.r = ctl.r;
        mv.link = ctl.sched == SCHED_LINK;
        mv.acc = mv.dense = false;
        sm.next_group = 0;
    }
    __syncthreads();
    // Test of the bounded wait: the last block leaves without arriving, so
    // the others' first barrier wait runs out.
    if (ctl.test_skip_barrier && blockIdx.x == gridDim.x - 1 && gridDim.x > 1) return;

    auto pow_share = [&]() {
        return pow_sum<T>(A.c, mv.link ? A.ideg : nullptr, n, mv.r);
    };
    // Block 0's duties of the last move, while it waits at a barrier.
    auto owed = [&]() {
        if (blockIdx.x == 0) write_owed(sc, A.st, A.log);
    };
    // The end of a move (thread 0, while its block waits at the move's last
    // barrier): the stop test and the re-derivation triggers of the stale
    // threshold, the solve's totals, and with the stale threshold the next
    // move's decisions.
    auto end_move = [&]() {
        const double l1 = sc.apr.x;
        const double sumr = (ctl.r == 1 && !mv.link) ? l1 : sc.apr.y;
        long long green = (long long)(sc.rsv & ((1ull << kCountBits) - 1ull));
        long long edges = (long long)(sc.rsv >> kCountBits);
        if (sc.all) {
            green = n;
            edges = ctl.nnz;
        }
        if (mv.acc) {
            // this move's cash C_t (gathered by its pass) against H_t 1; the
            // move is made whatever the tests say
            const bool converged = sc.moves >= 1 && l1 / fabs(sc.hsum) < ctl.tol;
            bool want_refresh = false;
            if (converged) {
                if (ctl.mixed && !sc.fresh) want_refresh = true;  // re-derive, then test again
                else sc.stop = ST_OK;
            } else if (ctl.mixed && ((ctl.refresh_factor > 0.0 && l1 < ctl.refresh_factor * s_l1_refresh) ||
                                     cash_stalled(l1, sc.stall_mark, sc.stall_count, ctl.stall_moves))) {
                want_refresh = true;
            }
            sc.want_refresh = want_refresh ? 1 : 0;
            sc.l1 = l1;
            sc.sumr = sumr;
            sc.mean = sumr / (double)n;
        }
        sc.hsum += sc.mm.x;
        sc.habs += sc.mm.y;
        sc.mabs = sc.mm.y;
        sc.moves++;
        sc.solve_moves++;
        sc.tot_green += green;
        sc.tot_edges += edges;
        sc.fresh = 0;
        if (sc.sched == SCHED_MASK) sc.mask_cursor++;
        if (sc.mode == MODE_PUSH) sc.push_moves++;
        if (sc.mode == MODE_PULL) sc.pull_moves++;
        sc.edges = edges;
        if (blockIdx.x == 0) {
            sc.rec.move = sc.moves - 1;
            sc.rec.green = green;
            sc.rec.edges = edges;
            sc.rec.mode = sc.mode;
            sc.rec.pad = 0;
            sc.rec.theta = sc.theta;
            sc.rec.l1 = sc.l1;
            sc.rec.hsum = sc.hsum;
            sc.owed = 1;
        }
        sc.p = rot3(sc.p);
        sm.next_group = 0;
        if (sc.stop >= 0 || sc.want_refresh) {
            sc.leave = 1;
        } else if (ctl.theta_lag) {
            // the tests that need no new statistics; the threshold from the
            // statistics just read
            sc.have_lag = 1;
            sc.iters++;
            const bool degenerate = !(fabs(sc.hsum) > 1e-12 * sc.habs) || sc.habs == 0.0;
            if (degenerate) sc.stop = ST_DEGENERATE;
            else if (sc.solve_moves >= ctl.max_steps) sc.stop = ST_NOCONV;
            else if (sc.now - sc.t_start > s_limit_ns || sc.iters > ctl.max_iters) sc.stop = ST_TIMEOUT;
            sc.leave = sc.stop >= 0 ? 1 : 0;
            set_move<T>(sc, ctl, mv, sm, A.masks, n, sc.l1, sc.mean);
        }
    };

    for (;;) {
        // A move of the stale threshold (after the first of the launch) has
        // no statistics pass and no barrier for it: its threshold comes from
        // the statistics of the cash before the previous move, and it
        // gathers its own cash's for the stop test.
        if (!(ctl.theta_lag && sc.have_lag)) {
            // ------------------------------------------ stats and control
            {
                NodeAcc<T> acc = kNoAcc<T>;
                node_pass<T, kHasW, kFar, PASS_STATS>(A, mv, sc.ax, sm, acc);
                if (mv.r > 2) acc.pr = pow_share();
                publish<T>(acc, &A.sw->slot[sc.p], ps, true);
            }
            auto control = [&]() {
                const SweepSlot* sl = &A.sw->slot[sc.p];
                const double2 apr = ldcg_pair(&sl->a);
                const double2 rts = ldcg_pair(&sl->reserve);
                const double l1 = apr.x;
                const double sumr = (ctl.r == 1 && !mv.link) ? l1 : apr.y;
                const double2 q = two_ratios(l1, fabs(sc.hsum), sumr, (double)n);
                if (threadIdx.x != 0) return;
                // (every block is done with the last move's slot; a launch
                // that ends here has no move that would clear it)
                if (blockIdx.x == 0) clear_slot(&A.sw->slot[rot3(rot3(sc.p))]);
                sc.l1 = l1;
                sc.sumr = sumr;
                sc.mean = q.y;
                sc.now = (unsigned long long)__double_as_longlong(rts.y);
                if (sc.iters == 0) sc.t_start = sc.now;
                sc.iters++;
                bool skip = false, want_refresh = false;
                const bool degenerate = !(fabs(sc.hsum) > 1e-12 * sc.habs) || sc.habs == 0.0;
                const bool converged = sc.moves >= 1 && q.x < ctl.tol;
                if (degenerate) {
                    sc.stop = ST_DEGENERATE;
                } else if (converged) {
                    if (ctl.mixed && !sc.fresh) {
                        want_refresh = true;  // re-derive, then test again
                        skip = true;
                    } else {
                        sc.stop = ST_OK;
                    }
                } else if (sc.solve_moves >= ctl.max_steps) {
                    sc.stop = ST_NOCONV;
                } else if (sc.now - sc.t_start > s_limit_ns || sc.iters > ctl.max_iters) {
                    sc.stop = ST_TIMEOUT;
                }
                if (sc.stop < 0 && !skip && ctl.mixed &&
                    ((ctl.refresh_factor > 0.0 && l1 < ctl.refresh_factor * s_l1_refresh) ||
                     cash_stalled(l1, sc.stall_mark, sc.stall_count, ctl.stall_moves)))
                    want_refresh = true;  // after this move
                sc.want_refresh = want_refresh ? 1 : 0;
                if (sc.stop >= 0 || skip) {
                    sc.leave = skip ? 2 : 1;
                    sc.p = rot3(sc.p);  // this slot holds the statistics
                }
                set_move<T>(sc, ctl, mv, sm, A.masks, n, l1, q.y);
            };
            if (!grid_barrier_with(&A.sw->bar, sc.target, ctl.barrier_limit_ns,
                                   blockIdx.x == 0 ? sc.ts[sc.tb] + 1 : nullptr, owed, control))
                goto aborted;
        }
        if (sc.leave) break;

        // ------------------------------------------------ top-k threshold
        // TOPFRAC: theta = the exact k-th largest |C| (k = ceil(f N)), one
        // radix pass and one grid barrier per digit
        if (sc.sched == SCHED_TOPFRAC) {
            if (threadIdx.x == 0) {
                const double f = (ctl.theta_arg > 0.0 && ctl.theta_arg <= 1.0) ? ctl.theta_arg : ctl.top_frac;
                long long k = (long long)ceil(f * (double)n);
                if (k < 1) k = 1;
                if (k > n) k = n;
                sc.tk_prefix = 0ull;
                sc.tk_remain = k;
            }
            __syncthreads();
            for (int hi = KeyOf<T>::bits; hi > 0; hi -= kRadixBits) {
                const int width = hi >= kRadixBits ? kRadixBits : hi;
                const int shift = hi - width;
                const unsigned int q = sc.tk_pass;
                sweep_radix_count<T>(A.c, n, A.sw->tk_hist[q % 3u], sc.tk_prefix, shift, width, sm.hist);
                if (!grid_barrier(&A.sw->bar, sc.target, ctl.barrier_limit_ns)) goto aborted;
                if (blockIdx.x == 0) {
                    unsigned int* old = A.sw->tk_hist[(q + 2u) % 3u];
                    for (int b = threadIdx.x; b < kRadixBins; b += blockDim.x) old[b] = 0u;
                }
                sweep_radix_pick(A.sw->tk_hist[q % 3u], shift, width, sc.tk_prefix, sc.tk_remain);
                if (threadIdx.x == 0) sc.tk_pass = q + 1u;
                __syncthreads();
            }
            if (threadIdx.x == 0) {
                sc.theta = KeyOf<T>::value(sc.tk_prefix);
                sc.theta_f = __double2float_ru(sc.theta);
                mv.th = std::is_same<T, float>::value ? (T)sc.theta_f : (T)sc.theta;
            }
            __syncthreads();
        }

        // --------------------------------------------------------- select
        {
            if (mv.acc && mv.r > 2) {
                NodeAcc<T> acc = kNoAcc<T>;
                acc.pr = pow_share();
                publish<T>(acc, &A.sw->slot[sc.p], ps, false);
                __syncthreads();  // (the scratch is used again; the selection clears cash)
            }
            if (threadIdx.x == 0) sm.next_group = 0;
            if (threadIdx.x == 0) mv.n_pieces = &A.sw->slot[sc.p].pieces;
            __syncthreads();
            NodeAcc<T> acc = kNoAcc<T>;
            if (sc.all) node_pass<T, kHasW, kFar, PASS_ALL>(A, mv, sc.ax, sm, acc);
            else node_pass<T, kHasW, kFar, PASS_SELECT>(A, mv, sc.ax, sm, acc);
            publish<T>(acc, &A.sw->slot[sc.p], ps, mv.acc, &sm.n_list);
        }
        {
            auto choose = [&]() {
                // every total of the move in one round of loads
                SweepSlot* sl = &A.sw->slot[sc.p];
                const double2 rts = ldcg_pair(&sl->reserve);
                const double2 mm = ldcg_pair(&sl->msum);
                const double2 apr = ldcg_pair(&sl->a);
                const unsigned long long np = __ldcg(&sl->pieces);
                if (threadIdx.x != 0) return;
                const unsigned long long rsv = (unsigned long long)__double_as_longlong(rts.x);
                if (sc.all) sc.mode = MODE_PULL;
                else if ((rsv & ((1ull << kCountBits) - 1ull)) == 0ull) sc.mode = MODE_NONE;
                else sc.mode = (double)(rsv >> kCountBits) >= sc.limit ? MODE_PULL : MODE_PUSH;
                sc.rsv = rsv;
                sc.mm = mm;
                sc.apr = apr;
                sc.n_pieces = (long long)np;
                if (mv.acc) sc.now = (unsigned long long)__double_as_longlong(rts.y);
                // every block is done with the last move's slot
                if (blockIdx.x == 0) clear_slot(&A.sw->slot[rot3(rot3(sc.p))]);
            };
            if (!grid_barrier_with(&A.sw->bar, sc.target, ctl.barrier_limit_ns,
                                   blockIdx.x == 0 ? sc.ts[sc.tb] + 3 : nullptr, owed, choose))
                goto aborted;
        }

        // ----------------------------------------------------------- move
        if (sc.mode == MODE_PUSH) {
            push_rows<T, kHasW, kFar>(A, sm, (int)sc.n_pieces);
            if (A.n_hubs) flush_hubs<T>(A, sm.hot);
        } else if (sc.mode == MODE_PULL) {
            if (!sc.all && !mv.dense) {
                dense_from_lists<T>(A, sm);
                if (!grid_barrier(&A.sw->bar, sc.target, ctl.barrier_limit_ns)) goto aborted;
            }
            // (four groups of 256 threads, each with its own tiles, so that a
            // barrier of one stalls a quarter of the SM. One tile for all
            // 1024: R-MAT 20, every node green, a pull 200 us against 98, FP64
            // 344 against 132; with four blocks of 256 an SM 101 and 140)
            pull_tiles<T, T, kHasW, true, kThreads, kSweepThreads / kThreads>(
                A.c, A.mt, A.t_ptr, A.t_src, A.t_w, A.tile_r, A.tile_e, A.ntiles, 0, 0,
                sm.pull[threadIdx.x / kThreads], &A.sw->slot[sc.p].chunk_next);
        }
        {
            // (the move's times stay until they are logged: the next move
            // has the other set)
            auto times = [&]() {
                if (threadIdx.x != 0 || blockIdx.x != 0) return;
                sc.tb ^= 1;
                sc.ts[sc.tb][0] = sc.ts[sc.tb][1] = sc.ts[sc.tb][2] = sc.ts[sc.tb ^ 1][6];
            };
            if (!grid_barrier_with(&A.sw->bar, sc.target, ctl.barrier_limit_ns,
                                   blockIdx.x == 0 ? sc.ts[sc.tb] + 5 : nullptr, end_move, times))
                goto aborted;
        }
        if (sc.leave) break;
    }
    if (lead) {
        write_owed(sc, A.st, A.log);
        A.st->l1 = sc.l1;
        A.st->sumr = sc.sumr;
        A.st->iters = sc.iters;
        A.st->t_start = sc.t_start;
        A.st->stall_mark = sc.stall_mark;
        A.st->stall_count = sc.stall_count;
        A.sw->bar.parity = (unsigned int)sc.p;
        A.sw->bar.tk_pass = sc.tk_pass;
        if (sc.stop >= 0) {
            A.st->done = 1;
            A.st->status = sc.stop;
            A.st->mode = MODE_NONE;
        } else {
            A.st->want_refresh = 1;
            if (sc.leave == 2) {  // the last test was of a cash to re-derive: no move
                A.st->skip_move = 1;
                A.st->mode = MODE_NONE;
            }
        }
        if (A.use_cond) {
            if (sc.stop >= 0) cudaGraphSetConditional(A.cond_loop, 0u);
            if (ctl.mixed) cudaGraphSetConditional(A.cond_refresh, sc.stop >= 0 ? 0u : 1u);
        }
    }
    return;
aborted:
    // A barrier wait gave up: end the solve with an error status.
    if (threadIdx.x == 0) {
        A.st->done = 1;
        A.st->status = ST_BARRIER;
        if (A.use_cond) {
            cudaGraphSetConditional(A.cond_loop, 0u);
            if (ctl.mixed) cudaGraphSetConditional(A.cond_refresh, 0u);
        }
    }
}

template <typename T, bool kHasW>
__global__ void __launch_bounds__(kSweepThreads, 1) k_sweep(SweepArgs<T> A) {
    sweep_moves<T, kHasW, false>(A);
}

// Chains whose node arrays take most of the L2 (see sweep_kernel).
template <typename T, bool kHasW>
__global__ void __launch_bounds__(kSweepThreads, 1) k_far_sweep(SweepArgs<T> A) {
    sweep_moves<T, kHasW, true>(A);
}

}  // namespace rlgl
