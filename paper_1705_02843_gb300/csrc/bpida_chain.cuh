// The 15-puzzle's Manhattan search for large work: the large steps of calls
// of many boards and of the serving loop (k_search_chain). Short steps run
// k_search's four-move step (bpida_device.cuh): its warps share one stack, so
// that their short runs spread over a warp's lanes sooner.
//
// Nothing here waits on another warp, block or kernel: every loop is bounded
// by the work it consumes.
#pragma once
#include "bpida_device.cuh"

namespace bp {

// Queue records of this search, with M_OPEN set in their metadata: bits
// 24..27 are the moves of the node still to be taken (bit 24 + m: move m);
// the node itself has been counted.
static constexpr uint32_t M_OPEN = 1u << 28;

// ---- the 15-puzzle search step: one child per lane and round ----
// A search lane holds one open node: a node that has been counted and has
// moves left to take. Each round every lane takes the lowest of its node's
// moves, counts and evaluates that child, and goes on with the child if it
// has moves of its own (the node itself, if it has moves left, goes to the
// lane's stack), else with the node's next move, else with the top of its
// stack. So a round builds exactly the nodes that are counted, where building
// all four candidates of a popped node builds four for the one that survives
// on average, and a node whose children are all pruned never reaches a stack.
//
// What bounds it is issue, the integer ALU pipe first. Against k_search's step
// (pop 32 nodes of a stack shared by the warp, build all four candidates of
// each, slots from ballots) on a pass of 2.2e9 nodes: 2.53 warp instructions
// per node instead of 4.29, ALU pipe 74.5 % of its peak, issue slots 71 % busy
// (20 warps per SM: the lanes' stacks fill shared memory). The 100 permutations
// of seeds 1001 to 1100 in one call 158.5 -> 125.4 ms, the 4096-board mix of
// seeds 100000 to 104095 576 -> 437 ms (all steps on k_search / the large ones
// on this kernel, same build). Tried and dropped, on other boards and earlier
// builds of the step: the same nodes on one stack per warp (pops and slots by
// ballot, 196.4 ms against 172.4); idle lanes paired with givers by rank, which
// always robs the lowest lanes (mix 98.4 against 95.5 ms with partners one
// flipped bit away); stacks of 16 entries and more warps (91.9 against 90.7
// ms); runs of up to 128 records (92.2 against 91.2 ms, and coarser time slices
// in the service).
//
// A node is four words: the board in the blank's frame (field j holds the
// tile of cell (p + j) mod 16, p the blank's cell, so that the neighbours up,
// left, right, down sit in fields 12, 15, 1, 4), z and w:
//   z  byte m: 12 + 4a, a the number of cells the blank can still move in
//      the direction of move m (up: its row r, left: its column c, right:
//      3 - c, down: 3 - r). Bit 4 of byte m is set when move m is legal.
//      With x the row or column distance of the tile that move m slides,
//      counted the same way (up: its goal row, left: its goal column, right
//      and down: 3 minus those), the tile slides away from its goal cell iff
//      x < a, i.e. iff bit 4 of 12 + 4a - 4x is set (no byte borrows).
//   w  bits 4, 12, 20, 28: the moves still to take (bit 8m + 4: move m);
//      bits 5..11: slack / 2 (the slack is even: f keeps the parity of
//      h(start) and limits rise by 2); bits 13..17: which record of the run
//      the node descends from.
struct Chain {
    static constexpr uint32_t MOVES = 0x10101010u;
    static constexpr uint32_t HALF_SLACK = 0x7Fu << 5;
    static constexpr int SLACK_SHIFT = 5, SLOT_SHIFT = 13, SLOTS = 32;
    __device__ static __forceinline__ int slot(uint32_t w) { return (int)((w >> SLOT_SHIFT) & (SLOTS - 1u)); }
    static constexpr int BYTES = 64;  // the moves' constants in shared memory
    // Move m turns the board left by k bits (up 16, left 4), and swaps its
    // halves on top (right 32 + 28, down 32 + 16); field 0, now the moved
    // tile t, becomes the blank, and the parent's blank cell, now field 4, 1,
    // 15 or 12, gets t: two multiply-adds, t * y on the low half and t * z on
    // the high half. w: what the blank's move adds to z.
    __device__ static void load(uint4 *t)
    {
        if (threadIdx.x < 4) {
            const int m = threadIdx.x;
            const uint32_t k = m == 1 ? 4u : m == 2 ? 28u : 16u;
            const uint32_t in = 1u << k;
            const uint32_t step = (4u << (8 * (3 - m))) - (4u << (8 * m));
            t[m] = m < 2 ? make_uint4(k, in - 1u, 0u, step) : make_uint4(k, 0u - 1u, in, step);
        }
    }
    // z of the blank at cell p
    __device__ static __forceinline__ uint32_t cells(uint32_t p)
    {
        const uint32_t r = p >> 2, c = p & 3u;
        return 0x0C0C0C0Cu + 4u * (r | (c << 8) | ((3u - c) << 16) | ((3u - r) << 24));
    }
    // the blank's cell
    __device__ static __forceinline__ uint32_t cell(uint32_t z)
    {
        return ((z & 255u) - 12u) + ((((z >> 8) & 255u) - 12u) >> 2);
    }
    // 4x in byte m
    __device__ static __forceinline__ uint32_t distance(uint32_t lo, uint32_t hi)
    {
        const uint32_t g = __byte_perm(lo, hi, 0x2076);
        return (g & 0x0C00000Cu) ^ (((g >> 2) & 0x000C0C00u) ^ 0x0C0C0000u);
    }
    // 12 + 4a - 4x in byte m: bit 4 set when move m's tile slides away from its goal cell
    __device__ static __forceinline__ uint32_t away(uint32_t lo, uint32_t hi, uint32_t z)
    {
        return z - distance(lo, hi);
    }
    __device__ static __forceinline__ uint64_t turn_left(uint64_t b, uint32_t k)
    {
        return k ? (b << k) | (b >> (64u - k)) : b;
    }
    // the four moves of a record (bits 24..27 of its metadata) and back
    __device__ static __forceinline__ uint32_t moves_from_rec(uint32_t m)
    {
        return ((m >> 20) & 0x10u) | ((m >> 13) & 0x1000u) | ((m >> 6) & 0x100000u) | ((m << 1) & 0x10000000u);
    }
    __device__ static __forceinline__ uint32_t moves_to_rec(uint32_t w)
    {
        return ((w << 20) & (1u << 24)) | ((w << 13) & (1u << 25)) | ((w << 6) & (1u << 26)) | ((w >> 1) & (1u << 27));
    }
};
// The lanes' stacks of open nodes {board lo, board hi, z, w} in shared memory:
// lane l owns column l of a warp's rows of 32 entries (a row is ROW bytes: the
// eight lanes of a quarter warp hit distinct banks at any mix of depths), so
// a push or a pop is one predicated access without a vote or a slot prefix.
// Row 0 holds what an empty stack pops, a node whose moves and child have no
// moves (z + the first move's step is 0), so an idle lane needs no test.
struct ChainStack {
    static constexpr uint32_t ROW = 512;
    static constexpr int ROUNDS = 4;  // rounds between two looks at the other lanes
    static constexpr int LOAD = 8;    // idle lanes that take the run's next records
    static constexpr uint32_t IDLE_Z = 4u - (4u << 24);  // less the first move's step
    static constexpr int SPILL = 4;   // entries a full lane moves to the overflow stack (>= ROUNDS)
    // bytes per warp for cap entries per lane
    __host__ __device__ static constexpr size_t bytes(int cap) { return (size_t)(cap + 1) * ROW; }
    __device__ static __forceinline__ void put_if(uint32_t p, uint32_t at, uint32_t lo, uint32_t hi, uint32_t z, uint32_t w)
    {
        asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q st.shared.v4.u32 [%1], {%2, %3, %4, %5}; }"
                     :: "r"(p), "r"(at), "r"(lo), "r"(hi), "r"(z), "r"(w) : "memory");
    }
    // the node keeps its value when p is nonzero
    __device__ static __forceinline__ void get_unless(uint32_t p, uint32_t at, uint32_t &lo, uint32_t &hi, uint32_t &z,
                                                      uint32_t &w)
    {
        asm volatile("{ .reg .pred q; setp.eq.u32 q, %5, 0; @q ld.shared.v4.u32 {%0, %1, %2, %3}, [%4]; }"
                     : "+r"(lo), "+r"(hi), "+r"(z), "+r"(w) : "r"(at), "r"(p) : "memory");
    }
    // A lane's next node {lo, hi, z, w}: the child {clo, chi, cz, cw} if it has
    // moves (the node, {lo, hi, z, rem}, goes to the stack if it has moves left,
    // more), else the node, else the top of the stack (empty: row 0). one is 1
    // in a register: the selects and sums then run on the multiply-add pipe.
    __device__ static __forceinline__ void next(uint32_t &lo, uint32_t &hi, uint32_t &z, uint32_t &w, uint32_t &sp,
                                                uint32_t clo, uint32_t chi, uint32_t cz, uint32_t cw, uint32_t moves,
                                                uint32_t rem, uint32_t more, uint32_t sp0, uint32_t one)
    {
        asm volatile("{ .reg .pred alive, push, pop; .reg .u32 any;\n\t"
                     "setp.ne.u32 alive, %6, 0;\n\t"
                     "setp.ne.and.u32 push, %7, 0, alive;\n\t"
                     "@push st.shared.v4.u32 [%4], {%0, %1, %2, %5};\n\t"
                     "mov.u32 %3, %5;\n\t"
                     "@alive mad.lo.u32 %0, %8, %12, 0;\n\t"
                     "@alive mad.lo.u32 %1, %9, %12, 0;\n\t"
                     "@alive mad.lo.u32 %2, %10, %12, 0;\n\t"
                     "@alive mov.u32 %3, %11;\n\t"
                     "or.b32 any, %6, %7;\n\t"
                     "setp.eq.u32 pop, any, 0;\n\t"
                     "@pop ld.shared.v4.u32 {%0, %1, %2, %3}, [%4+-512];\n\t"
                     "@push mad.lo.u32 %4, %12, 512, %4;\n\t"
                     "@pop mad.lo.u32 %4, %12, -512, %4;\n\t"
                     "max.u32 %4, %4, %13;\n\t"
                     "}"
                     : "+r"(lo), "+r"(hi), "+r"(z), "=&r"(w), "+r"(sp)
                     : "r"(rem), "r"(moves), "r"(more), "r"(clo), "r"(chi), "r"(cz), "r"(cw), "r"(one), "r"(sp0)
                     : "memory");
    }
    __device__ static __forceinline__ void copy(uint32_t to, uint32_t from)
    {
        uint32_t x = 0, y = 0, z = 0, w = 0;
        get_unless(0u, from, x, y, z, w);
        put_if(1u, to, x, y, z, w);
    }
};
// Entries of all warps' overflow stacks in global memory, which take the room of
// CHAIN_OVERFLOW_RECS records of each of the two hand-back queues (so that a
// workspace is no larger than one without them). At five 4-warp blocks on 152
// SMs a warp has 4139 entries, and the largest hand-back of a batch with a board
// of more than 1e11 nodes is 4.7 million records, of queues that hold 12.6
// million at least (6.1 million with 3072 entries, 8.5 with 2048, 15.0 with
// 1024, 23.5 with 512; the time is the same from 1024 up).
static constexpr int CHAIN_OVERFLOW_RECS = 1 << 22, CHAIN_OVERFLOW = 3 << 22;
static_assert(sizeof(uint4) * CHAIN_OVERFLOW == 2 * sizeof(Rec<4>) * CHAIN_OVERFLOW_RECS, "overflow stacks take records' room");

// A step searches with this kernel when it is predicted to expand at least
// CHAIN_MIN_NODES nodes (k_advance's sum over the step's instances, eight
// times their last iterations), else with k_search: this one is the faster
// one where the search itself is the time, and the slower one on short
// searches, whose time is how soon a record spreads over a warp's lanes. Both
// sides measured, k_search in every step / this kernel in all but the first /
// the rule: 512 40-move walks 2443 / 2787 / 2443 us, 64 50-to-60-move walks 2559 /
// 2893 / 2562 us, 700 of them 12.52 / 12.02 / 11.84 ms, 300 boards with 1 %
// permutations 13.07 / 12.54 / 12.36 ms, 100 permutations 430.9 / 327.9 /
// 327.7 ms; the service, 1000 30-to-50-move walks at once 8.54 / 8.93 / 8.48
// ms. The line is flat from 1e8 (walks of 40 moves, 4096 at once: 6.31 ms
// against 6.06) to 1e9 (the 700 walks: 12.13 ms).
static constexpr unsigned long long CHAIN_MIN_NODES = 300000000ull;

// Chain step: the records a warp works on, consecutive records of one
// instance in the pass's input: src[i] is record i.
template <int W> struct ChainRun {
    const Rec<W> *src;
    bool front;   // frontier records (a record's origin is its index)
    int first;    // record of slot 0
    unsigned inst;
    __device__ __forceinline__ uint32_t origin(uint32_t w) const
    {
        const int i = first + Chain::slot(w);
        return front ? (uint32_t)i : src[i].origin;
    }
};

// Chain step: an open node as a queue record.
template <int W>
__device__ __forceinline__ Rec<W> chain_rec(uint32_t lo, uint32_t hi, uint32_t z, uint32_t w, const ChainRun<W> &run)
{
    const uint32_t p = Chain::cell(z);
    Rec<W> r;
    r.b = (typename Geo<W>::B)Chain::turn_left(((uint64_t)hi << 32) | lo, 4u * p);
    r.meta = m_make(p, LAST_NONE, 2u * ((w & Chain::HALF_SLACK) >> Chain::SLACK_SHIFT)) | M_OPEN | Chain::moves_to_rec(w);
    r.inst = run.inst;
    r.origin = run.origin(w);
    r.pm = 0;
    return r;
}

// Chain step: hands back the top k entries of this lane's stack (k >= 0, its
// own for every lane) and, with held set, the node that the lane holds. Every
// lane of the warp calls it.
// (A call, like chain_goal: inlined, these paths spread the search loop over
// more instruction cache lines than it has.)
template <int W>
__device__ __noinline__ void chain_hand_back(Ctrl *ctrl, int Q, Rec<W> *out, int k, uint32_t sp, bool held, uint32_t lo,
                                             uint32_t hi, uint32_t z, uint32_t w, ChainRun<W> run)
{
    const int lane = threadIdx.x & 31;
    const int mine = k + (held ? 1 : 0);
    int x = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(FULL, x, d);
        if (lane >= d)
            x += y;
    }
    const int n = __shfl_sync(FULL, x, 31);
    if (n == 0)
        return;
    int base = 0;
    if (lane == 31)
        base = atomicAdd(&ctrl->out_count, n);
    base = __shfl_sync(FULL, base, 31);
    if (base + n > Q) {
        if (lane == 0)
            atomicOr(&ctrl->err, ERR_QUEUE);
        return;
    }
    base += x - mine;
    if (held)
        out[base++] = chain_rec<W>(lo, hi, z, w, run);
    for (int j = 1; j <= k; ++j) {
        uint32_t el, eh, ez, ew;
        el = eh = ez = ew = 0;
        ChainStack::get_unless(0u, sp - ChainStack::ROW * (uint32_t)j, el, eh, ez, ew);
        out[base++] = chain_rec<W>(el, eh, ez, ew, run);
    }
    __syncwarp();
}

// A goal that a lane counted, o its origin; aborted: null, or where
// first-solution mode stops the instance.
static __device__ __noinline__ void chain_goal(unsigned long long *goals, unsigned *origin, unsigned *aborted, uint32_t o)
{
    atomicAdd(goals, 1ull);
    atomicMin(origin, o);
    if (aborted)
        atomicOr(aborted, ABORT_FOUND);
}

// One warp works on a run of up to 32 records of one instance at a time; runs
// come from the pass's atomic queue, and once enough warps have run dry busy
// ones hand their open nodes to the next pass, as in k_search. REGS: registers
// per thread, 96 where the block size allows it (the unrolled rounds took 5 %
// longer with 64), 64 for blocks of more than CHAIN_WARPS warps.
static constexpr int CHAIN_WARPS = 16;
template <int REGS = 96>
__global__ void __maxnreg__(REGS) k_search_chain(const Dev<4> a)
{
    constexpr int W = 4;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_warps_done;
    __shared__ unsigned long long s_t_end, s_nodes;
    // 1 and -1, read from shared memory so that they stay multiplier operands
    // (sums then run on the multiply-add pipe, not on the integer ALU pipe,
    // which the logic of the step keeps busy)
    __shared__ uint32_t s_unit[2];
    if (threadIdx.x == 0) {
        atomicMin(&a.ctrl->t_start, global_ns());
        s_warps_done = 0;
        s_t_end = 0;
        s_nodes = 0;
        s_unit[0] = 1u;
        s_unit[1] = 0u - 1u;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the moves' constants, this lane's first stack entry, and the stack
    // pointer up to which ROUNDS more pushes fit
    Chain::load((uint4 *)smem);
    const uint32_t ctab = (uint32_t)__cvta_generic_to_shared(smem);
    const uint32_t sp0 = ctab + Chain::BYTES + (uint32_t)warp * (uint32_t)ChainStack::bytes(a.chain_cap) + ChainStack::ROW +
                         16u * (uint32_t)lane;
    const uint32_t sp_full = sp0 + ChainStack::ROW * (uint32_t)(a.chain_cap - ChainStack::ROUNDS);
    ChainStack::put_if(1u, sp0 - ChainStack::ROW, 0u, 0u, ChainStack::IDLE_Z, 0u);
    __syncthreads();
    const uint32_t one = *(volatile uint32_t *)&s_unit[0], neg1 = *(volatile uint32_t *)&s_unit[1];
    const Rec<W> *in = a.ctrl->qi ? a.q1 : a.q0;
    Rec<W> *out = a.ctrl->qi ? a.q0 : a.q1;
    const bool frontier = a.ctrl->first_pass != 0;
    const int n_act = a.ctrl->n_active;
    const int n_front = a.ctrl->n_front;
    const unsigned *act = a.ctrl->cur ? a.act1 : a.act0;
    const bool first_only = a.desc->first_only != 0;
    // this warp's overflow stack in global memory
    uint4 *covf = (uint4 *)a.ovf + ((size_t)blockIdx.x * (blockDim.x >> 5) + warp) * (size_t)a.ovf_cap;
    int ovf_n = 0;
    const unsigned lt = (1u << lane) - 1u;
    const uint64_t GOAL = goal_board<W>();
    const uint32_t GLO = (uint32_t)GOAL, GHI = (uint32_t)(GOAL >> 32);
    const int n_in = a.ctrl->n_in;
    const int total_warps = gridDim.x * (blockDim.x >> 5);
    const int chunk = max(1, min(Chain::SLOTS, n_in / (total_warps * 4)));
    int rounds = 0;
    bool stop = false;
    // counters of the runs' instance (see k_search)
    unsigned acc_inst = 0xffffffffu;
    unsigned long long acc_nodes = 0, tot_nodes = 0;
    uint32_t prn = 0;  // nonzero once a child was pruned: slack is even, so its f = limit + 2
    auto publish = [&]() {
        const bool pruned = __any_sync(FULL, prn != 0u);
        prn = 0;
        if (lane == 0 && acc_inst != 0xffffffffu) {
            if (acc_nodes)
                atomicAdd(&a.cnt.search_nodes[acc_inst], acc_nodes);
            if (pruned)
                atomicMin(&a.cnt.fnext_off[acc_inst], 2);
        }
        acc_nodes = 0;
    };
    // Every 32 rounds: 0 go on; DROP the instance is over its budget or has
    // its first solution (its work is dropped); STOP the pass hands back.
    enum { GO_ON = 0, DROP = 1, STOP = 2 };
    auto check = [&](unsigned inst0, bool budgeted, unsigned long long left, unsigned long long nodes,
                     unsigned long long &flushed) -> int {
        if (first_only) {
            int found = 0;
            if (lane == 0)
                found = (*(volatile unsigned *)&a.cnt.aborted[inst0] & ABORT_FOUND) != 0;
            if (__shfl_sync(FULL, found, 0))
                return DROP;
        }
        if (budgeted) {
            // publish this run's count; past the budget the
            // instance's remaining work is dropped
            int over = 0;
            if (lane == 0) {
                const unsigned long long before = atomicAdd(&a.cnt.search_nodes[inst0], nodes - flushed);
                over = before + (nodes - flushed) > left;
                if (over)
                    atomicOr(&a.cnt.aborted[inst0], ABORT_BUDGET);
            }
            flushed = nodes;
            if (__shfl_sync(FULL, over, 0))
                return DROP;
        }
        if (rounds >= a.tune.min_rounds) {
            // hand back once enough warps have run dry and the
            // pass has run long enough to pay for another one
            int go = 0;
            if (lane == 0 && *(volatile int *)&a.ctrl->exited >= a.tune.exit_threshold)
                go = global_ns() - *(volatile unsigned long long *)&a.ctrl->t_start >=
                     (unsigned long long)a.tune.min_pass_ns;
            // serving: the step's time slice is over
            if (lane == 0 && !go && slice_over(a))
                go = 1;
            if (__shfl_sync(FULL, go, 0))
                return STOP;
        }
        return GO_ON;
    };
    ChainRun<W> run;
    for (;;) {
        int h = 0;
        if (lane == 0)
            h = atomicAdd(&a.ctrl->head, chunk);
        h = __shfl_sync(FULL, h, 0);
        if (h >= n_in)
            break;
        const int end = min(h + chunk, n_in);
        int i = h;
        while (i < end) {
            // the run: records [i, stop_at) at most, all of one instance
            int stop_at = end;
            if (frontier && i < n_front) {
                int k0 = 0, k1 = n_act - 1;  // last problem with offset <= i
                while (k0 < k1) {
                    const int mid = (k0 + k1 + 1) >> 1;
                    if (a.offset[mid] <= i)
                        k0 = mid;
                    else
                        k1 = mid - 1;
                }
                run.front = true;
                run.src = a.scratch + region_of(a, k0, act[k0]) - a.offset[k0];
                run.inst = act[k0];
                stop_at = min(end, a.offset[k0] + a.count[k0]);
            } else {
                run.front = false;
                run.src = frontier ? in - n_front : in;
                run.inst = run.src[i].inst;
            }
            run.first = i;
            const unsigned inst0 = run.inst;
            // an instance whose node budget ran out, or that already found
            // its goal in first-solution mode, is dropped
            const unsigned long long left = a.cnt.budget_left[inst0];
            const bool budgeted = left != ~0ull;
            const bool dropped = (budgeted || first_only) &&
                                 __shfl_sync(FULL, *(volatile unsigned *)&a.cnt.aborted[inst0], 0) != 0u;
            if (inst0 != acc_inst) {
                publish();
                acc_inst = inst0;
            }
            __syncwarp();
            unsigned long long nodes = 0, flushed = 0;
            unsigned n32 = 0;  // this lane's nodes, in bits 8 and up
            // the node this lane holds and its stack pointer; vp is the entry
            // that it gives away next; a partner is lane ^ flip
            uint32_t lo = 0, hi = 0, z = ChainStack::IDLE_Z, w = 0, sp = sp0, vp = sp0;
            int flip = 1;
            int nxt = i;  // next record of the run
            auto goal_here = [&](uint32_t w) {
                chain_goal(&a.cnt.goals[inst0], &a.cnt.goal_origin[inst0], first_only ? &a.cnt.aborted[inst0] : nullptr,
                           run.origin(w));
            };
            // one round of every lane
            auto round = [&]() {
                // the lowest move left, and its child
                const uint32_t left4 = w & Chain::MOVES;
                const uint32_t bit = left4 & (left4 * neg1);
                const uint32_t rem = w ^ bit;
                uint32_t k, ylo, yhi, step;
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(k), "=r"(ylo), "=r"(yhi), "=r"(step) : "r"(__dp4a(bit, 0x03020100u, ctab)));
                // counted nodes in bits 8 and up (an idle lane has no bit)
                n32 = __dp4a(bit, 0x10101010u, n32);
                const uint32_t el = __funnelshift_l(hi, lo, k), eh = __funnelshift_l(lo, hi, k);
                const bool swap = bit >= 0x00100000u;
                const uint32_t tl = swap ? eh : el, th = swap ? el : eh;
                const uint32_t t = tl & 15u;
                const uint32_t clo = tl + t * ylo, chi = th + t * yhi;
                const uint32_t cz = z * one + step;
                const uint32_t inv = __byte_perm(bit, 0u, 0x0123);  // the inverse move
                // the child's moves; the inverse move takes its tile back,
                // so it goes towards iff this one went away (h rose)
                const uint32_t up = Chain::distance(clo, chi) * neg1 + cz;
                uint32_t cw = w & ~Chain::MOVES;
                if (!(up & inv))
                    cw = one * (0u - (1u << Chain::SLACK_SHIFT)) + cw;
                const uint32_t allowed = cz & ~inv & Chain::MOVES;
                uint32_t moves = allowed;
                if (!(cw & Chain::HALF_SLACK)) {
                    moves = allowed & ~up;
                    prn |= allowed & up;
                }
                if (__any_sync(FULL, clo == GLO)) {
                    if (clo == GLO && chi == GHI && cz == Chain::cells(0)) {
                        goal_here(cw);
                        moves = 0u;
                    }
                    __syncwarp();
                }
                ChainStack::next(lo, hi, z, w, sp, clo, chi, cz, cw | moves, moves, rem, rem & Chain::MOVES, sp0,
                                 one);
            };
            for (;;) {
                // idle lanes: each looks at one partner lane (its number
                // with one bit flipped, another bit each time) and takes an
                // entry from it, the bottom one first (the largest
                // subtrees); the giver's top entry fills the gap
                const unsigned idle = __ballot_sync(FULL, !(w & Chain::MOVES));
                bool ramp = false;  // many idle lanes: look again after one round
                if (idle) {
                    const int ni = __popc(idle), rank = __popc(idle & lt);
                    const bool dry = (idle >> lane) & 1u;
                    if (nxt < stop_at && ni >= ChainStack::LOAD) {
                        // records: each lane evaluates its own (those handed
                        // back as open nodes are counted already)
                        const bool v = dry && nxt + rank < stop_at;
                        Rec<4> r;
                        if (v)
                            r = run.src[nxt + rank];
                        const unsigned other = __ballot_sync(FULL, v && !run.front && r.inst != inst0);
                        // the first record of another instance ends the run
                        const int k = other ? __popc(idle & ((1u << (__ffs(other) - 1)) - 1u))
                                            : min(ni, stop_at - nxt);
                        if (v && rank < k && !dropped) {
                            const uint32_t p = m_blank(r.meta), last = m_last(r.meta);
                            const uint64_t fr = Chain::turn_left((uint64_t)r.b, (64u - 4u * p) & 63u);
                            const uint32_t half = (uint32_t)m_slack(r.meta) >> 1;
                            lo = (uint32_t)fr;
                            hi = (uint32_t)(fr >> 32);
                            z = Chain::cells(p);
                            w = (half << Chain::SLACK_SHIFT) | ((uint32_t)(nxt + rank - i) << Chain::SLOT_SHIFT);
                            if (r.meta & M_OPEN) {
                                w |= Chain::moves_from_rec(r.meta);
                            } else {
                                n32 += 1u << 8;
                                if (lo == GLO && hi == GHI && z == Chain::cells(0)) {
                                    goal_here(w);
                                } else {
                                    const uint32_t excl = last < 4u ? (0x10u << (8u * (3u - last))) : 0u;
                                    const uint32_t allowed = z & ~excl & Chain::MOVES;
                                    const uint32_t up = half ? 0u : Chain::away(lo, hi, z);
                                    prn |= allowed & up;
                                    w |= allowed & ~up;
                                }
                            }
                            if (!(w & Chain::MOVES)) {
                                z = ChainStack::IDLE_Z;
                                w = 0u;
                            }
                        }
                        nxt += k;
                        if (other)
                            stop_at = nxt;
                        __syncwarp();
                    } else if (ovf_n > 0) {
                        const int k = min(ni, ovf_n);
                        if (dry && rank < k) {
                            const uint4 e = covf[ovf_n - 1 - rank];
                            lo = e.x;
                            hi = e.y;
                            z = e.z;
                            w = e.w;
                        }
                        ovf_n -= k;
                    } else if (idle == FULL) {
                        break;  // (no record left: LOAD <= 32)
                    }
                    if (vp >= sp)
                        vp = sp0;
                    // what this lane offers: 0 idle, 1 nothing, 2 all but
                    // one of the moves of its node, else a stack entry
                    const uint32_t left4 = w & Chain::MOVES;
                    const uint32_t rest4 = left4 & (left4 - 1u);
                    const uint32_t mine = left4 ? (sp != sp0 ? vp : rest4 ? 2u : 1u) : 0u;
                    const uint32_t its = __shfl_xor_sync(FULL, mine, flip);
                    const bool take = mine == 0u && its > 1u, give = its == 0u && mine > 1u;
                    if (__any_sync(FULL, take && its == 2u)) {
                        const uint32_t a0 = __shfl_xor_sync(FULL, lo, flip), a1 = __shfl_xor_sync(FULL, hi, flip),
                                       a2 = __shfl_xor_sync(FULL, z, flip), a3 = __shfl_xor_sync(FULL, w, flip);
                        if (take && its == 2u) {
                            lo = a0;
                            hi = a1;
                            z = a2;
                            w = a3 & ~((a3 & Chain::MOVES) & (0u - (a3 & Chain::MOVES)));
                        }
                    }
                    flip = flip == 16 ? 1 : 2 * flip;
                    __syncwarp();
                    ChainStack::get_unless(take && its > 2u ? 0u : 1u, its, lo, hi, z, w);
                    __syncwarp();
                    if (give) {
                        if (mine == 2u) {
                            w ^= rest4;
                        } else {
                            sp -= ChainStack::ROW;
                            ChainStack::copy(vp, sp);
                            vp += ChainStack::ROW;
                        }
                    }
                    ramp = ni > 16;
                }
                const unsigned full = __ballot_sync(FULL, sp > sp_full);
                if (full) {
                    // full lanes move their bottom entries to the overflow
                    // stack, or to the next pass when that is full too, and
                    // their top entries fill the gap
                    const bool mine = (full >> lane) & 1u;
                    const int k = __popc(full) * ChainStack::SPILL;
                    if (lane == 0)
                        atomicAdd(&a.ctrl->spills, 1ull);
                    if (ovf_n + k <= a.ovf_cap) {
                        if (mine)
                            for (int j = 0; j < ChainStack::SPILL; ++j) {
                                uint32_t a0, a1, a2, a3;
                                a0 = a1 = a2 = a3 = 0;
                                ChainStack::get_unless(0u, sp0 + ChainStack::ROW * (uint32_t)j, a0, a1, a2, a3);
                                covf[ovf_n + j * __popc(full) + __popc(full & lt)] = make_uint4(a0, a1, a2, a3);
                            }
                        ovf_n += k;
                    } else {
                        chain_hand_back<4>(a.ctrl, a.Q, out, mine ? ChainStack::SPILL : 0,
                                           sp0 + ChainStack::ROW * ChainStack::SPILL, false, 0u, 0u, 0u, 0u, run);
                    }
                    if (mine)
                        for (int j = 0; j < ChainStack::SPILL; ++j) {
                            sp -= ChainStack::ROW;
                            ChainStack::copy(sp0 + ChainStack::ROW * (uint32_t)j, sp);
                        }
                    __syncwarp();
                }
                if (ramp) {
                    round();
                } else {
#pragma unroll
                    for (int turn = 0; turn < ChainStack::ROUNDS; ++turn)
                        round();
                }
                const int did = ramp ? 1 : ChainStack::ROUNDS;
                rounds += did;
                if ((rounds & 31) < did) {
                    nodes += __reduce_add_sync(FULL, n32 >> 8);
                    n32 = 0;
                    const int c = check(inst0, budgeted, left, nodes, flushed);
                    if (c == DROP) {
                        ovf_n = 0;
                        break;
                    }
                    if (c == STOP) {
                        stop = true;
                        break;
                    }
                }
            }
            // this run's counts
            nodes += __reduce_add_sync(FULL, n32 >> 8);
            acc_nodes += nodes - flushed;
            tot_nodes += nodes;
            if (budgeted)
                publish();
            if (stop) {
                chain_hand_back<W>(a.ctrl, a.Q, out, (int)((sp - sp0) / ChainStack::ROW), sp, (w & Chain::MOVES) != 0u, lo, hi,
                                   z, w, run);
                for (int j0 = 0; j0 < ovf_n; j0 += 32) {
                    const int j = j0 + lane;
                    uint4 e = make_uint4(0u, 0u, 0u, 0u);
                    if (j < ovf_n)
                        e = covf[j];
                    chain_hand_back<W>(a.ctrl, a.Q, out, 0, 0u, j < ovf_n, e.x, e.y, e.z, e.w, run);
                }
                hand_back_records<W>(a, frontier, n_act, n_front, act, in, out, nxt, end, lane);
                // input that no warp has taken yet goes back too
                for (;;) {
                    int h2 = 0;
                    if (lane == 0)
                        h2 = atomicAdd(&a.ctrl->head, chunk);
                    h2 = __shfl_sync(FULL, h2, 0);
                    if (h2 >= n_in)
                        break;
                    hand_back_records<W>(a, frontier, n_act, n_front, act, in, out, h2, min(h2 + chunk, n_in), lane);
                }
                break;
            }
            i = nxt;
        }
        if (stop)
            break;
    }
    publish();
    if (!stop && lane == 0)
        atomicAdd(&a.ctrl->exited, 1);
    // the last warp of a block publishes the block's end time and node
    // count; the last block to finish closes the pass
    if (lane == 0) {
        atomicMax(&s_t_end, global_ns());
        atomicAdd(&s_nodes, tot_nodes);
        __threadfence();
        if (atomicAdd(&s_warps_done, 1) == (int)(blockDim.x >> 5) - 1) {
            __threadfence();
            atomicMax(&a.ctrl->t_end, *(volatile unsigned long long *)&s_t_end);
            atomicAdd(&a.ctrl->search_nodes_total, *(volatile unsigned long long *)&s_nodes);
            __threadfence();
            if (atomicAdd(&a.ctrl->done_warps, 1) == (int)gridDim.x - 1) {
                __threadfence();
                a.ctrl->chain_passes += 1;
                end_of_pass<W>(a);
            }
        }
    }
}

}  // namespace bp
