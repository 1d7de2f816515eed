// ff_block.cuh - propagation sweep by blocks of four columns (arXiv
// 1703.02563, Sec. 3.1 Eq. 2 and the random search step; Sec. 3.2 for R_n = R n).
#pragma once
#include "ff_sweep.cuh"

namespace ffk {

// Level row that row v of a sweep's frame stands for.  The last strip's and cluster's
// rows past the frame (v >= V) take the last row's place: their warps form its
// addresses and load its first query, which they do not use.
__host__ __device__ constexpr int block_row(int v, int V, bool flipy) {
    const int r = v < V ? v : V - 1;
    return flipy ? V - 1 - r : r;
}

// ---------------------------------------------------------------------------
// matching error with the query's bytes as they are: per dimension one dp4a
// seeds the accumulator with -64 q and one adds the four weighted taps
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t sad_raw(uint32_t t00, uint32_t t10, uint32_t t01, uint32_t t11,
                                            uint32_t w, int4 s, uint32_t acc) {
    const uint32_t lo01 = __byte_perm(t00, t10, 0x5140);
    const uint32_t hi01 = __byte_perm(t00, t10, 0x7362);
    const uint32_t lo23 = __byte_perm(t01, t11, 0x5140);
    const uint32_t hi23 = __byte_perm(t01, t11, 0x7362);
    acc = __sad(__dp4a((int)__byte_perm(lo01, lo23, 0x5410), (int)w, s.x), 0, acc);
    acc = __sad(__dp4a((int)__byte_perm(lo01, lo23, 0x7632), (int)w, s.y), 0, acc);
    acc = __sad(__dp4a((int)__byte_perm(hi01, hi23, 0x5410), (int)w, s.z), 0, acc);
    acc = __sad(__dp4a((int)__byte_perm(hi01, hi23, 0x7632), (int)w, s.w), 0, acc);
    return acc;
}
__device__ __forceinline__ int4 query_seed(uint32_t q) {
    return make_int4(__dp4a((int)q, (int)0x000000C0u, 0), __dp4a((int)q, (int)0x0000C000u, 0),
                     __dp4a((int)q, (int)0x00C00000u, 0), __dp4a((int)q, (int)0xC0000000u, 0));
}

// all words of a feature vector by one thread
template <int C>
__device__ __forceinline__ uint32_t sad_point(const uint8_t *f2L, const TapRows &t,
                                              const uint8_t *q) {
    constexpr int NV = Geo<C>::P / 16, NWU = C == 3 ? 7 : 3;
    uint32_t acc = 0;
#pragma unroll
    for (int v = 0; v < NV; v++) {
        const Words<4> a = ldg_words<4>(f2L + t.r0 + t.c0 + 16 * v);
        const Words<4> b = ldg_words<4>(f2L + t.r0 + t.c1 + 16 * v);
        const Words<4> c = ldg_words<4>(f2L + t.r1 + t.c0 + 16 * v);
        const Words<4> d = ldg_words<4>(f2L + t.r1 + t.c1 + 16 * v);
        const Words<4> x = ldg_words<4>(q + 16 * v);
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (4 * v + j < NWU)
                acc = sad_raw(a.w[j], b.w[j], c.w[j], d.w[j], t.w, query_seed(x.w[j]), acc);
    }
    return acc;
}

struct SearchArgs {
    int t, dir, radius_q3;          // sweep that the search follows, direction word, R
    uint32_t seed, pair_id;
};

// Random search of one point (Sec. 3.1): the offset from Philox4x32-10,
// counter (y*W + x, t, L, dir), key (seed, pair_id); kept only if strictly better.
template <int C>
__device__ __forceinline__ void search_point(const SearchArgs &s, const uint8_t *f1L,
                                             const uint8_t *f2L, int W, int H, int L, int U, int V,
                                             int gx, int gy, uint32_t &flow, uint32_t &cost) {
    constexpr int P = Geo<C>::P;
    if (flow == kFlowInvalid) return;
    const int n = 1 << L, px = gx * n, py = gy * n;
    const int R = s.radius_q3 * n;
    const uint32_t span = 2u * (uint32_t)R + 1u;
    const uint4 rnd = philox4x32_10(
        make_uint4((uint32_t)(py * W + px), (uint32_t)s.t, (uint32_t)L, (uint32_t)s.dir), s.seed,
        s.pair_id);
    const int ox = (int)(rnd.x % span) - R, oy = (int)(rnd.y % span) - R;
    const int tx = clampi(8 * px + flow_x(flow) + ox, 0, 8 * (W - 1));
    const int ty = clampi(8 * py + flow_y(flow) + oy, 0, 8 * (H - 1));
    const uint32_t f = pack_flow(tx - 8 * px, ty - 8 * py);
    if (f == flow) return;
    const TapRows t = taps_of<P>(f, gx, gy, L, n >> 1, U, V);
    const uint32_t e = sad_point<C>(f2L, t, f1L + ((size_t)gy * U + gx) * P);
    if (e < cost) {
        flow = f;
        cost = e;
    }
}

// the random search on its own, over a whole level (when a match stops between
// a sweep's search and the next sweep, which otherwise does it)
template <int C>
__global__ void __launch_bounds__(128)
    k_search(const SearchArgs s, const uint8_t *f1L, const uint8_t *f2L, int W, int H, int L, int U,
             int V, uint32_t *flow, int *cost) {
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i >= U * V) return;
    uint32_t f = flow[i], c = (uint32_t)cost[i];
    const uint32_t f0 = f;
    search_point<C>(s, f1L, f2L, W, H, L, U, V, i % U, i / U, f, c);
    if (f != f0) {
        flow[i] = f;
        cost[i] = (int)c;
    }
}

constexpr int kBlkCols = 4;                  // columns decided per step
constexpr int kBlkRows = 4;                  // rows of a strip, one warp each
constexpr int kBlkCluster = 8;               // strips of a cluster
// Stager warps: Lab blocks take four, gray ones two; more only contend with the rows for
// issue slots.  One match from seeds, the other number of each (six frame sizes, 128x96 to
// 1920x1080): Lab with two 6-9% slower (1024x436 3.94 -> 4.23 ms), gray with four 7-10%
// (1242x375 3.41 -> 3.75 ms).
__host__ __device__ constexpr int blk_stagers(int C) { return C == 3 ? 4 : 2; }
__host__ __device__ constexpr int blk_threads(int C) { return (kBlkRows + blk_stagers(C) + 1) * 32; }
// CTAs per SM that the registers have to allow (0: as they come).  Gray: three, i.e. 80
// registers; with a few more only two fit, which costs 32 contexts on 640x480 frames
// 13.3 -> 16.6 ms, and with four, 72 registers, a lone 1242x375 pair takes 8% longer.
// Lab: two come (96 registers); three spill (1024x436: 8.4 -> 10.8 ms).
__host__ __device__ constexpr int blk_ctas(int C) { return C == 3 ? 0 : 3; }
constexpr int kBlkRing = 16;                 // staged blocks per row
// Levels up to this wide start the next sweep's launch early: its waiting CTAs hold
// room on the SMs (a 128x96 pair 973 -> 917 us, 1024x436 8.53 -> 8.45 ms; on every
// level the latter took 8.60 ms).
constexpr int kBlkOverlap = 512;
constexpr uint32_t kBlkNone = 0x80000000u;   // cost of a candidate that does not exist

struct BlockArgs {
    const uint8_t *f1L, *f2L;
    uint32_t *flow;                // level state, updated in place
    int *cost;
    unsigned long long *edge;      // [cluster][U] rows between clusters: (epoch << 32) | flow
    unsigned int *ticket;          // cluster counter of this launch (zeroed before)
    int *err;
    int W, H, L, U, V, d;
    int search;                    // the search of the sweep before is still to be done
    SearchArgs rs;
    uint32_t epoch;
    unsigned long long wait_ns;
    int force_timeout;
};

// what the stagers prepare for one row and block
struct BlockStage {
    uint32_t flow[4], cost[4];     // current values, after the pending random search
    uint32_t run[6];               // cost of current flow i at column j: 01 12 23 02 03 13
    uint32_t pad[2];
};

struct BlockShared {
    BlockStage stage[kBlkRows][kBlkRing];
    // Block + 1 of each staged block, released last.  Words of their own: a vector load is
    // a set of loads without an order among them, so one that held a tag and costs could
    // bring the tag of this block with the costs of the block there before.
    uint32_t tag[kBlkRows][kBlkRing];
    uint32_t cand[kBlkRows][16];   // costs of a step: H0-3, V0-3, V runs 01 12 23 02 03 13
    int done[kBlkRows];            // blocks each row has finished
    int abort, cluster;
};

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// address of the same shared-memory location in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t ld_cluster_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.relaxed.cluster.shared::cluster.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster_u64_if(uint32_t addr, unsigned long long v, bool pred) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t"
        "@p st.relaxed.cluster.shared::cluster.b64 [%0], %1;\n\t}" ::"r"(addr),
        "l"(v), "r"((int)pred)
        : "memory");
}
__device__ __forceinline__ void sts64_if(uint32_t addr, unsigned long long v, bool pred) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t"
        "@p st.volatile.shared.b64 [%0], %1;\n\t}" ::"r"(addr),
        "l"(v), "r"((int)pred)
        : "memory");
}
__device__ __forceinline__ void stg_u32_if(uint32_t *p, uint32_t v, bool pred) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p st.global.b32 [%0], %1;\n\t}" ::"l"(p),
        "r"(v), "r"((int)pred)
        : "memory");
}
// volatile accesses by 32-bit shared-memory address
__device__ __forceinline__ unsigned long long lds64s(uint32_t p) {
    unsigned long long v;
    asm volatile("ld.volatile.shared.b64 %0, [%1];" : "=l"(v) : "r"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint4 lds128s(uint32_t p) {
    uint4 r;
    asm volatile("ld.volatile.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
                 : "r"(p)
                 : "memory");
    return r;
}
__device__ __forceinline__ void sts32s(uint32_t p, uint32_t v) {
    asm volatile("st.volatile.shared.b32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}
// a flag and what it guards: the writer's lanes meet (__syncwarp) before one of them
// releases the flag; a reader acquires it before it loads the rest
__device__ __forceinline__ uint32_t lds32_acquire(uint32_t p) {
    uint32_t v;
    asm volatile("ld.acquire.cta.shared::cta.b32 %0, [%1];" : "=r"(v) : "r"(p) : "memory");
    return v;
}
__device__ __forceinline__ void sts32_release(uint32_t p, uint32_t v) {
    asm volatile("st.release.cta.shared::cta.b32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// packed 16-bit add (no carry between the halves)
__device__ __forceinline__ uint32_t add_s16x2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("add.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// dynamic shared memory: the row above each of the strip's rows, (1 << 32) | flow
// per column once it is decided
__host__ __device__ constexpr size_t block_smem_bytes(int U) {
    return (size_t)kBlkRows * ((U + kBlkCols - 1) / kBlkCols * kBlkCols) * 8;
}

// Poll k of a wait that found nothing; true when the warp must give up.  Every 64th looks
// at the clock and the CTA's abort flag, every 1024th (about 20 us) also whether another
// CTA or an earlier sweep of this direction has given up, so that one expiry ends the
// whole match: a load from global memory, which at every look would hold up the hand-over
// that is waited for.
__device__ __forceinline__ bool wait_over(int k, unsigned long long &t0, unsigned long long wait_ns,
                                          volatile int *abort_flag, int *err) {
    if (k & 63) return false;
    if ((k & 1023) == 0 && ld_relaxed_i32(err) != 0) *abort_flag = 1;
    return wait_expired(t0, wait_ns, abort_flag, err);
}

// One sweep in direction d, after the random search of the sweep before (which
// only changes a point's own value, so it can be done when the value is fetched).
//
// In the sweep's frame (u, v) a point takes the best of its current value, the
// value above it (u, v-1) and the one to its left (u-1, v), the later in that
// order on ties: a serial chain.  Here a warp owns a row and decides four columns
// per step.  A value that reaches column j of a block is the one left of the
// block, the one above a column i <= j, or the current one of a column i <= j; so
// 4 + 10 + 10 costs hold every outcome.  Those of current values (the points' own
// and six "runs" i -> j) do not depend on a neighbour and are staged ahead; the
// other 14 are evaluated at once, two lanes each, when the row above has decided
// the block; and the decision is then a chain of compares and selects.
//
//  * Row warps 0-3.  Decisions go to the row below as (1 << 32) | flow words: the
//    next warp's row of shared memory, the next CTA of the cluster's (distributed
//    shared memory), or, behind a cluster's last row, global memory.
//  * Stager warps: per block current values after the pending random search, and
//    the runs' costs; their loads also bring most of what the rows will read into L1.
//  * Loader warp (first CTA of a cluster): the global row above the cluster.
// Clusters take their rows in ticket order, so a row only waits for one that runs.
// Every wait is bounded and warp-uniform, and one that expires ends the others, as in
// the batch sweep.
//
// What bounds it: a step of ~1060 cycles (U/4 of them) and a row hand-over of ~870
// (V of them), both chains of dependent instructions of one warp (about 5 cycles
// each) with one tap load in them; 57% of the time are the hand-overs.  At 1024x436
// Lab the level-0 sweep takes 373 us with cold caches (650 with a step of one column of eight rows,
// ~920 cycles on each of U + V anti-diagonals).  Two columns per step would double
// the steps for about a tenth less of a hand-over; eight need 44 costs per step.
// Four rows per strip keep one row warp on each quarter of an SM.
template <int C>
__global__ void __cluster_dims__(kBlkCluster, 1, 1)
    __launch_bounds__(blk_threads(C), blk_ctas(C))
    k_sweep_block(const BlockArgs a) {
    constexpr int P = Geo<C>::P, LW = P / 8;   // bytes per vector; words of an evaluating lane
    constexpr unsigned FULL = 0xffffffffu;
    constexpr bool kEarly = C == 3;
    constexpr int kStagers = blk_stagers(C), kThreads = blk_threads(C);
    extern __shared__ __align__(16) unsigned long long vin_all[];   // [kBlkRows][4 NB]
    __shared__ __align__(16) BlockShared sm;
    volatile int *v_abort = &sm.abort;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int U = a.U, V = a.V, W = a.W, H = a.H, L = a.L, n = 1 << L, half = n >> 1;
    const int NB = (U + kBlkCols - 1) / kBlkCols, UP = NB * kBlkCols;
    const uint32_t rank = cluster_rank();
    for (int j = tid; j < kBlkRows * UP; j += kThreads) vin_all[j] = 0ull;
    for (int j = tid; j < kBlkRows * kBlkRing; j += kThreads) (&sm.tag[0][0])[j] = 0;
    if (tid < kBlkRows) sm.done[tid] = 0;
    if (tid == 0) sm.abort = 0;
    if (rank == 0 && tid == 0) sm.cluster = (int)atomicAdd(a.ticket, 1u);
    cluster_sync();   // (also: every CTA has started and cleared its rows)
    // Up to here nothing of the sweep before is touched: the launch may overlap its
    // end (programmatic dependent launch).
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int cluster = (int)ld_cluster_u32(mapa(smem_addr(&sm.cluster), 0));
    const int strip = cluster * kBlkCluster + (int)rank;
    const int v0 = strip * kBlkRows;
    const bool flipx = (a.d == 1 || a.d == 2), flipy = (a.d == 1 || a.d == 3);
    const uint8_t *__restrict__ f1L = a.f1L, *__restrict__ f2L = a.f2L;

    if (v0 >= V) {
        // no rows here
        launch_dependents();
    } else if (warp < kBlkRows) {
        // ================= a row =================
        const int v = v0 + warp;
        const int gy = block_row(v, V, flipy);
        const int py = gy * n;
        const bool live = v < V, has_v = v > 0;
        // this lane's evaluation: e 0-3 the left value at column e, 4-7 the value
        // above column e - 4 there, 8-13 the value above column i at a later
        // column j (01 12 23 02 03 13); two lanes share one, half of the words each
        const int e = min(lane >> 1, 13), h = lane & 1;
        const int src = e < 4 ? 0 : (e < 8 ? e - 4 : (int)((0x100210 >> (4 * (e - 8))) & 7));
        const int tgt = e < 8 ? (e & 3) : (int)((0x332321 >> (4 * (e - 8))) & 7);
        const bool left = e < 4;
        const uint32_t rowP = (uint32_t)U * P, wofs = 4 * LW * h;
        const uint8_t *__restrict__ qrow = f1L + (size_t)gy * rowP + wofs;
        // shared-memory addresses: the row above at this lane's source column, the
        // staged blocks, the costs of a step
        uint32_t vin = smem_addr(vin_all + (size_t)warp * UP);
        const uint32_t stage = smem_addr(sm.stage[warp]), cand = smem_addr(sm.cand[warp]);
        const uint32_t tags = smem_addr(sm.tag[warp]), done = smem_addr(&sm.done[warp]);
        // where the decisions go: the row below, in this CTA or the next of the
        // cluster, or the row in global memory behind the cluster's last strip
        const bool to_cta = warp + 1 < kBlkRows, to_peer = !to_cta && rank + 1 < kBlkCluster;
        uint32_t out = (to_peer ? mapa(smem_addr(vin_all), rank + 1)
                                : smem_addr(vin_all) + 8u * (uint32_t)((warp + 1) * UP)) +
                       8u * (lane & 3);
        const bool hands = lane < 4 && to_cta, hands_peer = lane < 4 && to_peer,
                   hands_far = lane < 4 && !to_cta && !to_peer;
        unsigned long long *edge = a.edge + (size_t)cluster * U + (lane & 3);
        // lanes 0-3 write the flows, 4-7 the costs
        uint32_t *state_row = (lane < 4 ? a.flow : reinterpret_cast<uint32_t *>(a.cost)) +
                              (size_t)gy * U + (flipx ? U - 1 - (lane & 3) : (lane & 3));
        const uint32_t want = (a.force_timeout && v == kBlkRows) ? 2u : 1u;
        const int loy = -8 * py, hiy = 8 * (H - 1) - 8 * py, by = half - loy;
        const uint32_t wstep = (uint32_t)(flipx ? 8 * n : -8 * n) & 0xffffu;   // window per column
        uint32_t lo0, hi0;                            // window of the block's first column
        {
            const int x = -8 * n * (flipx ? U - 1 : 0);
            lo0 = __byte_perm((uint32_t)x, (uint32_t)loy, 0x5410);
            hi0 = __byte_perm((uint32_t)(x + 8 * (W - 1)), (uint32_t)hiy, 0x5410);
        }
        int xcol = -8 * n * (flipx ? U - 1 - tgt : tgt);   // -8 x of this lane's target column
        uint32_t state = kFlowInvalid;                // this row's value at the column before
        Words<LW> qn;
        {
            const int u = min(tgt, U - 1);
            qn = ldg_words<LW>(qrow + (uint32_t)(flipx ? U - 1 - u : u) * P);
        }
        const int nb = live ? NB : 0;
#pragma unroll 1
        for (int b = 0; b < nb; b++) {
            // (past the right edge: the last column's window)
            const int lx = clampi(xcol, -8 * n * (U - 1), 0);
            xcol += flipx ? 8 * n * kBlkCols : -8 * n * kBlkCols;
            const uint32_t lo = __byte_perm((uint32_t)lx, (uint32_t)loy, 0x5410);
            const uint32_t hi = __byte_perm((uint32_t)(lx + 8 * (W - 1)), (uint32_t)hiy, 0x5410);
            const uint32_t slot = stage + (uint32_t)(b & (kBlkRing - 1)) * (uint32_t)sizeof(BlockStage);
            // What needs no neighbour: the staged block, the windows of the four columns, the
            // query.  For Lab frames before the wait, where it costs the rows below nothing;
            // for gray ones, whose evaluations are short, in the shadow of the tap loads.  (One
            // match from seeds, the other way round, same six sizes: Lab 1-5% slower, 1024x436
            // 3.94 -> 4.04 ms; gray 1-6%, 1242x375 3.41 -> 3.61 ms.)
            uint4 cf, cc, ca, cb;
            uint32_t lo1, hi1, lo2, hi2, lo3, hi3;
            int4 seed[LW];
            auto own_part = [&]() -> bool {
                // staged yet?  (A vote: the lanes need not see the same tag.)
                const uint32_t tag = tags + 4u * (uint32_t)(b & (kBlkRing - 1));
                unsigned long long t0 = 0;
                for (int k = 1; !__all_sync(FULL, lds32_acquire(tag) == (uint32_t)b + 1); k++)
                    if (wait_over(k, t0, a.wait_ns, v_abort, a.err)) return false;
                cf = lds128s(slot), cc = lds128s(slot + 16), ca = lds128s(slot + 32);
                cb = lds128s(slot + 48);
                lo1 = add_s16x2(lo0, wstep), hi1 = add_s16x2(hi0, wstep);
                lo2 = add_s16x2(lo1, wstep), hi2 = add_s16x2(hi1, wstep);
                lo3 = add_s16x2(lo2, wstep), hi3 = add_s16x2(hi2, wstep);
#pragma unroll
                for (int k = 0; k < LW; k++) seed[k] = query_seed(qn.w[k]);
                const int u = min((b + 1) * kBlkCols + tgt, U - 1);
                qn = ldg_words<LW>(qrow + (uint32_t)(flipx ? U - 1 - u : u) * P);
                return true;
            };
            if constexpr (kEarly) {
                if (!own_part()) goto finished;
            }
            // the values above
            unsigned long long va = 0;
            if (has_v) {
                unsigned long long t0 = 0;
                for (int k = 1;; k++) {
                    va = lds64s(vin + 8 * src);
                    if (__all_sync(FULL, (uint32_t)(va >> 32) == want)) break;
                    if (wait_over(k, t0, a.wait_ns, v_abort, a.err)) goto finished;
                }
            }
            // this lane's candidate, clamped into the frame; its taps and weights
            const uint32_t f = left ? state : (has_v ? (uint32_t)va : kFlowInvalid);
            const uint32_t fc = clamp_s16x2(f, lo, hi);
            const int sx = ((int)(int16_t)(fc & 0xffffu) + (half - lx)) >> L;
            const int sy = (((int)fc >> 16) + by) >> L;
            const int ix = min(sx >> 3, U - 1), iy = min(sy >> 3, V - 1);
            const uint32_t o00 = (uint32_t)iy * rowP + ((uint32_t)ix * P + wofs);
            const uint32_t dx = ix < U - 1 ? P : 0, dy = iy < V - 1 ? rowP : 0;
            const Words<LW> ta = ldg_words<LW>(f2L + o00), tb = ldg_words<LW>(f2L + (o00 + dx));
            const Words<LW> tc = ldg_words<LW>(f2L + (o00 + dy)),
                            td = ldg_words<LW>(f2L + (o00 + dx + dy));
            const uint32_t w = (uint32_t)(8 + 255 * (sx & 7)) * (uint32_t)(8 + 65535 * (sy & 7));
            if constexpr (!kEarly) {
                if (!own_part()) goto finished;
            }
            // The four flows above, waited for by other lanes than this one: behind a barrier of the
            // warp, which a vote is not.  Lab: one here, in the shadow of the tap loads (with the
            // loads behind the next one 8.43 -> 8.66 ms for the 1024x436 pair).  Gray: the one before
            // the costs are read (1242x375 pair 2.94 ms; here 3.04).
            uint4 vf0, vf1;
            if constexpr (kEarly) {
                __syncwarp();
                vf0 = lds128s(vin), vf1 = lds128s(vin + 16);
            }
            uint32_t acc0 = 0, acc1 = 0;
#pragma unroll
            for (int k = 0; k < LW; k += 2) {
                acc0 = sad_raw(ta.w[k], tb.w[k], tc.w[k], td.w[k], w, seed[k], acc0);
                acc1 = sad_raw(ta.w[k + 1], tb.w[k + 1], tc.w[k + 1], td.w[k + 1], w, seed[k + 1],
                               acc1);
            }
            acc0 += acc1;
            acc0 += __shfl_xor_sync(FULL, acc0, 1);
            if (f == kFlowInvalid) acc0 = kBlkNone;
            sts32s(cand + 4 * e, acc0);
            __syncwarp();
            const uint4 eh = lds128s(cand), ev = lds128s(cand + 16), ra = lds128s(cand + 32),
                        rb = lds128s(cand + 48);
            if constexpr (!kEarly) vf0 = lds128s(vin), vf1 = lds128s(vin + 16);
            // the better of current and above per column (the latter on ties), with
            // what it would cost at the later columns
            const bool p0 = ev.x <= cc.x, p1 = ev.y <= cc.y, p2 = ev.z <= cc.z, p3 = ev.w <= cc.w;
            const uint32_t bf0 = p0 ? clamp_s16x2(vf0.x, lo0, hi0) : cf.x;
            const uint32_t bf1 = p1 ? clamp_s16x2(vf0.z, lo1, hi1) : cf.y;
            const uint32_t bf2 = p2 ? clamp_s16x2(vf1.x, lo2, hi2) : cf.z;
            const uint32_t bf3 = p3 ? clamp_s16x2(vf1.z, lo3, hi3) : cf.w;
            const uint32_t bc0 = min(ev.x, cc.x), bc1 = min(ev.y, cc.y), bc2 = min(ev.z, cc.z),
                           bc3 = min(ev.w, cc.w);
            const uint32_t b01 = p0 ? ra.x : ca.x, b12 = p1 ? ra.y : ca.y, b23 = p2 ? ra.z : ca.z,
                           b02 = p0 ? ra.w : ca.w, b03 = p0 ? rb.x : cb.x, b13 = p1 ? rb.y : cb.y;
            // left to right: the value at the column before wins ties
            const bool k0 = eh.x <= bc0;
            const uint32_t d0 = k0 ? clamp_s16x2(state, lo0, hi0) : bf0;
            const uint32_t e1 = k0 ? eh.y : b01;
            uint32_t e2 = k0 ? eh.z : b02, e3 = k0 ? eh.w : b03;
            const bool k1 = e1 <= bc1;
            const uint32_t d1 = k1 ? clamp_s16x2(d0, lo1, hi1) : bf1;
            e2 = k1 ? e2 : b12;
            e3 = k1 ? e3 : b13;
            const bool k2 = e2 <= bc2;
            const uint32_t d2 = k2 ? clamp_s16x2(d1, lo2, hi2) : bf2;
            e3 = k2 ? e3 : b23;
            const bool k3 = e3 <= bc3;
            const uint32_t d3 = k3 ? clamp_s16x2(d2, lo3, hi3) : bf3;
            state = d3;
            // lane j hands on column j, lanes j and j + 4 write it
            const int j = lane & 3;
            const uint32_t df = j < 2 ? (j == 0 ? d0 : d1) : (j == 2 ? d2 : d3);
            const bool inside = b * kBlkCols + j < U;
            sts64_if(out, (1ull << 32) | df, hands);
            if (!to_cta) {
                st_cluster_u64_if(out, (1ull << 32) | df, hands_peer);
                st_relaxed_u64_if(edge, ((unsigned long long)a.epoch << 32) | df, hands_far && inside);
            }
            const uint32_t c0 = min(eh.x, bc0), c1 = min(e1, bc1), c2 = min(e2, bc2), c3 = min(e3, bc3);
            const uint32_t dc = j < 2 ? (j == 0 ? c0 : c1) : (j == 2 ? c2 : c3);
            stg_u32_if(state_row, lane < 4 ? df : dc, lane < 8 && inside);
            // (every lane has read the staged block: they met before the costs were read)
            if (lane == 0) sts32_release(done, (uint32_t)(b + 1));
            out += 8 * kBlkCols;
            vin += 8 * kBlkCols;
            edge += kBlkCols;
            state_row += flipx ? -kBlkCols : kBlkCols;
            lo0 = add_s16x2(lo3, wstep);
            hi0 = add_s16x2(hi3, wstep);
        }
        // rows past the frame's edge never hold a stager back
        if (!live && lane == 0) sts32s(done, NB + kBlkRing);
    } else if (warp < kBlkRows + kStagers) {
        // ================= a stager =================
        // pass p: blocks 2 p and 2 p + 1 of the four rows, one point per lane
        const int w = warp - kBlkRows;
        const int r = lane >> 3, i = lane & 3;
        const int v = v0 + r;
        const int gy = block_row(v, V, flipy);
        const int py = gy * n;
        const int loy = -8 * py, hiy = 8 * (H - 1) - 8 * py;
        for (int p = w; 2 * p < NB; p += kStagers) {
            // room: every row is past the block that used the slots before
            unsigned long long t0 = 0;
            for (int k = 1;; k++) {
                if (k > 1) __nanosleep(200);
                const bool ok = lane >= kBlkRows ||
                                (int)lds32_acquire(smem_addr(&sm.done[lane])) + kBlkRing >= 2 * p + 2;
                if (__all_sync(FULL, ok)) break;
                if (wait_over(k, t0, a.wait_ns, v_abort, a.err)) goto finished;
            }
            __syncwarp();          // (four lanes have looked, all will write)
            if (p == 0) launch_dependents();   // (the next sweep's launch may come in)
            const int u = 8 * p + (lane & 7);
            const bool in = v < V && u < U;
            uint32_t f = kFlowInvalid, c = 0x7fffffffu;
            int gx = 0;
            if (in) {
                gx = flipx ? U - 1 - u : u;
                f = a.flow[(size_t)gy * U + gx];
                c = (uint32_t)a.cost[(size_t)gy * U + gx];
                if (a.search) search_point<C>(a.rs, f1L, f2L, W, H, L, U, V, gx, gy, f, c);
            }
            // runs: lane i takes i -> i + 1 (lane 3: 0 -> 2), then lanes 0, 1 take i -> 3
            const uint32_t f0 = __shfl_sync(FULL, f, lane & ~3);
            const uint32_t fa = i == 3 ? f0 : f;
            uint32_t ra = kBlkNone, rb = kBlkNone;
            const int ja = i == 3 ? 2 : i + 1;
#pragma unroll 1
            for (int pass = 0; pass < 2; pass++) {
                const int j = pass == 0 ? ja : 3;
                const int uj = u - i + j;
                if ((pass == 0 || i < 2) && v < V && uj < U && fa != kFlowInvalid) {
                    const int gj = flipx ? U - 1 - uj : uj;
                    const int lx = -8 * n * gj;
                    const uint32_t fc = clamp_s16x2(
                        fa, __byte_perm((uint32_t)lx, (uint32_t)loy, 0x5410),
                        __byte_perm((uint32_t)(lx + 8 * (W - 1)), (uint32_t)hiy, 0x5410));
                    const TapRows t = taps_of<P>(fc, gj, gy, L, half, U, V);
                    const uint32_t s = sad_point<C>(f2L, t, f1L + ((size_t)gy * U + gj) * P);
                    if (pass == 0) ra = s;
                    else rb = s;
                }
            }
            const int slot = (2 * p + ((lane >> 2) & 1)) & (kBlkRing - 1);
            BlockStage *st = &sm.stage[r][slot];
            st->flow[i] = f;
            st->cost[i] = c;
            st->run[i] = ra;
            if (i < 2) st->run[4 + i] = rb;
            __syncwarp();
            if (i == 0) sts32_release(smem_addr(&sm.tag[r][slot]), (uint32_t)(u >> 2) + 1);
        }
    } else if (rank == 0 && strip > 0) {
        // ================= the loader: the row above this cluster =================
        const unsigned long long *srow = a.edge + (size_t)(cluster - 1) * U;
        int base = 0, k = 0;
        unsigned long long t0 = 0;
        while (base < U) {
            const int col = base + lane;
            unsigned long long x = 0;
            if (col < U) x = ld_relaxed_u64(srow + col);
            const bool ready = col >= U || (uint32_t)(x >> 32) == a.epoch;
            const unsigned m = __ballot_sync(FULL, ready);
            const int got = m == FULL ? 32 : __ffs(~m) - 1;
            if (lane < got && col < U) sts64(vin_all + col, (1ull << 32) | (uint32_t)x);
            // past the frame's right edge nothing is above, but the row waits for it
            if (lane < got && col >= U && col < UP) sts64(vin_all + col, (1ull << 32) | kFlowInvalid);
            if (got > 0) {
                base += got;
                t0 = 0;
                k = 0;
            } else if (wait_over(++k, t0, a.wait_ns, v_abort, a.err)) {
                break;
            }
        }
        for (int col = max(base, U) + lane; base >= U && col < UP; col += 32)
            sts64(vin_all + col, (1ull << 32) | kFlowInvalid);
    }
finished:
    __syncwarp();
    // no CTA leaves while a peer may still write into it
    cluster_sync();
}

}  // namespace ffk
