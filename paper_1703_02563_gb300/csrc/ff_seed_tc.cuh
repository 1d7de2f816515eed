// ff_seed_tc.cuh - the seeding search (arXiv 1703.02563, Sec. 3.1 Eq. 1 and
// Sec. 3.2 Eq. 4: the l candidates of every coarsest-grid point) on the
// 5th-generation tensor cores (tcgen05, accumulators in tensor memory).
//
// The exact top-8 of a query q by (|q - c|^2, index) only needs, per query, the
// ranking of key(c) = |c|^2 - 2 q.c, since |q|^2 is common.  The keys of all
// (query, candidate) pairs are one matrix product -- the one dense contraction
// of the method -- computed exactly on the bf16 tensor cores with FP32
// accumulation:
//   query row     = (-2 q_1 .. -2 q_D, 65536, 256, 1, 0 ..)
//   candidate row = (  c_1 ..   c_D,  h2,  h1, h0, 0 ..),  |c|^2 = h2 65536 + h1 256 + h0
// Every entry is an integer of magnitude <= 256 or a power of two (exact in
// bf16), every product is exact, and every partial sum stays below 2^24 in
// magnitude, so FP32 accumulation in any order returns the key exactly.
//
// The product is reduced where it is made: k_seed_tc keeps, per query, the
// eight tiles of 128 consecutive candidates with the least (least key, tile).
// They hold the top 8.  For take x = (k, i) of the top 8 in tile t outside
// them: each of the eight has a candidate of key <= (t's least key) <= k, and
// where that key equals k its tile, hence its index, comes before x's; so
// eight candidates come before x, which is not in the top 8.  k_seed_pick
// then ranks those 1024 candidates exactly.
#pragma once

#include <cuda_bf16.h>

#include "ff_kernels.cuh"

namespace ffk {

constexpr int kTcRows = 128;    // queries per CTA (MMA M) and candidates per tile (MMA N)
constexpr int kTcStages = 4;    // candidate tiles in flight per accumulator
// A tile's entry in a query's list: least key + kTcKeyBias (21 bits: keys are
// -|q|^2 .. 3 * 27 * 128^2) above the tile's number in the list (11 bits).
constexpr int kTcKeyBias = 27 * 128 * 128;
constexpr int kTcTileBits = 11;
constexpr int kTcChunkTiles = 1 << kTcTileBits;   // tiles of a chunk, at most
// Up to this many tiles of candidates the lists keep tiles of 32 candidates instead of
// 128.  Ranking 8 x 128 is then most of a search (19200 queries, 1200 candidates, Lab: 165 us;
// 70 with tiles of 32, which is 0.3 to 1.0 of the time at 10 to 235 tiles), while the
// product, whose epilogue inserts four times as often, takes over with more of them (0.95
// of the time on average at 294 tiles, 1.03 at 509).
constexpr int kTcFineTiles = 256;
constexpr int kTcFineRows = 32;
static_assert(kTcFineTiles * (kTcRows / kTcFineRows) <= kTcChunkTiles, "fine tiles of a chunk");
constexpr int kTcMaxKey = 3 * 27 * 128 * 128;     // no candidate's key is above it

// Byte offset of element (r, k) in a tile of 128 rows x K bf16 laid out for
// the tensor core without swizzling: 8-row x 16-byte core matrices, the K
// direction's core matrices 128 bytes apart, 8-row groups K * 16 bytes apart.
__host__ __device__ constexpr int tc_tile_offset(int r, int k, int K) {
    return (r >> 3) * (K * 16) + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2;
}

// The rows above (K = 16 gray, 32 Lab) in tiles of 128, straight from the
// level-0 features: the ncand candidates of the stride grid (padded with rows
// whose h2 is +inf, so that their keys are), then the nq queries (padded with
// zero rows).
template <int C>
__global__ void __launch_bounds__(128)
    k_seed_prep(const uint8_t *__restrict__ fq, const uint8_t *__restrict__ fc, int W, int N,
                int WS, int nq, int stride, int Wc, int ncand, uint8_t *__restrict__ qtile,
                uint8_t *__restrict__ ctile) {
    constexpr int D = 9 * C, K = C == 1 ? 16 : 32, P = Geo<C>::P;
    const int nct = (ncand + kTcRows - 1) / kTcRows;
    const bool query = (int)blockIdx.x >= nct;
    const int t = query ? blockIdx.x - nct : blockIdx.x, r = t * kTcRows + threadIdx.x;
    uint32_t w[P / 4];
#pragma unroll
    for (int k = 0; k < P / 4; k++) w[k] = 0;
    const bool real = r < (query ? nq : ncand);
    if (real) {
        const int wd = query ? WS : Wc, y = r / wd, x = r - y * wd, step = query ? N : stride;
        const uint4 *src = reinterpret_cast<const uint4 *>(
            (query ? fq : fc) + ((size_t)y * step * W + (size_t)x * step) * P);
#pragma unroll
        for (int v = 0; v < P / 16; v++) {
            const uint4 u = __ldg(src + v);
            w[4 * v] = u.x, w[4 * v + 1] = u.y, w[4 * v + 2] = u.z, w[4 * v + 3] = u.w;
        }
    }
    int nn = 0;
#pragma unroll
    for (int k = 0; k < P / 4; k++) nn = __dp4a((int)w[k], (int)w[k], nn);
    __align__(16) __nv_bfloat16 row[K];
#pragma unroll
    for (int d = 0; d < D; d++) {
        const int v = (int)(int8_t)(w[d >> 2] >> (8 * (d & 3)));
        row[d] = __int2bfloat16_rn(query ? -2 * v : v);
    }
    row[D] = real ? __int2bfloat16_rn(query ? 65536 : nn >> 16)
                  : (query ? __int2bfloat16_rn(0)
                           : __float2bfloat16(__int_as_float(0x7f800000)));
    row[D + 1] = __int2bfloat16_rn(!real ? 0 : (query ? 256 : (nn >> 8) & 255));
    row[D + 2] = __int2bfloat16_rn(!real ? 0 : (query ? 1 : nn & 255));
#pragma unroll
    for (int d = D + 3; d < K; d++) row[d] = __int2bfloat16_rn(0);
    uint8_t *tile = (query ? qtile : ctile) + (size_t)t * kTcRows * K * 2;
#pragma unroll
    for (int kg = 0; kg < K / 8; kg++)
        *reinterpret_cast<uint4 *>(tile + tc_tile_offset(threadIdx.x, kg * 8, K)) =
            reinterpret_cast<const uint4 *>(row)[kg];
}

__device__ __forceinline__ uint32_t tc_smem(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
// shared-memory matrix descriptor (no swizzle): start, K-direction core
// matrix offset, 8-row group offset, descriptor version 1
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}
__device__ __forceinline__ void mbar_init(uint64_t *m, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc_smem(m)), "r"(count));
}
__device__ __forceinline__ bool mbar_test(uint64_t *m, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(ok)
        : "r"(tc_smem(m)), "r"(parity), "r"(100000)
        : "memory");
    return ok != 0;
}
// Bounded wait for phase `parity` of m: false when the CTA's abort flag is up
// or wait_ns passed (then the error word gets FF_ETIMEOUT and the flag rises).
__device__ __forceinline__ bool mbar_wait(uint64_t *m, uint32_t parity, unsigned long long wait_ns,
                                          volatile int *abort_flag, int *err) {
    if (mbar_test(m, parity)) return true;
    const unsigned long long t0 = globaltimer_ns();
    while (!mbar_test(m, parity)) {
        if (*abort_flag) return false;
        if (globaltimer_ns() - t0 > wait_ns) {
            atomicCAS(err, 0, kErrTimeout);
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}
// The same for a whole warp, with one answer for all its lanes: what follows (the
// tensor-memory loads) takes every lane or none.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *m, uint32_t parity,
                                               unsigned long long wait_ns,
                                               volatile int *abort_flag, int *err) {
    if (__all_sync(0xffffffffu, mbar_test(m, parity))) return true;
    const unsigned long long t0 = globaltimer_ns();
    while (!__all_sync(0xffffffffu, mbar_test(m, parity))) {
        int stop = *abort_flag;
        if (!stop && globaltimer_ns() - t0 > wait_ns) {
            atomicCAS(err, 0, kErrTimeout);
            *abort_flag = 1;
            stop = 1;
        }
        if (__any_sync(0xffffffffu, stop)) return false;
    }
    return true;
}
// After giving up: the phase, abort or not, for a second at most.
__device__ __forceinline__ void mbar_drain(uint64_t *m, uint32_t parity) {
    const unsigned long long t0 = globaltimer_ns();
    while (!mbar_test(m, parity) && globaltimer_ns() - t0 < 1000000000ull) {
    }
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *m, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc_smem(m)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *m) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc_smem(m)) : "memory");
}
// one contiguous global -> shared copy, completing on mbarrier m
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes, uint64_t *m) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(tc_smem(dst)),
        "l"(src), "r"(bytes), "r"(tc_smem(m))
        : "memory");
}

template <int KS>
__host__ __device__ constexpr int tc_seed_smem_bytes() {
    return kTcRows * 16 * KS * 2 * (1 + 2 * kTcStages);
}

// The least of 128 consecutive 32-bit columns of each of this warp's 32
// tensor-memory lanes, reduced by the load itself; the loaded columns are not
// used.
__device__ __forceinline__ float tmem_min128(uint32_t taddr) {
    [[maybe_unused]] uint32_t r[128];
    uint32_t least;
    asm volatile(
        "tcgen05.ld.red.sync.aligned.32x32b.x128.min.f32 {%0, %1, %2, %3, %4, %5, %6, %7, %8,"
        " %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25,"
        " %26, %27, %28, %29, %30, %31, %32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42"
        ", %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %5"
        "9, %60, %61, %62, %63, %64, %65, %66, %67, %68, %69, %70, %71, %72, %73, %74, %75, %"
        "76, %77, %78, %79, %80, %81, %82, %83, %84, %85, %86, %87, %88, %89, %90, %91, %92, "
        "%93, %94, %95, %96, %97, %98, %99, %100, %101, %102, %103, %104, %105, %106, %107, %"
        "108, %109, %110, %111, %112, %113, %114, %115, %116, %117, %118, %119, %120, %121, %"
        "122, %123, %124, %125, %126, %127}, %128, [%129];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
          "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]),
          "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]),
          "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]),
          "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63]),
          "=r"(r[64]), "=r"(r[65]), "=r"(r[66]), "=r"(r[67]), "=r"(r[68]), "=r"(r[69]), "=r"(r[70]), "=r"(r[71]),
          "=r"(r[72]), "=r"(r[73]), "=r"(r[74]), "=r"(r[75]), "=r"(r[76]), "=r"(r[77]), "=r"(r[78]), "=r"(r[79]),
          "=r"(r[80]), "=r"(r[81]), "=r"(r[82]), "=r"(r[83]), "=r"(r[84]), "=r"(r[85]), "=r"(r[86]), "=r"(r[87]),
          "=r"(r[88]), "=r"(r[89]), "=r"(r[90]), "=r"(r[91]), "=r"(r[92]), "=r"(r[93]), "=r"(r[94]), "=r"(r[95]),
          "=r"(r[96]), "=r"(r[97]), "=r"(r[98]), "=r"(r[99]), "=r"(r[100]), "=r"(r[101]), "=r"(r[102]), "=r"(r[103]),
          "=r"(r[104]), "=r"(r[105]), "=r"(r[106]), "=r"(r[107]), "=r"(r[108]), "=r"(r[109]), "=r"(r[110]), "=r"(r[111]),
          "=r"(r[112]), "=r"(r[113]), "=r"(r[114]), "=r"(r[115]), "=r"(r[116]), "=r"(r[117]), "=r"(r[118]), "=r"(r[119]),
          "=r"(r[120]), "=r"(r[121]), "=r"(r[122]), "=r"(r[123]), "=r"(r[124]), "=r"(r[125]), "=r"(r[126]), "=r"(r[127]),
          "=r"(least)
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    asm volatile("" : "+r"(least));
    return __uint_as_float(least);
}

// The same for each 32 of the 128 columns: four loads, one wait.
#define FF_T8(d) "t" #d "0, t" #d "1, t" #d "2, t" #d "3, t" #d "4, t" #d "5, t" #d "6, t" #d "7"
#define FF_LD_MIN32(out, a, b, c, d, addr)                                                      \
    "tcgen05.ld.red.sync.aligned.32x32b.x32.min.f32 {" FF_T8(a) ", " FF_T8(b) ", " FF_T8(c)     \
    ", " FF_T8(d) "}, " out ", [" addr "];\n\t"
__device__ __forceinline__ void tmem_min32(uint32_t taddr, float (&least)[4]) {
    uint32_t m[4];
    asm volatile("{\n\t.reg .b32 t<170>;\n\t"
                 FF_LD_MIN32("%0", 1, 2, 3, 4, "%4")
                 FF_LD_MIN32("%1", 5, 6, 7, 8, "%5")
                 FF_LD_MIN32("%2", 9, 10, 11, 12, "%6")
                 FF_LD_MIN32("%3", 13, 14, 15, 16, "%7")
                 "tcgen05.wait::ld.sync.aligned;\n\t}"
                 : "=r"(m[0]), "=r"(m[1]), "=r"(m[2]), "=r"(m[3])
                 : "r"(taddr), "r"(taddr + 32), "r"(taddr + 64), "r"(taddr + 96)
                 : "memory");
#pragma unroll
    for (int s = 0; s < 4; s++) least[s] = __uint_as_float(m[s]);
}
#undef FF_LD_MIN32
#undef FF_T8

// (least key, tile) into a thread's list of eight
__device__ __forceinline__ void tile_insert(uint32_t (&l)[8], uint32_t x) {
#pragma unroll
    for (int e = 0; e < 8; e++) {
        const uint32_t lo = min(l[e], x);
        x = max(l[e], x);
        l[e] = lo;
    }
}

// Per CTA: 128 queries (tensor-memory lanes; epilogue thread = query row)
// against one chunk of candidates, 128 per tile; even tiles go through one
// 128-column accumulator, odd ones through the other, and each has its own
// issuing warp (4, 5), whose thread keeps four tiles of bulk copies in flight
// and issues the K/16 MMAs of a tile once its accumulator has been drained.
// Each thread of the epilogue warps (0-3) takes its row's least key out of the
// accumulator with one reducing tensor-memory load and puts (least key, tile)
// into its list of eight.  All waits are bounded; an issuing thread that gives up waits
// (bounded too) for its copies and products under way.  The list of chunk c and
// query row q is lists[(c * 128 nqt + q) * 8 ..], empty entries 0xffffffff.
//
// FINE: the lists' tiles have 32 candidates (tiles 4 t .. 4 t + 3 of a chunk are the
// product's tile t), so that k_seed_pick has a quarter of the candidates to rank, for four
// insertions per product here.
template <int KS, bool FINE>
__global__ void __launch_bounds__(192, 2)
    k_seed_tc(const uint8_t *__restrict__ qtile, const uint8_t *__restrict__ ctile, int nct,
              int chunk, uint32_t *__restrict__ lists, int *err, unsigned long long wait_ns) {
    constexpr int K = 16 * KS;
    constexpr uint32_t TILE_BYTES = kTcRows * K * 2;
    // dynamic shared memory (tc_seed_smem_bytes<KS>()): the query tile and the candidate ring
    extern __shared__ __align__(1024) uint8_t tc_dyn[];
    uint8_t *sA = tc_dyn;
    uint8_t(*sB)[TILE_BYTES] = reinterpret_cast<uint8_t(*)[TILE_BYTES]>(tc_dyn + TILE_BYTES);
    __shared__ __align__(8) uint64_t bar_a, full[2 * kTcStages], accf[2], acce[2];
    __shared__ uint32_t taddr_slot;
    __shared__ int abort_flag;
    volatile int *v_abort = &abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int qt = blockIdx.x;
    const int tile0 = blockIdx.y * chunk, ntiles = min(chunk, nct - tile0);
    if (tid == 0) {
        abort_flag = 0;
        mbar_init(&bar_a, 1);
        for (int s = 0; s < 2 * kTcStages; s++) mbar_init(&full[s], 1);
        for (int b = 0; b < 2; b++) {
            mbar_init(&accf[b], 1);
            mbar_init(&acce[b], 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(
            tc_smem(&taddr_slot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t taddr = taddr_slot;

    if (warp >= 4) {
        // ---------------- copies and MMAs of the tiles 2 n + g
        const int g = warp - 4, mine = (ntiles - g + 1) / 2;
        if (lane == 0) {
            uint64_t *fullg = full + g * kTcStages;
            uint8_t(*ring)[TILE_BYTES] = sB + g * kTcStages;
            const uint8_t *src = ctile + (size_t)(tile0 + g) * TILE_BYTES;
            auto copy = [&](int n) {
                mbar_expect_tx(&fullg[n % kTcStages], TILE_BYTES);
                bulk_copy(ring[n % kTcStages], src + (size_t)n * 2 * TILE_BYTES, TILE_BYTES,
                          &fullg[n % kTcStages]);
            };
            if (g == 0) {
                mbar_expect_tx(&bar_a, TILE_BYTES);
                bulk_copy(sA, qtile + (size_t)qt * TILE_BYTES, TILE_BYTES, &bar_a);
            }
            int sent = 0;          // copies so far; products so far: n
            while (sent < min(kTcStages, mine)) copy(sent++);
            // kind::f16, bf16 x bf16 -> f32, both K-major, N = 128, M = 128
            constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) |
                                       ((uint32_t)(kTcRows >> 3) << 17) |
                                       ((uint32_t)(kTcRows >> 4) << 24);
            const uint32_t d = taddr + (uint32_t)(g * kTcRows);
            const bool have_a = mbar_wait(&bar_a, 0, wait_ns, v_abort, err);
            int n = 0;
            for (; n < mine && have_a; n++) {
                const int s = n % kTcStages;
                if (!mbar_wait(&fullg[s], (n / kTcStages) & 1, wait_ns, v_abort, err)) break;
                if (n >= 1 && !mbar_wait(&acce[g], (n - 1) & 1, wait_ns, v_abort, err)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int ks = 0; ks < KS; ks++) {
                    const uint64_t da = tc_desc(tc_smem(sA) + ks * 256, 128, K * 16);
                    const uint64_t db = tc_desc(tc_smem(ring[s]) + ks * 256, 128, K * 16);
                    asm volatile(
                        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
                        "l"(da), "l"(db), "r"(idesc), "r"(ks));
                }
                asm volatile(
                    "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::
                        "r"(tc_smem(&accf[g]))
                    : "memory");
                // tile n - 1 has been drained, so its product is done with its stage
                if (n >= 1 && sent < mine) copy(sent++);
            }
            if (n < mine) {
                // gave up: no copy or product may still be under way when the CTA ends
                if (g == 0) mbar_drain(&bar_a, 0);
                for (int m = n; m < sent; m++) mbar_drain(&fullg[m % kTcStages], (m / kTcStages) & 1);
                if (n > 0) mbar_drain(&accf[g], (n - 1) & 1);
            }
        }
    } else {
        // ---------------- epilogue: warp w reads tensor-memory lanes 32 w .. +31
        // (thread = query row)
        const uint32_t ta = taddr + ((uint32_t)(warp * 32) << 16);
        uint32_t l[8];
#pragma unroll
        for (int e = 0; e < 8; e++) l[e] = 0xffffffffu;
        for (int t = 0; t < ntiles; t++) {
            const int g = t & 1;
            if (!mbar_wait_warp(&accf[g], (t >> 1) & 1, wait_ns, v_abort, err)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            constexpr int F = FINE ? 4 : 1;
            float least[4];
            if constexpr (FINE) tmem_min32(ta + (uint32_t)(g * kTcRows), least);
            else least[0] = tmem_min128(ta + (uint32_t)(g * kTcRows));
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&acce[g]);
#pragma unroll
            for (int f = 0; f < F; f++) {
                // key + bias in the low mantissa bits of 2^23 + key + bias (exact).  A fine
                // tile may be all padding (+inf): a key above every other stands for it.
                const float key = FINE ? fminf(least[f], (float)(kTcMaxKey + 1)) : least[f];
                tile_insert(l, (__float_as_uint(key + (float)(8388608 + kTcKeyBias)) << kTcTileBits) +
                                   (uint32_t)(F * t + f));
            }
        }
        const size_t row = ((size_t)blockIdx.y * gridDim.x + qt) * kTcRows + warp * 32 + lane;
        uint4 *dst = reinterpret_cast<uint4 *>(lists + row * 8);
        dst[0] = make_uint4(l[0], l[1], l[2], l[3]);
        dst[1] = make_uint4(l[4], l[5], l[6], l[7]);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 4) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(taddr));
    }
}

__device__ __forceinline__ bool lex_less(int d, int i, int D, int I) {
    return d < D || (d == D && i < I);
}

// A query's list across a warp: lane e holds its e-th best (distance, index).
struct KnnList {
    int D, I;
};
__device__ __forceinline__ void knn_insert(KnnList &l, int d, int i, int lane) {
    const bool less = lex_less(d, i, l.D, l.I);
    const int uD = __shfl_up_sync(0xffffffffu, l.D, 1), uI = __shfl_up_sync(0xffffffffu, l.I, 1);
    if (less) {
        const bool here = lane == 0 || !lex_less(d, i, uD, uI);
        l.D = here ? d : uD;
        l.I = here ? i : uI;
    }
}
// Puts every lane's (d, i) into the list that belongs among its first eight
// and does not come behind (capD, capI).  The eighth entry is looked at after
// each insertion, so that of many equal distances (flat image regions) only
// the first few are inserted.
__device__ __forceinline__ void knn_take(KnnList &l, int d, int i, int lane, int capD, int capI) {
    unsigned m = 0xffffffffu;
    for (;;) {
        int D = __shfl_sync(0xffffffffu, l.D, 7), I = __shfl_sync(0xffffffffu, l.I, 7);
        if (lex_less(capD, capI, D, I)) D = capD, I = capI;
        m &= __ballot_sync(0xffffffffu, lex_less(d, i, D, I));
        if (!m) return;
        const int s = __ffs(m) - 1;
        m &= m - 1;
        knn_insert(l, __shfl_sync(0xffffffffu, d, s), __shfl_sync(0xffffffffu, i, s), lane);
    }
}

// The warp's (d, i) pairs in order, through the warp's 32 words of buf (the
// empty ones, d = 0x7fffffff, last).
__device__ __forceinline__ KnnList knn_sort(int d, int i, int2 *buf, int lane) {
    int r = 0;
#pragma unroll
    for (int k = 0; k < 32; k++) {
        const int D = __shfl_sync(0xffffffffu, d, k), I = __shfl_sync(0xffffffffu, i, k);
        r += lex_less(D, I, d, i) || (D == d && I == i && k < lane);
    }
    __syncwarp();
    buf[r] = make_int2(d, i);
    __syncwarp();
    const int2 e = buf[lane];
    __syncwarp();
    return KnnList{e.x, e.y};
}

// What becomes of a finished list: its first `leaf` entries to the caller
// (idx, dist), and, for a match, the one of lowest matching error at the
// coarsest scale (Eq. 1), the earlier rank on ties, as the point's flow.
struct KnnOut {
    int leaf;
    int *idx, *dist;               // [queries][leaf], or NULL
    const uint8_t *f1L, *f2L;      // coarsest level
    int W, H, L, WL, HL;
    uint32_t *flow;                // [queries], or NULL
    int *cost;
};
// An int where a caller's array has it: the array may start at any byte.
__device__ __forceinline__ void store_any(int *p, int v) {
    if (((uintptr_t)p & 3) == 0) {
        *p = v;
    } else {
        uint8_t *b = reinterpret_cast<uint8_t *>(p);
#pragma unroll
        for (int k = 0; k < 4; k++) b[k] = (uint8_t)((uint32_t)v >> (8 * k));
    }
}
template <int C>
__device__ __forceinline__ void knn_finish(const KnnOut &o, int q, int lane, KnnList l) {
    constexpr int P = Geo<C>::P;
    const bool ok = lane < o.leaf && l.D != 0x7fffffff;
    if (o.idx && lane < o.leaf) {
        store_any(o.idx + (size_t)q * o.leaf + lane, ok ? l.I : -1);
        store_any(o.dist + (size_t)q * o.leaf + lane, ok ? l.D : -1);
    }
    if (!o.flow) return;
    const int gy = q / o.WL, gx = q - gy * o.WL;
    const int px = gx << o.L, py = gy << o.L;
    uint32_t f = kFlowInvalid;
    int e = kCostInvalid;
    if (ok) {
        uint32_t qw[P / 4];
#pragma unroll
        for (int w = 0; w < P / 4; w++) qw[w] = ldg32(o.f1L + (size_t)q * P + 4 * w);
        int fx = 8 * (l.I % o.W - px), fy = 8 * (l.I / o.W - py);
        clamp_flow(o.W, o.H, px, py, fx, fy);
        e = sad_full<C>(o.f2L, make_tap<P>(px, py, fx, fy, o.L, o.WL, o.HL), qw);
        f = pack_flow(fx, fy);
    }
    const int best = __reduce_min_sync(0xffffffffu, e);
    const int win = __ffs(__ballot_sync(0xffffffffu, e == best)) - 1;
    if (lane == win) {
        o.flow[q] = f;
        o.cost[q] = e;
    }
}

// A query's tile lists -> its top 8 (and, for a match, its coarsest flow); one
// warp per query.  The eight tiles of least (key, tile) come from its nch
// lists; the eighth's least key bounds the eighth distance, so few of their
// candidates are kept: those are collected and sorted once.  A tile has `trows`
// candidates: 32 (FINE), or a multiple of 128.
//
// What bounds it: the tiles' rows through L1, where rows a stride apart are lines of their
// own (8 x 128 of them per query, 19200 queries, Lab: 61 us with every pixel a candidate,
// 157 us with every eighth; 8 x 32: 53 us).  Halves of a row by a pair of lanes took 44 us
// there but 72 instead of 62 with every pixel.
template <int C, bool FINE>
__global__ void __launch_bounds__(128)
    k_seed_pick(const uint8_t *__restrict__ fq, const uint8_t *__restrict__ fc, int W, int N,
                int WS, int nq, int stride, int Wc, int ncand, const uint32_t *__restrict__ lists,
                int nqt, int nch, int chunk, int trows, const KnnOut out) {
    constexpr int P = Geo<C>::P, NV = P / 16, NW = Geo<C>::NW;
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ int2 s_buf[4][32];
    const int q = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    int2 *buf = s_buf[threadIdx.x >> 5];
    if (q >= nq) return;
    uint32_t qw[4 * NV];
    {
        const int gy = q / WS, gx = q - gy * WS;
        const uint4 *src = reinterpret_cast<const uint4 *>(
            fq + ((size_t)gy * N * W + (size_t)gx * N) * P);
#pragma unroll
        for (int v = 0; v < NV; v++) {
            const uint4 u = __ldg(src + v);
            qw[4 * v] = u.x, qw[4 * v + 1] = u.y, qw[4 * v + 2] = u.z, qw[4 * v + 3] = u.w;
        }
    }
    int qn = 0;
#pragma unroll
    for (int w = 0; w < NW; w++) qn = __dp4a((int)qw[w], (int)qw[w], qn);
    // the eight tiles (D: least key + bias, I: tile); a list is sorted
    KnnList best{0x7fffffff, 0x7fffffff};
    for (int c0 = 0; c0 < nch; c0 += 4) {
        const int c = c0 + (lane >> 3);
        int d = 0x7fffffff, t = 0x7fffffff;
        if (c < nch) {
            const uint32_t x = __ldg(lists + ((size_t)c * nqt * kTcRows + q) * 8 + (lane & 7));
            if (x != 0xffffffffu) {
                d = (int)(x >> kTcTileBits);
                t = c * chunk + (int)(x & ((1u << kTcTileBits) - 1));
            }
        }
        if (c0 == 0)
            best = nch == 1 ? KnnList{d, t} : knn_sort(d, t, buf, lane);
        else
            knn_take(best, d, t, lane, 0x7fffffff, 0x7fffffff);
    }
    const int D7 = __shfl_sync(FULL, best.D, 7);
    // (bD, bI): nothing behind it belongs to the top 8
    int bD = D7 == 0x7fffffff ? D7 : D7 - kTcKeyBias + qn, bI = 0x7fffffff;
    KnnList l{0x7fffffff, 0x7fffffff};
    int held = 0;                  // candidates in buf, all before (bD, bI) when they came
    // 128 candidates at a time: a stretch of a tile, or four fine tiles
    for (int k = 0; k < 8; k += FINE ? 4 : 1) {
        const int t = __shfl_sync(FULL, best.I, k);
        if (t == 0x7fffffff) break;
        // eight are known: may this tile, or one behind it, hold a better one?  (Uniform frames,
        // 76800 queries, Lab: the search 195 -> 147 us with every eighth pixel; others unchanged.)
        if (bI != 0x7fffffff) {
            const int c = t * trows, cy = c / Wc, first = (cy * W + (c - cy * Wc)) * stride;
            if (!lex_less(__shfl_sync(FULL, best.D, k) - kTcKeyBias + qn, first, bD, bI)) break;
        }
        const int end = FINE ? t * trows + 1 : min((t + 1) * trows, ncand);
        for (int o0 = t * trows; o0 < end; o0 += kTcRows) {
            uint4 r[4][NV];
            int idx[4];
            bool in[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                int c = o0 + 32 * j + lane;
                if (FINE) {
                    const int tj = __shfl_sync(FULL, best.I, k + j);
                    c = tj == 0x7fffffff ? ncand : tj * kTcFineRows + lane;
                }
                in[j] = c < ncand;
                idx[j] = min(c, ncand - 1);
                if (stride > 1) {
                    const int cy = idx[j] / Wc, cx = idx[j] - cy * Wc;
                    idx[j] = cy * stride * W + cx * stride;
                }
#pragma unroll
                for (int v = 0; v < NV; v++)
                    r[j][v] = __ldg(reinterpret_cast<const uint4 *>(fc + (size_t)idx[j] * P) + v);
            }
#pragma unroll
            for (int j = 0; j < 4; j++) {
                int dot = 0, nn = 0;
#pragma unroll
                for (int w = 0; w < NW; w++) {
                    const uint32_t cw = reinterpret_cast<const uint32_t *>(&r[j][0])[w];
                    dot = __dp4a((int)cw, (int)qw[w], dot);
                    nn = __dp4a((int)cw, (int)cw, nn);
                }
                const int d = nn + qn - 2 * dot;
                const bool hit = in[j] && lex_less(d, idx[j], bD, bI);
                const unsigned m = __ballot_sync(FULL, hit);
                if (!m) continue;
                if (held + __popc(m) > 32) {   // full: into the list, which lowers the bound
                    __syncwarp();
                    const int2 e = lane < held ? buf[lane] : make_int2(0x7fffffff, 0x7fffffff);
                    knn_take(l, e.x, e.y, lane, bD, bI);
                    knn_take(l, hit ? d : 0x7fffffff, idx[j], lane, bD, bI);
                    held = 0;
                    const int D = __shfl_sync(FULL, l.D, 7), I = __shfl_sync(FULL, l.I, 7);
                    if (lex_less(D, I, bD, bI)) bD = D, bI = I;
                } else {
                    if (hit) buf[held + __popc(m & ((1u << lane) - 1))] = make_int2(d, idx[j]);
                    held += __popc(m);
                }
            }
        }
    }
    __syncwarp();
    const int2 e = lane < held ? buf[lane] : make_int2(0x7fffffff, 0x7fffffff);
    if (__any_sync(FULL, l.D != 0x7fffffff))
        knn_take(l, e.x, e.y, lane, bD, bI);
    else
        l = knn_sort(e.x, e.y, buf, lane);
    knn_finish<C>(out, q, lane, l);
}

}  // namespace ffk
