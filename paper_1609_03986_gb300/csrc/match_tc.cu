// Brute-force Hamming matching on the 5th-generation tensor cores (Sec. 4's
// all-pairs distance computation, done as a dense contraction).
//
// Every descriptor bit b is expanded to the 4-bit E2M1 float 1 - 2 b (+1 or -1, two
// per byte), so the dot product of two expanded descriptors is (bits that agree) -
// (bits that differ) = 512 - 2 Hamming(q, t): one contraction gives the distance,
// with no popcount term.  The block-scaled fp4 MMA (kind::mxf4, every scale factor
// 2^0) issues twice the products per clock of the 8-bit kind; the products are +-1
// and the sums at most 512 in magnitude, so fp32 accumulation is exact.
//
// One launch serves a batch of matching problems (query set x train set pairs; a
// single hamming_match call is a batch of one).  All descriptors live in one
// expanded buffer (two TMA tensor maps over it: 128-row query boxes, 120-row train
// boxes).  The blocks work in pairs (clusters of two on the two SMs of a TPC, one block
// per SM, persistent); a pair's MMAs (cta_group::2, M = 256) take a tile of 256 queries,
// 128 in each block, and 240 train rows, 120 in each block's shared memory.  The units
// (problem, 256-query tile, 240-train tile) of all problems are shared out over the pairs
// (match_common.cuh); in a pair:
//   warp 0     TMA producer of its block's half: the query rows (128 rows x 256 B, 32 KB)
//              stay resident while consecutive units share them; train chunks (120 rows x
//              128 B, half of K) go through a 12-stage ring, 128-byte swizzle; both
//              blocks' copies complete on the first block's barriers;
//   warps 1-2  MMA issuers, in the pair's first block (even / odd units): per unit 6
//              tcgen05.mma (per 128-byte chunk of K = 256 values: K = 96, 96, 64) into one
//              of two TMEM accumulators (columns 0 and 256 of both blocks; the constant
//              scale factors in 496-511); their commits reach both blocks' barriers;
//              warp 2 also allocates TMEM;
//   warp 3     idle;
//   warps 4-23 epilogue of the block's 128 rows (one query row and 48 columns per
//              thread): three reducing TMEM loads (tcgen05.ld.red .max) bring the 48
//              values and the largest of each 16, and the accumulator is released at
//              once.  A group of 16 whose largest value is below the row's bound costs
//              nothing more: the bound is the smallest second-best distance any of the
//              row's five column groups holds (shared memory), and a column displaces one
//              of its own group's keys only with a larger value (later columns have
//              larger train indices).  The others take the top-two update (a tournament
//              over 64 v - column, unique values that break ties to the lower index).
//              When the pair leaves a query tile the row's two (distance << 32 | index)
//              keys go to a partial record.  In a launch of at most kFusedUnitsPerPair
//              units per pair the last block to leave a tile's half (an arrival counter
//              each) combines the records of its rows and writes their matches (ties to
//              the lowest train index, ratio test).
// match_merge_kernel does the same combination as a separate pass; it serves longer
// launches and the batches in which some problem has queries but an empty train set
// (no unit, so no block visits its tiles).  All mbarrier waits are bounded (sm103.h); on a timeout
// the block raises the device flag, lets its copies and MMAs end, frees TMEM.
//
// Why pairs and K = 96: shared memory (128 bytes per clock per SM) bounds the MMAs.  One
// block alone (M = 128, N = 240) reads 94 KB of operands per unit and the copies write
// 61 KB, 1,215 clocks (the kernel took 1,206 per unit; its MMAs at K = 64 need 960, and at
// K = 96 they are no faster than 846 because of the operand reads).  In a pair each block
// reads its own query rows but only half of the train rows, and copies half: 94 KB, 735
// clocks, next to 720 of MMAs (K = 96 issues 1.5 times the products of K = 64 per clock).
// Measured (GB300, whole calls; single blocks, K = 64 and an MMA thread of its own, and now):
// 16,384 x 1,048,576 descriptors 2,369 -> 1,768 us (about 945 clocks per unit), 10,000 x 10,000
// 46.4 -> 42.0 us, a batch of 64 images and 476 pairs (3.4e11 distances, extraction included)
// 67.0 -> 51.1 ms.  What is left above 720 clocks is the accumulators' round trip (MMA end, commit, TMEM loads of 20
// warps, arrivals of both blocks, next MMA: about 1,200 clocks for two accumulators in
// flight); three accumulators of 160 columns are slower (2,357 us: the epilogue's time per
// unit hardly depends on its columns).  Short walks are bound by the top-two updates of
// their first units instead; there the pairs of a tile exchange row bounds (single problems).
#include <cuda.h>

#include <cmath>
#include <new>

#include "match_common.cuh"
#include "sm103.h"

namespace latch {

namespace {

using namespace sm103;

constexpr int kRowsA = 128;             // query rows per block
constexpr int kRowsQ = 2 * kRowsA;      // query rows per tile (M of the pair's MMA)
constexpr int kColsB = 240;             // train rows per unit (N)
constexpr int kRowsB = kColsB / 2;      // of these in each block's shared memory
constexpr int kRowsP = kRowsQ;          // partial records per tile slot: one per query row
constexpr int kKBytes = kExpRowBytes;   // expanded descriptor: 512 x 4-bit
constexpr int kChunk = 128;             // K bytes per swizzle atom / TMA box
constexpr int kChunks = kKBytes / kChunk;
constexpr int kStages = 12;             // train chunks in flight (six units)
constexpr int kTileBytes = kRowsA * kChunk;   // 16 KB: a query chunk of 128 rows x 128 B (one TMA box)
constexpr int kStageBytes = kRowsB * kChunk;  // 15 KB: a train chunk of 120 rows x 128 B (one TMA box)
constexpr int kAccs = 2;                // TMEM accumulators in rotation (unit i uses i % kAccs)
constexpr int kAccStride = 256;          // accumulator a at TMEM columns [a kAccStride, +kColsB)
constexpr int kEpiWarps = 20;           // epilogue: 4 lane quarters x 5 column groups
constexpr int kEpiThreads = kEpiWarps * 32;
constexpr int kThreads = 128 + kEpiThreads;         // producer, two MMA issuers, an idle warp, then the epilogue
constexpr int kColGroups = kEpiWarps / 4;
constexpr int kColsPerThread = kColsB / kColGroups;  // accumulator columns one epilogue thread scans
constexpr int kLdCols = 16;                          // columns per tcgen05.ld
constexpr int kLds = kColsPerThread / kLdCols;       // loads per unit and thread
constexpr int kTmemCols = 512;
constexpr uint32_t kSfaCol = (kAccs - 1) * kAccStride + kColsB;  // scale factors of A: 4 columns (128 rows)
constexpr uint32_t kSfbCol = kSfaCol + 8;  // scale factors of B: 4 columns per 128 rows
constexpr uint32_t kScaleOne = 0x7F7F7F7Fu;  // four UE8M0 scale factors 2^0 (columns 496-511 all hold it)
constexpr uint32_t kIdesc64 = idesc_mxf4_e2m1(kRowsQ, kColsB);
constexpr uint32_t kIdesc96 = kIdesc64 | kIdescK96;
// A walk exchanges its row bounds with the tile's other pairs over its first units; beyond,
// updates are rare and the exchange costs more than it saves (16,384 x 1,048,576: 2,019 us
// when every unit of the walk does it, 1,755 with 64).
constexpr int32_t kShareUnits = 64;
constexpr int32_t kNoBound = 1024;      // a distance bound above every distance (512 bits)
constexpr int64_t kFusedUnitsPerPair = 64;  // longer launches combine the tiles' records in a separate pass
constexpr int64_t kWholeTilesPerPair = 8;   // batches with this many query tiles per pair share whole tiles
static_assert(kStageBytes % 1024 == 0 && kTileBytes % 1024 == 0, "128-byte swizzle atoms");
static_assert(kSfaCol % 8 == 0 && kSfbCol + 4 * ((kColsB + 127) / 128) <= kTmemCols, "TMEM columns overlap");
static_assert(kColsPerThread == kLds * kLdCols && kColsB == kColGroups * kColsPerThread, "epilogue column split");
static_assert(kColsB % 16 == 0 && kColsB <= 256 && kColsPerThread < 64 && kAccStride % 32 == 0, "unit shape");

// max(a, b, c) in one instruction.
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// mbar_wait by a whole warp, which goes on together.
__device__ __forceinline__ bool wait_all(uint64_t* bar, uint32_t parity, volatile int* abort) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort));
}

// Barrier of the epilogue threads (named barrier 1).
__device__ __forceinline__ void group_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory"); }

struct Smem {
    // offsets in the 1024-aligned dynamic buffer
    static constexpr int a = 0;                                        // [kChunks] boxes of 16 KB
    static constexpr int b = a + kChunks * kTileBytes;                 // [kStages] chunks of 15 KB
    static constexpr int part = b + kStages * kStageBytes;             // uint64 [kEpiThreads][2]
    static constexpr int bound = part + kEpiThreads * 16;              // int32 [kRowsA]
    static constexpr int bars = bound + kRowsA * 4;                    // uint64 barriers
    static constexpr int nbars = 2 * kStages + 2 + 2 * kAccs + 2;
    static constexpr int misc = bars + nbars * 8;                      // tmem base, abort flag, last-arrival flag
    static constexpr int total = misc + 16;
};
constexpr int kSmemBytes = Smem::total + 1024;
static_assert(kSmemBytes <= 227 * 1024, "shared memory per block");

// The fields of the current problem that the walk needs every unit are kept in
// registers (reading the problem table, a kernel parameter, with a run-time index
// costs hundreds of cycles per unit on the MMA warp's path).
struct UnitIter {
    int p;          // current problem (count once the walk is over)
    int count;      // problems in the batch
    int32_t m, n;   // query tile, train tile of the current unit
    int32_t cs;     // c': the block's share index in problem p
    int32_t ntl;    // train tiles of problem p
    int32_t g0;     // global index of problem p's first query tile
    int32_t t_row0; // first train row of problem p
    int32_t nt;     // train rows of problem p
    int64_t left;   // units left in the share, the current one included
    template <class B>
    __device__ __forceinline__ void set(const B& b, const Share& s) {
        p = s.p;
        m = s.m;
        n = s.n;
        cs = s.cs;
        left = s.left;
        if (p < count) {
            const MatchProblem& P = b.p[p];
            ntl = P.ntl;
            g0 = P.g0;
            t_row0 = P.t_row0;
            nt = P.nt;
        }
    }
    template <class B>
    __device__ __forceinline__ void init(const B& b, int64_t c) {
        count = b.count;
        set(b, first_share(b, c));
    }
    template <class B>
    __device__ __forceinline__ bool done(const B&) const { return p >= count; }
    template <class B>
    __device__ __forceinline__ int64_t g(const B&) const { return g0 + m; }
    template <class B>
    __device__ __forceinline__ int64_t slot(const B& b) const {
        return g0 + m + cs + static_cast<int64_t>(p) * (b.grid - 1);
    }
    template <class B>
    __device__ __forceinline__ bool last_of_tile(const B&) const { return left == 1 || n + 1 == ntl; }
    template <class B>
    __device__ __forceinline__ void next(const B& b, int64_t c) {
        if (--left == 0) {
            set(b, share_after(b, p, m, c));
            return;
        }
        if (++n == ntl) {
            n = 0;
            ++m;
        }
    }
};

// The block's walk as runs: a run is the consecutive units of one query tile (a run
// ends where its tile or its share ends, so consecutive runs are different tiles).
// The MMA issuers step through runs and count units inside them, which keeps the
// iterator off their per-unit path.
struct RunIter {
    UnitIter u;     // at the run's first unit
    int32_t len;    // units in the run
    template <class B>
    __device__ __forceinline__ void init(const B& b, int64_t c) {
        u.init(b, c);
        set(b);
    }
    template <class B>
    __device__ __forceinline__ void set(const B& b) {
        const int64_t rest = static_cast<int64_t>(u.ntl - u.n);
        len = u.done(b) ? 0 : static_cast<int32_t>(u.left < rest ? u.left : rest);
    }
    template <class B>
    __device__ __forceinline__ bool done(const B& b) const { return u.done(b); }
    template <class B>
    __device__ __forceinline__ void next(const B& b, int64_t c) {
        if (len == u.left) {
            u.set(b, share_after(b, u.p, u.m, c));  // the share ends with this run
        } else {
            u.left -= len;          // the run ends with its tile
            ++u.m;
            u.n = 0;
        }
        set(b);
    }
};

// Calls f(c') for the share index of every block that holds a record of query tile
// m of problem P, and returns how many there are.  With U >= G every share is
// non-empty and the owners are the contiguous range from the share of the tile's
// first unit to that of its last; with U < G every non-empty share holds one unit,
// so the owners are those of the tile's ntl units.
template <class B, class F>
__device__ __forceinline__ int64_t for_each_owner(const B& b, const MatchProblem& P, int64_t m, F&& f) {
    const int64_t U = static_cast<int64_t>(P.mt) * P.ntl;
    const int64_t u0 = m * P.ntl;
    if (U >= b.grid) {
        const int64_t clo = split_owner(u0, U, b.grid), chi = split_owner(u0 + P.ntl - 1, U, b.grid);
        for (int64_t cs = clo; cs <= chi; ++cs) f(cs);
        return chi - clo + 1;
    }
    for (int64_t u = u0; u < u0 + P.ntl; ++u) f(split_owner(u, U, b.grid));
    return P.ntl;
}

// Number of blocks that hold a record of query tile m of problem P.
template <class B>
__device__ __forceinline__ int64_t tile_owner_count(const B& b, const MatchProblem& P, int64_t m) {
    const int64_t U = static_cast<int64_t>(P.mt) * P.ntl;
    if (U < b.grid) return P.ntl;
    const int64_t u0 = m * P.ntl;
    return split_owner(u0 + P.ntl - 1, U, b.grid) - split_owner(u0, U, b.grid) + 1;
}

// Combines the partial records of row r of query tile m (global index g) of problem
// p over the blocks that own the tile's units.
template <class B>
__device__ __forceinline__ void combine_row(const B& b, int p, int64_t m, int64_t g, int r,
                                            const uint64_t* partials, uint64_t& k1, uint64_t& k2) {
    for_each_owner(b, b.p[p], m, [&](int64_t cs) {
        const uint64_t* rec = partials + ((g + cs + static_cast<int64_t>(p) * (b.grid - 1)) * kRowsP + r) * 2;
        top2_insert_u64(__ldcg(rec), k1, k2);
        top2_insert_u64(__ldcg(rec + 1), k1, k2);
    });
}

// The output record of a query from its two best keys (Sec. 4 ratio test).
__device__ __forceinline__ latch_match final_match(uint64_t k1, uint64_t k2, int k, int r_milli) {
    latch_match mres;
    mres.idx1 = k1 == kNoKey ? -1 : static_cast<int32_t>(k1 & 0xffffffffu);
    mres.dist1 = k1 == kNoKey ? 0xffff : static_cast<uint16_t>(k1 >> 32);
    const bool has2 = k == 2 && k2 != kNoKey;
    mres.idx2 = has2 ? static_cast<int32_t>(k2 & 0xffffffffu) : -1;
    mres.dist2 = has2 ? static_cast<uint16_t>(k2 >> 32) : 0xffff;
    if (k1 == kNoKey)
        mres.accepted = 0;
    else if (k == 1)
        mres.accepted = 1;
    else
        mres.accepted = (1000ll * mres.dist1 < static_cast<long long>(r_milli) * mres.dist2) ? 1 : 0;
    mres.pad[0] = mres.pad[1] = mres.pad[2] = 0;
    return mres;
}

// tile_cnt: per-query-tile arrival counters, zero at launch and zero again after a
// complete launch; NULL = leave the combination to match_merge_kernel.
// row_bounds (single problems): per query row the distance bound the pairs that share its
// tile have reached, as kNoBound - bound (0: none yet), zero at launch; NULL = each pair's
// own bounds only.
// kShare: row_bounds is given (a kernel of its own: the exchange's registers slow long walks
// by 3%).
template <int NP, bool kShare>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1) match_tc_kernel(const __grid_constant__ CUtensorMap tmq,
                                                              const __grid_constant__ CUtensorMap tmt,
                                                              const __grid_constant__ MatchBatchT<NP> batch,
                                                              uint64_t* __restrict__ partials,
                                                              int32_t* __restrict__ tile_cnt,
                                                              int32_t* __restrict__ row_bounds,
                                                              latch_match* __restrict__ out,
                                                              uint32_t* __restrict__ flags) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sA = smem + Smem::a;
    uint8_t* sB = smem + Smem::b;
    uint64_t* sPart = reinterpret_cast<uint64_t*>(smem + Smem::part);
    int32_t* sBound = reinterpret_cast<int32_t*>(smem + Smem::bound);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Smem::bars);
    uint64_t* full = bars;
    uint64_t* empty = bars + kStages;
    uint64_t* a_full = bars + 2 * kStages;
    uint64_t* a_empty = a_full + 1;
    uint64_t* acc_full = a_full + 2;               // [kAccs]
    uint64_t* acc_empty = acc_full + kAccs;        // [kAccs]
    uint64_t* mma_done = acc_empty + kAccs;        // [2]: one per MMA warp
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + Smem::misc);
    volatile int* abort = reinterpret_cast<volatile int*>(smem + Smem::misc + 4);
    volatile int* last_arrival = reinterpret_cast<volatile int*>(smem + Smem::misc + 8);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int rank = static_cast<int>(blockIdx.x & 1);  // in the pair; rank 0's block issues the MMAs
    const int64_t c = blockIdx.x >> 1;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        mbar_init(a_full, 1);
        mbar_init(a_empty, 2);  // both MMA warps commit once per query tile
        for (int i = 0; i < kAccs; ++i) {
            mbar_init(&acc_full[i], 1);
            mbar_init(&acc_empty[i], 2 * kEpiWarps);  // both blocks' epilogue warps (rank 0's barrier)
        }
        mbar_init(&mma_done[0], 1);
        mbar_init(&mma_done[1], 1);
        *abort = 0;
        fence_mbar_init();
    }
    if (warp == 0 && lane == 0) {
        prefetch_tmap(&tmq);
        prefetch_tmap(&tmt);
    }
    if (warp == 2) {
        tmem_alloc_pair(tmem_slot, kTmemCols);
        tc_fence_before();
    }
    for (int r = threadIdx.x; r < kRowsA; r += kThreads) sBound[r] = kNoBound;
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (warp >= 4 && warp < 8) {
        // block scale factors 2^0 in columns kSfaCol..511 of all 128 lanes (warp w may
        // address lane quarter w % 4)
        const uint32_t base = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
#pragma unroll
        for (uint32_t col = kSfaCol; col < kTmemCols; col += 8) tmem_st_32x32b_x8_same(base + col, kScaleOne);
        tmem_st_wait();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // both blocks' barriers and scale factors are there
    tc_fence_after();
    // everything above touched only this pair's shared memory and TMEM
    griddep_wait();
    griddep_launch_dependents();

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            UnitIter it;
            it.init(batch, c);
            int stage = 0;
            uint32_t ring = 0, a_par = 0;
            const uint32_t a_full0 = cluster_addr(smem_u32(a_full), 0), full0 = cluster_addr(smem_u32(full), 0);
            int64_t prev_g = -1;
            for (; !it.done(batch); it.next(batch, c)) {
                const MatchProblem& P = batch.p[it.p];
                const int64_t m = it.m, n = it.n;
                const int64_t g = it.g(batch);
                if (g != prev_g) {
                    if (prev_g >= 0) {
                        if (!mbar_wait(a_empty, a_par, abort)) break;
                        a_par ^= 1;
                    }
                    if (rank == 0) mbar_arrive_expect_tx(a_full, 2 * kChunks * kTileBytes);
                    for (int kc = 0; kc < kChunks; ++kc)
                        tma_load_2d_pair(sA + kc * kTileBytes, &tmq, kc * kChunk,
                                         static_cast<int32_t>(P.q_row0 + m * kRowsQ + rank * kRowsA), a_full0);
                    prev_g = g;
                }
                bool ok = true;
                for (int kc = 0; kc < kChunks; ++kc) {
                    if (!mbar_wait(&empty[stage], ring ^ 1, abort)) {
                        ok = false;
                        break;
                    }
                    if (rank == 0) mbar_arrive_expect_tx(&full[stage], 2 * kStageBytes);
                    tma_load_2d_pair(sB + stage * kStageBytes, &tmt, kc * kChunk,
                                     static_cast<int32_t>(it.t_row0 + n * kColsB + rank * kRowsB),
                                     full0 + 8u * static_cast<uint32_t>(stage));
                    if (++stage == kStages) {
                        stage = 0;
                        ring ^= 1;
                    }
                }
                if (!ok) break;
            }
            if (*abort) {
                // let copies still in flight land before the block exits (their barriers are in
                // the other block, which may have given up: a fixed time)
                const uint64_t t0 = globaltimer();
                while (globaltimer() - t0 < 50000000ull) {
                }
            }
        }
    } else if (warp == 1 || warp == 2) {
        // ---------------- MMA issuers: warp 1 issues the even units, warp 2 the odd ones
        // (a thread's tcgen05.mma waits until the tensor pipe takes it, so a single
        // issuer leaves the pipe idle while it waits on barriers between units; with two,
        // one issuer's waits overlap the other's MMAs).  Unit i uses accumulator i % 2
        // and stages 2 i, 2 i + 1 of the ring; both issuers walk every unit, wait for
        // every query tile and commit a_empty (count 2) at every tile's end. ----------------
        if (rank == 0) {
            // The whole warp walks the units and one elected lane issues: the loop's
            // counters are uniform (shuffles tell the compiler so), so the descriptors live in
            // uniform registers, as the MMA instruction takes them.  Issued from a branch of a
            // single lane with per-thread counters, every MMA took about 60 clocks more.
            const int mine = warp - 1;
            const bool issuer = elect_one();
            RunIter run;
            run.init(batch, c);
            uint32_t a_par = 0;
            // shared-memory descriptors of the first query box and train chunk; the others
            // differ only in the start-address field (bits 0-13: address / 16), so each MMA
            // adds a constant to them
            const uint64_t a_desc0 = umma_desc_sw128(smem_u32(sA));
            const uint64_t b_desc0 = umma_desc_sw128(smem_u32(sB));
            const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
            const uint32_t sfa = tm + kSfaCol, sfb = tm + kSfbCol;
            int i = 0;  // the run's first unit in the block's walk
            bool ok = true;
            for (; ok && !run.done(batch); run.next(batch, c)) {
                if (!wait_all(a_full, a_par, abort)) break;  // every run is a new query tile
                a_par ^= 1;
                const int end = __shfl_sync(0xffffffffu, i + run.len, 0);
                for (int j = i + ((i & 1) ^ mine); ok && j < end; j += 2) {
                    // unit j reads ring positions 2 j and 2 j + 1; its first MMA overwrites D.  The
                    // accumulator comes last: it is what the unit usually waits for, and the
                    // MMAs can follow at once
                    const int acc = j % kAccs;
#pragma unroll
                    for (int kc = 0; kc < kChunks; ++kc) {
                        const int pos = kChunks * j + kc;
                        ok = ok && wait_all(&full[pos % kStages], static_cast<uint32_t>(pos / kStages) & 1u, abort);
                    }
                    ok = ok && wait_all(&acc_empty[acc], static_cast<uint32_t>((j / kAccs) & 1) ^ 1u, abort);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d = tm + static_cast<uint32_t>(acc * kAccStride);
#pragma unroll
                    for (int kc = 0; kc < kChunks; ++kc) {
                        const int stage = (kChunks * j + kc) % kStages;
                        const uint64_t bd = b_desc0 + static_cast<uint64_t>((stage * kStageBytes) >> 4);
                        const uint64_t ad = a_desc0 + static_cast<uint64_t>((kc * kTileBytes) >> 4);
                        // 256 values: K = 96, 96, 64 (48, 48 and 32 bytes: none crosses the swizzle atom)
                        if (issuer) {
                            mma_mxf4_pair(d, ad, bd, kIdesc96, sfa, sfb, kc != 0);
                            mma_mxf4_pair(d, ad + 3, bd + 3, kIdesc96, sfa, sfb, 1);
                            mma_mxf4_pair(d, ad + 6, bd + 6, kIdesc64, sfa, sfb, 1);
                            mma_commit_pair(&empty[stage]);
                            if (kc == kChunks - 1) mma_commit_pair(&acc_full[acc]);
                        }
                        __syncwarp();
                    }
                }
                i = end;
                if (ok && issuer) mma_commit_pair(a_empty);
                __syncwarp();
            }
            // every issued MMA has finished before TMEM is released
            if (issuer) {
                mma_commit_pair(&mma_done[mine]);
                const uint64_t t0 = globaltimer();
                while (!mbar_try_wait(&mma_done[mine], 0) && globaltimer() - t0 < 200000000ull) {
                }
            }
            __syncwarp();
        }
    } else if (warp >= 4) {
        // ---------------- epilogue: kEpiWarps warps; thread = one query row x one
        // group of kColsPerThread accumulator columns.  The walk goes by runs (the
        // consecutive units of one query tile), so the per-unit path touches only
        // counters in registers; the problem table is read where a run ends. ----------------
        const int et = threadIdx.x - 128;  // 0 .. kEpiThreads-1 = cg * kRowsA + row_in_block
        const int quarter = warp & 3;      // TMEM lane quarter this warp may access
        const int cg = (warp - 4) >> 2;    // column group [cg * kColsPerThread, +kColsPerThread)
        const int col0 = cg * kColsPerThread;
        const int row_in_block = quarter * 32 + lane;
        const int row_in_tile = rank * kRowsA + row_in_block;
        const uint32_t acc_empty0 = cluster_addr(smem_u32(acc_empty), 0);
        const uint32_t lane_base = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + static_cast<uint32_t>(col0);
        const float kNegInf = __int_as_float(0xff800000);
        RunIter run;
        run.init(batch, c);
        int acc = 0;           // accumulator of the next unit (unit i uses i % kAccs)
        uint32_t acc_par = 0;  // bit a: the phase parity of accumulator a
        bool aborted = false;  // warp-uniform
        for (; !run.done(batch); run.next(batch, c)) {
            const UnitIter& u = run.u;  // the run's first unit
            uint64_t k1 = kNoKey, k2 = kNoKey;
            // 2 + the value (512 - 2 distance) of the thread's second-best key: the
            // thread's later columns have larger train indices, so one displaces a key
            // of the thread only with a larger value (values are even integers)
            float vown2 = kNegInf;
            // the thread's columns in the problem's last train tile that lie inside the
            // train set (the rest are rows of zeros or of the next problem)
            const int32_t n_last = u.ntl - 1;
            const int32_t lim_last = u.nt - n_last * kColsB - col0;
            // the top-two update from 16 of the thread's columns (group h: columns
            // 16 h .. 16 h + 15) of train tile n.  w = 64 v - j orders the columns by
            // value, then by lower index, and is unique (|v| <= 512, j < 64: exact in
            // fp32); the best two of the 16 by a tournament: (max, min) of each pair,
            // then three rounds of (a1, a2) + (b1, b2) -> (max, second max)
            auto update = [&](const float (&e)[kColsPerThread], int h, int32_t n, float vmin) {
                float t1[kLdCols / 2], t2[kLdCols / 2];
#pragma unroll
                for (int q = 0; q < kLdCols / 2; ++q) {
                    const int j = h * kLdCols + 2 * q;
                    const float wa = fmaf(e[j], 64.0f, -static_cast<float>(j));
                    const float wb = fmaf(e[j + 1], 64.0f, -static_cast<float>(j + 1));
                    t1[q] = fmaxf(wa, wb);
                    t2[q] = fminf(wa, wb);
                }
#pragma unroll
                for (int w = kLdCols / 4; w >= 1; w >>= 1)
#pragma unroll
                    for (int q = 0; q < w; ++q) {
                        const float lo = fminf(t1[q], t1[q + w]);
                        t1[q] = fmaxf(t1[q], t1[q + w]);
                        t2[q] = fmaxf(lo, fmaxf(t2[q], t2[q + w]));
                    }
                const float m1 = t1[0], m2 = t2[0];
                // the two best -> (distance << 32 | index) keys (-inf marks masked
                // columns); the second only where it can still enter (v >= vmin: w >=
                // 64 vmin - 63) or the thread holds fewer than two keys, so that its own
                // second-best stays defined
                const bool want2 = m2 >= fmaf(vmin, 64.0f, -63.0f) || k2 == kNoKey;
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const float mv = b == 0 ? m1 : m2;
                    if (mv != kNegInf && (b == 0 || want2)) {
                        const int32_t w = static_cast<int32_t>(mv);
                        const int32_t j = (-w) & 63;
                        const int32_t d = 256 - ((w + j) >> 7);  // v = (w + j) / 64, d = (512 - v) / 2
                        const uint32_t idx = static_cast<uint32_t>(n) * kColsB + static_cast<uint32_t>(col0 + j);
                        top2_insert_u64((static_cast<uint64_t>(d) << 32) | idx, k1, k2);
                    }
                }
                // the row's bound: the smallest second-best distance of its column groups
                if (k2 != kNoKey) {
                    const int32_t d2 = static_cast<int32_t>(k2 >> 32);
                    vown2 = static_cast<float>(514 - 2 * d2);
                    atomicMin(&sBound[row_in_block], d2);
                }
            };
            const int32_t n_end = u.n + run.len;
            // The first units of a walk are its dearest: as long as a row has met few columns
            // some row of nearly every warp takes an update.  The pairs that walk other parts
            // of the same tile tighten the row's bound together: column group 0 takes the
            // bound loaded a unit ago, publishes a lower one and loads again.  It is a bound
            // like the block's own (two keys at that distance are in some pair's record), so
            // the columns it excludes are in no final top two.
            int32_t seen = 0;
            const int32_t n_share = kShare && cg == 0 ? u.n + kShareUnits : u.n;
            const int32_t grow = static_cast<int32_t>(u.m) * kRowsQ + row_in_tile;
            for (int32_t n = u.n; n < n_end; ++n) {
                // after a failed wait a warp keeps walking the units without work, so that
                // every warp reaches the barriers at the ends of query tiles
                if (!aborted) aborted = !__all_sync(0xffffffffu, mbar_wait(&acc_full[acc], (acc_par >> acc) & 1u, abort));
                if (!aborted) {
                    acc_par ^= 1u << acc;
                    tc_fence_after();
                    if (kShare && n < n_share) {
                        const int32_t own = kNoBound - *static_cast<volatile int32_t*>(&sBound[row_in_block]);
                        if (seen > own) atomicMin(&sBound[row_in_block], kNoBound - seen);
                        if (own > seen) atomicMax(&row_bounds[grow], own);
                        seen = *static_cast<volatile int32_t*>(&row_bounds[grow]);
                    }
                    // the thread's columns (512 - 2 Hamming, exact integers) and the largest
                    // of each half in one round trip; the accumulator is free again as soon
                    // as they are in registers
                    const uint32_t base = lane_base + static_cast<uint32_t>(acc * kAccStride);
                    uint32_t v[kLds][kLdCols];
                    float mx[kLds];
#pragma unroll
                    for (int h = 0; h < kLds; ++h)
                        tmem_ld_red_max_32x32b_x16(base + static_cast<uint32_t>(h * kLdCols), v[h], mx[h]);
                    // some column group of the row holds two keys at distance <= bound, so a
                    // column enters the row's final top two only at a distance <= bound
                    // (equal: when its index is lower than a key's of another group), i.e.
                    // with a value >= 512 - 2 bound, and only above the thread's second best
                    const float vmin = fmaxf(
                        static_cast<float>(512 - 2 * *static_cast<volatile int32_t*>(&sBound[row_in_block])), vown2);
                    tmem_ld_wait();
#pragma unroll
                    for (int h = 0; h < kLds; ++h) tmem_arrived(v[h], mx[h]);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(acc_empty0 + 8u * static_cast<uint32_t>(acc));
                    float e[kColsPerThread];
#pragma unroll
                    for (int h = 0; h < kLds; ++h)
#pragma unroll
                        for (int j = 0; j < kLdCols; ++j) e[h * kLdCols + j] = __uint_as_float(v[h][j]);
                    if (n == n_last && lim_last < kColsPerThread) {
#pragma unroll
                        for (int h = 0; h < kLds; ++h) {
                            mx[h] = kNegInf;
#pragma unroll
                            for (int j = h * kLdCols; j < (h + 1) * kLdCols; ++j) {
                                if (j >= lim_last) e[j] = kNegInf;
                                mx[h] = fmaxf(mx[h], e[j]);
                            }
                        }
                    }
                    // only a group of 16 that reaches the row's bound takes the top-two update; one
                    // vote sends the warp on when none does, which is the usual case
                    static_assert(kLds == 3, "the vote below");
                    if (__any_sync(0xffffffffu, fmax3(mx[0], mx[1], mx[2]) >= vmin)) {
#pragma unroll
                        for (int h = 0; h < kLds; ++h)
                            if (__any_sync(0xffffffffu, mx[h] >= vmin)) update(e, h, n, vmin);
                    }
                }
                if (++acc == kAccs) acc = 0;
            }
            // the run ends where the block leaves its query tile: the column groups of
            // each row meet in shared memory; group 0 writes the row's partial record
            // (slot g + c')
            const MatchProblem& P = batch.p[u.p];
            const int64_t m = u.m;
            const int64_t g = u.g(batch);
            sPart[2 * et] = k1;
            sPart[2 * et + 1] = k2;
            group_sync();  // every thread is past the run's last bound read
            if (cg == 0) {
                sBound[row_in_block] = kNoBound;
#pragma unroll
                for (int q = 1; q < kColGroups; ++q) {
                    top2_insert_u64(sPart[2 * (q * kRowsA + row_in_block)], k1, k2);
                    top2_insert_u64(sPart[2 * (q * kRowsA + row_in_block) + 1], k1, k2);
                }
                if (batch.whole_tiles) {
                    // the block owns the whole tile: the row's two keys are final
                    const int64_t row = m * kRowsQ + row_in_tile;
                    if (row < P.nq) out[P.out0 + row] = final_match(k1, k2, P.k, P.r_milli);
                } else {
                    uint64_t* rec = partials + (u.slot(batch) * kRowsP + row_in_tile) * 2;
                    rec[0] = k1;
                    rec[1] = k2;
                    if (tile_cnt) __threadfence();  // the records are published before the arrival below
                }
            }
            group_sync();  // the shared records are free for the next run
            if (tile_cnt && !batch.whole_tiles) {
                // the last owner of the tile's half to arrive combines its records
                if (et == 0) {
                    int32_t* cnt = &tile_cnt[2 * g + rank];
                    const bool last = atomicAdd(cnt, 1) == tile_owner_count(batch, P, m) - 1;
                    if (last) *cnt = 0;  // no other block touches it again: leave it zero
                    *last_arrival = last;
                }
                group_sync();
                if (*last_arrival && cg == 0) {
                    __threadfence();
                    const int64_t row = m * kRowsQ + row_in_tile;
                    uint64_t f1 = kNoKey, f2 = kNoKey;
                    combine_row(batch, u.p, m, g, row_in_tile, partials, f1, f2);
                    if (row < P.nq) out[P.out0 + row] = final_match(f1, f2, P.k, P.r_milli);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort) atomicOr(flags, kFlagTimeout);
    cluster_sync();  // the other block's MMAs, copies and arrivals are over too
    if (warp == 2) {
        tc_fence_after();
        tmem_dealloc_pair(tmem, kTmemCols);
    }
}

// Combine the partial records of every query row; write one latch_match per query.
template <int NP>
__global__ void match_merge_kernel(const __grid_constant__ MatchBatchT<NP> batch,
                                   const uint64_t* __restrict__ partials, latch_match* __restrict__ out) {
    griddep_wait();
    const int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (q >= batch.queries) return;
    int lo = 0, hi = batch.count - 1;  // problem: largest p with out0 <= q
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (batch.p[mid].out0 <= q) lo = mid; else hi = mid - 1;
    }
    const MatchProblem& P = batch.p[lo];
    const int64_t ql = q - P.out0;
    uint64_t k1 = kNoKey, k2 = kNoKey;
    if (P.ntl > 0) {
        const int64_t m = ql / kRowsQ;
        combine_row(batch, lo, m, P.g0 + m, static_cast<int>(ql % kRowsQ), partials, k1, k2);
    }
    out[q] = final_match(k1, k2, P.k, P.r_milli);
}

// Bits -> E2M1 +-1 values (bit t of a descriptor -> 4-bit value t, kExpRowBytes per
// row); one thread per 32-bit descriptor word.
__global__ void expand_kernel(const uint32_t* __restrict__ in, int64_t nwords, uint4* __restrict__ out) {
    griddep_wait();
    griddep_launch_dependents();
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < nwords) out[i] = expand_word_e2m1(in[i]);
}

// The same for a single problem: the query set, then the train set behind it, and the
// matcher's arrival counters and row bounds cleared, in one launch.  (Two expansions and a memset in
// front of the matcher cost about 2 us more.)
__global__ void expand_two_kernel(const uint32_t* __restrict__ q, int64_t qwords, const uint32_t* __restrict__ t,
                                  int64_t twords, uint4* __restrict__ out, int32_t* __restrict__ counters,
                                  int32_t ncounters, int32_t* __restrict__ bounds, int32_t nbounds) {
    griddep_wait();
    griddep_launch_dependents();
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < ncounters) counters[i] = 0;
    if (i < nbounds) bounds[i] = 0;
    if (i < qwords)
        out[i] = expand_word_e2m1(q[i]);
    else if (i < qwords + twords)
        out[i] = expand_word_e2m1(t[i - qwords]);
}

bool make_map(CUtensorMap* map, const void* base, int64_t rows, int box_rows) {
    const EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {static_cast<cuuint64_t>(kKBytes), static_cast<cuuint64_t>(rows)};
    cuuint64_t strides[1] = {static_cast<cuuint64_t>(kKBytes)};
    cuuint32_t box[2] = {static_cast<cuuint32_t>(kChunk), static_cast<cuuint32_t>(box_rows)};
    cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

}  // namespace

cudaError_t launch_expand(const uint8_t* desc, int64_t n, uint8_t* out, cudaStream_t stream) {
    if (n == 0) return cudaSuccess;
    const int64_t nwords = n * 16;
    const int threads = 256;
    const int64_t grid = (nwords + threads - 1) / threads;
    return launch_chained(expand_kernel, dim3(static_cast<unsigned>(grid)), dim3(threads), 0, stream,
                          reinterpret_cast<const uint32_t*>(desc), nwords, reinterpret_cast<uint4*>(out));
}

int64_t match_tc_tiles(int64_t nq) { return (nq + kRowsQ - 1) / kRowsQ; }

// Fills tiles, unit offsets, query-tile prefixes and the split over the block pairs.  problems[i]
// must have q_row0, t_row0, nq, nt and out0 set.
void plan_match_batch(MatchBatch* b, int count, int64_t max_sms) {
    b->count = count;
    int64_t units = 0, g = 0, queries = 0;
    for (int i = 0; i < count; ++i) {
        MatchProblem& P = b->p[i];
        P.mt = static_cast<int32_t>(match_tc_tiles(P.nq));
        P.ntl = P.nq > 0 ? (P.nt + kColsB - 1) / kColsB : 0;
        P.unit0 = units;
        P.g0 = static_cast<int32_t>(g);
        units += static_cast<int64_t>(P.mt) * P.ntl;
        g += P.mt;
        queries = P.out0 + P.nq > queries ? P.out0 + P.nq : queries;
    }
    b->units = units;
    b->tiles = static_cast<int32_t>(g);
    b->queries = queries;
    const int64_t pairs = max_sms / 2 > 0 ? max_sms / 2 : 1;
    b->grid = units < pairs ? units : pairs;
    // whole query tiles dealt out to the pairs when there are enough of them to balance the
    // pairs (the one that walks a whole tile writes its matches directly, and a tile's walk
    // pays its start-up -- the first units' top-two updates -- once); not when some problem
    // has queries but no train rows (its tiles have no unit).  Tile g goes to pair g mod G:
    // cut into shares problem by problem, the few tiles of a problem fell on the same pairs
    // again and again where their number and G have a common divisor (2 tiles and 76 pairs:
    // on every second pair).  Matching of 1,128 image pairs on GB300, that way and this way:
    // 300 descriptors an image 957 / 269 us, 1,000 1,388 / 833, 2,340 3,150 / 2,181, 5,000
    // 7,507 / 7,014.
    bool whole = g >= kWholeTilesPerPair * b->grid;
    for (int i = 0; i < count; ++i)
        if (b->p[i].nq > 0 && b->p[i].ntl == 0) whole = false;
    b->whole_tiles = whole ? 1 : 0;
}

// Slots g + c' + p (G - 1) (UnitIter): tiles + count (G - 1) of them.
static size_t partial_record_bytes(const MatchBatch& b) {
    const int64_t shares = b.grid > 0 ? b.grid - 1 : 0;
    return static_cast<size_t>(b.tiles + static_cast<int64_t>(b.count) * shares) * kRowsP * 16;
}

size_t match_tc_partial_bytes(const MatchBatch& b) { return partial_record_bytes(b); }

// A counter for each half of a query tile.
size_t match_tc_counter_bytes(int64_t tiles) { return align_up(static_cast<size_t>(tiles) * 8, 256); }

// A launch over `problems` problems with `queries` query rows in total has at most
// queries / 256 + problems query tiles and at most `sms` / 2 block pairs.
size_t match_tc_partial_bound(int64_t queries, int64_t problems, int64_t sms) {
    const int64_t tiles = queries / kRowsQ + problems;
    return static_cast<size_t>(tiles + problems * (sms / 2 + 1)) * kRowsP * 16 + match_tc_counter_bytes(tiles) + 512;
}

size_t match_tc_batch_scratch_bytes(int64_t rows, const MatchBatch& b, int64_t counter_tiles) {
    const size_t exp_bytes = align_up(static_cast<size_t>(rows) * kKBytes, 1024);
    return exp_bytes + match_tc_counter_bytes(counter_tiles) + match_tc_partial_bytes(b) + 256;
}

// The batched layout's arrival counters: [expanded rows][counters][partials].
int32_t* match_tc_batch_counters(void* scratch, int64_t rows) {
    const size_t exp_bytes = align_up(static_cast<size_t>(rows) * kKBytes, 1024);
    return reinterpret_cast<int32_t*>(static_cast<uint8_t*>(scratch) + exp_bytes);
}

// Copies the header and the first b.count problems into the table of capacity NP.
template <int NP>
static void shrink(const MatchBatch& b, MatchBatchT<NP>* o) {
    o->count = b.count;
    o->tiles = b.tiles;
    o->whole_tiles = b.whole_tiles;
    o->units = b.units;
    o->grid = b.grid;
    o->queries = b.queries;
    for (int i = 0; i < b.count; ++i) o->p[i] = b.p[i];
}

template <int NP>
static cudaError_t set_match_attributes() {
    const cudaError_t e =
        cudaFuncSetAttribute(match_tc_kernel<NP, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess || NP > 1) return e;
    return cudaFuncSetAttribute(match_tc_kernel<NP, NP == 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
}

template <int NP>
static cudaError_t launch_match_np(const MatchBatch& full, const CUtensorMap& mapq, const CUtensorMap& mapt,
                                   uint64_t* partials, int32_t* tile_cnt, int32_t* row_bounds, latch_match* out,
                                   uint32_t* flags, cudaStream_t stream) {
    static unsigned long long attr_done = 0;
    {
        const cudaError_t e = once_per_device(&attr_done, set_match_attributes<NP>);
        if (e != cudaSuccess) return e;
    }
    MatchBatchT<NP>* b = new (std::nothrow) MatchBatchT<NP>;
    if (!b) return cudaErrorMemoryAllocation;
    shrink(full, b);
    cudaError_t e = cudaSuccess;
    if (b->units > 0)
        e = launch_chained(row_bounds ? match_tc_kernel<NP, NP == 1> : match_tc_kernel<NP, false>, dim3(static_cast<unsigned>(2 * b->grid)), dim3(kThreads), kSmemBytes,
                           stream, mapq, mapt, *b, partials, tile_cnt, row_bounds, out, flags);
    if (e == cudaSuccess && !tile_cnt && !b->whole_tiles && b->queries > 0) {
        const int threads = 256;
        const int64_t grid = (b->queries + threads - 1) / threads;
        e = launch_chained(match_merge_kernel<NP>, dim3(static_cast<unsigned>(grid)), dim3(threads), 0, stream, *b,
                           partials, out);
    }
    delete b;
    return e;
}

static cudaError_t launch_match_tc_bounds(const MatchBatch& b, const uint8_t* exp, int64_t rows, uint64_t* partials,
                                          int32_t* tile_cnt, int32_t* row_bounds, latch_match* out, uint32_t* flags,
                                          cudaStream_t stream) {
    if (b.queries == 0) return cudaSuccess;
    CUtensorMap mapq, mapt;
    if (b.units > 0 && !(make_map(&mapq, exp, rows, kRowsA) && make_map(&mapt, exp, rows, kRowsB)))
        return cudaErrorInvalidValue;
    // a short launch (at most kFusedUnitsPerPair units per pair) combines each query
    // tile's records itself, which saves the merge launch; a long one leaves them to
    // match_merge_kernel, because the combine at a tile's end (a fence and an atomic
    // round trip per block) holds the epilogue while the MMAs can run only an
    // accumulator's worth ahead.  Neither when some problem has queries but no train
    // rows (its tiles have no unit, so no block visits them).
    bool fused = b.units > 0 && tile_cnt != nullptr && b.units <= kFusedUnitsPerPair * b.grid;
    for (int i = 0; i < b.count; ++i)
        if (b.p[i].nq > 0 && b.p[i].ntl == 0) fused = false;
    if (!fused) tile_cnt = nullptr;
    if (b.count <= 1) return launch_match_np<1>(b, mapq, mapt, partials, tile_cnt, row_bounds, out, flags, stream);
    if (b.count <= 16) return launch_match_np<16>(b, mapq, mapt, partials, tile_cnt, nullptr, out, flags, stream);
    return launch_match_np<kMaxProblems>(b, mapq, mapt, partials, tile_cnt, nullptr, out, flags, stream);
}

cudaError_t launch_match_tc_rows(const MatchBatch& b, const uint8_t* exp, int64_t rows, uint64_t* partials,
                                 int32_t* tile_cnt, latch_match* out, uint32_t* flags, cudaStream_t stream) {
    return launch_match_tc_bounds(b, exp, rows, partials, tile_cnt, nullptr, out, flags, stream);
}

// Scratch: expanded rows (rows x kExpRowBytes), arrival counters, partial records.
// The expanded rows must already be filled (launch_expand).
cudaError_t launch_match_tc_batch(const MatchBatch& b, int64_t rows, int64_t counter_tiles, void* scratch,
                                  latch_match* out, uint32_t* flags, cudaStream_t stream) {
    uint8_t* base = static_cast<uint8_t*>(scratch);
    const size_t exp_bytes = align_up(static_cast<size_t>(rows) * kKBytes, 1024);
    const size_t cnt_bytes = match_tc_counter_bytes(counter_tiles);
    return launch_match_tc_rows(b, base, rows, reinterpret_cast<uint64_t*>(base + exp_bytes + cnt_bytes),
                                reinterpret_cast<int32_t*>(base + exp_bytes), out, flags, stream);
}

static void single_problem(MatchBatch* b, int32_t nq, int32_t nt, int64_t sms, int32_t k = 2, int32_t r = 800) {
    b->p[0].k = k;
    b->p[0].r_milli = r;
    b->p[0].q_row0 = 0;
    b->p[0].t_row0 = nq;
    b->p[0].nq = nq;
    b->p[0].nt = nt;
    b->p[0].out0 = 0;
    plan_match_batch(b, 1, sms);
}

size_t match_tc_scratch_bytes_sms(int64_t sms, int64_t nq, int64_t nt) {
    MatchBatch* b = new MatchBatch;
    single_problem(b, static_cast<int32_t>(nq), static_cast<int32_t>(nt), sms);
    const size_t r = match_tc_batch_scratch_bytes(nq + nt, *b, b->tiles);
    delete b;
    return r;
}

// Row bounds of a single problem (shared by the pairs of a tile), behind its scratch.
static size_t row_bound_bytes(int64_t nq) { return static_cast<size_t>((nq + kRowsQ - 1) / kRowsQ) * kRowsQ * 4; }

size_t match_tc_scratch_bytes(const latch_context* ctx, int64_t nq, int64_t nt) {
    return align_up(match_tc_scratch_bytes_sms(ctx->sm_count, nq, nt), 256) + row_bound_bytes(nq);
}

// `bounds`: the scratch has row_bound_bytes(nq) more, 256-byte aligned behind the rest.
static cudaError_t launch_match_single(const latch_context* ctx, const uint8_t* q, int32_t nq, const uint8_t* t,
                                       int32_t nt, int32_t k, int32_t r_milli, latch_match* out, void* scratch,
                                       bool bounds, cudaStream_t stream) {
    MatchBatch* b = new MatchBatch;
    single_problem(b, nq, nt, ctx->sm_count, k, r_milli);
    uint8_t* base = static_cast<uint8_t*>(scratch);
    int32_t* cnt = match_tc_batch_counters(scratch, static_cast<int64_t>(nq) + nt);
    // only pairs that share a tile have bounds to exchange, and only short walks gain (up to
    // about 500 units).  Without / with the exchange, us per call: 2,340 x 60,000 58.6 / 53.2,
    // 2,340 x 230,000 129.9 / 115.4, 5,000 x 230,000 195.1 / 184.9, 10,000 x 60,000 121.9 /
    // 117.9, 10,000 x 230,000 (500 units) 313.1 / 312.1; 10,000 x 1,048,576 1,128 / 1,156
    // and, with 1.2 pairs per tile, 16,384 x 230,000 448 / 461
    bounds = bounds && !b->whole_tiles && 2 * b->grid > 3 * b->tiles && b->units <= 512 * b->grid;
    int32_t* row_bounds =
        bounds ? reinterpret_cast<int32_t*>(
                     base + align_up(match_tc_scratch_bytes_sms(ctx->sm_count, nq, nt), 256))
               : nullptr;
    cudaError_t e = cudaSuccess;
    if (b->units > 0) {
        const int64_t qwords = static_cast<int64_t>(nq) * kDescWords, twords = static_cast<int64_t>(nt) * kDescWords;
        const int32_t ncounters = 2 * b->tiles;  // fewer than the query words
        const int32_t nbounds = bounds ? b->tiles * kRowsQ : 0;
        const int threads = 256;
        const int64_t work = qwords + twords > nbounds ? qwords + twords : nbounds;
        e = launch_chained(expand_two_kernel, dim3(static_cast<unsigned>((work + threads - 1) / threads)),
                           dim3(threads), 0, stream, reinterpret_cast<const uint32_t*>(q), qwords,
                           reinterpret_cast<const uint32_t*>(t), twords, reinterpret_cast<uint4*>(base), cnt, ncounters,
                           row_bounds, nbounds);
    }
    if (e == cudaSuccess) {
        const size_t exp_bytes = align_up((static_cast<size_t>(nq) + nt) * kKBytes, 1024);
        uint64_t* partials = reinterpret_cast<uint64_t*>(base + exp_bytes + match_tc_counter_bytes(b->tiles));
        e = launch_match_tc_bounds(*b, base, static_cast<int64_t>(nq) + nt, partials, cnt, row_bounds, out, ctx->d_flags,
                                   stream);
    }
    delete b;
    return e;
}

cudaError_t launch_match_tc(const latch_context* ctx, const uint8_t* q, int32_t nq, const uint8_t* t, int32_t nt,
                            int32_t k, int32_t r_milli, latch_match* out, void* scratch, cudaStream_t stream) {
    return launch_match_single(ctx, q, nq, t, nt, k, r_milli, out, scratch, true, stream);
}

}  // namespace latch

// ---------------------------------------------------------------------------
// Allocation-free variant of the tensor-core matcher.
//
// Some callers may not allocate device memory at all: a library embedded in a host
// application that owns every byte of HBM through its own pool (so a cudaMalloc
// from us could fail, or steal memory the application has budgeted), or a
// latency-bound pipeline where cudaMalloc/cudaFree would synchronise the device and
// stall the application's other streams.  hamming_match_noalloc serves them: its
// scratch (expanded operands, per-block partial results, status word)
// lives in the fixed array below, which the CUDA module reserves on every device
// that loads this library for as long as the process lives.
// ---------------------------------------------------------------------------

namespace latch {

constexpr size_t kStaticScratchBytes = size_t(16) << 20;  // 16 MiB
constexpr size_t kStaticFlagBytes = 256;  // status word: zero at load, raised by the kernels, cleared when read

}  // namespace latch

static __device__ __align__(256) uint8_t g_match_static_scratch[latch::kStaticScratchBytes];

#include <mutex>

namespace latch {
namespace {

constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
void* g_static_ptr[kMaxDevices] = {};

// Device address of g_match_static_scratch on `dev` (which must be current).  The
// symbol's host-side name is only a stand-in, so its address is looked up once per
// device and cached.
latch_status static_scratch(int dev, void** out) {
    if (dev < 0 || dev >= kMaxDevices) return fail(nullptr, LATCH_EUNSUPPORTED, "device index %d too large", dev);
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[dev]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_match_static_scratch);
        if (e != cudaSuccess || !p)
            return fail(nullptr, LATCH_ECUDA, "cudaGetSymbolAddress(static scratch): %s", cudaGetErrorString(e));
        g_static_ptr[dev] = p;
    }
    *out = g_static_ptr[dev];
    return LATCH_OK;
}

}  // namespace
}  // namespace latch

extern "C" latch_status hamming_match_noalloc(const uint8_t* d_query, int32_t nq, const uint8_t* d_train,
                                              int32_t nt, int32_t k, float ratio, latch_match* d_out,
                                              latch_stream_t stream) {
    using namespace latch;
    if (nq < 0 || nt < 0) return fail(nullptr, LATCH_EINVAL, "negative size");
    if (k != 1 && k != 2) return fail(nullptr, LATCH_EINVAL, "k = %d must be 1 or 2", k);
    if (!(ratio >= 0.0f && ratio <= 1.0f)) return fail(nullptr, LATCH_EINVAL, "ratio %g not in [0, 1]", ratio);
    if (nq > 0 && (!d_query || !d_out)) return fail(nullptr, LATCH_EINVAL, "NULL query or output");
    if (nq > 0 && nt > 0 && !d_train) return fail(nullptr, LATCH_EINVAL, "NULL train");
    if ((reinterpret_cast<uintptr_t>(d_query) | reinterpret_cast<uintptr_t>(d_train) |
         reinterpret_cast<uintptr_t>(d_out)) & 15)
        return fail(nullptr, LATCH_EINVAL, "descriptor and output pointers must be 16-byte aligned");
    if (nq == 0) return LATCH_OK;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return fail(nullptr, LATCH_ECUDA, "device query: %s", cudaGetErrorString(e));
    const size_t need = match_tc_scratch_bytes_sms(sms, nq, nt) + kStaticFlagBytes;
    if (need > kStaticScratchBytes)
        return fail(nullptr, LATCH_EINVAL,
                    "nq = %d, nt = %d needs %zu bytes of scratch; the static scratch holds %zu (about 60,000 "
                    "descriptors in total)",
                    nq, nt, need, kStaticScratchBytes);
    void* base = nullptr;
    latch_status st = static_scratch(dev, &base);
    if (st != LATCH_OK) return st;
    uint8_t* bytes = static_cast<uint8_t*>(base);
    uint32_t* flags = reinterpret_cast<uint32_t*>(bytes);  // sticky until hamming_match_noalloc_status reads it
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    // launch_match_tc reads only the SM count and the status-word pointer of its context
    latch_context shim;
    shim.device = dev;
    shim.sm_count = sms;
    shim.d_flags = flags;
    const int32_t r_milli = static_cast<int32_t>(std::round(static_cast<double>(ratio) * 1000.0));
    const bool bounds = (need + 255) / 256 * 256 + row_bound_bytes(nq) <= kStaticScratchBytes;  // left out where they do not fit
    e = launch_match_single(&shim, d_query, nq, d_train, nt, k, r_milli, d_out, bytes + kStaticFlagBytes, bounds, cs);
    if (e != cudaSuccess) return fail(nullptr, LATCH_ECUDA, "tensor match launch: %s", cudaGetErrorString(e));
    return LATCH_OK;
}

extern "C" latch_status hamming_match_noalloc_status(void) {
    using namespace latch;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(nullptr, LATCH_ECUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
    void* base = nullptr;
    latch_status st = static_scratch(dev, &base);
    if (st != LATCH_OK) return st;
    e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return fail(nullptr, LATCH_ECUDA, "earlier work failed: %s", cudaGetErrorString(e));
    uint32_t word = 0;
    e = cudaMemcpy(&word, base, sizeof(word), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && word) e = cudaMemset(base, 0, sizeof(word));
    if (e != cudaSuccess) return fail(nullptr, LATCH_ECUDA, "status word: %s", cudaGetErrorString(e));
    if (word & kFlagTimeout)
        return fail(nullptr, LATCH_ETIMEOUT, "a device-side wait of hamming_match_noalloc gave up (word 0x%x)", word);
    if (word) return fail(nullptr, LATCH_EDEVICE, "hamming_match_noalloc status word 0x%x", word);
    return LATCH_OK;
}
