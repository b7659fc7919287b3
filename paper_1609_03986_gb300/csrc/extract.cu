// LATCH descriptor extraction (Sec. 3.1 Eq. 1; Sec. 3.2).
//
// extract_lanes_kernel: one block of 32 warps per SM.  The launch's keypoints are taken
// in batches of up to 32 in their own order, one keypoint per lane; a batch's work is
// 64 chunks of 8 triplets.  Whole batches go round the blocks (batch r G + b to block
// b); the batches of the last, incomplete round are cut into chunk ranges, one per
// block (every block that evaluates a part of a batch builds the batch's windows).
// The block is a pipeline:
//   2 producers    per keypoint one TMA 2-D load of the image tile under its window
//                  (samples outside the image arrive as 0, the border reading) into a
//                  byte ring in shared memory; the box is that of the keypoint's scale
//                  class (at most three box sizes per launch);
//   12 builders    four groups of three warps, a keypoint per group: the 48x48 window
//                  through the per-(scale, bin) table of tile offsets (nearest pixel), a
//                  third of it per warp, into a staging buffer, column of words by column
//                  of words (word (cx, y) of the window at 48 cx + y);
//   16 evaluators  first copy the batch's staged words into tensor memory, window j in
//                  TMEM lane j of every lane quarter, and evaluate the triplets that no
//                  quarter holds from the staged windows, which frees the staging buffer
//                  for the next batch; then evaluate the others by Eq. 1, all 32 lanes on
//                  the same triplet: a patch is two or three columns of words, so as many
//                  8-row TMEM loads bring it, its rows are aligned by funnel shifts, and D1 - D2 =
//                  (sum C1^2 - sum C2^2) - 2 (sum A.C1 - sum A.C2) by __dp4a, all exact in
//                  32-bit integers.  A ballot gives a triplet's bit of all 32 keypoints;
//                  the bits are transposed and leave as whole rows, with the tensor
//                  matcher's expanded row when it is wanted.
//
// Why tensor memory: every lane needs 52.5 window words per triplet.  From shared memory
// (128 bytes per clock per SM) that alone is 840 wavefronts per keypoint, and it bound the
// kernel; tensor memory delivers 128 bytes per clock to each of the four SM partitions,
// so the loads no longer limit and shared memory holds tiles instead of two buffers of
// windows.  512 columns hold 504 of a window's 576 words.  As all four quarters hold the
// same keypoints, each keeps another part of the window, from another byte of a word on,
// and a triplet is evaluated in a quarter that holds its patches, where most of them start
// at a word and need no alignment (25 of 42 shifts are left on the seeded table).
// Instruction issue bounds the kernel: the evaluation's 125 instructions per triplet (56 of
// them dot products) are half of what a keypoint takes, sampling and copying its window, the
// waits and the output the other half.  The four quarters are the four partitions of an SM:
// plan_triplets levels them (to 0.2% of its own costs on the seeded table).
//
// Why a tile per keypoint: no sort by image cell is needed (it cost a memset and two
// launches in front of the extraction), builders need no barrier between keypoints, and at
// the density of photographs (about two keypoints per 32x32 cell) a cell's tile is as
// many bytes per keypoint as the keypoint's own.
//
// Keypoints whose window misses the image read only zeros, and so get the zero
// descriptor; one with a scale index outside the scale table is moved far outside for
// the same result and raises the context's device flag.
//
// Measured (GB300, whole calls back to back; before: windows in shared memory, cell sort):
// 257 keypoints of 321x243 47.2 -> 18.2 us, 2,000 of 640x480 45.2 -> 21.0 us, 10,000 of
// 1920x1080 92.2 -> 50.8 us, the same weighted 190 -> 124 us.
#include <cuda.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <type_traits>

#include "internal.h"
#include "sm103.h"

namespace latch {

namespace {

using namespace sm103;

constexpr int kGroups = 4;              // builder groups, one keypoint each at a time
constexpr int kGroupWarps = 3;
constexpr int kBuildWarps = kGroups * kGroupWarps;  // warps 0-11
constexpr int kProducers = 2;           // warps 12, 13 (14, 15 idle: register splits go by four warps)
constexpr int kEvalWarp0 = 16;          // warps 16-31 evaluate
constexpr int kEvalWarps = 16;
constexpr int kEvalThreads = 32 * kEvalWarps;
constexpr int kThreads = 32 * (kEvalWarp0 + kEvalWarps);
constexpr int kBatch = 32;              // keypoints per batch, one per lane
constexpr int kChunks = kBits / 8;      // chunks of 8 triplets per batch
constexpr int kWordCols = kWin / 4;     // 12 columns of words in a window
constexpr int kBlockWords = 32;         // a builder unit: 4 word columns x 8 rows, one word per lane
constexpr int kBlocks = kWordCols * kWin / kBlockWords;    // 18 units per window
constexpr int kWarpBlocks = kBlocks / kGroupWarps;         // 6 per builder warp
constexpr int kTmemCols = 512;
constexpr int kTmLast = kTmemCols - 8;  // last column an 8-column load may start at
constexpr int kStageWords = kWordCols * kWin + 1;          // odd: the 32 lanes' copies hit 32 banks
constexpr int kOutWords = 33;           // descriptor word w of lane l at 33 w + l
constexpr int kSlots = 8;               // tiles in flight at most, per producer
constexpr int kClasses = 3;             // tile box sizes per launch
// registers per thread after the split (1024 threads x 64 at launch)
constexpr int kBuildRegs = 48, kProducerRegs = 24, kEvalRegs = 80;
static_assert(kGroupWarps * 4 == kWordCols && kWarpBlocks * 8 == kWin, "a builder warp takes four word columns");
static_assert(kBuildWarps * kBuildRegs + 4 * kProducerRegs + kEvalWarps * kEvalRegs <= 32 * 64, "register split");

// What each TMEM lane quarter holds of a window (576 words do not fit its 512 columns):
// `nc` columns of words from byte column `b0` on, rows r0 .. r0 + nr - 1, word (k, r) at
// column k nr + r.  Each quarter lacks a different margin and starts at a different byte
// of a word, and a triplet goes to a quarter that holds its three patches, of these to
// one in which most of them start at a word (plan_triplets).  Those that fit none are
// evaluated from the staged windows in shared memory, before these are given back, by the
// warps of all quarters.
struct Quarter {
    int32_t b0, nc, r0, nr;
};
constexpr int kQuarters = 4;
__host__ __device__ constexpr Quarter quarter_of(int q) {
    return q == 0 ? Quarter{0, 12, 0, 42} : q == 1 ? Quarter{1, 12, 6, 42} : q == 2 ? Quarter{2, 10, 0, 48} : Quarter{7, 10, 0, 48};
}

struct TileClass {
    int32_t reach;      // |offset| of every window sample is at most this
    int32_t tw, th;     // box: bytes per row, rows
};

// Per-launch description of a batch of images (kernel parameters).
template <int NI>
struct ExtractParams {
    CUtensorMap map[NI * kClasses];  // map of image i and class c at i * kClasses + c
    const int32_t* n_dev;    // single-image launches: the keypoint count on the device (n is its bound), or NULL
    int32_t n;               // keypoints in this launch
    int32_t row0;            // row of the launch's first keypoint in the keypoint and output arrays
    int32_t min_batch;       // fewest keypoints per batch (latch_tuning.item_kps)
    int32_t nscales;
    int32_t count;           // images in this launch
    TileClass cls[kClasses];
    int8_t cls_of[LATCH_MAX_SCALES];
    int32_t width[NI], height[NI];
    int32_t first[NI];       // keypoints of the launch before image i
};

// The triplets as the evaluators read them (from constant memory: the index is the
// same for a whole warp, so the fields are unpacked once per warp), quarter by quarter
// and class by class: a word per patch (anchor, companions), bits 0-4 the byte shift
// times 8 (what a funnel shift takes), bits 16-25 the TMEM column of the patch's first
// word; bits 5-13 of the anchor's: the triplet's index.  A triplet's class has bit p set
// when patch p does not start at a word (its rows must be aligned); class 8 (kStaged): it
// is read from the staged windows, its patches' first words being those of the window (word
// (cx, y) at 48 cx + y), because the quarter does not hold it.
constexpr int kTripClasses = 9;
constexpr int kStaged = 8;
struct LaneTriplets {
    uint32_t e[3][kBits];
    int16_t start[kQuarters][kTripClasses + 1];  // first entry of each class
};

// Weights of the 8x8 patch pixels (row-major), a kernel parameter: with the pixel
// loops unrolled, every weight is a constant-bank operand of its multiply-add.
struct PatchWeights {
    int32_t w[64];
};

// The block's share of the launch as items: a batch and its chunk range [ca, cb).
struct Item {
    int32_t kp0, nk;  // first keypoint in the launch, keypoints
    int32_t ca, cb;
};

struct Work {
    int32_t n, bs;       // keypoints of the launch, per batch
    int32_t rounds, items;
    int32_t tail0;       // first batch of the incomplete round
    int32_t u0, u1;      // the block's chunk range in it
    __device__ __forceinline__ Item item(int i) const {
        Item it;
        int batch;
        if (i < rounds) {
            batch = i * static_cast<int>(gridDim.x) + static_cast<int>(blockIdx.x);
            it.ca = 0;
            it.cb = kChunks;
        } else {
            const int t = u0 / kChunks + (i - rounds);
            batch = tail0 + t;
            it.ca = max(u0, t * kChunks) - t * kChunks;
            it.cb = min(u1, (t + 1) * kChunks) - t * kChunks;
        }
        it.kp0 = batch * bs;
        it.nk = min(bs, n - it.kp0);
        return it;
    }
};

// Batch size: 32 (every lane busy) once the launch gives each block a batch or more.
// Below that a block builds bs windows for the chunks it evaluates of them, about
// kBuildCost bs + kEvalCost n / (G bs) clocks, least at bs = sqrt(kEvalCost n /
// (kBuildCost G)).
template <int NI>
__device__ __forceinline__ Work plan_work(const ExtractParams<NI>& prm, int n) {
    constexpr float kCostRatio = 60.0f;  // evaluation of a batch (16k clocks) / building a window (270 clocks)
    Work w;
    const uint32_t G = gridDim.x, b = blockIdx.x;
    w.n = n;
    w.bs = min(kBatch, max(prm.min_batch, static_cast<int>(sqrtf(kCostRatio * static_cast<float>(w.n) / static_cast<float>(G)))));
    const int nb = (w.n + w.bs - 1) / w.bs;
    w.rounds = static_cast<int>(static_cast<uint32_t>(nb) / G);
    w.tail0 = w.rounds * static_cast<int>(G);
    const uint32_t u = static_cast<uint32_t>(nb - w.tail0) * kChunks;  // below 64 G: the products fit 32 bits
    w.u0 = static_cast<int>(b * u / G);
    w.u1 = static_cast<int>((b + 1) * u / G);
    w.items = w.rounds + (w.u1 > w.u0 ? (w.u1 - 1) / kChunks - w.u0 / kChunks + 1 : 0);
    return w;
}

struct LanesSmem {  // static part
    uint32_t bits[2][kBits];                  // entry p of the triplet list: bit j = keypoint j's (double-buffered)
    uint32_t out[kEvalWarps * kOutWords];     // descriptor words of the item
    uint16_t entry[kBits];                    // list entry of each triplet
    uint32_t base[kProducers * kSlots];       // ring byte of the tile's sample at offset (-reach, -reach)
    uint64_t full[kProducers * kSlots], empty[kProducers * kSlots];  // tiles
    uint64_t staged, copied;                  // window staging buffer
    Work work;                                // the evaluators' copy (it would take registers)
    uint32_t tmem;
    int abort;
};

constexpr size_t kFixedSmem = 128 + static_cast<size_t>(kBatch) * kStageWords * 4;
constexpr int kRingBytes = static_cast<int>((227 * 1024 - sizeof(LanesSmem) - kFixedSmem) / 128 * 128);
constexpr size_t kDynSmem = kFixedSmem + kRingBytes;

// ---- evaluation --------------------------------------------------------------------

// Requests the word columns of a patch (its word `f`), 8 rows each, from the lane quarter
// at `tm` (whose column bits are zero) with `nr` rows per word column: two of a patch of
// at most 8 columns that starts at a word, else three.  kClamp: the third may lie past the
// last column (the patch does not need it then).
template <bool kThree, bool kClamp = false>
__device__ __forceinline__ void request(uint32_t (&w)[3][8], uint32_t f, uint32_t tm, uint32_t nr) {
    const uint32_t a = (f >> 16) + tm;
    tmem_ld_32x32b_x8(a, w[0]);
    tmem_ld_32x32b_x8(a + nr, w[1]);
    if constexpr (kThree) tmem_ld_32x32b_x8(kClamp ? min(a + 2 * nr, tm + kTmLast) : a + 2 * nr, w[2]);
}

// After tmem_ld_wait(): pins the loaded registers behind the wait (the compiler may move
// plain arithmetic above it).
template <bool kThree, int kRows>
__device__ __forceinline__ void arrive(uint32_t (&w)[3][8]) {
#pragma unroll
    for (int k = 0; k < (kThree ? 3 : 2); ++k)
#pragma unroll
        for (int r = 0; r < kRows; ++r) asm volatile("" : "+r"(w[k][r]));
}

// Aligns the rows: w[0][r] = pixels 0..3 and w[1][r] = pixels 4..7 of the patch row.
template <int kRows>
__device__ __forceinline__ void align(uint32_t (&w)[3][8], uint32_t f) {
#pragma unroll
    for (int r = 0; r < kRows; ++r) {  // (a funnel shift takes 5 bits of f)
        w[0][r] = __funnelshift_r(w[0][r], w[1][r], f);
        w[1][r] = __funnelshift_r(w[1][r], w[2][r], f);
    }
}

// The patch whose first word is `f`, aligned, from a staged window: two word columns, and a
// third where the patch reaches into it.
template <int kRows>
__device__ __forceinline__ void load_staged(uint32_t (&w)[3][8], uint32_t f, const uint32_t* window) {
    const uint32_t* x = window + (f >> 16);
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        w[0][r] = x[r];
        w[1][r] = x[kWin + r];
        w[2][r] = 0;
    }
    if ((f & 31u) > 64 - 8 * kRows) {
#pragma unroll
        for (int r = 0; r < kRows; ++r) w[2][r] = x[2 * kWin + r];
    }
    align<kRows>(w, f);
}

// The words of one triplet (LaneTriplets).
struct Words {
    uint32_t a, c1, c2;
    __device__ __forceinline__ int index() const { return static_cast<int>((a >> 5) & 511u); }
};
__device__ __forceinline__ Words words_of(const LaneTriplets& tt, int p) {
    return Words{tt.e[0][p], tt.e[1][p], tt.e[2][p]};
}

// sum A.C and sum C^2 over the 7 patch rows (pixel 8 of a row is not in the patch: masked
// in C, and A's is multiplied by it).
__device__ __forceinline__ void dot7(const uint32_t (&a)[3][8], const uint32_t (&c)[3][8], uint32_t& ac, uint32_t& cc) {
    ac = 0;
    cc = 0;
#pragma unroll
    for (int r = 0; r < 7; ++r) {
        const uint32_t hi = c[1][r] & 0x00ffffffu;
        ac = __dp4a(a[0][r], c[0][r], ac);
        cc = __dp4a(c[0][r], c[0][r], cc);
        ac = __dp4a(a[1][r], hi, ac);
        cc = __dp4a(hi, hi, cc);
    }
}

// D1 > D2 from the sums: D1 - D2 = sum C1^2 - sum C2^2 - 2 (sum A.C1 - sum A.C2).
__device__ __forceinline__ bool farther(uint32_t ac1, uint32_t cc1, uint32_t ac2, uint32_t cc2) {
    return (static_cast<int>(cc1) - static_cast<int>(cc2)) - 2 * (static_cast<int>(ac1) - static_cast<int>(ac2)) > 0;
}

// Eq. 1 for every fourth entry (those = `mine` mod 4) of one class' list entries [lo, hi):
// bits[p] = the bits of all lanes' keypoints.  The next triplet's first companion is
// requested under the second half of this one, its anchor at the end of it (the registers
// are free then): the other warps of the partition cover what is left of the wait.
template <int kClass>
__device__ __forceinline__ void eval_class(const LaneTriplets& tt, int lo, int hi, int mine, uint32_t tm, uint32_t nr,
                                           uint32_t* bits, int lane) {
    constexpr bool kA = kClass & 1, k1 = kClass & 2, k2 = kClass & 4;
    int p = lo + ((mine - lo) & 3);
    if (p >= hi) return;
    const int first = p;
    uint32_t a[3][8], c[3][8], d[3][8];
    Words f = words_of(tt, p);
    request<k1>(c, f.c1, tm, nr);
    request<kA>(a, f.a, tm, nr);
#pragma unroll 1
    for (; p < hi; p += 4) {
        const Words g = words_of(tt, p + 4 < hi ? p + 4 : first);
        tmem_ld_wait();
        arrive<k1, 7>(c);
        arrive<kA, 7>(a);
        request<k2>(d, f.c2, tm, nr);
        if constexpr (kA) align<7>(a, f.a);
        if constexpr (k1) align<7>(c, f.c1);
        uint32_t ac1, cc1, ac2, cc2;
        dot7(a, c, ac1, cc1);
        tmem_ld_wait();
        arrive<k2, 7>(d);
        request<k1>(c, g.c1, tm, nr);
        if constexpr (k2) align<7>(d, f.c2);
        dot7(a, d, ac2, cc2);
        request<kA>(a, g.a, tm, nr);
        const uint32_t b = __ballot_sync(0xffffffffu, farther(ac1, cc1, ac2, cc2));
        if (lane == 0) bits[p] = b;
        f = g;
    }
    tmem_ld_wait();
}

// Eq. 1 with weighted 8x8 patches (Sec. 3.2, weighing pixels in LATCH patches):
// D1 - D2 = sum w (C1 - C2)(C1 + C2 - 2 A), exact in int32 (|w (C1 - C2)(C1 + C2 - 2 A)|
// <= 255 * 255^2 per pixel, 64 pixels).
__device__ __forceinline__ bool farther_weighted(const uint32_t (&a)[3][8], const uint32_t (&c)[3][8],
                                                 const uint32_t (&d)[3][8], const PatchWeights& pw) {
    int acc = 0;
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t sel = 0x4440u | static_cast<uint32_t>(j & 3);
            const int av = static_cast<int>(__byte_perm(a[j >> 2][r], 0u, sel));
            const int cv = static_cast<int>(__byte_perm(c[j >> 2][r], 0u, sel));
            const int dv = static_cast<int>(__byte_perm(d[j >> 2][r], 0u, sel));
            acc += pw.w[r * 8 + j] * ((cv - dv) * (cv + dv - 2 * av));
        }
    return acc > 0;
}

// Eq. 1 for one triplet of any class of the quarter, not pipelined.
template <bool kWeighted>
__device__ __forceinline__ bool eval_held(const Words& f, uint32_t tm, uint32_t nr, const PatchWeights& pw) {
    constexpr int kRows = kWeighted ? 8 : 7;
    uint32_t a[3][8], c[3][8], d[3][8];
    request<true, true>(a, f.a, tm, nr);
    request<true, true>(c, f.c1, tm, nr);
    tmem_ld_wait();
    arrive<true, kRows>(a);
    arrive<true, kRows>(c);
    if constexpr (!kWeighted) request<true, true>(d, f.c2, tm, nr);
    align<kRows>(a, f.a);
    align<kRows>(c, f.c1);
    if constexpr (kWeighted) request<true, true>(d, f.c2, tm, nr);
    uint32_t ac1 = 0, cc1 = 0, ac2, cc2;
    if constexpr (!kWeighted) dot7(a, c, ac1, cc1);
    tmem_ld_wait();
    arrive<true, kRows>(d);
    align<kRows>(d, f.c2);
    if constexpr (kWeighted) return farther_weighted(a, c, d, pw);
    dot7(a, d, ac2, cc2);
    return farther(ac1, cc1, ac2, cc2);
}

// The same from the lane's staged window.  Its 42 to 63 shared-memory loads per triplet
// (128 bytes per clock per SM, for all four quarters) and its instructions take about equally
// long, some 250 clocks, and the builders wait for it: it serves the triplets that fit no
// quarter, about 40 of 512 of a random table.  It is what bounds tables of far-apart patches:
// 10,000 keypoints, every triplet across the window's diagonal, 72 us (the seeded table 51).
// Before, quarter 0 alone evaluated them, its missing rows selected from shared memory: 218
// and 53 us.
template <bool kWeighted>
__device__ __forceinline__ bool eval_staged(const Words& f, const uint32_t* window, const PatchWeights& pw) {
    constexpr int kRows = kWeighted ? 8 : 7;
    uint32_t a[3][8], c[3][8], d[3][8];
    load_staged<kRows>(a, f.a, window);
    load_staged<kRows>(c, f.c1, window);
    load_staged<kRows>(d, f.c2, window);
    if constexpr (kWeighted) return farther_weighted(a, c, d, pw);
    uint32_t ac1, cc1, ac2, cc2;
    dot7(a, c, ac1, cc1);
    dot7(a, d, ac2, cc2);
    return farther(ac1, cc1, ac2, cc2);
}

// Every fourth of the list entries [lo, hi) whose triplets lie in [t0, t1), one at a time:
// weighted patches, a part of the chunks, and (kFromStage) the staged class.
template <bool kWeighted, bool kFromStage>
__device__ __forceinline__ void eval_entries(const LaneTriplets& tt, const PatchWeights& pw, int lo, int hi, int mine,
                                             int t0, int t1, uint32_t tm, uint32_t nr, const uint32_t* window,
                                             uint32_t* bits, int lane) {
#pragma unroll 1
    for (int p = lo + ((mine - lo) & 3); p < hi; p += 4) {
        const Words f = words_of(tt, p);
        const int t = f.index();
        if (t < t0 || t >= t1) continue;
        bool bit;
        if constexpr (kFromStage)
            bit = eval_staged<kWeighted>(f, window, pw);
        else
            bit = eval_held<kWeighted>(f, tm, nr, pw);
        const uint32_t b = __ballot_sync(0xffffffffu, bit);
        if (lane == 0) bits[p] = b;
    }
}

// The warp's share (`mine` of 4) of the triplets [t0, t1) that its quarter holds.
template <bool kWeighted>
__device__ __forceinline__ void eval_quarter(const LaneTriplets& tt, const PatchWeights& pw, int quarter, int mine,
                                             int t0, int t1, uint32_t tm, uint32_t nr, uint32_t* bits, int lane) {
    const int16_t* start = tt.start[quarter];
    if (!kWeighted && t1 - t0 == kBits) {
        eval_class<0>(tt, start[0], start[1], mine, tm, nr, bits, lane);
        eval_class<1>(tt, start[1], start[2], mine, tm, nr, bits, lane);
        eval_class<2>(tt, start[2], start[3], mine, tm, nr, bits, lane);
        eval_class<3>(tt, start[3], start[4], mine, tm, nr, bits, lane);
        eval_class<4>(tt, start[4], start[5], mine, tm, nr, bits, lane);
        eval_class<5>(tt, start[5], start[6], mine, tm, nr, bits, lane);
        eval_class<6>(tt, start[6], start[7], mine, tm, nr, bits, lane);
        eval_class<7>(tt, start[7], start[kStaged], mine, tm, nr, bits, lane);
    } else {
        eval_entries<kWeighted, false>(tt, pw, start[0], start[kStaged], mine, t0, t1, tm, nr, nullptr, bits, lane);
    }
}

// Copies kRows rows (from row r of the quarter on) of the lane's staged window into the
// quarter, along the word columns; each word is joined from two of the window's.
template <int kRows>
__device__ __forceinline__ void copy_rows(const uint32_t* window, const Quarter& Q, int r, uint32_t tm) {
    static_assert(kRows == 12 || kRows == 6, "row split");
    const int c0 = Q.b0 >> 2;
    const uint32_t sh = 8u * static_cast<uint32_t>(Q.b0 & 3);
    const uint32_t* src = window + c0 * kWin + Q.r0 + r;
    uint32_t w[kRows];
#pragma unroll
    for (int q = 0; q < kRows; ++q) w[q] = src[q];
#pragma unroll 2
    for (int k = 0; k < Q.nc; ++k) {
        // (past the last word column: bytes that no patch uses)
        src += c0 + k + 1 < kWordCols ? kWin : 0;
        uint32_t v[kRows];
#pragma unroll
        for (int q = 0; q < kRows; ++q) {
            const uint32_t n = src[q];
            v[q] = __funnelshift_r(w[q], n, sh);
            w[q] = n;
        }
        const uint32_t to = tm + static_cast<uint32_t>(k * Q.nr + r);
        if constexpr (kRows == 12) {
            tmem_st_32x32b_x8(to, v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]);
            tmem_st_32x32b_x4(to + 8, v[8], v[9], v[10], v[11]);
        } else {
            tmem_st_32x32b_x4(to, v[0], v[1], v[2], v[3]);
            tmem_st_32x32b_x2(to + 4, v[4], v[5]);
        }
    }
}

template <int NI, bool kWeighted>
__global__ void __launch_bounds__(kThreads, 1) extract_lanes_kernel(
    const __grid_constant__ ExtractParams<NI> prm, const __grid_constant__ LaneTriplets tt,
    const __grid_constant__ PatchWeights pw, const latch_keypoint* __restrict__ kps,
    const uint2* __restrict__ toff, uint8_t* __restrict__ out, uint8_t* __restrict__ exp_out,
    uint32_t* __restrict__ flags) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ LanesSmem S;
    uint8_t* ring = smem_raw + (-smem_u32(smem_raw) & 127u);
    uint32_t* s_stage = reinterpret_cast<uint32_t*>(ring + kRingBytes);  // [kBatch][kStageWords]
    const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    volatile int* abort = &S.abort;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kProducers * kSlots; ++s) {
            mbar_init(&S.full[s], 1);
            mbar_init(&S.empty[s], kGroupWarps);
        }
        mbar_init(&S.staged, kBuildWarps);
        mbar_init(&S.copied, kEvalWarps);
        S.abort = 0;
        fence_mbar_init();
    }
    if (warp == kEvalWarp0) {
        tmem_alloc(&S.tmem, kTmemCols);
        tc_fence_before();
    }
    if (warp == kBuildWarps && lane < min(kClasses * prm.count, 32)) prefetch_tmap(&prm.map[lane]);
    __syncthreads();  // the last block-wide barrier: the roles meet only at mbarriers from here on
    tc_fence_after();
    // everything above and, in the evaluators, the triplet list touches only parameters,
    // shared memory and TMEM: it runs under the previous kernel's end
    auto start = [&]() {
        Work w;
        if (!prm.n_dev) w = plan_work(prm, prm.n);
        griddep_wait();
        griddep_launch_dependents();
        if (prm.n_dev) w = plan_work(prm, min(prm.n, max(0, *prm.n_dev)));
        return w;
    };

    if (warp < kBuildWarps) {
        // ================= builders =================
        set_max_regs_dec<kBuildRegs>();
        const Work work = start();
        const int g = warp / kGroupWarps, wi = warp - g * kGroupWarps;
        // the group takes the keypoints whose sequence number in the block is g mod kGroups
        const latch_keypoint* kp_launch = kps + prm.row0;
        // offset tables of an item's keypoints, lane = keypoint
        auto load_tables = [&](const Item& it) {
            if (lane >= it.nk) return 0u;
            const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(kp_launch + it.kp0 + lane) + 2);
            const uint32_t s = (w >> 8) & 0xffu;
            return (s < static_cast<uint32_t>(prm.nscales) ? s * kBins : 0u) + (w & (kBins - 1));
        };
        uint2 tab[kWarpBlocks];
        const uint2* tab_lane = toff + wi * kBlockWords + lane;  // the lane's word of unit q: kGroupWarps q units on
        // the lane's word of unit q: word column 4 wi + lane % 4, row 8 q + lane / 4
        const int cx = 4 * wi + (lane & 3), yl = lane >> 2;
        const uint32_t ring_addr = smem_u32(ring);
        const uint32_t stage_addr = smem_u32(s_stage) + 4u * static_cast<uint32_t>(cx * kWin + yl);
        int seq0 = 0;        // sequence number of the item's first keypoint
        bool ok = true;
        bool primed = false; // tab holds the group's next keypoint
        Item it = work.item(0);
        uint32_t tables = work.items > 0 ? load_tables(it) : 0u;
        for (int i = 0; i < work.items && ok; ++i) {
            // the next item's tables are on their way while this one is built
            const Item ni = work.item(i + 1);
            const uint32_t next_tables = i + 1 < work.items ? load_tables(ni) : 0u;
            const int j0 = (g - seq0) & (kGroups - 1);
            if (!primed && j0 < it.nk) {
                const uint32_t t = __shfl_sync(0xffffffffu, tables, j0);
#pragma unroll
                for (int q = 0; q < kWarpBlocks; ++q)
                    tab[q] = __ldg(tab_lane + t * (kBlocks * kBlockWords) + q * (kGroupWarps * kBlockWords));
                primed = true;
            }
            // the staging buffer is free once the evaluators have copied item i - 1
            if (i > 0) ok = mbar_wait_sleep<200>(&S.copied, (i - 1) & 1, abort);
            for (int j = j0; ok && j < it.nk; j += kGroups) {
                // the group's next keypoint: in this item or the first in the next one
                const bool same = j + kGroups < it.nk;
                const int nj = same ? j + kGroups : (g - seq0 - it.nk) & (kGroups - 1);
                const bool more = same || (i + 1 < work.items && nj < ni.nk);
                const uint32_t nt = __shfl_sync(0xffffffffu, same ? tables : next_tables, nj);
                const int seq = (seq0 + j) / kProducers, slot = (g & (kProducers - 1)) * kSlots + seq % kSlots;
                ok = mbar_wait_sleep<64>(&S.full[slot], static_cast<uint32_t>(seq / kSlots) & 1u, abort);
                if (!ok) break;
                const uint32_t t = ring_addr + S.base[slot];
                const uint32_t to = stage_addr + 4u * kStageWords * static_cast<uint32_t>(j);
                const uint2* next_tab = tab_lane + nt * (kBlocks * kBlockWords);
#pragma unroll
                for (int q = 0; q < kWarpBlocks; ++q) {
                    const uint2 e = tab[q];
                    const uint32_t b0 = lds_u8(t + (e.x & 0xffffu)), b1 = lds_u8(t + (e.x >> 16));
                    const uint32_t b2 = lds_u8(t + (e.y & 0xffffu)), b3 = lds_u8(t + (e.y >> 16));
                    // lands during the rest of this keypoint (the last keypoint's is not used)
                    tab[q] = __ldg(next_tab + q * (kGroupWarps * kBlockWords));
                    const uint32_t v = __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
                    sts_u32(to + 32u * q, v);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.empty[slot]);  // the tile is free for this warp
                primed = more;
            }
            __syncwarp();
            if (ok && lane == 0) mbar_arrive(&S.staged);
            seq0 += it.nk;
            it = ni;
            tables = next_tables;
        }
        if (!ok && lane == 0) atomicOr(flags, kFlagTimeout);
        return;
    }

    if (warp < kEvalWarp0) {
        set_max_regs_dec<kProducerRegs>();
        const int pw = warp - kBuildWarps;
        if (pw >= kProducers) return;
        const Work work = start();
        // ================= producers: tiles into byte rings =================
        // Producer pw takes the keypoints whose sequence number in the block is pw mod
        // kProducers, and has its part of the ring and of the slots.
        // tiles [oldest, seq) are in the ring in order; lane s remembers where slot s's tile
        // starts.  [head, limit): the free bytes behind the latest tile, up to the oldest
        // tile or the ring's end.  The warp's own chain of instructions is what limits how
        // fast it can issue, so everything per keypoint is prepared 32 at a time.
        constexpr int kPart = kRingBytes / kProducers / 128 * 128;
        uint8_t* part = ring + pw * kPart;
        uint64_t *full = S.full + pw * kSlots, *empty = S.empty + pw * kSlots;
        int head = 0, limit = kPart, my_start = 0, oldest = 0, seq = 0, seq0 = 0;
        bool ok = true;
        for (int i = 0; i < work.items && ok; ++i) {
            const Item it = work.item(i);
            int bytes = 0, tx = 0, ty = 0, ox = 0;
            const CUtensorMap* map = nullptr;
            if (lane < it.nk) {
                const int k = it.kp0 + lane;
                const latch_keypoint kp = kps[prm.row0 + k];
                int lo = 0, hi = prm.count - 1;  // image: largest i with first[i] <= k
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (prm.first[mid] <= k) lo = mid; else hi = mid - 1;
                }
                const bool bad = kp.scale_idx >= prm.nscales;
                if (bad) atomicOr(flags, kFlagBadScale);
                const int c = prm.cls_of[bad ? 0 : kp.scale_idx];
                const int r = prm.cls[c].reach;
                // a keypoint 1024 pixels outside sees as little of the image as any further out
                const int x = bad ? -1024 : min(max(kp.x, -1024), prm.width[lo] + 1024);
                const int y = min(max(kp.y, -1024), prm.height[lo] + 1024);
                tx = (x - r) & ~15;  // TMA: the first byte of a row is a multiple of 16
                ty = y - r;
                ox = x - r - tx;
                bytes = prm.cls[c].tw * prm.cls[c].th;
                map = &prm.map[lo * kClasses + c];
            }
            const int j0 = (pw - seq0) & (kProducers - 1);
            int size = __shfl_sync(0xffffffffu, bytes, j0);
            for (int j = j0; j < it.nk; j += kProducers) {
                size = (size + 127) & ~127;
                while (seq - oldest == kSlots || head + size > limit) {
                    if (seq - oldest < kSlots && limit == kPart && oldest < seq) {
                        head = 0;  // go round: free up to the oldest tile
                        limit = __shfl_sync(0xffffffffu, my_start, oldest % kSlots);
                        continue;
                    }
                    ok = __all_sync(0xffffffffu, mbar_wait_sleep<20>(&empty[oldest % kSlots],
                                                                     static_cast<uint32_t>(oldest / kSlots) & 1u, abort));
                    if (!ok) break;
                    if (++oldest == seq) {
                        head = 0;
                        limit = kPart;
                    } else {
                        const int tail = __shfl_sync(0xffffffffu, my_start, oldest % kSlots);
                        limit = tail >= head ? tail : kPart;
                    }
                }
                if (!ok) break;
                const int slot = seq % kSlots;
                if (lane == slot) my_start = head;
                if (lane == j) {
                    S.base[pw * kSlots + slot] = static_cast<uint32_t>(pw * kPart + head + ox);
                    mbar_arrive_expect_tx(&full[slot], static_cast<uint32_t>(bytes));
                    tma_load_2d(part + head, map, tx, ty, &full[slot]);
                }
                head += size;
                ++seq;
                size = __shfl_sync(0xffffffffu, bytes, j + kProducers);
            }
            seq0 += it.nk;
        }
        if (!ok) {  // let the copies in flight land before the block's memory is released
            if (lane == 0) {
                atomicOr(flags, kFlagTimeout);
                const uint64_t t0 = globaltimer();
                for (int s = seq > kSlots ? seq - kSlots : 0; s < seq; ++s)
                    while (!mbar_try_wait(&full[s % kSlots], static_cast<uint32_t>(s / kSlots) & 1u) &&
                           globaltimer() - t0 < 200000000ull) {
                    }
            }
            __syncwarp();
        }
        return;
    }

    // ================= evaluators =================
    set_max_regs_inc<kEvalRegs>();
    const int cw = warp - kEvalWarp0;
    const int ct = cw * 32 + lane;  // 0 .. kEvalThreads - 1
    const int quarter = warp & 3;   // TMEM lane quarter this warp may access
    // uniform over the warp, and known to be (shuffles), as TMEM addresses have to be
    const uint32_t tm = __shfl_sync(0xffffffffu, S.tmem, 0) + (static_cast<uint32_t>(quarter * 32) << 16);
    const Quarter Q = quarter_of(quarter);
    const uint32_t nr = static_cast<uint32_t>(Q.nr);
    {   // the triplet list's positions (only the evaluators use them)
        S.entry[(tt.e[0][ct] >> 5) & 511u] = static_cast<uint16_t>(ct);
        const Work w = start();
        if (ct == 0) S.work = w;
        bar_sync_id(5, kEvalThreads);
    }
    bool dead = false;  // after a failed wait: barriers without work, so that every warp reaches them
    for (int i = 0; i < S.work.items; ++i) {
        const Item it = S.work.item(i);
        uint32_t* bits = S.bits[i & 1];
        const int mine = (warp >> 2) & 3;
        const int t0 = __shfl_sync(0xffffffffu, 8 * it.ca, 0), t1 = __shfl_sync(0xffffffffu, 8 * it.cb, 0);
        if (!dead) dead = !__all_sync(0xffffffffu, mbar_wait_sleep<100>(&S.staged, i & 1, abort));
        if (!dead) {
            // copy the staged windows (lane = keypoint) into this quarter, 12 rows per warp
            tc_fence_after();
            const int r0 = 12 * (cw >> 2);
            if (r0 + 12 <= Q.nr)
                copy_rows<12>(s_stage + lane * kStageWords, Q, r0, tm);
            else
                copy_rows<6>(s_stage + lane * kStageWords, Q, r0, tm);
            tmem_st_wait();
            // ---- Eq. 1: this warp's share of the triplets that are read from the staged windows ----
            const int16_t* start = tt.start[quarter];
            eval_entries<kWeighted, true>(tt, pw, start[kStaged], start[kTripClasses], mine, t0, t1, tm, nr,
                                          s_stage + lane * kStageWords, bits, lane);
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.copied);
        }
        tc_fence_before();
        bar_sync_id(1 + quarter, 128);
        tc_fence_after();
        const int n = it.cb - it.ca;
        // ---- and of those that the quarter holds, in the chunks [ca, cb) ----
        if (!dead) eval_quarter<kWeighted>(tt, pw, quarter, mine, t0, t1, tm, nr, bits, lane);
        tc_fence_before();
        // all bits of the item are there, and (the buffers alternate) everybody is done with
        // the other buffer
        bar_sync_id(5, kEvalThreads);
        tc_fence_after();
        uint32_t* so = S.out;
        {   // warp cw: triplets 32 cw .. 32 cw + 31 of every keypoint, transposed: lane = keypoint
            uint32_t v = bits[S.entry[32 * cw + lane]];
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                constexpr uint32_t kMask[5] = {0x55555555u, 0x33333333u, 0x0f0f0f0fu, 0x00ff00ffu, 0x0000ffffu};
                const uint32_t m = kMask[o == 16 ? 4 : o == 8 ? 3 : o == 4 ? 2 : o == 2 ? 1 : 0];
                const uint32_t u = __shfl_xor_sync(0xffffffffu, v, o);
                v = (lane & o) ? (v & ~m) | ((u >> o) & m) : (v & m) | ((u << o) & ~m);
            }
            so[cw * kOutWords + lane] = v;  // word cw of the lane's descriptor
        }
        bar_sync_id(5, kEvalThreads);
        if (dead) continue;
        const size_t row = static_cast<size_t>(prm.row0) + it.kp0;
        if (n == kChunks) {
            // whole rows: 4 threads per 64-byte descriptor, 16 per 256-byte expanded row
            if (ct < 4 * it.nk) {
                const int r = ct >> 2, q = ct & 3;
                reinterpret_cast<uint4*>(out + row * kDescBytes)[ct] =
                    make_uint4(so[(4 * q) * kOutWords + r], so[(4 * q + 1) * kOutWords + r],
                               so[(4 * q + 2) * kOutWords + r], so[(4 * q + 3) * kOutWords + r]);
            }
            if (exp_out && ct < 16 * it.nk)
                reinterpret_cast<uint4*>(exp_out + row * kExpRowBytes)[ct] =
                    expand_word_e2m1(so[(ct & 15) * kOutWords + (ct >> 4)]);
        } else {
            // a part of the batch: descriptor bytes [ca, cb), expanded bytes [8 ca, 8 cb)
            const uint8_t* sb = reinterpret_cast<const uint8_t*>(so);
            for (int x = ct; x < n * it.nk; x += kEvalThreads) {
                const int r = x / n, c = it.ca + x - r * n;
                const uint32_t byte = sb[4 * ((c >> 2) * kOutWords + r) + (c & 3)];
                out[(row + r) * kDescBytes + c] = static_cast<uint8_t>(byte);
                if (exp_out)
                    reinterpret_cast<uint32_t*>(exp_out + (row + r) * kExpRowBytes)[c] = expand_byte_e2m1(byte);
            }
        }
    }
    if (dead && lane == 0) atomicOr(flags, kFlagTimeout);
    tc_fence_before();
    bar_sync_id(5, kEvalThreads);
    if (warp == kEvalWarp0) {
        tc_fence_after();
        tmem_dealloc(S.tmem, kTmemCols);
    }
}

}  // namespace

// Host-side precomputation for the extraction kernel ------------------------------

int window_reach(double scale) {
    // corner of the window: |a|, |e| <= 24, so |offset| <= 24 sqrt(2) scale, rounded
    return static_cast<int>(std::floor(24.0 * std::sqrt(2.0) * scale + 0.5 + 1e-6));
}

// Tile box of a reach: the window's samples at any column of a 16-byte granule.  Rows of
// an odd number of 16-byte granules start in 8 different bank groups (an even number
// gives 2 or 4), so the gathers along a rotated window collide less.
static TileClass tile_class(int reach) {
    TileClass t;
    t.reach = reach;
    t.tw = (2 * reach + 1 + 15 + 15) / 16 * 16;
    if ((t.tw / 16) % 2 == 0) t.tw += 16;
    t.th = 2 * reach + 1;
    return t;
}

// At most kClasses box sizes for the scale table: the scales sorted by reach are cut into
// groups, each served by its largest box, so that the bytes over the table are fewest.
static void tile_classes(const double* scales, int n, TileClass (&cls)[kClasses], int8_t (&cls_of)[LATCH_MAX_SCALES]) {
    int order[LATCH_MAX_SCALES];
    for (int i = 0; i < n; ++i) order[i] = i;
    for (int i = 1; i < n; ++i)
        for (int j = i; j > 0 && scales[order[j]] < scales[order[j - 1]]; --j) {
            const int t = order[j];
            order[j] = order[j - 1];
            order[j - 1] = t;
        }
    auto box = [&](int hi) { return tile_class(window_reach(scales[order[hi]])); };  // of sorted scale hi
    int64_t best = -1;
    int cut1 = n, cut2 = n;  // groups [0, cut1), [cut1, cut2), [cut2, n); empty ones allowed
    for (int a = 1; a <= n; ++a)
        for (int b = a; b <= n; ++b) {
            int64_t bytes = 0;
            const int ends[3] = {a, b, n};
            for (int c = 0, from = 0; c < 3; from = ends[c], ++c)
                if (ends[c] > from) {
                    const TileClass t = box(ends[c] - 1);
                    bytes += static_cast<int64_t>(t.tw) * t.th * (ends[c] - from);
                }
            if (best < 0 || bytes < best) {
                best = bytes;
                cut1 = a;
                cut2 = b;
            }
        }
    const int ends[3] = {cut1, cut2, n};
    for (int c = 0, from = 0; c < 3; from = ends[c], ++c) {
        cls[c] = box((ends[c] > from ? ends[c] : n) - 1);
        for (int i = from; i < ends[c]; ++i) cls_of[order[i]] = static_cast<int8_t>(c);
    }
}

// The kernel's offset table of every (scale, bin) from the (dx, dy) pairs of
// build_offset_tables: four 16-bit tile offsets per window word, relative to the sample
// at (-reach, -reach), in builder order (unit by unit, one word per lane).
void build_tile_offsets(const double* scales, int nscales, const int8_t* offsets, uint16_t* out) {
    TileClass cls[kClasses];
    int8_t cls_of[LATCH_MAX_SCALES];
    tile_classes(scales, nscales, cls, cls_of);
    for (int t = 0; t < nscales * kBins; ++t) {
        const TileClass& k = cls[cls_of[t / kBins]];
        const int8_t* src = offsets + static_cast<size_t>(t) * kWinPix * 2;
        uint16_t* dst = out + static_cast<size_t>(t) * kWinPix;
        for (int blk = 0; blk < kBlocks; ++blk)
            for (int l = 0; l < kBlockWords; ++l) {
                const int cx = 4 * (blk % 3) + (l & 3), y = 8 * (blk / 3) + (l >> 2);
                for (int q = 0; q < 4; ++q) {
                    const int8_t* d = src + 2 * (y * kWin + 4 * cx + q);
                    dst[(blk * kBlockWords + l) * 4 + q] =
                        static_cast<uint16_t>((d[1] + k.reach) * k.tw + d[0] + k.reach);
                }
            }
    }
}

// Whether quarter Q holds the patch of size x size pixels at (x0, y0), and the three word
// columns that a patch which does not start at a word is read from.
static bool patch_in(const Quarter& Q, int x0, int y0, int size) {
    const int x = x0 - Q.b0, y = y0 - Q.r0;
    return x >= 0 && x + size <= 4 * Q.nc && y >= 0 && y + size <= Q.nr &&
           ((x & 3) == 0 || ((x >> 2) + 2) * Q.nr + y <= kTmLast);
}

// The quarters (bit q) that hold the patch at (x0, y0).
struct PatchMasks {
    uint8_t at[kWin][kWin];
    explicit PatchMasks(int size) {
        for (int y = 0; y < kWin; ++y)
            for (int x = 0; x < kWin; ++x) {
                at[y][x] = 0;
                for (int q = 0; q < kQuarters; ++q)
                    at[y][x] |= static_cast<uint8_t>(patch_in(quarter_of(q), x, y, size) << q);
            }
    }
};

// Sets of the triplets that could move: bit k is triplet order(k).
struct TripletSet {
    uint64_t w[kBits / 64];
    int n;
    void add(int k) { w[k >> 6] |= uint64_t(1) << (k & 63), ++n; }
    void remove(int k) { w[k >> 6] &= ~(uint64_t(1) << (k & 63)), --n; }
    int first() const {
        int i = 0;
        while (!w[i]) ++i;
        return 64 * i + __builtin_ctzll(w[i]);
    }
};

// The triplet table as the evaluators read it (LaneTriplets) for patches of `size` x
// `size` pixels (7, or 8 when weighted): every triplet goes to the quarter in which it
// costs least, and then moves between quarters level their loads.  latch_extract plans
// whenever it is given another table than before, so a move takes the first of the sets of
// triplets that it costs the same, not a search of the table (that took 0.2-0.5 ms of host
// time a table, this 20-60 us: calls of 2,000 keypoints that alternate between two tables
// 253 -> 50 us each, with one table 37).
void plan_triplets(const latch_triplet* trip, int size, LaneTripletPlan* plan) {
    static const PatchMasks masks7(2 * kPatchR + 1), masks8(2 * kPatchR + 2);
    const PatchMasks& masks = size == 8 ? masks8 : masks7;
    // clocks of a triplet (as measured) by its level in a quarter: more with every patch that
    // does not start at a word (level = their number; the same for weighted patches), most
    // from the staged windows
    constexpr int kLevels = 5, kStagedLevel = 4;
    const int plain[kLevels] = {72, 81, 90, 99, 250}, weighted[kLevels] = {800, 800, 800, 800, 950};
    const int* cost = size == 8 ? weighted : plain;
    constexpr int kBuildCost = 10000;  // of a batch's windows, after the triplets read from the staged ones
    auto order = [](int k) { return k * 317 & (kBits - 1); };  // spread over the indices, so over the chunks
    uint8_t level[kBits][kQuarters], in[kBits];
    int load[kQuarters] = {}, staged[kQuarters] = {};  // clocks in all, and from the staged windows
    int nowhere = 0;
    TripletSet sets[kQuarters][kLevels][kQuarters][kLevels] = {};  // [quarter][level there][other quarter][level there]
    auto each_set = [&](int k, auto&& f) {
        const int t = order(k), q = in[t];
        for (int o = 0; o < kQuarters; ++o)
            if (o != q) f(sets[q][level[t][q]][o][level[t][o]], k);
    };
    for (int k = 0; k < kBits; ++k) {
        const int t = order(k);
        const uint8_t* c = &trip[t].ax;
        uint32_t held = 15;
        for (int p = 0; p < 3; ++p) held &= masks.at[c[2 * p + 1] - kPatchR][c[2 * p] - kPatchR];
        int best = 0;
        for (int q = 0; q < kQuarters; ++q) {
            const int b0 = quarter_of(q).b0 + kPatchR;
            const int shifts = (((c[0] - b0) & 3) != 0) + (((c[2] - b0) & 3) != 0) + (((c[4] - b0) & 3) != 0);
            level[t][q] = static_cast<uint8_t>(held >> q & 1 ? shifts : kStagedLevel);
            if (cost[level[t][q]] < cost[level[t][best]]) best = q;
        }
        // plain ones that no quarter holds go round and stay: the builders wait for them
        // (weighted ones take long enough next to the building)
        const bool fixed = !held && size != 8;
        if (fixed) best = nowhere++ % kQuarters;
        in[t] = static_cast<uint8_t>(best);
        load[best] += cost[level[t][best]];
        if (level[t][best] == kStagedLevel) staged[best] += cost[kStagedLevel];
        if (!fixed) each_set(k, [](TripletSet& s, int i) { s.add(i); });
    }
    // the changes of level by what they cost
    struct Change {
        int from, to, d;
    } changes[kLevels * kLevels];
    for (int i = 0; i < kLevels * kLevels; ++i) {
        const Change c{i / kLevels, i % kLevels, cost[i % kLevels] - cost[i / kLevels]};
        int j = i;
        for (; j > 0 && changes[j - 1].d > c.d; --j) changes[j] = changes[j - 1];
        changes[j] = c;
    }
    // each time the move that costs least among those out of the fullest quarter that has one:
    // it lowers the load of the two, and what a quarter reads from the staged windows and the
    // next batch's building, which waits for it, stay below that load
    for (int moves = 0; moves < 4 * kBits; ++moves) {
        int move = -1, to = 0;
        int below = INT32_MAX;
        while (move < 0) {
            int full = -1;
            for (int q = 0; q < kQuarters; ++q)
                if (load[q] < below && (full < 0 || load[q] > load[full])) full = q;
            if (full < 0) break;
            below = load[full];
            int least = 0;
            for (const Change& c : changes) {
                if (move >= 0 && c.d > least) break;
                for (int q = 0; q < kQuarters; ++q) {
                    const TripletSet& s = sets[full][c.from][q][c.to];
                    if (s.n == 0 || load[q] + cost[c.to] >= load[full]) continue;
                    if (c.to == kStagedLevel && staged[q] + cost[kStagedLevel] + kBuildCost >= load[full]) continue;
                    const int k = s.first();
                    if (move >= 0 && k >= move) continue;
                    move = k;
                    to = q;
                    least = c.d;
                }
            }
        }
        if (move < 0) break;
        const int t = order(move), from = in[t];
        each_set(move, [](TripletSet& s, int i) { s.remove(i); });
        load[from] -= cost[level[t][from]];
        if (level[t][from] == kStagedLevel) staged[from] -= cost[kStagedLevel];
        in[t] = static_cast<uint8_t>(to);
        load[to] += cost[level[t][to]];
        if (level[t][to] == kStagedLevel) staged[to] += cost[kStagedLevel];
        each_set(move, [](TripletSet& s, int i) { s.add(i); });
    }
    // the list, by quarter, class and index
    uint8_t cls[kBits];
    int count[kQuarters][kTripClasses] = {}, at = 0;
    for (int t = 0; t < kBits; ++t) {
        const uint8_t* c = &trip[t].ax;
        const int b0 = quarter_of(in[t]).b0 + kPatchR;
        cls[t] = kStaged;
        if (level[t][in[t]] != kStagedLevel)
            cls[t] = static_cast<uint8_t>((((c[0] - b0) & 3) != 0) | (((c[2] - b0) & 3) != 0) << 1 |
                                          (((c[4] - b0) & 3) != 0) << 2);
        ++count[in[t]][cls[t]];
    }
    for (int q = 0; q < kQuarters; ++q) {
        for (int i = 0; i < kTripClasses; ++i) {
            plan->start[q][i] = static_cast<int16_t>(at);
            at += count[q][i];
            count[q][i] = plan->start[q][i];  // from here on: the next entry
        }
        plan->start[q][kTripClasses] = static_cast<int16_t>(at);
    }
    for (int t = 0; t < kBits; ++t) {
        const uint8_t* c = &trip[t].ax;
        const Quarter from = cls[t] == kStaged ? Quarter{0, kWordCols, 0, kWin} : quarter_of(in[t]);
        const int e = count[in[t]][cls[t]]++;
        for (int p = 0; p < 3; ++p) {
            const int x = c[2 * p] - kPatchR - from.b0, y = c[2 * p + 1] - kPatchR - from.r0;
            plan->e[p][e] = static_cast<uint32_t>(8 * (x & 3)) | static_cast<uint32_t>((x >> 2) * from.nr + y) << 16 |
                            (p == 0 ? static_cast<uint32_t>(t) << 5 : 0u);
        }
    }
}

static constexpr int kBatchImages = 64;  // images per launch in the batched form
static_assert(sizeof(ExtractParams<kBatchImages>) + sizeof(LaneTriplets) + sizeof(PatchWeights) + 64 <= 32764,
              "kernel parameter space");

template <int NI, bool kWeighted>
static cudaError_t set_extract_attributes() {
    return cudaFuncSetAttribute(extract_lanes_kernel<NI, kWeighted>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(kDynSmem));
}

template <int NI>
static cudaError_t launch_chunk(const latch_context* ctx, const latch_image* imgs, const int64_t* kp0,
                                const int64_t* n, int i0, int i1, const latch_keypoint* d_kps, uint8_t* d_out,
                                uint8_t* exp_out, cudaStream_t stream, uint32_t* flags, const int32_t* n_dev) {
    static unsigned long long attr_done[2] = {0, 0};
    cudaError_t e = ctx->weighted ? once_per_device(&attr_done[1], set_extract_attributes<NI, true>)
                                  : once_per_device(&attr_done[0], set_extract_attributes<NI, false>);
    if (e != cudaSuccess) return e;
    const EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return cudaErrorNotSupported;
    struct Params {
        ExtractParams<NI> prm;
        LaneTriplets tt;
        PatchWeights pw;
    };
    Params* p = new (std::nothrow) Params;
    if (!p) return cudaErrorMemoryAllocation;
    ExtractParams<NI>& prm = p->prm;
    tile_classes(ctx->scales, ctx->nscales, prm.cls, prm.cls_of);
    prm.count = i1 - i0;
    prm.row0 = static_cast<int32_t>(kp0[i0]);
    prm.nscales = ctx->nscales;
    prm.min_batch = ctx->item_kps;
    prm.n_dev = n_dev;
    int64_t total = 0;
    for (int i = i0; i < i1; ++i) {
        const int j = i - i0;
        prm.width[j] = imgs[i].width;
        prm.height[j] = imgs[i].height;
        prm.first[j] = static_cast<int32_t>(total);
        total += n[i];
        cuuint64_t dims[2] = {static_cast<cuuint64_t>(imgs[i].width), static_cast<cuuint64_t>(imgs[i].height)};
        cuuint64_t strides[1] = {static_cast<cuuint64_t>(imgs[i].pitch)};
        cuuint32_t estr[2] = {1, 1};
        for (int c = 0; c < kClasses; ++c) {
            CUtensorMap* map = &prm.map[j * kClasses + c];
            if (c > 0 && prm.cls[c].tw == prm.cls[c - 1].tw && prm.cls[c].th == prm.cls[c - 1].th) {
                *map = map[-1];
                continue;
            }
            cuuint32_t box[2] = {static_cast<cuuint32_t>(prm.cls[c].tw), static_cast<cuuint32_t>(prm.cls[c].th)};
            if (enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t*>(imgs[i].data), dims, strides, box,
                    estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
                delete p;
                return cudaErrorInvalidValue;
            }
        }
    }
    prm.n = static_cast<int32_t>(total);
    static_assert(sizeof(LaneTriplets) == sizeof(ctx->trip_plan), "triplet table layout");
    memcpy(&p->tt, &ctx->trip_plan, sizeof(LaneTriplets));
    for (int i = 0; i < 64; ++i) p->pw.w[i] = ctx->patch_weights[i];
    e = launch_chained(ctx->weighted ? extract_lanes_kernel<NI, true> : extract_lanes_kernel<NI, false>,
                       dim3(static_cast<unsigned>(ctx->sm_count)), dim3(kThreads), kDynSmem, stream, prm, p->tt, p->pw,
                       d_kps, reinterpret_cast<const uint2*>(ctx->d_tile_offsets), d_out, exp_out, flags);
    delete p;
    return e;
}

cudaError_t launch_extract_batch(const latch_context* ctx, const latch_image* imgs, const int64_t* kp0,
                                 const int64_t* n, int count, const latch_keypoint* d_kps, uint8_t* d_out,
                                 cudaStream_t stream, uint8_t* exp_out, uint32_t* flags) {
    if (!flags) flags = ctx->d_flags;
    for (int i0 = 0; i0 < count; i0 += kBatchImages) {
        const int i1 = i0 + kBatchImages < count ? i0 + kBatchImages : count;
        int64_t nk = 0;
        for (int i = i0; i < i1; ++i) nk += n[i];
        if (nk == 0) continue;
        // the kernel parameters hold the images' tensor maps: the smallest instance that
        // fits keeps the launch's parameter block small
        const int ni = i1 - i0;
        const cudaError_t e =
            ni == 1    ? launch_chunk<1>(ctx, imgs, kp0, n, i0, i1, d_kps, d_out, exp_out, stream, flags, nullptr)
            : ni <= 4  ? launch_chunk<4>(ctx, imgs, kp0, n, i0, i1, d_kps, d_out, exp_out, stream, flags, nullptr)
            : ni <= 16 ? launch_chunk<16>(ctx, imgs, kp0, n, i0, i1, d_kps, d_out, exp_out, stream, flags, nullptr)
                       : launch_chunk<kBatchImages>(ctx, imgs, kp0, n, i0, i1, d_kps, d_out, exp_out, stream, flags,
                                                    nullptr);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_extract(const latch_context* ctx, const latch_image* img, const latch_keypoint* d_kps, int32_t n,
                           uint8_t* d_out, cudaStream_t stream) {
    const int64_t kp0 = 0, nn = n;
    return launch_extract_batch(ctx, img, &kp0, &nn, 1, d_kps, d_out, stream, nullptr);
}

cudaError_t launch_extract_dev_count(const latch_context* ctx, const latch_image* img, const latch_keypoint* d_kps,
                                     int32_t max_n, const int32_t* d_n, uint8_t* d_out, cudaStream_t stream) {
    if (max_n <= 0) return cudaSuccess;
    const int64_t kp0 = 0, nn = max_n;
    return launch_chunk<1>(ctx, img, &kp0, &nn, 0, 1, d_kps, d_out, nullptr, stream, ctx->d_flags, d_n);
}

}  // namespace latch
