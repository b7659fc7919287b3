// Dense per-pixel LATCH and windowed matching (Sec. 6: CLATCH for dense pixel
// matching, as an alternative to PatchMatch).
//
// Every pixel is an upright keypoint at scale 1, so a triplet (a, c1, c2) gives, at
// all pixels p at once,
//   D1(p) - D2(p) = sum over the 7x7 box of (A - C1)^2 - (A - C2)^2
//                 = box7[ (C2 - C1)(2A - C1 - C2) ](p),
// with A = I(p + a - 24 + d), C1, C2 likewise (Eq. 1; one product image per triplet,
// then a separable 7x7 box sum; all exact in int32, |box| <= 49 * 255 * 510).
//
// dense_extract_kernel: one block per 32x32-pixel tile and share of the triplets; the image
// region under the tile and every window (79 x 79 bytes, 0 outside the image) is staged
// once in shared memory.  Per round two triplets, from the two halves of the share:
//   phase A (304 threads, 2 x 38 rows x 4 segments): a thread forms the product image
//            along 14 pixels of one row (each patch's 14 bytes from five aligned
//            words) and writes 8 horizontal 7-sums;
//   phase B (256 threads, 2 x 32 columns x 4 segments): a thread adds 7 of them
//            vertically for 8 pixels of one column, and bit t of those pixels is
//            box > 0 (D1 > D2, strict).
// The horizontal sums are double-buffered, so one barrier separates the rounds;
// each phase-B thread gathers 32 consecutive bits per pixel in registers and
// writes the descriptor word once.
//
// dense_match_kernel: one block per 16x16 pixels of image A; the descriptors of B
// under the tile and its radius-R halo are staged in shared memory (by groups of eight
// cells, so that a warp's neighbouring descriptors hit different banks); each
// thread keeps its pixel's descriptor in registers and visits the (2R + 1)^2
// candidates in raster order of B (those inside B), computing XOR + population
// count (popc.cuh) and keeping the two smallest keys of distance and raster order, which
// is the lowest-raster-index tie rule.
#include <cstdint>

#include "internal.h"
#include "popc.cuh"
#include "sm103.h"

namespace latch {

namespace {

using namespace sm103;

constexpr int kTile = 32;                       // output pixels per tile side
constexpr int kRegion = kTile + kWin - 1;       // 79: staged image rows / columns
constexpr int kRegionPitch = 84;                // bytes per staged row (21 words: odd)
constexpr int kHRows = kTile + 2 * kPatchR;     // 38: rows of horizontal sums
constexpr int kHPitch = 36;                     // words per row of horizontal sums
constexpr int kSegs = 4;                        // 8-pixel segments per row / column
constexpr int kAThreads = kHRows * kSegs;       // 152 per triplet
constexpr int kBThreads = kTile * kSegs;        // 128 per triplet
constexpr int kDenseThreads = 320;
constexpr int kBlocksPerSm = 6;
constexpr int kMaxShares = 8;                   // a share is at least two descriptor words

struct DenseTriplets {
    latch_triplet t[kBits];
};

struct DenseSmem {
    uint8_t img[kRegion * kRegionPitch];
    uint8_t pad[16];                            // the last row's word loads may read past it
    uint16_t off[3][kBits];                     // staged-region offset of each patch's top-left pixel
    alignas(16) int32_t h[2][2][kHRows][kHPitch];  // [round parity][triplet slot][row][column]
};

// Three blocks per SM at 64 registers (24 bytes spilled); launch bounds of
// four and five blocks spill more and are slower.
__global__ void __launch_bounds__(kDenseThreads, 3) dense_extract_kernel(const uint8_t* __restrict__ img, int width,
                                                                      int height, int64_t pitch, int half,
                                                                      const __grid_constant__ DenseTriplets tr,
                                                                      uint32_t* __restrict__ out) {
    __shared__ __align__(16) DenseSmem S;
    const int tid = threadIdx.x;
    const int x0 = blockIdx.x * kTile, y0 = blockIdx.y * kTile;
    const int first = blockIdx.z * 2 * half;  // the share's triplets: [first, first + 2 half)
    griddep_wait();
    griddep_launch_dependents();
    // stage the region [x0 - 24, x0 + 55) x [y0 - 24, y0 + 55); samples outside read 0
    for (int i = tid; i < kRegion * kRegion; i += kDenseThreads) {
        const int rr = i / kRegion, cc = i - rr * kRegion;
        const int gy = y0 - kHalf + rr, gx = x0 - kHalf + cc;
        uint8_t v = 0;
        if (gx >= 0 && gx < width && gy >= 0 && gy < height) v = img[static_cast<int64_t>(gy) * pitch + gx];
        S.img[rr * kRegionPitch + cc] = v;
    }
    // patch at window point (x, y) of the pixel at tile offset (fx, fy): staged pixel
    // (fx + x - 3 + dx, fy + y - 3 + dy) for dx, dy in 0..6 -- the thread's base plus off
    for (int t = tid; t < 2 * half; t += kDenseThreads) {
        const uint8_t* c = &tr.t[first + t].ax;
        for (int p = 0; p < 3; ++p)
            S.off[p][t] = static_cast<uint16_t>((c[2 * p + 1] - kPatchR) * kRegionPitch + (c[2 * p] - kPatchR));
    }
    __syncthreads();

    // phase A role: slot ja, segment sa (pixels 8 sa .. 8 sa + 7), row ra of the
    // horizontal sums (image row y0 + ra - 3)
    const int ja = tid / kAThreads, la = tid - ja * kAThreads;
    const int sa = la / kHRows, ra = la - sa * kHRows;
    const uint8_t* abase = S.img + ra * kRegionPitch + kTile / kSegs * sa;
    // phase B role: slot jb, segment sb (rows 8 sb .. 8 sb + 7), column cb
    const int jb = tid / kBThreads, lb = tid - jb * kBThreads;
    const int sb = lb / kTile, cb = lb - sb * kTile;
    uint32_t bits[8] = {0, 0, 0, 0, 0, 0, 0, 0};

    // the 14 bytes at p as four words (byte i in byte i % 4 of word i / 4): five
    // aligned word loads and funnel shifts instead of 14 byte loads
    auto load14 = [](const uint8_t* p, uint32_t (&y)[4]) {
        const uintptr_t addr = reinterpret_cast<uintptr_t>(p);
        const uint32_t* w = reinterpret_cast<const uint32_t*>(addr & ~static_cast<uintptr_t>(3));
        const uint32_t sh = static_cast<uint32_t>(addr & 3u) * 8u;
        uint32_t x[5];
#pragma unroll
        for (int q = 0; q < 5; ++q) x[q] = w[q];
#pragma unroll
        for (int q = 0; q < 4; ++q) y[q] = __funnelshift_r(x[q], x[q + 1], sh);
    };
    auto byte_of = [](const uint32_t (&y)[4], int i) {
        return static_cast<int>(__byte_perm(y[i >> 2], 0u, 0x4440u | static_cast<uint32_t>(i & 3)));
    };
    auto phase_a = [&](int k) {
        const int t = ja * half + k;
        uint32_t ya[4], y1[4], y2[4];
        load14(abase + S.off[0][t], ya);
        load14(abase + S.off[1][t], y1);
        load14(abase + S.off[2][t], y2);
        int f[14];
#pragma unroll
        for (int i = 0; i < 14; ++i) {
            const int a = byte_of(ya, i), c1 = byte_of(y1, i), c2 = byte_of(y2, i);
            f[i] = (c2 - c1) * (2 * a - c1 - c2);
        }
        int h[8];
        h[0] = f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6];
#pragma unroll
        for (int j = 1; j < 8; ++j) h[j] = h[j - 1] + f[j + 6] - f[j - 1];
        int4* dst = reinterpret_cast<int4*>(&S.h[k & 1][ja][ra][kTile / kSegs * sa]);
        dst[0] = make_int4(h[0], h[1], h[2], h[3]);
        dst[1] = make_int4(h[4], h[5], h[6], h[7]);
    };

    if (tid < 2 * kAThreads) phase_a(0);
    __syncthreads();
    for (int k = 0; k < half; ++k) {
        if (tid < 2 * kBThreads) {
            const int32_t* hc = &S.h[k & 1][jb][kTile / kSegs * sb][cb];
            int hv[14];
#pragma unroll
            for (int i = 0; i < 14; ++i) hv[i] = hc[i * kHPitch];
            int v = hv[0] + hv[1] + hv[2] + hv[3] + hv[4] + hv[5] + hv[6];
            const uint32_t b = static_cast<uint32_t>(k & 31);
            bits[0] |= static_cast<uint32_t>(v > 0) << b;
#pragma unroll
            for (int j = 1; j < 8; ++j) {
                v += hv[j + 6] - hv[j - 1];
                bits[j] |= static_cast<uint32_t>(v > 0) << b;
            }
            if (b == 31) {
                // the descriptor word of triplet first + jb half + k, of the segment's 8 pixels
                const int w = (first + jb * half + k) >> 5;
                const int x = x0 + cb;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int y = y0 + kTile / kSegs * sb + j;
                    if (x < width && y < height) out[(static_cast<int64_t>(y) * width + x) * kDescWords + w] = bits[j];
                    bits[j] = 0;
                }
            }
        }
        if (k + 1 < half && tid < 2 * kAThreads) phase_a(k + 1);
        __syncthreads();
    }
}

constexpr int kMTile = 16;          // pixels of A per tile side
constexpr int kMatchThreads = kMTile * kMTile;
constexpr int kOrdBits = 12;        // staged row and column (less than 64 each) of a candidate
static_assert(kMTile + 2 * LATCH_DENSE_MAX_RADIUS <= 64, "staged rows and columns take 6 bits each");
constexpr uint32_t kNoKey = 0xffffffffu;

// Staged descriptors: eight neighbouring cells to a group of 512 bytes, chunk q (16
// bytes) of cell c at (c / 8) 512 + 128 q + (c % 8) 16.  Any eight neighbouring cells'
// chunks fill all 32 banks, a candidate's four chunks are one address and constant
// offsets, and the staging threads run along both the descriptors and the groups.
__device__ __forceinline__ const uint4* staged_cell(const uint4* s, int c) { return s + (c >> 3) * 32 + (c & 7); }

// Hamming distance of a descriptor to the one whose chunks are kStep chunks apart.
template <int kStep>
__device__ __forceinline__ int chunk_distance(const uint32_t (&a)[16], const uint4* c) {
    uint32_t x[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint4 v = c[kStep * q];
        x[4 * q] = v.x ^ a[4 * q], x[4 * q + 1] = v.y ^ a[4 * q + 1];
        x[4 * q + 2] = v.z ^ a[4 * q + 2], x[4 * q + 3] = v.w ^ a[4 * q + 3];
    }
    return popc16(x);
}

// One pixel per thread.  Keys distance << 12 | staged row << 6 | column are unique and
// order ties by raster index, so a distance costs the top two two minima and a maximum.
// The logic pipe (16 XORs and 16 adder operations, the top two: 35 at 64 lanes per clock) and
// the population-count pipe (9 counts at 16) bound it about equally; packed keys and the staged
// order take several of the logic pipe's operations per distance away.  Measured (GB300; with
// rotated chunks, compares and selects, and now): 640x480 at radius 2 / 8 / 16 30.9 -> 26.6, 298
// -> 238 and 1,786 -> 1,357 us, 1920x1080 at radius 8 1,902 -> 1,517 us.  At radius 0 a
// descriptor is read once and nothing is staged (staged, whose loads are 16 bytes from each of
// eight descriptors: 1001x601 14.2 -> 11.8 us, 1920x1080 46.2 -> 43.6).  Two pixels per thread (a
// candidate's loads serve both) took 10% more at 640x480, radius 8: too few warps.
__global__ void __launch_bounds__(kMatchThreads) dense_match_kernel(const uint4* __restrict__ da,
                                                                    const uint4* __restrict__ db, int width,
                                                                    int height, int radius, int k, int r_milli,
                                                                    latch_match* __restrict__ out) {
    extern __shared__ uint4 s_desc[];
    const int side = kMTile + 2 * radius, cells = side * side;
    const int x0 = blockIdx.x * kMTile, y0 = blockIdx.y * kMTile;
    griddep_wait();
    griddep_launch_dependents();
    if (radius > 0)
        for (int i = threadIdx.x; i < (cells + 7) / 8 * 32; i += kMatchThreads) {
            const int cell = (i >> 5) * 8 + (i & 7), q = (i >> 3) & 3;
            const int ry = cell / side, rx = cell - ry * side;
            const int gy = y0 - radius + ry, gx = x0 - radius + rx;
            if (cell < cells && gx >= 0 && gx < width && gy >= 0 && gy < height)
                s_desc[i] = db[(static_cast<int64_t>(gy) * width + gx) * 4 + q];
        }
    const int tx = threadIdx.x % kMTile, ty = threadIdx.x / kMTile;
    const int px = x0 + tx, py = y0 + ty;
    const bool live = px < width && py < height;
    const int64_t self = (static_cast<int64_t>(py) * width + px) * 4;
    uint32_t a[16];
    if (live) {
        const uint4* src = da + self;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 v = src[q];
            a[4 * q] = v.x, a[4 * q + 1] = v.y, a[4 * q + 2] = v.z, a[4 * q + 3] = v.w;
        }
    }
    uint32_t m1 = kNoKey, m2 = kNoKey;
    auto key_of = [](int d, int ry, int rx) {
        return (static_cast<uint32_t>(d) << kOrdBits) + static_cast<uint32_t>(ry << 6 | rx);
    };
    if (radius == 0) {  // each descriptor is read once: nothing to stage
        if (!live) return;
        m1 = key_of(chunk_distance<1>(a, db + self), ty, tx);
    } else {
        __syncthreads();
        if (!live) return;
        // staged rows and columns of the candidates inside B
        const int rx_lo = max(tx, radius - x0), rx_hi = min(tx + 2 * radius, width - 1 - x0 + radius);
        const int ry_lo = max(ty, radius - y0), ry_hi = min(ty + 2 * radius, height - 1 - y0 + radius);
        for (int ry = ry_lo; ry <= ry_hi; ++ry) {
            for (int rx = rx_lo; rx <= rx_hi; ++rx) {
                const uint32_t key = key_of(chunk_distance<8>(a, staged_cell(s_desc, ry * side + rx)), ry, rx);
                m2 = min(m2, max(m1, key));
                m1 = min(m1, key);
            }
        }
    }
    auto index = [&](uint32_t key) {
        const int ry = key >> 6 & 63, rx = key & 63;
        return (y0 - radius + ry) * width + x0 - radius + rx;
    };
    latch_match m;
    m.idx1 = index(m1);  // the pixel itself is always a candidate
    m.dist1 = static_cast<uint16_t>(m1 >> kOrdBits);
    const bool has2 = k == 2 && m2 != kNoKey;
    m.idx2 = has2 ? index(m2) : -1;
    m.dist2 = has2 ? static_cast<uint16_t>(m2 >> kOrdBits) : 0xffff;
    if (k == 1)
        m.accepted = 1;
    else
        m.accepted = (1000ll * m.dist1 < static_cast<long long>(r_milli) * m.dist2) ? 1 : 0;
    m.pad[0] = m.pad[1] = m.pad[2] = 0;
    out[static_cast<int64_t>(py) * width + px] = m;
}

}  // namespace

static size_t dense_match_smem_bytes(int radius) {
    if (radius == 0) return 0;
    const size_t side = static_cast<size_t>(kMTile + 2 * radius);
    return (side * side + 7) / 8 * 8 * kDescBytes;  // whole groups of eight cells
}

cudaError_t launch_dense_extract(const latch_context* ctx, const latch_image* img, uint8_t* d_out,
                                 cudaStream_t stream) {
    DenseTriplets tr;
    for (int t = 0; t < kBits; ++t) tr.t[t] = ctx->h_trip[t];
    const int tx = (img->width + kTile - 1) / kTile, ty = (img->height + kTile - 1) / kTile;
    // An SM holds three blocks; the triplets are shared out until there are about six per SM,
    // so that the last round of blocks is short (640x480, 300 tiles: 343 us with one share,
    // 234, 228 and 234 us with 2, 4 and 8, which stage the region more often).
    int shares = 1;
    while (shares < kMaxShares && static_cast<int64_t>(tx) * ty * shares < kBlocksPerSm * ctx->sm_count) shares *= 2;
    const dim3 grid(static_cast<unsigned>(tx), static_cast<unsigned>(ty), static_cast<unsigned>(shares));
    return launch_chained(dense_extract_kernel, grid, dim3(kDenseThreads), 0, stream, img->data, img->width,
                          img->height, img->pitch, kBits / (2 * shares), tr, reinterpret_cast<uint32_t*>(d_out));
}

static cudaError_t set_dense_match_attributes() {
    return cudaFuncSetAttribute(dense_match_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(dense_match_smem_bytes(kDenseMaxRadius)));
}

cudaError_t launch_dense_match(const uint8_t* d_a, const uint8_t* d_b, int32_t width, int32_t height, int32_t radius,
                               int32_t k, int32_t r_milli, latch_match* d_out, cudaStream_t stream) {
    static unsigned long long attr_done = 0;
    const cudaError_t e = once_per_device(&attr_done, set_dense_match_attributes);
    if (e != cudaSuccess) return e;
    const dim3 grid(static_cast<unsigned>((width + kMTile - 1) / kMTile),
                    static_cast<unsigned>((height + kMTile - 1) / kMTile));
    return launch_chained(dense_match_kernel, grid, dim3(kMatchThreads), dense_match_smem_bytes(radius), stream,
                          reinterpret_cast<const uint4*>(d_a), reinterpret_cast<const uint4*>(d_b), width, height,
                          radius, k, r_milli, d_out);
}

}  // namespace latch
