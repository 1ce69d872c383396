// Disparity fill (Sec. 3.1, last paragraph): a second disparity map of L0/R0
// by semi-global matching, which verifies the matching's own d0 where the
// joint consistency check removed the pixel (the disparity-only seeds are
// chosen in sff_seeds.cu).
//
// SGM as this library reads it (the paper gives no details):
//   grey = (R + 2G + B + 2) >> 2; census over a 9 x 7 window, bit k (row-major
//   window order, centre skipped) set when the neighbour is darker than the
//   centre, coordinates clamped; cost C(p, d) = popcount(census_L(x, y) ^
//   census_R(max(x - d, 0), y)); 8 directions r (4 axes, 4 diagonals)
//     L_r(p, d) = C(p, d) + min(L_r(p-r, d), L_r(p-r, d+-1) + P1,
//                               min_k L_r(p-r, k) + P2) - min_k L_r(p-r, k),
//   L_r(p, d) = C(p, d) at the first pixel of a path; disparity = argmin_d of
//   sum_r L_r(p, d), ties to the lowest d.
//
// L_r(p, d) lies in [0, 62 + P2], so with P2 <= 193 it is stored exactly in
// one byte.
//
// k_sgm_census: grey and census of both images from a shared-memory tile.
// k_sgm_cost:   the cost volume, one byte per pixel and disparity (a path
//               step then reads D bytes instead of D census words).
// k_sgm_paths:  the path lines of all directions; L_r to [dir][y][x][d].
// k_sgm_wta:    the 8 directions summed per disparity, the (sum, d) minimum.
#include <cstring>

#include "sff_internal.cuh"

namespace sff {
namespace {

constexpr int kDirs = 8;
constexpr int kWtaWarps = 8;   // warps per CTA of k_sgm_wta
constexpr int kCensusW = 9, kCensusH = 7;
constexpr int kTileX = 32, kTileY = 8;
constexpr unsigned kFull = 0xffffffffu;

struct SgmJob {
    const uint8_t* img[2];  // L0, R0
    int pitch, w, h, D, p1, p2;
    uint64_t* census[2];    // [y][x]
    uint8_t* cost;          // [y][x][D] matching costs
    uint8_t* paths;         // [dir][y][x][D]
    int16_t* disp;          // [y][x]
};

__constant__ int c_dir[kDirs][2] = {{1, 0}, {-1, 0}, {0, 1}, {0, -1}, {1, 1}, {-1, -1}, {1, -1}, {-1, 1}};

__global__ void __launch_bounds__(kTileX * kTileY) k_sgm_census(SgmJob S) {
    constexpr int TW = kTileX + kCensusW - 1, TH = kTileY + kCensusH - 1;
    __shared__ uint8_t tile[TH][TW];
    const uint8_t* img = blockIdx.z ? S.img[1] : S.img[0];  // no dynamic index into the parameter
    const int x0 = blockIdx.x * kTileX - kCensusW / 2, y0 = blockIdx.y * kTileY - kCensusH / 2;
    for (int k = threadIdx.y * kTileX + threadIdx.x; k < TW * TH; k += kTileX * kTileY) {
        const int tx = k % TW, ty = k / TW;
        const int gx = clampi(x0 + tx, 0, S.w - 1), gy = clampi(y0 + ty, 0, S.h - 1);
        const uint8_t* p = img + (size_t)gy * S.pitch + 3 * gx;
        tile[ty][tx] = (uint8_t)((p[0] + 2 * p[1] + p[2] + 2) >> 2);
    }
    __syncthreads();
    const int x = blockIdx.x * kTileX + threadIdx.x, y = blockIdx.y * kTileY + threadIdx.y;
    if (x >= S.w || y >= S.h) return;
    const int c = tile[threadIdx.y + kCensusH / 2][threadIdx.x + kCensusW / 2];
    uint64_t bits = 0;
    int k = 0;
#pragma unroll
    for (int j = 0; j < kCensusH; ++j)
#pragma unroll
        for (int i = 0; i < kCensusW; ++i) {
            if (i == kCensusW / 2 && j == kCensusH / 2) continue;
            bits |= (uint64_t)(tile[threadIdx.y + j][threadIdx.x + i] < c) << k;
            ++k;
        }
    (blockIdx.z ? S.census[1] : S.census[0])[(size_t)y * S.w + x] = bits;
}

// K bytes in registers: one access of 16, 8, 4 or 2 bytes.
template <int K>
struct Bytes;
template <>
struct Bytes<16> { using Vec = uint4; };
template <>
struct Bytes<8> { using Vec = uint2; };
template <>
struct Bytes<4> { using Vec = uint32_t; };
template <>
struct Bytes<2> { using Vec = uint16_t; };

// The costs of K consecutive disparities as 16-bit pairs: word j holds bytes j and
// K/2 + j.
__device__ __forceinline__ void unpack_pairs(const uint4& v, uint32_t (&c)[8]) {
    // costs are below 128, so the permute's sign-replicating selectors (bit 3
    // set) give the zero bytes
    const uint32_t lo[2] = {v.x, v.y}, hi[2] = {v.z, v.w};
#pragma unroll
    for (uint32_t j = 0; j < 8; ++j) {
        const uint32_t k = j & 3;
        asm("prmt.b32 %0, %1, %2, %3;"
            : "=r"(c[j])
            : "r"(lo[j >> 2]), "r"(hi[j >> 2]), "r"(k | (8 + k) << 4 | (4 + k) << 8 | (12 + k) << 12));
    }
}
__device__ __forceinline__ void unpack_pairs(const uint2& v, uint32_t (&c)[4]) {
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k)
        asm("prmt.b32 %0, %1, %2, %3;"
            : "=r"(c[k])
            : "r"(v.x), "r"(v.y), "r"(k | (8 + k) << 4 | (4 + k) << 8 | (12 + k) << 12));
}
__device__ __forceinline__ void unpack_pairs(const uint32_t& v, uint32_t (&c)[2]) {
    c[0] = v & 0x00ff00ffu;
    c[1] = (v >> 8) & 0x00ff00ffu;
}
__device__ __forceinline__ void unpack_pairs(const uint16_t& v, uint32_t (&c)[1]) {
    c[0] = __byte_perm((uint32_t)v, 0u, 0x4140);
}

// And back, every half below 256.
__device__ __forceinline__ void pack_four(const uint32_t* c, uint32_t& lo, uint32_t& hi) {
    const uint32_t a = __byte_perm(c[0], c[1], 0x6240), b = __byte_perm(c[2], c[3], 0x6240);
    lo = __byte_perm(a, b, 0x5410);
    hi = __byte_perm(a, b, 0x7632);
}
__device__ __forceinline__ void pack_pairs(const uint32_t (&c)[8], uint4& v) {
    pack_four(c, v.x, v.z);
    pack_four(c + 4, v.y, v.w);
}
__device__ __forceinline__ void pack_pairs(const uint32_t (&c)[4], uint2& v) { pack_four(c, v.x, v.y); }
__device__ __forceinline__ void pack_pairs(const uint32_t (&c)[2], uint32_t& v) { v = c[0] | c[1] << 8; }
__device__ __forceinline__ void pack_pairs(const uint32_t (&c)[1], uint16_t& v) {
    v = (uint16_t)__byte_perm(c[0], 0u, 0x4420);
}

// C(p, d) for every pixel.  One CTA per segment of kCostSeg pixels of a row:
// the right image's census words the segment needs (x - D + 1 .. the
// segment's end, positions clamped at 0) are staged in shared memory once; a
// thread keeps its disparity, so a warp reads 32 consecutive words, and the
// bytes are put together in shared memory for whole 16-byte stores.  Bound by
// the popcounts.  1242 x 375, D = 128: 59 us (J consecutive disparities per
// lane: the reads conflicted four ways) -> 36 us.
constexpr int kCostSeg = 64;
constexpr int kCostThreads = 256;

template <int D>
__global__ void __launch_bounds__(kCostThreads) k_sgm_cost(SgmJob S) {
    __shared__ uint64_t right[kCostSeg + D - 1], left[kCostSeg];
    __shared__ __align__(16) uint8_t out[kCostSeg * D];
    const int y = blockIdx.y, x0 = blockIdx.x * kCostSeg, t = threadIdx.x;
    const size_t row = (size_t)y * S.w;
    const int base = x0 - (D - 1);  // census position of right[0]
    for (int i = t; i < kCostSeg + D - 1; i += kCostThreads)
        right[i] = S.census[1][row + min(max(base + i, 0), S.w - 1)];
    if (t < kCostSeg) left[t] = S.census[0][row + min(x0 + t, S.w - 1)];
    __syncthreads();
    // right[k + D - 1 - d] is position x0 + k - d (already clamped)
    const int d = t % D;
#pragma unroll 4
    for (int k = t / D; k < kCostSeg; k += kCostThreads / D)
        out[k * D + d] = (uint8_t)__popcll(left[k] ^ right[k + D - 1 - d]);
    __syncthreads();
    const int bytes = min(kCostSeg, S.w - x0) * D;
    uint4* dst = reinterpret_cast<uint4*>(S.cost + (row + x0) * D);
    for (int i = t; i < bytes / 16; i += kCostThreads) dst[i] = reinterpret_cast<const uint4*>(out)[i];
}

// The path costs of one direction.  G lanes take a line's D disparities, K = D / G
// consecutive ones each, and a warp 32 / G neighbouring lines.  Two disparities
// share a 32-bit word as 16-bit halves: word j of a lane holds d = b + j and b +
// K/2 + j, so that the d - 1 and d + 1 neighbours of a word are the words beside it
// and only the two outer ones need a shuffle and a permute.  Every value stays
// below 2^16 and every difference taken is >= 0, so plain 32-bit adds and
// subtracts act on both halves:
//   L(p, d) = C + min(P, min(P(d - 1), P(d + 1)) + P1, m + P2) - m.
// Starting from P = m = 0 gives L = C at a line's first pixel.  Beyond the
// disparity range: 0x7fff.  The costs of the next pixels are in flight in registers.
constexpr int kAheadNarrow = 16, kAheadWide = 8;  // 8 and 4: 197 us

template <int D, int K>
__device__ __forceinline__ void path_lines(const SgmJob& S, int dir, int block) {
    constexpr int G = D / K, NP = K / 2, kAhead = K <= 4 ? kAheadNarrow : kAheadWide;
    static_assert(G >= 2 && G <= 32, "lanes per line");
    using Vec = typename Bytes<K>::Vec;
    const int rx = c_dir[dir][0], ry = c_dir[dir][1];
    const int lane = threadIdx.x & 31, gl = lane % G;
    const int line = block * (32 / G) + lane / G;
    const int W = S.w, H = S.h;
    // the line's first pixel: the pixels whose predecessor is outside the image
    int x, y, nlines;
    if (ry == 0) {
        nlines = H;
        y = line;
        x = rx > 0 ? 0 : W - 1;
    } else if (rx == 0) {
        nlines = W;
        x = line;
        y = ry > 0 ? 0 : H - 1;
    } else {
        nlines = W + H - 1;
        if (line < W) {
            x = line;
            y = ry > 0 ? 0 : H - 1;
        } else {
            x = rx > 0 ? 0 : W - 1;
            y = ry > 0 ? 1 + (line - W) : H - 2 - (line - W);
        }
    }
    // steps until the line leaves the image (0: no such line)
    const int n = line >= nlines ? 0
                                 : min(rx > 0 ? W - x : rx < 0 ? x + 1 : 1 << 30, ry > 0 ? H - y : ry < 0 ? y + 1 : 1 << 30);
    const int most = (int)__reduce_max_sync(kFull, (unsigned)n);
    const ptrdiff_t step = ((ptrdiff_t)ry * W + rx) * D;  // bytes from a pixel to the next
    const size_t p0 = n ? ((size_t)y * W + x) * D + gl * K : 0;
    const uint8_t* src = S.cost + p0;
    uint8_t* dst = S.paths + (size_t)dir * W * H * D + p0;
    Vec ahead[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
        ahead[u] = Vec{};
        if (u < n) ahead[u] = *reinterpret_cast<const Vec*>(src + u * step);
    }
    src += kAhead * step;
    const uint32_t p1x2 = (uint32_t)S.p1 * 0x00010001u, p2x2 = (uint32_t)S.p2 * 0x00010001u;
    const bool first = gl == 0, last = gl == G - 1;
    uint32_t prev[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) prev[j] = 0;
    uint32_t m2 = 0;  // the minimum over d, in both halves
    for (int t0 = 0; t0 < most; t0 += kAhead) {
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int t = t0 + u;
            uint32_t cost[NP];
            unpack_pairs(ahead[u], cost);
            if (t + kAhead < n) ahead[u] = *reinterpret_cast<const Vec*>(src);
            src += step;
            // the words below word 0 and above word NP - 1
            const uint32_t lo = __shfl_up_sync(kFull, prev[NP - 1], 1, G), hi = __shfl_down_sync(kFull, prev[0], 1, G);
            const uint32_t below = __byte_perm(first ? 0x7fff0000u : lo, prev[NP - 1], 0x5432);
            const uint32_t above = __byte_perm(prev[0], last ? 0x00007fffu : hi, 0x5432);
            const uint32_t mp2 = m2 + p2x2;
            uint32_t cur[NP];
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const uint32_t side = __vminu2(j > 0 ? prev[j - 1] : below, j < NP - 1 ? prev[j + 1] : above);
                cur[j] = __vminu2(__viaddmin_u16x2(side, p1x2, mp2), prev[j]) + (cost[j] - m2);
            }
            if (t < n) {
                Vec v;
                pack_pairs(cur, v);
                *reinterpret_cast<Vec*>(dst) = v;
            }
            dst += step;
            uint32_t mm[NP];
#pragma unroll
            for (int j = 0; j < NP; ++j) prev[j] = mm[j] = cur[j];
#pragma unroll
            for (int w = NP / 2; w >= 1; w >>= 1)
#pragma unroll
                for (int j = 0; j < w; ++j) mm[j] = __vminu2(mm[j], mm[j + w]);
            if constexpr (G == 32) {
                m2 = __reduce_min_sync(kFull, min(mm[0] & 0xffffu, mm[0] >> 16)) * 0x00010001u;
            } else {
                m2 = __vminu2(mm[0], __byte_perm(mm[0], 0u, 0x1032));
#pragma unroll
                for (int o = 1; o < G; o <<= 1) m2 = __vminu2(m2, __shfl_xor_sync(kFull, m2, o));
            }
        }
    }
}

// Two splits of a line.  The horizontal lines are the longest chains of steps (W,
// the others at most H) and few, so they get the shortest step: all lanes (16 at
// D = 32) on one line and the minimum by one redux.  The others share a warp: the
// fixed work of a step (addresses, loop, the minimum by shuffles) then serves
// several lines.  One warp per CTA, the horizontal ones first.
template <int D>
struct Split {
    static constexpr int kAcross = D >= 64 ? D / 32 : 2;  // disparities per lane, horizontal lines
    static constexpr int kOther = D >= 128 ? 16 : 8;
    __host__ __device__ static int blocks_across(int h) { return (h * (D / kAcross) + 31) / 32; }
    __host__ __device__ static int blocks(int lines) { return (lines * (D / kOther) + 31) / 32; }
};

// All directions.  Bound by the ALU pipe (67 % while the SMs are busy) and
// a tail of the horizontal lines (28 %).  1242 x 375, D = 128: 403 us (one line per
// warp, d +- 1 by permutes per word, costs through a cp.async ring) -> 231 us (every
// line on 8 lanes) -> 191 us.
template <int D>
__global__ void __launch_bounds__(32) k_sgm_paths(SgmJob S) {
    using P = Split<D>;
    const int across = P::blocks_across(S.h), b = (int)blockIdx.x;
    if (b < 2 * across) {
        path_lines<D, P::kAcross>(S, b & 1, b >> 1);
    } else {
        const int k = b - 2 * across, per = P::blocks(S.w + S.h - 1);
        path_lines<D, P::kOther>(S, 2 + k / per, k % per);
    }
}

// argmin over d of the sum of the 8 directions: K consecutive disparities per lane
// and direction, summed as 16-bit pairs.  Bound by HBM.  1242 x 375, D = 128:
// 96 us (one pixel per warp, 4 bytes a load) -> 72 us.
template <int D>
__global__ void __launch_bounds__(kWtaWarps * 32) k_sgm_wta(SgmJob S) {
    constexpr int K = Split<D>::kOther, G = D / K, kWords = K / 4;
    using Vec = typename Bytes<K>::Vec;
    const int lane = threadIdx.x & 31, gl = lane % G;
    const size_t np = (size_t)S.w * S.h;
    const size_t p = ((size_t)blockIdx.x * kWtaWarps + (threadIdx.x >> 5)) * (32 / G) + lane / G;
    const size_t o = min(p, np - 1) * D + gl * K;
    Vec v[kDirs];
#pragma unroll
    for (int r = 0; r < kDirs; ++r) v[r] = __ldcs(reinterpret_cast<const Vec*>(S.paths + (size_t)r * np * D + o));
    uint32_t even[kWords], odd[kWords];  // bytes 0 and 2, 1 and 3 of each word
#pragma unroll
    for (int j = 0; j < kWords; ++j) even[j] = odd[j] = 0;
#pragma unroll
    for (int r = 0; r < kDirs; ++r) {
        uint32_t w[kWords];
        memcpy(w, &v[r], sizeof w);
#pragma unroll
        for (int j = 0; j < kWords; ++j) {
            even[j] += w[j] & 0x00ff00ffu;
            odd[j] += (w[j] >> 8) & 0x00ff00ffu;
        }
    }
    // key = sum << 8 | d: the smallest key is the lowest sum, then the lowest d
    uint32_t key = 0xffffffffu;
#pragma unroll
    for (int j = 0; j < kWords; ++j) {
        const uint32_t d = gl * K + 4 * j;
        key = min(key, (even[j] << 16) >> 8 | d);
        key = min(key, (odd[j] << 16) >> 8 | (d + 1));
        key = min(key, (even[j] >> 16) << 8 | (d + 2));
        key = min(key, (odd[j] >> 16) << 8 | (d + 3));
    }
#pragma unroll
    for (int o2 = 1; o2 < G; o2 <<= 1) key = min(key, __shfl_xor_sync(kFull, key, o2));
    if (gl == 0 && p < np) S.disp[p] = (int16_t)(key & 0xff);
}

int check_sgm(const sff_sgm_params* P) {
    if (!P) return SFF_ERR_ARG;
    if (P->max_disp != 32 && P->max_disp != 64 && P->max_disp != 128 && P->max_disp != 256) return SFF_ERR_ARG;
    if (P->p1 < 0 || P->p2 < P->p1 || P->p2 > 193) return SFF_ERR_ARG;
    return SFF_OK;
}

struct SgmLayout {
    size_t census0, census1, cost, paths, total;
};

SgmLayout sgm_layout(int w, int h, int D) {
    const size_t np = (size_t)w * h;
    SgmLayout L;
    L.census0 = 0;
    L.census1 = align256(np * 8);
    L.cost = L.census1 + align256(np * 8);
    L.paths = L.cost + align256(np * D);
    L.total = L.paths + align256(np * kDirs * D);
    return L;
}

template <int D>
int launch_sgm(const SgmJob& S, cudaStream_t st) {
    const size_t np = (size_t)S.w * S.h;
    SFF_LAUNCH(k_sgm_cost<D>, dim3((S.w + kCostSeg - 1) / kCostSeg, S.h), kCostThreads, 0, st, S);
    using P = Split<D>;
    const int lines = S.w + S.h - 1;  // the diagonals have the most lines
    SFF_LAUNCH(k_sgm_paths<D>, dim3(2 * P::blocks_across(S.h) + (kDirs - 2) * P::blocks(lines)), 32, 0, st, S);
    constexpr int kPix = kWtaWarps * 32 / (D / P::kOther);  // pixels per CTA
    SFF_LAUNCH(k_sgm_wta<D>, dim3((unsigned)((np + kPix - 1) / kPix)), kWtaWarps * 32, 0, st, S);
    return SFF_OK;
}

}  // namespace
}  // namespace sff

extern "C" int sff_default_sgm_params(sff_sgm_params* out) {
    if (!out) return SFF_ERR_ARG;
    out->max_disp = 128;
    out->p1 = 10;
    out->p2 = 120;
    return SFF_OK;
}

extern "C" size_t sff_sgm_workspace_bytes(int32_t width, int32_t height, const sff_sgm_params* params) {
    if (sff::check_size(width, height) || sff::check_sgm(params)) return 0;
    return sff::sgm_layout(width, height, params->max_disp).total;
}

extern "C" int sff_sgm(const uint8_t* left_dev, const uint8_t* right_dev, int32_t pitch_bytes, int32_t width,
                       int32_t height, const sff_sgm_params* params, int16_t* disp_dev, void* workspace,
                       size_t workspace_bytes, void* stream) {
    using namespace sff;
    if (check_size(width, height) || check_sgm(params)) return SFF_ERR_ARG;
    if (!left_dev || !right_dev || !disp_dev || !workspace || pitch_bytes < 3 * width) return SFF_ERR_ARG;
    if (((uintptr_t)disp_dev & 1) || ((uintptr_t)workspace & 255)) return SFF_ERR_ARG;
    const SgmLayout L = sgm_layout(width, height, params->max_disp);
    if (workspace_bytes < L.total) return SFF_ERR_WORKSPACE;
    char* ws = reinterpret_cast<char*>(workspace);
    SgmJob S;
    S.img[0] = left_dev;
    S.img[1] = right_dev;
    S.pitch = pitch_bytes;
    S.w = width;
    S.h = height;
    S.D = params->max_disp;
    S.p1 = params->p1;
    S.p2 = params->p2;
    S.census[0] = reinterpret_cast<uint64_t*>(ws + L.census0);
    S.census[1] = reinterpret_cast<uint64_t*>(ws + L.census1);
    S.cost = reinterpret_cast<uint8_t*>(ws + L.cost);
    S.paths = reinterpret_cast<uint8_t*>(ws + L.paths);
    S.disp = disp_dev;
    cudaStream_t st = (cudaStream_t)stream;
    SFF_LAUNCH(k_sgm_census, dim3((width + kTileX - 1) / kTileX, (height + kTileY - 1) / kTileY, 2),
               dim3(kTileX, kTileY), 0, st, S);
    const int rc = S.D == 32 ? launch_sgm<32>(S, st) : S.D == 64 ? launch_sgm<64>(S, st)
                   : S.D == 128 ? launch_sgm<128>(S, st) : launch_sgm<256>(S, st);
    return rc != SFF_OK ? rc : launch_status();
}
