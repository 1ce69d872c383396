// Features of the paper's own matching cost (Sec. 3.1, "Matching Cost",
// Eq. 1): per pixel and scale the first three principal components phi of a
// dense SIFT descriptor, the principal axes computed over the descriptors of
// all four images.
//
// Readings (the paper names SIFTFlow's dense SIFT and the three principal
// components, nothing more):
//   - grey (R + 2G + B + 2) >> 2 of the scale's box-smoothed image (the
//     smoothing of the WHT features: n x n box, window -n/2 .. n/2 - 1,
//     clamped, rounded half up per channel);
//   - gradient with stride n, central differences, clamped; magnitude
//     sqrt(dx^2 + dy^2) in single precision; orientation sector k of 45
//     degrees by exact integer cross products with the sector rays;
//   - 4 x 4 cells of 3 x 3 samples at stride n around the pixel (offsets
//     -6 n .. 5 n, clamped), each cell's 8 bins summing its samples in
//     row-major order; 128 sums normalised, clipped at 0.2, renormalised,
//     quantised to min(255, (int)(v 512 + 0.5));
//   - axes: exact integer sums over the full-resolution descriptors of the
//     four images, covariance in double precision, 200 power iterations per
//     axis from the all-ones vector with deflation, sign of the largest
//     component positive; each dot product of an iteration as four partial
//     sums over the indices mod 4, each by fused multiply-adds in index
//     order, combined as (s0 + s1) + (s2 + s3);
//   - phi_c = sum_k fl(a_ck) q_k in single precision, minus fl(a_c . mean).
// Every floating-point operation is written out with the _rn intrinsics, in
// the order of the definition: fused multiply-adds only where the definition
// names them (the power iteration's dot products), no reassociation, so the
// results are reproducible bit for bit on any IEEE machine.
//
// k_sift_grey:    smoothed grey image of one scale (4 images, blockIdx.z).
// k_sift_desc:    gradients, cell sums and quantised descriptors of a tile of
//                 pixels, one thread per pixel.
// k_sift_cov:     sums and sums of products of the descriptors on the tensor
//                 cores, exact, into 64-bit integers.
// k_sift_axes:    one cluster of four CTAs: mean, covariance, power
//                 iterations, projection weights.
// k_sift_project: phi of every pixel of one scale of the four images.
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include <cuda_fp16.h>

#include "sff_internal.cuh"
#include "sff_tc.cuh"

namespace sff {
namespace {

constexpr int kDesc = 128;
// k_sift_desc: pixels per CTA (of one residue class mod n), the samples and
// the cell positions that their descriptors read
constexpr int kTileW = 32, kTileH = 16;
constexpr int kSampW = kTileW + 11, kSampH = kTileH + 11;
constexpr int kCellW = kTileW + 9, kCellH = kTileH + 9;
constexpr int kPowerIters = 200;

struct SiftJob {
    const uint8_t* rgb[4];
    int pitch, w, h, s, n;
    uint8_t* grey;           // [4][H][W]
    uint8_t* desc;           // [4][H][W][128]
    unsigned long long* s1;  // [128] sums
    unsigned long long* s2;  // [128][128] sums of products of (component - 128), entries j >= i
    double* axes;            // [3][128]
    float* proj;             // [3][128] single-precision axes, then [3] biases
    float* phi[4];           // [S][H][W][4] each
};

__device__ __forceinline__ const uint8_t* img_of(const SiftJob& J, int v) {
    return v == 0 ? J.rgb[0] : v == 1 ? J.rgb[1] : v == 2 ? J.rgb[2] : J.rgb[3];
}
__device__ __forceinline__ float* phi_of(const SiftJob& J, int v) {
    return v == 0 ? J.phi[0] : v == 1 ? J.phi[1] : v == 2 ? J.phi[2] : J.phi[3];
}

__global__ void k_sift_grey(SiftJob J) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y, v = blockIdx.z;
    if (x >= J.w) return;
    const uint8_t* img = img_of(J, v);
    int c[3];
    if (J.n == 1) {
        const uint8_t* p = img + (size_t)y * J.pitch + 3 * x;
        c[0] = p[0];
        c[1] = p[1];
        c[2] = p[2];
    } else {
        int sum[3] = {0, 0, 0};
        for (int j = -J.n / 2; j <= J.n / 2 - 1; ++j)
            for (int i = -J.n / 2; i <= J.n / 2 - 1; ++i) {
                const uint8_t* p = img + (size_t)clampi(y + j, 0, J.h - 1) * J.pitch + 3 * clampi(x + i, 0, J.w - 1);
                sum[0] += p[0];
                sum[1] += p[1];
                sum[2] += p[2];
            }
        const int a = J.n * J.n;
        for (int k = 0; k < 3; ++k) c[k] = (sum[k] + a / 2) / a;
    }
    J.grey[((size_t)v * J.h + y) * J.w + x] = (uint8_t)((c[0] + 2 * c[1] + c[2] + 2) >> 2);
}

// Sector k of a direction: [45 k, 45 k + 45) degrees, by sign and magnitude
// after a half turn of the lower half-plane (any sector for a zero gradient,
// whose magnitude is 0).
__device__ __forceinline__ int sector_of(int dx, int dy) {
    const bool lower = dy < 0 || (dy == 0 && dx < 0);
    if (lower) {
        dx = -dx;
        dy = -dy;
    }
    const int k = dx > 0 ? (dy < dx ? 0 : 1) : (-dx < dy ? 2 : 3);
    return lower ? k + 4 : k;
}

// Correctly rounded a / b for many a: with y = RN(1 / b), a faithful quotient
// q and the exact remainder r = a - q b, RN(q + r y) = RN(a / b) (Markstein,
// "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990, theorem on division).  q is faithful here because it is
// rounded once from a (y + lo) with y + lo within 2^-47 of 1 / b.  Needs 0 <=
// a <= 2^20 b with a and b in the normal range's middle (nothing below
// underflows): magnitudes are 0 or at least 1 and at most 9 x 361 per bin.
struct Divisor {
    float b, y, lo;
};
__device__ __forceinline__ Divisor divisor_of(float b) {
    Divisor d;
    d.b = b > 0.0f ? b : 1.0f;  // an all-zero descriptor stays all zero
    d.y = __frcp_rn(d.b);
    d.lo = __fmul_rn(__fmaf_rn(-d.b, d.y, 1.0f), d.y);
    return d;
}
__device__ __forceinline__ float quotient(float a, const Divisor& d) {
    const float q = __fmaf_rn(a, d.y, __fmul_rn(a, d.lo));
    return __fmaf_rn(__fmaf_rn(-q, d.b, a), d.y, q);
}

// Descriptors of a tile of kTileW x kTileH pixels whose coordinates share a
// residue mod n, one thread per pixel.  A cell's 8 sums depend only on its
// position, so they are computed once per position (kCellW x kCellH of them,
// two per pixel) and read by the 16 descriptors that contain the cell; the
// samples are n apart, hence the residue classes.  A bin's sum adds +0 for the
// samples of the other sectors, which leaves it bit-identical to adding only
// its own.  The thread reads its 128 values from shared memory three times
// (norm, clipped norm, result): holding them would leave 12 warps per SM.  The
// two halves of a position are separate planes, so that a warp's 16-byte
// reads are conflict-free.  Bound by issue: per value 2 + 7 + 11 operations.
// 1242 x 375, four images, four scales: 5127 us (each pixel's cells computed by
// four threads, IEEE divide routine, separate gradient kernel of 55 us) ->
// 929 us.
__global__ void __launch_bounds__(kTileW * kTileH, 3) k_sift_desc(SiftJob J) {
    __shared__ float4 cell[2][kCellW * kCellH];
    __shared__ float mag[kSampW * kSampH];
    __shared__ uint8_t bin[kSampW * kSampH];
    const int n = J.n, t = threadIdx.x;
    // residue (a, b) and tile
    const int a = (int)blockIdx.x % n, b = (int)blockIdx.y % n;
    const int x0 = a + n * kTileW * ((int)blockIdx.x / n), y0 = b + n * kTileH * ((int)blockIdx.y / n);
    if (x0 >= J.w || y0 >= J.h) return;  // CTA-uniform
    const size_t plane = (size_t)blockIdx.z * J.h * J.w;
    const uint8_t* g = J.grey + plane;
    // sample i of a row is image column x0 + n (i - 6), clamped
    for (int k = t; k < kSampW * kSampH; k += kTileW * kTileH) {
        const int x = clampi(x0 + n * (k % kSampW - 6), 0, J.w - 1), y = clampi(y0 + n * (k / kSampW - 6), 0, J.h - 1);
        const uint8_t* row = g + (size_t)y * J.w;
        const int dx = (int)row[min(x + n, J.w - 1)] - (int)row[max(x - n, 0)];
        const int dy = (int)g[(size_t)min(y + n, J.h - 1) * J.w + x] - (int)g[(size_t)max(y - n, 0) * J.w + x];
        mag[k] = __fsqrt_rn((float)(dx * dx + dy * dy));
        bin[k] = (uint8_t)sector_of(dx, dy);
    }
    __syncthreads();
    for (int k = t; k < kCellW * kCellH; k += kTileW * kTileH) {
        const int o = (k / kCellW) * kSampW + k % kCellW;
        float h[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) h[q] = 0.0f;
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const float m = mag[o + j * kSampW + i];
                const int s = bin[o + j * kSampW + i];
#pragma unroll
                for (int q = 0; q < 8; ++q) h[q] = __fadd_rn(h[q], s == q ? m : 0.0f);
            }
        cell[0][k] = make_float4(h[0], h[1], h[2], h[3]);
        cell[1][k] = make_float4(h[4], h[5], h[6], h[7]);
    }
    __syncthreads();
    const int px = t % kTileW, py = t / kTileW;
    const int x = x0 + n * px, y = y0 + n * py;
    if (x >= J.w || y >= J.h) return;
    const float4* c0 = &cell[0][py * kCellW + px];  // position of cell (0, 0); cells are 3 apart
    constexpr int kHalf = kCellW * kCellH;
    float ss = 0.0f;
#pragma unroll 1
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 v = c0[3 * j * kCellW + 3 * (i >> 1) + (i & 1) * kHalf];
            ss = __fadd_rn(ss, __fmul_rn(v.x, v.x));
            ss = __fadd_rn(ss, __fmul_rn(v.y, v.y));
            ss = __fadd_rn(ss, __fmul_rn(v.z, v.z));
            ss = __fadd_rn(ss, __fmul_rn(v.w, v.w));
        }
    const Divisor d1 = divisor_of(__fsqrt_rn(ss));
    ss = 0.0f;
#pragma unroll 1
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 v = c0[3 * j * kCellW + 3 * (i >> 1) + (i & 1) * kHalf];
            const float c[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float u = fminf(quotient(c[q], d1), 0.2f);
                ss = __fadd_rn(ss, __fmul_rn(u, u));
            }
        }
    const Divisor d2 = divisor_of(__fsqrt_rn(ss));
    uint8_t* out = J.desc + (plane + (size_t)y * J.w + x) * kDesc;
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
        uint32_t word[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 v = c0[3 * j * kCellW + 3 * (i >> 1) + (i & 1) * kHalf];
            const float c[4] = {v.x, v.y, v.z, v.w};
            uint32_t q8[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                // u 512 is exact, so one fused step rounds like the sum; adding
                // 2^23 towards zero leaves the truncated integer in the low bits
                const float u = quotient(fminf(quotient(c[q], d1), 0.2f), d2);
                q8[q] = __float_as_uint(__fadd_rz(fminf(__fmaf_rn(u, 512.0f, 0.5f), 255.0f), 8388608.0f));
            }
            word[i] = __byte_perm(__byte_perm(q8[0], q8[1], 0x0040), __byte_perm(q8[2], q8[3], 0x0040), 0x5410);
        }
        // one 32-byte store per cell row: whole sectors
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(out + 32 * j), "r"(word[0]),
                     "r"(word[1]), "r"(word[2]), "r"(word[3]), "r"(word[4]), "r"(word[5]), "r"(word[6]), "r"(word[7])
                     : "memory");
    }
}

// Sums of the descriptors and of their pairwise products over the four
// images' full-resolution descriptors: one matrix product S2 = Q Q^T on the
// tensor cores, Q = the 128 x count matrix of the descriptors less 128, in
// fp16 (integers -128..127, exact).  A product is at most 2^14 in magnitude, so
// the fp32 sums of kCovGroup = 1024 descriptors are exact in any order; then
// they are added to 32-bit integers in registers and, before those can
// overflow, to the 64-bit sums in memory.  Both operands are the same tile: a
// descriptor's 8 consecutive components are 16 bytes of an MN-major core
// matrix, so the conversion needs no transposition.  One CTA per SM; each step
// converts kCovStep descriptors that were loaded two steps earlier, one thread
// issues the MMAs, and the next steps fill other stages meanwhile.  Bound by the
// descriptor reads.  1242 x 375 (1.86 M descriptors): 1419 us (dp4a over a
// shared-memory transpose) -> 159 us.
constexpr int kCovStep = 128;                   // descriptors per step (K)
constexpr int kCovStages = 3;                   // steps in shared memory
constexpr int kCovGroup = 1024;                 // descriptors per exact fp32 sum
constexpr int kCovSteps = kCovGroup / kCovStep;
constexpr int kCovMaxGroups = 120;              // groups per 32-bit sum: 120 * 2^24 < 2^31
constexpr int kCovThreads = 512;
constexpr int kCovCtas = 152;                   // one per SM
constexpr int kCovStageBytes = kCovStep * kDesc * 2;
constexpr int kCovKGroup = kDesc * 16;          // bytes between K groups of 8 descriptors
constexpr int kCovSmemBytes = kCovStages * kCovStageBytes + 1024;  // + alignment slack
// instruction descriptor, kind::f16: fp32 D (bits 4-5 = 1), fp16 A and B (bits
// 7-12 = 0), both MN-major (bits 15, 16), N = M = 128
constexpr uint32_t kCovIdesc =
    (1u << 4) | (1u << 15) | (1u << 16) | ((uint32_t)(kDesc >> 3) << 17) | ((uint32_t)(kDesc >> 4) << 24);

__device__ unsigned int g_sift_status;  // bit 0: a bounded wait of k_sift_cov gave up; bit 1: its drain did

// 4 components as two fp16 pairs, each less 128 (1024 + b as a bit pattern,
// then an exact subtraction).
__device__ __forceinline__ uint2 centred_halves(uint32_t w) {
    const __half2 off = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));  // 1152
    const uint32_t lo = __byte_perm(w, 0x64646464u, 0x4140), hi = __byte_perm(w, 0x64646464u, 0x4342);
    const __half2 a = __hsub2(*reinterpret_cast<const __half2*>(&lo), off);
    const __half2 b = __hsub2(*reinterpret_cast<const __half2*>(&hi), off);
    return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}

__global__ void __launch_bounds__(kCovThreads, 1) k_sift_cov(SiftJob J, size_t count) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar[kCovStages];
    __shared__ uint32_t tmem_slot;
    __shared__ uint32_t s1[kDesc];
    uint8_t* sm = smem_raw + ((1024 - (smem_addr(smem_raw) & 1023)) & 1023);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) {
        for (int k = 0; k < kCovStages; ++k) mbar_init(&bar[k], 1);
        mbar_fence_init();
    }
    if (t < kDesc) s1[t] = 0;
    if (warp == 0) tmem_alloc(&tmem_slot, kDesc);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    const size_t steps_all = (count + kCovStep - 1) / kCovStep;
    const int steps = (int)((steps_all - blockIdx.x + gridDim.x - 1) / gridDim.x);  // grid <= steps_all
    // this thread's part of a step: descriptor 8 warp + lane % 8 (its K group
    // is the warp's), components 16 c .. 16 c + 15 for c = lane / 8 and c + 4; a
    // quarter warp then writes 128 contiguous bytes
    const int kd = 8 * warp + (lane & 7), c0 = lane >> 3;
    auto load = [&](int u, uint4 (&v)[2]) {
        const size_t d = ((size_t)blockIdx.x + (size_t)u * gridDim.x) * kCovStep + kd;
        const uint4* src = reinterpret_cast<const uint4*>(J.desc + d * kDesc);
        const bool in = u < steps && d < count;
#pragma unroll
        for (int r = 0; r < 2; ++r)  // past the end: 128 = a centred 0
            v[r] = in ? __ldg(src + c0 + 4 * r) : make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
        return in;
    };
    int acc[32];  // component i = 32 (warp % 4) + lane against components 32 (warp / 4) ..
#pragma unroll
    for (int e = 0; e < 32; ++e) acc[e] = 0;
    uint32_t part[2][8];  // 16-bit sums of this thread's components: even, odd bytes of each word
#pragma unroll
    for (int e = 0; e < 16; ++e) part[e >> 3][e & 7] = 0;
    auto flush = [&]() {  // the CTA's sums to memory
        const int i = 32 * (warp & 3) + lane;
#pragma unroll
        for (int e = 0; e < 32; ++e) {
            const int j = 32 * (warp >> 2) + e;
            if (j >= i) atomicAdd(J.s2 + i * kDesc + j, (unsigned long long)(long long)acc[e]);
            acc[e] = 0;
        }
        __syncthreads();
        if (t < kDesc) {
            atomicAdd(J.s1 + t, (unsigned long long)s1[t]);
            s1[t] = 0;
        }
        __syncthreads();
    };

    uint4 cur[2], nxt[2];
    bool cur_in = load(0, cur), nxt_in = load(1, nxt);
    bool ok = true, failed = false;
    int issued = 0, groups = 0;
    for (int u = 0; u < steps; ++u) {
        const int s = u % kCovStages;
        if (u >= kCovStages) ok = ok && mbar_wait(&bar[s], (unsigned)(u / kCovStages - 1) & 1u, kDefaultWaitNs);
        uint8_t* stage = sm + s * kCovStageBytes + warp * kCovKGroup + (lane & 7) * 16;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const uint32_t w[4] = {cur[r].x, cur[r].y, cur[r].z, cur[r].w};
            uint2 h[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                h[e] = centred_halves(w[e]);
                if (cur_in) {
                    part[r][2 * e] += w[e] & 0x00ff00ffu;
                    part[r][2 * e + 1] += (w[e] >> 8) & 0x00ff00ffu;
                }
            }
            // component groups 2 c and 2 c + 1 of 8
            uint4* dst = reinterpret_cast<uint4*>(stage + 256 * (c0 + 4 * r));
            dst[0] = make_uint4(h[0].x, h[0].y, h[1].x, h[1].y);
            dst[8] = make_uint4(h[2].x, h[2].y, h[3].x, h[3].y);
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) cur[r] = nxt[r];
        cur_in = nxt_in;
        nxt_in = load(u + 2, nxt);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the stage visible to the tensor cores
        tc_fence_before();
        if (!__syncthreads_and(ok)) {
            failed = true;
            break;
        }
        tc_fence_after();
        if (t == 0) {
            const uint32_t base = smem_addr(sm + s * kCovStageBytes);
#pragma unroll
            for (int k = 0; k < kCovStep / 16; ++k) {
                const uint64_t d = smem_desc(base + 2 * k * kCovKGroup, kCovKGroup, 128);
                tc_mma(tmem, d, d, kCovIdesc, u % kCovSteps != 0 || k > 0);
            }
            tc_commit(&bar[s]);
        }
        issued = u + 1;
        if (u % kCovSteps == kCovSteps - 1 || u == steps - 1) {
            // the group's sums out of tensor memory before the next MMA, which
            // follows the next barrier, starts them anew
            ok = __all_sync(0xffffffffu, mbar_wait(&bar[s], (unsigned)(u / kCovStages) & 1u, kDefaultWaitNs));
            if (ok) {
                tc_fence_after();
                uint32_t v[32];
                tmem_ld32(tmem + ((uint32_t)(32 * (warp & 3)) << 16), v, 32 * (warp >> 2));
                tmem_ld_wait(v);
                tc_fence_before();
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[e] += __float2int_rn(__uint_as_float(v[e]));
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    uint32_t* dst = s1 + 16 * (c0 + 4 * r) + 4 * (e >> 1) + (e & 1);
                    atomicAdd(dst, part[r][e] & 0xffffu);
                    atomicAdd(dst + 2, part[r][e] >> 16);
                    part[r][e] = 0;
                }
            if (++groups == kCovMaxGroups) {
                flush();
                groups = 0;
            }
        }
    }
    if (!failed && !__syncthreads_and(ok)) failed = true;
    if (failed) {
        // status, and the MMAs in flight complete before the tensor memory is released
        if (t == 0) {
            atomicOr(&g_sift_status, 1u);
            if (issued > 0 && !mbar_wait(&bar[(issued - 1) % kCovStages], (unsigned)((issued - 1) / kCovStages) & 1u,
                                         kDrainFactor * kDefaultWaitNs))
                atomicOr(&g_sift_status, 2u);
        }
    } else {
        flush();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, kDesc);
}

// Sum of the products of components i and j over the count descriptors, from
// the sums of the centred ones: (a - 128)(b - 128) = a b - 128 (a + b) + 128^2.
__device__ __forceinline__ double product_sum(const SiftJob& J, int i, int j, double count) {
    const long long c = (long long)J.s2[i < j ? i * kDesc + j : j * kDesc + i];
    return (double)(c + 128ll * (long long)(J.s1[i] + J.s1[j]) - 16384ll * (long long)count);
}

// The principal axes, by one cluster of kAxesCtas CTAs.  The FP64 pipe bounds
// it: a warp's DFMA holds its SM sub-partition for 64 clocks however many lanes
// are active, and the definition fixes the order of every sum, so an iteration
// is a chain of 32 dependent DFMAs for the matrix rows, 32 for each deflation
// dot product and 32 for the norm.  One thread per (row, residue mod 4) chain:
// 512 chains are 16 warps, one per sub-partition of four SMs, so the rows take
// one chain's time (2080 clocks) instead of the four that one SM needs.  A
// thread keeps its 32 covariance entries and the earlier axes' entries of its
// residue in registers; each row's sum goes to all four CTAs through
// distributed shared memory, one cluster barrier per iteration.  The dot
// products are computed by every warp for itself (its own sub-partition would
// idle otherwise), so they need no barrier.  5573 -> 3169 us (one CTA before).
constexpr int kAxesCtas = 4;
constexpr int kChain = kDesc / 4;  // terms of one residue's sum

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Stores v at the address that p has in the shared memory of CTA `rank`.
__device__ __forceinline__ void store_remote(double* p, int rank, double v) {
    asm volatile(
        "{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %0, %1;\n\tst.shared::cluster.f64 [a], %2;\n\t}" ::"r"(
            (unsigned)__cvta_generic_to_shared(p)),
        "r"(rank), "d"(v)
        : "memory");
}

// (s0 + s1) + (s2 + s3) of the partial sums of four neighbouring lanes (lane
// mod 4 = the residue), on every lane.
__device__ __forceinline__ double combine4(double s) {
    s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, 1));
    return __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, 2));
}

// Axis c by the power iteration.  cov: this thread's row at its residue; ax /
// axr: the earlier axes, whole in shared memory / at this thread's residue.
template <int c>
__device__ __forceinline__ void power_axis(const double (&cov)[kChain], const double (&axr)[2][kChain],
                                           double (*ax)[kDesc], double* v, double (*raw)[kDesc], double (*upd)[kDesc]) {
    const int i = threadIdx.x, r = i & 3;
    const int row = (int)blockIdx.x * (kDesc / kAxesCtas) + (i >> 2);
    v[i] = 1.0;
    __syncthreads();
    double vi = 0.0;
    for (int it = 0; it < kPowerIters; ++it) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < kChain; ++k) s = __fma_rn(cov[k], v[4 * k + r], s);
        s = combine4(s);
        // the buffers alternate: a CTA writes one again only after the next
        // barrier, which every CTA reaches when it has read it
        double* w = raw[it & 1];
        store_remote(w + row, r, s);
        cluster_barrier();
        double wi = w[i];
#pragma unroll
        for (int e = 0; e < c; ++e) {
            double t = 0.0;
#pragma unroll
            for (int k = 0; k < kChain; ++k) t = __fma_rn(axr[e][k], w[4 * k + r], t);
            wi = __dsub_rn(wi, __dmul_rn(combine4(t), ax[e][i]));
            w = upd[e];
            w[i] = wi;
            __syncthreads();
        }
        double t = 0.0;
#pragma unroll
        for (int k = 0; k < kChain; ++k) t = __fma_rn(w[4 * k + r], w[4 * k + r], t);
        const double nr = __dsqrt_rn(combine4(t));
        vi = nr > 0.0 ? __ddiv_rn(wi, nr) : 0.0;
        v[i] = vi;
        __syncthreads();
    }
    // the largest component (the first of equals) made positive; magnitudes
    // order like their bit patterns
    if (i < 32) {
        unsigned long long best = 0ull;
        int big = 0;
        for (int k = i; k < kDesc; k += 32) {
            const unsigned long long m = (unsigned long long)__double_as_longlong(v[k]) & 0x7fffffffffffffffull;
            if (k == i || m > best) {
                best = m;
                big = k;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long om = __shfl_xor_sync(0xffffffffu, best, o);
            const int ob = __shfl_xor_sync(0xffffffffu, big, o);
            if (om > best || (om == best && ob < big)) {
                best = om;
                big = ob;
            }
        }
        if (i == 0) raw[0][0] = v[big] < 0.0 ? -1.0 : 1.0;
    }
    __syncthreads();
    ax[c][i] = __dmul_rn(raw[0][0], vi);
    // no CTA writes raw[0] again (the next axis) before all have read the sign
    cluster_barrier();
}

__global__ void __cluster_dims__(kAxesCtas, 1, 1) __launch_bounds__(kDesc) k_sift_axes(SiftJob J, double count) {
    __shared__ double mean[kDesc], v[kDesc], ax[3][kDesc], raw[2][kDesc], upd[2][kDesc];
    const int i = threadIdx.x, r = i & 3;
    const int row = (int)blockIdx.x * (kDesc / kAxesCtas) + (i >> 2);
    mean[i] = __ddiv_rn((double)J.s1[i], count);
    __syncthreads();
    double cov[kChain], axr[2][kChain];
#pragma unroll
    for (int k = 0; k < kChain; ++k)
        cov[k] = __dsub_rn(__ddiv_rn(product_sum(J, row, 4 * k + r, count), count),
                           __dmul_rn(mean[row], mean[4 * k + r]));
    cluster_barrier();  // every CTA of the cluster runs before the first remote store
    power_axis<0>(cov, axr, ax, v, raw, upd);
#pragma unroll
    for (int k = 0; k < kChain; ++k) axr[0][k] = ax[0][4 * k + r];
    power_axis<1>(cov, axr, ax, v, raw, upd);
#pragma unroll
    for (int k = 0; k < kChain; ++k) axr[1][k] = ax[1][4 * k + r];
    power_axis<2>(cov, axr, ax, v, raw, upd);
    if (blockIdx.x != 0) return;  // the last cluster barrier is behind every remote store
    // axes, single-precision projection weights and biases fl(a_c . mean),
    // the bias a sequential sum
    for (int c = 0; c < 3; ++c) {
        J.axes[c * kDesc + i] = ax[c][i];
        J.proj[c * kDesc + i] = (float)ax[c][i];
    }
    if (i < 3) {
        double b = 0.0;
        for (int k = 0; k < kDesc; ++k) b = __dadd_rn(b, __dmul_rn(ax[i][k], mean[k]));
        J.proj[3 * kDesc + i] = (float)b;
    }
}

// phi of one scale, two pixels per thread, so that a weight is read from shared
// memory once for both.  The descriptors come through shared memory by coalesced
// asynchronous copies (a thread's own 128 bytes are four lines away from its
// neighbour's; rows padded by 16 bytes, conflict-free).  A byte becomes a float as the low bits of 2^23 (one
// byte permute), less 2^23: the conversion instruction runs at an eighth of
// the FP32 rate.  Bound by the FP32 pipe (7 operations per component and
// pixel; packed pairs issue half as often but pass at the same rate, and the
// assembler contracts their products and sums).  1242 x 375, four images:
// 105 us a scale (one pixel per thread, conversions) -> 84 us.
constexpr int kProjThreads = 128;

__global__ void __launch_bounds__(kProjThreads) k_sift_project(SiftJob J) {
    __shared__ float4 a[kDesc];  // the three weights of a component
    __shared__ uint4 row[2 * kProjThreads][kDesc / 16 + 1];
    const int v = blockIdx.y;
    const size_t np = (size_t)J.w * J.h;
    const size_t first = (size_t)blockIdx.x * (2 * kProjThreads);
    const uint4* desc = reinterpret_cast<const uint4*>(J.desc + ((size_t)v * np + first) * kDesc);
    const int chunks = (int)min((size_t)(2 * kProjThreads), np - first) * (kDesc / 16);
    for (int e = threadIdx.x; e < chunks; e += kProjThreads)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                         (unsigned)__cvta_generic_to_shared(&row[e / (kDesc / 16)][e % (kDesc / 16)])),
                     "l"(desc + e)
                     : "memory");
    for (int k = threadIdx.x; k < kDesc; k += kProjThreads)
        a[k] = make_float4(J.proj[k], J.proj[kDesc + k], J.proj[2 * kDesc + k], 0.0f);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    const size_t p0 = first + threadIdx.x, p1 = p0 + kProjThreads;
    if (p0 >= np) return;
    const uint4 *q0 = row[threadIdx.x], *q1 = row[p1 < np ? threadIdx.x + kProjThreads : threadIdx.x];
    float t[2][3] = {{0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}};
#pragma unroll 2
    for (int k16 = 0; k16 < kDesc / 16; ++k16) {  // 16 components per load, in index order
        const uint4 w0 = q0[k16], w1 = q1[k16];
        const uint32_t u[2][4] = {{w0.x, w0.y, w0.z, w0.w}, {w1.x, w1.y, w1.z, w1.w}};
#pragma unroll
        for (int b = 0; b < 16; ++b) {
            const float4 w = a[k16 * 16 + b];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float q =
                    __fsub_rn(__uint_as_float(__byte_perm(u[i][b >> 2], 0x4b000000u, 0x7650u + (b & 3))), 8388608.0f);
                t[i][0] = __fadd_rn(t[i][0], __fmul_rn(w.x, q));
                t[i][1] = __fadd_rn(t[i][1], __fmul_rn(w.y, q));
                t[i][2] = __fadd_rn(t[i][2], __fmul_rn(w.z, q));
            }
        }
    }
    float4* phi = reinterpret_cast<float4*>(phi_of(J, v)) + (size_t)J.s * np;
    const float b0 = J.proj[3 * kDesc], b1 = J.proj[3 * kDesc + 1], b2 = J.proj[3 * kDesc + 2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
        if (i == 0 || p1 < np)
            phi[i ? p1 : p0] =
                make_float4(__fsub_rn(t[i][0], b0), __fsub_rn(t[i][1], b1), __fsub_rn(t[i][2], b2), 0.0f);
}

struct SiftLayout {
    size_t grey, desc, s1, s2, axes, proj, total;
};

// scales: how many scales' descriptors are held at once.
SiftLayout sift_layout(int w, int h, int scales) {
    const size_t np = (size_t)w * h;
    SiftLayout L;
    L.grey = 0;
    L.desc = L.grey + align256(4 * np);
    L.s1 = L.desc + align256((size_t)scales * 4 * np * kDesc);
    L.s2 = L.s1 + align256(kDesc * 8);
    L.axes = L.s2 + align256(kDesc * kDesc * 8);
    L.proj = L.axes + align256(3 * kDesc * 8);
    L.total = L.proj + align256((3 * kDesc + 3) * sizeof(float));
    return L;
}

// The scratch that sff_sift_workspace_bytes asks for holds every scale's
// descriptors up to this size (2 KB per pixel, 4.0 GiB at most), so that the
// coarser scales' can be computed while the axes are; a larger image's holds
// one scale's.
constexpr size_t kOverlapPixels = (size_t)1 << 21;

int scratch_scales(int w, int h) { return (size_t)w * h <= kOverlapPixels ? SFF_MAX_SCALES : 1; }

// The stream on which the axes are computed, one per (device, caller stream),
// made at the first call on that pair and kept until exit.  Its priority is the
// highest: the axes' four CTAs take the first free SMs, while the caller's
// stream fills the others with descriptors.
struct AxesStream {
    cudaStream_t s = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
    std::mutex mu;  // held from a call's fork to its join: threads may share the caller's stream

    bool make() {
        int lo = 0, hi = 0;
        if (cudaDeviceGetStreamPriorityRange(&lo, &hi) == cudaSuccess &&
            cudaStreamCreateWithPriority(&s, cudaStreamNonBlocking, hi) == cudaSuccess &&
            cudaEventCreateWithFlags(&fork, cudaEventDisableTiming) == cudaSuccess &&
            cudaEventCreateWithFlags(&join, cudaEventDisableTiming) == cudaSuccess)
            return true;
        release();
        cudaGetLastError();
        return false;
    }
    void release() {
        if (join) cudaEventDestroy(join);
        if (fork) cudaEventDestroy(fork);
        if (s) cudaStreamDestroy(s);
    }
};
constexpr size_t kMaxAxesStreams = 64;  // further caller streams run everything in order
std::mutex g_axes_mu;
std::map<std::pair<int, cudaStream_t>, AxesStream> g_axes;

// cudaStreamPerThread names another stream in each thread, so its side streams (by
// device) belong to the thread and end with it.  One for all threads would stay part
// of a capture in one of them while another's call forks to it.
struct ThreadAxes {
    std::map<int, AxesStream> by_device;
    ~ThreadAxes() {
        for (auto& e : by_device) e.second.release();
    }
};
thread_local ThreadAxes t_axes;

template <class Map, class Key>
AxesStream* made_axes(Map& m, const Key& key) {
    const auto it = m.find(key);
    if (it != m.end()) return &it->second;
    if (m.size() >= kMaxAxesStreams) return nullptr;
    AxesStream& a = m[key];
    if (a.make()) return &a;
    m.erase(key);
    return nullptr;
}

AxesStream* axes_stream(cudaStream_t st) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    if (st == cudaStreamPerThread) return made_axes(t_axes.by_device, dev);
    std::lock_guard<std::mutex> lk(g_axes_mu);
    return made_axes(g_axes, std::make_pair(dev, st));
}

}  // namespace

// Reads (and with reset clears) the condition bits of the SIFT kernels, in
// stream order; the caller synchronises the stream.
int sift_status_read(cudaStream_t st, unsigned* out, bool reset) {
    static const unsigned zero = 0;
    if (cudaMemcpyFromSymbolAsync(out, g_sift_status, sizeof(unsigned), 0, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return SFF_ERR_CUDA;
    if (reset && cudaMemcpyToSymbolAsync(g_sift_status, &zero, sizeof(unsigned), 0, cudaMemcpyHostToDevice, st) !=
                     cudaSuccess)
        return SFF_ERR_CUDA;
    return SFF_OK;
}

}  // namespace sff

extern "C" size_t sff_sift_workspace_bytes(int32_t width, int32_t height) {
    if (sff::check_size(width, height)) return 0;
    return sff::sift_layout(width, height, sff::scratch_scales(width, height)).total;
}

extern "C" int sff_sift_features(const uint8_t* const* rgb_dev4, int32_t pitch_bytes, int32_t width, int32_t height,
                                 const sff_params* params, float* const* phi_dev4, void* workspace,
                                 size_t workspace_bytes, void* stream) {
    using namespace sff;
    if (check_size(width, height) || check_params(params) || !rgb_dev4 || !phi_dev4 || !workspace) return SFF_ERR_ARG;
    if (pitch_bytes < 3 * width || ((uintptr_t)workspace & 255)) return SFF_ERR_ARG;
    for (int v = 0; v < 4; ++v)
        if (!rgb_dev4[v] || !phi_dev4[v] || ((uintptr_t)phi_dev4[v] & 15)) return SFF_ERR_ARG;
    const int S = params->num_scales;
    // every scale's descriptors at once if the scratch holds them, else one scale's at a time
    const bool overlap = S > 1 && workspace_bytes >= sift_layout(width, height, S).total;
    const SiftLayout L = sift_layout(width, height, overlap ? S : 1);
    if (workspace_bytes < L.total) return SFF_ERR_WORKSPACE;
    char* ws = reinterpret_cast<char*>(workspace);
    SiftJob J;
    for (int v = 0; v < 4; ++v) {
        J.rgb[v] = rgb_dev4[v];
        J.phi[v] = phi_dev4[v];
    }
    J.pitch = pitch_bytes;
    J.w = width;
    J.h = height;
    J.grey = reinterpret_cast<uint8_t*>(ws + L.grey);
    J.desc = reinterpret_cast<uint8_t*>(ws + L.desc);
    J.s1 = reinterpret_cast<unsigned long long*>(ws + L.s1);
    J.s2 = reinterpret_cast<unsigned long long*>(ws + L.s2);
    J.axes = reinterpret_cast<double*>(ws + L.axes);
    J.proj = reinterpret_cast<float*>(ws + L.proj);
    cudaStream_t st = (cudaStream_t)stream;
    const dim3 g((width + 127) / 128, height, 4);
    const dim3 gp((unsigned)(((size_t)width * height + 2 * kProjThreads - 1) / (2 * kProjThreads)), 4);
    // the attribute is per device: set it on the current one at every call
    if (cudaFuncSetAttribute(k_sift_cov, cudaFuncAttributeMaxDynamicSharedMemorySize, kCovSmemBytes) != cudaSuccess)
        return SFF_ERR_CUDA;
    const size_t scale_bytes = 4 * (size_t)width * height * kDesc;
    uint8_t* const desc = J.desc;
    // scale s, its descriptors in slot s (overlap) or the only one
    auto at = [&](int s) {
        J.s = s;
        J.n = 1 << s;
        J.desc = desc + (overlap ? s * scale_bytes : 0);
    };
    auto descriptors = [&]() {
        SFF_LAUNCH(k_sift_grey, g, 128, 0, st, J);
        // the n residues of a tile column (row) side by side: their pixels share sectors
        const auto tiles = [&](int len, int tile) { return (unsigned)(J.n * ((len + J.n * tile - 1) / (J.n * tile))); };
        SFF_LAUNCH(k_sift_desc, dim3(tiles(width, kTileW), tiles(height, kTileH), 4), kTileW * kTileH, 0, st, J);
    };
    // the principal axes of the full-resolution descriptors
    at(0);
    descriptors();
    if (cudaMemsetAsync(J.s1, 0, L.axes - L.s1, st) != cudaSuccess) return SFF_ERR_CUDA;
    const size_t count = 4 * (size_t)width * height;
    const int blocks = (int)std::min<size_t>((count + kCovStep - 1) / kCovStep, kCovCtas);
    SFF_LAUNCH(k_sift_cov, dim3(blocks), kCovThreads, kCovSmemBytes, st, J, count);
    // The axes keep four SMs busy for 3 ms; the coarser scales' descriptors
    // need nothing of them and are computed beside (1242 x 375: 4.75 -> 3.93 ms
    // in all).
    AxesStream* side = overlap ? axes_stream(st) : nullptr;
    if (side) {
        std::lock_guard<std::mutex> lk(side->mu);
        if (cudaEventRecord(side->fork, st) != cudaSuccess || cudaStreamWaitEvent(side->s, side->fork, 0) != cudaSuccess)
            return SFF_ERR_CUDA;
        SFF_LAUNCH(k_sift_axes, dim3(kAxesCtas), kDesc, 0, side->s, J, (double)count);
        const bool joined = cudaEventRecord(side->join, side->s) == cudaSuccess;
        for (int s = 1; s < S; ++s) {
            at(s);
            descriptors();
        }
        if (cudaStreamWaitEvent(st, side->join, 0) != cudaSuccess || !joined) return SFF_ERR_CUDA;
    } else {
        SFF_LAUNCH(k_sift_axes, dim3(kAxesCtas), kDesc, 0, st, J, (double)count);
    }
    for (int s = 0; s < S; ++s) {
        at(s);
        if (!side && s > 0) descriptors();
        SFF_LAUNCH(k_sift_project, gp, kProjThreads, 0, st, J);
    }
    return launch_status();
}
