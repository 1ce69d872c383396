// Dense interpolation of the seeds (Sec. 3.2, "Interpolation Models" and
// "Edge-Aware Neighborhood"), with Euclidean distances in place of the
// geodesic ones (the trained boundary detector is not part of this stage).
//
// Every seed gets two local models, fitted by weighted least squares over
// its nearest seeds (weights exp(-alpha D / dist_unit), D the pixel
// distance):
//   a plane of the disparity d0 over the k_geo nearest seeds, in
//   coordinates centred at the seed;
//   an affine map x1 = A (x0 - c) + t of triangulated 3D points over the
//   k_motion nearest seeds with d0, d1 >= 1, c the weighted centroid.
// The linear parts get a ridge of 1e-9 * trace / dimension towards a flat
// plane and A = I.  Every pixel takes the models of its closest seed and
// evaluates them at its own position (d0, then reproject, transform,
// project back).  Ties in all distance orders go to the lower seed index.
//
// GB300 has little double-precision throughput, and the fits run in double
// precision, so the design spends double-precision instructions only on
// the sums and the solves:
//   - the seeds of sff_emit_seeds hold at most one seed per 3x3 block
//     (anchored at (0, 0)); a block map whose words pack the seed index, the
//     motion flag and the offset inside the block gives exact nearest-seed
//     searches by rings of blocks (ring r is at least 3r - 2 px away) with
//     no seed loads;
//   - the weight depends on the integer squared distance only: a table of
//     exp(-alpha sqrt(d2) / dist_unit) for d2 < 65536, the same expression
//     as inline, serves every fit;
//   - each seed's 3D points x0, x1 are triangulated once;
//   - the neighbourhoods are selected by counting (the k-th smallest
//     (d2, index) key by bisection), not by sorting;
//   - the selected neighbours are compacted into lists, so that the sums
//     run over them alone with every lane busy;
//   - the warp sums are a reduce-scatter (N - 1 additions for N values
//     instead of 5 N), and the plane and the three rows of the affine map
//     are solved by four lanes at once.
//
// k_interp_clear:  empty map, status, weight table.
// k_interp_prep:   map words and triangulated points of every seed.
// k_interp_models: one warp per one or two seeds: one pass over rings of blocks collects
//                  the candidates of both neighbourhoods, bisection selects
//                  them, the normal equations accumulate in double precision.
// k_interp_columns: per pixel column the closest seed in that column, for
//                  every row (a sweep down and up the block map).
// k_interp_pixels: per pixel the closest seed over the columns of its row,
//                  then its models evaluated in double precision.
#include "sff_internal.cuh"

namespace sff {
namespace {

constexpr int kBlock = 3;            // sparsification block of Sec. 3.2
constexpr int kModelWarps = 1;       // warps per CTA of k_interp_models
constexpr int kModelResident = 20;   // ... and CTAs per SM that its registers allow,
constexpr int kModelResidentLone = 12;  // in the form of one seed per warp
constexpr int kMinResidentPairs = 15;  // two seeds per warp only if this many fit an SM
constexpr int kMaxK = 1024;          // largest k_geo / k_motion
constexpr int kRegKeys = 16;         // candidate keys per lane held in registers during selection (half are, up to 256)
constexpr int kTighten = 4;          // the ring bound is within 1/16 of the k-th distance so far

// Candidate slots per seed: the rings up to the bound of the k-th nearest hold about
// 4/pi times k seeds plus a margin of whole rings; 4 k + 192 leaves room for uneven
// seed density (with k = 160, a lone seed in the middle of a 480 x 480 px hole in a
// dense seed lattice meets 833).  What does not fit is compacted to the members of
// both sets so far: at most k_geo - 1 + k_motion - 1 and those tied at either k-th
// distance, 256 each (the most lattice points on a circle that fit an image of 16384
// x 16384 px, counted), and a batch of 32 more.  `whole` slots always hold these; for
// small k 6 k + 256 slots are fewer, and candidates that do not fit raise
// kErrOverflow.  With 6 k + 256 at k = 160 an SM held 16 warps instead of 20: 659 ->
// 622 us, and 612 with one warp per CTA, whose resources are free as soon as it ends.
__host__ __device__ __forceinline__ int candidate_slots(int kg, int km) {
    const int k = kg > km ? kg : km, whole = kg + km + 2 * 256 + 32;
    const int slots = 6 * k + 256 < whole ? 6 * k + 256 : whole > 4 * k + 192 ? whole : 4 * k + 192;
    return (slots + 31) & ~31;
}
constexpr int kModelDoubles = 18;    // plane 3, [A | t] 12, centre 3
constexpr int kPointDoubles = 8;     // x0 3, x1 3, d0, pad
constexpr int kSumDoubles = 32;      // plane sums 9, motion N 10 and R 12, pad
constexpr int kWeightTable = 1 << 16;
constexpr unsigned kErrSeed = 1u, kErrOverflow = 2u;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kSms = 152, kSmemPerSm = 228 * 1024, kSmemPerCta = 1024;  // shared memory of an SM, and reserved per CTA

// Map word of a block: (seed index << 5) | (motion << 4) | (ox << 2) | oy,
// (ox, oy) the seed's offset inside its block; -1 for an empty block.
__device__ __forceinline__ int word_index(int w) { return w >> 5; }
__device__ __forceinline__ bool word_motion(int w) { return (w >> 4) & 1; }

struct InterpJob {
    const sff_seed* seeds;
    const int32_t* count;
    int capacity, w, h, gbw, gbh;
    int* map;          // [gbh][gbw] words
    double* pts;       // [capacity][kPointDoubles]
    double* wt;        // [kWeightTable]
    double* models;    // [capacity][kModelDoubles]
    double* sums;      // [capacity][kSumDoubles] normal equations
    int* motion;       // [capacity] motion neighbours
    unsigned* status;  // error bits
    int* lone_max;     // k_interp_models takes one seed per warp up to this many (see there)
    sff_interp_params p;
    double fb, inv_f;  // focal * baseline, 1 / focal
    int slots;         // candidate slots per warp of k_interp_models
    int resident;      // warps of k_interp_models that the GPU holds at once
};

__device__ __forceinline__ int seed_count(const InterpJob& J) { return min(*J.count, J.capacity); }

__device__ __forceinline__ double weight_of(const InterpJob& J, unsigned d2) {
    return d2 < (unsigned)kWeightTable ? J.wt[d2] : exp(-J.p.alpha * sqrt((double)d2) / J.p.dist_unit);
}

__global__ void k_interp_clear(InterpJob J) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < J.gbw * J.gbh) J.map[i] = -1;
    if (i < kWeightTable) J.wt[i] = exp(-J.p.alpha * sqrt((double)i) / J.p.dist_unit);
    if (i == 0) {
        const int n = seed_count(J);
        *J.status = 0u;
        const bool lone = n <= J.resident || (n > 2 * J.resident && n <= J.resident * 10 / 3) || 2 * n < J.gbw * J.gbh;
        *J.lone_max = lone ? n : -1;
    }
}

// Pinhole triangulation: Z = f B / d, X = (x - cx) Z / f, Y = (y - cy) Z / f.
__device__ __forceinline__ void triangulate(const InterpJob& J, double x, double y, double d, double* X) {
    const double Z = J.fb / d;
    X[0] = (x - J.p.cx) * Z / J.p.focal;
    X[1] = (y - J.p.cy) * Z / J.p.focal;
    X[2] = Z;
}

__global__ void k_interp_prep(InterpJob J) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= seed_count(J)) return;
    const sff_seed s = J.seeds[i];
    const bool motion = s.d0 >= 1 && s.d1 >= 1;
    // an index past the number of blocks implies a duplicate or an outside seed
    const bool inside = s.x >= 0 && s.y >= 0 && s.x < J.w && s.y < J.h && i < J.gbw * J.gbh;
    if (inside) {
        const int word = (i << 5) | ((int)motion << 4) | ((s.x % kBlock) << 2) | (s.y % kBlock);
        if (atomicCAS(J.map + (s.y / kBlock) * J.gbw + s.x / kBlock, -1, word) != -1) atomicOr(J.status, kErrSeed);
    } else {
        atomicOr(J.status, kErrSeed);
    }
    double X[kPointDoubles] = {0, 0, 0, 0, 0, 0, (double)s.d0, 0};
    if (motion) {
        triangulate(J, s.x, s.y, s.d0, X);
        triangulate(J, s.x + s.u, s.y + s.v, s.d1, X + 3);
    }
    double2* o = reinterpret_cast<double2*>(J.pts + (size_t)i * kPointDoubles);
#pragma unroll
    for (int k = 0; k < kPointDoubles / 2; ++k) o[k] = make_double2(X[2 * k], X[2 * k + 1]);
}

// Cell k of the Chebyshev ring r around a block: offsets (ox, oy).
__device__ __forceinline__ void ring_cell(int r, int k, int& ox, int& oy) {
    const int side = 2 * r + 1;
    if (r == 0) {
        ox = oy = 0;
    } else if (k < side) {  // top row
        ox = k - r;
        oy = -r;
    } else if (k < 2 * side) {  // bottom row
        ox = k - side - r;
        oy = r;
    } else {  // the two columns without their corners
        const int m = k - 2 * side;
        ox = (m & 1) ? r : -r;
        oy = (m >> 1) - r + 1;
    }
}

__device__ __forceinline__ int ring_cells(int r) { return r == 0 ? 1 : 8 * r; }

// Sums v[0 .. N) over groups of W lanes by recursive halving: on return lane l of
// a group holds in v[0 .. N / W) the totals of values l N / W ...
template <int N, int W>
__device__ __forceinline__ void reduce_scatter(double (&v)[N], int lane) {
    static_assert(W <= 32 && (W & (W - 1)) == 0 && N % W == 0, "whole halves");
#pragma unroll
    for (int o = W / 2, h = N / 2; o >= 1; o >>= 1, h >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double send = up ? v[i] : v[i + h];
            const double keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(kFull, send, o);
        }
    }
}

struct Candidates {
    const uint32_t* pos;  // (dy << 16) | (dx & 0xffff), offsets from the seed
    const int* word;
    int m;
};

__device__ __forceinline__ unsigned cand_d2(uint32_t p, int& dx, int& dy) {
    dx = (int)(int16_t)(p & 0xffffu);
    dy = (int)(int16_t)(p >> 16);
    return (unsigned)(dx * dx + dy * dy);
}

struct Threshold {
    unsigned D;  // a member has d2 < D, or d2 == D and index <= I
    int I;
};

// The index threshold among the candidates tied at distance D: the need-th
// smallest index of the set's members with d2 == D (need < number tied).
// Up to 32 tied members are ranked in registers; more fall back to
// bisection over the index.
__device__ int tie_threshold(const Candidates& C, bool motion, unsigned D, int need, int tied, int n, int* scratch,
                             int lane) {
    if (tied <= 32) {
        int filled = 0;
        for (int base = 0; base < C.m; base += 32) {
            const int j = base + lane;
            bool t = false;
            int idx = 0;
            if (j < C.m) {
                const int w = C.word[j];
                int dx, dy;
                t = (!motion || word_motion(w)) && cand_d2(C.pos[j], dx, dy) == D;
                idx = word_index(w);
            }
            const unsigned bt = __ballot_sync(kFull, t);
            if (t) scratch[filled + __popc(bt & ((1u << lane) - 1u))] = idx;
            filled += __popc(bt);
        }
        __syncwarp();
        const int v = lane < tied ? scratch[lane] : 0x7fffffff;
        int rank = 0;
        for (int u = 0; u < tied; ++u) rank += __shfl_sync(kFull, v, u) < v;
        __syncwarp();
        const unsigned hit = __ballot_sync(kFull, lane < tied && rank == need - 1);
        return __shfl_sync(kFull, v, __ffs(hit) - 1);
    }
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = lo + ((hi - lo) >> 1);
        int c = 0;
        for (int j = lane; j < C.m; j += 32) {
            const int w = C.word[j];
            int dx, dy;
            c += (!motion || word_motion(w)) && cand_d2(C.pos[j], dx, dy) == D && word_index(w) <= mid;
        }
        if ((int)__reduce_add_sync(kFull, c) >= need)
            hi = mid;
        else
            lo = mid + 1;
    }
    return lo;
}

// Bracket of the k-th smallest distance of a set: fewer than k members are nearer
// than lo, at least k within hi; `full`: exactly k are within hi, which need not be
// a member's distance itself.
struct Bracket {
    unsigned lo, hi;
    bool full;
};

// Runs f(each) with each(g) calling g(d2, motion key) for the lane's candidates,
// the motion key being d2 for a motion seed, past 2^31 for another; from keys held
// in registers when the candidates fit, else from shared memory.
template <class F>
__device__ __forceinline__ void with_keys(const Candidates& C, int lane, F f) {
    if (C.m <= 32 * kRegKeys) {
        unsigned key[kRegKeys];  // bit 31: no motion seed; the filler is farther than any bound
        const bool second = C.m > 16 * kRegKeys;
        auto load = [&](int t) {
            const int j = lane + 32 * t;
            key[t] = 0xffffffffu;
            if (j < C.m) {
                int dx, dy;
                key[t] = cand_d2(C.pos[j], dx, dy) | ((unsigned)!word_motion(C.word[j]) << 31);
            }
        };
#pragma unroll
        for (int t = 0; t < kRegKeys / 2; ++t) load(t);
        if (second)
#pragma unroll
            for (int t = kRegKeys / 2; t < kRegKeys; ++t) load(t);
        f([&](auto g) {
#pragma unroll
            for (int t = 0; t < kRegKeys / 2; ++t) g(key[t] & 0x7fffffffu, key[t]);
            if (second)
#pragma unroll
                for (int t = kRegKeys / 2; t < kRegKeys; ++t) g(key[t] & 0x7fffffffu, key[t]);
        });
    } else {
        f([&](auto g) {
            for (int j = lane; j < C.m; j += 32) {
                int dx, dy;
                const unsigned d2 = cand_d2(C.pos[j], dx, dy);
                g(d2, d2 | ((unsigned)!word_motion(C.word[j]) << 31));
            }
        });
    }
}

// Narrows the brackets of both sets, all candidates (k_geo) and the motion seeds
// among them (k_motion), by bisections that share their passes over the candidates,
// until they are full or at most hi >> shift wide (shift 31: lo = hi), and then, if
// asked for, counts the members below and at the distances that are not full
// (cnt[0..1] and cnt[2..3], zeros for a full one).  A set with lo = hi is left
// alone.  The counts of both sets share a word (at most 4352 candidates) and one
// reduction.  A dense field has about 200 candidates a seed, 7 of 16 keys per lane,
// and ends full after 5 or 6 passes from a bracket whose lower end is the nearest
// seed that the further rings can hold (10 from zero, and 10 more for the ring bound
// to the last integer): k_interp_models 309 M -> 226 M warp instructions, 714 -> 659
// us at 1242 x 375.  One routine serves the tightening of the ring bound and the final
// selection, so that its code exists once.
__device__ __noinline__ void narrow_both(const Candidates& C, int kg, int km, Bracket& A, Bracket& M, int shift,
                                         int lane, int* cnt) {
    A.full = M.full = false;
    with_keys(C, lane, [&](auto each) {
        for (;;) {
            const bool ga = !A.full && A.hi - A.lo > (A.hi >> shift), gm = !M.full && M.hi - M.lo > (M.hi >> shift);
            if (!ga && !gm) break;
            const unsigned midA = A.lo + ((A.hi - A.lo) >> 1), midM = M.lo + ((M.hi - M.lo) >> 1);
            unsigned c = 0;
            each([&](unsigned d2, unsigned mot) {
                if (d2 <= midA) c += 1u;
                if (mot <= midM) c += 1u << 16;
            });
            c = __reduce_add_sync(kFull, c);
            const int ca = c & 0xffffu, cm = c >> 16;
            auto step = [](Bracket& B, unsigned mid, int count, int k) {
                if (count < k) {
                    B.lo = mid + 1;
                } else {
                    B.hi = mid;
                    B.full = count == k;
                }
            };
            if (ga) step(A, midA, ca, kg);
            if (gm) step(M, midM, cm, km);
        }
        if (!cnt) return;
        unsigned below = 0, at = 0;
        if (!A.full || !M.full) {
            each([&](unsigned d2, unsigned mot) {
                if (d2 < A.hi) below += 1u;
                if (d2 == A.hi) at += 1u;
                if (mot < M.hi) below += 1u << 16;
                if (mot == M.hi) at += 1u << 16;
            });
            below = __reduce_add_sync(kFull, below);
            at = __reduce_add_sync(kFull, at);
        }
        cnt[0] = A.full ? 0 : (int)(below & 0xffffu);
        cnt[1] = A.full ? 0 : (int)(at & 0xffffu);
        cnt[2] = M.full ? 0 : (int)(below >> 16);
        cnt[3] = M.full ? 0 : (int)(at >> 16);
    });
}

// Thresholds of the k smallest (d2, index) keys of both neighbourhoods.
// `fa`/`fm` are the sizes of the two sets, BA / BM brackets of their k-th distances.
__device__ void select_both(const Candidates& C, int kg, int km, int fa, int fm, Bracket BA, Bracket BM, int n,
                            int* scratch, int lane, Threshold& A, Threshold& M) {
    A = Threshold{0xffffffffu, 0x7fffffff};
    M = Threshold{0xffffffffu, 0x7fffffff};
    const bool sa = fa > kg, sm = fm > km;
    if (!sa && !sm) return;
    int cnt[4];
    if (!sa) BA.lo = BA.hi;
    if (!sm) BM.lo = BM.hi;
    narrow_both(C, kg, km, BA, BM, 31, lane, cnt);
    if (sa) {
        A.D = BA.hi;
        if (!BA.full && kg - cnt[0] < cnt[1]) A.I = tie_threshold(C, false, A.D, kg - cnt[0], cnt[1], n, scratch, lane);
    }
    if (sm) {
        M.D = BM.hi;
        if (!BM.full && km - cnt[2] < cnt[3]) M.I = tie_threshold(C, true, M.D, km - cnt[2], cnt[3], n, scratch, lane);
    }
}

__device__ __forceinline__ bool selected(unsigned d2, int idx, unsigned D, int I) {
    return d2 < D || (d2 == D && idx <= I);
}

// Cholesky factorisation of one 4x4 matrix per lane (upper triangle u[10] row by
// row), and the solution of one right-hand side into b[4]; divisions by the
// diagonal are multiplications by its reciprocal.
struct Factor4 {
    double L[4][4], inv[4];
};
__device__ __forceinline__ void factor4(const double (&u)[10], Factor4& F) {
    auto& L = F.L;
    L[0][0] = u[0];
    L[1][0] = u[1];
    L[2][0] = u[2];
    L[3][0] = u[3];
    L[1][1] = u[4];
    L[2][1] = u[5];
    L[3][1] = u[6];
    L[2][2] = u[7];
    L[3][2] = u[8];
    L[3][3] = u[9];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        double s = L[j][j];
#pragma unroll
        for (int k = 0; k < j; ++k) s -= L[j][k] * L[j][k];
        const double ljj = sqrt(s > 0.0 ? s : 1e-300);
        F.inv[j] = 1.0 / ljj;
#pragma unroll
        for (int i = j + 1; i < 4; ++i) {
            double t = L[i][j];
#pragma unroll
            for (int k = 0; k < j; ++k) t -= L[i][k] * L[j][k];
            L[i][j] = t * F.inv[j];
        }
    }
}
__device__ __forceinline__ void solve4(const Factor4& F, double (&b)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        double t = b[i];
#pragma unroll
        for (int k = 0; k < i; ++k) t -= F.L[i][k] * b[k];
        b[i] = t * F.inv[i];
    }
#pragma unroll
    for (int i = 3; i >= 0; --i) {
        double t = b[i];
#pragma unroll
        for (int k = i + 1; k < 4; ++k) t -= F.L[k][i] * b[k];
        b[i] = t * F.inv[i];
    }
}

// Shared memory of one warp of k_interp_models: candidate positions and map words
// (J.slots each), the neighbour lists of its seeds (k_geo, k_motion position and
// word pairs each), 32 ints of scratch.
__host__ __device__ __forceinline__ size_t warp_smem_bytes(int slots, int kg, int km, int seeds) {
    return (size_t)slots * 8 + (size_t)seeds * (kg + km) * 8 + 128;
}

// The two neighbourhoods of seed si into la[kg] and lm[km]; false when the
// candidates do not fit the slots.
__device__ __forceinline__ bool select_neighbours(const InterpJob& J, int si, int n, uint32_t* pos, int* word, int* scratch,
                                                  uint2* la, uint2* lm, int& na, int& nm, int lane) {
    const int kg = J.p.k_geo, km = J.p.k_motion;
    const sff_seed s = J.seeds[si];
    const int bx = s.x / kBlock, by = s.y / kBlock;
    const int rmax = max(J.gbw, J.gbh);
    const unsigned lt = (1u << lane) - 1u;

    // Candidates by rings of blocks around the seed's block (ring q is at
    // least 3q - 2 px away).  First the rings until both neighbourhoods have
    // k members; a set's bound is the largest distance found when it got
    // them, and from then on a seed is kept only if it is within the bound
    // of a set it belongs to (so that sparse motion seeds do not drag every
    // seed in).  Then distances little above the k-th smallest of the candidates
    // replace the bounds, and the further rings that can still hold a member within
    // a bound are scanned.
    int fill = 0;                                          // candidates kept
    int fa = 0, fm = 0;                                    // ... of which motion seeds: fm
    unsigned far_a = 0, far_m = 0;                         // largest distance kept (all / motion)
    unsigned bound_a = 0xffffffffu, bound_m = 0xffffffffu;  // storage bounds, none yet
    // Compaction, when a batch would not fit the slots (motion seeds far
    // away behind many geometry-only seeds, e.g. the disparity fill's): the
    // k-th smallest distances of the candidates so far bound the final ones
    // from above (more candidates only lower them), so the candidates beyond
    // them are no members and are dropped, keeping the others in scan order.
    // far_a and far_m have to cover every candidate counted in fa and fm.
    auto compact = [&]() {
        const Candidates Cc{pos, word, fill};
        unsigned DA = bound_a, DM = bound_m;
        if (fa >= kg || fm >= km) {
            Bracket A{0u, fa >= kg ? far_a : 0u}, M{0u, fm >= km ? far_m : 0u};
            narrow_both(Cc, kg, km, A, M, 31, lane, nullptr);
            if (fa >= kg) DA = min(DA, A.hi);
            if (fm >= km) DM = min(DM, M.hi);
        }
        int kept = 0, kmot = 0;
        for (int base = 0; base < fill; base += 32) {
            const int j = base + lane;
            uint32_t pj = 0;
            int wj = -1;
            bool keep = false, mot = false;
            if (j < fill) {
                pj = pos[j];
                wj = word[j];
                int dx, dy;
                const unsigned d2 = cand_d2(pj, dx, dy);
                mot = word_motion(wj);
                keep = d2 <= DA || (mot && d2 <= DM);
            }
            const unsigned b = __ballot_sync(kFull, keep), bm = __ballot_sync(kFull, keep && mot);
            __syncwarp();  // the batch is read before any of it is overwritten
            if (keep) {
                const int slot = kept + __popc(b & lt);  // <= j
                pos[slot] = pj;
                word[slot] = wj;
            }
            __syncwarp();
            kept += __popc(b);
            kmot += __popc(bm);
        }
        fill = kept;
        fa = kept;
        fm = kmot;
        bound_a = DA;
        bound_m = DM;
    };
    auto scan = [&](int q) {
        unsigned ma = 0, mm = 0;
        for (int base = 0; base < ring_cells(q); base += 32) {
            const int k = base + lane;
            int w = -1, dx = 0, dy = 0;
            unsigned d2 = 0;
            if (k < ring_cells(q)) {
                int ox, oy;
                ring_cell(q, k, ox, oy);
                const int cx = bx + ox, cy = by + oy;
                if (cx >= 0 && cy >= 0 && cx < J.gbw && cy < J.gbh) w = J.map[cy * J.gbw + cx];
                if (w >= 0) {
                    dx = cx * kBlock + ((w >> 2) & 3) - s.x;
                    dy = cy * kBlock + (w & 3) - s.y;
                    d2 = (unsigned)(dx * dx + dy * dy);
                    if (!(d2 <= bound_a || (word_motion(w) && d2 <= bound_m))) w = -1;
                }
            }
            if (fill + __popc(__ballot_sync(kFull, w >= 0)) > J.slots) {
                // fa and fm count this ring's seeds already: a set may owe its k-th to them
                far_a = max(far_a, __reduce_max_sync(kFull, ma));
                far_m = max(far_m, __reduce_max_sync(kFull, mm));
                compact();
                if (w >= 0 && !(d2 <= bound_a || (word_motion(w) && d2 <= bound_m))) w = -1;
            }
            const unsigned has = __ballot_sync(kFull, w >= 0), mot = __ballot_sync(kFull, w >= 0 && word_motion(w));
            if (w >= 0) {
                const int slot = fill + __popc(has & lt);
                if (slot < J.slots) {
                    pos[slot] = ((uint32_t)(dy & 0xffff) << 16) | (uint32_t)(dx & 0xffff);
                    word[slot] = w;
                }
                ma = max(ma, d2);
                if (word_motion(w)) mm = max(mm, d2);
            }
            fill += __popc(has);
            fa += __popc(has);
            fm += __popc(mot);
        }
        far_a = max(far_a, __reduce_max_sync(kFull, ma));
        far_m = max(far_m, __reduce_max_sync(kFull, mm));
        if (bound_a == 0xffffffffu && fa >= kg) bound_a = far_a;
        if (bound_m == 0xffffffffu && fm >= km) bound_m = far_m;
    };
    int q = 0;
    for (; q <= rmax && (fa < kg || fm < km); ++q) scan(q);
    __syncwarp();
    if (fill > J.slots) return false;
    unsigned lo_a = 0, lo_m = 0;  // the k-th distances are at least these
    if (fa >= kg && fm >= km) {
        const Candidates C1{pos, word, fill};
        Bracket A{0u, bound_a}, M{0u, bound_m};
        narrow_both(C1, kg, km, A, M, kTighten, lane, nullptr);
        bound_a = A.hi;
        bound_m = M.hi;
        const unsigned near = (unsigned)(max(3 * q - 2, 0) * max(3 * q - 2, 0));  // the further rings' seeds
        lo_a = min(A.lo, near);
        lo_m = min(M.lo, near);
        for (; q <= rmax; ++q) {
            const long long b = 3 * q - 2;
            if (b * b > (long long)max(bound_a, bound_m)) break;
            scan(q);
        }
        __syncwarp();
    }
    const Candidates C{pos, word, fill};
    if (C.m > J.slots) return false;
    Threshold TA, TM;
    select_both(C, kg, km, fa, fm, Bracket{lo_a, min(bound_a, far_a)}, Bracket{lo_m, min(bound_m, far_m)}, n, scratch,
                lane, TA, TM);

    // the members of both neighbourhoods, compacted into lists
    na = nm = 0;
    for (int base = 0; base < C.m; base += 32) {
        const int j = base + lane;
        bool in_a = false, in_m = false;
        if (j < C.m) {
            const int w = C.word[j], idx = word_index(w);
            int dx, dy;
            const unsigned d2 = cand_d2(C.pos[j], dx, dy);
            in_a = selected(d2, idx, TA.D, TA.I);
            in_m = word_motion(w) && selected(d2, idx, TM.D, TM.I);
        }
        const unsigned ba = __ballot_sync(kFull, in_a), bm = __ballot_sync(kFull, in_m);
        const int qa = na + __popc(ba & lt), qm = nm + __popc(bm & lt);
        if (in_a && qa < kg) la[qa] = make_uint2(C.pos[j], (uint32_t)C.word[j]);
        if (in_m && qm < km) lm[qm] = make_uint2(C.pos[j], (uint32_t)C.word[j]);
        na += __popc(ba);
        nm += __popc(bm);
    }
    __syncwarp();
    return na <= kg && nm <= km;  // at most k members are selected
}

// One warp per two seeds (SP = 2): the whole warp selects each seed's neighbourhoods in
// turn, then the sums of both run side by side, 16 lanes per seed.  An FP64
// instruction holds its sub-partition's pipe for 64 clocks whatever its active
// lanes, so what counts is the number of warp instructions: with 32 lanes per seed
// the 80 motion neighbours took three rounds (2.5 needed) and the two reductions 47
// additions; 174 instead of 221 FP64 instructions per seed.  1242 x 375, default
// neighbourhoods: 778 -> 714 us (with the disparity fill's seeds 989 -> 879); four
// seeds per warp 887: their lists leave 12 warps per SM.
// Two each only where that is the better split, in us the call with two / one each
// (n seeds; R warps resident, SMs x 20 = 3040 at the default k):
//   - one each up to R, where every seed has a warp of its own at once (n = 368 102 /
//     75, 2885 122 / 104);
//   - two each up to 2 R, one round of the GPU instead of two (3691 126 / 135, 5105 145
//     / 150);
//   - one each again up to 10 R / 3, where the second round of two each is short (6774
//     209 / 189, 10009 257 / 249), and two each from there on (10856 226 / 240, 36976
//     632 / 684);
//   - but one each at any number of sparse seeds, fewer than half of the blocks: their
//     selections, which scan more rings, then outweigh the sums, and differ more from
//     warp to warp (4693 on 39195 blocks 352 / 313, 15110 on 51750 533 / 461, 59975 on
//     122574 1287 / 1306; 16012 on 30000, above half, 402 / 393).
// With larger neighbourhoods the second seed's lists cost more warps than the shared
// instructions save: SP = 1, one seed per warp at any number, where fewer than 15 warps
// of two would fit an SM (37749 seeds, us two / one: k 200/100, 16 warps, 951 / 960;
// 250/125, 13 warps, 1172 / 1120; 400/300 2167 / 1957; 1024/1024 13791 / 9911).
template <int SP>
__global__ void __launch_bounds__(kModelWarps * 32, SP == 2 ? kModelResident : kModelResidentLone)
    k_interp_models(InterpJob J) {
    constexpr int W = 16;  // lanes per seed of two, and half the lanes of a lone one's
    static_assert(SP == 1 || SP == 2, "seeds per warp");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n = seed_count(J);
    // one seed, its sums over all lanes (the line as a word of its own: with the rule's
    // comparisons here the kernel took 1 % more)
    const bool lone = SP == 1 || n <= *J.lone_max;
    const int s0 = (blockIdx.x * kModelWarps + wid) * (lone ? 1 : SP);
    if (s0 >= n) return;  // warp-uniform
    const int kg = J.p.k_geo, km = J.p.k_motion;
    unsigned char* mine = smem_raw + (size_t)wid * warp_smem_bytes(J.slots, kg, km, SP);
    uint32_t* pos = reinterpret_cast<uint32_t*>(mine);
    int* word = reinterpret_cast<int*>(mine + (size_t)J.slots * 4);
    uint2* lists = reinterpret_cast<uint2*>(mine + (size_t)J.slots * 8);
    int* scratch = reinterpret_cast<int*>(lists + SP * (kg + km));
    const int sub = lone ? 0 : lane / W, l = lane % W, si = s0 + sub;  // this lane's seed
    const int first = lone ? lane : l, step = lone ? 32 : W;          // its neighbours
    const auto halves = [&](double& v) { v += __shfl_xor_sync(kFull, v, W); };
    int na = 0, nm = 0;
#pragma unroll 1
    for (int k = 0; k < SP; ++k) {
        if (s0 + k >= n || (lone && k > 0)) break;
        int a, m;
        uint2* la = lists + k * (kg + km);
        if (!select_neighbours(J, s0 + k, n, pos, word, scratch, la, la + kg, a, m, lane)) {
            if (lane == 0) atomicOr(J.status, kErrOverflow);
            a = m = 0;  // the field is all zeros
        }
        if (sub == k) {
            na = a;
            nm = m;
        }
        __syncwarp();
    }
    const uint2 *la = lists + sub * (kg + km), *lm = la + kg;

    // plane sums and the motion centroid: M00 M01 M02 M11 M12 M22 b0 b1 b2,
    // then W, W x0 (3)
    double g[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) g[k] = 0.0;
    for (int t = first; t < na; t += step) {
        const uint2 c = la[t];
        int dx, dy;
        const unsigned d2 = cand_d2(c.x, dx, dy);
        const double wt = weight_of(J, d2);
        const double d = J.pts[(size_t)word_index((int)c.y) * kPointDoubles + 6];
        const double r0 = dx, r1 = dy;
        const double w0 = wt * r0, w1 = wt * r1;
        g[0] += w0 * r0;
        g[1] += w0 * r1;
        g[2] += w0;
        g[3] += w1 * r1;
        g[4] += w1;
        g[5] += wt;
        g[6] += w0 * d;
        g[7] += w1 * d;
        g[8] += wt * d;
    }
    for (int t = first; t < nm; t += step) {
        const uint2 c = lm[t];
        int dx, dy;
        const unsigned d2 = cand_d2(c.x, dx, dy);
        const double wt = weight_of(J, d2);
        const double* X = J.pts + (size_t)word_index((int)c.y) * kPointDoubles;
        g[9] += wt;
        g[10] += wt * X[0];
        g[11] += wt * X[1];
        g[12] += wt * X[2];
    }
    __syncwarp();
    reduce_scatter<16, W>(g, lane);
    if (lone) halves(g[0]);
    auto value = [&](int k) { return __shfl_sync(kFull, g[0], sub * W + k); };  // on lane k of the group
    double cen[3] = {0.0, 0.0, 0.0};
    {
        const double ws = value(9), c0 = value(10), c1 = value(11), c2 = value(12);
        if (nm > 0) {
            const double iw = 1.0 / ws;
            cen[0] = c0 * iw;
            cen[1] = c1 * iw;
            cen[2] = c2 * iw;
        }
    }
    // centred motion sums: N (upper triangle of [r 1][r 1]^T, 10) and
    // R[j][a] = sum w r_a x1_j (12), r = x0 - c
    constexpr int kSums = 32;
    double a[kSums];
#pragma unroll
    for (int k = 0; k < kSums; ++k) a[k] = 0.0;
    for (int t = first; t < nm; t += step) {
        const uint2 c = lm[t];
        int dx, dy;
        const unsigned d2 = cand_d2(c.x, dx, dy);
        const double wt = weight_of(J, d2);
        const double* X = J.pts + (size_t)word_index((int)c.y) * kPointDoubles;
        const double r[4] = {X[0] - cen[0], X[1] - cen[1], X[2] - cen[2], 1.0};
        const double wr[4] = {wt * r[0], wt * r[1], wt * r[2], wt};
        int e = 0;
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = p; q < 4; ++q) a[e++] += wr[p] * r[q];
#pragma unroll
        for (int jj = 0; jj < 3; ++jj)
#pragma unroll
            for (int p = 0; p < 4; ++p) a[10 + jj * 4 + p] += wr[p] * X[3 + jj];
    }
    __syncwarp();
    reduce_scatter<kSums, W>(a, lane);
    if (lone) {
#pragma unroll
        for (int i = 0; i < kSums / W; ++i) halves(a[i]);
    }

    // the sums go to k_interp_solve: plane sums first, then N and R
    if (si >= n || (lone && lane >= W)) return;
    double* sums = J.sums + (size_t)si * kSumDoubles;
    if (l < 9) sums[l] = g[0];
#pragma unroll
    for (int i = 0; i < kSums / W; ++i)
        if (l * (kSums / W) + i < 22) sums[9 + l * (kSums / W) + i] = a[i];
    if (l < 3) J.models[(size_t)si * kModelDoubles + 15 + l] = l == 0 ? cen[0] : l == 1 ? cen[1] : cen[2];
    if (l == 0) J.motion[si] = nm;
}

// The least-squares systems of every seed: the motion system (blockIdx.y 0, one
// thread factors its 4x4 matrix once and solves the three rows of [A | t]) and the
// plane (blockIdx.y 1; a 3x3 system, padded to 4x4 with an identity row, which
// leaves its solution unchanged).  Bound by the FP64 pipe, so by warp
// instructions: with the four systems on four neighbouring lanes the matrix was
// factored three times and a warp held 8 seeds; 1242 x 375: 70 -> 26 us.
__global__ void k_interp_solve(InterpJob J) {
    const int si = blockIdx.x * blockDim.x + threadIdx.x;
    if (si >= seed_count(J)) return;
    const double* S = J.sums + (size_t)si * kSumDoubles;
    double* out = J.models + (size_t)si * kModelDoubles;
    double u[10], b[4];
    Factor4 F;
    if (blockIdx.y == 1) {
        // M00 M01 M02 M11 M12 M22 into the padded upper triangle, b0 b1 b2
        u[0] = S[0];
        u[1] = S[1];
        u[2] = S[2];
        u[3] = 0.0;
        u[4] = S[3];
        u[5] = S[4];
        u[6] = 0.0;
        u[7] = S[5];
        u[8] = 0.0;
        u[9] = 1.0;
        const double lam = 1e-9 * (u[0] + u[4] + u[7]) / 3 + 1e-300;  // trace of the 3x3 system
        u[0] += lam;
        u[4] += lam;
        b[0] = S[6];
        b[1] = S[7];
        b[2] = S[8];
        b[3] = 0.0;
        factor4(u, F);
        solve4(F, b);
        out[0] = b[0];
        out[1] = b[1];
        out[2] = b[2];
        return;
    }
    if (J.motion[si] == 0) {
#pragma unroll
        for (int p = 0; p < 12; ++p) out[3 + p] = 0.0;
        return;
    }
#pragma unroll
    for (int k = 0; k < 10; ++k) u[k] = S[9 + k];
    const double lam = 1e-9 * (u[0] + u[4] + u[7] + u[9]) / 4 + 1e-300;
    u[0] += lam;
    u[4] += lam;
    u[7] += lam;
    factor4(u, F);
#pragma unroll
    for (int row = 0; row < 3; ++row) {
#pragma unroll
        for (int p = 0; p < 4; ++p) b[p] = S[19 + 4 * row + p];
        b[row] += lam;  // towards A = I
        solve4(F, b);
#pragma unroll
        for (int p = 0; p < 4; ++p) out[3 + 4 * row + p] = b[p];
    }
}

// Closest seed of every pixel, exactly, in two separable passes: the
// squared distance to a seed is (x - xs)^2 + (y - ys)^2, so the closest seed
// minimises (x - x')^2 + g(x', y)^2 over the columns x', g(x', y) being the
// distance from row y to the closest seed in column x'.  A tie inside a
// column is a tie of the total distance at every pixel of the row, so each
// pass keeps the lower seed index on ties and the result is the closest
// seed with the lowest index.
//
// k_interp_columns: col[y][x] = (g, index) of the closest seed in column x,
// or (0, -1) when the column holds no seed.  A CTA takes 32 columns, each
// cut into kColSegments runs of block rows, one thread per column and run:
// every thread records the first and last seed of its run, then sweeps its
// run down and up starting from the nearest seeds of the runs above and
// below.
constexpr int kColSegments = 16;

__global__ void __launch_bounds__(32 * kColSegments) k_interp_columns(InterpJob J, int2* col) {
    __shared__ int2 first_s[kColSegments][32], last_s[kColSegments][32];  // (row, index), index -1: none
    const int lane = threadIdx.x, seg = threadIdx.y;
    const int x = blockIdx.x * 32 + lane;
    if (seed_count(J) == 0 || *J.status) return;  // uniform over the CTA
    const bool live = x < J.w;
    const int bx = x / kBlock, ox = x % kBlock;
    const int per = (J.gbh + kColSegments - 1) / kColSegments;
    const int b0 = min(J.gbh, seg * per), b1 = min(J.gbh, b0 + per);
    // the seed of block row by in this column, or -1
    auto seed_row = [&](int by, int& idx) {
        const int w = J.map[by * J.gbw + bx];
        idx = word_index(w);
        return (w >= 0 && ((w >> 2) & 3) == ox) ? by * kBlock + (w & 3) : -1;
    };
    int2 f = make_int2(0, -1), l = make_int2(0, -1);
    if (live)
        for (int by = b0; by < b1; ++by) {
            int idx;
            const int sy = seed_row(by, idx);
            if (sy < 0) continue;
            if (f.y < 0) f = make_int2(sy, idx);
            l = make_int2(sy, idx);
        }
    first_s[seg][lane] = f;
    last_s[seg][lane] = l;
    __syncthreads();
    if (!live) return;
    int2 up = make_int2(0, -1), dn = make_int2(0, -1);  // nearest seeds above / below the run
    for (int q = seg - 1; q >= 0 && up.y < 0; --q) up = last_s[q][lane];
    for (int q = seg + 1; q < kColSegments && dn.y < 0; ++q) dn = first_s[q][lane];
    int ly = up.x, li = up.y;
    for (int by = b0; by < b1; ++by) {
        int idx;
        const int sy = seed_row(by, idx);
        const int y0 = by * kBlock;
        for (int y = y0; y < min(y0 + kBlock, J.h); ++y) {
            if (y == sy) {
                ly = sy;
                li = idx;
            }
            col[(size_t)y * J.w + x] = make_int2(y - ly, li);
        }
    }
    int ny = dn.x, ni = dn.y;
    for (int by = b1 - 1; by >= b0; --by) {
        int idx;
        const int sy = seed_row(by, idx);
        const int y0 = by * kBlock;
        for (int y = min(y0 + kBlock, J.h) - 1; y >= y0; --y) {
            if (y == sy) {
                ny = sy;
                ni = idx;
            }
            if (ni < 0) continue;
            const size_t pi = (size_t)y * J.w + x;
            const int2 a = col[pi];
            const int g = ny - y;
            if (a.y < 0 || g < a.x || (g == a.x && ni < a.y)) col[pi] = make_int2(g, ni);
        }
    }
}

// k_interp_pixels: per pixel the closest seed along its row of col (scanning
// outwards until the horizontal distance alone exceeds the best), then its
// models evaluated at the pixel: d0 from the plane, x0 from
// (x, y, max(d0, 1)), x1 = A (x0 - c) + t projected back.
__global__ void k_interp_pixels(InterpJob J, const int2* col, float4* field) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= J.w || y >= J.h) return;
    const size_t pi = (size_t)y * J.w + x;
    if (seed_count(J) == 0 || *J.status) {
        field[pi] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const int2* row = col + (size_t)y * J.w;
    long long bd = 0x7fffffffffffffffll;
    int best = 0x7fffffff;
    for (int dx = 0; dx < J.w; ++dx) {
        if ((long long)dx * dx > bd) break;
        const int xa = x - dx, xb = x + dx;
        if (xa >= 0) {
            const int2 c = row[xa];
            const long long d = (long long)dx * dx + (long long)c.x * c.x;
            if (c.y >= 0 && (d < bd || (d == bd && c.y < best))) {
                bd = d;
                best = c.y;
            }
        }
        if (dx > 0 && xb < J.w) {
            const int2 c = row[xb];
            const long long d = (long long)dx * dx + (long long)c.x * c.x;
            if (c.y >= 0 && (d < bd || (d == bd && c.y < best))) {
                bd = d;
                best = c.y;
            }
        }
    }
    if (best == 0x7fffffff) {  // unreachable while every seed is in the map
        field[pi] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const sff_seed s = J.seeds[best];
    const double* m = J.models + (size_t)best * kModelDoubles;
    const double d0 = m[0] * (x - s.x) + m[1] * (y - s.y) + m[2];
    float4 r = make_float4(0.f, 0.f, (float)d0, (float)d0);
    if (J.motion[best] > 0) {
        const double Z = J.fb / (d0 > 1.0 ? d0 : 1.0);
        const double X0[3] = {(x - J.p.cx) * Z * J.inv_f, (y - J.p.cy) * Z * J.inv_f, Z};
        const double* A = m + 3;
        const double* c = m + 15;
        double X1[3];
#pragma unroll
        for (int j = 0; j < 3; ++j)
            X1[j] = A[4 * j] * (X0[0] - c[0]) + A[4 * j + 1] * (X0[1] - c[1]) + A[4 * j + 2] * (X0[2] - c[2]) +
                    A[4 * j + 3];
        if (X1[2] > 0.0) {
            const double iz = 1.0 / X1[2];
            r.x = (float)(J.p.focal * X1[0] * iz + J.p.cx - x);
            r.y = (float)(J.p.focal * X1[1] * iz + J.p.cy - y);
            r.w = (float)(J.fb * iz);
        }
    }
    field[pi] = r;
}

struct InterpLayout {
    size_t map, pts, wt, models, sums, motion, nearest, status, total;
};

InterpLayout interp_layout(int w, int h, int capacity) {
    const int gbw = (w + kBlock - 1) / kBlock, gbh = (h + kBlock - 1) / kBlock;
    InterpLayout L;
    L.map = 0;
    L.pts = L.map + align256((size_t)gbw * gbh * sizeof(int));
    L.wt = L.pts + align256((size_t)capacity * kPointDoubles * sizeof(double));
    L.models = L.wt + align256((size_t)kWeightTable * sizeof(double));
    L.sums = L.models + align256((size_t)capacity * kModelDoubles * sizeof(double));
    L.motion = L.sums + align256((size_t)capacity * kSumDoubles * sizeof(double));
    L.nearest = L.motion + align256((size_t)capacity * sizeof(int));
    L.status = L.nearest + align256((size_t)w * h * sizeof(int2));
    L.total = L.status + 256;
    return L;
}

}  // namespace
}  // namespace sff

extern "C" int sff_default_interp_params(int32_t width, int32_t height, double focal, double baseline,
                                         sff_interp_params* out) {
    if (!out || width < 1 || height < 1 || !(focal > 0.0) || !(baseline > 0.0)) return SFF_ERR_ARG;
    out->k_geo = 160;
    out->k_motion = 80;
    out->alpha = 2.2;
    out->dist_unit = 20.0;
    out->focal = focal;
    out->baseline = baseline;
    out->cx = (width - 1) / 2.0;
    out->cy = (height - 1) / 2.0;
    return SFF_OK;
}

extern "C" size_t sff_interp_workspace_bytes(int32_t width, int32_t height, int32_t capacity) {
    if (sff::check_size(width, height) || capacity < 0) return 0;
    return sff::interp_layout(width, height, capacity).total;
}

extern "C" int sff_interpolate(const sff_seed* seeds_dev, const int32_t* count_dev, int32_t capacity, int32_t width,
                               int32_t height, const sff_interp_params* params, float* field_dev, void* workspace,
                               size_t workspace_bytes, void* stream) {
    using namespace sff;
    if (check_size(width, height) || !params || capacity < 0) return SFF_ERR_ARG;
    if (!seeds_dev || !count_dev || !field_dev || !workspace) return SFF_ERR_ARG;
    if (params->k_geo < 1 || params->k_geo > kMaxK || params->k_motion < 1 || params->k_motion > kMaxK ||
        !(params->alpha >= 0.0) || !(params->dist_unit > 0.0) || !(params->focal > 0.0) || !(params->baseline > 0.0))
        return SFF_ERR_ARG;
    if (((uintptr_t)field_dev & 15) || ((uintptr_t)workspace & 255) || ((uintptr_t)seeds_dev & 3)) return SFF_ERR_ARG;
    const InterpLayout L = interp_layout(width, height, capacity);
    if (workspace_bytes < L.total) return SFF_ERR_WORKSPACE;
    char* ws = reinterpret_cast<char*>(workspace);
    InterpJob J;
    J.seeds = seeds_dev;
    J.count = count_dev;
    J.capacity = capacity;
    J.w = width;
    J.h = height;
    J.gbw = (width + kBlock - 1) / kBlock;
    J.gbh = (height + kBlock - 1) / kBlock;
    J.map = reinterpret_cast<int*>(ws + L.map);
    J.pts = reinterpret_cast<double*>(ws + L.pts);
    J.wt = reinterpret_cast<double*>(ws + L.wt);
    J.models = reinterpret_cast<double*>(ws + L.models);
    J.sums = reinterpret_cast<double*>(ws + L.sums);
    J.motion = reinterpret_cast<int*>(ws + L.motion);
    J.status = reinterpret_cast<unsigned*>(ws + L.status);
    J.lone_max = reinterpret_cast<int*>(J.status + 1);
    J.p = *params;
    J.fb = params->focal * params->baseline;
    J.inv_f = 1.0 / params->focal;
    J.slots = candidate_slots(params->k_geo, params->k_motion);
    const size_t pair_smem = kModelWarps * warp_smem_bytes(J.slots, J.p.k_geo, J.p.k_motion, 2);
    const int per_sm = kModelWarps * min(kModelResident, (int)(kSmemPerSm / (pair_smem + kSmemPerCta)));
    const bool pairs = per_sm >= kMinResidentPairs;
    J.resident = kSms * per_sm;
    cudaStream_t st = (cudaStream_t)stream;
    const int clear = max(J.gbw * J.gbh, kWeightTable);
    SFF_LAUNCH(k_interp_clear, dim3((clear + 255) / 256), 256, 0, st, J);
    if (capacity > 0) {
        SFF_LAUNCH(k_interp_prep, dim3((capacity + 255) / 256), 256, 0, st, J);
        void (*const k_interp_models)(InterpJob) = pairs ? sff::k_interp_models<2> : sff::k_interp_models<1>;
        const size_t smem =
            pairs ? pair_smem : kModelWarps * warp_smem_bytes(J.slots, J.p.k_geo, J.p.k_motion, 1);
        if (smem > 48 * 1024 &&
            cudaFuncSetAttribute(k_interp_models, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            return SFF_ERR_CUDA;
        // pairs: enough warps for either split; those without a seed leave at once
        const int lone = min(capacity, max(J.resident * 10 / 3, J.gbw * J.gbh / 2));
        const int warps = pairs ? max((capacity + 1) / 2, lone) : capacity;
        SFF_LAUNCH(k_interp_models, dim3((warps + kModelWarps - 1) / kModelWarps), kModelWarps * 32, smem, st, J);
        SFF_LAUNCH(k_interp_solve, dim3((capacity + 63) / 64, 2), 64, 0, st, J);
    }
    int2* col = reinterpret_cast<int2*>(ws + L.nearest);
    SFF_LAUNCH(k_interp_columns, dim3((width + 31) / 32), dim3(32, kColSegments), 0, st, J, col);
    SFF_LAUNCH(k_interp_pixels, dim3((width + 127) / 128, height), 128, 0, st, J, col,
               reinterpret_cast<float4*>(field_dev));
    return launch_status();
}

extern "C" int sff_interp_status(const void* workspace, int32_t width, int32_t height, int32_t capacity,
                                 uint32_t* status_out) {
    using namespace sff;
    if (!workspace || !status_out || check_size(width, height) || capacity < 0) return SFF_ERR_ARG;
    const InterpLayout L = interp_layout(width, height, capacity);
    if (cudaMemcpy(status_out, reinterpret_cast<const char*>(workspace) + L.status, sizeof(uint32_t),
                   cudaMemcpyDeviceToHost) != cudaSuccess)
        return SFF_ERR_CUDA;
    return SFF_OK;
}
