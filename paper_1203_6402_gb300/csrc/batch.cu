// batch.cu -- many independent k-means|| problems in one call (kmpar_batch_run):
// Algorithm 2 (Sec. 3.3) and Lloyd's iteration (Sec. 1, Sec. 3.1) per problem,
// one thread block or cluster per problem, every step on the device.  The data-parallel
// pattern of Sec. 3.5 is applied across problems: a block owns its problem from
// the first center to the last centroid update, so no grid-wide synchronisation
// is needed and the blocks run in any order (largest problems first).
//
// Per problem (kBT threads a block; dense passes by tiles of rows and centers in shared
// memory, or, against few centers, a row per thread in registers):
//   init     i0 = floor(u n), D^2 = ||x - x_i0||^2, idx = 0, phi = sum D^2 (FP64)
//   round i  every x drawn with p = min(1, l D^2 / phi) (Philox, FP64 re-decision
//            of near draws), appended in ascending point order by an ordered
//            block compaction (no sort); D^2/idx against the batch
//   step 7   w_c = #{x : idx(x) = c} (shared-memory integer atomics)
//   step 8   weighted k-means++: per draw a blocked FP64 prefix over the masses,
//            the first candidate whose prefix exceeds u * total; each block of the
//            cluster holds a share of the candidates
//   Lloyd    assignment with the FP32 path's decision rule; centroids from a
//            stable counting sort by label (warp-private label counters,
//            __match_any_sync ranks) and compensated FP32 sums in ascending
//            point order, divided in FP64, rounded to FP32 once
// Most distances are never formed.  A row knows a reference it is near to (its candidate
// in the rounds and in Lloyd's first assignment, its center after): a center farther
// than 2 r + tau from the reference (r the row's distance to it, tau the reference's to
// some center) cannot be the row's nearest, so the centers within that reach are listed
// once per reference and a row examines its list.  In a round of several parts each part's
// candidates serve as references for the next part.  Lloyd keeps an upper bound (the exact
// distance to the row's center) and a lower one to all others between iterations, and
// sums again only the clusters whose members changed.  Rows beyond the lists go through the
// dense pass.  Margins of some 20 tie windows keep every center that is left out beyond
// the tie window, so all decisions are those of the dense passes.
// Distances are the exact FP32 difference form (ascending coordinates, one
// rounded subtraction and one FMA each), so every decision equals kmpar_fit's
// FP32 path on the same problem.
#include <float.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <vector>

#include <cooperative_groups.h>

#include "kmpar_internal.cuh"

namespace cg = cooperative_groups;

namespace kmp {
void set_thread_error(const std::string &m);

namespace {

constexpr int kBT = 256;          // threads per problem block
constexpr int kBW = kBT / 32;     // warps per block
constexpr int kBMaxCluster = 8;   // blocks per problem
constexpr int kBMinRows = 400;    // a finer cut for few problems ends here, where a row has some work (kBMinWork)
constexpr int kBMinWork = 2048;   // centers x padded coordinates
constexpr int kBRows = 128;       // rows of a tile
constexpr int kBCols = 64;        // centers of a tile
constexpr int kBXS = kBRows + 4, kBCS = kBCols + 4;   // floats per coordinate in shared memory
constexpr int kBMaxK = 512;
constexpr int kBMaxRounds = 16;
constexpr int kBMaxCap = 4096;    // per-round draw capacity

// device copy of one problem with its work-space offsets
struct BProb {
    int64_t x_off, n;
    int d, k;
    double ell;
    int rounds, max_iter;
    uint64_t seed;
    int64_t c_off, l_off, cand_off;   // outputs
    int64_t p_off, m_off;             // work space: per-point arrays, per-candidate arrays
    int64_t f_off, k_off;             // per-reference arrays (candidates or centers), per-center arrays
    int64_t s_off;                    // first float of the centers before an update
    int cap_round, cap_total;
};

struct BRes {
    long long m;
    double seed_cost, final_cost;
    int iters, status;
    unsigned long long sample_near, argmin_fp64, recluster_near;
};

struct BArgs {
    const float *X;
    const BProb *probs;
    const int32_t *order;    // problems of this launch, largest first
    float *centers;
    int32_t *labels_out;     // nullable
    int32_t *cand_out;       // nullable
    long long *w_out;        // nullable
    BRes *res;
    bool lists;              // the lists have their memory
    bool tiles;              // the launch has the shared memory of tiles and lists
    // work space
    float *D2;
    int32_t *idx, *lab, *perm;
    int32_t *cand;
    int32_t *w;
    float *rD2;
    unsigned int *rad;       // per reference: squared radius of its rows, then the one its list covers (< 0: none)
    int32_t *lcnt, *lst;     // its list
    float *tau2;             // squared distance to its nearest center (first assignment)
    float *drift;            // per center
    int32_t *flag;           // per center: its members changed
    float *cold;
};

constexpr int kBList = 16;   // entries of a reference's list
// Centers x padded coordinates from which a dense pass goes by tiles of rows.  Below, a tile is
// mostly its copies and its merge: 11 assignments of 2,975 x 15 to 6 centers take 0.23 ms a
// row per thread and 1.2 ms by tiles; 64 problems of 30,000 - 60,000 x 101, k = 30 - 60, 67 ms
// with the line at 64 centers and 72 at 32.  Above, the tiles' reuse counts: 64 problems of
// 500 - 3,000 rows, up to 60 centers, 3.8 ms with the rule and 4.6 ms with a row per thread
// alone; of 30,000 - 60,000 x 128, k = 200 - 256, 235 ms by tiles and 276 without.
template <int DP>
constexpr int kBTileWork = DP == 128 ? 8192 : 4096;
// Fewer rows go through the dense passes alone (lists, radii and their barriers cost more
// there than the few tiles they save).  With lists 512 problems of up to 200,000 rows,
// d = 32 - 128, take 305 ms instead of 577, 273 with the tiles below and step 8 over the
// whole cluster (22 -> 2.4 ms of the largest problem's time).
constexpr int kBListRows = 4096;
// Centers x coordinates of a dense pass from which lists pay: a row against its list costs some
// 15 to 30 ns of its block whatever the dimension (16 rows a warp), and its pairs' rows and
// centers are staged, by 16-byte copies where their rows allow it, else by 4-byte ones.
// 64 problems of 30,000 - 60,000 rows, k = 30 - 60, mixtures with R = 10, without lists / with:
// d = 128 75 ms / 42, d = 64 47 / 30; d = 101 55 / 65, d = 42 34 / 39.
constexpr int kBListWork = 8192, kBListWorkVec = 1024;
// After a list pass that left over 7/8 of the references without a list, or most rows open (the
// data do not separate), the problem goes on densely until its references are this many times
// as many.
constexpr int kBListRetry = 6;

enum { BM_FIRST = 0, BM_ROUND = 1, BM_ASSIGN = 2 };

// Deterministic block sum of one FP64 per thread: fixed shuffle tree, warps in
// order; the result is returned to every thread.
__device__ __forceinline__ double bsum_f64(double v, double *sh) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double r = 0.0;
    for (int i = 0; i < kBW; ++i) r += sh[i];
    return r;
}

__device__ __forceinline__ int bsum_i32(int v, int *sh) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    int r = 0;
    for (int i = 0; i < kBW; ++i) r += sh[i];
    return r;
}

// one term of the exact FP32 difference form: t = x - c rounded, a = fma(t, t, a)
__device__ __forceinline__ void sq_acc(float x, float c, float &a) {
    const float t = __fsub_rn(x, c);
    a = __fmaf_rn(t, t, a);
}

__device__ __forceinline__ void take_better(double v, int j, double &best, int &bj) {
    if (v < best || (v == best && j < bj)) { best = v; bj = j; }
}

// a distance known to be at most / at least the real one, from an exact FP32 square
__device__ __forceinline__ float upper_of(float v, float W) { return sqrtf(v * (1.f + W)) * (1.f + 1e-6f); }
__device__ __forceinline__ float lower_of(float v, float W) { return sqrtf(v * (1.f - 2.f * W)) * (1.f - 1e-6f); }
// ... of the runner-up v (center j; j < 0: the squares of all others are beyond FP32, which
// puts them that far and no farther)
__device__ __forceinline__ float runner_up(float v, int j, float W) { return lower_of(j >= 0 ? v : FLT_MAX, W); }

// Shared state of one block.
template <int DP>
struct BShared {
    float pick[(DP + 7) & ~7]; // step 8: the picked row, zero-padded
    double mass[kBMaxCluster]; // step 8: the blocks' masses
    int s_pick, s_first;       // step 8: the drawn candidate, the first one
    int lcount[kBRows];        // list_pass: entries per reference of the tile
    double red[kBW];
    int redi[kBW];
    int hist[kBW][kBMaxK];     // Lloyd: per-warp label counts, then the warps' running bases
    int base[kBMaxK + 1];      // Lloyd: cluster offsets
    int wpos[kBW];
    int s_int[4];
    int wl_tot[kBMaxK];        // Lloyd (rank 0): label totals over the cluster
    float drift[kBMaxK];       // Lloyd: per center, then the largest and second largest and whose the first is
    float s_m1, s_m2;
    int s_mi;
    int s_cnt;                 // rows listed by the block
    bool tiles;                // the launch's shared memory holds tiles
    int s_dead;                // list_pass: references of the block whose lists cover no row
    double s_dslot;
    int s_islot;
    unsigned long long s_uslot;
    unsigned long long s_near, s_fp64, s_rnear;
};

// dynamic shared memory of a block: a tile of rows and two of centers, or, in the row
// passes, kBStage rows a warp
constexpr int kBStage = 16;       // staged rows of X and of centers per warp and step
__host__ __device__ constexpr int stage_stride(int dp) { return ((dp >> 2) | 1) * 4; }   // floats, 16-byte units odd
__host__ __device__ constexpr size_t batch_smem(int dp) {
    const size_t tiles = sizeof(float) * dp * (kBXS + 2 * kBCS);
    const size_t stage = sizeof(float) * kBW * (2 * kBStage * stage_stride(dp) + 2 * kBStage);
    return tiles > stage ? tiles : stage;
}

// ... and of a launch whose problems have no use for tiles or lists (see uses_tiles): the rows
// a thread reads then find an L1 to stay in
constexpr size_t kBLeanSmem = 16 * 1024;

__device__ __forceinline__ void copy4(uint32_t dst, const float *src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void copy16(float *dst, const float *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// rows r = 0 .. B - 1 (row(r): the source, null past the end: zeros) to dst[q stride + r],
// consecutive threads along a row and then the next
template <typename F>
__device__ __forceinline__ void tile_copy(float *dst, int stride, int B, F row, const float *any, int d) {
    int r = threadIdx.x / d, q = threadIdx.x % d;
    const int dr = kBT / d, dq = kBT % d;
    while (r < B) {
        const float *src = row(r);
        copy4(static_cast<uint32_t>(__cvta_generic_to_shared(dst + q * stride + r)), src ? src + q : any, src != nullptr);
        r += dr;
        q += dq;
        if (q >= d) { q -= d; ++r; }
    }
}

// The exact FP32 distances of 128 rows (row(r), null: none) to cnt centers (center(j)),
// 64 centers at a time: a thread holds 4 rows x 8 centers of the tile and adds coordinate
// after coordinate (t = x - c, acc = fma(t, t, acc), ascending), so 32 independent chains
// keep the FP32 pipe busy and each shared-memory read feeds several; the next centers are
// copied while one tile is summed.  use(acc, c0) takes a tile's values: thread (ty, tx)'s
// rows 4 ty + i, centers c0 + (j / 4) 32 + j % 4 (past cnt: distances to 0).  About three
// times the rate of a row a thread with 8 chains over 32 centers.
template <int DP, typename R, typename K, typename U>
__device__ __forceinline__ void tile_scan(float *dsm, int d, const float *any, R row, int cnt, K center, U use) {
    float *xs = dsm, *cs = dsm + DP * kBXS;
    const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
    __syncthreads();   // the shared memory is free
    if (cnt > 0) {
        tile_copy(xs, kBXS, kBRows, row, any, d);
        tile_copy(cs, kBCS, kBCols, [&](int r) { return r < cnt ? center(r) : nullptr; }, any, d);
    }
    copies_commit();
    for (int t0 = 0, buf = 0; t0 < cnt; t0 += kBCols, buf ^= 1) {
        copies_wait();
        __syncthreads();   // this tile is in, and every thread is done with the one before
        if (t0 + kBCols < cnt)
            tile_copy(cs + (buf ^ 1) * DP * kBCS, kBCS, kBCols,
                      [&](int r) { return t0 + kBCols + r < cnt ? center(t0 + kBCols + r) : nullptr; }, any, d);
        copies_commit();
        float acc[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
        const float *xq = xs + ty * 4, *cq = cs + buf * DP * kBCS + tx * 4;
#pragma unroll 2
        for (int q = 0; q < d; ++q, xq += kBXS, cq += kBCS) {
            const float4 x = *reinterpret_cast<const float4 *>(xq);
            const float4 u = *reinterpret_cast<const float4 *>(cq), w = *reinterpret_cast<const float4 *>(cq + 32);
            const float xv[4] = {x.x, x.y, x.z, x.w}, cv[8] = {u.x, u.y, u.z, u.w, w.x, w.y, w.z, w.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) sq_acc(xv[i], cv[j], acc[i][j]);
        }
        use(acc, t0 + tx * 4);
    }
    copies_wait();
}

__device__ __forceinline__ bool lex_less(float v, int i, float w, int j) { return v < w || (v == w && i < j); }

// What a pass works on and writes; see dist_pass
struct BPass {
    const float *X, *C_rows;
    const int32_t *cand, *list;
    float *D2;
    int32_t *idx, *lab;
    float *dm, *lb;
    int32_t *flag;
    int d, begin, cnt;
    bool count;   // ASSIGN: count changed labels

    __device__ __forceinline__ int64_t number(int64_t r) const { return list ? (int64_t)list[r] : r; }
    __device__ __forceinline__ const float *crow(int j) const {
        return cand ? X + (int64_t)cand[j] * d : C_rows + (int64_t)j * d;
    }
};

// row pt with its smallest distance m1 (center n1, -1: none) and runner-up m2 (n2)
template <int MODE>
__device__ __forceinline__ void row_decide(const BPass &p, int64_t pt, float m1, int n1, float m2, int n2, int &chg,
                                           unsigned long long &nfp64) {
    const float W = fp32_tie_window(p.d);
    const float *xrow = p.X + pt * p.d;
    if (MODE == BM_FIRST) {
        p.D2[pt] = (n1 >= 0) ? m1 : __int_as_float(0x7f800000);
        p.idx[pt] = 0;
    } else if (MODE == BM_ASSIGN) {
        int l = n1 >= 0 ? n1 : 0;
        float stored = m1;
        if (n2 >= 0 && m2 <= m1 + W * m1) {
            double best = dist2_fp64(xrow, p.crow(n1), p.d);
            int bj = n1;
            take_better(dist2_fp64(xrow, p.crow(n2), p.d), n2, best, bj);
            if (bj == n2) { l = n2; stored = m2; }
            ++nfp64;
        }
        if (p.count && p.lab[pt] != l) {
            ++chg;
            if (p.flag) { p.flag[p.lab[pt]] = 1; p.flag[l] = 1; }
        }
        p.lab[pt] = l;
        p.dm[pt] = stored;
        p.lb[pt] = runner_up(l == n1 ? m2 : m1, n2, W);
    } else {
        const float old = p.D2[pt];
        const int oi = p.idx[pt];
        const float m32 = fminf(old, m1);
        const float lim = m32 + W * m32;
        const bool in_old = (oi >= 0) && old <= lim;
        const bool in1 = n1 >= 0 && m1 <= lim;
        const bool in2 = n2 >= 0 && m2 <= lim;
        int win = -1;
        float wv = old;
        if ((int)in_old + (int)in1 + (int)in2 >= 2) {
            double best = DBL_MAX;
            int bj = INT_MAX;
            if (in_old) take_better(dist2_fp64(xrow, p.X + (int64_t)p.cand[oi] * p.d, p.d), oi, best, bj);
            if (in1) take_better(dist2_fp64(xrow, p.crow(n1), p.d), n1, best, bj);
            if (in2) take_better(dist2_fp64(xrow, p.crow(n2), p.d), n2, best, bj);
            ++nfp64;
            if (bj == n1) { win = n1; wv = m1; }
            else if (bj == n2) { win = n2; wv = m2; }
        } else if (n1 >= 0 && m1 < old) {
            win = n1; wv = m1;
        }
        if (win >= 0) { p.D2[pt] = wv; p.idx[pt] = win; }
    }
}

// rows by tiles: 4 rows x 8 centers a thread
template <int DP, int MODE>
__device__ __noinline__ int rows_by_tile(const BPass p, float *dsm, int64_t r0, int64_t r1, unsigned long long *fp64_cnt) {
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    int chg = 0;
    unsigned long long nfp64 = 0;
    for (int64_t base = r0; base < r1; base += kBRows) {
        float b1[4], b2[4];
        int i1[4], i2[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { b1[i] = b2[i] = FLT_MAX; i1[i] = i2[i] = INT_MAX; }
        tile_scan<DP>(
            dsm, p.d, p.X,
            [&](int r) -> const float * { return base + r < r1 ? p.X + p.number(base + r) * p.d : nullptr; }, p.cnt,
            [&](int j) { return p.crow(p.begin + j); },
            [&](float (&acc)[4][8], int c0) {
                if (c0 - tx * 4 + kBCols > p.cnt) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (c0 + (j >> 2) * 32 + (j & 3) >= p.cnt) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) acc[i][j] = FLT_MAX;
                        }
                }
                // a row whose smallest value is not below its runner-up needs no more
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float m = acc[i][0];
#pragma unroll
                    for (int j = 1; j < 8; ++j) m = fminf(m, acc[i][j]);
                    if (m < b2[i]) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float v = acc[i][j];
                            if (v < b2[i]) {
                                const int c = p.begin + c0 + (j >> 2) * 32 + (j & 3);
                                if (v < b1[i]) { b2[i] = b1[i]; i2[i] = i1[i]; b1[i] = v; i1[i] = c; }
                                else { b2[i] = v; i2[i] = c; }
                            }
                        }
                    }
                }
            });
        // merge the 8 threads of a row, then thread tx = i decides the thread row's row i
        float m1 = FLT_MAX, m2 = FLT_MAX;
        int n1 = INT_MAX, n2 = INT_MAX;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float v1 = b1[i], v2 = b2[i];
            int j1 = i1[i], j2 = i2[i];
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                const float u1 = __shfl_xor_sync(0xffffffffu, v1, o), u2 = __shfl_xor_sync(0xffffffffu, v2, o);
                const int k1 = __shfl_xor_sync(0xffffffffu, j1, o), k2 = __shfl_xor_sync(0xffffffffu, j2, o);
                if (lex_less(u1, k1, v1, j1)) {
                    if (lex_less(v1, j1, u2, k2)) { v2 = v1; j2 = j1; } else { v2 = u2; j2 = k2; }
                    v1 = u1; j1 = k1;
                } else if (lex_less(u1, k1, v2, j2)) {
                    v2 = u1; j2 = k1;
                }
            }
            if (tx == i) { m1 = v1; m2 = v2; n1 = j1 == INT_MAX ? -1 : j1; n2 = j2 == INT_MAX ? -1 : j2; }
        }
        const int64_t at = base + ty * 4 + tx;
        if (tx < 4 && at < r1) row_decide<MODE>(p, p.number(at), m1, n1, m2, n2, chg, nfp64);
    }
    if (nfp64) atomicAdd(fp64_cnt, nfp64);
    return chg;
}

// a row per thread, its coordinates in registers (padded to DP with zeros: they add exact
// zeros to the sums); 8 chains, one per center, over centers 32 at a time.  Inlined: as a
// function of its own the compiler serialised the chains (11% fewer instructions an issue slot;
// 400 problems of 300 - 2,000 x 42, k = 30 - 60: 4.6 ms, inlined 3.8).
template <int DP, int MODE>
__device__ __forceinline__ int rows_by_thread(const BPass p, float *dsm, int64_t r0, int64_t r1,
                                           unsigned long long *fp64_cnt) {
    constexpr int B = 32, NCH = 8, P = DP / 2;
    const int tid = threadIdx.x, lane = tid & 31;
    float *stage = dsm + B * DP + (tid >> 5) * 32 * (P + 1);
    int chg = 0;
    unsigned long long nfp64 = 0;
    for (int64_t base = r0; base < r1; base += kBT) {
        const bool valid = base + tid < r1;
        const int64_t pt = valid ? p.number(base + tid) : 0;
        const float *xrow = p.X + pt * p.d;
        float xr[DP];
#pragma unroll
        for (int q = 0; q < DP; ++q) xr[q] = (valid && q < p.d) ? __ldg(xrow + q) : 0.f;
        float b1 = FLT_MAX, b2 = FLT_MAX;
        int i1 = -1, i2 = -1;
        auto take = [&](float a, int j) {
            if (a < b2) {
                if (a < b1) { b2 = b1; i2 = i1; b1 = a; i1 = j; }
                else { b2 = a; i2 = j; }
            }
        };
        for (int t0 = 0; t0 < p.cnt; t0 += B) {
            const int nt = min(B, p.cnt - t0);
            if (p.cnt > B || base == r0) {   // one tile stays for all the rows
                __syncthreads();
                for (int e = tid; e < B * DP; e += kBT) {
                    const int r = e / DP, q = e - r * DP;
                    dsm[e] = r < nt && q < p.d ? p.crow(p.begin + t0 + r)[q] : 0.f;
                }
                __syncthreads();
            }
            if (!valid) continue;
            int r = 0;
            for (; r + NCH <= nt; r += NCH) {
                float acc[NCH];
#pragma unroll
                for (int u = 0; u < NCH; ++u) acc[u] = 0.f;
#pragma unroll
                for (int q4 = 0; q4 < DP / 4; ++q4) {
                    float4 cv[NCH];
#pragma unroll
                    for (int u = 0; u < NCH; ++u) cv[u] = reinterpret_cast<const float4 *>(dsm + (r + u) * DP)[q4];
#pragma unroll
                    for (int u = 0; u < NCH; ++u) sq_acc(xr[4 * q4 + 0], cv[u].x, acc[u]);
#pragma unroll
                    for (int u = 0; u < NCH; ++u) sq_acc(xr[4 * q4 + 1], cv[u].y, acc[u]);
#pragma unroll
                    for (int u = 0; u < NCH; ++u) sq_acc(xr[4 * q4 + 2], cv[u].z, acc[u]);
#pragma unroll
                    for (int u = 0; u < NCH; ++u) sq_acc(xr[4 * q4 + 3], cv[u].w, acc[u]);
                }
#pragma unroll
                for (int u = 0; u < NCH; ++u) take(acc[u], p.begin + t0 + r + u);
            }
            for (; r < nt; ++r) {
                float a = 0.f;
#pragma unroll
                for (int q4 = 0; q4 < DP / 4; ++q4) {
                    const float4 u = reinterpret_cast<const float4 *>(dsm + r * DP)[q4];
                    sq_acc(xr[4 * q4 + 0], u.x, a);
                    sq_acc(xr[4 * q4 + 1], u.y, a);
                    sq_acc(xr[4 * q4 + 2], u.z, a);
                    sq_acc(xr[4 * q4 + 3], u.w, a);
                }
                take(a, p.begin + t0 + r);
            }
        }
        if (valid) row_decide<MODE>(p, pt, b1, i1, b2, i2, chg, nfp64);
    }
    if (nfp64) atomicAdd(fp64_cnt, nfp64);
    return chg;
}

// ... as a function of its own above 64 coordinates, where a block has the SM's registers
template <int DP, int MODE>
__device__ __noinline__ int rows_by_thread_wide(const BPass p, float *dsm, int64_t r0, int64_t r1,
                                                unsigned long long *fp64_cnt) {
    return rows_by_thread<DP, MODE>(p, dsm, r0, r1, fp64_cnt);
}

// One pass over the rows [r0, r1) of a problem (with `list`: the rows list[r0 .. r1))
// against `cnt` centers: the rows of C_rows (a center matrix, stride d) or, when cand is
// given, X rows cand[begin + r].  Each row's lexicographic (value, center number) top-2
// decides as the FP32 path does:
//   FIRST   D^2 = the single distance, idx = 0
//   ROUND   the current center is replaced by the best new one when nearer; two
//           or more of (current, best, runner-up) within the FP32 tie window are
//           re-decided in FP64 (difference form, no FMA), equal values keeping
//           the lower center number
//   ASSIGN  the best, re-decided in FP64 against the runner-up inside the window; takes
//           the distance to it and a lower bound of the distance to every other center
//           (dm, lb), and marks the centers that a row left or joined (flag; nullable)
// Sets *changed to the block's number of changed labels.
template <int DP, int MODE>
__device__ __forceinline__ void dist_pass(BShared<DP> &sh, float *dsm, const float *__restrict__ Xp, int64_t r0, int64_t r1,
                                          int d, const float *C_rows, const int32_t *__restrict__ cand, int begin, int cnt,
                                          float *D2, int32_t *idx, int32_t *lab, int *changed,
                                          unsigned long long *fp64_cnt, const int32_t *list = nullptr,
                                          float *dm = nullptr, float *lb = nullptr, int32_t *flag = nullptr) {
    const BPass p{Xp, C_rows, cand, list, D2, idx, lab, dm, lb, flag, d, begin, cnt, changed != nullptr};
    __syncthreads();
    int chg = 0;
    if (sh.tiles && cnt * DP >= kBTileWork<DP>) chg = rows_by_tile<DP, MODE>(p, dsm, r0, r1, fp64_cnt);
    else if constexpr (DP <= 64) chg = rows_by_thread<DP, MODE>(p, dsm, r0, r1, fp64_cnt);
    else chg = rows_by_thread_wide<DP, MODE>(p, dsm, r0, r1, fp64_cnt);
    if (MODE == BM_ASSIGN && changed) *changed = bsum_i32(chg, sh.redi);   // every thread
    __syncthreads();
}

// Exact FP32 distances of rows and centers of a warp's choice.  A warp brings up to kBStage
// rows of X (lane r < kBStage: row xr, null: none) and as many centers (cr) into its part of
// the shared memory, whole rows at a time, at a stride of an odd number of 16-byte units
// (a lane-per-row 16-byte read is then conflict-free), and lane p forms the distance of
// its center to staged row xi, or, once the sum passes lim, a value between lim and it.  Rows of 16-byte pieces (vec) take 16-byte copies.
__device__ __forceinline__ void stage_rows(float *dst, int ss, const float *row, int d, bool vec, int lane) {
    const unsigned long long mine = reinterpret_cast<unsigned long long>(row);
#pragma unroll 4
    for (int r = 0; r < kBStage; ++r) {
        const float *src = reinterpret_cast<const float *>(__shfl_sync(0xffffffffu, mine, r));
        if (!src) continue;
        float *to = dst + r * ss;
        if (vec) {
            if (4 * lane < d) copy16(to + 4 * lane, src + 4 * lane);   // d <= 128
        } else {
            for (int q = lane; q < d; q += 32)
                copy4(static_cast<uint32_t>(__cvta_generic_to_shared(to + q)), src + q, true);
        }
    }
}
__device__ __forceinline__ float stage_dist2(const float *x, const float *c, int d, bool vec, float lim) {
    float v = 0.f;
    if (vec) {
#pragma unroll 8
        for (int q = 0; q < d; q += 4) {
            if ((q & 31) == 0 && v > lim) return v;
            const float4 a = *reinterpret_cast<const float4 *>(x + q), b = *reinterpret_cast<const float4 *>(c + q);
            sq_acc(a.x, b.x, v);
            sq_acc(a.y, b.y, v);
            sq_acc(a.z, b.z, v);
            sq_acc(a.w, b.w, v);
        }
    } else {
#pragma unroll 4
        for (int q = 0; q < d; ++q) {
            if ((q & 15) == 0 && v > lim) return v;
            sq_acc(x[q], c[q], v);
        }
    }
    return v;
}

// The lists of up to kBStage rows of a warp (lane r < kBStage: its row x, n entries at
// l, center(j): an entry's coordinates; the other lanes n = 0): the (row, entry) pairs are
// dealt to lanes kBStage at a time; take(v, j) is called in the row's lane for each.
template <int DP, typename K, typename T>
__device__ __forceinline__ void warp_lists(float *ws, const float *x, int n, const int32_t *l, int d, bool vec, float lim,
                                           K center, T take) {
    constexpr int ss = stage_stride(DP);
    const int lane = threadIdx.x & 31;
    float *xs = ws, *cs = ws + kBStage * ss, *pv = cs + kBStage * ss;
    int32_t *pj = reinterpret_cast<int32_t *>(pv + kBStage);
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    const int excl = incl - n, P = __shfl_sync(0xffffffffu, incl, 31);
    const unsigned long long lp = reinterpret_cast<unsigned long long>(l);
    for (int p0 = 0; p0 < P; p0 += kBStage) {   // uniform per warp
        const int pi = p0 + lane;
        int r = 0;   // the pair's row: the first whose inclusive count exceeds pi
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (__shfl_sync(0xffffffffu, incl, r + o - 1) <= pi) r += o;
        const int32_t *lr = reinterpret_cast<const int32_t *>(__shfl_sync(0xffffffffu, lp, r));
        const int er = pi - __shfl_sync(0xffffffffu, excl, r);
        const float limr = __shfl_sync(0xffffffffu, lim, r);
        const int j = lane < kBStage && pi < P ? lr[er] : -1;
        if (p0 == 0) stage_rows(xs, ss, n > 0 ? x : nullptr, d, vec, lane);
        stage_rows(cs, ss, j >= 0 ? center(j) : nullptr, d, vec, lane);
        copies_commit();
        copies_wait();
        __syncwarp();
        if (j >= 0) {
            pv[lane] = stage_dist2(xs + r * ss, cs + lane * ss, d, vec, limr);
            pj[lane] = j;
        }
        __syncwarp();   // the values are there; the staged rows are read
        for (int q = max(excl, p0); q < min(incl, p0 + kBStage); ++q) take(pv[q - p0], pj[q - p0]);
        __syncwarp();
    }
}

// The largest D^2 among each reference's rows (rad: bits, zeroed before).
__device__ void radius_pass(int64_t r0, int64_t r1, const float *D2, const int32_t *ref, unsigned int *rad) {
    for (int64_t pt = r0 + threadIdx.x; pt < r1; pt += kBT) {
        const unsigned int v = __float_as_uint(D2[pt]);
        unsigned int *r = rad + ref[pt];
        if (v > *reinterpret_cast<volatile unsigned int *>(r)) atomicMax(r, v);
    }
}

// Lists of references [f0, f1) (rows of the problem when cand is given: X rows cand[i];
// else the centers themselves, left off their own lists): the centers (rows of C_rows, or
// X rows ccand[begin + j]) within 2 r + tau, r^2 = rad[i], tau the distance to the nearest
// of them (want_tau; else 0).  A list that overflows is taken again at half the radius,
// three times at most.  On return rad[i] holds the bits of the squared radius covered
// (-1: none; sh.s_dead of the block's), lcnt and lst the list (numbers from begin, in no order).
template <int DP>
__device__ __noinline__ void list_pass(BShared<DP> &sh, float *dsm, const float *__restrict__ Xp, int f0, int f1, int d,
                                       const int32_t *__restrict__ cand, const float *C_rows,
                                       const int32_t *__restrict__ ccand, int begin, int cnt, bool want_tau,
                                       unsigned int *rad, int32_t *lcnt, int32_t *lst, float *tau2) {
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const float W = fp32_tie_window(d);
    const float INF = __int_as_float(0x7f800000);
    auto center = [&](int j) -> const float * {
        return ccand ? Xp + (int64_t)ccand[begin + j] * d : C_rows + (int64_t)(begin + j) * d;
    };
    __syncthreads();
    if (tid == 0) sh.s_dead = 0;
    __syncthreads();
    for (int base = f0; base < f1; base += kBRows) {   // uniform per block
        auto row = [&](int r) -> const float * {
            const int i = base + r;
            return i < f1 ? (cand ? Xp + (int64_t)cand[i] * d : C_rows + (int64_t)i * d) : nullptr;
        };
        // thread (ty, tx) looks at the values of references base + 4 ty + i
        float r2[4], tau[4];
        bool active[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int f = base + ty * 4 + i;
            active[i] = f < f1;
            r2[i] = active[i] ? __uint_as_float(rad[f]) : 0.f;
            tau[i] = 0.f;
        }
        if (want_tau) {
#pragma unroll
            for (int i = 0; i < 4; ++i) tau[i] = INF;
            tile_scan<DP>(dsm, d, Xp, row, cnt, center, [&](float (&acc)[4][8], int c0) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (c0 + (j >> 2) * 32 + (j & 3) < cnt) tau[i] = fminf(tau[i], acc[i][j]);
            });
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) tau[i] = fminf(tau[i], __shfl_xor_sync(0xffffffffu, tau[i], o));
        }
        for (int level = 0; level < 4; ++level) {
            if (!__syncthreads_or(active[0] || active[1] || active[2] || active[3])) break;
            float reach2[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float reach = 2.f * sqrtf(r2[i]) + sqrtf(tau[i]);
                reach2[i] = reach * reach * (1.f + 24.f * W);
                if (tx == 0) sh.lcount[ty * 4 + i] = 0;
            }
            tile_scan<DP>(dsm, d, Xp, row, cnt, center, [&](float (&acc)[4][8], int c0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (!active[i]) continue;
                    const int f = base + ty * 4 + i;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int c = c0 + (j >> 2) * 32 + (j & 3);
                        if (c < cnt && !(acc[i][j] > reach2[i]) && (cand || c != f)) {
                            const int at = atomicAdd(&sh.lcount[ty * 4 + i], 1);
                            if (at < kBList) lst[(size_t)f * kBList + at] = begin + c;
                        }
                    }
                }
            });
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (!active[i]) continue;
                const int n = sh.lcount[ty * 4 + i], f = base + ty * 4 + i;
                if (n <= kBList) {
                    active[i] = false;
                    if (tx == 0) {
                        rad[f] = __float_as_uint(r2[i]);
                        lcnt[f] = n;
                    }
                } else {
                    r2[i] *= 0.25f;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int f = base + ty * 4 + i;
            if (tx != 0 || f >= f1) continue;
            if (active[i]) {
                rad[f] = __float_as_uint(-1.f);
                lcnt[f] = 0;
                atomicAdd(&sh.s_dead, 1);
            }
            if (want_tau) tau2[f] = tau[i];
        }
        __syncthreads();
    }
}

// block-ordered append of the taken rows to list[*count ..); every thread of the block calls
__device__ __forceinline__ void block_append(bool take, int32_t row, int32_t *list, int *count) {
    const int lane = threadIdx.x & 31;
    const unsigned m = __ballot_sync(0xffffffffu, take);
    int b = 0;
    if (lane == 0 && m) b = atomicAdd(count, __popc(m));
    b = __shfl_sync(0xffffffffu, b, 0);
    if (take) list[b + __popc(m & ((1u << lane) - 1u))] = row;
}

// Rows [r0, r1) against the lists of their references; rows beyond them to open (room for
// the block's rows), their number to sh.s_cnt.
//   ROUND   ref = idx, distance D2, centers X rows cand[j]; D2 / idx updated
//   ASSIGN  ref = idx, distance D2 (overwritten: the distance to the chosen center; idx
//           becomes the lower bound lb, the same memory), centers C rows
template <int MODE, int DP>
__device__ __noinline__ void lists_rows(BShared<DP> &sh, float *dsm, const float *__restrict__ Xp, int64_t r0, int64_t r1,
                                        int d, bool vec, const float *C_rows, const int32_t *cand,
                                        const unsigned int *rad, const int32_t *lcnt, const int32_t *lst,
                                        const float *tau2, float *D2, int32_t *idx, int32_t *lab, int32_t *open,
                                        unsigned long long *fp64_cnt) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const float W = fp32_tie_window(d);
    float *ws = dsm + wid * (2 * kBStage * stage_stride(DP) + 2 * kBStage);
    unsigned long long nfp64 = 0;
    __syncthreads();
    if (tid == 0) sh.s_cnt = 0;
    __syncthreads();
    auto crow = [&](int j) -> const float * {
        return MODE == BM_ROUND ? Xp + (int64_t)cand[j] * d : C_rows + (int64_t)j * d;
    };
    for (int64_t base = r0 + wid * kBStage; base < r1; base += kBW * kBStage) {   // uniform per warp
        const int64_t pt = base + lane;
        const bool mine = lane < kBStage && pt < r1;
        int a = 0, n = 0;
        float dd = 0.f, cov = -1.f;
        if (mine) {
            a = idx[pt];
            dd = D2[pt];
            cov = __uint_as_float(rad[a]);
            n = lcnt[a];
        }
        const bool op = mine && (!(dd <= cov) || (MODE == BM_ASSIGN && n == 0));
        if (op || !mine) n = 0;
        const float *xrow = Xp + (mine ? pt : r0) * d;
        float b1 = FLT_MAX, b2 = FLT_MAX;
        int i1 = -1, i2 = -1;
        warp_lists<DP>(ws, xrow, n, lst + (size_t)a * kBList, d, vec,
                       MODE == BM_ROUND ? dd * (1.f + 4.f * W) : FLT_MAX, crow, [&](float v, int j) {
            if (v < b1 || (v == b1 && j < i1)) { b2 = b1; i2 = i1; b1 = v; i1 = j; }
            else if (v < b2 || (v == b2 && j < i2)) { b2 = v; i2 = j; }
        });
        if (n > 0 && MODE == BM_ASSIGN) {
            int best = i1 >= 0 ? i1 : 0;
            float stored = b1;
            if (i2 >= 0 && b2 <= b1 + W * b1) {
                double bv = dist2_fp64(xrow, crow(i1), d);
                int bj = i1;
                take_better(dist2_fp64(xrow, crow(i2), d), i2, bv, bj);
                if (bj == i2) { best = i2; stored = b2; }
                ++nfp64;
            }
            const float off = (2.f * sqrtf(cov) + sqrtf(tau2[a])) * (1.f - 1e-6f) - upper_of(dd, W);
            lab[pt] = best;
            D2[pt] = stored;
            reinterpret_cast<float *>(idx)[pt] =
                fmaxf(0.f, fminf(off, runner_up(best == i1 ? b2 : b1, i2, W)));
        } else if (n > 0) {
            const float m32 = fminf(dd, b1), lim = m32 + W * m32;
            const bool in_old = dd <= lim, in1 = i1 >= 0 && b1 <= lim, in2 = i2 >= 0 && b2 <= lim;
            int win = -1;
            float wv = dd;
            if ((int)in_old + (int)in1 + (int)in2 >= 2) {
                double best = DBL_MAX;
                int bj = INT_MAX;
                if (in_old) take_better(dist2_fp64(xrow, crow(a), d), a, best, bj);
                if (in1) take_better(dist2_fp64(xrow, crow(i1), d), i1, best, bj);
                if (in2) take_better(dist2_fp64(xrow, crow(i2), d), i2, best, bj);
                ++nfp64;
                if (bj == i1) { win = i1; wv = b1; }
                else if (bj == i2) { win = i2; wv = b2; }
            } else if (i1 >= 0 && b1 < dd) {
                win = i1; wv = b1;
            }
            if (win >= 0) { D2[pt] = wv; idx[pt] = win; }
        }
        block_append(op, (int32_t)pt, open, &sh.s_cnt);
    }
    if (nfp64) atomicAdd(fp64_cnt, nfp64);
    __syncthreads();
}

// After a centroid update: rows whose bounds hold keep their center (its distance is
// recomputed only when it moved); the others are listed as pending (pend, number in
// sh.s_cnt) and their distance goes into their center's radius.
template <int DP>
__device__ __noinline__ void bounds_rows(BShared<DP> &sh, float *dsm, const float *__restrict__ Xp, int64_t r0, int64_t r1,
                                         int d, bool vec, const float *C, const int32_t *lab, float *dm, float *lb,
                                         unsigned int *rad, int32_t *pend) {
    constexpr int ss = stage_stride(DP);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const float W = fp32_tie_window(d);
    float *xs = dsm + wid * (2 * kBStage * ss + 2 * kBStage), *cs = xs + kBStage * ss;
    __syncthreads();
    if (tid == 0) sh.s_cnt = 0;
    __syncthreads();
    for (int64_t base = r0 + wid * kBStage; base < r1; base += kBW * kBStage) {   // uniform per warp
        const int64_t pt = base + lane;
        const bool mine = lane < kBStage && pt < r1;
        int a = 0;
        float v = 0.f, lo = 0.f;
        bool moved = false;
        if (mine) {
            a = lab[pt];
            moved = sh.drift[a] != 0.f;
            lo = lb[pt] - (a == sh.s_mi ? sh.s_m2 : sh.s_m1);
            v = dm[pt];
        }
        if (__any_sync(0xffffffffu, moved)) {
            stage_rows(xs, ss, moved ? Xp + pt * d : nullptr, d, vec, lane);
            stage_rows(cs, ss, moved ? C + (int64_t)a * d : nullptr, d, vec, lane);
            copies_commit();
            copies_wait();
            __syncwarp();
            if (moved) {
                v = stage_dist2(xs + lane * ss, cs + lane * ss, d, vec, FLT_MAX);
                dm[pt] = v;
            }
            __syncwarp();   // the staged rows are read
        }
        const bool pd = mine && !(lo > 0.f && upper_of(v, W) < lo);
        if (mine) lb[pt] = pd ? 0.f : lo;
        if (pd) {
            const unsigned int bits = __float_as_uint(v);
            if (bits > *reinterpret_cast<volatile unsigned int *>(rad + a)) atomicMax(rad + a, bits);
        }
        block_append(pd, (int32_t)pt, pend, &sh.s_cnt);
    }
    __syncthreads();
}

// The pending rows (np of them) against the lists of their centers; the rows beyond them
// stay, compacted, in pend (number in sh.s_cnt).  Returns the thread's changed labels.
template <int DP>
__device__ __noinline__ int pending_rows(BShared<DP> &sh, float *dsm, const float *__restrict__ Xp, int np, int d,
                                         bool vec, const float *C, const unsigned int *rad, const int32_t *lcnt,
                                         const int32_t *lst, int32_t *lab, float *dm, float *lb, int32_t *pend,
                                         int32_t *flag, unsigned long long *fp64_cnt) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const float W = fp32_tie_window(d);
    float *ws = dsm + wid * (2 * kBStage * stage_stride(DP) + 2 * kBStage);
    int chg = 0;
    unsigned long long nfp64 = 0;
    __syncthreads();
    if (tid == 0) sh.s_cnt = 0;
    __syncthreads();
    auto crow = [&](int j) -> const float * { return C + (int64_t)j * d; };
    for (int base = 0; base < np; base += kBW * kBStage) {   // uniform per block
        const int at = base + wid * kBStage + lane;
        const bool mine = lane < kBStage && at < np;
        int32_t pt = 0;
        int a = 0, n = 0;
        float dd = 0.f, cov = -1.f;
        if (mine) {
            pt = pend[at];
            a = lab[pt];
            dd = dm[pt];
            cov = __uint_as_float(rad[a]);
            n = lcnt[a];
        }
        // (a row whose own center's square is beyond FP32 has the dense pass's label and value)
        const bool op = mine && !(dd <= cov && dd < FLT_MAX);
        if (op || !mine) n = 0;
        const float *xrow = Xp + (int64_t)pt * d;
        float b1 = dd, b2 = FLT_MAX;
        int i1 = a, i2 = -1;
        warp_lists<DP>(ws, xrow, n, lst + (size_t)a * kBList, d, vec, FLT_MAX, crow, [&](float v, int j) {
            if (v < b1 || (v == b1 && j < i1)) { b2 = b1; i2 = i1; b1 = v; i1 = j; }
            else if (v < b2 || (v == b2 && j < i2)) { b2 = v; i2 = j; }
        });
        if (mine && !op) {
            int best = i1;
            float stored = b1;
            if (i2 >= 0 && b2 <= b1 + W * b1) {
                double bv = dist2_fp64(xrow, crow(i1), d);
                int bj = i1;
                take_better(dist2_fp64(xrow, crow(i2), d), i2, bv, bj);
                if (bj == i2) { best = i2; stored = b2; }
                ++nfp64;
            }
            if (best != a) {
                ++chg;
                flag[a] = 1;
                flag[best] = 1;
                lab[pt] = best;
                dm[pt] = stored;
            }
            const float off = 2.f * sqrtf(cov) * (1.f - 1e-6f) - upper_of(dd, W);
            lb[pt] = fmaxf(0.f, fminf(off, runner_up(best == i1 ? b2 : b1, i2, W)));
        }
        __syncthreads();   // the chunk's entries are read before rows are put back over them
        block_append(op, pt, pend, &sh.s_cnt);
    }
    if (nfp64) atomicAdd(fp64_cnt, nfp64);
    __syncthreads();
    return chg;
}

// the block's FP64 sum of v[r0 .. r1): a thread's rows in ascending order, then the block
template <int DP>
__device__ __forceinline__ double sum_rows_of(BShared<DP> &sh, const float *v, int64_t r0, int64_t r1) {
    double acc = 0.0;
    for (int64_t pt = r0 + threadIdx.x; pt < r1; pt += kBT) acc += (double)v[pt];
    return bsum_f64(acc, sh.red);
}

// Block-wide exclusive prefix of one FP64 per thread in thread order (warp scans,
// then the warp totals in order); returns the thread's exclusive prefix and the
// total (to every thread).
__device__ __forceinline__ double bscan_f64(double v, double *sh, double *total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    __syncthreads();
    if (lane == 31) sh[wid] = incl;
    __syncthreads();
    double before = 0.0, tot = 0.0;
    for (int i = 0; i < kBW; ++i) {
        if (i < wid) before += sh[i];
        tot += sh[i];
    }
    *total = tot;
    double excl = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) excl = 0.0;
    return before + excl;
}

__device__ __forceinline__ int bmin_i32(int v, int *sh) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    int r = INT_MAX;
    for (int i = 0; i < kBW; ++i) r = min(r, sh[i]);
    return r;
}

__device__ __forceinline__ int bmax_i32(int v, int *sh) { return -bmin_i32(-v, sh); }

// ---- a problem split over a thread-block cluster of CS blocks (CS = 1: one block)
// Barrier of the cluster (hardware; its arrive/wait pair orders memory at cluster
// scope, and the fence makes the global writes of this block visible first).
template <int CS>
__device__ __forceinline__ void csync() {
    if (CS > 1) {
        __threadfence();
        cg::this_cluster().sync();
    } else {
        __syncthreads();
    }
}

// Sum over the cluster's blocks, in rank order, of a block-uniform value: every
// block gets the same result.
template <int CS, typename T>
__device__ __forceinline__ T csum(T v, T *slot) {
    if (CS == 1) return v;
    __syncthreads();
    if (threadIdx.x == 0) *slot = v;
    cg::this_cluster().sync();
    T r = 0;
    for (int q = 0; q < CS; ++q) r += *cg::this_cluster().map_shared_rank(slot, q);
    cg::this_cluster().sync();   // no block overwrites its slot before every block has read it
    return r;
}

// Exclusive prefix in rank order and total of a block-uniform count.
template <int CS>
__device__ __forceinline__ int cprefix(int v, int *slot, int *total) {
    if (CS == 1) { *total = v; return 0; }
    __syncthreads();
    if (threadIdx.x == 0) *slot = v;
    cg::this_cluster().sync();
    const int me = (int)cg::this_cluster().block_rank();
    int before = 0, tot = 0;
    for (int q = 0; q < CS; ++q) {
        const int c = *cg::this_cluster().map_shared_rank(slot, q);
        if (q < me) before += c;
        tot += c;
    }
    cg::this_cluster().sync();
    *total = tot;
    return before;
}

// Knuth's TwoSum: (s, c) += x with s the rounded sum and c the accumulated
// rounding errors (all FP32, each operation rounded to nearest)
__device__ __forceinline__ void two_sum_add(float &s, float &c, float x) {
    const float t = __fadd_rn(s, x);
    const float bp = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(x, bp));
    c = __fadd_rn(c, e);
    s = t;
}

// One problem per cluster of CS blocks (CS = 1: one block).  Block rank r of the
// cluster owns the contiguous rows [r0, r1); every per-point step runs on the
// block's own rows, and the cluster combines in rank order: phi and the Lloyd
// cost and change counts (sums), the round draws (each block appends its draws in
// ascending point order after those of the lower ranks), and Lloyd's counting sort
// (label offsets over (rank, warp) in order).
template <int DP, int CS>
__global__ void __launch_bounds__(kBT, DP == 128 ? 1 : 2) batch_kernel(BArgs a, int first) {
    __shared__ BShared<DP> sh;
    extern __shared__ __align__(16) float dsm[];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int rank = CS > 1 ? (int)cg::this_cluster().block_rank() : 0;
    const int pi = a.order[first + blockIdx.x / CS];
    const BProb P = a.probs[pi];
    const float *X = a.X + P.x_off;
    const int64_t n = P.n;
    const int d = P.d, k = P.k;
    const int64_t per = (n + CS - 1) / CS;
    const int64_t r0 = min(n, (int64_t)rank * per), r1 = min(n, r0 + per);
    float *D2 = a.D2 + P.p_off;
    int32_t *idx = a.idx + P.p_off, *lab = a.lab + P.p_off, *perm = a.perm + P.p_off;
    int32_t *cand = a.cand + P.m_off, *w = a.w + P.m_off;
    float *rD2 = a.rD2 + P.m_off;
    float *C = a.centers + P.c_off;
    unsigned int *rad = a.rad + P.f_off;
    int32_t *lcnt = a.lcnt + P.f_off, *lst = a.lst + P.f_off * kBList;
    float *tau2 = a.tau2 + P.f_off;
    float *drift = a.drift + P.k_off, *cold = a.cold + P.s_off;
    int32_t *flag = a.flag + P.k_off;
    // rows of 16-byte pieces
    const bool vec = (d & 3) == 0 && ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(C)) & 15u) == 0;
    if (tid == 0) {
        sh.tiles = a.tiles;
        sh.s_near = 0; sh.s_fp64 = 0; sh.s_rnear = 0;
        if (rank == 0) {
            // Alg. 2 step 1: the first center, uniform over the problem's points
            const double u = uniform53(0, 0, TAG_INIT, P.seed);
            int64_t i0 = (int64_t)floor(__dmul_rn(u, (double)n));
            if (i0 >= n) i0 = n - 1;
            cand[0] = (int32_t)i0;
        }
    }
    csync<CS>();
    // step 2: D^2 to the first center and psi
    dist_pass<DP, BM_FIRST>(sh, dsm, X, r0, r1, d, nullptr, cand, 0, 1, D2, idx, nullptr, nullptr, &sh.s_fp64);
    double phi = csum<CS>(sum_rows_of(sh, D2, r0, r1), &sh.s_dslot);
    int m = 1, status = KMPAR_OK;
    int fail = 0;   // references of the last list pass if it left most rows open
    for (int r = 1; r <= P.rounds; ++r) {
        // step 4: independent draws of the block's rows; p and the near-draw rule as
        // in the single-problem path
        auto draw = [&](int64_t pt, bool &take, unsigned long long &near) {
            const float dd = D2[pt];
            double pr = 0.0;
            if (phi > 0.0) pr = fmin(1.0, __ddiv_rn(__dmul_rn(P.ell, (double)dd), phi));
            const double u = uniform53((uint64_t)pt, (uint32_t)r, TAG_SAMPLE, P.seed);
            if (dd > 0.f && fabs(u - pr) <= 1e-5) {
                // the FP32 D^2 could decide this draw: use the FP64 distance of the definition
                const double d64 = dist2_fp64(X + pt * d, X + (int64_t)cand[idx[pt]] * d, d);
                pr = fmin(1.0, __ddiv_rn(__dmul_rn(P.ell, d64), phi));
            }
            if (fabs(u - pr) <= 1e-6) ++near;
            take = u < pr;
        };
        // the block's place among the cluster's draws (a counting pass first)
        int mine = 0;
        if (CS > 1) {
            unsigned long long dummy = 0;
            int cntl = 0;
            for (int64_t pt = r0 + tid; pt < r1; pt += kBT) {
                bool take;
                draw(pt, take, dummy);
                cntl += take;
            }
            mine = bsum_i32(cntl, sh.redi);
        }
        int appended_all = 0;
        const int before_blocks = cprefix<CS>(mine, &sh.s_islot, &appended_all);
        int appended = 0;
        unsigned long long near = 0;
        for (int64_t base = r0; base < r1; base += kBT) {
            const int64_t pt = base + tid;
            bool take = false;
            if (pt < r1) draw(pt, take, near);
            const unsigned mask = __ballot_sync(0xffffffffu, take);
            if (lane == 0) sh.wpos[wid] = __popc(mask);
            __syncthreads();
            int before = 0, tot = 0;
            for (int i = 0; i < kBW; ++i) {
                if (i < wid) before += sh.wpos[i];
                tot += sh.wpos[i];
            }
            if (take) {
                const int pos = before_blocks + appended + before + __popc(mask & ((1u << lane) - 1u));
                if (pos < P.cap_round) cand[m + pos] = (int32_t)pt;
            }
            appended += tot;
            __syncthreads();   // wpos is rewritten by the next chunk
        }
        if (near) atomicAdd(&sh.s_near, near);
        if (CS == 1) appended_all = appended;
        if (appended_all > P.cap_round) { status = KMPAR_ERR_CAPACITY; break; }
        csync<CS>();           // the batch's row numbers are visible to the whole cluster
        // step 5: D^2 and idx against the batch, then phi.  While the references (the
        // candidates before a part of the batch) are few against the rows, their lists
        // settle most rows; a first round starts with a dense part.
        const bool lists = a.lists && a.tiles && n >= kBListRows && n >= 8 * (int64_t)(m + appended_all) &&
                           appended_all * d >= (vec ? kBListWorkVec : kBListWork);
        const int parts = max(1, min(4, appended_all / 64));
        for (int part = 0, from = 0; part == 0 || from < appended_all; ++part) {
            const int b0 = m + from;
            const bool by_list = lists && b0 > 1 && b0 >= kBListRetry * fail;
            // (the first part of a first round is dense, what lists have failed for all at once)
            if (by_list || (lists && b0 == 1)) from = min(appended_all, (int)((int64_t)appended_all * (part + 1) / parts));
            else from = appended_all;
            const int b1 = m + from;
            if (!by_list) {
                dist_pass<DP, BM_ROUND>(sh, dsm, X, r0, r1, d, nullptr, cand, b0, b1 - b0, D2, idx, nullptr, nullptr,
                                        &sh.s_fp64);
                csync<CS>();
                continue;
            }
            for (int j = rank * kBT + tid; j < b0; j += CS * kBT) rad[j] = 0u;
            csync<CS>();
            radius_pass(r0, r1, D2, idx, rad);
            csync<CS>();
            const int per_f = (b0 + CS - 1) / CS;
            list_pass<DP>(sh, dsm, X, min(b0, rank * per_f), min(b0, (rank + 1) * per_f), d, cand, nullptr, cand, b0, b1 - b0,
                          false, rad, lcnt, lst, nullptr);
            csync<CS>();
            if (8 * csum<CS>(sh.s_dead, &sh.s_islot) > 7 * b0) {   // (nor are there rows to look at)
                fail = b0;
                dist_pass<DP, BM_ROUND>(sh, dsm, X, r0, r1, d, nullptr, cand, b0, b1 - b0, D2, idx, nullptr, nullptr,
                                        &sh.s_fp64);
                csync<CS>();
                continue;
            }
            lists_rows<BM_ROUND, DP>(sh, dsm, X, r0, r1, d, vec, nullptr, cand, rad, lcnt, lst, nullptr, D2, idx, nullptr,
                                     perm + r0, &sh.s_fp64);
            const int no = sh.s_cnt;
            const int64_t open = csum<CS>(no, &sh.s_islot);
            fail = 8 * open > (r == 1 ? 7 : 6) * n ? b0 : 0;   // (round 1 still has clusters without a candidate)
            __syncthreads();
            dist_pass<DP, BM_ROUND>(sh, dsm, X, 0, no, d, nullptr, cand, b0, b1 - b0, D2, idx, nullptr, nullptr, &sh.s_fp64,
                                    perm + r0);
            csync<CS>();
        }
        phi = csum<CS>(sum_rows_of(sh, D2, r0, r1), &sh.s_dslot);
        m += appended_all;
    }
    BRes res{};
    res.m = m;
    if (status == KMPAR_OK) {
        // step 7: weights
        for (int j = (int)(rank * kBT) + tid; j < m; j += CS * kBT) w[j] = 0;
        csync<CS>();
        for (int64_t pt = r0 + tid; pt < r1; pt += kBT) atomicAdd(&w[idx[pt]], 1);
        csync<CS>();
        // step 8: weighted k-means++ over the m candidates, block r holding a contiguous
        // share [j0, j1) of them.  Each draw: the blocks' masses meet in every block, the one
        // that the target falls into picks, and all lower their candidates' D^2.  The
        // weights, the D^2 and the first Q coordinates (as many as fit, [q][candidate]:
        // consecutive threads then read consecutive words) stay in shared memory.
        bool warn = false;
        {
            const int per_m = (m + CS - 1) / CS;
            const int j0 = min(m, rank * per_m), ml = min(m, j0 + per_m) - j0;
            const int cap = (int)((a.tiles ? batch_smem(DP) : kBLeanSmem) / sizeof(float));
            const int mls = per_m | 1;   // odd: the transposing stores below meet no bank twice
            const bool in_smem = 2 * per_m <= cap;
            const int Q = in_smem ? min((cap - 2 * per_m) / mls & ~7, (d + 7) & ~7) : 0;
            float *rd = in_smem ? dsm : rD2 + j0;
            int32_t *ww = in_smem ? reinterpret_cast<int32_t *>(dsm + per_m) : w + j0;
            float *xT = dsm + 2 * per_m;
            __syncthreads();   // the passes before are done with the shared memory
            for (int j = tid; j < ml; j += kBT) {
                rd[j] = __int_as_float(0x7f800000);
                if (in_smem) ww[j] = w[j0 + j];
            }
            for (int j = wid; j < ml; j += kBW) {
                const float *src = X + (int64_t)cand[j0 + j] * d;
                for (int q = lane; q < Q; q += 32) xT[q * mls + j] = q < d ? __ldg(src + q) : 0.f;
            }
            __syncthreads();
            const int q = (ml + kBT - 1) / kBT;
            const int lo = min(ml, tid * q), hi = min(ml, lo + q);
            for (int t = 0; t < k; ++t) {
                double local = 0.0;
                for (int j = lo; j < hi; ++j)
                    local += t == 0 ? (double)ww[j] : __dmul_rn((double)ww[j], (double)rd[j]);
                double mine, total = 0.0, before = 0.0;
                double excl = bscan_f64(local, sh.red, &mine);
                int owner = -1;
                const double u = uniform53((uint64_t)t, 0, TAG_RECLUSTER, P.seed);
                double target;
                if (CS > 1) {
                    if (tid < CS) *cg::this_cluster().map_shared_rank(&sh.mass[rank], tid) = mine;
                    cg::this_cluster().sync();
                    for (int r = 0; r < CS; ++r) total += sh.mass[r];
                    target = __dmul_rn(u, total);
                    double run = 0.0;
                    for (int r = 0; r < CS; ++r) {
                        if (r == rank) before = run;
                        run += sh.mass[r];
                        if (owner < 0 && run > target) owner = r;
                    }
                    if (owner < 0)   // rounded past every prefix: the last block with mass
                        for (int r = 0; r < CS; ++r) owner = sh.mass[r] > 0.0 ? r : owner;
                    excl += before;
                } else {
                    total = mine;
                    target = __dmul_rn(u, total);
                    owner = 0;
                }
                if (!(total > 0.0)) {
                    // positive mass exhausted: the remaining centers repeat the first chosen one
                    if (rank == 0) {
                        const int64_t src = t > 0 ? cand[sh.s_first] : cand[0];
                        for (int s2 = t; s2 < k; ++s2)
                            for (int qq = tid; qq < d; qq += kBT) C[(int64_t)s2 * d + qq] = X[src * d + qq];
                    }
                    warn = true;
                    break;
                }
                if (rank == owner) {
                    // the first candidate whose prefix exceeds the target; a thread whose share
                    // ends well before it or starts well after it has none
                    int hit = INT_MAX;
                    double cum0 = 0.0, cum = 0.0, run = excl;
                    const double slack = 1e-9 * total;
                    if (target >= excl - slack && target <= excl + local + slack)
                        for (int j = lo; j < hi; ++j) {
                            const double e = t == 0 ? (double)ww[j] : __dmul_rn((double)ww[j], (double)rd[j]);
                            const double pre = run;
                            run = run + e;
                            if (run > target) { hit = j; cum0 = pre; cum = run; break; }
                        }
                    int pick = bmin_i32(hit, sh.redi);
                    if (pick == INT_MAX) {
                        // the target rounded past every prefix: the last candidate with positive mass
                        int lastp = -1;
                        for (int j = lo; j < hi; ++j)
                            if ((t == 0 ? (double)ww[j] : __dmul_rn((double)ww[j], (double)rd[j])) > 0.0) lastp = j;
                        pick = bmax_i32(lastp, sh.redi);
                        if (tid == 0) atomicAdd(&sh.s_rnear, 1ull);
                    } else if (hit == pick &&
                               (fabs(target - cum0) <= 1e-6 * total || fabs(cum - target) <= 1e-6 * total)) {
                        atomicAdd(&sh.s_rnear, 1ull);
                    }
                    pick += j0;
                    if (CS == 1) {
                        if (tid == 0) sh.s_pick = pick;
                    } else if (tid < CS) {
                        *cg::this_cluster().map_shared_rank(&sh.s_pick, tid) = pick;
                    }
                }
                if (CS > 1) cg::this_cluster().sync();
                else __syncthreads();
                const int pick = sh.s_pick;
                if (t == 0 && tid == 0) sh.s_first = pick;
                const float *prow = X + (int64_t)cand[pick] * d;
                for (int qq = tid; qq < ((DP + 7) & ~7); qq += kBT) {
                    const float v = qq < d ? prow[qq] : 0.f;
                    sh.pick[qq] = v;   // the pick's row, zero-padded to DP
                    if (rank == owner && qq < d) C[(int64_t)t * d + qq] = v;
                }
                __syncthreads();
                // D^2 of every candidate to the centers drawn so far, in the exact FP32
                // chain (t = x_q - c_q, fma, q ascending; padded zeros add 0).  The partial
                // sums never decrease, so once one reaches the candidate's D^2 the rest
                // cannot lower it and is skipped (most candidates are far from the pick).
                for (int j = tid; j < ml; j += kBT) {
                    const float lim = rd[j];
                    float v = 0.f;
                    int q0 = 0;
                    for (; q0 < Q && !(v >= lim); q0 += 8) {
                        float xr[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) xr[e] = xT[(q0 + e) * mls + j];
#pragma unroll
                        for (int e = 0; e < 8; ++e) sq_acc(xr[e], sh.pick[q0 + e], v);
                    }
                    const float *xj = X + (int64_t)cand[j0 + j] * d;
                    for (; q0 < d && !(v >= lim); q0 += 8) {
                        float xr[8];
                        if (vec) {
#pragma unroll
                            for (int e = 0; e < 8; e += 4) {
                                float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
                                if (q0 + e < d) f = __ldg(reinterpret_cast<const float4 *>(xj + q0 + e));
                                xr[e] = f.x; xr[e + 1] = f.y; xr[e + 2] = f.z; xr[e + 3] = f.w;
                            }
                        } else {
#pragma unroll
                            for (int e = 0; e < 8; ++e) xr[e] = q0 + e < d ? __ldg(xj + q0 + e) : 0.f;
                        }
#pragma unroll
                        for (int e = 0; e < 8; ++e) sq_acc(xr[e], sh.pick[q0 + e], v);
                    }
                    if (v < lim) rd[j] = v;
                }
                __syncthreads();
            }
        }
        if (warn) status = KMPAR_WARN_FEW_CANDIDATES;
        csync<CS>();           // the seed centers are visible to the whole cluster
        // Lloyd's iteration from the seed centers: dm (in place of D2) the exact distance to a
        // row's center, lb (in place of idx) a lower bound of those to the others
        float *dm = D2, *lb = reinterpret_cast<float *>(idx);
        bool center_lists = a.lists && a.tiles && n >= kBListRows && n >= 8 * (int64_t)k && k * d >= (vec ? kBListWorkVec : kBListWork) &&
                            m >= kBListRetry * fail;
        const bool first_lists = center_lists && n >= 8 * (int64_t)m;
        int it = 0;
        double cost = 0.0;
        for (;; ++it) {
            int chg = 0;
            if (it == 0 && first_lists) {
                for (int j = rank * kBT + tid; j < m; j += CS * kBT) rad[j] = 0u;
                csync<CS>();
                radius_pass(r0, r1, D2, idx, rad);
                csync<CS>();
                const int per_f = (m + CS - 1) / CS;
                list_pass<DP>(sh, dsm, X, min(m, rank * per_f), min(m, (rank + 1) * per_f), d, cand, C, nullptr, 0, k, true,
                              rad, lcnt, lst, tau2);
                csync<CS>();
                lists_rows<BM_ASSIGN, DP>(sh, dsm, X, r0, r1, d, vec, C, nullptr, rad, lcnt, lst, tau2, D2, idx, lab,
                                          perm + r0, &sh.s_fp64);
                const int no = sh.s_cnt;
                if (8 * (int64_t)csum<CS>(no, &sh.s_islot) > 7 * n) center_lists = false;
                __syncthreads();
                dist_pass<DP, BM_ASSIGN>(sh, dsm, X, 0, no, d, C, nullptr, 0, k, nullptr, nullptr, lab, nullptr, &sh.s_fp64,
                                         perm + r0, dm, lb);
            } else if (it > 0 && center_lists) {
                // drifts since the last assignment, the largest two
                for (int j = tid; j < k; j += kBT) sh.drift[j] = drift[j];
                for (int j = rank * kBT + tid; j < k; j += CS * kBT) rad[j] = 0u;
                __syncthreads();
                if (wid == 0) {
                    float m1 = 0.f, m2 = 0.f;
                    int mi = -1;
                    for (int j = lane; j < k; j += 32) {
                        const float v = sh.drift[j];
                        if (v > m1) { m2 = m1; m1 = v; mi = j; }
                        else m2 = fmaxf(m2, v);
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const float u1 = __shfl_xor_sync(0xffffffffu, m1, o), u2 = __shfl_xor_sync(0xffffffffu, m2, o);
                        const int ui = __shfl_xor_sync(0xffffffffu, mi, o);
                        if (u1 > m1 || (u1 == m1 && ui < mi)) { m2 = fmaxf(m1, u2); m1 = u1; mi = ui; }
                        else m2 = fmaxf(m2, u1);
                    }
                    if (lane == 0) { sh.s_m1 = m1; sh.s_m2 = m2; sh.s_mi = mi; }
                }
                csync<CS>();
                bounds_rows<DP>(sh, dsm, X, r0, r1, d, vec, C, lab, dm, lb, rad, perm + r0);
                const int np = sh.s_cnt;
                csync<CS>();
                const int per_f = (k + CS - 1) / CS;
                list_pass<DP>(sh, dsm, X, min(k, rank * per_f), min(k, (rank + 1) * per_f), d, nullptr, C, nullptr, 0, k,
                              false, rad, lcnt, lst, nullptr);
                csync<CS>();
                const int tc = pending_rows<DP>(sh, dsm, X, np, d, vec, C, rad, lcnt, lst, lab, dm, lb, perm + r0, flag,
                                                &sh.s_fp64);
                const int no = sh.s_cnt;
                if (2 * (int64_t)csum<CS>(no, &sh.s_islot) > n) center_lists = false;   // (the dense pass settles most rows)
                __syncthreads();
                dist_pass<DP, BM_ASSIGN>(sh, dsm, X, 0, no, d, C, nullptr, 0, k, nullptr, nullptr, lab, &chg, &sh.s_fp64,
                                         perm + r0, dm, lb, flag);
                chg += bsum_i32(tc, sh.redi);
            } else {
                dist_pass<DP, BM_ASSIGN>(sh, dsm, X, r0, r1, d, C, nullptr, 0, k, nullptr, nullptr, lab,
                                         it > 0 ? &chg : nullptr, &sh.s_fp64, nullptr, dm, lb, it > 0 ? flag : nullptr);
            }
            const double part = sum_rows_of(sh, dm, r0, r1);
            cost = csum<CS>(part, &sh.s_dslot);
            if (it > 0) chg = csum<CS>(chg, &sh.s_islot);
            if (it == 0) res.seed_cost = cost;
            if (it > 0 && chg == 0) break;
            if (it == P.max_iter) break;
            // stable counting sort by label: warp wr of block r owns the contiguous rows
            // [r0 + wr npw, r0 + (wr+1) npw); offsets run over (rank, warp) in order
            const int64_t npw = (r1 - r0 + kBW - 1) / kBW;
            const int64_t w0 = min(r1, r0 + (int64_t)wid * npw), w1 = min(r1, w0 + npw);
            for (int l = tid; l < kBW * kBMaxK; l += kBT) (&sh.hist[0][0])[l] = 0;
            __syncthreads();
            for (int64_t c0 = w0; c0 < w1; c0 += 32) {
                const int64_t pt = c0 + lane;
                const int l = pt < w1 ? lab[pt] : -1;
                const unsigned peers = __match_any_sync(0xffffffffu, l);
                if (l >= 0 && lane == __ffs(peers) - 1) sh.hist[wid][l] += __popc(peers);
                __syncwarp();
            }
            csync<CS>();
            if (rank == 0) {
                // label totals over the cluster, their prefix, then every (rank, warp)
                // count replaced by its running offset (written into the owning block)
                for (int l = tid; l < k; l += kBT) {
                    int tot = 0;
                    for (int q2 = 0; q2 < CS; ++q2) {
                        const int(*hq)[kBMaxK] = CS > 1 ? cg::this_cluster().map_shared_rank(sh.hist, q2) : sh.hist;
                        for (int i = 0; i < kBW; ++i) tot += hq[i][l];
                    }
                    sh.wl_tot[l] = tot;
                }
                __syncthreads();
                if (tid == 0) {
                    int acc = 0;
                    for (int l = 0; l < k; ++l) {
                        sh.base[l] = acc;
                        acc += sh.wl_tot[l];
                    }
                    sh.base[k] = acc;
                }
                __syncthreads();
                for (int l = tid; l < k; l += kBT) {
                    int run2 = sh.base[l];
                    for (int q2 = 0; q2 < CS; ++q2) {
                        int(*hq)[kBMaxK] = CS > 1 ? cg::this_cluster().map_shared_rank(sh.hist, q2) : sh.hist;
                        for (int i = 0; i < kBW; ++i) {
                            const int c = hq[i][l];
                            hq[i][l] = run2;
                            run2 += c;
                        }
                    }
                }
                __syncthreads();
                if (CS > 1)
                    for (int q2 = 1; q2 < CS; ++q2) {
                        int *bq = cg::this_cluster().map_shared_rank(sh.base, q2);
                        for (int l = tid; l <= k; l += kBT) bq[l] = sh.base[l];
                    }
            }
            csync<CS>();
            for (int64_t c0 = w0; c0 < w1; c0 += 32) {
                const int64_t pt = c0 + lane;
                const int l = pt < w1 ? lab[pt] : -1;
                const unsigned peers = __match_any_sync(0xffffffffu, l);
                if (l >= 0) perm[sh.hist[wid][l] + __popc(peers & ((1u << lane) - 1u))] = (int32_t)pt;
                __syncwarp();
                if (l >= 0 && lane == __ffs(peers) - 1) sh.hist[wid][l] += __popc(peers);
                __syncwarp();
            }
            csync<CS>();
            // centroids: member coordinates in ascending point order, compensated FP32;
            // the (center, coordinate) pairs are shared out over the cluster
            for (int64_t pq = (int64_t)rank * kBT + tid; pq < (int64_t)k * d; pq += (int64_t)CS * kBT) {
                const int j = (int)(pq / d), qq = (int)(pq % d);
                const int b0 = sh.base[j], b1 = sh.base[j + 1];
                cold[pq] = C[pq];
                // an empty cluster keeps its center, one with the same members has it already
                if (b1 == b0 || (it > 0 && !flag[j])) continue;
                float s = 0.f, c = 0.f;
                int i = b0;
                for (; i + 8 <= b1; i += 8) {   // eight loads in flight, then the serial sum
                    float v[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] = __ldg(X + (int64_t)perm[i + e] * d + qq);
#pragma unroll
                    for (int e = 0; e < 8; ++e) two_sum_add(s, c, v[e]);
                }
                for (; i < b1; ++i) two_sum_add(s, c, X[(int64_t)perm[i] * d + qq]);
                C[pq] = (float)(((double)s + (double)c) / (double)(b1 - b0));
            }
            csync<CS>();
            // how far each center moved, rounded up (0 only when it is the same)
            for (int j = rank * kBW + wid; j < k; j += CS * kBW) {
                float t2 = 0.f;
                bool diff = false;
                for (int qq = lane; qq < d; qq += 32) {
                    const float t = __fsub_rn(C[(int64_t)j * d + qq], cold[(int64_t)j * d + qq]);
                    t2 = __fmaf_rn(t, t, t2);
                    diff |= t != 0.f;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) t2 += __shfl_xor_sync(0xffffffffu, t2, o);
                diff = __any_sync(0xffffffffu, diff);
                if (lane == 0) {
                    drift[j] = diff ? fmaxf(upper_of(t2, fp32_tie_window(d)), 1e-18f) : 0.f;
                    flag[j] = 0;
                }
            }
            csync<CS>();
        }
        res.iters = it;
        res.final_cost = cost;
        if (a.labels_out)
            for (int64_t pt = r0 + tid; pt < r1; pt += kBT) a.labels_out[P.l_off + pt] = lab[pt];
    }
    if (a.cand_out)
        for (int j = rank * kBT + tid; j < m && j < P.cap_total; j += CS * kBT) a.cand_out[P.cand_off + j] = cand[j];
    if (a.w_out && status != KMPAR_ERR_CAPACITY)
        for (int j = rank * kBT + tid; j < m; j += CS * kBT) a.w_out[P.cand_off + j] = w[j];
    const unsigned long long nr = csum<CS>(sh.s_near, &sh.s_uslot);
    const unsigned long long nf = csum<CS>(sh.s_fp64, &sh.s_uslot);
    const unsigned long long nrc = csum<CS>(sh.s_rnear, &sh.s_uslot);
    if (rank == 0 && tid == 0) {
        res.status = status;
        res.sample_near = nr;
        res.argmin_fp64 = nf;
        res.recluster_near = nrc;
        a.res[pi] = res;
    }
}

}  // namespace
}  // namespace kmp

// ------------------------------------------------------------------ host side
namespace kmp {
namespace {

// l + 10 sqrt(l) + 64 (the round count is a sum of independent draws with mean at
// most l and variance at most l), lowered by KMPAR_ROUND_CAPACITY when set
int batch_round_capacity(double ell) {
    double c = ell + 10.0 * std::sqrt(ell) + 64.0;
    if (c > 2.0e9) c = 2.0e9;
    int cap = (int)std::ceil(c);
    if (const char *v = std::getenv("KMPAR_ROUND_CAPACITY")) {
        char *end = nullptr;
        const unsigned long long x = std::strtoull(v, &end, 10);
        if (*v && end && *end == 0 && x > 0 && x < (unsigned long long)cap) cap = (int)x;
    }
    return cap;
}

kmpar_status batch_fail(kmpar_status s, const std::string &m) {
    kmp::set_thread_error(m);
    return s;
}

// rows per block a problem is cut into: problems larger than this run as a cluster
// (kmpar_batch_set_split; 0: never split)
std::atomic<int64_t> g_rows_per_block{25000};

int padded_dim(int d) { return d <= 32 ? 32 : (d <= 64 ? 64 : 128); }

// blocks of a problem at rpb rows a block; below the set size (full) blocks of little work
// a row stay larger, or their barriers outweigh it (one problem of some 10,000 x 3, k = 5,
// box: 0.96 ms in one block, 1.30 in eight)
int cluster_size(const kmpar_problem &p, int64_t rpb, int64_t full) {
    const int64_t work = (int64_t)p.k * padded_dim(p.d);
    if (rpb < full && work < kBMinWork) rpb = std::max(rpb, std::min(full, (int64_t)kBMinRows * kBMinWork / work));
    int cs = 1;
    while (rpb > 0 && cs < 8 && (p.n + cs - 1) / cs > rpb) cs *= 2;
    return cs;
}

// whether a problem's passes may go by tiles or lists; a launch of which none may takes
// little shared memory (400 problems of 300 - 2,000 x 15 and 42, k = 30 - 60: 4.9 ms with
// the tiles' 92 KB a block, 3.9 without)
bool uses_tiles(const kmpar_problem &p) {
    const double most = std::max((double)p.k, p.ell);   // centers of a pass
    const int dp = padded_dim(p.d);
    return most * dp >= 2.0 * (dp == 128 ? kBTileWork<128> : kBTileWork<64>) ||
           (p.n >= kBListRows && most * p.d >= (p.d % 4 == 0 ? kBListWorkVec : kBListWork));
}

template <int DP, int CS>
cudaError_t launch_cs(const kmp::BArgs &a, int first, int count, cudaStream_t s) {
    if (count == 0) return cudaSuccess;
    const size_t smem = a.tiles ? kmp::batch_smem(DP) : kmp::kBLeanSmem;
    const cudaError_t ea = cudaFuncSetAttribute(kmp::batch_kernel<DP, CS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)kmp::batch_smem(DP));
    if (ea != cudaSuccess) return ea;
    if (CS == 1) {
        kmp::batch_kernel<DP, 1><<<count, kmp::kBT, smem, s>>>(a, first);
    } else {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(count * CS));
        cfg.blockDim = dim3(kmp::kBT);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = CS;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kmp::batch_kernel<DP, CS>, a, first);
        if (e != cudaSuccess) return e;
    }
    kmp::count_launches(1);
    return cudaGetLastError();
}

template <int DP>
cudaError_t launch_class(const kmp::BArgs &a, int cs, int first, int count, cudaStream_t s) {
    switch (cs) {
        case 1: return launch_cs<DP, 1>(a, first, count, s);
        case 2: return launch_cs<DP, 2>(a, first, count, s);
        case 4: return launch_cs<DP, 4>(a, first, count, s);
        case 8: return launch_cs<DP, 8>(a, first, count, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace
}  // namespace kmp

extern "C" {

kmpar_status kmpar_batch_set_split(int32_t rows_per_block) {
    if (rows_per_block < 0) return kmp::batch_fail(KMPAR_ERR_ARG, "rows_per_block < 0");
    kmp::g_rows_per_block.store(rows_per_block, std::memory_order_relaxed);
    return KMPAR_OK;
}

int64_t kmpar_batch_cand_capacity(double ell, int32_t rounds) {
    if (!(ell > 0.0) || rounds < 0) return 0;
    return 1 + (int64_t)rounds * kmp::batch_round_capacity(ell);
}

kmpar_status kmpar_batch_run(const float *X, const kmpar_problem *problems, int32_t count, float *centers_out,
                             int32_t *labels_out, int32_t *cand_out, int64_t *w_out, kmpar_problem_result *results,
                             void *stream) {
    using namespace kmp;
    if (count < 0 || (count > 0 && (!X || !problems || !centers_out || !results)))
        return batch_fail(KMPAR_ERR_ARG, "NULL pointer or negative count");
    if (count == 0) return KMPAR_OK;
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<BProb> hp((size_t)count);
    std::vector<double> work((size_t)count);
    int64_t p_tot = 0, m_tot = 0, f_tot = 0, k_tot = 0, s_tot = 0;
    for (int i = 0; i < count; ++i) {
        const kmpar_problem &q = problems[i];
        if (q.n < 1 || q.n >= (int64_t)INT32_MAX || q.d < 1 || q.d > 128 || q.k < 1 || q.k > kBMaxK ||
            !(q.ell > 0.0) || !std::isfinite(q.ell) || q.rounds < 0 || q.rounds > kBMaxRounds || q.max_iter < 0 ||
            q.x_offset < 0 || q.c_offset < 0 || q.l_offset < 0 || q.cand_offset < 0)
            return batch_fail(KMPAR_ERR_ARG, "problem " + std::to_string(i) + ": argument out of range");
        const int cap = batch_round_capacity(q.ell);
        if (cap > kBMaxCap)
            return batch_fail(KMPAR_ERR_UNSUPPORTED,
                              "problem " + std::to_string(i) + ": l + 10 sqrt(l) + 64 exceeds 4096 per round");
        BProb &b = hp[(size_t)i];
        b.x_off = q.x_offset; b.n = q.n; b.d = q.d; b.k = q.k; b.ell = q.ell; b.rounds = q.rounds;
        b.max_iter = q.max_iter; b.seed = q.seed; b.c_off = q.c_offset; b.l_off = q.l_offset;
        b.cand_off = q.cand_offset;
        b.cap_round = cap;
        b.cap_total = 1 + q.rounds * cap;
        b.p_off = p_tot;
        b.m_off = m_tot;
        b.f_off = f_tot;
        b.k_off = k_tot;
        b.s_off = s_tot;
        p_tot += q.n;
        m_tot += b.cap_total;
        f_tot += std::max(b.cap_total, q.k);
        k_tot += q.k;
        s_tot += (int64_t)q.k * q.d;
        // distance evaluations of the rounds and of Lloyd, times the padded dimension
        work[(size_t)i] = (double)q.n * padded_dim(q.d) * (1.0 + q.rounds * q.ell + (double)(q.max_iter + 1) * q.k);
    }
    // a call whose blocks would leave SMs idle cuts its problems finer, down to blocks of
    // kBMinRows rows (64 problems of 500 - 3,000 rows, d = 15 and 42: 3.8 ms a block each,
    // 1.8 ms at 780 rows a block)
    const int64_t full = g_rows_per_block.load(std::memory_order_relaxed);
    int64_t rpb = full;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        sms = 0;
    while (rpb >= 2 * kBMinRows) {
        int64_t blocks = 0;
        for (int i = 0; i < count && blocks < sms; ++i) blocks += cluster_size(problems[i], rpb, full);
        if (blocks >= sms) break;
        rpb /= 2;
    }
    // one launch per (dimension class, cluster size), largest problems first in each
    std::vector<int32_t> order;
    order.reserve((size_t)count);
    struct Cls { int dp, cs, first, count; };
    std::vector<Cls> classes;
    for (int c = 0; c < 3; ++c) {
        const int lo = c == 0 ? 1 : (c == 1 ? 33 : 65), hi = c == 0 ? 32 : (c == 1 ? 64 : 128);
        for (int cs = 8; cs >= 1; cs /= 2) {
            std::vector<int32_t> ids;
            for (int i = 0; i < count; ++i)
                if (problems[i].d >= lo && problems[i].d <= hi && cluster_size(problems[i], rpb, full) == cs) ids.push_back(i);
            if (ids.empty()) continue;
            std::stable_sort(ids.begin(), ids.end(), [&](int32_t x, int32_t y) { return work[x] > work[y]; });
            classes.push_back({c == 0 ? 32 : (c == 1 ? 64 : 128), cs, (int)order.size(), (int)ids.size()});
            order.insert(order.end(), ids.begin(), ids.end());
        }
    }
    // one device block holds the table, the order, the results and the work space
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t o_probs = 0;
    const size_t o_order = o_probs + up(sizeof(BProb) * (size_t)count);
    const size_t o_res = o_order + up(sizeof(int32_t) * (size_t)count);
    const size_t o_d2 = o_res + up(sizeof(BRes) * (size_t)count);
    const size_t o_idx = o_d2 + up(sizeof(float) * (size_t)p_tot);
    const size_t o_lab = o_idx + up(sizeof(int32_t) * (size_t)p_tot);
    const size_t o_perm = o_lab + up(sizeof(int32_t) * (size_t)p_tot);
    const size_t o_cand = o_perm + up(sizeof(int32_t) * (size_t)p_tot);
    const size_t o_w = o_cand + up(sizeof(int32_t) * (size_t)m_tot);
    const size_t o_rd2 = o_w + up(sizeof(int32_t) * (size_t)m_tot);
    const size_t o_drift = o_rd2 + up(sizeof(float) * (size_t)m_tot);
    const size_t o_flag = o_drift + up(sizeof(float) * (size_t)k_tot);
    const size_t o_cold = o_flag + up(sizeof(int32_t) * (size_t)k_tot);
    const size_t o_rad = o_cold + up(sizeof(float) * (size_t)s_tot);   // from here on: the lists
    const size_t o_lcnt = o_rad + up(sizeof(int32_t) * (size_t)f_tot);
    const size_t o_lst = o_lcnt + up(sizeof(int32_t) * (size_t)f_tot);
    const size_t o_tau = o_lst + up(sizeof(int32_t) * (size_t)f_tot * kBList);
    const size_t total = o_tau + up(sizeof(float) * (size_t)f_tot);
    unsigned char *ws = nullptr;
    cudaError_t e = scratch_alloc(reinterpret_cast<void **>(&ws), total, s);
    const bool lists = e == cudaSuccess;
    if (e == cudaErrorMemoryAllocation) {   // without the lists every pass is dense
        (void)cudaGetLastError();
        e = scratch_alloc(reinterpret_cast<void **>(&ws), o_rad, s);
    }
    if (e != cudaSuccess)
        return batch_fail(e == cudaErrorMemoryAllocation ? KMPAR_ERR_OOM : KMPAR_ERR_CUDA,
                          std::string("batch work space: ") + cudaGetErrorString(e));
    std::vector<BRes> hres((size_t)count);
    const int nside = (int)classes.size() - 1;
    std::vector<cudaStream_t> side((size_t)std::max(0, nside), nullptr);
    std::vector<cudaEvent_t> ev_join((size_t)std::max(0, nside), nullptr);
    cudaEvent_t ev_fork = nullptr;
    BArgs a{};
    a.X = X;
    a.probs = reinterpret_cast<const BProb *>(ws + o_probs);
    a.order = reinterpret_cast<const int32_t *>(ws + o_order);
    a.centers = centers_out;
    a.labels_out = labels_out;
    a.cand_out = cand_out;
    a.w_out = reinterpret_cast<long long *>(w_out);
    a.res = reinterpret_cast<BRes *>(ws + o_res);
    a.D2 = reinterpret_cast<float *>(ws + o_d2);
    a.idx = reinterpret_cast<int32_t *>(ws + o_idx);
    a.lab = reinterpret_cast<int32_t *>(ws + o_lab);
    a.perm = reinterpret_cast<int32_t *>(ws + o_perm);
    a.cand = reinterpret_cast<int32_t *>(ws + o_cand);
    a.w = reinterpret_cast<int32_t *>(ws + o_w);
    a.rD2 = reinterpret_cast<float *>(ws + o_rd2);
    a.lists = lists;
    a.rad = reinterpret_cast<unsigned int *>(ws + o_rad);
    a.lcnt = reinterpret_cast<int32_t *>(ws + o_lcnt);
    a.lst = reinterpret_cast<int32_t *>(ws + o_lst);
    a.tau2 = reinterpret_cast<float *>(ws + o_tau);
    a.drift = reinterpret_cast<float *>(ws + o_drift);
    a.flag = reinterpret_cast<int32_t *>(ws + o_flag);
    a.cold = reinterpret_cast<float *>(ws + o_cold);
    e = cudaMemcpyAsync(ws + o_probs, hp.data(), sizeof(BProb) * (size_t)count, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(ws + o_order, order.data(), sizeof(int32_t) * (size_t)count, cudaMemcpyHostToDevice, s);
    // the classes run concurrently: the caller's stream and side streams forked from
    // it and joined back (also valid inside a stream capture)
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev_fork, cudaEventDisableTiming);
    for (int i = 0; i < nside && e == cudaSuccess; ++i) {
        e = cudaStreamCreateWithFlags(&side[(size_t)i], cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev_join[(size_t)i], cudaEventDisableTiming);
    }
    if (e == cudaSuccess) e = cudaEventRecord(ev_fork, s);
    for (int i = 0; i < nside && e == cudaSuccess; ++i) e = cudaStreamWaitEvent(side[(size_t)i], ev_fork, 0);
    for (size_t c = 0; c < classes.size() && e == cudaSuccess; ++c) {
        const Cls &q = classes[c];
        a.tiles = false;
        for (int i = 0; i < q.count; ++i) a.tiles |= uses_tiles(problems[order[(size_t)(q.first + i)]]);
        cudaStream_t cs = c == 0 ? s : side[c - 1];
        if (q.dp == 32) e = launch_class<32>(a, q.cs, q.first, q.count, cs);
        else if (q.dp == 64) e = launch_class<64>(a, q.cs, q.first, q.count, cs);
        else e = launch_class<128>(a, q.cs, q.first, q.count, cs);
    }
    for (int i = 0; i < nside && e == cudaSuccess; ++i) {
        e = cudaEventRecord(ev_join[(size_t)i], side[(size_t)i]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ev_join[(size_t)i], 0);
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(hres.data(), ws + o_res, sizeof(BRes) * (size_t)count, cudaMemcpyDeviceToHost, s);
    const cudaError_t ef = cudaFreeAsync(ws, s);
    if (e == cudaSuccess) e = ef;
    const cudaError_t es = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = es;
    for (int i = 0; i < nside; ++i) {
        if (side[(size_t)i]) cudaStreamDestroy(side[(size_t)i]);
        if (ev_join[(size_t)i]) cudaEventDestroy(ev_join[(size_t)i]);
    }
    if (ev_fork) cudaEventDestroy(ev_fork);
    if (e != cudaSuccess) return batch_fail(KMPAR_ERR_CUDA, std::string("batch kernels: ") + cudaGetErrorString(e));
    kmpar_status worst = KMPAR_OK;
    for (int i = 0; i < count; ++i) {
        const BRes &r = hres[(size_t)i];
        kmpar_problem_result &o = results[i];
        o.m = r.m;
        o.seed_cost = r.seed_cost;
        o.final_cost = r.final_cost;
        o.iters = r.iters;
        o.status = r.status;
        o.sample_near = (int64_t)r.sample_near;
        o.argmin_fp64 = (int64_t)r.argmin_fp64;
        o.recluster_near = (int64_t)r.recluster_near;
        if (r.status == KMPAR_ERR_CAPACITY) worst = KMPAR_ERR_CAPACITY;
        else if (r.status == KMPAR_WARN_FEW_CANDIDATES && worst == KMPAR_OK) worst = KMPAR_WARN_FEW_CANDIDATES;
    }
    if (worst == KMPAR_ERR_CAPACITY) kmp::set_thread_error("a problem's round drew more points than its capacity");
    return worst;
}

}  // extern "C"
