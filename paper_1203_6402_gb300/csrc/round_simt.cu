// round_simt.cu -- the per-round data-parallel pass of k-means|| (Alg. 2 steps
// 1-2, 4-5 of Bahmani et al., Sec. 3.3) and the nearest-center scan that Lloyd's
// iteration and phi_X(C) (Sec. 3.1) reuse, on CUDA cores in exact FP32.
//
// Kernels:
//   pick_first_kernel   Alg. 2 step 1: i0 = floor(u n), row gathered as candidate 0
//   first_dist_kernel   Alg. 2 step 2: D^2 to the first center, per-block FP64 sums
//   nearest_tile_kernel d^2(x, C') for the batch C' (or all k centers), top-2 per
//                       row, FP64 re-decision of near ties, D^2/idx/labels update,
//                       per-block FP64 partial of phi
//   sample_kernel       Alg. 2 step 4: p = min(1, l D^2/phi), Philox draw,
//                       warp-aggregated atomic append
//   sort_batch_kernel   ascending order of the round's draws (one CTA, bitonic)
//   gather_kernel       candidate rows copied out of X
//   sum_f64_kernel      fixed-order FP64 sum of per-block partials
#include <float.h>

#include <algorithm>

#include "kmpar_internal.cuh"

namespace kmp {

// How the resident refine covers a pass of cap_rows centers: `parts` launches of
// `rows` centers each (`hold` rows of shared memory, `warps` warps per CTA).
// parts = 0: the per-row kernel (refine_kernel) is used instead.
struct ResidentPlan {
    int parts, rows, hold, warps;
};
ResidentPlan resident_plan(int cap_rows, int d);

enum { MODE_ROUND = 1, MODE_ASSIGN = 2 };

struct NearestParams {
    const float *X;
    int64_t n;
    int d;
    const float *C;        // center rows, stride d
    int c_begin, c_cnt;    // ASSIGN: static range; ROUND: taken from st
    const DevState *st;
    float *D2;             // ROUND: in/out
    int32_t *idx;          // ROUND: in/out
    int32_t *labels;       // ASSIGN: out (nullable)
    const int32_t *prev;   // ASSIGN: previous labels (nullable)
    int *changed;          // ASSIGN: +number of labels != prev (nullable)
    double *partials;      // per-block FP64 sum of the stored distances (nullable)
    unsigned long long *fp64_cnt, *wide_cnt;
};

// lexicographic (value, index) improvement
__device__ __forceinline__ void take_if_better(double v, int j, double &best, int &bj) {
    if (v < best || (v == best && j < bj)) { best = v; bj = j; }
}

// The decision for row pt once its lexicographic (value, center) best and runner-up
// (b1, i1), (b2, i2) are known (INT_MAX: none): writes the row's outputs, returns the
// stored distance; chg: a label changed.
template <int MODE>
__device__ __forceinline__ float nearest_decide(const NearestParams &p, int64_t pt, float b1, int i1, float b2, int i2,
                                                int &chg) {
    const int d = p.d;
    const float *xrow = p.X + pt * (int64_t)d;
    const float W = fp32_tie_window(d);
    if (i1 == INT_MAX) i1 = -1;
    if (i2 == INT_MAX) i2 = -1;
    float stored = 0.f;
    if constexpr (MODE == MODE_ASSIGN) {
        // a row whose distances are all NaN/inf keeps label 0 (labels stay in range)
        int lab = i1 >= 0 ? i1 : 0;
        stored = b1;
        if (i2 >= 0 && b2 <= b1 + W * b1) {
            // the FP32 order of the two best may differ from the FP64 order
            double best = dist2_fp64(xrow, p.C + (int64_t)i1 * d, d);
            int bj = i1;
            take_if_better(dist2_fp64(xrow, p.C + (int64_t)i2 * d, d), i2, best, bj);
            if (bj == i2) { lab = i2; stored = b2; }
            atomicAdd(p.fp64_cnt, 1ull);
        }
        if (p.labels) p.labels[pt] = lab;
        if (p.prev) chg = (p.prev[pt] != lab);
    } else {
        const float old = p.D2[pt];
        const int oi = p.idx[pt];
        const float m32 = fminf(old, b1);
        const float lim = m32 + W * m32;
        const bool in_old = (oi >= 0) && old <= lim;
        const bool in1 = i1 >= 0 && b1 <= lim;
        const bool in2 = i2 >= 0 && b2 <= lim;
        int win = -1;
        float wv = old;
        if ((int)in_old + (int)in1 + (int)in2 >= 2) {
            double best = DBL_MAX;
            int bj = INT_MAX;
            if (in_old) take_if_better(dist2_fp64(xrow, p.C + (int64_t)oi * d, d), oi, best, bj);
            if (in1) take_if_better(dist2_fp64(xrow, p.C + (int64_t)i1 * d, d), i1, best, bj);
            if (in2) take_if_better(dist2_fp64(xrow, p.C + (int64_t)i2 * d, d), i2, best, bj);
            atomicAdd(p.fp64_cnt, 1ull);
            if (in1 && in2) atomicAdd(p.wide_cnt, 1ull);
            if (bj == i1) { win = i1; wv = b1; }
            else if (bj == i2) { win = i2; wv = b2; }
        } else if (i1 >= 0 && b1 < old) {
            win = i1; wv = b1;
        }
        if (win >= 0) {
            p.D2[pt] = wv;
            p.idx[pt] = win;
            stored = wv;
        } else {
            stored = old;
        }
    }
    return stored;
}

// (value, index) order with the lower index first on equal values
__device__ __forceinline__ bool lex_lt(float v, int i, float w, int j) { return v < w || (v == w && i < j); }

// top-2 of the union of two top-2 lists
__device__ __forceinline__ void top2_merge(float &b1, int &i1, float &b2, int &i2, float c1, int j1, float c2, int j2) {
    if (lex_lt(c1, j1, b1, i1)) {
        // c1 is the new best; second = best of (b1, c2)
        if (lex_lt(b1, i1, c2, j2)) { b2 = b1; i2 = i1; } else { b2 = c2; i2 = j2; }
        b1 = c1; i1 = j1;
    } else if (lex_lt(c1, j1, b2, i2)) {
        b2 = c1; i2 = j1;
    }
}

// The scan for d <= 32, and for few centers up to d = 128: a row a thread, its coordinates in registers, 64 centers at a
// time in shared memory.  With so few coordinates the tiled scan's handling of its tile's
// results outweighs the sums (3e6 x 3 against 100: 0.36 ms, tiled 0.8; 1e6 x 32 against
// 100: 0.59, 0.68; at 50 coordinates 200,000 rows against 300 take 0.62, tiled 0.52), as
// does a tile's padding to 32 or 64 centers where there are few (see few_centers).
constexpr int kNearThreads = 128;

template <int DP, int MODE>
__global__ void __launch_bounds__(kNearThreads) nearest_kernel(NearestParams p) {
    constexpr int TC = DP <= 64 ? 64 : 32;
    __shared__ __align__(16) float tile[TC * DP];
    __shared__ double red[32];
    __shared__ int redi[32];

    const int tid = threadIdx.x;
    const int64_t pt = (int64_t)blockIdx.x * kNearThreads + tid;
    const bool valid = pt < p.n;
    const int d = p.d;
    const float *xrow = p.X + (valid ? pt : 0) * (int64_t)d;

    float xr[DP];
#pragma unroll
    for (int q = 0; q < DP; ++q) xr[q] = (valid && q < d) ? __ldg(xrow + q) : 0.f;

    int begin, cnt;
    if constexpr (MODE == MODE_ASSIGN) {
        begin = p.c_begin; cnt = p.c_cnt;
    } else {
        begin = p.st->batch_begin; cnt = p.st->batch_cnt;
    }

    float b1 = FLT_MAX, b2 = FLT_MAX;
    int i1 = INT_MAX, i2 = INT_MAX;
    for (int t0 = 0; t0 < cnt; t0 += TC) {
        const int nt = min(TC, cnt - t0);
        __syncthreads();
        for (int e = tid; e < TC * DP; e += kNearThreads) {
            const int r = e / DP, q = e - r * DP;
            tile[e] = (r < nt && q < d) ? __ldg(p.C + (int64_t)(begin + t0 + r) * d + q) : 0.f;
        }
        __syncthreads();
        if (valid) {
            for (int r = 0; r < nt; ++r) {
                float acc = 0.f;
                const float4 *c4 = reinterpret_cast<const float4 *>(tile + r * DP);
#pragma unroll
                for (int q4 = 0; q4 < DP / 4; ++q4) {
                    const float4 c = c4[q4];
                    float t;
                    t = __fsub_rn(xr[4 * q4 + 0], c.x); acc = __fmaf_rn(t, t, acc);
                    t = __fsub_rn(xr[4 * q4 + 1], c.y); acc = __fmaf_rn(t, t, acc);
                    t = __fsub_rn(xr[4 * q4 + 2], c.z); acc = __fmaf_rn(t, t, acc);
                    t = __fsub_rn(xr[4 * q4 + 3], c.w); acc = __fmaf_rn(t, t, acc);
                }
                const int j = begin + t0 + r;
                if (acc < b2) {
                    if (acc < b1) { b2 = b1; i2 = i1; b1 = acc; i1 = j; }
                    else { b2 = acc; i2 = j; }
                }
            }
        }
    }

    float stored = 0.f;
    int chg = 0;
    if (valid) stored = nearest_decide<MODE>(p, pt, b1, i1, b2, i2, chg);
    const double s = block_sum_f64(valid ? (double)stored : 0.0, red);
    if (tid == 0 && p.partials) p.partials[blockIdx.x] = s;
    if constexpr (MODE == MODE_ASSIGN) {
        if (p.changed) {
            int c = warp_sum_i32(chg);
            __syncthreads();
            if ((tid & 31) == 0) redi[tid >> 5] = c;
            __syncthreads();
            if (tid == 0) {
                int tot = 0;
                for (int i = 0; i < kNearThreads / 32; ++i) tot += redi[i];
                if (tot) atomicAdd(p.changed, tot);
            }
        }
    }
}

// The exact FP32 nearest-center scan, tiled like a GEMM.  A block of 8 x RT threads takes
// BM rows and walks the centers 8 TN at a time; a thread holds 4 x TN distances of its
// tile in registers and adds coordinate after coordinate (t = x - c, acc = fma(t, t, acc),
// ascending: the chain of dist2_fp32), so the FP32 pipe always has 4 TN independent
// chains a thread and each shared-memory read feeds several.  Rows (resident while
// d <= kTileK) and centers lie in shared memory coordinate-major with 16 bytes of padding
// a coordinate, brought in by 4-byte asynchronous copies (the transposition costs no
// registers); the next tile of centers is copied while one is summed.  A thread meets its
// centers in ascending order; the 8 threads of a row merge their top two.  (The FP32 pipe
// gives packed pairs no more lanes: in a loop of this shape 8 x 4 scalar chains ran at 31 T
// operations/s of 40.3, packed ones at 30.)  Bound by FP32 issue: the cost of 1e6 x 42
// against 500 centers 2.23 -> 1.96 ms, a fit of 200k x 50, k = 300 11.9 -> 8.9 ms, against a
// row per thread with its coordinates in registers.
constexpr int kTileK = 96;    // coordinates resident: two blocks an SM
constexpr int kTileChunk = 64;   // coordinates of a step when the rows are not resident

__device__ __forceinline__ void cp_async4_zfill(uint32_t dst, const float *src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(valid ? 4 : 0) : "memory");
}

// coordinates q0 .. q0 + kn - 1 of rows first .. first + B - 1 (rows at or past `limit` as
// zeros) to dst[q * stride + r], consecutive threads along a row and then the next
template <int THREADS>
__device__ __forceinline__ void tile_copy(float *dst, int stride, int B, const float *src, int64_t first, int64_t limit,
                                          int d, int q0, int kn) {
    int r = threadIdx.x / kn, q = threadIdx.x % kn;
    const int dr = THREADS / kn, dq = THREADS % kn;
    uint32_t to = static_cast<uint32_t>(__cvta_generic_to_shared(dst + q * stride + r));
    const uint32_t step = 4u * (dq * stride + dr), wrap = 4u * (kn * stride - 1);
    const float *from = src + (first + r) * d + q0 + q;
    const int64_t fs = (int64_t)dr * d + dq, fw = d - kn;
    const int lim = (int)min((int64_t)B, limit - first);
#pragma unroll 4
    while (r < B) {
        const bool ok = r < lim;
        cp_async4_zfill(to, ok ? from : src, ok);
        r += dr;
        q += dq;
        from += fs;
        to += step;
        if (q >= kn) { q -= kn; ++r; from += fw; to -= wrap; }
    }
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int MODE, int BM, int TN>
__global__ void __launch_bounds__(2 * BM, BM == 128 ? 2 : 8) nearest_tile_kernel(NearestParams p, int kc) {
    constexpr int TM = 4, threads = 2 * BM, BN = 8 * TN;
    constexpr int XS = BM + 4, CS = BN + 4;   // floats per coordinate
    extern __shared__ __align__(16) float tsm[];
    __shared__ double red[32];
    __shared__ int redi[32];
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3, d = p.d;
    const bool resident = d <= kc;
    float *xb = tsm, *cb = tsm + (resident ? 1 : 2) * kc * XS;   // rows (two buffers in steps), centers (two)
    const int64_t base = (int64_t)blockIdx.x * BM;
    int begin, cnt;
    if constexpr (MODE == MODE_ASSIGN) {
        begin = p.c_begin; cnt = p.c_cnt;
    } else {
        begin = p.st->batch_begin; cnt = p.st->batch_cnt;
    }
    const int chunks = (d + kc - 1) / kc, steps = ((cnt + BN - 1) / BN) * chunks;
    auto issue = [&](int s) {   // step s: tile s / chunks of the centers, chunk s % chunks of the coordinates
        const int t = s / chunks, q0 = (s - t * chunks) * kc, kn = min(kc, d - q0);
        if (!resident || s == 0)
            tile_copy<threads>(xb + (resident ? 0 : (s & 1) * kc * XS), XS, BM, p.X, base, p.n, d, q0, kn);
        tile_copy<threads>(cb + (s & 1) * kc * CS, CS, BN, p.C, begin + (int64_t)t * BN, begin + (int64_t)cnt, d, q0, kn);
    };
    float b1[TM], b2[TM];
    int i1[TM], i2[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) { b1[i] = b2[i] = FLT_MAX; i1[i] = i2[i] = INT_MAX; }
    float acc[TM][TN];
    if (steps > 0) issue(0);
    cp_async_commit();
    for (int s = 0; s < steps; ++s) {
        cp_async_wait<0>();
        __syncthreads();   // step s is in, and every thread is done with step s - 1
        if (s + 1 < steps) issue(s + 1);
        cp_async_commit();
        const int t = s / chunks, ch = s - t * chunks, kn = min(kc, d - ch * kc);
        if (ch == 0) {
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
        }
        const float *xq = xb + (resident ? 0 : (s & 1) * kc * XS) + ty * 4, *cq = cb + (s & 1) * kc * CS + tx * 4;
#pragma unroll 2
        for (int q = 0; q < kn; ++q, xq += XS, cq += CS) {
            float x[TM], c[TN];
            const float4 xv = *reinterpret_cast<const float4 *>(xq);
            x[0] = xv.x; x[1] = xv.y; x[2] = xv.z; x[3] = xv.w;
#pragma unroll
            for (int j = 0; j < TN; j += 4) {   // columns 4 tx .. + 3 of each 32
                const float4 v = *reinterpret_cast<const float4 *>(cq + 8 * j);
                c[j] = v.x; c[j + 1] = v.y; c[j + 2] = v.z; c[j + 3] = v.w;
            }
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    const float u = __fsub_rn(x[i], c[j]);
                    acc[i][j] = __fmaf_rn(u, u, acc[i][j]);
                }
        }
        if (ch + 1 < chunks) continue;
        // the thread's centers of this tile, ascending: a row whose smallest value is not
        // below its runner-up needs no look at the others (after the first tiles, most)
        const int c0 = t * BN + tx * 4;   // column j: c0 + (j / 4) 32 + j % 4
        if (t * BN + BN > cnt) {   // pad columns hold the distance to 0
#pragma unroll
            for (int j = 0; j < TN; ++j)
                if (c0 + (j >> 2) * 32 + (j & 3) >= cnt) {
#pragma unroll
                    for (int i = 0; i < TM; ++i) acc[i][j] = FLT_MAX;
                }
        }
#pragma unroll
        for (int r = 0; r < TM; ++r) {
            float m = acc[r][0];
#pragma unroll
            for (int j = 1; j < TN; ++j) m = fminf(m, acc[r][j]);
            if (m < b2[r]) {
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    const float a = acc[r][j];
                    if (a < b2[r]) {
                        const int c = begin + c0 + (j >> 2) * 32 + (j & 3);
                        if (a < b1[r]) { b2[r] = b1[r]; i2[r] = i1[r]; b1[r] = a; i1[r] = c; }
                        else { b2[r] = a; i2[r] = c; }
                    }
                }
            }
        }
    }
    auto number = [&](int r) -> int64_t {
        const int64_t at = base + r;
        return at < p.n ? at : -1;
    };
    // merge the 8 threads of a row, then thread tx = r decides the thread row's row r
    float m1 = FLT_MAX, m2 = FLT_MAX;
    int n1 = INT_MAX, n2 = INT_MAX;
#pragma unroll
    for (int r = 0; r < TM; ++r) {
        float v1 = b1[r], v2 = b2[r];
        int j1 = i1[r], j2 = i2[r];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            const float u1 = __shfl_xor_sync(0xffffffffu, v1, o), u2 = __shfl_xor_sync(0xffffffffu, v2, o);
            const int k1 = __shfl_xor_sync(0xffffffffu, j1, o), k2 = __shfl_xor_sync(0xffffffffu, j2, o);
            top2_merge(v1, j1, v2, j2, u1, k1, u2, k2);
        }
        if (tx == r) { m1 = v1; m2 = v2; n1 = j1; n2 = j2; }
    }
    const int64_t pt = tx < TM ? number(ty * 4 + tx) : -1;
    float stored = 0.f;
    int chg = 0;
    if (pt >= 0) stored = nearest_decide<MODE>(p, pt, m1, n1, m2, n2, chg);
    const double s = block_sum_f64(pt >= 0 ? (double)stored : 0.0, red);
    if (tid == 0 && p.partials) p.partials[blockIdx.x] = s;
    if constexpr (MODE == MODE_ASSIGN) {
        if (p.changed) {
            int c = warp_sum_i32(chg);
            __syncthreads();
            if ((tid & 31) == 0) redi[tid >> 5] = c;
            __syncthreads();
            if (tid == 0) {
                int tot = 0;
                for (int i = 0; i < threads / 32; ++i) tot += redi[i];
                if (tot) atomicAdd(p.changed, tot);
            }
        }
    }
}

// rows per block of the scan: small sets are cut finer, so that more SMs take part (40,000
// rows in blocks of 128 are two a SM; from there on the larger tile's reuse counts for more).
// Up to 32 coordinates a row per thread holds them in registers and needs no tile of rows.
static int scan_rows(int64_t n, int d) { return d > 32 && n <= 40000 ? 32 : 128; }

int assign_num_partials(int64_t n, int d) { return (int)((n + scan_rows(n, d) - 1) / scan_rows(n, d)); }

// dynamic shared memory of a tile kernel at d coordinates: rows (two buffers in steps) and
// two buffers of centers
constexpr size_t tile_smem(int d, int BM, int BN) {
    return sizeof(float) * (d <= kTileK ? d * (BM + 4 + 2 * (BN + 4)) : kTileChunk * 2 * (BM + 4 + BN + 4));
}

template <int MODE, int BM, int TN>
static cudaError_t launch_tiles(const NearestParams &p, int grid, cudaStream_t s) {
    constexpr size_t at_k = tile_smem(kTileK, BM, 8 * TN), steps = tile_smem(kTileK + 1, BM, 8 * TN);
    constexpr size_t most = at_k > steps ? at_k : steps;
    // the limit belongs to the process: always the kernel's largest size, whatever this
    // call takes, so that no call lowers it under another one
    if (most > 40 * 1024) {   // (the static shared memory counts too)
        const cudaError_t e = cudaFuncSetAttribute(nearest_tile_kernel<MODE, BM, TN>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
        if (e != cudaSuccess) return e;
    }
    nearest_tile_kernel<MODE, BM, TN><<<grid, 2 * BM, tile_smem(p.d, BM, 8 * TN), s>>>(p, p.d <= kTileK ? p.d : kTileChunk);
    return cudaGetLastError();
}

// Few centers against many rows (more than the 40,000 cut into small blocks), by the number of
// centers (an assignment's) or the capacity for them (a round's; that of l = 12 is 110).
// 2e6 x 33 against 1 center: 0.30 ms a row a thread, 0.41 tiled; x 97 0.52, 0.78;
// against 30: 1.0 and 0.7.
static bool few_centers(int mode, int64_t n, int d, int cnt_hint) {
    return d <= 128 && scan_rows(n, d) == 128 && cnt_hint <= (mode == MODE_ASSIGN ? 8 : 110);
}

template <int MODE>
static cudaError_t launch_nearest_mode(const NearestParams &p, int cnt_hint, cudaStream_t s) {
    const int grid = assign_num_partials(p.n, p.d);
    const bool small = scan_rows(p.n, p.d) == 32, narrow = cnt_hint <= 32;
    count_launches(1);
    if (p.d <= 4) nearest_kernel<4, MODE><<<grid, kNearThreads, 0, s>>>(p);
    else if (p.d <= 8) nearest_kernel<8, MODE><<<grid, kNearThreads, 0, s>>>(p);
    else if (p.d <= 16) nearest_kernel<16, MODE><<<grid, kNearThreads, 0, s>>>(p);
    else if (p.d <= 32) nearest_kernel<32, MODE><<<grid, kNearThreads, 0, s>>>(p);
    else if (few_centers(MODE, p.n, p.d, cnt_hint)) {
        if (p.d <= 48) nearest_kernel<48, MODE><<<grid, kNearThreads, 0, s>>>(p);
        else if (p.d <= 64) nearest_kernel<64, MODE><<<grid, kNearThreads, 0, s>>>(p);
        else if (p.d <= 96) nearest_kernel<96, MODE><<<grid, kNearThreads, 0, s>>>(p);
        else nearest_kernel<128, MODE><<<grid, kNearThreads, 0, s>>>(p);
    } else if (small) return narrow ? launch_tiles<MODE, 32, 4>(p, grid, s) : launch_tiles<MODE, 32, 8>(p, grid, s);
    else return narrow ? launch_tiles<MODE, 128, 4>(p, grid, s) : launch_tiles<MODE, 128, 8>(p, grid, s);
    return cudaGetLastError();
}

// Alg. 2 step 2: D^2 to the first center, idx = 0.  128 rows a block, up to kFirstPiece
// coordinates at a time through shared memory, coordinate-major at an odd stride: all of a
// piece is on its way at once (asynchronous copies along the rows), and a lane then walks
// its row.  Bound by reading X; with loads of 32 lanes a row, eight rows in flight, most lanes
// idle in a row of 3 to 24 coordinates: 9e6 x 8 525 us, so 126; 4.8e6 x 42 432, 201; 2e6 x
// 128 500, 249.
constexpr int kFirstRows = 128, kFirstPiece = 64, kFirstStride = kFirstRows + 1;

__global__ void __launch_bounds__(kFirstRows) first_dist_kernel(const float *__restrict__ X, int64_t n, int d,
                                                               const float *__restrict__ C, float *__restrict__ D2,
                                                               int32_t *__restrict__ idx, double *partials) {
    extern __shared__ __align__(16) float fsm[];   // min(d, kFirstPiece) x kFirstStride
    __shared__ float cq[kFirstPiece];
    __shared__ double red[32];
    const int tid = threadIdx.x;
    const int64_t base = (int64_t)blockIdx.x * kFirstRows, R = base + tid;
    float v = 0.f;
    for (int q0 = 0; q0 < d; q0 += kFirstPiece) {
        const int kn = min(kFirstPiece, d - q0);
        __syncthreads();   // the walkers of the last piece are done
        tile_copy<kFirstRows>(fsm, kFirstStride, kFirstRows, X, base, n, d, q0, kn);
        cp_async_commit();
        if (tid < kn) cq[tid] = C[q0 + tid];
        cp_async_wait<0>();
        __syncthreads();
#pragma unroll 8
        for (int q = 0; q < kn; ++q) {
            const float t = __fsub_rn(fsm[q * kFirstStride + tid], cq[q]);
            v = __fmaf_rn(t, t, v);
        }
    }
    // (a distance that is not below the largest float counts as infinite)
    const float stored = v < FLT_MAX ? v : __int_as_float(0x7f800000);
    if (R < n) {
        D2[R] = stored;
        idx[R] = 0;
    }
    const double s = block_sum_f64(R < n ? (double)stored : 0.0, red);
    if (tid == 0) partials[blockIdx.x] = s;
}

// ------------------------------------------------------------------ init
__global__ void pick_first_kernel(const float *X, int64_t n, int d, uint64_t seed, DevState *st,
                                  int32_t *cand, float *C) {
    __shared__ int64_t s_i0;
    if (threadIdx.x == 0) {
        const double u = uniform53(0, 0, TAG_INIT, seed);
        int64_t i0 = (int64_t)floor(__dmul_rn(u, (double)n));
        if (i0 >= n) i0 = n - 1;
        s_i0 = i0;
        st->i0 = (int32_t)i0;
        cand[0] = (int32_t)i0;
        st->m = 1;
        st->part_open = -1;
        st->batch_begin = 0;
        st->batch_cnt = 1;
        st->drawn = 0;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < d; q += blockDim.x) C[q] = X[s_i0 * (int64_t)d + q];
}

cudaError_t launch_init_first(Ctx &c) {
    pick_first_kernel<<<1, 128, 0, c.stream>>>(c.X, c.n, c.d, c.seed, c.st, c.cand, c.C);
    count_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int grid = (int)((c.n + kFirstRows - 1) / kFirstRows);
    const size_t smem = sizeof(float) * (size_t)std::min(c.d, kFirstPiece) * kFirstStride;
    first_dist_kernel<<<grid, kFirstRows, smem, c.stream>>>(c.X, c.n, c.d, c.C, c.D2, c.idx, c.partials);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return launch_phi_finalize(c, grid, &c.st->phi, &c.st->phi_hist[0]);
}

// ------------------------------------------------------------------ sampling
__global__ void sample_kernel(const float *__restrict__ D2, const int32_t *__restrict__ idx,
                              const float *__restrict__ X, const float *__restrict__ C, int64_t n, int d,
                              double ell, uint32_t round, uint64_t seed, DevState *st, int32_t *drawn,
                              int cap) {
    const double phi = st->phi;
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += stride) {
        const int64_t i = base + threadIdx.x;
        bool take = false;
        if (i < n) {
            const float dd = D2[i];
            double pr = 0.0;
            if (phi > 0.0) pr = fmin(1.0, __ddiv_rn(__dmul_rn(ell, (double)dd), phi));
            const double u = uniform53((uint64_t)i, round, TAG_SAMPLE, seed);
            if (dd > 0.f && fabs(u - pr) <= 1e-5) {
                // the FP32 D^2 could decide this draw: use the FP64 distance of the definition
                const double d64 = dist2_fp64(X + i * (int64_t)d, C + (int64_t)idx[i] * d, d);
                pr = fmin(1.0, __ddiv_rn(__dmul_rn(ell, d64), phi));
                atomicAdd(&st->sample_refined, 1ull);
            }
            if (fabs(u - pr) <= 1e-6) atomicAdd(&st->sample_near, 1ull);
            take = u < pr;
        }
        const unsigned mask = __ballot_sync(0xffffffffu, take);
        if (mask) {
            const int leader = __ffs(mask) - 1;
            int b = 0;
            if (lane == leader) b = atomicAdd(&st->drawn, __popc(mask));
            b = __shfl_sync(0xffffffffu, b, leader);
            if (take) {
                const int pos = b + __popc(mask & ((1u << lane) - 1u));
                if (pos < cap) drawn[pos] = (int32_t)i;
                else st->overflow = 1;
            }
        }
    }
}

// one CTA: bitonic sort of this round's draws (ascending point order), appended to
// the candidate list; the batch range is published in st for the next kernels.
__global__ void __launch_bounds__(1024) sort_batch_kernel(const int32_t *drawn, int cap, int round,
                                                          DevState *st, int32_t *cand) {
    extern __shared__ int32_t keys[];
    const int total = st->drawn;
    const int cnt = min(total, cap);
    int P = 1;
    while (P < cnt) P <<= 1;
    for (int e = threadIdx.x; e < P; e += blockDim.x) keys[e] = e < cnt ? drawn[e] : INT_MAX;
    for (int size = 2; size <= P; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            __syncthreads();
            for (int e = threadIdx.x; e < P; e += blockDim.x) {
                const int o = e ^ stride;
                if (o > e) {
                    const bool asc = (e & size) == 0;
                    const int a = keys[e], b = keys[o];
                    if ((a > b) == asc) { keys[e] = b; keys[o] = a; }
                }
            }
        }
    }
    __syncthreads();
    const int m0 = st->m;
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) cand[m0 + e] = keys[e];
    __syncthreads();
    if (threadIdx.x == 0) {
        st->batch_begin = m0;
        st->batch_cnt = cnt;
        st->m = m0 + cnt;
        st->round_added[round - 1] = total;
        st->drawn = 0;
    }
}

__global__ void gather_kernel(const float *__restrict__ X, int d, const DevState *st, const int32_t *cand,
                              float *C) {
    const int begin = st->batch_begin, cnt = st->batch_cnt;
    const int64_t total = (int64_t)cnt * d;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / d;
        const int q = (int)(e - r * d);
        C[(begin + r) * d + q] = X[(int64_t)cand[begin + r] * d + q];
    }
}

__global__ void __launch_bounds__(1024) sum_f64_kernel(const double *parts, int nparts, double *out,
                                                      double *copy) {
    __shared__ double sh[32];
    double v = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) v += parts[i];
    const double s = block_sum_f64(v, sh);
    if (threadIdx.x == 0) {
        *out = s;
        if (copy) *copy = s;
    }
}

cudaError_t launch_sum_f64(const double *parts, int nparts, double *out, double *copy, cudaStream_t s) {
    sum_f64_kernel<<<1, 1024, 0, s>>>(parts, nparts, out, copy);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_phi_finalize(Ctx &c, int nparts, double *out, double *hist_slot) {
    return launch_sum_f64(c.partials, nparts, out, hist_slot, c.stream);
}

cudaError_t launch_round(Ctx &c, int round) {
    cudaError_t e;
    if (c.sampling == 1) {
        if ((e = launch_sample_exact(c, round)) != cudaSuccess) return e;
    } else {
        const int sgrid = c.num_sms * 8;
        sample_kernel<<<sgrid, 256, 0, c.stream>>>(c.D2, c.idx, c.X, c.C, c.n, c.d, c.ell, (uint32_t)round,
                                                   c.seed, c.st, c.drawn, c.cap_round);
        count_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    int P = 1;
    while (P < c.cap_round) P <<= 1;
    sort_batch_kernel<<<1, 1024, P * sizeof(int32_t), c.stream>>>(c.drawn, c.cap_round, round, c.st, c.cand);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int64_t gtot = (int64_t)c.cap_round * c.d;
    const int ggrid = (int)std::min<int64_t>((gtot + 255) / 256, (int64_t)c.num_sms * 16);
    gather_kernel<<<ggrid, 256, 0, c.stream>>>(c.X, c.d, c.st, c.cand, c.C);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    count_launches(2);
    return launch_round_distance(c, round);
}

cudaError_t launch_sum_rows(const float *v, int64_t n, double *partials, int max_parts, double *out, double *copy,
                            cudaStream_t s);

// Whether the round passes filter rows by their candidate (see the round filter): the
// lists take a screening pass over the old candidates, at most cap_total of them, so
// they have to be few against the rows, and its 25 launches cost some 60 us a round, which
// a dense pass of under 4e7 rows x candidates does not (seeding of 30,000 x 64, l = 100:
// 1.55 ms without, 1.67 with; 100,000 x 64, l = 200: 2.21, 2.13).
bool round_filter_sizes(const Ctx &c) {
    return c.rounds > 0 && tc::tc_norms_in_epilogue(c.tc_fmt) && c.d % 4 == 0 &&
           resident_plan(c.cap_round, c.d).parts == 0 && (int64_t)c.cap_total <= c.n / 8 &&
           (double)c.n * c.cap_round >= 4e7;
}
static bool round_filter_usable(const Ctx &c) {
    return c.rf_rows != nullptr && ((reinterpret_cast<uintptr_t>(c.X) | reinterpret_cast<uintptr_t>(c.C)) & 15u) == 0;
}

// The part of the round's batch that the next distance pass covers: part s of S equal
// ones, or all that is left when the filter left most rows open in the pass before (the
// data does not separate, and every part would go over all rows again) or hardly any
// (nothing is left to save); s = S: the whole batch again.  filter: the pass may use lists;
// where they left most rows open, the next try waits until there are kListRetry times as many
// references (a round's list pass over data that do not separate costs a fifth of it).
constexpr int kListRetry = 6;

__global__ void round_part_kernel(DevState *st, int s, int S, int filter, const int *open_cnt, int64_t n) {
    if (st->list_refs > 0) {   // the outcome of the last list pass
        const int64_t open = *open_cnt;
        st->part_open = (int32_t)open;
        st->list_fail = open * 4 > 3 * n ? st->list_refs : 0;
        st->list_refs = 0;
    }
    if (s == 0) {
        st->part_begin = st->batch_begin;
        st->part_total = st->batch_cnt;
        st->part_next = 0;
    }
    const int total = st->part_total, from = st->part_next;
    if (s == S) {
        st->batch_begin = st->part_begin;
        st->batch_cnt = total;
        return;
    }
    const int64_t open = st->part_open;
    const bool skip = filter && st->list_fail > 0 && st->part_begin + from < kListRetry * (int64_t)st->list_fail;
    const bool rest = skip || s == S - 1 || (open >= 0 && (open * 4 > 3 * n || open * 50 < n));
    const int to = rest ? total : max(from, (int)((int64_t)total * (s + 1) / S));
    st->batch_begin = st->part_begin + from;
    st->batch_cnt = to - from;
    st->part_next = to;
    st->list_skip = skip && to > from;
    st->list_refs = filter && !skip && to > from ? st->batch_begin : 0;
}

// Parts of a round's batch.  A part's candidates filter the parts after it, so the dense
// pass of a later part covers fewer rows; a part costs about 9 ns a row beyond its
// screening (2 ps a row and candidate at d = 128), which parts of about 5,000
// candidates outweigh.
static int round_parts(const Ctx &c) {
    if (!round_filter_usable(c)) return 1;
    return std::max(1, std::min(4, c.cap_round / 5000));
}

// Alg. 2 step 5: D^2/idx against the batch just appended, then phi
cudaError_t launch_round_distance(Ctx &c, int round) {
    cudaError_t e;
    if (c.precision != KMPAR_FP32) {
        const int S = round_parts(c);
        const bool planned = round_filter_usable(c);   // (S > 1 only then)
        for (int s = 0; s < S; ++s) {
            c.round_part = s;
            if (planned) {
                // (the first pass of the first round has no filter)
                round_part_kernel<<<1, 1, 0, c.stream>>>(c.st, s, S, s + c.rounds_done > 0, c.rf_cnt, c.n);
                count_launches(1);
            }
            if ((e = launch_tc_pass(c, 1, c.C, 0, nullptr, nullptr, nullptr, nullptr, 0, nullptr, nullptr)) !=
                cudaSuccess)
                return e;
        }
        c.round_part = 0;
        if (S > 1) {
            round_part_kernel<<<1, 1, 0, c.stream>>>(c.st, S, S, 0, c.rf_cnt, c.n);
            count_launches(1);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        return launch_sum_rows(c.D2, c.n, c.partials, c.sum_blocks, &c.st->phi, &c.st->phi_hist[round], c.stream);
    }
    cudaEvent_t ev = nullptr;
    if ((e = timing_begin(c, &ev)) != cudaSuccess) return e;
    NearestParams p{};
    p.X = c.X; p.n = c.n; p.d = c.d; p.C = c.C; p.st = c.st; p.D2 = c.D2; p.idx = c.idx;
    p.partials = c.partials; p.fp64_cnt = &c.st->argmin_fp64; p.wide_cnt = &c.st->argmin_wide;
    if ((e = launch_nearest_mode<MODE_ROUND>(p, c.cap_round, c.stream)) != cudaSuccess) return e;
    if ((e = timing_end(c, ev, 0)) != cudaSuccess) return e;
    return launch_phi_finalize(c, assign_num_partials(c.n, c.d), &c.st->phi, &c.st->phi_hist[round]);
}

cudaError_t launch_assign(const float *X, int64_t n, int d, const float *C, int k, int32_t *labels,
                          const int32_t *prev, int *changed, double *partials, int,
                          unsigned long long *fp64_cnt, cudaStream_t s) {
    NearestParams p{};
    p.X = X; p.n = n; p.d = d; p.C = C; p.c_begin = 0; p.c_cnt = k;
    p.labels = labels; p.prev = prev; p.changed = changed; p.partials = partials;
    p.fp64_cnt = fp64_cnt; p.wide_cnt = fp64_cnt;
    return launch_nearest_mode<MODE_ASSIGN>(p, k, s);
}

// ------------------------------------------------------------------ generator export
__global__ void uniforms_kernel(int64_t count, uint32_t round, uint32_t tag, uint64_t seed, double *out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = uniform53((uint64_t)i, round, tag, seed);
}

cudaError_t launch_uniforms(int64_t count, uint32_t round, uint32_t tag, uint64_t seed, double *out,
                            cudaStream_t s) {
    const int grid = (int)std::min<int64_t>((count + 255) / 256, 4096);
    uniforms_kernel<<<grid > 0 ? grid : 1, 256, 0, s>>>(count, round, tag, seed, out);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace kmp

namespace kmp {
cudaError_t configure_refine_kernels();

cudaError_t configure_round_kernels() {
    cudaError_t e = cudaFuncSetAttribute(sort_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kMaxRoundCap * (int)sizeof(int32_t));
    if (e != cudaSuccess) return e;
    return configure_refine_kernels();
}
}  // namespace kmp

// ------------------------------------------------------------------ tensor-core passes
namespace kmp {

// deterministic FP64 sum of a float array: fixed per-block ranges, fixed trees
__global__ void __launch_bounds__(256) sum_rows_kernel(const float *__restrict__ v, int64_t n, int64_t per_block,
                                                      double *partials) {
    __shared__ double sh[32];
    const int64_t b0 = (int64_t)blockIdx.x * per_block;
    const int64_t b1 = min(n, b0 + per_block);
    double acc = 0.0;
    if ((per_block & 3) == 0 && (reinterpret_cast<uintptr_t>(v) & 15u) == 0) {
        // four consecutive values per thread and step, added in index order
        for (int64_t i = b0 + 4 * threadIdx.x; i < b1; i += 4 * blockDim.x) {
            if (i + 4 <= b1) {
                const float4 q = __ldg(reinterpret_cast<const float4 *>(v + i));
                acc += (double)q.x;
                acc += (double)q.y;
                acc += (double)q.z;
                acc += (double)q.w;
            } else {
                for (int64_t j = i; j < b1; ++j) acc += (double)v[j];
            }
        }
    } else {
        for (int64_t i = b0 + threadIdx.x; i < b1; i += blockDim.x) acc += (double)v[i];
    }
    const double s = block_sum_f64(acc, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

cudaError_t launch_sum_rows(const float *v, int64_t n, double *partials, int max_parts, double *out, double *copy,
                            cudaStream_t s) {
    int64_t per = 1024;
    int64_t nb = (n + per - 1) / per;
    if (nb > max_parts) {
        per = (n + max_parts - 1) / max_parts;
        nb = (n + per - 1) / per;
    }
    if (nb < 1) nb = 1;
    sum_rows_kernel<<<(int)nb, 256, 0, s>>>(v, n, per, partials);
    count_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_sum_f64(partials, (int)nb, out, copy, s);
}

// The decision for row R once its best and runner-up candidates (b1, i1), (b2, i2)
// have exact FP32 values (i2 = -1: none), taken exactly as nearest_decide takes
// it.  Lloyd: the label is the best, re-decided in FP64 against the runner-up
// when their FP32 values lie within the tie window.  Round: the current center
// is replaced by the best new candidate when nearer; when two or more of (current,
// best, runner-up) lie within the tie window they are re-decided in FP64, equal
// FP64 values keeping the lower center number.  Returns 1 when a Lloyd label
// changed.
template <int MODE>
__device__ __forceinline__ int decide_top2(const float *__restrict__ X, int d, const float *__restrict__ C, int64_t R,
                                           float b1, int i1, float b2, int i2, float *D2, int32_t *idx,
                                           int32_t *labels, const int32_t *prev, float *dmin,
                                           unsigned long long *fp64_cnt, unsigned long long *wide_cnt) {
    const float W = fp32_tie_window(d);
    const float *xrow = X + R * d;
    if (MODE == MODE_ASSIGN) {
        int lab = i1 != INT_MAX ? i1 : 0;
        float stored = b1;
        if (i2 >= 0 && b2 <= b1 + W * b1) {
            double best = dist2_fp64(xrow, C + (int64_t)i1 * d, d);
            int bj = i1;
            take_if_better(dist2_fp64(xrow, C + (int64_t)i2 * d, d), i2, best, bj);
            if (bj == i2) { lab = i2; stored = b2; }
            atomicAdd(fp64_cnt, 1ull);
        }
        if (labels) labels[R] = lab;
        if (dmin) dmin[R] = stored;
        return (prev && prev[R] != lab) ? 1 : 0;
    } else {
        const float old = D2[R];
        const int oi = idx[R];
        const float m32 = fminf(old, b1);
        const float lim = m32 + W * m32;
        const bool in_old = (oi >= 0) && old <= lim;
        const bool in1 = i1 != INT_MAX && b1 <= lim;
        const bool in2 = i2 >= 0 && b2 <= lim;
        int win = -1;
        float wv = old;
        if ((int)in_old + (int)in1 + (int)in2 >= 2) {
            double best = DBL_MAX;
            int bj = INT_MAX;
            if (in_old) take_if_better(dist2_fp64(xrow, C + (int64_t)oi * d, d), oi, best, bj);
            if (in1) take_if_better(dist2_fp64(xrow, C + (int64_t)i1 * d, d), i1, best, bj);
            if (in2) take_if_better(dist2_fp64(xrow, C + (int64_t)i2 * d, d), i2, best, bj);
            atomicAdd(fp64_cnt, 1ull);
            if (in1 && in2) atomicAdd(wide_cnt, 1ull);
            if (bj == i1) { win = i1; wv = b1; }
            else if (bj == i2) { win = i2; wv = b2; }
        } else if (i1 != INT_MAX && b1 < old) {
            win = i1; wv = b1;
        }
        if (win >= 0) { D2[R] = wv; idx[R] = win; }
        return 0;
    }
}

// screening statistics of a pass: rows screened, rows the pair screening left
// undecided, and (after the list pass) rows that needed the exact scan
__global__ void count_fixups_kernel(const int *fix_cnt, const int *exact_cnt, int64_t n, const int *rows_cnt,
                                    DevState *st, int count_rows) {
    st->screen_fallback += (unsigned long long)*fix_cnt;
    if (count_rows) st->screen_rows += (unsigned long long)(rows_cnt ? (int64_t)*rows_cnt : n);
    st->screen_exact += (unsigned long long)(exact_cnt ? *exact_cnt : *fix_cnt);
}

cudaError_t count_fixups(Ctx &c, const int *exact_cnt, const int *rows_cnt = nullptr) {
    count_fixups_kernel<<<1, 1, 0, c.stream>>>(c.fix_cnt, exact_cnt, c.n, rows_cnt, c.st, c.round_part == 0);
    count_launches(1);
    return cudaGetLastError();
}

// the two halves of count_fixups when the undecided rows pass through several stages
__global__ void count_stage_kernel(const int *fallback_cnt, const int *exact_cnt, int64_t n, const int *rows_cnt,
                                   DevState *st, int count_rows) {
    if (fallback_cnt) {   // the rows the pair screening left, all refined from their own lists
        st->screen_fallback += (unsigned long long)*fallback_cnt;
        st->screen_listed += (unsigned long long)*fallback_cnt;
        if (count_rows) st->screen_rows += (unsigned long long)(rows_cnt ? (int64_t)*rows_cnt : n);
    }
    if (exact_cnt) st->screen_exact += (unsigned long long)*exact_cnt;
}

// Exact FP32 distances and the decision for the rows the tensor screening has
// brought down to one pair of adjacent centers (cand1 = the pair's first center,
// -1: none).  Both centers of the pair get the exact FP32 difference form
// (ascending coordinates, bit-identical to dist2_fp32); the row is certain when
// every center outside the pair is, by the screening bound, beyond the tie window
// of the pair's best exact value.  Certain rows take the CUDA-core decision
// (decide_top2) on the pair; the others go to the fix-up list.
__host__ __device__ __forceinline__ int refine_stride(int d) { return d + ((6 - (d & 3)) & 3); }   // = 2 mod 4

__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}

struct ScreenBound {
    const float *xnorm;            // ||x'||^2 per point (x' = x - anchor)
    const unsigned int *cmax_bits; // max ||c'|| of the batch
    const DevState *st;            // ROUND: batch range
    float ep, en, ec;              // E(x, c) = ep ||x'|| ||c'|| + en (||x'||^2 + ||c'||^2) + ec ||x'|| max ||c'||
    int32_t *fix_rows;
    int *fix_cnt;
    float *ub;                     // per listed row: exact FP32 upper bound of its deciding distance
};

// rows whose screening is not certain go to the fix-up list: one atomic per warp
__device__ __forceinline__ void append_fixups(const ScreenBound &sb, bool fix, int64_t R) {
    const unsigned m = __ballot_sync(0xffffffffu, fix);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    int base = 0;
    if (lane == 0) base = atomicAdd(sb.fix_cnt, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (fix) sb.fix_rows[base + __popc(m & ((1u << lane) - 1u))] = (int32_t)R;
}

// screened values arrive with their low 6 mantissa bits cleared (relative change
// below 2^-17); twice that is allowed for
constexpr float kKeyTrunc = 1.6e-5f;

// The certainty test.  m = the exact FP32 d^2 that decides the row: the pair's
// best in Lloyd, the nearer of the current center and the pair's best in a round
// (a center farther than the current one changes nothing unless it falls in the
// tie window).  v2 = a lower bound of the screened value (s = ||c'||^2 - 2 x'.c')
// of every center not examined exactly.  Such a center c has d^2 = s + ||x'||^2
// >= v2 - E(x, c) + ||x'||^2.  A center with ||c'|| > ||x'|| + sqrt(m (1 + 2W)) is
// farther than m (1 + 2W) by the triangle inequality; every nearer one has
// ||c'|| <= ceff, so E(x, c) <= Eo.  If the bound exceeds m (1 + 2W), no FP32 value
// outside the examined centers can win or fall in the tie window of the best
// (W = fp32_tie_window covers both FP32 errors).
__device__ __forceinline__ bool bound_certain(const ScreenBound &sb, float xnorm, float m, float v2lo, int d) {
    const float xn = fmaxf(xnorm, 0.f);
    const float X = sqrtf(xn);
    const float cmax = __uint_as_float(*sb.cmax_bits);
    const float W = fp32_tie_window(d);
    const float lim = fmaxf(m, 0.f) * (1.f + 2.f * W);
    const float ceff = fminf(cmax, X + sqrtf(lim));
    const float Eo = sb.ep * X * ceff + sb.en * (xn + ceff * ceff) + sb.ec * X * cmax;
    return (v2lo - Eo + xn) > lim + 1e-30f;
}

// the pair screening's v2 arrives key-truncated: lowered by that truncation (stays
// +inf when there is no other center)
__device__ __forceinline__ bool pair_certain(const ScreenBound &sb, float xnorm, float m, float v2, int d) {
    const float v2lo = v2 >= 0.f ? v2 * (1.f - kKeyTrunc) : v2 * (1.f + kKeyTrunc);
    return bound_certain(sb, xnorm, m, v2lo, d);
}

// a lower bound of the real d^2 of every center outside the examined ones, from
// their smallest screened value (key-truncated v2, lowered): v2lo - E + ||x'||^2
// with E at the largest center norm (no triangle-inequality cut: this bound is
// kept for Lloyd's next iteration, where it has to hold for every center)
__device__ __forceinline__ float outside_lb(const ScreenBound &sb, float xnorm, float v2) {
    const float v2lo = v2 >= 0.f ? v2 * (1.f - kKeyTrunc) : v2 * (1.f + kKeyTrunc);
    const float xn = fmaxf(xnorm, 0.f);
    const float X = sqrtf(xn);
    const float cmax = __uint_as_float(*sb.cmax_bits);
    const float E = sb.ep * X * cmax + sb.en * (xn + cmax * cmax) + sb.ec * X * cmax;
    return v2lo - E + xn;
}

// Lloyd's bounds of a row for the next iteration, as distances: u >= the real
// distance to its center, l <= the real distance to every other center (FP32
// values carry at most W relative error; 1e-6 covers the rounding of these few
// operations).  l = 0: no bound.
__device__ __forceinline__ float bound_upper(float best, float W) { return sqrtf(best * (1.f + W)) * (1.f + 1e-6f); }
__device__ __forceinline__ float bound_lower(float l2, float xnorm, float W) {
    const float v = l2 * (1.f - 2.f * W) - 2.f * W * fmaxf(xnorm, 0.f);
    return v > 0.f ? sqrtf(v) * (1.f - 1e-6f) : 0.f;
}

// the distance that decides a row whose nearest screened center has exact FP32
// value b1 (FLT_MAX: none): see bound_certain
template <int MODE>
__device__ __forceinline__ float deciding(const float *D2, int64_t R, float b1) {
    return MODE == MODE_ROUND ? fminf(D2[R], b1) : b1;
}

// exact FP32 difference form of one row against one center, both in shared memory
// (8-byte loads when the row start is 8-byte aligned)
__device__ __forceinline__ float dist2_smem(const float *xa, const float *ca, int d, bool pairs) {
    float s = 0.f;
    if (pairs) {
        const float2 *x2 = reinterpret_cast<const float2 *>(xa);
        const float2 *c2 = reinterpret_cast<const float2 *>(ca);
#pragma unroll 4
        for (int p = 0; p < (d >> 1); ++p) {
            const float2 a = x2[p], c = c2[p];
            float t = __fsub_rn(a.x, c.x);
            s = __fmaf_rn(t, t, s);
            t = __fsub_rn(a.y, c.y);
            s = __fmaf_rn(t, t, s);
        }
        if (d & 1) {
            const float t = __fsub_rn(xa[d - 1], ca[d - 1]);
            s = __fmaf_rn(t, t, s);
        }
    } else {
#pragma unroll 4
        for (int q = 0; q < d; ++q) {
            const float t = __fsub_rn(xa[q], ca[q]);
            s = __fmaf_rn(t, t, s);
        }
    }
    return s;
}

// exact FP32 difference form of one row against several centers at once (rows in
// shared memory, 8-byte aligned): the chains are independent, so their FMA
// latencies overlap; each chain is still summed in ascending coordinates, so every
// value is bit-identical to dist2_fp32
template <int NC>
__device__ __forceinline__ void dist2_smem_multi(const float *xa, const float *const (&ca)[NC], int d, float (&s)[NC]) {
#pragma unroll
    for (int u = 0; u < NC; ++u) s[u] = 0.f;
    const float2 *x2 = reinterpret_cast<const float2 *>(xa);
#pragma unroll 2
    for (int p = 0; p < (d >> 1); ++p) {
        const float2 a = x2[p];
#pragma unroll
        for (int u = 0; u < NC; ++u) {
            const float2 c = reinterpret_cast<const float2 *>(ca[u])[p];
            float t = __fsub_rn(a.x, c.x);
            s[u] = __fmaf_rn(t, t, s[u]);
            t = __fsub_rn(a.y, c.y);
            s[u] = __fmaf_rn(t, t, s[u]);
        }
    }
    if (d & 1) {
#pragma unroll
        for (int u = 0; u < NC; ++u) {
            const float t = __fsub_rn(xa[d - 1], ca[u][d - 1]);
            s[u] = __fmaf_rn(t, t, s[u]);
        }
    }
}

// the pair's exact values in (value, center number) order; i2 = -1 when the pair
// has one real center
__device__ __forceinline__ void pair_top2(float va, int ja, float vb, int jb, bool has_b, float &b1, int &i1,
                                          float &b2, int &i2) {
    if (has_b && (vb < va || (vb == va && jb < ja))) { b1 = vb; i1 = jb; b2 = va; i2 = ja; }
    else { b1 = va; i1 = ja; b2 = has_b ? vb : FLT_MAX; i2 = has_b ? jb : -1; }
}

// Per-row copies: a warp takes 32 rows; asynchronous copies bring its 32 point
// rows and their pairs of center rows into shared memory (row stride = 2 mod 4:
// 8-byte aligned, conflict-free lane-per-row reads), then each lane sums its row.
template <int MODE>
__global__ void __launch_bounds__(256) refine_kernel(const float *__restrict__ X, int64_t n, int d,
                                                    const float *__restrict__ C, int c_cnt,
                                                    const int32_t *__restrict__ cand1, const float *__restrict__ v2s,
                                                    ScreenBound sb, float *D2, int32_t *idx, int32_t *labels,
                                                    const int32_t *prev, int *changed, float *dmin,
                                                    unsigned long long *fp64_cnt, unsigned long long *wide_cnt) {
    extern __shared__ __align__(16) float rsm[];
    const int ds = refine_stride(d);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float *xs = rsm + wid * 96 * ds;   // 32 point rows
    float *cs = xs + 32 * ds;          // 32 pairs of center rows
    const int64_t w0 = (int64_t)blockIdx.x * blockDim.x + wid * 32;
    const int nw = (int)max((int64_t)0, min((int64_t)32, n - w0));
    const int64_t R = w0 + lane;
    const int end = MODE == MODE_ROUND ? sb.st->batch_begin + sb.st->batch_cnt : c_cnt;
    int j = -1;
    if (lane < nw) j = cand1[R];
    const bool even = (d & 1) == 0;   // rows 8-byte aligned in global memory
    for (int rr = 0; rr < nw; ++rr) {
        const int jr = __shfl_sync(0xffffffffu, j, rr);
        if (jr < 0) continue;
        const int nc = jr + 1 < end ? 2 : 1;
        const float *xr = X + (w0 + rr) * d;
        const float *cr = C + (int64_t)jr * d;
        float *ct = cs + 2 * rr * ds;
        if (even) {
            for (int p = lane; p < (d >> 1); p += 32) {
                cp_async8(xs + rr * ds + 2 * p, xr + 2 * p);
                for (int u = 0; u < nc; ++u) cp_async8(ct + u * ds + 2 * p, cr + (int64_t)u * d + 2 * p);
            }
        } else {
            for (int q = lane; q < d; q += 32) {
                cp_async4(xs + rr * ds + q, xr + q);
                for (int u = 0; u < nc; ++u) cp_async4(ct + u * ds + q, cr + (int64_t)u * d + q);
            }
        }
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    bool fix = lane < nw && j < 0;
    int chg = 0;
    if (lane < nw && j >= 0) {
        const bool has_b = j + 1 < end;
        const float *ct = cs + 2 * lane * ds;
        const float *cp[2] = {ct, has_b ? ct + ds : ct};
        float v[2];
        dist2_smem_multi<2>(xs + lane * ds, cp, d, v);
        const float va = v[0], vb = has_b ? v[1] : 0.f;
        float b1, b2;
        int i1, i2;
        pair_top2(va, j, vb, j + 1, has_b, b1, i1, b2, i2);
        const float m = deciding<MODE>(D2, R, b1);
        if (pair_certain(sb, sb.xnorm[R], m, v2s[R], d))
            chg = decide_top2<MODE>(X, d, C, R, b1, i1, b2, i2, D2, idx, labels, prev, dmin, fp64_cnt, wide_cnt);
        else {
            fix = true;
            sb.ub[R] = m;
        }
    } else if (fix) {
        sb.ub[R] = deciding<MODE>(D2, R, FLT_MAX);
    }
    append_fixups(sb, fix, R);
    if (MODE == MODE_ASSIGN && changed) {
        const int c = warp_sum_i32(chg);
        if (lane == 0 && c) atomicAdd(changed, c);
    }
}

// Per-row refine for rows of d = 0 mod 4 floats (16-byte aligned): one thread per
// row sums every center of its screened group (G adjacent centers) with G
// interleaved exact FP32 chains (ascending coordinates, bit-identical to
// dist2_fp32) from 16-byte loads of the point row and the center rows; no
// shared-memory staging, so the kernel runs at full occupancy and the rows come
// through L1.  The lexicographic top-2 of the group then goes through the same
// certainty test and decision as a pair.
template <int MODE, int G>
__global__ void __launch_bounds__(256) refine_direct_kernel(const float *__restrict__ X, int64_t n, int d,
                                                           const float *__restrict__ C, int c_cnt,
                                                           const int32_t *__restrict__ cand1,
                                                           const float *__restrict__ v2s, ScreenBound sb, float *D2,
                                                           int32_t *idx, int32_t *labels, const int32_t *prev,
                                                           int *changed, float *dmin, unsigned long long *fp64_cnt,
                                                           unsigned long long *wide_cnt, const int32_t *order,
                                                           const int *nrows_dev, float *ubd, float *lbd) {
    // (the rows a compact round pass leaves undecided are listed by position, as its
    // lists are)
    // rows in the order given (a permutation of 0..n-1, e.g. the rows sorted by
    // their previous label: neighbouring threads then mostly read the same center
    // rows, which L1 serves), or in storage order.  nrows_dev: a compact pass over
    // the rows order[0 .. *nrows_dev), whose screening results are by position.
    const int64_t T = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = T < (nrows_dev ? (int64_t)*nrows_dev : n);
    const int64_t R = order && valid ? (int64_t)order[T] : T;
    const int64_t Ri = nrows_dev ? T : R;
    const int lane = threadIdx.x & 31;
    const int end = MODE == MODE_ROUND ? sb.st->batch_begin + sb.st->batch_cnt : c_cnt;
    const int j = valid ? cand1[Ri] : -1;
    if (MODE == MODE_ASSIGN && lbd && valid) lbd[R] = 0.f;   // no bound unless the row is certified below
    bool fix = valid && j < 0;
    int chg = 0;
    if (valid && j >= 0) {
        const float4 *x4 = reinterpret_cast<const float4 *>(X + R * d);
        const float4 *c4[G];
#pragma unroll
        for (int u = 0; u < G; ++u) c4[u] = reinterpret_cast<const float4 *>(C + (int64_t)min(j + u, end - 1) * d);
        float v[G];
#pragma unroll
        for (int u = 0; u < G; ++u) v[u] = 0.f;
#pragma unroll 2
        for (int p = 0; p < (d >> 2); ++p) {
            const float4 x = __ldg(x4 + p);
#pragma unroll
            for (int u = 0; u < G; ++u) {
                const float4 c = __ldg(c4[u] + p);
                float t;
                t = __fsub_rn(x.x, c.x); v[u] = __fmaf_rn(t, t, v[u]);
                t = __fsub_rn(x.y, c.y); v[u] = __fmaf_rn(t, t, v[u]);
                t = __fsub_rn(x.z, c.z); v[u] = __fmaf_rn(t, t, v[u]);
                t = __fsub_rn(x.w, c.w); v[u] = __fmaf_rn(t, t, v[u]);
            }
        }
        // lexicographic (value, center number) top-2 over the group's real centers
        float b1 = FLT_MAX, b2 = FLT_MAX;
        int i1 = INT_MAX, i2 = -1;
#pragma unroll
        for (int u = 0; u < G; ++u) {
            if (j + u < end) {
                if (v[u] < b1) { b2 = b1; i2 = i1 == INT_MAX ? -1 : i1; b1 = v[u]; i1 = j + u; }
                else if (v[u] < b2) { b2 = v[u]; i2 = j + u; }
            }
        }
        if (i2 < 0) b2 = FLT_MAX;
        const float m = deciding<MODE>(D2, R, b1);
        const float v2r = v2s[Ri];
        if (pair_certain(sb, sb.xnorm[R], m, v2r, d)) {
            chg = decide_top2<MODE>(X, d, C, R, b1, i1, b2, i2, D2, idx, labels, prev, dmin, fp64_cnt, wide_cnt);
            if (MODE == MODE_ASSIGN && lbd) {
                // the group's runner-up (exact FP32) and the bound outside the group
                const float W = fp32_tie_window(d);
                const bool first = labels[R] == i1;
                const float runner = first ? b2 : b1;
                ubd[R] = bound_upper(first ? b1 : b2, W);
                lbd[R] = bound_lower(fminf(runner, outside_lb(sb, sb.xnorm[R], v2r)), sb.xnorm[R], W);
            }
        } else {
            fix = true;
            sb.ub[R] = m;
        }
    } else if (fix) {
        sb.ub[R] = deciding<MODE>(D2, R, FLT_MAX);
    }
    append_fixups(sb, fix, MODE == MODE_ROUND ? Ri : R);
    if (MODE == MODE_ASSIGN && changed) {
        const int c = warp_sum_i32(chg);
        if (lane == 0 && c) atomicAdd(changed, c);
    }
}

// Centers resident in shared memory (used when lane-per-row reads are conflict-free:
// d odd or d = 2 mod 4).  Persistent CTAs copy the pass's centers once; each warp
// then walks 32-row blocks of X.  A block is contiguous in X, so flat 16-byte
// asynchronous copies bring it in, double-buffered per warp, and the next block's
// screening results are loaded while the current block is summed.  A pass whose
// centers exceed shared memory runs as a few launches, each holding the slice
// [part_lo, part_lo + part_rows) of the centers (plus the next row, the partner of
// a pair that ends the slice): a row is refined by the launch whose slice holds its
// screened pair, and rows without one are listed for the fix-up by the first.
__host__ __device__ __forceinline__ int resident_center_floats(int cap_rows, int d) { return (cap_rows * d + 3) & ~3; }
__host__ __device__ __forceinline__ int resident_block_floats(int d) { return (32 * d + 3) & ~3; }

template <int MODE>
__global__ void __launch_bounds__(512) refine_resident_kernel(
    const float *__restrict__ X, int64_t n, int d, const float *__restrict__ C, int cap_rows, int part_lo,
    int part_rows, int hold_rows, const int32_t *__restrict__ cand1, const float *__restrict__ v2s, ScreenBound sb,
    float *D2, int32_t *idx, int32_t *labels, const int32_t *prev, int *changed, float *dmin,
    unsigned long long *fp64_cnt, unsigned long long *wide_cnt) {
    extern __shared__ __align__(16) float rsm[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int begin = MODE == MODE_ROUND ? sb.st->batch_begin : 0;
    const int cnt = MODE == MODE_ROUND ? min(sb.st->batch_cnt, cap_rows) : cap_rows;
    const int lo = part_lo, hi = min(cnt, part_lo + part_rows);
    if (lo > 0 && lo >= hi) return;   // uniform per block: the batch ends before this slice
    const int nhold = max(0, min(cnt, hi + 1) - lo);   // <= hold_rows
    const int xfl = resident_block_floats(d);
    float *Cs = rsm;
    float *xb = rsm + resident_center_floats(hold_rows, d) + wid * 2 * xfl;
    {
        const float *src = C + (int64_t)(begin + lo) * d;
        const int nf = nhold * d;
        if ((reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
            for (int f = threadIdx.x; f < (nf >> 2); f += blockDim.x) cp_async16(Cs + 4 * f, src + 4 * f);
            for (int f = (nf & ~3) + threadIdx.x; f < nf; f += blockDim.x) cp_async4(Cs + f, src + f);
        } else {
            for (int f = threadIdx.x; f < nf; f += blockDim.x) cp_async4(Cs + f, src + f);
        }
        cp_async_commit();
    }
    const int64_t nb = (n + 31) / 32;
    const int64_t gw = (int64_t)blockIdx.x * nwarps + wid, W = (int64_t)gridDim.x * nwarps;
    // a block starts at 32 b d floats = 128 b d bytes: 16-byte aligned when X is
    const bool xal = (reinterpret_cast<uintptr_t>(X) & 15u) == 0;
    auto issue = [&](int64_t b, float *dst) {
        const int64_t r0 = b * 32;
        const int nf = (int)min((int64_t)32, n - r0) * d;
        const float *src = X + r0 * d;
        if (xal) {
            for (int f = lane; f < (nf >> 2); f += 32) cp_async16(dst + 4 * f, src + 4 * f);
            for (int f = (nf & ~3) + lane; f < nf; f += 32) cp_async4(dst + f, src + f);
        } else {
            for (int f = lane; f < nf; f += 32) cp_async4(dst + f, src + f);
        }
    };
    // screening results of block b for this lane's row
    auto fetch = [&](int64_t b, int &j, float &v2, float &xn) {
        const int64_t R = b * 32 + lane;
        j = -1;
        v2 = 0.f;
        xn = 0.f;
        if (b < nb && R < n) {
            j = cand1[R];
            v2 = v2s[R];
            xn = sb.xnorm[R];
        }
    };
    if (gw < nb) issue(gw, xb);
    cp_async_commit();
    int jn;
    float v2n, xnn;
    fetch(gw, jn, v2n, xnn);
    cp_async_wait<1>();   // the centers (the first block may still be in flight)
    __syncthreads();
    const bool pairs = (d & 1) == 0;
    int chg = 0, it = 0;
    for (int64_t b = gw; b < nb; b += W, ++it) {
        const float *cur = xb + (it & 1) * xfl;
        if (b + W < nb) issue(b + W, xb + ((it + 1) & 1) * xfl);
        cp_async_commit();
        int j = jn;
        const float v2 = v2n, xn = xnn;
        fetch(b + W, jn, v2n, xnn);
        const int64_t R = b * 32 + lane;
        const bool valid = R < n;
        cp_async_wait<1>();   // this block is in (the next one may be pending)
        __syncwarp();
        const int jl = j - begin;   // batch-local pair start (j = -1: none)
        const bool screened = j >= 0 && jl >= 0 && jl < cnt;
        bool fix = valid && !screened && lo == 0;
        if (valid && screened && jl >= lo && jl < hi) {
            const bool has_b = jl + 1 < cnt;
            const float *xa = cur + lane * d;
            const float *ca = Cs + (int64_t)(jl - lo) * d;
            float va, vb = 0.f;
            if (pairs) {
                const float *cp[2] = {ca, has_b ? ca + d : ca};
                float v[2];
                dist2_smem_multi<2>(xa, cp, d, v);
                va = v[0];
                if (has_b) vb = v[1];
            } else {
                va = dist2_smem(xa, ca, d, false);
                if (has_b) vb = dist2_smem(xa, ca + d, d, false);
            }
            float b1, b2;
            int i1, i2;
            pair_top2(va, j, vb, j + 1, has_b, b1, i1, b2, i2);
            const float m = deciding<MODE>(D2, R, b1);
            if (pair_certain(sb, xn, m, v2, d))
                chg += decide_top2<MODE>(X, d, C, R, b1, i1, b2, i2, D2, idx, labels, prev, dmin, fp64_cnt, wide_cnt);
            else {
                fix = true;
                sb.ub[R] = m;
            }
        } else if (fix) {
            sb.ub[R] = deciding<MODE>(D2, R, FLT_MAX);
        }
        append_fixups(sb, fix, R);
        __syncwarp();   // the buffer is refilled two blocks later
    }
    cp_async_wait<0>();
    if (MODE == MODE_ASSIGN && changed) {
        const int c = warp_sum_i32(chg);
        if (lane == 0 && c) atomicAdd(changed, c);
    }
}

// warps of a resident refine CTA holding all cap_rows centers (0: they do not fit,
// or the stride is not conflict-free)
int resident_warps(int cap_rows, int d) {
    if (!((d & 1) || (d & 3) == 2)) return 0;
    const size_t budget = 200u * 1024u;
    const size_t cbytes = sizeof(float) * (size_t)resident_center_floats(cap_rows, d);
    if (cbytes >= budget) return 0;
    const size_t per_warp = sizeof(float) * 2 * (size_t)resident_block_floats(d);
    const int w = (int)((budget - cbytes) / per_warp);
    return w < 4 ? 0 : (w > 16 ? 16 : w);
}

size_t resident_smem_bytes(int cap_rows, int d, int warps) {
    return sizeof(float) * ((size_t)resident_center_floats(cap_rows, d) + (size_t)warps * 2 * resident_block_floats(d));
}

ResidentPlan resident_plan(int cap_rows, int d) {
    const int w1 = resident_warps(cap_rows, d);
    if (w1 > 0) return {1, cap_rows, cap_rows, w1};
    if (!((d & 1) || (d & 3) == 2)) return {0, 0, 0, 0};
    // slices: 8 warps, the rest of the 200 KB for one slice of centers plus the
    // partner row; each launch reads X once, so at most 3 of them
    const int warps = 8;
    const size_t per_warp = sizeof(float) * 2 * (size_t)resident_block_floats(d);
    if (warps * per_warp + sizeof(float) * 66 * (size_t)d + 16 > 200u * 1024u) return {0, 0, 0, 0};
    const size_t cfloats = (200u * 1024u - warps * per_warp) / sizeof(float);
    const int hold = (int)((cfloats - 3) / (size_t)d);   // resident_center_floats adds at most 3
    const int rows = (hold - 1) & ~1;
    if (rows < 64) return {0, 0, 0, 0};
    const int parts = (cap_rows + rows - 1) / rows;
    if (parts > 3) return {0, 0, 0, 0};
    return {parts, rows, rows + 1, warps};
}

// warps per refine CTA: 96 staged rows (32 points, 32 pairs of centers) of
// refine_stride(d) floats each, within 200 KB
int refine_warps(int d) {
    const int w = (int)((200u * 1024u) / (96u * 4u * (unsigned)refine_stride(d)));
    return w > 8 ? 8 : (w < 1 ? 1 : w);
}

size_t refine_smem_bytes(int d) { return sizeof(float) * refine_warps(d) * 96 * (size_t)refine_stride(d); }

// Rows the screening could not settle, scanned exactly against every center of the
// pass.  A CTA takes tiles of 32 listed rows, four per warp; the centers stream
// through shared memory in chunks of 64 (asynchronous copies, double-buffered) and
// lane l sums centers l and l + 32 of each chunk for the warp's four rows in the
// exact FP32 difference form in ascending coordinates (bit-identical to
// dist2_fp32): per coordinate pair four broadcast and two conflict-free 8-byte
// shared loads (row stride 2 mod 4) feed 32 FP32 operations, and every center chunk
// serves 32 rows.  A lexicographic top-2 per row is merged across the warp, then the
// same decision as nearest_decide (decide_top2).  Persistent: the row count is read
// on the device.
constexpr int kFxWarpRows = 4;
constexpr int kFxRows = 8 * kFxWarpRows;
constexpr int kFxCent = 64;

template <int MODE>
__global__ void __launch_bounds__(256) fixup_kernel(const float *__restrict__ X, int d, const float *__restrict__ C,
                                                   int c_cnt, int c_pairs, const DevState *st,
                                                   const int32_t *__restrict__ rows, const int *rows_cnt, float *D2,
                                                   int32_t *idx, int32_t *labels, const int32_t *prev, int *changed,
                                                   float *dmin, unsigned long long *fp64_cnt,
                                                   unsigned long long *wide_cnt) {
    extern __shared__ __align__(16) float fsm[];
    const int ds = refine_stride(d);
    float *xs = fsm;                   // kFxRows x ds point rows (row wid + 8 r of the tile: xs + (wid + 8 r) ds)
    float *cs = fsm + kFxRows * ds;    // 2 x kFxCent x ds center rows
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nrows = *rows_cnt;
    const int begin = MODE == MODE_ROUND ? st->batch_begin : 0;
    const int cnt = MODE == MODE_ROUND ? st->batch_cnt : c_cnt;
    const int nchunk = (cnt + kFxCent - 1) / kFxCent;
    const float FMAX = FLT_MAX;
    auto issue = [&](int ch) {
        float *dst = cs + (ch & 1) * kFxCent * ds;
        const int j0 = ch * kFxCent;
        const int nc = min(kFxCent, cnt - j0);
        for (int rr = wid; rr < nc; rr += 8) {
            const float *src = C + (int64_t)(begin + j0 + rr) * d;
            if (c_pairs)
                for (int p = lane; p < (d >> 1); p += 32) cp_async8(dst + rr * ds + 2 * p, src + 2 * p);
            for (int q = (c_pairs ? (d & ~1) : 0) + lane; q < d; q += 32) cp_async4(dst + rr * ds + q, src + q);
        }
    };
    for (int t0 = blockIdx.x * kFxRows; t0 < nrows; t0 += gridDim.x * kFxRows) {   // uniform per block
        const int nr = min(kFxRows, nrows - t0);
        __syncthreads();   // the previous tile's readers are done with xs and cs
#pragma unroll
        for (int r = 0; r < kFxWarpRows; ++r) {
            const int tr = wid + 8 * r;
            if (tr < nr) {
                const float *src = X + (int64_t)rows[t0 + tr] * d;
                for (int q = lane; q < d; q += 32) xs[tr * ds + q] = __ldg(src + q);
            }
        }
        if (nchunk > 0) issue(0);
        cp_async_commit();
        float b1[kFxWarpRows], b2[kFxWarpRows];
        int i1[kFxWarpRows], i2[kFxWarpRows];
#pragma unroll
        for (int r = 0; r < kFxWarpRows; ++r) { b1[r] = FMAX; b2[r] = FMAX; i1[r] = INT_MAX; i2[r] = INT_MAX; }
        for (int ch = 0; ch < nchunk; ++ch) {
            if (ch + 1 < nchunk) issue(ch + 1);
            cp_async_commit();
            cp_async_wait<1>();
            __syncthreads();   // chunk ch and the point rows are visible
            const float *cb = cs + (ch & 1) * kFxCent * ds;
            const float *c0 = cb + lane * ds, *c1 = cb + (lane + 32) * ds;
            float a0[kFxWarpRows], a1[kFxWarpRows];
#pragma unroll
            for (int r = 0; r < kFxWarpRows; ++r) { a0[r] = 0.f; a1[r] = 0.f; }
            const float2 *p0 = reinterpret_cast<const float2 *>(c0);
            const float2 *p1 = reinterpret_cast<const float2 *>(c1);
#pragma unroll 2
            for (int p = 0; p < (d >> 1); ++p) {
                const float2 u = p0[p], v = p1[p];
#pragma unroll
                for (int r = 0; r < kFxWarpRows; ++r) {
                    const float2 x = reinterpret_cast<const float2 *>(xs + (wid + 8 * r) * ds)[p];
                    float t = __fsub_rn(x.x, u.x);
                    a0[r] = __fmaf_rn(t, t, a0[r]);
                    t = __fsub_rn(x.y, u.y);
                    a0[r] = __fmaf_rn(t, t, a0[r]);
                    t = __fsub_rn(x.x, v.x);
                    a1[r] = __fmaf_rn(t, t, a1[r]);
                    t = __fsub_rn(x.y, v.y);
                    a1[r] = __fmaf_rn(t, t, a1[r]);
                }
            }
            if (d & 1) {
#pragma unroll
                for (int r = 0; r < kFxWarpRows; ++r) {
                    const float xe = xs[(wid + 8 * r) * ds + d - 1];
                    float t = __fsub_rn(xe, c0[d - 1]);
                    a0[r] = __fmaf_rn(t, t, a0[r]);
                    t = __fsub_rn(xe, c1[d - 1]);
                    a1[r] = __fmaf_rn(t, t, a1[r]);
                }
            }
            const int jl0 = ch * kFxCent + lane, jl1 = jl0 + 32;
#pragma unroll
            for (int r = 0; r < kFxWarpRows; ++r) {
                if (jl0 < cnt && lex_lt(a0[r], begin + jl0, b2[r], i2[r])) {
                    if (lex_lt(a0[r], begin + jl0, b1[r], i1[r])) {
                        b2[r] = b1[r]; i2[r] = i1[r]; b1[r] = a0[r]; i1[r] = begin + jl0;
                    } else {
                        b2[r] = a0[r]; i2[r] = begin + jl0;
                    }
                }
                if (jl1 < cnt && lex_lt(a1[r], begin + jl1, b2[r], i2[r])) {
                    if (lex_lt(a1[r], begin + jl1, b1[r], i1[r])) {
                        b2[r] = b1[r]; i2[r] = i1[r]; b1[r] = a1[r]; i1[r] = begin + jl1;
                    } else {
                        b2[r] = a1[r]; i2[r] = begin + jl1;
                    }
                }
            }
            __syncthreads();   // every reader is done with this buffer before it is refilled
        }
        cp_async_wait<0>();
#pragma unroll
        for (int r = 0; r < kFxWarpRows; ++r) {
            float v1 = b1[r], v2 = b2[r];
            int j1 = i1[r], j2 = i2[r];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float c1v = __shfl_xor_sync(0xffffffffu, v1, o), c2v = __shfl_xor_sync(0xffffffffu, v2, o);
                const int k1 = __shfl_xor_sync(0xffffffffu, j1, o), k2 = __shfl_xor_sync(0xffffffffu, j2, o);
                top2_merge(v1, j1, v2, j2, c1v, k1, c2v, k2);
            }
            const int tr = wid + 8 * r;
            if (lane == 0 && tr < nr) {
                const int64_t R = rows[t0 + tr];
                if (j2 == INT_MAX) { j2 = -1; v2 = FMAX; }
                if (decide_top2<MODE>(X, d, C, R, v1, j1, v2, j2, D2, idx, labels, prev, dmin, fp64_cnt, wide_cnt) &&
                    changed)
                    atomicAdd(changed, 1);
            }
        }
    }
}

// Fix-up with the pass's centers resident in shared memory (used when they fit):
// persistent CTAs copy the centers once (row stride 2 mod 4: lane l reading center
// l of a consecutive run is conflict-free with 8-byte loads); then one warp per
// listed row: the row is staged, lane l sums centers l, l + 32, ... in the exact
// FP32 difference form (bit-identical to dist2_fp32), a lexicographic top-2 is
// merged across the warp and decided by decide_top2.  No center is read from
// global memory more than once per CTA.  Listed row t goes to CTA t mod G (G CTAs),
// so when the rows outnumber the warps the warps that take a second row are spread
// one or two per SM instead of filling the first SMs.
template <int MODE>
__global__ void __launch_bounds__(512) fixup_resident_kernel(const float *__restrict__ X, int d,
                                                            const float *__restrict__ C, int c_cnt, int cap_rows,
                                                            int c_pairs, const DevState *st,
                                                            const int32_t *__restrict__ rows, const int *rows_cnt,
                                                            float *D2, int32_t *idx, int32_t *labels,
                                                            const int32_t *prev, int *changed, float *dmin,
                                                            unsigned long long *fp64_cnt,
                                                            unsigned long long *wide_cnt) {
    extern __shared__ __align__(16) float fsm[];
    const int ds = refine_stride(d);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int nrows = *rows_cnt;
    if ((int)blockIdx.x >= nrows) return;   // uniform per block: nothing for this CTA
    const int begin = MODE == MODE_ROUND ? st->batch_begin : 0;
    const int cnt = MODE == MODE_ROUND ? min(st->batch_cnt, cap_rows) : c_cnt;
    float *Cs = fsm;                                   // cap_rows x ds
    float *xs = fsm + (size_t)cap_rows * ds + wid * ds; // this warp's point row
    for (int rr = wid; rr < cnt; rr += nwarps) {
        const float *src = C + (int64_t)(begin + rr) * d;
        if (c_pairs)
            for (int p = lane; p < (d >> 1); p += 32) cp_async8(Cs + rr * ds + 2 * p, src + 2 * p);
        for (int q = (c_pairs ? (d & ~1) : 0) + lane; q < d; q += 32) cp_async4(Cs + rr * ds + q, src + q);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    const float FMAX = FLT_MAX;
    for (int t = wid * gridDim.x + blockIdx.x; t < nrows; t += gridDim.x * nwarps) {   // uniform per warp
        const int64_t R = rows[t];
        for (int q = lane; q < d; q += 32) xs[q] = __ldg(X + R * d + q);
        __syncwarp();
        float b1 = FMAX, b2 = FMAX;
        int i1 = INT_MAX, i2 = INT_MAX;
        // lane l: centers l, l + 32, l + 64, l + 96 summed together, then the next 128
        for (int j0 = lane; j0 < cnt; j0 += 128) {
            const float *cp[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) cp[u] = Cs + (size_t)min(j0 + 32 * u, cnt - 1) * ds;
            float v[4];
            dist2_smem_multi<4>(xs, cp, d, v);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int jl = j0 + 32 * u;
                if (jl < cnt) {
                    const int j = begin + jl;
                    if (lex_lt(v[u], j, b2, i2)) {
                        if (lex_lt(v[u], j, b1, i1)) { b2 = b1; i2 = i1; b1 = v[u]; i1 = j; }
                        else { b2 = v[u]; i2 = j; }
                    }
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float c1 = __shfl_xor_sync(0xffffffffu, b1, o), c2 = __shfl_xor_sync(0xffffffffu, b2, o);
            const int j1 = __shfl_xor_sync(0xffffffffu, i1, o), j2 = __shfl_xor_sync(0xffffffffu, i2, o);
            top2_merge(b1, i1, b2, i2, c1, j1, c2, j2);
        }
        if (lane == 0) {
            if (i2 == INT_MAX) { i2 = -1; b2 = FMAX; }
            if (decide_top2<MODE>(X, d, C, R, b1, i1, b2, i2, D2, idx, labels, prev, dmin, fp64_cnt, wide_cnt) &&
                changed)
                atomicAdd(changed, 1);
        }
        __syncwarp();   // the staged row is read before the next one overwrites it
    }
}

// warps of a resident fix-up CTA (0: the centers do not fit; use fixup_kernel)
int fixup_resident_warps(int cap_rows, int d) {
    const size_t budget = 200u * 1024u;
    const size_t cbytes = sizeof(float) * (size_t)cap_rows * refine_stride(d);
    const size_t per_warp = sizeof(float) * (size_t)refine_stride(d);
    if (cbytes + 16 * per_warp > budget) return 0;
    return 16;
}

size_t fixup_smem_bytes(int d) { return sizeof(float) * (size_t)(kFxRows + 2 * kFxCent) * refine_stride(d); }

cudaError_t launch_fixup(const Ctx &c, int mode_round, const float *C, int k, int32_t *labels, const int32_t *prev,
                         int *changed, float *dmin, const int32_t *rows, const int *rows_cnt) {
    // 8-byte center copies need d even and 8-byte aligned rows
    const int c_pairs = (c.d % 2 == 0) && (reinterpret_cast<uintptr_t>(C) % 8 == 0);
    const int cap_rows = mode_round ? c.cap_round : k;
    const int rw = fixup_resident_warps(cap_rows, c.d);
    if (rw > 0) {
        const size_t sm = sizeof(float) * ((size_t)cap_rows + rw) * refine_stride(c.d);
        if (mode_round)
            fixup_resident_kernel<MODE_ROUND><<<c.num_sms, 32 * rw, sm, c.stream>>>(
                c.X, c.d, C, 0, cap_rows, c_pairs, c.st, rows, rows_cnt, c.D2, c.idx, nullptr, nullptr,
                nullptr, nullptr, &c.st->argmin_fp64, &c.st->argmin_wide);
        else
            fixup_resident_kernel<MODE_ASSIGN><<<c.num_sms, 32 * rw, sm, c.stream>>>(
                c.X, c.d, C, k, cap_rows, c_pairs, c.st, rows, rows_cnt, nullptr, nullptr, labels, prev,
                changed, dmin, &c.st->argmin_fp64, &c.st->argmin_wide);
        count_launches(1);
        return cudaGetLastError();
    }
    const int grid = c.num_sms * 4;   // persistent: the row count is only known on the device
    const size_t sm = fixup_smem_bytes(c.d);
    const int pairs = c_pairs;
    if (mode_round)
        fixup_kernel<MODE_ROUND><<<grid, 256, sm, c.stream>>>(c.X, c.d, C, 0, pairs, c.st, rows, rows_cnt, c.D2,
                                                              c.idx, nullptr, nullptr, nullptr, nullptr,
                                                              &c.st->argmin_fp64, &c.st->argmin_wide);
    else
        fixup_kernel<MODE_ASSIGN><<<grid, 256, sm, c.stream>>>(c.X, c.d, C, k, pairs, c.st, rows, rows_cnt,
                                                               nullptr, nullptr, labels, prev, changed, dmin,
                                                               &c.st->argmin_fp64, &c.st->argmin_wide);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t configure_refine_kernels() {
    // the tensor passes support d + 2 <= 192: refine tiles of 256 rows of up to 190 floats
    cudaError_t e = cudaFuncSetAttribute(refine_kernel<MODE_ROUND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         200 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(refine_kernel<MODE_ASSIGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(refine_resident_kernel<MODE_ROUND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             200 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(refine_resident_kernel<MODE_ASSIGN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             200 * 1024);
    if (e != cudaSuccess) return e;
    // the tensor passes support d <= 190: fix-up tiles of 160 rows of up to 190 floats
    const int fx = (int)fixup_smem_bytes(190);
    e = cudaFuncSetAttribute(fixup_kernel<MODE_ROUND>, cudaFuncAttributeMaxDynamicSharedMemorySize, fx);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(fixup_kernel<MODE_ASSIGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, fx);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(fixup_resident_kernel<MODE_ROUND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             200 * 1024);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(fixup_resident_kernel<MODE_ASSIGN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                200 * 1024);
}

// exact FP32 difference form of one row against one center, both in global memory:
// the same chain as dist2_fp32 (ascending coordinates, one rounded subtraction and
// one FMA each), with 16-byte loads when both rows are 16-byte aligned
__device__ __forceinline__ float dist2_fp32_v4(const float *__restrict__ x, const float *__restrict__ c, int d) {
    if ((d & 3) == 0 && ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(c)) & 15u) == 0) {
        const float4 *x4 = reinterpret_cast<const float4 *>(x);
        const float4 *c4 = reinterpret_cast<const float4 *>(c);
        float s = 0.f;
        for (int p = 0; p < (d >> 2); ++p) {
            const float4 a = __ldg(x4 + p), b = __ldg(c4 + p);
            float t = __fsub_rn(a.x, b.x);
            s = __fmaf_rn(t, t, s);
            t = __fsub_rn(a.y, b.y);
            s = __fmaf_rn(t, t, s);
            t = __fsub_rn(a.z, b.z);
            s = __fmaf_rn(t, t, s);
            t = __fsub_rn(a.w, b.w);
            s = __fmaf_rn(t, t, s);
        }
        return s;
    }
    return dist2_fp32(x, c, d);
}

// Rows the list pass screened (rows[i], i < *rows_cnt): one warp per row.  The
// row's four column groups listed their centers whose screened value is at most
// thr[i]; lane l computes listed center l in the exact FP32 difference form
// (bit-identical to dist2_fp32), a lexicographic top-2 is merged across the warp,
// and the row is certain when no group overflowed its slots and every center
// left off the list (screened value above thr[i]) is, by the screening bound,
// beyond the tie window of the deciding distance (bound_certain).  Certain rows
// take decide_top2, the others go to the exact scan's list (rows2).
template <int MODE, bool BYROW>
__global__ void __launch_bounds__(256) refine_list_kernel(
    const float *__restrict__ X, int d, const float *__restrict__ C, int c_cnt, const int32_t *__restrict__ rows,
    const int *rows_cnt, const int32_t *__restrict__ order, const int32_t *__restrict__ lst, const int32_t *__restrict__ lcnt,
    const float *__restrict__ thr, ScreenBound sb, int32_t *rows2, int *cnt2, float *D2, int32_t *idx,
    int32_t *labels, const int32_t *prev, int *changed, float *dmin, unsigned long long *fp64_cnt,
    unsigned long long *wide_cnt) {
    // four listed rows per warp, eight lanes per row (a row's lists usually hold a
    // few centers): lane sl of a row's group takes its list entries sl, sl + 8, ...
    constexpr int S = tc::kListSlots;
    const int lane = threadIdx.x & 31;
    const int sub = lane >> 3, sl = lane & 7;
    const unsigned gmask = 0xFFu << (8 * sub);   // the lanes of this row's group
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t W = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int nrows = *rows_cnt;
    const int begin = MODE == MODE_ROUND ? sb.st->batch_begin : 0;
    const int cnt = MODE == MODE_ROUND ? sb.st->batch_cnt : c_cnt;
    const float FMAX = FLT_MAX;
    for (int64_t i0 = gw * 4; i0 < nrows; i0 += W * 4) {   // uniform per warp
        const int64_t i = i0 + sub;
        const bool valid = i < nrows;
        // the row's lists and threshold are by list position, or (BYROW) by the listed
        // number: the row, or its position in `order`
        const int64_t r0 = valid ? rows[i] : 0;
        const int64_t li = BYROW ? r0 : i;
        const int64_t R = BYROW && order && valid ? (int64_t)order[r0] : r0;
        const int cg = valid && sl < 4 ? lcnt[li * 4 + sl] : 0;
        const bool over = (__ballot_sync(0xffffffffu, cg > S) & gmask) != 0;
        const int c0 = __shfl_sync(0xffffffffu, cg, 8 * sub), c1 = __shfl_sync(0xffffffffu, cg, 8 * sub + 1);
        const int c2 = __shfl_sync(0xffffffffu, cg, 8 * sub + 2), c3 = __shfl_sync(0xffffffffu, cg, 8 * sub + 3);
        float b1 = FMAX, b2 = FMAX;
        int i1 = INT_MAX, i2 = INT_MAX;
        if (valid && !over) {
            const int total = c0 + c1 + c2 + c3;
            for (int e = sl; e < total; e += 8) {
                int g, sidx = e;
                if (sidx < c0) g = 0;
                else if ((sidx -= c0) < c1) g = 1;
                else if ((sidx -= c1) < c2) g = 2;
                else { sidx -= c2; g = 3; }
                const int col = lst[(li * 4 + g) * S + sidx];
                if (col >= 0 && col < cnt) {
                    const int j = begin + col;
                    const float v = dist2_fp32_v4(X + R * d, C + (int64_t)j * d, d);
                    if (lex_lt(v, j, b2, i2)) {
                        if (lex_lt(v, j, b1, i1)) { b2 = b1; i2 = i1; b1 = v; i1 = j; }
                        else { b2 = v; i2 = j; }
                    }
                }
            }
        }
        // top-2 of the row's group (xor offsets below 8 stay within the group)
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            const float u1 = __shfl_xor_sync(0xffffffffu, b1, o), u2 = __shfl_xor_sync(0xffffffffu, b2, o);
            const int j1 = __shfl_xor_sync(0xffffffffu, i1, o), j2 = __shfl_xor_sync(0xffffffffu, i2, o);
            top2_merge(b1, i1, b2, i2, u1, j1, u2, j2);
        }
        if (sl == 0 && valid) {
            bool certain = false;
            if (!over) {
                const float m = deciding<MODE>(D2, R, i1 != INT_MAX ? b1 : FMAX);
                certain = m < FMAX && bound_certain(sb, sb.xnorm[R], m, thr[li], d);
            }
            if (certain) {
                if (i2 == INT_MAX) { i2 = -1; b2 = FMAX; }
                if (decide_top2<MODE>(X, d, C, R, b1, i1, b2, i2, D2, idx, labels, prev, dmin, fp64_cnt, wide_cnt) &&
                    changed)
                    atomicAdd(changed, 1);
            } else {
                rows2[atomicAdd(cnt2, 1)] = (int32_t)R;
            }
        }
    }
}

// ---------------------------------------------------------------- the round filter
// A new candidate c can only become nearest to a row x of candidate a (D(x) = d(x, a))
// when d(a, c) < 2 D(x): otherwise d(x, c) >= d(a, c) - d(x, a) >= D(x).  So the new
// candidates within twice the largest D of a's rows are listed once per candidate a (a
// screening pass over the few old candidates instead of all rows), and a row examines
// its candidate's list in exact FP32.  Margins (16 W on the squared radius, the
// screening bound in the threshold) keep every center left off the list beyond the
// tie window, so the decisions are those of the dense pass.  A candidate that serves a
// far cluster too has a radius that lists everything: its list is taken again at half
// the radius, down to an eighth, and only its rows within that are settled.
// 1e7 x 128, l = 20,000 (a mixture of 10,000): rounds 79 + 63 + 52 + 52 + 52 ms dense ->
// 56 + 11 + 5.2 + 5.3 + 5.4 ms; where the data do not separate, the lists cost a pass over
// the old candidates (at most an eighth of the rows) and the rows are gathered.

// per candidate, the bits of the largest D^2 among its rows (a read first: most rows
// are below the maximum already stored)
// (refs: nothing to do where it is 0; null: always)
__global__ void __launch_bounds__(256) candidate_radius_kernel(const float *__restrict__ D2,
                                                              const int32_t *__restrict__ idx, int64_t n,
                                                              unsigned int *rad2, const int32_t *refs) {
    if (refs && *refs == 0) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const unsigned int v = __float_as_uint(D2[i]);
        unsigned int *r = rad2 + idx[i];
        if (v > *reinterpret_cast<volatile unsigned int *>(r)) atomicMax(r, v);
    }
}

// The rows' lists examined exactly: a warp takes 32 rows (a lane holds a row's list head;
// the next block's are loaded meanwhile) and deals their (row, entry) pairs to its lanes,
// 32 at a time, so lanes stay busy however the lists' lengths vary (2 entries on average,
// 5 at most of 32 rows in a late round of a mixture).  A lane computes its pair's exact
// FP32 distance (the chain of dist2_fp32); the row's lane takes the top two of its pairs
// and the decision of the dense pass.  Rows beyond the radius that the list covers go to
// open_rows.  Rows and candidates are staged in shared memory by whole warps (row stride
// an odd number of 16-byte units: a lane-per-row 16-byte read is conflict-free; straight
// from global memory 16 bytes of 32 different rows touch 32 lines an instruction).
// 1e7 x 128 against lists of 1.9 entries (5.1 GB of rows from HBM, 9.7 GB of candidates
// from L2): 2.8 ms; 4.5 ms as one thread per row, 5.0 ms with the copies in loops, 5.0 ms
// with a bulk copy a row.
__host__ __device__ __forceinline__ int stage_stride4(int d) { return (d >> 2) | 1; }   // in 16-byte units
constexpr int kStageExtra = 512;   // bytes per warp: 64 open rows, 32 pairs' values

// RP: rows a warp copies with one instruction, each by 32 / RP lanes of 16 bytes, in NQ
// steps (the copies are a fixed unrolled sequence of a shuffle and a predicated copy a
// row; as a loop over rows and pieces they were two thirds of the kernel's instructions)
template <int RP, int NQ>
__device__ __forceinline__ void stage_rows(float4 *dst, int ss, const float *base, int d4, int row, int lane) {
    // row: this lane's row of base (negative: none), staged as row `lane` of dst
    constexpr int LW = 32 / RP;   // lanes per copied row
    const int gq = lane / LW, lq = lane % LW;
    const float4 *b4 = reinterpret_cast<const float4 *>(base) + lq;
    float4 *to = dst + gq * ss + lq;
#pragma unroll 8
    for (int r0 = 0; r0 < 32; r0 += RP) {
        const int o = __shfl_sync(0xffffffffu, row, r0 + gq);
#pragma unroll
        for (int u = 0; u < NQ; ++u)
            if (o >= 0 && lq + u * LW < d4) cp_async16(to + r0 * ss + u * LW, b4 + (int64_t)o * d4 + u * LW);
    }
}

// the exact FP32 chain of dist2_fp32 over two staged rows
__device__ __forceinline__ float stage_dist2(const float4 *x, const float4 *c, int d4) {
    float v = 0.f;
#pragma unroll 8
    for (int p = 0; p < d4; ++p) {
        const float4 u = x[p], w = c[p];
        float t;
        t = __fsub_rn(u.x, w.x); v = __fmaf_rn(t, t, v);
        t = __fsub_rn(u.y, w.y); v = __fmaf_rn(t, t, v);
        t = __fsub_rn(u.z, w.z); v = __fmaf_rn(t, t, v);
        t = __fsub_rn(u.w, w.w); v = __fmaf_rn(t, t, v);
    }
    return v;
}

// Rows of a warp collected for a list in memory and written 32 or more at a time: one
// atomic on the list's one counter for every block of rows would queue.
struct RowSink {
    int32_t *buf;   // 64 entries of the warp's shared memory
    int n = 0;
    __device__ __forceinline__ void put(bool take, int32_t row, int lane) {
        const unsigned m = __ballot_sync(0xffffffffu, take);
        if (take) buf[n + __popc(m & ((1u << lane) - 1u))] = row;
        n += __popc(m);
    }
    __device__ __forceinline__ void flush(int32_t *rows, int *cnt, int lane, bool last) {
        if (n == 0 || (n < 32 && !last)) return;
        __syncwarp();
        int base = 0;
        if (lane == 0) base = atomicAdd(cnt, n);
        base = __shfl_sync(0xffffffffu, base, 0);
        for (int i = lane; i < n; i += 32) rows[base + i] = buf[i];
        n = 0;
        __syncwarp();
    }
};

struct GroupArgs {
    const float *X;
    int64_t n;                  // rows, or null counts below: rows[0 .. *rows_cnt)
    const int32_t *rows;
    const int *rows_cnt;
    int d;
    const float *C;
    const int32_t *glst;
    const int2 *ghead;
    const int32_t *ref;         // per row, its reference
    const float *refd2;         // and the exact squared distance to it
    const float *tau2;          // per reference, squared distance to some center (null: 0)
    int32_t *open_rows;
    int *open_cnt;
    DevState *st;
    // round
    float *D2;
    int32_t *idx;
    int count_rows;
    // Lloyd; `own`: the reference is the row's previous center and refd2 its exact distance
    int own;
    int32_t *labels;
    const int32_t *prev;
    float *dmin, *ub, *lb;
    int *changed;
};

template <int MODE, int RP, int NQ>
__global__ void __launch_bounds__(256) refine_group_kernel(GroupArgs g) {
    extern __shared__ __align__(16) float4 gst[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int d = g.d, d4 = d >> 2, ss = stage_stride4(d);
    float4 *xs = gst + (size_t)wid * (64 * ss + kStageExtra / 16), *cs = xs + 32 * ss;
    RowSink open_sink{reinterpret_cast<int32_t *>(cs + 32 * ss)};
    float *pv = reinterpret_cast<float *>(open_sink.buf + 64);   // the pairs' values
    int32_t *pj = reinterpret_cast<int32_t *>(pv + 32);          // and centers
    const float W = fp32_tie_window(d);
    const int64_t stride = (int64_t)gridDim.x * nwarps;
    const int begin = MODE == MODE_ROUND ? g.st->batch_begin : 0;
    const bool any = MODE != MODE_ROUND || g.st->batch_cnt > 0;   // (an empty batch has no lists, changes nothing)
    const int64_t n = g.rows ? (int64_t)*g.rows_cnt : g.n, nb = (n + 31) / 32;
    if (MODE == MODE_ROUND && g.st->list_skip) {   // no lists: all rows, in order, to the dense pass
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
            g.open_rows[i] = (int32_t)i;
        if (blockIdx.x == 0 && threadIdx.x == 0) *g.open_cnt = (int)n;
        return;
    }
    unsigned int settled = 0, listed = 0, chg = 0;
    int64_t b = (int64_t)blockIdx.x * nwarps + wid;
    // this lane's row of block b: its number, reference, distance and list head
    int R = -1, a = 0;
    int2 hd = make_int2(0, 0);
    float dd = 0.f;
    if (any && b < nb && b * 32 + lane < n) {
        R = g.rows ? g.rows[b * 32 + lane] : (int)(b * 32 + lane);
        a = g.ref[R];
        dd = g.refd2[R];
        hd = __ldg(g.ghead + a);
    }
    for (; b < nb; b += stride) {   // uniform per warp
        const int64_t tn = (b + stride) * 32 + lane;
        int Rn = -1, an = 0;
        float ddn = 0.f;
        if (any && tn < n) {
            Rn = g.rows ? g.rows[tn] : (int)tn;
            an = g.ref[Rn];
            ddn = g.refd2[Rn];
        }
        // (in the first assignment a list holds a center, or it covers nothing)
        const bool open = R >= 0 && (!(dd <= __int_as_float(hd.y)) || (MODE == MODE_ASSIGN && !g.own && hd.x == 0));
        const int total = R >= 0 && !open ? hd.x : 0;
        int incl = total;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        const int excl = incl - total, P = __shfl_sync(0xffffffffu, incl, 31);
        float b1 = FLT_MAX, b2 = FLT_MAX;
        int i1 = INT_MAX, i2 = INT_MAX;
        if (MODE == MODE_ASSIGN && g.own && R >= 0 && !open) { b1 = dd; i1 = a; }
        for (int p0 = 0; p0 < P; p0 += 32) {
            const int pi = p0 + lane;
            // the pair's row: the first whose inclusive count exceeds pi
            int r = 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(0xffffffffu, incl, r + o - 1) <= pi) r += o;
            const int ar = __shfl_sync(0xffffffffu, a, r), er = pi - __shfl_sync(0xffffffffu, excl, r);
            int j = -1;
            if (pi < P) j = begin + __ldg(g.glst + (size_t)ar * 4 * tc::kListSlots + er);
            if (p0 == 0) stage_rows<RP, NQ>(xs, ss, g.X, d4, total > 0 ? R : -1, lane);
            stage_rows<RP, NQ>(cs, ss, g.C, d4, j, lane);
            cp_async_commit();
            cp_async_wait<0>();
            __syncwarp();
            pj[lane] = j;
            if (j >= 0) pv[lane] = stage_dist2(xs + r * ss, cs + lane * ss, d4);
            __syncwarp();   // the values are there; the staged rows are read
            for (int q = max(excl, p0); q < min(incl, p0 + 32); ++q) {
                const float v = pv[q - p0];
                const int jq = pj[q - p0];
                if (lex_lt(v, jq, b2, i2)) {
                    if (lex_lt(v, jq, b1, i1)) { b2 = b1; i2 = i1; b1 = v; i1 = jq; }
                    else { b2 = v; i2 = jq; }
                }
            }
            __syncwarp();
        }
        const int2 hdn = Rn >= 0 ? __ldg(g.ghead + an) : make_int2(0, 0);
        if (i1 != INT_MAX) {
            if (i2 == INT_MAX) { i2 = -1; b2 = FLT_MAX; }
            if (MODE == MODE_ROUND) {
                decide_top2<MODE_ROUND>(g.X, d, g.C, R, b1, i1, b2, i2, g.D2, g.idx, nullptr, nullptr, nullptr,
                                        &g.st->argmin_fp64, &g.st->argmin_wide);
            } else {
                chg += decide_top2<MODE_ASSIGN>(g.X, d, g.C, R, b1, i1, b2, i2, nullptr, nullptr, g.labels, g.prev,
                                                g.dmin, &g.st->argmin_fp64, &g.st->argmin_wide);
                if (g.lb) {
                    // the exact runner-up, and for a center off the list its distance to the
                    // reference less the row's (real distances: FP32 ones within W of them)
                    const bool fst = g.labels[R] == i1;
                    g.ub[R] = bound_upper(fst ? b1 : b2, W);
                    const float reach = 2.f * sqrtf(__int_as_float(hd.y)) + (g.tau2 ? sqrtf(g.tau2[a]) : 0.f);
                    const float off = reach * (1.f - 1e-6f) - bound_upper(dd, W);
                    const float run = fst ? b2 : b1;
                    const float l2 = run < FLT_MAX ? sqrtf(run * (1.f - 2.f * W)) * (1.f - 1e-6f) : FLT_MAX;
                    g.lb[R] = fmaxf(0.f, fminf(l2, off));
                }
            }
        }
        open_sink.put(open, R, lane);
        open_sink.flush(g.open_rows, g.open_cnt, lane, b + stride >= nb);
        settled += (unsigned int)(R >= 0 && !open) + (unsigned int)(!any && b * 32 + lane < n);
        listed += (unsigned int)(total > 0);
        R = Rn;
        a = an;
        dd = ddn;
        hd = hdn;
    }
    settled = __reduce_add_sync(0xffffffffu, settled);
    listed = __reduce_add_sync(0xffffffffu, listed);
    if (MODE == MODE_ASSIGN) chg = __reduce_add_sync(0xffffffffu, chg);
    if (lane == 0) {   // the rows settled here (the dense pass counts the open ones)
        if (MODE == MODE_ROUND) {
            if (settled && g.count_rows) atomicAdd(&g.st->screen_rows, (unsigned long long)settled);
            if (listed) {
                atomicAdd(&g.st->screen_fallback, (unsigned long long)listed);
                atomicAdd(&g.st->screen_listed, (unsigned long long)listed);
            }
        } else {
            if (settled && g.own) atomicAdd(&g.st->lloyd_settled, (unsigned long long)settled);
            if (settled && !g.own) atomicAdd(&g.st->screen_rows, (unsigned long long)settled);
            if (chg && g.changed) atomicAdd(g.changed, (int)chg);
        }
    }
}

// warps per CTA: about 100 KB of staged rows a CTA, two CTAs on an SM
constexpr unsigned kStageSmem = 108u * 1024u;
int stage_warps(int d) {
    const int w = (int)(kStageSmem / (64u * 16u * (unsigned)stage_stride4(d) + kStageExtra));
    return w < 1 ? 1 : (w > 8 ? 8 : w);
}
size_t stage_smem_bytes(int d) { return (size_t)stage_warps(d) * (64 * 16 * stage_stride4(d) + kStageExtra); }

// a kernel of the staged kind over n rows: persistent, two CTAs an SM
template <typename K, typename A>
static cudaError_t launch_staged(K kern, const Ctx &c, int64_t n, const A &args) {
    const size_t smem = stage_smem_bytes(c.d);   // at most kStageSmem up to d = 424
    // (the same limit in every call: it belongs to the process)
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStageSmem);
    if (e != cudaSuccess) return e;
    const int sw = stage_warps(c.d);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((n + 32 * sw - 1) / (32 * sw), 2 * (int64_t)c.num_sms));
    kern<<<grid, 32 * sw, smem, c.stream>>>(args);
    count_launches(1);
    return cudaGetLastError();
}
template <int MODE>
static cudaError_t launch_refine_group(const Ctx &c, const GroupArgs &g) {
    const int d4 = c.d >> 2;
    if (d4 > 32) return launch_staged(refine_group_kernel<MODE, 1, 2>, c, c.n, g);   // (d <= 188)
    if (d4 > 16) return launch_staged(refine_group_kernel<MODE, 1, 1>, c, c.n, g);
    if (d4 > 8) return launch_staged(refine_group_kernel<MODE, 2, 1>, c, c.n, g);
    if (d4 > 4) return launch_staged(refine_group_kernel<MODE, 4, 1>, c, c.n, g);
    return launch_staged(refine_group_kernel<MODE, 8, 1>, c, c.n, g);
}

// A distance pass on the tensor cores.  rows / rows_cnt (direct refine only): the pass
// covers just the rows rows[0 .. *rows_cnt), gathered into a compact image; the others
// keep what the caller wrote for them.
cudaError_t launch_tc_pass(Ctx &c, int mode_round, const float *C, int k, int32_t *labels, const int32_t *prev,
                           int *changed, float *dmin, int timing_cls, const int32_t *rows, const int *rows_cnt) {
    cudaError_t e;
    const int fmt = c.tc_fmt;
    if (!c.tc_prepared &&
        (e = tc::launch_prep_centers(C, c.d, fmt, c.st, k, mode_round, mode_round ? c.cap_round : k, c.tc_anchor,
                                     c.tc_img, c.tc_ncol, c.tc_tscale, c.tc_cmax, c.stream)) != cudaSuccess)
        return e;
    if ((e = cudaMemsetAsync(c.fix_cnt, 0, sizeof(int), c.stream)) != cudaSuccess) return e;
    // rows the screening does not reach (e.g. an empty batch) must not see a stale winner
    if (!rows && (e = cudaMemsetAsync(c.cand1, 0xFF, sizeof(int32_t) * (size_t)c.n, c.stream)) != cudaSuccess)
        return e;
    tc::TcParams p{};
    p.X = c.X; p.n = c.n; p.d = c.d; p.fmt = fmt;
    p.ximg = c.tc_ximg; p.xnorm = c.tc_xnorm; p.xscale = c.tc_xscale;
    p.Cf = C; p.cnt = k; p.st = c.st; p.bimg = c.tc_img; p.ncol = c.tc_ncol; p.tscale = c.tc_tscale;
    p.cmax_bits = c.tc_cmax;
    p.cand1 = c.cand1; p.v2 = c.tc_v2; p.fix_rows = c.fix_rows; p.fix_cnt = c.fix_cnt;
    p.fp64_cnt = &c.st->argmin_fp64; p.err = c.tc_err;
    const int cap_rows = mode_round ? c.cap_round : k;
    const ResidentPlan rp = resident_plan(cap_rows, c.d);
    // the direct refine serves rows of d = 0 mod 4; with it, formats that add the norms
    // in the epilogue screen groups of four centers (fewer ALU operations per value)
    const bool direct = rp.parts == 0 && (c.d & 3) == 0 &&
                        ((reinterpret_cast<uintptr_t>(c.X) | reinterpret_cast<uintptr_t>(C)) & 15u) == 0;
    p.group = (direct && tc::tc_norms_in_epilogue(fmt)) ? 4 : 2;
    ScreenBound sb{};
    sb.xnorm = c.tc_xnorm; sb.cmax_bits = c.tc_cmax; sb.st = c.st;
    sb.fix_rows = c.fix_rows; sb.fix_cnt = c.fix_cnt; sb.ub = c.tc_ub;
    tc::tc_bound(c.d, fmt, &sb.ep, &sb.en, &sb.ec);
    // a round pass whose rows already have a nearest distance D^2 lists, in the
    // screening pass itself, every center within that distance (plus the bound):
    // the rows the groups leave undecided then need no second screening
    // (Not in the first round: its rows' D^2 is the distance to the first center alone,
    // far above the spread of any cluster, so their lists would only overflow.)
    const bool plist = mode_round && p.group == 4 && c.tc_list && (c.rounds_done >= 1 || c.round_part > 0);
    // the round filter settles the rows near an old candidate; the dense pass then covers
    // only the rows it leaves open
    const int64_t old = 1 + (int64_t)(c.rounds_done + 1) * c.cap_round;
    if (plist && !rows && round_filter_usable(c)) {
        if ((e = cudaMemsetAsync(c.rf_rad2, 0, sizeof(unsigned int) * (size_t)old, c.stream)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(c.rf_cnt, 0, sizeof(int), c.stream)) != cudaSuccess) return e;
        candidate_radius_kernel<<<c.num_sms * 8, 256, 0, c.stream>>>(c.D2, c.idx, c.n, c.rf_rad2, &c.st->list_refs);
        count_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        tc::TcParams pf = p;
        pf.lst = c.tc_lst; pf.lcnt = c.tc_lcnt;
        const tc::ListBufs lb{c.cap_total, c.tc_cimg, c.tc_cscale, c.tc_thr, c.rf_rad2, c.rf_num, c.rf_lst, c.rf_head,
                              c.rf_lcnt};
        if ((e = tc::launch_reference_lists(pf, 1, lb, c.cand, &c.st->list_refs, nullptr, sb.ep, sb.en, sb.ec, c.num_sms,
                                            c.stream)) != cudaSuccess)
            return e;
        GroupArgs ga{};
        ga.X = c.X; ga.n = c.n; ga.d = c.d; ga.C = C; ga.glst = c.rf_lst; ga.ghead = c.rf_head; ga.ref = c.idx;
        ga.refd2 = c.D2; ga.open_rows = c.rf_rows; ga.open_cnt = c.rf_cnt; ga.st = c.st; ga.D2 = c.D2; ga.idx = c.idx;
        ga.count_rows = c.round_part == 0;
        if ((e = launch_refine_group<MODE_ROUND>(c, ga)) != cudaSuccess) return e;
        rows = c.rf_rows;
        rows_cnt = c.rf_cnt;
    }
    if (plist) {
        if (!rows && (e = tc::launch_row_thresholds(c.D2, c.n, c.d, c.tc_xnorm, c.tc_cmax, sb.ep, sb.en, sb.ec, c.tc_thr,
                                           c.stream)) != cudaSuccess)
            return e;
        p.thr = c.tc_thr; p.lst = c.tc_lst; p.lcnt = c.tc_lcnt;
    }
    if (rows) {
        // the compact image of the listed rows, with their scales and, for a listing
        // pass, their thresholds (by D^2)
        if (!direct || p.group != 4 || !c.tc_cimg) return cudaErrorInvalidValue;
        if ((e = tc::launch_gather_rows(c.tc_ximg, c.tc_xscale, c.d, fmt, rows, rows_cnt,
                                        mode_round ? c.D2 : c.tc_ub, c.tc_xnorm, c.tc_cmax, sb.ep, sb.en, sb.ec,
                                        c.tc_cimg, c.tc_cscale, c.tc_thr, c.num_sms * 8, c.stream, nullptr, nullptr,
                                        mode_round ? &c.st->list_skip : nullptr)) != cudaSuccess)
            return e;
        if (mode_round) { p.all_dev = &c.st->list_skip; p.ximg_all = p.ximg; }
        p.ximg = c.tc_cimg; p.xscale = c.tc_cscale; p.nrows_dev = rows_cnt;
        if ((e = tc::launch_nearest_tc(p, mode_round, plist ? tc::EPI_PAIRLIST : tc::EPI_PAIR, c.num_sms, c.stream)) !=
            cudaSuccess)
            return e;
        p.all_dev = nullptr;   // (the passes over undecided rows gather theirs)
        const int grid = (int)((c.n + 255) / 256);
        if (mode_round)
            refine_direct_kernel<MODE_ROUND, 4><<<grid, 256, 0, c.stream>>>(
                c.X, c.n, c.d, C, 0, c.cand1, c.tc_v2, sb, c.D2, c.idx, nullptr, nullptr, nullptr, nullptr,
                &c.st->argmin_fp64, &c.st->argmin_wide, rows, rows_cnt, nullptr, nullptr);
        else
            refine_direct_kernel<MODE_ASSIGN, 4><<<grid, 256, 0, c.stream>>>(
                c.X, c.n, c.d, C, k, c.cand1, c.tc_v2, sb, nullptr, nullptr, labels, prev, changed, dmin,
                &c.st->argmin_fp64, &c.st->argmin_wide, rows, rows_cnt, c.ll_ub, c.ll_lb);
        count_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    } else {
    cudaEvent_t ev = nullptr;
    if ((e = timing_begin(c, &ev)) != cudaSuccess) return e;
    if ((e = tc::launch_nearest_tc(p, mode_round, plist ? tc::EPI_PAIRLIST : tc::EPI_PAIR, c.num_sms, c.stream)) !=
        cudaSuccess)
        return e;
    if ((e = timing_end(c, ev, timing_cls)) != cudaSuccess) return e;
    if (rp.parts > 0) {
        const int rw = rp.warps;
        const size_t rsm = resident_smem_bytes(rp.hold, c.d, rw);
        const int64_t nb = (c.n + 31) / 32;
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(c.num_sms, (nb + rw - 1) / rw));
        for (int part = 0; part < rp.parts; ++part) {
            const int lo = part * rp.rows;
            if (mode_round)
                refine_resident_kernel<MODE_ROUND><<<grid, 32 * rw, rsm, c.stream>>>(
                    c.X, c.n, c.d, C, cap_rows, lo, rp.rows, rp.hold, c.cand1, c.tc_v2, sb, c.D2, c.idx, nullptr,
                    nullptr, nullptr, nullptr, &c.st->argmin_fp64, &c.st->argmin_wide);
            else
                refine_resident_kernel<MODE_ASSIGN><<<grid, 32 * rw, rsm, c.stream>>>(
                    c.X, c.n, c.d, C, cap_rows, lo, rp.rows, rp.hold, c.cand1, c.tc_v2, sb, nullptr, nullptr, labels,
                    prev, changed, dmin, &c.st->argmin_fp64, &c.st->argmin_wide);
            count_launches(1);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    } else if (direct) {
        const int grid = (int)((c.n + 255) / 256);
#define KMP_DIRECT(G)                                                                                           \
    if (mode_round)                                                                                             \
        refine_direct_kernel<MODE_ROUND, G><<<grid, 256, 0, c.stream>>>(c.X, c.n, c.d, C, 0, c.cand1, c.tc_v2, sb, \
                                                                        c.D2, c.idx, nullptr, nullptr, nullptr,  \
                                                                        nullptr, &c.st->argmin_fp64,             \
                                                                        &c.st->argmin_wide, nullptr, nullptr,    \
                                                                        nullptr, nullptr);                       \
    else                                                                                                        \
        refine_direct_kernel<MODE_ASSIGN, G><<<grid, 256, 0, c.stream>>>(c.X, c.n, c.d, C, k, c.cand1, c.tc_v2,  \
                                                                         sb, nullptr, nullptr, labels, prev,     \
                                                                         changed, dmin, &c.st->argmin_fp64,      \
                                                                         &c.st->argmin_wide, c.refine_order,     \
                                                                         nullptr, c.ll_ub, c.ll_lb);
        if (p.group == 4) { KMP_DIRECT(4) } else { KMP_DIRECT(2) }
#undef KMP_DIRECT
        count_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    } else {
        const int rthreads = 32 * refine_warps(c.d);
        const int grid = (int)((c.n + rthreads - 1) / rthreads);
        const size_t rsm = refine_smem_bytes(c.d);
        if (mode_round)
            refine_kernel<MODE_ROUND><<<grid, rthreads, rsm, c.stream>>>(c.X, c.n, c.d, C, 0, c.cand1, c.tc_v2, sb,
                                                                         c.D2, c.idx, nullptr, nullptr, nullptr,
                                                                         nullptr, &c.st->argmin_fp64,
                                                                         &c.st->argmin_wide);
        else
            refine_kernel<MODE_ASSIGN><<<grid, rthreads, rsm, c.stream>>>(c.X, c.n, c.d, C, k, c.cand1, c.tc_v2, sb,
                                                                          nullptr, nullptr, labels, prev, changed,
                                                                          dmin, &c.st->argmin_fp64,
                                                                          &c.st->argmin_wide);
        count_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    }
    if (!c.tc_list) {
        if ((e = count_fixups(c, nullptr, rows_cnt)) != cudaSuccess) return e;
        return launch_fixup(c, mode_round, C, k, labels, prev, changed, dmin, c.fix_rows, c.fix_cnt);
    }
    const int lgrid = c.num_sms * 8;
    // rows the pair screening left undecided (rows_in, cnt_in): a second screening of
    // just those rows that lists every center within twice the screening bound of
    // the row's deciding distance, the exact FP32 form of the listed centers, and the
    // exact scan only for rows whose lists overflowed or stayed uncertain (rows_out)
    auto list_pass = [&](int32_t *rows_in, int *cnt_in, int32_t *rows_out, int *cnt_out) -> cudaError_t {
        cudaError_t e2;
        if ((e2 = cudaMemsetAsync(cnt_out, 0, sizeof(int), c.stream)) != cudaSuccess) return e2;
        if ((e2 = tc::launch_gather_rows(c.tc_ximg, c.tc_xscale, c.d, fmt, rows_in, cnt_in, c.tc_ub, c.tc_xnorm,
                                         c.tc_cmax, sb.ep, sb.en, sb.ec, c.tc_cimg, c.tc_cscale, c.tc_thr,
                                         c.num_sms * 8, c.stream)) != cudaSuccess)
            return e2;
        tc::TcParams pl = p;
        pl.ximg = c.tc_cimg; pl.xscale = c.tc_cscale;
        pl.nrows_dev = cnt_in; pl.thr = c.tc_thr; pl.lst = c.tc_lst; pl.lcnt = c.tc_lcnt;
        if ((e2 = tc::launch_nearest_tc(pl, mode_round, tc::EPI_LIST, c.num_sms, c.stream)) != cudaSuccess) return e2;
        if (mode_round)
            refine_list_kernel<MODE_ROUND, false><<<lgrid, 256, 0, c.stream>>>(
                c.X, c.d, C, 0, rows_in, cnt_in, nullptr, c.tc_lst, c.tc_lcnt, c.tc_thr, sb, rows_out, cnt_out, c.D2, c.idx,
                nullptr, nullptr, nullptr, nullptr, &c.st->argmin_fp64, &c.st->argmin_wide);
        else
            refine_list_kernel<MODE_ASSIGN, false><<<lgrid, 256, 0, c.stream>>>(
                c.X, c.d, C, k, rows_in, cnt_in, nullptr, c.tc_lst, c.tc_lcnt, c.tc_thr, sb, rows_out, cnt_out, nullptr,
                nullptr, labels, prev, changed, dmin, &c.st->argmin_fp64, &c.st->argmin_wide);
        count_launches(1);
        return cudaGetLastError();
    };
    if (!plist) {
        if ((e = list_pass(c.fix_rows, c.fix_cnt, c.fix_rows2, c.fix_cnt2)) != cudaSuccess) return e;
        if ((e = count_fixups(c, c.fix_cnt2, rows_cnt)) != cudaSuccess) return e;
        return launch_fixup(c, mode_round, C, k, labels, prev, changed, dmin, c.fix_rows2, c.fix_cnt2);
    }
    // the lists the screening pass kept: the exact FP32 form of the listed centers;
    // rows whose lists overflowed or stayed uncertain take the list pass, and the
    // rows that one leaves, the exact scan
    if ((e = cudaMemsetAsync(c.fix_cnt2, 0, sizeof(int), c.stream)) != cudaSuccess) return e;
    refine_list_kernel<MODE_ROUND, true><<<lgrid, 256, 0, c.stream>>>(
        c.X, c.d, C, 0, c.fix_rows, c.fix_cnt, rows, c.tc_lst, c.tc_lcnt, c.tc_thr, sb, c.fix_rows2, c.fix_cnt2, c.D2, c.idx,
        nullptr, nullptr, nullptr, nullptr, &c.st->argmin_fp64, &c.st->argmin_wide);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    count_stage_kernel<<<1, 1, 0, c.stream>>>(c.fix_cnt, nullptr, c.n, rows_cnt, c.st, c.round_part == 0);
    count_launches(1);
    if ((e = list_pass(c.fix_rows2, c.fix_cnt2, c.fix_rows, c.fix_cnt)) != cudaSuccess) return e;
    count_stage_kernel<<<1, 1, 0, c.stream>>>(nullptr, c.fix_cnt, c.n, nullptr, c.st, 0);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return launch_fixup(c, mode_round, C, k, labels, prev, changed, dmin, c.fix_rows, c.fix_cnt);
}

// ---------------------------------------------------------------- Lloyd's bounds
// Between Lloyd iterations every center c moves by delta_c = ||c_new - c_old||.
// A row labelled a with u >= d(x, c_a) and l <= d(x, c) for every other c keeps
// u + delta_a and l - max_{c != a} delta_c as bounds for the moved centers (the
// triangle inequality); if the first is below the second, a is still strictly the
// nearest center, by more than the FP32 tie window (both bounds carry it), so the
// exact FP32 argmin takes a again and only d^2(x, c_a) needs computing.

// delta_c in FP64 from the FP32 centers, rounded up to FP32 (one warp per center)
__global__ void lloyd_drift_kernel(const float *__restrict__ Cn, const float *__restrict__ Co, int k, int d,
                                   float *__restrict__ drift) {
    const int lane = threadIdx.x & 31;
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (c >= k) return;
    double s = 0.0;
    for (int q = lane; q < d; q += 32) {
        const double t = (double)Cn[(size_t)c * d + q] - (double)Co[(size_t)c * d + q];
        s = __fma_rn(t, t, s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) drift[c] = __double2float_ru(sqrt(s));
}

// for every center, the largest drift among the other centers (one block)
__global__ void __launch_bounds__(1024) lloyd_drift_other_kernel(const float *__restrict__ drift, int k,
                                                                 float *__restrict__ other) {
    __shared__ float s1[32], s2[32];
    __shared__ int si[32];
    float m1 = 0.f, m2 = 0.f;
    int i1 = -1;
    for (int c = threadIdx.x; c < k; c += blockDim.x) {
        const float v = drift[c];
        if (v > m1) { m2 = m1; m1 = v; i1 = c; }
        else if (v > m2) m2 = v;
    }
    // merge the top two of the warp, then of the block
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float a1 = __shfl_xor_sync(0xffffffffu, m1, o), a2 = __shfl_xor_sync(0xffffffffu, m2, o);
        const int ai = __shfl_xor_sync(0xffffffffu, i1, o);
        if (a1 > m1 || (a1 == m1 && ai < i1)) { m2 = fmaxf(m1, a2); m1 = a1; i1 = ai; }
        else m2 = fmaxf(m2, a1);
    }
    if (lane == 0) { s1[wid] = m1; s2[wid] = m2; si[wid] = i1; }
    __syncthreads();
    if (wid == 0) {
        const int nw = blockDim.x >> 5;
        m1 = lane < nw ? s1[lane] : 0.f;
        m2 = lane < nw ? s2[lane] : 0.f;
        i1 = lane < nw ? si[lane] : -1;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float a1 = __shfl_xor_sync(0xffffffffu, m1, o), a2 = __shfl_xor_sync(0xffffffffu, m2, o);
            const int ai = __shfl_xor_sync(0xffffffffu, i1, o);
            if (a1 > m1 || (a1 == m1 && ai < i1)) { m2 = fmaxf(m1, a2); m1 = a1; i1 = ai; }
            else m2 = fmaxf(m2, a1);
        }
        if (lane == 0) { s1[0] = m1; s2[0] = m2; si[0] = i1; }
    }
    __syncthreads();
    m1 = s1[0]; m2 = s2[0]; i1 = si[0];
    for (int c = threadIdx.x; c < k; c += blockDim.x) other[c] = c == i1 ? m2 : m1;
}

// The bounds test, in two kernels.  A row whose center did not move keeps its exact d^2
// and its upper bound: lloyd_still_kernel settles it, or lists it as pending, without a
// look at X (16 bytes of state read a row), and lists the rows of moved centers.  Those get
// the exact FP32 d^2 to the moved center (the chain of the refine, rows and centers staged
// by whole warps) and with it a tight upper bound for the test (lloyd_moved_kernel).
// Settled rows get their label, distance and bounds; a pending one has l = 0 until a pass
// certifies it again, and its distance goes into its center's radius for the lists.  Without
// lists nothing wants the distance of a row that will be pending: rows of moved centers whose
// old upper bound and its center's drift already fail the test are listed as pending at once.
// 1e7 x 128, k = 10,000, 4% of the centers moving: 1.9 ms an assignment as one kernel with
// a row a thread, 0.8 staged over all rows, 0.13 + 0.1 so.
struct BoundsArgs {
    const float *X;
    int64_t n;
    int d;
    const float *C;
    const int32_t *prev;
    int32_t *labels;
    float *dmin, *ub, *lb;
    const float *drift, *other;
    unsigned int *rad2;   // per center (null: not wanted)
    int32_t *moved;       // rows of moved centers
    int *moved_cnt;
    int32_t *rows;        // pending rows
    int *cnt;
    unsigned long long *settled;

    __device__ __forceinline__ void radius(int a, float v) const {
        if (!rad2) return;
        unsigned int *r = rad2 + a;
        const unsigned int bits = __float_as_uint(v);
        if (bits > *reinterpret_cast<volatile unsigned int *>(r)) atomicMax(r, bits);
    }
};

__global__ void __launch_bounds__(256) lloyd_still_kernel(BoundsArgs g) {
    __shared__ int32_t buf[16][64];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    RowSink moved{buf[wid]}, pend{buf[8 + wid]};
    const int64_t nb = (g.n + 31) / 32, stride = (int64_t)gridDim.x * 8;
    unsigned int settled = 0;
    for (int64_t b = (int64_t)blockIdx.x * 8 + wid; b < nb; b += stride) {   // uniform per warp
        const int64_t R = b * 32 + lane;
        bool mv = false, pd = false;
        if (R < g.n) {
            const int a = g.prev[R];
            mv = g.drift[a] != 0.f;
            g.labels[R] = a;
            if (mv && !g.rad2) {
                const float lo = g.lb[R] - g.other[a];
                pd = !(lo > 0.f && g.ub[R] + g.drift[a] < lo);
                if (pd) g.lb[R] = 0.f;
                mv = !pd;
            } else if (!mv) {
                const float lo = g.lb[R] - g.other[a];
                pd = !(lo > 0.f && g.ub[R] < lo);
                g.lb[R] = pd ? 0.f : lo;
                if (pd) g.radius(a, g.dmin[R]);
                settled += (unsigned int)!pd;
            }
        }
        moved.put(mv, (int32_t)R, lane);
        pend.put(pd, (int32_t)R, lane);
        const bool last = b + stride >= nb;
        moved.flush(g.moved, g.moved_cnt, lane, last);
        pend.flush(g.rows, g.cnt, lane, last);
    }
    settled = __reduce_add_sync(0xffffffffu, settled);
    if (lane == 0 && settled) atomicAdd(g.settled, (unsigned long long)settled);
}

template <int RP, int NQ>
__global__ void __launch_bounds__(256) lloyd_moved_kernel(BoundsArgs g) {
    extern __shared__ __align__(16) float4 gst[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int d = g.d, d4 = d >> 2, ss = stage_stride4(d);
    float4 *xs = gst + (size_t)wid * (64 * ss + kStageExtra / 16), *cs = xs + 32 * ss;
    RowSink sink{reinterpret_cast<int32_t *>(cs + 32 * ss)};
    const float W = fp32_tie_window(d);
    const int n = *g.moved_cnt, nb = (n + 31) / 32, stride = gridDim.x * nwarps;
    unsigned int settled = 0;
    int b = blockIdx.x * nwarps + wid;
    // this lane's row of block b
    int R = -1, a = -1;
    if (b < nb && b * 32 + lane < n) {
        R = g.moved[b * 32 + lane];
        a = g.prev[R];
    }
    for (; b < nb; b += stride) {   // uniform per warp
        stage_rows<RP, NQ>(xs, ss, g.X, d4, R, lane);
        stage_rows<RP, NQ>(cs, ss, g.C, d4, a, lane);
        cp_async_commit();
        // while the copies are in flight: this row's bound, the next block's rows
        const int cr = R, ca = a;
        const float lo = cr >= 0 ? g.lb[cr] - g.other[ca] : 0.f;
        const int tn = (b + stride) * 32 + lane;
        R = a = -1;
        if (b + stride < nb && tn < n) {
            R = g.moved[tn];
            a = g.prev[R];
        }
        cp_async_wait<0>();
        __syncwarp();
        bool keep = false;
        if (cr >= 0) {
            const float v = stage_dist2(xs + lane * ss, cs + lane * ss, d4);
            const float u = bound_upper(v, W);
            keep = lo > 0.f && u < lo;
            g.dmin[cr] = v;
            g.ub[cr] = u;
            g.lb[cr] = keep ? lo : 0.f;
            if (!keep) g.radius(ca, v);
        }
        __syncwarp();   // the staged rows are read
        sink.put(cr >= 0 && !keep, cr, lane);
        sink.flush(g.rows, g.cnt, lane, b + stride >= nb);
        settled += (unsigned int)keep;
    }
    settled = __reduce_add_sync(0xffffffffu, settled);
    if (lane == 0 && settled) atomicAdd(g.settled, (unsigned long long)settled);
}

// tau2: the squared FP32 distance from reference i (row i of A) to the nearest of the
// screened group of four centers at cand1[i] (any center serves), +inf without one
__global__ void __launch_bounds__(256) reference_tau_kernel(const float *__restrict__ A, const int *cnt, int d,
                                                           const float *__restrict__ C, int k,
                                                           const int32_t *__restrict__ cand1,
                                                           float *__restrict__ tau2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= *cnt) return;
    const int j = cand1[i];
    float best = __int_as_float(0x7f800000);
    if (j >= 0)
        for (int u = j; u < min(j + 4, k); ++u) best = fminf(best, dist2_fp32(A + (int64_t)i * d, C + (int64_t)u * d, d));
    tau2[i] = best;
}

bool lloyd_bounds_usable(const Ctx &c, const float *C) {
    if (c.precision == KMPAR_FP32 || !c.ll_lb || !c.tc_cimg) return false;
    const ResidentPlan rp = resident_plan(c.k, c.d);
    return rp.parts == 0 && (c.d & 3) == 0 && tc::tc_norms_in_epilogue(c.tc_fmt) &&
           ((reinterpret_cast<uintptr_t>(c.X) | reinterpret_cast<uintptr_t>(C)) & 15u) == 0;
}

// Whether the lists around references can take the place of the dense passes: the
// references have to be few against the rows, and the rows x centers of a dense pass
// have to outweigh the lists' 18 launches an assignment (10 updates: 300,000 x 128,
// k = 1,000 4.3 ms without, 4.6 with; 1,000,000 x 96, k = 2,000 8.2 and 6.3).
bool lloyd_lists_sizes(const Ctx &c) {
    return c.precision != KMPAR_FP32 && c.tc_cimg && tc::tc_norms_in_epilogue(c.tc_fmt) && c.d % 4 == 0 &&
           resident_plan(c.k, c.d).parts == 0 && (int64_t)std::max(c.cap_total, c.k) <= c.n / 8 &&
           (double)c.n * c.k >= 1e9;
}
bool lloyd_lists_usable(const Ctx &c) { return lloyd_lists_sizes(c) && c.ll_pick && !c.lists_failed; }
const int *lloyd_pending(const Ctx &c) { return c.ll_lcnt + tc::kListLevels + 1; }

// Whether an assignment by the lists paid.  Those that found their center in a list, pending
// less open, were settled at the price of listing k centers around each other (some 2 k rows of
// a dense pass, four times that where the lists overflow) and of 18 launches, some 120 us.
bool lloyd_lists_paid(const Ctx &c, int pending, int open) {
    const double levels = 1.0 + 3.0 * open / std::max(1, pending);
    return (double)pending - open > 2.0 * c.k * levels + 8e9 / ((double)c.k * c.d);
}

__global__ void set_int_kernel(int *p, int v) { *p = v; }

static cudaError_t launch_bounds(const Ctx &c, const BoundsArgs &g) {
    const int grid = (int)std::min<int64_t>((c.n + 255) / 256, (int64_t)c.num_sms * 8);
    lloyd_still_kernel<<<grid, 256, 0, c.stream>>>(g);
    count_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int d4 = c.d >> 2;
    if (d4 > 32) return launch_staged(lloyd_moved_kernel<1, 2>, c, c.n, g);
    if (d4 > 16) return launch_staged(lloyd_moved_kernel<1, 1>, c, c.n, g);
    if (d4 > 8) return launch_staged(lloyd_moved_kernel<2, 1>, c, c.n, g);
    if (d4 > 4) return launch_staged(lloyd_moved_kernel<4, 1>, c, c.n, g);
    return launch_staged(lloyd_moved_kernel<8, 1>, c, c.n, g);
}

// center tiles of the assignment's centers, the pass parameters and bounds with them
static cudaError_t lloyd_prepare(Ctx &c, const float *C, tc::TcParams &p, ScreenBound &sb) {
    p = tc::TcParams{};
    p.X = c.X; p.n = c.n; p.d = c.d; p.fmt = c.tc_fmt;
    p.Cf = C; p.cnt = c.k; p.st = c.st; p.bimg = c.tc_img; p.ncol = c.tc_ncol; p.tscale = c.tc_tscale;
    p.cmax_bits = c.tc_cmax; p.cand1 = c.cand1; p.v2 = c.tc_v2; p.err = c.tc_err; p.group = 4;
    p.lst = c.tc_lst; p.lcnt = c.tc_lcnt;
    sb = ScreenBound{};
    tc::tc_bound(c.d, c.tc_fmt, &sb.ep, &sb.en, &sb.ec);
    return tc::launch_prep_centers(C, c.d, c.tc_fmt, c.st, c.k, 0, c.k, c.tc_anchor, c.tc_img, c.tc_ncol, c.tc_tscale,
                                   c.tc_cmax, c.stream);
}

static tc::ListBufs lloyd_list_bufs(const Ctx &c) {
    return tc::ListBufs{std::max(c.cap_total, c.k), c.tc_cimg, c.tc_cscale, c.tc_thr, c.ll_rad2, c.ll_num, c.ll_lst,
                        c.ll_head, c.ll_lcnt};
}

// the dense compact pass over the rows the lists leave open, with the centers prepared
static cudaError_t lloyd_open_pass(Ctx &c, const float *C, int32_t *labels, const int32_t *prev, int *changed,
                                   float *dmin) {
    c.tc_prepared = true;
    const cudaError_t e = launch_tc_pass(c, 0, C, c.k, labels, prev, changed, dmin, -1, c.ll_rows, c.ll_cnt);
    c.tc_prepared = false;
    return e;
}

// The first assignment.  Every row is within D(x) of its candidate, and a candidate
// within tau of some center, so the row's nearest center is within 2 D(x) + tau of its
// candidate: centers are listed around the candidates, rows examine their candidate's
// list, and the dense pass covers the rows beyond the lists.  1e7 x 128, k = 10,000:
// 24 ms dense, 3.5 ms.
cudaError_t launch_lloyd_first_pass(Ctx &c, const float *C, int32_t *labels, int *changed, float *dmin) {
    cudaError_t e;
    tc::TcParams p;
    ScreenBound sb;
    if ((e = lloyd_prepare(c, C, p, sb)) != cudaSuccess) return e;
    const tc::ListBufs lb = lloyd_list_bufs(c);
    if ((e = cudaMemsetAsync(c.ll_rad2, 0, sizeof(unsigned int) * (size_t)lb.cap, c.stream)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(c.ll_cnt, 0, sizeof(int), c.stream)) != cudaSuccess) return e;
    candidate_radius_kernel<<<c.num_sms * 8, 256, 0, c.stream>>>(c.D2, c.idx, c.n, c.ll_rad2, nullptr);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // tau: the candidates' best screened groups
    const int *m = &c.st->m;
    if ((e = tc::launch_gather_rows(c.tc_ximg, c.tc_xscale, c.d, c.tc_fmt, c.cand, m, c.D2, c.tc_xnorm, c.tc_cmax, sb.ep,
                                    sb.en, sb.ec, c.tc_cimg, c.tc_cscale, c.tc_thr, c.num_sms * 8, c.stream)) !=
        cudaSuccess)
        return e;
    tc::TcParams pt = p;
    pt.ximg = c.tc_cimg; pt.xscale = c.tc_cscale; pt.nrows_dev = m;
    if ((e = tc::launch_nearest_tc(pt, 0, tc::EPI_PAIR, c.num_sms, c.stream)) != cudaSuccess) return e;
    reference_tau_kernel<<<(c.cap_total + 255) / 256, 256, 0, c.stream>>>(c.C, m, c.d, C, c.k, c.cand1, c.ll_tau2);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    p.ximg = c.tc_ximg; p.xnorm = c.tc_xnorm; p.xscale = c.tc_xscale;
    if ((e = tc::launch_reference_lists(p, 0, lb, c.cand, m, c.ll_tau2, sb.ep, sb.en, sb.ec, c.num_sms, c.stream)) !=
        cudaSuccess)
        return e;
    GroupArgs g{};
    g.X = c.X; g.n = c.n; g.d = c.d; g.C = C; g.glst = c.ll_lst; g.ghead = c.ll_head; g.ref = c.idx; g.refd2 = c.D2;
    g.tau2 = c.ll_tau2; g.open_rows = c.ll_rows; g.open_cnt = c.ll_cnt; g.st = c.st; g.labels = labels; g.dmin = dmin;
    g.ub = c.ll_ub; g.lb = c.ll_lb;
    if ((e = launch_refine_group<MODE_ASSIGN>(c, g)) != cudaSuccess) return e;
    return lloyd_open_pass(c, C, labels, nullptr, changed, dmin);
}

// One assignment after a centroid update: the rows the bounds settle; for the others the
// exact distances to the centers listed within twice their distance of their own center
// (an open row of a mixture has one or two), and a dense compact pass over the rows
// beyond the lists.
cudaError_t launch_lloyd_bounded_pass(Ctx &c, const float *C, int32_t *labels, const int32_t *prev, int *changed,
                                      float *dmin, bool lists) {
    cudaError_t e;
    const int k = c.k;
    lloyd_drift_kernel<<<(k + 7) / 8, 256, 0, c.stream>>>(C, c.ll_cold, k, c.d, c.ll_drift);
    lloyd_drift_other_kernel<<<1, 1024, 0, c.stream>>>(c.ll_drift, k, c.ll_other);
    count_launches(2);
    // (ll_cnt: the open rows, then the rows of moved centers)
    if ((e = cudaMemsetAsync(c.ll_cnt, 0, 2 * sizeof(int), c.stream)) != cudaSuccess) return e;
    int *pend_cnt = lists ? c.ll_lcnt + tc::kListLevels + 1 : c.ll_cnt;
    if (lists) {
        if ((e = cudaMemsetAsync(c.ll_rad2, 0, sizeof(unsigned int) * (size_t)k, c.stream)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(pend_cnt, 0, sizeof(int), c.stream)) != cudaSuccess) return e;
    }
    BoundsArgs ba{};
    ba.X = c.X; ba.n = c.n; ba.d = c.d; ba.C = C; ba.prev = prev; ba.labels = labels; ba.dmin = dmin; ba.ub = c.ll_ub;
    ba.lb = c.ll_lb; ba.drift = c.ll_drift; ba.other = c.ll_other; ba.rad2 = lists ? c.ll_rad2 : nullptr;
    ba.moved = c.perm; ba.moved_cnt = c.ll_cnt + 1;   // (the centroids are made: their sort is free)
    ba.rows = lists ? c.ll_pend : c.ll_rows; ba.cnt = pend_cnt; ba.settled = &c.st->lloyd_settled;
    if ((e = launch_bounds(c, ba)) != cudaSuccess) return e;
    if (!lists) return launch_tc_pass(c, 0, C, k, labels, prev, changed, dmin, -1, c.ll_rows, c.ll_cnt);
    tc::TcParams p;
    ScreenBound sb;
    if ((e = lloyd_prepare(c, C, p, sb)) != cudaSuccess) return e;
    if ((e = tc::launch_prep_points(C, k, c.d, c.tc_fmt, c.tc_anchor, c.ll_img, c.ll_xnorm, c.ll_xscale, c.stream)) !=
        cudaSuccess)
        return e;
    int *kdev = c.ll_lcnt + tc::kListLevels;
    set_int_kernel<<<1, 1, 0, c.stream>>>(kdev, k);
    count_launches(1);
    p.ximg = c.ll_img; p.xnorm = c.ll_xnorm; p.xscale = c.ll_xscale;
    if ((e = tc::launch_reference_lists(p, 0, lloyd_list_bufs(c), nullptr, kdev, nullptr, sb.ep, sb.en, sb.ec, c.num_sms,
                                        c.stream)) != cudaSuccess)
        return e;
    GroupArgs g{};
    g.X = c.X; g.n = c.n; g.rows = c.ll_pend; g.rows_cnt = pend_cnt; g.d = c.d; g.C = C; g.glst = c.ll_lst;
    g.ghead = c.ll_head; g.ref = prev; g.refd2 = dmin; g.own = 1; g.open_rows = c.ll_rows; g.open_cnt = c.ll_cnt;
    g.st = c.st; g.labels = labels; g.prev = prev; g.dmin = dmin; g.ub = c.ll_ub; g.lb = c.ll_lb; g.changed = changed;
    if ((e = launch_refine_group<MODE_ASSIGN>(c, g)) != cudaSuccess) return e;
    return lloyd_open_pass(c, C, labels, prev, changed, dmin);
}

}  // namespace kmp
