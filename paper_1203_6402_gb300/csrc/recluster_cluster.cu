// recluster_cluster.cu -- Alg. 2 step 8 (weighted k-means++, Alg. 1 with
// multiplicities, Sec. 4.2) one draw at a time in one thread-block cluster.
//
// The k draws form a chain: draw t needs D^2 to the t centers before it.  What
// bounds a draw is therefore latency, not work, and everything here is laid out to
// keep the chain short:
//   * CS CTAs of 512 threads (CS = 1, 2, 4, 8 or 16) hold the candidates' D^2 and
//     weights in shared memory and their rows as far as they fit (coordinates in
//     groups of four, one 16-byte conflict-free load per lane and group); the rest
//     of the rows comes from a transposed copy in L2, one coalesced load per group.
//   * a draw is two one-way messages over distributed shared memory, each an
//     st.async that completes an mbarrier of the receiver: every CTA's mass total
//     to every CTA, then the picked row from the owning CTA to every CTA.  No
//     cluster barrier, no fence and no poll of global memory is on the chain.
//   * masses are 96-bit integers (w D^2 in units of 2^eb): FP64 additions take 66
//     cycles here and share a pipe of two lanes per SM, an integer add with carry
//     takes a few cycles, and integer sums are exact, so they do not depend on the
//     order and every prefix is that of the definition (a mass below the unit, that
//     is below 2^-75 of the largest one, counts as one unit).
//   * a warp none of whose D^2 fell keeps its total.
// A draw over 4,933 candidates of 42 coordinates takes 2.9 us (about 5,800 cycles: 400
// masses, 1,600 totals there, 600 the owner, 400 the candidate and row out, 1,550 row
// there, 1,600 D^2); 5.9 us with cluster barriers and FP64 scans.
//
// Draw t (exchange x): warp gw = aw rank + wid (wid < aw, 16 where there are candidates for as
// many warps) owns the 32 cpw consecutive candidates from 32 cpw gw, lane l the cpw from there + l cpw, so the order of the
// prefix is lane by lane.  Warp 0 of every CTA scans its CTA's 16 warp totals, sends
// their sum to every CTA, waits for all CS sums and finds the CTA whose prefix passes
// the target u_t * total (exact integers: u_t is a multiple of 2^-53); the owner's
// warp 0 finds the warp and the candidate and sends header and row to all.
// A header can also say "masses ran out" or "new unit" (after the first draw, and
// when the largest mass has fallen by 2^16: the masses are then formed again).
//
// Buffers and barriers alternate by the parity of x: a CTA can send exchange x + 2
// only after it has received every CTA's x + 1, which is sent after all its warps are
// done with x.  Every wait is bounded; one that runs out sets the error word and
// the CTA goes to the closing cluster barrier.
#include <algorithm>
#include <atomic>

#include "kmpar_internal.cuh"

namespace kmp {

namespace {

constexpr int kRdWarps = 16;
constexpr int kRdThreads = 32 * kRdWarps;
constexpr int kRdMaxCl = 16;
constexpr int kRdSmemBudget = 224 * 1024;
constexpr unsigned long long kRdWait = 4000000000ull;   // ~2 s
constexpr int kRdUnset = 1 << 20;                        // no unit yet: every positive mass counts as 1
constexpr uint32_t kExpInf = 2000u, kExpNan = 3000u;     // "exponents" of an infinite and a NaN D^2

__device__ __forceinline__ uint32_t rd_s32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint32_t rd_map(uint32_t addr, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
__device__ __forceinline__ void rd_bar_init(uint64_t *b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(rd_s32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void rd_arm(uint64_t *b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(rd_s32(b)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void rd_arrive(uint64_t *b) {
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(rd_s32(b)) : "memory");
}
__device__ __forceinline__ bool rd_try(uint64_t *b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(rd_s32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait, the same answer in every lane of the warp
__device__ __forceinline__ bool rd_wait(uint64_t *b, uint32_t parity, unsigned long long limit, int *err) {
    if (__all_sync(0xffffffffu, rd_try(b, parity))) return true;
    const unsigned long long t0 = clock64();
    for (;;) {
        if (__all_sync(0xffffffffu, rd_try(b, parity))) return true;
        if (__any_sync(0xffffffffu, clock64() - t0 > limit)) {
            if ((threadIdx.x & 31) == 0) atomicCAS(err, 0, 2);
            return false;
        }
    }
}
// 16 bytes into a CTA of the cluster, counted by a barrier of that CTA
__device__ __forceinline__ void rd_send(uint32_t addr, uint4 v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
                 "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void rd_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// 96-bit unsigned integers
struct U96 {
    uint32_t a, b, c;
};
__device__ __forceinline__ U96 operator+(U96 x, U96 y) {
    U96 r;
    asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
        : "=r"(r.a), "=r"(r.b), "=r"(r.c)
        : "r"(x.a), "r"(x.b), "r"(x.c), "r"(y.a), "r"(y.b), "r"(y.c));
    return r;
}
__device__ __forceinline__ U96 operator-(U96 x, U96 y) {
    U96 r;
    asm("sub.cc.u32 %0, %3, %6;\n\tsubc.cc.u32 %1, %4, %7;\n\tsubc.u32 %2, %5, %8;"
        : "=r"(r.a), "=r"(r.b), "=r"(r.c)
        : "r"(x.a), "r"(x.b), "r"(x.c), "r"(y.a), "r"(y.b), "r"(y.c));
    return r;
}
__device__ __forceinline__ bool operator>(U96 x, U96 y) {   // the borrow of y - x
    uint32_t r;
    asm("{\n\t.reg .u32 t;\n\tsub.cc.u32 t, %1, %4;\n\tsubc.cc.u32 t, %2, %5;\n\tsubc.cc.u32 t, %3, %6;\n\t"
        "subc.u32 %0, 0, 0;\n\t}"
        : "=r"(r)
        : "r"(y.a), "r"(y.b), "r"(y.c), "r"(x.a), "r"(x.b), "r"(x.c));
    return r != 0u;
}
__device__ __forceinline__ U96 rd_shfl(U96 v, int src) {
    return {__shfl_sync(0xffffffffu, v.a, src), __shfl_sync(0xffffffffu, v.b, src), __shfl_sync(0xffffffffu, v.c, src)};
}
__device__ __forceinline__ U96 rd_warp_sum(U96 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v = v + U96{__shfl_xor_sync(0xffffffffu, v.a, o), __shfl_xor_sync(0xffffffffu, v.b, o),
                    __shfl_xor_sync(0xffffffffu, v.c, o)};
    return v;
}
// inclusive prefixes over the first N lanes (16: the lanes beyond keep partial sums)
template <int N>
__device__ __forceinline__ U96 rd_incl(U96 v, int lane) {
#pragma unroll
    for (int o = 1; o < N; o <<= 1) {
        U96 u = {__shfl_up_sync(0xffffffffu, v.a, o), __shfl_up_sync(0xffffffffu, v.b, o),
                 __shfl_up_sync(0xffffffffu, v.c, o)};
        if (lane < o) u = U96{0u, 0u, 0u};
        v = v + u;
    }
    return v;
}
// floor(x U / 2^53) for x < 2^95, U < 2^53
__device__ __forceinline__ U96 rd_scale(U96 x, unsigned long long U) {
    using u128 = unsigned __int128;
    const u128 v = ((u128)x.c << 64) | (((unsigned long long)x.b << 32) | x.a);
    const u128 t1 = v >> 48, t0 = v & (((u128)1 << 48) - 1);
    const u128 r = (t1 * U + ((t0 * U) >> 48)) >> 5;
    return {(uint32_t)r, (uint32_t)(r >> 32), (uint32_t)(r >> 64)};
}

// the unit's exponent for masses below 2^(E - 126): m of them sum to less than 2^95
__device__ __forceinline__ int rd_unit(uint32_t E, int m) { return (int)E - 126 + (32 - __clz(m)) - 95; }

// w D^2 in units of 2^eb (at least 1 when positive), and E with w D^2 < 2^(E - 126)
// (0: no mass; kExpInf, kExpNan: D^2 is not finite)
__device__ __forceinline__ U96 rd_mass(uint32_t w, float d2, int eb, uint32_t &E) {
    const uint32_t bits = __float_as_uint(d2) & 0x7fffffffu;
    E = 0;
    if (w == 0u || bits == 0u) return {0u, 0u, 0u};
    const uint32_t e8 = bits >> 23;
    if (e8 == 255u) {
        E = (bits & 0x7fffffu) ? kExpNan : kExpInf;
        return {1u, 0u, 0u};
    }
    const uint32_t e = max(e8, 1u);
    unsigned long long p = (unsigned long long)w * ((bits & 0x7fffffu) | (e8 ? 0x800000u : 0u));
    E = e + (32 - __clz(w));
    const int s = (int)e - 150 - eb;   // at most 70
    if (s < 0) {
        p = s > -64 ? p >> -s : 0ull;
        if (p == 0ull) p = 1ull;
    }
    const uint32_t lo = (uint32_t)p, hi = (uint32_t)(p >> 32), sh = s > 0 ? (uint32_t)s : 0u;
    const uint32_t x0 = lo << (sh & 31u), x1 = __funnelshift_l(lo, hi, sh), x2 = __funnelshift_l(hi, 0u, sh);
    if (sh < 32u) return {x0, x1, x2};
    if (sh < 64u) return {0u, x0, x1};
    return {0u, 0u, x0};
}

struct RdArgs {
    const float *C;          // candidates, row-major
    const float4 *CT4;       // [group of four coordinates][slot], or null (rows then come from C)
    const long long *w;
    DevState *st;
    int m, d, k;
    uint64_t seed;
    int cs, cpw;             // CTAs, candidates per lane
    int aw;                  // warps of a CTA that hold candidates
    int qs4;                 // coordinate groups kept in shared memory
    int32_t *chosen;
    float *centers;
    int *err;
    unsigned long long wait;
};

// slot s of the transposed copy and of the CTAs' arrays (cpw x 32 slots per warp,
// lanes adjacent) holds candidate slot_cand(s)
__host__ __device__ __forceinline__ int slot_cand(int s, int cpw) {
    const int lane = s & 31, c = s >> 5;
    return (c / cpw) * 32 * cpw + lane * cpw + c % cpw;
}

// four coordinates of candidate j, zero-padded past d
__device__ __forceinline__ float4 rd_coords(const float *__restrict__ C, int j, int d, int q4) {
    const float *r = C + (int64_t)j * d;
    const int q = 4 * q4;
    float4 v;
    v.x = q < d ? __ldg(r + q) : 0.f;
    v.y = q + 1 < d ? __ldg(r + q + 1) : 0.f;
    v.z = q + 2 < d ? __ldg(r + q + 2) : 0.f;
    v.w = q + 3 < d ? __ldg(r + q + 3) : 0.f;
    return v;
}

// t = x - c rounded, s = fma(t, t, s), coordinates ascending: the FP32 chain of
// dist2_fp32 (padded coordinates are 0 on both sides and add an exact 0)
__device__ __forceinline__ void rd_acc(float &s, float4 x, float4 c) {
    float t = __fsub_rn(x.x, c.x); s = __fmaf_rn(t, t, s);
    t = __fsub_rn(x.y, c.y); s = __fmaf_rn(t, t, s);
    t = __fsub_rn(x.z, c.z); s = __fmaf_rn(t, t, s);
    t = __fsub_rn(x.w, c.w); s = __fmaf_rn(t, t, s);
}

__host__ __device__ __forceinline__ size_t rd_smem_bytes(int d4, int cpw, int aw, int qs4) {
    const size_t nc = (size_t)cpw * 32 * aw;
    return 16 * (size_t)(2 * kRdMaxCl + 2 * kRdWarps + 2 * (d4 + 1)) + 16 * nc * qs4 + 8 * nc;
}

// where the coordinates beyond shared memory come from
enum { RD_SMEM = 0, RD_L2 = 1, RD_ROWS = 2 };   // nowhere; the transposed copy; the row-major candidates

// D^2 of slot ls against the new center cn (its lane's candidate; `first`: the first
// center).  Partial sums of non-negative terms never decrease: once every lane's has
// reached its D^2 (a vote every 16 coordinates in shared memory, 32 beyond) the rest is
// skipped.  Returns whether the lane's D^2 fell.
template <int SRC>
__device__ __forceinline__ bool rd_update(const RdArgs &a, const float4 *rows, float *dl, const uint32_t *wl,
                                          const float4 *cn, int ls, int s0, int NC, int d4, bool first) {
    const bool act = wl[ls] != 0u;
    const float lim = first ? __uint_as_float(0x7f800000u) : dl[ls];
    float v = 0.f;
    bool open = __any_sync(0xffffffffu, act && !(v >= lim));   // (false: every D^2 is 0)
    const float4 *x = rows + ls;
    int q4 = 0;
    while (open && q4 + 4 <= a.qs4) {
        const float4 x0 = x[0], x1 = x[NC], x2 = x[2 * NC], x3 = x[3 * NC];
        rd_acc(v, x0, cn[q4]);
        rd_acc(v, x1, cn[q4 + 1]);
        rd_acc(v, x2, cn[q4 + 2]);
        rd_acc(v, x3, cn[q4 + 3]);
        q4 += 4;
        x += 4 * NC;
        open = __any_sync(0xffffffffu, act && !(v >= lim));
    }
    if (open) {
        for (; q4 < a.qs4; ++q4, x += NC) rd_acc(v, *x, cn[q4]);
        if (SRC != RD_SMEM) {
            const size_t mpt = (size_t)NC * a.cs;
            const int j = SRC == RD_ROWS ? min(slot_cand(s0 + ls, a.cpw), a.m - 1) : 0;
            const float4 *src = a.CT4 + (size_t)q4 * mpt + s0 + ls;
            while (open && q4 < d4) {
                // eight loads in flight: an L2 load takes some 600 cycles
                float4 g[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    g[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (q4 + u < d4) g[u] = SRC == RD_L2 ? __ldg(src + u * mpt) : rd_coords(a.C, j, a.d, q4 + u);
                }
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (q4 + u < d4) rd_acc(v, g[u], cn[q4 + u]);
                q4 += 8;
                src += 8 * mpt;
                open = __any_sync(0xffffffffu, act && !(v >= lim));
            }
        }
    }
    const bool fell = act && (first || v < lim);
    if (fell) dl[ls] = v;
    return fell;
}

template <int SRC>
__global__ void __launch_bounds__(kRdThreads, 1) recluster_draws_kernel(RdArgs a) {
    extern __shared__ __align__(16) unsigned char rd_sm[];
    __shared__ uint64_t bar_tot[2], bar_row[2], bar_loc;
    const int d = a.d, d4 = (d + 3) >> 2, cpw = a.cpw, NC = cpw * 32 * a.aw, m = a.m, CS = a.cs;
    uint4 *tot = reinterpret_cast<uint4 *>(rd_sm);               // [2][CS]
    uint4 *wtot = tot + 2 * kRdMaxCl;                             // [2][16 warps]
    uint4 *row = wtot + 2 * kRdWarps;                             // [2][header, d4 groups]
    float4 *rows = reinterpret_cast<float4 *>(row + 2 * (d4 + 1));   // [qs4][NC]
    float *dl = reinterpret_cast<float *>(rows + (size_t)a.qs4 * NC);
    uint32_t *wl = reinterpret_cast<uint32_t *>(dl + NC);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int mine = wid < a.aw ? cpw : 0;   // candidates of a lane of this warp
    uint32_t rank_u;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank_u));
    const int rank = (int)rank_u;
    const uint32_t tot_bytes = 16u * CS, row_bytes = 16u * (d4 + 1);
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            rd_bar_init(&bar_tot[i], 1);
            rd_bar_init(&bar_row[i], 1);
        }
        rd_bar_init(&bar_loc, kRdWarps);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int i = 0; i < 2; ++i) {
            rd_arm(&bar_tot[i], tot_bytes);
            rd_arm(&bar_row[i], row_bytes);
        }
    }
    // this CTA's candidates
    const int s0 = rank * NC;
    for (int s = tid; s < NC; s += kRdThreads) {
        const int j = slot_cand(s0 + s, cpw);
        wl[s] = j < m ? (uint32_t)a.w[j] : 0u;
        dl[s] = 0.f;
    }
    for (int f = tid; f < a.qs4 * NC; f += kRdThreads) {
        const int s = f % NC, q4 = f / NC;
        const int j = slot_cand(s0 + s, cpw);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (j < m)
            v = SRC == RD_L2 ? __ldg(a.CT4 + (size_t)q4 * NC * CS + s0 + s) : rd_coords(a.C, j, d, q4);
        rows[(size_t)q4 * NC + s] = v;
    }
    __syncthreads();
    rd_cluster_sync();   // every CTA's barriers are initialised and armed

    const uint32_t a_tot = rd_s32(tot), a_row = rd_s32(row);
    const uint32_t a_bt = rd_s32(&bar_tot[0]), a_br = rd_s32(&bar_row[0]);
    // draw 0: masses w, below 2^31
    uint32_t curE = 127u + 31u;
    int eb = rd_unit(curE, m), t = 0, pick0 = 0;
    bool dirty = true, ok = true, first = true;
    U96 wsum = {0u, 0u, 0u};
    uint32_t wE = 0;
    for (uint32_t x = 0;; ++x) {
        const uint32_t b = x & 1u, par = (x >> 1) & 1u;
        // ---- the warp's mass total
        if (dirty) {
            U96 s = {0u, 0u, 0u};
            uint32_t E = 0;
            for (int i = 0; i < mine; ++i) {
                const int ls = (wid * cpw + i) * 32 + lane;
                uint32_t Ei;
                s = s + rd_mass(wl[ls], t == 0 ? 1.f : dl[ls], eb, Ei);
                E = max(E, Ei);
            }
            wsum = rd_warp_sum(s);
            wE = __reduce_max_sync(0xffffffffu, E);
            dirty = false;
        }
        if (lane == 0) {
            wtot[b * kRdWarps + wid] = make_uint4(wsum.a, wsum.b, wsum.c, wE);
            rd_arrive(&bar_loc);   // the total and this warp's D^2 are written (read by warp 0)
        }
        __syncwarp();
        if (wid == 0) {
            const uint4 rw = philox4x32_10((uint32_t)t, 0u, 0u, TAG_RECLUSTER, (uint32_t)a.seed,
                                           (uint32_t)(a.seed >> 32));
            const unsigned long long U = ((unsigned long long)(rw.x >> 5) << 26) + (rw.y >> 6);   // u = U / 2^53
            // ---- the CTA's total to every CTA
            ok = rd_wait(&bar_loc, x & 1u, a.wait, a.err);
            if (!ok) break;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (lane < kRdWarps) v = wtot[b * kRdWarps + lane];
            const U96 wi = rd_incl<16>(U96{v.x, v.y, v.z}, lane);   // prefixes of the warps
            const U96 ctot = rd_shfl(wi, kRdWarps - 1);
            const uint32_t cE = __reduce_max_sync(0xffffffffu, v.w);
            if (lane < CS)
                rd_send(rd_map(a_tot + 16u * (b * kRdMaxCl + rank), lane),
                        make_uint4(ctot.a, ctot.b, ctot.c, cE),
                        rd_map(a_bt + 8u * b, lane));
            // ---- the owning CTA, from all totals
            ok = rd_wait(&bar_tot[b], par, a.wait, a.err);
            if (!ok) break;
            if (lane == 0) rd_arm(&bar_tot[b], tot_bytes);
            v = make_uint4(0u, 0u, 0u, 0u);
            if (lane < CS) v = tot[b * kRdMaxCl + lane];
            const U96 ls = {v.x, v.y, v.z};
            const U96 incl = rd_incl<16>(ls, lane);
            const U96 total = rd_shfl(incl, kRdMaxCl - 1);
            const uint32_t gE = __reduce_max_sync(0xffffffffu, v.w);
            int code = 0, neb = 0;
            if (gE == 0u || gE == kExpNan) code = -1;                              // no mass left
            else if (gE != kExpInf && (eb == kRdUnset || gE + 16u < curE)) {        // a new unit
                code = -2;
                neb = (int)gE;
            }
            if (code != 0) {
                if (rank == 0)
                    for (int q4 = lane; q4 <= d4; q4 += 32)
                        for (int r = 0; r < CS; ++r)
                            rd_send(rd_map(a_row + 16u * (b * (d4 + 1) + q4), r), make_uint4((uint32_t)code, neb, 0, 0),
                                    rd_map(a_br + 8u * b, r));
            } else {
                U96 target = rd_scale(total, U);                            // floor(u total) < total
                if (gE == kExpInf) target = total - U96{1u, 0u, 0u};         // the last candidate with any mass
                // total > target: some CTA's prefix passes it
                const int owner = __ffs(__ballot_sync(0xffffffffu, lane < kRdMaxCl && incl > target)) - 1;
                if (owner == rank) {
                    // ---- the warp, then the lane, then the lane's candidate
                    U96 before = rd_shfl(incl - ls, owner);
                    const int lw = __ffs(__ballot_sync(0xffffffffu, lane < kRdWarps && before + wi > target)) - 1;
                    if (lw > 0) before = before + rd_shfl(wi, lw - 1);
                    U96 es = {0u, 0u, 0u};
                    for (int i = 0; i < cpw; ++i) {
                        const int sl = (lw * cpw + i) * 32 + lane;
                        uint32_t Ei;
                        es = es + rd_mass(wl[sl], t == 0 ? 1.f : dl[sl], eb, Ei);
                    }
                    const U96 ei = before + rd_incl<32>(es, lane);
                    const int hl = __ffs(__ballot_sync(0xffffffffu, ei > target)) - 1;
                    int ps = 0;
                    U96 cum0 = {0u, 0u, 0u}, cum = cum0;
                    if (lane == hl) {
                        cum0 = ei - es;
                        for (int i = 0; i < cpw; ++i) {
                            ps = (lw * cpw + i) * 32 + lane;
                            uint32_t Ei;
                            cum = cum0 + rd_mass(wl[ps], t == 0 ? 1.f : dl[ps], eb, Ei);
                            if (cum > target) break;
                            cum0 = cum;
                        }
                    }
                    ps = __shfl_sync(0xffffffffu, ps, hl);
                    const int pick = slot_cand(s0 + ps, cpw);
                    for (int q4 = lane; q4 <= d4; q4 += 32) {   // group d4 stands for the header
                        uint4 v = make_uint4((uint32_t)pick, 0u, 0u, 0u);
                        if (q4 < d4) {
                            const float4 g = q4 < a.qs4 ? rows[(size_t)q4 * NC + ps]
                                             : SRC == RD_L2 ? __ldg(a.CT4 + (size_t)q4 * NC * CS + s0 + ps)
                                                            : rd_coords(a.C, pick, d, q4);
                            v = make_uint4(__float_as_uint(g.x), __float_as_uint(g.y), __float_as_uint(g.z),
                                           __float_as_uint(g.w));
                        }
                        const uint32_t dst = a_row + 16u * (b * (d4 + 1) + (q4 < d4 ? q4 + 1 : 0));
                        for (int r = 0; r < CS; ++r) rd_send(rd_map(dst, r), v, rd_map(a_br + 8u * b, r));
                    }
                    if (lane == hl) {
                        // 1e-6 of the total, off the chain
                        const U96 win = rd_scale(total, 9007199255ull);
                        if (!(target - cum0 > win) || !(cum - target > win)) atomicAdd(&a.st->recluster_near, 1ull);
                    }
                }
            }
        }
        // ---- the picked row
        ok = rd_wait(&bar_row[b], par, a.wait, a.err);
        if (!ok) break;
        if (tid == 0) rd_arm(&bar_row[b], row_bytes);
        const uint4 *rb = row + b * (d4 + 1);
        const uint4 hdr = rb[0];
        if ((int)hdr.x == -2) {
            curE = hdr.y;
            eb = rd_unit(curE, m);
            dirty = true;
            continue;
        }
        if ((int)hdr.x == -1) {
            // positive mass exhausted: the remaining draws repeat the first center
            if (rank == 0) {
                const int src = pick0;
                for (int s = t + tid; s < a.k; s += kRdThreads) a.chosen[s] = src;
                if (tid == 0) a.st->warn = 1;
                for (int s = t; s < a.k; ++s)
                    for (int q = tid; q < d; q += kRdThreads) a.centers[(int64_t)s * d + q] = a.C[(int64_t)src * d + q];
            }
            break;
        }
        if (t == 0) pick0 = (int)hdr.x;
        const float4 *cn = reinterpret_cast<const float4 *>(rb + 1);
        if (rank == 0 && wid == 1) {
            const float *cf = reinterpret_cast<const float *>(cn);
            for (int q = lane; q < d; q += 32) a.centers[(int64_t)t * d + q] = cf[q];
            if (lane == 0) a.chosen[t] = (int32_t)hdr.x;
        }
        if (++t == a.k) break;
        // ---- D^2 against the new center.  Partial sums of non-negative terms never
        // decrease: once every lane's has reached its D^2 the rest is skipped
        bool fell = false;
        for (int i = 0; i < mine; ++i)
            fell |= rd_update<SRC>(a, rows, dl, wl, cn, (wid * cpw + i) * 32 + lane, s0, NC, d4, first);
        dirty = __any_sync(0xffffffffu, fell) || dirty;
        if (first) {
            first = false;
            dirty = true;
            eb = kRdUnset;   // the unit follows from the first D^2
        }
        __syncwarp();
    }
    if (!ok) {
        // messages of the other CTAs may still be on their way here
        const unsigned long long t0 = clock64();
        while (clock64() - t0 < 200000ull) __nanosleep(200);
    }
    __syncwarp();
    rd_cluster_sync();   // no CTA leaves while another may still write its shared memory
}

// candidates (m x d, row-major) -> groups of four coordinates by slot, zero-padded:
// eight lanes read 128 consecutive bytes of a row
__global__ void __launch_bounds__(256) transpose4_kernel(const float *__restrict__ C, int m, int d, int cpw,
                                                         int slots, float4 *__restrict__ CT4) {
    const int d4 = (d + 3) >> 2;
    const int64_t n = (int64_t)slots * ((d4 + 7) / 8) * 8;
    for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < n; f += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = f >> 3;
        const int s = (int)(g % slots), q4 = (int)(g / slots) * 8 + (int)(f & 7);
        if (q4 >= d4) continue;
        const int j = slot_cand(s, cpw);
        CT4[(size_t)q4 * slots + s] = j < m ? rd_coords(C, j, d, q4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

}  // namespace

// How the draws kernel covers m candidates of d coordinates: the fewest CTAs with one
// candidate per lane, max_cs beyond max_cs x 512 candidates, more where that brings all
// coordinates into shared memory, and else as many leading groups of coordinates there as
// fit.  The cooperative grid form takes over (cs = 0) when a draw would read more than
// 512 KB a CTA from L2: measured, us a draw, this form / the grid: 4,933 x 42 2.9 / 8.6,
// 9,925 x 42 3.8 / 8.7 (nothing from L2); 9,876 x 128 (320 KB) 7.7 / 9.3, 19,960 x 96 (384 KB)
// 8.2 / 9.5, 39,809 x 128 (1.1 MB) 15.9 / 10.3.
ReclusterPlan recluster_plan(int m, int d, int max_cs) {
    const int d4 = (d + 3) >> 2;
    const size_t budget = kRdSmemBudget;
    int cs = 1;
    while (cs < max_cs && m > cs * kRdThreads) cs *= 2;
    ReclusterPlan first{};
    for (int c = cs; c <= max_cs; c *= 2) {
        ReclusterPlan p{};
        p.cs = c;
        p.cpw = std::max(1, (m + c * kRdThreads - 1) / (c * kRdThreads));
        p.aw = std::min(kRdWarps, (m + c * 32 * p.cpw - 1) / (c * 32 * p.cpw));
        p.slots = c * p.cpw * 32 * p.aw;
        const size_t base = rd_smem_bytes(d4, p.cpw, p.aw, 0);
        if (base > budget) return ReclusterPlan{};
        const int fit = (int)((budget - base) / (16 * (size_t)p.cpw * 32 * p.aw));
        p.qs4 = fit >= d4 ? d4 : fit & ~3;
        if (p.qs4 == d4) return p;
        if (c == cs) first = p;
    }
    if ((size_t)(d4 - first.qs4) * first.cpw * 32 * first.aw * 16 > 512u * 1024u) return ReclusterPlan{};
    return first;
}

static const void *rd_kernels[3] = {(const void *)recluster_draws_kernel<RD_SMEM>,
                                    (const void *)recluster_draws_kernel<RD_L2>,
                                    (const void *)recluster_draws_kernel<RD_ROWS>};

// the largest cluster the device holds (16 CTAs need the non-portable attribute);
// asked once per device, as is the kernels' shared memory
cudaError_t recluster_max_cluster(int dev, int *max_cs) {
    static std::atomic<int> known[64];
    const bool slot = dev >= 0 && dev < 64;
    if (slot && (*max_cs = known[dev].load()) > 0) return cudaSuccess;
    for (const void *kern : rd_kernels) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRdSmemBudget);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kRdMaxCl);
    cfg.blockDim = dim3(kRdThreads);
    cfg.dynamicSmemBytes = kRdSmemBudget;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kRdMaxCl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    *max_cs = 8;
    if (cudaOccupancyMaxActiveClusters(&n, rd_kernels[RD_L2], &cfg) != cudaSuccess) cudaGetLastError();
    else if (n >= 1) *max_cs = kRdMaxCl;
    if (slot) known[dev].store(*max_cs);
    return cudaSuccess;
}

// The draws kernel with plan p; CT4 (p.slots x ceil(d / 4) float4) may be null: the
// groups beyond shared memory then come from the row-major candidates.
cudaError_t launch_recluster_draws(Ctx &c, float *centers, const ReclusterPlan &p, float *CT4) {
    cudaError_t e;
    const int d4 = (c.d + 3) >> 2;
    float4 *ct = p.qs4 < d4 ? reinterpret_cast<float4 *>(CT4) : nullptr;
    if (ct) {
        const int64_t work = (int64_t)p.slots * ((d4 + 7) / 8) * 8;
        transpose4_kernel<<<(int)std::min<int64_t>((work + 255) / 256, (int64_t)c.num_sms * 16), 256, 0, c.stream>>>(
            c.C, c.m_host, c.d, p.cpw, p.slots, ct);
        count_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    RdArgs a{};
    a.C = c.C; a.CT4 = ct; a.w = c.w; a.st = c.st; a.m = c.m_host; a.d = c.d; a.k = c.k; a.seed = c.seed;
    a.cs = p.cs; a.cpw = p.cpw; a.aw = p.aw; a.qs4 = p.qs4; a.chosen = c.chosen; a.centers = centers; a.err = c.rc_err;
    a.wait = kRdWait;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.cs);
    cfg.blockDim = dim3(kRdThreads);
    cfg.dynamicSmemBytes = rd_smem_bytes(d4, p.cpw, p.aw, p.qs4);
    cfg.stream = c.stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)p.cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void *args[] = {&a};
    e = cudaLaunchKernelExC(&cfg, rd_kernels[p.qs4 == d4 ? RD_SMEM : ct ? RD_L2 : RD_ROWS], args);
    count_launches(1);
    return e;
}

}  // namespace kmp
