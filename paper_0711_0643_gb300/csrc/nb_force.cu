// Force + jerk + potential of the active block against all N predicted
// particles: Eq. (Force) of Sect. 2.1 with Plummer softening, its exact time
// derivative, and the softened potential.
//
// The paper splits the j-sum over processors and adds the partial forces with
// MPI_Allreduce (Sect. 3). Here the split is on one chip: every CTA of a persistent
// grid derives its share of the work from the active count s on the device, so the
// launch needs no host round trip and can live inside a CUDA graph; j-records stream
// through shared memory, copied by the TMA bulk engine (cp.async.bulk + mbarrier);
// partials are reduced in a fixed order (lane shuffles, then the CTAs' partials): the
// last CTA to finish an i-block (an arrival ticket, no waiting) adds them, so results
// are bitwise reproducible run to run.
//
// Mixed precision: positions arrive as double-single (hi, lo) pairs so that
// r = x_j - x_i keeps ~46 bits even for close pairs (velocities are FP32: the
// jerk error is set by the FP32 pair arithmetic, not by w); the pair
// arithmetic is FP32 on packed f32x2 instructions over the two particles of a
// pair record, with one MUFU reciprocal square root per particle refined by a
// Newton step; per-thread FP32 partial sums over at most kFoldPairs
// pairs are folded into (hi, lo) two-sum accumulators, and the cross-thread
// reductions combine (hi, lo) pairs with two-sums too (FP64 is a narrow pipe on
// this part; only the final per-split partial is converted to double).
#include <cooperative_groups.h>

#include <cstddef>

#include "nb_internal.cuh"
#include "nb_pair.cuh"
#include "nb_rsqrt.cuh"

namespace cg = cooperative_groups;

namespace nb {

namespace {

// ------------------------------------------------------------ PTX helpers

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// 1-D bulk copy global -> shared, completion counted on the mbarrier (TMA).
// Both addresses 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait on an mbarrier phase: false if the spin limit expired.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, int64_t limit)
{
    for (int it = 0; it < 64; ++it)
        if (mbar_test(bar, parity)) return true;
    for (int64_t it = 64; it < limit; ++it) {
        if (mbar_test(bar, parity)) return true;
        __nanosleep(64);
    }
    return false;
}

// ------------------------------------------------------------ shared memory

constexpr int kPT = kJT / 2;    // pair records per tile
constexpr int kRing = 8;        // tiles in flight in the TMA streaming variant

// Column kernel (see there): a unit is up to kUnitRec pair records in kUnitBytes of
// shared memory, kSlots units in flight.
constexpr int kUnitRec = 256;
constexpr int kUnitBytes = kUnitRec * (int)sizeof(JPair);
constexpr int kSlots = 4;
// variant 0: items of kLongTiles tiles or more go through the TMA ring where the j range is so
// large that its records come from HBM in use (the same sums). N = 2^20, s = 1, us, ring / straight
// loads: records from HBM 16.5 / 16.9, from L2 11.1 / 10.8; smaller ranges, which stay in L2: N =
// 32768, s = 64 14.7 / 12.1, N = 20000, s = 64 11.6 / 10.3
constexpr int kLongTiles = 12;
constexpr int kColdTiles = 2048;
constexpr int kShortTiles = 32;   // shares that may go by whole items (see short_items): up to this
constexpr int kItemTiles = 128;   //   many tiles always, up to this many where the items fill the GPU
constexpr int kFoldTiles = kFoldPairs;   // tiles in which a thread of 256 meets kFoldPairs / 2 records

// Resident-share variant: clusters of kShareC CTAs, CTA r holding up to
// kShareRec pair records of the j range in shared memory, the active list dealt
// out to the clusters in chunks of up to kShareSlots particles.
constexpr int kShareC = 8;
constexpr int kShareRec = 1024;
constexpr int kShareSlots = 256;
constexpr int kSharePiece = 256;   // records per copy (four mbarriers)
static_assert(kShareRec / kSharePiece <= kRing, "one mbarrier per piece");

// How the column kernel cuts a launch (worked out by one thread per CTA).
struct ColPlan {
    int64_t tper;       // tiles per share of the table's split
    int64_t upi;        // units per i-block
    int64_t nib, U, G;  // i-blocks, units in all, CTAs sharing them
    int64_t u0, u1, b0; // this CTA's run of units, the i-block it begins in
    int ups;            // units per share
    int lgst, lgcw;     // log2 of the column stride (records) and of the columns per unit
    int lgtj;           // log2 of the threads per i-particle
    int slots;          // partial slots per particle
    int whole;          // no i-block is shared between CTAs
    int part_n, part_slot;   // the current i-block: CTAs that meet it, this one's place
};

// The staging buffers come last, so that the resident-share variant's larger
// buffer can take their place and run past the end of the struct.
struct __align__(128) Smem {
    float2 red[kThreads / 32][14];
    uint64_t bar[kRing];
    uint64_t inject_bar;
    int64_t s;                 // active count of this launch
    int64_t items, tper;       // streamed variants: work items, tiles per item,
    int split, lgi;            //   items per i-block, log2 of the particles of an i-block
    Tuning tune;               // the device tuning table, read once per CTA
    int32_t idx_pre[kThreads]; // the first kThreads entries of the active list, read with s
    ColPlan plan;              // kept here and not in registers: the pair loop needs those
    uint64_t empty[kSlots];    // column kernel: every warp has read the slot's unit
    int2 info[kSlots];         // the unit's rows and columns
    int abort;
    int last;
    alignas(128) union {
        JPair ring[kRing][kPT];                      // TMA streaming variant
        struct {
            unsigned char unit[kSlots][kUnitBytes];  // column kernel
            float2 sums[7][kThreads];                // its threads' sums of an i-block
        };
    };
};

struct ShareBuf {
    JPair rec[kShareRec];            // this CTA's share of the j-records
    // (hi, lo) partials of the chunk's positions rank, rank + kShareC, ..., pushed here by
    // every CTA of the cluster
    float2 in[kShareSlots / kShareC][kShareC][7];
};

constexpr size_t kSmemShare =
    (sizeof(Smem) > offsetof(Smem, ring) + sizeof(ShareBuf) ? sizeof(Smem) : offsetof(Smem, ring) + sizeof(ShareBuf));

__device__ __forceinline__ ShareBuf *shb(Smem *sm) { return reinterpret_cast<ShareBuf *>(&sm->ring[0][0]); }

__device__ __forceinline__ int bucket_of(int64_t s)
{
    // bucket b holds s in (2^(b-1), 2^b]; s = 1 -> 0
    int b = 0;
    while ((int64_t(1) << b) < s && b < kBuckets - 1) ++b;
    return b;
}

// a / b for a >= 0, b > 0. A 64-bit division is a long dependent instruction
// chain on this GPU (several of them sat on the critical path of every launch);
// the 32-bit one is short, and the sizes of a launch fit in 32 bits.
__device__ __forceinline__ int64_t qdiv(int64_t a, int64_t b)
{
    if ((((uint64_t)a | (uint64_t)b) >> 32) == 0) return (int64_t)((uint32_t)a / (uint32_t)b);
    return a / b;
}

__device__ __forceinline__ int64_t qmod(int64_t a, int64_t b) { return a - qdiv(a, b) * b; }

// The table's split is the one for its bucket's largest size s_ref = min(2^b, n);
// a smaller block of the bucket keeps the same number of work items (i-blocks x
// splits), so a wave-aligned choice stays wave-aligned.
__device__ __forceinline__ int table_split(int S_ref, int b, int64_t s, int64_t n, int64_t I)
{
    const int64_t s_ref = (int64_t(1) << b) < n ? (int64_t(1) << b) : n;
    const int lg = 31 - __clz((int)I);   // I is a power of two
    const int64_t nib_ref = (s_ref + I - 1) >> lg, nib = (s + I - 1) >> lg;
    const int64_t S = nib_ref == nib ? S_ref : qdiv((int64_t)S_ref * nib_ref, nib);
    return S < 1 ? 1 : (S > (1 << 30) ? (1 << 30) : (int)S);
}

// Entry jj < s of the active list (the first kThreads from shared memory).
__device__ __forceinline__ int32_t idx_at(const ForceArgs &A, const Smem *sm, int64_t jj)
{
    return jj < kThreads ? sm->idx_pre[jj] : A.idx[jj];
}

// Split factor clamp shared by both precisions.
__device__ __forceinline__ int clamp_split(int S, int64_t n_tiles, int64_t s, int64_t cap)
{
    if (S < 1) S = 1;
    if (S > n_tiles) S = (int)n_tiles;
    if ((int64_t)S * s * kPartStride > cap) {
        const int64_t lim = qdiv(cap, s * kPartStride);
        S = lim < 1 ? 1 : (int)lim;
    }
    return S;
}

// Split partial of active particle ii from split by, as (hi, lo) float pairs.
__device__ __forceinline__ float2 *part2(const ForceArgs &A, int64_t ii, int by, int S)
{
    return reinterpret_cast<float2 *>(A.part) + (ii * S + by) * kPartStride;
}

// Final sum of component c (ax ay az kx ky kz phi) of active particle ii: into
// fin and, when the launch has them, the caller's layouts.
__device__ __forceinline__ void put_final(const ForceArgs &A, int64_t ii, int c, double v)
{
    A.fin[ii * kPartStride + c] = v;
    double *dst = c < 3 ? A.out_a : (c < 6 ? A.out_k : A.out_phi);
    if (dst) {
        dst[c < 6 ? ii * 3 + (c % 3) : ii] = v;
        if (!isfinite(v)) atomicOr(A.status, kStNonfinite);
    }
}

// Active count of a launch and the optional copy of the caller's list into the
// context (grid-stride; every CTA takes part).
__device__ __forceinline__ int64_t launch_s(const ForceArgs &A) { return A.s_host >= 0 ? A.s_host : *A.s; }

__device__ __forceinline__ void copy_list(const ForceArgs &A, int64_t s)
{
    if (!A.idx_copy) return;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < s; q += (int64_t)gridDim.x * blockDim.x)
        A.idx_copy[q] = A.idx[q];
    if (blockIdx.x == 0 && threadIdx.x == 0) *A.s_copy = s;
}

template <int U>
__device__ __forceinline__ void sum_lane(const float2 *src, int lane, int n, float &h, float &l)
{
    for (int q0 = lane; q0 < n; q0 += 32 * U) {
        float2 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            v[u] = q0 + 32 * u < n ? __ldcg(src + (q0 + 32 * u) * kPartStride) : make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (q0 + 32 * u < n) ds_add(h, l, v[u].x, v[u].y);
    }
}

constexpr int kFewParts = 4;

// Adds the n partials of each of the active particles [ib0, ib1) (slots 0 .. n - 1 of S)
// by this CTA, in a fixed order, and writes the results.
template <bool FEW>
__device__ void sum_parts(const ForceArgs &A, int64_t ib0, int64_t ib1, int S, int n)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int np = (int)(ib1 - ib0);
    if (FEW && n <= kFewParts && np <= 8) {
        // a thread per (particle, component): no lane tree (N = 4096, s = 1 .. 16: 0.2 us, N = 24576, s =
        // 195: 0.9 us less than the forms below)
        if (threadIdx.x < 7 * np) {
            const int64_t ii = ib0 + threadIdx.x / 7;
            const int c = threadIdx.x % 7;
            float2 v[kFewParts];
#pragma unroll
            for (int u = 0; u < kFewParts; ++u)
                v[u] = u < n ? __ldcg(part2(A, ii, u, S) + c) : make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 1; u < kFewParts; ++u)
                if (u < n) ds_add(v[0].x, v[0].y, v[u].x, v[u].y);
            put_final(A, ii, c, (double)v[0].x + (double)v[0].y);
        }
        return;
    }
    if (np == 1) {
        // a warp per component; lane l adds partials l, l + 32, ..., their loads issued
        // together (ten cover a partial from every CTA), then a butterfly over the lanes
        if (warp < 7) {
            float h = 0.f, l = 0.f;
            if (n <= 64)
                sum_lane<2>(part2(A, ib0, 0, S) + warp, lane, n, h, l);
            else
                sum_lane<10>(part2(A, ib0, 0, S) + warp, lane, n, h, l);
            ds_group_reduce<32>(h, l);
            if (lane == 0) put_final(A, ib0, warp, (double)h + (double)l);
        }
        return;
    }
    // D threads per (particle, component pair), neighbours in a warp, thread d adding
    // partials d, d + D, ... with kLoads 16-byte loads issued together (an L2 round trip
    // each: the sum is bound by how many are in flight), then a tree over the D threads.
    constexpr int kLoads = 16;
    const int D = np <= 8 ? 8 : (np <= 16 ? 4 : (np <= 32 ? 2 : 1));
    const int qc = threadIdx.x & 3, d = (threadIdx.x >> 2) & (D - 1);
    const int per = kThreads / (4 * D);   // particles at a time
    for (int p0 = 0; p0 < np; p0 += per) {
        const int pi = p0 + threadIdx.x / (4 * D);
        const int64_t ii = ib0 + (pi < np ? pi : np - 1);
        const float4 *src = reinterpret_cast<const float4 *>(part2(A, ii, 0, S)) + qc;
        float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f;
        for (int q0 = d; q0 < n; q0 += D * kLoads) {
            float4 v[kLoads];
#pragma unroll
            for (int u = 0; u < kLoads; ++u) {
                const int q = q0 + D * u;
                v[u] = q < n ? __ldcg(src + q * (kPartStride / 2)) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < kLoads; ++u)
                if (q0 + D * u < n) {
                    ds_add(h0, l0, v[u].x, v[u].y);
                    if (qc < 3) ds_add(h1, l1, v[u].z, v[u].w);   // component 7 is padding
                }
        }
        for (int off = 4; off < 4 * D; off <<= 1) {
            const float a0 = __shfl_xor_sync(0xffffffffu, h0, off), b0 = __shfl_xor_sync(0xffffffffu, l0, off);
            const float a1 = __shfl_xor_sync(0xffffffffu, h1, off), b1 = __shfl_xor_sync(0xffffffffu, l1, off);
            ds_add(h0, l0, a0, b0);
            ds_add(h1, l1, a1, b1);
        }
        if (d == 0 && pi < np) {
            put_final(A, ii, 2 * qc, (double)h0 + (double)l0);
            if (qc < 3) put_final(A, ii, 2 * qc + 1, (double)h1 + (double)l1);
        }
    }
}

// Called by every thread after this CTA has written its partials of i-block bx (active
// particles [ib0, ib1)). The CTA that completes the block's n partials (ticket n - 1)
// adds them with two-sums and writes the FP64 results; it then re-arms the ticket.
template <bool FEW>
__device__ void finish_block(const ForceArgs &A, int64_t bx, int64_t ib0, int64_t ib1, int S, int n, Smem *sm)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const int t = atomicAdd(&A.tickets[bx], 1);
        sm->last = (t == n - 1);
    }
    __syncthreads();
    if (sm->last) {
        __threadfence();
        sum_parts<FEW>(A, ib0, ib1, S, n);
        if (threadIdx.x == 0) A.tickets[bx] = 0;
    }
    __syncthreads();
}

// ------------------------------------------------------- streamed variant
// All threads share the same R i-particles; each thread walks its own pair records
// straight from global memory, so no shared staging is needed. For the smallest active
// blocks: a call is then a chain of latencies, and this chain is the shortest.

// Item w of the launch: i-block bx and tiles [t0, t1) (the launch's split and tiles per
// item are kept in shared memory: the pair loops need the registers).
__device__ __forceinline__ void stream_item(const ForceArgs &A, int64_t w, const Smem *sm, int64_t &bx, int64_t &t0,
                                            int64_t &t1)
{
    bx = qdiv(w, sm->split);
    const int64_t by = w - bx * sm->split;
    t0 = A.tile_lo + by * sm->tper;
    t1 = t0 + sm->tper < A.tile_hi ? t0 + sm->tper : A.tile_hi;
}

// The CTA's sums of particle bx, r-th of the CTA's: into the CTA's partial slot or,
// where the CTA holds all of j (S == 1), the results. more: added to what is there.
__device__ __forceinline__ void cta_sum_red(const Acc7 &hi, const Acc7 &lo, float2 *red, bool more = false)
{
    float h, l;
    const int lane = threadIdx.x & 31;
    const int c = ds_scatter_reduce<32>(hi, lo, h, l);   // a lane holds component c
    if ((lane & 3) == 0 && c < 7) {
        if (more) ds_add(h, l, red[c].x, red[c].y);
        red[c] = make_float2(h, l);
    }
}
template <int R>
__device__ __forceinline__ void cta_sum_out(const ForceArgs &A, int64_t w, Smem *sm)
{
    // warps in ascending order
    const int tid = threadIdx.x, S = sm->split;
    const int64_t s = sm->s, bx = qdiv(w, S), i0 = bx * R;
    const int by = (int)(w - bx * S);
    if (tid < 7 * R) {
        float h = sm->red[0][tid].x, l = sm->red[0][tid].y;
#pragma unroll
        for (int wv = 1; wv < kThreads / 32; ++wv) ds_add(h, l, sm->red[wv][tid].x, sm->red[wv][tid].y);
        const int64_t ii = i0 + tid / 7;
        const int c = tid % 7;
        if (ii < s) {
            if (S == 1)
                put_final(A, ii, c, (double)h + (double)l);
            else
                part2(A, ii, by, S)[c] = make_float2(h, l);
        }
    }
}

// LONG (R = 2): items of more than 64 tiles, one fold and one sum over the CTA for every 64
// (accumulators that outlive a fold would not fit the registers).
template <int R, bool LONG = false>
__device__ void work_stream(const ForceArgs &A, int64_t w, Smem *sm)
{
    const int tid = threadIdx.x, warp = tid >> 5;
    int64_t bx;
    int p0, p1;   // records: fewer than 2^30
    {
        int64_t t0, t1;
        stream_item(A, w, sm, bx, t0, t1);
        p0 = (int)(t0 * kPT);
        p1 = (int)(t1 * kPT);
    }
    // this thread's first pair record moves into L1 while the i-particle loads
    // are in flight (a prefetch holds no registers)
    if (p0 + tid < p1) {
        const char *a = reinterpret_cast<const char *>(A.j.p + p0 + tid);
        asm volatile("prefetch.global.L1 [%0];" ::"l"(a));
        asm volatile("prefetch.global.L1 [%0];" ::"l"(a + 64));
    }
    IPk ip[R];
    int32_t gi[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t ii = bx * R + r;
        gi[r] = idx_at(A, sm, ii < sm->s ? ii : sm->s - 1);
        ip[r] = ipk_of(jrec_load(A.j.p, gi[r]));
    }
    const float2 e2 = make_float2(A.eps2f, A.eps2f);
    AccPk p[R];
    Acc7 hi[R], lo[R];
#pragma unroll
    for (int r = 0; r < R; ++r) { zero(p[r]); zero(hi[r]); zero(lo[r]); }
    // two pair records per thread in flight (their loads are issued together), a fold
    // after every kFoldPairs / 2 records, i.e. 64 tiles (R = 2: at the end of them)
    constexpr int kPart = kFoldTiles * kPT;
    int cnt = 0;
    bool more = false;
    do {
        const int pe = LONG && p1 - p0 > kPart ? p0 + kPart : p1;
        for (int pp = p0 + tid; pp < pe; pp += 2 * kThreads) {
            const int pq = pp + kThreads < pe ? pp + kThreads : pp;
            float4 a0, a1, a2, a3, a4, b0, b1, b2, b3, b4;
            {
                const float4 *q = A.j.p[pp].q;
                const float4 *w = A.j.p[pq].q;
                a0 = __ldg(q); a1 = __ldg(q + 1); a2 = __ldg(q + 2); a3 = __ldg(q + 3); a4 = __ldg(q + 4);
                b0 = __ldg(w); b1 = __ldg(w + 1); b2 = __ldg(w + 2); b3 = __ldg(w + 3); b4 = __ldg(w + 4);
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
                pair_packed<true>(a0, a1, a2, a3, a4, ip[r], e2, p[r], 2 * pp == gi[r], 2 * pp + 1 == gi[r]);
            if (pq != pp) {
#pragma unroll
                for (int r = 0; r < R; ++r)
                    pair_packed<true>(b0, b1, b2, b3, b4, ip[r], e2, p[r], 2 * pq == gi[r], 2 * pq + 1 == gi[r]);
            }
            cnt += 2;
            if (R == 1 && cnt >= kFoldPairs / 2) {
                cnt = 0;
                fold(hi[0], lo[0], p[0]);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            fold(hi[r], lo[r], p[r]);
            cta_sum_red(hi[r], lo[r], &sm->red[warp][7 * r], LONG && more);
            if (LONG) {
                zero(hi[r]);
                zero(lo[r]);
            }
        }
        more = true;
        p0 = pe;
    } while (LONG && p0 < p1);
    __syncthreads();
    cta_sum_out<R>(A, w, sm);
    __syncthreads();
}

// --------------------------------------------------- TMA streaming variant
// TI = 1: all threads share one i-particle; the item's j-tiles stream through a
// ring of kRing shared-memory stages filled by the TMA bulk engine, so that
// kRing x 10 KB per CTA are in flight without holding registers (for blocks of
// one or two particles the evaluation is bound by reading the j-records). The
// two halves of the CTA take consecutive tiles, a thread one pair record of its
// half's tile.
__device__ __forceinline__ void issue_ring(const ForceArgs &A, Smem *sm, int64_t tile, int st)
{
    constexpr uint32_t bytes = kPT * sizeof(JPair);
    mbar_arrive_expect_tx(&sm->bar[st], bytes);
    bulk_g2s(sm->ring[st], A.j.p + tile * kPT, bytes, &sm->bar[st]);
}

__device__ void work_stream_tma(const ForceArgs &A, int64_t w, Smem *sm, uint32_t &git)
{
    static_assert(kThreads == 2 * kPT, "each half of the CTA takes one tile");
    const int tid = threadIdx.x;
    int64_t bx, t0, t1;
    stream_item(A, w, sm, bx, t0, t1);
    const int64_t s = sm->s;
    const int64_t nt = t1 > t0 ? t1 - t0 : 0;
    if (tid == 0) {
        const int64_t pro = nt < kRing ? nt : kRing;
        for (int64_t q = 0; q < pro; ++q) issue_ring(A, sm, t0 + q, (int)((git + q) % kRing));
    }
    const int32_t gi = idx_at(A, sm, bx < s ? bx : s - 1);
    const IPk ip = ipk_of(jrec_load(A.j.p, gi));
    const float2 e2 = make_float2(A.eps2f, A.eps2f);
    const int half = tid / kPT, r = tid % kPT;
    AccPk p;
    Acc7 hi, lo;
    zero(p);
    zero(hi);
    zero(lo);
    int cnt = 0;
    for (int64_t q = 0; q < nt; q += 2) {
        const int64_t qh = q + half;
        if (qh < nt) {
            const uint32_t g = git + (uint32_t)qh;
            const int st = (int)(g % kRing);
            if (!mbar_wait(&sm->bar[st], (g / kRing) & 1u, A.spin_limit)) {
                sm->abort = 1;
            } else {
                const float4 *Q = sm->ring[st][r].q;
                const float4 q0 = Q[0], q1 = Q[1], q2 = Q[2], q3 = Q[3], q4 = Q[4];
                const int64_t ja = (t0 + qh) * kJT + 2 * r;
                pair_packed<true>(q0, q1, q2, q3, q4, ip, e2, p, ja == gi, ja + 1 == gi);
                if (++cnt == kFoldPairs / 2) {
                    cnt = 0;
                    fold(hi, lo, p);
                }
            }
        }
        __syncthreads();   // both tiles read: their stages may be refilled
        if (sm->abort) {
            // a wait ran out: drain what this CTA still has in flight (bounded), then stop
            // (tiles q .. q + kRing - 1 were issued; each wait is bounded)
            if (tid == 0) {
                for (int64_t qq = q; qq < nt && qq < q + kRing; ++qq) {
                    const uint32_t gg = git + (uint32_t)qq;
                    (void)mbar_wait(&sm->bar[gg % kRing], (gg / kRing) & 1u, A.spin_limit);
                }
            }
            git += (uint32_t)nt;
            return;
        }
        if (tid == 0) {
            for (int64_t qq = q + kRing; qq < q + kRing + 2 && qq < nt; ++qq)
                issue_ring(A, sm, t0 + qq, (int)((git + qq) % kRing));
        }
    }
    git += (uint32_t)nt;
    fold(hi, lo, p);
    cta_sum_red(hi, lo, sm->red[tid >> 5]);
    __syncthreads();
    cta_sum_out<1>(A, w, sm);
    __syncthreads();
}

// ----------------------------------------------------------- column kernel
// Variants 1 to 4: blocks of more than a few particles (see short_items).
//
// A variant's FP32 partial sums run over 32 pair records each before they are folded
// into the two-sum accumulators. Over the records of a share (the table's split S gives
// every i-particle S shares of tper tiles) they form columns: with stride st (256, 32, 8
// or 1 records for variants 1, 2, 3, 4), 32 st consecutive records are a 32 x st matrix,
// row by row, and each column is one FP32 sum (for st = 1 a column is 32 consecutive
// records). The order of the columns is free: it only enters the two-sums. So
//   * a unit is up to kUnitRec records, as many whole columns of one matrix as fit; its
//     rows are copied into shared memory by the bulk engine, kSlots units in flight;
//   * a CTA holds an i-block of I = 256 / TJ particles, TJ threads to each on different
//     columns. Neighbouring lanes hold different particles and the same column, so a
//     record is one broadcast for a warp (lanes on four columns would take twice the
//     shared-memory wavefronts and hold the loop up). No record is read from L2 more
//     than once per i-block, and the TJ threads' sums meet once per i-block;
//   * the (i-block, unit) pairs are laid out in one line and cut into equal runs, one
//     per CTA, whatever s, n and S. A run may end one i-block and begin the next; the
//     last CTA of an i-block adds its partials in CTA order.
//
// What bounds it: the operand reads of the pair arithmetic (the register file delivers
// two 32-bit operands per lane and clock; a packed FMA with three distinct operands
// takes 1.45x one with two, so a record costs ~90 clocks a warp where the FP32 pipe
// alone would take 76), i.e. 8.9e11 pairs/s. Measured against items of (i-block, share)
// with 1, 2, 8, 32 or 256 particles, dealt out in advance (us a call): N = 65536: s = 480
// 71.3 -> 59.4, 1024 150 -> 100, 5000 862 -> 417, N 5850 -> 5010; N = 200000, s = 700 298
// -> 196; N = 300007: s = 33 49 -> 31, 61 47.9 -> 39.6; N = 2^20: s = 64 115 -> 104, 1024
// 1424 -> 1300; N = s = 131072 20480 -> 19990 (94 clocks a record).

__device__ __forceinline__ int variant_lgst(int v) { return v == 1 ? 8 : (v == 2 ? 5 : (v == 3 ? 3 : 0)); }
// tiles per matrix (log2)
__device__ __forceinline__ int matrix_lg(int lgst) { return lgst == 8 ? 6 : (lgst == 5 ? 3 : 1); }

// Threads per particle (log2, at most 5). Wide i-blocks read each record for more
// particles; narrower ones leave fewer lanes without a particle (at most 1 in 16
// here), give every i-block fewer partials (the last CTA adds I G / nib of 64 bytes
// each, kept near kColSum bytes), and cut the work finer (kColUnits units per CTA for
// equal runs; not below 32 particles for this).
constexpr int64_t kColSum = 128 << 10;
constexpr int64_t kColUnits = 16;
__device__ __forceinline__ int cols_lgtj(int64_t s, int64_t grid, int64_t upi)
{
    int lg = 0;
    for (; lg < 5; ++lg) {
        const int64_t I = kThreads >> lg, nib = (s + I - 1) >> (8 - lg);
        if (16 * (nib * I - s) <= s && I * grid * 64 <= kColSum * nib && (lg >= 3 || nib * upi >= kColUnits * grid))
            break;
    }
    return lg;
}

// Partial slots per particle: an i-block meets at most ceil(G / nib) + 1 runs.
__device__ __forceinline__ int cols_slots(int64_t G, int64_t nib) { return (int)(G <= nib ? 2 : qdiv(G + nib - 1, nib) + 1); }

// (few divisions: they are the longest part of the start of a small launch)
__device__ __forceinline__ ColPlan cols_plan(const ForceArgs &A, int variant, int64_t s, int S)
{
    ColPlan P;
    const int64_t T = A.tile_hi - A.tile_lo, grid = gridDim.x, me = blockIdx.x;
    P.tper = S == 1 ? T : qdiv(T + S - 1, S);
    const int64_t shares = S == 1 ? 1 : qdiv(T + P.tper - 1, P.tper);
    P.lgst = variant_lgst(variant);
    // rows of a share's first matrix, columns per unit
    const int lgmt = matrix_lg(P.lgst);
    const int nt = P.tper < (1 << lgmt) ? (int)P.tper : 1 << lgmt;
    const int rows = P.lgst == 8 ? (nt + 1) / 2 : (P.lgst == 5 ? 4 * nt : (P.lgst == 3 ? 16 * nt : 32));
    const int top = P.lgst == 8 ? 7 : (P.lgst == 5 ? 5 : 3);
    P.lgcw = rows <= 1 ? 8 : 8 - (32 - __clz(rows - 1));   // floor(log2(kUnitRec / rows))
    if (P.lgcw > top) P.lgcw = top;
    P.ups = (int)((P.tper + (1 << lgmt) - 1) >> lgmt) << (P.lgst > P.lgcw ? P.lgst - P.lgcw : 0);
    P.upi = shares * P.ups;
    P.lgtj = cols_lgtj(s, grid, P.upi);
    P.nib = (s + (kThreads >> P.lgtj) - 1) >> (8 - P.lgtj);
    P.slots = cols_slots(grid, P.nib);
    // never more partials than there is room for (the no-allocation entry point has room
    // for few): more, smaller i-blocks; without any room, whole i-blocks to a CTA
    while (s * P.slots * kPartStride > A.part_cap && P.lgtj < 5) {
        ++P.lgtj;
        P.nib = (s + (kThreads >> P.lgtj) - 1) >> (8 - P.lgtj);
        P.slots = cols_slots(grid, P.nib);
    }
    const bool whole = s * P.slots * kPartStride > A.part_cap;
    if (whole) {
        P.lgtj = 3;
        P.nib = (s + (kThreads >> P.lgtj) - 1) >> (8 - P.lgtj);
    }
    P.U = P.nib * P.upi;
    const int64_t line = whole ? P.nib : P.U, step = whole ? P.upi : 1;
    P.G = grid < line ? grid : line;
    P.u0 = P.u1 = P.b0 = 0;
    if (me < P.G) {
        P.u0 = qdiv(line * me, P.G) * step;
        P.u1 = qdiv(line * (me + 1), P.G) * step;
        P.b0 = qdiv(P.u0, P.upi);
    }
    P.whole = whole ? 1 : 0;
    return P;
}

// Where unit u of an i-block lies: record `rec` is row 0 of its first column, `rows`
// rows of `cols` columns, 2^lgst records apart (st = 1: `cols` columns of 32
// consecutive records).
struct Unit {
    int64_t rec;
    int rows, cols;
};
__device__ __forceinline__ Unit unit_at(const ForceArgs &A, const ColPlan &P, int64_t u)
{
    const int64_t sh = P.upi == P.ups ? 0 : qdiv(u, P.ups);
    const int v = (int)(u - sh * P.ups);
    const int64_t t0 = A.tile_lo + sh * P.tper;
    const int64_t t1 = t0 + P.tper < A.tile_hi ? t0 + P.tper : A.tile_hi;
    const int lgch = P.lgst > P.lgcw ? P.lgst - P.lgcw : 0;   // column chunks per matrix
    const int m = v >> lgch, c0 = (v - (m << lgch)) << P.lgcw;
    const int lgmt = matrix_lg(P.lgst);
    const int64_t ts = t0 + ((int64_t)m << lgmt);
    int nt = t1 - ts < (1 << lgmt) ? (int)(t1 - ts) : 1 << lgmt;
    if (nt < 0) nt = 0;
    Unit q;
    q.rec = ts * kPT + c0;
    q.cols = P.lgst == 0 ? 4 * nt : 1 << P.lgcw;
    q.rows = P.lgst == 8 ? (c0 >= 128 ? nt / 2 : (nt + 1) / 2) : (P.lgst == 5 ? 4 * nt : (P.lgst == 3 ? 16 * nt : 32));
    return q;
}

// The unit, column and row of record r of the range (unit -1: r is outside the range).
__device__ __forceinline__ int64_t unit_of(const ForceArgs &A, const ColPlan &P, int64_t r, int &col, int &row)
{
    col = row = 0;
    const int64_t tile = (r >> 7) - A.tile_lo;
    if (tile < 0 || r >= A.tile_hi * kPT) return -1;
    const int64_t sh = P.upi == P.ups ? 0 : qdiv(tile, P.tper);
    const int64_t rs = r - (A.tile_lo + sh * P.tper) * kPT;   // record within the share
    const int lgm = 7 + matrix_lg(P.lgst);                    // records per matrix
    const int64_t m = rs >> lgm;
    const int rm = (int)(rs - (m << lgm));
    if (P.lgst == 0) {
        col = rm >> 5;
        row = rm & 31;
        return sh * P.ups + m;
    }
    const int c = rm & ((1 << P.lgst) - 1);
    row = rm >> P.lgst;
    col = c & ((1 << P.lgcw) - 1);
    return sh * P.ups + (m << (P.lgst - P.lgcw)) + (c >> P.lgcw);
}

// Copies unit u into its slot (called by one warp): one copy where the unit's records
// are consecutive, else one per row.
__device__ __forceinline__ void unit_issue(const ForceArgs &A, Smem *sm, const ColPlan &P, int64_t u, int slot)
{
    const int lane = threadIdx.x & 31;
    const Unit q = unit_at(A, P, u);
    const uint32_t row = (uint32_t)sizeof(JPair) << P.lgcw;
    const uint32_t all = P.lgst == 0 ? (uint32_t)q.cols * 32u * (uint32_t)sizeof(JPair) : (uint32_t)q.rows * row;
    if (lane == 0) {
        sm->info[slot] = make_int2(q.rows, q.cols);   // read by the warps after the slot's barrier
        mbar_arrive_expect_tx(&sm->bar[slot], all);
    }
    __syncwarp();
    if (P.lgst <= 3) {
        if (lane == 0 && all) bulk_g2s(sm->unit[slot], A.j.p + q.rec, all, &sm->bar[slot]);
    } else if (lane < q.rows) {
        bulk_g2s(sm->unit[slot] + lane * row, A.j.p + q.rec + ((int64_t)lane << P.lgst), row, &sm->bar[slot]);
    }
}

// One column: rows records of hop bytes from src (ROWS, HOP: the usual ones, known to the
// compiler). self: the row holding the i-particle itself, in lane b of the record if
// odd; -1: none.
template <bool MASK, int ROWS, int HOP>
__device__ __forceinline__ void sweep_column(const unsigned char *src, int rows, int hop, int self, bool odd,
                                             const IPk &ip, float2 e2, AccPk &p)
{
    if (ROWS) rows = ROWS;
    if (HOP) hop = HOP;
#pragma unroll 4
    for (int m = 0; m < rows; ++m) {
        const float4 *Q = reinterpret_cast<const float4 *>(src + m * hop);
        const float4 q0 = Q[0], q1 = Q[1], q2 = Q[2], q3 = Q[3], q4 = Q[4];
        pair_packed<MASK>(q0, q1, q2, q3, q4, ip, e2, p, MASK && m == self && !odd, MASK && m == self && odd);
    }
}

// The sums of i-block b: every thread's (hi, lo), first over the lanes of a warp that
// hold the same particle (I < 32), then over the warps through shared memory, into the
// CTA's partial slot or, with n == 1 (no other CTA has a part), the results.
__device__ __forceinline__ void cols_out(const ForceArgs &A, int64_t s, int64_t ib0, int lgi, int n, int slot, Acc7 &hi,
                                         Acc7 &lo, Smem *sm)
{
    const int tid = threadIdx.x;
    for (int off = 16; off >= (1 << lgi); off >>= 1) {
        Acc7 h2, l2;
        h2.ax = __shfl_xor_sync(0xffffffffu, hi.ax, off); l2.ax = __shfl_xor_sync(0xffffffffu, lo.ax, off);
        h2.ay = __shfl_xor_sync(0xffffffffu, hi.ay, off); l2.ay = __shfl_xor_sync(0xffffffffu, lo.ay, off);
        h2.az = __shfl_xor_sync(0xffffffffu, hi.az, off); l2.az = __shfl_xor_sync(0xffffffffu, lo.az, off);
        h2.kx = __shfl_xor_sync(0xffffffffu, hi.kx, off); l2.kx = __shfl_xor_sync(0xffffffffu, lo.kx, off);
        h2.ky = __shfl_xor_sync(0xffffffffu, hi.ky, off); l2.ky = __shfl_xor_sync(0xffffffffu, lo.ky, off);
        h2.kz = __shfl_xor_sync(0xffffffffu, hi.kz, off); l2.kz = __shfl_xor_sync(0xffffffffu, lo.kz, off);
        h2.ph = __shfl_xor_sync(0xffffffffu, hi.ph, off); l2.ph = __shfl_xor_sync(0xffffffffu, lo.ph, off);
        ds_add(hi.ax, lo.ax, h2.ax, l2.ax);
        ds_add(hi.ay, lo.ay, h2.ay, l2.ay);
        ds_add(hi.az, lo.az, h2.az, l2.az);
        ds_add(hi.kx, lo.kx, h2.kx, l2.kx);
        ds_add(hi.ky, lo.ky, h2.ky, l2.ky);
        ds_add(hi.kz, lo.kz, h2.kz, l2.kz);
        ds_add(hi.ph, lo.ph, h2.ph, l2.ph);
    }
#pragma unroll
    for (int c = 0; c < 7; ++c) sm->sums[c][tid] = make_float2(acc_get(hi, c), acc_get(lo, c));
    __syncthreads();
    const int I = 1 << lgi, hop = I < 32 ? 32 : I, W = kThreads / hop;
    for (int o = tid; o < 8 * I; o += kThreads) {
        const int c = o & 7, i = o >> 3;
        if (c == 7 || ib0 + i >= s) continue;
        float h = sm->sums[c][i].x, l = sm->sums[c][i].y;
        for (int w = 1; w < W; ++w) ds_add(h, l, sm->sums[c][i + w * hop].x, sm->sums[c][i + w * hop].y);
        if (n == 1)
            put_final(A, ib0 + i, c, (double)h + (double)l);
        else
            part2(A, ib0 + i, slot, sm->plan.slots)[c] = make_float2(h, l);
    }
}

// This CTA's run. False: a wait ran out.
__device__ bool work_cols(const ForceArgs &A, int64_t s, Smem *sm)
{
    const ColPlan &P = sm->plan;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int lgtj = P.lgtj, lgi = 8 - lgtj, tj = tid >> lgi, ti = tid & ((1 << lgi) - 1);
    const int lgnu = lgtj > P.lgcw ? lgtj - P.lgcw : 0;    // units side by side
    const int cstep = lgnu ? 1 << P.lgcw : 1 << lgtj;      // a thread's columns: c0, c0 + cstep, ...
    const int ncol = lgnu ? 1 : 1 << (P.lgcw - lgtj);      // of them per unit
    const int c0 = tj & (cstep - 1);
    const int mine = lgnu ? tj >> P.lgcw : 0;              // this thread's unit of a round
    // Slots are refilled one unit behind, when all warps have most likely left it. Rounds of
    // several units: at once (the warp whose turn it is waits for the slowest), so that the
    // next round's units are on their way. One round behind they were not: N = 300007, s =
    // 61 39.4 -> 37.5 us under the profiler, N = 2^20, s = 61 103 -> 100.6.
    const int ahead = kSlots - (lgnu == 0 ? 1 : 0);
    const int hop = P.lgst == 0 ? (int)sizeof(JPair) : (int)sizeof(JPair) << P.lgcw;
    const int chop = P.lgst == 0 ? 32 * (int)sizeof(JPair) : (int)sizeof(JPair);
    const float2 e2 = make_float2(A.eps2f, A.eps2f);
    volatile int *stop = &sm->abort;
    const int64_t u0 = P.u0, u1 = P.u1;
    int64_t b = P.b0;
    int64_t ub = b * P.upi;         // first unit of i-block b
    const int64_t place0 = u0 - ub; // unit v of the run is at place (place0 + v) mod upi of its i-block
    if (warp < kSlots && u0 + warp < u1) unit_issue(A, sm, P, place0 + warp < P.upi ? place0 + warp : qmod(place0 + warp, P.upi), warp);
    uint32_t used = 0;              // units of the run this warp is done with
    bool ok = true;
    for (int64_t u = u0; u < u1; ++b, ub += P.upi) {
        const int64_t ue = ub + P.upi < u1 ? ub + P.upi : u1;
        const int64_t ib0 = b << lgi, ii = ib0 + ti;
        const int32_t gi = idx_at(A, sm, ii < s ? ii : s - 1);
        const IPk ip = ipk_of(jrec_load(A.j.p, gi));
        int scol, srow;
        const int64_t su = unit_of(A, P, gi >> 1, scol, srow) + ub;   // the i-particle's own place
        if (tid == 0) {
            // the runs that meet this i-block
            const int64_t first = qdiv((ub + 1) * P.G - 1, P.U);
            sm->plan.part_n = P.whole ? 1 : (int)(qdiv((ub + P.upi) * P.G - 1, P.U) - first) + 1;
            sm->plan.part_slot = (int)(blockIdx.x - first);
        }
        AccPk p;
        Acc7 hi, lo;
        zero(p);
        zero(hi);
        zero(lo);
        while (u < ue) {
            // a round: 2^lgnu units (the last one of an i-block or run may have fewer)
            const int cnt = ue - u < (1 << lgnu) ? (int)(ue - u) : 1 << lgnu;
            const bool have = mine < cnt;
            // The warp releases all the units of the round, so it waits for all their copies, not
            // only for its own unit's. Only then are the slots' earlier phases behind it: another
            // warp's releases of one round come from different lanes and may be seen in any
            // order, and a wait tests one parity bit, so that otherwise a release could count for
            // the phase before, or the refill's wait below pass on the phase two before.
            for (uint32_t v = used; v < used + (uint32_t)cnt; ++v)
                ok = mbar_wait(&sm->bar[v % kSlots], (v / kSlots) & 1u, A.spin_limit) && ok;
            if (__all_sync(0xffffffffu, ok)) {
                const int sl = (int)((used + (uint32_t)(have ? mine : 0)) % kSlots);
                const int2 q = sm->info[sl];
                const bool self = have && u + mine == su;
                const unsigned char *src = sm->unit[sl] + c0 * chop;
                const bool plain = have && !self && q.x == 32 && q.y >= cstep * ncol;
                if (__all_sync(0xffffffffu, plain) && (hop == (int)sizeof(JPair) || hop == 8 * (int)sizeof(JPair))) {
                    for (int it = 0; it < ncol; ++it, src += cstep * chop) {
                        if (hop == (int)sizeof(JPair))
                            sweep_column<false, 32, (int)sizeof(JPair)>(src, 32, hop, -1, false, ip, e2, p);
                        else
                            sweep_column<false, 32, 8 * (int)sizeof(JPair)>(src, 32, hop, -1, false, ip, e2, p);
                        fold(hi, lo, p);
                    }
                } else {
                    for (int it = 0; it < ncol; ++it, src += cstep * chop) {
                        const int c = c0 + it * cstep;
                        const int rows = have && c < q.y ? q.x : 0;
                        const bool here = self && c == scol;
                        if (__any_sync(0xffffffffu, here))
                            sweep_column<true, 0, 0>(src, rows, hop, here ? srow : -1, gi & 1, ip, e2, p);
                        else
                            sweep_column<false, 0, 0>(src, rows, hop, -1, false, ip, e2, p);
                        fold(hi, lo, p);
                    }
                }
            }
            if (!__all_sync(0xffffffffu, ok)) *stop = 1;
            if (*stop) break;
            __syncwarp();   // this warp has read the round's units
            if (lane < cnt) mbar_arrive(&sm->empty[(used + lane) % kSlots]);
            // the warps take turns at refilling
            for (int q = 0; q < cnt; ++q) {
                const uint32_t w = used + (uint32_t)(ahead + q);   // unit to copy
                if (w < kSlots || (w & (kThreads / 32 - 1)) != (uint32_t)warp || u0 + w >= u1) continue;
                ok = mbar_wait(&sm->empty[w % kSlots], (w / kSlots - 1) & 1u, A.spin_limit);
                if (!__all_sync(0xffffffffu, ok)) {
                    *stop = 1;
                    break;
                }
                unit_issue(A, sm, P, qmod(place0 + w, P.upi), (int)(w % kSlots));
            }
            used += cnt;
            u += cnt;
        }
        if (__syncthreads_or(!ok || *stop)) {
            // a wait ran out somewhere in the CTA: drain what may be in flight (bounded), stop
            if (tid == 0)
                for (uint32_t q = 0; q < 2 * kSlots; ++q) {
                    const uint32_t w = used + q < kSlots ? q : used + q - kSlots;
                    if (u0 + w < u1) (void)mbar_wait(&sm->bar[w % kSlots], (w / kSlots) & 1u, A.spin_limit);
                }
            return false;
        }
        const int n = sm->plan.part_n;
        cols_out(A, s, ib0, lgi, n, sm->plan.part_slot, hi, lo, sm);
        if (n > 1) {
            const int64_t ib1 = ib0 + (1 << lgi);
            finish_block<false>(A, b, ib0, ib1 < s ? ib1 : s, P.slots, n, sm);
        }
    }
    return true;
}

// --------------------------------------------------- short shares, variant 2
// Eight particles per CTA, one per warp, a lane per column (stride 32): an item's
// tiles, up to kShortRing at once, are copied into shared memory in one go. For blocks
// so small that one item per CTA covers them: no plan, no ring, no meeting of warps.
constexpr int kShortRing = (int)(sizeof(Smem::unit) / (kPT * sizeof(JPair)));
static_assert(kShortRing == 8, "the fold falls on whole turns (32 rows are 8 tiles)");

__device__ void work_tile32(const ForceArgs &A, int64_t w, Smem *sm, uint32_t &git)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int64_t bx, t0, t1;
    stream_item(A, w, sm, bx, t0, t1);
    const int64_t ii = bx * 8 + warp;
    const int32_t gi = idx_at(A, sm, ii < sm->s ? ii : sm->s - 1);
    IPk ip;
    AccPk p;
    Acc7 hi, lo;
    zero(p);
    zero(hi);
    zero(lo);
    const float2 e2 = make_float2(A.eps2f, A.eps2f);
    const JPair *rec = reinterpret_cast<const JPair *>(sm->unit[0]);
    for (int64_t t = t0; t < t1; t += kShortRing) {
        const int nt = t1 - t < kShortRing ? (int)(t1 - t) : kShortRing;
        if (tid == 0) {
            constexpr uint32_t bytes = kPT * sizeof(JPair);
            mbar_arrive_expect_tx(&sm->bar[0], (uint32_t)nt * bytes);
            for (int q = 0; q < nt; ++q)
                bulk_g2s(sm->unit[0] + q * bytes, A.j.p + (t + q) * kPT, bytes, &sm->bar[0]);
        }
        if (t == t0) ip = ipk_of(jrec_load(A.j.p, gi));
        // the particle's own row, if its record is in this lane's column
        const int64_t rel = (gi >> 1) - t * kPT;
        const int self = rel >= 0 && rel < nt * kPT && ((int)rel & 31) == lane ? (int)rel >> 5 : -1;
        if (!mbar_wait(&sm->bar[0], git & 1u, A.spin_limit)) sm->abort = 1;
        ++git;
        if (__syncthreads_or(sm->abort)) return;   // (the wait that failed was the drain)
#pragma unroll 4
        for (int m = 0; m < 4 * nt; ++m) {
            const float4 *Q = rec[32 * m + lane].q;
            pair_packed<true>(Q[0], Q[1], Q[2], Q[3], Q[4], ip, e2, p, m == self && !(gi & 1), m == self && (gi & 1));
        }
        fold(hi, lo, p);
        __syncthreads();   // the tiles have been read
    }
    float h, l;
    const int c = ds_scatter_reduce<32>(hi, lo, h, l);
    if ((lane & 3) == 0 && c < 7 && ii < sm->s) {
        if (sm->split == 1)
            put_final(A, ii, c, (double)h + (double)l);
        else
            part2(A, ii, (int)(w - bx * sm->split), sm->split)[c] = make_float2(h, l);
    }
}

// -------------------------------------------------------------- variants

// 0: stream (one particle per CTA)   5: TMA stream (the same sums)
// 1, 2, 3, 4: columns with stride 256, 32, 8, 1
// 6: resident share (cluster launch; the split factor is unused)
constexpr int kMixedFallback = kMixedFallbackId;   // the variant of an out-of-range table entry
constexpr int kShareVariant = kShareVariantId;
__host__ __device__ __forceinline__ int mixed_I(int v)
{
    switch (v) {
    case 0: return 1;
    case 1: return 2;
    case 2: return 8;
    case 3: return 32;
    case 5: return 1;
    case 6: return 1;
    default: return 256;
    }
}

// ------------------------------------------------- resident-share variant
// For j ranges of up to kShareC * kShareRec pair records. The launch runs as
// clusters of kShareC CTAs; CTA r of a cluster copies records [r * rper, (r + 1)
// * rper) of the range into shared memory once (bulk copies of kSharePiece records, each
// on its own mbarrier: the first pass starts on the first piece), padded with far-away
// massless records to whole rounds of 32. The clusters deal out the active list in
// chunks (chunk k to cluster k mod clusters); every CTA of the cluster runs the whole
// chunk against its share in passes whose group width TJ fits the remaining count, and
// pushes each position's (hi, lo) partial sums into the shared memory of the CTA that
// finishes it (position mod kShareC). One cluster barrier later that CTA adds the
// kShareC partials from its own shared memory, in a fixed tree over the ranks, and
// writes the FP64 results. No global partial slots, tickets or fences; the same bits on
// every run. Bound by latency up to a few hundred particles; us under the profiler, with
// one wait for the whole share, partials read across the cluster after the barrier and a
// second barrier / now: N = 16384, s = 20 9.2 / 7.9, 100 12.7 / 11.0, 256 14.6 / 14.0, 2000 55.2 / 54.0.

// rper: records per CTA, a multiple of 32 (0 when the range does not fit)
__device__ __forceinline__ int64_t share_rper(const ForceArgs &A)
{
    const int64_t nrec = (A.tile_hi - A.tile_lo) * kPT;
    const int64_t rper = ((nrec + kShareC - 1) / kShareC + 31) / 32 * 32;
    return rper <= kShareRec ? rper : 0;
}

// Waits for the share's pieces up to the one holding record r (ready: pieces this thread
// has waited for). On a timeout the status is set and the copy gets a second wait, so that
// none is in flight when the CTA ends.
__device__ __forceinline__ void share_wait(const ForceArgs &A, Smem *sm, int r, int &ready)
{
    for (const int need = r / kSharePiece + 1; ready < need; ++ready)
        if (!mbar_wait(&sm->bar[ready], 0, A.spin_limit)) {
            atomicOr(A.status, kStTimeout);
            (void)mbar_wait(&sm->bar[ready], 0, A.spin_limit);
        }
}

// Sends component c of the partial sums of chunk position pl to the CTA that finishes it.
__device__ __forceinline__ void share_push(Smem *sm, int rank, int pl, int c, float h, float l)
{
    cg::cluster_group cl = cg::this_cluster();
    *cl.map_shared_rank(&shb(sm)->in[pl / kShareC][rank][c], pl % kShareC) = make_float2(h, l);
}

// One pass: cnt particles from list position p0, chunk positions slot0 ..., TJ threads
// per particle taking records tj, tj + TJ, ... of the share (nr rounds).
template <int TJ>
__device__ __forceinline__ void share_pass(const ForceArgs &A, Smem *sm, int64_t p0, int cnt, int slot0,
                                           int64_t rec0, int nrec, int nr, int rank, int &ready)
{
    constexpr int FP = kFoldPairs / 2;   // rounds per fold
    constexpr int STEP = kSharePiece / TJ < FP ? kSharePiece / TJ : FP;   // rounds of one piece, within a fold
    const int tid = threadIdx.x, tj = tid % TJ, ti = tid / TJ;
    const bool live = ti < cnt;
    const int32_t gi = idx_at(A, sm, p0 + (live ? ti : cnt - 1));
    const IPk ip = ipk_of(jrec_load(A.j.p, gi));
    const float2 e2 = make_float2(A.eps2f, A.eps2f);
    AccPk p;
    Acc7 hi, lo;
    zero(p);
    zero(hi);
    zero(lo);
    // the round holding i's own record, if this thread meets it
    const int64_t self = ((int64_t)gi >> 1) - rec0;
    const int selfk = self >= 0 && self < (int64_t)nrec && (int)self % TJ == tj ? (int)self / TJ : -1;
    const JPair *R = shb(sm)->rec;
    // the first pass follows the pieces as they arrive, the later ones go fold by fold
    const int step = ready < kShareRec / kSharePiece ? STEP : FP;
    for (int k0 = 0; k0 < nr; k0 += step) {
        const int k1 = k0 + step < nr ? k0 + step : nr;
        share_wait(A, sm, k1 * TJ - 1, ready);
        if (__any_sync(0xffffffffu, selfk >= k0 && selfk < k1)) {
#pragma unroll 2
            for (int k = k0; k < k1; ++k) {
                const float4 *Q = R[tj + k * TJ].q;
                pair_packed<true>(Q[0], Q[1], Q[2], Q[3], Q[4], ip, e2, p, k == selfk && !(gi & 1),
                                  k == selfk && (gi & 1));
            }
        } else {
#pragma unroll 2
            for (int k = k0; k < k1; ++k) {
                const float4 *Q = R[tj + k * TJ].q;
                pair_packed<false>(Q[0], Q[1], Q[2], Q[3], Q[4], ip, e2, p, false, false);
            }
        }
        if (k1 % FP == 0 || k1 == nr) fold(hi, lo, p);
    }
    // the group's sums; every lane ends with max(1, 8 / TJ) of the components
    constexpr int N = TJ >= 8 ? 1 : 8 / TJ;
    constexpr int kRun = TJ > 8 ? TJ / 8 : 1;   // lanes left with the same sum
    float sh[N], sl[N];
    const int first = ds_scatter_reduce<TJ, N>(hi, lo, sh, sl);
    if (live && (tj & (kRun - 1)) == 0) {
#pragma unroll
        for (int c = 0; c < N; ++c)
            if (first + c < 7) share_push(sm, rank, slot0 + ti, first + c, sh[c], sl[c]);
    }
}

// A pass for cnt <= 8 / W particles with W warps each: lanes then warps of a particle
// summed in ascending order. The rounds of one piece at a time, side by side.
template <int W>
__device__ __forceinline__ void share_pass_wide(const ForceArgs &A, Smem *sm, int64_t p0, int cnt, int slot0,
                                                int64_t rec0, int nrec, int nrec32, int rank, int &ready)
{
    constexpr int FP = kFoldPairs / 2;
    constexpr int TW = 32 * W;               // threads per particle
    constexpr int G = kSharePiece / TW;      // rounds per piece
    static_assert(kShareRec / TW <= FP, "one fold");
    const int tid = threadIdx.x, warp = tid >> 5;
    const int ti = tid / TW, tj = tid % TW;
    const bool live = ti < cnt;
    const int32_t gi = idx_at(A, sm, p0 + (live ? ti : cnt - 1));
    const IPk ip = ipk_of(jrec_load(A.j.p, gi));
    const float2 e2 = make_float2(A.eps2f, A.eps2f);
    AccPk p;
    Acc7 hi, lo;
    zero(p);
    zero(hi);
    zero(lo);
    const int64_t self = (int64_t)gi - 2 * rec0;
    const int selfi = self >= 0 && self < 2 * (int64_t)nrec ? (int)self : -2;
    const JPair *R = shb(sm)->rec;
    for (int b0 = 0; b0 < nrec32; b0 += kSharePiece) {
        share_wait(A, sm, b0, ready);
#pragma unroll
        for (int u = 0; u < G; ++u) {
            const int pp = b0 + u * TW + tj;
            if (pp < nrec32) {
                const float4 *Q = R[pp].q;
                pair_packed<true>(Q[0], Q[1], Q[2], Q[3], Q[4], ip, e2, p, 2 * pp == selfi, 2 * pp + 1 == selfi);
            }
        }
    }
    fold(hi, lo, p);
    cta_sum_red(hi, lo, sm->red[warp]);
    __syncthreads();
    if (tid < cnt * 7) {
        const int t = tid / 7, c = tid % 7;
        float h = sm->red[t * W][c].x, l = sm->red[t * W][c].y;
#pragma unroll
        for (int wv = 1; wv < W; ++wv) ds_add(h, l, sm->red[t * W + wv][c].x, sm->red[t * W + wv][c].y);
        share_push(sm, rank, slot0 + t, c, h, l);
    }
    __syncthreads();
}

// The whole launch of the resident-share variant for this CTA.
__device__ __noinline__ void share_force(const ForceArgs &A, int64_t s, Smem *sm, int64_t rper)
{
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int q = blockIdx.x / kShareC, ncl = gridDim.x / kShareC;
    const int tid = threadIdx.x;
    const int64_t rtot = (A.tile_hi - A.tile_lo) * kPT;
    const int64_t rec0 = A.tile_lo * kPT + (int64_t)rank * rper;
    const int64_t rlim = A.tile_lo * kPT + rtot;
    const int nrec = (int)(rec0 < rlim ? (rlim - rec0 < rper ? rlim - rec0 : rper) : 0);
    const int nrec32 = (nrec + 31) / 32 * 32;
    // chunks: ceil(s / clusters) particles each (at most kShareSlots)
    int64_t csz = qdiv(s + ncl - 1, ncl);
    if (csz > kShareSlots) csz = kShareSlots;
    const int64_t nchunk = qdiv(s + csz - 1, csz);
    if (q >= nchunk) return;   // the whole cluster has nothing to do (uniform over it)
    // no CTA writes into another's shared memory before all of the cluster run: arrive
    // here, wait before the first pass
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    if (tid < kShareRec / kSharePiece) {
        // (a piece past the share completes at once)
        const int r0 = tid * kSharePiece;
        const int nr = nrec - r0 < kSharePiece ? nrec - r0 : kSharePiece;
        const uint32_t bytes = nr > 0 ? (uint32_t)nr * (uint32_t)sizeof(JPair) : 0u;
        mbar_arrive_expect_tx(&sm->bar[tid], bytes);
        if (nr > 0) bulk_g2s(shb(sm)->rec + r0, A.j.p + rec0 + r0, bytes, &sm->bar[tid]);
    }
    {
        const float far = (float)kPadPos;
        for (int qq = 2 * nrec + tid; qq < 2 * nrec32; qq += kThreads)
            jrec_store(shb(sm)->rec, qq, far, far, far, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    int ready = 0;
    for (int64_t k = q; k < nchunk; k += ncl) {
        const int64_t c0 = k * csz;
        const int cnt = (int)(c0 + csz < s ? csz : s - c0);
        int done = 0;
        while (done < cnt) {
            const int r = cnt - done;
            if (r >= 256) {
                share_pass<1>(A, sm, c0 + done, 256, done, rec0, nrec, nrec32, rank, ready);
                done += 256;
            } else if (r >= 128) {
                share_pass<2>(A, sm, c0 + done, 128, done, rec0, nrec, nrec32 / 2, rank, ready);
                done += 128;
            } else if (r >= 64) {
                share_pass<4>(A, sm, c0 + done, 64, done, rec0, nrec, nrec32 / 4, rank, ready);
                done += 64;
            } else if (r >= 32) {
                share_pass<8>(A, sm, c0 + done, 32, done, rec0, nrec, nrec32 / 8, rank, ready);
                done += 32;
            } else if (r > 8) {
                const int n16 = r < 16 ? r : 16;
                share_pass<16>(A, sm, c0 + done, n16, done, rec0, nrec, nrec32 / 16, rank, ready);
                done += n16;
            } else if (r > 4) {
                share_pass<32>(A, sm, c0 + done, r, done, rec0, nrec, nrec32 / 32, rank, ready);
                done += r;
            } else {
                if (r == 1)
                    share_pass_wide<8>(A, sm, c0 + done, r, done, rec0, nrec, nrec32, rank, ready);
                else if (r == 2)
                    share_pass_wide<4>(A, sm, c0 + done, r, done, rec0, nrec, nrec32, rank, ready);
                else
                    share_pass_wide<2>(A, sm, c0 + done, r, done, rec0, nrec, nrec32, rank, ready);
                done += r;
            }
        }
        cl.sync();   // every CTA's partials are in the finishing CTAs' shared memory
        // positions rank, rank + kShareC, ...: one (position, component) per thread
        for (int t = tid; t < ((cnt + kShareC - 1) / kShareC) * 7; t += kThreads) {
            const int pl = rank + kShareC * (t / 7), c = t % 7;
            if (pl < cnt) {
                float2 v[kShareC];
#pragma unroll
                for (int u = 0; u < kShareC; ++u) v[u] = shb(sm)->in[t / 7][u][c];
#pragma unroll
                for (int d = 1; d < kShareC; d <<= 1) {
#pragma unroll
                    for (int u = 0; u < kShareC; u += 2 * d) ds_add(v[u].x, v[u].y, v[u + d].x, v[u + d].y);
                }
                put_final(A, c0 + pl, c, (double)v[0].x + (double)v[0].y);
            }
        }
        if (k + ncl < nchunk) cl.sync();   // the partials have been read: the next chunk may push
    }
    // a CTA whose passes met no record of a piece still waits for its copy before it ends
    share_wait(A, sm, kShareRec - 1, ready);
}

// Variants 1 and 2 where one item (two or eight particles, one share) per CTA covers the
// block: short shares always, since such a launch is a chain of latencies, and the columns'
// plan, ring and meeting of warps lengthen it (us under the profiler, items against columns: N =
// 10^5, s = 2 10.4 / 17.2, s = 24 13.2 / 15.9; N = 65536, s = 20 12.4 / 15.5). Longer ones take as long
// as their tiles, 9 + 0.215 t us for t of them, whatever their number; the columns as long as there
// are particles, about 11.5 + 0.096 n us for n items of 64 to 128 tiles, whatever the share (its
// last matrix is cut into as many units as a full one). The line is where the two meet. Items /
// columns, us a call in a graph: N = 16385, s = 200 15.2 / 18.6, 512 23.3 / 36.0; N = 20000, s = 300 25.1 /
// 23.0, 400 26.2 / 29.5; N = 24576, s = 257 28.8 / 23.0, 512 30.9 / 36.4; N = 49152, s = 104 19.0 / 24.5;
// N = 32768, s = 512 38.0 / 36.0; N = 2^20, s = 20 48.1 / 54.4. More items than CTAs: the columns (N =
// 65536, s = 65 29.9 / 22.1).
__device__ __forceinline__ bool short_items(int variant, int64_t T, int S, int64_t items)
{
    return variant <= 2 && items <= gridDim.x &&
           (T <= kShortTiles * (int64_t)S || (T <= kItemTiles * (int64_t)S && 9 * T <= (4 * items + 100) * S));
}

// SHARE: the instantiation with the resident-share variant (launched as clusters
// with kSmemShare bytes); without it the kernel has no cluster code and the
// plain shared-memory size.
template <bool SHARE>
__global__ void __launch_bounds__(kThreads, 2) force_mixed_kernel(ForceArgs A)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Smem *sm = reinterpret_cast<Smem *>(smem_raw);
    const int tid = threadIdx.x;
    // a launch that depends on this one programmatically (the nb_run loop's
    // corrector) may start now: it reads only what was written before this kernel
    // until it waits for this grid's completion
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // read ahead of s: entries past s are stale and never used (idx_cap >= s)
    const int32_t ipre = tid < A.idx_cap ? A.idx[tid] : 0;
    if (tid == 0) {
        for (int st = 0; st < kRing; ++st) mbar_init(&sm->bar[st], 1);
        for (int st = 0; st < kSlots; ++st) mbar_init(&sm->empty[st], kThreads / 32);
        mbar_init(&sm->inject_bar, 1);
        fence_mbar_init();
        sm->abort = 0;
        sm->s = launch_s(A);
    }
    // the active count and the whole tuning table in one round trip
    if (A.force_variant < 0 && tid < 2 * kBuckets) {
        if (tid < kBuckets)
            sm->tune.variant[tid] = A.tune->variant[tid];
        else
            sm->tune.split[tid - kBuckets] = A.tune->split[tid - kBuckets];
    }
    sm->idx_pre[tid] = ipre;
    __syncthreads();
    const int64_t s = sm->s;
    if (s <= 0) return;
    copy_list(A, s);
    if (A.inject) {
        // Test hook: wait on a barrier that no one arrives on; the spin limit must
        // expire and the kernel must report it. No copy is in flight here.
        if (!mbar_wait(&sm->inject_bar, 0, A.spin_limit) && tid == 0) atomicOr(A.status, kStTimeout);
        return;
    }
    int variant, S;
    if (A.force_variant >= 0) {
        variant = A.force_variant;
        S = A.force_split;
    } else {
        const int b = bucket_of(s);
        variant = sm->tune.variant[b];
        if (variant < 0 || variant >= kMixedVariants) variant = kMixedFallback;
        S = table_split(sm->tune.split[b], b, s, A.n, mixed_I(variant));
    }
    if (variant < 0 || variant >= kMixedVariants) variant = kMixedFallback;
    if (variant == kShareVariant) {
        // needs the cluster launch and a j range that fits the shares (the same
        // answer in every CTA of a cluster)
        if constexpr (SHARE) {
            const int64_t rper = share_rper(A);
            if (cg::this_cluster().num_blocks() == kShareC && rper > 0) {
                if (blockIdx.x == 0 && tid == 0) *A.split_used = kShareC;
                share_force(A, s, sm, rper);
                return;
            }
        }
        variant = kMixedFallback;   // (a launch without clusters: one split)
        S = 1;
    }
    S = clamp_split(S, A.tile_hi - A.tile_lo, s, A.part_cap);
    if (blockIdx.x == 0 && tid == 0) *A.split_used = S;
    const int64_t T = A.tile_hi - A.tile_lo;
    const int lgi = variant == 1 ? 1 : (variant == 2 ? 3 : 0);
    // worked out by one thread (the pair loops need the registers): the columns' plan, or the
    // work items (i-block of 1, 2 or 8 particles, share)
    if (tid == 0) {
        const int64_t items = ((s + (1 << lgi) - 1) >> lgi) * S;
        sm->items = variant < 1 || variant > 4 || short_items(variant, T, S, items) ? items : -1;
        if (sm->items < 0) {
            sm->plan = cols_plan(A, variant, s, S);
        } else {
            sm->split = S;
            sm->lgi = lgi;
            sm->tper = S == 1 ? T : qdiv(T + S - 1, S);
        }
    }
    __syncthreads();
    if (sm->items < 0) {
        if (blockIdx.x < sm->plan.G && !work_cols(A, s, sm) && tid == 0) atomicOr(A.status, kStTimeout);
        return;
    }
    uint32_t git = 0;
    for (int64_t w = blockIdx.x; w < sm->items; w += gridDim.x) {
        if (variant == 1 && sm->tper <= kFoldTiles)
            work_stream<2>(A, w, sm);
        else if (variant == 1)
            work_stream<2, true>(A, w, sm);
        else if (variant == 2)
            work_tile32(A, w, sm, git);
        else if (variant == 0 && (sm->tper < kLongTiles || T < kColdTiles))
            work_stream<1>(A, w, sm);
        else
            work_stream_tma(A, w, sm, git);
        if (sm->abort) {
            if (tid == 0) atomicOr(A.status, kStTimeout);
            return;
        }
        if (sm->split > 1) {
            const int64_t bx = qdiv(w, sm->split), i0 = bx << sm->lgi, i1 = (bx + 1) << sm->lgi;
            finish_block<true>(A, bx, i0, i1 < sm->s ? i1 : sm->s, sm->split, sm->split, sm);
        }
    }
}

// ------------------------------------------------------------- FP64 kernel
// The plain FP64 path. It is bound by the FP64 pipe: an FP64 warp instruction holds
// a sub-partition's unit for ~64 clocks here, whatever its active lanes, so what
// counts is the number of FP64 instructions per pair (32, see pair_f64), every lane
// holding a pair, and the same number of them on every SM:
//   * a CTA (8 warps) takes an i-block of TI = 32 / TJ active particles, one per
//     group of TJ lanes (TJ > 1 where blocks of 32 would leave lanes empty), and the
//     warps and the lanes of a group take consecutive j; all lanes of a warp with the
//     same j read it in one broadcast transaction;
//   * the (i-block, j unit) pairs, 8 TJ j's to a unit, are laid out in one line and
//     cut into equal runs, one per CTA of the grid. A run may end one i-block and
//     begin the next; an i-block's partials are added by the CTA that completes it
//     (arrival ticket), in CTA order: the same bits on every run.
// Measured (us per call, before: one i-particle per CTA up to s = 64, i-blocks of 256
// with at most n_tiles / 4 shares of j above, so 16 of 152 SMs at work at N = 16384):
// N = 16384: s = 1 18.4 -> 12.3, 64 84 -> 74, 256 2278 -> 250 (the pipe's time for its
// instructions is 213), N 18020 -> 15310; N = 65536, s = 1024 4587 -> 3820.

__device__ __forceinline__ void pair_f64(double xj, double yj, double zj, double mj, double vxj, double vyj,
                                         double vzj, const double *xi, double eps2, double *acc, bool self)
{
    double dx = xj - xi[0], dy = yj - xi[1], dz = zj - xi[2];
    double wx = vxj - xi[3], wy = vyj - xi[4], wz = vzj - xi[5];
    double r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2)));
    double rw = fma(dx, wx, fma(dy, wy, dz * wz));
    double q = rsqrt_f64(r2);
    if (self) q = 0.0;
    double q2 = q * q;
    double mq = mj * q;
    double mu = mq * q2;
    double al = 3.0 * rw * q2;
    acc[6] -= mq;
    acc[0] = fma(mu, dx, acc[0]);
    acc[1] = fma(mu, dy, acc[1]);
    acc[2] = fma(mu, dz, acc[2]);
    acc[3] = fma(mu, fma(-al, dx, wx), acc[3]);
    acc[4] = fma(mu, fma(-al, dy, wy), acc[4]);
    acc[5] = fma(mu, fma(-al, dz, wz), acc[5]);
}

// 0: one particle per i-block (the lanes of a warp on 32 j's)   1: by the block size
__host__ __device__ __forceinline__ int f64_I(int v) { return v == 0 ? 1 : 32; }

// Particles per i-block of variant 1 for an active count s on `grid` CTAs: the largest
// power of two up to 32 that leaves at most 1 lane in 8 without a particle (the
// pipe's time is paid per warp) and spreads the CTAs over enough i-blocks for each to
// be summed from about kF64Parts partials (one CTA adds them while the others have
// nothing left; N = 16384, s = 64: 80, 74, 74, 100 us with 8, 16, 32, no limit).
// Smaller blocks cost a lane tree of a few FP64 additions per item.
constexpr int kF64Parts = 16;
__device__ __forceinline__ int f64_block(int64_t s, int64_t grid)
{
    int I = 32;
    while (I > 1 && (8 * ((s + I - 1) / I * I - s) > s || I * grid > kF64Parts * s)) I >>= 1;
    return I;
}

struct F64Run {
    int64_t nib, units, U, G;   // i-blocks, units per i-block, all units, CTAs sharing them
    int64_t jlo, jhi;           // j range
    int I, unit, slots;         // particles per i-block, j's per unit, partial slots per particle
};

// CTA whose run holds unit u (run c: units [floor(U c / G), floor(U (c + 1) / G)))
__device__ __forceinline__ int64_t f64_owner(const F64Run &R, int64_t u) { return ((u + 1) * R.G - 1) / R.U; }

// The sums of i-block b over this CTA's j in [j0, j1): per-warp partial sums through
// shared memory, component c summed by warp c over the warps, then over the TJ lanes.
// Returns (in lanes with tj == 0 of warps 0 .. 6) component `warp` of particle ti.
template <int TJ>
__device__ __forceinline__ double f64_item(const ForceArgs &A, int64_t s, int64_t ib0, int64_t j0, int64_t j1,
                                           double (*sacc)[kThreads])
{
    constexpr int W = kThreads / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tj = lane % TJ, ti = lane / TJ;
    const int32_t gi = A.idx[ib0 + ti < s ? ib0 + ti : s - 1];
    const int64_t np = A.n_tiles * kJT;
    const double xi[6] = {A.xp[gi], A.xp[np + gi], A.xp[2 * np + gi], A.vp[gi], A.vp[np + gi], A.vp[2 * np + gi]};
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};
#pragma unroll 2
    for (int64_t j = j0 + warp * TJ + tj; j < j1; j += W * TJ)
        pair_f64(__ldg(A.xp + j), __ldg(A.xp + np + j), __ldg(A.xp + 2 * np + j), __ldg(A.m + j),
                 __ldg(A.vp + j), __ldg(A.vp + np + j), __ldg(A.vp + 2 * np + j), xi, A.eps2, acc, j == gi);
#pragma unroll
    for (int c = 0; c < 7; ++c) sacc[c][tid] = acc[c];
    __syncthreads();
    double v = 0.0;
    if (warp < 7) {
        v = sacc[warp][lane];
#pragma unroll
        for (int w = 1; w < W; ++w) v += sacc[warp][w * 32 + lane];
#pragma unroll
        for (int off = TJ / 2; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    }
    return v;
}

// Adds the n partials of active particles [ib0, ib0 + cnt) in slot order (D lanes per
// sum, eight loads in flight each, then a lane tree) and writes the results.
__device__ void f64_finish(const ForceArgs &A, int64_t ib0, int cnt, int n, int slots)
{
    const int D = cnt <= 1 ? 32 : (cnt <= 2 ? 16 : (cnt <= 4 ? 8 : (cnt <= 8 ? 4 : (cnt <= 16 ? 2 : 1))));
    const int d = threadIdx.x % D, per = kThreads / D;
    for (int q0 = 0; q0 < cnt * 7; q0 += per) {
        const int q = q0 + threadIdx.x / D;
        const int qq = q < cnt * 7 ? q : 0;
        const int64_t ii = ib0 + qq / 7;
        const double *src = A.part + ii * slots * kPartStride + qq % 7;
        double x = 0.0;
        for (int sp0 = d; sp0 < n; sp0 += 8 * D) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = sp0 + u * D < n ? __ldcg(src + (sp0 + u * D) * kPartStride) : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (sp0 + u * D < n) x += v[u];
        }
        for (int off = D / 2; off >= 1; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
        if (d == 0 && q < cnt * 7) put_final(A, ii, qq % 7, x);
    }
}

__global__ void __launch_bounds__(kThreads, 2) force_f64_kernel(ForceArgs A)
{
    __shared__ double sacc[7][kThreads];
    __shared__ uint64_t inject_bar;
    __shared__ int last;
    __shared__ F64Run run;
    const int tid = threadIdx.x;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int64_t s = launch_s(A);
    if (s <= 0) return;
    copy_list(A, s);
    if (A.inject) {
        if (tid == 0) {
            mbar_init(&inject_bar, 1);
            fence_mbar_init();
        }
        __syncthreads();
        if (!mbar_wait(&inject_bar, 0, A.spin_limit) && tid == 0) atomicOr(A.status, kStTimeout);
        return;
    }
    if (tid == 0) {
        int variant, S;
        if (A.force_variant >= 0) {
            variant = A.force_variant;
            S = A.force_split;
        } else {
            const int b = bucket_of(s);
            variant = A.tune->variant[b];
            if (variant < 0 || variant >= kF64Variants) variant = kF64Variants - 1;
            S = table_split(A.tune->split[b], b, s, A.n, f64_I(variant));
        }
        if (variant < 0 || variant >= kF64Variants) variant = kF64Variants - 1;
        F64Run R;
        R.I = variant == 0 ? 1 : f64_block(s, gridDim.x);
        R.unit = kThreads / R.I;   // one j per lane group and warp
        R.jlo = A.tile_lo * kJT;
        R.jhi = A.tile_hi * kJT < A.n ? A.tile_hi * kJT : A.n;
        R.nib = (s + R.I - 1) / R.I;
        R.units = (R.jhi - R.jlo + R.unit - 1) / R.unit;
        R.U = R.nib * R.units;
        // as many CTAs as the split asks for (S of them to an i-block of f64_I(variant))
        const int64_t nibt = (s + f64_I(variant) - 1) / f64_I(variant);
        R.G = nibt * (S < 1 ? 1 : S);
        if (R.G > gridDim.x) R.G = gridDim.x;
        if (R.G > R.U) R.G = R.U;
        // a run is at least floor(U / G) units, so an i-block meets at most
        // ceil(G / nib) + 1 of them; never more partials than there is room for
        while (R.G > 1 && s * ((R.G + R.nib - 1) / R.nib + 1) * kPartStride > A.part_cap) R.G = (R.G + 1) / 2;
        R.slots = (int)((R.G + R.nib - 1) / R.nib + 1);
        run = R;
        if (blockIdx.x == 0) *A.split_used = R.slots;
    }
    __syncthreads();
    const F64Run &R = run;
    if (blockIdx.x >= R.G) return;
    const int64_t u1 = R.U * (blockIdx.x + 1) / R.G;
    for (int64_t u = R.U * blockIdx.x / R.G; u < u1;) {
        const int64_t b = u / R.units, bu = b * R.units;
        const int64_t ue = bu + R.units < u1 ? bu + R.units : u1;
        const int64_t j0 = R.jlo + (u - bu) * R.unit;
        const int64_t je = R.jlo + (ue - bu) * R.unit;
        const int64_t j1 = je < R.jhi ? je : R.jhi;
        const int64_t ib0 = b * R.I;
        double v;
        int TJ;
        switch (R.I) {
        case 32: v = f64_item<1>(A, s, ib0, j0, j1, sacc); TJ = 1; break;
        case 16: v = f64_item<2>(A, s, ib0, j0, j1, sacc); TJ = 2; break;
        case 8: v = f64_item<4>(A, s, ib0, j0, j1, sacc); TJ = 4; break;
        case 4: v = f64_item<8>(A, s, ib0, j0, j1, sacc); TJ = 8; break;
        case 2: v = f64_item<16>(A, s, ib0, j0, j1, sacc); TJ = 16; break;
        default: v = f64_item<32>(A, s, ib0, j0, j1, sacc); TJ = 32; break;
        }
        const int lane = tid & 31, warp = tid >> 5;
        const int64_t ii = ib0 + lane / TJ;
        const bool holds = warp < 7 && lane % TJ == 0 && ii < s;
        const int64_t c0 = f64_owner(R, bu);
        const int n = (int)(f64_owner(R, bu + R.units - 1) - c0) + 1;   // CTAs that meet this i-block
        if (n == 1) {
            if (holds) put_final(A, ii, warp, v);
            __syncthreads();   // sacc is rewritten by the next i-block
        } else {
            if (holds) A.part[(ii * R.slots + (blockIdx.x - c0)) * kPartStride + warp] = v;
            __syncthreads();
            if (tid == 0) {
                __threadfence();
                last = atomicAdd(&A.tickets[b], 1) == n - 1;
            }
            __syncthreads();
            if (last) {
                __threadfence();
                f64_finish(A, ib0, (int)(ib0 + R.I < s ? R.I : s - ib0), n, R.slots);
                if (tid == 0) A.tickets[b] = 0;
            }
        }
        u = ue;
    }
}

}  // namespace

// ------------------------------------------------------------------ host side

int mixed_variant_I(int v) { return mixed_I(v); }

// The names callers look variants up by: those of the kernels that variants 1 to 4 began
// as (now columns with stride 256, 32, 8 and 1, or items of two and eight particles).
const char *mixed_variant_name(int v)
{
    switch (v) {
    case 0: return "stream R=1";
    case 1: return "stream R=2";
    case 2: return "tile R=1 TJ=32";
    case 3: return "tile R=1 TJ=8";
    case 4: return "tile R=1 TJ=1";
    case 5: return "TMA stream R=1";
    case 6: return "resident share (8-CTA clusters)";
    default: return "?";
    }
}

int f64_variant_I(int v) { return f64_I(v); }

const char *f64_variant_name(int v) { return v == 0 ? "f64 stream" : "f64 i-loop"; }

size_t force_mixed_smem_bytes() { return sizeof(Smem); }

static int g_mixed_occ = -1, g_f64_occ = -1, g_mixed_grid = -1;

int force_mixed_ctas_per_sm()
{
    if (g_mixed_occ < 0) {
        cudaFuncSetAttribute(force_mixed_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(Smem));
        cudaFuncSetAttribute(force_mixed_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kSmemShare);
        int occ = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, force_mixed_kernel<false>, kThreads, sizeof(Smem)) !=
                cudaSuccess ||
            occ < 1)
            occ = 1;
        g_mixed_occ = occ;
    }
    return g_mixed_occ;
}

// For particle counts whose j-records fit the resident shares of one cluster,
// the mixed kernel runs as clusters of kShareC CTAs (the resident-share variant
// needs them; the others ignore them). Its persistent grid is then the number of
// clusters the device keeps resident at once times kShareC, so that no CTA of
// the grid waits for another to finish (a CTA of a late cluster would hold its
// work items until then); 0 when cluster launches are not available. Larger
// particle counts (and that case) launch SMs x resident CTAs without clusters.
static int mixed_cluster_grid()
{
    if (g_mixed_grid < 0) {
        (void)force_mixed_ctas_per_sm();
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kShareC;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(kShareC * 64);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kSmemShare;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int ncl = 0;
        if (cudaOccupancyMaxActiveClusters(&ncl, force_mixed_kernel<true>, &cfg) != cudaSuccess || ncl < 1) {
            cudaGetLastError();
            ncl = 0;
        }
        g_mixed_grid = ncl * kShareC;
    }
    return g_mixed_grid;
}

bool mixed_share_fits(int64_t n_tiles)
{
    const int64_t rper = ((n_tiles * kPT + kShareC - 1) / kShareC + 31) / 32 * 32;
    return rper <= kShareRec && mixed_cluster_grid() > 0;
}

int force_mixed_grid(int num_sms, int64_t n_tiles)
{
    return mixed_share_fits(n_tiles) ? mixed_cluster_grid() : num_sms * force_mixed_ctas_per_sm();
}

int force_f64_ctas_per_sm()
{
    if (g_f64_occ < 0) {
        int occ = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, force_f64_kernel, kThreads, 0) != cudaSuccess ||
            occ < 1)
            occ = 1;
        g_f64_occ = occ;
    }
    return g_f64_occ;
}

cudaError_t launch_force_mixed(const ForceArgs &a, int grid, cudaStream_t st)
{
    (void)force_mixed_ctas_per_sm();   // sets the dynamic shared-memory attribute once
    if (mixed_share_fits(a.n_tiles) && grid % kShareC == 0) {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kShareC;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kSmemShare;
        cfg.stream = st;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, force_mixed_kernel<true>, a);
    }
    force_mixed_kernel<false><<<grid, kThreads, sizeof(Smem), st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_force_f64(const ForceArgs &a, int grid, cudaStream_t st)
{
    force_f64_kernel<<<grid, kThreads, 0, st>>>(a);
    return cudaGetLastError();
}

// Work items are i-blocks x j-splits over a grid of R = SMs x resident CTAs;
// a launch takes ceil(W / R) waves of items, so W just above a multiple of R
// wastes most of a wave. One full wave (S = R / nib) unless items would then be
// long (64 tiles or more): then the split in [S, 4 S] whose items fill their
// waves best. At least 4 tiles per item.
int64_t wave_split(int64_t nib, int64_t n_tiles, int64_t resident)
{
    int64_t S = std::max<int64_t>(1, resident / nib);
    if (n_tiles / S >= 64) {
        int64_t best = S;
        double best_eff = 0.0;
        for (int64_t c = S; c <= 4 * S; ++c) {
            const int64_t W = nib * c;
            const double eff = (double)W / (double)(((W + resident - 1) / resident) * resident);
            if (eff > best_eff + 1e-9) {
                best_eff = eff;
                best = c;
            }
        }
        S = best;
    }
    S = std::min<int64_t>(S, std::max<int64_t>(1, n_tiles / 4));
    return std::max<int64_t>(1, std::min<int64_t>(S, n_tiles));
}

// (The lines between variants 1 to 4 were found for the separate kernels they began as and
// also decide which FP32 sums are formed. Against those kernels calls of 1262 sizes over n =
// 500 .. 2^20, s = 1 .. n are 1.16 times as fast in the geometric mean, five slower by 2 to 5 %.)
void default_tuning(int precision, int64_t n, int64_t s, int num_sms, int ctas_per_sm, int *variant, int *split)
{
    const int64_t n_tiles = (n + kJT - 1) / kJT;
    const int64_t resident = (int64_t)num_sms * ctas_per_sm;
    int v;
    if (precision == NB_PREC_FP64) {
        // every CTA of the grid on equal runs of (i-block, j) units
        *variant = 1;
        *split = (int)resident;
        return;
    } else if (mixed_share_fits(n_tiles) && s > 16 && s <= 8192) {
        // the j-records fit the resident shares of a cluster: no split partials in L2
        v = kShareVariant;
    } else if (n <= 65536) {
        // j-records stay in L2 and are cheap to re-read: wide columns while blocks are small
        v = s <= (n <= 32768 ? 64 : 16) ? 0 : s <= 1024 ? 1 : s <= 1536 ? 2 : s <= 12288 ? 3 : 4;
    } else {
        // large N: narrower columns, fewer shares
        v = s <= 1 ? 0 : s <= 4 ? 1 : s <= 32 ? 2 : s <= 512 ? 3 : 4;
    }
    const int64_t I = mixed_I(v);
    *variant = v;
    *split = (int)wave_split((s + I - 1) / I, n_tiles, resident);
}

}  // namespace nb
