// Perturber lists of binaries (Sect. 3.1 of the paper): for each binary, the
// stars that perturb its internal motion, in the order a serial scan over the
// star index finds them, at most nmax of them, with the count of all.
//
// The paper gives the threshold as a force of about 10^-7 relative to a mean
// force. It is read here as the tidal perturbation of the binary: star j at
// distance r_j from the binary's centre of mass accelerates the two members
// differently by about 2 m_j d / r_j^3 (d their separation), against the
// binary's internal acceleration m_b / d^2, and it is a perturber when the ratio
// 2 m_j d^3 / (m_b r_j^3) reaches gamma. The test is taken without roots, on
// sixth powers, as (2 m_j)^2 d^6 >= (gamma m_b)^2 r_j^6, every FP64 operation an
// explicit round-to-nearest one in a fixed order (the decision is an integer
// result and must not depend on operation fusing).
//
// A CTA takes B binaries and walks the stars once for all of them, in segments in
// ascending index. Every warp tests its 32 stars of a round against the B binaries
// and leaves the ballots as bits in shared memory, without a barrier; after a
// segment, warp b walks binary b's words in order and writes the list entries, so
// the list comes out in the serial order by construction (the paper restores that
// order after its parallel search by broadcasting and sorting the lists). A j-range
// restricts the scan to one rank's share of the stars; lists of consecutive ranges
// concatenated in range order and cut at nmax give the list of the whole range.
//
// What bounds it: the FP64 test is 14 FP64 instructions, ~64 clocks each on a
// sub-partition's unit: 83 % FP64 pipe at 828 us for 1638 binaries x 16384 stars. The
// decision needs FP64 only where the two sides are close, so an FP32 test on the
// double-single positions (packed f32x2, two stars at a time) decides wherever they
// differ by 2^-16 or more, and only a warp with an undecided star evaluates the FP64
// test (~1e-4 of the rounds on Plummer models). Same lists and counts, bit for
// bit. Measured: 828 -> 59 us (issue-bound).
#include "nb_internal.cuh"

namespace nb {
namespace {

constexpr int kPertThreads = 256;
constexpr int kPertWarps = kPertThreads / 32;
constexpr int kPertSeg = 8192;          // stars per segment (a multiple of kPertThreads)
constexpr float kPertWindow = 0x1p-16f; // relative window of the FP32 test (see test_f32)

__device__ __forceinline__ double d2_of(double ux, double uy, double uz, double wx, double wy, double wz)
{
    const double dx = __dsub_rn(ux, wx), dy = __dsub_rn(uy, wy), dz = __dsub_rn(uz, wz);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// One binary: the FP64 test's constants and the FP32 test's (every float twice, the
// operands of the packed instructions on two stars).
struct __align__(16) Bin {
    float4 x, y, z;          // -cm as double-single: (hi, hi, lo, lo) per component
    float4 k;                // (-K, -K, w K, w K): K = d^6 / (gamma m_b)^2 4^e
    double cm[3], d6, rhs;
    int i, j;                // members; i < 0: an invalid pair (or none)
    float K, cabs;           // K (0: invalid pair, NaN: the FP32 test never decides), |cm_x| + |cm_y| + |cm_z|
};

// The masses are scaled by 2^-e for the FP32 test, K by 4^e: the same sides. e = 0 unless
// the first and the last star are both outside the masses it takes (see star_tm2), which
// then stand for the unit of mass: without it a call whose stars are all outside pays for
// both tests (N = 16384, 1638 binaries, masses times 2^22: 877 us, 832 with the FP64 test
// alone, now 61).
constexpr int kMassLo = -34, kMassBits = 42;   // |m| 2^-e in [2^-34, 2^8)
__device__ __forceinline__ int mass_exp(const PertArgs &P)
{
    if (P.j_lo >= P.j_hi) return 0;
    const int a = ((__double2hiint(P.m[P.j_lo]) >> 20) & 0x7ff) - 1023;
    const int z = ((__double2hiint(P.m[P.j_hi - 1]) >> 20) & 0x7ff) - 1023;
    const bool fits = (unsigned)(a - kMassLo) < kMassBits || (unsigned)(z - kMassLo) < kMassBits;
    return fits || z < -120 || z > 120 ? 0 : z;
}

__device__ void load_bin(const PertArgs &P, int32_t b, int e, Bin &q)
{
    const float nan = __int_as_float(0x7fffffff);
    q.i = q.j = -1;
    q.K = q.cabs = 0.f;      // an invalid pair: a sure no
    q.x = q.y = q.z = q.k = make_float4(0.f, 0.f, 0.f, 0.f);
    q.d6 = q.rhs = q.cm[0] = q.cm[1] = q.cm[2] = 0.0;
    if (b >= P.nbin) return;
    const int32_t i = P.pairs[2 * b], k = P.pairs[2 * b + 1];
    if (i < 0 || k < 0 || i >= P.n || k >= P.n || i == k) return;
    const double mi = P.m[i], mk = P.m[k];
    const double mb = __dadd_rn(mi, mk);
    double xi[3], xk[3];
    float4 c4[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        xi[c] = P.x[c * P.np + i];
        xk[c] = P.x[c * P.np + k];
        q.cm[c] = __ddiv_rn(__dadd_rn(__dmul_rn(mi, xi[c]), __dmul_rn(mk, xk[c])), mb);
        const float h = __double2float_rn(q.cm[c]), l = __double2float_rn(__dsub_rn(q.cm[c], (double)h));
        c4[c] = make_float4(-h, -h, -l, -l);
        q.cabs += fabsf(h);
    }
    q.x = c4[0];
    q.y = c4[1];
    q.z = c4[2];
    const double d2 = d2_of(xi[0], xi[1], xi[2], xk[0], xk[1], xk[2]);
    q.d6 = __dmul_rn(__dmul_rn(d2, d2), d2);
    const double gm = __dmul_rn(P.gamma, mb);
    q.rhs = __dmul_rn(gm, gm);
    // FP64 sides that could leave the normal range (their masses are up to 2^128 where e is
    // not 0), and a K outside [2^-55, 2^100], are not for the FP32 test
    const double top = e == 0 ? 0x1p800 : 0x1p600, low = e == 0 ? 0x1p-800 : 0x1p-600;
    const bool normal = q.d6 >= low && q.d6 <= top && q.rhs >= low && q.rhs <= top;
    const double K = __dmul_rn(__ddiv_rn(q.d6, q.rhs), __hiloint2double((1023 + 2 * e) << 20, 0));
    q.K = normal && K >= 0x1p-55 && K <= 0x1p100 ? __double2float_rn(K) : nan;
    q.k = make_float4(-q.K, -q.K, kPertWindow * q.K, kPertWindow * q.K);
    q.i = i;
    q.j = k;
}

// The FP32 test of two stars against a binary: d = r^6 - L with L = K (2 m_j 2^-e)^2; the
// star is a perturber if d < 0, and that is certain where |d| >= w L.
// Errors. Each component of r is a double-single difference: the high parts subtract
// exactly when they are within a factor two of one another, so its error is at most
// 2^-23 of itself plus 2^-45 X, X = the two positions' sizes. star_tm2 admits a star
// only where 2^-45 X is below 2^-20 of the threshold distance L^(1/6), so it moves r^6
// near the threshold by at most 6 x 2^-20 L = 2^-17.4 L; the roundings relative to r
// add 2^-18.8 L, L itself is within 2^-21.4 of its exact value and the FP64 test rounds
// at 2^-50: 2^-16.8 L in all, so a |d| of 2^-16 L or more has the exact sign. Farther
// from the threshold the margin only grows. L is in [2^-121, 2^118], an r^6 that overflows is +inf (a sure no), one
// that underflows is far below L; NaN (a star or binary not admitted, non-finite
// positions) compares false: undecided.
struct Star2 {
    float2 xh, xl, yh, yl, zh, zl;   // double-single positions of two stars
    float2 tm2;                      // (2 m 2^-e)^2, NaN where the FP32 test is not to decide
};

__device__ __forceinline__ float star_tm2(double m, int e, float sabs, float cmax, float kmin)
{
    // FP64 conversions and comparisons share the narrow pipe: the mass as FP32 by bit
    // fields (truncated, 2^-23) for |m| 2^-e in [2^-34, 2^8)
    const int hi = (__double2hiint(m) & 0x7fffffff) - e * (1 << 20);
    const float f = __int_as_float(__funnelshift_l(__double2loint(m), hi - (896 << 20), 3));
    const float q = (2.f * f) * (2.f * f);
    const float t = 0x1p-25f * (sabs + cmax), t2 = t * t;
    return (unsigned)(hi - ((1023 + kMassLo) << 20)) < (unsigned)(kMassBits << 20) && kmin * q >= (t2 * t2) * t2
               ? q
               : __int_as_float(0x7fffffff);
}

__device__ __forceinline__ Star2 load_stars(const PertArgs &P, int64_t j0, int64_t j1, int e, float cmax,
                                            float kmin)
{
    const float2 ax = __ldg(P.x2 + j0), ay = __ldg(P.x2 + P.np + j0), az = __ldg(P.x2 + 2 * P.np + j0);
    const float2 bx = __ldg(P.x2 + j1), by = __ldg(P.x2 + P.np + j1), bz = __ldg(P.x2 + 2 * P.np + j1);
    const double ma = __ldg(P.m + j0), mb = __ldg(P.m + j1);
    Star2 t;
    t.xh = make_float2(ax.x, bx.x);
    t.xl = make_float2(ax.y, bx.y);
    t.yh = make_float2(ay.x, by.x);
    t.yl = make_float2(ay.y, by.y);
    t.zh = make_float2(az.x, bz.x);
    t.zl = make_float2(az.y, bz.y);
    t.tm2 = make_float2(star_tm2(ma, e, fabsf(ax.x) + fabsf(ay.x) + fabsf(az.x), cmax, kmin),
                        star_tm2(mb, e, fabsf(bx.x) + fabsf(by.x) + fabsf(bz.x), cmax, kmin));
    return t;
}

// d and w L of the two stars
__device__ __forceinline__ void test_f32(const Star2 &t, const Bin &q, float2 &d, float2 &wl)
{
    const float4 cx = q.x, cy = q.y, cz = q.z, ck = q.k;
    const float2 dx = __fadd2_rn(__fadd2_rn(t.xh, make_float2(cx.x, cx.y)), __fadd2_rn(t.xl, make_float2(cx.z, cx.w)));
    const float2 dy = __fadd2_rn(__fadd2_rn(t.yh, make_float2(cy.x, cy.y)), __fadd2_rn(t.yl, make_float2(cy.z, cy.w)));
    const float2 dz = __fadd2_rn(__fadd2_rn(t.zh, make_float2(cz.x, cz.y)), __fadd2_rn(t.zl, make_float2(cz.z, cz.w)));
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    d = __ffma2_rn(__fmul2_rn(r2, r2), r2, __fmul2_rn(make_float2(ck.x, ck.y), t.tm2));
    wl = __fmul2_rn(make_float2(ck.z, ck.w), t.tm2);
}

// The FP64 test of star j, every operation rounded separately in the oracle's order.
__device__ __noinline__ bool test_f64(const double *x, const double *m, int64_t np, const Bin &q, int64_t j)
{
    const double r2 = d2_of(x[j], x[np + j], x[2 * np + j], q.cm[0], q.cm[1], q.cm[2]);
    const double r6 = __dmul_rn(__dmul_rn(r2, r2), r2);
    const double tm = __dmul_rn(2.0, m[j]);
    return __dmul_rn(__dmul_rn(tm, tm), q.d6) >= __dmul_rn(q.rhs, r6);
}

template <int B>
__global__ void __launch_bounds__(kPertThreads, 4) perturbers_kernel(PertArgs P)
{
    static_assert(B <= kPertWarps, "one warp per binary writes the lists");
    __shared__ Bin bins[B];
    __shared__ unsigned bits[B][kPertSeg / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int e = mass_exp(P);
    for (int64_t b0 = (int64_t)blockIdx.x * B; b0 < P.nbin; b0 += (int64_t)gridDim.x * B) {
        __syncthreads();   // the previous binaries have been used
        if (lane == 0 && warp < B) load_bin(P, (int32_t)(b0 + warp < P.nbin ? b0 + warp : P.nbin), e, bins[warp]);
        __syncthreads();
        float cmax = 0.f, kmin = 0x1p100f;   // over the CTA's binaries
#pragma unroll
        for (int b = 0; b < B; ++b) {
            cmax = fmaxf(cmax, bins[b].cabs);
            if (bins[b].K > 0.f) kmin = fminf(kmin, bins[b].K);
        }
        // warp b's binary (the lists are written by warps 0 .. B - 1)
        const int bw = warp < B ? warp : 0;
        const bool writes = warp < B && b0 + warp < P.nbin;
        const bool valid = writes && bins[bw].i >= 0;
        int32_t *list = P.lists + (b0 + bw) * P.nmax;
        int found = 0;   // the same in every lane of warp b
        for (int64_t s0 = P.j_lo; s0 < P.j_hi; s0 += kPertSeg) {
            const int cnt = (int)(P.j_hi - s0 < kPertSeg ? P.j_hi - s0 : kPertSeg);
            const int words = (cnt + 31) / 32;
            // a warp takes the stars of words w and w + kPertWarps together
            for (int w = warp; w < words; w += 2 * kPertWarps) {
                const int64_t ja = s0 + 32 * w + lane, jb = ja + 32 * kPertWarps;
                const bool la = ja < P.j_hi, lb = jb < P.j_hi;
                const Star2 t = load_stars(P, la ? ja : P.j_hi - 1, lb ? jb : P.j_hi - 1, e, cmax, kmin);
                unsigned mine_a = 0, mine_b = 0;
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    float2 d, wl;
                    test_f32(t, bins[b], d, wl);
                    bool ya = la && d.x < 0.f, yb = lb && d.y < 0.f;
                    const bool sure = fabsf(d.x) >= wl.x && fabsf(d.y) >= wl.y;
                    if (!__all_sync(0xffffffffu, sure)) {
                        if (!(fabsf(d.x) >= wl.x))
                            ya = la && bins[b].i >= 0 && test_f64(P.x, P.m, P.np, bins[b], ja);
                        if (!(fabsf(d.y) >= wl.y))
                            yb = lb && bins[b].i >= 0 && test_f64(P.x, P.m, P.np, bins[b], jb);
                    }
                    const unsigned va = __ballot_sync(0xffffffffu, ya), vb = __ballot_sync(0xffffffffu, yb);
                    if (lane == b) {
                        mine_a = va;
                        mine_b = vb;
                    }
                }
                if (lane < B) {
                    bits[lane][w] = mine_a;
                    if (w + kPertWarps < words) bits[lane][w + kPertWarps] = mine_b;
                }
            }
            __syncthreads();
            if (valid) {
                // the members do not count as their own perturbers
                if (lane < 2) {
                    const int64_t mem = (lane == 0 ? bins[bw].i : bins[bw].j) - s0;
                    if (mem >= 0 && mem < cnt) atomicAnd(&bits[bw][mem >> 5], ~(1u << (mem & 31)));
                }
                __syncwarp();
                for (int w0 = 0; w0 < words; w0 += 32) {
                    unsigned m = w0 + lane < words ? bits[bw][w0 + lane] : 0u;
                    const int c = __popc(m);
                    int incl = c;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, incl, off);
                        if (lane >= off) incl += y;
                    }
                    int pos = found + incl - c;
                    const int32_t j0 = (int32_t)(s0 + 32 * (w0 + lane));
                    for (; m && pos < P.nmax; m &= m - 1u) list[pos++] = j0 + __ffs(m) - 1;
                    found += __shfl_sync(0xffffffffu, incl, 31);
                }
            }
            __syncthreads();   // the bits are rewritten by the next segment
        }
        if (writes) {
            // (an invalid pair: an empty list and a negative count)
            for (int64_t q = found + lane; q < P.nmax; q += 32) list[q] = -1;
            if (lane == 0) P.counts[b0 + warp] = valid ? found : -1;
        }
    }
}

template <int B>
cudaError_t launch_B(const PertArgs &p, cudaStream_t st)
{
    const int64_t grid = ((int64_t)p.nbin + B - 1) / B;
    perturbers_kernel<B><<<(int)(grid < 65535 ? grid : 65535), kPertThreads, 0, st>>>(p);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_perturbers(const PertArgs &p, cudaStream_t st)
{
    if (p.nbin <= 0) return cudaSuccess;
    // With more binaries to a CTA each star is read less often, with fewer there are more
    // CTAs to hide a round's latency (N = 16384, us with 1, 2, 4, 8 to a CTA: 300
    // binaries 25, 28, 37, 55; 1638 binaries 82, 70, 59, 72; 3000 140, 106, 92, 97). The lines
    // leave at least two CTAs of 2 or 4 binaries to each of the 152 SMs; a star's cost does
    // not depend on N.
    if (p.nbin >= 1216) return launch_B<4>(p, st);
    if (p.nbin >= 608) return launch_B<2>(p, st);
    return launch_B<1>(p, st);
}

}  // namespace nb
