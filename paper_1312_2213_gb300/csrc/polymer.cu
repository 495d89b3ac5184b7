// polymer.cu -- multicanonical sweeps of a single flexible bead-spring polymer
// (paper: polymer paragraph and Eq. 7; the benchmark's parameters: FENE bonds
// K = 40, R = 1.5, Lennard-Jones 12-6 between beads |i-j| >= 2 with eps = sigma
// = 1, cut at 2.5 and shifted; single-bead moves in a cube of side 0.3).
//
// G lanes of a warp per walker (G = 1, 2, 4, 8, 16 or 32; 32/G walkers share a
// warp).
// The beads are visited in order; for bead i every lane of the walker's group
// evaluates the old and the new pair energies with its partner beads
// j = lane, lane + G, ... in FP32 and keeps a compensated (Kahan) sum (the old
// bond energies come from a per-walker cache, updated on acceptance); the lane
// sums are added in FP32 over the group and the total is converted once to 64-bit
// fixed point (2^-32 energy units).  Nothing on the hot path uses FP64, whose
// rate on GB300 is a small fraction of FP32.
//
// Exactness: master coordinates are int64 on a 2^-44 grid and a move adds
// (u - 2^31) * 1229 grid units per axis (a cube of side 1229/4096 = 0.30005), so
// the coordinates of an accepted move are exact and identical to any other
// implementation that draws the same words.  The FP32 pair terms use shadows
// relative to the walker's bead 0 at the start of each sweep, kept as unevaluated
// float pairs (hi + lo): a difference (hi_i - hi_j) + (lo_i - lo_j) keeps the
// separation of two beads to ~1e-7 of itself however far the chain extends, so
// the rounding of FP32 energy changes stays unbiased when walk-in selects moves
// by the sign of their energy change.  The running
// energy is an exact sum of the fixed-point energy changes; it is refreshed from
// scratch after every iterate call, and the largest difference is recorded.
// Acceptance inside the window: d = ln W(b') - ln W(b) from a fixed-point table,
// accept iff d >= 0 or ln(u 2^-32) < d (the FP32 logarithm of each bead's
// acceptance word is taken once a sweep); outside the window a move is accepted
// iff it does not increase the distance to the window (walk-in).  Visits are
// counted in the block's 32-bit shared-memory counters, which the block's last
// warp to finish adds to the 64-bit histogram (an iterate longer than they can
// hold runs as several launches), so that walkers crowding one bin (right after
// they walk in, say) do not queue on one global counter.
#include <type_traits>

#include "muca_device.cuh"
#include "muca_internal.h"

namespace muca {

bool polymer_supported(int N) { return N >= 2 && N <= kPolyMaxN; }

// (sigma/r)^2 from the hardware's approximate reciprocal (PTX rcp.approx.ftz.f32, at most one
// ulp off: the r^-12 term then carries a few ulp, a few 1e-8 of the pair's error scale
// |v| + |r v'|, which is 48 (sigma/r)^12 and more).  A correctly rounded reciprocal took a
// quarter of the sweep's time at N = 128.
__device__ __forceinline__ float lj_energy(float r2, const PolyArgs &a)
{
    float rr;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rr) : "f"(r2));
    const float ir2 = rr * a.lj_sigma2;  // sigma = 1 in model 0
    const float ir6 = ir2 * ir2 * ir2;
    const float v = 4.0f * (ir6 * ir6 - ir6) - a.lj_shift;
    return r2 < a.lj_rc2 ? v : 0.0f;
}

__device__ __forceinline__ float fene_energy(float r2, const PolyArgs &a)
{
    if (a.model == 1) {  // rest length r0: -(K/2) R^2 ln(1 - ((r - r0)/R)^2)
        const float x = (__fsqrt_rn(r2) - a.fene_r0) * a.fene_invR;
        return -a.fene_KR2_half * log1pf(-x * x);
    }
    return -a.fene_KR2_half * log1pf(-r2 * a.fene_invR2);
}

// A bond of squared length r2 is intact: r < R (model 0), |r - r0| < R (model 1).
__device__ __forceinline__ bool fene_intact(float r2, const PolyArgs &a)
{
    if (a.model == 1) return fabsf((__fsqrt_rn(r2) - a.fene_r0) * a.fene_invR) < 1.0f;
    return r2 < 1.0f / a.fene_invR2;
}

// Offset on the 2^-44 grid as an unevaluated pair hi + lo of floats.
__device__ __forceinline__ void grid_to_ff(long long d, float &hi, float &lo)
{
    hi = (float)d;
    lo = (float)(d - (long long)hi);
    hi *= 0x1p-44f;
    lo *= 0x1p-44f;
}

__device__ __forceinline__ long long warp_sum_ll(long long q)
{
#pragma unroll
    for (int off = 16; off; off >>= 1) q += __shfl_xor_sync(0xffffffffu, q, off);
    return q;
}

// A 2^-32 fixed-point value as a float, from its two 32-bit halves (32-bit
// conversions only).
__device__ __forceinline__ float q32_to_float(long long v)
{
    return (float)(int)(v >> 32) + (float)(uint32_t)v * 0x1p-32f;
}

// lnu < q32_to_float(v) for v < 0 and lnu in (-23, 0] or -inf, without conversion instructions (their
// latency is on the attempt's chain): 16-bit integers become floats under an exponent of 2^23, and
// 65536 h + l rounds once, as the conversion does.  Whole parts below -2^21 are all the same.
__device__ __forceinline__ bool less_than_q32(float lnu, long long v)
{
    const uint32_t lo = (uint32_t)v;
    const float h = __uint_as_float(0x4B000000u | (lo >> 16)) - 8388608.0f;
    const float l = __uint_as_float(0x4B000000u | (lo & 0xFFFFu)) - 8388608.0f;
    const float whole = __int_as_float(0x4B400000 + max((int)(v >> 32), -(1 << 21))) - 12582912.0f;
    return lnu < fmaf(fmaf(h, 65536.0f, l), 0x1p-32f, whole);
}

__device__ __forceinline__ int poly_bin(long long E, const PolyArgs &a)
{
    const long long b = ((E - a.elo_q) * a.bin_k) >> 32;
    return b < -1 ? -1 : (b > (long long)a.B ? a.B : (int)b);
}

// poly_bin of a relative energy r = E - elo_q: the upper half of the 64-bit product r k, modulo 2^64
// as poly_bin forms it (an overlapping initial chain can have an energy beyond that product), from
// the 32-bit halves of r.
__device__ __forceinline__ int poly_bin_rel(long long r, const PolyArgs &a)
{
    const int v = (int)((uint32_t)(r >> 32) * (uint32_t)a.bin_k + __umulhi((uint32_t)r, (uint32_t)a.bin_k));
    return min(max(v, -1), a.B);
}

// llrint(v 2^32) for the sum of G lanes, each below 2^22: |v| <= 2^26 up to 16 lanes, 2^27 for 32.
// Conversion instructions have twice the latency of additions, and this is on the attempt's chain, so
// v is cut into integers by adding 1.5 2^23 (the integer, at most 2^22, then sits in the low mantissa
// bits): v = U h + r with U = 16 (32 for 32 lanes), 2^12 r = m + x, q = U 2^32 h + 2^20 m + rint(2^20 x),
// every difference exact (a multiple of v's last place that is no longer than v).  Only the last
// step rounds, to nearest even beside even terms, as the conversion of v would.
template <int G>
__device__ __forceinline__ long long float_to_q32(float v)
{
    const float M = 12582912.0f;
    const int MB = 0x4B400000;
    constexpr int U = G > 16 ? 32 : 16;
    const float th = fmaf(v, 1.0f / U, M), r = fmaf(th - M, (float)-U, v);
    const float tm = fmaf(r, 4096.0f, M), x = fmaf(r, 4096.0f, -(tm - M));
    const float tl = fmaf(x, 1048576.0f, M);
    const int h = __float_as_int(th) - MB, m = __float_as_int(tm) - MB, l = __float_as_int(tl) - MB;
    return (long long)m * (1 << 20) + l + ((long long)(h * U) << 32);
}

// n visits of a bin: a shared-memory reduction without a returned value, so nothing
// waits for it.
__device__ __forceinline__ void count_visits(unsigned *h, unsigned n)
{
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(h)), "r"(n) : "memory");
}

// Random-walk initial chain (thread per walker): bead k = bead k-1 + unit vector
// from Marsaglia's method on tag-2 Philox words, rounded to the grid, redrawn (up
// to 64 times) while an earlier bead is closer than 0.9.  Binary64 with explicit
// round-to-nearest operations (run once).
__global__ void k_poly_init(const PolyArgs a)
{
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= a.p) return;
    const int N = a.N;
    const uint32_t wid = (uint32_t)(w + a.walker_offset);
    long long *X = a.X + (size_t)w * 3 * N;
    X[0] = X[N] = X[2 * N] = 0;
    uint32_t draw = 0;
    for (int k = 1; k < N; ++k) {
        long long cand[3] = {0, 0, 0};
        for (int attempt = 0; attempt < 64; ++attempt) {
            double v1 = 0.0, v2 = 0.0, s = 0.5;
            for (int tries = 0; tries < 4096; ++tries) {
                const uint4 u = philox4x32_10(make_uint4(draw++, 0u, wid, kTagPolyInit), a.key0, a.key1);
                v1 = __dsub_rn(__dmul_rn((double)u.x, 0x1p-31), 1.0);
                v2 = __dsub_rn(__dmul_rn((double)u.y, 0x1p-31), 1.0);
                s = __dadd_rn(__dmul_rn(v1, v1), __dmul_rn(v2, v2));
                if (s < 1.0 && s > 0.0) break;
            }
            const double f = __dmul_rn(2.0, __dsqrt_rn(__dsub_rn(1.0, s)));
            const double uh[3] = {__dmul_rn(v1, f), __dmul_rn(v2, f), __dsub_rn(1.0, __dmul_rn(2.0, s))};
            for (int c = 0; c < 3; ++c)
                cand[c] = X[c * N + k - 1] + (long long)rint(__dmul_rn(__dmul_rn(uh[c], a.init_bond), 0x1p44));
            bool ok = true;
            for (int j = 0; j < k - 1 && ok; ++j) {
                const double dx = __dmul_rn((double)(cand[0] - X[j]), 0x1p-44);
                const double dy = __dmul_rn((double)(cand[1] - X[N + j]), 0x1p-44);
                const double dz = __dmul_rn((double)(cand[2] - X[2 * N + j]), 0x1p-44);
                const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
                if (d2 < a.init_d2min) ok = false;
            }
            if (ok) break;
        }
        for (int c = 0; c < 3; ++c) X[c * N + k] = cand[c];
    }
}

// Energy from scratch, one warp per walker (FP32 pairs relative to bead 0,
// Kahan per lane, exact fixed-point warp sum).  With track != 0 the largest
// change against the running energy is recorded in state->drift_max_q.
__global__ void k_poly_energy(const PolyArgs a, int track)
{
    extern __shared__ __align__(16) float sh[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, N = a.N;
    const int w = blockIdx.x * (blockDim.x >> 5) + wib;
    if (w >= a.p) return;
    float *xs = sh + (size_t)wib * 6 * N;  // hi[3N], lo[3N]
    float *xl = xs + 3 * N;
    const long long *X = a.X + (size_t)w * 3 * N;
    const long long A0 = X[0], A1 = X[N], A2 = X[2 * N];
    for (int j = lane; j < N; j += 32) {
        grid_to_ff(X[j] - A0, xs[j], xl[j]);
        grid_to_ff(X[N + j] - A1, xs[N + j], xl[N + j]);
        grid_to_ff(X[2 * N + j] - A2, xs[2 * N + j], xl[2 * N + j]);
    }
    __syncwarp();
    float s = 0.0f, c = 0.0f;
    for (int i = 0; i < N; ++i) {
        const float xi = xs[i], yi = xs[N + i], zi = xs[2 * N + i];
        const float li = xl[i], mi = xl[N + i], ni = xl[2 * N + i];
        for (int j = lane; j < N; j += 32) {
            if (j <= i) continue;
            const float dx = (xi - xs[j]) + (li - xl[j]), dy = (yi - xs[N + j]) + (mi - xl[N + j]),
                        dz = (zi - xs[2 * N + j]) + (ni - xl[2 * N + j]);
            const float r2 = dx * dx + dy * dy + dz * dz;
            const float v = (j - i == 1) ? fene_energy(r2, a) : lj_energy(r2, a);
            const float y = v - c;
            const float t = s + y;
            c = (t - s) - y;
            s = t;
        }
    }
    long long q = __float2ll_rn(s * 0x1p32f) - __float2ll_rn(c * 0x1p32f);
    q = warp_sum_ll(q);
    if (lane == 0) {
        if (track) {
            const long long d = q - a.E[w];
            atomicMax(&a.state->drift_max_q, (unsigned long long)(d < 0 ? -d : d));
        }
        a.E[w] = q;
        a.bin[w] = poly_bin(q, a);
    }
}

template <int G>
__device__ __forceinline__ bool group_any(bool p, int gi)
{
    const unsigned bal = __ballot_sync(0xffffffffu, p);
    return G == 32 ? bal != 0u : ((bal >> (gi * G)) & ((1u << (G & 31)) - 1u)) != 0u;
}

// Spherical rotation of bead i (move set 1): the pivot is a bonded neighbour,
// the new position pivot + d n with d = |r_i - r_pivot| and n a unit vector from
// Marsaglia's method on (m.z, m.w) and then on tag-4 blocks (64 i + t), two pairs
// a block, at most 64 pairs.  Every step is a correctly rounded binary64
// operation on exact grid values, so the new grid position is bit-identical to
// any implementation that follows the same steps.  poly_unit draws n and returns
// false when no point was found (the move is then rejected).
__device__ bool poly_unit(int i, uint32_t g, uint32_t wid, const uint4 m, const uint32_t (&rk)[20], double n[3])
{
    double v1 = 0.0, v2 = 0.0, s = 0.0;
    bool found = false;
    uint4 blk = make_uint4(0u, 0u, m.z, m.w);
    for (int t = 0; t < 64 && !found; ++t) {
        if (t & 1) blk = philox4x32_10_rk(make_uint4((uint32_t)(64 * i + (t >> 1)), g, wid, kTagPolySphere), rk);
        const uint32_t aw = (t == 0) ? m.z : ((t & 1) ? blk.x : blk.z);
        const uint32_t bw = (t == 0) ? m.w : ((t & 1) ? blk.y : blk.w);
        v1 = __dsub_rn(__dmul_rn((double)aw, 0x1p-31), 1.0);
        v2 = __dsub_rn(__dmul_rn((double)bw, 0x1p-31), 1.0);
        s = __dadd_rn(__dmul_rn(v1, v1), __dmul_rn(v2, v2));
        found = s < 1.0 && s > 0.0;
    }
    if (!found) return false;
    const double f = __dmul_rn(2.0, __dsqrt_rn(__dsub_rn(1.0, s)));
    n[0] = __dmul_rn(v1, f);
    n[1] = __dmul_rn(v2, f);
    n[2] = __dsub_rn(1.0, __dmul_rn(2.0, s));
    return true;
}

// One axis' share (dd, squared by the caller) of d and the new grid coordinate of one axis.
__device__ __forceinline__ double poly_axis_diff(long long x, long long pivot)
{
    return __dmul_rn((double)(x - pivot), 0x1p-44);
}
__device__ __forceinline__ double poly_distance(double dx, double dy, double dz)
{
    return __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
}
__device__ __forceinline__ long long poly_rotated(long long pivot, double n, double d)
{
    return pivot + (long long)rint(__dmul_rn(__dmul_rn(n, d), 0x1p44));
}

// Packed pairs of floats (PTX f32x2): one instruction for the same operation on both halves, each
// rounded as the scalar one.
using float_pair = unsigned long long;
__device__ __forceinline__ float_pair pair_of(float lo, float hi)
{
    float_pair r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void halves_of(float_pair v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ float_pair add_pair(float_pair a, float_pair b)
{
    float_pair r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float_pair mul_pair(float_pair a, float_pair b)
{
    float_pair r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float_pair fma_pair(float_pair a, float_pair b, float_pair c)
{
    float_pair r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// LJ energies (lj_energy) of a bead at minus (px, py, pz) with two partners, each coordinate a
// float pair hi + lo; the partners' coordinates are packed, the bead's are in both halves.
// (The squares do not see the sign of a separation; n6 = -(sigma/r)^6.)
__device__ __forceinline__ void lj_two(const float4 &j0, const float4 &j1, const float4 &j2, const float4 &b0,
                                       const float4 &b1, const float4 &b2, const PolyArgs &a, float &v0, float &v1)
{
    const float_pair dx = add_pair(add_pair(pair_of(j0.x, j0.y), pair_of(b0.x, b0.y)),
                                   add_pair(pair_of(j1.z, j1.w), pair_of(b1.z, b1.w)));
    const float_pair dy = add_pair(add_pair(pair_of(j0.z, j0.w), pair_of(b0.z, b0.w)),
                                   add_pair(pair_of(j2.x, j2.y), pair_of(b2.x, b2.y)));
    const float_pair dz = add_pair(add_pair(pair_of(j1.x, j1.y), pair_of(b1.x, b1.y)),
                                   add_pair(pair_of(j2.z, j2.w), pair_of(b2.z, b2.w)));
    const float_pair r2 = fma_pair(dz, dz, fma_pair(dx, dx, mul_pair(dy, dy)));
    float r0, r1;
    halves_of(r2, r0, r1);
    const float_pair n2 = mul_pair(pair_of(rcp_approx(r0), rcp_approx(r1)), pair_of(-a.lj_sigma2, -a.lj_sigma2));
    const float_pair n6 = mul_pair(mul_pair(n2, n2), n2);
    const float_pair v = fma_pair(fma_pair(n6, n6, n6), pair_of(4.0f, 4.0f), pair_of(-a.lj_shift, -a.lj_shift));
    halves_of(v, v0, v1);
    v0 = r0 < a.lj_rc2 ? v0 : 0.0f;
    v1 = r1 < a.lj_rc2 ? v1 : 0.0f;
}

// Energy of a new bond over the separation (bx, by, bz), NaN if it breaks.
__device__ __forceinline__ float bond_or_nan(float bx, float by, float bz, const PolyArgs &a)
{
    const float r2n = bx * bx + by * by + bz * bz;
    return fene_intact(r2n, a) ? fene_energy(r2n, a) : __int_as_float(0x7fffffff);
}

// A bead's float-pair shadow.
struct Shadow {
    float c[6];  // x, y, z, lo x, lo y, lo z
};
__device__ __forceinline__ float bond_between(const Shadow &p, const Shadow &r, const PolyArgs &a)
{
    return bond_or_nan((p.c[0] - r.c[0]) + (p.c[3] - r.c[3]), (p.c[1] - r.c[1]) + (p.c[4] - r.c[4]),
                       (p.c[2] - r.c[2]) + (p.c[5] - r.c[5]), a);
}

// Shared memory of one walker's slot.  The shadows of all beads are in pos, two partners of a lane
// (beads j and j + G) side by side so that one packed instruction takes both: 4-vectors
// (x x' y y'), (z z' lo x, lo x'), (lo y, lo y', lo z, lo z'), nP of each.  With at most one partner
// a lane (ONE, N <= G) both halves hold bead j, and the packed instruction takes the moved bead's
// old and proposed place at once.  eb[j] is the energy of
// the bond (j - 1, j), 0 at both ends.  The chunk of beads being visited (poly_chunk of them at a
// time): minus the bead's old and proposed shadow, each number twice (twelve 2-vectors in six
// 4-vectors, in the order of pos; ONE: old and proposed side by side, three), and rec = (energy
// change of the left bond, left bead where it was / left bead moved; of the right bond, right bead
// where it is; ln of the acceptance word); a change is NaN where the bond breaks.
// Beads of a chunk: one a lane, two at 8 lanes (up to 5 % faster with 2048 walkers).  More beads than lanes
// to prepare them cost shared memory and hide nothing: with 16 in every grouping a one-lane warp's 32
// slots of N = 13 took 87 KB, two warps an SM, and 32768 walkers 6.13 ms for 46 sweeps instead of 1.62.
template <int G>
__host__ __device__ constexpr int poly_chunk() { return G == 8 ? 16 : G; }

template <int G, int MOVES, bool ONE>
struct PolySlot {
    static constexpr int BV = ONE ? 3 : 6;  // 4-vectors of a chunk bead
    float4 *pos;     // [3][nP]
    float4 *bead;    // [CH][BV]
    float4 *rec;     // [CH]
    long long *nx;   // [CH][3] (MOVES) proposed grid position, or the rotation's unit vector
    uint32_t *how;   // [CH] (MOVES) kReady, kLate, kNoPoint; else [CH][3] the random words of the step
    float *nr;       // [CH] energy of the right bond with the bead moved
    float *eb;       // [N + 1]
    int nP;
    static __host__ __device__ int pairs(int N) { return ONE ? G : (N <= G ? N : (N + 2 * G - 1) / (2 * G) * G); }
    // beads of a chunk that have records (a short chain's chunk is the chain; 16 lanes: always 16, which
    // the unrolled loop counts on)
    static __host__ __device__ int records(int N) { return (G == 16 && !MOVES) || N > poly_chunk<G>() ? poly_chunk<G>() : N; }
    static __host__ __device__ size_t bytes(int N)
    {
        const size_t b = (size_t)48 * pairs(N) + (size_t)records(N) * (16 * BV + 16 + (MOVES ? 28 : 12) + 4) + 4 * (size_t)(N + 1);
        // (an odd number of 16-byte units where several walkers share a warp, for the banks)
        return G < 16 ? ((b + 15) / 16 | 1) * 16 : (b + 15) / 16 * 16;
    }
    __device__ PolySlot(unsigned char *p, int N)
    {
        const int CH = records(N);
        nP = pairs(N);
        pos = (float4 *)p;
        bead = pos + 3 * nP;
        rec = bead + BV * CH;
        nx = (long long *)(rec + CH);
        how = (uint32_t *)(MOVES ? nx + 3 * CH : nx);
        nr = (float *)(how + (MOVES ? CH : 3 * CH));
        eb = nr + CH;
    }
    // component c (in the order x y | z lx | ly lz of pos) of bead j
    __device__ float *at(int j, int c) const
    {
        if (ONE) return (float *)(pos + (c >> 1) * nP + j) + 2 * (c & 1);
        const int idx = j / (2 * G) * G + j % G, half = (j / G) & 1;
        return (float *)(pos + (c >> 1) * nP + idx) + 2 * (c & 1) + half;
    }
    __device__ void set(int j, int c, float v) const
    {
        if (ONE) *(float2 *)at(j, c) = make_float2(v, v);
        else *at(j, c) = v;
    }
    __device__ Shadow get(int j) const
    {
        return Shadow{{*at(j, 0), *at(j, 1), *at(j, 2), *at(j, 3), *at(j, 4), *at(j, 5)}};
    }
    __device__ void put(int j, const Shadow &s) const
    {
#pragma unroll
        for (int c = 0; c < 6; ++c) set(j, c, s.c[c]);
    }
    // minus component c of the proposed shadow of chunk bead t
    __device__ float proposed(int t, int c) const
    {
        return ONE ? ((float *)(bead + 3 * t))[2 * c + 1] : ((float *)(bead + 6 * t + 3))[2 * c];
    }
    __device__ void set_proposed(int t, int c, float v) const
    {
        if (ONE) ((float *)(bead + 3 * t))[2 * c + 1] = -v;
        else *(float2 *)((float *)(bead + 6 * t + 3) + 2 * c) = make_float2(-v, -v);
    }
    __device__ Shadow get_proposed(int t) const
    {
        return Shadow{{-proposed(t, 0), -proposed(t, 1), -proposed(t, 2), -proposed(t, 3), -proposed(t, 4),
                       -proposed(t, 5)}};
    }
    __device__ void put_bead(int t, const Shadow &o, const Shadow &n) const
    {
        float4 *b = bead + BV * t;
        if (ONE) {
            b[0] = make_float4(-o.c[0], -n.c[0], -o.c[1], -n.c[1]);
            b[1] = make_float4(-o.c[2], -n.c[2], -o.c[3], -n.c[3]);
            b[2] = make_float4(-o.c[4], -n.c[4], -o.c[5], -n.c[5]);
        } else {
            b[0] = make_float4(-o.c[0], -o.c[0], -o.c[1], -o.c[1]);
            b[1] = make_float4(-o.c[2], -o.c[2], -o.c[3], -o.c[3]);
            b[2] = make_float4(-o.c[4], -o.c[4], -o.c[5], -o.c[5]);
            b[BV - 3] = make_float4(-n.c[0], -n.c[0], -n.c[1], -n.c[1]);
            b[BV - 2] = make_float4(-n.c[2], -n.c[2], -n.c[3], -n.c[3]);
            b[BV - 1] = make_float4(-n.c[4], -n.c[4], -n.c[5], -n.c[5]);
        }
    }
};

// LJ energy changes of chunk bead t with this lane's partners of 4-vector k: of both (new minus old),
// or of the one (ONE, d1 unused).
template <class SLOT, bool ONE>
__device__ __forceinline__ void lj_changes(const SLOT &S, int t, int k, const PolyArgs &a, float &d0, float &d1)
{
    const float4 j0 = S.pos[k], j1 = S.pos[S.nP + k], j2 = S.pos[2 * S.nP + k];
    const float4 *own = S.bead + SLOT::BV * t;
    float vo0, vo1, vn0, vn1;
    lj_two(j0, j1, j2, own[0], own[1], own[2], a, vo0, vo1);
    if (ONE) {  // (old, new) of one partner
        d0 = vo1 - vo0;
        d1 = 0.0f;
        return;
    }
    lj_two(j0, j1, j2, own[SLOT::BV - 3], own[SLOT::BV - 2], own[SLOT::BV - 1], a, vn0, vn1);
    d0 = vn0 - vo0;
    d1 = vn1 - vo1;
}

__device__ __forceinline__ void kahan_add(float &s, float &c, float v)
{
    const float y = v - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
}
enum : uint32_t { kReady = 0u, kLate = 1u, kNoPoint = 2u, kLateNext = 3u };

// Sweeps: G lanes per walker, 32/G walkers a warp, all on the same bead i.  The two bonds of bead i
// (FENE) are taken by lanes 0 and 1 of the group, the other partners (LJ, |i - j| >= 2) by lanes
// j mod G, in ascending order, so the FP32 sums do not depend on anything else.
//
// Bound by issue and by fixed latencies (3.4 warps a scheduler at 4096 walkers), so what is not pair
// work is taken out of the serial loop: a bead is visited once a sweep and stands still until then,
// so its random words, its proposed position and the energies of its new bonds (the left one for
// both outcomes of the bead before it) are known before the loop reaches it.  Every lane prepares
// its own beads of the next poly_chunk beads, and the attempt only reads them.  Accepted moves reach
// the int64 master coordinates behind the chunk, in parallel again.  Pair energies are evaluated for
// two partners at once in packed instructions (lj_two).  With rotations (MOVES) a proposal about
// bead i - 1 needs that bead's outcome: its unit vector is prepared, the position (binary64, one
// axis a lane) made when the bead is reached.
//
// NP > 0 (shifts, NP 4-vectors of partners a lane; kOnePartner: N <= G): the pair terms of bead
// i + 1 do not depend on the outcome of bead i, which is bonded to it, so they are evaluated beside
// the sum, the conversion, the table load and the decision of bead i, whose latencies they fill.
// NP = 0 evaluates them in the attempt (any N).
constexpr int kOnePartner = 5;
template <int G, int MOVES, int NP>
__global__ void __launch_bounds__(kMaxSweepBlock) k_sweep_polymer(const PolyArgs a)
{
    constexpr int W = 32 / G;
    constexpr int CH = poly_chunk<G>();
    constexpr bool ONE = NP == kOnePartner;
    // One or two lanes a walker have no others to prepare bonds beside them, so they evaluate the two
    // bonds of an attempt in it, of one outcome of the bead before instead of both (N = 5, 32768 walkers,
    // 122 sweeps: 1.32 against 1.51 ms, one lane); with rotations every grouping does.
    constexpr bool LATE = MOVES || G <= 2;
    constexpr bool HOLD = !MOVES && G == 1;  // the bead's master coordinates and step stay in registers
    constexpr int NV = ONE ? 1 : (NP > 0 ? NP : 1);  // 4-vectors evaluated ahead
    using Slot = PolySlot<G, MOVES, ONE>;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5, N = a.N;
    const int gi = lane / G, li = lane % G;
    const int spb = wpb * W, slot = wib * W + gi;
    const size_t sst = Slot::bytes(N);
    const Slot S(smem + slot * sst, N);
    // the block's histogram counters and its count of finished warps, behind all slots
    unsigned *hs = (unsigned *)(smem + spb * sst);
    unsigned *done = hs + a.B;
    for (int i = threadIdx.x; i <= a.B; i += blockDim.x) hs[i] = 0u;
    __syncthreads();
    const int w0 = (blockIdx.x * wpb + wib) * W;
    if (w0 >= a.p) return;  // whole warps only; no block-wide barrier follows
    const int w = w0 + gi;
    const bool active = w < a.p;
    const bool counts = active && li == 0;  // the lane that counts its walker's visits
    const bool visits = counts && a.record == 0;
    const int wr = active ? w : w0;  // a group past the last walker shadows the warp's first one, read-only
    const uint32_t wid = (uint32_t)(wr + a.walker_offset);
    long long *Xg = a.X + (size_t)wr * 3 * N;
    long long E = a.E[wr] - a.elo_q;  // energies relative to the window
    int b = poly_bin_rel(E, a);
    bool inside = (unsigned)b < (unsigned)a.B;
    long long lw = __ldg(a.lnWq + (inside ? b : 0));  // ln W of the current bin
    const uint32_t g0 = (uint32_t)(a.state->sweep_counter + a.sweep_base);
    // metrics: accepted moves and tunnelling between bins 0 and B-1 (group-uniform values)
    unsigned long long nacc = 0;
    unsigned ev = 0;
    int tst = (active && a.tun) ? a.tun[w] : 0;
    const float kStep = (float)a.step_q * 0x1p-44f;
    for (int64_t sw = 0; sw < a.sweeps; ++sw) {
        const uint32_t g = g0 + (uint32_t)sw;
        const long long A0 = Xg[0], A1 = Xg[N], A2 = Xg[2 * N];
        for (int j = li; j < N; j += G) {
            Shadow p;
            grid_to_ff(Xg[j] - A0, p.c[0], p.c[3]);
            grid_to_ff(Xg[N + j] - A1, p.c[1], p.c[4]);
            grid_to_ff(Xg[2 * N + j] - A2, p.c[2], p.c[5]);
            S.put(j, p);
        }
        __syncwarp();
        for (int j = li; j <= N; j += G) {
            float v = 0.0f;
            if (j > 0 && j < N) {
                const Shadow p = S.get(j - 1), r = S.get(j);
                const float dx = (p.c[0] - r.c[0]) + (p.c[3] - r.c[3]);
                const float dy = (p.c[1] - r.c[1]) + (p.c[4] - r.c[4]);
                const float dz = (p.c[2] - r.c[2]) + (p.c[5] - r.c[5]);
                v = fene_energy(dx * dx + dy * dy + dz * dz, a);
            }
            S.eb[j] = v;
        }
#pragma unroll 1
        for (int c0 = 0; c0 < N; c0 += CH) {
            // ---- prepare the chunk, a bead a lane
            long long x_own[3] = {0, 0, 0};  // HOLD: this lane's bead of the chunk
            int s_own[3] = {0, 0, 0};
#pragma unroll 1
            for (int t = li; t < CH; t += G) {
                const int j = c0 + t;
                if (j >= N) break;
                const uint4 r = philox4x32_10_rk(make_uint4((uint32_t)j, g, wid, kTagSweep), a.rk);
                // move (u - 2^31) * 1229 grid units per axis: exact on the int64 master
                // coordinates; the float-pair shadow moves by the same amount in FP32
                // (the shadows are rebuilt exactly from the masters every sweep)
                const int sx = (int)(r.x ^ 0x80000000u), sy = (int)(r.y ^ 0x80000000u), sz = (int)(r.z ^ 0x80000000u);
                const Shadow p = S.get(j);
                const float dx = (float)sx * kStep, dy = (float)sy * kStep, dz = (float)sz * kStep;
                const float xo = p.c[0], yo = p.c[1], zo = p.c[2];
                float xn = xo + dx, yn = yo + dy, zn = zo + dz;
                float lxn = p.c[3] + ((xo - xn) + dx), lyn = p.c[4] + ((yo - yn) + dy), lzn = p.c[5] + ((zo - zn) + dz);
                if (MOVES) {
                    const long long X0 = Xg[j], X1 = Xg[N + j], X2 = Xg[2 * N + j];
                    long long n0 = X0 + (long long)sx * (long long)a.step_q, n1 = X1 + (long long)sy * (long long)a.step_q,
                              n2 = X2 + (long long)sz * (long long)a.step_q;
                    const uint4 mv = philox4x32_10_rk(make_uint4((uint32_t)j, g, wid, kTagPolyMove), a.rk);
                    uint32_t how = kReady;
                    if (mv.x >= 0x80000000u) {  // spherical rotation about a bonded neighbour
                        double n[3];
                        const bool next = j == 0 || (j != N - 1 && (mv.y & 1u));
                        if (!poly_unit(j, g, wid, mv, a.rk, n)) {
                            how = kNoPoint;
                        } else if (G > 2 && next) {  // about bead j + 1, not visited yet
                            // (one or two lanes take both pivots in the attempt: the binary64 work once)
                            const long long P0 = Xg[j + 1], P1 = Xg[N + j + 1], P2 = Xg[2 * N + j + 1];
                            const double d = poly_distance(poly_axis_diff(X0, P0), poly_axis_diff(X1, P1),
                                                           poly_axis_diff(X2, P2));
                            n0 = poly_rotated(P0, n[0], d);
                            n1 = poly_rotated(P1, n[1], d);
                            n2 = poly_rotated(P2, n[2], d);
                            grid_to_ff(n0 - A0, xn, lxn);
                            grid_to_ff(n1 - A1, yn, lyn);
                            grid_to_ff(n2 - A2, zn, lzn);
                        } else {  // about bead j - 1: when it has been visited
                            how = next ? kLateNext : kLate;
                            n0 = __double_as_longlong(n[0]);
                            n1 = __double_as_longlong(n[1]);
                            n2 = __double_as_longlong(n[2]);
                        }
                    }
                    S.nx[3 * t] = n0;
                    S.nx[3 * t + 1] = n1;
                    S.nx[3 * t + 2] = n2;
                    S.how[t] = how;
                } else if (HOLD) {
                    x_own[0] = Xg[j];
                    x_own[1] = Xg[N + j];
                    x_own[2] = Xg[2 * N + j];
                    s_own[0] = sx;
                    s_own[1] = sy;
                    s_own[2] = sz;
                } else {
                    S.how[3 * t] = r.x;
                    S.how[3 * t + 1] = r.y;
                    S.how[3 * t + 2] = r.z;
                }
                S.put_bead(t, p, Shadow{{xn, yn, zn, lxn, lyn, lzn}});
                // the acceptance test u 2^-32 < exp(d) is taken as ln(u 2^-32) < d: the logarithm
                // (FP32, -inf for u = 0) is taken here, off the serial path
                S.rec[t] = make_float4(0.0f, 0.0f, 0.0f, logf((float)r.w * 0x1p-32f));
            }
            __syncwarp();
            if (!LATE) {
#pragma unroll 1
                for (int t = li; t < CH; t += G) {
                    const int j = c0 + t;
                    if (j >= N) break;
                    // (the bead before the chunk stands where pos has it)
                    const Shadow p = S.get_proposed(t);
                    const float l0 = bond_between(p, S.get(max(j - 1, 0)), a);
                    const float l1 = bond_between(p, S.get_proposed(max(t - 1, 0)), a);
                    const float r = bond_between(p, S.get(min(j + 1, N - 1)), a);
                    S.nr[t] = r;
                    S.rec[t].x = j > 0 ? l0 - S.eb[j] : 0.0f;
                    S.rec[t].y = l1;
                    S.rec[t].z = j + 1 < N ? r - S.eb[j + 1] : 0.0f;
                }
                __syncwarp();
#pragma unroll 1
                for (int t = li; t < CH; t += G)
                    if (t > 0 && c0 + t < N) S.rec[t].y -= S.nr[t - 1];  // (only used if bead t - 1 moved: not NaN)
                __syncwarp();
            }
            // ---- the attempts, one after the other
            const int nt = min(CH, N - c0);
            uint32_t accs = 0u;   // accepted beads of the chunk (group-uniform)
            bool acc = false;     // the bead before was moved
            const int kc = min(li, 5);  // G >= 8: the shadow component this lane writes
            // The unrolled loop, in two versions: for a warp with a walker that is not inside the window yet
            // (some chains that start with beads on top of each other take long), and for one without
            // (inside, none leaves the window again).
            auto unrolled = [&](auto walk) {
                constexpr bool WALK = decltype(walk)::value;
                const long long span = a.ehi_q - a.elo_q;
                long long dist = b < 0 ? -E : E - span;  // outside: distance to the window
                float4 rec_n = S.rec[0];
                float own_n = S.proposed(0, kc);
                float dn[2 * NV];  // pair terms of the next attempt
#pragma unroll
                for (int m = 0; m < NV; ++m) lj_changes<Slot, ONE>(S, 0, G * m + li, a, dn[2 * m], dn[2 * m + 1]);
#pragma unroll 1
                for (int t = 0; t < nt; ++t) {
                    const int i = c0 + t, tn = min(t + 1, CH - 1);  // (behind the chunk's end: not used)
                    const float4 rec = rec_n;
                    const float own = own_n;
                    rec_n = S.rec[tn];
                    own_n = S.proposed(tn, kc);
                    // the sums as in the other loop below; a broken bond (NaN) or a lane sum that is too
                    // large makes the walker's sum NaN, and the move is rejected
                    float s = 0.0f + (li == 0 ? (acc ? rec.y : rec.x) : (li == 1 ? rec.z : 0.0f)), c = 0.0f;
                    const unsigned u = (unsigned)(li - i + 1);
#pragma unroll
                    for (int m = 0; m < NV; ++m) {
                        const int j = li + 2 * G * m;
                        if (u + 2 * G * m > 2u && j < N) kahan_add(s, c, dn[2 * m]);
                        if (!ONE && u + 2 * G * m + G > 2u && j + G < N) kahan_add(s, c, dn[2 * m + 1]);
                    }
#pragma unroll
                    for (int m = 0; m < NV; ++m) lj_changes<Slot, ONE>(S, tn, G * m + li, a, dn[2 * m], dn[2 * m + 1]);
                    float lane_sum = fabsf(s) < 4194304.0f ? s - c : __int_as_float(0x7fffffff);
#pragma unroll
                    for (int off = G / 2; off; off >>= 1) lane_sum += __shfl_xor_sync(0xffffffffu, lane_sum, off);
                    const long long En = E + float_to_q32<G>(lane_sum);
                    const int bn = poly_bin_rel(En, a);
                    const bool lands = (unsigned)bn < (unsigned)a.B && lane_sum == lane_sum;
                    const long long lwn = __ldg(a.lnWq + (lands ? bn : 0));
                    const long long dq = lwn - lw;
                    acc = lands && (dq >= 0 || less_than_q32(rec.w, dq));
                    const long long dnew = bn < 0 ? -En : (bn >= a.B ? En - span : 0);
                    if (WALK) acc = inside ? acc : dnew <= dist && lane_sum == lane_sum;
                    // (selects: a branch costs more latency than what it skips)
                    if (acc && li < 6) S.set(i, kc, -own);
                    E = acc ? En : E;
                    b = acc ? bn : b;
                    lw = acc ? lwn : lw;
                    if (WALK) {
                        inside = acc ? lands : inside;
                        dist = acc ? dnew : dist;
                    }
                    accs |= acc ? 1u << t : 0u;
                    __syncwarp();
                    if (visits && (!WALK || inside)) count_visits(&hs[b], 1u);
                }
            };
            if (NP > 0 && !a.trace) {
                if (__any_sync(0xffffffffu, !inside)) unrolled(std::true_type{});
                else unrolled(std::false_type{});
            } else {
            // (The loop for anything: rotations, any G, traces.)
#pragma unroll 1
            for (int t = 0; t < nt; ++t) {
                const int i = c0 + t;
                bool no_point = false;
                if (MOVES) {
                    const uint32_t how = S.how[t];
                    no_point = how == kNoPoint;
                    const bool turn = how == kLate || (G <= 2 && how == kLateNext);
                    if (__any_sync(0xffffffffu, turn)) {
                        // about bead i - 1, where it is now; lanes 0, 1, 2 of the group an axis each
                        // (fewer lanes take the axes in turn)
                        const int pv = G <= 2 && how == kLateNext ? i + 1 : (i > 0 ? i - 1 : 0);
                        double dd[3];
                        if (G >= 4) {
                            const int c = min(li, 2);
                            const double own = poly_axis_diff(Xg[c * N + i], Xg[c * N + pv]);
#pragma unroll
                            for (int k = 0; k < 3; ++k) dd[k] = __shfl_sync(0xffffffffu, own, gi * G + min(k, G - 1));
                        } else {
#pragma unroll
                            for (int k = 0; k < 3; ++k) dd[k] = poly_axis_diff(Xg[k * N + i], Xg[k * N + pv]);
                        }
                        const double d = poly_distance(dd[0], dd[1], dd[2]);
                        if (turn) {
                            for (int c = li; c < 3; c += G) {
                                const long long nn =
                                    poly_rotated(Xg[c * N + pv], __longlong_as_double(S.nx[3 * t + c]), d);
                                float hi, lo;
                                grid_to_ff(nn - (c == 0 ? A0 : (c == 1 ? A1 : A2)), hi, lo);
                                S.nx[3 * t + c] = nn;
                                S.set_proposed(t, c, hi);
                                S.set_proposed(t, 3 + c, lo);
                            }
                        }
                        __syncwarp();
                    }
                }
                const float4 rec = S.rec[t];
                // the bonds (i-1, i) and (i, i+1): lanes 0 and 1 of the group, or the walker's only lane
                // for both when G = 1; a broken bond counts as unchanged (the move is rejected)
                float s = 0.0f, c = 0.0f;
                bool broken = false;
                float vb[2] = {0.0f, 0.0f};
#pragma unroll
                for (int k = 0; k < (G == 1 ? 2 : 1); ++k) {
                    const bool left = (G == 1) ? k == 0 : li == 0;
                    float d = left ? (acc ? rec.y : rec.x) : rec.z;
                    if (LATE) {
                        d = 0.0f;
                        if ((G == 1 || li < 2) && (left ? i > 0 : i + 1 < N)) {
                            vb[k] = bond_between(S.get_proposed(t), S.get(left ? i - 1 : i + 1), a);
                            d = vb[k] - S.eb[left ? i : i + 1];
                        }
                    }
                    if (G == 1 || li < 2) {
                        broken = broken || d != d;
                        kahan_add(s, c, d == d ? d : 0.0f);
                    }
                }
                // the other partners, in order, compensated (Kahan); li + 2 G m - i + 1 is 0, 1, 2 for
                // the bonded beads and i itself
                const unsigned u = (unsigned)(li - i + 1);
#pragma unroll 1
                for (int e = (G == 1 ? 1 : 0); li + 2 * G * e < N; ++e) {
                    // (one lane: the pair i / 2 is the bead and one bonded to it, so the others only)
                    const int m = G == 1 && e <= i / 2 ? e - 1 : e;
                    float d0, d1;
                    lj_changes<Slot, ONE>(S, t, G * m + li, a, d0, d1);
                    if (u + 2 * G * m > 2u) kahan_add(s, c, d0);
                    if (!ONE && u + 2 * G * m + G > 2u && li + 2 * G * m + G < N) kahan_add(s, c, d1);
                }
                // |lane sum| >= 2^22 only for overlapping beads: such a move is rejected
                const bool huge = !(fabsf(s) < 4194304.0f);
                const bool refused = group_any<G>(huge || broken, gi) || no_point;
                // the lanes' compensated sums added in FP32 by a butterfly: every lane adds the same
                // two operands at every step (a + b = b + a exactly), so all lanes of the group end
                // with the same sum, converted once to 2^-32 fixed point
                float lane_sum = s - c;
#pragma unroll
                for (int off = G / 2; off; off >>= 1) lane_sum += __shfl_xor_sync(0xffffffffu, lane_sum, off);
                const long long q = float_to_q32<G>(lane_sum);  // (a refused move's is not used)
                const long long En = E + q;
                const int bn = poly_bin_rel(En, a);
                const bool lands = (unsigned)bn < (unsigned)a.B;
                const long long lwn = __ldg(a.lnWq + (lands ? bn : 0));
                const long long dq = lwn - lw;
                // accept iff d >= 0 or ln(u 2^-32) < d
                acc = lands && (dq >= 0 || rec.w < q32_to_float(dq));
                if (!inside) {  // walking in: not further from the window than before
                    const long long span = a.ehi_q - a.elo_q;
                    const long long dold = (b < 0) ? -E : E - span;
                    const long long dnew = (bn < 0) ? -En : (bn >= a.B ? En - span : 0);
                    acc = dnew <= dold;
                }
                acc = acc && !refused;
                if (a.trace) {  // parity inspection only
                    const bool any_huge = group_any<G>(huge, gi), any_broken = group_any<G>(broken, gi) || no_point;
                    PolyTraceRec r;
                    r.dq = any_huge ? 0 : q;
                    r.E = (acc ? En : E) + a.elo_q;
                    r.bn = any_huge ? poly_bin_rel(E, a) : bn;
                    r.b = acc ? bn : b;
                    r.flags = (acc ? 1 : 0) | (any_broken ? 2 : 0) | (any_huge ? 4 : 0);
                    r.pad = 0;
                    if (counts)
                        a.trace[((size_t)w * (size_t)a.trace_sweeps + (size_t)(a.sweep_base + sw)) * (size_t)N + i] = r;
                }
                if (acc) {
                    for (int k = li; k < 6; k += G) S.set(i, k, -S.proposed(t, k));
                    if (LATE) {
                        if (G == 1) {
                            if (i > 0) S.eb[i] = vb[0];
                            if (i + 1 < N) S.eb[i + 1] = vb[1];
                        } else if (li < 2) {
                            S.eb[li == 0 ? i : i + 1] = vb[0];
                        }
                    }
                    if (MOVES && counts) {
                        Xg[i] = S.nx[3 * t];
                        Xg[N + i] = S.nx[3 * t + 1];
                        Xg[2 * N + i] = S.nx[3 * t + 2];
                    }
                    E = En;
                    b = bn;
                    lw = lwn;
                    inside = lands;
                    accs |= 1u << t;
                }
                __syncwarp();
                if (visits && inside) count_visits(&hs[b], 1u);
            }
            }
            nacc += (unsigned)__popc(accs);
            // the bond into the next chunk (the others are rebuilt with the next sweep)
            if (!LATE && li == 0 && ((accs >> (nt - 1)) & 1u) && c0 + nt < N) S.eb[c0 + nt] = S.nr[nt - 1];
            // ---- the accepted moves on the master coordinates (32 x 32-bit products: the grid step fits an int)
            if (HOLD) {
                if (active && ((accs >> li) & 1u)) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) Xg[c * N + c0 + li] = x_own[c] + (long long)s_own[c] * (long long)a.step_q;
                }
            } else if (!MOVES && active) {
#pragma unroll 1
                for (int t = li; t < nt; t += G) {
                    if ((accs >> t) & 1u) {
#pragma unroll
                        for (int c = 0; c < 3; ++c)
                            Xg[c * N + c0 + t] += (long long)(int)(S.how[3 * t + c] ^ 0x80000000u) * (long long)a.step_q;
                    }
                }
            }
            __syncwarp();  // the chunk's records are rewritten
        }
        if (a.record == 1 && counts && inside) count_visits(&hs[b], 1u);
        tunnel_step(b, 0, a.B - 1, tst, ev);
        __syncwarp();
    }
    // the block's last warp to finish adds the counters to the histogram (the launch's sweeps
    // fit the 32-bit counters: launch_g splits longer iterates)
    __threadfence_block();  // this warp's visits are counted before it reports
    __syncwarp();
    const int nwarps = min(wpb, (a.p - blockIdx.x * spb + W - 1) / W);  // warps of the block with walkers
    unsigned last = 0u;
    if (lane == 0) last = (atomicAdd(done, 1u) == (unsigned)nwarps - 1u);
    if (__shfl_sync(0xffffffffu, last, 0)) {
        __threadfence_block();
        for (int i = lane; i < a.B; i += 32) {
            const unsigned c = hs[i];
            if (c) atomicAdd(a.H + i, (unsigned long long)c);
        }
    }
    const bool lead = li == 0 && active;
    flush_metrics(a.metrics, lead ? nacc : 0ull, lead ? ev : 0u);
    if (lead && a.tun) a.tun[w] = (uint8_t)tst;
    if (!active) return;  // (no warp-wide operation follows)
    // recentre on bead 0 (an exact grid shift) and write back
    const long long A0 = Xg[0], A1 = Xg[N], A2 = Xg[2 * N];
    __syncwarp(__activemask());
    for (int t = li; t < N; t += G) {
        Xg[t] -= A0;
        Xg[N + t] -= A1;
        Xg[2 * N + t] -= A2;
    }
    if (li == 0) {
        a.E[w] = E + a.elo_q;
        a.bin[w] = b;
    }
}

__global__ void k_poly_lnwq(const double *lnW, long long *lnWq, int B)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B) lnWq[b] = __double2ll_rn(__dmul_rn(lnW[b], 0x1p32));
}

__global__ void k_poly_unpack(const PolyArgs a, double *coords, double *energies)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n = (long long)a.p * a.N;
    if (t >= n) return;
    const int w = (int)(t / a.N), j = (int)(t - (t / a.N) * a.N);
    const long long *X = a.X + (size_t)w * 3 * a.N;
    for (int c = 0; c < 3; ++c) coords[t * 3 + c] = (double)X[c * a.N + j] * 0x1p-44;
    if (j == 0) energies[w] = (double)a.E[w] * 0x1p-32;
}

cudaError_t launch_poly_init(const PolyArgs &a, cudaStream_t s)
{
    k_poly_init<<<(a.p + 127) / 128, 128, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_poly_energy(const PolyArgs &a, int track_drift, cudaStream_t s)
{
    const int wpb = 4;
    const size_t smem = (size_t)wpb * 6 * a.N * sizeof(float);
    k_poly_energy<<<(a.p + wpb - 1) / wpb, wpb * 32, smem, s>>>(a, track_drift);
    return cudaGetLastError();
}

// Shared memory of one warp of the sweep: 32/G walkers' slots.
template <int G, int MOVES, int NP>
static size_t poly_warp_smem(const PolyArgs &a)
{
    return (size_t)(32 / G) * (NP == kOnePartner ? PolySlot<G, MOVES, true>::bytes(a.N) : PolySlot<G, MOVES, false>::bytes(a.N));
}

constexpr size_t kPolySmemMax = 227u * 1024u;

// The block's 32-bit histogram counters (one per bin), after the warps' shared memory.
static size_t poly_hist_smem(const PolyArgs &a)
{
    return ((size_t)(a.B + 1) * sizeof(unsigned) + 15) / 16 * 16;
}

// Warps a block when the caller has set none: the walkers' warps spread evenly over the SMs (the
// fullest SM sets the time: 256-thread blocks put 16 warps on most SMs and 8 on the rest at 4096
// walkers, where 14 everywhere do), in blocks of at most eight warps.
static int poly_auto_warps(int p, int walkers_a_warp)
{
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm < 1)
        return 8;
    const int warps = (p + walkers_a_warp - 1) / walkers_a_warp, each = (warps + nsm - 1) / nsm;
    const int blocks = (each + 7) / 8;
    return (each + blocks - 1) / blocks;
}

template <int G, int MOVES, int NP>
static cudaError_t launch_g(const PolyArgs &a, int block, cudaStream_t s)
{
    // as many warps of the requested block as fit the shared memory of one block
    int wpb = block > 0 ? block / 32 : poly_auto_warps(a.p, 32 / G);
    const size_t per_warp = poly_warp_smem<G, MOVES, NP>(a), hist = poly_hist_smem(a);
    if (hist + (size_t)wpb * per_warp > kPolySmemMax)
        wpb = hist < kPolySmemMax ? (int)((kPolySmemMax - hist) / per_warp) : 0;
    if (wpb < 1) return cudaErrorInvalidValue;
    block = 32 * wpb;
    const int spb = wpb * (32 / G);
    const size_t smem = (size_t)wpb * per_warp + hist;
    const int nblk = (a.p + spb - 1) / spb;
    cudaError_t e = allow_dynamic_smem(k_sweep_polymer<G, MOVES, NP>, kPolySmemMax);
    if (e != cudaSuccess) return e;
    // one launch per chunk of sweeps whose visits fit the block's 32-bit counters (spb N a sweep
    // at most), or fewer ("flush_every")
    int64_t fe = (int64_t)(0xFFFFFFFFu / (unsigned)(spb * a.N));
    if (a.flush_every > 0 && a.flush_every < fe) fe = a.flush_every;
    for (int64_t s0 = 0; s0 < a.sweeps; s0 += fe) {
        PolyArgs c = a;
        c.sweep_base = s0;
        c.sweeps = (a.sweeps - s0 < fe) ? a.sweeps - s0 : fe;
        c.trace_sweeps = a.sweeps;
        k_sweep_polymer<G, MOVES, NP><<<nblk, block, smem, s>>>(c);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Lanes per walker: the fixed cost of an attempt (group reductions, the bin and
// weight lookups, the decision) is shared by the 32/G walkers of a warp, the pair
// terms are spread over G lanes.  A request for a grouping whose warp does not fit
// the shared memory of a block falls back to the next larger G.  Measured on GB300
// with 2048 walkers (pilot window, N = 13, 751 sweeps): 21.7, 14.3,
// 10.7, 7.0, 4.5 and 7.3 ms with 1, 2, 4, 8, 16 and 32 lanes (the last before it ran as 16).
// Fewer lanes share the fixed cost among more walkers but leave 2048 G / 32 warps to hide
// latency and prepare more beads one after the other, and only 16 has the loops unrolled by the
// partners of a lane; so 16 is the default.
// (What fits is still counted in the bytes of a slot that holds a whole sweep's random words: the
// lanes decide the rounding of the FP32 sums, so a request keeps the grouping it always had.  The
// slots above are smaller where this line matters.)
static bool poly_fits(const PolyArgs &a, int g)
{
    const size_t slot = (size_t)((7 * a.N + 3) & ~3) * sizeof(float) + (size_t)a.N * (a.moves ? 2 : 1) * sizeof(uint4);
    return (size_t)(32 / g) * slot + poly_hist_smem(a) <= kPolySmemMax;
}

int poly_lanes(const PolyArgs &a, int requested)
{
    int g = (requested == 1 || requested == 2 || requested == 4 || requested == 8 || requested == 16 ||
             requested == 32) ? requested : 16;
    if (g == 1 && !poly_fits(a, 1)) g = 2;
    if (g == 2 && !poly_fits(a, 2)) g = 4;
    // With at most a bead a lane, further lanes only add zeros to the same sums, so a smaller grouping
    // gives the same bits: 32768 walkers of N = 2, 305 sweeps, 1.09 ms with 2 lanes (4: 2.15, 8: 4.0,
    // 32: 14.0 ms), of N = 3, 203 sweeps, 4.96 ms with 16 (32: 10.8).
    if (a.N == 2 && (g == 4 || g == 8 || g == 32)) g = 2;
    if (a.N <= 16 && g == 32) g = 16;
    return g;
}

cudaError_t launch_poly_sweep(const PolyArgs &a, int block, cudaStream_t s)
{
    if (!polymer_supported(a.N)) return cudaErrorInvalidValue;
    switch (poly_lanes(a, a.lanes)) {
    case 1: return a.moves ? launch_g<1, 1, 0>(a, block, s) : launch_g<1, 0, 0>(a, block, s);
    case 2: return a.moves ? launch_g<2, 1, 0>(a, block, s) : launch_g<2, 0, 0>(a, block, s);
    case 4: return a.moves ? launch_g<4, 1, 0>(a, block, s) : launch_g<4, 0, 0>(a, block, s);
    case 8: return a.moves ? launch_g<8, 1, 0>(a, block, s) : launch_g<8, 0, 0>(a, block, s);
    case 16:  // the default: unrolled by the partners of a lane
        if (a.N <= 16) return a.moves ? launch_g<16, 1, 0>(a, block, s) : launch_g<16, 0, kOnePartner>(a, block, s);
        if (a.moves) return launch_g<16, 1, 0>(a, block, s);
        switch ((a.N + 31) / 32) {
        case 1: return launch_g<16, 0, 1>(a, block, s);
        case 2: return launch_g<16, 0, 2>(a, block, s);
        case 3: return launch_g<16, 0, 3>(a, block, s);
        default: return launch_g<16, 0, 4>(a, block, s);
        }
    default: return a.moves ? launch_g<32, 1, 0>(a, block, s) : launch_g<32, 0, 0>(a, block, s);
    }
}

cudaError_t launch_poly_lnwq(const double *lnW, long long *lnWq, int B, cudaStream_t s)
{
    k_poly_lnwq<<<(B + 255) / 256, 256, 0, s>>>(lnW, lnWq, B);
    return cudaGetLastError();
}

cudaError_t launch_poly_unpack(const PolyArgs &a, double *coords, double *energies, cudaStream_t s)
{
    const long long n = (long long)a.p * a.N;
    k_poly_unpack<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, coords, energies);
    return cudaGetLastError();
}

}  // namespace muca
