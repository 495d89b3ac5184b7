// update.cu -- everything between two sweeps of the parallel multicanonical
// loop (paper, Fig. 1: "the histograms are merged, the new weights are
// estimated and distributed to all processes again"):
//   k_merge       integer sum of the per-block histograms (exact, so the
//                 result does not depend on how walkers are grouped);
//   k_recursion   accumulated-statistics weight recursion in log form
//                 ("use the full statistics of previous iterations ...
//                 implemented with logarithmic weights"), plus the flatness
//                 statistics of the merged histogram;
//   k_thresholds  the integer acceptance table T[b][c] = floor(2^32 exp(d)),
//                 d = ln W(target) - ln W(b) (- beta dE for the multimagnetic
//                 ensemble, Eq. 3), or "always" for d >= 0;
//   k_reweight    Eq. (2): canonical averages from the merged histogram.
// All binary64 arithmetic of the recursion and the thresholds uses explicit
// round-to-nearest intrinsics (this file is also built with -fmad=false), so
// the results are the same bits on every run and every compiler.
#include <cooperative_groups.h>

#include <cfloat>

#include "muca_device.cuh"
#include "muca_internal.h"

namespace muca {

#define kNegInf (__longlong_as_double((long long)0xfff0000000000000ULL))

// Merge: 32 bins x 8 slot rows a block.  A thread that walked all ceil(p / block) slots of its bin
// alone waited for one L2 round trip after the other (52 us for 128 slots of 8193 bins, 34 us for
// the nine systems of the mix); eight rows take 6.3 and 4.6 us.  (A row still goes slot by slot: a
// slot's count is cleared before the next is read.)
constexpr int kMergeBins = 32, kMergeRows = 8;

__device__ __forceinline__ void merge_body(const UpdateArgs &a)
{
    __shared__ unsigned long long part[kMergeRows][kMergeBins];
    const int tx = threadIdx.x % kMergeBins, ty = threadIdx.x / kMergeBins;
    const int b = blockIdx.x * kMergeBins + tx;
    if (blockIdx.x * kMergeBins >= a.B) return;  // whole blocks only
    unsigned long long s = 0ull;
    if (b < a.B) {
#pragma unroll 4
        for (int k = ty; k < a.nblocks; k += kMergeRows) {
            unsigned long long *p = a.Hpart + (size_t)k * a.B + b;
            const unsigned long long v = *p;
            s += v;
            if (v) *p = 0ull;
        }
    }
    part[ty][tx] = s;
    __syncthreads();
    if (ty == 0 && b < a.B) {
#pragma unroll
        for (int r = 1; r < kMergeRows; ++r) s += part[r][tx];
        a.H[b] = s;
    }
}

__global__ void __launch_bounds__(kMergeBins *kMergeRows) k_merge(const UpdateArgs a) { merge_body(a); }

__global__ void __launch_bounds__(kMergeBins *kMergeRows) k_merge_batch(const UpdateArgs *__restrict__ arr)
{
    merge_body(arr[blockIdx.y]);
}

// The sequential sum acc <- RN(acc + r_k) of the recursion, with its roundings, a window of
// kPrefixWindow terms at a time.  A dependent binary64 addition takes 64 cycles on GB300, 252 us for
// the 8192 terms of L = 64 Potts; the windows take about 15 where the sum is smooth.
// While acc stays in one binade [2^e, 2^(e+1)) it is an integer multiple A of u = 2^(e-52) and
// RN(A u + r) = u (A + round(r / u)), where a tie rounds to an even sum: a term with a fractional
// part of exactly one half adds f + ((A + f) & 1), f = floor(r / u).  So every term is a map of A
// that depends on A through its parity alone, such maps compose associatively, and a window is an
// integer scan of (increment for even A, increment for odd A).  The scan is right up to the first
// term at which the sum leaves 2^52 < A < 2^53 or whose |r| is not below 2^e; that term is added in
// binary64 and the next window starts behind it.  acc = 0 (bins not visited yet) passes over zero
// terms.  For negative acc everything is mirrored, as rounding to nearest even is.
// A window costs about as much as twenty additions, so behind the term that ended one early some
// more are added singly: eight, or, where the window got less than kPrefixWorth terms far (a sum
// that wanders about small values crosses binades at every few terms), four times as many as the
// last time; at worst all are.  (These numbers had the least cost over the ln W of the mix's
// systems and of L = 32, of init 1..64, worth 16..64, factors 2 and 4.)
constexpr int kRecThreads = 256;
constexpr int kPrefixPerThread = 2;
constexpr int kPrefixWindow = kRecThreads * kPrefixPerThread;
constexpr int kPrefixWorth = 16, kPrefixSerialMax = 2048;

struct PrefixShared {
    long long tot[kRecThreads / 32][2];  // each warp's composed map
    int first;                           // first term of the window that the scan cannot take
    double acc;                          // sum before that term
};

__device__ __forceinline__ void prefix_term(double r, bool neg, bool zero, int e, long long &f, bool &tie, bool &bad)
{
    const unsigned long long bits = (unsigned long long)__double_as_longlong(r);
    unsigned long long m = bits & 0x000fffffffffffffull;
    int er = (int)((bits >> 52) & 0x7ffull);
    f = 0;
    tie = false;
    if (zero) {
        bad = (bits << 1) != 0ull;  // (+-0 leaves +0 as it is)
        return;
    }
    if (er) m |= 0x0010000000000000ull;
    else er = 1;
    const int sh = e - er;  // r / u = m 2^-sh
    bad = sh <= 0 && m != 0ull;  // |r| >= 2^e, infinite or NaN
    if (bad || sh > 54 || m == 0ull) return;  // (sh > 54: |r / u| < 1/4)
    const unsigned long long fl = m >> sh, rem = m & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
    tie = rem == half;
    const bool minus = ((bits >> 63) != 0ull) != neg;
    const long long up = (long long)(fl + (rem > half ? 1ull : 0ull));
    f = tie ? (minus ? -(long long)fl - 1 : (long long)fl) : (minus ? -up : up);
}

__device__ __forceinline__ long long prefix_step(long long d, long long f, bool tie, long long A)
{
    return d + f + (tie ? ((A + d + f) & 1ll) : 0ll);
}

// r[k] <- r_0 + ... + r_k for k < n, every sum rounded as in sequence; r in shared memory; the
// whole block (kRecThreads) calls it.
__device__ void exact_prefix(double *r, int n, PrefixShared &ps)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double acc = 0.0;
    // a short sum is made as it stands, and so is the start of a longer one, where acc is no larger
    // than the terms yet
    int s = 0, serial = n <= 128 ? n : 16, streak = 1;
    while (s < n) {
        if (serial > 0) {
            const int end = min(s + serial, n);
            if (tid == 0) {
                // eight terms read ahead while the eight before them are added
                const int full = s + (end - s) / 8 * 8;
                double nx[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) nx[i] = r[min(s + i, end - 1)];
#pragma unroll 1
                for (int k = s; k < full; k += 8) {
                    double x[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) x[i] = nx[i];
#pragma unroll
                    for (int i = 0; i < 8; ++i) nx[i] = r[min(k + 8 + i, end - 1)];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        acc = __dadd_rn(acc, x[i]);
                        x[i] = acc;
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) r[k + i] = x[i];
                }
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (full + i < end) {
                        acc = __dadd_rn(acc, nx[i]);
                        r[full + i] = acc;
                    }
                ps.acc = acc;
            }
            __syncthreads();
            acc = ps.acc;
            s = end;
            serial = 0;
            __syncthreads();  // ps is rewritten by the next window
            continue;
        }
        const unsigned long long ab = (unsigned long long)__double_as_longlong(acc);
        const int e = (int)((ab >> 52) & 0x7ffull);
        const bool zero = ab == 0ull, neg = (ab >> 63) != 0ull;
        if (!zero && (e == 0 || e == 0x7ff)) {  // subnormal or not finite
            serial = 64;
            continue;
        }
        const int end = min(s + kPrefixWindow, n);
        const long long A0 = zero ? 0ll : (long long)((ab & 0x000fffffffffffffull) | 0x0010000000000000ull);
        const int k0 = s + tid * kPrefixPerThread;
        long long f[kPrefixPerThread];
        bool tie[kPrefixPerThread], bad[kPrefixPerThread];
        long long d0 = 0, d1 = 0;  // this thread's terms: increment for even A, for odd A
#pragma unroll
        for (int i = 0; i < kPrefixPerThread; ++i) {
            prefix_term(k0 + i < end ? r[k0 + i] : 0.0, neg, zero, e, f[i], tie[i], bad[i]);
            d0 = prefix_step(d0, f[i], tie[i], 0ll);
            d1 = prefix_step(d1, f[i], tie[i], 1ll);
        }
        // inclusive scan of the maps over the warp, then over the warps before this one; without a
        // tie in the warp (most have none) both parities move alike
        long long i0 = d0, i1 = d1;
        if (__any_sync(0xffffffffu, d0 != d1)) {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long p0 = __shfl_up_sync(0xffffffffu, i0, o), p1 = __shfl_up_sync(0xffffffffu, i1, o);
                if (lane >= o) {
                    const long long n0 = p0 + ((p0 & 1ll) ? i1 : i0), n1 = p1 + (((p1 + 1ll) & 1ll) ? i1 : i0);
                    i0 = n0;
                    i1 = n1;
                }
            }
        } else {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long p0 = __shfl_up_sync(0xffffffffu, i0, o);
                if (lane >= o) i0 += p0;
            }
            i1 = i0;
        }
        if (lane == 31) {
            ps.tot[warp][0] = i0;
            ps.tot[warp][1] = i1;
        }
        if (tid == 0) {
            ps.first = end;
            ps.acc = acc;
        }
        __syncthreads();
        long long A = A0;
        long long t0[kRecThreads / 32 - 1], t1[kRecThreads / 32 - 1];  // (read together, not in a chain)
#pragma unroll
        for (int w = 0; w < kRecThreads / 32 - 1; ++w) {
            t0[w] = ps.tot[w][0];
            t1[w] = ps.tot[w][1];
        }
#pragma unroll
        for (int w = 0; w < kRecThreads / 32 - 1; ++w)
            if (w < warp) A += (A & 1ll) ? t1[w] : t0[w];
        long long x0 = __shfl_up_sync(0xffffffffu, i0, 1), x1 = __shfl_up_sync(0xffffffffu, i1, 1);
        if (lane == 0) x0 = x1 = 0ll;
        A += (A & 1ll) ? x1 : x0;
        // the sums behind this thread's terms, while they stay inside the binade
        long long a[kPrefixPerThread];
        int bad_at = end;
#pragma unroll
        for (int i = 0; i < kPrefixPerThread; ++i) {
            A += prefix_step(0ll, f[i], tie[i], A);
            a[i] = A;
            const bool in = zero || (A > 0x0010000000000000ll && A < 0x0020000000000000ll);
            if (k0 + i < bad_at && (bad[i] || !in)) bad_at = k0 + i;
        }
        const int wmin = __reduce_min_sync(0xffffffffu, bad_at);
        if (lane == 0 && wmin < end) atomicMin(&ps.first, wmin);
        __syncthreads();
        const int v = ps.first;
#pragma unroll
        for (int i = 0; i < kPrefixPerThread; ++i) {
            if (k0 + i < v) {
                const double val = zero ? 0.0
                                        : __longlong_as_double((long long)((ab & 0xfff0000000000000ull) |
                                                                           ((unsigned long long)a[i] & 0x000fffffffffffffull)));
                r[k0 + i] = val;
                if (k0 + i == v - 1) ps.acc = val;
            }
        }
        __syncthreads();
        acc = ps.acc;
        if (v < end) {
            streak = v - s < kPrefixWorth ? min(4 * streak, kPrefixSerialMax) : 8;
            serial = streak;
        }
        s = v;
        __syncthreads();  // ps is rewritten by the next window
    }
}

// Recursion over the ordered reachable bins r_0 < ... < r_{K-1}.  For each
// neighbouring pair with h0 = H(r_k) > 0 and h1 = H(r_{k+1}) > 0:
//   g = h0 h1 / (h0 + h1);  G_k += g;  kappa = g / G_k;
//   lnR_k += kappa (ln h0 - ln h1),
// then ln W(r_0) = 0 and ln W(r_{k+1}) = ln W(r_k) + lnR_k, summed in order
// (exact_prefix).  The pairs are independent: a block takes kRecPairs of them, one logarithm and
// one pair a thread, so that they spread over the SMs (GB300 has two FP64 lanes a clock and SM, and
// 8193 bins on one SM took over 200 us); the last block to finish sums them up.  The whole
// recursion took 489 us for 8193 bins on one SM with one thread adding, and takes 50; 86 and 29
// for the 1025 bins of L = 32 Ising, 301 and 49 for the mix.  What is left is latency: the chains of
// FP64 operations (log, three divisions: about 10 us in all) and the windows of the sum.
constexpr int kRecPairs = 63;

__device__ __forceinline__ int recursion_blocks(int nreach) { return max(1, (nreach - 1 + kRecPairs - 1) / kRecPairs); }

// The iteration's metrics become the "last" ones (and are added to the totals);
// the open counters restart.  Runs once per update, after the sweeps' atomics.
__device__ __forceinline__ void close_metrics(const UpdateArgs &a)
{
    unsigned long long *m = a.metrics;
    if (!m) return;
    m[2] = m[0];
    m[3] = m[1];
    m[4] += m[0];
    m[5] += m[1];
    const unsigned long long sc = a.state->sweep_counter;
    m[6] = sc - m[7];
    m[7] = sc;
    m[0] = 0ull;
    m[1] = 0ull;
}

// Scratch of an update (UpdateArgs::scratch): the count of finished blocks, each block's
// {min, max, sum} of its bins' counts and, for the plain rule, ln W(r_k) - ln max(H(r_k), 1).
__device__ __forceinline__ void recursion_body(const UpdateArgs &a, double *sm)
{
    __shared__ double slog[kRecPairs + 1];
    __shared__ unsigned long long red[3][kRecThreads / 32];
    __shared__ PrefixShared ps;
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nblk = recursion_blocks(a.nreach);
    if ((int)blockIdx.x >= nblk) return;  // whole blocks only (batches size the grid for the largest system)
    unsigned *done = (unsigned *)a.scratch;
    unsigned long long *part = (unsigned long long *)a.scratch + 1;
    double *plain = (double *)(part + 3 * nblk);
    // the weights the merged histogram was sampled with; the last block overwrites lnW afterwards
    for (int b = blockIdx.x * kRecThreads + tid; b < a.B; b += nblk * kRecThreads) a.lnW_sampled[b] = a.lnW[b];
    const int base = blockIdx.x * kRecPairs;
    unsigned long long h = 0ull, mn = ~0ull, mx = 0ull, sum = 0ull;
    const int k = base + tid;
    if (tid <= kRecPairs && k < a.nreach) {
        h = a.H[a.rlist[k]];
        slog[tid] = h ? dm_log(__ull2double_rn(h)) : 0.0;
        if (tid < kRecPairs || k == a.nreach - 1) mn = mx = sum = h;  // (the bin two blocks share counts once)
        if (a.recursion == 1) plain[k] = __dsub_rn(a.lnW[a.rlist[k]], slog[tid]);
    }
    __syncthreads();
    if (a.recursion != 1 && tid < kRecPairs && k + 1 < a.nreach) {
        const unsigned long long h1 = a.H[a.rlist[k + 1]];
        if (h != 0ull && h1 != 0ull) {
            const double x0 = __ull2double_rn(h), x1 = __ull2double_rn(h1);
            const double g = __ddiv_rn(__dmul_rn(x0, x1), __dadd_rn(x0, x1));
            const double G = __dadd_rn(a.G[k], g);
            a.G[k] = G;
            const double kappa = __ddiv_rn(g, G);
            a.lnR[k] = __dadd_rn(a.lnR[k], __dmul_rn(kappa, __dsub_rn(slog[tid], slog[tid + 1])));
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const unsigned long long n = __shfl_xor_sync(0xffffffffu, mn, o), x = __shfl_xor_sync(0xffffffffu, mx, o);
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        mn = n < mn ? n : mn;
        mx = x > mx ? x : mx;
    }
    if (lane == 0) {
        red[0][warp] = mn;
        red[1][warp] = mx;
        red[2][warp] = sum;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < kRecThreads / 32; ++w) {
            mn = red[0][w] < mn ? red[0][w] : mn;
            mx = red[1][w] > mx ? red[1][w] : mx;
            sum += red[2][w];
        }
        part[3 * blockIdx.x] = mn;
        part[3 * blockIdx.x + 1] = mx;
        part[3 * blockIdx.x + 2] = sum;
        __threadfence();
        s_last = atomicAdd(done, 1u) == (unsigned)nblk - 1u;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (a.recursion == 1) {
        // the plain rule W(n+1) = W(n)/H(n) in log form: x_k = ln W(r_k) - ln max(H(r_k), 1),
        // ln W(r_k) = x_k - x_0 (an unvisited bin keeps its weight)
        const double x0 = __ldcg(plain);
        for (int i = tid; i < a.nreach; i += kRecThreads) a.lnW[a.rlist[i]] = __dsub_rn(__ldcg(plain + i), x0);
    } else {
        for (int i = tid; i + 1 < a.nreach; i += kRecThreads) sm[i] = __ldcg(a.lnR + i);
    }
    __syncthreads();
    if (warp == kRecThreads / 32 - 1) {  // while the first warp starts on the sum
        mn = ~0ull;
        mx = sum = 0ull;
        for (int i = lane; i < nblk; i += 32) {
            const unsigned long long n = __ldcg(part + 3 * i), x = __ldcg(part + 3 * i + 1);
            sum += __ldcg(part + 3 * i + 2);
            mn = n < mn ? n : mn;
            mx = x > mx ? x : mx;
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const unsigned long long n = __shfl_xor_sync(0xffffffffu, mn, o), x = __shfl_xor_sync(0xffffffffu, mx, o);
            sum += __shfl_xor_sync(0xffffffffu, sum, o);
            mn = n < mn ? n : mn;
            mx = x > mx ? x : mx;
        }
        if (lane == 0) {
            const double mean = __ddiv_rn(__ull2double_rn(sum), (double)a.nreach);
            a.state->flat_min = __ull2double_rn(mn);
            a.state->flat_mean = mean;
            a.state->flat_max = __ull2double_rn(mx);
            a.state->flat = (mn > 0ull) && (__ddiv_rn(__ull2double_rn(mn), mean) >= a.flat_ratio);
            a.state->iteration += 1ull;
            *done = 0u;  // ready for the next update
            close_metrics(a);
        }
    }
    if (a.recursion != 1) {
        exact_prefix(sm, a.nreach - 1, ps);
        if (tid == 0) a.lnW[a.rlist[0]] = 0.0;
        for (int i = tid; i + 1 < a.nreach; i += kRecThreads) a.lnW[a.rlist[i + 1]] = sm[i];
    }
}

__global__ void __launch_bounds__(kRecThreads) k_recursion(const UpdateArgs a)
{
    extern __shared__ double sm[];
    recursion_body(a, sm);
}

__global__ void __launch_bounds__(kRecThreads) k_recursion_batch(const UpdateArgs *__restrict__ arr)
{
    extern __shared__ double sm[];
    const UpdateArgs a = arr[blockIdx.y];
    recursion_body(a, sm);
}

__device__ __forceinline__ void thresholds_body(const UpdateArgs &a, int i)
{
    if (a.system == kPolymer) return;  // its weights go to the fixed-point table instead (k_poly_lnwq)
    const int C = num_cols(a.system);
    if (i >= a.B * C) return;
    const int b = i / C, c = i - (i / C) * C;
    int b2, dE = 0;
    if (a.system == kIsing) {
        b2 = b + c - 2;
    } else if (a.system == kPotts) {
        dE = c - 4;
        b2 = b + dE;
    } else {
        const int sidx = c / 5, k = c - 5 * (c / 5);
        dE = 4 * (k - 2);
        b2 = b - 1 + 2 * sidx;
    }
    uint32_t t = 0u;
    if (a.reach[b] && b2 >= 0 && b2 < a.B && a.reach[b2]) {
        double d = __dsub_rn(a.lnW[b2], a.lnW[b]);
        if (a.system == kMuma) d = __dsub_rn(d, __dmul_rn(a.beta, (double)dE));
        if (d >= 0.0) {
            t = kAlways;
        } else {
            const double scaled = __dmul_rn(dm_exp(d), 4294967296.0);
            t = (scaled >= 4294967296.0) ? kAlways : (uint32_t)floor(scaled);
        }
    }
    a.T[i] = t;
}

__global__ void k_thresholds(const UpdateArgs a) { thresholds_body(a, blockIdx.x * blockDim.x + threadIdx.x); }

__global__ void k_thresholds_batch(const UpdateArgs *__restrict__ arr)
{
    thresholds_body(arr[blockIdx.y], blockIdx.x * blockDim.x + threadIdx.x);
}

__global__ void k_advance(DevState *st, long long sweeps) { st->sweep_counter += (unsigned long long)sweeps; }

__global__ void k_advance_batch(DevState *const *states, const SpinSweepArgs *sys, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) states[i]->sweep_counter += (unsigned long long)sys[i].sweeps;  // each system's own count
}

__global__ void k_init_weights(const UpdateArgs a)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= a.B) return;
    const double v = a.reach[b] ? 0.0 : kNegInf;  // unreachable bins never carry weight
    a.lnW[b] = v;
    a.lnW_sampled[b] = v;
    a.G[b] = 0.0;
    a.lnR[b] = 0.0;
    a.H[b] = 0ull;
}

// Initial lattices from the INIT stream: word i%4 of Philox((i/4, 0, walker, 0)).
// Ising/MUMA: s = -1 (bit 1) iff the word's top bit is set; Potts: s = mulhi(u, q).
__global__ void k_init_spins(int system, int L, int q, int p, int pstride, uint32_t k0, uint32_t k1,
                             int walker_offset, uint32_t *lat, int32_t *bin)
{
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= p) return;
    const uint32_t wid = (uint32_t)(w + walker_offset);
    const int WR = (system == kPotts) ? potts_words_per_row(L) : ising_words_per_row(L);
    const int bits = (system == kPotts) ? 4 : 1;
    uint32_t *my = lat + w;
    uint4 u = make_uint4(0u, 0u, 0u, 0u);
    for (int y = 0; y < L; ++y) {
        for (int j = 0; j < WR; ++j) {
            uint32_t word = 0u;
            for (int x = j * 32 / bits; x < (j + 1) * 32 / bits && x < L; ++x) {
                const int i = y * L + x;
                if ((i & 3) == 0) u = philox4x32_10(make_uint4((uint32_t)(i / 4), 0u, wid, kTagInit), k0, k1);
                const uint32_t r = (i & 3) == 0 ? u.x : ((i & 3) == 1 ? u.y : ((i & 3) == 2 ? u.z : u.w));
                const uint32_t v = (system == kPotts) ? __umulhi(r, (uint32_t)q) : (r >> 31);
                word |= v << ((x * bits) & 31);
            }
            my[(y * WR + j) * pstride] = word;
        }
    }
    // bin of the initial state, from scratch
    int E = 0, nminus = 0;
    for (int y = 0; y < L; ++y)
        for (int x = 0; x < L; ++x) {
            const int yd = (y + 1) % L, xr = (x + 1) % L;
            if (system == kPotts) {
                auto nib = [&](int yy, int xx) {
                    return (my[(yy * WR + (4 * xx) / 32) * pstride] >> ((4 * xx) & 31)) & 15u;
                };
                const uint32_t s = nib(y, x);
                E -= (int)(s == nib(y, xr)) + (int)(s == nib(yd, x));
            } else {
                auto bt = [&](int yy, int xx) { return (my[(yy * WR + xx / 32) * pstride] >> (xx & 31)) & 1u; };
                const int s = bt(y, x) ? -1 : 1, sr = bt(y, xr) ? -1 : 1, sd = bt(yd, x) ? -1 : 1;
                E -= s * sr + s * sd;
                nminus += (s < 0);
            }
        }
    const int N = L * L;
    if (system == kIsing) bin[w] = (E + 2 * N) / 4;
    else if (system == kPotts) bin[w] = E + 2 * N;
    else bin[w] = N - nminus;  // (M + N)/2 = number of +1 spins
}

__global__ void k_unpack_spins(int system, int L, int p, int pstride, const uint32_t *lat, int8_t *out)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long N = (long long)L * L;
    if (idx >= (long long)p * N) return;
    const int w = (int)(idx / N), i = (int)(idx - (idx / N) * N);
    const int y = i / L, x = i - (i / L) * L;
    if (system == kPotts) {
        const int WR = potts_words_per_row(L);
        const uint32_t word = lat[(size_t)(y * WR + (4 * x) / 32) * pstride + w];
        out[idx] = (int8_t)((word >> ((4 * x) & 31)) & 15u);
    } else {
        const int WR = ising_words_per_row(L);
        const uint32_t word = lat[(size_t)(y * WR + x / 32) * pstride + w];
        out[idx] = ((word >> (x & 31)) & 1u) ? (int8_t)-1 : (int8_t)1;
    }
}

// Eq. (2) with O a function of the binned variable; ln Omega(b) = ln H(b) -
// ln W(b), W being the weights H was sampled with.  Fixed-order tree
// reductions, so repeated calls give identical results.
// One log and three exponentials a bin in binary64, of which an SM does two lanes a clock: 8193 bins
// on one SM took 214 us.  So a cluster of kReweightCtas blocks works as one block of 1024 threads
// would, thread t on bins t, t + 1024, ...: the partial results of all threads go to every block through
// distributed shared memory, and each makes the same tree of 1024 (the sums keep their order).
constexpr int kReweightCtas = 8, kReweightThreads = 128, kReweightAll = kReweightCtas * kReweightThreads;

template <class OP>
__device__ double reweight_reduce(double v, double *red, OP op)
{
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const int t = (int)cl.block_rank() * kReweightThreads + threadIdx.x;
    cl.sync();  // the last reduction has been read everywhere
    for (int r = 0; r < kReweightCtas; ++r) cl.map_shared_rank(red, r)[t] = v;
    cl.sync();
    for (int s = kReweightAll / 2; s > 0; s >>= 1) {
        for (int i = threadIdx.x; i < s; i += kReweightThreads) red[i] = op(red[i], red[i + s]);
        __syncthreads();
    }
    return red[0];
}

__global__ void __cluster_dims__(kReweightCtas, 1, 1) __launch_bounds__(kReweightThreads)
    k_reweight(const UpdateArgs a, double beta, double *out4, double *lnP)
{
    extern __shared__ double sx[];  // this block's values of x_b: bin t + 1024 i at 128 i + its thread
    __shared__ double red[kReweightAll];
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const int rank = (int)cl.block_rank(), tid = rank * kReweightThreads + threadIdx.x, bs = kReweightAll, B = a.B, N = a.N;
    auto own = [](int b) { return b / kReweightAll * kReweightThreads + b % kReweightThreads; };
    auto energy = [&](int b) {
        if (a.system == kPolymer) return a.e_lo + a.bin_w * (b + 0.5);
        return (a.system == kIsing) ? (double)(4 * b - 2 * N) : (double)(b - 2 * N);
    };
    auto plus = [](double x, double y) { return x + y; };
    auto larger = [](double x, double y) { return fmax(x, y); };
    const double NEG_INF = kNegInf;
    double m = NEG_INF;
    for (int b = tid; b < B; b += bs) {
        double x = NEG_INF;
        const unsigned long long h = a.H[b];
        if (a.reach[b] && h) {
            const double lnOmega = log((double)h) - a.lnW_sampled[b];
            x = (a.system == kMuma) ? lnOmega : lnOmega - beta * energy(b);
        }
        sx[own(b)] = x;
        m = fmax(m, x);
    }
    m = reweight_reduce(m, red, larger);
    double z = 0.0;
    for (int b = tid; b < B; b += bs)
        if (sx[own(b)] > NEG_INF) z += exp(sx[own(b)] - m);
    const double lse = m + log(reweight_reduce(z, red, plus));
    double a1 = 0.0, a2 = 0.0;
    for (int b = tid; b < B; b += bs) {
        const double x = sx[own(b)];
        const double lp = (x > NEG_INF) ? x - lse : NEG_INF;
        if (lnP) lnP[b] = lp;
        if (x > NEG_INF) {
            const double P = exp(lp);
            const double v = (a.system == kMuma) ? fabs((double)(2 * b - N)) : energy(b);
            a1 += P * v;
            a2 += P * v * v;
        }
    }
    a1 = reweight_reduce(a1, red, plus);
    a2 = reweight_reduce(a2, red, plus);
    // polymer: log-sum-exp of ln Omega itself (the normalisation of ln Z)
    double lnNorm = 0.0;
    if (a.system == kPolymer) {
        double m2 = NEG_INF;
        for (int b = tid; b < B; b += bs)
            if (sx[own(b)] > NEG_INF) m2 = fmax(m2, sx[own(b)] + beta * energy(b));
        m2 = reweight_reduce(m2, red, larger);
        double z2 = 0.0;
        for (int b = tid; b < B; b += bs)
            if (sx[own(b)] > NEG_INF) z2 += exp(sx[own(b)] + beta * energy(b) - m2);
        lnNorm = m2 + log(reweight_reduce(z2, red, plus));
    }
    auto x_of = [&](int b) -> double { return cl.map_shared_rank(sx, b % kReweightAll / kReweightThreads)[own(b)]; };
    if (tid == 0) {
        if (a.system == kPolymer) {
            out4[0] = a1;
            out4[1] = a2;
            out4[2] = beta * beta * (a2 - a1 * a1) / N;
            out4[3] = lse - lnNorm;
        } else if (a.system == kMuma) {
            out4[0] = a1 / N;
            out4[1] = a2 / ((double)N * N);
            out4[2] = a.beta * N * (out4[1] - out4[0] * out4[0]);
            const int b0 = N / 2, bm = N;
            out4[3] = (x_of(b0) > NEG_INF && x_of(bm) > NEG_INF) ? x_of(b0) - x_of(bm) : __longlong_as_double(0x7ff8000000000000LL);
        } else {
            out4[0] = a1;
            out4[1] = a2;
            out4[2] = beta * beta * (a2 - a1 * a1) / N;
            const double g0 = (a.system == kIsing) ? 2.0 : (double)a.q;
            if (x_of(0) > NEG_INF) out4[3] = lse + log(g0) - (x_of(0) - beta * (double)(2 * N));
            else out4[3] = __longlong_as_double(0x7ff8000000000000LL);
        }
    }
    cl.sync();  // no block leaves while its shared memory may be read
}

__global__ void k_det_math(int fn, const double *in, double *out, long long n)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = fn == 0 ? dm_exp(in[i]) : dm_log(in[i]);
}

// ---------------------------------------------------------------------------
cudaError_t launch_det_math(int fn, const double *in, double *out, long long n, cudaStream_t s)
{
    k_det_math<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(fn, in, out, n);
    return cudaGetLastError();
}

// Launch shape of the recursion: its blocks, and shared memory for the last block's terms.
static int recursion_grid(int nreach) { return nreach > kRecPairs ? (nreach - 1 + kRecPairs - 1) / kRecPairs : 1; }
static size_t recursion_smem(int nreach) { return (size_t)nreach * sizeof(double); }

size_t update_scratch_bytes(int bins)
{
    return sizeof(unsigned long long) * (1 + 3 * (size_t)recursion_grid(bins) + (size_t)bins);
}

cudaError_t launch_merge(const UpdateArgs &a, cudaStream_t s)
{
    k_merge<<<(a.B + kMergeBins - 1) / kMergeBins, kMergeBins * kMergeRows, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_recursion(const UpdateArgs &a, cudaStream_t s)
{
    const size_t smem = recursion_smem(a.nreach);
    if (smem > 40u * 1024u) {  // above what a launch may ask for without the attribute
        const cudaError_t e = allow_dynamic_smem(k_recursion, recursion_smem(kPolyMaxBins));
        if (e != cudaSuccess) return e;
    }
    k_recursion<<<recursion_grid(a.nreach), kRecThreads, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_thresholds(const UpdateArgs &a, cudaStream_t s)
{
    const int n = a.B * num_cols(a.system);
    k_thresholds<<<(n + 255) / 256, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_merge_batch(const UpdateArgs *d_args, int n, int max_bins, cudaStream_t s)
{
    k_merge_batch<<<dim3((max_bins + kMergeBins - 1) / kMergeBins, n), kMergeBins * kMergeRows, 0, s>>>(d_args);
    return cudaGetLastError();
}

cudaError_t launch_recursion_batch(const UpdateArgs *d_args, int n, int max_nreach, cudaStream_t s)
{
    k_recursion_batch<<<dim3(recursion_grid(max_nreach), n), kRecThreads, recursion_smem(max_nreach), s>>>(d_args);
    return cudaGetLastError();
}

cudaError_t prepare_recursion_batch()
{
    return allow_dynamic_smem(k_recursion_batch, recursion_smem(kPolyMaxBins));  // (no system has more bins)
}

cudaError_t launch_thresholds_batch(const UpdateArgs *d_args, int n, int max_cells, cudaStream_t s)
{
    k_thresholds_batch<<<dim3((max_cells + 255) / 256, n), 256, 0, s>>>(d_args);
    return cudaGetLastError();
}

cudaError_t launch_advance_batch(DevState *const *d_states, const SpinSweepArgs *d_sys, int n, cudaStream_t s)
{
    k_advance_batch<<<(n + 127) / 128, 128, 0, s>>>(d_states, d_sys, n);
    return cudaGetLastError();
}

cudaError_t launch_advance(DevState *st, int64_t sweeps, cudaStream_t s)
{
    k_advance<<<1, 1, 0, s>>>(st, (long long)sweeps);
    return cudaGetLastError();
}

cudaError_t launch_init_lnW(const UpdateArgs &a, cudaStream_t s)
{
    k_init_weights<<<(a.B + 255) / 256, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_init_spins(int system, int L, int q, int p, int pstride, uint32_t key0, uint32_t key1,
                              int walker_offset, uint32_t *lattice, int32_t *bin, cudaStream_t s)
{
    k_init_spins<<<(p + 127) / 128, 128, 0, s>>>(system, L, q, p, pstride, key0, key1, walker_offset, lattice, bin);
    return cudaGetLastError();
}

cudaError_t launch_unpack_spins(int system, int L, int p, int pstride, const uint32_t *lattice, int8_t *out,
                                cudaStream_t s)
{
    const long long n = (long long)p * L * L;
    k_unpack_spins<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(system, L, p, pstride, lattice, out);
    return cudaGetLastError();
}

cudaError_t launch_reweight(const UpdateArgs &a, double beta, double *out4, double *lnP, cudaStream_t s)
{
    // (at most 12288 bins: 12 KB a block, within what a launch may ask for without an attribute)
    const size_t smem = (size_t)((a.B + kReweightAll - 1) / kReweightAll) * kReweightThreads * sizeof(double);
    k_reweight<<<kReweightCtas, kReweightThreads, smem, s>>>(a, beta, out4, lnP);
    return cudaGetLastError();
}

// Eq. (2) with per-bin sums of an Ising run (samples n, sum |M|, sum M^2 per bin):
// <O>_beta = sum_b S_O(b) e^{x_b} / sum_b n(b) e^{x_b}, x_b = -beta E_b - ln W(b),
// E_b = 4b - 2N, W the weights the sums were sampled with.  One block; out =
// {<|M|>/N, <M^2>/N^2, beta N (<M^2>/N^2 - (<|M|>/N)^2)}, NaN without samples.
__global__ void __launch_bounds__(256) k_reweight_obs(const unsigned long long *__restrict__ sums,
                                                      const double *__restrict__ lnW, int B, int N, double beta,
                                                      double *out)
{
    __shared__ double red[4][256];
    const int t = threadIdx.x;
    double m = -INFINITY;
    for (int b = t; b < B; b += 256)
        if (sums[3 * b] > 0ull) m = fmax(m, -beta * (double)(4 * b - 2 * N) - lnW[b]);
    red[0][t] = m;
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
        if (t < o) red[0][t] = fmax(red[0][t], red[0][t + o]);
        __syncthreads();
    }
    const double mx = red[0][0];
    __syncthreads();
    double z = 0.0, a1 = 0.0, a2 = 0.0;
    if (mx > -INFINITY) {
        for (int b = t; b < B; b += 256) {
            if (sums[3 * b] == 0ull) continue;
            const double f = exp(-beta * (double)(4 * b - 2 * N) - lnW[b] - mx);
            z += f * (double)sums[3 * b];
            a1 += f * (double)sums[3 * b + 1];
            a2 += f * (double)sums[3 * b + 2];
        }
    }
    red[1][t] = z;
    red[2][t] = a1;
    red[3][t] = a2;
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
        if (t < o) {
            red[1][t] += red[1][t + o];
            red[2][t] += red[2][t + o];
            red[3][t] += red[3][t + o];
        }
        __syncthreads();
    }
    if (t == 0) {
        if (!(mx > -INFINITY)) {
            out[0] = out[1] = out[2] = NAN;
        } else {
            const double m1 = red[2][0] / red[1][0] / N, m2 = red[3][0] / red[1][0] / ((double)N * N);
            out[0] = m1;
            out[1] = m2;
            out[2] = beta * N * (m2 - m1 * m1);
        }
    }
}

cudaError_t launch_reweight_obs(const unsigned long long *sums, const double *lnW_sampled, int B, int N, double beta,
                                double *out3, cudaStream_t s)
{
    k_reweight_obs<<<1, 256, 0, s>>>(sums, lnW_sampled, B, N, beta, out3);
    return cudaGetLastError();
}

}  // namespace muca
