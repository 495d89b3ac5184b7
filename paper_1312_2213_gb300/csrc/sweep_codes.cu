// sweep_codes.cu -- producer/consumer form with precomputed site codes (Ising,
// MUMA and Potts).
#include "muca_device.cuh"
#include "muca_internal.h"
#include "muca_checks.cuh"
#include "sweep_common.cuh"

namespace muca {

// ---------------------------------------------------------------------------
// Producer/consumer form with precomputed site codes (Ising and MUMA).
// Shared memory holds the thresholds and the histogram counters (column-major, see
// below).  The producer warps write, per row, the walkers' random
// words (clamped, see clamp_words), their old row and, for every site, two column
// bytes holding 4 c: c0 for "left
// neighbour as it was" and c1 for "left neighbour flipped", both without the up
// neighbour (which only the consumer knows: the row above is final only after
// the consumer has swept it) and, for the last site, without its right
// neighbour (site 0 of the same row).  Four sites are handled at once with
// bytewise arithmetic on the row's anti-aligned bits.  The consumer subtracts the up term
// (and the right term of the last site), makes addresses and bin moves from the bytes
// with byte dot products, and runs a speculative chain: both candidate thresholds of a
// site are loaded while the site before it is decided.  (A variant that stored
// (threshold, next-row) pairs to save the moves was slower: its 8-byte random loads
// doubled the bank conflicts on the critical chain.)
// Bound by that chain: 39 cycles a site, of which two shared-memory loads and their
// selects and compares; the producers alone need 36 (L = 32).  Cycles a site, 8192
// walkers spread over all bins, before / after the column-major table, the joined
// rows and the shorter Philox rounds: Ising L = 32 50.7 / 42.6, MUMA 50.3 / 43.5;
// Ising L = 64 (2048 walkers) 50.9 / 42.9, L = 16 59.4 / 48.6, L = 8 (64) 74.5 / 60.0.
template <int L, int WR>
__device__ __forceinline__ uint32_t row_bit(const uint32_t (&r)[WR], int x)
{
    return (r[x >> 5] >> (x & 31)) & 1u;
}

// Sites x..x+3 (x % 4 == 0) of a packed row as bytes 4 [bit].
template <int WR>
__device__ __forceinline__ uint32_t nibble_fours(const uint32_t (&r)[WR], int x)
{
    return (((r[x >> 5] >> (x & 31)) & 15u) * (0x00204081u << 2)) & 0x04040404u;
}

// Code-form table of Ising and MUMA: column-major, T[c][b] at word c NB + b, the counters of the bins
// behind the C columns.  A code byte is then worth NB bytes a unit of 4 c, and one dp2a makes a
// threshold's address from the packed codes of four sites and the walker's bin address (NB in the
// 16-bit half that meets the site's byte), where rows of C + 1 words a bin took an extraction and an
// addition, and a multiplication for the bin's move.
// Ising codes travel as 4 c + 0x78; the consumer flips the top bits behind the up neighbour's term,
// which leaves the signed byte 4 (c - 2): the bin's move in bytes, added by one dp4a.
template <int SYS>
constexpr uint32_t kCodeBias = SYS == kIsing ? 0x78787878u : 0u;

// The random words handed to a code-form consumer are min(u, 2^32 - 2).  With
// that clamp the acceptance "T == always or u < T" becomes the single compare
// u' < T: for T = 2^32 - 1 (always) every u' is below it, and for any smaller T
// the only changed word, 2^32 - 1, is rejected before and after.
__device__ __forceinline__ uint4 clamp_words(uint4 u)
{
    u.x = min(u.x, 0xFFFFFFFEu);
    u.y = min(u.y, 0xFFFFFFFEu);
    u.z = min(u.z, 0xFFFFFFFEu);
    u.w = min(u.w, 0xFFFFFFFEu);
    return u;
}

// Producer warps per consumer warp in the Ising/MUMA code form.  One Philox4x32-10 block costs a
// scheduler 88 cycles of multiply and logic throughput and a single warp alone about 134
// cycles, so one producer cannot keep up with its consumer; the row's
// site groups are split over the producers (on other schedulers), which arrive
// together on the row's FULL barrier.
constexpr int kCodeProducers = 2;

// Warp roles of a code-form block of one or two walker warps (ncw).  The block
// has 4 ncw warps, laid out so that, with warp w issuing from scheduler w mod 4,
// every consumer has a scheduler to itself (its serial chain is what sets the
// pace) and the two producers of a consumer share another one:
//   ncw = 1: [C0, idle, P0.0, P0.1]
//   ncw = 2: [C0, C1, P0.0, P1.0, idle, idle, P0.1, P1.1]   (Pc.k: part k for consumer c)
// Idle warps only take part in the block-wide barriers of the histogram flush.
enum { kRoleConsumer = 0, kRoleProducer = 1, kRoleIdle = 2 };
struct CodeRole {
    int kind, pair, part;
};
__device__ __forceinline__ CodeRole code_role(int warp, int ncw)
{
    if (ncw == 1) {
        if (warp == 0) return CodeRole{kRoleConsumer, 0, 0};
        if (warp == 1) return CodeRole{kRoleIdle, 0, 0};
        return CodeRole{kRoleProducer, 0, warp - 2};
    }
    const int sch = warp & 3, grp = warp >> 2;
    if (sch < 2) return grp == 0 ? CodeRole{kRoleConsumer, sch, 0} : CodeRole{kRoleIdle, 0, 0};
    return CodeRole{kRoleProducer, sch - 2, grp};
}
constexpr int kCodeWarpsPerWalkerWarp = 4;

// Lanes of a consumer warp that run the protocol (and arrive on EMPTY) when `left` walkers are left
// for it: those with a walker, or all of a warp that has none.  (Lanes without a walker beside others
// with one took a loop of their own, which the warp then ran after the walkers': 10 % at p = 1000.)
__device__ __forceinline__ unsigned code_consumer_lanes(int left) { return left > 0 && left < 32 ? (unsigned)left : 32u; }

// A lane whose wait gives up (`bad`) takes no further part in the launch's hand-overs: it writes no slot,
// reads none and arrives nowhere, so its partners' waits run out as well, within the same bound, and no
// lane ever decides on a slot that is being rewritten (its codes need not fit its lattice and bin, which
// could walk off the table).

// The producer's rows of nsw sweeps.
template <int SYS, int L, int PART>
__device__ __forceinline__ void produce_tn(int64_t nsw, uint32_t g0, uint32_t wid, const uint32_t (&rk)[20],
                                           const uint32_t *__restrict__ lat, int ps, uint4 *ring_u, uint2 *ring_c,
                                           uint32_t *ring_r, unsigned long long *full, unsigned long long *empty, int &k,
                                           bool &bad, int drop_k)
{
    constexpr int WR = ising_words_per_row(L);
    constexpr int G = L / 4;
    constexpr size_t SU = (size_t)G * 32, SC = (size_t)G * 32, SR = (size_t)WR * 32;
    // Rolling rows: o = row y (old), d = row y+1 (old; row 0 final for y = L-1), nn = row y+2
    // prefetched one row ahead, on into the next sweep.  The producer runs at most kRing rows ahead of
    // the consumer and L >= 2 kRing, so every row it reads has its value for its sweep (rows y, y+1, y+2
    // not yet swept; rows 0 and 1 already swept when they are read behind rows L-2 and L-1).  At the
    // first sweep nothing is in flight.
    uint32_t o[WR], d[WR], nn[WR];
#pragma unroll
    for (int j = 0; j < WR; ++j) {
        o[j] = lat[j * ps];
        d[j] = lat[(WR + j) * ps];
    }
#pragma unroll 1
    for (int64_t sw = 0; sw < nsw; ++sw) {
        const PhiloxLane pl = philox_lane(g0 + (uint32_t)sw, wid, rk);
#pragma unroll 1
        for (int y = 0; y < L; ++y) {
            const int slot = k % kRing;
            // the row's random words are made while the answer about the slot is under way
            constexpr int g_lo = PART * G / kCodeProducers, g_hi = (PART + 1) * G / kCodeProducers, NG = g_hi - g_lo;
            bool free_slot = mbar_try(&empty[slot], (unsigned)(((k / kRing) & 1) ^ 1));
            uint4 words[NG];
            constexpr int PB = NG < 4 ? NG : 4;
#pragma unroll
            for (int i = 0; i + PB <= NG; i += PB) {
                uint4 c[PB];
                philox4x32_10_groups<PB>((uint32_t)(y * G + g_lo + i), pl, rk, c);
#pragma unroll
                for (int e = 0; e < PB; ++e) words[i + e] = clamp_words(c[e]);
            }
            for (int i = NG / PB * PB; i < NG; ++i) words[i] = clamp_words(philox4x32_10_group((uint32_t)(y * G + g_lo + i), pl, rk));
            if (!free_slot && !mbar_wait(&empty[slot], (unsigned)(((k / kRing) & 1) ^ 1))) {
                bad = true;
                return;
            }
            const int y2 = (y + 2 < L) ? y + 2 : y + 2 - L;
#pragma unroll
            for (int j = 0; j < WR; ++j) nn[j] = lat[(y2 * WR + j) * ps];
            uint4 *wu = ring_u + slot * SU;
            uint2 *wc = ring_c + slot * SC;
            uint32_t *wr = ring_r + slot * SR;
            if (PART == 0) {
#pragma unroll
                for (int j = 0; j < WR; ++j) wr[j * 32] = o[j];
            }
            // anti-aligned neighbours of the whole row at once: left, right (none for the last site: the
            // consumer adds it) and down
            uint32_t la[WR], ra[WR], da[WR];
#pragma unroll
            for (int j = 0; j < WR; ++j) {
                constexpr int last = (L - 1) & 31;  // bit of the row's last site in its word
                const uint32_t from_left = (j > 0) ? o[j - 1] >> 31 : (o[WR - 1] >> last) & 1u;
                const uint32_t from_right = (j + 1 < WR) ? o[(j + 1) % WR] << 31 : o[j] & (1u << last);
                la[j] = o[j] ^ ((o[j] << 1) | from_left);
                ra[j] = o[j] ^ ((o[j] >> 1) | from_right);
                da[j] = o[j] ^ d[j];
            }
#pragma unroll
            for (int gq = g_lo; gq < g_hi; ++gq) {
                wu[gq * 32] = words[gq - g_lo];
                // per byte 4 [anti-aligned], and from them the columns as byte offsets 4 c: 4 (4 - count)
                // without the up neighbour, for the left neighbour as it was (k0) and flipped (k1)
                const int x = 4 * gq;
                const uint32_t A = nibble_fours<WR>(la, x), BD = nibble_fours<WR>(ra, x) + nibble_fours<WR>(da, x);
                uint32_t k0 = 0x10101010u - A - BD, k1 = 0x0C0C0C0Cu + A - BD;
                // the row's first site does not see the site decided before it: one code for both outcomes
                if (gq == 0) k1 = __byte_perm(k0, k1, 0x7650u);
                if (SYS == kMuma) {
                    const uint32_t s5 = nibble_fours<WR>(o, x) * 5u;
                    k0 += s5;
                    k1 += s5;
                }
                wc[gq * 32] = make_uint2(k0 + kCodeBias<SYS>, k1 + kCodeBias<SYS>);
            }
            if (k != drop_k) mbar_arrive(&full[slot]);
            ++k;
#pragma unroll
            for (int j = 0; j < WR; ++j) {
                o[j] = d[j];
                d[j] = nn[j];
            }
        }
    }
}

// The consumer's rows of nsw sweeps, one after the other without a break: the next row's hand-over,
// its first codes and both candidates of its first threshold are taken up while the last four sites of
// a row are decided (with a fresh start at every row a row cost 270 cycles beside 39 a site).
template <int SYS, int L, int RECORD>
__device__ __forceinline__ void consume_tn(int64_t nsw, uint32_t *__restrict__ lat, int ps, int &bR,
                                           uint32_t *__restrict__ sTH, const uint4 *__restrict__ ring_u,
                                           const uint2 *__restrict__ ring_c, const uint32_t *__restrict__ ring_r,
                                           unsigned long long *full, unsigned long long *empty, int &k, bool &bad,
                                           unsigned long long *obs, unsigned long long &nacc, int r_lo, int r_hi,
                                           int &tst, unsigned &ev)
{
    constexpr int WR = ising_words_per_row(L);
    constexpr int C = (SYS == kMuma) ? 10 : 5;
    constexpr int NB = L * L + 1;
    constexpr int G = L / 4;
    constexpr size_t SU = (size_t)G * 32, SC = (size_t)G * 32, SR = (size_t)WR * 32;
    // The chain works in 32-bit shared-window byte addresses: bB = table base + 4 bin.
    const int sbase = (int)__cvta_generic_to_shared(sTH);
    constexpr int TOFF = (SYS == kMuma) ? 0 : 8 * NB;  // Ising: codes count from column 2
    auto th = [sbase](int addr) -> uint32_t {
        uint32_t v;
        asm("ld.shared.u32 %0, [%1 + %2];" : "=r"(v) : "r"(checked_addr(addr + TOFF, sbase) - TOFF), "n"(TOFF));
        return v;
    };
    // bB + NB x byte i of w (signed for Ising)
    auto at = [](uint32_t w, int i, int b) -> int {
        const int n = NB << (16 * (i & 1));
        if (SYS == kMuma) return (int)(i < 2 ? __dp2a_lo((unsigned)n, w, (unsigned)b) : __dp2a_hi((unsigned)n, w, (unsigned)b));
        return i < 2 ? __dp2a_lo(n, (int)w, b) : __dp2a_hi(n, (int)w, b);
    };
    // codes of four sites with the up neighbour's term (bytes 4 [anti-aligned])
    auto settle = [](uint2 c, uint32_t up4) -> uint2 {
        constexpr uint32_t flip = (SYS == kMuma) ? 0u : 0x80808080u;
        return make_uint2((c.x - up4) ^ flip, (c.y - up4) ^ flip);
    };

    // A row is decided in units of U sites (one word): the whole row up to L = 32, halves at L = 64,
    // where 64 unrolled sites stalled on instruction fetch (48.0 cycles a site, 42.9 in halves).
    constexpr int U = (L % 32 == 0) ? 32 : L, NU = L / U, WU = (U + 31) / 32;
    const int k_end = k + (int)(nsw * L);
    int bB = sbase + 4 * bR;
    uint32_t up[WR], cur[WU], nxt[WU];
    uint2 cdn = make_uint2(0u, 0u);
    uint32_t T0 = 0u, T1 = 0u;
    bool accP = false;  // the site decided before
    if (!mbar_wait(&full[k % kRing], (unsigned)((k / kRing) & 1))) bad = true;
    if (!bad) {
        const int slot = k % kRing;
#pragma unroll
        for (int j = 0; j < WR; ++j) up[j] = lat[((L - 1) * WR + j) * ps];
#pragma unroll
        for (int j = 0; j < WU; ++j) nxt[j] = ring_r[slot * SR + j * 32];
        const uint32_t ua0[1] = {up[0] ^ nxt[0]};
        cdn = settle(ring_c[slot * SC], nibble_fours<1>(ua0, 0));
        T0 = T1 = th(at(cdn.x, 0, bB));
    }
#pragma unroll 1
    for (int64_t sw = 0; sw < nsw && !bad; ++sw) {
        unsigned na = 0;
        // two rows an iteration from L = 32 up (2-4 % there; L = 16 rows are short enough that the
        // larger body costs more than the loop overhead it saves)
        constexpr int kRowUnroll = (L >= 32) ? 2 : 1;
        uint32_t s0 = 0u;  // site 0 of the row, decided
#pragma unroll kRowUnroll
        for (int yu = 0; yu < L * NU; ++yu) {
            const int y = yu / NU, h = yu % NU;  // row and unit (constants of the unrolled pair at NU = 2)
            const bool row_end = h == NU - 1;
            const int slot = k % kRing, slot_n = row_end ? (k + 1) % kRing : slot;
            const uint4 *ru = ring_u + slot * SU + (size_t)h * (U / 4) * 32;
            const uint2 *rc = ring_c + slot * SC + (size_t)h * (U / 4) * 32;
            uint32_t ua[WU], old[WU];
#pragma unroll
            for (int j = 0; j < WU; ++j) {
                old[j] = cur[j] = nxt[j];
                ua[j] = up[h * WU + j] ^ cur[j];  // up neighbour anti-aligned
            }
            const uint32_t sLast = row_bit<U, WU>(cur, U - 1);
            uint2 cd = cdn, cnext = cdn;
            uint4 u = make_uint4(0u, 0u, 0u, 0u);
            uint32_t mv = 0u;   // MUMA: the four sites' moves in bytes, +-4
            bool next = false;  // the next row is there
#pragma unroll
            for (int x = 0; x < U; ++x) {
                const int j4 = x & 3;
                if (j4 == 0) {
                    u = ru[(x / 4) * 32];
                    cd = cdn;
                    // s = -1 (bit set): one bin up, else one down; 0xFC = -4, 0xFC ^ 0xF8 = 4
                    if (SYS == kMuma) mv = (nibble_fours<WU>(old, x) * 0x3Eu) ^ 0xFCFCFCFCu;
                    if (x + 4 < U) cdn = settle(rc[(x / 4 + 1) * 32], nibble_fours<WU>(ua, x + 4));
                    if (x + 8 == U && row_end) next = mbar_try(&full[slot_n], (unsigned)(((k + 1) / kRing) & 1));
                    if (x + 4 == U) {
                        // the next unit; behind the last row (or a wait that gave up) an earlier row's codes
                        // are read and not used
                        if (row_end && !next && !(sw + 1 == nsw && y == L - 1))
                            bad = !mbar_wait(&full[slot_n], (unsigned)(((k + 1) / kRing) & 1));
                        const int hn = row_end ? 0 : h + 1;
#pragma unroll
                        for (int j = 0; j < WU; ++j) nxt[j] = ring_r[slot_n * SR + (hn * WU + j) * 32];
                        cnext = ring_c[slot_n * SC + (size_t)hn * (U / 4) * 32];
                    }
                }
                if (h == 0 && x == 4) s0 = row_bit<U, WU>(cur, 0);
                if (row_end && x == U - 2) {
                    // the last site's right neighbour is site 0 of this row, final by now (its code is the
                    // top byte, so nothing is borrowed from)
                    const uint32_t ra = (s0 ^ sLast) << 26;
                    cd.x -= ra;
                    cd.y -= ra;
                }
                if (x == U - 1) {
                    // (the first four sites of this row's first unit, or of the row above's next unit)
                    const uint32_t ua0[1] = {((NU == 1) ? cur[0] : up[row_end ? 0 : h + 1]) ^ nxt[0]};
                    cdn = settle(cnext, nibble_fours<1>(ua0, 0));
                }
                const uint32_t uw = word_of(u, j4);
                // the bin's address if this site is accepted
                const int bA = (SYS == kMuma) ? __dp4a((int)mv, 1 << (8 * j4), bB)
                                              : __dp4a((int)(accP ? cd.y : cd.x), 1 << (8 * j4), bB);
                const uint32_t T = accP ? T1 : T0;
                // both candidates of the next site's threshold (behind the last site: of the next row's
                // first, whose two codes are the same)
                const int jn = (x + 1) & 3;
                T0 = th(at((jn == 0) ? cdn.x : cd.x, jn, bB));
                T1 = th(at((jn == 0) ? cdn.y : cd.y, jn, bA));
                const bool acc = uw < T;  // the producer's clamp makes this "always or u < T"
                if (acc) cur[x >> 5] ^= 1u << (x & 31);
                bB = acc ? bA : bB;
                if (RECORD == 0)
                    asm volatile("red.shared.add.u32 [%0 + %2], %1;" ::"r"(checked_addr(bB + 4 * C * NB, sbase) - 4 * C * NB),
                                 "r"(1u), "n"(4 * C * NB)
                                 : "memory");
                accP = acc;
            }
#pragma unroll
            for (int j = 0; j < WU; ++j) {
                lat[(y * WR + h * WU + j) * ps] = cur[j];
                na += (unsigned)__popc(old[j] ^ cur[j]);
                up[h * WU + j] = cur[j];
            }
            if (row_end) {
                mbar_arrive(&empty[slot]);  // after the row is stored: the producer reads it later
                ++k;
                if (bad) break;
            }
        }
        nacc += na;
        if (bad) break;
        const int bin = (bB - sbase) / 4;
        if (RECORD == 1) atomicAdd(&sTH[checked_word(bin + C * NB)], 1u);
        if (SYS == kIsing && obs) {
            int pc = 0;  // -1 spins of the final rows
#pragma unroll 1
            for (int j = 0; j < L * WR; ++j) pc += __popc(lat[j * ps]);
            record_observables(obs, bin, L * L, pc);
        }
        tunnel_step(bin, r_lo, r_hi, tst, ev);
    }
    k = k_end;
    bR = (bB - sbase) / 4;
}

__host__ __device__ constexpr size_t tn_ring_bytes(int L)
{
    return (size_t)kRing * ((size_t)(L / 4) * 32 * 16 + (size_t)(L / 4) * 32 * 8 + (size_t)((L + 31) / 32) * 32 * 4);
}

// put(i, T[i]) for i < n by the whole block, eight loads a thread in flight (one after the other they
// took an L2 round trip each: 46,000 thresholds of q-Potts at L = 48 by 256 threads).
template <class PUT>
__device__ __forceinline__ void stage_table(const uint32_t *__restrict__ T, int n, PUT put)
{
    constexpr int U = 8;
    int i = threadIdx.x;
    for (; i + (U - 1) * (int)blockDim.x < n; i += U * blockDim.x) {
        uint32_t t[U];
#pragma unroll
        for (int e = 0; e < U; ++e) t[e] = T[i + e * (int)blockDim.x];
#pragma unroll
        for (int e = 0; e < U; ++e) put(i + e * (int)blockDim.x, t[e]);
    }
    for (; i < n; i += blockDim.x) put(i, T[i]);
}

template <int SYS, int L>
__device__ __forceinline__ void sweep_block_tn(const SpinSweepArgs &a, int w0, int slot_id, uint32_t *smem)
{
    constexpr int C = num_cols(SYS);
    constexpr int NB = L * L + 1;
    constexpr int G = L / 4;
    constexpr int NP = kCodeProducers;
    const int ncw = blockDim.x / (32 * kCodeWarpsPerWalkerWarp);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const CodeRole role = code_role(warp, ncw);
    const bool producer = role.kind == kRoleProducer, consumer = role.kind == kRoleConsumer;
    const int pair = role.pair, part = role.part;
    int drop_k = (blockIdx.x == 0 && producer && pair == 0 && part == 0) ? a.debug_drop_row : -1;
    uint32_t *sTH = smem;
    const size_t th_bytes = ((size_t)NB * (C + 1) * 4 + 15) / 16 * 16;
    char *rbase = (char *)smem + th_bytes + (size_t)pair * tn_ring_bytes(L);
    uint4 *ring_u = (uint4 *)rbase + lane;
    uint2 *ring_c = (uint2 *)(rbase + (size_t)kRing * G * 32 * 16) + lane;
    uint32_t *ring_r = (uint32_t *)(rbase + (size_t)kRing * (G * 32 * 16 + G * 32 * 8)) + lane;
    unsigned long long *bars = (unsigned long long *)((char *)smem + th_bytes + (size_t)ncw * tn_ring_bytes(L));
    unsigned long long *full = bars + (size_t)pair * 2 * kRing, *empty = full + kRing;

    const int tid = threadIdx.x;
    stage_table(a.T, NB * C, [&](int i, uint32_t t) {
        const int b = i / C, c = i - (i / C) * C;
        sTH[c * NB + b] = t;
    });
    for (int b = tid; b < NB; b += blockDim.x) sTH[C * NB + b] = 0u;
    // the rings' codes start on a middle column, so that codes read ahead of a row that never came
    // (a wait that gave up, the end of the last sweep) still address the table
    for (int i = tid; i < ncw * kRing * G * 32; i += blockDim.x) {
        const int pr = i / (kRing * G * 32);
        ((uint2 *)((char *)smem + th_bytes + (size_t)pr * tn_ring_bytes(L) + (size_t)kRing * G * 32 * 16))[i - pr * kRing * G * 32] =
            make_uint2(0x08080808u + kCodeBias<SYS>, 0x08080808u + kCodeBias<SYS>);
    }
    if (tid == 0)  // per pair: FULL[kRing] (NP producer warps arrive), EMPTY[kRing] (the consumer)
        for (int i = 0; i < ncw * 2 * kRing; ++i)
            mbar_init(bars + i, ((i / kRing) % 2 == 0) ? 32 * NP : code_consumer_lanes(a.p - w0 - 32 * (i / (2 * kRing))));
    set_block_spin_limit(a.spin_limit);
    checks_begin(NB * (C + 1), a.debug_check);
    __syncthreads();

    const int w = w0 + pair * 32 + lane;
    const bool active = w < a.p;
    const bool some = w - lane < a.p;  // this warp has walkers
    const uint32_t wid = (uint32_t)(w + a.walker_offset);
    const uint32_t g0 = (uint32_t)a.state->sweep_counter;
    uint32_t *lat = a.lattice + (active ? w : 0);
    int bR = active ? a.bin[w] : 0;
    unsigned long long *Hb = a.Hpart + (size_t)slot_id * NB;
    int k = 0;
    bool bad = false;
    const int r_lo = a.bin_lo, r_hi = a.bin_hi;
    int tst = (consumer && active && a.tun) ? a.tun[w] : 0;
    unsigned ev = 0;
    unsigned long long nacc = 0;
    for (int64_t s0 = 0; s0 < a.sweeps; s0 += a.flush_every) {
        const int64_t nsw = (a.sweeps < s0 + a.flush_every) ? a.sweeps - s0 : (int64_t)a.flush_every;
        const uint32_t g = g0 + (uint32_t)s0;
        if (bad) {  // (a wait of this lane gave up: see code_consumer_lanes)
        } else if (producer) {
            if (part == 0)
                produce_tn<SYS, L, 0>(nsw, g, wid, a.rk, lat, a.pstride, ring_u, ring_c, ring_r, full, empty, k, bad, drop_k);
            else
                produce_tn<SYS, L, 1>(nsw, g, wid, a.rk, lat, a.pstride, ring_u, ring_c, ring_r, full, empty, k, bad, -1);
        } else if (consumer && !some) {  // a consumer warp with no walkers keeps the barrier protocol
#pragma unroll 1
            for (int64_t r = 0; r < nsw * L; ++r) {
                const int slot = k % kRing;
                if (!mbar_wait(&full[slot], (unsigned)((k / kRing) & 1))) {
                    bad = true;
                    break;
                }
                mbar_arrive(&empty[slot]);
                ++k;
            }
        } else if (consumer && active) {
            if (a.record == 0)
                consume_tn<SYS, L, 0>(nsw, lat, a.pstride, bR, sTH, ring_u, ring_c, ring_r, full, empty, k, bad,
                                      a.obs, nacc, r_lo, r_hi, tst, ev);
            else
                consume_tn<SYS, L, 1>(nsw, lat, a.pstride, bR, sTH, ring_u, ring_c, ring_r, full, empty, k, bad,
                                      a.obs, nacc, r_lo, r_hi, tst, ev);
        }
        __syncthreads();
        for (int b = tid; b < NB; b += blockDim.x) {
            const uint32_t c = sTH[C * NB + b];
            if (c) {
                Hb[b] += c;
                sTH[C * NB + b] = 0u;
            }
        }
        rebase_rows(k, drop_k, kRing);
        __syncthreads();
    }
    if (bad) atomicOr(const_cast<int *>(&a.state->err), 1);
    if (consumer && active) {
        a.bin[w] = bR;
        if (a.tun) a.tun[w] = (uint8_t)tst;
    }
    flush_metrics(a.metrics, nacc, ev);
    checks_end(a.state);
}

// PER_SM: blocks of 64 walkers (256 threads) an SM is to hold; 1 leaves the registers to the compiler.
template <int SYS, int L, int PER_SM>
__global__ void __launch_bounds__(PER_SM > 1 ? 256 : kMaxSweepBlock, PER_SM) k_sweep_spin_tn(const SpinSweepArgs a)
{
    extern __shared__ __align__(16) uint32_t smem[];
    sweep_block_tn<SYS, L>(a, blockIdx.x * (blockDim.x / kCodeWarpsPerWalkerWarp), blockIdx.x, smem);
}

static size_t potts_tn_smem_bytes(int L, int B, int walkers_per_block);

size_t spin_sweep_tn_smem_bytes(int system, int L, int B, int walkers_per_block)
{
    if (system == kPotts) return potts_tn_smem_bytes(L, B, walkers_per_block);
    const int ncw = walkers_per_block / 32;
    return ((size_t)B * (num_cols(system) + 1) * 4 + 15) / 16 * 16 + (size_t)ncw * tn_ring_bytes(L) +
           (size_t)ncw * 2 * kRing * sizeof(unsigned long long);
}

// ---------------------------------------------------------------------------
// Code form for Potts.  The producer warp draws both words of every site and
// makes the proposal v = (s + 1 + mulhi(u, q-1)) mod q itself.  Per row it
// writes the acceptance words, the old and the proposed row (one byte a site)
// and two code bytes a site, c = 4 + dE without the up neighbour: c0 with the
// left neighbour as it was, c1 with the left neighbour recoloured to its own
// proposal.  With ne(n, s) = [n != s], a neighbour n adds ne(n, v) - ne(n, s) to
// dE; the producer evaluates it four sites at a time on bytes.  The consumer
// adds the up neighbour's term the same way, four sites at a time, from the
// final row above (kept in bytes), and the last site's right neighbour (site 0
// of the same row, final by then) once a row.  The chain itself is the one of
// the Ising code form.  RD is the ring depth in rows (potts_tn_depth).
__device__ __forceinline__ uint32_t nib_half_to_bytes(uint32_t w, int half)  // 4 nibbles -> 4 bytes
{
    const uint32_t t = __byte_perm(w, 0u, half ? 0x3322u : 0x1100u);
    return (t & 0x000F000Fu) | ((t >> 4) & 0x0F000F00u);
}

__device__ __forceinline__ uint32_t bytes_to_nibs(uint32_t w0, uint32_t w1)  // 8 bytes (< 16) -> 8 nibbles
{
    return __byte_perm(w0 | (w0 >> 4), w1 | (w1 >> 4), 0x6420u);
}

// Potts producers.  A Potts site takes two random words and eight neighbour comparisons, about 35
// instructions against the consumer's 18; one warp issues an instruction every 2.5 cycles at best and
// the multiply and logic pipes of a scheduler sustain a Philox block in 88 cycles, so production (not
// the chain) bounds the blocks of two walker warps and is spread over more warps than the Ising
// form's.  The block has 12 warps for two walker warps, 8 for one, warp w on scheduler w mod 4:
//   ncw = 2: [C0, C1, P0.0, P1.0,  P0.3, P1.3, P0.1, P1.1,  P0.4, P1.4, P0.2, P1.2]
//   ncw = 1: [C0, P0.0, P0.1, P0.2,  -, P0.3, P0.4, P0.5]
// so a consumer shares its scheduler with one or two of its producers or with none.
// Where the ring has four rows (L <= 32) four producers take whole rows in turn (produce_potts_rows).
// With two rows (L = 48 and 64) all work on the same row: parts 0..n-1 own contiguous groups of four
// sites, and a part beyond the first draws the block of the site left of its own once more.
// Cycles a site with three producers on words of every row / as described (the consumer's unrolled
// loop included, which pays since all producers run one code): q = 8 L = 32, 8192 walkers 72.7 / 57.8
// (4096 walkers 60.2 / 47.6), L = 24 77.6 / 61.0, L = 16 90.0 / 63.9 (q = 10, 2048 walkers 71.3 / 52.8),
// L = 8 127 / 74; q = 10 L = 48, 2048 walkers 56.1 / 48.9; L = 64, 8192 walkers 81.5 / 77.6 (four parts
// 81.4: production bounds it, two rows being all that fits beside the table), 4096 walkers 63.4 / 54.0.
__host__ __device__ constexpr int potts_parts(int ncw) { return ncw == 2 ? 5 : 6; }  // of a row (L = 48, 64)
__host__ __device__ constexpr int potts_part_groups(int L, int ncw, int part)
{
    // as even as whole groups allow, the surplus with the first parts
    return L / 4 / potts_parts(ncw) + (part < L / 4 % potts_parts(ncw) ? 1 : 0);
}
__host__ __device__ constexpr int potts_part_max(int L)  // most groups a part has, over both layouts
{
    return potts_part_groups(L, 2, 0) > potts_part_groups(L, 1, 0) ? potts_part_groups(L, 2, 0) : potts_part_groups(L, 1, 0);
}
__device__ __forceinline__ CodeRole potts_role(int warp, int ncw)
{
    if (ncw == 1)
        return warp == 0 ? CodeRole{kRoleConsumer, 0, 0}
                         : (warp == 4 ? CodeRole{kRoleIdle, 0, 0} : CodeRole{kRoleProducer, 0, warp < 4 ? warp - 1 : warp - 2});
    if (warp < 2) return CodeRole{kRoleConsumer, warp, 0};
    const int pair = warp & 1, row = warp >> 2;
    return CodeRole{kRoleProducer, pair, (warp & 2) ? row : row + 2};
}
// Threads of a block.  An idle warp holds registers: with eight warps two 32-walker blocks of L = 16 fit
// an SM, with the six that four producers need three do, so a launch of more blocks than SMs drops the
// last two (q = 8, 16384 walkers in 32-walker blocks, 585 sweeps: 11.4 / 9.6 ms; L = 8, 2343 sweeps,
// 11.1 / 8.6; L = 24, 32768 walkers, 130 sweeps, 9.3 / 7.5).  Where every block can have an SM to itself the idle
// warps cost nothing, and a batch may place its blocks better with them: the nine-system mix with 332 walkers
// as a graph of five iterations of 25 sweeps takes 10.95 ms, with six warps 12.25 (why is not known).
constexpr int potts_threads(int ncw) { return ncw == 2 ? 384 : 256; }
constexpr int kPottsThreadsDense = 192;  // one walker warp, four producers

// The split table (L = 64, see potts_split_full): the acceptance words travel as their
// upper 16 bits, two to a 32-bit word (uint2 per 4 sites instead of uint4).
template <int L>
struct PottsSplit {
    static constexpr bool on = L > 48;
};

// The 16-bit stand-ins of the split table.  A threshold T keeps 0xFFFF only for "always"
// and min(T >> 16, 0xFFFE) otherwise; a random word u travels as min(u >> 16, 0xFFFE).  Then
// the upper halves decide exactly wherever they differ (u < T when the half of u is the
// smaller, u >= T when it is the larger, u < T whenever T is "always"), and only equal
// halves -- never with T "always" -- need the full words.
__host__ __device__ __forceinline__ uint16_t split_hi(uint32_t T)
{
    return T == kAlways ? (uint16_t)0xFFFFu : (uint16_t)((T >> 16) < 0xFFFEu ? (T >> 16) : 0xFFFEu);
}

// The split table's 16-bit counters, emptied into the block's 64-bit slot: every bin's
// count is taken and cleared with one atomic AND while the consumers keep counting.
// Producer part 1 of every consumer warp scans one F-th of the bins (b = slice mod F) after
// every row it hands over, so every bin is scanned once every F rows and no row carries the
// whole table.  Having produced row k it knows its consumer has finished row k - RD, so the
// consumer counts at most F + RD rows between two scans of a bin, and F + RD <= 2^16 / (32 L
// x consumer warps) keeps every counter below 2^16.  Words are read eight at a time so the
// loads overlap; the AND runs only where a count is not zero.
template <int RS>
__device__ __forceinline__ void split_scan(uint32_t *sTH, unsigned long long *Hb, int B, int lane, int slice, int F)
{
    const int sbase = (int)__cvta_generic_to_shared(sTH);
    for (int b0 = slice + F * lane; b0 < B; b0 += F * 8 * 32) {
        uint32_t w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int b = b0 + F * 32 * i;
            w[i] = 0u;
            if (b < B)
                asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w[i]) : "r"(checked_addr(sbase + 4 * (b * RS + RS - 1), sbase)));
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int b = b0 + F * 32 * i;
            if (w[i] >> 16) {
                const uint32_t old = atomicAnd(&sTH[b * RS + RS - 1], 0xFFFFu);
                atomicAdd(&Hb[b], (unsigned long long)(old >> 16));
            }
        }
    }
}

// Codes travel as CSC c + bias with c = 4 + dE (without the up neighbour), CSC = 4 bytes a column (2
// with the split table); the consumer flips the top bits behind the up neighbour's term, which leaves
// the signed byte CSC (c - 4): the threshold's place in the bin's row, and RSW of it the bin's move.
template <int L>
struct PottsCode {
    static constexpr int CSC = L > 48 ? 2 : 4;
    static constexpr int SH = CSC == 4 ? 2 : 3;
    static constexpr uint32_t BIAS = (0x80u - 4u * CSC) * 0x01010101u;
    static constexpr uint32_t REST = 0x80808080u;  // dE = 0 at every site
};
__device__ __forceinline__ uint32_t ne16(uint32_t a, uint32_t b)  // per byte 16 [a != b], bytes < 16
{
    return ((a ^ b) + 0x0F0F0F0Fu) & 0x10101010u;
}

// Four sites of a row: bytes ob (old colours), those left (ob_prev, with its last proposal in the top
// byte of pprev), right (ob_next) and below (db); r: the sites' two Philox blocks.  Returns the two
// codes and the proposals in pb; last: the group holds the row's last site, whose right neighbour the
// consumer adds; first: the row's first site does not see the site decided before it.
template <int L>
__device__ __forceinline__ uint2 potts_group(const uint4 (&r)[2], uint32_t q, uint32_t ob, uint32_t ob_prev, uint32_t ob_next,
                                             uint32_t db, uint32_t pprev, bool first, uint32_t mask_last, uint32_t &pb)
{
    using PC = PottsCode<L>;
    const uint32_t qm1 = q - 1u;
    const uint32_t wrap = (0x80u - q) * 0x01010101u;  // per byte: top bit set iff v >= q
    // proposals v = (s + 1 + mulhi(u, q - 1)) mod q, four bytes at once
    const uint32_t t01 = __byte_perm(__umulhi(r[0].x, qm1), __umulhi(r[0].z, qm1), 0x0040u);
    const uint32_t t23 = __byte_perm(__umulhi(r[1].x, qm1), __umulhi(r[1].z, qm1), 0x0040u);
    pb = ob + 0x01010101u + __byte_perm(t01, t23, 0x5410u);
    pb -= (((pb + wrap) & 0x80808080u) >> 7) * q;
    const uint32_t R = __funnelshift_r(ob, ob_next, 8);   // right neighbours (old)
    const uint32_t Lo = __funnelshift_l(ob_prev, ob, 8);  // left neighbours (old)
    const uint32_t Lp = __funnelshift_l(pprev, pb, 8);    // left neighbours (recoloured)
    const uint32_t nRp = ne16(R, pb) & mask_last, nRo = ne16(R, ob) & mask_last;
    const uint32_t sp = 0x40404040u + nRp + ne16(db, pb);
    const uint32_t so = nRo + ne16(db, ob);
    // 16 c: every byte stays in [16, 112] and no partial result borrows across bytes
    const uint32_t c0 = sp + ne16(Lo, pb) - so - ne16(Lo, ob);
    uint32_t c1 = sp + ne16(Lp, pb) - so - ne16(Lp, ob);
    if (first) c1 = __byte_perm(c0, c1, 0x7650u);
    return make_uint2((c0 >> PC::SH) + PC::BIAS, (c1 >> PC::SH) + PC::BIAS);
}

// With a ring of RD = 4 rows, four producers: producer `part` makes every fourth row alone, always in
// the ring's slot `part` (L is a multiple of four), so no block is drawn twice and three rows are on
// the way while one is consumed.
template <int L, int RD>
__device__ __forceinline__ void produce_potts_rows(int64_t nsw, uint32_t sweep0, uint32_t wid, const uint32_t (&rk)[20],
                                                   const uint32_t *__restrict__ lat, int ps, uint32_t q, int part,
                                                   void *ring_u, uint2 *ring_c, uint2 *ring_op, unsigned long long *full,
                                                   unsigned long long *empty, int &k, bool &bad, int drop_k)
{
    static_assert(L % 8 == 0 && L % RD == 0 && !PottsSplit<L>::on, "whole nibble words a row, whole turns of the ring");
    constexpr int WR = L / 8;
    constexpr size_t S = (size_t)(L / 4) * 32;
    // Rows as in produce_tn: when slot `part` is free the consumer has finished the row four before, so
    // from L = 16 up the two rows of the next turn (y + 4, y + 5) have their values for it and are
    // loaded a turn ahead.
    constexpr bool AHEAD = L >= 16;
    uint32_t o[WR], d[WR], on[WR], dn[WR];
    auto load = [&](int y, uint32_t (&a)[WR], uint32_t (&b)[WR]) {
        const int y0 = y < L ? y : y - L, y1 = y + 1 < L ? y + 1 : y + 1 - L;
#pragma unroll
        for (int e = 0; e < WR; ++e) {
            a[e] = lat[(y0 * WR + e) * ps];
            b[e] = lat[(y1 * WR + e) * ps];
        }
    };
    if (AHEAD) load(part, on, dn);
    uint4 *wu = (uint4 *)ring_u + part * S;
    uint2 *wc = ring_c + part * S;
    uint2 *wop = ring_op + part * S;
    k += part;
#pragma unroll 1
    for (int64_t sw = 0; sw < nsw; ++sw) {
        const PhiloxLane pl = philox_lane(sweep0 + (uint32_t)sw, wid, rk);
#pragma unroll 1
        for (int y = part; y < L; y += RD) {
            if (!mbar_wait(&empty[part], (unsigned)(((k / RD) & 1) ^ 1))) {
                bad = true;
                return;
            }
            if (AHEAD) {
#pragma unroll
                for (int e = 0; e < WR; ++e) {
                    o[e] = on[e];
                    d[e] = dn[e];
                }
                load(y + RD, on, dn);
            } else {
                load(y, o, d);
            }
            uint32_t ob_prev = nib_half_to_bytes(o[WR - 1], 1), pprev = 0u;
            uint32_t ob = nib_half_to_bytes(o[0], 0);
#pragma unroll 1
            for (int i = 0; i < WR; ++i) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int j = 2 * i + h;
                    uint4 rr[2];
                    philox4x32_10_groups<2>((uint32_t)(y * (L / 2) + 2 * j), pl, rk, rr);
                    const uint32_t ob_next = nib_half_to_bytes(h == 0 ? o[0] : o[1 % WR], h ^ 1);
                    uint32_t pb;
                    const uint2 c = potts_group<L>(rr, q, ob, ob_prev, ob_next, nib_half_to_bytes(d[0], h), pprev, j == 0,
                                                   (h == 1 && i == WR - 1) ? 0x00FFFFFFu : 0xFFFFFFFFu, pb);
                    wu[j * 32] = clamp_words(make_uint4(rr[0].y, rr[0].w, rr[1].y, rr[1].w));
                    wc[j * 32] = c;
                    wop[j * 32] = make_uint2(ob, pb);
                    ob_prev = ob;
                    ob = ob_next;
                    pprev = pb;
                }
                // the next word becomes word 0
                const uint32_t t0 = o[0], t1 = d[0];
#pragma unroll
                for (int e = 0; e + 1 < WR; ++e) {
                    o[e] = o[e + 1];
                    d[e] = d[e + 1];
                }
                o[WR - 1] = t0;
                d[WR - 1] = t1;
            }
            if (k != drop_k) mbar_arrive(&full[part]);
            k += RD;
        }
    }
    k -= part;
}

// The producer's rows of nsw sweeps: groups [g0, g0 + ng) of every row, the same code for every part.
template <int L, int RD>
__device__ __forceinline__ void produce_potts_tn(int64_t nsw, uint32_t sweep0, uint32_t wid, const uint32_t (&rk)[20],
                                                 const uint32_t *__restrict__ lat, int ps, uint32_t q, int part, int g0,
                                                 int ng, void *ring_u, uint2 *ring_c, uint2 *ring_op,
                                                 unsigned long long *full, unsigned long long *empty, int &k, bool &bad,
                                                 int drop_k, uint32_t *sTH, unsigned long long *Hb, int B, int F, int &since)
{
    constexpr bool SPLIT = PottsSplit<L>::on;
    constexpr int RSW = 5;  // words a split row (only the split table is scanned)
    static_assert(L % 8 == 0, "whole nibble words a row");
    constexpr int WR = L / 8;
    constexpr int NGM = potts_part_max(L);
    constexpr int NA = (2 + NGM) / 2 + 1;  // words of the part's groups and one group on either side
    constexpr size_t S = (size_t)(L / 4) * 32;
    const uint32_t qm1 = q - 1u;
    // Rolling rows as in produce_tn, of this part's words: word e is word g0 / 2 - 1 + e of the row,
    // cyclic.
    int off[NA + 1];
#pragma unroll
    for (int e = 0; e <= NA; ++e) off[e] = (g0 / 2 - 1 + e + WR * 4) % WR * ps;
    const int odd = 16 * (g0 & 1);
    uint32_t o[NA + 1], d[NA + 1], nn[NA + 1];
#pragma unroll
    for (int e = 0; e <= NA; ++e) {
        o[e] = lat[off[e]];
        d[e] = lat[WR * ps + off[e]];
    }
    const uint32_t mask_last = (g0 + ng == L / 4) ? 0x00FFFFFFu : 0xFFFFFFFFu;
#pragma unroll 1
    for (int64_t sw = 0; sw < nsw; ++sw) {
        const PhiloxLane pl = philox_lane(sweep0 + (uint32_t)sw, wid, rk);
#pragma unroll 1
        for (int y = 0; y < L; ++y) {
            const int slot = k % RD;
            bool free_slot = mbar_try(&empty[slot], (unsigned)(((k / RD) & 1) ^ 1));
            // the part's groups at even halves of words: group g0 + i is half i & 1 of word 1 + i / 2
            uint32_t ow[NA], dw[NA];
#pragma unroll
            for (int e = 0; e < NA; ++e) {
                ow[e] = __funnelshift_r(o[e], o[e + 1], odd);
                dw[e] = __funnelshift_r(d[e], d[e + 1], odd);
            }
            uint32_t ob_prev = nib_half_to_bytes(ow[0], 1);  // the four sites left of group g0 (cyclic)
            uint32_t pprev = 0u;
            if (g0 > 0) {
                // proposal of site 4 g0 - 1 (the second site of its Philox block): the c1
                // column of site 4 g0 has it as its recoloured left neighbour
                const uint4 r = philox4x32_10_group((uint32_t)(y * (L / 2) + 2 * g0 - 1), pl, rk);
                uint32_t v = (ob_prev >> 24) + 1u + __umulhi(r.z, qm1);
                v = (v >= q) ? v - q : v;
                pprev = v << 24;
            }
            uint32_t ob = nib_half_to_bytes(ow[1], 0);
            uint4 *wu = (uint4 *)ring_u + slot * S;
            uint2 *wu16 = (uint2 *)ring_u + slot * S;
            uint2 *wc = ring_c + slot * S;
            uint2 *wop = ring_op + slot * S;
#pragma unroll
            for (int i = 0; i < NGM; ++i) {
                if (i < ng) {
                    const int j = g0 + i;
                    uint4 r[2];
                    philox4x32_10_groups<2>((uint32_t)(y * (L / 2) + 2 * j), pl, rk, r);
                    const uint32_t ob_next = nib_half_to_bytes(ow[(3 + i) / 2], (3 + i) & 1);
                    const uint32_t db = nib_half_to_bytes(dw[(2 + i) / 2], i & 1);
                    uint32_t pb;
                    const uint2 c = potts_group<L>(r, q, ob, ob_prev, ob_next, db, pprev, j == 0,
                                                   i == ng - 1 ? mask_last : 0xFFFFFFFFu, pb);
                    if (i == 0) {
                        if (!free_slot && !mbar_wait(&empty[slot], (unsigned)(((k / RD) & 1) ^ 1))) {
                            bad = true;
                            return;
                        }
                        // (also behind the last row: rows 0 and 1 as this sweep leaves them)
                        const int y2 = (y + 2 < L) ? y + 2 : y + 2 - L;
#pragma unroll
                        for (int e = 0; e <= NA; ++e) nn[e] = lat[y2 * WR * ps + off[e]];
                    }
                    if (SPLIT)  // upper halves, clamped to 0xFFFE (split_hi)
                        wu16[j * 32] = make_uint2(__vminu2((r[0].y >> 16) | (r[0].w & 0xFFFF0000u), 0xFFFEFFFEu),
                                                  __vminu2((r[1].y >> 16) | (r[1].w & 0xFFFF0000u), 0xFFFEFFFEu));
                    else
                        wu[j * 32] = clamp_words(make_uint4(r[0].y, r[0].w, r[1].y, r[1].w));
                    wc[j * 32] = c;
                    wop[j * 32] = make_uint2(ob, pb);
                    ob_prev = ob;
                    ob = ob_next;
                    pprev = pb;
                }
            }
            if (k != drop_k) mbar_arrive(&full[slot]);
            ++k;
            if (SPLIT && part == 1) {  // empty one F-th of the 16-bit counters (split_scan)
                split_scan<RSW>(sTH, Hb, B, (int)(threadIdx.x & 31), since, F);
                if (++since == F) since = 0;
            }
#pragma unroll
            for (int e = 0; e <= NA; ++e) {
                o[e] = d[e];
                d[e] = nn[e];
            }
        }
    }
}

// The full acceptance test behind the split table: the walker's acceptance word
// recomputed from its Philox block (block `blk` of the sweep, word y for even
// sites and w for odd ones) against the full threshold T[bin][col] in global
// memory.  Only the row redo (potts_redo_row) calls it, for sites whose upper halves tie.
__device__ __forceinline__ bool potts_split_full(const uint32_t *__restrict__ Tg, int bin, int col, uint32_t blk,
                                                uint32_t g, uint32_t wid, uint32_t key0, uint32_t key1, int odd)
{
    const uint4 r = philox4x32_10_rolled(make_uint4(blk, g, wid, kTagSweep), key0, key1);
    const uint32_t u = odd ? r.w : r.y;
    const uint32_t T = Tg[bin * 9 + col];
    return T == kAlways || u < T;
}

// Row layout of the Potts tables: 11 words a bin (9 thresholds, the counter, a pad word that
// makes the stride odd, so that the bins of a warp's walkers spread over all 32 banks: 1-2 %
// faster than 10 words), 10 at L = 48 (where the 11th would not fit), or at L = 64 the split
// row of 5 words: the 9 upper halves of the thresholds and a 16-bit
// counter, the high half of word 4 (whose low half is column 8).  A visit adds 2^16 to
// word 4, so column 8 never changes; a producer warp empties the 16-bit counters every
// few rows (split_scan) before they can wrap.  Codes are scaled to byte offsets into a
// row (4 c, or 2 c for halfword entries), and a bin move of (c - 4) rows is
// (cs - 4 CSC) MS bytes.
template <int L>
struct PottsRow {
    static constexpr bool split = PottsSplit<L>::on;
    static constexpr int RSW = split ? 5 : (L <= 32 ? 11 : 10);  // words a row
    static constexpr int HW = split ? 4 : 9;               // counter word
    static constexpr uint32_t ONE = split ? 0x10000u : 1u;  // one visit
    static constexpr int CSH = split ? 16 : 0;             // counter shift in its word
    static constexpr int CSC = split ? 2 : 4;              // code scale
    static constexpr int C4 = 4 * CSC;                     // scaled code of dE = 0
    static constexpr int MS = 4 * RSW / CSC;               // bytes a row per unit of scaled code
};

// The row redo behind the split table.  The consumer's pass decides every site on the
// 16-bit stand-ins alone (split_hi), a tie (probability 2^-16 where the threshold is not
// "always") counting as a rejection, and only notes that the row had one.  A lane whose row had a tie then replays the row from its start
// along two trajectories at once: the pass's own (its visits are taken back out of the
// block's 64-bit histogram slot) and the exact one, on which a tie is decided on the full
// words (potts_split_full) and whose visits are added to the slot.  The exact trajectory
// rewrites the row (lattice and up row), the bin and the acceptance count, before the
// ring slot is released.  Up to the first tie the two trajectories coincide.
template <int L>
__device__ __forceinline__ void potts_redo_row(uint32_t *__restrict__ lat, int ps, int y, int sbase, int b0, int &bB,
                                            const uint2 *__restrict__ ru16, const uint2 *__restrict__ rc,
                                            const uint2 *__restrict__ rop, const uint32_t *__restrict__ uOld,
                                            uint32_t *__restrict__ uNew, unsigned long long *Hb, int record,
                                            unsigned &nacc, uint32_t g, uint32_t wid, uint32_t key0, uint32_t key1,
                                            const uint32_t *__restrict__ Tg)
{
    using R = PottsRow<L>;
    constexpr int W4 = L / 4, WR = L / 8;
    auto th = [sbase](int addr) -> uint32_t {
        uint32_t v;
        asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(checked_addr(addr, sbase)));
        return v;
    };
    int bw = b0, br = b0;    // byte addresses of the bins: the pass's trajectory, the exact one
    bool pw = false, pr = false;  // the left neighbour's decision on each
    uint32_t f0w = 0u, f0r = 0u, fprev = 0u;
    unsigned naw = 0u, nar = 0u;
#pragma unroll 1
    for (int j = 0; j < W4; ++j) {
        const uint2 op = rop[j * 32];
        const uint32_t ubw = uOld[j * 32];
        const uint32_t np = ne16(ubw, op.y) >> PottsCode<L>::SH, no = ne16(ubw, op.x) >> PottsCode<L>::SH;
        const uint32_t cx = rc[j * 32].x + np - no - PottsCode<L>::BIAS, cy = rc[j * 32].y + np - no - PottsCode<L>::BIAS;
        const uint2 h = ru16[j * 32];
        uint32_t amw = 0u, amr = 0u;
#pragma unroll 1
        for (int i = 0; i < 4; ++i) {
            const int x = 4 * j + i;
            const uint32_t uw = ((i < 2 ? h.x : h.y) >> (16 * (i & 1))) & 0xFFFFu;
            int cw = (int)(((pw ? cy : cx) >> (8 * i)) & 0xffu);
            int cr = (int)(((pr ? cy : cx) >> (8 * i)) & 0xffu);
            if (x == L - 1) {  // right neighbour: site 0 of this row, final on each trajectory
                cw += R::CSC * ((int)(f0w != (op.y >> 24)) - (int)(f0w != (op.x >> 24)));
                cr += R::CSC * ((int)(f0r != (op.y >> 24)) - (int)(f0r != (op.x >> 24)));
            }
            const bool aw = uw < th(bw + cw);
            const uint32_t Tr = th(br + cr);
            bool ar = uw < Tr;
            if (uw == Tr)
                ar = potts_split_full(Tg, (br - sbase) / (4 * R::RSW), cr / R::CSC, (uint32_t)(y * (L / 2) + x / 2), g,
                                      wid, key0, key1, x & 1);
            if (aw) {
                bw += (cw - R::C4) * R::MS;
                amw |= 0xffu << (8 * i);
            }
            if (ar) {
                br += (cr - R::C4) * R::MS;
                amr |= 0xffu << (8 * i);
            }
            if (record == 0) {
                atomicAdd(&Hb[(bw - sbase) / (4 * R::RSW)], ~0ull);  // minus one: the pass counted it
                atomicAdd(&Hb[(br - sbase) / (4 * R::RSW)], 1ull);
            }
            pw = aw;
            pr = ar;
        }
        naw += (unsigned)__popc(amw);
        nar += (unsigned)__popc(amr);
        const uint32_t fr = op.x ^ ((op.x ^ op.y) & amr);
        if (j == 0) {
            f0r = fr & 0xffu;
            f0w = (op.x ^ ((op.x ^ op.y) & amw)) & 0xffu;
        }
        uNew[j * 32] = fr;
        if (j & 1) lat[(y * WR + (j >> 1)) * ps] = bytes_to_nibs(fprev, fr);
        fprev = fr;
    }
    bB = br;
    nacc += nar - naw;  // modulo 2^32, like the count itself
}

// The consumer's rows of nsw sweeps, joined as in consume_tn: the next row is asked for two byte words
// ahead, and its first site's threshold is loaded for both outcomes of the row's last.  A row is a
// loop over its byte words (4 sites each), unrolled (by two it took 55.8 cycles a site at L = 32 with
// 4096 walkers, in full 47.6; the longer rows of the split table by four: by two 60.2, in full 59.7,
// by four 54.0), with the last
// word, which holds the last site's right-neighbour term, peeled.  The final row above
// lives in a per-lane shared-memory row (bytes).  With the split table there are
// two such rows, read and written in turn (the row being decided reads one and
// writes the other), so that a redo still has the row above; otherwise one row
// is rewritten word by word as the current row completes.
template <int L, int RD, int RECORD>
__device__ __forceinline__ void consume_potts_tn(int64_t nsw, uint32_t sweep0, uint32_t *__restrict__ lat, int ps, int &bR,
                                                 uint32_t *__restrict__ sTH, const void *__restrict__ ring_u_,
                                                 const uint2 *__restrict__ ring_c, const uint2 *__restrict__ ring_op,
                                                 uint32_t *__restrict__ sU, unsigned long long *full,
                                                 unsigned long long *empty, int &k, bool &bad, unsigned long long &nacc,
                                                 int r_lo, int r_hi, int &tst, unsigned &ev, uint32_t wid, uint32_t key0,
                                                 uint32_t key1, const uint32_t *__restrict__ Tg, unsigned long long *Hb)
{
    static_assert(L % 8 == 0, "whole nibble words a row");
    using R = PottsRow<L>;
    using PC = PottsCode<L>;
    constexpr bool SPLIT = R::split;
    constexpr int WR = L / 8;
    constexpr int W4 = L / 4;
    constexpr size_t S = (size_t)W4 * 32;
    static_assert(!SPLIT || L % 2 == 0, "the up rows alternate: row L - 1 must leave its values in the first");
    constexpr int kWordUnroll = SPLIT ? 4 : W4;
    const uint4 *ring_u = (const uint4 *)ring_u_;
    const uint2 *ring_u16 = (const uint2 *)ring_u_;
    // As in the Ising consumer: 32-bit shared-window byte addresses (bB = table base + 4 RSW bin),
    // clamped acceptance words, one compare (split: upper halves).
    const int sbase = (int)__cvta_generic_to_shared(sTH);
    constexpr int TOFF = R::C4;  // signed codes count from column 4
    auto th = [sbase](int addr) -> uint32_t {
        uint32_t v;
        if (SPLIT)
            asm("ld.shared.u16 %0, [%1 + %2];" : "=r"(v) : "r"(checked_addr(addr + TOFF, sbase) - TOFF), "n"(TOFF));
        else
            asm("ld.shared.u32 %0, [%1 + %2];" : "=r"(v) : "r"(checked_addr(addr + TOFF, sbase) - TOFF), "n"(TOFF));
        return v;
    };
    auto hist = [sbase](int addr) {
        asm volatile("red.shared.add.u32 [%0 + %2], %1;" ::"r"(checked_addr(addr + 4 * R::HW, sbase) - 4 * R::HW),
                     "r"(R::ONE), "n"(4 * R::HW)
                     : "memory");
    };
    // threshold address and bin move of byte i of settled codes
    auto at = [](uint32_t c, int i, int b) -> int { return __dp4a((int)c, 1 << (8 * i), b); };
    constexpr int MOVE = 4 * R::RSW / PC::CSC;
    auto moved = [](uint32_t c, int i, int b) -> int { return __dp4a((int)c, MOVE << (8 * i), b); };
    // codes with the up neighbour's term added (bytes CSC (c - 4))
    auto settle = [](uint2 c, uint2 op, uint32_t ubw) -> uint2 {
        const uint32_t np = ne16(ubw, op.y) >> PC::SH, no = ne16(ubw, op.x) >> PC::SH;
        return make_uint2((c.x + np - no) ^ PC::REST, (c.y + np - no) ^ PC::REST);
    };
    const int k_end = k + (int)(nsw * L);
    int bB = sbase + bR * 4;
    uint2 opn = make_uint2(0u, 0u), cdn = opn;
    uint32_t T0 = 0u, T1 = 0u;
    bool accP = false;  // the site decided before
    bool tie = false;
    // decide the current site (codes of its word c, byte i; threshold T0 or T1 by the previous
    // decision) and load both candidates of the next site, byte jn of the codes n
    auto site = [&](uint32_t uw, const uint2 &c, int i, const uint2 &n, int jn, uint32_t &am) {
        const int bA = moved(accP ? c.y : c.x, i, bB);
        const uint32_t T = accP ? T1 : T0;
        T0 = th(at(n.x, jn, bB));
        T1 = th(at(n.y, jn, bA));
        const bool acc = uw < T;  // the producer's clamp makes this "always or u < T"
        if (SPLIT) tie |= uw == T;  // upper halves equal: the row is redone (potts_redo_row)
        if (acc) am |= 0xffu << (8 * i);
        bB = acc ? bA : bB;
        if (RECORD == 0) hist(bB);
        accP = acc;
    };
    if (!mbar_wait(&full[k % RD], (unsigned)((k / RD) & 1))) bad = true;
    if (!bad) {
        const int slot = k % RD;
        opn = ring_op[slot * S];
        cdn = settle(ring_c[slot * S], opn, sU[0]);
        T0 = T1 = th(at(cdn.x, 0, bB));
    }
#pragma unroll 1
    for (int64_t sw = 0; sw < nsw && !bad; ++sw) {
        unsigned na = 0;
#pragma unroll 1
        for (int y = 0; y < L; ++y) {
            const int slot = k % RD, slot_n = (k + 1) % RD;
            const uint4 *ru = ring_u + slot * S;
            const uint2 *ru16 = ring_u16 + slot * S;
            const uint2 *rc = ring_c + slot * S;
            const uint2 *rop = ring_op + slot * S;
            const uint32_t *uOld = (SPLIT && (y & 1)) ? sU + S : sU;  // the row above
            uint32_t *uNew = (SPLIT && !(y & 1)) ? sU + S : sU;       // this row, as it is decided
            const int b0 = bB;
            // the acceptance words of byte word j (split: their upper halves)
            auto words = [&](int j) -> uint4 {
                if (SPLIT) {
                    const uint2 h = ru16[j * 32];
                    return make_uint4(h.x & 0xFFFFu, h.x >> 16, h.y & 0xFFFFu, h.y >> 16);
                }
                return ru[j * 32];
            };
            uint32_t fprev = 0u;
#pragma unroll kWordUnroll
            for (int j = 0; j < W4 - 1; ++j) {
                const uint2 op = opn, cd = cdn;
                const uint4 u = words(j);
                opn = rop[(j + 1) * 32];
                cdn = settle(rc[(j + 1) * 32], opn, uOld[(j + 1) * 32]);
                uint32_t am = 0u;
                site(u.x, cd, 0, cd, 1, am);
                site(u.y, cd, 1, cd, 2, am);
                site(u.z, cd, 2, cd, 3, am);
                site(u.w, cd, 3, cdn, 0, am);
                na += (unsigned)__popc(am);  // 0xff per accepted site: 8 x accepted (divided at the end)
                const uint32_t f = op.x ^ ((op.x ^ op.y) & am);
                uNew[j * 32] = f;
                if (j & 1) lat[(y * WR + (j >> 1)) * ps] = bytes_to_nibs(fprev, f);
                fprev = f;
            }
            {
                constexpr int j = W4 - 1;
                bool next = mbar_try(&full[slot_n], (unsigned)(((k + 1) / RD) & 1));
                const uint2 op = opn;
                uint2 cd = cdn;
                const uint4 u = words(j);
                uint32_t am = 0u;
                site(u.x, cd, 0, cd, 1, am);
                site(u.y, cd, 1, cd, 2, am);
                // the last site's right neighbour is site 0 of this row, final by now (word 0 is written);
                // its code is the top byte
                const uint32_t f0 = uNew[0];
                const uint32_t t = (PC::CSC << 24) * (uint32_t)((int)((f0 & 0xffu) != (op.y >> 24)) - (int)((f0 & 0xffu) != (op.x >> 24)));
                cd.x += t;
                cd.y += t;
                // the next row; behind the last one (or a wait that gave up) an earlier row's codes
                // are read and not used
                if (!next && !(sw + 1 == nsw && y == L - 1))
                    bad = !mbar_wait(&full[slot_n], (unsigned)(((k + 1) / RD) & 1));
                opn = ring_op[slot_n * S];
                const uint2 rcn = ring_c[slot_n * S];
                site(u.z, cd, 2, cd, 3, am);
                cdn = settle(rcn, opn, f0);
                site(u.w, cd, 3, cdn, 0, am);
                na += (unsigned)__popc(am);
                const uint32_t f = op.x ^ ((op.x ^ op.y) & am);
                uNew[j * 32] = f;
                lat[(y * WR + WR - 1) * ps] = bytes_to_nibs(fprev, f);
                if (SPLIT && tie) {
                    potts_redo_row<L>(lat, ps, y, sbase, b0, bB, ru16, rc, rop, uOld, uNew, Hb, RECORD, na, sweep0 + (uint32_t)sw,
                                      wid, key0, key1, Tg);
                    cdn = settle(rcn, opn, uNew[0]);
                    T0 = T1 = th(at(cdn.x, 0, bB));
                    tie = false;
                }
            }
            mbar_arrive(&empty[slot]);  // after the row is stored: the producer reads it later
            ++k;
            if (bad) break;
        }
        nacc += na >> 3;
        if (bad) break;
        const int word = (bB - sbase) / 4;
        if (RECORD == 1) atomicAdd(&sTH[checked_word(word + R::HW)], R::ONE);
        tunnel_step(word, r_lo, r_hi, tst, ev);
    }
    k = k_end;
    bR = (bB - sbase) / 4;
}

// Shared memory a consumer warp owns: RD ring rows (acceptance words 16 B, or their
// upper halves 8 B at L = 64, codes 8 B, old/proposed bytes 8 B, per group of 4 sites
// and lane) and its up row (two at L = 64).
__host__ __device__ constexpr size_t tnp_warp_bytes(int L, int RD)
{
    return (size_t)RD * (size_t)(L / 4) * 32 * ((L > 48 ? 8 : 16) + 8 + 8) + (size_t)(L > 48 ? 2 : 1) * (L / 4) * 32 * 4;
}

// Bytes of the Potts threshold + counter table: PottsRow<L>::RSW words a bin (11, 10 at
// L = 48, the split rows of 5 at L = 64).
__host__ __device__ constexpr size_t tnp_table_bytes(int L, int B)
{
    return ((size_t)B * (L > 48 ? 20 : (L > 32 ? 40 : 44)) + 15) / 16 * 16;
}

template <int L, int RD>
__device__ __forceinline__ void sweep_block_tnp(const SpinSweepArgs &a, int w0, int slot_id, uint32_t *smem)
{
    using R = PottsRow<L>;
    constexpr int C = 9;
    constexpr int RS = R::RSW;  // words a table row
    constexpr size_t S = (size_t)(L / 4) * 32;
    const int ncw = blockDim.x == (unsigned)potts_threads(2) ? 2 : 1;
    // (from lane 0, so that the compiler knows it is the same for the warp)
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const CodeRole role = potts_role(warp, ncw);
    constexpr bool ROWS = RD == 4;            // producers take whole rows in turn, else groups of every row
    const int NP = ROWS ? RD : potts_parts(ncw);  // further producers are idle
    const int pair = role.pair, part = role.part;
    const bool producer = role.kind == kRoleProducer && part < NP, consumer = role.kind == kRoleConsumer;
    int g0 = 0, ng = 0;  // a producer's groups of the row
    for (int i = 0; i <= part && producer && !ROWS; ++i) {
        g0 += ng;
        ng = potts_part_groups(L, ncw, i);
    }
    // (the test hook's row: with whole rows in turn, of the producer whose turn it is)
    int drop_k = (blockIdx.x == 0 && producer && pair == 0 && (ROWS || part == 0)) ? a.debug_drop_row : -1;
    uint32_t *sTH = smem;
    const size_t th_bytes = tnp_table_bytes(L, a.B);
    constexpr size_t UB = R::split ? 8 : 16;  // ring bytes of a group's acceptance words
    char *rbase = (char *)smem + th_bytes + (size_t)pair * tnp_warp_bytes(L, RD);
    void *ring_u = R::split ? (void *)((uint2 *)rbase + lane) : (void *)((uint4 *)rbase + lane);
    uint2 *ring_c = (uint2 *)(rbase + (size_t)RD * S * UB) + lane;
    uint2 *ring_op = (uint2 *)(rbase + (size_t)RD * S * (UB + 8)) + lane;
    uint32_t *sU = (uint32_t *)(rbase + (size_t)RD * S * (UB + 16)) + lane;
    unsigned long long *bars = (unsigned long long *)((char *)smem + th_bytes + (size_t)ncw * tnp_warp_bytes(L, RD));
    unsigned long long *full = bars + (size_t)pair * 2 * RD, *empty = full + RD;

    const int tid = threadIdx.x;
    if (R::split) {  // halfword rows: 9 upper halves (split_hi), the 16-bit counter
        uint16_t *h = (uint16_t *)smem;
        stage_table(a.T, a.B * C, [&](int i, uint32_t t) { h[i + i / C] = split_hi(t); });
        for (int b = tid; b < a.B; b += blockDim.x) h[b * 10 + C] = (uint16_t)0;
    } else {
        stage_table(a.T, a.B * C, [&](int i, uint32_t t) { sTH[i + (RS - C) * (i / C)] = t; });
        for (int b = tid; b < a.B; b += blockDim.x)
            for (int c = C; c < RS; ++c) sTH[b * RS + c] = 0u;
    }
    // as in the Ising form: codes read ahead of a row that never came address the table
    for (int i = tid; i < ncw * RD * (int)S; i += blockDim.x) {
        char *rb = (char *)smem + th_bytes + (size_t)(i / (RD * (int)S)) * tnp_warp_bytes(L, RD) + (size_t)RD * S * UB;
        const int e = i % (RD * (int)S);
        ((uint2 *)rb)[e] = make_uint2(PottsCode<L>::REST, PottsCode<L>::REST);
        ((uint2 *)(rb + (size_t)RD * S * 8))[e] = make_uint2(0u, 0u);
    }
    if (tid == 0)  // per pair: FULL[RD] (NP producer warps arrive), EMPTY[RD] (the consumer)
        for (int i = 0; i < ncw * 2 * RD; ++i)
            mbar_init(bars + i, ((i / RD) % 2 == 0) ? (ROWS ? 32 : 32 * NP) : code_consumer_lanes(a.p - w0 - 32 * (i / (2 * RD))));
    set_block_spin_limit(a.spin_limit);
    checks_begin(a.B * RS, a.debug_check);
    __syncthreads();

    const int w = w0 + pair * 32 + lane;
    const bool active = w < a.p;
    const bool some = w - lane < a.p;  // this warp has walkers
    const uint32_t wid = (uint32_t)(w + a.walker_offset);
    const uint32_t g_first = (uint32_t)a.state->sweep_counter;
    uint32_t *lat = a.lattice + (active ? w : 0);
    int bR = (active ? a.bin[w] : 0) * RS;
    unsigned long long *Hb = a.Hpart + (size_t)slot_id * a.B;
    int k = 0;
    bool bad = false;
    const int r_lo = a.bin_lo * RS, r_hi = a.bin_hi * RS;
    int tst = (consumer && active && a.tun) ? a.tun[w] : 0;
    unsigned ev = 0;
    unsigned long long nacc = 0;
    // rows between two scans of the split table's 16-bit counters (split_scan)
    const int F = R::split ? 65535 / (ncw * 32 * L) - RD : 0;
    int since = 0;
    if (consumer && active) {  // the row above row 0: row L-1 as the previous launch left it
        constexpr int WR = L / 8;
#pragma unroll
        for (int j = 0; j < L / 4; ++j)
            sU[j * 32] = nib_half_to_bytes(lat[((L - 1) * WR + (j >> 1)) * a.pstride], j & 1);
    }
    for (int64_t s0 = 0; s0 < a.sweeps; s0 += a.flush_every) {
        const int64_t nsw = (a.sweeps < s0 + a.flush_every) ? a.sweeps - s0 : (int64_t)a.flush_every;
        const uint32_t g = g_first + (uint32_t)s0;
        if (bad) {  // (a wait of this lane gave up: see code_consumer_lanes)
        } else if (producer) {
            if constexpr (ROWS)
                produce_potts_rows<L, RD>(nsw, g, wid, a.rk, lat, a.pstride, (uint32_t)a.q, part, ring_u, ring_c, ring_op, full,
                                          empty, k, bad, drop_k);
            else
                produce_potts_tn<L, RD>(nsw, g, wid, a.rk, lat, a.pstride, (uint32_t)a.q, part, g0, ng, ring_u, ring_c, ring_op,
                                    full, empty, k, bad, drop_k, sTH, Hb, a.B, F, since);
        } else if (consumer && !some) {  // a consumer warp with no walkers keeps the barrier protocol
#pragma unroll 1
            for (int64_t r = 0; r < nsw * L; ++r) {
                const int slot = k % RD;
                if (!mbar_wait(&full[slot], (unsigned)((k / RD) & 1))) {
                    bad = true;
                    break;
                }
                mbar_arrive(&empty[slot]);
                ++k;
            }
        } else if (consumer && active) {
            if (a.record == 0)
                consume_potts_tn<L, RD, 0>(nsw, g, lat, a.pstride, bR, sTH, ring_u, ring_c, ring_op, sU, full, empty, k, bad,
                                           nacc, r_lo, r_hi, tst, ev, wid, a.key0, a.key1, a.T, Hb);
            else
                consume_potts_tn<L, RD, 1>(nsw, g, lat, a.pstride, bR, sTH, ring_u, ring_c, ring_op, sU, full, empty, k, bad,
                                           nacc, r_lo, r_hi, tst, ev, wid, a.key0, a.key1, a.T, Hb);
        }
        __syncthreads();
        for (int b = tid; b < a.B; b += blockDim.x) {
            const uint32_t c = sTH[b * RS + R::HW] >> R::CSH;
            if (c) {
                Hb[b] += c;
                sTH[b * RS + R::HW] -= c << R::CSH;
            }
        }
        rebase_rows(k, drop_k, RD);
        __syncthreads();
    }
    if (bad) atomicOr(const_cast<int *>(&a.state->err), 1);
    if (consumer && active) {
        a.bin[w] = bR / RS;
        if (a.tun) a.tun[w] = (uint8_t)tst;
    }
    flush_metrics(a.metrics, nacc, ev);
    checks_end(a.state);
}

template <int L, int RD>
// At most 64 walkers (384 threads) a block: the L = 48 and 64 forms need more than the 128
// registers a thread that 512-thread blocks would leave.
__global__ void __launch_bounds__(potts_threads(2), 1) k_sweep_potts_tn(const SpinSweepArgs a)
{
    extern __shared__ __align__(16) uint32_t smem[];
    sweep_block_tnp<L, RD>(a, blockIdx.x * (blockDim.x == (unsigned)potts_threads(2) ? 64 : 32), blockIdx.x, smem);
}

// Rows of the ring: four up to L = 32, two at L = 48 and 64, where four do not fit beside the table (at
// L = 64 they would beside 32-walker blocks, not beside the default 64).
constexpr int potts_tn_depth(int L) { return L <= 32 ? 4 : 2; }

static size_t potts_tn_smem_bytes(int L, int B, int walkers_per_block)
{
    const int ncw = walkers_per_block / 32, RD = potts_tn_depth(L);
    return tnp_table_bytes(L, B) + (size_t)ncw * tnp_warp_bytes(L, RD) +
           (size_t)ncw * 2 * RD * sizeof(unsigned long long);
}

static bool potts_tn_fits(int L, int B, int walkers_per_block)
{
    return L >= 8 && L % 8 == 0 && sweep_L_supported(L) &&
           potts_tn_smem_bytes(L, B, walkers_per_block) <= 227u * 1024u;
}

// SMs of the current device (152 on GB300, also if it cannot be asked).
static int device_sms()
{
    int dev = 0, nsm = 0;
    const bool known = cudaGetDevice(&dev) == cudaSuccess &&
                       cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && nsm > 0;
    return known ? nsm : 152;
}

template <int SYS, int L, int PER_SM>
static cudaError_t launch_per_sm_tn(const SpinSweepArgs &a, int block, cudaStream_t s, int *per_sm)
{
    const size_t smem = spin_sweep_tn_smem_bytes(SYS, L, a.B, block);
    const int largest = spin_sweep_tn_fits(SYS, L, a.B, 64) ? 64 : 32;
    cudaError_t e = allow_dynamic_smem(k_sweep_spin_tn<SYS, L, PER_SM>, spin_sweep_tn_smem_bytes(SYS, L, a.B, largest));
    if (e != cudaSuccess) return e;
    const int nblk = (a.p + block - 1) / block;
    return launch_sweep_kernel(k_sweep_spin_tn<SYS, L, PER_SM>, a, nblk, kCodeWarpsPerWalkerWarp * block, smem, s, per_sm);
}

// L = 8: the registers the compiler takes leave room for two blocks an SM; with more walkers than two
// blocks an SM hold, four in 64 registers a thread are faster (65536 walkers, 585 sweeps: Ising 5.90 / 5.15 ms,
// MUMA 6.10 / 5.46; 16384 walkers, 2343 sweeps: 6.9 / 7.4 and 7.2 / 7.4).  MUMA with fewer walkers takes the
// form with room for three (2048 walkers, 4687 sweeps: 9.1 / 8.5 ms; Ising is 1 % slower with it).  L = 12
// and 16 with room for three gain 4-8 % at 65536 walkers and lose up to 20 % below; from L = 24 up the
// tables leave two blocks, then one.
template <int SYS, int L>
static cudaError_t launch_one_tn(const SpinSweepArgs &a, int block, cudaStream_t s, int *per_sm)
{
    if constexpr (L == 8) {
        if (a.p > 2 * 64 * device_sms()) return launch_per_sm_tn<SYS, L, 4>(a, block, s, per_sm);
        return launch_per_sm_tn<SYS, L, SYS == kMuma ? 3 : 1>(a, block, s, per_sm);
    } else {
        return launch_per_sm_tn<SYS, L, 1>(a, block, s, per_sm);
    }
}

template <int SYS>
static cudaError_t launch_sys_tn(int L, const SpinSweepArgs &a, int block, cudaStream_t s, int *per_sm)
{
    switch (L) {
    case 8: return launch_one_tn<SYS, 8>(a, block, s, per_sm);
    case 12: return launch_one_tn<SYS, 12>(a, block, s, per_sm);
    case 16: return launch_one_tn<SYS, 16>(a, block, s, per_sm);
    case 24: return launch_one_tn<SYS, 24>(a, block, s, per_sm);
    case 32: return launch_one_tn<SYS, 32>(a, block, s, per_sm);
    case 48: return launch_one_tn<SYS, 48>(a, block, s, per_sm);
    case 64: return launch_one_tn<SYS, 64>(a, block, s, per_sm);
    default: return cudaErrorInvalidValue;
    }
}

bool spin_sweep_tn_fits(int system, int L, int B, int walkers_per_block)
{
    if (system == kPotts)
        return (walkers_per_block == 32 || walkers_per_block == 64) && potts_tn_fits(L, B, walkers_per_block);
    return (system == kIsing || system == kMuma) && L >= 2 * kRing &&
           (walkers_per_block == 32 || walkers_per_block == 64) &&
           spin_sweep_tn_smem_bytes(system, L, B, walkers_per_block) <= 227u * 1024u;
}

template <int L>
static cudaError_t launch_one_tnp(const SpinSweepArgs &a, int block, cudaStream_t s, int *per_sm)
{
    constexpr int RD = potts_tn_depth(L);
    const size_t smem = potts_tn_smem_bytes(L, a.B, block);
    const int largest = potts_tn_fits(L, a.B, 64) ? 64 : 32;
    cudaError_t e = allow_dynamic_smem(k_sweep_potts_tn<L, RD>, potts_tn_smem_bytes(L, a.B, largest));
    if (e != cudaSuccess) return e;
    const int nblk = (a.p + block - 1) / block;
    const int threads = RD == 4 && block == 32 && nblk > device_sms() ? kPottsThreadsDense : potts_threads(block / 32);
    return launch_sweep_kernel(k_sweep_potts_tn<L, RD>, a, nblk, threads, smem, s, per_sm);
}

static cudaError_t launch_potts_tn(int L, const SpinSweepArgs &a, int block, cudaStream_t s, int *per_sm)
{
    switch (L) {
    case 8: return launch_one_tnp<8>(a, block, s, per_sm);
    case 16: return launch_one_tnp<16>(a, block, s, per_sm);
    case 24: return launch_one_tnp<24>(a, block, s, per_sm);
    case 32: return launch_one_tnp<32>(a, block, s, per_sm);
    case 48: return launch_one_tnp<48>(a, block, s, per_sm);
    case 64: return launch_one_tnp<64>(a, block, s, per_sm);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_spin_sweep_tn(int system, int L, const SpinSweepArgs &a, int block, cudaStream_t s, int *per_sm)
{
    if (!spin_sweep_supported(system, L) || !spin_sweep_tn_fits(system, L, a.B, block)) return cudaErrorInvalidValue;
    switch (system) {
    case kIsing: return launch_sys_tn<kIsing>(L, a, block, s, per_sm);
    case kMuma: return launch_sys_tn<kMuma>(L, a, block, s, per_sm);
    case kPotts: return launch_potts_tn(L, a, block, s, per_sm);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace muca
