// Draw-ahead form of a sweep call: the acceptance masks of a block of steps are
// drawn by the whole GPU one launch ahead of the update that uses them.
//
// The draws of Sec. 5.3's role do not depend on the spins (the random-number
// contract fixes them by site and step), and they are nearly all of a sweep's
// work: about 13 of its 14 instructions per attempt.  A step of a lattice that
// does not fill the GPU is bound by something else, the synchronisation between
// the steps.  So one launch holds two roles:
//   update  the first CTAs: each holds a tile of rows (all columns) with `halo`
//           rows on either side and runs the block's steps on it without any
//           other CTA; a step spoils one more row at either end of the tile, so
//           that a block of `halo` steps leaves the tile's own rows right.  The
//           redundant rows cost only bit logic (8 operations per 32 sites);
//   draw    all other CTAs: the masks of the next block, into another buffer.
// The next launch updates what this one drew; a launch boundary is the only
// synchronisation between CTAs.
//
// Bound: draws at 1750 per ns on the whole GPU (below); where the lattice is small,
// the chain of steps of a tile (62 ns a step at L = 64, 110 .. 220 ns above) and 2 to
// 3 us per launch.  Measured, one call, before (step launches or one-launch forms)
// and with this form: L = 64, 1000 sweeps 239 -> 170 us; 256, 1000: 1072 -> 316;
// 320, 500: 2985 -> 223; 512, 1000: 4885 -> 383; 1024, 500: 2850 -> 460; 2048, 200:
// 1446 -> 585; 4096, 200: 3546 -> 2193 (1530 attempts per ns of 946); 65536, 4: 12449 ->
// 11150 (1540 of 1380).  Persistent CTAs that wait for one another on flags instead
// of launches were no faster (a block's hand-over costs them 3.4 us); CTAs of one
// cluster are, where they can hold the lattice.
//
// Layout of a tile: the two checkerboard colours of a row are kept apart, 32
// sites of one colour per word, so that a step works on full words: bit k of
// word w of colour p in row y is the site x = 64 w + 2 k + o, o = (y + p) & 1.
// The neighbours of a site of colour p are of the other colour q: the bit at
// the same place in rows y - 1 and y + 1, and in row y the bit at the same
// place and the one before (o = 0) or behind it (o = 1).  With a the site's spin
// and n1 .. n4 its neighbours, S3 = n1 ^ n2 ^ n3 and M3 = maj(n1, n2, n3):
//   two or more anti-aligned  (a ^ M3) | ((a ^ S3) & (a ^ n4))
//   one or three              S3 ^ n4
// and since a draw below thr8 is below thr4 too, Eq. 5 of Sec. 4 is
//   flip = two or more | (P4 & one or three) | P8.
#include "ahead.h"
#include "handle.h"
#include "sweep_device.cuh"

#include <algorithm>
#include <atomic>

namespace ising {

namespace {

// Steps whose masks an update thread holds or has on the way: their latency (about
// a microsecond with the L2 busy) against the time of a step, within 160 KiB.
// (two CTAs a SM: 98 KiB).
__host__ __device__ constexpr uint32_t stages_of(uint32_t kw, bool field, bool two) { return two ? 2 : (field && kw == 4) ? 4 : 8; }

// Threads per CTA.  One lattice: one CTA per SM, so that an update, which the next
// launch waits for, has an SM to itself.  Several lattices: two CTAs per SM, so that
// one draws while the other waits for rows and masks.
constexpr uint32_t kThreads = 512, kBatchThreads = 256;

constexpr uint32_t kChunk = 8;     // steps of a stage of the one-warp form
constexpr uint32_t kWarpStages = 8;
constexpr uint32_t kClusterThreads = 256, kClusterChunk = 4, kClusterStages = 8;  // of the cluster form: update threads, steps of a stage, stages
constexpr uint32_t kBuffers = 3, kClusterBuffers = 2;  // mask buffers, used in turn
constexpr uint32_t kWaitLimit = 1u << 22;  // polls of a wait for masks on their way into shared memory
constexpr uint32_t kPublishedLimit = 1u << 12;  // polls for a word that is there already

template <int V>
struct Parity {
    static constexpr int value = V;
};

__device__ __forceinline__ uint32_t shared_addr(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// Bits 0, 2, .. 62 of v as one word.
__device__ __forceinline__ uint32_t even_bits(uint64_t v)
{
    uint32_t h[2] = {(uint32_t)v & 0x55555555u, (uint32_t)(v >> 32) & 0x55555555u};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        h[i] = (h[i] | (h[i] >> 1)) & 0x33333333u;
        h[i] = (h[i] | (h[i] >> 2)) & 0x0F0F0F0Fu;
        h[i] = (h[i] | (h[i] >> 4)) & 0x00FF00FFu;
    }
    return __byte_perm(h[0], h[1], 0x6420);
}
// The inverse: bit k of v at bit 2 k.
__device__ __forceinline__ uint64_t spread_bits(uint32_t v)
{
    uint32_t h[2] = {__byte_perm(v, 0u, 0x4140), __byte_perm(v, 0u, 0x4342)};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        h[i] = (h[i] | (h[i] << 4)) & 0x0F0F0F0Fu;
        h[i] = (h[i] | (h[i] << 2)) & 0x33333333u;
        h[i] = (h[i] | (h[i] << 1)) & 0x55555555u;
    }
    return (uint64_t)h[0] | ((uint64_t)h[1] << 32);
}

// ------------------------------------------------------------------ draw --
// One item: the masks of one word of one colour for K sweeps from the block's sweep sw.
// A widening multiplication keeps its pipe for 4 cycles and the ALU for 2 of them, so
// a call of 4 draws (16.4 multiplications, 27 ALU operations, 8 insertions) takes 86
// cycles of a sub-partition at best; 92 measured: 1756 draws per ns with K = 4, 1616
// with K = 1.  16 warps a SM are enough for that.  (Insertions kept off the multiply
// pipe, carry chains, funnel shifts, keys in registers: no faster or slower.)
// The first Philox round, and the half of the second that works on its result,
// depend on the site and the colour only: they are done once for the K steps.
// The mask planes of a step: P4 and P8, or in a field the five of field_planes.
template <bool FIELD>
constexpr int kPlanes = FIELD ? 5 : 2;

// a: the lattice (AheadArgs or AheadJob); masks, step_bytes, t0: the block's buffer,
// its stride and first sweep index.  BAND: the masks are those of the rows from
// a.d_row0 on, of a lattice whose Philox groups may need the second counter word.
template <bool FIELD, int K, bool BAND, typename A>
__device__ __forceinline__ void draw_item(const A &a, char *masks, size_t step_bytes, uint32_t t0, uint32_t p, uint32_t sw,
                                          uint32_t idx)
{
    constexpr int NP = kPlanes<FIELD>;
    const uint32_t t = t0 + sw;
    // mask order: pair of rows, word, row of the pair
    const uint32_t pair = a.by_wc.quotient(idx >> 1), w = (idx >> 1) - pair * a.wc;
    uint32_t g0, g_hi = 0u;
    if constexpr (BAND) {
        uint32_t y = a.d_row0 + 2u * pair + (idx & 1u);
        if (y >= a.L) y -= a.L;
        const uint64_t g = (uint64_t)y * (a.L >> 3) + w * 8u;
        g0 = (uint32_t)g;
        g_hi = (uint32_t)(g >> 32);
    } else {
        g0 = (2u * pair + (idx & 1u)) * (a.L >> 3) + w * 8u;
    }
    const uint32_t x2k = (a.c3base | p) ^ a.key.k1[0];
    uint32_t c0[K], c2[K], c3[K], m[K][NP];
    {
        // the step's uniform values, lane k those of sweep t + k % K
        const uint64_t pb = (uint64_t)(t + (threadIdx.x & (K - 1u))) * kPhiloxMulB;
        const uint64_t pa = (uint64_t)((uint32_t)(pb >> 32) ^ a.key.k0[0]) * kPhiloxMulA;
        const uint32_t v0 = (uint32_t)pb ^ a.key.k0[1], v2 = (uint32_t)(pa >> 32) ^ a.key.k1[1];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            c0[k] = K == 1 ? v0 : __shfl_sync(0xFFFFFFFFu, v0, k);
            c2[k] = K == 1 ? v2 : __shfl_sync(0xFFFFFFFFu, v2, k);
            c3[k] = K == 1 ? (uint32_t)pa : __shfl_sync(0xFFFFFFFFu, (uint32_t)pa, k);
#pragma unroll
            for (int j = 0; j < NP; ++j) m[k][j] = 0u;
        }
        if constexpr (BAND)
            if (a.L > 131072u) {  // the second counter word is not 0 everywhere
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const uint64_t qb = (uint64_t)(t + k) * kPhiloxMulB;
                    const uint64_t qa = (uint64_t)((uint32_t)(qb >> 32) ^ g_hi ^ a.key.k0[0]) * kPhiloxMulA;
                    c2[k] = (uint32_t)(qa >> 32) ^ a.key.k1[1];
                    c3[k] = (uint32_t)qa;
                }
            }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const uint64_t pa = (uint64_t)(g0 + q) * kPhiloxMulA;
        const uint64_t pb = (uint64_t)((uint32_t)(pa >> 32) ^ x2k) * kPhiloxMulB;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            uint32_t u[4] = {(uint32_t)(pb >> 32) ^ c0[k], (uint32_t)pb, (uint32_t)pa ^ c2[k], c3[k]};
            philox_rounds_from<2>(u[0], u[1], u[2], u[3], a.key);
#pragma unroll
            for (int l = 0; l < 4; ++l)
#pragma unroll
                for (int j = 0; j < NP; ++j)
                    asm("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %1, %2;\n\t@p or.b32 %0, %0, %3;\n\t}"
                        : "+r"(m[k][j])
                        : "r"(u[l]), "r"(a.thr[j]), "r"(1u << (4 * q + l)));
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        char *const step = masks + (size_t)(2u * (sw + k) + p) * step_bytes;
        if constexpr (FIELD) {
            reinterpret_cast<uint4 *>(step)[idx] = make_uint4(m[k][0], m[k][1], m[k][2], m[k][3]);
            reinterpret_cast<uint32_t *>(step + step_bytes / 5u * 4u)[idx] = m[k][4];  // behind 16 bytes a word
        } else {
            reinterpret_cast<uint2 *>(step)[idx] = make_uint2(m[k][0], m[k][1]);
        }
    }
}

// The warps of the launch take tickets for 32 items each (consecutive words of
// one colour and group of sweeps: nwords is a multiple of 64).
template <bool FIELD, bool BAND, bool TWO>
__device__ __forceinline__ void draw_role(const AheadArgs &a)
{
    const uint32_t lane = threadIdx.x & 31u, per_group = BAND ? (a.d_words + 31u) / 32u : a.nwords / 32u;
    const size_t step_bytes = BAND ? (size_t)a.d_words * (FIELD ? 20u : 8u) : a.step_bytes;
    uint32_t next = lane == 0 ? atomicAdd(a.d_ticket, 1u) : 0u;
    for (;;) {
        const uint32_t it = __shfl_sync(0xFFFFFFFFu, next, 0);
        if (it >= a.d_tickets) return;
        if (lane == 0) next = atomicAdd(a.d_ticket, 1u);  // back before this item is done
        const uint32_t gp = a.by_group.quotient(it);
        uint32_t idx = (it - gp * per_group) * 32u + lane;
        if constexpr (BAND) idx = min(idx, a.d_words - 1u);  // (the last ticket of a group repeats its last word)
        if (!(FIELD && TWO) && a.d_k == 4u)
            draw_item<FIELD, 4, BAND>(a, a.d_masks, step_bytes, a.d_t0, gp & 1u, (gp >> 1) * 4u, idx);
        else if (a.d_k == 2u)
            draw_item<FIELD, 2, BAND>(a, a.d_masks, step_bytes, a.d_t0, gp & 1u, (gp >> 1) * 2u, idx);
        else
            draw_item<FIELD, 1, BAND>(a, a.d_masks, step_bytes, a.d_t0, gp & 1u, gp >> 1, idx);
    }
}

// ---------------------------------------------------------------- update --
// Asynchronous copies to shared memory: each thread fetches only what it reads
// itself, so that waiting for its own copies is enough.
__device__ __forceinline__ void copy_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async8(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(shared_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(shared_addr(bar)) : "memory");
}
// A bounded wait for the phase of the given parity; false when it runs out.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint32_t limit)
{
    for (uint32_t n = 0; n < limit; ++n) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(shared_addr(bar)), "r"(parity)
                     : "memory");
        if (done) return true;
    }
    return false;
}
// Announces `bytes` on the barrier of a stage; the copy then completes it.
__device__ __forceinline__ void copy_bulk(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(shared_addr(bar)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(shared_addr(dst)),
                 "l"(src), "r"(bytes), "r"(shared_addr(bar))
                 : "memory");
}

// The words of a run of KW rows of one column, both colours, from the rows' 64-bit
// words and back (KW is even and runs start at even rows: a row's parity is k's).
template <int KW>
__device__ __forceinline__ void load_run(const uint64_t *p, uint32_t wc, uint32_t (&v)[2][KW])
{
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const uint64_t word = __ldcg(p + k * wc);
        const uint32_t e = even_bits(word), o = even_bits(word >> 1);
        v[0][k] = (k & 1) ? o : e;
        v[1][k] = (k & 1) ? e : o;
    }
}
template <int KW>
__device__ __forceinline__ void store_run(uint64_t *p, uint32_t wc, const uint32_t (&v)[2][KW])
{
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const uint32_t e = (k & 1) ? v[1][k] : v[0][k], o = (k & 1) ? v[0][k] : v[1][k];
        __stcg(p + k * wc, spread_bits(e) | (spread_bits(o) << 1));
    }
}

// A function of three bits by its table: bit (4 a + 2 b + c) of LUT.
template <int LUT>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(d) : "r"(a), "r"(b), "r"(c), "n"(LUT));
    return d;
}

// One step of parity P on a run: hz the horizontal neighbours' words, up / dn the
// words above and below the run, m the masks.
template <int KW, int P>
__device__ __forceinline__ void step_run(uint32_t (&v)[2][KW], const uint32_t (&hz)[KW], uint32_t up, uint32_t dn,
                                         const uint4 (&m)[KW / 2])
{
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const uint32_t p4 = (k & 1) ? m[k / 2].z : m[k / 2].x, p8 = (k & 1) ? m[k / 2].w : m[k / 2].y;
        const uint32_t n1 = v[1 - P][k];
        const uint32_t n2 = ((k + P) & 1) ? __funnelshift_r(n1, hz[k], 1) : __funnelshift_l(hz[k], n1, 1);
        const uint32_t n3 = k == 0 ? up : v[1 - P][k - 1], n4 = k == KW - 1 ? dn : v[1 - P][k + 1];
        const uint32_t s3 = lop3<0x96>(n1, n2, n3), m3 = lop3<0xE8>(n1, n2, n3), x = v[P][k];
        const uint32_t two = lop3<0xBE>(x, m3, lop3<0x18>(x, s3, n4));      // (x ^ m3) | ((x ^ s3) & (x ^ n4))
        const uint32_t drawn = lop3<0x28>(s3, n4, p4) | p8;                  // ((s3 ^ n4) & p4) | p8
        v[P][k] = lop3<0x1E>(x, two, drawn);                                 // x ^ (two | drawn)
    }
}
// The same in a field H.  With sigma the spin in units of the field's sign, a flip
// has the class (sigma, c), c the number of anti-aligned neighbours.  Classes sigma =
// +1 are always taken from c = kA (3, 4 or 5) on, classes sigma = -1 from c = kB on,
// and kA + kB <= 5 (the neighbour sums n > -|H| and n < -|H| are different ones): five
// planes hold all draws, P0 .. P2 for sigma = +1, c = 0 .. 2, P3 for (+1, 3) or else
// (-1, 1), P4 for (+1, 4) or else (-1, 0); a class that is always taken gets an all-one
// word.  The thresholds of one sigma grow with c, so that "c >= j and below the j-th"
// for j = 0 .. c adds nothing to "below the c-th".
template <int KW, int P>
__device__ __forceinline__ void step_run_field(const AheadArgs &a, uint32_t (&v)[2][KW], const uint32_t (&hz)[KW], uint32_t up,
                                               uint32_t dn, const uint4 (&m)[KW], const uint2 (&m4)[KW / 2])
{
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const uint32_t p4 = (k & 1) ? m4[k / 2].y : m4[k / 2].x;
        const uint32_t n1 = v[1 - P][k];
        const uint32_t n2 = ((k + P) & 1) ? __funnelshift_r(n1, hz[k], 1) : __funnelshift_l(hz[k], n1, 1);
        const uint32_t n3 = k == 0 ? up : v[1 - P][k - 1], n4 = k == KW - 1 ? dn : v[1 - P][k + 1];
        const uint32_t s3 = n1 ^ n2 ^ n3, m3 = (n1 & n2) | (n3 & (n1 | n2));
        const uint32_t x = v[P][k];
        const uint32_t t = (x ^ s3) & (x ^ n4);
        const uint32_t b0 = s3 ^ n4, b1 = (x ^ m3) ^ t, b2 = (x ^ m3) & t;  // c = b0 + 2 b1 + 4 b2
        const uint32_t ge1 = b0 | b1 | b2, ge2 = b1 | b2, ge3 = (b0 & b1) | b2;
        uint32_t plus = m[k].x | (ge1 & m[k].y);
        plus |= ge2 & m[k].z;
        plus |= (ge3 & (m[k].w | a.plus3)) | (b2 & (p4 | a.plus4));
        const uint32_t minus = ge2 | (ge1 & (m[k].w | a.minus1)) | (p4 | a.minus0);
        v[P][k] = x ^ (((x ^ a.flipped) & plus) | (~(x ^ a.flipped) & minus));
    }
}
// After the step of parity 1: +1 spins of the run, and the anti-aligned bonds of
// its sites of parity 1 (every bond of the lattice once), by the bit-sliced sum
// b0 + 2 b1 + 4 b2 of a site's four.
template <int KW>
__device__ __forceinline__ void count_run(const uint32_t (&v)[2][KW], const uint32_t (&hz)[KW], uint32_t up, uint32_t dn,
                                          uint32_t &cu, uint32_t &ca)
{
    cu = ca = 0u;
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const uint32_t n1 = v[0][k], x = v[1][k];
        const uint32_t n2 = ((k + 1) & 1) ? __funnelshift_r(n1, hz[k], 1) : __funnelshift_l(hz[k], n1, 1);
        const uint32_t n3 = k == 0 ? up : v[0][k - 1], n4 = k == KW - 1 ? dn : v[0][k + 1];
        const uint32_t s3 = n1 ^ n2 ^ n3, m3 = (n1 & n2) | (n3 & (n1 | n2));
        const uint32_t t = (x ^ s3) & (x ^ n4), h = x ^ m3;
        cu += __popc(x) + __popc(n1);
        ca += __popc(s3 ^ n4) + 2 * __popc(h ^ t) + 4 * __popc(h & t);
    }
}

// A sweep is counted when it is recorded, and the call's last one always.
struct Counting {
    uint32_t phase, slot;
    __device__ __forceinline__ bool next(const AheadArgs &a, bool last)
    {
        const bool rec = a.record_every != 0u && phase + 1 == a.record_every;
        if (a.record_every) phase = rec ? 0u : phase + 1;
        return rec || last;
    }
};

// The state of a run after a counted sweep, for the counting CTAs of a later launch:
// row k of colour q of the lattice's run c (row group times wc plus word) at
// c 2 KW + q KW + k.
template <int KW>
__device__ __forceinline__ void store_snapshot(uint32_t *p, const uint32_t (&v)[2][KW])
{
    if constexpr (KW == 2) {
        *reinterpret_cast<uint4 *>(p) = make_uint4(v[0][0], v[0][1], v[1][0], v[1][1]);
    } else {
#pragma unroll
        for (int k = 0; k < 2 * KW; k += 4)
            *reinterpret_cast<uint4 *>(p + k) =
                make_uint4(v[k / KW][k % KW], v[k / KW][k % KW + 1], v[k / KW][k % KW + 2], v[k / KW][k % KW + 3]);
    }
}
template <int KW>
__device__ __forceinline__ void store_snapshot(const AheadArgs &a, uint32_t slot, uint32_t c, const uint32_t (&v)[2][KW])
{
    store_snapshot<KW>(a.u_snaps + (size_t)slot * (2u * a.nwords) + c * (2u * KW), v);
}

// One tile through the block: threads hold KW rows of one column each (a run).
// SNAPS: counted sweeps may go out as snapshots (where there is a buffer for them), else
// the tile counts its own rows.
// BAND: the tile is one of a band of rows and holds tile_words words of a row, and one
// on either side, whose sites of the colour spoil from the far end, one a step.
template <uint32_t THREADS, int KW, bool FIELD, bool SNAPS, bool BAND, bool TWO>
__device__ __forceinline__ void update_tile(const AheadArgs &a, uint32_t tile, unsigned char *smem)
{
    constexpr uint32_t ST = stages_of(KW, FIELD, TWO);
    constexpr uint32_t NQ = FIELD ? KW : KW / 2;                  // 16-byte mask units of a run and step
    const uint32_t tid = threadIdx.x, wc = a.wc, L = a.L;
    const uint32_t tw = BAND ? a.tile_words + 2u : wc;            // words of a row of the tile
    const uint32_t nruns = (a.tile_rows + 2 * a.halo) / KW, nthr = nruns * tw;  // threads with a run
    const uint32_t nbar = (nthr + 31u) & ~31u;
    // [ST][NQ][THREADS]: (P4, P8) of two rows, or the first four planes of a row
    uint4 *const ring = reinterpret_cast<uint4 *>(smem);
    // in a field [ST][KW / 2][THREADS]: the fifth plane of two rows
    uint2 *const ring4 = reinterpret_cast<uint2 *>(ring + ST * NQ * THREADS);
    // [2][KW][THREADS]: the two colours
    uint32_t *const X = reinterpret_cast<uint32_t *>(ring4 + (FIELD ? ST * (KW / 2) * THREADS : 0u));
    uint32_t *const cnt = X + 2 * KW * THREADS;                   // [samples of the block, last state][2]
    const bool whole = a.halo == 0u;                              // the tile is the lattice
    const bool snaps = SNAPS && a.u_snaps != nullptr;
    if (!snaps) {
        for (uint32_t k = tid; k < 2 * a.u_slots; k += THREADS) cnt[k] = 0u;
        __syncthreads();
    }
    if (tid < nbar) {
        // (a thread past the last run repeats the last one's work)
        const uint32_t c = min(tid, nthr - 1u), run = (BAND ? a.by_tw : a.by_wc).quotient(c), w = c - run * tw;
        const uint32_t groups = L / KW;                           // row groups of the lattice
        uint32_t r0 = tile * a.tile_rows, gw = w;                 // the tile's first own row; the word in the lattice's row
        bool mine = tid < nthr && run >= a.halo / KW && run < (a.halo + a.tile_rows) / KW;
        if constexpr (BAND) {
            const uint32_t ty = tile / a.tiles_x, tx = tile - ty * a.tiles_x, w0 = tx * a.tile_words;
            r0 = a.u_row0 + ty * a.tile_rows;
            gw = w0 + w + wc - 1u;
            while (gw >= wc) gw -= wc;
            mine = mine && w >= 1u && w <= a.tile_words && w0 + w - 1u < wc;
        }
        uint32_t group = (r0 + L - a.halo) / KW + run;            // the run's row group
        while (group >= groups) group -= groups;
        const uint32_t xl = c - w + (w == 0 ? tw - 1u : w - 1u), xr = c - w + (w + 1u == tw ? 0u : w + 1u);
        const uint32_t xu = (KW - 1) * THREADS + (run == 0 ? nthr - tw + w : c - tw);
        const uint32_t xd = c + tw >= nthr ? w : c + tw;
        // the steps after which this warp's rows are of no more use: a step spoils a
        // row at either end of the tile
        uint32_t useful = a.u_steps;
        if (!whole) useful = min(useful, __reduce_max_sync(0xFFFFFFFFu, (min(run, nruns - 1u - run) + 1u) * KW - 1u));

        // the masks of the next step not yet asked for, into its stage
        size_t first = (size_t)(group * (KW / 2)) * wc + gw;      // the run's first pair of rows
        size_t step_bytes = a.step_bytes;
        if constexpr (BAND) {
            uint32_t y = group * KW + L - a.u_mask_row0;          // in the rows that have masks
            if (y >= L) y -= L;
            first = (size_t)(y / 2u) * wc + gw;
            step_bytes = (size_t)a.u_words * (FIELD ? 20u : 8u);
        }
        const char *msrc = a.u_masks + first * (FIELD ? 32u : 16u), *msrc4 = a.u_masks + step_bytes / 5u * 4u + first * 8u;
        const uint32_t mdst = shared_addr(ring + c), mdst4 = shared_addr(ring4 + c);
        uint32_t fetched = 0;
        auto fetch = [&]() {
            if (fetched < useful) {
                const uint32_t st = fetched & (ST - 1u);
#pragma unroll
                for (int k = 0; k < KW / 2; ++k) {
                    if constexpr (FIELD) {
                        copy_async16(mdst + (st * NQ + 2 * k) * THREADS * 16u, msrc + (size_t)k * wc * 32u);
                        copy_async16(mdst + (st * NQ + 2 * k + 1) * THREADS * 16u, msrc + (size_t)k * wc * 32u + 16u);
                        copy_async8(mdst4 + (st * (KW / 2) + k) * THREADS * 8u, msrc4 + (size_t)k * wc * 8u);
                    } else {
                        copy_async16(mdst + (st * NQ + k) * THREADS * 16u, msrc + k * wc * 16u);
                    }
                }
            }
            copy_commit();
            msrc += step_bytes;
            msrc4 += step_bytes;
            ++fetched;
        };
#pragma unroll
        for (uint32_t s = 0; s < ST; ++s) fetch();

        uint32_t v[2][KW];
        load_run<KW>(a.src + (size_t)(group * KW) * wc + gw, wc, v);
#pragma unroll
        for (int k = 0; k < KW; ++k) {
            X[k * THREADS + c] = v[0][k];
            X[(KW + k) * THREADS + c] = v[1][k];
        }
        Counting cn{a.u_phase, 0u};
        uint4 m[NQ];
        uint2 m4[KW / 2];
        auto masks_of = [&](uint32_t s) {
            copy_wait<ST - 1>();
            const uint32_t st = s & (ST - 1u);
#pragma unroll
            for (int k = 0; k < (int)NQ; ++k) m[k] = ring[(st * NQ + k) * THREADS + c];
            if constexpr (FIELD) {
#pragma unroll
                for (int k = 0; k < KW / 2; ++k) m4[k] = ring4[(st * (KW / 2) + k) * THREADS + c];
            }
        };
        masks_of(0);
        asm volatile("bar.sync 1, %0;" ::"r"(nbar) : "memory");

        auto step = [&](auto parity, uint32_t s, bool count) {
            constexpr int P = decltype(parity)::value;
            if (s < useful) {
                const uint32_t *const B = X + (1 - P) * KW * THREADS;
                uint32_t hz[KW];
#pragma unroll
                for (int k = 0; k < KW; ++k) hz[k] = B[k * THREADS + (((k + P) & 1) ? xr : xl)];
                const uint32_t up = B[xu], dn = B[xd];
                if constexpr (FIELD)
                    step_run_field<KW, P>(a, v, hz, up, dn, m, m4);
                else
                    step_run<KW, P>(v, hz, up, dn, m);
#pragma unroll
                for (int k = 0; k < KW; ++k) X[(P * KW + k) * THREADS + c] = v[P][k];
                // the next step's masks, while the others reach the barrier
                fetch();  // into the stage of this step, whose masks are in registers
                masks_of(s + 1u);
                if (P == 1 && count) {
                    if (snaps) {
                        if (mine) store_snapshot<KW>(a, cn.slot, group * wc + w, v);
                    } else {
                        uint32_t cu, ca;
                        count_run<KW>(v, hz, up, dn, cu, ca);
                        cu = __reduce_add_sync(0xFFFFFFFFu, mine ? cu : 0u);
                        ca = __reduce_add_sync(0xFFFFFFFFu, mine ? ca : 0u);
                        if ((tid & 31u) == 0) {
                            atomicAdd(&cnt[2 * cn.slot], cu);
                            atomicAdd(&cnt[2 * cn.slot + 1], ca);
                        }
                    }
                }
            }
            asm volatile("bar.sync 1, %0;" ::"r"(nbar) : "memory");
        };
        for (uint32_t s = 0; s < a.u_steps; s += 2) {
            const bool count = cn.next(a, a.u_last != 0u && s + 2 == a.u_steps);
            step(Parity<0>{}, s, false);
            step(Parity<1>{}, s + 1u, count);
            if (count) ++cn.slot;
        }
        copy_wait<0>();
        // the block's samples (the last counter, if it is none, is the state after the call)
        for (uint32_t k = tid; !snaps && k < a.u_slots; k += nbar) {
            const unsigned long long up = cnt[2 * k], anti = cnt[2 * k + 1];
            if (k < a.u_recs) {
                atomicAdd(a.acc + 2 * (size_t)(a.u_slot0 + k), up);
                atomicAdd(a.acc + 2 * (size_t)(a.u_slot0 + k) + 1, anti);
            }
            if (a.u_last != 0u && k + 1 == a.u_slots) {
                atomicAdd(a.final_acc, up);
                atomicAdd(a.final_acc + 1, anti);
            }
        }
        if (mine) store_run<KW>(a.dst + (size_t)(group * KW) * wc + gw, wc, v);
    }
    __syncthreads();  // the tile's shared memory is free again
}

// L = 64: one warp holds the lattice, two rows a lane; the rows above and below come by
// shuffles and a step has no barrier.  Another warp fetches the masks, in chunks
// of several steps.
__device__ __forceinline__ void update_warp(const AheadArgs &a, unsigned char *smem)
{
    __shared__ __align__(8) uint64_t full[kWarpStages], empty[kWarpStages];
    const uint32_t tid = threadIdx.x, lane = tid & 31u;
    // (1000 sweeps, M/E every tenth: 181 us with a loop of single steps that read their
    // masks one step ahead, 154 with a chunk's 8 steps unrolled on masks in registers: 62 ns
    // a step, of 39 instructions)
    uint4 *const ring = reinterpret_cast<uint4 *>(smem);          // [kWarpStages][kChunk][lane]
    if (tid == 0) {
        for (uint32_t k = 0; k < kWarpStages; ++k) {
            mbar_init(&full[k]);
            mbar_init(&empty[k]);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const uint32_t limit = a.hold_step ? 1u << 12 : kWaitLimit;
    if (tid == 32) {
        uint32_t f = 0;  // chunks asked for
        const uint4 *from = reinterpret_cast<const uint4 *>(a.u_masks);
        for (uint32_t s = 0; s < a.u_steps; s += kChunk, ++f, from += kChunk * 32) {
            const uint32_t st = f % kWarpStages;
            if (f >= kWarpStages && !mbar_wait(&empty[st], (f / kWarpStages - 1u) & 1u, 4 * limit)) break;
            // (failure testing: the held step's chunk and those behind it never arrive)
            if (a.hold_step != 0u && a.hold_step - 1u < a.u_step0 + s + kChunk) break;
            copy_bulk(ring + st * kChunk * 32, from, min(kChunk, a.u_steps - s) * 512u, &full[st]);
        }
        // no copy is on its way when the CTA goes on
        for (uint32_t k = f > kWarpStages ? f - kWarpStages : 0u; k < f; ++k)
            (void)mbar_wait(&full[k % kWarpStages], k / kWarpStages & 1u, limit);
    } else if (tid < 32) {
        uint32_t v[2][2];
        load_run<2>(a.src + lane * 2, 1u, v);
        const uint4 *const mp = ring + lane;
        const uint32_t above = lane - 1u, below = lane + 1u;
        uint32_t until = a.record_every - a.u_phase;                  // sweeps to the next recorded one (0: none)
        uint32_t *snap = a.u_snaps + lane * 4u;
        auto record = [&]() {
            store_snapshot<2>(snap, v);
            snap += 2u * a.nwords;
        };
        auto step = [&](auto parity, const uint4 &mj) {
            constexpr int P = decltype(parity)::value;
            const uint32_t up = __shfl_sync(0xFFFFFFFFu, v[1 - P][1], above);
            const uint32_t dn = __shfl_sync(0xFFFFFFFFu, v[1 - P][0], below);
            // a row is one word: its horizontal neighbours are its own bits
            const uint32_t hz[2] = {v[1 - P][0], v[1 - P][1]};
            const uint4 m[1] = {mj};
            step_run<2, P>(v, hz, up, dn, m);
        };
        uint4 m[kChunk];                                              // a chunk's masks
        bool good = __all_sync(0xFFFFFFFFu, mbar_wait(&full[0], 0u, limit));
        if (good) {
#pragma unroll
            for (uint32_t j = 0; j < kChunk; ++j) m[j] = mp[j * 32];
            uint32_t st = 0, turn = 0;
            for (uint32_t left = a.u_steps;;) {
                // each step's masks make room for those of the same step of the next chunk
                uint32_t next_st = st + 1u;
                if (next_st == kWarpStages) {
                    next_st = 0u;
                    turn ^= 1u;
                }
                const uint4 *const next = mp + next_st * (kChunk * 32);
                if (left > kChunk) {
                    good = __all_sync(0xFFFFFFFFu, mbar_wait(&full[next_st], turn, limit));
                    if (!good) break;
                }
                bool ended = false;
#pragma unroll
                for (uint32_t j = 0; j < kChunk; j += 2) {
                    step(Parity<0>{}, m[j]);
                    m[j] = next[j * 32];
                    step(Parity<1>{}, m[j + 1]);
                    m[j + 1] = next[(j + 1) * 32];
                    if (--until == 0u) {
                        record();
                        until = a.record_every;
                    }
                    if (left <= j + 2u) {                             // a block's steps are even
                        ended = true;
                        break;
                    }
                }
                if (ended) break;
                left -= kChunk;
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[st]);
                st = next_st;
            }
        }
        if (good && a.u_slots > a.u_recs) record();                   // the state after the call
        if (!good && lane == 0 && a.err) atomicExch(a.err, 1u);
        store_run<2>(a.dst + lane * 2, 1u, v);
    }
    __syncthreads();
}

// M and E of the snapshots of the launch before, a thread a run.
template <int KW>
__device__ __forceinline__ void count_role(const AheadArgs &a, uint32_t cta)
{
    const uint32_t wc = a.wc, runs = a.nwords / KW, per = (runs + 31u) & ~31u;  // threads a snapshot: whole warps
    for (uint32_t i = cta * kThreads + threadIdx.x; i < a.c_slots * per; i += a.count_ctas * kThreads) {
        const uint32_t slot = i / per, c = min(i - slot * per, runs - 1u), w = c - a.by_wc.quotient(c) * wc;
        const bool real = i - slot * per < runs;
        const uint32_t *const B = a.c_snaps + (size_t)slot * (2u * a.nwords);
        const uint32_t left = c - w + (w == 0 ? wc - 1u : w - 1u), right = c - w + (w + 1u == wc ? 0u : w + 1u);
        uint32_t v[2][KW], hz[KW], cu, ca;
#pragma unroll
        for (int k = 0; k < KW; ++k) {
            v[0][k] = B[c * 2 * KW + k];
            v[1][k] = B[c * 2 * KW + KW + k];
            hz[k] = B[(((k + 1) & 1) ? right : left) * 2 * KW + k];
        }
        const uint32_t up = B[(c < wc ? runs - wc + c : c - wc) * 2 * KW + KW - 1], dn = B[(c + wc >= runs ? c + wc - runs : c + wc) * 2 * KW];
        count_run<KW>(v, hz, up, dn, cu, ca);
        cu = __reduce_add_sync(0xFFFFFFFFu, real ? cu : 0u);
        ca = __reduce_add_sync(0xFFFFFFFFu, real ? ca : 0u);
        if ((threadIdx.x & 31u) == 0u) {
            if (slot < a.c_recs) {
                atomicAdd(a.acc + 2 * (size_t)(a.c_slot0 + slot), (unsigned long long)cu);
                atomicAdd(a.acc + 2 * (size_t)(a.c_slot0 + slot) + 1, (unsigned long long)ca);
            }
            if (a.c_last != 0u && slot + 1 == a.c_slots) {
                atomicAdd(a.final_acc, (unsigned long long)cu);
                atomicAdd(a.final_acc + 1, (unsigned long long)ca);
            }
        }
    }
}

// TWO: two CTAs share a SM (8 rows a thread, and 4 in a field).
template <int KW, bool WARP, bool FIELD, bool TWO>
__global__ void __launch_bounds__(kThreads, TWO ? 2 : 1) k_ahead(const __grid_constant__ AheadArgs a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    // The first launch of a call (it only draws) starts after all work before it.
    // A later one draws into a buffer, and takes tickets from a counter, that no
    // launch still running uses (three and four in turn), so its draws need not
    // wait: of what the stream has written they read the counter alone, by atomics in the
    // L2, which a launch that has ended has cleared.  Updates and counts need what the
    // launch before wrote.
    const uint32_t early = a.update_ctas + a.count_ctas;
    if (blockIdx.x < early || early == 0u) dependent_launch_wait();
    dependent_launch_trigger();
    if (blockIdx.x < a.update_ctas) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *a.next_ticket = 0u;
        if constexpr (WARP)
            update_warp(a, smem);
        else
            for (uint32_t t = blockIdx.x; t < a.tiles; t += a.update_ctas) update_tile<kThreads, KW, FIELD, true, false, TWO>(a, t, smem);
    } else if (blockIdx.x < early) {
        count_role<KW>(a, blockIdx.x - a.update_ctas);
    }
    if (a.d_tickets != 0u) draw_role<FIELD, false, TWO>(a);
}

// --------------------------------------------------------------- cluster --
// A lattice of 320^2 .. 512^2 held by the CTAs of one cluster: each has its tile of rows and
// a halo of a.halo rows on either side, which its neighbours' boundary rows refresh every
// a.halo steps through distributed shared memory, so that a block of many sweeps is one
// launch and the halo is short.
//
// Bound: the chain of steps, 290 cycles each (a barrier 70, shared memory 35, 45
// dependent instructions; an exchange 600 every 16 steps), with the draws beside it.  The
// tiles of separate launches need 230 cycles a step and 2.8 us a launch: 1000
// sweeps of 512 478 -> 383 us (M/E every hundredth), 500 of 320 237 -> 223 (every sweep); 256 (2 us of 32 sweeps a launch) is no faster than with tiles, 1024 is bound by its
// draws.  One row a thread, 8 rows of halo, and 4 rows a lane with shuffles in place of
// the barrier took as long within 5 %.

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of a shared variable of this CTA in the one of the given rank.
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// 16 bytes into a peer's shared memory; the peer's barrier counts them.
__device__ __forceinline__ void store_peer16(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "r"(x),
                 "r"(y), "r"(z), "r"(w), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(shared_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy_bulk_part(uint32_t dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
                 "r"(bytes), "r"(shared_addr(bar))
                 : "memory");
}

// Shared memory of update_cluster: the masks of a.stages chunks of kClusterChunk steps, the
// two colours of the rows, two inboxes of halo rows.
__host__ __device__ inline uint32_t cluster_step_bytes(uint32_t rows, uint32_t wc) { return rows * wc * 8u; }
__host__ __device__ inline uint32_t cluster_smem(uint32_t rows, uint32_t halo, uint32_t wc, uint32_t stages)
{
    return stages * kClusterChunk * cluster_step_bytes(rows, wc) + 4u * kClusterThreads * 4u + 2u * (2u * halo * wc * 8u);
}

__device__ __forceinline__ void update_cluster(const AheadArgs &a, unsigned char *smem)
{
    constexpr uint32_t CH = kClusterChunk, T = kClusterThreads;
    constexpr int KW = 2;                                              // rows of a run
    __shared__ __align__(8) uint64_t full[kClusterStages], empty[kClusterStages], inbox_bar[2];
    const uint32_t tid = threadIdx.x, wc = a.wc, L = a.L, rank = blockIdx.x, ranks = a.update_ctas;
    const uint32_t R = a.tile_rows, H = a.halo, rows = R + 2 * H;
    const uint32_t nthr = rows / KW * wc, nbar = (nthr + 31u) & ~31u;  // threads with a run; in whole warps
    const uint32_t sb = cluster_step_bytes(rows, wc), ST = a.stages;
    unsigned char *const ring = smem;                                  // [ST][CH][pair of rows][word][row of the pair]
    uint32_t *const X = reinterpret_cast<uint32_t *>(smem + ST * CH * sb);  // [2][KW][T]: the two colours
    uint4 *const inbox = reinterpret_cast<uint4 *>(X + 2 * KW * T);    // [2][runs of both halos]
    const uint32_t inbox_bytes = 2u * H * wc * 8u;
    if (tid == 0) {
        for (uint32_t k = 0; k < ST; ++k) {
            mbar_init(&full[k]);
            mbar_init(&empty[k]);
        }
        mbar_init(&inbox_bar[0]);
        mbar_init(&inbox_bar[1]);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const uint32_t limit = a.hold_step ? 1u << 12 : kWaitLimit;
    const uint32_t r0 = rank * R;
    if (tid >= nbar) {
        // the warp that fetches masks
        cluster_sync();
        if (tid == nbar) {
            const uint32_t y0 = r0 >= H ? r0 - H : r0 + L - H;  // the first row with masks; the rows may go on at row 0
            const uint32_t bytes1 = min(rows, L - y0) * wc * 8u, bytes2 = sb - bytes1;
            uint32_t f = 0;
            const char *from = a.u_masks;
            for (uint32_t s = 0; s < a.u_steps; s += CH, ++f) {
                const uint32_t st = f % ST, n = min(CH, a.u_steps - s);
                if (f >= ST && !mbar_wait(&empty[st], (f / ST - 1u) & 1u, 4 * limit)) break;
                // (failure testing, as in update_warp)
                if (a.hold_step != 0u && a.hold_step - 1u < a.u_step0 + s + CH) break;
                mbar_expect(&full[st], n * sb);
                uint32_t dst = shared_addr(ring + st * CH * sb);
                for (uint32_t j = 0; j < n; ++j, from += a.step_bytes, dst += sb) {
                    copy_bulk_part(dst, from + (size_t)y0 * wc * 8u, bytes1, &full[st]);
                    if (bytes2) copy_bulk_part(dst + bytes1, from, bytes2, &full[st]);
                }
            }
            // no copy is on its way when the CTA goes on
            for (uint32_t k = f > ST ? f - ST : 0u; k < f; ++k) (void)mbar_wait(&full[k % ST], k / ST & 1u, limit);
        }
        __syncwarp();
    } else {
        // (a thread past the last run repeats the last one's work)
        const uint32_t c = min(tid, nthr - 1u), run = a.by_wc.quotient(c), w = c - run * wc;
        const uint32_t groups = L / KW, hr = H / KW, rr = R / KW;
        uint32_t group = (r0 + L - H) / KW + run;                      // the run's row group
        while (group >= groups) group -= groups;
        const bool own = run >= hr && run < hr + rr, mine = own && tid < nthr;
        const uint32_t xl = c - w + (w == 0 ? wc - 1u : w - 1u), xr = c - w + (w + 1u == wc ? 0u : w + 1u);
        const uint32_t xu = (KW - 1) * T + (run == 0 ? nthr - wc + w : c - wc);
        const uint32_t xd = c + wc >= nthr ? w : c + wc;
        uint32_t v[2][KW];
        load_run<KW>(a.src + (size_t)(group * KW) * wc + w, wc, v);
#pragma unroll
        for (int k = 0; k < KW; ++k) {
            X[k * T + c] = v[0][k];
            X[(KW + k) * T + c] = v[1][k];
        }
        // where this run's rows go in the peers' inboxes, and come from in this one's
        const uint32_t up_rank = rank == 0 ? ranks - 1u : rank - 1u, dn_rank = rank + 1u == ranks ? 0u : rank + 1u;
        const bool to_up = mine && run < 2u * hr, to_dn = mine && run >= rr;
        const uint32_t put_up = peer_addr(shared_addr(inbox + run * wc + w), up_rank), bar_up = peer_addr(shared_addr(inbox_bar), up_rank);
        const uint32_t put_dn = peer_addr(shared_addr(inbox + (to_dn ? run - rr : 0u) * wc + w), dn_rank),
                       bar_dn = peer_addr(shared_addr(inbox_bar), dn_rank);
        const uint32_t take = (run < hr ? run : run >= rr ? run - rr : 0u) * wc + w;
        // no peer writes here before the barriers are ready; every peer has loaded its rows
        cluster_sync();

        // after a wait for masks has run out the others hardly wait; rows of peers always
        // come, if late
        uint32_t patience = limit;
        bool good = true, received = true;
        auto wait_masks = [&](uint64_t *bar, uint32_t parity) {
            if (!mbar_wait(bar, parity, patience)) {
                good = false;
                patience = 1u;
            }
        };
        // the masks of a chunk's steps, read while the threads gather at the barrier before it
        uint4 m[CH][1];
        const unsigned char *const mp = ring + c * 16u;
        auto masks_of = [&](uint32_t stage) {
            const unsigned char *p = mp + stage * (CH * sb);
#pragma unroll
            for (uint32_t j = 0; j < CH; ++j, p += sb) m[j][0] = *reinterpret_cast<const uint4 *>(p);
        };
        wait_masks(&full[0], 0u);
        masks_of(0);
        asm volatile("bar.sync 1, %0;" ::"r"(nbar) : "memory");
        // steps for which this warp's rows are right after an exchange: a step spoils a
        // row at either end of the tile
        const uint32_t useful = __reduce_max_sync(0xFFFFFFFFu, (min(run, rows / KW - 1u - run) + 1u) * KW - 1u);
        uint32_t phase = 0, exchanges = 0;                             // steps since the last exchange; exchanges
        uint32_t st = 0, turn = 0;                                     // the chunk's stage and its parity
        uint32_t until = a.record_every - a.u_phase;                   // sweeps to the next recorded one (0: none)
        uint32_t *snap = a.u_snaps + (size_t)(group * wc + w) * (2 * KW);
        if (tid == 0 && a.u_steps > H) mbar_expect(&inbox_bar[0], inbox_bytes);
        auto step = [&](auto parity, const uint4 (&mj)[1]) {
            constexpr int P = decltype(parity)::value;
            const uint32_t *const B = X + (1 - P) * KW * T;
            uint32_t hz[KW];
#pragma unroll
            for (int k = 0; k < KW; ++k) hz[k] = B[k * T + (((k + P) & 1) ? xr : xl)];
            const uint32_t up = B[xu], dn = B[xd];
            step_run<KW, P>(v, hz, up, dn, mj);
#pragma unroll
            for (int k = 0; k < KW; ++k) X[(P * KW + k) * T + c] = v[P][k];
        };
        auto record = [&]() {
            if (mine) store_snapshot<KW>(snap, v);
            snap += 2 * a.nwords;
        };
        for (uint32_t left = a.u_steps;;) {
            // a chunk is 4 steps, the last one 2 or 4
            const bool active = phase < useful;
            if (active) step(Parity<0>{}, m[0]);
            asm volatile("bar.sync 1, %0;" ::"r"(nbar) : "memory");
            if (active) step(Parity<1>{}, m[1]);
            if (--until == 0u) {
                record();
                until = a.record_every;
            }
            if (left <= 2u) break;
            asm volatile("bar.sync 1, %0;" ::"r"(nbar) : "memory");
            if (active) step(Parity<0>{}, m[2]);
            asm volatile("bar.sync 1, %0;" ::"r"(nbar) : "memory");
            if (active) step(Parity<1>{}, m[3]);
            if (--until == 0u) {
                record();
                until = a.record_every;
            }
            if (left <= 4u) break;
            left -= CH;
            phase += CH;
            uint32_t next_st = st + 1u;
            if (next_st == ST) {
                next_st = 0u;
                turn ^= 1u;
            }
            if (phase == H) {
                // exchange: boundary rows out, halo rows in
                phase = 0u;
                const uint32_t e = exchanges & 1u, off = e * inbox_bytes;
                if (to_up) store_peer16(put_up + off, v[0][0], v[0][1], v[1][0], v[1][1], bar_up + e * 8u);
                if (to_dn) store_peer16(put_dn + off, v[0][0], v[0][1], v[1][0], v[1][1], bar_dn + e * 8u);
                // (the next exchange's bytes may come as soon as this one's have gone)
                if (tid == 0 && received) mbar_expect(&inbox_bar[1u - e], inbox_bytes);
                asm volatile("bar.sync 1, %0;" ::"r"(nbar) : "memory");
                if (!own) {
                    received = received && mbar_wait(&inbox_bar[e], exchanges >> 1 & 1u, 4 * limit);
                    const uint4 q = inbox[e * (inbox_bytes / 16u) + take];
                    v[0][0] = q.x;
                    v[0][1] = q.y;
                    v[1][0] = q.z;
                    v[1][1] = q.w;
#pragma unroll
                    for (int k = 0; k < KW; ++k) {
                        X[k * T + c] = v[0][k];
                        X[(KW + k) * T + c] = v[1][k];
                    }
                }
                ++exchanges;
            }
            wait_masks(&full[next_st], turn);
            masks_of(next_st);
            asm volatile("bar.sync 1, %0;" ::"r"(nbar) : "memory");
            if (tid == 0) mbar_arrive(&empty[st]);
            st = next_st;
        }
        if (a.u_slots > a.u_recs) record();                            // the state after the call
        if (!(good && received) && a.err) atomicExch(a.err, 1u);
        if (mine) store_run<KW>(a.dst + (size_t)(group * KW) * wc + w, wc, v);
    }
    cluster_sync();  // no peer writes into a CTA that has ended
}

// How many updates' writes are visible here: published with release order by a thread that
// has waited for them, read with acquire order (and then a CTA barrier) by one that has not.
__device__ __forceinline__ void publish(unsigned int *done, uint32_t n)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(done), "r"(n) : "memory");
}
__device__ __forceinline__ bool published(const unsigned int *done, uint32_t n, uint32_t limit)
{
    for (uint32_t k = 0; k < limit; ++k) {
        uint32_t v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(done) : "memory");
        if (v >= n) return true;
    }
    return false;
}

// The launches of a call take turns: draws of block b and counts of block b - 2, and the
// update of block b.  The update starts when the draws have ended; it lets the next draws
// start at once, which need not wait for it: what they write was read, and what they
// count was written, by launches that ended before the update began.  That they have ended
// does not make their writes visible to a launch that did not wait for them, and the
// buffers are used again every other block: so the update publishes, before it lets the
// draws start, what it has waited for, and the draws acquire that (it is there when they
// start).  One CTA of the draws stays until the update before has ended, for the next
// update, which waits for the draws alone.
__global__ void __launch_bounds__(kThreads, 1) k_ahead_draw(const __grid_constant__ AheadArgs a)
{
    if (a.c_wait != 0u) dependent_launch_wait();  // the call's last counts
    dependent_launch_trigger();
    bool go = true;
    if (a.d_after != 0u) {
        const bool late = threadIdx.x == 0 && !published(a.done, a.d_after, kPublishedLimit);
        if (late && a.err) atomicExch(a.err, 1u);
        go = __syncthreads_or(late) == 0;
    }
    if (go && blockIdx.x < a.count_ctas) count_role<2>(a, blockIdx.x);
    if (go && a.d_tickets != 0u) draw_role<false, false, false>(a);
    if (blockIdx.x + 1u == gridDim.x) {
        dependent_launch_wait();
        if (threadIdx.x == 0) *a.next_ticket = 0u;
    }
}

__global__ void __launch_bounds__(kClusterThreads + 32, 1) k_ahead_cluster(const __grid_constant__ AheadArgs a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    dependent_launch_wait();
    // (the last thread, of the warp that fetches masks: the others need not wait for it)
    const bool last = threadIdx.x + 1u == blockDim.x;
    if (blockIdx.x == 0 && last) publish(a.done, a.u_before);
    if (blockIdx.x != 0 || last) dependent_launch_trigger();
    __syncwarp();
    update_cluster(a, smem);
}

// Large lattices: a launch draws the masks of a band of rows (and of the rows that the
// band's tiles spoil) for a block of sweeps and updates the band before from one copy of
// the lattice to the other.
template <bool FIELD>
__global__ void __launch_bounds__(kThreads, 2) k_ahead_band(const __grid_constant__ AheadArgs a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    // (waits as in k_ahead)
    if (blockIdx.x < a.update_ctas || a.update_ctas == 0u) dependent_launch_wait();
    dependent_launch_trigger();
    if (blockIdx.x < a.update_ctas) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *a.next_ticket = 0u;
        for (uint32_t t = blockIdx.x; t < a.tiles; t += a.update_ctas) update_tile<kThreads, FIELD ? 4 : 8, FIELD, false, true, true>(a, t, smem);
    }
    if (a.d_tickets != 0u) draw_role<FIELD, true, true>(a);
}

// ----------------------------------------------------------------- batch --
// Bound: the draws, 1750 per ns (a lattice's keys come from registers here: 1700), as
// soon as the lattices together have some 64 M attempts a block; the tiles take the SMs
// for about a fifth as long.  Measured, strips in one persistent launch (batch.cu) and
// this: four sizes 256 .. 2048 at 32 temperatures, 100 sweeps 15043 -> 12885 us (1380
// attempts per ns); 32 of 512^2, 500 sweeps 10612 -> 3213; one of 2048^2 10998 -> 1554; 128
// of 64^2 1284 -> 638.
//
// Many lattices: launch b draws block b of every lattice that has one and updates
// block b - 1.  Lattices have blocks of their own length; they are sorted by the
// number of their blocks, so that those still running come first.

// The job that item `i` of a launch belongs to, by the running sums of the jobs.
__device__ __forceinline__ uint32_t find_job(const AheadJob *jobs, uint32_t n, uint32_t i, uint32_t AheadJob::*start)
{
    uint32_t lo = 0, hi = n;
    while (hi - lo > 1u) {
        const uint32_t mid = (lo + hi) / 2u;
        if (jobs[mid].*start <= i)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

// early: this CTA has not waited for the launch before.  It reads the table of the lattices
// and the run's first sweep indices, which the copies before the run wrote where an earlier
// run's were: that the run's first launch has waited for them is acquired here, beside the
// first ticket (it published that before it let the next one start).
__device__ __forceinline__ void batch_draw_role(const AheadBatchArgs &a, bool early)
{
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t next = lane == 0 ? atomicAdd(a.d_ticket, 1u) : 0u;
    if (early && lane == 0 && !published(a.done, 1u, kPublishedLimit)) {
        atomicExch(a.err, 1u);
        next = a.d_tickets;
    }
    __syncwarp();
    for (;;) {
        const uint32_t it = __shfl_sync(0xFFFFFFFFu, next, 0);
        if (it >= a.d_tickets) return;
        if (lane == 0) next = atomicAdd(a.d_ticket, 1u);  // back before this item is done
        const uint32_t ji = find_job(a.jobs, a.d_jobs, it, &AheadJob::ticket_start);
        const AheadJob j = a.jobs[ji];
        const uint32_t local = it - j.ticket_start, gp = j.by_group.quotient(local);
        const uint32_t sw = (gp >> 1) * 4u;
        if (sw >= j.sweeps - a.block * j.block_sweeps) continue;  // past the lattice's last sweep
        const uint32_t idx = (local - gp * (j.nwords / 32u)) * 32u + lane;
        char *const masks = j.masks + (size_t)(a.block % kBuffers) * j.mask_bytes;
        const uint32_t t0 = a.t0[j.index] + a.block * j.block_sweeps;
        if (j.field)
            draw_item<true, 4, false>(j, masks, j.step_bytes, t0, gp & 1u, sw, idx);
        else
            draw_item<false, 4, false>(j, masks, j.step_bytes, t0, gp & 1u, sw, idx);
    }
}

// The arguments of a tile's block, as the one-lattice form has them.
__device__ __forceinline__ void batch_tile_args(const AheadBatchArgs &a, const AheadJob &j, AheadArgs &t)
{
    const uint32_t ub = a.block - 1u, done = ub * j.block_sweeps, n = min(j.block_sweeps, j.sweeps - done);
    const uint32_t t0 = a.t0[j.index], re = j.record_every;
    t.L = j.L;
    t.wc = j.wc;
    t.nwords = j.nwords;
    t.by_wc = j.by_wc;
    t.plus3 = j.plus3;
    t.plus4 = j.plus4;
    t.minus0 = j.minus0;
    t.minus1 = j.minus1;
    t.flipped = j.flipped;
    t.step_bytes = j.step_bytes;
    t.record_every = re;
    t.acc = j.acc;
    t.final_acc = j.final_acc;
    t.tile_rows = j.tile_rows;
    t.halo = j.halo;
    t.u_steps = 2u * n;
    t.src = (ub & 1u) ? j.odd : j.even;
    t.dst = (ub & 1u) ? j.even : j.odd;
    t.u_masks = j.masks + (size_t)(ub % kBuffers) * j.mask_bytes;
    t.u_phase = re ? (t0 + done) % re : 0u;
    t.u_recs = re ? (t.u_phase + n) / re : 0u;
    t.u_slot0 = re ? (t0 % re + done) / re : 0u;
    t.u_last = done + n == j.sweeps ? 1u : 0u;
    t.u_slots = t.u_recs + ((t.u_last && !(re && (t.u_phase + n) % re == 0u)) ? 1u : 0u);
}

__global__ void __launch_bounds__(kBatchThreads, 2) k_ahead_batch(const __grid_constant__ AheadBatchArgs a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ AheadArgs t;
    // (waits as in k_ahead; the first launch copies the lattices whose last block
    // would otherwise end in their second buffer)
    const bool early = blockIdx.x >= a.update_ctas && a.block != 0u;
    if (!early) dependent_launch_wait();
    const bool first = a.block == 0u && blockIdx.x == 0;
    if (first && threadIdx.x == 0) publish(a.done, 1u);
    if (!first || threadIdx.x == 0) dependent_launch_trigger();
    if (a.block == 0u) {
        // groups of CTAs, each for every so many-th lattice (one CTA a lattice took 200 us for
        // one of 4096^2)
        const uint32_t parts = max(1u, gridDim.x / a.d_jobs), groups = gridDim.x / parts, group = blockIdx.x / parts;
        for (uint32_t k = group; group < groups && k < a.d_jobs; k += groups) {
            const AheadJob &j = a.jobs[k];
            if (j.copy_from)
                for (uint32_t i = blockIdx.x % parts * kBatchThreads + threadIdx.x; i < j.nwords; i += parts * kBatchThreads)
                    j.even[i] = j.copy_from[i];
        }
    } else if (blockIdx.x < a.update_ctas) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *a.next_ticket = 0u;
        for (uint32_t g = blockIdx.x; g < a.u_tiles; g += a.update_ctas) {
            const uint32_t ji = find_job(a.jobs, a.u_jobs, g, &AheadJob::tile_start);
            const AheadJob &j = a.jobs[ji];
            if (threadIdx.x == 0) batch_tile_args(a, j, t);
            __syncthreads();
            const uint32_t tile = g - j.tile_start;
            if (!j.field) {
                if (j.kw == 2)
                    update_tile<kBatchThreads, 2, false, false, false, false>(t, tile, smem);
                else if (j.kw == 4)
                    update_tile<kBatchThreads, 4, false, false, false, false>(t, tile, smem);
                else
                    update_tile<kBatchThreads, 8, false, false, false, true>(t, tile, smem);
            } else if (j.kw == 2) {
                update_tile<kBatchThreads, 2, true, false, false, false>(t, tile, smem);
            } else {
                update_tile<kBatchThreads, 4, true, false, false, false>(t, tile, smem);
            }
        }
    }
    if (a.d_tickets != 0u) batch_draw_role(a, early);
}

using AheadKernel = void (*)(AheadArgs);

AheadKernel pick_kernel(const AheadPlan &p)
{
    if (p.band_rows) return p.field ? k_ahead_band<true> : k_ahead_band<false>;
    if (p.field)
        return p.kw == 2 ? k_ahead<2, false, true, false>
               : p.kw != 4 ? nullptr
               : p.two     ? k_ahead<4, false, true, true>
                           : k_ahead<4, false, true, false>;
    if (p.warp) return k_ahead<2, true, false, false>;
    return p.kw == 2   ? k_ahead<2, false, false, false>
           : p.kw == 4 ? k_ahead<4, false, false, false>
           : p.kw == 8 ? k_ahead<8, false, false, true>
                       : nullptr;
}

constexpr int kMaxDevices = 64;
constexpr int kMaxSmem = 200 * 1024;
constexpr size_t kTicketBytes = 256;  // the ticket counters at the start of the scratch
constexpr size_t kDoneWord = 32;      // and the cluster form's count of updates, on a line of its own

FastDiv fast_div(uint32_t d)
{
    FastDiv f{};
    f.shift = 24;
    while ((1u << (f.shift - 24)) < d) ++f.shift;
    f.mul = (uint32_t)(((1ull << f.shift) + d - 1) / d);
    return f;
}

// SMs of the current device; a kernel's shared-memory limit is raised once per device.
cudaError_t prepare_device(AheadKernel kern, uint32_t which, int *sms)
{
    static std::atomic<int> sms_of[kMaxDevices], ready[kMaxDevices];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool cached = dev >= 0 && dev < kMaxDevices;
    *sms = cached ? sms_of[dev].load(std::memory_order_relaxed) : 0;
    if (*sms <= 0) {
        e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        if (cached) sms_of[dev].store(*sms, std::memory_order_relaxed);
    }
    if (!cached || !(ready[dev].load(std::memory_order_acquire) >> which & 1)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return e;
        if (cached) ready[dev].fetch_or(1 << which, std::memory_order_release);
    }
    return cudaSuccess;
}

}  // namespace

// The plan by size.  L <= 192: one CTA holds the lattice, in registers for the
// whole block, and blocks are long: 256 sweeps a launch, at L = 64 1024, whose draws take
// the whole GPU 2 us (256: calls queued on 8 streams of their own, 1000 sweeps 0.30 ms and
// 0.22, 10^5 16.1 and 12.2; one stream 11.6 and 11.0).
// Above, tiles of full rows: the taller the halo, the fewer launches and the more
// redundant rows; a tile and its halo are at most 4096 words of a colour (8 rows a
// thread), so that both shrink as rows get longer.  Measured (us for a call, M/E
// every tenth sweep), tile and halo:
//   L =  256, 1000 sweeps: 32 + 64: 352, 32 + 32: 405, 64 + 32: 425, one CTA: 416
//   L =  512, 1000 sweeps: 32 + 64: 461, 32 + 32: 482, 64 + 32: 558 (every sweep: 32 + 32 is 8 % ahead)
//   L = 1024,  500 sweeps: 64 + 32: 447, 32 + 32: 470, 32 + 16: 607
//   L = 2048,  200 sweeps: 64 + 32: 606, 64 + 16: 630, 32 + 16: 659
//   L = 4096,  200 sweeps: 32 + 16: 2225, 16 + 8: 2399
// Above 8192 tiles are parts of rows and a launch takes a band of rows: the masks of
// all would be 64 times the lattice a block.  Measured against the step kernels (two
// launches a sweep): L = 65536, 4 sweeps 12252 -> 11083 us (1550 attempts per ns), 8 sweeps
// 24481 -> 21766; 16384, 40 sweeps 8510 -> 6808; 8256, 40 sweeps 2456 -> 1804.  Two CTAs
// of the largest tiles share a SM, and with draws (L = 2048, 200 sweeps: 606 us with
// one, 585 with two; 4096 2225 and 2137; 8192, 40 sweeps 1848 and 1748).  In a field (20
// bytes of masks a word and step instead of 8) the bands start above 4096, for tiles of
// half the words.  Measured with M/E every sweep, the field step kernel (L = 64 .. 512:
// the one-launch field kernels) against this form: 200 sweeps of L = 64 547 -> 102 us, 512
// 1384 -> 249, 704 5568 -> 347, 2048 5593 -> 922, 20 of 4096 689 -> 335, 40 of 8256 3769 ->
// 2620, 8 of 32768 9718 -> 7849.  There too two CTAs share a SM above L = 1024 (with one,
// and items of 4 sweeps: 2048 1018, 4096 200 sweeps 3745 and 3225, 32768 9119; below, where
// the chain of steps counts, one CTA is faster: 1024 567 and 622).  min_sweeps: a call
// has one launch more than it has blocks, and the one-launch forms (L = 64, 128, 256) and
// two step launches per sweep (above) are as fast on shorter calls.  Measured at the edges,
// form of the configuration and this form, M/E every sweep (and none): L = 1024, 5 sweeps 60
// -> 46 us (45 -> 34); 1536, 5 57 -> 57 (45 -> 46), 6 69 -> 65 (51 -> 50); 1984, 6 73 -> 77
// (60 -> 60), 7 85 -> 78 (67 -> 69), 9 96 -> 78 (82 -> 81); 2048, 10 100 -> 88; 8256, 4 273
// -> 255; 32768, 5 3867 -> 3671.  In a field: 2048, 1 54 -> 52 (42 -> 44), 2 83 -> 59; 4096, 4
// 161 -> 128; 4160, 4 165 -> 134, 6 225 -> 166; 8256, 4 407 -> 402, 6 600 -> 477; 32768, 4
// 4882 -> 4012.
AheadPlan ahead_plan(uint64_t L, bool field)
{
    AheadPlan p{};
    if (L % 64 != 0 || L < 64) return p;
    const uint32_t wc = (uint32_t)(L / 64);
    p.field = field;
    if (L > (field ? 4096 : 8192)) {
        // tiles of 64 rows (80 with the halo of a block of 4 sweeps, 10 runs of 8; in a field
        // 32 rows, 12 runs of 4) and as many words as fill 512 threads with two more, in
        // equal parts of a row; bands of about 2^20 words, at least 512 rows (16 more are
        // drawn twice)
        p.kw = field ? 4 : 8;
        p.two = true;
        p.tile_rows = field ? 32 : 64;
        p.halo = 8;
        p.block_sweeps = 4;
        p.min_sweeps = 4;
        const uint32_t words = kThreads / ((p.tile_rows + 2 * p.halo) / p.kw) - 2;
        p.tiles_x = (wc + words - 1) / words;
        p.tile_words = (wc + p.tiles_x - 1) / p.tiles_x;
        p.band_rows = std::min((uint32_t)L, std::max(512u, (1u << 20) / wc / 64 * 64));
        p.mask_bytes = (size_t)2 * p.block_sweeps * std::min<uint64_t>(L, p.band_rows + 2 * p.halo) * wc * (field ? 20 : 8);
        return p;
    }
    if (L <= 192) {
        p.tile_rows = (uint32_t)L;
        p.halo = 0;
    } else {
        p.tile_rows = L >= 1024 && L <= 2048 ? 64 : L <= 4096 ? 32 : 16;
        p.halo = L <= 256 ? 64 : L <= 2048 ? 32 : L <= 4096 ? 16 : 8;
        if (field) {  // at most 2048 words of a colour: five planes of masks take the shared memory of 4 rows a thread
            p.tile_rows = L <= 1024 || L > 2048 ? std::min(p.tile_rows, L <= 1024 ? 64u : 16u) : 32u;
            p.halo = std::min(p.halo, L <= 1024 ? 32u : L <= 2048 ? 16u : 8u);
        }
    }
    p.warp = L == 64 && !field;
    p.block_sweeps = p.halo ? p.halo / 2 : p.warp ? 1024 : 256;
    p.min_sweeps = field ? (L <= 512 && (L & (L - 1)) == 0 ? 5 : L > 2048 ? 4 : 1)
                         : L == 64 ? 200 : L == 128 ? 100 : L == 256 ? 10 : L < 1024 ? 3 : L < 1536 ? 5 : L < 1856 ? 6 : L < 2048 ? 9 : 10;
    const uint32_t rows = p.tile_rows + 2 * p.halo, most = p.halo ? kThreads : kThreads / 2;
    for (p.kw = 2; rows / p.kw * wc > most;) p.kw *= 2;
    p.two = p.kw == 8 || (field && p.kw == 4 && L > 1024);
    p.tiles = (uint32_t)(L / p.tile_rows);
    // one tile a CTA, or several the same number each: of 66 tiles 2 on two CTAs take
    // twice as long as the others; 128 tiles (L = 4096) on 64 CTAs 2137 us, on 128 2228
    // (a CTA that updates draws nothing before the launch before has ended: fewer of
    // them where a CTA has an SM to itself)
    const uint32_t most_ctas = p.two ? 128 : 64;
    const uint32_t each = p.tiles <= 96 ? 1 : std::max(2u, (p.tiles + most_ctas - 1) / most_ctas);
    p.update_ctas = (p.tiles + each - 1) / each;
    p.step_bytes = (uint32_t)(L * wc * (field ? 20 : 8));
    p.mask_bytes = (size_t)2 * p.block_sweeps * p.step_bytes;
    p.snap_bytes = L <= 2048 ? (size_t)p.block_sweeps * L * wc * 8 : 0;
    return p;
}

namespace {

// The mask planes' thresholds of a lattice, and in a field what step_run_field needs.
template <typename A>
void set_planes(A &a, const ising_lattice *h, bool field)
{
    if (!field) {
        a.thr[0] = h->thr4;
        a.thr[1] = h->thr8;
        return;
    }
    const FieldTable &ft = h->field;
    const uint32_t i = h->H > 0.0 ? 1 : 0;  // the spin direction of sigma = +1
    const uint32_t kA = i ? ft.k_up : ft.k_dn, kB = i ? ft.k_dn : ft.k_up;
    const uint32_t *const plus = ft.thr + 8 * i, *const minus = ft.thr + 8 * (1 - i);
    a.thr[0] = plus[0];
    a.thr[1] = plus[1];
    a.thr[2] = plus[2];
    a.thr[3] = kA > 3 ? plus[3] : kB > 1 ? minus[1] : 0u;
    a.thr[4] = kA > 4 ? plus[4] : kB > 0 ? minus[0] : 0u;
    a.plus3 = kA > 3 ? 0u : ~0u;
    a.plus4 = kA > 4 ? 0u : ~0u;
    a.minus0 = kB > 0 ? 0u : ~0u;
    a.minus1 = kB > 1 ? 0u : ~0u;
    a.flipped = i ? 0u : ~0u;
}

cudaError_t launch_ahead(const AheadPlan &pl, AheadArgs a, bool dependent, cudaStream_t s)
{
    const AheadKernel kern = pick_kernel(pl);
    if (!kern) return cudaErrorInvalidValue;
    int sms = 0;
    cudaError_t e = prepare_device(kern, pl.band_rows ? 16 + pl.field : pl.warp ? 0 : pl.kw / 2 + (pl.field ? 8 : 0) + (pl.field && pl.two ? 1 : 0), &sms);
    if (e != cudaSuccess) return e;
    if (pl.band_rows) a.nwords = (a.d_words + 31) / 32 * 32;  // for the tickets
    a.update_ctas = !a.u_steps ? 0u : pl.band_rows ? std::min(a.tiles, (uint32_t)sms) : pl.update_ctas;
    const uint32_t per = (a.nwords / pl.kw + 31u) & ~31u;
    a.count_ctas = a.c_slots ? std::min<uint32_t>((a.c_slots * per + kThreads - 1) / kThreads, pl.two ? 64u : 16u) : 0u;
    // 1756 attempts/ns in items of 4 sweeps, 1708 in items of 2, 1616 one by one; the masks
    // of 4 sweeps in a field do not fit the registers of two CTAs a SM
    a.d_k = a.d_sweeps % 4 == 0 && !(pl.field && pl.two) ? 4 : a.d_sweeps % 2 == 0 ? 2 : 1;
    a.d_tickets = a.d_sweeps / a.d_k * 2u * (a.nwords / 32u);
    const uint32_t early = a.update_ctas + a.count_ctas, warps = kThreads / 32u;
    const uint32_t grid = std::max(early, std::min<uint32_t>((uint32_t)sms * (pl.two ? 2u : 1u), early + (a.d_tickets + warps - 1) / warps));
    const size_t smem = !a.u_steps ? 0
                        : pl.warp  ? kWarpStages * kChunk * 512
                                   : (stages_of(pl.kw, pl.field, pl.two) * (pl.field ? 20 : 8) + 8) * pl.kw * kThreads + (a.u_snaps ? 0 : (size_t)a.u_slots * 8);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

}  // namespace

size_t ahead_bytes(const AheadPlan &pl, uint64_t L)
{
    return kTicketBytes + (pl.cluster ? kClusterBuffers : kBuffers) * pl.mask_bytes + 2 * pl.snap_bytes + (pl.halo && !pl.cluster ? (size_t)(L * L / 8) : 0);
}

// Blocks of 4 sweeps (the rest of a division by 4 first), each in bands of rows.
static cudaError_t band_sweeps(const AheadPlan &pl, AheadArgs a, char *masks, unsigned int *tickets, uint64_t *spins, uint64_t *other,
                               size_t bytes, uint64_t t0, uint64_t nsweeps, uint64_t full, cudaStream_t s)
{
    const uint32_t L = a.L, halo = pl.halo, bands = (L + pl.band_rows - 1) / pl.band_rows;
    const uint64_t first = nsweeps % full ? nsweeps % full : full, nblocks = 1 + (nsweeps - first + full - 1) / full;
    uint64_t *src = spins, *dst = other;
    cudaError_t e = cudaSuccess;
    if (nblocks % 2 == 1) {
        e = cudaMemcpyAsync(other, spins, bytes, cudaMemcpyDeviceToDevice, s);
        std::swap(src, dst);
    }
    a.tile_words = pl.tile_words;
    a.tiles_x = pl.tiles_x;
    a.by_tw = fast_div(pl.tile_words + 2);
    const uint32_t re = a.record_every;
    uint64_t i = 0, rec_done = 0, done = 0;  // items before; samples and sweeps of the blocks before the one updated
    for (uint64_t b = 0; b <= nblocks; ++b) {
        const uint64_t drawn = b == 0 ? 0 : first + (b - 1) * full;
        for (uint32_t k = 0; k < bands && e == cudaSuccess; ++k, ++i) {
            // draw band k of block b, update the band before
            if (i > 0) {
                const uint64_t ub = k ? b : b - 1, t = t0 + done, n = ub == 0 ? first : full;
                const uint32_t uk = k ? k - 1 : bands - 1, rows = std::min(pl.band_rows, L - uk * pl.band_rows);
                a.u_steps = (uint32_t)(2 * n);
                a.src = src;
                a.dst = dst;
                a.u_masks = masks + ((i - 1) % kBuffers) * pl.mask_bytes;
                a.u_row0 = uk * pl.band_rows;
                a.u_mask_row0 = bands == 1 ? 0u : (a.u_row0 + L - halo) % L;
                a.u_words = (bands == 1 ? L : rows + 2 * halo) * a.wc;
                a.tiles = rows / pl.tile_rows * pl.tiles_x;
                a.u_phase = re ? (uint32_t)(t % re) : 0u;
                a.u_recs = re ? (uint32_t)((t + n) / re - t / re) : 0u;
                a.u_slot0 = (uint32_t)rec_done;
                a.u_last = done + n == nsweeps;
                a.u_slots = a.u_recs + ((a.u_last && !(re && (t + n) % re == 0)) ? 1u : 0u);
                if (uk == bands - 1) {  // the block's last band
                    std::swap(src, dst);
                    done += n;
                    rec_done += a.u_recs;
                }
            }
            if (b == nblocks && k > 0) return e;
            a.d_sweeps = b == nblocks ? 0u : (uint32_t)(b == 0 ? first : full);
            if (a.d_sweeps) {
                const uint32_t row0 = k * pl.band_rows, rows = std::min(pl.band_rows, L - row0);
                a.d_t0 = (uint32_t)(t0 + drawn);
                a.d_row0 = bands == 1 ? 0u : (row0 + L - halo) % L;
                a.d_words = (bands == 1 ? L : rows + 2 * halo) * a.wc;
                a.by_group = fast_div((a.d_words + 31) / 32);
            }
            a.d_masks = masks + (i % kBuffers) * pl.mask_bytes;
            a.d_ticket = tickets + i % 4;
            a.next_ticket = tickets + (i + 2) % 4;
            e = launch_ahead(pl, a, i > 0, s);
        }
        if (e != cudaSuccess) break;
    }
    return e;
}

static uint32_t cluster_threads(const AheadPlan &p, uint32_t wc) { return (((p.tile_rows + 2 * p.halo) / 2 * wc + 31u) & ~31u) + 32u; }
static uint32_t cluster_smem_of(const AheadPlan &p, uint32_t wc) { return cluster_smem(p.tile_rows + 2 * p.halo, p.halo, wc, p.stages); }

// Whether this GPU (a partition may not) has room for a cluster of the plan.
static bool cluster_fits(const AheadPlan &pl, uint32_t wc)
{
    static std::atomic<signed char> known[kMaxDevices][17];  // by device, CTAs
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return false;
    std::atomic<signed char> &fits = known[dev][pl.tiles];
    if (fits.load(std::memory_order_acquire) == 0) {
        const AheadKernel kern = k_ahead_cluster;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(pl.tiles);
        cfg.blockDim = dim3(cluster_threads(pl, wc));
        cfg.dynamicSmemBytes = cluster_smem_of(pl, wc);
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = pl.tiles;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int n = 0;
        const bool ok = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) == cudaSuccess &&
                        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                        cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n >= 1;
        if (!ok) cudaGetLastError();
        fits.store(ok ? 1 : -1, std::memory_order_release);
    }
    return fits.load(std::memory_order_acquire) > 0;
}

// Calls of 192 sweeps and more: the first block's draws overlap nothing and the blocks
// start short, so that calls of 64 and 128 take 72 and 100 us at 512 and with tiles
// 65 and 93.
AheadPlan cluster_plan(uint64_t L, uint64_t nsweeps)
{
    AheadPlan p{};
    if (L % 64 != 0 || L < 320 || L > 512 || nsweeps < 192) return p;
    const uint32_t wc = (uint32_t)(L / 64);
    p.cluster = true;
    p.kw = 2;
    p.tile_rows = 32;
    p.halo = 16;
    p.tiles = p.update_ctas = (uint32_t)(L / p.tile_rows);
    p.stages = kClusterStages;
    p.block_sweeps = 128;  // (256: 1 % faster at 512 with twice the scratch; 64: 8 % slower)
    p.min_sweeps = 192;
    p.step_bytes = (uint32_t)(L * wc * 8);
    p.mask_bytes = (size_t)2 * p.block_sweeps * p.step_bytes;
    p.snap_bytes = (size_t)p.block_sweeps * L * wc * 8;
    if (!cluster_fits(p, wc)) p.kw = 0;
    return p;
}

// The launches of the cluster form (k_ahead_draw and k_ahead_cluster in turn).
static cudaError_t cluster_sweeps(const AheadPlan &pl, AheadArgs a, char *masks, char *snaps, unsigned int *tickets, uint64_t *spins,
                                  uint64_t t0, uint64_t nsweeps, uint64_t full, cudaStream_t s)
{
    const AheadKernel kern = k_ahead_cluster, draw = k_ahead_draw;
    int sms = 0;
    cudaError_t e = prepare_device(draw, 18, &sms);
    if (e != cudaSuccess) return e;
    a.stages = pl.stages;
    a.src = a.dst = spins;
    a.update_ctas = pl.tiles;
    a.done = tickets + kDoneWord;
    cudaLaunchAttribute attr[2]{};
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = pl.tiles;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t dc{}, uc{};
    dc.blockDim = dim3(kThreads);
    uc.gridDim = dim3(pl.tiles);
    uc.blockDim = dim3(cluster_threads(pl, a.wc));
    uc.dynamicSmemBytes = cluster_smem_of(pl, a.wc);
    dc.stream = uc.stream = s;
    dc.attrs = uc.attrs = attr;
    uc.numAttrs = 2;
    // Blocks start short, since nothing overlaps the first one's draws, and with the rest of
    // a division by 4 (items of 4 sweeps are the cheapest to draw).
    uint64_t left = nsweeps, done = 0, rec_done = 0, grow = std::min<uint64_t>(full, 32);
    struct Counted {
        uint32_t slots = 0, recs = 0, slot0 = 0, last = 0;
        const uint32_t *snaps = nullptr;
    } counted[2];  // of the blocks before
    const uint32_t re = a.record_every;
    for (uint64_t b = 0;; ++b) {
        uint64_t n = std::min(left, grow);
        if (left % 4 && n < left && n > 4) n -= 4 - left % 4;
        grow = std::min<uint64_t>(full, 2 * grow);
        left -= n;
        const Counted c = counted[0];
        if (n == 0 && c.slots == 0) {
            if (counted[1].slots == 0) return cudaSuccess;
            counted[0] = counted[1];
            counted[1] = Counted{};
            continue;
        }
        a.c_slots = c.slots;
        a.c_recs = c.recs;
        a.c_slot0 = c.slot0;
        a.c_last = c.last;
        a.c_snaps = c.snaps;
        a.c_wait = n == 0;
        // block b - 2: its counts, and the buffer of masks that its update read
        a.d_after = n != 0 && b >= 2 ? (uint32_t)(b - 1) : 0u;
        a.d_t0 = (uint32_t)(t0 + done);
        a.d_sweeps = (uint32_t)n;
        a.d_masks = masks + (b % kClusterBuffers) * pl.mask_bytes;
        a.d_ticket = tickets + b % 4;
        a.next_ticket = tickets + (b + 2) % 4;
        a.d_k = n % 4 == 0 ? 4 : n % 2 == 0 ? 2 : 1;
        a.d_tickets = a.d_sweeps / a.d_k * 2u * (a.nwords / 32u);
        const DrawGrid g = draw_grid((uint32_t)sms, kThreads, a.c_slots, a.nwords / pl.kw, a.d_tickets);
        a.count_ctas = g.count_ctas;
        dc.gridDim = dim3(g.grid);
        dc.numAttrs = b > 0 ? 1 : 0;
        if ((e = cudaLaunchKernelEx(&dc, draw, a)) != cudaSuccess) return e;
        counted[0] = counted[1];
        counted[1] = Counted{};
        if (n == 0) continue;
        const uint64_t t = t0 + done;
        a.u_steps = (uint32_t)(2 * n);
        a.u_step0 = (uint32_t)(2 * done);
        a.u_before = (uint32_t)b;
        a.u_masks = a.d_masks;
        a.u_snaps = reinterpret_cast<uint32_t *>(snaps + (b % 2) * pl.snap_bytes);
        a.u_phase = re ? (uint32_t)(t % re) : 0u;
        a.u_recs = re ? (uint32_t)((t + n) / re - t / re) : 0u;
        a.u_last = left == 0;
        a.u_slots = a.u_recs + ((a.u_last && !(re && (t + n) % re == 0)) ? 1u : 0u);
        counted[1].slots = a.u_slots;
        counted[1].recs = a.u_recs;
        counted[1].slot0 = (uint32_t)rec_done;
        counted[1].last = a.u_last;
        counted[1].snaps = a.u_snaps;
        if ((e = cudaLaunchKernelEx(&uc, kern, a)) != cudaSuccess) return e;
        done += n;
        rec_done += a.u_recs;
    }
}

cudaError_t ahead_sweeps(ising_lattice *h, const AheadPlan &pl, void *lattice, uint64_t L, uint64_t t0, uint64_t nsweeps, uint32_t record_every,
                         uint64_t nrec, unsigned int *err, uint32_t hold_step, uint64_t max_block)
{
    const uint32_t full = (uint32_t)std::min<uint64_t>(pl.block_sweeps, max_block);
    const size_t bytes = (size_t)(L * L / 8);
    unsigned int *const tickets = static_cast<unsigned int *>(h->scratch.p);
    char *const masks = static_cast<char *>(h->scratch.p) + kTicketBytes;
    char *const snaps = masks + (pl.cluster ? kClusterBuffers : kBuffers) * pl.mask_bytes;
    uint64_t *const spins = static_cast<uint64_t *>(lattice);
    uint64_t *const other = pl.halo ? reinterpret_cast<uint64_t *>(snaps + 2 * pl.snap_bytes) : spins;
    AheadArgs a{};
    a.key = h->key;
    a.step_bytes = pl.step_bytes;
    set_planes(a, h, pl.field);
    a.c3base = h->stream_id << 1;
    a.L = (uint32_t)L;
    a.wc = a.L / 64;
    a.by_wc = fast_div(a.wc);
    if (!pl.band_rows) {
        a.nwords = a.L * a.wc;
        a.by_group = fast_div(a.nwords / 32);
    }
    a.tiles = pl.tiles;
    a.tile_rows = pl.tile_rows;
    a.halo = pl.halo;
    a.record_every = record_every;
    a.acc = h->d_acc;
    a.final_acc = h->d_acc + 2 * nrec;
    a.err = err;
    a.hold_step = hold_step;
    if (pl.cluster) {
        const cudaError_t e = cudaMemsetAsync(tickets, 0, kTicketBytes, h->stream);
        return e != cudaSuccess ? e : cluster_sweeps(pl, a, masks, snaps, tickets, spins, t0, nsweeps, full, h->stream);
    }
    if (pl.band_rows) {
        const cudaError_t e = cudaMemsetAsync(tickets, 0, kTicketBytes, h->stream);
        return e != cudaSuccess ? e : band_sweeps(pl, a, masks, tickets, spins, other, bytes, t0, nsweeps, full, h->stream);
    }
    // Counting in the launch after the update takes work off its chain of steps, but
    // costs a launch at the end and the snapshots' traffic: M/E every sweep, counted by
    // the tiles and from snapshots, 1000 sweeps of 256 490 and 365 us, 1000 of 512 625 and
    // 496, 200 of 2048 667 and 618, 200 of 4096 2183 and 2246; 10 sweeps of 4096 165 and
    // 203.
    const bool snapshots = pl.warp || (nsweeps >= 32 && L <= 2048);
    // Blocks.  Items of 4 sweeps are the cheapest to draw, so a call that is long
    // enough starts with the rest of a division by 4.  Where an update takes long
    // (one CTA holds the lattice), blocks start short, but for the cheap draws of L = 64:
    // nothing overlaps the first one's draws.
    uint64_t drawn = 0, done = 0, rec_done = 0, prev = 0, grow = pl.halo || pl.warp ? full : std::min<uint64_t>(full, 32);
    auto next_block = [&]() -> uint64_t {
        const uint64_t left = nsweeps - drawn;
        if (full % 4 != 0 || (left <= 7 && L < 2048)) return std::min<uint64_t>(left, full);
        if (left % 4) return left % 4;
        if (pl.halo && left % full) return left % full;
        const uint64_t n = std::min(left, grow);
        grow = std::min<uint64_t>(full, 4 * grow);
        return n;
    };
    uint64_t nblocks = 0;
    for (; drawn < nsweeps; ++nblocks) drawn += next_block();
    drawn = 0;
    grow = pl.halo || pl.warp ? full : std::min<uint64_t>(full, 32);
    cudaError_t e = cudaMemsetAsync(tickets, 0, kTicketBytes, h->stream);
    if (e != cudaSuccess) return e;
    const uint64_t *src = spins;
    if (pl.halo && nblocks % 2 == 1) {
        e = cudaMemcpyAsync(other, spins, bytes, cudaMemcpyDeviceToDevice, h->stream);
        if (e != cudaSuccess) return e;
        src = other;
    }
    // launch b draws block b, updates block b - 1 and counts the snapshots of block b - 2
    for (uint64_t b = 0; b < nblocks + (snapshots ? 2 : 1); ++b) {
        const uint64_t n = drawn < nsweeps ? next_block() : 0;
        a.c_slots = snapshots ? a.u_slots : 0u;
        a.c_recs = a.u_recs;
        a.c_slot0 = a.u_slot0;
        a.c_last = a.u_last;
        a.c_snaps = a.u_snaps;
        a.u_steps = (uint32_t)(2 * prev);
        a.u_recs = a.u_slots = a.u_last = 0u;
        if (prev) {
            const uint64_t t = t0 + done;
            a.u_step0 = (uint32_t)(2 * done);
            a.src = src;
            a.dst = src == spins ? other : spins;
            a.u_masks = masks + ((b - 1) % kBuffers) * pl.mask_bytes;
            a.u_snaps = snapshots ? reinterpret_cast<uint32_t *>(snaps + (b % 2) * pl.snap_bytes) : nullptr;
            a.u_phase = record_every ? (uint32_t)(t % record_every) : 0u;
            a.u_recs = record_every ? (uint32_t)((t + prev) / record_every - t / record_every) : 0u;
            a.u_slot0 = (uint32_t)rec_done;
            a.u_last = done + prev == nsweeps;
            a.u_slots = a.u_recs + ((a.u_last && !(record_every && (t + prev) % record_every == 0)) ? 1u : 0u);
            src = a.dst;
            done += prev;
            rec_done += a.u_recs;
        }
        a.d_t0 = (uint32_t)(t0 + drawn);
        a.d_sweeps = (uint32_t)n;
        a.d_masks = masks + (b % kBuffers) * pl.mask_bytes;
        a.d_ticket = tickets + b % 4;
        a.next_ticket = tickets + (b + 2) % 4;
        if (!a.u_steps && !n && !a.c_slots) break;
        if ((e = launch_ahead(pl, a, b > 0, h->stream)) != cudaSuccess) return e;
        drawn += n;
        prev = n;
    }
    return cudaSuccess;
}

// ------------------------------------------------------------ batch, host --
namespace {

// Lattices up to this many words of a colour are one tile (L <= 256, in a field 192):
// 128 lattices of 256^2, 500 sweeps, in one tile each 3176 us, in four with halos 3685;
// 16 of 320^2 877 and 773; 16 of 256^2 in a field (with 16 of 512^2) 2451 and 2287.
uint32_t whole_words(const AheadJob &j) { return j.field ? 576 : 1024; }

// The tiles of a lattice in a batch for blocks of s sweeps: the lattice, or full rows
// with halos, at most 8 rows a thread (in a field 4).  False if there are none.
bool batch_tiles(AheadJob &j, uint32_t s)
{
    const uint32_t most = kBatchThreads * (j.field ? 4 : 8);
    j.block_sweeps = s;
    if (j.nwords <= whole_words(j)) {
        j.tile_rows = j.L;
        j.halo = 0;
    } else {
        j.halo = 2 * s;
        j.tile_rows = 0;
        for (uint32_t t : {64u, 32u, 16u})
            if (t >= j.halo && j.L % t == 0 && (t + 2 * j.halo) * j.wc <= most) {
                j.tile_rows = t;
                break;
            }
        if (!j.tile_rows) return false;
    }
    const uint32_t rows = j.tile_rows + 2 * j.halo;
    for (j.kw = 2; rows / j.kw * j.wc > kBatchThreads;) j.kw *= 2;
    return rows * j.wc <= most;
}

}  // namespace

// Blocks: the shortest (4 sweeps) for large lattices; longer ones for small lattices,
// whose steps take as long but draw less, and where all together would not fill the
// GPU for some 40 us a launch.
bool AheadBatch::plan(const std::vector<ising_lattice *> &hs, const std::vector<uint64_t> &sweeps,
                      const std::vector<uint32_t> &record_every)
{
    const size_t n = hs.size();
    jobs.assign(n, AheadJob{});
    std::vector<uint32_t> cap(n);
    double work = 0;
    for (size_t i = 0; i < n; ++i) {
        AheadJob &j = jobs[i];
        const ising_lattice *h = hs[i];
        if (h->L > 4096) return false;
        j.key = h->key;
        set_planes(j, h, h->H != 0.0);
        j.c3base = h->stream_id << 1;
        j.L = (uint32_t)h->L;
        j.wc = j.L / 64;
        j.nwords = j.L * j.wc;
        j.by_wc = fast_div(j.wc);
        j.by_group = fast_div(j.nwords / 32);
        j.field = h->H != 0.0;
        j.step_bytes = j.nwords * (j.field ? 20 : 8);
        j.sweeps = (uint32_t)sweeps[i];
        j.record_every = record_every[i];
        j.index = (uint32_t)i;
        for (cap[i] = j.nwords <= whole_words(j) ? 64 : 16; cap[i] >= 4 && !batch_tiles(j, cap[i]);) cap[i] /= 2;
        if (cap[i] < 4) return false;
        uint32_t s = 4;
        while (s < cap[i] && s < j.sweeps && (uint64_t)2 * s * j.L * j.L <= (4u << 20)) s *= 2;
        j.block_sweeps = s;
        work += (double)s * j.L * j.L;
    }
    for (bool grown = true; work < (double)(64u << 20) && grown;) {
        grown = false;
        for (size_t i = 0; i < n; ++i)
            if (jobs[i].block_sweeps < cap[i] && jobs[i].block_sweeps < jobs[i].sweeps) {
                work += (double)jobs[i].block_sweeps * jobs[i].L * jobs[i].L;
                jobs[i].block_sweeps *= 2;
                grown = true;
            }
    }
    size_t bytes = 0, cnt_slots = 0;
    smem = 0;
    for (AheadJob &j : jobs) {
        if (!batch_tiles(j, j.block_sweeps)) return false;
        j.nblocks = (j.sweeps + j.block_sweeps - 1) / j.block_sweeps;
        j.mask_bytes = (size_t)2 * j.block_sweeps * j.step_bytes;
        bytes += kBuffers * j.mask_bytes + (j.halo ? (size_t)j.nwords * 8 : 0);
        cnt_slots = std::max<size_t>(cnt_slots, j.block_sweeps + 1);
        smem = std::max<size_t>(smem, (size_t)(stages_of(j.kw, j.field, j.kw == 8) * (j.field ? 20 : 8) + 8) * j.kw * kBatchThreads);
    }
    smem += cnt_slots * 8;
    std::stable_sort(jobs.begin(), jobs.end(), [](const AheadJob &x, const AheadJob &y) { return x.nblocks > y.nblocks; });
    uint64_t tiles = 0, tickets = 0;
    for (AheadJob &j : jobs) {
        j.tile_start = (uint32_t)tiles;
        j.ticket_start = (uint32_t)tickets;
        tiles += j.L / j.tile_rows;
        tickets += (uint64_t)(j.block_sweeps / 4) * 2 * (j.nwords / 32);
    }
    if (tickets >= (1ull << 31)) return false;
    total_tiles = (uint32_t)tiles;
    total_tickets = (uint32_t)tickets;
    table_bytes = (kTicketBytes + n * sizeof(AheadJob) + 255) & ~(size_t)255;
    scratch_bytes = table_bytes + bytes;
    return true;
}

cudaError_t AheadBatch::upload(void *scratch, const std::vector<ising_lattice *> &hs,
                               const std::vector<unsigned long long *> &acc, const std::vector<unsigned long long *> &final_acc,
                               cudaStream_t s)
{
    d_scratch = static_cast<char *>(scratch);
    char *at = d_scratch + table_bytes;
    for (AheadJob &j : jobs) {
        ising_lattice *h = hs[j.index];
        uint64_t *const spins = static_cast<uint64_t *>(h->d_spins);
        j.masks = at;
        at += kBuffers * j.mask_bytes;
        uint64_t *const other = j.halo ? reinterpret_cast<uint64_t *>(at) : spins;
        if (j.halo) at += (size_t)j.nwords * 8;
        const bool swap = j.halo && j.nblocks % 2 == 1;  // the last block ends in the lattice
        j.even = swap ? other : spins;
        j.odd = swap ? spins : other;
        j.copy_from = swap ? spins : nullptr;
        j.acc = acc[j.index];
        j.final_acc = final_acc[j.index];
    }
    cudaError_t e = cudaMemcpyAsync(d_scratch + kTicketBytes, jobs.data(), jobs.size() * sizeof(AheadJob), cudaMemcpyHostToDevice, s);
    return e == cudaSuccess ? cudaStreamSynchronize(s) : e;
}

cudaError_t AheadBatch::enqueue(const uint32_t *d_t0, unsigned int *d_err, cudaStream_t s)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_ahead_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem / 2);
    unsigned int *const tickets = reinterpret_cast<unsigned int *>(d_scratch);
    if (e == cudaSuccess) e = cudaMemsetAsync(tickets, 0, kTicketBytes, s);
    if (e != cudaSuccess) return e;
    AheadBatchArgs a{};
    a.jobs = reinterpret_cast<const AheadJob *>(d_scratch + kTicketBytes);
    a.t0 = d_t0;
    a.done = tickets + kDoneWord;
    a.err = d_err;
    size_t drawing = jobs.size(), updating = 0;  // the first so many jobs have a block b, a block b - 1
    for (uint32_t b = 0;; ++b) {
        updating = b ? drawing : 0;
        while (drawing && jobs[drawing - 1].nblocks <= b) --drawing;
        if (!drawing && !updating) return cudaSuccess;
        a.block = b;
        a.d_jobs = (uint32_t)drawing;
        a.u_jobs = (uint32_t)updating;
        a.d_tickets = drawing == jobs.size() ? total_tickets : jobs[drawing].ticket_start;
        a.u_tiles = updating == 0 ? 0u : updating == jobs.size() ? total_tiles : jobs[updating].tile_start;
        a.update_ctas = std::min<uint32_t>(a.u_tiles, (uint32_t)sms);
        a.d_ticket = tickets + b % 4;
        a.next_ticket = tickets + (b + 2) % 4;
        const uint32_t warps = kBatchThreads / 32;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(std::max(1u, std::min(2 * (uint32_t)sms, a.update_ctas + (a.d_tickets + warps - 1) / warps)));
        cfg.blockDim = dim3(kBatchThreads);
        cfg.dynamicSmemBytes = b ? smem : 0;
        cfg.stream = s;
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = b ? 1 : 0;
        if ((e = cudaLaunchKernelEx(&cfg, k_ahead_batch, a)) != cudaSuccess) return e;
    }
}

}  // namespace ising
