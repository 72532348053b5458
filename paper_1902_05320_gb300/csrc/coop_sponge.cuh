// coop_sponge.cuh -- whole sponges (Section 3.2, Eq. 11-18) on the cooperative
// state of coop.cuh, one message per warp, at any length, alignment and output
// size.  A block's words are requested before the permutation that precedes
// their absorption; they are shifted, padded and split into halves during its
// last rounds.
#pragma once

#include <cstdint>

#include "coop.cuh"
#include "runtime.cuh"
#include "sponge.cuh"

namespace kb {

// The aligned 32-bit words that hold a lane word's message bytes, as loaded (a
// word without a message byte is not loaded and reads as zero).
struct RawWord {
    uint32_t w0, w1, w2;
};

// `left`: message bytes from q on (zero or negative: none).
__device__ __forceinline__ RawWord ld_raw(const uint8_t *q, int64_t left) {
    const uintptr_t start = reinterpret_cast<uintptr_t>(q);
    const uint32_t *a = reinterpret_cast<const uint32_t *>(start & ~uintptr_t(3));
    const uint32_t o = uint32_t(start & 3);
    const uint32_t n = left >= 8 ? 8u : left > 0 ? uint32_t(left) : 0u;
    RawWord r;
    r.w0 = n ? *a : 0u;
    r.w1 = o + n > 4 ? a[1] : 0u;
    r.w2 = o + n > 8 ? a[2] : 0u;
    return r;
}

// The lane word (lo, hi) of a raw word at alignment o (its address mod 4): the
// message bytes, then the domain byte where the message ends (left bytes on), then
// zeros; `end`: the last word of the padded block, which takes 0x80.
__device__ __forceinline__ void pad_raw(const RawWord &r, uint32_t o, int64_t left, bool end, uint32_t domain,
                                        uint32_t &lo, uint32_t &hi) {
    lo = __funnelshift_r(r.w0, r.w1, 8 * o);
    hi = __funnelshift_r(r.w1, r.w2, 8 * o);
    if (left < 8) {
        const uint32_t n = left > 0 ? uint32_t(left) : 0u;
        lo &= __funnelshift_lc(0xFFFFFFFFu, 0u, 8 * n);
        hi &= n > 4 ? __funnelshift_lc(0xFFFFFFFFu, 0u, 8 * (n - 4)) : 0u;
        if (left >= 0) {
            if (left < 4) lo ^= domain << (8 * n);
            else hi ^= domain << (8 * (n - 4));
        }
    }
    if (end) hi ^= 0x80000000u;
}

// The part of a sponge whose next block is a full one too: `count` times, XORs the
// halves in e into the state and permutes, while the next block's words arrive and
// become the new e.  `next`: the first byte of the block after the one in e.  Nothing
// is padded here, and a thread's two addresses move on by a block each time
// (rate % 4 == 0).
__device__ __forceinline__ void coop_full_blocks(const Coop &c, uint32_t (&a)[2], uint32_t (&e)[2], uintptr_t next,
                                                 uint32_t rate, uint64_t count) {
    const int nwords = int(rate / 8);
    const bool have0 = c.on && c.lane(0) < nwords, have1 = c.on && c.lane(1) < nwords;
    const uint32_t *q0 = reinterpret_cast<const uint32_t *>((next + 8u * uint32_t(c.lane(0))) & ~uintptr_t(3));
    const uint32_t *q1 = reinterpret_cast<const uint32_t *>((next + 8u * uint32_t(c.lane(1))) & ~uintptr_t(3));
    const uint32_t sh = 8 * uint32_t(next & 3), step = rate / 4;
    RawWord r0{0, 0, 0}, r1{0, 0, 0};
    for (; count; --count) {
        a[0] ^= e[0];
        a[1] ^= e[1];
        if (have0) {
            r0.w0 = *q0;
            r0.w1 = q0[1];
            if (sh) r0.w2 = q0[2];
        }
        if (have1) {
            r1.w0 = *q1;
            r1.w1 = q1[1];
            if (sh) r1.w2 = q1[2];
        }
        q0 += step;
        q1 += step;
        c.permute(a, [&] {
            e[0] = c.half(__funnelshift_r(r0.w0, r0.w1, sh), __funnelshift_r(r0.w1, r0.w2, sh));
            e[1] = c.half(__funnelshift_r(r1.w0, r1.w1, sh), __funnelshift_r(r1.w1, r1.w2, sh));
        });
    }
}

// Writes bytes [0, take) of the state's rate part to dst.  Every thread of the warp
// calls it.
__device__ __forceinline__ void coop_squeeze(const Coop &c, const uint32_t (&a)[2], uint8_t *dst, uint32_t take) {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const uint32_t w = c.unhalf(a[s]);
        const uint32_t at = 8u * uint32_t(c.lane(s)) + 4u * uint32_t(c.h);
        if (c.on && at < take) {
            uint8_t *q = dst + at;
            const uint32_t nb = take - at < 4 ? take - at : 4;
            if (nb == 4 && (reinterpret_cast<uintptr_t>(q) & 3) == 0) *reinterpret_cast<uint32_t *>(q) = w;
            else
                for (uint32_t b = 0; b < nb; ++b) q[b] = uint8_t(w >> (8 * b));
        }
    }
}

// One sponge: the message of len bytes at p (PREFIX >= 0: that byte comes before
// it), dlen output bytes to dst.  Every thread of the warp calls it with the same
// arguments.  ONLY: the kernel hashes nothing else and has one such warp a block;
// the next one may then be set up at once where there are `few` blocks (few_warps),
// and from the last message block on where there are many: its blocks are placed while this
// kernel's still stand and would crowd some SMs, where such warps slow one another
// (1824 leaves of 1000 bytes a call: 63 to 96 us from run to run set up at once,
// 57.5 late; 200 ragged messages 14.4 at once, 16.8 late).
template <int PREFIX = -1, bool ONLY = false>
__device__ __forceinline__ void coop_sponge(const Coop &c, const uint8_t *p, uint64_t len, int variant, uint8_t *dst,
                                            uint32_t dlen, bool few = false) {
    constexpr int kShift = PREFIX >= 0 ? 1 : 0;  // bytes before the message
    const uint32_t rate = uint32_t(variant_rate(variant));
    const int nwords = int(rate / 8);
    const uint32_t domain = rt_domain(variant);
    const uint64_t vlen = len + kShift;
    const uint64_t nfull = vlen / rate;
    const uint32_t nsq = dlen > rate ? (dlen - 1) / rate : 0;
    const uint64_t total = nfull + 1 + nsq;  // permutations
    const uint32_t o = uint32_t((reinterpret_cast<uintptr_t>(p) - kShift) & 3);  // the same for every lane word
    if (ONLY && few) launch_next();
    uint32_t a[2] = {0, 0}, e[2] = {0, 0};
    RawWord raw[2] = {};
    int64_t left[2] = {-1, -1};
    // This thread's words of block i (i <= nfull).
    auto request = [&](uint64_t i) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int k = c.lane(s);
            raw[s] = RawWord{0, 0, 0};
            if (c.on && k < nwords) {
                const uint64_t at = i * rate + 8u * uint32_t(k);
                left[s] = int64_t(vlen - at);
                if (kShift && at == 0) raw[s] = ld_raw(p, left[s] - 1 < 7 ? left[s] - 1 : 7);
                else raw[s] = ld_raw(p + at - kShift, left[s]);
            }
        }
    };
    // Their padded halves.
    auto convert = [&](uint64_t i) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int k = c.lane(s);
            uint32_t lo = 0, hi = 0;
            if (c.on && k < nwords) {
                RawWord r = raw[s];
                uint32_t sh = o;
                if (kShift && i == 0 && k == 0) {  // bytes 0..6 of the message behind the prefix byte
                    const uint32_t om = (o + 1) & 3;
                    const uint32_t m0 = __funnelshift_r(r.w0, r.w1, 8 * om), m1 = __funnelshift_r(r.w1, r.w2, 8 * om);
                    r = RawWord{(m0 << 8) | uint32_t(PREFIX & 0xff), __funnelshift_l(m0, m1, 8), 0};
                    sh = 0;
                }
                pad_raw(r, sh, left[s], i == nfull && k == nwords - 1, domain, lo, hi);
            }
            e[s] = c.half(lo, hi);
        }
    };
    request(0);
    convert(0);
    uint64_t i = 0;
    if (nfull > 2) {
        coop_full_blocks(c, a, e, reinterpret_cast<uintptr_t>(p) + rate - kShift, rate, nfull - 1);
        i = nfull - 1;
    }
    for (; i < total; ++i) {
        a[0] ^= e[0];
        a[1] ^= e[1];
        e[0] = e[1] = 0;
        const bool more = i < nfull;
        if (ONLY && !more) launch_next();
        if (more) request(i + 1);
        c.permute(a, [&] {
            if (more) convert(i + 1);
        });
        if (i >= nfull) {  // output block i - nfull
            const uint32_t base = uint32_t(i - nfull) * rate;
            coop_squeeze(c, a, dst + base, dlen - base < rate ? dlen - base : rate);
        }
    }
}

}  // namespace kb
