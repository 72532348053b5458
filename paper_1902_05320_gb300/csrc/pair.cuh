// pair.cuh -- one sponge state in two neighbouring threads of a warp: thread h = 0
// holds the low, h = 1 the high 32-bit word of each of the 25 lanes.  For batches
// that give each SM sub-partition at most one warp this way (and less than half
// of one with a thread per message): the 180 ALU instructions of a round become 90
// per thread, and a 64-bit rotation needs the partner's word:
// (own << n) | (partner >> (32 - n)), n < 32, the same on both threads, and with the
// two words' roles exchanged for n >= 32, so 29 shuffles a round (24 of rho, 5 of
// theta) carry everything and no thread differs from its partner but in iota.
//
// Measured on GB300, us a permutation against the number of states: 2.82 up to
// 9,728 (one warp per sub-partition; a thread per state takes 4.47), 4.97 up to
// 19,456, where a thread per state still takes 4.47.  A sub-partition issues a
// shuffle per 4 cycles, 116 a round beside 180 of ALU work, so the lone warp's 243
// are latency; rotations on the multiply pipe (keccak_core.cuh) are slower here
// (3.03), since the ALU is not what binds.
#pragma once

#include <cstdint>

#include "keccak_core.cuh"
#include "runtime.cuh"
#include "sponge.cuh"

namespace kb {

__device__ __forceinline__ uint32_t pair_partner(uint32_t v) { return __shfl_xor_sync(0xffffffffu, v, 1); }

template <int N>
__device__ __forceinline__ uint32_t pair_rotl(uint32_t own) {
    if constexpr (N == 0) return own;
    const uint32_t other = pair_partner(own);
    if constexpr (N < 32) return funnel_l<N>(other, own);
    else return funnel_l<N - 32>(own, other);
}

template <int X, int Y>
__device__ __forceinline__ uint32_t pair_theta_rho_pi(const uint32_t (&S)[25], const uint32_t (&C)[5],
                                                      const uint32_t (&R)[5]) {
    constexpr int SX = (X + 3 * Y) % 5;
    constexpr int SRC = SX + 5 * X;
    return pair_rotl<rho_offset(SRC)>(xor3(S[SRC], C[(SX + 4) % 5], R[(SX + 1) % 5]));
}

template <int Y>
__device__ __forceinline__ void pair_row(const uint32_t (&S)[25], const uint32_t (&C)[5], const uint32_t (&R)[5],
                                         uint32_t (&N)[25]) {
    const uint32_t B[5] = {pair_theta_rho_pi<0, Y>(S, C, R), pair_theta_rho_pi<1, Y>(S, C, R),
                           pair_theta_rho_pi<2, Y>(S, C, R), pair_theta_rho_pi<3, Y>(S, C, R),
                           pair_theta_rho_pi<4, Y>(S, C, R)};
#pragma unroll
    for (int x = 0; x < 5; ++x) N[x + 5 * Y] = chi3(B[x], B[(x + 1) % 5], B[(x + 2) % 5]);
}

// Round ir; lo_mask = h - 1 (all ones on the threads with the low words).
__device__ __forceinline__ void pair_round(uint32_t (&S)[25], uint32_t h, uint32_t lo_mask, int ir) {
    uint32_t C[5], R[5], N[25];
#pragma unroll
    for (int x = 0; x < 5; ++x) C[x] = xor3(xor3(S[x], S[x + 5], S[x + 10]), S[x + 15], S[x + 20]);
#pragma unroll
    for (int x = 0; x < 5; ++x) R[x] = pair_rotl<1>(C[x]);
    pair_row<0>(S, C, R, N);
    pair_row<1>(S, C, R, N);
    pair_row<2>(S, C, R, N);
    pair_row<3>(S, C, R, N);
    pair_row<4>(S, C, R, N);
    // The constant's high word is bit 31 alone or nothing: a sum will do.
    N[0] = (N[0] ^ (c_rc.w[2 * ir] & lo_mask)) + c_rc.w[2 * ir + 1] * h;
#pragma unroll
    for (int i = 0; i < 25; ++i) S[i] = N[i];
}

// Keccak-f[1600]; every thread of the warp calls it.  h: which word of the lanes
// this thread holds (its lane number's last bit).  TAIL: rounds [TAIL, 24) are
// unrolled, so that the last one keeps only the lanes that are used.
template <int TAIL = 24, int UNROLL = 4>
__device__ __forceinline__ void pair_permute(uint32_t (&S)[25], uint32_t h) {
    const uint32_t lo_mask = h - 1u;
#pragma unroll 1
    for (int r = 0; r < TAIL; r += UNROLL) {
#pragma unroll
        for (int j = 0; j < UNROLL; ++j) pair_round(S, h, lo_mask, r + j);
    }
#pragma unroll
    for (int r = TAIL; r < 24; ++r) pair_round(S, h, lo_mask, r);
}

// Bytes [p, p + nvalid) as a little-endian 32-bit word, nvalid <= 4, any
// alignment; loads only the aligned words that hold a valid byte.
__device__ __forceinline__ uint32_t ld_u32_any(const uint8_t *p, uint32_t nvalid) {
    if (nvalid == 0) return 0;
    const uintptr_t start = reinterpret_cast<uintptr_t>(p);
    const uint32_t *a = reinterpret_cast<const uint32_t *>(start & ~uintptr_t(3));
    const uint32_t o = uint32_t(start & 3);
    const uint32_t w0 = *a;
    const uint32_t w1 = o + nvalid > 4 ? a[1] : 0u;
    const uint32_t v = __funnelshift_r(w0, w1, 8 * o);
    return nvalid < 4 ? v & ((1u << (8 * nvalid)) - 1u) : v;
}

// Writes bytes [0, nbytes) of the rate part to dst.
template <int RATE>
__device__ __forceinline__ void pair_squeeze(const uint32_t (&S)[25], bool active, uint32_t h, uint8_t *dst,
                                             uint32_t nbytes) {
    const bool whole = ((reinterpret_cast<uintptr_t>(dst) | nbytes) & 3) == 0;
#pragma unroll
    for (int k = 0; k < RATE / 8; ++k) {
        const uint32_t at = 8 * k + 4 * h;
        if (!active || at >= nbytes) continue;
        if (whole) {
            *reinterpret_cast<uint32_t *>(dst + at) = S[k];
        } else {
            const uint32_t nb = nbytes - at < 4 ? nbytes - at : 4;
            for (uint32_t b = 0; b < nb; ++b) dst[at + b] = uint8_t(S[k] >> (8 * b));
        }
    }
}

// A message of one block (len < RATE, dlen <= RATE; dlen <= 8 OUT lanes).  Words are
// taken whole, in part or not at all by branches on the common length.
template <int RATE, int DOMAIN, int OUT>
__device__ __forceinline__ void pair_one_block(bool active, const uint8_t *p, uint32_t len, uint8_t *dst,
                                               uint32_t dlen) {
    const uint32_t h = threadIdx.x & 1u;
    uint32_t S[25];
    const uintptr_t q = reinterpret_cast<uintptr_t>(p) + 4 * h;
    const uint32_t *w = reinterpret_cast<const uint32_t *>(q & ~uintptr_t(3));
    const uint32_t o = uint32_t(q & 3);
#pragma unroll
    for (int k = 0; k < 25; ++k) {
        S[k] = 0;
        if (k >= RATE / 8) continue;
        if (uint32_t(8 * k + 8) <= len) {
            if (active) S[k] = __funnelshift_r(w[2 * k], o ? w[2 * k + 1] : 0u, 8 * o);
        } else if (uint32_t(8 * k) <= len) {
            const uint32_t at = 8 * k + 4 * h, left = len > at ? len - at : 0;
            if (active) S[k] = ld_u32_any(p + at, left < 4 ? left : 4u);
            if (len / 4 == at / 4) S[k] ^= uint32_t(DOMAIN) << (8 * (len & 3));
        }
        if (k == RATE / 8 - 1) S[k] ^= h << 31;
    }
    pair_permute<22, 2>(S, h);
    pair_squeeze<8 * OUT>(S, active, h, dst, dlen);
}

// One sponge in the pair: the message of len bytes at p, dlen output bytes to dst.
// Every thread of the warp calls it with the same len, dlen and rate; `active` is
// false for a pair without a message.  A full block's aligned words are loaded
// before the permutation that precedes its absorption, every other word by each
// thread; at an unaligned p the threads exchange them, since state word j takes
// bytes of aligned words j and j + 1.
template <int RATE, int DOMAIN>
__device__ __forceinline__ void pair_sponge(bool active, const uint8_t *p, uint64_t len, uint8_t *dst, uint32_t dlen) {
    constexpr int kWords = RATE / 8;
    const uint32_t h = threadIdx.x & 1u;
    const uint64_t nfull = len / RATE;
    const uint32_t rem = uint32_t(len - nfull * RATE);
    const uint32_t nsq = dlen > uint32_t(RATE) ? (dlen - 1) / RATE : 0;
    const uint32_t sh = uint32_t(reinterpret_cast<uintptr_t>(p) & 3) * 8;  // the same for every block (RATE % 4 == 0)
    uint32_t S[25], w[kWords + 1];
#pragma unroll
    for (int k = 0; k < 25; ++k) S[k] = 0;
    auto fetch = [&](uint64_t i) {  // aligned words 2k + h of full block i, and the one past them for h = 0
        const uint32_t *q = reinterpret_cast<const uint32_t *>((reinterpret_cast<uintptr_t>(p) & ~uintptr_t(3)) +
                                                               i * RATE) + h;
#pragma unroll
        for (int k = 0; k < kWords; ++k) w[k] = active ? q[2 * k] : 0u;
        w[kWords] = active && sh && h == 0 ? q[2 * kWords] : 0u;
    };
    const bool unaligned = __any_sync(0xffffffffu, sh != 0);
    if (nfull) fetch(0);
    for (uint64_t i = 0; i <= nfull + nsq; ++i) {
        if (i < nfull) {
            if (unaligned) {
#pragma unroll
                for (int k = 0; k < kWords; ++k) {
                    const uint32_t next = pair_partner(h ? w[k] : w[k + 1]);  // to h = 1: word 2k + 2; to h = 0: 2k + 1
                    S[k] ^= __funnelshift_r(w[k], next, sh);
                }
            } else {
#pragma unroll
                for (int k = 0; k < kWords; ++k) S[k] ^= w[k];
            }
            if (i + 1 < nfull) fetch(i + 1);
        } else if (i == nfull) {
            launch_next();  // not before: the next kernel's blocks would crowd some SMs
#pragma unroll
            for (int k = 0; k < kWords; ++k) {
                const uint32_t at = 8 * k + 4 * h;
                const uint32_t left = rem > at ? rem - at : 0;
                uint32_t v = active ? ld_u32_any(p + nfull * RATE + at, left < 4 ? left : 4u) : 0u;
                if (rem / 4 == at / 4) v ^= uint32_t(DOMAIN) << (8 * (rem & 3));
                if (k == kWords - 1 && h) v ^= 0x80000000u;
                S[k] ^= v;
            }
        } else {
            pair_squeeze<RATE>(S, active, h, dst + (i - nfull - 1) * RATE, RATE);
        }
        pair_permute(S, h);
    }
    pair_squeeze<RATE>(S, active, h, dst + uint64_t(nsq) * RATE, dlen - nsq * RATE);
}

}  // namespace kb
