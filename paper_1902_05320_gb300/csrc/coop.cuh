// coop.cuh -- one sponge state across thirty threads of a warp: the form for
// batches too small to fill the GPU with a thread per message, and for long
// messages, where one message's chain of permutations sets the time.
//
// The state is bit-interleaved (each lane as its even and its odd bits, 32-bit
// words): a lane rotation by n is then a rotation of each half by about n/2, an
// odd n also swapping the halves, so a thread rotates its own words and the swap
// is only a matter of where they are stored.  Thread (x, h, p) holds, of column x
// and half h, rows 2p and 2p + 1 (the second row of p = 2 does not exist and
// stays zero; lanes 30 and 31 idle along).  Per round (Eq. 10):
//   theta: the parity of the thread's rows; by shuffles the three parts of C[x-1]
//          of its half and of C[x+1] of the other half, which rotated by one
//          (even half) or not at all (odd half) is its half of rot(C[x+1], 1);
//   rho:   rotations by per-thread amounts;
//   pi:    stores to shared memory at per-thread addresses;
//   chi:   the thread's rows of columns x, x+1 and x+2, loaded back;
//   iota:  the constant's half, masked to the threads of lane (0, 0).
//
// What bounds it.  Probed on GB300: a sub-partition issues one 4-byte shuffle,
// shared store or load of a warp per 4 cycles (an 8-byte load per 5 to 8), whatever
// the number of active lanes, beside latencies of 26 (shuffle) and about 25
// cycles (shared load).  So the exchanges a thread makes set latency and
// throughput alike: here 6 shuffles, 2 stores and 3 8-byte loads, 134 cycles a
// round, 1.55 us a permutation where one thread per state takes 4.47 and a lane
// per thread (18 shuffles) took 2.36.  Ten threads a state (2 shuffles, 5 stores,
// 15 loads, three states a warp) measured 1.98: better than this form and than two
// threads a state (pair.cuh) only for 12 to 18 states per SM, and by at most a
// fifth.  Sixteen-byte loads measured no faster there.
//
// Two buffers alternate, so a round's stores never meet the last round's loads
// and one warp barrier a round suffices.  The loads have no bank conflict, the
// stores two words on some banks.
#pragma once

#include <cstdint>

#include "keccak_core.cuh"

namespace kb {

// The round constants' even and odd halves.
struct CoopRcTable {
    uint32_t w[48];
};
__host__ __device__ constexpr CoopRcTable make_coop_rc() {
    CoopRcTable t{};
    for (int i = 0; i < 24; ++i) {
        t.w[2 * i] = even_half(round_constant(i));
        t.w[2 * i + 1] = odd_half(round_constant(i));
    }
    return t;
}
static __constant__ CoopRcTable c_coop_rc = make_coop_rc();

// rho_offset of lanes (0..4, y), six bits each.
__host__ __device__ constexpr uint32_t coop_rho_row(int y) {
    uint32_t v = 0;
    for (int x = 0; x < 5; ++x) v |= uint32_t(rho_offset(x + 5 * y)) << (6 * x);
    return v;
}

__device__ __forceinline__ uint32_t coop_rot(uint32_t v, uint32_t s) { return __funnelshift_l(v, v, s); }
__device__ __forceinline__ uint32_t coop_shfl(uint32_t v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ void coop_st(uint32_t a, uint32_t v) {
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void coop_ld2(uint32_t a, uint32_t (&v)[2]) {
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(a) : "memory");
}

struct Coop {
    static constexpr int kBufWords = 64;              // 60 words of a state and a place nothing reads
    static constexpr int kWarpWords = 2 * kBufWords;  // shared memory of a warp, in words

    int x, h, p;             // column, half, part
    bool on;                 // works on the state (lanes 30 and 31 do not)
    int src_m, src_p;        // first lanes of C[x-1], this half, and of C[x+1], the other
    uint32_t rot1;           // theta's rotation of the fetched half: 1 on the even half, else 0
    uint32_t rot[2];         // rho amounts
    uint32_t wr[2];          // shared addresses its rotated words go to (buffer 0)
    uint32_t rd[3];          // shared addresses of its rows of columns x, x+1, x+2 (buffer 0)
    uint32_t rc_even, rc_odd;  // masks of the round constant's halves: lane (0, 0) only

    // Word of half h of lane (x, y) within one buffer.
    __device__ __forceinline__ static uint32_t word(int x, int y, int h) { return uint32_t(12 * x + 6 * h + y); }
    // Lane index x + 5y of this thread's row s; 25 or more where the row does not exist.
    __device__ __forceinline__ int lane(int s) const { return x + 5 * (2 * p + s); }

    // warp_mem: kWarpWords words of this warp, 8-byte aligned.  Every thread of
    // the warp calls it.
    __device__ __forceinline__ explicit Coop(uint32_t *warp_mem) {
        const int t = int(threadIdx.x & 31);
        for (int i = t; i < kWarpWords; i += 32) warp_mem[i] = 0;
        __syncwarp();
        on = t < 30;
        x = on ? t / 6 : 0;
        h = on ? (t / 3) & 1 : 0;
        p = on ? t % 3 : 0;
        const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(warp_mem));
        rot1 = h ? 0u : 1u;
        src_m = 6 * ((x + 4) % 5) + 3 * h;
        src_p = 6 * ((x + 1) % 5) + 3 * (h ^ 1);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int y = 2 * p + s;
            const uint32_t rho = p == 0 ? coop_rho_row(s) : p == 1 ? coop_rho_row(2 + s) : coop_rho_row(4);
            // Even n rotates each half by n/2; odd n sends the even half to the
            // odd one by (n-1)/2, the odd to the even by (n+1)/2.
            const int n = int((rho >> (6 * x)) & 63u);
            rot[s] = uint32_t((n + (h & n & 1)) >> 1);
            // pi (Eq. 6): lane (x, y) becomes lane (y, 2x + 3y).
            wr[s] = base + 4 * (on && y < 5 ? word(y, (2 * x + 3 * y) % 5, h ^ (n & 1)) : uint32_t(kBufWords - 4));
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) rd[k] = base + 4 * word((x + k) % 5, 2 * p, h);
        rc_even = on && x == 0 && p == 0 && h == 0 ? 0xffffffffu : 0u;
        rc_odd = on && x == 0 && p == 0 && h == 1 ? 0xffffffffu : 0u;
    }

    template <int BUF>
    __device__ __forceinline__ void round(uint32_t (&a)[2], int ir) const {
        constexpr uint32_t kOff = 4u * BUF * kBufWords;
        const uint32_t rcw = (c_coop_rc.w[2 * ir] & rc_even) | (c_coop_rc.w[2 * ir + 1] & rc_odd);
        const uint32_t par = a[0] ^ a[1];  // Eq. 2
        const uint32_t q0 = coop_shfl(par, src_p), q1 = coop_shfl(par, src_p + 1), q2 = coop_shfl(par, src_p + 2);
        const uint32_t m0 = coop_shfl(par, src_m), m1 = coop_shfl(par, src_m + 1), m2 = coop_shfl(par, src_m + 2);
        const uint32_t q = coop_rot(xor3(q0, q1, q2), rot1);  // Eq. 3
        const uint32_t m = xor3(m0, m1, m2);
        coop_st(wr[0] + kOff, coop_rot(xor3(a[0], m, q), rot[0]));  // Eq. 4, rho, pi
        coop_st(wr[1] + kOff, coop_rot(xor3(a[1], m, q), rot[1]));
        __syncwarp();
        uint32_t b0[2], b1[2], b2[2];
        coop_ld2(rd[0] + kOff, b0);
        coop_ld2(rd[1] + kOff, b1);
        coop_ld2(rd[2] + kOff, b2);
        a[0] = chi3(b0[0], b1[0], b2[0]) ^ rcw;  // Eq. 7, 9
        a[1] = chi3(b0[1], b1[1], b2[1]);
    }

    // Keccak-f[1600]; every thread of the warp calls it.  work() is independent
    // of the state: its instructions fill the waits of the last four rounds.
    template <class W>
    __device__ __forceinline__ void permute(uint32_t (&a)[2], W work) const {
#pragma unroll 1
        for (int i = 0; i < 20; i += 4) {
            round<0>(a, i);
            round<1>(a, i + 1);
            round<0>(a, i + 2);
            round<1>(a, i + 3);
        }
        work();
        round<0>(a, 20);
        round<1>(a, 21);
        round<0>(a, 22);
        round<1>(a, 23);
    }

    // This thread's half of a 64-bit word (lo, hi): its bits h, h+2, h+4, ... packed.
    __device__ __forceinline__ uint32_t half(uint32_t lo, uint32_t hi) const {
        auto pack = [](uint32_t v) {  // even bits of v into the low 8 bits of each half word
            v &= 0x55555555u;
            v = (v | (v >> 1)) & 0x33333333u;
            v = (v | (v >> 2)) & 0x0F0F0F0Fu;
            return v | (v >> 4);
        };
        return __byte_perm(pack(lo >> h), pack(hi >> h), 0x6420);
    }

    // The low (h = 0) or high (h = 1) 32-bit word of the lane whose half this
    // thread holds in `own`.  Every thread of the warp calls it.
    __device__ __forceinline__ uint32_t unhalf(uint32_t own) const {
        const uint32_t other = coop_shfl(own, int(threadIdx.x & 31) + (on ? (h ? -3 : 3) : 0));
        const uint32_t e = h ? other : own, o = h ? own : other;
        uint32_t z = __byte_perm(e, o, h ? 0x7632 : 0x5410);  // 16 even bits, then 16 odd bits
        z = __byte_perm(z, z, 0x3120);
        uint32_t t;
        t = (z ^ (z >> 4)) & 0x00F000F0u; z ^= t ^ (t << 4);
        t = (z ^ (z >> 2)) & 0x0C0C0C0Cu; z ^= t ^ (t << 2);
        t = (z ^ (z >> 1)) & 0x22222222u; z ^= t ^ (t << 1);
        return z;
    }
};

}  // namespace kb
