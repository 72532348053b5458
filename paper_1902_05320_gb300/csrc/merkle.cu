// merkle.cu -- tree mode (Section 4: digests combined pairwise, level after
// level, up to one root; the paper leaves it to future work with
// reductions).
//
// Node format: leaf = SHA3-256(0x00 || leaf bytes), inner node =
// SHA3-256(0x01 || left || right); levels are reduced one at a time and an odd
// last node is carried up unchanged.  All levels are written back to back
// (leaf digests first, root last) so that callers can also take proofs.
//
// Kernels: one thread per leaf (the prefixed message is read through a
// one-byte funnel shift of the leaf's aligned words), then the levels above
// (0x01 || left || right is exactly one 65-byte block at rate 136), one thread
// per parent node: one launch per level while a level has more than kClimbPerSm
// parents per SM, and above that climbing launches that reduce up to four
// levels each with a warp per node.  Few leaves take a warp each as well.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "coop_sponge.cuh"
#include "keccak_core.cuh"
#include "runtime.cuh"
#include "sponge.cuh"

namespace kb {
namespace {

constexpr int kRate = Variant<1>::rate;   // SHA3-256
constexpr int kDomain = Variant<1>::domain;

// Lane word g of the virtual message 0x00 || leaf, built from leaf words g-1
// and g: the byte that falls off the top of word g-1 becomes byte 0 of word g.
// `carry` holds the high half of leaf word g-1 (prefix << 24 for g = 0).
__device__ __forceinline__ void prefixed_word(uint32_t &carry, uint32_t lo, uint32_t hi, uint32_t &vlo,
                                              uint32_t &vhi) {
    vlo = __funnelshift_l(carry, lo, 8);
    vhi = __funnelshift_l(lo, hi, 8);
    carry = hi;
}

// Leaves at 8-byte aligned addresses with leaf_bytes % 8 == 0.
// XORs block b of the padded message 0x00 || leaf (leaf_bytes bytes at p,
// mwords = leaf_bytes / 8 words, nfull full blocks, rem bytes in the last)
// into the state.  The prefix byte is shifted in through one-byte funnel
// shifts of the leaf's aligned 8-byte words; carry holds the byte carried
// between words (0 before block 0).
__device__ __forceinline__ void absorb_leaf_block_a8(uint32_t (&A)[25], uint32_t (&B)[25], const uint8_t *p,
                                                     uint64_t b, uint64_t nfull, uint32_t rem, uint64_t mwords,
                                                     uint32_t &carry) {
    const uint64_t g0 = b * (kRate / 8);
    if (b < nfull) {
#pragma unroll
        for (int k = 0; k < kRate / 8; ++k) {
            uint32_t lo, hi, vlo, vhi;
            ld_word_a8(p + 8 * (g0 + k), lo, hi);
            prefixed_word(carry, lo, hi, vlo, vhi);
            PlainRep::xor_word(A[k], B[k], vlo, vhi);
        }
    } else {
#pragma unroll
        for (int k = 0; k < kRate / 8; ++k) {
            uint32_t lo = 0, hi = 0, vlo, vhi;
            if (g0 + k < mwords) ld_word_a8(p + 8 * (g0 + k), lo, hi);
            prefixed_word(carry, lo, hi, vlo, vhi);
            if (uint32_t(k) == rem / 8) {
                const uint32_t sh = (rem % 8) * 8;
                if (sh < 32) vlo ^= uint32_t(kDomain) << sh;
                else vhi ^= uint32_t(kDomain) << (sh - 32);
            }
            if (k == kRate / 8 - 1) vhi ^= 0x80000000u;
            PlainRep::xor_word(A[k], B[k], vlo, vhi);
        }
    }
}

// The state after absorbing 0x00 || leaf and its padding, permuted:
// SHA3-256 of the prefixed leaf sits in lanes 0..3.
__device__ __forceinline__ void leaf_state_a8(const uint8_t *p, uint64_t leaf_bytes, uint32_t (&A)[25],
                                              uint32_t (&B)[25]) {
    const uint64_t vlen = leaf_bytes + 1;  // prefixed message length
    const uint64_t nfull = vlen / kRate;
    const uint32_t rem = uint32_t(vlen - nfull * kRate);
#pragma unroll
    for (int k = 0; k < 25; ++k) A[k] = B[k] = 0;
    uint32_t carry = 0x00u << 24;  // leaf prefix byte
    for (uint64_t b = 0; b <= nfull; ++b) {
        absorb_leaf_block_a8(A, B, p, b, nfull, rem, leaf_bytes / 8, carry);
        PlainRep::permute<false>(A, B);
    }
}

__global__ void __launch_bounds__(kThreads, kMinBlocks)
    k_merkle_leaves_a8(const uint8_t *buf, uint64_t n_leaves, uint64_t leaf_bytes,
                       uint8_t *out) {
    launch_wait();
    const uint64_t step = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n_leaves; i += step) {
        uint32_t A[25], B[25];
        leaf_state_a8(buf + i * leaf_bytes, leaf_bytes, A, B);
        squeeze<kRate, PlainRep, 32>(A, B, out + 32 * i, 32);
    }
}

// Leaves at any alignment and of any size.  XORs block b of the padded message
// 0x00 || leaf (leaf at p, nfull full blocks, rem bytes in the last) into the state.
// The block's bytes are leaf bytes from 136 b - 1 on: lanes 1..16 are funnel shifts
// of the aligned 32-bit words that hold them, lane 0 alone, which takes the prefix
// in block 0, is read byte-exactly.  (Every lane byte-exactly, as before, was 45
// instructions a lane: 2^18 leaves of 1001 bytes 670 us a tree.)
__device__ __forceinline__ void absorb_leaf_block_any(uint32_t (&A)[25], uint32_t (&B)[25], const uint8_t *p,
                                                      uint64_t b, uint64_t nfull, uint32_t rem) {
    const bool full = b < nfull;
    const uint32_t valid = full ? uint32_t(kRate) : rem;  // message bytes in this block, the prefix among them
    uint32_t lo = 0, hi = 0;
    const uint32_t first = valid < 8 ? valid : 8u;  // of them in lane 0
    if (b == 0) {
        if (first > 1) ld_word_any(p, first - 1, lo, hi);
        hi = __funnelshift_l(lo, hi, 8);
        lo = lo << 8;  // prefix byte 0x00
    } else if (first) {
        ld_word_any(p + (b * kRate - 1), first, lo, hi);
    }
    if (rem < 8 && !full) {
        if (rem < 4) lo ^= uint32_t(kDomain) << (8 * rem);
        else hi ^= uint32_t(kDomain) << (8 * (rem - 4));
    }
    PlainRep::xor_word(A[0], B[0], lo, hi);
    // Lanes 1..16, leaf bytes from 136 b + 7 on.
    const uint8_t *q = p + b * kRate + 7;
    const uintptr_t start = reinterpret_cast<uintptr_t>(q);
    const uint32_t *a = reinterpret_cast<const uint32_t *>(start & ~uintptr_t(3));
    const uint32_t sh = uint32_t(start & 3) * 8;
    if (full) {
        uint32_t prev = *a;
#pragma unroll
        for (int k = 1; k < kRate / 8; ++k) {
            const uint32_t w1 = a[2 * k - 1];
            const uint32_t w2 = (k + 1 < kRate / 8 || sh != 0) ? a[2 * k] : 0u;
            PlainRep::xor_word(A[k], B[k], __funnelshift_r(prev, w1, sh), __funnelshift_r(w1, w2, sh));
            prev = w2;
        }
    } else {
        // Aligned words 0 .. nw-1 hold the bytes; those past the message are masked.
        const uint32_t left = rem > 8 ? rem - 8 : 0u;
        const uint32_t nw = left ? uint32_t(((start + left - 1) >> 2) - (start >> 2)) + 1 : 0u;
        int rb = int(8 * rem) - 64;  // message bits still to come, from lane k on
        uint32_t prev = nw ? *a : 0u;
#pragma unroll
        for (int k = 1; k < kRate / 8; ++k) {
            const uint32_t w1 = uint32_t(2 * k - 1) < nw ? a[2 * k - 1] : 0u;
            const uint32_t w2 = uint32_t(2 * k) < nw ? a[2 * k] : 0u;
            uint32_t vl = __funnelshift_r(prev, w1, sh), vh = __funnelshift_r(w1, w2, sh);
            prev = w2;
            vl &= __funnelshift_lc(0xFFFFFFFFu, 0u, uint32_t(max(rb, 0)));
            vh &= __funnelshift_lc(0xFFFFFFFFu, 0u, uint32_t(max(rb - 32, 0)));
            if (uint32_t(rb) < 32u) vl ^= uint32_t(kDomain) << rb;
            else if (uint32_t(rb - 32) < 32u) vh ^= uint32_t(kDomain) << (rb - 32);
            if (k == kRate / 8 - 1) vh ^= 0x80000000u;
            rb -= 64;
            PlainRep::xor_word(A[k], B[k], vl, vh);
        }
    }
}

__global__ void __launch_bounds__(kThreads, kMinBlocks)
    k_merkle_leaves_any(const uint8_t *buf, uint64_t n_leaves, uint64_t leaf_bytes,
                        uint8_t *out) {
    launch_wait();
    const uint64_t step = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t vlen = leaf_bytes + 1;
    const uint64_t nfull = vlen / kRate;
    const uint32_t rem = uint32_t(vlen - nfull * kRate);
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n_leaves; i += step) {
        const uint8_t *p = buf + i * leaf_bytes;
        uint32_t A[25], B[25];
#pragma unroll
        for (int k = 0; k < 25; ++k) A[k] = B[k] = 0;
        for (uint64_t b = 0; b <= nfull; ++b) {
            absorb_leaf_block_any(A, B, p, b, nfull, rem);
            PlainRep::permute<false>(A, B);
        }
        squeeze<kRate, PlainRep, 32>(A, B, out + 32 * i, 32);
    }
}

// Parent j of one level: SHA3-256(0x01 || in[2j] || in[2j+1]); for an odd
// count the last child is copied to out[count/2].  `in` is 32-byte aligned.
// No __restrict__: in the top-of-tree kernel a level written by the block is
// read back by it after a barrier, so the loads must stay coherent ones.
__device__ __forceinline__ void merkle_parent(const uint8_t *in, uint64_t count, uint8_t *out, uint64_t j) {
    const uint64_t pairs = count / 2;
    if (j == pairs) {
        const uint4 *s = reinterpret_cast<const uint4 *>(in + 32 * (count - 1));
        uint4 *d = reinterpret_cast<uint4 *>(out + 32 * j);
        d[0] = s[0];
        d[1] = s[1];
        return;
    }
    uint32_t A[25], B[25];
#pragma unroll
    for (int k = 0; k < 25; ++k) A[k] = B[k] = 0;
    const uint4 *q = reinterpret_cast<const uint4 *>(in + 64 * j);
    uint32_t carry = 0x01u << 24;  // node prefix byte
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const uint4 v = q[t];
        uint32_t vlo, vhi;
        prefixed_word(carry, v.x, v.y, vlo, vhi);
        PlainRep::set_word(A[2 * t], B[2 * t], vlo, vhi);
        prefixed_word(carry, v.z, v.w, vlo, vhi);
        PlainRep::set_word(A[2 * t + 1], B[2 * t + 1], vlo, vhi);
    }
    // Word 8: the last child byte, then the domain byte at message offset 65.
    uint32_t vlo = (carry >> 24) | (uint32_t(kDomain) << 8), vhi = 0;
    PlainRep::set_word(A[8], B[8], vlo, vhi);
    B[kRate / 8 - 1] ^= 0x80000000u;
    PlainRep::permute<true>(A, B);
    squeeze<kRate, PlainRep, 32>(A, B, out + 32 * j, 32);
}

// One level, one thread per parent.
__global__ void __launch_bounds__(kThreads, kMinBlocks)
    k_merkle_level(const uint8_t *in, uint64_t count, uint8_t *out) {
    launch_wait();
    const uint64_t parents = count / 2 + (count & 1);
    const uint64_t step = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t j = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; j < parents; j += step)
        merkle_parent(in, count, out, j);
}

// ---- many small trees, one thread per tree ----------------------------------

// The state holding the padded block of 0x01 || left || right (digests as
// eight little-endian 32-bit words each), ready to permute.
__device__ __forceinline__ void load_node_block(uint32_t (&A)[25], uint32_t (&B)[25], const uint32_t (&l)[8],
                                                const uint32_t (&r)[8]) {
#pragma unroll
    for (int k = 0; k < 25; ++k) A[k] = B[k] = 0;
    uint32_t carry = 0x01u << 24;  // node prefix byte
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const uint32_t lo = t < 4 ? l[2 * t] : r[2 * (t - 4)];
        const uint32_t hi = t < 4 ? l[2 * t + 1] : r[2 * (t - 4) + 1];
        uint32_t vlo, vhi;
        prefixed_word(carry, lo, hi, vlo, vhi);
        PlainRep::set_word(A[t], B[t], vlo, vhi);
    }
    PlainRep::set_word(A[8], B[8], (carry >> 24) | (uint32_t(kDomain) << 8), 0u);
    B[kRate / 8 - 1] ^= 0x80000000u;
}

// Few leaves: one warp each (coop_sponge.cuh), which takes a third of the time of a
// thread for a leaf's chain of permutations.
__global__ void __launch_bounds__(32)
    k_merkle_leaves_coop(const uint8_t *buf, uint64_t leaf_bytes, uint8_t *out, bool few) {
    __shared__ __align__(16) uint32_t mem[Coop::kWarpWords];
    const Coop c(mem);
    const uint64_t i = blockIdx.x;
    launch_wait();
    coop_sponge<0, true>(c, buf + i * leaf_bytes, leaf_bytes, 1, out + 32 * i, 32, few);
}

// Levels where a permutation's latency, not the ALU pipe's throughput, sets the
// time: up to kClimbLevels of them in one launch, one warp per node (coop.cuh).
// Block b takes children [16b, 16b + 16) of the first level and all nodes above
// them, up to one: 8 nodes, then 4, 2 and 1, handed on in shared memory; an odd
// last node of a level is carried up.  The blocks' ranges nest (the parents of
// nodes [16b, 16b + 16) are nodes [8b, 8b + 8) of the next level), so every node
// is the one the level-by-level reduction gives, and each is written out.
//
// A node takes 1.6 us alone on its SM, more beside others (the warps of an SM share
// its path to shared memory), where one thread per node took 4.5 whatever their
// number.  Eight warps and four levels a launch measured best: 1000 leaves of 1001
// bytes to the root 115 -> 47.9 us; 49.5 with four warps and three levels, 48.3 with
// two and two, 70.7 with sixteen and five.  From kClimbPerSm parents per SM on down
// this is the shorter way.
constexpr int kClimbWarps = 8, kClimbLevels = 4;
constexpr uint64_t kClimbPerSm = 16;

__global__ void __launch_bounds__(32 * kClimbWarps)
    k_merkle_climb(const uint8_t *in, uint64_t count, uint8_t *out, int levels) {
    __shared__ __align__(16) uint32_t mem[kClimbWarps][Coop::kWarpWords];
    __shared__ __align__(16) uint32_t node[2][2 * kClimbWarps][8];  // digests of the level below and of this one
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Coop c(mem[warp]);
    uint64_t cnt = count;                            // nodes of the level below
    uint64_t base = uint64_t(blockIdx.x) * 2 * kClimbWarps;  // this block's first of them
    launch_wait();
    if (threadIdx.x < 4 * kClimbWarps) {  // 16 bytes a thread; plain loads: an earlier launch wrote them
        const uint64_t i = base + threadIdx.x / 2;
        if (i < cnt)
            *reinterpret_cast<uint4 *>(&node[0][threadIdx.x / 2][4 * (threadIdx.x & 1)]) =
                reinterpret_cast<const uint4 *>(in)[2 * i + (threadIdx.x & 1)];
    }
    __syncthreads();
    for (int l = 0; l < levels; ++l) {
        const uint32_t (*child)[8] = node[l & 1];
        const uint64_t parents = cnt / 2 + (cnt & 1);
        if (l + 1 == levels) launch_next();
        const uint64_t q = base / 2 + warp;  // this warp's parent, child[2 * warp] and the next
        if (warp < uint32_t(kClimbWarps) >> l && q < parents) {
            if (2 * q + 1 < cnt) {
                // 0x01 || left || right, 65 bytes and their padding, in lanes 0..8 and 16.
                const uint32_t *d = child[2 * warp];  // sixteen words: the two digests are neighbours
                uint32_t a[2];
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const int k = c.lane(s);
                    uint32_t lo = 0, hi = 0;
                    if (k < 8) {
                        lo = __funnelshift_l(k ? d[2 * k - 1] : 0x01000000u, d[2 * k], 8);
                        hi = __funnelshift_l(d[2 * k], d[2 * k + 1], 8);
                    } else if (k == 8) {
                        lo = (d[15] >> 24) | (uint32_t(kDomain) << 8);
                    } else if (k == kRate / 8 - 1) {
                        hi = 0x80000000u;
                    }
                    a[s] = c.on && k < kRate / 8 ? c.half(lo, hi) : 0u;
                }
                c.permute(a, [] {});
                const uint32_t w = c.unhalf(a[0]);
                if (c.on && c.p == 0 && c.x < 4) {
                    node[(l & 1) ^ 1][warp][2 * c.x + c.h] = w;
                    reinterpret_cast<uint32_t *>(out + 32 * q)[2 * c.x + c.h] = w;
                }
            } else if (lane < 8) {
                const uint32_t w = child[2 * warp][lane];
                node[(l & 1) ^ 1][warp][lane] = w;
                reinterpret_cast<uint32_t *>(out + 32 * q)[lane] = w;
            }
        }
        __syncthreads();
        out += 32 * parents;
        cnt = parents;
        base /= 2;
    }
}

// Stack of subtree digests: sizes are distinct powers of two (the binary
// digits of the leaves seen so far), so 40 entries cover trees below 2^39.
constexpr int kStackDepth = 40;

// Tree t = leaves [t*L, (t+1)*L) of leaf_bytes each.  Leaves are hashed in
// order; equal-size subtrees on the stack merge at once, and the remaining
// ones merge right to left at the end, which builds exactly the level-by-
// level tree with odd nodes carried up.  Every leaf block and every node is
// one pass of a single loop around one permutation call site, so the kernel
// holds one copy of the permutation's code.
template <bool A8>
__global__ void __launch_bounds__(kThreads)
    k_merkle_many(const uint8_t *__restrict__ buf, uint64_t n_trees, uint64_t leaves_per_tree, uint64_t leaf_bytes,
                  uint8_t *__restrict__ roots) {
    const uint64_t step = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t vlen = leaf_bytes + 1;
    const uint64_t nfull = vlen / kRate;
    const uint32_t rem = uint32_t(vlen - nfull * kRate);
    enum Mode { kLeaf, kMerge, kFold };
    for (uint64_t t = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < n_trees; t += step) {
        uint32_t stack[kStackDepth][8];
        uint64_t size[kStackDepth];
        int top = 0;
        uint32_t cur[8];  // the digest being merged or folded
        uint32_t A[25], B[25];
        uint64_t leaf = 0, blk = 0, sz = 0;
        uint32_t carry = 0;
        int j = 0;  // fold position
        Mode mode = kLeaf;
        const uint8_t *first_leaf = buf + t * leaves_per_tree * leaf_bytes;
        for (;;) {
            if (mode == kLeaf) {
                const uint8_t *p = first_leaf + leaf * leaf_bytes;
                if (blk == 0) {
#pragma unroll
                    for (int k = 0; k < 25; ++k) A[k] = B[k] = 0;
                    carry = 0x00u << 24;  // leaf prefix byte
                }
                if constexpr (A8) absorb_leaf_block_a8(A, B, p, blk, nfull, rem, leaf_bytes / 8, carry);
                else absorb_leaf_block_any(A, B, p, blk, nfull, rem);
            } else {
                uint32_t l[8];
                const int li = mode == kMerge ? top - 1 : j;
#pragma unroll
                for (int k = 0; k < 8; ++k) l[k] = stack[li][k];
                load_node_block(A, B, l, cur);
            }
            PlainRep::permute<false>(A, B);
            if (mode == kLeaf && blk < nfull) {
                ++blk;
                continue;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                cur[2 * k] = A[k];
                cur[2 * k + 1] = B[k];
            }
            if (mode == kFold) {
                if (j == 0) break;  // cur is the root
                --j;
                continue;
            }
            if (mode == kLeaf) {
                sz = 1;
                blk = 0;
                ++leaf;
            } else {  // kMerge: cur = node(stack[top - 1], cur)
                sz *= 2;
                --top;
            }
            if (top > 0 && size[top - 1] == sz) {
                mode = kMerge;
                continue;
            }
            if (leaf < leaves_per_tree) {
#pragma unroll
                for (int k = 0; k < 8; ++k) stack[top][k] = cur[k];
                size[top++] = sz;
                mode = kLeaf;
                continue;
            }
            // All leaves are in: fold the stack's subtrees into cur, right to left.
            if (top == 0) break;  // cur is the root
            j = top - 1;
            mode = kFold;
        }
        uint4 *o = reinterpret_cast<uint4 *>(roots + 32 * t);
        o[0] = make_uint4(cur[0], cur[1], cur[2], cur[3]);
        o[1] = make_uint4(cur[4], cur[5], cur[6], cur[7]);
    }
}

}  // namespace

uint64_t merkle_nodes(uint64_t n_leaves) {
    if (n_leaves == 0) return 0;
    uint64_t total = 0, n = n_leaves;
    for (;;) {
        total += n;
        if (n == 1) break;
        n = (n + 1) / 2;
    }
    return total;
}

namespace {

int launch_leaves(const uint8_t *buf, uint64_t n_leaves, uint64_t leaf_bytes, uint8_t *out, cudaStream_t stream,
                  const DeviceInfo &dev) {
    if (n_leaves == 0) return KB_OK;
    const uint64_t sms = uint64_t(dev.sm_count > 0 ? dev.sm_count : 1);
    const uint64_t few = leaf_bytes + 1 < uint64_t(kRate) ? kCoopOnePerSm : kCoopPerSm;
    if (n_leaves <= few * sms)
        return cuda_status(
            launch_overlapped(k_merkle_leaves_coop, unsigned(n_leaves), 32, 0, stream, buf, leaf_bytes, out,
                              few_warps(n_leaves, dev.sm_count)));
    const bool a8 = ((reinterpret_cast<uintptr_t>(buf) | leaf_bytes) & 7) == 0 && leaf_bytes > 0;
    // One thread per leaf and as many blocks as that takes: a leaf is a long
    // chain of permutations, and the block scheduler's dynamic placement
    // balances the last wave better than a fixed grid-stride split (measured
    // 5% faster on 4 GiB of 8 KiB leaves).
    const uint64_t grid = std::min<uint64_t>((n_leaves + kThreads - 1) / kThreads, uint64_t(INT32_MAX));
    return cuda_status(launch_overlapped(a8 ? k_merkle_leaves_a8 : k_merkle_leaves_any, unsigned(grid), kThreads, 0,
                                         stream, buf, n_leaves, leaf_bytes, out));
}

// Every level above the n leaf digests at `nodes`, written after them: one
// launch per level while a level has more than kClimbPerSm parents per SM (there
// a thread per parent is as quick or the ALU pipe's throughput sets the time),
// then climbing launches of up to kClimbLevels levels each.
int launch_upper_levels(uint8_t *nodes, uint64_t n, cudaStream_t stream, const DeviceInfo &dev) {
    uint8_t *level = nodes;
    while (n > 1) {
        const uint64_t parents = n / 2 + (n & 1);
        if (parents > kClimbPerSm * uint64_t(dev.sm_count > 0 ? dev.sm_count : 1)) {
            const uint64_t grid = std::min<uint64_t>((parents + kThreads - 1) / kThreads, uint64_t(INT32_MAX));
            if (launch_overlapped(k_merkle_level, unsigned(grid), kThreads, 0, stream, level, n, level + 32 * n) !=
                cudaSuccess)
                return KB_ERR_CUDA;
            level += 32 * n;
            n = parents;
            continue;
        }
        int levels = 0;
        for (uint64_t m = n; levels < kClimbLevels && m > 1; m = m / 2 + (m & 1)) ++levels;
        const uint64_t blocks = (n + 2 * kClimbWarps - 1) / (2 * kClimbWarps);
        if (launch_overlapped(k_merkle_climb, unsigned(blocks), 32 * kClimbWarps, 0, stream, level, n, level + 32 * n,
                              levels) != cudaSuccess)
            return KB_ERR_CUDA;
        for (int l = 0; l < levels; ++l) {
            level += 32 * n;
            n = n / 2 + (n & 1);
        }
    }
    return KB_OK;
}

}  // namespace

int launch_merkle_levels(const uint8_t *buf, uint64_t n_leaves, uint64_t leaf_bytes, uint8_t *nodes,
                         cudaStream_t stream, const DeviceInfo &dev) {
    int rc = launch_leaves(buf, n_leaves, leaf_bytes, nodes, stream, dev);
    if (rc != KB_OK) return rc;
    return launch_upper_levels(nodes, n_leaves, stream, dev);
}

int launch_merkle_many(const uint8_t *buf, uint64_t n_trees, uint64_t leaves_per_tree, uint64_t leaf_bytes,
                       uint8_t *roots, cudaStream_t stream, const DeviceInfo & /*dev*/) {
    // Leaves on 8-byte boundaries (buffer and leaf size) take the aligned
    // 8-byte loads; others the byte-exact reads.
    const bool a8 = ((reinterpret_cast<uintptr_t>(buf) | leaf_bytes) & 7) == 0;
    // One thread per tree and as many blocks as that takes: the block
    // scheduler balances the last wave, where a grid-stride split would give
    // some threads one tree more than others.
    const uint64_t grid = std::min<uint64_t>((n_trees + kThreads - 1) / kThreads, uint64_t(INT32_MAX));
    if (a8)
        k_merkle_many<true><<<unsigned(grid), kThreads, 0, stream>>>(buf, n_trees, leaves_per_tree, leaf_bytes,
                                                                      roots);
    else
        k_merkle_many<false><<<unsigned(grid), kThreads, 0, stream>>>(buf, n_trees, leaves_per_tree, leaf_bytes,
                                                                       roots);
    return cuda_status(cudaGetLastError());
}

uint64_t merkle_message_leaves(uint64_t len, uint64_t chunk_bytes) {
    return len == 0 ? 1 : (len + chunk_bytes - 1) / chunk_bytes;
}

int launch_merkle_message(const uint8_t *msg, uint64_t len, uint64_t chunk_bytes, uint8_t *nodes,
                          cudaStream_t stream, const DeviceInfo &dev) {
    const uint64_t n = merkle_message_leaves(len, chunk_bytes);
    const uint64_t full = len / chunk_bytes;
    int rc = launch_leaves(msg, full, chunk_bytes, nodes, stream, dev);
    if (rc != KB_OK) return rc;
    if (full < n) {  // the short (or empty) last chunk
        const uint64_t last = len - full * chunk_bytes;
        if ((rc = launch_leaves(msg + full * chunk_bytes, 1, last, nodes + 32 * full, stream, dev)) != KB_OK) return rc;
    }
    return launch_upper_levels(nodes, n, stream, dev);
}

}  // namespace kb
