// keccak_p.cu -- the permutation alone: Keccak-p[b, n_r] (Section 3.1, Table 1
// widths, Eq. 10) applied in place to a batch of raw states, for every width
// b = 25w (w = 1, 2, 4, ..., 64) and any number of rounds n_r, with the round
// indices of FIPS 202 Algorithm 7 (the last n_r of 12 + 2l).  This is the
// tool for reduced-round and small-width experiments; the hashing entry
// points use the fixed Keccak-f[1600].
//
// The round constant of width w is the 64-bit one truncated to w bits (its
// bits sit at 2^j - 1 for j <= l), and rc has period 255, so one table of 255
// lanes serves all widths and all round indices.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>

#include "coop.cuh"
#include "keccak_core.cuh"
#include "runtime.cuh"

namespace kb {
namespace {

struct Rc255 {
    uint64_t v[255];
};
__host__ __device__ constexpr Rc255 make_rc255() {
    int seq[255] = {};
    unsigned R = 1;  // rc(t) for t = 0..254, the register stepped once per t
    for (int t = 0; t < 255; ++t) {
        seq[t] = int(R & 1u);
        R <<= 1;
        if (R & 0x100u) R ^= 0x100u | 0x1u | 0x10u | 0x20u | 0x40u;
    }
    Rc255 out{};
    for (int ir = 0; ir < 255; ++ir) {
        uint64_t v = 0;
        for (int j = 0; j <= 6; ++j)
            if (seq[(j + 7 * ir) % 255]) v |= uint64_t(1) << ((1 << j) - 1);
        out.v[ir] = v;
    }
    return out;
}
static __constant__ Rc255 c_rc255 = make_rc255();

// Widths up to 32: lane x + 5y in one 32-bit register that holds its w bits
// 32/w times over (bit z of the lane at bits z, z + w, z + 2w, ...).  As 32 is
// a multiple of w, rotating the register by n rotates every copy of the lane
// by n within its w bits, so a lane rotation is one funnel shift with no
// mask; XOR, AND and NOT keep the copies equal, and the round constant is
// replicated the same way.  Only the low w bits are stored back.
template <int W>
struct SmallLanes {
    static constexpr uint32_t mask = W == 32 ? 0xffffffffu : ((1u << W) - 1u);
    static constexpr uint32_t spread = 0xffffffffu / mask;  // 1 at bits 0, w, 2w, ...
    __device__ static __forceinline__ uint32_t load(uint32_t v) { return (v & mask) * spread; }
    __device__ static __forceinline__ uint32_t store(uint32_t v) { return v & mask; }
    __device__ static __forceinline__ uint32_t rot(uint32_t x, int n) {
        return n % W == 0 ? x : __funnelshift_l(x, x, uint32_t(n % W));
    }
};

template <int W>
__device__ __forceinline__ void small_round(uint32_t (&A)[25], int ir) {
    using L = SmallLanes<W>;
    uint32_t C[5], D[5], Bv[25];
#pragma unroll
    for (int x = 0; x < 5; ++x) C[x] = A[x] ^ A[x + 5] ^ A[x + 10] ^ A[x + 15] ^ A[x + 20];
#pragma unroll
    for (int x = 0; x < 5; ++x) D[x] = C[(x + 4) % 5] ^ L::rot(C[(x + 1) % 5], 1);
#pragma unroll
    for (int y = 0; y < 5; ++y)
#pragma unroll
        for (int x = 0; x < 5; ++x) {
            // pi: B[y, 2x+3y] takes rho(A[x, y])
            const int src = x + 5 * y;
            Bv[y + 5 * ((2 * x + 3 * y) % 5)] = L::rot(A[src] ^ D[x], rho_offset(src));
        }
#pragma unroll
    for (int y = 0; y < 5; ++y)
#pragma unroll
        for (int x = 0; x < 5; ++x)
            A[x + 5 * y] = chi3(Bv[x + 5 * y], Bv[(x + 1) % 5 + 5 * y], Bv[(x + 2) % 5 + 5 * y]);
    A[0] ^= L::load(uint32_t(c_rc255.v[ir]));
}

// States move between global memory and registers through shared memory:
// each warp takes tiles of 32 consecutive 200-byte states (6.4 KB), copied
// with coalesced 8-byte accesses (the warp touches 256 contiguous bytes per
// access), and each thread then reads its own state from shared memory.
// A warp takes one tile and ends; the SM's other warps compute while its copies
// (cp.async, 8 bytes each) are in flight, and warps synchronise only among their
// own threads.  Reading the states straight from global memory, each thread 25
// accesses 200 bytes apart, leaves the reduced rounds waiting on memory.  2^22
// states: 12 rounds of width 1600 463 us, 4 rounds 250, 18 rounds of width 200 397;
// with two buffers a warp in a grid that strides over the tiles, which is half the
// warps per SM and equal shares (k_sha3_uniform64_tma says why those end late), 501,
// 303 and 422.  What is left of the 4 rounds is HBM's (1.68 GB, 251 us at the
// measured copy rate).
constexpr uint32_t kWarpTile = 32;                                   // states per warp tile
constexpr uint32_t kTileWords = kWarpTile * 25;                      // uint2 words of a tile (6.4 KB)
constexpr size_t kTileSmem = size_t(kThreads / 32) * kTileWords * sizeof(uint2);  // per block

// This warp's tile, permuted state by state by f(uint2 *state) in shared memory
// and written back in place.
template <class F>
__device__ __forceinline__ void run_tile(uint64_t *states, uint64_t n, uint2 *sm, F f) {
    const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
    const uint64_t first = (uint64_t(blockIdx.x) * (blockDim.x / 32) + wib) * kWarpTile;
    launch_wait();
    if (first >= n) return;
    const uint32_t cnt = uint32_t(n - first < kWarpTile ? n - first : uint64_t(kWarpTile));
    uint2 *mine = sm + wib * kTileWords;
    uint2 *g = reinterpret_cast<uint2 *>(states + 25 * first);
    const uint32_t sbase = static_cast<uint32_t>(__cvta_generic_to_shared(mine));
    for (uint32_t j = lane; j < cnt * 25; j += 32)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sbase + 8 * j), "l"(g + j) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    if (lane < cnt) f(mine + 25 * lane);
    __syncwarp();
    for (uint32_t j = lane; j < cnt * 25; j += 32) g[j] = mine[j];
}

// (At 7 blocks per SM 18 rounds of width 200 take 397 us, 407 with registers to spare.)
template <int W>
__global__ void __launch_bounds__(kThreads, 7) k_keccak_p_small(uint64_t *states, int first_ir, int nr, uint64_t n) {
    using L = SmallLanes<W>;
    extern __shared__ uint2 sm[];
    const int ir0 = ((first_ir % 255) + 255) % 255;  // rc has period 255 (Algorithm 5)
    run_tile(states, n, sm, [&](uint2 *s) {
        uint32_t A[25];
#pragma unroll
        for (int k = 0; k < 25; ++k) A[k] = L::load(s[k].x);
        int ir = ir0;
        for (int r = 0; r < nr; ++r) {
            small_round<W>(A, ir);
            ir = ir == 254 ? 0 : ir + 1;
        }
#pragma unroll
        for (int k = 0; k < 25; ++k) s[k] = make_uint2(L::store(A[k]), 0u);
    });
}

// One round of Keccak-p[1600] (Eq. 10) with round-constant index ir of the
// period-255 table, in place.
__device__ __forceinline__ void p1600_round(uint32_t (&L)[25], uint32_t (&H)[25], int ir) {
    uint32_t NL[25], NH[25];
    plain_round_body(L, H, NL, NH);
    const uint64_t rc = c_rc255.v[ir];
    NL[0] ^= uint32_t(rc);
    NH[0] += uint32_t(rc >> 32);  // bit 31 alone or nothing: the sum is the XOR, off the ALU pipe
#pragma unroll
    for (int k = 0; k < 25; ++k) {
        L[k] = NL[k];
        H[k] = NH[k];
    }
}

// Width 64: n_r rounds of the plain 32-bit-half round of the hashing kernels
// on registers L, H from round-constant index first_ir.  Keccak-f[1600]
// itself (first_ir 0, 24 rounds) runs the hashing kernels' permutation;
// other round ranges run four rounds per loop pass, so that the compiler
// renames the state between rounds instead of copying it.
__device__ __forceinline__ void p1600_rounds(uint32_t (&L)[25], uint32_t (&H)[25], int first_ir, int nr) {
    if (first_ir == 0 && nr == 24) {
        keccak_f1600_plain<false, 20>(L, H);
        return;
    }
    int ir = ((first_ir % 255) + 255) % 255, r = 0;  // rc has period 255 (Algorithm 5)
#pragma unroll 1
    for (; r + 4 <= nr; r += 4) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            p1600_round(L, H, ir);
            ir = ir == 254 ? 0 : ir + 1;
        }
    }
    for (; r < nr; ++r) {
        p1600_round(L, H, ir);
        ir = ir == 254 ? 0 : ir + 1;
    }
}

// STAGED: states pass through shared memory as in k_keccak_p_small, which
// pays off when the rounds are few (the memory latency is then a large part
// of a state's time); without it each thread reads and writes its own state
// directly, which keeps blocks free of barriers when the rounds dominate.
template <bool STAGED>
__global__ void __launch_bounds__(kThreads) k_keccak_p_1600(uint64_t *states, int first_ir, int nr, uint64_t n) {
    if constexpr (STAGED) {
        extern __shared__ uint2 sm[];
        run_tile(states, n, sm, [&](uint2 *s) {
            uint32_t L[25], H[25];
#pragma unroll
            for (int k = 0; k < 25; ++k) {
                const uint2 v = s[k];
                L[k] = v.x;
                H[k] = v.y;
            }
            p1600_rounds(L, H, first_ir, nr);
#pragma unroll
            for (int k = 0; k < 25; ++k) s[k] = make_uint2(L[k], H[k]);
        });
    } else {
        launch_wait();
        const uint64_t step = uint64_t(gridDim.x) * blockDim.x;
        for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += step) {
            uint2 *s = reinterpret_cast<uint2 *>(states + 25 * i);
            uint32_t L[25], H[25];
#pragma unroll
            for (int k = 0; k < 25; ++k) {
                const uint2 v = s[k];
                L[k] = v.x;
                H[k] = v.y;
            }
            p1600_rounds(L, H, first_ir, nr);
#pragma unroll
            for (int k = 0; k < 25; ++k) s[k] = make_uint2(L[k], H[k]);
        }
    }
}

// Few states of width 64 and rounds within Keccak-f[1600]'s 24: a warp each
// (coop.cuh), a third of the time of one thread's chain of rounds.
__global__ void __launch_bounds__(32) k_keccak_p_1600_coop(uint64_t *states, int first_ir, int nr, bool few) {
    __shared__ __align__(16) uint32_t mem[Coop::kWarpWords];
    const Coop c(mem);
    if (few) launch_next();
    launch_wait();
    uint2 *st = reinterpret_cast<uint2 *>(states + 25 * uint64_t(blockIdx.x));
    uint32_t a[2] = {0, 0};
#pragma unroll
    for (int s = 0; s < 2; ++s)
        if (c.on && c.lane(s) < 25) {
            const uint2 w = st[c.lane(s)];
            a[s] = c.half(w.x, w.y);
        }
    int r = first_ir;
    const int end = first_ir + nr;
#pragma unroll 1
    for (; r + 2 <= end; r += 2) {
        c.round<0>(a, r);
        c.round<1>(a, r + 1);
    }
    if (r < end) c.round<0>(a, r);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const uint32_t w = c.unhalf(a[s]);
        if (c.on && c.lane(s) < 25) reinterpret_cast<uint32_t *>(st)[2 * c.lane(s) + c.h] = w;
    }
}

template <class K>
int launch_tiled(K kernel, uint64_t *states, int first_ir, int nr, uint64_t n, cudaStream_t stream) {
    const uint64_t grid = (n + kThreads - 1) / kThreads;  // 2^31 blocks would be 55 TB of states
    return cuda_status(launch_overlapped(kernel, unsigned(grid), kThreads, kTileSmem, stream, states, first_ir, nr, n));
}

template <int W>
int launch_small(uint64_t *states, int first_ir, int nr, uint64_t n, cudaStream_t stream) {
    return launch_tiled(k_keccak_p_small<W>, states, first_ir, nr, n, stream);
}

}  // namespace

int launch_keccak_p(uint64_t *states, int b, int nr, uint64_t n, cudaStream_t stream, const DeviceInfo &dev) {
    int l = -1;
    for (int k = 0; k <= 6; ++k)
        if (b == 25 * (1 << k)) l = k;
    if (l < 0) return KB_ERR_INVALID;
    const int first_ir = 12 + 2 * l - nr;
    switch (l) {
        case 0: return launch_small<1>(states, first_ir, nr, n, stream);
        case 1: return launch_small<2>(states, first_ir, nr, n, stream);
        case 2: return launch_small<4>(states, first_ir, nr, n, stream);
        case 3: return launch_small<8>(states, first_ir, nr, n, stream);
        case 4: return launch_small<16>(states, first_ir, nr, n, stream);
        case 5: return launch_small<32>(states, first_ir, nr, n, stream);
        default: {
            if (first_ir >= 0 && n <= kCoopPerSm * uint64_t(dev.sm_count > 0 ? dev.sm_count : 1))
                return cuda_status(
                    launch_overlapped(k_keccak_p_1600_coop, unsigned(n), 32, 0, stream, states, first_ir, nr,
                                      few_warps(n, dev.sm_count)));
            // Staged through shared memory below 16 rounds (2^22 states: 12 rounds
            // 574 us read directly, 463 staged; 14 rounds 560 and 532; 18 rounds
            // 647 and 669; 24 rounds 839 and 875).
            if (nr < 16) return launch_tiled(k_keccak_p_1600<true>, states, first_ir, nr, n, stream);
            const uint64_t g = std::min<uint64_t>((n + kThreads - 1) / kThreads, uint64_t(INT32_MAX));
            return cuda_status(
                launch_overlapped(k_keccak_p_1600<false>, unsigned(g), kThreads, 0, stream, states, first_ir, nr, n));
        }
    }
}

}  // namespace kb
