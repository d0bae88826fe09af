// Metropolis chains (Sec. 4.2) on bit-planes of the terms.
//
// For one term <x|phi> is b omega 2^{-|v|/2} i^{q(x)} where the constraints F_k . x = s_k (column
// k of F, k not in v) hold, and zero elsewhere, with the Z4 form
//     q(x) = sum_p d_p x_p + 2 sum_{p<q} J_pq x_p x_q,   J = M F^T (symmetric),
//     d_p = gamma_p + 2 F_p . M_p + 2 F_p . (s & v)      (mod 4)
// (Eqs. (amplitude), (amplitude1) with the Pauli product written out: the sign u . w of
// U_C^{-1} X(x) U_C = i^mu X(u) Z(w) is the diagonal F_p . M_p because M F^T is symmetric).
// A proposal y = x ^ e_j changes q by +-d_j + 2 J_j . x and constraint i by its bit at j, so a
// chain's state is two phase bits and one bit per constraint for every term, and all of it is
// bitwise over the terms: k_mc_planes stores J, d, the constraints' bits and targets as
// planes (one bit per term), a thread owns 64 terms (two words) and J_j . x is the XOR of
// the planes J_jq over the set bits q of x, about n / 2 loads for 64 terms.  The state moves
// 2 + 2 + (constraints) bits per (chain, term) and pass instead of the 96 or 128 of the
// Pauli pair (u, w); what is left is the FP32 sum over the terms.
//
// Planes are stored with the words of a 256-term tile in the order (w, k): term 128 k + 32 w + l
// of the tile is bit l of component k of column 4 tile + w.  A thread sums its 64 terms as
// leaves (k = 0) + (k = 1) and then a binary tree over l, the four columns of a tile in
// order, the tiles in FP64.
#include <string.h>

#include "lrs_device.cuh"

namespace {

constexpr int MC_TPB = 256;    // threads per block
constexpr int MC_COLS = 128;   // most columns of a block
constexpr int MC_TERMS = 256;  // terms per tile (cap is a multiple of 256)
constexpr int MC_CG = 32;      // most chains of a block

// ---- bulk-copy helpers (1-D cp.async.bulk completing on an mbarrier) ----------
constexpr unsigned long long MC_WAIT_NS = 1000000000ull;   // 1 s
__device__ __forceinline__ uint32_t mc_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long mc_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mc_bar_init(uint32_t bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mc_bar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mc_bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ bool mc_bar_try(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}
// Wait for the phase of the given parity; false after MC_WAIT_NS.
__device__ __forceinline__ bool mc_bar_wait(uint32_t bar, uint32_t parity) {
    if (mc_bar_try(bar, parity)) return true;
    const unsigned long long t0 = mc_ns();
    while (!mc_bar_try(bar, parity))
        if (mc_ns() - t0 > MC_WAIT_NS) return false;
    return true;
}

// ---- planes -----------------------------------------------------------------------------
// cols = cap / 64 columns of 64 terms.
struct McView {
    int n;
    int64_t cols;
    uint2* J;        // [n (n - 1) / 2 + 1][cols]: J_pq, p > q, row p (p - 1) / 2 + q; the last row zero
    uint2* D;        // [n][2][cols]: d_p, bits 0 and 1
    uint4* K;        // [n][pairs][cols]: coefficients of constraints 2 i (x, y) and 2 i + 1 (z, w) at qubit p
    uint4* target;   // [pairs][cols]: s at the two constraints
    int pairs;       // (n + 1) / 2
    float2* base;    // [64][cols]: b omega 2^{-|v|/2} / 2 of term (k, l), row 32 k + l (0: no contribution)
    uint8_t* mf;     // [cols / 4]: constraints of the tile (the most of its terms)
};
__host__ __device__ __forceinline__ int mc_pairs(int n) { return n * (n - 1) / 2; }
// Chain states: [plane][chain][cols] of two words, phase bits 0 and 1 and the parities J_j1 . x
// and J_j2 . x of the last pass's proposals; then [pair][chain][cols] of four, the syndromes
// of the constraints.
constexpr int MC_PLANES = 4;

// A block takes a tile: its F in shared memory, and MC_SETS sets of 256 threads (a term each) that
// share out the rows of J and the pairs of constraints, with the gridDim.y blocks of the tile where
// there are fewer tiles than SMs.  (With one set, two warps a scheduler waited for one product
// after the other: 130 us for four tiles at n = 57 and 520 us for 2^17 terms, now 17 and
// 196.)  Padding terms have no weight and get no constraints: as |0^n> they have n of them,
// which every chain would carry through the last tile.
constexpr int MC_SETS = 4;
__device__ __forceinline__ void mc_set_sync(int set) {
    asm volatile("bar.sync %0, 256;" ::"r"(set + 1) : "memory");
}

__global__ void __launch_bounds__(256 * MC_SETS) k_mc_planes(TermsView T, McView V) {
    extern __shared__ uint64_t sF[];          // [n][256]
    __shared__ uint32_t sws[MC_SETS][2][64][16];   // words of a set of planes for the tile, double-buffered
    __shared__ int s_mf;
    const int n = T.n, set = threadIdx.x >> 8, tid = threadIdx.x & 255, lane = tid & 31, wi = tid >> 5;
    const int first = blockIdx.y * MC_SETS + set, sets = gridDim.y * MC_SETS;   // of the tile's sets
    const int64_t tile = blockIdx.x, a = tile * MC_TERMS + tid;
    const int slot = (wi & 3) * 2 + (wi >> 2);   // word of this warp within the tile
    uint32_t(*sw)[64][16] = sws[set];
    for (int p = set; p < n; p += MC_SETS) sF[p * 256 + tid] = T.F[(int64_t)p * T.cap + a];
    const uint64_t glo = T.glo[a], ghi = T.ghi[a], v = T.v[a], s = T.s[a];
    const uint32_t om = T.omega[a];
    const bool dead = ((om >> 3) & 1u) != 0u;
    const uint64_t out = dead || a >= T.chi ? 0ull : ~v & T.nmask;
    if (threadIdx.x == 0) s_mf = 0;
    __syncthreads();
    if (set == 0) atomicMax(&s_mf, __popcll(out));
    if (first == 0) {
        float2 b = make_float2(0.f, 0.f);
        if (!dead) {
            b = z8_scale(T.coef[a], (int)(om & 7u), __popcll(v) + (int)(om >> 8));
            b = make_float2(0.5f * b.x, 0.5f * b.y);   // the pass multiplies by +-2 (k_mc_pass)
        }
        V.base[(int64_t)((wi >> 2) * 32 + lane) * V.cols + tile * 4 + (wi & 3)] = b;
    }
    __syncthreads();
    const int mf = s_mf;
    const int64_t row = V.cols * 2;   // words per plane
    int buf = 0;
    for (int p = first; p < n; p += sets, buf ^= 1) {
        const uint64_t Mp = T.M[(int64_t)p * T.cap + a], Fp = sF[p * 256 + tid];
#pragma unroll 4
        for (int q = 0; q < p; ++q) {
            const uint32_t w = __ballot_sync(0xffffffffu, par64(Mp & sF[q * 256 + tid]));
            if (lane == 0) sw[buf][q][slot] = w;
        }
        const uint32_t lo = __ballot_sync(0xffffffffu, (uint32_t)getb(glo, p));
        const uint32_t hi =
            __ballot_sync(0xffffffffu, (uint32_t)getb(ghi, p) ^ par64(Fp & Mp) ^ par64(Fp & s & v));
        if (lane == 0) {
            sw[buf][62][slot] = lo;
            sw[buf][63][slot] = hi;
        }
        mc_set_sync(set);
        for (int e = tid; e < p * 8; e += 256)
            reinterpret_cast<uint32_t*>(V.J)[((int64_t)p * (p - 1) / 2 + (e >> 3)) * row + tile * 8 + (e & 7)] =
                sw[buf][e >> 3][e & 7];
        if (tid < 16)
            reinterpret_cast<uint32_t*>(V.D)[(2 * p + (tid >> 3)) * row + tile * 8 + (tid & 7)] = sw[buf][62 + (tid >> 3)][tid & 7];
    }
    uint64_t ks = out;
    const int slot4 = (wi & 3) * 4 + (wi >> 2);   // word of this warp in a set of pairs
    for (int i = 0; 2 * i < mf; ++i) {
        const int k0 = ks ? ffs64(ks) : -1;   // constraint 2 i of this term: qubit k0, or none
        ks &= ks - 1;
        const int k1 = ks ? ffs64(ks) : -1;
        ks &= ks - 1;
        if (i % sets != first) continue;
#pragma unroll 4
        for (int p = 0; p <= n; ++p) {
            const uint64_t r = p < n ? sF[p * 256 + tid] : s;   // last: the targets
            const uint32_t w0 = __ballot_sync(0xffffffffu, k0 >= 0 ? (uint32_t)getb(r, k0) : 0u);
            const uint32_t w1 = __ballot_sync(0xffffffffu, k1 >= 0 ? (uint32_t)getb(r, k1) : 0u);
            if (lane == 0) {
                sw[buf][p][slot4] = w0;
                sw[buf][p][slot4 + 2] = w1;
            }
        }
        mc_set_sync(set);
        for (int e = tid; e < (n + 1) * 16; e += 256) {
            const int p = e >> 4;
            uint4* dst = p < n ? V.K + ((int64_t)p * V.pairs + i) * V.cols : V.target + (int64_t)i * V.cols;
            reinterpret_cast<uint32_t*>(dst)[tile * 16 + (e & 15)] = sw[buf][p][e & 15];
        }
        buf ^= 1;
    }
    if (blockIdx.y > 0) return;
    if (threadIdx.x == 0) V.mf[tile] = (uint8_t)mf;
    if (threadIdx.x < 8) reinterpret_cast<uint32_t*>(V.J)[mc_pairs(n) * row + tile * 8 + threadIdx.x] = 0u;
}

__device__ __forceinline__ uint2 operator^(uint2 a, uint2 b) { return make_uint2(a.x ^ b.x, a.y ^ b.y); }
__device__ __forceinline__ uint2 operator&(uint2 a, uint2 b) { return make_uint2(a.x & b.x, a.y & b.y); }

__device__ __forceinline__ uint4 operator^(uint4 a, uint4 b) {
    return make_uint4(a.x ^ b.x, a.y ^ b.y, a.z ^ b.z, a.w ^ b.w);
}

// (lo, hi) += +-(dl, dh) + 2 par, in Z4 planes
__device__ __forceinline__ void z4_step(uint2& lo, uint2& hi, uint2 dl, uint2 dh, bool minus, uint2 par) {
    if (minus) dh = dh ^ dl;
    hi = hi ^ dh ^ (lo & dl) ^ par;
    lo = lo ^ dl;
}

// row of J_pq (the zero row for p == q)
__device__ __forceinline__ int mc_row(int p, int q, int zero) {
    const int hi = p > q ? p : q, lo = p > q ? q : p;
    return p == q ? zero : hi * (hi - 1) / 2 + lo;
}

// State of every (chain, term) at the chains' strings: q(x) by adding the set bits (Z4 sums, so in
// any order), and the syndromes.  `split` threads of a warp (a power of two, their columns tbx = 32
// / split apart) share the set bits and the pairs of constraints of a (chain, column): with
// few chains of few terms one thread's loads, one batch after the other, were all there was to wait
// for (8 chains of 1000 terms at n = 57: 121 us, now 29).
__global__ void __launch_bounds__(MC_TPB) k_mc_start(McView V, int64_t C, uint2* __restrict__ S,
                                                     const uint64_t* __restrict__ xs, uint64_t nmask, int tbx, int split,
                                                     int64_t cblocks) {
    // chains fastest: the blocks that read one column range's planes run together
    const int tid = threadIdx.x, part = tid / tbx % split;
    int64_t c = blockIdx.x % cblocks * (MC_TPB / (tbx * split)) + tid / (tbx * split);
    int64_t col = blockIdx.x / cblocks * tbx + tid % tbx;
    const bool on = c < C && col < V.cols;
    if (split == 1 && !on) return;
    if (!on) c = col = 0;   // for the exchanges
    const uint64_t x = xs[c] & nmask;
    const uint2* J = V.J + col;
    uint2 lo = make_uint2(0u, 0u), hi = lo;
    uint64_t r = x;
    for (int k = 0; k < part; ++k) r &= r - 1;
    while (r) {
        const int p = ffs64(r);
        for (int k = 0; k < split; ++k) r &= r - 1;
        uint2 par = make_uint2(0u, 0u);
        const uint2* Jp = J + (int64_t)(p * (p - 1) / 2) * V.cols;
        uint64_t below = x & (bit64(p) - 1);
        while (below) {
            uint2 t[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                t[u] = make_uint2(0u, 0u);
                if (below) t[u] = __ldg(Jp + (int64_t)ffs64(below) * V.cols);
                below &= below - 1;
            }
            par = par ^ (t[0] ^ t[1]) ^ (t[2] ^ t[3]);
        }
        z4_step(lo, hi, __ldg(V.D + (int64_t)(2 * p) * V.cols + col), __ldg(V.D + (int64_t)(2 * p + 1) * V.cols + col), false,
                par);
    }
    for (int off = tbx; off < tbx * split; off <<= 1) {
        uint2 l2, h2;
        l2.x = __shfl_xor_sync(0xffffffffu, lo.x, off);
        l2.y = __shfl_xor_sync(0xffffffffu, lo.y, off);
        h2.x = __shfl_xor_sync(0xffffffffu, hi.x, off);
        h2.y = __shfl_xor_sync(0xffffffffu, hi.y, off);
        hi = hi ^ h2 ^ (lo & l2);
        lo = lo ^ l2;
    }
    if (!on) return;
    const int64_t plane = C * V.cols;
    uint2* st = S + c * V.cols + col;
    if (part == 0) {
        st[0] = lo;
        st[plane] = hi;
    }
    uint4* sy = reinterpret_cast<uint4*>(S + MC_PLANES * plane) + c * V.cols + col;
    const int pairs = (V.mf[col >> 2] + 1) >> 1;
    for (int i = part; i < pairs; i += split) {
        uint4 y = __ldg(V.target + (int64_t)i * V.cols + col);
        const uint4* Ki = V.K + (int64_t)i * V.cols + col;
        uint64_t w = x;
        while (w) {
            uint4 t[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                t[u] = make_uint4(0u, 0u, 0u, 0u);
                if (w) t[u] = __ldg(Ki + (int64_t)ffs64(w) * V.pairs * V.cols);
                w &= w - 1;
            }
            y = y ^ (t[0] ^ t[1]) ^ (t[2] ^ t[3]);
        }
        sy[i * plane] = y;
    }
}

// One pass over the states for one or two steps.  Two steps: the proposals j1 = j_t and
// j2 = j_{t+1} come from the counter RNG and do not depend on the chain, so one pass forms
// <y|psi> for every string step t + 1 may propose: y1 = x ^ e_j1, y1 ^ e_j2 (step t accepted)
// and x ^ e_j2 (rejected); the accept kernel then takes both decisions in order, and the
// planes of J are read from DRAM once per two steps.  The flips accepted after the previous
// pass (pend) are applied first, with the parities that pass left.  Each term's
// contribution and the order of the sums are those of a single step.
//
// The FP32 sums are what bounds it: per (term, sum) a sign and live factor (+-2 or +-0, built
// from two adjacent bits of a nibble and multiplied onto half the coefficient, which is
// exact), a swap of the two parts, and one fused multiply-add each.
// n = 50, chi = 2^20, 256 chains: 574 us per two-step pass and 37 for its accept test
// (2.1 ms with 16-byte Pauli states); n = 40, chi = 2^16, 1024 chains: 136 us.
// The block's coefficients (64 rows of tbx columns) are copied once by cp.async.bulk; the wait
// is bounded (1 s) and a block that gives up sets *err and leaves its sums unwritten.
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {   // two FP32 additions
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// What a pass reads of a chain, gathered once per block: the string, the flips to apply and to
// propose, and the rows of J at the set bits of x, J_j1q | J_j2q << 16 (rows of zeros for
// q = j and up to a multiple of eight).
struct McChain {
    uint64_t x;
    int p1, p2, j1, j2;
    int nq, reserved;
    uint32_t row[64];
};

template <int STEPS>
__global__ void __launch_bounds__(MC_TPB, 3) k_mc_pass(McView V, int64_t C, uint2* __restrict__ S,
                                                       const uint64_t* __restrict__ cx,
                                                       const int32_t* __restrict__ pend,
                                                       const int32_t* __restrict__ jprop, float2* __restrict__ partial,
                                                       int cg, int64_t groups, int tbx, int* err) {
    constexpr int NE = STEPS == 2 ? 3 : 1;   // strings evaluated
    extern __shared__ __align__(128) float2 sbase[];   // [64][tbx], then McChain[cg]
    __shared__ __align__(8) uint64_t full;
    McChain* chains = reinterpret_cast<McChain*>(sbase + 64 * tbx);
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t c0 = blockIdx.x % groups * cg, tb = blockIdx.x / groups;
    const int nc = (int)(C - c0 < cg ? C - c0 : cg);
    const int nsub = MC_TPB / tbx, tc = tid % tbx;
    const int64_t col0 = tb * tbx;
    const int nb = (int)(V.cols - col0 < tbx ? V.cols - col0 : tbx);   // a multiple of 4
    const int zero = mc_pairs(V.n);
    const uint32_t bar = mc_smem(&full);
    if (tid == 0) {
        mc_bar_init(bar);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // err[1] is a one-shot test request (lrs_debug_inject_wait_timeout): block 0 takes it
        // and expects 16 bytes that no copy delivers, so the bounded wait runs out
        uint32_t extra = 0;
        if (blockIdx.x == 0 && *(volatile int*)&err[1] != 0) {
            *(volatile int*)&err[1] = 0;
            extra = 16;
        }
        mc_bar_expect(bar, (uint32_t)(64 * nb * sizeof(float2)) + extra);
    }
    if (tid < 32) {
        __syncwarp();
        for (int r = tid; r < 64; r += 32)
            mc_bulk_load(mc_smem(sbase + r * tbx), V.base + (int64_t)r * V.cols + col0, (uint32_t)(nb * sizeof(float2)), bar);
    }
    for (int ci = tid >> 5; ci < nc; ci += MC_TPB / 32) {   // a warp per chain
        McChain& ch = chains[ci];
        const int64_t c = c0 + ci;
        const uint64_t x = cx[c];
        const int j1 = jprop[c], j2 = STEPS == 2 ? jprop[C + c] : 0, nq = __popcll(x);
        if (lane == 0) {
            ch.x = x;
            ch.p1 = pend[c];
            ch.p2 = pend[C + c];
            ch.j1 = j1;
            ch.j2 = j2;
            ch.nq = nq;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int q = lane + 32 * h;
            if (getb(x, q))
                ch.row[__popcll(x & (bit64(q) - 1))] =
                    (uint32_t)mc_row(j1, q, zero) | (uint32_t)(STEPS == 2 ? mc_row(j2, q, zero) : zero) << 16;
        }
        if (lane < ((8 - nq) & 7)) ch.row[nq + lane] = (uint32_t)zero | (uint32_t)zero << 16;
    }
    __syncthreads();
    if (__syncthreads_or(!mc_bar_wait(bar, 0u))) {
        // every copy has landed or is waited for once more (bounded) before the block leaves
        if (tid == 0) {
            mc_bar_wait(bar, 0u);
            atomicExch(err, 1);
        }
        return;
    }
    const bool in = tc < nb;
    const int64_t col = col0 + (in ? tc : 0), plane = C * V.cols, n_tiles = V.cols >> 2;
    const int mf2 = (V.mf[col >> 2] + 1) >> 1;   // pairs of constraints of the tile
    const int mfw = __reduce_max_sync(0xffffffffu, mf2);
    const uint32_t row8 = (uint32_t)V.cols * 8u;   // bytes of a plane (cols <= 2^28)
    const char* Jc = reinterpret_cast<const char*>(V.J + col);
    const char* Dc = reinterpret_cast<const char*>(V.D + col);
    auto J = [&](uint32_t r) { return __ldg(reinterpret_cast<const uint2*>(Jc + (uint64_t)r * row8)); };
    auto D = [&](uint32_t r) { return __ldg(reinterpret_cast<const uint2*>(Dc + (uint64_t)r * row8)); };
    const float2* bp = sbase + tc;
    const uint2 none = make_uint2(0u, 0u);
    for (int i0 = 0; i0 < nc; i0 += nsub) {
        const int ci = i0 + tid / tbx < nc ? i0 + tid / tbx : 0;
        const bool on = in && i0 + tid / tbx < nc;
        const McChain& ch = chains[ci];
        const int64_t c = c0 + ci;
        const uint64_t x = ch.x;
        const int p1 = ch.p1, p2 = ch.p2, j1 = ch.j1, j2 = ch.j2;
        uint2* st = S + c * V.cols + col;
        uint2 lo = st[0], hi = st[plane];
        const bool moved = p1 >= 0 || p2 >= 0;
        uint2 old1 = none, old2 = none;
        if (p1 >= 0) old1 = st[2 * plane];
        if (p2 >= 0) old2 = st[3 * plane];
        // J_j . x for the proposals
        uint2 par1 = none, par2 = none;
#pragma unroll 1
        for (int k = 0; k < ch.nq; k += 8) {
            uint2 t1[8], t2[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const uint32_t r = ch.row[k + u];
                t1[u] = J(r & 0xffffu);
                if (STEPS == 2) t2[u] = J(r >> 16);
            }
#pragma unroll
            for (int u = 0; u < 8; u += 2) {
                par1 = par1 ^ t1[u] ^ t1[u + 1];
                if (STEPS == 2) par2 = par2 ^ t2[u] ^ t2[u + 1];
            }
        }
        if (moved) {   // the flips accepted after the previous pass, in order
            uint64_t xo = x ^ (p1 >= 0 ? bit64(p1) : 0ull) ^ (p2 >= 0 ? bit64(p2) : 0ull);
            if (p1 >= 0) {
                z4_step(lo, hi, D(2 * p1), D(2 * p1 + 1), getb(xo, p1) != 0, old1);
                xo ^= bit64(p1);
                if (p2 >= 0) old2 = old2 ^ J(mc_row(p1, p2, zero));
            }
            if (p2 >= 0) z4_step(lo, hi, D(2 * p2), D(2 * p2 + 1), getb(xo, p2) != 0, old2);
            if (on) {
                st[0] = lo;
                st[plane] = hi;
            }
        }
        if (on) {
            st[2 * plane] = par1;
            if (STEPS == 2) st[3 * plane] = par2;
        }
        // phases of y1, y1 ^ e_j2, x ^ e_j2 and the terms whose constraints fail there
        uint2 L[NE], H[NE], dead[NE];
        L[0] = lo;
        H[0] = hi;
        z4_step(L[0], H[0], D(2 * j1), D(2 * j1 + 1), getb(x, j1) != 0, par1);
        if (STEPS == 2) {
            const uint2 dl = D(2 * j2), dh = D(2 * j2 + 1), j12 = J(mc_row(j1, j2, zero));
            L[NE / 2] = L[0];
            H[NE / 2] = H[0];
            z4_step(L[NE / 2], H[NE / 2], dl, dh, getb(x ^ bit64(j1), j2) != 0, par2 ^ j12);
            L[NE - 1] = lo;
            H[NE - 1] = hi;
            z4_step(L[NE - 1], H[NE - 1], dl, dh, getb(x, j2) != 0, par2);
        }
#pragma unroll
        for (int e = 0; e < NE; ++e) dead[e] = none;
        uint4* sy = reinterpret_cast<uint4*>(S + MC_PLANES * plane) + c * V.cols + col;
        const uint4* K = V.K + col;
        const int64_t krow = (int64_t)V.pairs * V.cols;
#pragma unroll 1
        for (int i = 0; i < mfw; ++i, K += V.cols, sy += plane) {
            if (i >= mf2) continue;   // this tile has fewer
            uint4 y = *sy;
            const uint4 k1 = __ldg(K + j1 * krow);
            uint4 k2;
            if (STEPS == 2) k2 = __ldg(K + j2 * krow);
            if (moved) {
                if (p1 >= 0) y = y ^ __ldg(K + p1 * krow);
                if (p2 >= 0) y = y ^ __ldg(K + p2 * krow);
                if (on) *sy = y;
            }
            const uint4 y1 = y ^ k1;
            dead[0].x |= y1.x | y1.z;
            dead[0].y |= y1.y | y1.w;
            if (STEPS == 2) {
                dead[NE / 2].x |= (y1.x ^ k2.x) | (y1.z ^ k2.z);
                dead[NE / 2].y |= (y1.y ^ k2.y) | (y1.w ^ k2.w);
                dead[NE - 1].x |= (y.x ^ k2.x) | (y.z ^ k2.z);
                dead[NE - 1].y |= (y.y ^ k2.y) | (y.w ^ k2.w);
            }
        }
        // the sums, one string at a time (rolled: registers for three blocks an SM)
#pragma unroll 1
        for (int e = 0; e < NE; ++e) {
            uint64_t f2 = 0, u = 0;
            if (__any_sync(0xffffffffu, (dead[0].x & dead[0].y) != 0xffffffffu)) {
#pragma unroll 1
                for (int it = 0; it < 4; ++it) {
                    // leaves l = l0 + 4 t, l0 = bits 0 and 1 of l; nibble t of N: live, phase
                    // bit 1, phase bit 0
                    const int l0 = (it >> 1) + 2 * (it & 1);
                    constexpr uint32_t one = 0x11111111u;
                    const uint32_t N0 =
                        (~dead[0].x >> l0 & one) | (H[0].x >> l0 & one) << 1 | (L[0].x >> l0 & one) << 2;
                    const uint32_t N1 =
                        (~dead[0].y >> l0 & one) | (H[0].y >> l0 & one) << 1 | (L[0].y >> l0 & one) << 2;
                    const float2* b0 = bp + l0 * tbx;
                    uint64_t v[8];   // complex pairs
#pragma unroll
                    for (int t = 0; t < 8; ++t) {
                        const float2 ba = b0[4 * t * tbx], bb = b0[(32 + 4 * t) * tbx];
                        // b i^m, m = 2 hi + lo: (x, y) or (-y, x), times (-1)^hi
                        const float fa = __uint_as_float((N0 << (30 - 4 * t)) & 0xC0000000u);
                        const float fb = __uint_as_float((N1 << (30 - 4 * t)) & 0xC0000000u);
                        const bool sa = (N0 & (4u << (4 * t))) != 0, sb = (N1 & (4u << (4 * t))) != 0;
                        const float re = fmaf(fb, sb ? -bb.y : bb.x, fa * (sa ? -ba.y : ba.x));
                        const float im = fmaf(fb, sb ? bb.x : bb.y, fa * (sa ? ba.x : ba.y));
                        asm("mov.b64 %0, {%1, %2};" : "=l"(v[t]) : "f"(re), "f"(im));
                    }
#pragma unroll
                    for (int h = 4; h > 0; h >>= 1)   // bits 4, 3, 2 of l
#pragma unroll
                        for (int t = 0; t < h; ++t) v[t] = add2(v[t], v[t + h]);
                    // bit 1, then bit 0
                    u = (it & 1) ? add2(u, v[0]) : v[0];
                    if (it == 1) f2 = u;
                    if (it == 3) f2 = add2(f2, u);
                }
            }
            // the four columns of the tile in order
            const float2 f = make_float2(__uint_as_float((uint32_t)f2), __uint_as_float((uint32_t)(f2 >> 32)));
            float2 acc = f;
#pragma unroll
            for (int w = 1; w < 4; ++w) {
                acc.x += __shfl_down_sync(0xffffffffu, f.x, w);
                acc.y += __shfl_down_sync(0xffffffffu, f.y, w);
            }
            if (on && (lane & 3) == 0) partial[((int64_t)e * C + c) * n_tiles + (col >> 2)] = acc;
            if (NE == 3) {   // next string
                L[0] = L[NE / 2];
                H[0] = H[NE / 2];
                dead[0] = dead[NE / 2];
                L[NE / 2] = L[NE - 1];
                H[NE / 2] = H[NE - 1];
                dead[NE / 2] = dead[NE - 1];
            }
        }
    }
}

// |sum over tiles|^2 of chain c in FP64, by each group of 256 threads; valid in the group's
// first warp's lane 0.  (The last five levels of the tree by shuffles: same pairs.)
__device__ __forceinline__ double chain_reduce(const float2* __restrict__ partial, int64_t c,
                                               int64_t n_tiles) {
    const int tid = threadIdx.x & 255;
    double re = 0.0, im = 0.0;
    for (int64_t t = tid; t < n_tiles; t += 256) {
        const float2 p = partial[c * n_tiles + t];
        re += (double)p.x;
        im += (double)p.y;
    }
    __shared__ double sre[768], sim[768];
    sre[threadIdx.x] = re;
    sim[threadIdx.x] = im;
    __syncthreads();
    for (int off = 128; off >= 64; off >>= 1) {
        if (tid < off) {
            sre[threadIdx.x] += sre[threadIdx.x + off];
            sim[threadIdx.x] += sim[threadIdx.x + off];
        }
        __syncthreads();
    }
    if (tid >= 32) return 0.0;
    re = sre[threadIdx.x] + sre[threadIdx.x + 32];
    im = sim[threadIdx.x] + sim[threadIdx.x + 32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        re += __shfl_down_sync(0xffffffffu, re, off);
        im += __shfl_down_sync(0xffffffffu, im, off);
    }
    return re * re + im * im;
}

__device__ __forceinline__ int draw_j(uint64_t seed, int64_t c, int64_t step, int n) {
    const uint64_t r = sm64_at(sm64_key(seed, (uint64_t)c), (uint64_t)(2 * step));
    return (int)(((r >> 32) * (uint64_t)n) >> 32);
}

__global__ void k_chains_set(const double* __restrict__ amp, int64_t C, const uint64_t* xs, uint64_t nmask,
                             uint64_t* cx, double* cp, int32_t* pend) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    const double re = amp[2 * c], im = amp[2 * c + 1];
    cx[c] = xs[c] & nmask;
    cp[c] = re * re + im * im;
    pend[c] = -1;
    pend[C + c] = -1;
}

// Per-call parameters live in device memory so that a captured graph of steps
// can be replayed: step t of a launch uses global step P->step0 + t.
__global__ void k_mc_set(McParams* P, uint64_t seed, int64_t step0) {
    P->seed = seed;
    P->step0 = step0;
}
__global__ void k_mc_advance(McParams* P, int64_t by) { P->step0 += by; }

__global__ void k_metro_first(int64_t C, const McParams* __restrict__ P, int n, int32_t* jprop, int32_t* jprop2) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    jprop[c] = draw_j(P->seed, c, P->step0, n);
    if (jprop2) jprop2[c] = draw_j(P->seed, c, P->step0 + 1, n);
}

// FP64 accept test (Sec. 4.2) and the proposal index of the next step.
__global__ void k_metro_accept(const float2* __restrict__ partial, int64_t n_tiles,
                               const McParams* __restrict__ P, int64_t t, int n, uint64_t* cx, double* cp,
                               int32_t* pend, int32_t* jprop, uint64_t* trace, int64_t C) {
    const int64_t c = blockIdx.x;
    const double py = chain_reduce(partial, c, n_tiles);
    const uint64_t seed = P->seed;
    const int64_t step = P->step0 + t;
    if (threadIdx.x == 0) {
        const double px = cp[c];
        const int j = jprop[c];
        bool acc;
        if (py >= px) {
            acc = true;
        } else {
            const double r = sm64_unit(sm64_at(sm64_key(seed, (uint64_t)c), (uint64_t)(2 * step + 1)));
            acc = r < py / px;
        }
        if (acc) {
            cx[c] ^= 1ull << j;
            cp[c] = py;
            pend[c] = j;
        } else {
            pend[c] = -1;
        }
        pend[C + c] = -1;
        if (trace) trace[c] = cx[c];
        jprop[c] = draw_j(seed, c, step + 1, n);
    }
}

// The two decisions of a two-step pass (steps t and t + 1), each the FP64 test of
// k_metro_accept with the same draws: step t + 1 compares the sum of the string it
// proposes from the state step t left.  Sums in partial: [0] y1, [1] y1 ^ e_j2,
// [2] x ^ e_j2; proposals j1 = jprop[c], j2 = jprop[C + c].
__global__ void k_metro_accept2(const float2* __restrict__ partial, int64_t n_tiles,
                                const McParams* __restrict__ P, int64_t t, int n, uint64_t* cx, double* cp,
                                int32_t* pend, int32_t* jprop, uint64_t* trace, int64_t C) {
    // the three sums, by as many groups of 256 threads as the block has (three or one)
    __shared__ double prob[3];
    const int64_t c = blockIdx.x;
    for (int r = threadIdx.x >> 8; r < 3; r += blockDim.x >> 8) {
        const double pr = chain_reduce(partial + r * C * n_tiles, c, n_tiles);
        if ((threadIdx.x & 255) == 0) prob[r] = pr;
        __syncthreads();
    }
    const double p1 = prob[0], p2a = prob[1], p2r = prob[2];
    if (threadIdx.x == 0) {
        const uint64_t seed = P->seed;
        const uint64_t key = sm64_key(seed, (uint64_t)c);
        const int64_t step = P->step0 + t;
        const int j1 = jprop[c], j2 = jprop[C + c];
        uint64_t x = cx[c];
        double px = cp[c];
        bool a1;
        if (p1 >= px) a1 = true;
        else a1 = sm64_unit(sm64_at(key, (uint64_t)(2 * step + 1))) < p1 / px;
        if (a1) {
            x ^= 1ull << j1;
            px = p1;
        }
        if (trace) trace[c] = x;
        const double py = a1 ? p2a : p2r;
        bool a2;
        if (py >= px) a2 = true;
        else a2 = sm64_unit(sm64_at(key, (uint64_t)(2 * (step + 1) + 1))) < py / px;
        if (a2) {
            x ^= 1ull << j2;
            px = py;
        }
        if (trace) trace[C + c] = x;
        cx[c] = x;
        cp[c] = px;
        pend[c] = a1 ? j1 : -1;
        pend[C + c] = a2 ? j2 : -1;
        jprop[c] = draw_j(seed, c, step + 2, n);
        jprop[C + c] = draw_j(seed, c, step + 3, n);
    }
}

// Metropolis-Hastings with an independent learned proposal q: accept y with
// probability min(1, P(y) q(x) / (P(x) q(y))), FP64; the uniform of step t of
// chain c is uniform(seed, c, t).
__global__ void k_mh_accept(const double* __restrict__ ampy, const uint64_t* __restrict__ y,
                            const float* __restrict__ lqy, uint64_t seed, int64_t step, int64_t C,
                            uint64_t* cx, double* cp, float* lqx, uint64_t* trace, int64_t* accepts) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    const double py = ampy[2 * c] * ampy[2 * c] + ampy[2 * c + 1] * ampy[2 * c + 1];
    const double px = cp[c];
    bool acc;
    if (px <= 0.0) {
        acc = true;
    } else {
        const double ratio = (py / px) * exp((double)lqx[c] - (double)lqy[c]);
        const double r = sm64_unit(sm64_at(sm64_key(seed, (uint64_t)c), (uint64_t)step));
        acc = ratio >= 1.0 || r < ratio;
    }
    if (acc) {
        cx[c] = y[c];
        cp[c] = py;
        lqx[c] = lqy[c];
        if (accepts) accepts[c] += 1;
    }
    if (trace) trace[c] = cx[c];
}

// Term-sharded steps: the FP64 sum over tiles of each chain's partial <y|psi_shard>
// (not squared: the shards' sums add before P(y) is formed).
// The pass has applied the pending flips, so they are cleared.
__global__ void k_metro_partial_out(const float2* __restrict__ partial, int64_t n_tiles, double* __restrict__ amp,
                                    int32_t* pend, int64_t C) {
    const int64_t c = blockIdx.x;
    double re = 0.0, im = 0.0;
    for (int64_t t = threadIdx.x; t < n_tiles; t += blockDim.x) {
        const float2 p = partial[c * n_tiles + t];
        re += (double)p.x;
        im += (double)p.y;
    }
    __shared__ double sre[256], sim[256];
    sre[threadIdx.x] = re;
    sim[threadIdx.x] = im;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) {
            sre[threadIdx.x] += sre[threadIdx.x + off];
            sim[threadIdx.x] += sim[threadIdx.x + off];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        amp[2 * c] = sre[0];
        amp[2 * c + 1] = sim[0];
        pend[c] = -1;
        pend[C + c] = -1;
    }
}

// The FP64 accept test of step `step` (Sec. 4.2) on the summed amplitudes of the
// proposals: the same rule and draws as k_metro_accept.
__global__ void k_metro_accept_amp(const double* __restrict__ amp, int64_t C, uint64_t seed, int64_t step,
                                   const int32_t* __restrict__ jprop, uint64_t* cx, double* cp, int32_t* pend,
                                   uint64_t* trace) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    const double py = amp[2 * c] * amp[2 * c] + amp[2 * c + 1] * amp[2 * c + 1];
    const double px = cp[c];
    const int j = jprop[c];
    bool acc;
    if (py >= px) {
        acc = true;
    } else {
        const double r = sm64_unit(sm64_at(sm64_key(seed, (uint64_t)c), (uint64_t)(2 * step + 1)));
        acc = r < py / px;
    }
    if (acc) {
        cx[c] ^= 1ull << j;
        cp[c] = py;
        pend[c] = j;
    } else {
        pend[c] = -1;
    }
    pend[C + c] = -1;
    if (trace) trace[c] = cx[c];
}

// Chains without states (ctx->mc_direct): the strings that step `step` proposes.
__global__ void k_mc_strings(int64_t C, uint64_t seed, int64_t step, int n, const uint64_t* __restrict__ cx,
                             uint64_t* __restrict__ y, int32_t* __restrict__ jprop) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    const int j = draw_j(seed, c, step, n);
    jprop[c] = j;
    y[c] = cx[c] ^ bit64(j);
}

__global__ void k_chains_set_prob(const double* __restrict__ amp, int64_t C, double* cp) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < C) cp[c] = amp[2 * c] * amp[2 * c] + amp[2 * c + 1] * amp[2 * c + 1];
}

__global__ void k_metro_out(int64_t C, const uint64_t* cx, const double* cp, uint64_t* x_out,
                            double* p_out) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    if (x_out) x_out[c] = cx[c];
    if (p_out) p_out[c] = cp[c];
}

}  // namespace

// Pointers into ctx->mc_planes (layout of McView).
static size_t mc_layout(const lrs_ctx* ctx, McView* V) {
    const int n = ctx->n;
    const int64_t cols = ctx->cap / 64;
    const size_t plane = (size_t)cols * sizeof(uint2);
    char* p = (char*)ctx->mc_planes;
    size_t at = 0;
    auto take = [&](size_t planes) {
        char* q = p + at;
        at += planes * plane;
        return q;
    };
    McView v;
    v.n = n;
    v.cols = cols;
    v.base = (float2*)take(64);
    v.J = (uint2*)take(mc_pairs(n) + 1);
    v.D = (uint2*)take(2 * n);
    v.pairs = (n + 1) / 2;
    v.K = (uint4*)take((size_t)2 * n * v.pairs);
    v.target = (uint4*)take((size_t)2 * v.pairs);
    v.mf = (uint8_t*)take(1);   // cols / 4 bytes
    if (V) *V = v;
    return at;
}

size_t mc_planes_bytes(const lrs_ctx* ctx) { return mc_layout(ctx, nullptr); }
size_t mc_state_bytes(const lrs_ctx* ctx, int64_t chains) {
    return (size_t)(MC_PLANES + 2 * ((ctx->n + 1) / 2)) * chains * (ctx->cap / 64) * sizeof(uint2);
}

// Columns per block: 128, fewer (a power of two) for a context of fewer terms, whose
// blocks then take several chains at a time.
static int mc_columns(int64_t cols) {
    int t = MC_COLS;
    while (t > 4 && t / 2 >= cols) t /= 2;
    return t;
}

// States and P(x) of the chains at strings x.
static lrs_status mc_start(lrs_ctx* ctx, const uint64_t* x, cudaStream_t st) {
    const int64_t C = ctx->n_chains;
    if (!ctx->mc_direct) {
        McView V;
        mc_layout(ctx, &V);
        // as many threads a (chain, column) as leave no more than two rounds of 2048 an SM
        int split = 8;
        while (split > 1 && C * V.cols * split > (int64_t)4096 * ctx->sm_count) split /= 2;
        const int tbx = split > 1 ? 32 / split : mc_columns(V.cols), nsub = MC_TPB / (tbx * split);
        const int64_t cblocks = (C + nsub - 1) / nsub, blocks = (V.cols + tbx - 1) / tbx * cblocks;
        if (blocks > 0x7FFFFFFF) return lrs_fail(LRS_ERR_UNSUPPORTED, "chain start grid too large");
        k_mc_start<<<(unsigned)blocks, MC_TPB, 0, st>>>(V, C, (uint2*)ctx->Q, x, ctx->nmask, tbx, split, cblocks);
        LRS_LAUNCH_CHECK("chain start kernel");
    }
    double* amp = nullptr;
    lrs_status rc = launch_amplitude_start(ctx, x, C, &amp, st);
    if (rc != LRS_OK) return rc;
    k_chains_set<<<(unsigned)((C + 127) / 128), 128, 0, st>>>(amp, C, x, ctx->nmask, ctx->cx, ctx->cp, ctx->pend);
    LRS_LAUNCH_CHECK("chains_set kernel");
    return LRS_OK;
}

lrs_status launch_chains_init(lrs_ctx* ctx, const uint64_t* x, cudaStream_t st) {
    // the planes of the current terms, then the chains' states and probabilities
    if (ctx->mc_direct) return mc_start(ctx, x, st);
    McView V;
    mc_layout(ctx, &V);
    const size_t smem = (size_t)ctx->n * 256 * sizeof(uint64_t);
    if (!lrs_capturing(st))
        LRS_CUDA(cudaFuncSetAttribute(k_mc_planes, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(62 * 256 * sizeof(uint64_t))));
    const int64_t tiles = ctx->cap / MC_TERMS;
    int parts = 8;
    while (parts > 1 && tiles * parts > ctx->sm_count) parts /= 2;
    k_mc_planes<<<dim3((unsigned)tiles, (unsigned)parts), 256 * MC_SETS, smem, st>>>(ctx->view(), V);
    LRS_LAUNCH_CHECK("chain planes kernel");
    return mc_start(ctx, x, st);
}

// One pass of `steps` (1 or 2) steps.
static lrs_status mc_pass(lrs_ctx* ctx, int steps, const int32_t* jprop, float2* partial, cudaStream_t st) {
    McView V;
    mc_layout(ctx, &V);
    const int64_t C = ctx->n_chains;
    const int tbx = mc_columns(V.cols), nsub = MC_TPB / tbx;
    const int64_t tblocks = (V.cols + tbx - 1) / tbx;
    // chains per block: up to the tuned number and what leaves room for three blocks per
    // SM, fewer while the grid is under four rounds of them (a block's coefficients are
    // one copy of 64 KB)
    const int64_t want = ((int64_t)12 * ctx->sm_count + tblocks - 1) / tblocks;
    int64_t cg = (C + want - 1) / want;
    if (cg < nsub) cg = nsub;
    if (cg > ctx->tune_mc_cg) cg = ctx->tune_mc_cg;
    if (cg > MC_CG) cg = MC_CG;
    const int64_t groups = (C + cg - 1) / cg, blocks = tblocks * groups;
    if (blocks > 0x7FFFFFFF) return lrs_fail(LRS_ERR_UNSUPPORTED, "Metropolis grid too large");
    const size_t smem = (size_t)64 * tbx * sizeof(float2) + cg * sizeof(McChain);
    const auto kernel = steps == 2 ? k_mc_pass<2> : k_mc_pass<1>;
    kernel<<<(unsigned)blocks, MC_TPB, smem, st>>>(V, C, (uint2*)ctx->Q, ctx->cx, ctx->pend, jprop, partial, (int)cg,
                                                   groups, tbx, ctx->mc_err_d);
    LRS_LAUNCH_CHECK("metropolis pass kernel");
    return LRS_OK;
}

static lrs_status mc_attributes(cudaStream_t st) {
    // inside a graph capture the attributes were set by an earlier uncaptured call
    if (lrs_capturing(st)) return LRS_OK;
    const int most = (int)(64 * MC_COLS * sizeof(float2) + MC_CG * sizeof(McChain));
    LRS_CUDA(cudaFuncSetAttribute(k_mc_pass<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    LRS_CUDA(cudaFuncSetAttribute(k_mc_pass<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    return LRS_OK;
}

// Enqueue steps t0 .. t0 + count - 1 (relative to P->step0) of the flip chains.
static lrs_status enqueue_steps(lrs_ctx* ctx, int64_t t0, int64_t count, float2* partial, int32_t* jprop,
                                uint64_t* trace, cudaStream_t st) {
    const int64_t C = ctx->n_chains;
    const int64_t n_tiles = ctx->cap / MC_TERMS;
    lrs_status rc;
    int64_t t = t0;
    if (ctx->tune_mc_lookahead == 2) {
        for (; t + 1 < t0 + count; t += 2) {
            if ((rc = mc_pass(ctx, 2, jprop, partial, st)) != LRS_OK) return rc;
            // three groups where the sums are long, or where there are too few chains to fill the GPU
            const int tpb = n_tiles >= 1024 || C <= 2 * ctx->sm_count ? 768 : 256;
            k_metro_accept2<<<(unsigned)C, tpb, 0, st>>>(partial, n_tiles, ctx->mc_par, t, ctx->n, ctx->cx,
                                                          ctx->cp, ctx->pend, jprop,
                                                          trace ? trace + t * C : nullptr, C);
            LRS_LAUNCH_CHECK("metropolis two-step accept kernel");
        }
    }
    for (; t < t0 + count; ++t) {
        if ((rc = mc_pass(ctx, 1, jprop, partial, st)) != LRS_OK) return rc;
        k_metro_accept<<<(unsigned)C, 256, 0, st>>>(partial, n_tiles, ctx->mc_par, t, ctx->n, ctx->cx,
                                                     ctx->cp, ctx->pend, jprop,
                                                     trace ? trace + t * C : nullptr, C);
        LRS_LAUNCH_CHECK("metropolis accept kernel");
    }
    return LRS_OK;
}

// One CUDA graph holding LRS_MC_GRAPH_STEPS steps followed by step0 += steps;
// rebuilt whenever one of the buffers it was captured with changes: each of them by its own
// address, as any may come back to an old one alone (fewer chains after more reallocate cx, cp and
// pend, and may find the states and planes where they were).
static lrs_status mc_graph(lrs_ctx* ctx, float2* partial, int32_t* jprop, cudaGraphExec_t* out) {
    const void* key[9] = {partial, jprop, ctx->Q, ctx->mc_planes, ctx->cx, ctx->cp, ctx->pend,
                          (void*)(intptr_t)((ctx->n_chains * 128 + ctx->tune_mc_cg) * 4 + ctx->tune_mc_lookahead),
                          (void*)(intptr_t)ctx->cap};
    if (ctx->mc_exec && memcmp(key, ctx->mc_key, sizeof(key)) == 0) {
        *out = (cudaGraphExec_t)ctx->mc_exec;
        return LRS_OK;
    }
    if (ctx->mc_exec) cudaGraphExecDestroy((cudaGraphExec_t)ctx->mc_exec);
    ctx->mc_exec = nullptr;
    if (!ctx->cap_stream) LRS_CUDA(cudaStreamCreateWithFlags((cudaStream_t*)&ctx->cap_stream, cudaStreamNonBlocking));
    cudaStream_t cs = (cudaStream_t)ctx->cap_stream;
    LRS_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    lrs_status rc = enqueue_steps(ctx, 0, LRS_MC_GRAPH_STEPS, partial, jprop, nullptr, cs);
    if (rc == LRS_OK) {
        k_mc_advance<<<1, 1, 0, cs>>>(ctx->mc_par, LRS_MC_GRAPH_STEPS);
        if (cudaGetLastError() != cudaSuccess) rc = lrs_fail(LRS_ERR_CUDA, "graph advance kernel");
    }
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(cs, &g);
    if (rc != LRS_OK) {
        if (g) cudaGraphDestroy(g);
        return rc;
    }
    if (e != cudaSuccess) return lrs_cuda_check(e, "cudaStreamEndCapture");
    cudaGraphExec_t ex = nullptr;
    e = cudaGraphInstantiate(&ex, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return lrs_cuda_check(e, "cudaGraphInstantiate");
    ctx->mc_exec = ex;
    memcpy(ctx->mc_key, key, sizeof(key));
    *out = ex;
    return LRS_OK;
}

// The mapped host words of the propose kernels: [0] a stage wait gave up, [1] a
// one-shot test request (lrs_debug_inject_wait_timeout).
lrs_status mc_flags(lrs_ctx* ctx) {
    if (ctx->mc_err_h) return LRS_OK;
    LRS_CUDA(cudaHostAlloc((void**)&ctx->mc_err_h, 2 * sizeof(int), cudaHostAllocMapped));
    ctx->mc_err_h[0] = 0;
    ctx->mc_err_h[1] = 0;
    LRS_CUDA(cudaHostGetDevicePointer((void**)&ctx->mc_err_d, ctx->mc_err_h, 0));
    return LRS_OK;
}

// Strings that every chain without states proposes (ybuf, their flips in jbuf).
static lrs_status mc_propose_strings(lrs_ctx* ctx, uint64_t seed, int64_t step, cudaStream_t st) {
    const int64_t C = ctx->n_chains;
    lrs_status rc = lrs_ensure((void**)&ctx->jbuf, &ctx->jbuf_bytes, (size_t)C * sizeof(int32_t));
    if (rc != LRS_OK) return rc;
    k_mc_strings<<<(unsigned)((C + 127) / 128), 128, 0, st>>>(C, seed, step, ctx->n, ctx->cx, ctx->ybuf, ctx->jbuf);
    LRS_LAUNCH_CHECK("proposal strings kernel");
    return LRS_OK;
}

// Steps of chains without states: the amplitudes of the proposed strings over all terms, the same
// draws and the same FP64 test.  No memory per (chain, term), at an amplitude call per step
// (41 strings of 2^24 terms at n = 40: 25 ms).
static lrs_status mc_direct_steps(lrs_ctx* ctx, int64_t steps, uint64_t seed, int64_t step0, uint64_t* trace,
                                  cudaStream_t st) {
    const int64_t C = ctx->n_chains;
    for (int64_t t = 0; t < steps; ++t) {
        double* amp = nullptr;
        lrs_status rc = mc_propose_strings(ctx, seed, step0 + t, st);
        if (rc == LRS_OK) rc = launch_amplitude_start(ctx, ctx->ybuf, C, &amp, st);
        if (rc == LRS_OK) rc = launch_metropolis_accept(ctx, amp, seed, step0 + t, trace ? trace + t * C : nullptr, st);
        if (rc != LRS_OK) return rc;
    }
    return LRS_OK;
}

lrs_status launch_metropolis(lrs_ctx* ctx, int64_t steps, uint64_t seed, int64_t step0,
                             uint64_t* x_out, double* p_out, uint64_t* trace, cudaStream_t st) {
    const int64_t C = ctx->n_chains;
    if (ctx->mc_direct) {
        const lrs_status rd = mc_direct_steps(ctx, steps, seed, step0, trace, st);
        if (rd != LRS_OK) return rd;
        k_metro_out<<<(unsigned)((C + 127) / 128), 128, 0, st>>>(C, ctx->cx, ctx->cp, x_out, p_out);
        LRS_LAUNCH_CHECK("metropolis out kernel");
        return LRS_OK;
    }
    const int64_t n_tiles = ctx->cap / MC_TERMS;
    void* scr = nullptr;
    // partial sums: three per chain and tile for two-step passes; proposals j_t, j_{t+1}
    const size_t part_bytes = 3 * (size_t)C * n_tiles * sizeof(float2);
    lrs_status rc = lrs_scratch(ctx, part_bytes + 2 * (size_t)C * sizeof(int32_t) + 256, &scr);
    if (rc != LRS_OK) return rc;
    if (!ctx->mc_par) LRS_CUDA(cudaMalloc(&ctx->mc_par, sizeof(McParams)));
    lrs_status rf = mc_flags(ctx);
    if (rf != LRS_OK) return rf;
    if (*(volatile int*)ctx->mc_err_h) {   // set by an earlier propose launch that gave up waiting
        *(volatile int*)ctx->mc_err_h = 0;
        return lrs_fail(LRS_ERR_TIMEOUT, "a Metropolis propose kernel gave up waiting for its copies");
    }
    // inside a graph capture the steps are captured as plain launches (no nested graph)
    const bool capturing = lrs_capturing(st);
    if ((rc = mc_attributes(st)) != LRS_OK) return rc;
    float2* partial = (float2*)scr;
    int32_t* jprop = (int32_t*)((char*)scr + ((part_bytes + 255) & ~(size_t)255));
    k_mc_set<<<1, 1, 0, st>>>(ctx->mc_par, seed, step0);
    k_metro_first<<<(unsigned)((C + 127) / 128), 128, 0, st>>>(C, ctx->mc_par, ctx->n, jprop, jprop + C);
    LRS_LAUNCH_CHECK("metropolis first kernel");
    int64_t done = 0;
    if (!trace && !capturing && steps >= LRS_MC_GRAPH_STEPS) {
        // replay a captured graph of LRS_MC_GRAPH_STEPS steps (one launch instead of 2 per step)
        cudaGraphExec_t ex = nullptr;
        rc = mc_graph(ctx, partial, jprop, &ex);
        if (rc != LRS_OK) return rc;
        for (; done + LRS_MC_GRAPH_STEPS <= steps; done += LRS_MC_GRAPH_STEPS)
            LRS_CUDA(cudaGraphLaunch(ex, st));
    }
    rc = enqueue_steps(ctx, trace ? 0 : 0, steps - done, partial, jprop, trace, st);
    if (rc != LRS_OK) return rc;
    k_metro_out<<<(unsigned)((C + 127) / 128), 128, 0, st>>>(C, ctx->cx, ctx->cp, x_out, p_out);
    LRS_LAUNCH_CHECK("metropolis out kernel");
    return LRS_OK;
}

// One term-sharded proposal: every chain's partial amplitude of its proposal y over
// this context's terms (the pending flip of the previous step is applied to Q first).
lrs_status launch_metropolis_propose(lrs_ctx* ctx, uint64_t seed, int64_t step, double* amp, cudaStream_t st) {
    const int64_t C = ctx->n_chains;
    lrs_status rc;
    if (ctx->mc_direct) {
        if ((rc = mc_propose_strings(ctx, seed, step, st)) != LRS_OK) return rc;
        return launch_amplitude(ctx, ctx->ybuf, C, amp, nullptr, st);
    }
    const int64_t n_tiles = ctx->cap / MC_TERMS;
    void* scr = nullptr;
    if ((rc = lrs_scratch(ctx, (size_t)C * n_tiles * sizeof(float2), &scr)) != LRS_OK) return rc;
    if (!ctx->mc_par) LRS_CUDA(cudaMalloc(&ctx->mc_par, sizeof(McParams)));
    if ((rc = lrs_ensure((void**)&ctx->jbuf, &ctx->jbuf_bytes, (size_t)C * sizeof(int32_t))) != LRS_OK) return rc;
    if ((rc = mc_flags(ctx)) != LRS_OK) return rc;
    if (*(volatile int*)ctx->mc_err_h) {
        *(volatile int*)ctx->mc_err_h = 0;
        return lrs_fail(LRS_ERR_TIMEOUT, "a Metropolis propose kernel gave up waiting for its copies");
    }
    if ((rc = mc_attributes(st)) != LRS_OK) return rc;
    k_mc_set<<<1, 1, 0, st>>>(ctx->mc_par, seed, step);
    k_metro_first<<<(unsigned)((C + 127) / 128), 128, 0, st>>>(C, ctx->mc_par, ctx->n, ctx->jbuf, nullptr);
    LRS_LAUNCH_CHECK("metropolis first kernel");
    float2* partial = (float2*)scr;
    if ((rc = mc_pass(ctx, 1, ctx->jbuf, partial, st)) != LRS_OK) return rc;
    k_metro_partial_out<<<(unsigned)C, 256, 0, st>>>(partial, n_tiles, amp, ctx->pend, C);
    LRS_LAUNCH_CHECK("metropolis partial amplitude kernel");
    return LRS_OK;
}

lrs_status launch_metropolis_accept(lrs_ctx* ctx, const double* amp, uint64_t seed, int64_t step, uint64_t* trace,
                                    cudaStream_t st) {
    const int64_t C = ctx->n_chains;
    k_metro_accept_amp<<<(unsigned)((C + 127) / 128), 128, 0, st>>>(amp, C, seed, step, ctx->jbuf, ctx->cx, ctx->cp,
                                                                     ctx->pend, trace);
    LRS_LAUNCH_CHECK("metropolis accept kernel");
    return LRS_OK;
}

lrs_status launch_chains_set_prob(lrs_ctx* ctx, const double* amp, cudaStream_t st) {
    const int64_t C = ctx->n_chains;
    k_chains_set_prob<<<(unsigned)((C + 127) / 128), 128, 0, st>>>(amp, C, ctx->cp);
    LRS_LAUNCH_CHECK("chain probability kernel");
    return LRS_OK;
}

lrs_status mh_buffers(lrs_ctx* ctx, int64_t C) {
    if (C <= ctx->mh_cap) return LRS_OK;
    cudaFree(ctx->ybuf); cudaFree(ctx->lqy); cudaFree(ctx->lqx); cudaFree(ctx->ampy);
    ctx->ybuf = nullptr; ctx->lqy = nullptr; ctx->lqx = nullptr; ctx->ampy = nullptr;
    ctx->mh_cap = 0;
    LRS_CUDA(cudaMalloc(&ctx->ybuf, (size_t)C * sizeof(uint64_t)));
    LRS_CUDA(cudaMalloc(&ctx->lqy, (size_t)C * sizeof(float)));
    LRS_CUDA(cudaMalloc(&ctx->lqx, (size_t)C * sizeof(float)));
    LRS_CUDA(cudaMalloc(&ctx->ampy, (size_t)C * 2 * sizeof(double)));
    ctx->mh_cap = C;
    return LRS_OK;
}

lrs_status launch_metropolis_learned(lrs_ctx* ctx, lrs_mlp* mlp, int64_t steps, uint64_t seed, int64_t step0,
                                     uint64_t* x_out, double* p_out, uint64_t* trace, int64_t* accepts,
                                     cudaStream_t st) {
    const int64_t C = ctx->n_chains;
    lrs_status rc = mh_buffers(ctx, C);
    if (rc != LRS_OK) return rc;
    // log q of the current states under the current network
    rc = lrs_mlp_forward(mlp, ctx->cx, C, nullptr, ctx->lqx, st);
    if (rc != LRS_OK) return rc;
    for (int64_t t = 0; t < steps; ++t) {
        const int64_t step = step0 + t;
        rc = lrs_mlp_sample(mlp, C, seed, step * C, ctx->ybuf, ctx->lqy, st);
        if (rc != LRS_OK) return rc;
        rc = launch_amplitude(ctx, ctx->ybuf, C, ctx->ampy, nullptr, st);
        if (rc != LRS_OK) return rc;
        k_mh_accept<<<(unsigned)((C + 127) / 128), 128, 0, st>>>(ctx->ampy, ctx->ybuf, ctx->lqy, seed, step, C,
                                                                  ctx->cx, ctx->cp, ctx->lqx,
                                                                  trace ? trace + t * C : nullptr, accepts);
        LRS_LAUNCH_CHECK("learned MH accept kernel");
    }
    ctx->q_stale = true;
    k_metro_out<<<(unsigned)((C + 127) / 128), 128, 0, st>>>(C, ctx->cx, ctx->cp, x_out, p_out);
    LRS_LAUNCH_CHECK("metropolis out kernel");
    return LRS_OK;
}

// Rebuild the states for the chains' current strings (after learned moves).  The strings are
// copied into the learned proposal's buffer (free at this point) because chains_set
// rewrites cx.
lrs_status launch_chains_refresh(lrs_ctx* ctx, cudaStream_t st) {
    const int64_t C = ctx->n_chains;
    if (!ctx->ybuf || ctx->mh_cap < C) return lrs_fail(LRS_ERR_STATE, "chain refresh without a learned-move buffer");
    LRS_CUDA(cudaMemcpyAsync(ctx->ybuf, ctx->cx, (size_t)C * 8, cudaMemcpyDeviceToDevice, st));
    const lrs_status rc = mc_start(ctx, ctx->ybuf, st);
    if (rc != LRS_OK) return rc;
    ctx->q_stale = false;
    return LRS_OK;
}
