// Batched amplitudes <x|psi> = sum_alpha b_alpha <x|phi_alpha> (Eqs. (amplitude),
// (amplitude1)).
//
// For each (x, term) the Pauli Q = prod_{p: x_p = 1} U_C^{-1} X_p U_C is written
// i^mu X(u) Z(w); taking the rows in increasing p,
//     z ^= w & F_p;  u ^= F_p;  w ^= M_p,   mu = x.gamma + 2 parity(z)  (mod 4).
// The rows are grouped four at a time (Four Russians): for the current term the
// block builds a shared table, per 4-row chunk c and pattern q of x's bits
// 4c..4c+3, of (u_q, w_q, z_q) restricted to those rows; a chunk then enters as
//     z ^= (w & u_q) ^ z_q;  u ^= u_q;  w ^= w_q.
// One thread owns XP strings x and walks the block's tile of terms, so its
// chi-sum is a private FP32 Kahan sum (no cross-thread reduction); the tile
// partials are summed in FP64 by k_amp_reduce.
#include <string.h>

#include <atomic>

#include "lrs_device.cuh"

namespace {

constexpr int AMP_XT = 128;   // threads per block
// strings per thread (independent chains for ILP): each term's tables and barrier
// serve 1024 strings
constexpr int AMP_XP = 8, AMP_XB = AMP_XT * AMP_XP;

struct AmpEntry {
    uint64_t u, w, z;
};

// PK (n <= 62): only parity(z) enters mu, and parity(z_after) = parity(z) +
// parity(w & u_q) + parity(z_q), so a table entry keeps parity(z_q) in bit 63 of u_q
// and the lookups XOR-accumulate w & u_q (one popcount per string at the end): two
// 8-byte tables (u_q, w_q) instead of three, each a conflict-free 128-byte row per
// chunk.
// Register budget: five blocks per SM (96 registers, eight strings per thread).
// ERR: also sum |b_alpha <x|phi_alpha>| over the terms that contribute at x (one FP32
// add per contributing (x, term)), written to magp[i * n_tiles + tile]: the input of
// the per-result error bound of k_amp_reduce.
// One block of the amplitude launch: term tile `tile`, strings xblk * AMP_XB ... (shared
// by the single-circuit kernel and the batched kernel of several circuits).
template <int NCH, bool PK, bool ERR>
__device__ __forceinline__ void amp_block(const TermsView& T, const uint64_t* __restrict__ xs, int64_t batch,
                                          int64_t tt, float2* __restrict__ partial, int64_t n_tiles,
                                          float* __restrict__ magp, int64_t tile,
                                          int64_t xblk) {
    // One barrier per term: while the block evaluates term a from table slot a, it
    // builds the table of term a + 1 (from the rows stored in the previous interval)
    // and stores the rows of term a + 2; tables and rows are double-buffered, the
    // per-term scalars (read while the scalars of a + 2 are written) triple-buffered.
    __shared__ AmpEntry tab[2][PK ? 1 : NCH][16];
    __shared__ uint64_t tabU[2][PK ? NCH : 1][16], tabW[2][PK ? NCH : 1][16];
    __shared__ uint64_t sF[2][64], sM[2][64];
    __shared__ float2 val8[3][8];           // b e^{i pi k/4} 2^{-(|v|+h)/2}, k = 0..7
    __shared__ float val_abs[3];            // |b| 2^{-(|v|+h)/2} (ERR)
    __shared__ uint64_t sc[3][4];           // glo, ghi, v, s
    __shared__ uint32_t sc_live[3];
    const int n = T.n;
    const int tid = threadIdx.x;
    const int64_t xb = xblk * AMP_XB;
    uint64_t xv[AMP_XP];
#pragma unroll
    for (int k = 0; k < AMP_XP; ++k) {
        const int64_t i = xb + tid + k * AMP_XT;
        xv[k] = i < batch ? (xs[i] & T.nmask) : 0ull;   // bits >= n are ignored
    }
    KahanC acc[AMP_XP];
    float mag[ERR ? AMP_XP : 1];
#pragma unroll
    for (int k = 0; k < AMP_XP; ++k) acc[k].init();
#pragma unroll
    for (int k = 0; k < (ERR ? AMP_XP : 1); ++k) mag[k] = 0.f;

    const int64_t a0 = tile * tt;
    const int64_t a1 = (a0 + tt < T.cap) ? a0 + tt : T.cap;
    // register prefetch of the next term: threads < n hold rows, threads 64..66 scalars
    // (thread 66 keeps its own copy of v: it must not read sc[2], which thread 65
    // writes in the same barrier interval)
    uint64_t pf = 0, pm = 0, pv = 0;
    auto prefetch = [&](int64_t a) {
        if (tid < n) {
            pf = T.F[(int64_t)tid * T.cap + a];
            pm = T.M[(int64_t)tid * T.cap + a];
        } else if (tid == 64) {
            pf = T.glo[a]; pm = T.ghi[a];
        } else if (tid == 65) {
            pf = T.v[a]; pm = T.s[a];
        } else if (tid == 66) {
            pf = T.omega[a];
            const float2 b = T.coef[a];
            pm = (uint64_t)__float_as_uint(b.x) | ((uint64_t)__float_as_uint(b.y) << 32);
            pv = T.v[a];
        }
    };
    // thread-owned stores of the prefetched term into row slot rs and scalar slot ss
    auto store = [&](int rs, int ss) {
        if (tid < n) { sF[rs][tid] = pf; sM[rs][tid] = pm; }
        if (tid == 64) { sc[ss][0] = pf; sc[ss][1] = pm; }
        if (tid == 65) { sc[ss][2] = pf; sc[ss][3] = pm; }
        if (tid == 66) {
            const uint32_t om = (uint32_t)pf;
            const float2 b = make_float2(__uint_as_float((uint32_t)pm), __uint_as_float((uint32_t)(pm >> 32)));
            sc_live[ss] = ((om >> 3) & 1u) ? 0u : 1u;
            const int e0 = __popcll(pv) + (int)(om >> 8);
#pragma unroll
            for (int k = 0; k < 8; ++k) val8[ss][k] = z8_scale(b, k + (int)(om & 7u), e0);
            if (ERR) val_abs[ss] = ldexpf(hypotf(b.x, b.y), -(e0 >> 1)) * ((e0 & 1) ? 0.70710678f : 1.f);
        }
    };
    // the Four-Russians table of the term whose rows are in slot ts, into table slot ts
    auto build = [&](int ts) {
        for (int e = tid; e < NCH * 16; e += AMP_XT) {
            const int c = e >> 4, q = e & 15;
            uint64_t u = 0, w = 0, z = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int r = 4 * c + b;
                if (((q >> b) & 1) && r < n) {
                    const uint64_t Fr = sF[ts][r];
                    z ^= w & Fr;
                    u ^= Fr;
                    w ^= sM[ts][r];
                }
            }
            if (PK) {
                tabU[ts][c][q] = u | ((uint64_t)par64(z) << 63);
                tabW[ts][c][q] = w;
            } else {
                tab[ts][c][q].u = u;
                tab[ts][c][q].w = w;
                tab[ts][c][q].z = z;
            }
        }
    };
    if (a0 < a1) { prefetch(a0); store(0, 0); }
    if (a0 + 1 < a1) { prefetch(a0 + 1); store(1, 1); }
    if (a0 + 2 < a1) prefetch(a0 + 2);
    __syncthreads();
    if (a0 < a1) build(0);
    __syncthreads();
    for (int64_t a = a0; a < a1; ++a) {
        const int kt = (int)(a - a0);
        const int tb = kt & 1, ss = kt % 3;
        if (a + 1 < a1) build(tb ^ 1);
        if (a + 2 < a1) store(tb, (kt + 2) % 3);
        if (a + 3 < a1) prefetch(a + 3);
        const bool live = sc_live[ss] != 0u;
        if (live) {
            const uint64_t glo = sc[ss][0], ghi = sc[ss][1], v = sc[ss][2], s = sc[ss][3];
            const uint64_t nv = ~v & T.nmask, sv = s & v;
    #pragma unroll
            for (int k = 0; k < AMP_XP; ++k) {
                const uint64_t x = xv[k];
                uint64_t u = 0, w = 0;
                uint32_t zpar;
                if (PK) {
                    // only the parity of sum_c popc(w_c & u_q) enters, and that is the
                    // parity of the XOR of the terms: one popcount per string
                    uint64_t zx = 0;
    #pragma unroll
                    for (int c = 0; c < NCH; ++c) {
                        const int q = (int)((x >> (4 * c)) & 15u);
                        const uint64_t Eu = tabU[tb][c][q], Ew = tabW[tb][c][q];
                        zx ^= w & Eu;   // w has no bit 63
                        u ^= Eu;
                        w ^= Ew;
                    }
                    zpar = ((uint32_t)__popcll(zx) + (uint32_t)(u >> 63)) & 1u;
                    u &= ~(1ull << 63);
                } else {
                    uint64_t z = 0;
    #pragma unroll
                    for (int c = 0; c < NCH; ++c) {
                        const AmpEntry& E = tab[tb][c][(int)((x >> (4 * c)) & 15u)];
                        z ^= (w & E.u) ^ E.z;
                        u ^= E.u;
                        w ^= E.w;
                    }
                    zpar = par64(z);
                }
                const int mu = __popcll(x & glo) + 2 * __popcll(x & ghi) + 2 * (int)zpar;
                if (((u ^ s) & nv) == 0) {
                    const int sign = (int)par64(u & (w ^ sv));
                    acc[k].add(val8[ss][(2 * mu + 4 * sign) & 7]);
                    if (ERR) mag[k] += val_abs[ss];
                }
            }
        }
        __syncthreads();   // slot tb ^ 1 and the next rows and scalars are complete
    }
#pragma unroll
    for (int k = 0; k < AMP_XP; ++k) {
        const int64_t i = xb + tid + k * AMP_XT;
        if (i < batch) {
            partial[i * n_tiles + tile] = acc[k].value();
            if (ERR) magp[i * n_tiles + tile] = mag[ERR ? k : 0];
        }
    }
}

template <int NCH, bool PK, bool ERR>
__global__ void __launch_bounds__(AMP_XT, 5) k_amplitude(TermsView T, const uint64_t* __restrict__ xs,
                                                      int64_t batch, int64_t tt,
                                                      float2* __restrict__ partial, int64_t n_tiles,
                                                      float* __restrict__ magp) {
    amp_block<NCH, PK, ERR>(T, xs, batch, tt, partial, n_tiles, magp, blockIdx.x, blockIdx.y);
}

// Several circuits of the same width in one launch: block b runs block b - first[c]
// of circuit c's own launch shape (term tile fastest), so every circuit gets exactly the
// partial sums of its single-circuit launch; the table is a kernel parameter, so the
// circuit lookup and every value read from it are warp-uniform.
#define LRS_AMP_BATCH_MAX 12
struct AmpBatch {
    int count;
    int64_t first[LRS_AMP_BATCH_MAX + 1];
    TermsView T[LRS_AMP_BATCH_MAX];
    const uint64_t* xs[LRS_AMP_BATCH_MAX];
    int64_t batch[LRS_AMP_BATCH_MAX], tt[LRS_AMP_BATCH_MAX], n_tiles[LRS_AMP_BATCH_MAX];
    float2* partial[LRS_AMP_BATCH_MAX];
    double* out[LRS_AMP_BATCH_MAX];
};

template <int NCH, bool PK>
__global__ void __launch_bounds__(AMP_XT, 5) k_amplitude_batch(const __grid_constant__ AmpBatch B) {
    const int64_t b = blockIdx.x;
    int c = 0;
#pragma unroll 1
    for (int i = 1; i < B.count; ++i)
        if (B.first[i] <= b) c = i;
    const int64_t local = b - B.first[c];
    amp_block<NCH, PK, false>(B.T[c], B.xs[c], B.batch[c], B.tt[c], B.partial[c], B.n_tiles[c], nullptr, local % B.n_tiles[c], local / B.n_tiles[c]);
}

// FP64 sum of the block partials of each x, and (magp != NULL) the error bound of
// that sum against the exact chi-sum:
//   |a_gpu - a| <= (8u + 8 tt u^2)(1 + tt u)(1 + 1e-4) M + n_tiles 2^-52 P,
// u = 2^-24, M = sum over contributing terms of |b_alpha <x|phi_alpha>| (FP32 sums of
// the tiles), P = sum over tiles of |partial|.  Per addend: the FP32 coefficient and
// the FP32 phase/sqrt2 factors of z8_scale give at most 4u |a_alpha|; the Kahan sum of
// a tile of tt addends adds (2u + O(tt u^2)) per real component, 2 sqrt2 u |a_alpha|
// for the complex pair; the final s - c rounding u; M itself is an FP32 sum of tt
// positive values (relative tt u) of magnitudes computed to 1e-4.  The FP64 sum of
// n_tiles partials adds at most n_tiles 2^-53 P per component.
__global__ void k_amp_reduce(const float2* __restrict__ partial, const float* __restrict__ magp, int64_t n_tiles,
                             int64_t batch, int64_t tt, double* __restrict__ out, float* __restrict__ err) {
    const int64_t xi = blockIdx.x;
    if (xi >= batch) return;
    double re = 0.0, im = 0.0, m = 0.0, pa = 0.0;
    for (int64_t t = threadIdx.x; t < n_tiles; t += blockDim.x) {
        const float2 p = partial[xi * n_tiles + t];
        re += (double)p.x;
        im += (double)p.y;
        if (magp) {
            m += (double)magp[xi * n_tiles + t];
            pa += hypot((double)p.x, (double)p.y);
        }
    }
    __shared__ double sre[256], sim[256], sm[256], spa[256];
    sre[threadIdx.x] = re;
    sim[threadIdx.x] = im;
    sm[threadIdx.x] = m;
    spa[threadIdx.x] = pa;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) {
            sre[threadIdx.x] += sre[threadIdx.x + off];
            sim[threadIdx.x] += sim[threadIdx.x + off];
            sm[threadIdx.x] += sm[threadIdx.x + off];
            spa[threadIdx.x] += spa[threadIdx.x + off];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[2 * xi] = sre[0];
        out[2 * xi + 1] = sim[0];
        if (magp) {
            const double u = 5.9604644775390625e-8, ttd = (double)tt;
            const double c = (8.0 * u + 8.0 * ttd * u * u) * (1.0 + ttd * u) * (1.0 + 1e-4);
            err[xi] = (float)((c * sm[0] + (double)n_tiles * 2.220446049250313e-16 * spa[0]) * (1.0 + 1e-6));
        }
    }
}

// The FP64 tile sums of several circuits in one launch: block b is string b - xfirst[c]
// of circuit c (same summation order as k_amp_reduce).
__global__ void k_amp_reduce_batch(const __grid_constant__ AmpBatch B, int64_t total) {
    const int64_t b = blockIdx.x;
    if (b >= total) return;
    int c = 0;
#pragma unroll 1
    for (int i = 1; i < B.count; ++i)
        if (B.first[i] <= b) c = i;
    const int64_t xi = b - B.first[c];
    const float2* partial = B.partial[c];
    const int64_t n_tiles = B.n_tiles[c];
    double re = 0.0, im = 0.0;
    for (int64_t t = threadIdx.x; t < n_tiles; t += blockDim.x) {
        const float2 p = partial[xi * n_tiles + t];
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
        B.out[c][2 * xi] = sre[0];
        B.out[c][2 * xi + 1] = sim[0];
    }
}

// ---- bit-sliced amplitudes -------------------------------------------------------------
// <x|phi> = b omega 2^{-|v|/2} i^{q(x)} where F_k . x = s_k for every k not in v (F_k: column k
// of F), else 0, with the Z4 form
//     q(x) = sum_p d_p x_p + 2 sum_{p<q} J_pq x_p x_q,   J = M F^T,
//     d_p = gamma_p + 2 F_p . M_p + 2 F_p . (s & v),
// or, with sum_p lo_p x_p = P + 2 sum_{p<q} lo_p lo_q x_p x_q (P its parity, lo_p = d_p mod 2),
//     q(x) = P + 2 (hi . x + sum_p x_p (L_p . x)),   L_p = (J_pq + lo_p lo_q) over q < p.
// k_amp_prep writes lo, hi, the rows L_p and the constraints of every term once (a warp per
// term); k_amp_sliced evaluates these linear forms on 32 strings at a time, bit i of a word
// belonging to string i: a form is the XOR, over chunks of six qubits, of one entry of a
// table of the chunk's 64 XORs of string words, which depends on the strings only
// and serves every term.  Per (term, 1024 strings) that is about n^2 / 12 + 1.5 n + n / 6 per
// constraint shared-memory loads of 128 bytes and three integer instructions each, where one
// string per thread takes 8 ceil(n / 4) + 16 instructions for 32 strings.  4096 strings: n = 50,
// chi = 2^20 34.3 -> 12.0 ms, n = 40, chi = 2^16 with bounds 1.95 -> 0.69 ms; 1024 strings of 64
// terms 79 -> 31 us; integer issue bounds it (ALU pipe 72% busy).
constexpr int AS_WARPS = 8, AS_TPB = 32 * AS_WARPS;
constexpr int AS_CB = 6;       // qubits per chunk
constexpr int AS_TERMS = 32;   // terms whose words the block collects before summing
enum { AMP_INFO = 0, AMP_VAL, AMP_LO, AMP_HI, AMP_ROWS };   // record: header, rows L_0.., constraints

struct AmpPrep {
    uint64_t* rec;   // [slots][words]
    int words, rows;   // rows = chunks * AS_CB
    // the launch's terms: r0 .. r0 + rl - 1 of every tile of tt terms; term r0 + j of tile t in
    // slot t rl + j
    int64_t tt, r0;
    int rl;
};

// Records of a launch's terms, eight terms of tile blockIdx.y a block (rl is a multiple of 8): a
// warp per term, lane c holding rows c and c + 32.
__global__ void __launch_bounds__(256) k_amp_prep(TermsView T, AmpPrep P) {
    __shared__ uint64_t sF[8][64];
    const int n = T.n, lane = threadIdx.x & 31;
    const int64_t j = blockIdx.x * 8 + (threadIdx.x >> 5), r = P.r0 + j, a = (int64_t)blockIdx.y * P.tt + r;
    if (r >= P.tt || a >= T.cap) return;
    const uint64_t v = T.v[a], s = T.s[a], glo = T.glo[a], ghi = T.ghi[a];
    const uint32_t om = T.omega[a];
    uint64_t F[2], M[2], J[2] = {0, 0};   // on their way before the flags are known
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int q = lane + 32 * c;
        F[c] = q < n ? T.F[(int64_t)q * T.cap + a] : 0ull;
        M[c] = q < n ? T.M[(int64_t)q * T.cap + a] : 0ull;
    }
    uint64_t* rec = P.rec + ((int64_t)blockIdx.y * P.rl + j) * P.words;
    const bool live = ((om >> 3) & 1u) == 0u;
    const uint64_t out = ~v & T.nmask;
    const int mf = __popcll(out);
    if (lane == 0) {
        const float2 b = T.coef[a];
        const int e0 = __popcll(v) + (int)(om >> 8);
        const float2 val = z8_scale(b, (int)(om & 7u), e0);
        const float mag = ldexpf(hypotf(b.x, b.y), -(e0 >> 1)) * ((e0 & 1) ? 0.70710678f : 1.f);
        rec[AMP_INFO] = (uint64_t)((uint32_t)mf | (live ? 1u << 8 : 0u)) | (uint64_t)__float_as_uint(mag) << 32;
        rec[AMP_VAL] = (uint64_t)__float_as_uint(val.x) | (uint64_t)__float_as_uint(val.y) << 32;
    }
    if (!live) return;
    uint32_t hi[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int q = lane + 32 * c;
        hi[c] = (uint32_t)getb(ghi, q) ^ par64(F[c] & M[c]) ^ par64(F[c] & s & v);
    }
    uint64_t* rows = sF[threadIdx.x >> 5];
    rows[lane] = F[0];
    rows[lane + 32] = F[1];
    __syncwarp();
    lrs_products(rows, n, M[0], M[1], J[0], J[1]);
    const uint64_t hw = (uint64_t)__ballot_sync(0xffffffffu, hi[0]) | (uint64_t)__ballot_sync(0xffffffffu, hi[1]) << 32;
    if (lane == 0) {
        rec[AMP_LO] = glo;
        rec[AMP_HI] = hw & T.nmask;
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int p = lane + 32 * c;
        if (p < P.rows) rec[AMP_ROWS + p] = p < n ? (J[c] ^ (getb(glo, p) ? glo : 0ull)) & (bit64(p) - 1) : 0ull;
    }
    // constraints: the columns of F outside v
    uint64_t ks = out;
    for (int k = 0; k < mf; ++k) {
        const int q = ffs64(ks);
        ks &= ks - 1;
        const uint64_t col = (uint64_t)__ballot_sync(0xffffffffu, (uint32_t)getb(F[0], q)) |
                             (uint64_t)__ballot_sync(0xffffffffu, (uint32_t)getb(F[1], q)) << 32;
        if (lane == 0) rec[AMP_ROWS + P.rows + k] = col;
    }
    if (lane == 0) {
        rec[AMP_ROWS + P.rows + n] = s;       // targets: s_k of the k-th qubit outside v
        rec[AMP_ROWS + P.rows + n + 1] = v;
    }
}

// Linear form w over the first NC chunks: XOR of table entries of this lane's column.  `tab` is the
// shared address of the lane's column; the table starts on an 8 KB boundary, so that
// masking the pattern (times 128 bytes) out of the word and adding the address is one
// three-input operation.
template <int C>
__device__ __forceinline__ uint32_t amp_entry(uint32_t tab, uint32_t lo, uint32_t hi) {
    constexpr int sh = AS_CB * C - 7;
    uint32_t t, a, r;
    if (sh < 0)
        t = lo << (sh < 0 ? -sh : 0);
    else if (sh < 32)
        t = __funnelshift_r(lo, hi, sh >= 0 ? sh : 0);
    else
        t = hi >> (sh >= 32 ? sh - 32 : 0);
    asm("lop3.b32 %0, %1, 0x1f80, %2, 0xea;" : "=r"(a) : "r"(t), "r"(tab));   // (t & 0x1f80) | tab
    asm("ld.shared.u32 %0, [%1 + %2];" : "=r"(r) : "r"(a), "n"(C * 64 * 128));
    return r;
}
template <int NC, int C = 0>
__device__ __forceinline__ uint32_t amp_form(uint32_t tab, uint64_t w) {
    const uint32_t lo = (uint32_t)w, hi = (uint32_t)(w >> 32);
    if constexpr (C + 2 < NC)
        return amp_entry<C>(tab, lo, hi) ^ amp_entry<C + 1>(tab, lo, hi) ^ amp_form<NC, C + 2>(tab, w);
    else if constexpr (C + 2 == NC)
        return amp_entry<C>(tab, lo, hi) ^ amp_entry<C + 1>(tab, lo, hi);
    else
        return amp_entry<C>(tab, lo, hi);
}
template <int P>   // the string words of qubit P
__device__ __forceinline__ uint32_t amp_bit(uint32_t tab) {
    uint32_t r;
    asm("ld.shared.u32 %0, [%1 + %2];" : "=r"(r) : "r"(tab), "n"((P / AS_CB * 64 + (1 << P % AS_CB)) * 128));
    return r;
}

// Rows p = C AS_CB .. of the quadratic part: sum over p of x_p (L_p . x), chunk row by chunk
// row, the next chunk's rows loaded while this one's are evaluated.
struct AmpRows {
    ulonglong2 r[AS_CB / 2];
};
__device__ __forceinline__ AmpRows amp_load(const ulonglong2* __restrict__ rows, int c) {
    AmpRows R;
#pragma unroll
    for (int i = 0; i < AS_CB / 2; ++i) R.r[i] = __ldg(rows + c * (AS_CB / 2) + i);
    return R;
}
template <int NC, int C>
__device__ __forceinline__ void amp_rows(uint32_t tab, const ulonglong2* __restrict__ rows, const AmpRows& cur, int n,
                                         uint32_t& acc) {
    AmpRows next = cur;
    if constexpr (C + 1 < NC) next = amp_load(rows, C + 1);
    constexpr int P = C * AS_CB;
    if (P > 0) acc ^= amp_form<C + 1>(tab, cur.r[0].x) & amp_bit<P>(tab);
    if (C + 1 < NC || P + 1 < n) acc ^= amp_form<C + 1>(tab, cur.r[0].y) & amp_bit<P + 1>(tab);
    if (C + 1 < NC || P + 2 < n) {
        acc ^= amp_form<C + 1>(tab, cur.r[1].x) & amp_bit<P + 2>(tab);
        acc ^= amp_form<C + 1>(tab, cur.r[1].y) & amp_bit<P + 3>(tab);
    }
    if (C + 1 < NC || P + 4 < n) {
        acc ^= amp_form<C + 1>(tab, cur.r[2].x) & amp_bit<P + 4>(tab);
        acc ^= amp_form<C + 1>(tab, cur.r[2].y) & amp_bit<P + 5>(tab);
    }
    if constexpr (C + 1 < NC) amp_rows<NC, C + 1>(tab, rows, next, n, acc);
}

// Kahan sum of the complex pair s with the negated compensation nc, both parts at once (the
// operations of KahanC::add, packed), where `on` is not zero.
__device__ __forceinline__ void kahan_add2(uint64_t& s, uint64_t& nc, float x, float y, uint32_t on) {
    asm("{\n"
        " .reg .pred p;\n .reg .b64 a, t, d, m;\n"
        " setp.ne.u32 p, %4, 0;\n"
        " mov.b64 a, {%2, %3};\n"
        " mov.b64 m, {%5, %5};\n"
        " add.rn.f32x2 a, a, %1;\n"        // x - c
        " add.rn.f32x2 t, %0, a;\n"
        " fma.rn.f32x2 d, t, m, %0;\n"     // s - t
        " @p add.rn.f32x2 %1, a, d;\n"     // -((t - s) - (x - c))
        " @p mov.b64 %0, t;\n"
        "}"
        : "+l"(s), "+l"(nc)
        : "f"(x), "f"(y), "r"(on), "f"(-1.f));
}

// A block: 8 warps, G = 32 / wl term tiles (wl string words of 32 strings each, a power of
// two: 32 for 1024 strings and one tile).  Lane (g, l) = (lane / wl, lane % wl) holds
// word l for tile g.  The warps first evaluate AS_TERMS terms of every tile, one term each at
// a time, leaving three words per lane and term (live, phase bits); then thread (warp, lane)
// adds up the four strings 4 warp .. 4 warp + 3 of its lane's word, in term order, so every
// string's Kahan sum over a tile is the one a single thread would form; a sum that a later
// launch continues (more) is left as it stands, its compensation in `comp`.
// The table takes 8 KB per chunk (72 KB at n = 50): two blocks an SM.
template <int NC, bool ERR>
__global__ void __launch_bounds__(AS_TPB, 2) k_amp_sliced(AmpPrep P, int n, uint64_t nmask, const uint64_t* __restrict__ xs,
                                                          int64_t batch, int64_t cap, int64_t n_tiles, int wl,
                                                          int64_t tgroups, bool more, float2* __restrict__ partial,
                                                          float2* __restrict__ comp, float* __restrict__ magp) {
    // shared memory: table (on an 8 KB boundary), then the collected words and values, whose
    // place holds the string words while the table is built
    extern __shared__ __align__(16) unsigned char dyn[];
    const uint32_t dyn0 = (uint32_t)__cvta_generic_to_shared(dyn);
    const uint32_t tab0 = (dyn0 + 8191u) & ~8191u;
    uint32_t* tabw = reinterpret_cast<uint32_t*>(dyn + (tab0 - dyn0));                             // [NC][64][32]
    uint32_t(*sw)[3][32] = reinterpret_cast<uint32_t(*)[3][32]>(tabw + NC * 64 * 32);              // live, phase bits
    uint32_t(*sx)[32] = &sw[0][0];                                                                 // [NC AS_CB][32]
    float2(*sval)[32] = reinterpret_cast<float2(*)[32]>(&sw[AS_TERMS][0][0]);                      // [AS_TERMS][32]
    float(*smag)[32] = reinterpret_cast<float(*)[32]>(&sval[AS_TERMS][0]);                         // [AS_TERMS][32] (ERR)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t tg = blockIdx.x % tgroups, xb = blockIdx.x / tgroups;
    const int G = 32 / wl, g = lane / wl, l = lane % wl;
    // string words: warp per word, ballots over its 32 strings
    for (int w = warp; w < wl; w += AS_WARPS) {
        const int64_t i = (xb * wl + w) * 32 + lane;
        const uint64_t x = i < batch ? xs[i] & nmask : 0ull;
        for (int p = 0; p < NC * AS_CB; ++p) {
            const uint32_t b = __ballot_sync(0xffffffffu, p < 64 && ((x >> (p & 63)) & 1ull) != 0);
            if (lane < G) sx[p][lane * wl + w] = b;
        }
    }
    __syncthreads();
    for (int c = warp; c < NC; c += AS_WARPS) {
        uint32_t* t = tabw + c * 64 * 32 + lane;
        uint32_t cur = 0;
        t[0] = 0;
#pragma unroll
        for (int k = 1; k < 64; ++k) {   // Gray code: one XOR an entry
            const int bit = __ffs(k) - 1;
            cur ^= sx[c * AS_CB + bit][lane];
            t[(k ^ (k >> 1)) * 32] = cur;
        }
    }
    __syncthreads();
    const int64_t tile = tg * G + g;
    // this launch's terms of this lane's tile, and the slot of the first
    const int64_t end = tile < n_tiles ? (tile * P.tt + P.tt < cap ? P.tt : cap - tile * P.tt) - P.r0 : 0;
    const int len = end < P.rl ? (int)end : P.rl;   // 0 or less: none
    const int64_t slot0 = tile * P.rl;
    const bool used = (xb * wl + l) * 32 < batch;   // lanes past the batch's words
    uint32_t tl;   // opaque and after the barrier: the table's loads depend on it
    asm volatile("add.u32 %0, %1, %2;" : "=r"(tl) : "r"(tab0), "r"(4u * lane) : "memory");
    uint64_t sum[4], nc[4];   // complex pairs
    float mag[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        sum[k] = nc[k] = 0;
        mag[k] = 0.f;
    }
    if (P.r0 > 0) {   // as the launch before left them
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t i = (xb * wl + l) * 32 + 4 * warp + k;
            if (tile >= n_tiles || i >= batch) continue;
            sum[k] = reinterpret_cast<const uint64_t*>(partial)[i * n_tiles + tile];
            nc[k] = reinterpret_cast<const uint64_t*>(comp)[i * n_tiles + tile];
            if (ERR) mag[k] = magp[i * n_tiles + tile];
        }
    }
    for (int c0 = 0; c0 < P.rl; c0 += AS_TERMS) {
#pragma unroll 1
        for (int t = warp; t < AS_TERMS && c0 + t < P.rl; t += AS_WARPS) {
            const bool have = c0 + t < len;
            const uint64_t* rec = P.rec + (have ? slot0 + c0 + t : 0) * P.words;
            const ulonglong2 head = __ldg(reinterpret_cast<const ulonglong2*>(rec));
            const ulonglong2 lin = __ldg(reinterpret_cast<const ulonglong2*>(rec + AMP_LO));
            const bool on = have && used && ((uint32_t)head.x >> 8 & 1u);
            {   // the warp's next record on its way
                const char* nx = reinterpret_cast<const char*>(rec + (int64_t)AS_WARPS * P.words) + l * 128;
                if (c0 + t + AS_WARPS < len && l * 16 < AMP_ROWS + P.rows)
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(nx));
            }
            const int mf = on ? (int)(head.x & 255u) : 0;
            uint32_t live = on ? 0xffffffffu : 0u;
            const uint64_t* cons = rec + AMP_ROWS + P.rows;
            const uint64_t tgt = mf > 0 ? __ldg(cons + n) : 0ull;
            uint64_t ks = mf > 0 ? ~__ldg(cons + n + 1) & nmask : 0ull;
            const int most = __reduce_max_sync(0xffffffffu, mf);
#pragma unroll 1
            for (int k = 0; k < most; ++k) {
                if (k < mf) {
                    const uint32_t y = amp_form<NC>(tl, __ldg(cons + k));
                    const uint32_t want = 0u - (uint32_t)((tgt & ks & (0ull - ks)) != 0);
                    ks &= ks - 1;
                    live &= ~(y ^ want);
                }
                if (!__any_sync(0xffffffffu, live != 0u)) break;
            }
            uint32_t ph0 = 0, ph1 = 0;
            if (__any_sync(0xffffffffu, live != 0u)) {
                ph0 = amp_form<NC>(tl, lin.x);
                ph1 = amp_form<NC>(tl, lin.y);
                const ulonglong2* rows = reinterpret_cast<const ulonglong2*>(rec + AMP_ROWS);
                amp_rows<NC, 0>(tl, rows, amp_load(rows, 0), n, ph1);
            }
            sw[t][0][lane] = live;
            sw[t][1][lane] = ph0;
            sw[t][2][lane] = ph1;
            if (l == 0) {
                sval[t][g] = make_float2(__uint_as_float((uint32_t)head.y), __uint_as_float((uint32_t)(head.y >> 32)));
                if (ERR) smag[t][g] = __uint_as_float((uint32_t)(head.x >> 32));
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int t = 0; t < AS_TERMS && c0 + t < P.rl; ++t) {
            const uint32_t live = sw[t][0][lane] >> (4 * warp) & 15u;
            if (!__any_sync(0xffffffffu, live != 0u)) continue;
            const uint32_t q0 = sw[t][1][lane] >> (4 * warp), q1 = sw[t][2][lane] >> (4 * warp);
            const float2 b = sval[t][g];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool odd = (q0 >> k) & 1u;   // i^m b, m = q0 + 2 q1
                const uint32_t neg = (q1 << (31 - k)) & 0x80000000u;
                const uint32_t rx = __float_as_uint(odd ? -b.y : b.x), ry = __float_as_uint(odd ? b.x : b.y);
                kahan_add2(sum[k], nc[k], __uint_as_float(rx ^ neg), __uint_as_float(ry ^ neg), live & (1u << k));
                if (ERR && (live >> k & 1u)) mag[k] += smag[t][g];
            }
        }
        __syncthreads();
    }
    if (tile < n_tiles) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t i = (xb * wl + l) * 32 + 4 * warp + k;
            if (i < batch) {
                if (more) {
                    reinterpret_cast<uint64_t*>(partial)[i * n_tiles + tile] = sum[k];
                    reinterpret_cast<uint64_t*>(comp)[i * n_tiles + tile] = nc[k];
                } else {
                    partial[i * n_tiles + tile] =
                        make_float2(__uint_as_float((uint32_t)sum[k]) + __uint_as_float((uint32_t)nc[k]),
                                    __uint_as_float((uint32_t)(sum[k] >> 32)) + __uint_as_float((uint32_t)(nc[k] >> 32)));
                }
                if (ERR) magp[i * n_tiles + tile] = mag[k];
            }
        }
    }
}

struct AmpPlan {
    int64_t xblocks, n_tiles, tt;
};

// Term tiles so that the grid covers every SM several times.
AmpPlan amp_plan(const lrs_ctx* ctx, int64_t batch, int per_block) {
    AmpPlan P;
    P.xblocks = (batch + per_block - 1) / per_block;
    const int64_t target = (int64_t)ctx->sm_count * ctx->tune_amp_bps;
    int64_t nt = (target + P.xblocks - 1) / P.xblocks;
    const int64_t maxt = (ctx->cap + 31) / 32;
    if (nt > maxt) nt = maxt;
    if (nt < 1) nt = 1;
    P.tt = ((ctx->cap + nt - 1) / nt + 7) & ~(int64_t)7;   // tiles start at multiples of 8 terms
    P.n_tiles = (ctx->cap + P.tt - 1) / P.tt;
    return P;
}

template <int NCH>
lrs_status launch_amp_t(lrs_ctx* ctx, const uint64_t* x, int64_t batch, float2* partial,
                        const AmpPlan& P, float* magp, cudaStream_t st) {
    dim3 grid((unsigned)P.n_tiles, (unsigned)P.xblocks);
    const bool pk = ctx->n <= 62;
    const TermsView T = ctx->view();
    if (pk && magp)
        k_amplitude<NCH, true, true><<<grid, AMP_XT, 0, st>>>(T, x, batch, P.tt, partial, P.n_tiles, magp);
    else if (pk)
        k_amplitude<NCH, true, false><<<grid, AMP_XT, 0, st>>>(T, x, batch, P.tt, partial, P.n_tiles, nullptr);
    else if (magp)
        k_amplitude<NCH, false, true><<<grid, AMP_XT, 0, st>>>(T, x, batch, P.tt, partial, P.n_tiles, magp);
    else
        k_amplitude<NCH, false, false><<<grid, AMP_XT, 0, st>>>(T, x, batch, P.tt, partial, P.n_tiles, nullptr);
    LRS_LAUNCH_CHECK("amplitude kernel");
    return LRS_OK;
}

template <int NC>
lrs_status launch_sliced_t(lrs_ctx* ctx, const AmpPrep& R, const uint64_t* x, int64_t batch, const AmpPlan& P, int wl,
                           float2* partial, float2* comp, float* magp, cudaStream_t st) {
    // up to 8 KB to the table's boundary, the table, the collected words and values
    const size_t smem = 8192 + (size_t)NC * 8192 +
                        (size_t)AS_TERMS * 32 * (3 * sizeof(uint32_t) + sizeof(float2) + (magp ? sizeof(float) : 0));
    const auto kernel = magp ? k_amp_sliced<NC, true> : k_amp_sliced<NC, false>;
    // also under capture (it is no stream operation): the call that sized the scratch may have been
    // one with the other choice of bounds
    LRS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int64_t G = 32 / wl, tgroups = (P.n_tiles + G - 1) / G;
    const int64_t blocks = tgroups * ((batch + 32 * wl - 1) / (32 * wl));
    if (blocks > 0x7FFFFFFF) return lrs_fail(LRS_ERR_UNSUPPORTED, "amplitude grid too large");
    kernel<<<(unsigned)blocks, AS_TPB, smem, st>>>(R, ctx->n, ctx->nmask, x, batch, ctx->cap, P.n_tiles, wl, tgroups,
                                                   R.r0 + R.rl < P.tt, partial, comp, magp);
    LRS_LAUNCH_CHECK("amplitude kernel");
    return LRS_OK;
}

// Scratch of a call.  What it needs must not shrink as the batch grows, or a call of fewer strings
// would reallocate the scratch that a captured call still addresses: so the partial sums are
// counted by a bound that grows with the batch, and the records are as many for every batch.
//
// Partial sums of at most `batch` strings: n_tiles <= ceil(target / xblocks), and never more than
// target or cap / 32 (the sums themselves: 1024 x 1216 at 1024 strings, 4097 x 244 at 4097).
size_t amp_partials(const lrs_ctx* ctx, int64_t batch) {
    const int64_t target = (int64_t)ctx->sm_count * ctx->tune_amp_bps, maxt = (ctx->cap + 31) / 32;
    const int64_t a = batch * (target < maxt ? target : maxt), b = AMP_XB * (target + (batch + AMP_XB - 1) / AMP_XB);
    return (size_t)(a < b ? a : b);
}
// Records: of all terms, or AMP_REC_BYTES of them; a call then takes several launches, each over
// some terms of every tile.
constexpr size_t AMP_REC_BYTES = (size_t)512 << 20;
AmpPrep amp_records(const lrs_ctx* ctx, int64_t* count) {
    AmpPrep R;
    memset(&R, 0, sizeof(R));
    R.rows = (ctx->n + AS_CB - 1) / AS_CB * AS_CB;
    R.words = (AMP_ROWS + R.rows + ctx->n + 2 + 15) & ~15;   // lines of 128 bytes
    const int64_t most = (int64_t)(AMP_REC_BYTES / (R.words * sizeof(uint64_t)));
    *count = ctx->cap < most ? ctx->cap : most;
    return R;
}
// Terms of a tile per launch with `count` slots: all, or equal parts that are whole rounds of
// AS_TERMS (0: not even one round).
int amp_range(const AmpPlan& P, int64_t cap, int64_t count) {
    if (count >= cap) return (int)P.tt;
    const int64_t most = count / P.n_tiles / AS_TERMS * AS_TERMS;
    if (most <= 0) return 0;
    const int64_t parts = (P.tt + most - 1) / most;
    return (int)(((P.tt + parts - 1) / parts + AS_TERMS - 1) / AS_TERMS * AS_TERMS);
}

// Tile sums of the batch by the sliced kernel, R.rl terms of every tile at a time.  (Some whole
// tiles at a time either left too few blocks for the GPU or took records for a quarter of the
// terms, 3.2 GB at n = 40, chi = 2^24, and reached fewer string words a block: 41 strings
// there 46.4 -> 24.5 ms, 1024 strings 54.7 -> 54.9; 4096 strings at n = 50, chi = 2^20 12.0 ms
// either way.)
lrs_status launch_sliced(lrs_ctx* ctx, const uint64_t* x, int64_t batch, float2* partial, float2* comp, const AmpPlan& P,
                         AmpPrep R, float* magp, cudaStream_t st) {
    // string words of a block: 32 (1024 strings), fewer for a batch that has fewer, whose
    // blocks then take several tiles, as long as that leaves a block per SM (gates and 100
    // amplitudes of 300001 terms: 5.57 ms, with two blocks per SM 5.79 ms; with 3 strings of
    // 2048 terms, 32 tiles a block made two blocks and 17 us more than the string-per-thread
    // kernel)
    int wl = 32;
    while (wl > 1 && batch <= 16 * wl && P.n_tiles * (wl / 2) >= (int64_t)32 * ctx->sm_count) wl /= 2;
    R.tt = P.tt;
    for (R.r0 = 0; R.r0 < P.tt; R.r0 += R.rl) {
        k_amp_prep<<<dim3((unsigned)(R.rl / 8), (unsigned)P.n_tiles), 256, 0, st>>>(ctx->view(), R);
        LRS_LAUNCH_CHECK("amplitude prep kernel");
        lrs_status rc;
        switch (R.rows / AS_CB) {
            case 1: rc = launch_sliced_t<1>(ctx, R, x, batch, P, wl, partial, comp, magp, st); break;
            case 2: rc = launch_sliced_t<2>(ctx, R, x, batch, P, wl, partial, comp, magp, st); break;
            case 3: rc = launch_sliced_t<3>(ctx, R, x, batch, P, wl, partial, comp, magp, st); break;
            case 4: rc = launch_sliced_t<4>(ctx, R, x, batch, P, wl, partial, comp, magp, st); break;
            case 5: rc = launch_sliced_t<5>(ctx, R, x, batch, P, wl, partial, comp, magp, st); break;
            case 6: rc = launch_sliced_t<6>(ctx, R, x, batch, P, wl, partial, comp, magp, st); break;
            case 7: rc = launch_sliced_t<7>(ctx, R, x, batch, P, wl, partial, comp, magp, st); break;
            case 8: rc = launch_sliced_t<8>(ctx, R, x, batch, P, wl, partial, comp, magp, st); break;
            case 9: rc = launch_sliced_t<9>(ctx, R, x, batch, P, wl, partial, comp, magp, st); break;
            case 10: rc = launch_sliced_t<10>(ctx, R, x, batch, P, wl, partial, comp, magp, st); break;
            default: rc = launch_sliced_t<11>(ctx, R, x, batch, P, wl, partial, comp, magp, st); break;
        }
        if (rc != LRS_OK) return rc;
    }
    return LRS_OK;
}

lrs_status launch_amp_kernels(lrs_ctx* ctx, const uint64_t* x, int64_t batch, double* out,
                              float2* partial, const AmpPlan& P, cudaStream_t st,
                              float* magp = nullptr, float* err = nullptr) {
    if (P.xblocks > 65535) return lrs_fail(LRS_ERR_UNSUPPORTED, "amplitude batch too large");
    lrs_status rc;
    switch ((ctx->n + 3) / 4) {
        case 1: rc = launch_amp_t<1>(ctx, x, batch, partial, P, magp, st); break;
        case 2: rc = launch_amp_t<2>(ctx, x, batch, partial, P, magp, st); break;
        case 3: rc = launch_amp_t<3>(ctx, x, batch, partial, P, magp, st); break;
        case 4: rc = launch_amp_t<4>(ctx, x, batch, partial, P, magp, st); break;
        case 5: rc = launch_amp_t<5>(ctx, x, batch, partial, P, magp, st); break;
        case 6: rc = launch_amp_t<6>(ctx, x, batch, partial, P, magp, st); break;
        case 7: rc = launch_amp_t<7>(ctx, x, batch, partial, P, magp, st); break;
        case 8: rc = launch_amp_t<8>(ctx, x, batch, partial, P, magp, st); break;
        case 9: rc = launch_amp_t<9>(ctx, x, batch, partial, P, magp, st); break;
        case 10: rc = launch_amp_t<10>(ctx, x, batch, partial, P, magp, st); break;
        case 11: rc = launch_amp_t<11>(ctx, x, batch, partial, P, magp, st); break;
        case 12: rc = launch_amp_t<12>(ctx, x, batch, partial, P, magp, st); break;
        case 13: rc = launch_amp_t<13>(ctx, x, batch, partial, P, magp, st); break;
        case 14: rc = launch_amp_t<14>(ctx, x, batch, partial, P, magp, st); break;
        case 15: rc = launch_amp_t<15>(ctx, x, batch, partial, P, magp, st); break;
        default: rc = launch_amp_t<16>(ctx, x, batch, partial, P, magp, st); break;
    }
    if (rc != LRS_OK) return rc;
    k_amp_reduce<<<(unsigned)batch, 256, 0, st>>>(partial, magp, P.n_tiles, batch, P.tt, out, err);
    LRS_LAUNCH_CHECK("amplitude reduce kernel");
    return LRS_OK;
}

}  // namespace

// Scratch of `full` bytes, or of at least `least` where so much cannot be had.  Scratch that is
// enough for `least` is not given up before a larger one is there (a captured call may address
// it), and an allocation that has failed is not tried again for as much until the terms' storage
// changes: such calls reallocate nothing, neither each time nor under capture.
static lrs_status amp_scratch(lrs_ctx* ctx, size_t full, size_t least, cudaStream_t st) {
    if (ctx->scratch_bytes >= full) return LRS_OK;
    const bool keep = ctx->scratch_bytes >= least, tried = ctx->amp_oom != 0 && full >= ctx->amp_oom;
    if (keep && (tried || lrs_capturing(st))) return LRS_OK;
    if (!tried) {
        void* p = keep ? nullptr : ctx->scratch;
        size_t have = keep ? 0 : ctx->scratch_bytes;
        const lrs_status rc = lrs_ensure(&p, &have, full, ctx->alloc_limit);
        if (rc == LRS_OK || !keep) {
            if (keep) cudaFree(ctx->scratch);
            ctx->scratch = p;
            ctx->scratch_bytes = have;
        }
        if (rc != LRS_ERR_OOM) return rc;
        ctx->amp_oom = full;
        if (keep) return LRS_OK;
    }
    void* scr = nullptr;
    return lrs_scratch(ctx, least, &scr);
}

// The sliced kernels and the reduction, with scratch for partial sums and their compensations,
// bounds (err), amplitudes (*amp_out) and records: as many of the records as the scratch that
// could be had holds, and the string-per-thread kernel where that is too few.
static lrs_status launch_amp_scratch(lrs_ctx* ctx, const uint64_t* x, int64_t batch, const AmpPlan& P, double* out,
                                     double** amp_out, float* err, cudaStream_t st) {
    auto round = [](size_t bytes) { return (bytes + 255) & ~(size_t)255; };
    const size_t amps = round((size_t)batch * 2 * sizeof(double));
    // bounds and amplitudes have their place in every call, as the sums do
    const size_t most = amp_partials(ctx, batch), need = 2 * round(most * sizeof(float2)) + round(most * sizeof(float)) + amps;
    // without records: the sums of this call and what it asked for
    const size_t sums = (size_t)batch * P.n_tiles;
    const size_t least = round(sums * sizeof(float2)) + (err ? round(sums * sizeof(float)) : 0) + (amp_out ? amps : 0);
    int64_t records;
    AmpPrep R = amp_records(ctx, &records);
    const size_t rec_bytes = R.words * sizeof(uint64_t);
    lrs_status rc = amp_scratch(ctx, need + (size_t)records * rec_bytes, least, st);
    if (rc != LRS_OK) return rc;
    const size_t room = ctx->scratch_bytes > need ? (ctx->scratch_bytes - need) / rec_bytes : 0;
    if ((size_t)records > room) records = (int64_t)room;
    R.rl = amp_range(P, ctx->cap, records);
    char* at = (char*)ctx->scratch;
    auto take = [&](size_t bytes) {
        char* q = at;
        at += round(bytes);
        return q;
    };
    float2* partial = (float2*)take(sums * sizeof(float2));
    float* magp = err ? (float*)take(sums * sizeof(float)) : nullptr;
    if (amp_out) out = *amp_out = (double*)take(amps);
    if (R.rl == 0) return launch_amp_kernels(ctx, x, batch, out, partial, P, st, magp, err);
    float2* comp = (float2*)take(sums * sizeof(float2));
    R.rec = (uint64_t*)((char*)ctx->scratch + need);
    if ((rc = launch_sliced(ctx, x, batch, partial, comp, P, R, magp, st)) != LRS_OK) return rc;
    k_amp_reduce<<<(unsigned)batch, 256, 0, st>>>(partial, magp, P.n_tiles, batch, P.tt, out, err);
    LRS_LAUNCH_CHECK("amplitude reduce kernel");
    return LRS_OK;
}

// Amplitudes of the chains' start strings into scratch (*amp_out, 2 doubles per x), on the
// term tiles of 512 strings per block.
lrs_status launch_amplitude_start(lrs_ctx* ctx, const uint64_t* x, int64_t batch, double** amp_out, cudaStream_t st) {
    AmpPlan P = amp_plan(ctx, batch, 512);
    P.xblocks = (batch + AMP_XB - 1) / AMP_XB;
    return launch_amp_scratch(ctx, x, batch, P, nullptr, amp_out, nullptr, st);
}

lrs_status launch_amplitude(lrs_ctx* ctx, const uint64_t* x, int64_t batch, double* out, float* err,
                            cudaStream_t st) {
    if (batch == 0) return LRS_OK;
    const AmpPlan P = amp_plan(ctx, batch, AMP_XB);
    if (P.xblocks > 65535) return lrs_fail(LRS_ERR_UNSUPPORTED, "amplitude batch too large");
    return launch_amp_scratch(ctx, x, batch, P, out, nullptr, err, st);
}

template <int NCH>
static lrs_status launch_amp_batch_t(const AmpBatch& B, int64_t blocks, bool pk, cudaStream_t st) {
    if (pk)
        k_amplitude_batch<NCH, true><<<(unsigned)blocks, AMP_XT, 0, st>>>(B);
    else
        k_amplitude_batch<NCH, false><<<(unsigned)blocks, AMP_XT, 0, st>>>(B);
    LRS_LAUNCH_CHECK("batched amplitude kernel");
    return LRS_OK;
}

// Amplitudes of several circuits of the same width (count <= LRS_AMP_BATCH_MAX per
// launch pair): one amplitude launch and one reduction launch for all of them, each
// circuit with the tile plan and partial buffer of its own single launch.
lrs_status launch_amplitude_batch(lrs_ctx* const* ctxs, const uint64_t* const* xs, const int64_t* batch,
                                  double* const* out, int32_t count, cudaStream_t st) {
    const int n = ctxs[0]->n;
    // Large circuits one after the other by the sliced kernel (each fills the GPU); small
    // ones, where its launches per circuit would add up, together.  The line: 2^23 (x, term)
    // per circuit take about 60 us either way.
    double work = 0.0;
    for (int32_t i = 0; i < count; ++i) work += (double)ctxs[i]->cap * (double)batch[i];
    if (work >= (double)count * 8388608.0) {
        for (int32_t i = 0; i < count; ++i) {
            const lrs_status rc = launch_amplitude(ctxs[i], xs[i], batch[i], out[i], nullptr, st);
            if (rc != LRS_OK) return rc;
        }
        return LRS_OK;
    }
    for (int32_t base = 0; base < count; base += LRS_AMP_BATCH_MAX) {
        AmpBatch B;
        memset(&B, 0, sizeof(B));
        int64_t xfirst[LRS_AMP_BATCH_MAX + 1];
        int k = 0;
        int64_t blocks = 0, strings = 0;
        const int32_t end = (count - base < LRS_AMP_BATCH_MAX) ? count : base + LRS_AMP_BATCH_MAX;
        for (int32_t i = base; i < end; ++i) {
            if (batch[i] == 0) continue;
            lrs_ctx* c = ctxs[i];
            const AmpPlan P = amp_plan(c, batch[i], AMP_XB);
            if (P.xblocks > 65535) return lrs_fail(LRS_ERR_UNSUPPORTED, "amplitude batch too large");
            void* scr = nullptr;
            lrs_status rc = lrs_scratch(c, amp_partials(c, batch[i]) * sizeof(float2), &scr);
            if (rc != LRS_OK) return rc;
            B.first[k] = blocks;
            B.T[k] = c->view();
            B.xs[k] = xs[i];
            B.batch[k] = batch[i];
            B.tt[k] = P.tt;
            B.n_tiles[k] = P.n_tiles;
            B.partial[k] = (float2*)scr;
            B.out[k] = out[i];
            xfirst[k] = strings;
            blocks += P.n_tiles * P.xblocks;
            strings += batch[i];
            ++k;
        }
        if (k == 0) continue;
        if (blocks > 0x7FFFFFFF) return lrs_fail(LRS_ERR_UNSUPPORTED, "batched amplitude grid too large");
        B.count = k;
        B.first[k] = blocks;
        xfirst[k] = strings;
        AmpBatch R = B;   // the reduction indexes strings instead of blocks
        for (int j = 0; j <= k; ++j) R.first[j] = xfirst[j];
        lrs_status rc;
        const bool pk = n <= 62;
        switch ((n + 3) / 4) {
            case 1: rc = launch_amp_batch_t<1>(B, blocks, pk, st); break;
            case 2: rc = launch_amp_batch_t<2>(B, blocks, pk, st); break;
            case 3: rc = launch_amp_batch_t<3>(B, blocks, pk, st); break;
            case 4: rc = launch_amp_batch_t<4>(B, blocks, pk, st); break;
            case 5: rc = launch_amp_batch_t<5>(B, blocks, pk, st); break;
            case 6: rc = launch_amp_batch_t<6>(B, blocks, pk, st); break;
            case 7: rc = launch_amp_batch_t<7>(B, blocks, pk, st); break;
            case 8: rc = launch_amp_batch_t<8>(B, blocks, pk, st); break;
            case 9: rc = launch_amp_batch_t<9>(B, blocks, pk, st); break;
            case 10: rc = launch_amp_batch_t<10>(B, blocks, pk, st); break;
            case 11: rc = launch_amp_batch_t<11>(B, blocks, pk, st); break;
            case 12: rc = launch_amp_batch_t<12>(B, blocks, pk, st); break;
            case 13: rc = launch_amp_batch_t<13>(B, blocks, pk, st); break;
            case 14: rc = launch_amp_batch_t<14>(B, blocks, pk, st); break;
            case 15: rc = launch_amp_batch_t<15>(B, blocks, pk, st); break;
            default: rc = launch_amp_batch_t<16>(B, blocks, pk, st); break;
        }
        if (rc != LRS_OK) return rc;
        k_amp_reduce_batch<<<(unsigned)strings, 256, 0, st>>>(R, strings);
        LRS_LAUNCH_CHECK("batched amplitude reduce kernel");
    }
    return LRS_OK;
}

// ---------------------------------------------------------------------------------
// Allocation-free variant of lrs_amplitude.
//
// Some callers cannot call cudaMalloc at the point where they need amplitudes:
// a serving loop whose framework allocator has already reserved all device
// memory, or code that must not take the allocator's locks or its latency on
// a hot path.  For them the block partial sums live in a fixed file-scope
// device array instead of the context's growable scratch buffer.  The array
// is allocated when the library is loaded and stays on every GPU that loads
// the library until the process exits.
// ---------------------------------------------------------------------------------
#define LRS_NOALLOC_PARTIALS (2u * 1024u * 1024u)   // float2 entries = 16 MiB

static __device__ __align__(256) float2 g_noalloc_partials[LRS_NOALLOC_PARTIALS];

// Device address of g_noalloc_partials, looked up once per device.  In host
// code the symbol name is only a host-side stand-in, so it is never passed to a
// kernel directly.  The address is published through an atomic, so first calls
// racing from several host threads each look it up (same value) without a data
// race; a failed lookup publishes nothing and the next call tries again.
static std::atomic<void*> g_noalloc_addr[128];

static lrs_status noalloc_address(int device, float2** out) {
    if (device < 0 || device >= 128) return lrs_fail(LRS_ERR_UNSUPPORTED, "device index %d", device);
    void* p = g_noalloc_addr[device].load(std::memory_order_acquire);
    if (!p) {
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_partials);
        if (e != cudaSuccess) return lrs_cuda_check(e, "cudaGetSymbolAddress(g_noalloc_partials)");
        g_noalloc_addr[device].store(p, std::memory_order_release);
    }
    *out = (float2*)p;
    return LRS_OK;
}

extern "C" lrs_status lrs_amplitude_noalloc(lrs_ctx* ctx, const uint64_t* x, int64_t batch,
                                            double* out, void* stream) {
    if (!ctx) return lrs_fail(LRS_ERR_ARG, "ctx is NULL");
    if (!ctx->have_terms) return lrs_fail(LRS_ERR_STATE, "no terms");
    if (batch < 0) return lrs_fail(LRS_ERR_ARG, "batch < 0");
    if (batch > 0 && (!x || !out)) return lrs_fail(LRS_ERR_ARG, "NULL buffer");
    LRS_CUDA(cudaSetDevice(ctx->device));
    float2* partial = nullptr;
    lrs_status rc = noalloc_address(ctx->device, &partial);   // first call on a device: set-up
    if (rc != LRS_OK) return rc;
    if (batch == 0) return LRS_OK;
    const AmpPlan P = amp_plan(ctx, batch, AMP_XB);
    if ((uint64_t)batch * (uint64_t)P.n_tiles > (uint64_t)LRS_NOALLOC_PARTIALS)
        return lrs_fail(LRS_ERR_ARG,
                        "lrs_amplitude_noalloc: %lld partial sums (batch x term tiles) exceed the "
                        "fixed buffer of %u; use a smaller batch or lrs_amplitude",
                        (long long)(batch * P.n_tiles), LRS_NOALLOC_PARTIALS);
    return launch_amp_kernels(ctx, x, batch, out, partial, P, (cudaStream_t)stream);
}
