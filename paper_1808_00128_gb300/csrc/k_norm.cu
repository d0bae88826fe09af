// Norm estimation (Sec. 4.3): eta_l = 2^n |<phi_{A_l}|psi>|^2.
//
// Per (A, term) the sum is taken over y' = G (s + x), x in Z2^v (Lemma (Inner Product) with
// G^-1 = F^T):
//   <phi_A|phi>^* ~ (-1)^{|s|} sum over y' with f_k . y' = s_k (k not in v) of
//                   i^{q_A(y') + q_J(y') + 2 (F s) . y'},
// q_A and q_J the Z4 forms with off-diagonal A and J = M F^T and diagonals A_cc, gamma_c; f_k =
// column k of F.  The constraints in reduced echelon form give y'_p = h_p . y + c_p over
// the m = |v| free variables y, and both forms restrict to y separately:
//   k_norm_prep   per term (a warp each): J, the echelon form, and q_J + 2 (F s) . y'
//                 restricted to the free variables, as one record of bit rows
//   k_norm_draw   per 32 equatorial states: A_l from the counter RNG, transposed so that one
//                 32-bit word holds entry (i, k) of 32 matrices
//   k_norm        per (32 states, term) a warp: q_A restricted and added, then the exponential
//                 sum by pairwise elimination (Lemma (Exponential Sum)) on 32 forms at once
//   k_norm_reduce the FP64 sum over term tiles
//
// The elimination is integer-pipe bound, so its words are what counts.  One form per thread
// (rows as 64-bit words) spends 32 lanes x ~8 instructions on every row of every pivot
// pair; with bit f of a word belonging to form f, entry (i, k) of 32 forms takes two
// three-input operations a pivot pair, whatever their pivots are: 13.2 -> 7.4 thousand warp
// instructions per (term, 32 states) at n = 50, 302 -> 182 ms at chi = 2^20, L = 512, and
// 6.83 -> 3.79 ms at n = 40, chi = 2^16, L = 256.  Lane k of the warp holds columns k and
// k + 32 in registers, row i at register i; the pivots are always the first two live
// rows, which is made so in every form by adding to the second the first row that the
// pivot row is joined to (a change of basis of that form alone), and the rows move up by
// two as they are updated, so every register index is a constant.  The integer pipe is 75%
// busy; the code of a term (some 40 KB, nearly straight) and three warps a scheduler
// are what is left.  Measured and not kept: more stages of row counts (14.5 against 11.6 ms on a
// sixteenth of that call: the instruction cache), folds by tables of XORs (12.3), a
// group of states per warp instead of per block (13.4).
#include "lrs_device.cuh"

namespace {

constexpr int NRM_WINDOW = 16;   // rows searched for the pivot row's partner
constexpr int NRM_STRIDE = 66;   // words per row of A in shared memory; column 64 and row n are zero
constexpr int NRM_END = 10;      // variables left to the per-form elimination
constexpr int NRM_SYNC = 4;      // terms between the barriers of a block
constexpr int NRM_VEC = 88;      // entries of the shared vectors: past the last row that a step reads (stage)
constexpr int NRM_CHUNK = 32;    // terms whose values a cooperating block collects at a time

// Record of a term: `rows` words of bit rows, then six header words, then the pivots as bytes
// (14 words beside the rows: near the memory limit the scratch of a call is mostly these
// records).  Rows 0..m-1: the restricted form of J between free variables (bit k of row k:
// its odd diagonal).  Rows from m on: h of every constraint (n - m of them); or, for a term
// with few free variables (norm_basis), the y' of every free variable (m vectors over the
// n qubits) and the constant vector c.
struct NormPrep {
    uint64_t* rec;          // [cap][words]
    int words, rows;
    uint32_t *A, *ad;       // [group][n][64] and [group][2][64]: entries, diagonal planes
};
enum { REC_FREE = 0, REC_LO, REC_HI, REC_CONST, REC_INFO, REC_COEF, REC_PIV, REC_HEAD = REC_PIV + 8 };

// Few free variables: q_A is evaluated on the basis (m + 1 matrix-vector products and
// m^2 / 2 dot products over the lanes) instead of folding n - m constraints one by one, whose
// cost grows with (n - m)^2.  2 m + 1 rows have to fit the record; 16 variables keep the
// products below the folds' cost for every n.
__host__ __device__ constexpr bool norm_basis(int n, int m) { return m <= 16 && 2 * m + 1 <= n; }

__device__ __forceinline__ uint64_t shfl64(uint64_t v, int src) {
    return __shfl_sync(0xffffffffu, (unsigned long long)v, src);
}

// ---- A_l in M_n from the counter RNG ------------------------------------------------
// The diagonal as two bit-planes (words 0 and 1 of the stream of l), the upper triangle
// from words 2.. in the order (0,1), (0,2), .., (0,n-1), (1,2), .., one bit each.
// One block per 32 states: lane l draws word j of its state, and 64 ballots turn the
// 32 words into the bit-sliced entries 64 j .. 64 j + 63.  States past L repeat state L - 1, and
// their sums are dropped.  (As zero matrices they left sparse forms, whose isolated variables
// sent the whole group through the elimination form by form: 16 states of the n = 57 QAOA at
// chi = 2^17 9.4 ms, repeated 2.3.)
constexpr int DRAW_WARPS = 8;
__global__ void __launch_bounds__(32 * DRAW_WARPS) k_norm_draw(int n, int64_t L, uint64_t seed, NormPrep P) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t g = blockIdx.x, l = g * 32 + lane;
    const uint64_t key = sm64_key(seed, (uint64_t)(l < L ? l : L - 1));
    uint32_t* A = P.A + g * n * 64;
    const int entries = n * (n - 1) / 2;
    const int words = 2 + (entries + 63) / 64;
    for (int j = warp; j < words; j += DRAW_WARPS) {
        const uint64_t w = sm64_at(key, (uint64_t)j);
        uint32_t e0 = 0, e1 = 0;
#pragma unroll
        for (int t = 0; t < 32; ++t) {
            const uint32_t b0 = __ballot_sync(0xffffffffu, (uint32_t)w >> t & 1u);
            const uint32_t b1 = __ballot_sync(0xffffffffu, (uint32_t)(w >> 32) >> t & 1u);
            if (lane == t) { e0 = b0; e1 = b1; }
        }
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const uint32_t e = half ? e1 : e0;
            const int b = lane + 32 * half;
            if (j < 2) {
                P.ad[(g * 2 + j) * 64 + b] = b < n ? e : 0u;
                if (j == 0 && b < n) A[b * 64 + b] = e;
            } else {
                int k = (j - 2) * 64 + b;
                if (k >= entries) continue;
                int r = 0;
                while (k >= n - 1 - r) { k -= n - 1 - r; ++r; }
                const int c = r + 1 + k;
                A[r * 64 + c] = e;
                A[c * 64 + r] = e;
            }
        }
    }
}

// ---- per-term record ------------------------------------------------------------------
// A warp per term, lane c holding rows c and c + 32.  (One thread per term was a serial
// chain of some 25 thousand instructions; a small call waited for it.)
__device__ __forceinline__ uint64_t drop_bits(uint64_t x, uint64_t keep, uint64_t nmask) {
    // bits of x at the positions in `keep`, moved together (the others removed from the top)
    for (uint64_t out = ~keep & nmask; out;) {
        const int p = 63 - __clzll((long long)out);
        out ^= bit64(p);
        const uint64_t low = bit64(p) - 1;
        x = (x & low) | ((x >> 1) & ~low);
    }
    return x;
}

__global__ void __launch_bounds__(256) k_norm_prep(TermsView T, NormPrep P) {
    __shared__ uint64_t sF[8][64];
    const int n = T.n, lane = threadIdx.x & 31;
    const int64_t alpha = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (alpha >= T.chi) return;   // warp-uniform; padding terms need no record
    const uint64_t nmask = T.nmask, v = T.v[alpha], s = T.s[alpha], glo = T.glo[alpha], ghi = T.ghi[alpha];
    uint64_t F[2], M[2], J[2] = {0, 0}, f[2] = {0, 0};
    uint32_t d[2], con[2] = {0, 0};
    int pivot[2] = {0, 0};
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int q = lane + 32 * c;
        F[c] = q < n ? T.F[(int64_t)q * T.cap + alpha] : 0ull;
        M[c] = q < n ? T.M[(int64_t)q * T.cap + alpha] : 0ull;
        // diagonal of q_J + 2 (F s) . y' (Z4)
        d[c] = (uint32_t)getb(glo, q) | ((uint32_t)getb(ghi, q) ^ par64(F[c] & s)) << 1;
    }
    uint64_t* rows = sF[threadIdx.x >> 5];
    rows[lane] = F[0];
    rows[lane + 32] = F[1];
    __syncwarp();
    lrs_products(rows, n, M[0], M[1], J[0], J[1]);
#pragma unroll
    for (int c = 0; c < 2; ++c) J[c] &= ~bit64(lane + 32 * c);
    // constraint i in lane i % 32: column k_i of F (k_i the i-th qubit outside v) and s_{k_i}
    const uint64_t out = ~v & nmask;
    const int mf = __popcll(out), m = n - mf;
    {
        uint64_t ks = out;
        for (int i = 0; i < mf; ++i) {
            const int k = ffs64(ks);
            ks &= ks - 1;
            const uint64_t col = (uint64_t)__ballot_sync(0xffffffffu, (uint32_t)getb(F[0], k)) |
                                 (uint64_t)__ballot_sync(0xffffffffu, (uint32_t)getb(F[1], k)) << 32;
            if (lane == (i & 31)) {
                f[i >> 5] = col;
                con[i >> 5] = (uint32_t)getb(s, k);
            }
        }
    }
    // reduced echelon form (the columns are independent: F is invertible); the pivot of
    // constraint i is its lowest bit when it is processed, then cleared from all others
    uint64_t pivots = 0;
    for (int i = 0; i < mf; ++i) {
        const uint64_t fi = shfl64(i < 32 ? f[0] : f[1], i & 31);
        const uint32_t ci = __shfl_sync(0xffffffffu, i < 32 ? con[0] : con[1], i & 31);
        const int p = ffs64(fi);
        pivots |= bit64(p);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (lane + 32 * c == i) {
                pivot[c] = p;
            } else if (getb(f[c], p)) {
                f[c] ^= fi;
                con[c] ^= ci;
            }
        }
    }
    // substitute y'_p = h . y + c into q_J, one constraint at a time (see fold in k_norm)
    const uint64_t freev = nmask & ~pivots;
    uint64_t act = nmask;
    uint32_t kc = 0;
    for (int i = 0; i < mf; ++i) {
        const int src = i & 31;
        const int p = __shfl_sync(0xffffffffu, i < 32 ? pivot[0] : pivot[1], src);
        const uint64_t h = shfl64(i < 32 ? f[0] : f[1], src) & ~bit64(p);
        const uint32_t ci = __shfl_sync(0xffffffffu, i < 32 ? con[0] : con[1], src);
        act &= ~bit64(p);
        const uint64_t q = shfl64(p < 32 ? J[0] : J[1], p & 31) & act;
        uint32_t dp = __shfl_sync(0xffffffffu, p < 32 ? d[0] : d[1], p & 31) & 3u;
        if (ci) {
            kc += dp;
            dp = (4u - dp) & 3u;
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int r = lane + 32 * c;
            const uint32_t hr = (uint32_t)getb(h, r), qr = (uint32_t)getb(q, r);
            d[c] += 2u * (qr & ci) + hr * dp + 2u * (hr & qr);
            if (hr) J[c] ^= q ^ ((dp & 1u) ? h : 0ull);
            if (qr) J[c] ^= h;
        }
    }
    const uint64_t lo_n = (uint64_t)__ballot_sync(0xffffffffu, d[0] & 1u) |
                          (uint64_t)__ballot_sync(0xffffffffu, d[1] & 1u) << 32;
    const uint64_t hi_n = (uint64_t)__ballot_sync(0xffffffffu, (d[0] >> 1) & 1u) |
                          (uint64_t)__ballot_sync(0xffffffffu, (d[1] >> 1) & 1u) << 32;
    uint64_t* rec = P.rec + alpha * P.words;
    uint64_t* head = rec + P.rows;
    const bool basis = norm_basis(n, m);
    if (basis) {
        uint64_t b[2] = {bit64(lane), bit64(lane + 32)}, cv = 0;
        for (int i = 0; i < mf; ++i) {
            const int p = __shfl_sync(0xffffffffu, i < 32 ? pivot[0] : pivot[1], i & 31);
            const uint64_t h = shfl64(i < 32 ? f[0] : f[1], i & 31);
            const uint32_t ci = __shfl_sync(0xffffffffu, i < 32 ? con[0] : con[1], i & 31);
            if (ci) cv |= bit64(p);
#pragma unroll
            for (int c = 0; c < 2; ++c)
                if (getb(h, lane + 32 * c)) b[c] |= bit64(p);
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int r = lane + 32 * c;
            if (r < n && getb(freev, r)) rec[m + __popcll(freev & (bit64(r) - 1))] = b[c];
        }
        if (lane == 0) rec[2 * m] = cv;
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int r = lane + 32 * c;
        if (r < n && getb(freev, r)) {
            const uint64_t row = (J[c] & ~bit64(r)) | ((uint64_t)(d[c] & 1u) << r);
            rec[__popcll(freev & (bit64(r) - 1))] = drop_bits(row & freev, freev, nmask);
        }
        if (r < mf && !basis) {
            rec[m + r] = drop_bits(f[c] & freev, freev, nmask);
            reinterpret_cast<uint8_t*>(head + REC_PIV)[r] = (uint8_t)pivot[c];
        }
    }
    const uint64_t cm = (uint64_t)__ballot_sync(0xffffffffu, con[0]) | (uint64_t)__ballot_sync(0xffffffffu, con[1]) << 32;
    if (lane == 0) {
        const uint32_t om = T.omega[alpha];
        const uint32_t ph = ((om & 7u) + 4u * (uint32_t)__popcll(s & ~v) - 2u * kc) & 7u;
        head[REC_FREE] = freev;
        head[REC_LO] = drop_bits(lo_n & freev, freev, nmask);
        head[REC_HI] = drop_bits(hi_n & freev, freev, nmask);
        head[REC_CONST] = cm;
        // m, phase, live, basis; |v| + h
        head[REC_INFO] = (uint64_t)((uint32_t)m | ph << 8 | (((om >> 3) & 1u) ? 0u : 1u) << 16 | (basis ? 1u << 17 : 0u)) |
                         (uint64_t)((uint32_t)__popcll(v) + (om >> 8)) << 32;
        const float2 b = T.coef[alpha];
        head[REC_COEF] = (uint64_t)__float_as_uint(b.x) | (uint64_t)__float_as_uint(b.y) << 32;
    }
}

// ---- bit-sliced elimination --------------------------------------------------------------
// Work area of a warp in shared memory.
struct NormWarp {
    uint4 pa[80];            // per column: pivot row, second row, linear planes
    uint2 pb[NRM_VEC];       // per column: the two vectors of a rank-2 update
    uint32_t off[80];        // first word of row (natural index of the variable) in A
    union {
        uint32_t rows[NRM_END][32];   // last rows, one form per lane
        uint32_t mat[16][32];         // q_A on the basis, and its diagonal planes
    };
    uint32_t diag[2][16];
    uint64_t rec[2][80];     // record of this term and the next
};
static_assert(sizeof(NormWarp) % 16 == 0, "the warps' areas follow one another");

// c ^ (a & b) as one instruction (at n = 50, chi = 2^20, L = 512: 248 -> 207 ms against the same
// expressions in C)
__device__ __forceinline__ uint32_t xand(uint32_t c, uint32_t a, uint32_t b) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0x6a;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

// 0xffffffff where bit I of w is set, else 0 (sign-replicating byte permute: two
// instructions per bit at most, the shift shared by the word's four bytes)
template <int I>
__device__ __forceinline__ uint32_t bit_mask(uint32_t w) {
    constexpr uint32_t sel = 0x8888u + 0x1111u * (I >> 3);
    const uint32_t t = w << (7 - (I & 7));
    uint32_t r;
    asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(t), "n"(sel));
    return r;
}
__device__ __forceinline__ uint32_t lane_mask(uint64_t w, int pos) { return 0u - (uint32_t)getb(w, pos); }

// lane l's word, as the mask over l of the words' bit `lane` (32 x 32 bit transpose across
// the warp; Warren, Hacker's Delight, ch. 7)
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane) {
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) {
        const uint32_t mk = sh == 16 ? 0x0000ffffu : sh == 8 ? 0x00ff00ffu : sh == 4 ? 0x0f0f0f0fu
                            : sh == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, sh);
        x = (lane & sh) ? (((y >> sh) & mk) | (x & ~mk)) : ((x & mk) | ((y & mk) << sh));
    }
    return x;
}

// Sliced state of 32 forms: S[c][i] = entry (row a + i, own column c), linear planes L0 and
// L1 (the coefficient of the lift variable X), sign planes of X = 0 and of X.
template <int NR, int NC>
struct Forms {
    uint32_t S[NC][NR];
    uint32_t L0[NC], L1[NC];
    uint32_t s0, s1;
    int a, m;
};

// Eliminates variables a and a + 1 in all 32 forms; false (nothing changed) when in some form
// variable a is joined to no other.  R rows are live at most (m - a <= R).  C columns a
// lane: positions lane and lane + 32, or (C = 1) the position pos = lane (mod 32) in
// [a, a + 32), kept twice in the shared vectors so that no index wraps.
template <int R, int C, int NR, int NC>
__device__ __forceinline__ bool eliminate_pair(Forms<NR, NC>& Z, NormWarp& W, int lane, int pos) {
    const int b = C == 2 ? Z.a : (Z.a & 31);
    uint32_t p1[C], p2[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
        p1[c] = Z.S[c][0];
        p2[c] = Z.S[c][1];
        if (C == 1 && pos < Z.a) p1[c] = 0;   // a column that has left
        const uint4 e = make_uint4(p1[c], Z.L0[c] ^ p2[c], Z.L1[c], 0u);
        W.pa[lane + 32 * c] = e;
        if (C == 1) W.pa[lane + 32] = e;
    }
    __syncwarp();
    const uint4 ea = W.pa[b], eb = W.pa[b + 1];
    // linear planes of a, and of its partner
    const uint32_t c10 = ea.y ^ eb.x, c11 = ea.z;
    uint32_t found = eb.x, c20 = eb.y, c21 = eb.z;
    // a + 1 becomes a + 1 plus the first later neighbour of a, in the forms where it is none
#pragma unroll
    for (int j0 = 2; j0 < (R < NRM_WINDOW ? R : NRM_WINDOW); j0 += 4) {
        if (found == 0xffffffffu) break;   // one word for all lanes: uniform
        uint4 e[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (j0 + u < R) e[u] = W.pa[b + j0 + u];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (j0 + u >= R) break;
            const uint32_t sel = e[u].x & ~found;
            found |= e[u].x;
#pragma unroll
            for (int c = 0; c < C; ++c) p2[c] = xand(p2[c], sel, Z.S[c][j0 + u]);
            c20 = xand(c20, sel, e[u].y);
            c21 = xand(c21, sel, e[u].z);
        }
    }
    if (found != 0xffffffffu) return false;
    Z.s0 = xand(Z.s0, c10, c20);
    Z.s1 = xand(xand(Z.s1, c10, c21), c11, c20 ^ c21);
#pragma unroll
    for (int c = 0; c < C; ++c) {
        if (C == 1 && pos < Z.a) p2[c] = 0;
        Z.L0[c] = xand(xand(Z.L0[c], p2[c], p1[c] ^ c10), c20, p1[c]);
        Z.L1[c] = xand(xand(Z.L1[c], c11, p2[c]), c21, p1[c]);
        W.pb[lane + 32 * c] = make_uint2(p1[c], p2[c]);
        if (C == 1) W.pb[lane + 32] = make_uint2(p1[c], p2[c]);
    }
    __syncwarp();
#pragma unroll
    for (int i = 2; i < R; i += 2) {
        const uint4 w = *reinterpret_cast<const uint4*>(&W.pb[b + i]);   // b is even
#pragma unroll
        for (int c = 0; c < C; ++c) {
            Z.S[c][i - 2] = xand(xand(Z.S[c][i], w.x, p2[c]), w.y, p1[c]);
            Z.S[c][i - 1] = xand(xand(Z.S[c][i + 1], w.z, p2[c]), w.w, p1[c]);
        }
    }
#pragma unroll
    for (int c = 0; c < C; ++c) Z.S[c][R - 2] = Z.S[c][R - 1] = 0;
    Z.a += 2;
    return true;
}

// What one form (lane) still needs after the sliced steps: rows by relative index, by
// scalar pairwise elimination.  `rows`: this lane's rows, `st` words apart.
template <class Word>
__device__ __forceinline__ void finish_form(Word* rows, int st, int r, Word L0, Word L1, uint32_t& s0, uint32_t& s1,
                                            uint32_t& z0, uint32_t& z1, int& e) {
    Word act = r == 8 * (int)sizeof(Word) ? ~(Word)0 : (((Word)1 << r) - 1);
    for (Word cand = act; cand;) {
        const Word ba = cand & (0 - cand);
        const int a = sizeof(Word) == 4 ? __ffs((int)ba) - 1 : ffs64((uint64_t)ba);
        cand ^= ba;
        const Word ra = rows[a * st] & act & ~ba;
        if (!ra) continue;   // isolated: stays so
        const Word bb = ra & (0 - ra);
        const int b = sizeof(Word) == 4 ? __ffs((int)bb) - 1 : ffs64((uint64_t)bb);
        const Word m1 = ra & ~bb;
        act &= ~(ba | bb);
        cand &= ~bb;
        const Word m2 = rows[b * st] & act;
        const bool a0 = (L0 & ba) != 0, b0 = (L0 & bb) != 0, a1 = (L1 & ba) != 0, b1 = (L1 & bb) != 0;
        s0 ^= (uint32_t)(a0 && b0);
        s1 ^= (uint32_t)((a0 && b1) != (a1 && (b0 != b1)));
        L0 ^= (m1 & m2) ^ (a0 ? m2 : 0) ^ (b0 ? m1 : 0);
        L1 ^= (a1 ? m2 : 0) ^ (b1 ? m1 : 0);
        e += 1;
        for (Word w = (m1 | m2) & act; w;) {
            const Word lb = w & (0 - w);
            w ^= lb;
            const int i = sizeof(Word) == 4 ? __ffs((int)lb) - 1 : ffs64((uint64_t)lb);
            Word x = 0;
            if (m1 & lb) x ^= m2;
            if (m2 & lb) x ^= m1;
            rows[i * st] ^= x;
        }
    }
    e += sizeof(Word) == 4 ? __popc((unsigned)act) : __popcll((uint64_t)act);
    z0 = (L0 & act) != 0;
    z1 = ((L0 ^ L1) & act) != 0;
}

// The rest of the elimination form by form: row words are transposed so that lane f holds
// form f.  The usual case leaves at most NRM_END variables; more only when in some form
// a variable is joined to no other (a probability of 2^(1-r) per form with r variables
// left, A being uniform), on local arrays.
template <int R, int C>
__device__ __noinline__ void finish_long(const uint32_t (&S)[C][R], const uint32_t (&L)[2][C], int a, int r, int lane,
                                         uint32_t& s0, uint32_t& s1, uint32_t& z0, uint32_t& z1, int& e) {
    uint64_t rows[64];
    auto gather = [&](uint32_t x0, uint32_t x1) -> uint64_t {
        const uint32_t t = transpose32(x0, lane);
        if (C == 2) return ((uint64_t)transpose32(x1, lane) << 32 | t) >> a;
        return __funnelshift_r(t, t, a & 31);
    };
#pragma unroll 1
    for (int i = 0; i < r; ++i) rows[i] = gather(S[0][i], S[C - 1][i]);
    const uint64_t M0 = gather(L[0][0], L[0][C - 1]), M1 = gather(L[1][0], L[1][C - 1]);
    finish_form<uint64_t>(rows, 1, r, M0, M1, s0, s1, z0, z1, e);
}

template <int R, int C, int NR, int NC>
__device__ __forceinline__ void finish_many(Forms<NR, NC>& Z, int lane, uint32_t& s0, uint32_t& s1, uint32_t& z0,
                                            uint32_t& z1, int& e) {
    uint32_t S[C][R], L[2][C];
    // volatile: the compiler would otherwise store the rows in every step for this rare path
    volatile uint32_t* out = &S[0][0];
#pragma unroll
    for (int c = 0; c < C; ++c) {
#pragma unroll
        for (int i = 0; i < R; ++i) out[c * R + i] = Z.S[c][i];
        L[0][c] = Z.L0[c];
        L[1][c] = Z.L1[c];
    }
    finish_long<R, C>(S, L, Z.a, Z.m - Z.a, lane, s0, s1, z0, z1, e);
}

// Sliced steps while more than LOW variables are left, R rows at most.  A step starts at
// a <= NR - LOW - 2 (a even, m <= NR) and reads R entries of the shared vectors from there; with one
// column a lane from a mod 32.
template <int R, int C, int LOW, int NR, int NC>
__device__ __forceinline__ bool stage(Forms<NR, NC>& Z, NormWarp& W, int lane, int pos) {
    static_assert((C == 1 ? 30 : NR - LOW - 2) + R <= NRM_VEC, "a step reads past the shared vectors");
#pragma unroll 1
    while (Z.m - Z.a > LOW)
        if (!eliminate_pair<R, C>(Z, W, lane, pos)) return false;
    return true;
}

// Stages of falling row counts (a step costs its rows): two columns a lane above 32
// variables, one below.  Few stages: the warps of an SM run the same code at the same
// time (k_norm), and what matters for that is that it stays short.
template <int NR, int NC>
__device__ __forceinline__ void exponential_sum(Forms<NR, NC>& Z, NormWarp& W, int lane, uint32_t& s0, uint32_t& s1,
                                                uint32_t& z0, uint32_t& z1, int& e) {
    int pos = lane;
    e = 0;
    bool ok = true;
    if constexpr (NR > 32) {
        if constexpr (NR > 40) ok = stage<NR, 2, 40>(Z, W, lane, pos);
        if (ok) ok = stage<(NR < 40 ? NR : 40), 2, 32>(Z, W, lane, pos);
        if (!ok) {
            s0 = (Z.s0 >> lane) & 1u;
            s1 = (Z.s1 >> lane) & 1u;
            finish_many<NR, 2>(Z, lane, s0, s1, z0, z1, e);
        } else {
            // 32 or fewer variables are left: one live column a lane
            const bool low = lane >= Z.a;
            pos = low ? lane : lane + 32;
#pragma unroll
            for (int i = 0; i < 32; ++i) Z.S[0][i] = low ? Z.S[0][i] : Z.S[NC - 1][i];
            Z.L0[0] = low ? Z.L0[0] : Z.L0[NC - 1];
            Z.L1[0] = low ? Z.L1[0] : Z.L1[NC - 1];
        }
    }
    constexpr int R1 = NR < 32 ? NR : 32;
    if (ok) {
        if constexpr (R1 > 16) ok = stage<R1, 1, 16>(Z, W, lane, pos);
        if constexpr (R1 > NRM_END)
            if (ok) ok = stage<(R1 < 16 ? R1 : 16), 1, NRM_END>(Z, W, lane, pos);
        s0 = (Z.s0 >> lane) & 1u;
        s1 = (Z.s1 >> lane) & 1u;
        if (!ok) {
            finish_many<R1, 1>(Z, lane, s0, s1, z0, z1, e);
        } else {
            const int r = Z.m - Z.a;
            const uint32_t valid = (1u << r) - 1u;   // r <= NRM_END
#pragma unroll
            for (int i = 0; i < (NR < NRM_END ? NR : NRM_END); ++i) {
                if (i >= r) break;
                const uint32_t t = transpose32(Z.S[0][i], lane);
                W.rows[i][lane] = __funnelshift_r(t, t, Z.a & 31) & valid;
            }
            const uint32_t t0 = transpose32(Z.L0[0], lane), t1 = transpose32(Z.L1[0], lane);
            finish_form<uint32_t>(&W.rows[0][lane], 32, r, __funnelshift_r(t0, t0, Z.a & 31) & valid,
                                  __funnelshift_r(t1, t1, Z.a & 31) & valid, s0, s1, z0, z1, e);
        }
    }
    e += Z.a >> 1;
    __syncwarp();   // the next term rewrites the shared vectors
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}

// Warps of a block, one block per SM: what the registers allow (the matrix takes nr words, or
// 2 nr above 32 rows, and the step some 50).
constexpr int norm_warps(int nr) { return nr <= 40 ? 16 : nr <= 52 ? 12 : 8; }

// words of A and its diagonal planes in shared memory, rounded to 16 bytes
__host__ __device__ constexpr int norm_a_words(int n) { return ((n + 3) * NRM_STRIDE + 3) & ~3; }

// q_A on the basis: vec[k] = y' of free variable k (k < m), vec[m] = the constant c.  Lane q holds
// entries q and q + 32 of A vec[k]; a form's value on a pair of vectors is the XOR over
// the lanes that the other vector selects.
__device__ __noinline__ uint2 basis_products(const uint64_t* vec, int m, int n, const uint32_t* __restrict__ sA,
                                             const uint32_t* __restrict__ sD, NormWarp& W, int lane) {
    uint32_t klo = 0, khi = 0;
    uint32_t* mat = &W.mat[0][0];   // [m][32]
    uint32_t* dg = W.diag[0];       // diagonal planes
    const uint32_t* A0 = sA + lane;   // columns past n are zero
    const uint32_t* A1 = sA + (lane + 32 < n ? lane + 32 : 64);
#pragma unroll 1
    for (int k = m; k >= 0; --k) {
        const uint64_t bk = vec[k];
        uint32_t y0 = 0, y1 = 0, t0 = 0, t1 = 0, lo = 0, hi = 0;
        for (uint64_t w = bk; w; w &= w - 1) {   // A b_k, and its part from earlier qubits only
            const int j = ffs64(w);
            const uint32_t w0 = A0[j * NRM_STRIDE], w1 = A1[j * NRM_STRIDE], dl = sD[j];
            y0 ^= w0;
            y1 ^= w1;
            if (j < lane) t0 ^= w0;
            if (j < lane + 32) t1 ^= w1;
            hi ^= sD[NRM_STRIDE + j] ^ (lo & dl);
            lo ^= dl;
        }
        const uint32_t b0 = lane_mask(bk, lane), b1 = lane_mask(bk, lane + 32);
        hi ^= __reduce_xor_sync(0xffffffffu, (t0 & b0) ^ (t1 & b1));   // q_A(b_k) = lo + 2 hi
        if (k == m) {
            klo = lo;
            khi = hi;
        } else {
            const uint64_t cv = vec[m];   // with the constant: + 2 b_k . A c
            hi ^= __reduce_xor_sync(0xffffffffu, (y0 & lane_mask(cv, lane)) ^ (y1 & lane_mask(cv, lane + 32)));
            if (lane == 0) {
                dg[k] = lo;
                dg[16 + k] = hi;
                mat[k * 32 + k] = lo;     // as in A: the odd diagonal, which the lift takes out
            }
#pragma unroll 1
            for (int i = 0; i < k; ++i) {
                const uint64_t bi = vec[i];
                const uint32_t x =
                    __reduce_xor_sync(0xffffffffu, (y0 & lane_mask(bi, lane)) ^ (y1 & lane_mask(bi, lane + 32)));
                if (lane == 0) {
                    mat[k * 32 + i] = x;
                    mat[i * 32 + k] = x;
                }
            }
        }
    }
    __syncwarp();
    return make_uint2(klo, khi);
}

// The value 2^{n/2} conj<phi_A|..> contribution of one term to 32 states (lane f: state f of the
// group); false where it is zero.
template <int NR>
__device__ __forceinline__ bool norm_value(const uint64_t* rec, int rows, int n, const uint32_t* __restrict__ sA,
                                           const uint32_t* __restrict__ sD, NormWarp& W, int lane, float2& val) {
    constexpr int NC = NR > 32 ? 2 : 1;
    const uint64_t* head = rec + rows;
    const uint64_t info = head[REC_INFO], freev = head[REC_FREE];
    const int m = (int)(info & 255u), mf = n - m;
    Forms<NR, NC> Z;
    Z.a = 0;
    Z.m = m;
    Z.s0 = Z.s1 = 0;
    // natural index of every free variable, row n (zeros) past the last
#pragma unroll
    for (int c = 0; c < NC; ++c) W.off[lane + 32 * c] = (uint32_t)(n * NRM_STRIDE);
    __syncwarp();
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int q = lane + 32 * c;
        if (getb(freev, q)) W.off[__popcll(freev & (bit64(q) - 1))] = (uint32_t)(q * NRM_STRIDE);
    }
    __syncwarp();
    uint32_t col[NC], dlo[NC], dhi[NC];
    uint64_t jr[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int q = lane + 32 * c;
        const uint32_t o = W.off[q];
        col[c] = q < m ? (o * 993u) >> 16 : 64u;   // o / NRM_STRIDE
        jr[c] = q < m ? rec[q] : 0ull;
        dlo[c] = sD[col[c]];
        dhi[c] = sD[NRM_STRIDE + col[c]];
    }
    uint32_t klo = 0, khi = 0;   // constant part of q_A (Z4 planes)
    if (!((info >> 17) & 1u)) {
        // S = A + J between free variables
#pragma unroll
        for (int i = 0; i < NR; i += 4) {
            const uint4 o = *reinterpret_cast<const uint4*>(&W.off[i]);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const uint32_t* A = sA + col[c];
                const uint32_t j = i < 32 ? (uint32_t)jr[c] : (uint32_t)(jr[c] >> 32);
                switch (i & 31) {   // constant
#define NRM_ROW(b)                                                 \
        case b:                                                        \
            Z.S[c][i] = A[o.x] ^ bit_mask<b>(j);                       \
            Z.S[c][i + 1] = A[o.y] ^ bit_mask<b + 1>(j);               \
            Z.S[c][i + 2] = A[o.z] ^ bit_mask<b + 2>(j);               \
            Z.S[c][i + 3] = A[o.w] ^ bit_mask<b + 3>(j);               \
            break;
                    NRM_ROW(0) NRM_ROW(4) NRM_ROW(8) NRM_ROW(12) NRM_ROW(16) NRM_ROW(20) NRM_ROW(24) NRM_ROW(28)
#undef NRM_ROW
                }
            }
        }
        // fold the constraints into q_A: y'_p = h . y + c.  With q = row p as the earlier folds left
        // it and d its diagonal (-d if c), rows gain h q^T + q h^T + d h h^T, diagonals d h + 2 h q,
        // linear terms 2 q if c.
        const uint8_t* piv = reinterpret_cast<const uint8_t*>(head + REC_PIV);
        const uint64_t cm = head[REC_CONST];
#pragma unroll 1
        for (int i = 0; i < mf; ++i) {
            const uint32_t* Ap = sA + (int)piv[i] * NRM_STRIDE;
            uint32_t q[NC], hm[NC], hq[NC];
            uint32_t dl = sD[piv[i]], dh = sD[NRM_STRIDE + piv[i]];
#pragma unroll
            for (int c = 0; c < NC; ++c) q[c] = Ap[col[c]];
#pragma unroll 1
            for (int k = 0; k < i; ++k) {
                const uint32_t w = Ap[piv[k]];
                const uint64_t hk = rec[m + k];
#pragma unroll
                for (int c = 0; c < NC; ++c) q[c] ^= w & lane_mask(hk, lane + 32 * c);
                if (getb(cm, k)) dh ^= w;
            }
            const uint64_t h = rec[m + i];
            if (getb(cm, i)) {
                khi ^= dh ^ (klo & dl);
                klo ^= dl;
                dh ^= dl;
#pragma unroll
                for (int c = 0; c < NC; ++c) dhi[c] ^= q[c];
            }
            __syncwarp();   // the previous pass has been read
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                hm[c] = lane_mask(h, lane + 32 * c);
                const uint32_t t = dl & hm[c];
                dhi[c] ^= (dlo[c] & t) ^ (hm[c] & (dh ^ q[c]));
                dlo[c] ^= t;
                hq[c] = q[c] ^ t;
                W.pb[lane + 32 * c] = make_uint2(q[c], hm[c]);
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < NR; r += 2) {
                if (r >= 40 && r % 4 == 0 && r >= m) break;
                const uint4 w = *reinterpret_cast<const uint4*>(&W.pb[r]);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    Z.S[c][r] = xand(xand(Z.S[c][r], w.x, hm[c]), w.y, hq[c]);
                    Z.S[c][r + 1] = xand(xand(Z.S[c][r + 1], w.z, hm[c]), w.w, hq[c]);
                }
            }
        }
    } else {
        const uint2 kc = basis_products(rec + m, m, n, sA, sD, W, lane);
        klo = kc.x;
        khi = kc.y;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            dlo[c] = c == 0 && lane < m ? W.diag[0][lane] : 0u;
            dhi[c] = c == 0 && lane < m ? W.diag[1][lane] : 0u;
#pragma unroll
            for (int i = 0; i < NR; ++i) Z.S[c][i] = 0u;
        }
        if (lane < m) {
#pragma unroll
            for (int i = 0; i < (NR < 16 ? NR : 16); ++i)
                if (i < m) Z.S[0][i] = W.mat[i][lane] ^ (0u - ((uint32_t)(jr[0] >> i) & 1u));
        }
    }
    __syncwarp();
    // the whole form's diagonal, and the lift to Z2: S_ik += odd_i odd_k, odd on X
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const uint32_t jl = lane_mask(head[REC_LO], lane + 32 * c), jh = lane_mask(head[REC_HI], lane + 32 * c);
        Z.L0[c] = dhi[c] ^ jh ^ (dlo[c] & jl);
        Z.L1[c] = dlo[c] ^ jl;
        reinterpret_cast<uint32_t*>(W.pb)[lane + 32 * c] = Z.L1[c];
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < NR; r += 4) {
        const uint4 w = reinterpret_cast<const uint4*>(W.pb)[r >> 2];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            Z.S[c][r] = xand(Z.S[c][r], w.x, Z.L1[c]);
            Z.S[c][r + 1] = xand(Z.S[c][r + 1], w.y, Z.L1[c]);
            Z.S[c][r + 2] = xand(Z.S[c][r + 2], w.z, Z.L1[c]);
            Z.S[c][r + 3] = xand(Z.S[c][r + 3], w.w, Z.L1[c]);
        }
    }
    __syncwarp();
    uint32_t s0, s1, z0, z1;
    int e;
    exponential_sum(Z, W, lane, s0, s1, z0, z1, e);
    if (z0 && z1) return false;
    // sum = ((1 + i) W0 + (1 - i) W1) / 2, W0 and W1 each 0 or +-2^e (signs s0, s0 ^ s1),
    // as sqrt2^both 2^e1 e^{i pi phz / 4}
    const uint32_t t0 = s0, t1 = s0 ^ s1;
    int phz, e1 = e, both = 0;
    if (!z0 && !z1) {
        phz = (t0 ? 4 : 0) + (t0 == t1 ? 0 : 2);
    } else {
        both = 1;
        e1 = e - 1;
        phz = z1 ? (t0 ? 5 : 1) : (t1 ? 3 : 7);
    }
    const int kc = (int)((klo >> lane) & 1u) + 2 * (int)((khi >> lane) & 1u);
    const int ph = (int)((info >> 8) & 7u) - phz - 2 * kc;
    const int E = (int)(info >> 32) - 2 * e1 - both;
    const uint64_t cf = head[REC_COEF];
    val = z8_scale(make_float2(__uint_as_float((uint32_t)cf), __uint_as_float((uint32_t)(cf >> 32))), ph, E);
    return true;
}

// Terms of tile t: [t tt, (t + 1) tt).  Wide grids give each warp a tile of its own; with
// COOP the block's warps share one tile and the values are added in term order by one
// warp, so that a small call still has all warps busy.  The sums (one Kahan
// sum per state over a tile, in term order) are the same either way.
// With the warps of an SM at different places in the code the kernel waited for instructions
// half the time (348 ms at n = 50, chi = 2^20, L = 512 with blocks of four warps, 248 with this
// and a barrier each term).  So an SM runs one block, whose warps meet every NRM_SYNC terms
// (on a sixteenth of that call: 13.3 ms with a barrier each term, 12.4 every four, 12.5
// every sixteen).
template <int NR, bool COOP>
__global__ void __launch_bounds__(32 * norm_warps(NR), 1)
    k_norm(int n, int64_t chi, int64_t cap, NormPrep P, int64_t L, int64_t groups, int64_t tt,
           float2* __restrict__ partial, int64_t n_tiles) {
    constexpr int NW = norm_warps(NR);
    extern __shared__ __align__(16) uint32_t sA[];   // [n + 1][NRM_STRIDE], sD, the warps' areas, COOP values
    uint32_t* sD = sA + (n + 1) * NRM_STRIDE;        // [2][NRM_STRIDE] diagonal planes
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    NormWarp* sW = reinterpret_cast<NormWarp*>(sA + norm_a_words(n));
    float2(*sVal)[32] = reinterpret_cast<float2(*)[32]>(sW + NW);
    uint32_t* sUse = reinterpret_cast<uint32_t*>(sVal + NRM_CHUNK);
    const int64_t g = blockIdx.x % groups, tb = blockIdx.x / groups;
    for (int i = tid; i < (n + 1) * NRM_STRIDE; i += 32 * NW) {
        const int r = i / NRM_STRIDE, c = i - r * NRM_STRIDE;
        sA[i] = (r < n && c < n) ? P.A[(g * n + r) * 64 + c] : 0u;
    }
    for (int i = tid; i < 2 * NRM_STRIDE; i += 32 * NW) {
        const int r = i / NRM_STRIDE, c = i - r * NRM_STRIDE;
        sD[i] = c < n ? P.ad[(g * 2 + r) * 64 + c] : 0u;
    }
    NormWarp& W = sW[warp];
    for (int i = lane; i < NRM_VEC; i += 32) {
        W.pb[i] = make_uint2(0u, 0u);
        if (i >= 80) break;
        W.pa[i] = make_uint4(0u, 0u, 0u, 0u);
        W.off[i] = (uint32_t)(n * NRM_STRIDE);
    }
    const int64_t tile = COOP ? tb : tb * NW + warp;
    const int64_t a0 = tile * tt, a1 = tile < n_tiles ? (a0 + tt < cap ? a0 + tt : cap) : a0;
    const int step = COOP ? NW : 1;
    auto fetch = [&](int64_t alpha, int buf) {   // record of alpha into this warp's buffer
        if (alpha < a1 && alpha < chi) {
            const char* src = reinterpret_cast<const char*>(P.rec + alpha * P.words);
            for (int i = lane; i < P.words / 2; i += 32) cp_async16(reinterpret_cast<char*>(W.rec[buf]) + 16 * i, src + 16 * i);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    KahanC acc;
    acc.init();
    fetch(a0 + (COOP ? warp : 0), 0);
    // rounds are the same number for every warp of the block: one term each
    constexpr int RC = (NRM_CHUNK + NW - 1) / NW;   // rounds per chunk (COOP)
    const int rounds = COOP ? RC : (int)tt;
    int buf = 0;
#pragma unroll 1
    for (int64_t c0 = a0; c0 < a0 + tt; c0 += COOP ? NRM_CHUNK : tt) {
        const int64_t c1 = COOP ? (c0 + NRM_CHUNK < a1 ? c0 + NRM_CHUNK : a1) : a1;
#pragma unroll 1
        for (int r = 0; r < rounds; ++r) {
            const int64_t alpha = c0 + (COOP ? warp : 0) + (int64_t)r * step;
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            if (r % NRM_SYNC == 0) __syncthreads();
            __syncwarp();
            if (alpha >= c1) continue;
            int64_t next = alpha + step;
            if (COOP && next >= c0 + NRM_CHUNK) next = c0 + NRM_CHUNK + warp;
            fetch(next, buf ^ 1);
            float2 val = make_float2(0.f, 0.f);
            bool use = true;   // padding terms (weight 0) take part in the sum
            if (alpha < chi) {
                const uint64_t* rec = W.rec[buf];
                use = (rec[P.rows + REC_INFO] >> 16) & 1u;   // a projected-out term does not
                if (use) use = norm_value<NR>(rec, P.rows, n, sA, sD, W, lane, val);
            }
            buf ^= 1;
            if (COOP) {
                sVal[alpha - c0][lane] = val;
                const uint32_t u = __ballot_sync(0xffffffffu, use);
                if (lane == 0) sUse[alpha - c0] = u;
            } else if (use) {
                acc.add(val);
            }
        }
        if (COOP) {
            __syncthreads();
            if (warp == 0)
                for (int i = 0; i < (int)(c1 - c0); ++i)
                    if ((sUse[i] >> lane) & 1u) acc.add(sVal[i][lane]);
            __syncthreads();
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    const int64_t l = g * 32 + lane;
    if (l < L && tile < n_tiles && (!COOP || warp == 0)) partial[l * n_tiles + tile] = acc.value();
}

// ov (may be NULL) receives the FP64 sums themselves, 2^{n/2} <phi_{A_l}|psi> (the
// per-term values carry the 2^{n/2}), for term-sharded estimates; eta (may be NULL)
// their squared magnitude.
__global__ void k_norm_reduce(const float2* __restrict__ partial, int64_t n_tiles, int64_t L,
                              double* __restrict__ eta, double* __restrict__ ov) {
    const int64_t l = blockIdx.x;
    if (l >= L) return;
    double re = 0.0, im = 0.0;
    for (int64_t t = threadIdx.x; t < n_tiles; t += blockDim.x) {
        const float2 p = partial[l * n_tiles + t];
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
        if (eta) eta[l] = sre[0] * sre[0] + sim[0] * sim[0];
        if (ov) {
            ov[2 * l] = sre[0];
            ov[2 * l + 1] = sim[0];
        }
    }
}

__global__ void k_norm_eta(const double* __restrict__ ov, int64_t L, double* __restrict__ eta) {
    const int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l < L) eta[l] = ov[2 * l] * ov[2 * l] + ov[2 * l + 1] * ov[2 * l + 1];
}

}  // namespace

template <int NR>
static lrs_status launch_norm_t(lrs_ctx* ctx, const NormPrep& P, int64_t L, int64_t tt, float2* partial,
                                int64_t n_tiles, cudaStream_t st) {
    constexpr int NW = norm_warps(NR);
    const int64_t groups = (L + 31) / 32;
    // a tile per warp once that gives every SM two blocks
    const bool coop = n_tiles * groups < (int64_t)ctx->sm_count * NW * 2;
    constexpr size_t values = NRM_CHUNK * (32 * sizeof(float2) + sizeof(uint32_t));
    constexpr size_t most = norm_a_words(NR) * sizeof(uint32_t) + NW * sizeof(NormWarp) + values;
    const size_t smem = norm_a_words(ctx->n) * sizeof(uint32_t) + NW * sizeof(NormWarp) + (coop ? values : 0);
    const int64_t blocks = (coop ? n_tiles : (n_tiles + NW - 1) / NW) * groups;
    if (blocks > 0x7FFFFFFF) return lrs_fail(LRS_ERR_UNSUPPORTED, "norm estimate grid too large");
    const auto kernel = coop ? k_norm<NR, true> : k_norm<NR, false>;
    if (!lrs_capturing(st))
        LRS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
    kernel<<<(unsigned)blocks, 32 * NW, smem, st>>>(ctx->n, ctx->chi, ctx->cap, P, L, groups, tt, partial, n_tiles);
    LRS_LAUNCH_CHECK("norm kernel");
    return LRS_OK;
}

lrs_status launch_norm_eta(const double* ov, int64_t L, double* eta, cudaStream_t st) {
    k_norm_eta<<<(unsigned)((L + 255) / 256), 256, 0, st>>>(ov, L, eta);
    LRS_LAUNCH_CHECK("norm eta kernel");
    return LRS_OK;
}

lrs_status launch_norm_estimate(lrs_ctx* ctx, int64_t L, uint64_t seed, double* eta, double* ov,
                                cudaStream_t st) {
    if ((L + 63) / 64 > 65535) return lrs_fail(LRS_ERR_UNSUPPORTED, "L too large");
    // tile of terms per sum: keep the partial buffer at <= 2048 tiles per A
    int64_t tt = 32;
    while ((ctx->cap + tt - 1) / tt > ctx->tune_norm_tiles) tt *= 2;
    const int64_t n_tiles = (ctx->cap + tt - 1) / tt;
    const int64_t groups = (L + 31) / 32;
    void* scr = nullptr;
    // scratch: partial sums, then the per-term records and the equatorial states
    NormPrep P;
    P.rows = (ctx->n + 1) & ~1;
    P.words = P.rows + REC_HEAD;
    const size_t part_bytes = ((size_t)L * n_tiles * sizeof(float2) + 255) & ~(size_t)255;
    const size_t rec_bytes = (size_t)ctx->cap * P.words * sizeof(uint64_t);
    const size_t a_words = (size_t)groups * (ctx->n + 2) * 64;
    lrs_status rc = lrs_scratch(ctx, part_bytes + rec_bytes + a_words * sizeof(uint32_t), &scr);
    if (rc != LRS_OK) return rc;
    float2* partial = (float2*)scr;
    P.rec = (uint64_t*)((char*)scr + part_bytes);
    P.A = (uint32_t*)((char*)scr + part_bytes + rec_bytes);
    P.ad = P.A + (size_t)groups * ctx->n * 64;
    k_norm_prep<<<(unsigned)((ctx->chi + 7) / 8), 256, 0, st>>>(ctx->view(), P);
    LRS_LAUNCH_CHECK("norm prep kernel");
    k_norm_draw<<<(unsigned)groups, 32 * DRAW_WARPS, 0, st>>>(ctx->n, L, seed, P);
    LRS_LAUNCH_CHECK("equatorial state kernel");
    switch ((ctx->n + 3) / 4) {
        case 1: rc = launch_norm_t<4>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 2: rc = launch_norm_t<8>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 3: rc = launch_norm_t<12>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 4: rc = launch_norm_t<16>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 5: rc = launch_norm_t<20>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 6: rc = launch_norm_t<24>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 7: rc = launch_norm_t<28>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 8: rc = launch_norm_t<32>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 9: rc = launch_norm_t<36>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 10: rc = launch_norm_t<40>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 11: rc = launch_norm_t<44>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 12: rc = launch_norm_t<48>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 13: rc = launch_norm_t<52>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 14: rc = launch_norm_t<56>(ctx, P, L, tt, partial, n_tiles, st); break;
        case 15: rc = launch_norm_t<60>(ctx, P, L, tt, partial, n_tiles, st); break;
        default: rc = launch_norm_t<64>(ctx, P, L, tt, partial, n_tiles, st); break;
    }
    if (rc != LRS_OK) return rc;
    k_norm_reduce<<<(unsigned)L, 256, 0, st>>>(partial, n_tiles, L, eta, ov);
    LRS_LAUNCH_CHECK("norm reduce kernel");
    return LRS_OK;
}
