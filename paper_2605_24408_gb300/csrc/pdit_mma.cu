// Annealed p-dit sweep with the influence entries of many replicas formed by
// tensor-core products (zero diagonals; first: symmetric instances, entries
// of D and F in 0..127).
//
// The two influence entries of Eq. 3 for the updating location i and each
// candidate j (one-term table of Eq. 2, I[m][c] = sum_y D[m][y] F[c][p(y)])
// are, with a = p(i),
//   I[j][a]    = sum_y D[j][y] q[y],   q[y] = F[a][p(y)],
//   I[i][p(j)] = sum_c F[p(j)][c] g[c],   g[c] = D[i][p^-1(c)].
// Both matrices are the instance's own; only the vectors q and g belong to
// the replica, N bytes gathered from one row each. So the replicas of a CTA
// update the same location in lock step, and one update of all of them is
// two contractions, D x [q_1 .. q_R] and F x [g_1 .. g_R], with fixed left
// operands: no table and no permuted matrix per replica, and an accepted swap
// exchanges four bytes and updates the p-diagonal h[x] = I[x][p(x)].
//
// Products are mma.sync m16n8k16, f16 in and binary32 out. A byte b read as
// the low half of a 16-bit word is the f16 subnormal b 2^-24, so operands
// need no conversion; every product, sum and swap energy is an integer
// multiple of 2^-48 whose multiplier stays below 2^24 (2 N 127^2 + 2 127^2 at
// N = 256), hence exact in binary32. Energies stay in that unit throughout;
// draws are those of eq5_draw_core and eq5_draw_exact, so the trajectories
// equal those of the other kernels and of the CPU oracle.
//
// LPR threads (16 or 32) run one replica; thread t owns the K locations
// t*K + k. Steps of one update: the gathers (each replica's threads), a CTA
// barrier, the products (each warp holds its rows of D or F for all
// replicas), a barrier, and energies, draw and swap (each replica's threads).
// General instances (ASYM: D or F not symmetric) keep Eq. 2's two-term table,
//   T[j][a]    = sum_y D[j][y] F[a][p(y)] + D[y][j] F[p(y)][a],
//   T[i][p(j)] = sum_c F[p(j)][c] D[i][p^-1(c)] + F[c][p(j)] D[p^-1(c)][i]:
// the same products of twice the depth, [D | D^T] and [F | F^T] against
// [q; q'] and [g; g']. A unit of energy is then 2^-48 itself.
// Wide instances (symmetric, an entry above 127, none above 2047; N <= 128)
// keep 16-bit tables, which read as f16 are their entries times 2^-24 too, and
// split a vector's entries into their low 5 bits and the rest: two products
// whose sums stay below 2^24 (N 2047 63), joined as int32; energies, h and the
// swap are int32, states' energies 64 bits. N = 61, 512 replicas x 500 sweeps:
// 24.3 ms (60.6 ms with the table kernels); 1.1 to 1.8 times their speed with
// 64 replicas, 1.6 (N = 33) to 6.6 (N = 112) with 4096.
//
// Bound: the latency of an update's chain of about 450 instructions a warp
// (N = 100: issue slots 45% busy, shared-memory pipe 67%, tensor pipe 26%).
// The launch bound of two CTAs an SM holds 16 lanes at 16 warps an SM; at 97
// to 128 locations registers do (128 a thread; the spills are 36 / 64 bytes of
// stores / loads at 97, 94 / 196 at 113 locations, 150 / 304 in the wide form),
// below 81 fewer would do. With few replicas an SM other kernels are faster
// (few_replicas in pdit_host.cu). Byte permutes that form a gather's address from
// its row's, warp-uniform control and replicas paired in warps from the first
// took N = 100, 4096 replicas, from 2.13e9 to 2.39e9 updates/s (1.12e9 with
// the dot-product kernel); N = 256, 2048 replicas: 7.3e8 (1.6e8 with the table
// kernels). Bytes instead of f16 words for the vectors, with h in registers,
// cut the wavefronts by a fifth but were slower (2.03e9: more instructions);
// products formed one location ahead by warps of their own were too (1.78e9);
// two accumulators a tile, the scaled row's load ahead of the gathers and a
// total by butterfly changed nothing.
#include <type_traits>

#include "pdit_f16.cuh"
#include "pdit_sweep.cuh"

namespace pdit {

template <int K_, int LPR_, int FORM_ = kMmSymmetric>
struct MmShape {
    static constexpr int K = K_, LPR = LPR_, FORM = FORM_;
    static constexpr bool ASYM = FORM == kMmGeneral, WIDE = FORM == kMmWide;
    using V = typename std::conditional<WIDE, int, float>::type;      // energies and influence entries
    using E = typename std::conditional<WIDE, long long, int>::type;  // energies of states
    static constexpr int NP = K * LPR;            // padded size
    static constexpr int MT = NP / 16;            // 16-row tiles of D and of F; 16-deep steps of a product
    static constexpr int NW = LPR == 16 ? 8 : 16; // warps per CTA
    static constexpr int T = 32 * NW;
    static constexpr int R = 16;                  // replica slots per CTA
    static constexpr int JT = (MT + NW / 2 - 1) / (NW / 2);  // row tiles per warp
    static constexpr bool REGS = MT <= 8 && !ASYM;         // the warp's rows stay in registers
    // Row strides. Tables, bytes: 256 where the fragments are read once, so
    // that a gather's address is its row's with the byte index for the low
    // byte (one byte permute); else 16 x odd, so that 8 rows x 16 bytes read
    // by a warp fall in 32 distinct banks. Vectors, bytes: 32 mod 64, the same
    // for 64-bit reads, and the two replicas of a warp, 2 rows apart, store to
    // disjoint banks. Results, floats: 4 mod 16, so that the four column pairs
    // of a fragment store hit distinct banks and the two replicas of a warp,
    // 4 rows apart (crow), read disjoint ones.
    static constexpr int VS = 32 * (MT | 1);
    static constexpr int DS = WIDE ? VS : REGS ? 256 : 16 * (MT | 1);
    static constexpr int CS = NP + 4;
    static constexpr int PS = 8 * LPR;            // permutation bytes of a replica (8 per thread)
    // shared memory (the tables first: their rows are 256-byte aligned)
    static constexpr int TT = NP * DS, VT = R * VS;  // from a table, a vector, to its transpose's
    static constexpr int NT2 = ASYM ? 2 : 1;      // the transposes after D and F, their vectors after q and g
    static constexpr int NV2 = ASYM || WIDE ? 2 : 1;  // (wide: the high parts after the low ones)
    static constexpr int oD = 0, oF = oD + NT2 * NP * DS, oVq = oF + NT2 * NP * DS, oVg = oVq + NV2 * R * VS,
                         oC = oVg + NV2 * R * VS,
                         oR = oC + 4 * R * CS, oH = oR + 4 * R * CS, oP = oH + 4 * R * CS, oI = oP + R * PS,
                         oDr = oI + R * PS, oX = oDr + 8 * NP, bytes = oX + 16;
    // result row of the replica in vector row v: bits 1 and 2 of v trade places
    __host__ __device__ static constexpr int crow(int v) {
        return LPR == 32 ? v : (v & ~6) | ((v & 2) << 1) | ((v & 4) >> 1);
    }
    // Orders. Locations (rows and columns of D, the vector q, the results C,
    // h): t*K + k at pos(t, k), pairs of a thread's locations together, so
    // that it moves two as one word. Facilities (F, the vector g, the
    // results R): their own order. Permutation bytes: 8 per thread.
    __host__ __device__ static constexpr int pos(int t, int k) {
        return k < (K & ~1) ? (k >> 1) * 2 * LPR + 2 * t + (k & 1) : (K - 1) * LPR + t;
    }
    __device__ static int loc(int j) { return pos(j / K, j % K); }
    __device__ static int pbyte(int j) { return (j / K) * 8 + j % K; }
    // byte of facility c in the inverse permutation: the inverse of pos
    __device__ static int ibyte(int c) {
        if (c >= (K & ~1) * LPR) return (c - (K - 1) * LPR) * 8 + K - 1;
        return ((c % (2 * LPR)) >> 1) * 8 + 2 * (c / (2 * LPR)) + (c & 1);
    }
};

// Byte k of the eight in v.
__device__ __forceinline__ int byte8(const uint2 v, int k) {
    return (int)__byte_perm(k < 4 ? v.x : v.y, 0, 0x4440 | (k & 3));
}

__device__ __forceinline__ int lds_s32(uint32_t a) {
    int v;
    asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ int lds_u16(uint32_t a) {
    int v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}

template <int K, typename V>
struct MmVals {
    V v[K];
};

// Weight of an outcome d above the least dmin: binary32 units of `scale`, or
// integers of half the energy.
__device__ __forceinline__ unsigned long long mm_weight(float d, float dmin, float scale, float beta) {
    return eq5_weight_f((d - dmin) * scale, beta);
}
__device__ __forceinline__ unsigned long long mm_weight(int d, int dmin, float, float beta) {
    return eq5_weight(2 * (d - dmin), beta);
}
__device__ __forceinline__ float mm_top(float) { return __int_as_float(0x7F800000); }
__device__ __forceinline__ int mm_top(int) { return 0x7FFFFFFF; }
__device__ __forceinline__ float mm_min(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ int mm_min(int a, int b) { return min(a, b); }

// The exact draw (eq5_draw_exact) for one replica's LPR threads; beyond n
// where no outcome has a weight.
template <int K, int LPR, typename V>
__device__ __noinline__ int mm_exact_draw(const MmVals<K, V> d, int n, int t, float scale, float beta,
                                          unsigned long long draw, unsigned mask) {
    V dmin = mm_top(V());
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (t * K + k < n) dmin = mm_min(dmin, d.v[k]);
#pragma unroll
    for (int o = LPR / 2; o; o >>= 1) dmin = mm_min(dmin, __shfl_xor_sync(mask, dmin, o, LPR));
    unsigned long long pre[K];
    unsigned long long lsum = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (t * K + k < n) lsum += mm_weight(d.v[k], dmin, scale, beta);
        pre[k] = lsum;
    }
    unsigned long long incl = lsum;
#pragma unroll
    for (int o = 1; o < LPR; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(mask, incl, o, LPR);
        if (t >= o) incl += y;
    }
    const unsigned long long total = __shfl_sync(mask, incl, LPR - 1, LPR);
    const unsigned long long excl = incl - lsum;
    const unsigned long long tdraw = __umul64hi(draw, total);
    int j = 0x7FFFFFFF;
#pragma unroll
    for (int k = K - 1; k >= 0; --k)
        if (tdraw >= excl && excl + pre[k] > tdraw) j = t * K + k;
#pragma unroll
    for (int o = LPR / 2; o; o >>= 1) j = min(j, __shfl_xor_sync(mask, j, o, LPR));
    return j;
}

// Address of entry byte8(v, k) of the table row at `row`.
template <class S>
__device__ __forceinline__ uint32_t entry(uint32_t row, const uint2 v, int k) {
    if constexpr (S::WIDE)
        return row + 2u * (uint32_t)byte8(v, k);
    else if constexpr (S::DS == 256)
        return __byte_perm(k < 4 ? v.x : v.y, row, 0x7650 | (k & 3));
    else
        return row + (uint32_t)byte8(v, k);
}

// The table entry at an address.
template <class S>
__device__ __forceinline__ int lds_entry(uint32_t a) {
    return S::WIDE ? lds_u16(a) : lds_u8(a);
}

// The fragment of a wide table: 16-bit entries are f16 numbers as they stand.
template <int DS>
__device__ __forceinline__ void mm_frag_wide(const uint8_t *tab, int row0, int s, int lane, uint32_t (&a)[4]) {
    const uint8_t *p = tab + (row0 + (lane >> 2)) * DS + 32 * s + 8 * (lane & 3);
    const uint2 x = *reinterpret_cast<const uint2 *>(p);
    const uint2 y = *reinterpret_cast<const uint2 *>(p + 8 * DS);
    a[0] = x.x;
    a[1] = y.x;
    a[2] = x.y;
    a[3] = y.y;
}

// D and F of an instance into the CTA's tables (zero outside n x n),
// and the warp's rows into registers where they stay there. Ends with the
// CTA synchronised.
template <class S>
__device__ __forceinline__ void mm_stage(const int32_t *D, const int32_t *F, int n, unsigned char *sm,
                                         uint32_t (&A)[S::JT][S::REGS ? S::MT : 1][4]) {
    uint32_t *z = reinterpret_cast<uint32_t *>(sm + S::oD);
    for (int w = threadIdx.x; w < 2 * S::NT2 * S::NP * S::DS / 4; w += S::T) z[w] = 0u;
    __syncthreads();
    for (int idx = threadIdx.x; idx < n * n; idx += S::T) {
        const int x = idx / n, y = idx - x * n;
        if constexpr (S::WIDE) {
            *reinterpret_cast<uint16_t *>(sm + S::oD + S::loc(x) * S::DS + 2 * S::loc(y)) = (uint16_t)D[idx];
            *reinterpret_cast<uint16_t *>(sm + S::oF + x * S::DS + 2 * y) = (uint16_t)F[idx];
            continue;
        }
        sm[S::oD + S::loc(x) * S::DS + S::loc(y)] = (uint8_t)D[idx];
        sm[S::oF + x * S::DS + y] = (uint8_t)F[idx];
        if constexpr (S::ASYM) {
            sm[S::oD + S::TT + S::loc(y) * S::DS + S::loc(x)] = (uint8_t)D[idx];
            sm[S::oF + S::TT + y * S::DS + x] = (uint8_t)F[idx];
        }
    }
    __syncthreads();
    if constexpr (S::REGS) {
        const int w = __shfl_sync(kFull, threadIdx.x >> 5, 0);
        const uint8_t *tab = sm + (w < S::NW / 2 ? S::oD : S::oF);
#pragma unroll
        for (int jt = 0; jt < S::JT; ++jt) {
            const int m = min(w % (S::NW / 2) + jt * (S::NW / 2), S::MT - 1);
#pragma unroll
            for (int s = 0; s < S::MT; ++s) {
                if constexpr (S::WIDE)
                    mm_frag_wide<S::DS>(tab, 16 * m, s, threadIdx.x & 31, A[jt][s]);
                else
                    mm_frag<S::DS>(tab, 16 * m, s, threadIdx.x & 31, A[jt][s]);
            }
        }
    }
}

// This warp's row tiles of D x [q] or F x [g] for NT x 8 replicas.
template <class S, int NT>
__device__ __forceinline__ void mm_products(unsigned char *sm, int w, const uint32_t (&A)[S::JT][S::REGS ? S::MT : 1][4]) {
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, q = lane & 3;
    const bool second = w >= S::NW / 2;
    const int m0 = w % (S::NW / 2);
    if (m0 >= S::MT) return;
    const uint8_t *tab = sm + (second ? S::oF : S::oD);
    const unsigned char *v = sm + (second ? S::oVg : S::oVq) + g * S::VS + 8 * q;
    constexpr int NA = S::WIDE ? 2 : 1;  // wide: the high parts' products by themselves
    float acc[S::JT][NA * NT][4];
#pragma unroll
    for (int jt = 0; jt < S::JT; ++jt)
#pragma unroll
        for (int nt = 0; nt < NA * NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[jt][nt][e] = 0.0f;
#pragma unroll
    for (int d = 0; d < S::NT2 * S::MT; ++d) {
        const int s = d % S::MT, tr = d / S::MT;  // the second half: the transposes
        uint2 b[NA * NT];
#pragma unroll
        for (int nt = 0; nt < NA * NT; ++nt)
            b[nt] = *reinterpret_cast<const uint2 *>(v + (tr + nt / NT) * S::VT + 8 * (nt % NT) * S::VS + 32 * s);
#pragma unroll
        for (int jt = 0; jt < S::JT; ++jt) {
            const int m = m0 + jt * (S::NW / 2);
            if (S::MT % (S::NW / 2) != 0 && jt == S::JT - 1 && m >= S::MT) continue;
            if constexpr (S::REGS) {
#pragma unroll
                for (int nt = 0; nt < NA * NT; ++nt) mma_f16(acc[jt][nt], A[jt][s], b[nt]);
            } else {
                uint32_t a[4];
                mm_frag<S::DS>(tab + tr * S::TT, 16 * m, s, lane, a);
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) mma_f16(acc[jt][nt], a, b[nt]);
            }
        }
    }
    // columns 2q and 2q + 1 of a tile go to result rows crow(2q) and, one on, crow(2q + 1)
    using V = typename S::V;
    V *out = reinterpret_cast<V *>(sm + (second ? S::oR : S::oC)) + S::crow(2 * q) * S::CS + g;
#pragma unroll
    for (int jt = 0; jt < S::JT; ++jt) {
        const int m = m0 + jt * (S::NW / 2);
        if (m >= S::MT) break;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            V *o = out + 8 * nt * S::CS + 16 * m;
            V x[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if constexpr (S::WIDE)  // units of 2^-48: low + 32 high
                    x[e] = (int)(acc[jt][nt][e] * (0.5f * kMmScale)) + 32 * (int)(acc[jt][NT + nt][e] * (0.5f * kMmScale));
                else
                    x[e] = acc[jt][nt][e];
            }
            o[0] = x[0];
            o[S::CS] = x[1];
            o[8] = x[2];
            o[S::CS + 8] = x[3];
        }
    }
}

// p-diagonal entries of this thread's locations, h[x] = sum_y D[y][x]
// F[p(y)][p(x)] (symmetric; general form: and the transposes'), from the replica's permutation bytes (integers);
// one row of each table at a time.
template <class S>
__device__ __forceinline__ void mm_diagonal(const unsigned char *sm, const uint8_t *pb, int n, int t, int (&h)[S::K]) {
    constexpr int K = S::K;
    int px[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        h[k] = 0;
        px[k] = pb[t * 8 + k];
    }
#pragma unroll 2
    for (int y = 0; y < n; ++y) {
        const uint8_t *dr = sm + S::oD + S::loc(y) * S::DS, *fr = sm + S::oF + pb[S::pbyte(y)] * S::DS;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if constexpr (S::WIDE)
                h[k] += (int)reinterpret_cast<const uint16_t *>(dr)[S::pos(t, k)] *
                        (int)reinterpret_cast<const uint16_t *>(fr)[px[k]];
            else
                h[k] += (int)dr[S::pos(t, k)] * (int)fr[px[k]];
            if constexpr (S::ASYM) h[k] += (int)dr[S::TT + S::pos(t, k)] * (int)fr[S::TT + px[k]];
        }
    }
}

template <int LPR, typename E>
__device__ __forceinline__ E mm_sum(E v, unsigned mask) {
#pragma unroll
    for (int o = LPR / 2; o; o >>= 1) v += __shfl_xor_sync(mask, v, o, LPR);
    return v;
}

// One block of up to 16 replicas: part `part` of their sweeps (see
// part_begin), r0 the local id of the first.
template <class S>
__device__ __forceinline__ void mm_run_block(const SweepArgs &a, int r0, int part, unsigned char *sm,
                                             const uint32_t (&A)[S::JT][S::REGS ? S::MT : 1][4]) {
    constexpr int K = S::K, LPR = S::LPR;
    constexpr bool ASYM = S::ASYM, WIDE = S::WIDE;
    using V = typename S::V;
    using Acc = typename S::E;
    constexpr float kScale = ASYM ? 0.5f * kMmScale : kMmScale;
    const int tid = threadIdx.x, w = __shfl_sync(kFull, tid >> 5, 0), lane = tid & 31;
    const int half = LPR == 16 ? lane >> 4 : 0;
    const int t = lane & (LPR - 1);
    const unsigned mask = LPR == 32 ? kFull : 0xFFFFu << (16 * half);
    const int n = a.n;
    const int count = min(a.groups, a.replicas - r0);  // replicas of this block
    // vector row of this thread's replica; the two of a warp are 2 apart.
    // More than 8 replicas fill the warps two by two.
    const int v0 = LPR == 32 ? w : (w & 1) + 4 * (w >> 1);
    const int slot = v0 + 2 * half;
    const int idx = LPR == 16 && count > 8 ? 2 * w + half : slot;
    const bool live = idx < count;
    const bool warp_live = (LPR == 16 && count > 8 ? 2 * w : v0) < count;
    const int r = r0 + idx;
    const uint32_t grep = a.rep_base + (uint32_t)r;
    V *sC = reinterpret_cast<V *>(sm + S::oC) + S::crow(slot) * S::CS;
    V *sR = reinterpret_cast<V *>(sm + S::oR) + S::crow(slot) * S::CS;
    V *sH = reinterpret_cast<V *>(sm + S::oH) + S::crow(slot) * S::CS;
    uint8_t *pb = sm + S::oP + slot * S::PS;
    uint8_t *ib = sm + S::oI + slot * S::PS;
    float *drow = reinterpret_cast<float *>(sm + S::oDr);
    volatile int *flag = reinterpret_cast<volatile int *>(sm + S::oX);
    // shared-window addresses
    const uint32_t base32 = (uint32_t)__cvta_generic_to_shared(sm);
    const uint32_t aP = base32 + S::oP + slot * S::PS, aI = aP + (S::oI - S::oP);
    const uint32_t aC = base32 + S::oC + 4 * S::crow(slot) * S::CS, aR = aC + (S::oR - S::oC), aH = aC + (S::oH - S::oC);
    int32_t *gp = a.perm + (size_t)r * n;
    int32_t *gbp = a.best_perm + (size_t)r * n;
    const bool fresh = part == 0 && a.fresh;

    // (|E| <= n^2 127^2 < 2^31, and twice that in the general form's sums;
    // wide: 64 bits)
    // (the best sweep and the accepted swaps stay in global memory)
    Acc E = 0, bestE = 0;
    bool reached = false;
    if (warp_live) {
        // ---- permutation: bytes by thread, and its inverse. A slot without
        // a replica holds the identity.
        int32_t *tmp = reinterpret_cast<int32_t *>(sC);
        uint32_t *wrd = reinterpret_cast<uint32_t *>(sR);
        for (int m = t; m < S::NP; m += LPR) tmp[m] = m;
        __syncwarp();
        if (live) {
            if (fresh) {
                for (int q = t; 4 * q < n; q += LPR) {
                    const uint4 o = philox4x32_10(a.inst, grep, 0xFFFFFFFFu, (uint32_t)q, a.key0, a.key1);
                    wrd[4 * q] = o.x;
                    wrd[4 * q + 1] = o.y;
                    wrd[4 * q + 2] = o.z;
                    wrd[4 * q + 3] = o.w;
                }
                __syncwarp(mask);
                if (t == 0) {
                    for (int k = n - 1; k >= 1; --k) {
                        const int j = (int)__umulhi(wrd[k], (uint32_t)(k + 1));
                        const int x = tmp[k];
                        tmp[k] = tmp[j];
                        tmp[j] = x;
                    }
                }
            } else {
                for (int m = t; m < n; m += LPR) tmp[m] = __ldcg(gp + m);
            }
        }
        __syncwarp();
        for (int j = t; j < S::NP; j += LPR) {
            const int c = tmp[j];
            pb[S::pbyte(j)] = (uint8_t)c;
            ib[S::ibyte(c)] = (uint8_t)S::loc(j);
        }
        __syncwarp();
        // ---- p-diagonal and energy: E = sum_x h[x] (Eq. 1 regrouped)
        int h[K];
        Acc esum = 0;
        mm_diagonal<S>(sm, pb, n, t, h);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            esum += h[k];
            // an entry beyond n: an energy of +infinity, a weight of 0
            if constexpr (WIDE)
                sH[S::pos(t, k)] = h[k];
            else
                sH[S::pos(t, k)] = t * K + k < n ? (float)h[k] * kMmUnit : __int_as_float(0xFF800000);
        }
        esum = mm_sum<LPR>(esum, kFull);
        if constexpr (S::ASYM) esum >>= 1;
        if (live) {
            if (fresh) {
                E = bestE = esum;
                for (int m = t; m < n; m += LPR) gbp[m] = tmp[m];
                if (t == 0) {
                    a.best_sweep[r] = -1;
                    a.accepted[r] = 0;
                    note_target(a, bestE, -1, reached);
                }
            } else {
                E = (Acc)__ldcg(a.energy + r);
                bestE = (Acc)__ldcg(a.best_energy + r);
                if (E != esum && t == 0) atomicOr(a.status, 1);
            }
        }
        __syncwarp();
    }
    const int s_begin = part_begin(a, part);
    const int s_end = part >= a.segments - 1 ? a.sweep_end : part_begin(a, part + 1);
    auto beta_of = [&](int s) {
        return a.mode == 1 || a.mode == 2 ? (!live ? 0.0f : a.mode == 1 ? a.beta[a.rung[r]] : a.beta[r]) : a.beta[s];
    };
    int par = 0;
    const uint32_t aV = base32 + S::oVq + slot * S::VS + 4 * t;  // this thread's words of q; g at + oVg - oVq

    for (int s = s_begin; s < s_end; ++s) {
        if (a.stop) {
            // one read of the instance's flag for the whole block
            __syncthreads();
            if (tid == 0) *flag = *reinterpret_cast<volatile int *>(a.done);
            __syncthreads();
            if (*flag) break;
        }
        // (never 0, so that an infinite energy always has weight 0; a beta
        // that is not a number stays one, so that the exact draw decides)
        const float kb = min_nan(-beta_of(s) * kLog2e * (WIDE ? 2.0f : kScale), -1e-37f);
        uint32_t rhi = 0;  // high words of the draws of LPR locations
        int moves = 0;
        // location i = ti K + ki
        for (int i = 0, ti = 0, ki = 0; i < n; ++i) {
            if ((i & (LPR - 1)) == 0 && warp_live) {
                // Philox(inst, replica, sweep, location) for the next LPR locations
                rhi = philox4x32_10(a.inst, grep, (uint32_t)s, (uint32_t)(i + t), a.key0, a.key1).y;
            }
            const int xi = S::pos(ti, ki);
            const uint32_t aDi = base32 + S::oD + xi * S::DS;
            const uint32_t aDr = base32 + S::oDr + par * 4 * S::NP;  // 2 D_ij (D_ij + D_ji) units
            uint2 p8 = make_uint2(0, 0);
            int pi = 0, qb[K], qt[ASYM ? K : 1];  // F_ab, F_ba of this thread's locations
            uint32_t aFi = 0;
            // ---- vectors
            if constexpr (WIDE) {
                if (tid < S::NP) asm volatile("st.shared.b32 [%0], %1;" ::"r"(aDr + 4 * tid), "r"(2 * lds_u16(aDi + 2 * tid)));
            } else if (tid < S::NP) {
                const float x = ASYM ? (float)(lds_u8(aDi + tid) + lds_u8(aDi + S::TT + tid)) * kMmUnit
                                     : (float)lds_u8(aDi + tid) * (2.0f * kMmUnit);
                asm volatile("st.shared.f32 [%0], %1;" ::"r"(aDr + 4 * tid), "f"(x));
            }
            if (warp_live) {
                pi = lds_u8(aP + 8 * ti + ki);
                p8 = lds_u64(aP + 8 * t);
                const uint2 i8 = lds_u64(aI + 8 * t);
                aFi = base32 + S::oF + pi * S::DS;
                auto put = [&](uint32_t at, const int (&x)[K]) {
#pragma unroll
                    for (int k = 0; k < K; k += 2) {
                        const uint32_t v = k + 1 < K ? __byte_perm(x[k], x[k + 1 < K ? k + 1 : k], 0x5410) : (uint32_t)x[k];
#pragma unroll
                        for (int part = 0; part < (WIDE ? 2 : 1); ++part) {  // low 5 bits, the bits above
                            const uint32_t y = !WIDE ? v : part == 0 ? v & 0x001F001Fu : (v >> 5) & 0x003F003Fu;
                            if (k + 1 < K)
                                asm volatile("st.shared.b32 [%0], %1;" ::"r"(at + part * S::VT + k * 2 * LPR), "r"(y));
                            else
                                asm volatile("st.shared.b16 [%0], %1;" ::"r"(at + part * S::VT - 2 * t + k * 2 * LPR),
                                             "h"((uint16_t)y));
                        }
                    }
                };
                int gb[K];
#pragma unroll
                for (int k = 0; k < K; ++k) gb[k] = lds_entry<S>(entry<S>(aDi, i8, k));
#pragma unroll
                for (int k = 0; k < K; ++k) qb[k] = lds_entry<S>(entry<S>(aFi, p8, k));
                put(aV + (S::oVg - S::oVq), gb);
                put(aV, qb);
                if constexpr (ASYM) {
#pragma unroll
                    for (int k = 0; k < K; ++k) gb[k] = lds_u8(entry<S>(aDi, i8, k) + S::TT);
#pragma unroll
                    for (int k = 0; k < K; ++k) qt[k] = lds_u8(entry<S>(aFi, p8, k) + S::TT);
                    put(aV + (S::oVg - S::oVq) + S::VT, gb);
                    put(aV + S::VT, qt);
                }
            }
            __syncthreads();
            // ---- products
            if (count > 8)
                mm_products<S, 2>(sm, w, A);
            else
                mm_products<S, 1>(sm, w, A);
            __syncthreads();
            if (warp_live) {
                // ---- swap energies, half of Eq. 3, up to the common h_i:
                // I[i][p(j)] + I[j][p(i)] - h_j + 2 D_ij F_ab
                V hi;  // I[i][p(i)]
                MmVals<K, V> e;
                V hk[K];
                float mq[WIDE ? 1 : K], pre[K], lsum = 0.0f;
                if constexpr (WIDE) {
                    hi = lds_s32(aR + 4 * pi);
#pragma unroll
                    for (int k = 0; k < K; ++k) {
                        const uint32_t x = 4 * S::pos(t, k);
                        hk[k] = lds_s32(aH + x);
                        e.v[k] = lds_s32(aDr + x) * qb[k] + lds_s32(aR + 4 * byte8(p8, k)) + (lds_s32(aC + x) - hk[k]);
                        const float w = ex2_approx(__int2float_rn(e.v[k] - hi) * kb);
                        pre[k] = t * K + k < n ? w : 0.0f;
                    }
                } else {
                hi = lds_f32(aR + 4 * pi);
#pragma unroll
                for (int k = 0; k < K; ++k)  // 2^23 + F_ab (F_ab + F_ba)
                    mq[k] = __int_as_float(0x4B000000 | (ASYM ? qb[k] + qt[ASYM ? k : 0] : qb[k]));
#pragma unroll
                for (int k = 0; k + 1 < K; k += 2) {
                    const uint32_t x = 4 * k * LPR + 8 * t;
                    const float2 c = lds_f64(aC + x);
                    const float2 h = lds_f64(aH + x);
                    const float2 d = lds_f64(aDr + x);
                    const float2 rr = make_float2(lds_f32(aR + 4 * byte8(p8, k)), lds_f32(aR + 4 * byte8(p8, k + 1)));
                    const float2 q = sub2(make_float2(mq[k], mq[k + 1]), two(8388608.0f));
                    const float2 v = fma2(d, q, add2(rr, sub2(c, h)));
                    hk[k] = h.x;
                    hk[k + 1] = h.y;
                    e.v[k] = v.x;
                    e.v[k + 1] = v.y;
                }
                if constexpr (K & 1) {
                    constexpr int k = K - 1;
                    const uint32_t x = 4 * (k * LPR + t);
                    hk[k] = lds_f32(aH + x);
                    e.v[k] = fmaf(lds_f32(aDr + x), mq[k] - 8388608.0f, lds_f32(aR + 4 * byte8(p8, k)) + (lds_f32(aC + x) - hk[k]));
                }
                // ---- binary32 draw, kept where it is certainly the exact
                // one (eq5_draw_core): no interval end within m of t
                const float bias = -kb * hi;
#pragma unroll
                for (int k = 0; k + 1 < K; k += 2) {
                    const float2 x = fma2(make_float2(e.v[k], e.v[k + 1]), two(kb), two(bias));
                    pre[k] = ex2_approx(x.x);
                    pre[k + 1] = ex2_approx(x.y);
                }
                if constexpr (K & 1) pre[K - 1] = ex2_approx(fmaf(e.v[K - 1], kb, bias));
                }
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    lsum += pre[k];
                    pre[k] = lsum;
                }
                float incl = lsum;
#pragma unroll
                for (int o = 1; o < LPR; o <<= 1) {
                    const float y = __shfl_up_sync(kFull, incl, o, LPR);
                    if (t >= o) incl += y;
                }
                const float total = __shfl_sync(kFull, incl, LPR - 1, LPR);
                const uint32_t dhi = __shfl_sync(kFull, rhi, i & (LPR - 1), LPR);
                const float tt = __uint2float_rn(dhi >> 8) * 5.9604644775390625e-08f * total;
                const float mg = total < kDrawLimit ? kDrawMargin * total : __int_as_float(0x7FC00000);
                const float base = (incl - lsum) - tt;
                float near = fabsf(base), z = base;
                int kk = 0;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    z = pre[k] + base;
                    near = fminf(near, fabsf(z));
                    kk += (int)((uint32_t)__float_as_int(z) >> 31);
                }
                const unsigned ball = __ballot_sync(kFull, base < 0.0f && z > 0.0f && near > mg) & mask;
                // the drawn location tj K + kj and its facility, from its owner
                int v = __shfl_sync(kFull, (t << 8) | kk | (int)(__byte_perm(p8.x, p8.y, kk) << 16), __ffs(ball) - 1);
                if (__any_sync(kFull, ball == 0)) {
                    const uint32_t dlo = philox4x32_10(a.inst, grep, (uint32_t)s, (uint32_t)i, a.key0, a.key1).x;
                    const int jx = mm_exact_draw<K, LPR>(e, n, t, kScale, beta_of(s), ((unsigned long long)dhi << 32) | dlo, kFull);
                    if (ball == 0) {
                        const int js = jx < n ? jx : i;  // (no outcome has a weight: the location stays)
                        const int tx = js / K, kx = js - tx * K;
                        v = (tx << 8) | kx | (lds_u8(aP + 8 * tx + kx) << 16);
                    }
                }
                const int tj = (v >> 8) & 0xFF, kj = v & 0xFF;
                // ---- apply the swap i <-> j (facilities a = p(i), b = p(j))
                const bool sw = tj != ti || kj != ki;
                if (__any_sync(kFull, sw)) {
                    const int fb = (v >> 16) & 0xFF;
                    const int xj = S::pos(tj, kj);
                    const uint32_t aFj = base32 + S::oF + fb * S::DS, aDj = base32 + S::oD + xj * S::DS;
                    V rs, cs, dq, dd;  // dq: what the swap adds to both moved entries of h, D_ij F_ab (D_ij F_ba + D_ji F_ab)
                    V hw[WIDE ? K : 1];
                    float2 hn[WIDE ? 1 : K / 2 + 1];
                    if constexpr (WIDE) {
                        rs = lds_s32(aR + 4 * fb);
                        cs = lds_s32(aC + 4 * xj);
                        dq = (lds_s32(aDr + 4 * xj) >> 1) * lds_u16(aFi + 2 * fb);
                        dd = (rs - hi) + (cs - lds_s32(aH + 4 * xj)) + 2 * dq;
                        // h[m] += (D_im - D_jm) (F_b,p(m) - F_a,p(m))
#pragma unroll
                        for (int k = 0; k < K; ++k) {
                            const int u = (lds_s32(aDr + 4 * S::pos(t, k)) >> 1) - lds_u16(aDj + 2 * S::pos(t, k));
                            hw[k] = hk[k] + u * (lds_u16(entry<S>(aFj, p8, k)) - qb[k]);
                        }
                    } else {
                    rs = lds_f32(aR + 4 * fb);
                    cs = lds_f32(aC + 4 * xj);
                    const float hs = lds_f32(aH + 4 * xj);
                    if constexpr (ASYM) {
                        const int fab = lds_u8(aFi + fb), fba = lds_u8(aFi + S::TT + fb);
                        dq = (float)(lds_u8(aDi + xj) * fba + lds_u8(aDi + S::TT + xj) * fab) * kMmUnit;
                        dd = lds_f32(aDr + 4 * xj) * (float)(fab + fba);
                    } else {
                        dq = 0.5f * lds_f32(aDr + 4 * xj) * (float)lds_u8(aFi + fb);
                        dd = 2.0f * dq;
                    }
                    dd = (rs - hi) + (cs - hs) + dd;
                    // h[m] += (D_im - D_jm) (F_b,p(m) - F_a,p(m))
                    auto word = [&](uint32_t at) {  // a pair of a row of D at this thread's locations
                        uint32_t x;
                        asm volatile("ld.shared.u16 %0, [%1];" : "=r"(x) : "r"(at + 2 * t));
                        return x;
                    };
                    auto units = [](uint32_t x) {  // 2^-25 + entry units
                        return make_float2(__int_as_float((int)__byte_perm(x, 0x33000000u, 0x7540)),
                                           __int_as_float((int)__byte_perm(x, 0x33000000u, 0x7541)));
                    };
                    auto ones = [](int x) { return __int_as_float(0x4B000000 | x); };  // 2^23 + entry
#pragma unroll
                    for (int k = 0; k + 1 < K; k += 2) {
                        float2 u;
                        if constexpr (ASYM)
                            u = sub2(units(word(aDi + k * LPR)), units(word(aDj + k * LPR)));
                        else
                            u = sub2(fma2(lds_f64(aDr + 4 * k * LPR + 8 * t), two(0.5f), two(kMmOne)),
                                     units(word(aDj + k * LPR)));
                        const float2 fbk = make_float2(ones(lds_u8(entry<S>(aFj, p8, k))), ones(lds_u8(entry<S>(aFj, p8, k + 1))));
                        const float2 fak = ASYM ? make_float2(ones(qb[k]), ones(qb[k + 1])) : make_float2(mq[k], mq[k + 1]);
                        float2 x = fma2(u, sub2(fbk, fak), make_float2(hk[k], hk[k + 1]));
                        if constexpr (ASYM) {
                            const float2 ut = sub2(units(word(aDi + S::TT + k * LPR)), units(word(aDj + S::TT + k * LPR)));
                            const float2 ft = make_float2(ones(lds_u8(entry<S>(aFj, p8, k) + S::TT)),
                                                          ones(lds_u8(entry<S>(aFj, p8, k + 1) + S::TT)));
                            x = fma2(ut, sub2(ft, make_float2(ones(qt[k]), ones(qt[k + 1]))), x);
                        }
                        hn[k / 2] = x;
                    }
                    if constexpr (K & 1) {
                        constexpr int k = K - 1;
                        auto unit = [&](uint32_t row) { return __int_as_float(0x33000000 | lds_u8(row + k * LPR + t)); };
                        const float u = (ASYM ? unit(aDi) : fmaf(lds_f32(aDr + 4 * (k * LPR + t)), 0.5f, kMmOne)) - unit(aDj);
                        float x = fmaf(u, ones(lds_u8(entry<S>(aFj, p8, k))) - (ASYM ? ones(qb[k]) : mq[k]), hk[k]);
                        if constexpr (ASYM)
                            x = fmaf(unit(aDi + S::TT) - unit(aDj + S::TT),
                                     ones(lds_u8(entry<S>(aFj, p8, k) + S::TT)) - ones(qt[k]), x);
                        hn[K / 2].x = x;
                    }
                    }
                    __syncwarp();  // reads of h and p by the replica's threads done
                    if (sw) {
                        if constexpr (WIDE) {
#pragma unroll
                            for (int k = 0; k < K; ++k) sH[S::pos(t, k)] = hw[k];
                            E += 2 * dd;
                        } else {
#pragma unroll
                        for (int k = 0; k + 1 < K; k += 2) *reinterpret_cast<float2 *>(sH + k * LPR + 2 * t) = hn[k / 2];
                        if constexpr (K & 1) sH[(K - 1) * LPR + t] = hn[K / 2].x;
                        E += (int)(dd * kScale);
                        }
                        moves += 1;
                    }
                    __syncwarp();
                    if (sw && t < 2) {  // one moved facility and location each
                        const bool first = t == 0;
                        sH[first ? xi : xj] = (first ? rs : cs) + dq;
                        pb[first ? 8 * ti + ki : 8 * tj + kj] = (uint8_t)(first ? fb : pi);
                        ib[S::ibyte(first ? fb : pi)] = (uint8_t)(first ? xi : xj);
                    }
                    __syncwarp();
                    if (live && E < bestE) {
                        bestE = E;
                        const uint2 b8 = *reinterpret_cast<const uint2 *>(pb + 8 * t);
#pragma unroll
                        for (int k = 0; k < K; ++k)
                            if (t * K + k < n) gbp[t * K + k] = byte8(b8, k);
                        if (t == 0) {
                            a.best_sweep[r] = s;
                            note_target(a, bestE, s, reached);
                        }
                    }
                    __syncwarp();
                }
            }
            par ^= 1;
            if (++ki == K) {
                ki = 0;
                ++ti;
            }
        }
        if (live && t == 0) atomicAdd(reinterpret_cast<unsigned long long *>(a.accepted + r), (unsigned long long)moves);
    }

    // ---- audit (the last unit of a call; a resumed unit begins with the same
    // check): Eq. 1 of the final permutation equals the tracked energy; write
    // back
    if (warp_live) {
        if (a.audit && part >= a.segments - 1) {
            int h[K];
            Acc eq1 = 0;
            mm_diagonal<S>(sm, pb, n, t, h);
#pragma unroll
            for (int k = 0; k < K; ++k) eq1 += h[k];
            eq1 = mm_sum<LPR>(eq1, kFull);
            if constexpr (S::ASYM) eq1 >>= 1;
            if (live && t == 0 && eq1 != E) atomicOr(a.status, 1);
        }
        if (live) {
            for (int m = t; m < n; m += LPR) gp[m] = pb[S::pbyte(m)];
            if (t == 0) {
                a.energy[r] = E;
                a.best_energy[r] = bestE;
            }
        }
    }
}

// Persistent: CTAs take (block of replicas, part) units in order, part k of
// every block before part k + 1 (one part: one unit per block); see
// dot_kernel for why the wait for the part before ends.
template <class S>
__global__ void __launch_bounds__(S::T, S::LPR == 16 ? 2 : 1) mm_kernel(const SweepArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    uint32_t A[S::JT][S::REGS ? S::MT : 1][4];
    mm_stage<S>(a.D, a.F, a.n, smem, A);
    volatile int *x = reinterpret_cast<volatile int *>(smem + S::oX);
    const int blocks = (a.replicas + a.groups - 1) / a.groups;
    const int parts = a.segments > 1 ? a.segments : 1;
    const long long units = (long long)blocks * parts;
    for (;;) {
        if (threadIdx.x == 0) {
            const int item = atomicAdd(a.queue, 1);
            int go = item < units ? 1 : 0;
            const int part = go ? item / blocks : 0, b = item - part * blocks;
            if (go && part > 0) go = wait_part(a, b, part);
            x[1] = b;
            x[2] = part;
            x[3] = go;
        }
        __syncthreads();
        const int b = x[1], part = x[2], go = x[3];
        if (!go) break;
        mm_run_block<S>(a, b * a.groups, part, smem, A);
        if (parts > 1) __threadfence();
        __syncthreads();
        if (parts > 1 && threadIdx.x == 0) publish_part(a, b, part + 1);
    }
}

// Persistent multi-instance kernel: CTAs take (instance, block of replicas)
// units from `queue` and restage the tables when they move to another
// instance. Every instance of a launch shares the compiled shape.
template <class S>
__global__ void __launch_bounds__(S::T, S::LPR == 16 ? 2 : 1)
    mm_batch_kernel(const SweepArgs *__restrict__ descs, const BatchUnit *__restrict__ units, int nunits, int *queue) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ SweepArgs sa;
    __shared__ int s_unit;
    uint32_t A[S::JT][S::REGS ? S::MT : 1][4];
    int cur = -1;
    for (;;) {
        if (threadIdx.x == 0) s_unit = atomicAdd(queue, 1);
        __syncthreads();
        const int u = s_unit;
        if (u >= nunits) break;
        const BatchUnit bu = units[u];
        if (bu.inst != cur) {
            const int *src = reinterpret_cast<const int *>(descs + bu.inst);
            int *dst = reinterpret_cast<int *>(&sa);
            for (int w = threadIdx.x; w < (int)(sizeof(SweepArgs) / sizeof(int)); w += S::T) dst[w] = src[w];
            mm_stage<S>(descs[bu.inst].D, descs[bu.inst].F, descs[bu.inst].n, smem, A);
            cur = bu.inst;
        }
        __syncthreads();
        mm_run_block<S>(sa, bu.r0, 0, smem, A);
        __syncthreads();
    }
}

// One launch, a query of the single-instance kernel's shape, or the
// occupancy of the multi-instance kernel.
struct MmCall {
    const SweepArgs *args = nullptr;   // launch the single-instance kernel
    const SweepArgs *descs = nullptr;  // launch the multi-instance kernel
    const BatchUnit *units = nullptr;
    int nunits = 0;
    int *queue = nullptr;
    int grid = 0;
    cudaStream_t st = nullptr;
    MmInfo *info = nullptr;
    int *batch_blocks = nullptr;
};

template <int K, int LPR, int FORM>
static int mm_one(const MmCall &c) {
    using S = MmShape<K, LPR, FORM>;
    const bool batch = c.descs || c.batch_blocks;
    const cudaError_t e =
        batch ? cudaFuncSetAttribute(mm_batch_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::bytes)
              : cudaFuncSetAttribute(mm_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::bytes);
    if (e != cudaSuccess) return (int)e;
    if (c.batch_blocks)
        return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(c.batch_blocks, mm_batch_kernel<S>, S::T, S::bytes);
    if (c.info) {
        c.info->threads = S::T;
        c.info->slots = S::R;
        c.info->lanes = LPR;
        c.info->k = K;
        c.info->smem = S::bytes;
        return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c.info->blocks_per_sm, mm_kernel<S>, S::T, S::bytes);
    }
    if (batch)
        mm_batch_kernel<S><<<c.grid, S::T, S::bytes, c.st>>>(c.descs, c.units, c.nunits, c.queue);
    else
        mm_kernel<S><<<c.grid, S::T, S::bytes, c.st>>>(*c.args);
    return (int)cudaGetLastError();
}

template <int FORM>
static int mm_dispatch_form(int n, const MmCall &c) {
    if (n <= 128) {
        switch ((n + 15) / 16) {
        case 3: return mm_one<3, 16, FORM>(c);
        case 4: return mm_one<4, 16, FORM>(c);
        case 5: return mm_one<5, 16, FORM>(c);
        case 6: return mm_one<6, 16, FORM>(c);
        case 7: return mm_one<7, 16, FORM>(c);
        default: return mm_one<8, 16, FORM>(c);
        }
    }
    if constexpr (FORM != kMmWide)
        if ((n + 31) / 32 == 5) return mm_one<5, 32, FORM>(c);
    if constexpr (FORM == kMmSymmetric) {  // (the general form's four tables end at 160 locations)
        switch ((n + 31) / 32) {
        case 6: return mm_one<6, 32, FORM>(c);
        case 7: return mm_one<7, 32, FORM>(c);
        default: return mm_one<8, 32, FORM>(c);
        }
    }
    return (int)cudaErrorInvalidValue;
}

static int mm_dispatch(int n, int form, const MmCall &c) {
    if (n <= 32 || n > kMmMax[form]) return (int)cudaErrorInvalidValue;
    return form == kMmGeneral ? mm_dispatch_form<kMmGeneral>(n, c)
         : form == kMmWide    ? mm_dispatch_form<kMmWide>(n, c)
                              : mm_dispatch_form<kMmSymmetric>(n, c);
}

int mm_query(int n, int form, MmInfo *info) {
    MmCall c;
    c.info = info;
    return mm_dispatch(n, form, c);
}

int mm_launch(const SweepArgs &a, int form, int grid, cudaStream_t st) {
    MmCall c;
    c.args = &a;
    c.grid = grid;
    c.st = st;
    return mm_dispatch(a.n, form, c);
}

int mm_batch_blocks_per_sm(int n, int form, int *blocks) {
    MmCall c;
    c.batch_blocks = blocks;
    return mm_dispatch(n, form, c);
}

int mm_batch_launch(int n, int form, const SweepArgs *descs, const BatchUnit *units, int nunits, int *queue, int grid,
                    cudaStream_t st) {
    MmCall c;
    c.descs = descs;
    c.units = units;
    c.nunits = nunits;
    c.queue = queue;
    c.grid = grid;
    c.st = st;
    return mm_dispatch(n, form, c);
}

}  // namespace pdit
