// Annealed p-dit sweep with the influence entries of many replicas formed by
// tensor-core products (symmetric instances, zero diagonals, entries of D and
// F in 0..127).
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
//
// Bound: shared-memory wavefronts (93 per update at N = 100, 69% of the
// pipe's cycles), then the latency of the three phases. Measured at N = 100,
// 4096 replicas: 2.13e9 updates/s against 1.22e9 with the dot-product kernel;
// N = 256, 2048 replicas: 7.4e8 against 1.8e8 with the table kernels.
#include "pdit_sweep.cuh"

namespace pdit {

template <int K_, int LPR_>
struct MmShape {
    static constexpr int K = K_, LPR = LPR_;
    static constexpr int NP = K * LPR;            // padded size
    static constexpr int MT = NP / 16;            // 16-row tiles of D and of F; 16-deep steps of a product
    static constexpr int NW = LPR == 16 ? 8 : 16; // warps per CTA
    static constexpr int T = 32 * NW;
    static constexpr int R = 16;                  // replica slots per CTA
    static constexpr int JT = (MT + NW / 2 - 1) / (NW / 2);  // row tiles per warp
    static constexpr bool REGS = MT <= 8;         // the warp's rows stay in registers
    // Row strides. Tables, bytes: 16 x odd, so that 8 rows x 16 bytes read by
    // a warp fall in 32 distinct banks. Vectors, bytes: 32 mod 64, the same
    // for 64-bit reads. Results, floats: 4 mod 16, so that the four column
    // pairs of a fragment store and the replicas of one warp (r, r + 4) hit
    // distinct banks.
    static constexpr int DS = 16 * (MT | 1);
    static constexpr int VS = 32 * (MT | 1);
    static constexpr int CS = NP + 4;
    static constexpr int PS = 8 * LPR;            // permutation bytes of a replica (8 per thread)
    // shared memory
    static constexpr int oD = 0, oF = oD + NP * DS, oVq = oF + NP * DS, oVg = oVq + R * VS, oC = oVg + R * VS,
                         oR = oC + 4 * R * CS, oH = oR + 4 * R * CS, oP = oH + 4 * R * CS, oI = oP + R * PS,
                         oDr = oI + R * PS, oX = oDr + 8 * NP, bytes = oX + 16;
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

constexpr float kMmUnit = 3.552713678800501e-15f;   // 2^-48: one unit of energy / 2
constexpr float kMmScale = 5.62949953421312e14f;    // 2^49: energy per unit
constexpr float kMmOne = 2.98023223876953125e-08f;  // 2^-25: the unit in its last place

// Two binary32 operations at once (each rounded as the single one).
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 d;
    asm("{ .reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; add.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z; }"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    float2 d;
    asm("{ .reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; sub.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z; }"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{ .reg .b64 x, y, z, w; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; mov.b64 w, {%6, %7}; "
        "fma.rn.f32x2 z, x, y, w; mov.b64 {%0, %1}, z; }"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float2 two(float v) { return make_float2(v, v); }

// Byte k of the eight in v.
__device__ __forceinline__ int byte8(const uint2 v, int k) {
    return (int)__byte_perm(k < 4 ? v.x : v.y, 0, 0x4440 | (k & 3));
}

template <int K>
struct MmVals {
    float v[K];
};

// The exact draw (eq5_draw_exact) for one replica's LPR threads.
template <int K, int LPR>
__device__ __noinline__ int mm_exact_draw(const MmVals<K> d, int n, int t, float beta, unsigned long long draw,
                                          unsigned mask) {
    float dmin = __int_as_float(0x7F800000);
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (t * K + k < n) dmin = fminf(dmin, d.v[k]);
#pragma unroll
    for (int o = LPR / 2; o; o >>= 1) dmin = fminf(dmin, __shfl_xor_sync(mask, dmin, o, LPR));
    unsigned long long pre[K];
    unsigned long long lsum = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (t * K + k < n) lsum += eq5_weight_f((d.v[k] - dmin) * kMmScale, beta);
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

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], const uint2 b) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// The 16 x 16 fragment of rows row0.. of a table at depth step s. Depth order
// within a step: a thread's four consecutive bytes are the fragment's (2q,
// 2q + 1) and (2q + 8, 2q + 9), as in the vectors.
template <int DS>
__device__ __forceinline__ void mm_frag(const uint8_t *tab, int row0, int s, int lane, uint32_t (&a)[4]) {
    const uint8_t *p = tab + (row0 + (lane >> 2)) * DS + 16 * s + 4 * (lane & 3);
    const uint32_t x = *reinterpret_cast<const uint32_t *>(p);
    const uint32_t y = *reinterpret_cast<const uint32_t *>(p + 8 * DS);
    a[0] = __byte_perm(x, 0, 0x4140);
    a[1] = __byte_perm(y, 0, 0x4140);
    a[2] = __byte_perm(x, 0, 0x4342);
    a[3] = __byte_perm(y, 0, 0x4342);
}

// D and F of an instance into the CTA's tables (bytes, zero outside n x n),
// and the warp's rows into registers where they stay there. Ends with the
// CTA synchronised.
template <class S>
__device__ __forceinline__ void mm_stage(const int32_t *D, const int32_t *F, int n, unsigned char *sm,
                                         uint32_t (&A)[S::JT][S::REGS ? S::MT : 1][4]) {
    uint32_t *z = reinterpret_cast<uint32_t *>(sm + S::oD);
    for (int w = threadIdx.x; w < 2 * S::NP * S::DS / 4; w += S::T) z[w] = 0u;
    __syncthreads();
    for (int idx = threadIdx.x; idx < n * n; idx += S::T) {
        const int x = idx / n, y = idx - x * n;
        sm[S::oD + S::loc(x) * S::DS + S::loc(y)] = (uint8_t)D[idx];
        sm[S::oF + x * S::DS + y] = (uint8_t)F[idx];
    }
    __syncthreads();
    if constexpr (S::REGS) {
        const int w = threadIdx.x >> 5;
        const uint8_t *tab = sm + (w < S::NW / 2 ? S::oD : S::oF);
#pragma unroll
        for (int jt = 0; jt < S::JT; ++jt) {
            const int m = min(w % (S::NW / 2) + jt * (S::NW / 2), S::MT - 1);
#pragma unroll
            for (int s = 0; s < S::MT; ++s) mm_frag<S::DS>(tab, 16 * m, s, threadIdx.x & 31, A[jt][s]);
        }
    }
}

// This warp's row tiles of D x [q] or F x [g] for NT x 8 replicas.
template <class S, int NT>
__device__ __forceinline__ void mm_products(unsigned char *sm, const uint32_t (&A)[S::JT][S::REGS ? S::MT : 1][4]) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, q = lane & 3;
    const bool second = w >= S::NW / 2;
    const int m0 = w % (S::NW / 2);
    if (m0 >= S::MT) return;
    const uint8_t *tab = sm + (second ? S::oF : S::oD);
    const unsigned char *v = sm + (second ? S::oVg : S::oVq) + g * S::VS + 8 * q;
    float acc[S::JT][NT][4];
#pragma unroll
    for (int jt = 0; jt < S::JT; ++jt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[jt][nt][e] = 0.0f;
#pragma unroll
    for (int s = 0; s < S::MT; ++s) {
        uint2 b[NT];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) b[nt] = *reinterpret_cast<const uint2 *>(v + 8 * nt * S::VS + 32 * s);
#pragma unroll
        for (int jt = 0; jt < S::JT; ++jt) {
            const int m = m0 + jt * (S::NW / 2);
            if (S::MT % (S::NW / 2) != 0 && jt == S::JT - 1 && m >= S::MT) continue;
            if constexpr (S::REGS) {
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) mma_f16(acc[jt][nt], A[jt][s], b[nt]);
            } else {
                uint32_t a[4];
                mm_frag<S::DS>(tab, 16 * m, s, lane, a);
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) mma_f16(acc[jt][nt], a, b[nt]);
            }
        }
    }
    float *out = reinterpret_cast<float *>(sm + (second ? S::oR : S::oC));
#pragma unroll
    for (int jt = 0; jt < S::JT; ++jt) {
        const int m = m0 + jt * (S::NW / 2);
        if (m >= S::MT) break;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            float *o = out + (8 * nt + 2 * q) * S::CS + 16 * m + g;
            o[0] = acc[jt][nt][0];
            o[S::CS] = acc[jt][nt][1];
            o[8] = acc[jt][nt][2];
            o[S::CS + 8] = acc[jt][nt][3];
        }
    }
}

// p-diagonal entries of this thread's locations, h[x] = sum_y D[x][y]
// F[p(x)][p(y)], from the replica's permutation bytes (integers).
template <class S>
__device__ __forceinline__ void mm_diagonal(const unsigned char *sm, const uint8_t *pb, int n, int t, int (&h)[S::K]) {
    constexpr int K = S::K;
    const uint8_t *fr[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        h[k] = 0;
        fr[k] = sm + S::oF + pb[t * 8 + k] * S::DS;
    }
    for (int y = 0; y < n; ++y) {
        const int py = pb[S::pbyte(y)];
        const uint8_t *dc = sm + S::oD + S::loc(y);
#pragma unroll
        for (int k = 0; k < K; ++k) h[k] += (int)dc[S::pos(t, k) * S::DS] * (int)fr[k][py];
    }
}

template <int LPR>
__device__ __forceinline__ int mm_sum(int v, unsigned mask) {
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
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int half = LPR == 16 ? lane >> 4 : 0;
    const int t = lane & (LPR - 1);
    const unsigned mask = LPR == 32 ? kFull : 0xFFFFu << (16 * half);
    const int n = a.n;
    const int count = min(a.groups, a.replicas - r0);  // replicas of this block
    // slot of this thread's replica; the two of a warp are 4 apart (row strides)
    const int slot = LPR == 32 ? w : (w & 3) + 8 * (w >> 2) + 4 * half;
    const bool live = slot < count;
    const bool warp_live = LPR == 32 ? live : (w & 3) + 8 * (w >> 2) < count;
    const int r = r0 + slot;
    const uint32_t grep = a.rep_base + (uint32_t)r;
    float *sC = reinterpret_cast<float *>(sm + S::oC) + slot * S::CS;
    float *sR = reinterpret_cast<float *>(sm + S::oR) + slot * S::CS;
    float *sH = reinterpret_cast<float *>(sm + S::oH) + slot * S::CS;
    uint8_t *pb = sm + S::oP + slot * S::PS;
    uint8_t *ib = sm + S::oI + slot * S::PS;
    float *drow = reinterpret_cast<float *>(sm + S::oDr);
    volatile int *flag = reinterpret_cast<volatile int *>(sm + S::oX);
    int32_t *gp = a.perm + (size_t)r * n;
    int32_t *gbp = a.best_perm + (size_t)r * n;
    const bool fresh = part == 0 && a.fresh;

    // (|E| <= n^2 127^2 < 2^31)
    int E = 0, bestE = 0, bsweep = -1;
    long long acc_moves = 0;
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
        int h[K], esum = 0;
        mm_diagonal<S>(sm, pb, n, t, h);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            esum += h[k];
            // an entry beyond n: an energy of +infinity, a weight of 0
            sH[S::pos(t, k)] = t * K + k < n ? (float)h[k] * kMmUnit : __int_as_float(0xFF800000);
        }
        esum = mm_sum<LPR>(esum, kFull);
        if (live) {
            if (fresh) {
                E = bestE = esum;
                for (int m = t; m < n; m += LPR) gbp[m] = tmp[m];
                if (t == 0) note_target(a, bestE, -1, reached);
            } else {
                E = (int)__ldcg(a.energy + r);
                bestE = (int)__ldcg(a.best_energy + r);
                bsweep = __ldcg(a.best_sweep + r);
                acc_moves = __ldcg(a.accepted + r);
                if (E != esum && t == 0) atomicOr(a.status, 1);
            }
        }
        __syncwarp();
    }
    const int s_begin = part_begin(a, part);
    const int s_end = part >= a.segments - 1 ? a.sweep_end : part_begin(a, part + 1);
    const float beta_fixed = a.sweep_end <= a.sweep_begin || !live ? 0.0f
                           : a.mode == 1 ? a.beta[a.rung[r]] : a.mode == 2 ? a.beta[r] : 0.0f;
    int par = 0;

    for (int s = s_begin; s < s_end; ++s) {
        if (a.stop) {
            // one read of the instance's flag for the whole block
            __syncthreads();
            if (tid == 0) *flag = *reinterpret_cast<volatile int *>(a.done);
            __syncthreads();
            if (*flag) break;
        }
        const float beta = (a.mode == 1 || a.mode == 2) ? beta_fixed : a.beta[s];
        // (never 0, so that an infinite energy always has weight 0)
        const float kb = fminf(-beta * kLog2e * kMmScale, -1e-37f);
        uint32_t rlo = 0, rhi = 0;
        int moves = 0;
        // location i = ti K + ki
        for (int i = 0, ti = 0, ki = 0; i < n; ++i) {
            if ((i & (LPR - 1)) == 0 && warp_live) {
                // Philox(inst, replica, sweep, location) for the next LPR locations
                const uint4 rw = philox4x32_10(a.inst, grep, (uint32_t)s, (uint32_t)(i + t), a.key0, a.key1);
                rlo = rw.x;
                rhi = rw.y;
            }
            const int xi = S::pos(ti, ki);
            const uint8_t *Drow = sm + S::oD + xi * S::DS;
            float *dr = drow + par * S::NP;  // 2 D_ij units
            uint2 p8 = make_uint2(0, 0);
            int pi = 0, qb[K];
            const uint8_t *Frow = sm;
            // ---- vectors
            if (tid < S::NP) dr[tid] = (float)Drow[tid] * (2.0f * kMmUnit);
            if (warp_live) {
                pi = pb[8 * ti + ki];
                p8 = *reinterpret_cast<const uint2 *>(pb + 8 * t);
                const uint2 i8 = *reinterpret_cast<const uint2 *>(ib + 8 * t);
                Frow = sm + S::oF + pi * S::DS;
                int gb[K];
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    gb[k] = Drow[byte8(i8, k)];
                    qb[k] = Frow[byte8(p8, k)];
                }
                unsigned char *vq = sm + S::oVq + slot * S::VS, *vg = sm + S::oVg + slot * S::VS;
#pragma unroll
                for (int k = 0; k + 1 < K; k += 2) {
                    *reinterpret_cast<uint32_t *>(vg + k * 2 * LPR + 4 * t) = (uint32_t)gb[k] + 65536u * (uint32_t)gb[k + 1];
                    *reinterpret_cast<uint32_t *>(vq + k * 2 * LPR + 4 * t) = (uint32_t)qb[k] + 65536u * (uint32_t)qb[k + 1];
                }
                if constexpr (K & 1) {
                    *reinterpret_cast<uint16_t *>(vg + (K - 1) * 2 * LPR + 2 * t) = (uint16_t)gb[K - 1];
                    *reinterpret_cast<uint16_t *>(vq + (K - 1) * 2 * LPR + 2 * t) = (uint16_t)qb[K - 1];
                }
            }
            __syncthreads();
            // ---- products
            if (count > 8)
                mm_products<S, 2>(sm, A);
            else
                mm_products<S, 1>(sm, A);
            __syncthreads();
            if (warp_live) {
                // ---- swap energies, half of Eq. 3, up to the common h_i:
                // I[i][p(j)] + I[j][p(i)] - h_j + 2 D_ij F_ab
                const float hi = sR[pi];  // I[i][p(i)]
                MmVals<K> e;
                float hk[K], mq[K], di[K];
#pragma unroll
                for (int k = 0; k < K; ++k) mq[k] = __int_as_float(0x4B000000 | qb[k]);  // 2^23 + F_ab
#pragma unroll
                for (int k = 0; k + 1 < K; k += 2) {
                    const int x = k * LPR + 2 * t;
                    const float2 c = *reinterpret_cast<const float2 *>(sC + x);
                    const float2 h = *reinterpret_cast<const float2 *>(sH + x);
                    const float2 d = *reinterpret_cast<const float2 *>(dr + x);
                    const float2 rr = make_float2(sR[byte8(p8, k)], sR[byte8(p8, k + 1)]);
                    const float2 q = sub2(make_float2(mq[k], mq[k + 1]), two(8388608.0f));
                    const float2 v = fma2(d, q, add2(rr, sub2(c, h)));
                    hk[k] = h.x;
                    hk[k + 1] = h.y;
                    di[k] = d.x;
                    di[k + 1] = d.y;
                    e.v[k] = v.x;
                    e.v[k + 1] = v.y;
                }
                if constexpr (K & 1) {
                    constexpr int k = K - 1;
                    const int x = k * LPR + t;
                    hk[k] = sH[x];
                    di[k] = dr[x];
                    e.v[k] = fmaf(di[k], mq[k] - 8388608.0f, sR[byte8(p8, k)] + (sC[x] - hk[k]));
                }
                // ---- binary32 draw, kept where it is certainly the exact
                // one (eq5_draw_core): no interval end within m of t
                const float bias = -kb * hi;
                float pre[K], lsum = 0.0f;
#pragma unroll
                for (int k = 0; k + 1 < K; k += 2) {
                    const float2 x = fma2(make_float2(e.v[k], e.v[k + 1]), two(kb), two(bias));
                    pre[k] = ex2_approx(x.x);
                    pre[k + 1] = ex2_approx(x.y);
                }
                if constexpr (K & 1) pre[K - 1] = ex2_approx(fmaf(e.v[K - 1], kb, bias));
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
                int tj, kj, fb;  // the drawn location tj K + kj and its facility
                if (ball) {
                    const int own = __ffs(ball) - 1;
                    const int v = __shfl_sync(mask, kk | (int)(__byte_perm(p8.x, p8.y, kk) << 8), own);
                    tj = own & (LPR - 1);
                    kj = v & 0xFF;
                    fb = (v >> 8) & 0xFF;
                } else {
                    const uint32_t dlo = __shfl_sync(mask, rlo, i & (LPR - 1), LPR);
                    const int js = mm_exact_draw<K, LPR>(e, n, t, beta, ((unsigned long long)dhi << 32) | dlo, mask);
                    tj = js / K;
                    kj = js - tj * K;
                    fb = pb[8 * tj + kj];
                }
                __syncwarp();
                // ---- apply the swap i <-> j (facilities fa = p(i), fb = p(j))
                const bool sw = tj != ti || kj != ki;
                if (__any_sync(kFull, sw)) {
                    const int xj = S::pos(tj, kj);
                    const uint8_t *Fb = sm + S::oF + fb * S::DS;
                    const uint8_t *Dj = sm + S::oD + xj * S::DS;
                    const float rs = sR[fb], cs = sC[xj], hs = sH[xj];
                    const float dq = 0.5f * dr[xj] * (float)Frow[fb];  // D_ij F_ab
                    // h[m] += (D_im - D_jm) (F_b,p(m) - F_a,p(m))
                    float2 hn[K / 2 + 1];
#pragma unroll
                    for (int k = 0; k + 1 < K; k += 2) {
                        const uint32_t dj = *reinterpret_cast<const uint16_t *>(Dj + k * LPR + 2 * t);
                        // 2^-25 + D_jm units
                        const float2 mj = make_float2(__int_as_float(__byte_perm(dj, 0x33000000u, 0x7540)),
                                                      __int_as_float(__byte_perm(dj, 0x33000000u, 0x7541)));
                        const float2 u = sub2(fma2(make_float2(di[k], di[k + 1]), two(0.5f), two(kMmOne)), mj);
                        const float2 v = sub2(make_float2(__int_as_float(0x4B000000 | (int)Fb[byte8(p8, k)]),
                                                          __int_as_float(0x4B000000 | (int)Fb[byte8(p8, k + 1)])),
                                              make_float2(mq[k], mq[k + 1]));
                        hn[k / 2] = fma2(u, v, make_float2(hk[k], hk[k + 1]));
                    }
                    if constexpr (K & 1) {
                        constexpr int k = K - 1;
                        const float mj = __int_as_float(0x33000000 | (int)Dj[k * LPR + t]);
                        const float v = __int_as_float(0x4B000000 | (int)Fb[byte8(p8, k)]) - mq[k];
                        hn[K / 2].x = fmaf(fmaf(di[k], 0.5f, kMmOne) - mj, v, hk[k]);
                    }
                    __syncwarp();  // reads of h and p by the replica's threads done
                    if (sw) {
#pragma unroll
                        for (int k = 0; k + 1 < K; k += 2) *reinterpret_cast<float2 *>(sH + k * LPR + 2 * t) = hn[k / 2];
                        if constexpr (K & 1) sH[(K - 1) * LPR + t] = hn[K / 2].x;
                        E += (int)(((rs - hi) + (cs - hs) + 2.0f * dq) * kMmScale);
                        moves += 1;
                    }
                    __syncwarp();
                    if (sw && t == 0) {
                        sH[xi] = rs + dq;
                        sH[xj] = cs + dq;
                        pb[8 * ti + ki] = (uint8_t)fb;
                        pb[8 * tj + kj] = (uint8_t)pi;
                        ib[S::ibyte(pi)] = (uint8_t)xj;
                        ib[S::ibyte(fb)] = (uint8_t)xi;
                    }
                    __syncwarp();
                    if (live && E < bestE) {
                        bestE = E;
                        bsweep = s;
                        const uint2 b8 = *reinterpret_cast<const uint2 *>(pb + 8 * t);
#pragma unroll
                        for (int k = 0; k < K; ++k)
                            if (t * K + k < n) gbp[t * K + k] = byte8(b8, k);
                        if (t == 0) note_target(a, bestE, s, reached);
                    }
                }
            }
            par ^= 1;
            if (++ki == K) {
                ki = 0;
                ++ti;
            }
        }
        acc_moves += moves;
    }

    // ---- audit (the last unit of a call): Eq. 1 of the final permutation
    // equals the tracked energy; write back
    if (warp_live) {
        if (part >= a.segments - 1) {
            int h[K], eq1 = 0;
            mm_diagonal<S>(sm, pb, n, t, h);
#pragma unroll
            for (int k = 0; k < K; ++k) eq1 += h[k];
            eq1 = mm_sum<LPR>(eq1, kFull);
            if (live && t == 0 && eq1 != E) atomicOr(a.status, 1);
        }
        if (live) {
            for (int m = t; m < n; m += LPR) gp[m] = pb[S::pbyte(m)];
            if (t == 0) {
                a.energy[r] = E;
                a.best_energy[r] = bestE;
                a.best_sweep[r] = bsweep;
                a.accepted[r] = acc_moves;
            }
        }
    }
}

// Persistent: CTAs take (block of replicas, part) units in order, part k of
// every block before part k + 1 (one part: one unit per block); see
// dot_kernel for why the wait for the part before ends.
template <class S>
__global__ void __launch_bounds__(S::T, S::LPR == 16 ? 2 : 1) mm_kernel(const SweepArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
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

template <int K, int LPR>
static int mm_one(const SweepArgs &a, int grid, cudaStream_t st, MmInfo *info) {
    using S = MmShape<K, LPR>;
    auto fn = mm_kernel<S>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, S::bytes);
    if (e != cudaSuccess) return (int)e;
    if (info) {
        info->threads = S::T;
        info->slots = S::R;
        info->lanes = LPR;
        info->k = K;
        info->smem = S::bytes;
        return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(&info->blocks_per_sm, fn, S::T, S::bytes);
    }
    fn<<<grid, S::T, S::bytes, st>>>(a);
    return (int)cudaGetLastError();
}

static int mm_dispatch(int n, const SweepArgs &a, int grid, cudaStream_t st, MmInfo *info) {
    if (n <= 128) {
        switch ((n + 15) / 16) {
        case 1: return mm_one<1, 16>(a, grid, st, info);
        case 2: return mm_one<2, 16>(a, grid, st, info);
        case 3: return mm_one<3, 16>(a, grid, st, info);
        case 4: return mm_one<4, 16>(a, grid, st, info);
        case 5: return mm_one<5, 16>(a, grid, st, info);
        case 6: return mm_one<6, 16>(a, grid, st, info);
        case 7: return mm_one<7, 16>(a, grid, st, info);
        default: return mm_one<8, 16>(a, grid, st, info);
        }
    }
    switch ((n + 31) / 32) {
    case 5: return mm_one<5, 32>(a, grid, st, info);
    case 6: return mm_one<6, 32>(a, grid, st, info);
    case 7: return mm_one<7, 32>(a, grid, st, info);
    case 8: return mm_one<8, 32>(a, grid, st, info);
    default: return (int)cudaErrorInvalidValue;
    }
}

int mm_query(int n, MmInfo *info) { return mm_dispatch(n, SweepArgs{}, 0, nullptr, info); }

int mm_launch(const SweepArgs &a, int grid, cudaStream_t st) { return mm_dispatch(a.n, a, grid, st, nullptr); }

}  // namespace pdit
