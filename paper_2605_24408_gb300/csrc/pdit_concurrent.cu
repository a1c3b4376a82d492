// Concurrent updates (mode 3) of symmetric instances with zero diagonals and
// entries of D and F in 0..127, up to 128 locations: one CTA per replica.
//
// Every location proposes from the same state, so an iteration needs all N^2
// swap energies at once, and those are products. With the permuted flow
// G[x][y] = F[p(x)][p(y)] and S = D G + G D (S[x][y] = I[x][p(y)] + I[y][p(x)]
// in Eq. 2's one-term table), Eq. 3 is
//   dE(x, y) = 2 S[x][y] - S[x][x] - S[y][y] + 4 D[x][y] G[x][y],
// and the energy of a state is half the trace of S. So an iteration is a
// rebuild of G (a byte gather), a product of depth 2N, the energies in the
// accumulators, N draws of four lanes each, and the matching; an iteration
// that accepts nothing leaves the state and its energies as they are.
//
// Layout. Rows of the products are "slots": slot 8 t + 2 q + e is location
// 4 MT q + 2 t + e, so that in mma.sync's accumulator, where lane (g, q) has
// columns 8 t + 2 q + {0, 1} of every tile t, a lane owns 4 MT consecutive
// outcomes of its two rows, and a draw is a serial sum with a scan of four
// lanes. Columns of D and G in memory are locations; the rows, 16 x odd bytes
// apart, fall in distinct banks for 8 rows x 16 bytes. Bytes enter the
// products as f16 subnormals (see pdit_mma.cu); |dE| and every partial sum
// stay below 2^24, exact in binary32.
//
// Matching: a proposal whose priority (energy change, then location) is the
// least among those left at both of its locations is accepted, in rounds;
// that is the set the greedy pass in priority order accepts. Acceptance and
// energies are exact, so the trajectories equal the table kernels'.
//
// Bound: an iteration's latency, about 17000 clocks at N = 100, 7000 of them
// the two products (two warps a scheduler reach half of mma.sync's rate; loads
// of a step ahead of its products made no difference) and 2000 to 4000 the
// matching, two CTAs an SM overlapped. N = 100, 4096 replicas x 60 iterations:
// 7.0 ms (7.8 ms with both products at this size too, 8.8 ms with two warps a
// row tile; 21.6 ms with the table kernels, which update every table entry for
// every accepted swap); N = 12, 64 replicas: 0.21 ms (0.57 ms).
#include "pdit_f16.cuh"
#include "pdit_sweep.cuh"

namespace pdit {

template <int MT_>
struct CcShape {
    static constexpr int MT = MT_, NT = 2 * MT, NP = 16 * MT, T = 32 * MT, LC = 4 * MT;
    static constexpr int GS = 16 * (MT | 1);  // row stride of D and G, bytes
    static constexpr int FS = 256;            // of F: an entry's address is its row's with the column for the low byte
    static constexpr int CTAS = (MT >= 7 ? 512 : MT >= 5 ? 640 : 768) / T;  // resident CTAs an SM aimed at (more spill)
    // S = J + J^T, J = D G exchanged through shared memory, at 97 to 112
    // locations, where it is faster; else both products. 4096 replicas x 60
    // iterations, J or both: N = 100 7.0 or 7.8 ms; N = 96 5.8 or 5.2, N = 64
    // 2.2 or 2.0 (J's memory leaves fewer CTAs an SM); N = 128: J leaves one;
    // N = 32 0.64 or 0.61, N = 16 0.32 or 0.31 (as many CTAs, but the products
    // are short and the exchange is not).
    static constexpr bool TR = MT == 7;
    static constexpr int CS = NP + 4;  // row stride of J, floats: the transposed reads of a warp in distinct banks (NP = 112)
    // shared memory, bytes (F first: its rows are 256-byte aligned)
    static constexpr int oF = 0, oD = oF + NP * FS, oG = oD + NP * GS, oP = oG + NP * GS, oS = oP + 128,
                         oB = oS + 4 * (NP + 8), oTk = oB + 2 * 4 * 128, oX = oTk + 128,
                         oJ = oX + 32, bytes = oJ + (TR ? 4 * NP * CS : 0);
    __host__ __device__ static constexpr int slot(int x) {
        return 8 * ((x % LC) >> 1) + 2 * (x / LC) + (x & 1);
    }
    __host__ __device__ static constexpr int loc(int v) { return LC * ((v & 7) >> 1) + 2 * (v >> 3) + (v & 1); }
    // index of location x in the diagonal: the four lanes' runs two words apart
    __host__ __device__ static constexpr int diag(int x) { return x + 2 * (x / LC); }
};

constexpr float kCcScale = 2.81474976710656e14f;  // 2^48: energy per 1.0

template <int LC>
struct CcRow {
    float v[LC];
};

// The exact draw (eq5_draw_exact) for the four lanes of each row; q: the
// lane's place, v: its outcomes LC q + k. Returns the outcome.
template <int LC>
__device__ __noinline__ int cc_exact_draw(const CcRow<LC> d, int n, int q, float beta, unsigned long long draw) {
    float dmin = __int_as_float(0x7F800000);
#pragma unroll
    for (int k = 0; k < LC; ++k) dmin = fminf(dmin, d.v[k]);
    dmin = fminf(dmin, __shfl_xor_sync(kFull, dmin, 1));
    dmin = fminf(dmin, __shfl_xor_sync(kFull, dmin, 2));
    unsigned long long lsum = 0;
#pragma unroll 4
    for (int k = 0; k < LC; ++k)
        if (LC * q + k < n) lsum += eq5_weight_f((d.v[k] - dmin) * kCcScale, beta);
    unsigned long long incl = lsum;
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(kFull, incl, o, 4);
        if (q >= o) incl += y;
    }
    const unsigned long long total = __shfl_sync(kFull, incl, 3, 4);
    const unsigned long long tdraw = __umul64hi(draw, total);
    unsigned long long run = incl - lsum;
    int j = 0x7FFFFFFF;
    if (tdraw >= run && tdraw < incl) {
#pragma unroll 4
        for (int k = 0; k < LC; ++k)
            if (LC * q + k < n) {
                run += eq5_weight_f((d.v[k] - dmin) * kCcScale, beta);
                if (run > tdraw && j == 0x7FFFFFFF) j = LC * q + k;
            }
    }
    j = min(j, __shfl_xor_sync(kFull, j, 1));
    return min(j, __shfl_xor_sync(kFull, j, 2));
}

// G from the permutation, S and the swap energies (units of 2^-48) in `acc`.
// Begins after a CTA barrier, ends with the diagonal of S visible to the CTA.
template <class S>
__device__ __forceinline__ void cc_energies(unsigned char *sm, int n, float (&acc)[S::NT][4]) {
    constexpr int MT = S::MT, NT = S::NT, LC = S::LC, GS = S::GS;
    const int tid = threadIdx.x, lane = tid & 31, m = tid >> 5;
    const int g = lane >> 2, q = lane & 3;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm);
    {
        // thread: four columns of every eighth slot
        const int r0 = tid / LC, c4 = 4 * (tid % LC);
        const uint32_t py = *reinterpret_cast<const uint32_t *>(sm + S::oP + c4);
        const uint8_t *px = sm + S::oP + LC * (r0 >> 1) + (r0 & 1);
        unsigned char *out = sm + S::oG + r0 * GS + c4;
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const uint32_t row = base + S::oF + (uint32_t)px[2 * t] * S::FS;
            const int b0 = lds_u8(__byte_perm(py, row, 0x7650)), b1 = lds_u8(__byte_perm(py, row, 0x7651));
            const int b2 = lds_u8(__byte_perm(py, row, 0x7652)), b3 = lds_u8(__byte_perm(py, row, 0x7653));
            *reinterpret_cast<uint32_t *>(out + 8 * t * GS) =
                __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
        }
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[t][e] = 0.0f;
    const unsigned char *bD = sm + S::oD + g * GS + 4 * q, *bG = sm + S::oG + g * GS + 4 * q;
#pragma unroll 1
    for (int s = 0; s < MT; ++s) {
        uint32_t aD[4], aG[4];
        mm_frag<GS>(sm + S::oD, 16 * m, s, lane, aD);
        mm_frag<GS>(sm + S::oG, 16 * m, s, lane, aG);
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const uint32_t x = *reinterpret_cast<const uint32_t *>(bG + 8 * t * GS + 16 * s);
            const uint32_t y = *reinterpret_cast<const uint32_t *>(bD + 8 * t * GS + 16 * s);
            mma_f16(acc[t], aD, make_uint2(__byte_perm(x, 0, 0x4140), __byte_perm(x, 0, 0x4342)));
            if constexpr (!S::TR)
                mma_f16(acc[t], aG, make_uint2(__byte_perm(y, 0, 0x4140), __byte_perm(y, 0, 0x4342)));
        }
    }
    // diagonal: rows 16 m + g and 16 m + 8 + g are columns 2 q + e = g of tiles 2 m, 2 m + 1
    float *diag = reinterpret_cast<float *>(sm + S::oS);
    float d0 = 0.0f, d1 = 0.0f;
#pragma unroll
    for (int t = 0; t < MT; ++t)
        if (t == m) {
            d0 = g & 1 ? acc[2 * t][1] : acc[2 * t][0];
            d1 = g & 1 ? acc[2 * t + 1][3] : acc[2 * t + 1][2];
        }
    float *J = reinterpret_cast<float *>(sm + S::oJ) + (16 * m + g) * S::CS;
    if constexpr (S::TR) {
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            *reinterpret_cast<float2 *>(J + 8 * t + 2 * q) = make_float2(acc[t][0], acc[t][1]);
            *reinterpret_cast<float2 *>(J + 8 * S::CS + 8 * t + 2 * q) = make_float2(acc[t][2], acc[t][3]);
        }
        d0 += d0;
        d1 += d1;
    }
    const int x0 = LC * (g >> 1) + 4 * m + (g & 1), x1 = x0 + 2;  // locations of this lane's rows
    if (q == g >> 1) {
        // a location beyond n: energies of +infinity, weights of 0
        diag[S::diag(x0)] = x0 < n ? d0 : __int_as_float(0xFF800000);
        diag[S::diag(x1)] = x1 < n ? d1 : __int_as_float(0xFF800000);
    }
    __syncthreads();
    if constexpr (S::TR) {
        const float *Jt = reinterpret_cast<const float *>(sm + S::oJ) + 2 * q * S::CS + 16 * m + g;
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            acc[t][0] += Jt[8 * t * S::CS];
            acc[t][1] += Jt[(8 * t + 1) * S::CS];
            acc[t][2] += Jt[8 * t * S::CS + 8];
            acc[t][3] += Jt[(8 * t + 1) * S::CS + 8];
        }
    }
    const float s0 = diag[S::diag(x0)], s1 = diag[S::diag(x1)];
    const float *dq = diag + (LC + 2) * q;
    const unsigned char *rD = sm + S::oD + (16 * m + g) * GS + LC * q, *rG = rD + (S::oG - S::oD);
    // 4 D G of two columns: 4 (2^-25 + D) units less their 2^-23, times (2^23 + G) less 2^23
    auto pair = [](uint32_t d, uint32_t f, int at, float2 v) {
        const float2 a = make_float2(__int_as_float((int)__byte_perm(d, 0x34000000u, at ? 0x7542 : 0x7540)),
                                     __int_as_float((int)__byte_perm(d, 0x34000000u, at ? 0x7543 : 0x7541)));
        const float2 b = make_float2(__int_as_float((int)__byte_perm(f, 0x4B000000u, at ? 0x7542 : 0x7540)),
                                     __int_as_float((int)__byte_perm(f, 0x4B000000u, at ? 0x7543 : 0x7541)));
        return fma2(sub2(a, two(4.0f * kMmOne)), sub2(b, two(8388608.0f)), v);
    };
#pragma unroll
    for (int k = 0; k < MT; ++k) {
        const uint32_t dA = *reinterpret_cast<const uint32_t *>(rD + 4 * k);
        const uint32_t gA = *reinterpret_cast<const uint32_t *>(rG + 4 * k);
        const uint32_t dB = *reinterpret_cast<const uint32_t *>(rD + 8 * GS + 4 * k);
        const uint32_t gB = *reinterpret_cast<const uint32_t *>(rG + 8 * GS + 4 * k);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float(&c)[4] = acc[2 * k + h];
            const float2 sj = *reinterpret_cast<const float2 *>(dq + 4 * k + 2 * h);
            const float2 u0 = fma2(make_float2(c[0], c[1]), two(2.0f), sub2(two(-s0), sj));
            const float2 u1 = fma2(make_float2(c[2], c[3]), two(2.0f), sub2(two(-s1), sj));
            const float2 v0 = pair(dA, gA, h, u0), v1 = pair(dB, gB, h, u1);
            c[0] = v0.x;
            c[1] = v0.y;
            c[2] = v1.x;
            c[3] = v1.y;
        }
    }
}

// One part of a replica's iterations.
template <class S>
__device__ __forceinline__ void cc_run_replica(const SweepArgs &a, int r, int part, unsigned char *sm) {
    constexpr int NT = S::NT, NP = S::NP, LC = S::LC;
    const int tid = threadIdx.x, lane = tid & 31, m = tid >> 5;
    const int g = lane >> 2, q = lane & 3;
    const int n = a.n;
    const uint32_t grep = a.rep_base + (uint32_t)r;
    int32_t *gp = a.perm + (size_t)r * n;
    int32_t *gbp = a.best_perm + (size_t)r * n;
    uint8_t *pb = sm + S::oP;
    const float *diag = reinterpret_cast<const float *>(sm + S::oS);
    uint32_t *best = reinterpret_cast<uint32_t *>(sm + S::oB);  // two rounds' least priorities, by location
    uint8_t *taken = sm + S::oTk;
    volatile int *flag = reinterpret_cast<volatile int *>(sm + S::oX);
    const bool fresh = part == 0 && a.fresh;

    // ---- permutation
    if (m == 0) {
        if (fresh) {
            int32_t *wrd = reinterpret_cast<int32_t *>(sm + S::oB), *tmp = wrd + 128;
            fisher_yates<1>(a, grep, n, lane, wrd, tmp, 0);
            __syncwarp();
            for (int x = lane; x < NP; x += 32) pb[x] = (uint8_t)(x < n ? tmp[x] : x);
        } else {
            for (int x = lane; x < NP; x += 32) pb[x] = (uint8_t)(x < n ? __ldcg(gp + x) : x);
        }
    }
    __syncthreads();
    for (int x = tid; x < 128; x += S::T) best[x] = 0xFFFFFFFFu;
    float e[NT][4];
    cc_energies<S>(sm, n, e);
    // energy of the state, half the trace of S (the first warp)
    auto energy = [&]() {
        int v = 0;
        for (int x = lane; x < n; x += 32) v += (int)(diag[S::diag(x)] * kCcScale);
        return __reduce_add_sync(kFull, v) >> 1;
    };
    int E = 0, bestE = 0, bsweep = -1;  // kept by the first warp
    long long accepted = 0;
    bool reached = false;
    if (m == 0) {
        const int now = energy();
        if (fresh) {
            E = bestE = now;
            for (int x = lane; x < n; x += 32) gbp[x] = pb[x];
            if (lane == 0) note_target(a, bestE, -1, reached);
        } else {
            E = (int)__ldcg(a.energy + r);
            bestE = (int)__ldcg(a.best_energy + r);
            bsweep = __ldcg(a.best_sweep + r);
            accepted = __ldcg(a.accepted + r);
            if (E != now && lane == 0) atomicOr(a.status, 1);
        }
    }
    const int s_begin = part_begin(a, part);
    const int s_end = part >= a.segments - 1 ? a.sweep_end : part_begin(a, part + 1);
    const int row0 = LC * (g >> 1) + 4 * m + (g & 1);  // location of row half 0; half 1: + 2
    int par = 0;
    for (int s = s_begin; s < s_end; ++s) {
        if (a.stop) {
            __syncthreads();
            if (tid == 0) *flag = *reinterpret_cast<volatile int *>(a.done);
            __syncthreads();
            if (*flag) break;
        }
        const float beta = a.beta[s];
        if (!sweep_moves(beta)) continue;
        // (never 0, so that an infinite energy always has weight 0)
        const float kb = fminf(-beta * kLog2e * kCcScale, -1e-37f);
        // Philox(inst, replica, iteration, location): lanes 0, 2 of a row pair have half 0's, 1, 3 half 1's
        const uint4 rw = philox4x32_10(a.inst, grep, (uint32_t)s, (uint32_t)(row0 + 2 * (q & 1)), a.key0, a.key1);
        // ---- proposals: one row of the quad's two at a time; lane q keeps row q's (q < 2)
        int pj = -1, pd = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = row0 + 2 * h;
            // prefix sums of four outcomes each (the draw's at most 17
            // roundings, 1.0e-6 of the total, leave 1.5e-5 its slack)
            float pre[S::MT], lsum = 0.0f;
#pragma unroll
            for (int k = 0; k < S::MT; ++k) {
                const float2 x = mul2(make_float2(e[2 * k][2 * h], e[2 * k][2 * h + 1]), two(kb));
                const float2 y = mul2(make_float2(e[2 * k + 1][2 * h], e[2 * k + 1][2 * h + 1]), two(kb));
                lsum += (ex2_approx(x.x) + ex2_approx(x.y)) + (ex2_approx(y.x) + ex2_approx(y.y));
                pre[k] = lsum;
            }
            float incl = lsum;
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                const float y = __shfl_up_sync(kFull, incl, o, 4);
                if (q >= o) incl += y;
            }
            const float total = __shfl_sync(kFull, incl, 3, 4);
            const uint32_t dhi = __shfl_sync(kFull, rw.y, h, 4);
            const float tt = __uint2float_rn(dhi >> 8) * 5.9604644775390625e-08f * total;
            const float mg = total < kDrawLimit ? kDrawMargin * total : __int_as_float(0x7FC00000);
            const float base = (incl - lsum) - tt;
            // the four outcomes around the draw, then the one: boundaries lo < 0 < hi
            float lo = base, v[4] = {e[0][2 * h], e[0][2 * h + 1], e[1][2 * h], e[1][2 * h + 1]};
            int kk = 0;
#pragma unroll
            for (int k = 1; k < S::MT; ++k) {
                const float z = pre[k - 1] + base;
                if (z < 0.0f) {
                    lo = z;
                    kk = 4 * k;
                    v[0] = e[2 * k][2 * h];
                    v[1] = e[2 * k][2 * h + 1];
                    v[2] = e[2 * k + 1][2 * h];
                    v[3] = e[2 * k + 1][2 * h + 1];
                }
            }
            float hi = lo + ex2_approx(v[0] * kb), dsel = v[0];
            const int k4 = kk;
#pragma unroll
            for (int k = 1; k < 4; ++k) {
                const float z = hi + ex2_approx(v[k] * kb);
                if (hi < 0.0f) {
                    lo = hi;
                    hi = z;
                    kk = k4 + k;
                    dsel = v[k];
                }
            }
            // the lane whose interval certainly holds the draw (eq5_draw_core)
            const unsigned ball = __ballot_sync(kFull, fminf(-lo, hi) > mg);
            const unsigned mine = (ball >> (lane & 28)) & 15u;
            int src = __ffs(mine) - 1;
            int js = __shfl_sync(kFull, LC * q + kk, src, 4);
            float d = __shfl_sync(kFull, dsel, src, 4);
            if (__any_sync(kFull, mine == 0 && i < n)) {
                CcRow<LC> row;
#pragma unroll
                for (int k = 0; k < LC; ++k) row.v[k] = e[k / 2][2 * h + (k & 1)];
                const uint32_t dlo = __shfl_sync(kFull, rw.x, h, 4);
                const int jx = cc_exact_draw<LC>(row, n, q, beta, ((unsigned long long)dhi << 32) | dlo);
                float dx = 0.0f;
#pragma unroll
                for (int k = 0; k < LC; ++k)
                    if (LC * q + k == jx) dx = row.v[k];
                dx = __shfl_sync(kFull, dx, (jx / LC) & 3, 4);
                if (mine == 0) {
                    js = jx;
                    d = dx;
                }
            }
            if (q == h && i < n) {
                pj = js == i ? -1 : js;
                pd = (int)(d * kCcScale);
            }
        }
        // ---- matching: lanes q < 2 of a quad carry location i's proposal
        // priority: |dE| < 2^23 (4 N 127^2 + 4 127^2 at N = 128), then the location
        const int i = row0 + 2 * (q & 1);
        const uint32_t key = ((uint32_t)(pd + 8388608) << 7) | (uint32_t)i;
        if (tid < 32) reinterpret_cast<uint32_t *>(taken)[tid] = 0u;
        bool won = false;
        __syncthreads();
        for (;;) {
            uint32_t *now = best + 128 * par;
            const bool left = pj >= 0 && !won && !taken[i] && !taken[pj];
            if (left) {
                atomicMin(now + i, key);
                atomicMin(now + pj, key);
            }
            // the other round's entries for the next one
            for (int x = tid; x < 128; x += S::T) best[128 * (par ^ 1) + x] = 0xFFFFFFFFu;
            par ^= 1;
            if (!__syncthreads_or(left)) break;
            if (left && now[i] == key && now[pj] == key) {
                won = true;
                taken[i] = 1;
                taken[pj] = 1;
            }
            __syncthreads();
        }
        if (won) {
            const uint8_t x = pb[i];
            pb[i] = pb[pj];
            pb[pj] = x;
        }
        const int swaps = __syncthreads_count(won);
        if (swaps == 0) continue;
        cc_energies<S>(sm, n, e);
        if (m == 0) {
            accepted += swaps;
            E = energy();
            if (E < bestE) {
                bestE = E;
                bsweep = s;
                for (int x = lane; x < n; x += 32) gbp[x] = pb[x];
                if (lane == 0) note_target(a, bestE, s, reached);
            }
        }
    }

    // ---- audit (the last unit of a call; a resumed unit begins with the same
    // check): Eq. 1 of the final permutation, from D and F, equals the energy
    if (m == 0) {
        if (part >= a.segments - 1) {
            int eq1 = 0;  // (n^2 127^2 < 2^31)
            for (int x = lane; x < n; x += 32)
                for (int y = 0; y < n; ++y)
                    eq1 += (int)sm[S::oD + S::slot(x) * S::GS + y] * (int)sm[S::oF + pb[x] * S::FS + pb[y]];
            eq1 = __reduce_add_sync(kFull, eq1);
            if (lane == 0 && eq1 != E) atomicOr(a.status, 1);
        }
        for (int x = lane; x < n; x += 32) gp[x] = pb[x];
        if (lane == 0) {
            a.energy[r] = E;
            a.best_energy[r] = bestE;
            a.best_sweep[r] = bsweep;
            a.accepted[r] = accepted;
        }
    }
}

// Persistent: CTAs take (replica, part) units in order, part k of every
// replica before part k + 1; see dot_kernel for why the wait for the part
// before ends.
template <class S>
__global__ void __launch_bounds__(S::T, S::CTAS) concurrent_kernel(const SweepArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    for (int w = threadIdx.x; w < S::oP / 4; w += S::T) reinterpret_cast<uint32_t *>(smem)[w] = 0u;
    __syncthreads();
    for (int idx = threadIdx.x; idx < a.n * a.n; idx += S::T) {
        const int x = idx / a.n, y = idx - x * a.n;
        smem[S::oD + S::slot(x) * S::GS + y] = (uint8_t)a.D[idx];
        smem[S::oF + x * S::FS + y] = (uint8_t)a.F[idx];
    }
    volatile int *x = reinterpret_cast<volatile int *>(smem + S::oX);
    const int parts = a.segments > 1 ? a.segments : 1;
    const long long units = (long long)a.replicas * parts;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) {
            const int item = atomicAdd(a.queue, 1);
            int go = item < units ? 1 : 0;
            const int part = go ? item / a.replicas : 0, r = item - part * a.replicas;
            if (go && part > 0) go = wait_part(a, r, part);
            x[1] = r;
            x[2] = part;
            x[3] = go;
        }
        __syncthreads();
        const int r = x[1], part = x[2], go = x[3];
        if (!go) break;
        cc_run_replica<S>(a, r, part, smem);
        if (parts > 1) {
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) publish_part(a, r, part + 1);
        }
    }
}

template <int MT>
static int cc_one(const SweepArgs *a, int grid, cudaStream_t st, CcInfo *info) {
    using S = CcShape<MT>;
    const cudaError_t e =
        cudaFuncSetAttribute(concurrent_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::bytes);
    if (e != cudaSuccess) return (int)e;
    if (info) {
        info->threads = S::T;
        info->smem = S::bytes;
        return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(&info->blocks_per_sm, concurrent_kernel<S>, S::T,
                                                                  S::bytes);
    }
    concurrent_kernel<S><<<grid, S::T, S::bytes, st>>>(*a);
    return (int)cudaGetLastError();
}

static int cc_dispatch(int n, const SweepArgs *a, int grid, cudaStream_t st, CcInfo *info) {
    switch (n < 1 ? 0 : (n + 15) / 16) {
    case 1: return cc_one<1>(a, grid, st, info);
    case 2: return cc_one<2>(a, grid, st, info);
    case 3: return cc_one<3>(a, grid, st, info);
    case 4: return cc_one<4>(a, grid, st, info);
    case 5: return cc_one<5>(a, grid, st, info);
    case 6: return cc_one<6>(a, grid, st, info);
    case 7: return cc_one<7>(a, grid, st, info);
    case 8: return cc_one<8>(a, grid, st, info);
    default: return (int)cudaErrorInvalidValue;
    }
}

int concurrent_query(int n, CcInfo *info) { return cc_dispatch(n, nullptr, 0, nullptr, info); }

int concurrent_launch(const SweepArgs &a, int grid, cudaStream_t st) { return cc_dispatch(a.n, &a, grid, st, nullptr); }

}  // namespace pdit
