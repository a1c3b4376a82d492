// Annealed p-dit sweep for symmetric instances of at most 32 locations: one
// warp per replica, lane m owns location m.
//
// A replica of this size is one dependent chain (gathers, weights, prefix
// sums, draw, swap), and few replicas share an SM, so its latency is the
// time. The influence table of Eq. 2 in the one-term form, I[m][c] = sum_y
// D[m][y] F[c][p(y)], is kept twice: lane m holds row m in registers and its
// copy in shared memory, where an update gathers its two entries (a row read
// at distinct columns and a column, no loop). A swap's rank-1 change of the
// table is added during the next update's draw, in the shadow of its shuffles,
// and the energies of the next location, formed during the draw, are brought
// to the state after a swap i <-> s (facilities a, b) by the same change: with
// u_m = D_im - D_sm and v(c) = F_bc - F_ac,
//   I'[j][p(w)] = I[j][p(w)] + u_j v(p(w)),  I'[w][c] = I[w][c] + u_w v(c),
// entries at i and s trading places; where w = s, the column is that of a,
// from the present location's gathers.
//
// V is binary32 where every entry and energy is an integer below 2^24
// (8 (n + 2) max|D| max|F| < 2^24: exact, and two products per instruction),
// else int32.
//
// Bound: the latency of the chain, 560 clocks an update at N = 12 (64
// replicas, 0.42 of the updates swap) and 850 at N = 30 (0.84 swap), against
// 1070 and 1700 with the dot-product kernel; one warp alone issues about one
// instruction in three clocks. N = 30, 1024 replicas, 5000 sweeps: 61.4 ms (125
// ms with the dot-product kernel, 72 ms with the table changed in the swap
// itself). The row's copy is stored in every update, changed or not.
#include <type_traits>

#include "pdit_sweep.cuh"

namespace pdit {

__device__ __forceinline__ void add_scaled4(float (&t)[4], float u, const float4 v) {
    asm("{ .reg .b64 a, b, c; mov.b64 a, {%0, %1}; mov.b64 b, {%2, %2}; mov.b64 c, {%3, %4}; fma.rn.f32x2 a, b, c, a; "
        "mov.b64 {%0, %1}, a; }"
        : "+f"(t[0]), "+f"(t[1])
        : "f"(u), "f"(v.x), "f"(v.y));
    asm("{ .reg .b64 a, b, c; mov.b64 a, {%0, %1}; mov.b64 b, {%2, %2}; mov.b64 c, {%3, %4}; fma.rn.f32x2 a, b, c, a; "
        "mov.b64 {%0, %1}, a; }"
        : "+f"(t[2]), "+f"(t[3])
        : "f"(u), "f"(v.z), "f"(v.w));
}
__device__ __forceinline__ void add_scaled4(int (&t)[4], int u, const int4 v) {
    t[0] += u * v.x;
    t[1] += u * v.y;
    t[2] += u * v.z;
    t[3] += u * v.w;
}
template <typename V>
struct Vec4;
template <>
struct Vec4<int> {
    using type = int4;
    __device__ static int4 of(const int (&t)[4]) { return make_int4(t[0], t[1], t[2], t[3]); }
};
template <>
struct Vec4<float> {
    using type = float4;
    __device__ static float4 of(const float (&t)[4]) { return make_float4(t[0], t[1], t[2], t[3]); }
};

template <int NP, typename V>
__device__ __forceinline__ void run_small_replica(const SweepArgs &a, int r, int part, int lane, const V *sD,
                                                  const V *sF, V *sT, V *sv, int32_t *sp) {
    constexpr int DS = NP + 1, S = NP + 4;  // row strides of D (lanes down a column) and of the table
    using V4 = typename Vec4<V>::type;
    const int n = a.n;
    const bool act = lane < n;
    const int row = act ? lane : 0;
    const uint32_t grep = a.rep_base + (uint32_t)r;
    int32_t *gp = a.perm + (size_t)r * n;
    int32_t *gbp = a.best_perm + (size_t)r * n;
    const bool fresh = part == 0 && a.fresh;

    // ---- permutation
    if (fresh) {
        fisher_yates<1>(a, grep, n, lane, reinterpret_cast<int32_t *>(sv), sp, 0);
    } else if (act) {
        sp[lane] = __ldcg(gp + lane);
    }
    __syncwarp();
    int p = act ? sp[lane] : 0;

    // ---- table rows, p-diagonal h[m] = I[m][p(m)], energy E = sum_m h[m]
    V T[NP / 4][4];
#pragma unroll
    for (int c = 0; c < NP; ++c) T[c / 4][c % 4] = 0;
    for (int y = 0; y < n; ++y) {
        const V dm = act ? sD[row * DS + y] : (V)0;
        const V4 *f4 = reinterpret_cast<const V4 *>(sF + sp[y] * NP);  // F symmetric
#pragma unroll
        for (int q = 0; q < NP / 4; ++q) add_scaled4(T[q], dm, f4[q]);
    }
    V *mine = sT + row * S;
    auto store = [&]() {
        if (act) {
#pragma unroll
            for (int q = 0; q < NP / 4; ++q) reinterpret_cast<V4 *>(mine)[q] = Vec4<V>::of(T[q]);
        }
    };
    store();
    __syncwarp();
    V h = act ? mine[p] : (V)0;
    const long long esum = warp_sum((long long)h);
    // (binary32 instances: |E| <= n^2 max|D| max|F| < 2^31)
    using Acc = typename std::conditional<std::is_same<V, float>::value, int, long long>::type;
    Acc E, bestE;
    long long acc_moves;
    int bsweep;
    bool reached = false;
    if (fresh) {
        E = bestE = (Acc)esum;
        bsweep = -1;
        acc_moves = 0;
        if (act) gbp[lane] = p;
        if (lane == 0) note_target(a, bestE, -1, reached);
    } else {
        E = (Acc)__ldcg(a.energy + r);
        bestE = (Acc)__ldcg(a.best_energy + r);
        bsweep = __ldcg(a.best_sweep + r);
        acc_moves = __ldcg(a.accepted + r);
        if (E != esum && lane == 0) atomicOr(a.status, 1);
    }
    const int s_begin = part_begin(a, part);
    const int s_end = part >= a.segments - 1 ? a.sweep_end : part_begin(a, part + 1);
    const float beta_fixed = a.sweep_end <= a.sweep_begin ? 0.0f
                           : a.mode == 1 ? a.beta[a.rung[r]] : a.mode == 2 ? a.beta[r] : 0.0f;
    const V djj = sD[row * DS + row];

    // Eq. 3 for location i against this lane's (one-term units), and what it
    // was formed from: p(i), F[p(i)][p(j)], I[i][p(j)], I[j][p(i)], h_i, D_ij
    struct Energy {
        V d, fab, rv, cv, hi, dij;
        int fa;
    };
    auto finish = [&](Energy &e, int i) {
        V d = 2 * ((e.rv - e.hi) + (e.cv - h));
        if (a.zero_diag)
            d += 4 * (e.dij * e.fab);
        else
            d += (sD[i * DS + i] + djj - 2 * e.dij) * (sF[e.fa * NP + e.fa] + sF[p * NP + p] - 2 * e.fab);
        e.d = lane == i ? (V)0 : d;
    };
    auto energy = [&](int i, int fa) {
        Energy e;
        e.fa = fa;
        e.rv = sT[i * S + p];
        e.cv = mine[e.fa];
        e.fab = sF[e.fa * NP + p];
        e.hi = sT[i * S + e.fa];
        e.dij = sD[i * DS + row];
        finish(e, i);
        return e;
    };
    Energy e = energy(0, __shfl_sync(kFull, p, 0));
    V pu = 0;  // the last swap's u, until the table has it (its v is in sv)
    if (lane < NP) sv[lane] = 0;
    __syncwarp();
    for (int s = s_begin; s < s_end; ++s) {
        if (a.stop) {
            int f = 0;
            if (lane == 0) f = *reinterpret_cast<volatile int *>(a.done);
            if (__shfl_sync(kFull, f, 0)) break;
        }
        const float beta = (a.mode == 1 || a.mode == 2) ? beta_fixed : a.beta[s];
        const float kb = -beta * kLog2e;
        // Philox(inst, replica, sweep, location) of every location
        const uint4 rw = philox4x32_10(a.inst, grep, (uint32_t)s, (uint32_t)lane, a.key0, a.key1);
        const float ul = __uint2float_rn(rw.y >> 8) * 5.9604644775390625e-08f;
        int moves = 0;
        for (int i = 0; i < n; ++i) {
            __syncwarp();  // the reads of the table for this update's energies are done
            const int nxt = i + 1 < n ? i + 1 : 0;
            const float u01 = __shfl_sync(kFull, ul, i);
            const int fnxt = __shfl_sync(kFull, p, nxt);
            // ---- the binary32 draw of eq5_draw_core, one outcome a lane; the
            // total comes from a butterfly beside the prefix sums, and the
            // pending change of the table goes in between
            const float w = act ? ex2_approx((float)e.d * kb) : 0.0f;
            float incl = w, total = w;
#pragma unroll
            for (int q = 0; q < NP / 4; ++q) add_scaled4(T[q], pu, reinterpret_cast<const V4 *>(sv)[q]);
            store();
#pragma unroll
            for (int o = 1; o < (NP > 16 ? 32 : 16); o <<= 1) {
                const float y = __shfl_up_sync(kFull, incl, o), z = __shfl_xor_sync(kFull, total, o);
                if (lane >= o) incl += y;
                total += z;
            }
            __syncwarp();
            Energy en = energy(nxt, fnxt);
            const float tt = u01 * total;
            const float mg = total < kDrawLimit ? kDrawMargin * total : __int_as_float(0x7FC00000);
            const unsigned own = __ballot_sync(kFull, act && tt - mg >= incl - w && tt + mg < incl);
            int js = __ffs(own) - 1;
            if (!own) {
                const int dc[1] = {(int)e.d};
                const unsigned long long draw = ((unsigned long long)__shfl_sync(kFull, rw.y, i) << 32) |
                                                (unsigned long long)__shfl_sync(kFull, rw.x, i);
                js = eq5_draw_exact<1, 1>(dc, [&](int) { return p; }, n, lane, beta, draw, 0, 0, nullptr).x;
                if (!sweep_moves(beta)) js = i;
            }
            pu = 0;
            if (js != i) {
                // ---- swap i <-> js (facilities fa = p(i), fb = p(js))
                const int fa = e.fa, fb = __shfl_sync(kFull, p, js);
                const V rs = __shfl_sync(kFull, e.rv, js), fab = __shfl_sync(kFull, e.fab, js);
                E += (int)__shfl_sync(kFull, e.d, js);
                const V u = act ? e.dij - sD[js * DS + row] : (V)0;
                if (lane == i) p = fb;
                if (lane == js) p = fa;
                const V fap = sF[fa * NP + p], v = sF[fb * NP + p] - fap;  // v(p'(j))
                // h[m] += u_m v(p(m)); the two moved entries from I[i][fb], I[js][fa]
                h = (lane == i ? rs : lane == js ? e.cv : h) + u * v;
                // the next location after the swap
                const int tau = lane == i ? js : lane == js ? i : lane;
                const V uw = __shfl_sync(kFull, u, nxt);
                const V rt = __shfl_sync(kFull, en.rv, tau), ft = __shfl_sync(kFull, en.fab, tau);
                const bool isw = nxt == js;
                en.fa = isw ? fa : nxt == i ? fb : en.fa;
                const V vw = sF[fb * NP + en.fa] - sF[fa * NP + en.fa];
                en.rv = rt + uw * v;
                en.cv = (isw ? e.cv : en.cv) + u * vw;
                en.fab = isw ? fap : ft;
                en.hi = en.hi + uw * vw;
                if (isw) en.hi = __shfl_sync(kFull, h, nxt);
                finish(en, nxt);
                pu = u;
                __syncwarp();  // the table's reads of sv are done
                if (lane < NP) sv[lane] = sF[fb * NP + lane] - sF[fa * NP + lane];
                moves += 1;
                if (E < bestE) {
                    bestE = E;
                    bsweep = s;
                    if (act) gbp[lane] = p;
                    if (lane == 0) note_target(a, bestE, s, reached);
                }
                __syncwarp();
            }
            e = en;
        }
        acc_moves += moves;
    }

    // ---- audit (the last unit of a call): the energy of the tracked table
    // against Eq. 1 of the final permutation, from D and F
    if (part >= a.segments - 1) {
        __syncwarp();
        if (act) sp[lane] = p;
        __syncwarp();
        long long eq1 = 0;
        if (act)
            for (int y = 0; y < n; ++y) eq1 += (long long)sD[row * DS + y] * (long long)sF[p * NP + sp[y]];
        eq1 = warp_sum(eq1);
        if (lane == 0 && eq1 != E) atomicOr(a.status, 1);
    }
    if (act) gp[lane] = p;
    if (lane == 0) {
        a.energy[r] = E;
        a.best_energy[r] = bestE;
        a.best_sweep[r] = bsweep;
        a.accepted[r] = acc_moves;
    }
}

// Shared memory (32-bit words): F (n x NP), then per warp the table copy
// (n x NP+4), a column factor and the permutation (NP each), then D (n x NP+1).
template <int NP, typename V>
__global__ void __launch_bounds__(512) small_kernel(const SweepArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int n = a.n;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    V *sF = reinterpret_cast<V *>(smem);
    V *sW = sF + n * NP + w * (n * (NP + 4) + 2 * NP);
    V *sD = sF + n * NP + (blockDim.x >> 5) * (n * (NP + 4) + 2 * NP);
    for (int idx = threadIdx.x; idx < n * NP; idx += blockDim.x) {
        const int m = idx / NP, c = idx - m * NP;
        sF[idx] = c < n ? (V)a.F[m * n + c] : (V)0;
        sD[m * (NP + 1) + c] = c < n ? (V)a.D[m * n + c] : (V)0;
    }
    __syncthreads();
    V *sv = sW + n * (NP + 4);
    int32_t *sp = reinterpret_cast<int32_t *>(sv + NP);
    // work units in order, as in dot_kernel: part k of every replica, then
    // part k + 1, each after the replica's previous part
    const int K = a.segments > 1 ? a.segments : 1;
    const long long units = (long long)a.replicas * K;
    for (;;) {
        int item = 0, go = 0;
        if (lane == 0) {
            item = atomicAdd(a.queue, 1);
            go = item < units ? 1 : 0;
            if (go && K > 1 && item >= a.replicas) go = wait_part(a, item % a.replicas, item / a.replicas);
        }
        item = __shfl_sync(kFull, item, 0);
        if (!__shfl_sync(kFull, go, 0)) break;
        const int part = item / a.replicas, r = item - part * a.replicas;
        run_small_replica<NP, V>(a, r, part, lane, sD, sF, sW, sv, sp);
        if (K > 1) {
            __threadfence();
            __syncwarp();
            if (lane == 0) publish_part(a, r, part + 1);
        }
        __syncwarp();
    }
}

template <int NP, typename V>
static int small_one(const SweepArgs *a, int n, int grid, int warps, cudaStream_t st, SmallInfo *info) {
    auto fn = small_kernel<NP, V>;
    if (warps < 1 || 32 * warps > 512) return (int)cudaErrorInvalidValue;
    const size_t smem = 4 * ((size_t)n * NP + (size_t)n * (NP + 1) + (size_t)warps * (n * (NP + 4) + 2 * NP));
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    if (info) {
        info->smem = smem;
        return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(&info->blocks_per_sm, fn, 32 * warps, smem);
    }
    fn<<<grid, 32 * warps, smem, st>>>(*a);
    return (int)cudaGetLastError();
}

template <typename V>
static int small_dispatch(const SweepArgs *a, int n, int grid, int warps, cudaStream_t st, SmallInfo *info) {
    if (n <= 16) return small_one<16, V>(a, n, grid, warps, st, info);
    if (n <= 24) return small_one<24, V>(a, n, grid, warps, st, info);
    if (n <= 32) return small_one<32, V>(a, n, grid, warps, st, info);
    return (int)cudaErrorInvalidValue;
}

int small_query(int n, bool f32, int warps, SmallInfo *info) {
    return f32 ? small_dispatch<float>(nullptr, n, 0, warps, nullptr, info)
               : small_dispatch<int>(nullptr, n, 0, warps, nullptr, info);
}

int small_launch(const SweepArgs &a, bool f32, int grid, int warps, cudaStream_t st) {
    return f32 ? small_dispatch<float>(&a, a.n, grid, warps, st, nullptr)
               : small_dispatch<int>(&a, a.n, grid, warps, st, nullptr);
}

}  // namespace pdit
