// Annealed p-dit sweep for symmetric instances of at most 32 locations: one
// warp per replica, lane m owns location m.
//
// A replica of this size is one dependent chain (products or gathers, weights,
// prefix sums, draw, swap), and few replicas share an SM, so its latency is
// the time. The influence table of Eq. 2 in the one-term form, I[m][c] =
// sum_y D[m][y] F[c][p(y)], is kept twice: lane m holds row m in registers and
// its copy in shared memory. An update gathers its two entries from shared
// memory (a row read at distinct columns and a column, no loop); an accepted
// swap adds its rank-1 change to the registers and stores them, so the copy is
// written but never read back to be changed. The energies of the next location
// are formed while the present draw runs and formed again only after a swap.
#include "pdit_sweep.cuh"

namespace pdit {

template <int NP>
__device__ __forceinline__ void run_small_replica(const SweepArgs &a, int r, int part, int lane, const int32_t *sD,
                                                  const int32_t *sF, int32_t *sT, int32_t *sv, int32_t *sp) {
    constexpr int DS = NP + 1, S = NP + 4;  // row strides of D (lanes down a column) and of the table
    const int n = a.n;
    const bool act = lane < n;
    const int row = act ? lane : 0;
    const uint32_t grep = a.rep_base + (uint32_t)r;
    int32_t *gp = a.perm + (size_t)r * n;
    int32_t *gbp = a.best_perm + (size_t)r * n;
    const bool fresh = part == 0 && a.fresh;

    // ---- permutation
    if (fresh) {
        fisher_yates<1>(a, grep, n, lane, sv, sp, 0);
    } else if (act) {
        sp[lane] = __ldcg(gp + lane);
    }
    __syncwarp();
    int p = act ? sp[lane] : 0;

    // ---- table rows, p-diagonal h[m] = I[m][p(m)], energy E = sum_m h[m]
    int T[NP];
#pragma unroll
    for (int c = 0; c < NP; ++c) T[c] = 0;
    for (int y = 0; y < n; ++y) {
        const int dm = act ? sD[row * DS + y] : 0;
        const int4 *f4 = reinterpret_cast<const int4 *>(sF + sp[y] * NP);  // F symmetric
#pragma unroll
        for (int q = 0; q < NP / 4; ++q) {
            const int4 f = f4[q];
            T[4 * q] += dm * f.x;
            T[4 * q + 1] += dm * f.y;
            T[4 * q + 2] += dm * f.z;
            T[4 * q + 3] += dm * f.w;
        }
    }
    int32_t *mine = sT + row * S;
    auto store = [&]() {
        if (act) {
#pragma unroll
            for (int q = 0; q < NP / 4; ++q)
                reinterpret_cast<int4 *>(mine)[q] = make_int4(T[4 * q], T[4 * q + 1], T[4 * q + 2], T[4 * q + 3]);
        }
    };
    store();
    __syncwarp();
    int h = act ? mine[p] : 0;
    const long long esum = warp_sum((long long)h);
    long long E, bestE, acc_moves;
    int bsweep;
    bool reached = false;
    if (fresh) {
        E = bestE = esum;
        bsweep = -1;
        acc_moves = 0;
        if (act) gbp[lane] = p;
        if (lane == 0) note_target(a, bestE, -1, reached);
    } else {
        E = __ldcg(a.energy + r);
        bestE = __ldcg(a.best_energy + r);
        bsweep = __ldcg(a.best_sweep + r);
        acc_moves = __ldcg(a.accepted + r);
        if (E != esum && lane == 0) atomicOr(a.status, 1);
    }
    const int s_begin = part_begin(a, part);
    const int s_end = part >= a.segments - 1 ? a.sweep_end : part_begin(a, part + 1);
    const float beta_fixed = a.sweep_end <= a.sweep_begin ? 0.0f
                           : a.mode == 1 ? a.beta[a.rung[r]] : a.mode == 2 ? a.beta[r] : 0.0f;
    const int djj = sD[row * DS + row];

    // Eq. 3 for location i against this lane's (one-term units)
    auto energy = [&](int i) {
        const int fa = __shfl_sync(kFull, p, i);
        const int rv = sT[i * S + p], hi = sT[i * S + fa], cv = mine[fa];
        const int dij = sD[i * DS + row], fab = sF[fa * NP + p];
        int d = 2 * ((rv - hi) + (cv - h));
        if (a.zero_diag)
            d += 4 * dij * fab;
        else
            d += (sD[i * DS + i] + djj - 2 * dij) * (sF[fa * NP + fa] + sF[p * NP + p] - 2 * fab);
        return lane == i ? 0 : d;
    };
    int d = energy(0);
    for (int s = s_begin; s < s_end; ++s) {
        if (a.stop) {
            int f = 0;
            if (lane == 0) f = *reinterpret_cast<volatile int *>(a.done);
            if (__shfl_sync(kFull, f, 0)) break;
        }
        const float beta = (a.mode == 1 || a.mode == 2) ? beta_fixed : a.beta[s];
        // Philox(inst, replica, sweep, location) of every location
        const uint4 rw = philox4x32_10(a.inst, grep, (uint32_t)s, (uint32_t)lane, a.key0, a.key1);
        for (int i = 0; i < n; ++i) {
            const int nxt = i + 1 < n ? i + 1 : 0;
            int dn = energy(nxt);
            const int dc[1] = {d};
            const int3 sel = eq5_draw_regs<1, 1>(
                dc, [&](int) { return p; }, n, lane, beta, __shfl_sync(kFull, rw.y, i),
                [&]() { return __shfl_sync(kFull, rw.x, i); }, draw_tag(i, s), 0, nullptr);
            const int js = sel.x;
            if (js != i) {
                // ---- swap i <-> js (facilities fa = p(i), fb = p(js)): I += u (x) v
                const int fb = sel.z, fa = __shfl_sync(kFull, p, i);
                const int u = act ? sD[i * DS + row] - sD[js * DS + row] : 0;
                if (lane < NP) sv[lane] = sF[fb * NP + lane] - sF[fa * NP + lane];
                if (lane == i) p = fb;
                if (lane == js) p = fa;
                __syncwarp();
#pragma unroll
                for (int q = 0; q < NP / 4; ++q) {
                    const int4 v = reinterpret_cast<const int4 *>(sv)[q];
                    T[4 * q] += u * v.x;
                    T[4 * q + 1] += u * v.y;
                    T[4 * q + 2] += u * v.z;
                    T[4 * q + 3] += u * v.w;
                }
                store();
                E += sel.y;
                acc_moves += 1;
                if (E < bestE) {
                    bestE = E;
                    bsweep = s;
                    if (act) gbp[lane] = p;
                    if (lane == 0) note_target(a, bestE, s, reached);
                }
                __syncwarp();
                h = act ? mine[p] : 0;
                dn = energy(nxt);
            }
            d = dn;
        }
    }

    // ---- audit (the last unit of a call): the energy of the tracked table
    // against Eq. 1 of the final permutation, from D and F
    if (part >= a.segments - 1) {
        __syncwarp();
        if (act) sp[lane] = p;
        __syncwarp();
        long long eq1 = 0;
        if (act)
            for (int y = 0; y < n; ++y) eq1 += (long long)sD[row * DS + y] * sF[p * NP + sp[y]];
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

// Shared memory (int32): D (n x NP+1), F (n x NP, 16-byte rows), then per warp
// the table copy (n x NP+4), a column factor and the permutation (NP each).
template <int NP>
__global__ void __launch_bounds__(512) small_kernel(const SweepArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int n = a.n;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t *sF = reinterpret_cast<int32_t *>(smem);
    int32_t *sW = sF + n * NP + w * (n * (NP + 4) + 2 * NP);
    int32_t *sD = sF + n * NP + (blockDim.x >> 5) * (n * (NP + 4) + 2 * NP);
    for (int idx = threadIdx.x; idx < n * NP; idx += blockDim.x) {
        const int m = idx / NP, c = idx - m * NP;
        sF[idx] = c < n ? a.F[m * n + c] : 0;
        sD[m * (NP + 1) + c] = c < n ? a.D[m * n + c] : 0;
    }
    __syncthreads();
    int32_t *sv = sW + n * (NP + 4), *sp = sv + NP;
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
        run_small_replica<NP>(a, r, part, lane, sD, sF, sW, sv, sp);
        if (K > 1) {
            __threadfence();
            __syncwarp();
            if (lane == 0) publish_part(a, r, part + 1);
        }
        __syncwarp();
    }
}

template <int NP>
static int small_one(const SweepArgs *a, int n, int grid, int warps, cudaStream_t st, SmallInfo *info) {
    auto fn = small_kernel<NP>;
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

static int small_dispatch(const SweepArgs *a, int n, int grid, int warps, cudaStream_t st, SmallInfo *info) {
    if (n <= 16) return small_one<16>(a, n, grid, warps, st, info);
    if (n <= 24) return small_one<24>(a, n, grid, warps, st, info);
    if (n <= 32) return small_one<32>(a, n, grid, warps, st, info);
    return (int)cudaErrorInvalidValue;
}

int small_query(int n, int warps, SmallInfo *info) { return small_dispatch(nullptr, n, 0, warps, nullptr, info); }

int small_launch(const SweepArgs &a, int grid, int warps, cudaStream_t st) {
    return small_dispatch(&a, a.n, grid, warps, st, nullptr);
}

}  // namespace pdit
