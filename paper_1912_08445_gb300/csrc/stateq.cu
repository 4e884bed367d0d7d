// K4 statistical equilibrium (eq. 'ourALI'), validity check (Sec. 6.1), convergence
// measure, LTE start and Ng acceleration (Sec. 3.4).
#include <cmath>
#include <cstring>
#include <algorithm>
#include "common.cuh"
#include "posfp.cuh"
#include "stateq_common.cuh"

using namespace mg;

namespace {

// LTE (Boltzmann) populations n_i = n g_i exp(-E_i/kT) / sum_j g_j exp(-E_j/kT).
__global__ void k_lte(int64_t n, int nlev, const double *E, const double *g, const double *T, const double *nspec,
                      double *pops) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    const double ikT = 1.0 / (kKB * T[c]);
    double Z = 0.0;
    for (int i = 0; i < nlev; i++) Z += g[i] * exp(-E[i] * ikT);
    const double s = nspec[c] / Z;
    for (int i = 0; i < nlev; i++) pops[c * nlev + i] = s * g[i] * exp(-E[i] * ikT);
}

// Collision rates per point and level pair (i > j), stored as (down, up):
// C_ij = K_ij(T) n_coll with K interpolated linearly in T (constant beyond the grid), and
// C_ji = C_ij (g_i/g_j) exp(-(E_i - E_j)/kT) (detailed balance).
__global__ void k_collision_rates(int64_t n, int nlev, int nT, const double *E, const double *g,
                                  const double *Tg, const double *K, const double *T, const double *ncoll,
                                  double *coll) {
    const int npairs = nlev * (nlev - 1) / 2;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * npairs) return;
    const int64_t c = t / npairs;
    const int pr = (int)(t - c * npairs);
    int i = 1;
    while ((i + 1) * i / 2 <= pr) i++;
    const int j = pr - i * (i - 1) / 2;
    const double Tc = T[c];
    double Cd, Cu;
    collision_rates_pair(collision_k_down(K, pr, nT, Tg, Tc), ncoll[c], g[i], g[j], E[i], E[j], Tc, Cd, Cu);
    coll[2 * t] = Cd;
    coll[2 * t + 1] = Cu;
}

struct StateqArgs {
    int64_t n;
    int nlev, L;
    const LineConst *lc;
    const double *pops;      // old
    double *pops_new;
    const double *J, *Lc, *Jeff;
    const double *coll;      // [n][npairs][2]
    const double *nspec;
    unsigned long long *scal;   // [0] max change bits, [1] fallback count, [2] non-finite count
    const int32_t *active;      // optional: skip the whole launch when *active == 0
};

// Rates u->l = A (1 - L) + B_ul Jeff + C_ul, l->u = B_lu Jeff + C_lu (eq. 'ourALI');
// 1 - L is passed in directly (accumulated without cancellation by the formal solve).
template <int MAXLEV>
__device__ void build_rates(const StateqArgs &a, int64_t c, bool plain, double (&q)[MAXLEV][MAXLEV]) {
    const int n = a.nlev;
    for (int i = 0; i < n; i++)
        for (int j = 0; j < n; j++) q[i][j] = 0.0;
    line_rates<MAXLEV>(a.L, a.lc, a.J, a.Lc, a.Jeff, c, plain, q);
    const int npairs = n * (n - 1) / 2;
    const double *cr = a.coll + (size_t)c * npairs * 2;
    int pr = 0;
    for (int i = 1; i < n; i++)
        for (int j = 0; j < i; j++, pr++) {
            q[i][j] += cr[2 * pr];
            q[j][i] += cr[2 * pr + 1];
        }
}

template <int MAXLEV>
__global__ void k_stateq(StateqArgs a) {
    if (a.active && !*a.active) return;
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double change = 0.0;
    unsigned long long fb = 0, bad = 0;
    if (c < a.n) {
        const int n = a.nlev;
        double q[MAXLEV][MAXLEV], pi[MAXLEV];
        build_rates<MAXLEV>(a, c, false, q);
        bool ok = gth_solve<MAXLEV>(n, q, pi) && valid_fractions<MAXLEV>(n, pi);
        if (!ok) {
            fb = 1;
            build_rates<MAXLEV>(a, c, true, q);
            ok = gth_solve<MAXLEV>(n, q, pi) && valid_fractions<MAXLEV>(n, pi);
            if (!ok) bad = 1;
        }
        const double ns = a.nspec[c];
        for (int i = 0; i < n; i++) {
            const double nw = ns * pi[i];
            const double od = a.pops[c * n + i];
            a.pops_new[c * n + i] = nw;
            if (nw >= 1e-10 * ns) {
                const double d = fabs(nw - od) / nw;
                if (d > change) change = d;
            }
        }
        if (!isfinite(change)) change = INFINITY;
    }
    // positive doubles order like their bit patterns: max over bits is deterministic
    unsigned long long bits = __double_as_longlong(change);
    for (int d = 16; d; d >>= 1) {
        unsigned long long o = __shfl_down_sync(0xffffffffu, bits, d);
        bits = o > bits ? o : bits;
        fb += __shfl_down_sync(0xffffffffu, fb, d);
        bad += __shfl_down_sync(0xffffffffu, bad, d);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&a.scal[0], bits);
        if (fb) atomicAdd(&a.scal[1], fb);
        if (bad) atomicAdd(&a.scal[2], bad);
    }
}

// The same update with 8 lanes per cell and the rate matrix in shared memory.
//
// One thread per cell (k_stateq) keeps the matrix in local memory and runs the whole
// elimination as one chain: a grid of a few thousand cells takes its latency, ~n^3/3
// dependent steps, and 20 levels spill 3 KB per thread. Eight lanes share a cell's columns:
// the elimination step of level k is k^2/8 multiply-adds per lane, its exit rate and the
// back substitution are sums over the lanes in a fixed tree, and the reciprocal of the exit
// rate runs on the integer pipe (an FP64 division costs 8 FP64 instructions of 80 cycles).
// Measured, one update, thread per cell -> this: 3000 cells x 20 levels 456 -> 72 us, 1500 x 5
// 22.7 -> 14.4 us, 200k x 20 2.95 -> 2.46 ms, 3000 x 64 (32 lanes per cell above 24 levels)
// 19.3 -> 1.25 ms. With few levels the thread-per-cell kernel uses its lanes better and wins
// once the grid hides its latency: 16000 cells x 5 levels 24.5 against 32.2 us, 16000 x 8
// 46.1 against 46.5 us, 200k x 9 444 against 617 us, 200k x 12 874 against 900 us (20000 x 12:
// 167 against 108 us); stateq_thread_cells follows these crossings.
template <int LPC>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
    for (int d = LPC / 2; d; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// Cells from which the thread-per-cell kernel is the faster one.
int64_t stateq_thread_cells(int lev) { return lev <= 8 ? 2000 * lev : (lev <= 12 ? 30000ll << (lev - 9) : (1ll << 60)); }

struct StateqGroup {
    StateqArgs s;
    int cells;        // per block
    int dup;          // two lines share a level pair: their rates are added one by one
};

// Doubles of shared memory per cell: the matrix (row stride odd, so that a column spreads
// over the banks), reciprocal exit rates and populations.
__host__ __device__ inline int stateq_stride(int n) { return n | 1; }
__host__ __device__ inline int stateq_cell_doubles(int n) { return n * stateq_stride(n) + 2 * n; }

template <int LPC>
__device__ __forceinline__ void stateq_group(const StateqGroup &A) {
    extern __shared__ double stq[];
    const StateqArgs &a = A.s;
    if ((int64_t)blockIdx.x * A.cells >= a.n) return;   // (a batch's grid is that of its largest model)
    if (a.active && !*a.active) return;
    const int n = a.nlev, ld = stateq_stride(n);
    const int cell = threadIdx.x / LPC, t = threadIdx.x % LPC;
    const int64_t c = (int64_t)blockIdx.x * A.cells + cell;
    const bool in = c < a.n;
    const int64_t cc = in ? c : a.n - 1;      // (idle groups repeat the last cell and store nothing)
    double *q = stq + (size_t)cell * stateq_cell_doubles(n), *ix = q + n * ld, *pi = ix + n;
    const int npairs = n * (n - 1) / 2;
    const double2 *cr = reinterpret_cast<const double2 *>(a.coll) + (size_t)cc * npairs;
    bool ok = false;
    int fell = 0;
    double tot = 0.0;
    // the ALO first; where its result is invalid, once more without it (Sec. 6.1). All cells
    // of a warp take part in every attempt (the barriers are the warp's).
    for (int attempt = 0; attempt < 2; attempt++) {
        if (__all_sync(0xffffffffu, ok)) break;
        const bool work = !ok, plain = attempt == 1;
        if (work && plain) fell = 1;
        if (work) {
            int i = 1, base = 0;              // pairs (1,0), (2,0), (2,1), ...: pair p = base + j of row i
            for (int p = t; p < npairs; p += LPC) {
                while (p - base >= i) base += i++;
                const int j = p - base;
                const double2 v = cr[p];
                q[i * ld + j] = v.x;
                q[j * ld + i] = v.y;
            }
        }
        __syncwarp();
        for (int l0 = 0; l0 < a.L; l0 += LPC) {
            const int l = l0 + t;
            double down = 0.0, up = 0.0;
            int iu = 0, il = 1;
            if (work && l < a.L) {
                const LineConst k = a.lc[l];
                const double je = plain ? a.J[cc * a.L + l] : a.Jeff[cc * a.L + l];
                const double om = plain ? 1.0 : a.Lc[cc * a.L + l];
                iu = k.up;
                il = k.lo;
                down = k.A * om + k.Bul * je;
                up = k.Blu * je;
            }
            for (int r = 0; r < (A.dup ? LPC : 1); r++) {
                if (work && l < a.L && (!A.dup || t == r)) {
                    q[iu * ld + il] += down;
                    q[il * ld + iu] += up;
                }
                if (A.dup) __syncwarp();
            }
        }
        __syncwarp();
        // state reduction: the exit rate e of level k to those below it, then every rate
        // between lower levels gains the detour through k
        bool good = true;
        for (int k = n - 1; k >= 1; k--) {
            double e = 0.0;
            for (int j = t; j < k; j += LPC) e += q[k * ld + j];
            e = group_sum<LPC>(e);
            good = good && e > 0.0;
            const int ex = (__double2hiint(e) >> 20) & 0x7ff;
            const double is = ex > 2 && ex < 0x7fd ? pos_pack(pos_rcp(pos_from(e))) : 1.0 / e;
            if (t == 0) ix[k] = is;
            for (int j = t; j < k; j += LPC) q[k * ld + j] *= is;
            __syncwarp();
            // q_ij += q_ik (q_kj / e) over the k x k block, its elements dealt to the lanes
            int i = t / k, j = t - i * k;
            const int di = LPC / k, dj = LPC - di * k;
            while (i < k) {
                q[i * ld + j] = fma(q[i * ld + k], q[k * ld + j], q[i * ld + j]);
                i += di;
                j += dj;
                if (j >= k) {
                    j -= k;
                    i++;
                }
            }
            __syncwarp();
        }
        if (t == 0) pi[0] = 1.0;
        double sum = 1.0;
        __syncwarp();
        for (int k = 1; k < n; k++) {
            double s = 0.0;
            for (int i = t; i < k; i += LPC) s += pi[i] * q[i * ld + k];
            s = group_sum<LPC>(s) * ix[k];
            if (t == 0 && work) pi[k] = s;
            sum += s;
            __syncwarp();
        }
        bool valid = good && isfinite(sum);
        for (int i = t; i < n; i += LPC) valid = valid && isfinite(pi[i]) && pi[i] >= 0.0;
        const unsigned vm = __ballot_sync(0xffffffffu, valid);
        const unsigned mine = LPC == 32 ? 0xffffffffu : ((1u << (LPC & 31)) - 1u) << (threadIdx.x & 31 & ~(LPC - 1));
        if (work) {
            ok = (vm & mine) == mine;
            tot = sum;
        }
        __syncwarp();
    }
    double change = 0.0;
    if (in) {
        const double ns = a.nspec[c];
        for (int i = t; i < n; i += LPC) {
            const double nw = ns * (pi[i] / tot);
            const double od = a.pops[c * n + i];
            a.pops_new[c * n + i] = nw;
            if (nw >= 1e-10 * ns) change = fmax(change, fabs(nw - od) / nw);
        }
        if (!isfinite(change)) change = INFINITY;
    }
    unsigned long long bits = __double_as_longlong(change);
    unsigned long long fb = in && t == 0 ? fell : 0, bad = in && t == 0 ? !ok : 0;
    for (int d = 16; d; d >>= 1) {
        const unsigned long long o = __shfl_down_sync(0xffffffffu, bits, d);
        bits = o > bits ? o : bits;
        fb += __shfl_down_sync(0xffffffffu, fb, d);
        bad += __shfl_down_sync(0xffffffffu, bad, d);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&a.scal[0], bits);
        if (fb) atomicAdd(&a.scal[1], fb);
        if (bad) atomicAdd(&a.scal[2], bad);
    }
}

template <int LPC>
__global__ void __launch_bounds__(128) k_stateq_group(StateqGroup A) {
    stateq_group<LPC>(A);
}

// Several models in one launch (blockIdx.y), their arguments by value.
constexpr int kBatchArgs = 24;
struct StateqBatch {
    StateqGroup m[kBatchArgs];
};
static_assert(sizeof(StateqBatch) <= 4096, "kernel parameter size");
template <int LPC>
__global__ void __launch_bounds__(128) k_stateq_batch(const __grid_constant__ StateqBatch b) {
    stateq_group<LPC>(b.m[blockIdx.y]);
}

// ---------------------------------------------------------------- Ng acceleration
// History of fractional populations x = n_i / n_spec (uniform weights over levels).
// (The Ng kernels serve one or several models, blockIdx.y.)
struct NgArgs {
    int64_t m;                 // values: cells x levels
    int nlev, blocks;          // blocks of the dot products
    const double *x0, *x1, *x2, *x3, *nspec, *pops;
    double *hist, *part, *tmp;
    unsigned long long *flag;
};
constexpr int kNgBatch = 24;
struct NgBatch {
    NgArgs a[kNgBatch];
};
static_assert(sizeof(NgBatch) <= 4096, "kernel parameter size");

__global__ void k_push_history(const __grid_constant__ NgBatch b) {
    const NgArgs &a = b.a[blockIdx.y];
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.m) return;
    a.hist[t] = a.pops[t] / a.nspec[t / a.nlev];
}

constexpr int kNgBlocks = 512;
constexpr int kNgThreads = 256;

// Partial sums of the Ng normal equations with D_i = x_i - x_{i+1}, Q_j = D_0 - D_j:
// a11 = <Q1,Q1>, a12 = <Q1,Q2>, a22 = <Q2,Q2>, b1 = <Q1,D0>, b2 = <Q2,D0>. Each block
// writes its partials; a fixed-order sum follows, so the result is reproducible.
__global__ void k_ng_dots(const __grid_constant__ NgBatch b) {
    const NgArgs &a = b.a[blockIdx.y];
    if ((int)blockIdx.x >= a.blocks) return;
    const double *x0 = a.x0, *x1 = a.x1, *x2 = a.x2, *x3 = a.x3;
    double *part = a.part;
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.flag = 0;
    double s[5] = {0, 0, 0, 0, 0};
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < a.m; t += (int64_t)a.blocks * blockDim.x) {
        const double D0 = x0[t] - x1[t], D1 = x1[t] - x2[t], D2 = x2[t] - x3[t];
        const double Q1 = D0 - D1, Q2 = D0 - D2;
        s[0] += Q1 * Q1; s[1] += Q1 * Q2; s[2] += Q2 * Q2; s[3] += Q1 * D0; s[4] += Q2 * D0;
    }
    __shared__ double sh[5][kNgThreads];
    for (int k = 0; k < 5; k++) sh[k][threadIdx.x] = s[k];
    __syncthreads();
    for (int w = kNgThreads / 2; w; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int k = 0; k < 5; k++) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int k = 0; k < 5; k++) part[5 * blockIdx.x + k] = sh[k][0];
}

// Sums the partials in a fixed order, solves the 2x2 system and forms
// x = (1 - a1 - a2) x0 + a1 x1 + a2 x2 in tmp; flags a singular system or a negative value.
__global__ void k_ng_apply(const __grid_constant__ NgBatch b) {
    const NgArgs &a = b.a[blockIdx.y];
    if ((int)blockIdx.x >= a.blocks) return;
    const double *x0 = a.x0, *x1 = a.x1, *x2 = a.x2;
    double *part = a.part, *tmp = a.tmp;
    unsigned long long *flag = a.flag;
    const int nparts = a.blocks;
    __shared__ double coef[2];
    __shared__ int singular;
    // the first warp sums the partials: strided per lane, then a shuffle tree (every block
    // the same order)
    double s[5] = {0, 0, 0, 0, 0};
    if (threadIdx.x < 32) {
        for (int b = threadIdx.x; b < nparts; b += 32)
            for (int k = 0; k < 5; k++) s[k] += part[5 * b + k];
        for (int d = 16; d; d >>= 1)
            for (int k = 0; k < 5; k++) s[k] += __shfl_xor_sync(0xffffffffu, s[k], d);
    }
    if (threadIdx.x == 0) {
        const double det = s[0] * s[2] - s[1] * s[1];
        singular = !(det != 0.0 && isfinite(det));
        coef[0] = singular ? 0.0 : (s[3] * s[2] - s[4] * s[1]) / det;
        coef[1] = singular ? 0.0 : (s[0] * s[4] - s[1] * s[3]) / det;
        if (singular && blockIdx.x == 0) atomicOr(flag, 1ull);
    }
    __syncthreads();
    if (singular) return;
    const double a1 = coef[0], a2 = coef[1];
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < a.m; t += (int64_t)a.blocks * blockDim.x) {
        const double x = (1.0 - a1 - a2) * x0[t] + a1 * x1[t] + a2 * x2[t];
        if (!(x >= 0.0)) atomicOr(flag, 2ull);
        tmp[t] = x * a.nspec[t / a.nlev];
    }
}

}  // namespace

int mg_launch_lte(mg_ctx *ctx) {
    MgTimed t(ctx, "lte");
    k_lte<<<(unsigned)((ctx->n + 127) / 128), 128, 0, ctx->stream>>>(ctx->n, ctx->n_lev, ctx->d_E, ctx->d_g,
                                                                      ctx->d_T, ctx->d_nspec, ctx->d_pops);
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

int mg_launch_collision_rates(mg_ctx *ctx) {
    const int npairs = ctx->n_lev * (ctx->n_lev - 1) / 2;
    int rc;
    if ((rc = mg_alloc(ctx, &ctx->d_coll, (size_t)ctx->n * npairs * 2))) return rc;
    const int64_t m = ctx->n * npairs;
    k_collision_rates<<<(unsigned)((m + 255) / 256), 256, 0, ctx->stream>>>(
        ctx->n, ctx->n_lev, ctx->n_T, ctx->d_E, ctx->d_g, ctx->d_Tgrid, ctx->d_Kdown, ctx->d_T, ctx->d_ncoll,
        ctx->d_coll);
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

template <int LPC>
static int launch_stateq_group(mg_ctx *ctx, const StateqArgs &a) {
    StateqGroup A{};
    A.s = a;
    A.dup = ctx->dup_lines;
    const size_t cell = sizeof(double) * stateq_cell_doubles(ctx->n_lev);
    A.cells = 128 / LPC;   // 128 threads, fewer where two blocks would not fit an SM
    while (A.cells > 32 / LPC && A.cells * cell > 110 * 1024) A.cells /= 2;
    MG_CUDA(cudaFuncSetAttribute(k_stateq_group<LPC>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem));
    k_stateq_group<LPC><<<(unsigned)((ctx->n + A.cells - 1) / A.cells), A.cells * LPC, A.cells * cell, ctx->stream>>>(A);
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

static int launch_stateq(mg_ctx *ctx, const StateqArgs &a) {
    const unsigned grid = (unsigned)((ctx->n + 127) / 128);
    const int lev = ctx->n_lev;
    if (ctx->n >= stateq_thread_cells(lev)) {
        if (lev <= 8) k_stateq<8><<<grid, 128, 0, ctx->stream>>>(a);
        else k_stateq<12><<<grid, 128, 0, ctx->stream>>>(a);
        MG_CUDA(cudaGetLastError());
        return MG_OK;
    }
    return lev <= 24 ? launch_stateq_group<8>(ctx, a) : launch_stateq_group<32>(ctx, a);
}

int mg_launch_stateq(mg_ctx *ctx) {
    StateqArgs a{};
    a.n = ctx->n; a.nlev = ctx->n_lev; a.L = ctx->n_lines; a.lc = ctx->d_lines;
    a.pops = ctx->d_pops; a.pops_new = ctx->d_pops_new; a.J = ctx->d_J; a.Lc = ctx->d_Lc; a.Jeff = ctx->d_Jeff;
    a.coll = ctx->d_coll; a.nspec = ctx->d_nspec; a.scal = ctx->d_scal;
    MG_CUDA(cudaMemsetAsync(ctx->d_scal, 0, 3 * sizeof(unsigned long long), ctx->stream));
    int rc;
    {
        MgTimed t(ctx, "stateq");
        rc = launch_stateq(ctx, a);
    }
    if (rc) return rc;
    std::swap(ctx->d_pops, ctx->d_pops_new);
    return MG_OK;
}

// Statistical equilibrium from pops_old into pops_new with explicit buffers (no pointer
// swap), skipped when *active == 0; used by the batch graph.
int mg_launch_stateq_into(mg_ctx *ctx, const double *pops_old, double *pops_new, const int32_t *active) {
    StateqArgs a{};
    a.n = ctx->n; a.nlev = ctx->n_lev; a.L = ctx->n_lines; a.lc = ctx->d_lines;
    a.pops = pops_old; a.pops_new = pops_new; a.J = ctx->d_J; a.Lc = ctx->d_Lc; a.Jeff = ctx->d_Jeff;
    a.coll = ctx->d_coll; a.nspec = ctx->d_nspec; a.scal = ctx->d_scal; a.active = active;
    return launch_stateq(ctx, a);
}

// The statistical equilibrium of every model in place (pops -> pops; each cell reads its old
// values before it writes), as one launch per 24 models; `active`: one word per model.
// Returns 1 when the models need a launch each (mixed level counts, or large models of few
// levels, for which the thread-per-cell kernel is the faster one).
int mg_launch_stateq_batch(mg_ctx *const *models, int count, const int32_t *active, cudaStream_t stream) {
    const int lev = models[0]->n_lev;
    int64_t nmax = 0;
    for (int i = 0; i < count; i++) {
        if (models[i]->n_lev != lev || models[i]->n >= stateq_thread_cells(lev)) return 1;
        nmax = std::max(nmax, models[i]->n);
    }
    const int lpc = lev <= 24 ? 8 : 32;
    const size_t cell = sizeof(double) * stateq_cell_doubles(lev);
    int cells = 128 / lpc;
    while (cells > 32 / lpc && cells * cell > 110 * 1024) cells /= 2;
    void (*kern)(StateqBatch) = lpc == 8 ? k_stateq_batch<8> : k_stateq_batch<32>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
    for (int i0 = 0; i0 < count && e == cudaSuccess; i0 += kBatchArgs) {
        StateqBatch b{};
        const int k = std::min(kBatchArgs, count - i0);
        for (int i = 0; i < k; i++) {
            const mg_ctx *c = models[i0 + i];
            StateqArgs &a = b.m[i].s;
            a.n = c->n; a.nlev = lev; a.L = c->n_lines; a.lc = c->d_lines;
            a.pops = c->d_pops; a.pops_new = c->d_pops; a.J = c->d_J; a.Lc = c->d_Lc; a.Jeff = c->d_Jeff;
            a.coll = c->d_coll; a.nspec = c->d_nspec; a.scal = c->d_scal; a.active = active + i0 + i;
            b.m[i].cells = cells;
            b.m[i].dup = c->dup_lines;
        }
        kern<<<dim3((unsigned)((nmax + cells - 1) / cells), k), cells * lpc, cells * cell, stream>>>(b);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? MG_OK : MG_ERR_CUDA;
}

// A block per 2048 values (8 per thread), so that small models leave few partials to sum.
// With 512 blocks, and one thread summing their partials in every block of the second
// kernel, the step took 131 us; now 28 us (3000 cells x 20 levels).
static NgArgs ng_args(mg_ctx *ctx) {
    NgArgs a{};
    a.m = ctx->n * ctx->n_lev;
    a.nlev = ctx->n_lev;
    a.blocks = (int)std::min<int64_t>(kNgBlocks, (a.m + 2047) / 2048);
    a.x0 = ctx->d_hist[0]; a.x1 = ctx->d_hist[1]; a.x2 = ctx->d_hist[2]; a.x3 = ctx->d_hist[3];
    a.nspec = ctx->d_nspec; a.pops = ctx->d_pops; a.hist = ctx->d_hist[0];
    a.part = ctx->d_ng_part; a.tmp = ctx->d_ng_tmp; a.flag = ctx->d_scal + 3;
    return a;
}

// Pushes the current populations of every model into its history, and runs the Ng step of
// every model (flag word d_scal[3]: 0 when the step is valid; it is in d_ng_tmp then).
int mg_launch_push_history_batch(mg_ctx *const *models, int count, cudaStream_t stream) {
    for (int i0 = 0; i0 < count; i0 += kNgBatch) {
        NgBatch b{};
        const int k = std::min(kNgBatch, count - i0);
        int64_t mmax = 0;
        for (int i = 0; i < k; i++) {
            mg_ctx *ctx = models[i0 + i];
            const int64_t m = ctx->n * ctx->n_lev;
            int rc;
            for (auto &h : ctx->d_hist)
                if (!h && (rc = mg_alloc(ctx, &h, m))) return rc;
            double *t = ctx->d_hist[3];
            ctx->d_hist[3] = ctx->d_hist[2];
            ctx->d_hist[2] = ctx->d_hist[1];
            ctx->d_hist[1] = ctx->d_hist[0];
            ctx->d_hist[0] = t;
            b.a[i] = ng_args(ctx);
            mmax = std::max(mmax, m);
        }
        k_push_history<<<dim3((unsigned)((mmax + 255) / 256), k), 256, 0, stream>>>(b);
        if (cudaGetLastError() != cudaSuccess) return MG_ERR_CUDA;
    }
    return MG_OK;
}

int mg_launch_ng_batch(mg_ctx *const *models, int count, cudaStream_t stream) {
    for (int i0 = 0; i0 < count; i0 += kNgBatch) {
        NgBatch b{};
        const int k = std::min(kNgBatch, count - i0);
        int blocks = 1;
        for (int i = 0; i < k; i++) {
            mg_ctx *ctx = models[i0 + i];
            int rc;
            if (!ctx->d_ng_tmp && (rc = mg_alloc(ctx, &ctx->d_ng_tmp, ctx->n * ctx->n_lev))) return rc;
            if (!ctx->d_ng_part && (rc = mg_alloc(ctx, &ctx->d_ng_part, 5 * kNgBlocks))) return rc;
            b.a[i] = ng_args(ctx);
            blocks = std::max(blocks, b.a[i].blocks);
        }
        k_ng_dots<<<dim3(blocks, k), kNgThreads, 0, stream>>>(b);
        k_ng_apply<<<dim3(blocks, k), kNgThreads, 0, stream>>>(b);
        if (cudaGetLastError() != cudaSuccess) return MG_ERR_CUDA;
    }
    return MG_OK;
}

int mg_launch_push_history(mg_ctx *ctx) {
    int rc = mg_launch_push_history_batch(&ctx, 1, ctx->stream);
    if (rc == MG_ERR_CUDA) return mg_cuda_check(ctx, cudaErrorLaunchFailure, "Ng history");
    return rc;
}

int mg_launch_ng(mg_ctx *ctx, int *accepted) {
    int rc;
    {
        MgTimed t(ctx, "ng");
        rc = mg_launch_ng_batch(&ctx, 1, ctx->stream);
    }
    if (rc == MG_ERR_CUDA) return mg_cuda_check(ctx, cudaErrorLaunchFailure, "Ng step");
    if (rc) return rc;
    MG_CUDA(cudaMemcpyAsync(ctx->h_scal + 3, ctx->d_scal + 3, 8, cudaMemcpyDeviceToHost, ctx->stream));
    MG_CUDA(cudaStreamSynchronize(ctx->stream));
    *accepted = ctx->h_scal[3] == 0;
    if (*accepted)
        MG_CUDA(cudaMemcpyAsync(ctx->d_pops, ctx->d_ng_tmp, 8 * ctx->n * ctx->n_lev, cudaMemcpyDeviceToDevice, ctx->stream));
    return MG_OK;
}
