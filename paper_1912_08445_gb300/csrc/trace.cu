// K1: ray tracing by neighbour walk (Sec. 3.2) with the velocity-step rule (Sec. 3.1.1).
// This translation unit is compiled with --fmad=false: every floating-point decision of
// the walk (projections, distances, velocity steps) is reproducible bit for bit.
#include <cmath>
#include <algorithm>
#include <mutex>
#include "common.cuh"
#include "kept.h"

using namespace mg;

namespace {

struct TraceArgs {
    int64_t n;
    int32_t R;
    int32_t geometry;
    const double *pos, *vel, *b, *dirs;
    const float4 *posf;                // (x, y, z, reach) in FP32, for the filter: the reach of a cell is
                                       // the largest |x| + |y| + |z| of it and its neighbours
    const int64_t *nbr_off;
    const int32_t *nbr_idx;
    const uint8_t *bdy;
    double dshift_frac;
    int64_t max_steps;
    // count pass
    int32_t *len, *xlen;
    // fill pass
    const int64_t *ray_off;
    int32_t *cells, *xcum;
    double *ds, *vpar;
    float *dsf, *vparf;                // FP32 copies
    int32_t *err;
    // cells of each half-ray recorded by the count pass: tmp[k * n R + t] for k < cap_tmp
    int32_t *tmp;
    int32_t cap_tmp;
};

// Points inserted between two consecutive points by the velocity-step rule: when the
// line-of-sight velocity changes by dv > f min(b_a, b_b), ceil(dv/(f min)) - 1 points.
__device__ __forceinline__ int32_t velocity_inserts(double va, double ba, double vb, double bb, double f) {
    double dv = fabs(vb - va);
    // (widths are positive: they compare like their bits)
    double wmin = __double_as_longlong(ba) < __double_as_longlong(bb) ? ba : bb;
    double lim = f * wmin;
    if (dv > lim) {
        // The FP32 quotient (relative error below 4e-7) decides the ceiling unless it lies that
        // close to a whole number; an FP64 division costs eight FP64 instructions.
        const float q = __fdiv_rn((float)dv, (float)lim), near = rintf(q);
        if (q < 1e6f && fabsf(q - near) > 1e-6f * q) return (int32_t)ceilf(q) - 1;
        return (int32_t)ceil(dv / lim) - 1;
    }
    return 0;
}

// Records one element of the half-ray. The count pass records only the cell (its count,
// and the first cells for the replay); the fill pass also the path length, the
// line-of-sight velocity and the expanded-point count of the velocity-step rule.
template <bool FILL>
__device__ __forceinline__ bool emit(const TraceArgs &a, int64_t base, int32_t &len, int32_t &x, int32_t cell,
                                     double ds, double vp, double &va, double &ba) {
    if (len >= a.max_steps) return false;
    if (FILL) {
        double bb = a.b[cell];
        int32_t ns = velocity_inserts(va, ba, vp, bb, a.dshift_frac);
        x += ns + 1;
        a.cells[base + len] = cell;
        a.xcum[base + len] = x;
        a.ds[base + len] = ds;
        a.vpar[base + len] = vp;
        a.dsf[base + len] = (float)ds;
        a.vparf[base + len] = (float)vp;
        va = vp;
        ba = bb;
    } else if (a.tmp && len < a.cap_tmp) {
        a.tmp[(int64_t)len * a.n * a.R + base] = cell;   // base = thread index in the count pass
    }
    len++;
    return true;
}

// 3D point cloud: from the current cell, the neighbour with a strictly larger projection
// on the ray that lies closest to the ray (ties: smaller squared distance, smaller
// projection, smaller index); stop after a boundary cell or at a dead end.
//
// The decisions are those of the FP64 expressions below, bit for bit, but most of them
// are taken in FP32 (64x the FP64 rate on this GPU) with a rigorous error bound, and FP64
// is evaluated only where the bound cannot decide:
// - a candidate is valid when s > s_cur: the FP32 projection decides unless it lies
//   within its error bound of s_cur, where the FP64 projection decides;
// - the FP32 squared distance d of every valid candidate comes with an error bound Ed(d), so
//   that the FP64 value lies in [lo, hi] = [d - Ed, d + Ed]. The FP64 winner's lo is at most
//   the smallest hi, that of the smallest d. The three smallest d are kept: when the
//   second's lo lies above that hi, the first is the winner; when the third's does, the
//   first two are evaluated in FP64 and the winner is chosen with the exact tie-breaks;
//   otherwise every valid candidate with lo <= hi is. (A non-finite d leaves the choice to
//   the last.)
// The bounds follow from |fl32(a) - a| <= u|a| (u = 2^-24) for the conversions of the
// positions and the direction and for each FP32 operation, with |x|_1 bounded by the reaches
// of the current cell and of the origin (P below); they are doubled for margin. They are the
// same for every candidate of a step: bounds per candidate took more instructions than the
// distances themselves (20k-point cloud, 960k half-rays: 2.02 ms, per step 1.41 ms). Bounds for
// the whole model (1.42 ms) decide nothing near the centre of a model with many scales: 20k
// points over five decades of radius took 36.0 ms, bounds per candidate 5.7 ms, per step 4.1 ms.
struct Bounds32 {
    float margin;          // of |s32 - s_cur|
    float e1, e0, e2;      // Ed(d) = e1 sqrt(d) + e0 + e2 d
    __device__ Bounds32(float P) {
        constexpr float k2u = 1.2e-7f;   // 2u with margin
        const float Es = k2u * 7.0f * P;                                // |s32 - s64|
        margin = Es + k2u * 4.0f * P;                                   // and of s_cur and the difference
        const float Ep = 2.0f * (Es + 0.6e-7f * 8.0f * P);              // |p32 - p64| per component
        e1 = 1.1f * 2.0f * Ep * 1.7322f;                                // |p|_1 <= sqrt(3 d)
        e0 = 1.1f * 9.0f * Ep * Ep;
        e2 = 1.1f * 2.0f * k2u;
    }
    __device__ float err(float d) const { return e1 * sqrtf(d) + e0 + e2 * d; }
};

__device__ __forceinline__ double proj64(const TraceArgs &a, int64_t c, double xo0, double xo1, double xo2,
                                         double n0, double n1, double n2) {
    const double dx = a.pos[3 * c] - xo0;
    const double dy = a.pos[3 * c + 1] - xo1;
    const double dz = a.pos[3 * c + 2] - xo2;
    return dx * n0 + dy * n1 + dz * n2;
}

// FP32 squared distance of candidate c from the ray and whether it lies ahead of s_cur.
__device__ __forceinline__ bool ahead32(const TraceArgs &a, int64_t c, const float4 pc, const float4 po, float n0f,
                                        float n1f, float n2f, float scf, const Bounds32 &B, double s_cur, double xo0,
                                        double xo1, double xo2, double n0, double n1, double n2, float &d2) {
    const float dx = pc.x - po.x, dy = pc.y - po.y, dz = pc.z - po.z;
    const float sf = __fmaf_rn(dz, n2f, __fmaf_rn(dy, n1f, dx * n0f));
    const float px = __fmaf_rn(-sf, n0f, dx), py = __fmaf_rn(-sf, n1f, dy), pz = __fmaf_rn(-sf, n2f, dz);
    d2 = __fmaf_rn(pz, pz, __fmaf_rn(py, py, px * px));
    const float diff = sf - scf;
    if (diff > B.margin) return true;
    if (diff < -B.margin) return false;
    return proj64(a, c, xo0, xo1, xo2, n0, n1, n2) > s_cur;   // inconclusive in FP32
}

template <bool FILL>
__device__ void walk_3d(const TraceArgs &a, int64_t o, int r, int64_t base, int32_t &len, int32_t &x,
                        bool &dead, bool &overflow) {
    const double n0 = a.dirs[3 * r], n1 = a.dirs[3 * r + 1], n2 = a.dirs[3 * r + 2];
    const double xo0 = a.pos[3 * o], xo1 = a.pos[3 * o + 1], xo2 = a.pos[3 * o + 2];
    const double vo0 = a.vel[3 * o], vo1 = a.vel[3 * o + 1], vo2 = a.vel[3 * o + 2];
    const float n0f = (float)n0, n1f = (float)n1, n2f = (float)n2;
    const float4 po = a.posf[o];
    int64_t cur = o;
    double s_cur = 0.0;
    double va = 0.0, ba = a.b[o];
    len = 0;
    x = 0;
    dead = false;
    overflow = false;
    for (;;) {
        const float scf = (float)s_cur;
        const Bounds32 B((a.posf[cur].w + po.w) * 1.0001f);
        const int64_t e0 = a.nbr_off[cur], e1 = a.nbr_off[cur + 1];
        // pass 1: the three smallest FP32 distances among the valid candidates, four
        // candidates' gathers in flight at a time
        float d1 = INFINITY, d2 = INFINITY, d3 = INFINITY;
        int32_t c1 = -1, c2 = -1;
        bool full = false;   // a distance that is not finite leaves the choice to FP64
        for (int64_t e = e0; e < e1; e += 4) {
            int32_t id[4];
            float4 pc[4];
#pragma unroll
            for (int k = 0; k < 4; k++) id[k] = a.nbr_idx[e + k < e1 ? e + k : e0];
#pragma unroll
            for (int k = 0; k < 4; k++) pc[k] = a.posf[id[k]];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                if (e + k >= e1) break;
                float d;
                if (!ahead32(a, id[k], pc[k], po, n0f, n1f, n2f, scf, B, s_cur, xo0, xo1, xo2, n0, n1, n2, d)) continue;
                full = full || !(d < INFINITY);
                const bool l1 = d < d1, l2 = d < d2;
                d3 = l2 ? d2 : fminf(d3, d);
                c2 = l1 ? c1 : (l2 ? id[k] : c2);
                d2 = l1 ? d1 : (l2 ? d : d2);
                c1 = l1 ? id[k] : c1;
                d1 = l1 ? d : d1;
            }
        }
        int64_t best = -1;
        double bs = 0.0, bd2 = 0.0;
        const float hi = d1 + B.err(d1);
        full = full || !(hi < INFINITY);
        // FP64 distance of one candidate, with the tie-breaks
        auto consider = [&](int64_t c) {
            const double dx = a.pos[3 * c] - xo0;
            const double dy = a.pos[3 * c + 1] - xo1;
            const double dz = a.pos[3 * c + 2] - xo2;
            const double s = dx * n0 + dy * n1 + dz * n2;
            const double px = dx - s * n0, py = dy - s * n1, pz = dz - s * n2;
            const double dd = px * px + py * py + pz * pz;
            const bool better = (best < 0) || (dd < bd2) || (dd == bd2 && s < bs) || (dd == bd2 && s == bs && c < best);
            if (better) { best = c; bs = s; bd2 = dd; }
        };
        if (!full && (c2 < 0 || d2 - B.err(d2) > hi)) {
            best = c1;
            bs = proj64(a, c1, xo0, xo1, xo2, n0, n1, n2);
        } else if (!full && (!(d3 < INFINITY) || d3 - B.err(d3) > hi)) {
            consider(c1);
            consider(c2);
        } else if (c1 >= 0 || full) {
            for (int64_t e = e0; e < e1; e++) {
                const int64_t c = a.nbr_idx[e];
                float d;
                if (!ahead32(a, c, a.posf[c], po, n0f, n1f, n2f, scf, B, s_cur, xo0, xo1, xo2, n0, n1, n2, d)) continue;
                if (!full && d - B.err(d) > hi) continue;
                consider(c);
            }
        }
        if (best < 0) { dead = true; return; }
        const double vp = FILL ? n0 * (a.vel[3 * best] - vo0) + n1 * (a.vel[3 * best + 1] - vo1) +
                                     n2 * (a.vel[3 * best + 2] - vo2)
                               : 0.0;
        if (!emit<FILL>(a, base, len, x, (int32_t)best, bs - s_cur, vp, va, ba)) { overflow = true; return; }
        s_cur = bs;
        cur = best;
        if (a.bdy[best]) return;
    }
}

// Fill pass of a half-ray whose cells the count pass recorded: the same projections,
// path lengths, line-of-sight velocities and velocity steps as the walk, without the
// neighbour search.
__device__ int32_t replay_3d(const TraceArgs &a, int64_t o, int r, int64_t t, int64_t base, int32_t n_cells) {
    const double n0 = a.dirs[3 * r], n1 = a.dirs[3 * r + 1], n2 = a.dirs[3 * r + 2];
    const double xo0 = a.pos[3 * o], xo1 = a.pos[3 * o + 1], xo2 = a.pos[3 * o + 2];
    const double vo0 = a.vel[3 * o], vo1 = a.vel[3 * o + 1], vo2 = a.vel[3 * o + 2];
    double s_cur = 0.0, va = 0.0, ba = a.b[o];
    int32_t len = 0, x = 0;
    for (int32_t k = 0; k < n_cells; k++) {
        const int64_t c = a.tmp[(int64_t)k * a.n * a.R + t];
        const double dx = a.pos[3 * c] - xo0;
        const double dy = a.pos[3 * c + 1] - xo1;
        const double dz = a.pos[3 * c + 2] - xo2;
        const double s = dx * n0 + dy * n1 + dz * n2;
        const double vp = n0 * (a.vel[3 * c] - vo0) + n1 * (a.vel[3 * c + 1] - vo1) + n2 * (a.vel[3 * c + 2] - vo2);
        emit<true>(a, base, len, x, (int32_t)c, s - s_cur, vp, va, ba);
        s_cur = s;
    }
    return x;
}

// Spherically symmetric shells on +z: crossings of the ray with sphere j at
// s = -r_o mu +- sqrt(r_j^2 - r_o^2 (1 - mu^2)), in increasing s; an empty core below the
// first radius carries no path length; a first radius of 0 is a centre point.
template <bool FILL>
__device__ void walk_sph1d(const TraceArgs &a, int64_t o, int r, int64_t base, int32_t &len, int32_t &x,
                           bool &overflow) {
    const double mu = a.dirs[3 * r + 2];
    const double ro = a.pos[3 * o + 2];
    const double p2 = ro * ro * (1.0 - mu * mu);
    const double vro = a.vel[3 * o + 2];
    const int64_t N = a.n;
    const double r0 = a.pos[2];
    double va = 0.0, ba = a.b[o];
    double s_prev = 0.0;
    len = 0;
    x = 0;
    overflow = false;
    int64_t j = o;
    bool through_core = false;
    const bool inward = (mu < 0.0 && ro > 0.0);
    if (inward) {
        for (j = o - 1; j >= 0; j--) {
            const double rj = a.pos[3 * j + 2];
            const double q = rj * rj - p2;
            if (rj == 0.0 && p2 == 0.0) {
                const double s = -ro * mu;
                if (!emit<FILL>(a, base, len, x, (int32_t)j, s - s_prev, -vro * mu, va, ba)) { overflow = true; return; }
                s_prev = s;
                j--;
                break;
            }
            if (!(q > 0.0) || rj == 0.0) break;
            const double s = -ro * mu - sqrt(q);
            const double vp = a.vel[3 * j + 2] * (ro * mu + s) / rj - vro * mu;
            if (!emit<FILL>(a, base, len, x, (int32_t)j, s - s_prev, vp, va, ba)) { overflow = true; return; }
            s_prev = s;
        }
        if (j < 0 && r0 > 0.0) through_core = true;
        j = j + 1;
        if (j == 0 && r0 == 0.0) j = 1;
    }
    const int64_t jstart = inward ? j : o + 1;
    for (int64_t k = jstart; k < N; k++) {
        const double rk = a.pos[3 * k + 2];
        const double q = rk * rk - p2;
        if (q < 0.0) continue;
        const double s = -ro * mu + sqrt(q);
        const bool core_chord = through_core && k == jstart;
        if (!(s > s_prev) && !core_chord) continue;
        const double dsv = core_chord ? 0.0 : s - s_prev;
        const double vp = (rk > 0.0 ? a.vel[3 * k + 2] * (ro * mu + s) / rk : 0.0) - vro * mu;
        if (!emit<FILL>(a, base, len, x, (int32_t)k, dsv, vp, va, ba)) { overflow = true; return; }
        s_prev = s;
    }
}

// One thread per (origin, direction); consecutive threads take consecutive origins of the
// same direction so that neighbouring walks share cache lines.
template <bool FILL>
__global__ void k_trace(TraceArgs a) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.n * a.R) return;
    const int r = (int)(t / a.n);
    const int64_t o = t - (int64_t)r * a.n;
    const int64_t ray = o * a.R + r;
    const int64_t base = FILL ? a.ray_off[ray] : t;
    int32_t len = 0, x = 0;
    bool dead = false, overflow = false;
    if (FILL && a.tmp && a.geometry == MG_GEOM_3D) {
        const int32_t n_cells = a.len[ray];
        if (n_cells <= a.cap_tmp) {
            const int32_t xl = replay_3d(a, o, r, t, base, n_cells);
            a.xlen[ray] = a.xlen[ray] < 0 ? -xl - 1 : xl;
            return;
        }
    }
    if (a.geometry == MG_GEOM_SPHERICAL_1D) walk_sph1d<FILL>(a, o, r, base, len, x, overflow);
    else walk_3d<FILL>(a, o, r, base, len, x, dead, overflow);
    if (overflow) atomicOr(a.err, 1);
    if (!FILL) {
        a.len[ray] = len;
        a.xlen[ray] = dead ? -1 : 0;   // dead-end flag
    } else {
        // the expanded length, with the count pass's dead-end flag as the sign (-x - 1)
        a.xlen[ray] = a.xlen[ray] < 0 ? -x - 1 : x;
    }
}

// ---------------------------------------------------------------- exclusive scan
// Exclusive prefix sum of int32 counts into int64 offsets, in three passes: per-block
// sums, a single-block scan of the block sums, then per-block scans with their offsets.
constexpr int kScanBlock = 1024;

__device__ __forceinline__ int64_t warp_incl_scan(int64_t v) {
    const int lane = threadIdx.x & 31;
    for (int d = 1; d < 32; d <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += y;
    }
    return v;
}

__device__ int64_t block_excl_scan(int64_t v, int64_t *total) {
    __shared__ int64_t wsum[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int64_t inc = warp_incl_scan(v);
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    if (w == 0) {
        int64_t s = (lane < (int)(blockDim.x >> 5)) ? wsum[lane] : 0;
        s = warp_incl_scan(s);
        wsum[lane] = s;
    }
    __syncthreads();
    int64_t off = w ? wsum[w - 1] : 0;
    if (total) *total = wsum[(blockDim.x >> 5) - 1];
    __syncthreads();
    return off + inc - v;
}

__global__ void k_scan_blocks(const int32_t *cnt, int64_t m, int64_t *bsum) {
    int64_t i = (int64_t)blockIdx.x * kScanBlock + threadIdx.x;
    int64_t v = i < m ? cnt[i] : 0;
    int64_t tot;
    block_excl_scan(v, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void k_scan_sums(int64_t *bsum, int64_t nb) {
    // single block: sequential chunks of kScanBlock
    int64_t carry = 0;
    for (int64_t c0 = 0; c0 < nb; c0 += kScanBlock) {
        int64_t i = c0 + threadIdx.x;
        int64_t v = i < nb ? bsum[i] : 0;
        int64_t tot;
        int64_t ex = block_excl_scan(v, &tot);
        if (i < nb) bsum[i] = ex + carry;
        carry += tot;
        __syncthreads();
    }
}

__global__ void k_scan_apply(const int32_t *cnt, int64_t m, const int64_t *bsum, int64_t *out) {
    int64_t i = (int64_t)blockIdx.x * kScanBlock + threadIdx.x;
    int64_t v = i < m ? cnt[i] : 0;
    int64_t ex = block_excl_scan(v, nullptr);
    if (i < m) out[i] = bsum[blockIdx.x] + ex;
    if (i == m - 1) out[m] = bsum[blockIdx.x] + ex + v;
}

// ---------------------------------------------------------------- statistics
constexpr int kStatBlocks = 304, kStatThreads = 256;

// Two kernels' worth of blocks per SM, each adding its sums once (a warp each made 81 us of
// contention on four words of 960k half-rays).
__global__ void __launch_bounds__(kStatThreads) k_ray_stats(int64_t n, int R, int P, const int32_t *pf, const int32_t *pb,
                                                            const int32_t *len, const int32_t *xlen,
                                                            unsigned long long *st) {
    // st: [0] elements, [1] expanded, [2] max pair length, [3] dead ends
    unsigned long long el = 0, ex = 0, mx = 0, dead = 0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * R; t += (int64_t)gridDim.x * blockDim.x) {
        int32_t xv = xlen[t];
        if (xv < 0) { dead++; xv = -xv - 1; }
        el += (unsigned long long)len[t];
        ex += (unsigned long long)xv;
    }
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * P; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t o = t / P;
        const int p = (int)(t - o * P);
        int32_t a = xlen[o * R + pf[p]], b = xlen[o * R + pb[p]];
        a = a < 0 ? -a - 1 : a;
        b = b < 0 ? -b - 1 : b;
        mx = max(mx, (unsigned long long)(a + b + 1));
    }
    __shared__ unsigned long long sh[4][kStatThreads / 32];
    for (int d = 16; d; d >>= 1) {
        el += __shfl_down_sync(0xffffffffu, el, d);
        ex += __shfl_down_sync(0xffffffffu, ex, d);
        dead += __shfl_down_sync(0xffffffffu, dead, d);
        unsigned long long m2 = __shfl_down_sync(0xffffffffu, mx, d);
        mx = m2 > mx ? m2 : mx;
    }
    if ((threadIdx.x & 31) == 0) {
        const int w = threadIdx.x >> 5;
        sh[0][w] = el; sh[1][w] = ex; sh[2][w] = mx; sh[3][w] = dead;
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        unsigned long long v = sh[threadIdx.x][0];
        for (int w = 1; w < kStatThreads / 32; w++)
            v = threadIdx.x == 2 ? max(v, sh[2][w]) : v + sh[threadIdx.x][w];
        if (threadIdx.x == 2) atomicMax(&st[2], v);
        else if (v) atomicAdd(&st[threadIdx.x], v);
    }
}

}  // namespace

// Exclusive prefix sum of m counts into d_out[m + 1]; bsum: scratch of one word per block.
static int scan_counts(mg_ctx *ctx, const int32_t *d_cnt, int64_t m, int64_t *d_out, int64_t *bsum) {
    const int64_t nb = (m + kScanBlock - 1) / kScanBlock;
    k_scan_blocks<<<(unsigned)nb, kScanBlock, 0, ctx->stream>>>(d_cnt, m, bsum);
    k_scan_sums<<<1, kScanBlock, 0, ctx->stream>>>(bsum, nb);
    k_scan_apply<<<(unsigned)nb, kScanBlock, 0, ctx->stream>>>(d_cnt, m, bsum, d_out);
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

__global__ void k_posf(int64_t n, const double *__restrict__ pos, const int64_t *__restrict__ nbr_off,
                       const int32_t *__restrict__ nbr_idx, float4 *__restrict__ posf) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    auto at = [&](int64_t c) { return make_float3((float)pos[3 * c], (float)pos[3 * c + 1], (float)pos[3 * c + 2]); };
    auto size = [](const float3 p) { return fabsf(p.x) + fabsf(p.y) + fabsf(p.z); };
    const float3 p = at(i);
    // (as bits: non-negative floats order like them, and a NaN is the largest)
    unsigned m = __float_as_uint(size(p)) & 0x7fffffffu;
    for (int64_t e = nbr_off[i]; e < nbr_off[i + 1]; e++) m = max(m, __float_as_uint(size(at(nbr_idx[e]))) & 0x7fffffffu);
    posf[i] = make_float4(p.x, p.y, p.z, __uint_as_float(m));
}

// Stream-ordered pool for a trace's scratch, one per device: allocating and freeing up to
// gigabytes at every trace cost 1 ms of a 5.3 ms trace of 20k points. It keeps at most 1 GiB
// between traces (the release threshold; the rest goes back at the next synchronisation)
// and is given back with the device's last context. CUDA orders a block's reuse after the
// work that used it, on whatever streams and threads.
constexpr int kPoolDevices = 64;
static std::mutex g_pool_mu;
static cudaMemPool_t g_pool[kPoolDevices] = {};
static int g_pool_refs[kPoolDevices] = {};

void mg_pool_retain(int device) {
    if (device < 0 || device >= kPoolDevices) return;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (g_pool_refs[device]++ > 0) return;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    unsigned long long keep = 1ull << 30;
    if (cudaMemPoolCreate(&g_pool[device], &props) != cudaSuccess) {
        g_pool[device] = nullptr;   // plain allocations then
    } else if (cudaMemPoolSetAttribute(g_pool[device], cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaMemPoolDestroy(g_pool[device]);
        g_pool[device] = nullptr;
    }
    cudaGetLastError();
}

void mg_pool_release(int device) {
    if (device < 0 || device >= kPoolDevices) return;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (--g_pool_refs[device] > 0) return;
    if (g_pool[device]) cudaMemPoolDestroy(g_pool[device]);
    g_pool[device] = nullptr;
}

// Temporaries of one trace, given back on every return (in stream order, or by cudaFree,
// which waits for the kernels that may still use them).
struct TraceScratch {
    mg_ctx *ctx;
    cudaMemPool_t pool;
    std::vector<void *> held;
    explicit TraceScratch(mg_ctx *c) : ctx(c), pool(nullptr) {
        if (c->device >= 0 && c->device < kPoolDevices) {
            std::lock_guard<std::mutex> lk(g_pool_mu);
            pool = g_pool[c->device];
        }
    }
    cudaError_t take(void **q, size_t bytes) {
        return pool ? cudaMallocFromPoolAsync(q, bytes, pool, ctx->stream) : cudaMalloc(q, bytes);
    }
    template <typename T>
    cudaError_t get(T **p, size_t count) {
        void *q = nullptr;
        const size_t bytes = std::max<size_t>(1, count) * sizeof(T);
        cudaError_t e = take(&q, bytes);
        if (e != cudaSuccess && mg_release_idle_rays(ctx)) e = take(&q, bytes);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return e;
        }
        held.push_back(q);
        *p = static_cast<T *>(q);
        return e;
    }
    void give_back() {
        for (void *q : held) {
            if (pool) cudaFreeAsync(q, ctx->stream);
            else cudaFree(q);
        }
        held.clear();
    }
    ~TraceScratch() { give_back(); }
};

template <typename T>
static int ray_buffer(mg_ctx *ctx, T **p, int64_t &cap, int64_t count) {
    return kept_buffer(cap, count, [&](int64_t n) { return mg_alloc(ctx, p, n); });
}

int mg_launch_trace(mg_ctx *ctx) {
    const int64_t nr = ctx->n * ctx->R;
    int rc;
    TraceScratch sc(ctx);
    int32_t *d_len = nullptr, *d_xlen = nullptr, *d_tmp = nullptr;
    float4 *posf = nullptr;
    int64_t *bsum = nullptr;
    cudaError_t ce;
    if ((ce = sc.get(&d_len, nr)) || (ce = sc.get(&d_xlen, nr)) ||
        (ce = sc.get(&bsum, (nr + kScanBlock - 1) / kScanBlock)) ||
        (ctx->geometry == MG_GEOM_3D && (ce = sc.get(&posf, ctx->n))))
        return mg_fail(ctx, MG_ERR_OOM, std::string("cudaMalloc failed: ") + cudaGetErrorString(ce));
    // The ray store is written in place: solves and images of the old rays come first. Those
    // of this stream do; after a change of stream, wait for all (as the frees of a replaced
    // store do).
    if (ctx->stream_changed) MG_CUDA(cudaDeviceSynchronize());
    ctx->stream_changed = false;
    ctx->traced = false;
    struct InUse {           // the store is this trace's until it returns, and then the rays' if it succeeded
        mg_ctx *c;
        explicit InUse(mg_ctx *ctx) : c(ctx) { c->rays_idle = false; }
        ~InUse() { c->rays_idle = !c->traced; }
    } in_use(ctx);
    if ((rc = ray_buffer(ctx, &ctx->d_ray_off, ctx->ray_off_cap, nr + 1))) return rc;
    MG_CUDA(cudaMemsetAsync(ctx->d_err, 0, sizeof(int32_t), ctx->stream));
    TraceArgs a{};
    a.n = ctx->n; a.R = ctx->R; a.geometry = ctx->geometry;
    a.pos = ctx->d_pos; a.vel = ctx->d_vel; a.b = ctx->d_b; a.dirs = ctx->d_dirs;
    a.nbr_off = ctx->d_nbr_off; a.nbr_idx = ctx->d_nbr_idx; a.bdy = ctx->d_bdy;
    a.dshift_frac = ctx->opt.dshift_frac; a.max_steps = ctx->opt.max_steps;
    a.len = d_len; a.xlen = d_xlen; a.err = ctx->d_err;
    if (ctx->geometry == MG_GEOM_3D)
        k_posf<<<(unsigned)((ctx->n + 127) / 128), 128, 0, ctx->stream>>>(ctx->n, ctx->d_pos, ctx->d_nbr_off,
                                                                         ctx->d_nbr_idx, posf);
    a.posf = posf;
    // Record up to cap_tmp cells per half-ray in the count pass, in scratch of at most
    // 32 GiB and a quarter of the free device memory (given back after tracing; half-rays with
    // more cells, or all of them without scratch, are walked again by the fill pass).
    int32_t cap_tmp = 128;
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
        cudaGetLastError();
        free_b = 0;
    }
    const double budget = std::min(32.0 * (1 << 30), 0.25 * (double)free_b);
    while (cap_tmp > 0 && (double)nr * cap_tmp * 4.0 > budget) cap_tmp /= 2;
    if (ctx->geometry == MG_GEOM_3D && cap_tmp > 0) sc.get(&d_tmp, (size_t)nr * cap_tmp);
    a.tmp = d_tmp;
    a.cap_tmp = d_tmp ? cap_tmp : 0;
    const int bs = 128;
    const unsigned grid = (unsigned)((nr + bs - 1) / bs);
    {
        MgTimed t(ctx, "trace_count");
        k_trace<false><<<grid, bs, 0, ctx->stream>>>(a);
    }
    MG_CUDA(cudaGetLastError());
    if ((rc = scan_counts(ctx, d_len, nr, ctx->d_ray_off, bsum))) return rc;
    int64_t total = 0;
    int32_t kerr = 0;
    MG_CUDA(cudaMemcpyAsync(&total, ctx->d_ray_off + nr, 8, cudaMemcpyDeviceToHost, ctx->stream));
    MG_CUDA(cudaMemcpyAsync(&kerr, ctx->d_err, 4, cudaMemcpyDeviceToHost, ctx->stream));
    MG_CUDA(cudaStreamSynchronize(ctx->stream));
    if (kerr) {
        return mg_fail(ctx, MG_ERR_CAPACITY, "ray tracing: a half-ray exceeded max_steps");
    }
    auto store = [&]() {
        int64_t *c = ctx->ray_cap;
        return ray_buffer(ctx, &ctx->d_cells, c[0], total) || ray_buffer(ctx, &ctx->d_xcum, c[1], total) ||
               ray_buffer(ctx, &ctx->d_ds, c[2], total) || ray_buffer(ctx, &ctx->d_vpar, c[3], total) ||
               ray_buffer(ctx, &ctx->d_dsf, c[4], total) || ray_buffer(ctx, &ctx->d_vparf, c[5], total);
    };
    if (store()) {           // once more without what the buffers held before
        mg_free(ctx->d_cells); mg_free(ctx->d_xcum); mg_free(ctx->d_ds);
        mg_free(ctx->d_vpar); mg_free(ctx->d_dsf); mg_free(ctx->d_vparf);
        for (int64_t &c : ctx->ray_cap) c = 0;
        if (store()) return MG_ERR_OOM;
    }
    a.ray_off = ctx->d_ray_off; a.cells = ctx->d_cells; a.xcum = ctx->d_xcum; a.ds = ctx->d_ds; a.vpar = ctx->d_vpar;
    a.dsf = ctx->d_dsf; a.vparf = ctx->d_vparf;
    {
        MgTimed t(ctx, "trace_fill");
        k_trace<true><<<grid, bs, 0, ctx->stream>>>(a);
    }
    MG_CUDA(cudaGetLastError());
    MG_CUDA(cudaMemsetAsync(ctx->d_scal, 0, 4 * sizeof(unsigned long long), ctx->stream));
    k_ray_stats<<<kStatBlocks, kStatThreads, 0, ctx->stream>>>(ctx->n, ctx->R, ctx->P, ctx->d_pf, ctx->d_pb, d_len, d_xlen,
                                                              ctx->d_scal);
    MG_CUDA(cudaGetLastError());
    unsigned long long st[4];
    MG_CUDA(cudaMemcpyAsync(st, ctx->d_scal, sizeof(st), cudaMemcpyDeviceToHost, ctx->stream));
    sc.give_back();   // before the synchronisation, at which the pool lets go of what it does not keep
    MG_CUDA(cudaStreamSynchronize(ctx->stream));
    ctx->n_elements = (int64_t)st[0];
    ctx->n_expanded = (int64_t)st[1];
    ctx->max_pair_len = (int64_t)st[2];
    ctx->n_dead = (int64_t)st[3];
    ctx->traced = true;
    return MG_OK;
}
