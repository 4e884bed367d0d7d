// K3 in mixed precision: the Feautrier formal solve of Sec. 3.3-3.4 in FP32 (the
// statistical equilibrium that follows stays in FP64). Intensities are carried in units
// of I0 = 1e-20 W m^-2 Hz^-1 sr^-1 and the float line data are scaled (chi x 1e5,
// eta x 1e25) so that no FP32 quantity underflows. The line opacity of bin a_q at a point
// is chi_l = X 2^(-x'^2), with X = chi_int c / (nu_l b sqrt(pi)) and the profile
// argument x' in units of sqrt(log2 e) Doppler widths; for a line that overlaps no other
// line the source function S = eta_int/chi_int is frequency independent.
//
// Two kernels:
// - k_feautrier_warp (the common case: lines that do not overlap) gives each warp one
//   origin and a group of G lines, with the bins of those lines across its lanes (NB
//   per lane), and sweeps every ray pair through a per-warp ring of staged points; the
//   persistent k_feautrier_batch runs the same work item over a queue of models.
// - k_feautrier_mixed (lines that overlap, so that a bin sums several lines) gives each
//   origin a CTA and stages every ray pair whole in shared memory.
//
// Per point and bin the sweep costs one ex2 and one rcp (MUFU) and a handful of FMA-
// and ALU-pipe ops, in the rescaled Rybicki-Hummer recursion described with the FP64
// kernel:
//   dtau = max((chi_prev + chi) ds/2, dtau_min),  t = (dtau_prev + dtau)/2,
//   Phi = t + Phi iota,  iota = 1/(1 + dtau Phi),  psi = (t S + psi) iota.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include "common.cuh"

using namespace mg;

namespace {

constexpr float kSqrtLog2e = 1.2011224087864498f;
constexpr float kSqrt2 = 1.4142135623730951f;
constexpr float kInvSqrt8 = 0.35355339059327373f;   // 1/(2 sqrt 2)
constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcpf(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Line data of one or several models (blockIdx.y), arguments by value.
struct LineArgs {
    int64_t n;
    int L, nlev;
    const double *pops;
    const LineConst *lc;
    double *line;
    float *linef;
    unsigned long long *scal;   // [4]: negative line opacities
};
constexpr int kLineBatch = 48;
struct LineBatch {
    LineArgs m[kLineBatch];
};
static_assert(sizeof(LineBatch) <= 4096, "kernel parameter size");

__global__ void k_line_data_f32(const __grid_constant__ LineBatch b) {
    const LineArgs &a = b.m[blockIdx.y];
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.n * a.L) return;
    const int64_t c = t / a.L;
    const int l = (int)(t - c * a.L);
    const LineConst k = a.lc[l];
    const double nu_ = a.pops[c * a.nlev + k.up], nl_ = a.pops[c * a.nlev + k.lo];
    const double eta = k.pre * nu_ * k.A;
    const double chi = k.pre * (nl_ * k.Blu - nu_ * k.Bul);
    a.line[2 * t] = eta;
    a.line[2 * t + 1] = chi;
    if (chi < 0.0) atomicAdd(a.scal + 4, 1ull);
    // (eta, chi) times the profile normalisation c / (nu_l sqrt(pi)): the line opacity of a
    // bin is then chi' 2^(-x'^2) / b, and S = eta'/chi' keeps the scale kEtaScale/kChiScale
    const double kl = kC / (k.nu * kSqrtPi);
    a.linef[2 * t] = (float)(eta * (kEtaScale / kChiScale) * kl);
    a.linef[2 * t + 1] = (float)(chi * kl);
}

// Clears the words that a batch's line data ([4]) and population update ([0..2]) count in.
struct ScalBatch {
    unsigned long long *scal[256];
};
__global__ void k_clear_words(const __grid_constant__ ScalBatch b, int count, int update) {
    const int m = threadIdx.x;
    if (m >= count) return;
    b.scal[m][4] = 0;
    if (update) b.scal[m][0] = b.scal[m][1] = b.scal[m][2] = 0;
}

struct MixArgs {
    int64_t n;
    int32_t R, P, L, Q;
    const int32_t *pf, *pb;
    const int64_t *ray_off;
    const int32_t *cells, *xcum;
    const float *ds, *vpar, *b;
    const float *line;           // [n][L][2] (eta, chi) times c/(nu_l sqrt(pi)), eta also times kEtaScale/kChiScale
    const float *nu_ghz;         // [L]
    const double *roots, *weights;
    const int32_t *ovl_off;
    const Overlap *ovl;
    float chi_min, dtau_min, inv_chi_min;
    float delta_min;             // dtau_min / sqrt 2
    float q_nofloor;             // q' = chi_min ds/(2 sqrt 2) from which 2 q' >= delta_min in FP32
    float qscale;                // chi_min/(2 sqrt 2): q' of an interval per unit length
    float planck_a, planck_b;    // B'(nu) = a nu_G^3 / expm1(b nu_G): a = 2h 1e27/c^2/I0, b = h 1e9/(k T_cmb)
    double *J, *Lout, *Jeff, *Lc, *Jnu;
    int32_t kmax;
    int32_t overlap;             // some line overlaps another
    int32_t skip;                // leave out far points
    int32_t *err;
    unsigned long long *work;    // optional: point-bin updates the warp kernel executed
};

__device__ __forceinline__ float planck_f(const MixArgs &a, float nu_g) {
    return a.planck_a * nu_g * nu_g * nu_g / expm1f(a.planck_b * nu_g);
}

// CTA kernel (overlapping lines). Stages half-ray (o, r) in FP32, point x of the half at
// pair index base + dir x:
//   pt[k]    = (ds_k / 2, v_k, sqrt(log2 e)/b_k, 0)
//   ln[k][l] = (X_l, S_l) of every line l.
__device__ void stage_half32(const MixArgs &a, int64_t o, int r, int base, int dir, float4 *pt, float2 *ln) {
    const int L = a.L;
    const int64_t off = a.ray_off[o * a.R + r];
    const int len = (int)(a.ray_off[o * a.R + r + 1] - off);
    for (int e = threadIdx.x; e < len; e += blockDim.x) {
        const int64_t c = a.cells[off + e];
        const int64_t prev = e ? a.cells[off + e - 1] : o;
        const int x0 = e ? a.xcum[off + e - 1] : 0;
        const int ns = a.xcum[off + e] - x0 - 1;
        const float pv = e ? a.vpar[off + e - 1] : 0.0f;
        const float ve = a.vpar[off + e];
        const float hds = 0.5f * a.ds[off + e] / (float)(ns + 1);
        const float bp = a.b[prev], bc = a.b[c];
        const float2 *lp = reinterpret_cast<const float2 *>(a.line) + prev * L;
        const float2 *lq = reinterpret_cast<const float2 *>(a.line) + c * L;
        for (int j = 1; j <= ns + 1; j++) {
            const float w = (float)j / (float)(ns + 1);
            const int idx = base + dir * (x0 + j - 1);
            const float bb = (1.0f - w) * bp + w * bc;
            const float ib = 1.0f / bb;
            // the path length is stored with the point farther from the origin
            pt[idx] = make_float4(hds, (1.0f - w) * pv + w * ve, kSqrtLog2e * ib, 0.0f);
            for (int l = 0; l < L; l++) {
                const float2 p0 = lp[l], p1 = lq[l];
                const float et = (1.0f - w) * p0.x + w * p1.x;
                const float ch = (1.0f - w) * p0.y + w * p1.y;
                const float X = ch * ib;
                const float S = ch > 0.0f ? et / ch : 0.0f;
                ln[(size_t)idx * L + l] = make_float2(X, S);
            }
        }
    }
}

struct Side32 {
    float phi_iota, psi, dtau;
};

// Opacity and emissivity at point k for bin (l, aq); fast path: line l alone.
template <bool OVL>
__device__ __forceinline__ void point32(const MixArgs &a, int l, float aq, float A1, int k, const float4 *pt,
                                        const float2 *ln, float &chi, float &S, float &chil, float &etal) {
    const float4 p = pt[k];
    if (!OVL) {
        const float2 d = ln[(size_t)k * a.L + l];
        const float x = fmaf(-p.y, A1, aq) * p.z;
        const float e = ex2f(-x * x);
        chil = d.x * e;
        etal = chil * d.y;
        if (chil >= a.chi_min) {
            chi = chil;
            S = d.y;
        } else {   // opacity floor: S = eta / chi_min
            chi = a.chi_min;
            S = etal * a.inv_chi_min;
        }
        return;
    }
    // general case: sum over the lines that can reach this bin
    float ch = 0.f, et = 0.f;
    const int o0 = a.ovl_off[l], o1 = a.ovl_off[l + 1];
    const float base = fmaf(-p.y, A1, aq);
    for (int i = o0; i < o1; i++) {
        const Overlap ov = a.ovl[i];
        const float2 d = ln[(size_t)k * a.L + ov.l2];
        const float x = ((float)ov.dnl + (float)ov.rat * base) * p.z;
        const float c2 = d.x * ex2f(-x * x);
        ch += c2;
        et += c2 * d.y;
        if (i == o0) { chil = c2; etal = c2 * d.y; }
    }
    chi = fmaxf(ch, a.chi_min);
    S = et / chi;
}

template <bool OVL>
__device__ __forceinline__ Side32 sweep32(const MixArgs &a, int l, float aq, float A1, float nu_og, int kstart,
                                          int kend, int step, const float4 *pt, const float2 *ln, float &chi_o,
                                          float &S_o, float &chil_o, float &etal_o) {
    float chi_p, S_p, cl, el;
    point32<OVL>(a, l, aq, A1, kstart, pt, ln, chi_p, S_p, cl, el);
    const float I = planck_f(a, nu_og * (1.0f - pt[kstart].y * (float)(1.0 / kC)));
    float Phi, iota, psi, dt_p;
    // boundary row (first interval)
    {
        const int k = kstart + step;
        float chi, S;
        point32<OVL>(a, l, aq, A1, k, pt, ln, chi, S, cl, el);
        const float hds = pt[kstart].x;   // interval (kstart, k): stored with the farther point
        const float dt = fmaxf((chi_p + chi) * hds, a.dtau_min);
        Phi = fmaf(0.5f, dt, 1.0f);
        iota = rcpf(fmaf(dt, Phi, 1.0f));
        psi = fmaf(0.5f * dt, S_p, I) * iota;
        dt_p = dt;
        chi_p = chi;
        S_p = S;
        if (k == kend) {
            chi_o = chi; S_o = S; chil_o = cl; etal_o = el;
            return Side32{Phi * iota, psi, dt_p};
        }
    }
    for (int k = kstart + 2 * step;; k += step) {
        float chi, S;
        point32<OVL>(a, l, aq, A1, k, pt, ln, chi, S, cl, el);
        const float hds = pt[k - step].x;
        const float dt = fmaxf((chi_p + chi) * hds, a.dtau_min);
        const float t = 0.5f * (dt_p + dt);
        Phi = fmaf(Phi, iota, t);
        iota = rcpf(fmaf(dt, Phi, 1.0f));
        psi = fmaf(t, S_p, psi) * iota;
        dt_p = dt;
        chi_p = chi;
        S_p = S;
        if (k == kend) {
            chi_o = chi; S_o = S; chil_o = cl; etal_o = el;
            break;
        }
    }
    return Side32{Phi * iota, psi, dt_p};
}

// Shared memory of the CTA kernel: pt [kmax] float4, ln [kmax][L] float2, then acc
// [L][Q] float4 at the next 16-byte boundary.
__host__ __device__ constexpr size_t mixed_acc_offset(int kmax, int L) {
    return (16 * (size_t)kmax + 8 * (size_t)kmax * L + 15) & ~(size_t)15;
}
static_assert(mixed_acc_offset(3, 3) % 16 == 0 && mixed_acc_offset(3, 3) >= 16 * 3 + 8 * 9, "acc alignment");
static_assert(mixed_acc_offset(4, 2) == 16 * 4 + 8 * 8, "no padding when kmax * L is even");

template <bool OVL>
__global__ void __launch_bounds__(256) k_feautrier_mixed(MixArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = a.L, Q = a.Q;
    const int kmax = a.kmax;
    float4 *pt = reinterpret_cast<float4 *>(smem_raw);
    float2 *ln = reinterpret_cast<float2 *>(pt + kmax);
    // [L*Q]: (sum u, L, Jeff, 1-L); starts on a 16-byte boundary (kmax * L may be odd)
    float4 *acc = reinterpret_cast<float4 *>(smem_raw + mixed_acc_offset(kmax, L));
    const int64_t o = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    for (int f = threadIdx.x; f < L * Q; f += blockDim.x) acc[f] = make_float4(0.f, 0.f, 0.f, 0.f);
    const float bo = a.b[o];
    const float2 *lo = reinterpret_cast<const float2 *>(a.line) + o * L;
    for (int p = 0; p < a.P; p++) {
        const int rf = a.pf[p], rb = a.pb[p];
        const int64_t ofb = a.ray_off[o * a.R + rb], ofl = a.ray_off[o * a.R + rf];
        const int lb = (int)(a.ray_off[o * a.R + rb + 1] - ofb);
        const int lf = (int)(a.ray_off[o * a.R + rf + 1] - ofl);
        const int Kb = lb ? a.xcum[ofb + lb - 1] : 0;
        const int Kf = lf ? a.xcum[ofl + lf - 1] : 0;
        const int K = Kb + 1 + Kf;
        if (K > kmax) {
            if (threadIdx.x == 0) atomicOr(a.err, 2);
            continue;
        }
        __syncthreads();
        stage_half32(a, o, rb, Kb - 1, -1, pt, ln);
        stage_half32(a, o, rf, Kb + 1, +1, pt, ln);
        if (threadIdx.x == 0) pt[Kb] = make_float4(0.f, 0.f, kSqrtLog2e / bo, 0.f);
        for (int l = threadIdx.x; l < L; l += blockDim.x) {
            const float2 d = lo[l];
            const float X = d.y / bo;
            ln[(size_t)Kb * L + l] = make_float2(X, d.y > 0.f ? d.x / d.y : 0.f);
        }
        __syncthreads();
        for (int l = warp; l < L; l += nwarps) {
            const float nu_g = a.nu_ghz[l];
            for (int q = lane; q < Q; q += 32) {
                const float aq = (float)(a.roots[q] * a.b[o]);
                const float A1 = 1.0f + aq * (float)(1.0 / kC);
                const float nu_og = nu_g * A1;
                float u, lam, uml, oml, chi_o = 0.f, S_o = 0.f, chil = 0.f, etal = 0.f;
                if (K == 1) {
                    const float I = planck_f(a, nu_og);
                    point32<OVL>(a, l, aq, A1, Kb, pt, ln, chi_o, S_o, chil, etal);
                    u = I; lam = 0.f; uml = I; oml = 1.f;
                } else {
                    Side32 sb{1.f, 0.f, 0.f}, sf{1.f, 0.f, 0.f};
                    if (Kb > 0) sb = sweep32<OVL>(a, l, aq, A1, nu_og, 0, Kb, +1, pt, ln, chi_o, S_o, chil, etal);
                    if (Kf > 0) sf = sweep32<OVL>(a, l, aq, A1, nu_og, K - 1, Kb, -1, pt, ln, chi_o, S_o, chil, etal);
                    if (Kb == 0 || Kf == 0) {
                        const float Io = planck_f(a, nu_og);
                        if (Kb == 0) sb.psi = Io;
                        if (Kf == 0) sf.psi = Io;
                    }
                    const float sig = 2.0f / (sb.dtau + sf.dtau);
                    const float pi2 = sb.phi_iota + sf.phi_iota;
                    const float iD = 1.0f / fmaf(sig, pi2, 1.0f);
                    const float ps = sig * (sb.psi + sf.psi);
                    u = (S_o + ps) * iD;
                    lam = iD;
                    uml = ps * iD;
                    oml = sig * pi2 * iD;
                }
                const float ichi = 1.0f / chi_o;
                const float eta_o = S_o * chi_o;
                float4 r = acc[l * Q + q];
                r.x += u;
                r.y += lam * chil * ichi;
                r.z += uml + lam * (eta_o - etal) * ichi;
                r.w += oml + lam * (chi_o - chil) * ichi;
                acc[l * Q + q] = r;
            }
        }
    }
    __syncthreads();
    // per-line weighted sums over bins, fixed order, in FP64
    const double invP = 1.0 / a.P;
    for (int t = threadIdx.x; t < 4 * L; t += blockDim.x) {
        const int l = t >> 2, k = t & 3;
        double s = 0.0;
        for (int q = 0; q < Q; q++) {
            const float4 r = acc[l * Q + q];
            const float v = k == 0 ? r.x : (k == 1 ? r.y : (k == 2 ? r.z : r.w));
            s += a.weights[q] * (double)v;
        }
        s *= invP;
        if (k == 0 || k == 2) s *= (double)kI0;
        double *dst = k == 0 ? a.J : (k == 1 ? a.Lout : (k == 2 ? a.Jeff : a.Lc));
        dst[o * L + l] = s;
    }
    if (a.Jnu)
        for (int f = threadIdx.x; f < L * Q; f += blockDim.x) a.Jnu[o * L * Q + f] = (double)acc[f].x * invP * (double)kI0;
}


// ---------------------------------------------------------------------------------
// Warp-per-(origin, line group) variant for models whose lines do not overlap (the
// common case). A warp serves G lines and every lane NB (line, bin) results (BinLanes and
// LineLanes below), so each shared-memory read and loop step is shared by NB updates.
// The warp loops over all ray pairs of its origin and stages the expanded points through
// a private ring of kRing points (one point per lane per refill): no CTA barrier is ever
// needed, and the pair sums are kept per lane in a fixed order. The boundary row is the
// interior update started from the virtual state (Phi iota = 1, psi = I, dtau = 0).
// The opacity floor: chi = max(chi_l, chi_min) and S_eff = S min(chi_l/chi_min, 1),
// which is eta/chi with chi floored. The warp kernel carries opacities in units of
// chi_min (and the interval factor q times chi_min, so that dtau is unchanged): the floor
// is then max(chi', 1) and the source's min(chi', 1), with no multiplication by
// 1/chi_min per bin.
//
// The ray elements behind the ring come from an element window in shared memory (one
// element per lane). A window serves refills until its points are used up; meanwhile
// the next window is filled asynchronously (cp.async): its records (xcum, cell, v, ds)
// are issued on the first refill from the current window, and the gathers through the
// cell index (b and the line data) half-way through that refill's sweep, so a window is
// normally complete when it is needed. The last window of a half-ray prefetches the
// first window of the next half-ray.
constexpr int kRing = 32;
constexpr int kWarps2 = 4;   // warps per block of most launch variants
constexpr int kWin = 32;   // elements top, top-1, ..., top-31 of a half-ray

// Element window of one warp, double-buffered: one slot per lane. Element e of the
// half-ray sits at slot top - e; element -1 (reached when top < 31) is the origin itself:
// xcum 0, cell o, v 0. Slots 0 .. 30 own the points of a refill; slot 31 only serves as
// the predecessor (towards the origin) of slot 30.
template <int G>
struct ElemWin {
    int32_t x1[2][kWin];      // xcum[e]: the element's expanded points are xcum[e-1] .. xcum[e]-1
    int32_t cell[2][kWin];
    float ds[2][kWin];
    float2 vb[2][kWin];        // (line-of-sight velocity, width b) of the element's cell
    float2 ln[2][G][kWin];    // scaled (eta, chi) of the warp's lines at the element's cell
};

__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Issues the copies of the records of elements top .. top-31 of the half-ray at `off`
// into buffer bf (lane i: slot i).
template <int G>
__device__ __forceinline__ void win_records(const MixArgs &a, int64_t off, int top, int32_t o, ElemWin<G> &w,
                                            int bf) {
    const int i = threadIdx.x & 31;
    const int e = top - i;
    if (e >= 0) {
        const int64_t k = off + e;
        cp_async4(&w.x1[bf][i], a.xcum + k);
        cp_async4(&w.cell[bf][i], a.cells + k);
        cp_async4(&w.vb[bf][i].x, a.vpar + k);
        cp_async4(&w.ds[bf][i], a.ds + k);
    } else {
        w.x1[bf][i] = 0;
        w.cell[bf][i] = o;
        w.vb[bf][i].x = 0.0f;
        w.ds[bf][i] = 0.0f;
    }
    cp_async_commit();
}

// Issues the gathers through the cell index of buffer bf; the records must have landed
// (each lane reads only the slots it copied itself).
template <int G>
__device__ __forceinline__ void win_gathers(const MixArgs &a, int l0, ElemWin<G> &w, int bf) {
    const int i = threadIdx.x & 31;
    const int64_t c = w.cell[bf][i];
    cp_async4(&w.vb[bf][i].y, a.b + c);
    const float2 *lc = reinterpret_cast<const float2 *>(a.line) + c * a.L;
#pragma unroll
    for (int k = 0; k < G; k++) cp_async8(&w.ln[bf][k][i], lc + (l0 + k < a.L ? l0 + k : a.L - 1));
    cp_async_commit();
}

// Scalars of the sweep, held in registers (not re-read from the argument block).
struct SweepK {
    float dmin;              // floor of delta = dtau/sqrt 2
    float planck_a, planck_b;
};

// B_nu / I0 at nu_g GHz; e^x - 1 from one ex2 (x = h nu / k T_cmb is O(1) at line
// frequencies, so the subtraction costs no precision there).
__device__ __forceinline__ float planck_k(const SweepK &k, float nu_g) {
    return k.planck_a * nu_g * nu_g * nu_g * rcpf(ex2f(k.planck_b * kLog2e * nu_g) - 1.0f);
}

// One staged point of the ring. The per-point scalars are stored twice so that a bin
// pair reads them as the operand pairs of packed FP32x2 arithmetic:
//   a = (g_z, g_z, -g_y, -g_y) with g_y = sqrt(log2 e) v/b and g_z = sqrt(log2 e)(1 - v/c)/b,
//       so that the profile argument of bin a_q is x' = a_q g_z - g_y;
//   q = (q', q') with q' = chi_min ds/(2 sqrt 2) of the interval from the adjacent point
//       away from the origin (the half-width interval factor that yields delta =
//       dtau/sqrt 2 from opacities in units of chi_min).
// The line data of a point are (X', X', S, S) per line, X' = X/chi_min: the line opacity
// in units of chi_min is chi' = X' 2^(-x'^2), the floored opacity max(chi', 1), and the
// floored source S_eff = S min(chi', 1), which is eta/chi with chi = max(chi_l, chi_min)
// (exactly S where the line is not floored; finite for any finite S).
struct Ring {
    float4 a[kRing];
    float2 q[kRing];
    int4 own[kRing];   // per element with points to sweep: (slot, first point + its position, x0, points)
};

// Expanded point x (sub-point j = x - x0 + 1 of np of the interval from slot i + 1, the
// element's predecessor towards the origin, to slot i, its own cell): geometry part.
struct PointGeo {
    float gz, gy, ib;
    float2 w0, w1;
};
template <int G>
__device__ __forceinline__ PointGeo point_geometry(const ElemWin<G> &w, int bf, int i, int j, int np) {
    // exactly 1 at the element's own cell, so that a thick neighbour cannot leak into it
    const float wt = j == np ? 1.0f : (float)j * rcpf((float)np);
    PointGeo p;
    // interpolations (1 - w) p0 + w p1 in packed pairs; w = 1 gives p1 exactly
    p.w1 = make_float2(wt, wt);
    p.w0 = make_float2(1.0f - wt, 1.0f - wt);
    const float2 vbi = __ffma2_rn(p.w1, w.vb[bf][i], __fmul2_rn(p.w0, w.vb[bf][i + 1]));
    p.ib = rcpf(vbi.y);
    const float pz = kSqrtLog2e * p.ib;
    p.gy = vbi.x * pz;
    p.gz = (1.0f - vbi.x * (float)(1.0 / kC)) * pz;
    return p;
}

// Line part: (X', S) of the warp's G lines; returns the largest X'.
template <int G>
__device__ __forceinline__ float point_lines(const MixArgs &a, const ElemWin<G> &w, int bf, int i, const PointGeo &p,
                                             float2 (&out)[G]) {
    const float ibc = p.ib * a.inv_chi_min;
    float Xmax = 0.0f;
#pragma unroll
    for (int k = 0; k < G; k++) {
        const float2 e = __ffma2_rn(p.w1, w.ln[bf][k][i], __fmul2_rn(p.w0, w.ln[bf][k][i + 1]));   // (eta, chi)
        const float X = fmaxf(e.y, 0.0f) * ibc;
        // (a line whose opacity is below the smallest normal float has no source here)
        const float S = e.y >= 1.17549435e-38f ? e.x * rcpf(e.y) : 0.0f;
        out[k] = make_float2(X, S);
        Xmax = fmaxf(Xmax, X);
    }
    return Xmax;
}

// Per-bin sweep state in the variables delta = dtau/sqrt 2, Phi^ = sqrt 2 Phi and
// psi^ = sqrt 2 psi, in which the recursion carries no factor 1/2:
//   s = delta_prev + delta,  Phi^ = s + Phi^_prev iota_prev,  iota = 1/(1 + delta Phi^),
//   psi^ = (s S_prev + psi^_prev) iota.
// Bins 2p and 2p+1 of a lane form pair p and are updated together with packed FP32x2
// arithmetic (fma/mul/add on float2); an odd last bin is updated alone.
template <int NB>
struct BinState {
    static constexpr int NP = NB / 2;
    static constexpr bool ODD = (NB & 1) != 0;
    float2 aq2[NP > 0 ? NP : 1], chi_p2[NP > 0 ? NP : 1], S_p2[NP > 0 ? NP : 1], d_p2[NP > 0 ? NP : 1];
    float2 Phi2[NP > 0 ? NP : 1], iota2[NP > 0 ? NP : 1], psi2[NP > 0 ? NP : 1];
    float aq1, chi_p1, S_p1, d_p1, Phi1, iota1, psi1;
    __device__ __forceinline__ float aq(int i) const {
        return i < 2 * NP ? ((i & 1) ? aq2[i >> 1].y : aq2[i >> 1].x) : aq1;
    }
    __device__ __forceinline__ void set_aq(int i, float v) {
        if (i < 2 * NP) {
            if (i & 1) aq2[i >> 1].y = v; else aq2[i >> 1].x = v;
        } else {
            aq1 = v;
        }
    }
};

__device__ __forceinline__ float2 ex2f2(const float2 t) { return make_float2(ex2f(-t.x), ex2f(-t.y)); }

// The far end of a half: the boundary row is the interior update from the virtual state
// Phi^ iota = sqrt 2, psi^ = sqrt 2 I, delta = 0.
template <int NB>
__device__ __forceinline__ void first_point(const SweepK &k, BinState<NB> &st, const float4 A, const float4 D,
                                            const float nu_g, const float v) {
    const float2 gz = make_float2(A.x, A.y), ngy = make_float2(A.z, A.w);
    const float2 X = make_float2(D.x, D.y), S = make_float2(D.z, D.w);
    const float dop = 1.0f - v * (float)(1.0 / kC);
#pragma unroll
    for (int p = 0; p < BinState<NB>::NP; p++) {
        const float2 x = __ffma2_rn(st.aq2[p], gz, ngy);
        const float2 chil = __fmul2_rn(X, ex2f2(__fmul2_rn(x, x)));
        st.chi_p2[p] = make_float2(fmaxf(chil.x, 1.0f), fmaxf(chil.y, 1.0f));
        st.S_p2[p] = __fmul2_rn(S, make_float2(fminf(chil.x, 1.0f), fminf(chil.y, 1.0f)));
        st.Phi2[p] = make_float2(kSqrt2, kSqrt2);
        st.iota2[p] = make_float2(1.0f, 1.0f);
        st.d_p2[p] = make_float2(0.0f, 0.0f);
        st.psi2[p] = make_float2(kSqrt2 * planck_k(k, nu_g * (1.0f + st.aq2[p].x * (float)(1.0 / kC)) * dop),
                                 kSqrt2 * planck_k(k, nu_g * (1.0f + st.aq2[p].y * (float)(1.0 / kC)) * dop));
    }
    if constexpr (BinState<NB>::ODD) {
        const float x = fmaf(st.aq1, gz.x, ngy.x);
        const float chil = X.x * ex2f(-x * x);
        st.chi_p1 = fmaxf(chil, 1.0f);
        st.S_p1 = S.x * fminf(chil, 1.0f);
        st.Phi1 = kSqrt2;
        st.iota1 = 1.0f;
        st.d_p1 = 0.0f;
        st.psi1 = kSqrt2 * planck_k(k, nu_g * (1.0f + st.aq1 * (float)(1.0 / kC)) * dop);
    }
}

// Update with the interval (previous point, this point); qp = (q, q) of that interval,
// A and D the point's ring entries. FLOOR = false drops the dtau floor where the caller
// knows that it cannot bind (q' >= q_nofloor): the result is the same bit for bit.
template <int NB, bool FLOOR = true>
__device__ __forceinline__ void step_point(const SweepK &k, BinState<NB> &st, const float4 A, const float4 D,
                                           const float2 qp) {
    const float2 gz = make_float2(A.x, A.y), ngy = make_float2(A.z, A.w);
    const float2 X = make_float2(D.x, D.y), S = make_float2(D.z, D.w);
#pragma unroll
    for (int p = 0; p < BinState<NB>::NP; p++) {
        const float2 x = __ffma2_rn(st.aq2[p], gz, ngy);
        const float2 chil = __fmul2_rn(X, ex2f2(__fmul2_rn(x, x)));
        const float2 chi = make_float2(fmaxf(chil.x, 1.0f), fmaxf(chil.y, 1.0f));
        const float2 Sx = __fmul2_rn(S, make_float2(fminf(chil.x, 1.0f), fminf(chil.y, 1.0f)));
        const float2 d0 = __fmul2_rn(__fadd2_rn(st.chi_p2[p], chi), qp);
        const float2 dl = FLOOR ? make_float2(fmaxf(d0.x, k.dmin), fmaxf(d0.y, k.dmin)) : d0;
        const float2 sm = __fadd2_rn(st.d_p2[p], dl);
        st.Phi2[p] = __ffma2_rn(st.Phi2[p], st.iota2[p], sm);
        const float2 den = __ffma2_rn(dl, st.Phi2[p], make_float2(1.0f, 1.0f));
        st.iota2[p] = make_float2(rcpf(den.x), rcpf(den.y));
        st.psi2[p] = __fmul2_rn(__ffma2_rn(sm, st.S_p2[p], st.psi2[p]), st.iota2[p]);
        st.d_p2[p] = dl;
        st.chi_p2[p] = chi;
        st.S_p2[p] = Sx;
    }
    if constexpr (BinState<NB>::ODD) {
        const float x = fmaf(st.aq1, gz.x, ngy.x);
        const float chil = X.x * ex2f(-x * x);
        const float chi = fmaxf(chil, 1.0f);
        const float Sx = S.x * fminf(chil, 1.0f);
        const float d0 = (st.chi_p1 + chi) * qp.x;
        const float dl = FLOOR ? fmaxf(d0, k.dmin) : d0;
        const float sm = st.d_p1 + dl;
        st.Phi1 = fmaf(st.Phi1, st.iota1, sm);
        st.iota1 = rcpf(fmaf(dl, st.Phi1, 1.0f));
        st.psi1 = fmaf(sm, st.S_p1, st.psi1) * st.iota1;
        st.d_p1 = dl;
        st.chi_p1 = chi;
        st.S_p1 = Sx;
    }
}

// (Phi^ iota, psi^, delta) of every bin.
template <int NB>
__device__ __forceinline__ void bin_results(const BinState<NB> &st, float (&pi)[NB], float (&ps)[NB],
                                            float (&dt)[NB]) {
#pragma unroll
    for (int p = 0; p < BinState<NB>::NP; p++) {
        const float2 pp = __fmul2_rn(st.Phi2[p], st.iota2[p]);
        pi[2 * p] = pp.x;
        pi[2 * p + 1] = pp.y;
        ps[2 * p] = st.psi2[p].x;
        ps[2 * p + 1] = st.psi2[p].y;
        dt[2 * p] = st.d_p2[p].x;
        dt[2 * p + 1] = st.d_p2[p].y;
    }
    if constexpr (BinState<NB>::ODD) {
        pi[NB - 1] = st.Phi1 * st.iota1;
        ps[NB - 1] = st.psi1;
        dt[NB - 1] = st.d_p1;
    }
}

// How the (line, bin) results of a warp lie on its lanes.
//
// BinLanes: G lane groups of 32/G lanes, a line each; a lane has NB bins of its line, swept in
// pairs of bins. It fits any number of bins to the lanes.
//
// LineLanes: a lane has the same NB/G bins (lane, lane + 32, ...) of all G lines, swept in
// pairs of lines. The profile argument a_q g_z - g_y and its exponential are the same for every
// line of a species (the bins are in Doppler widths), so they are computed once per bin
// for all G lines: per pair and point 9 packed ops, 2 rcp and 4 max/min, and per point and
// bin 2 ops, one ex2 and a copy, against 11 packed ops, 2 ex2, 2 rcp and 4 max/min per pair
// in BinLanes. Points of the ring carry (X, X, S, S) of a line pair without duplicates.
// Measured, BinLanes -> LineLanes: disc of 32k cells (19 lines x 63 bins, G = 4, NB = 8) 197.5 -> 180.6 ms;
// clumpy 50k (4 x 31, G = 4, NB = 4) 9.07 -> 8.69 ms.
template <int G_, int NB_>
struct BinLanes {
    static constexpr int G = G_, NB = NB_, LPG = 32 / G, kRingLines = G;
    BinState<NB> st;
    float nu_g;
    float4 Do;              // the origin's line data
    int grp;

    __device__ __forceinline__ int line(int) const { return grp; }
    __device__ __forceinline__ int bin(int i) const { return (threadIdx.x & 31) - grp * LPG + LPG * i; }
    __device__ __forceinline__ float aq(int i) const { return st.aq(i); }
    __device__ __forceinline__ void init(const MixArgs &a, int64_t o, int l0, float bo, float ibo) {
        grp = (threadIdx.x & 31) / LPG;
        const int lc = l0 + grp < a.L ? l0 + grp : a.L - 1;
        nu_g = a.nu_ghz[lc];
        const float2 dl = reinterpret_cast<const float2 *>(a.line)[o * a.L + lc];
        const float Xo = fmaxf(dl.y, 0.0f) * (ibo * a.inv_chi_min);   // in units of chi_min
        const float So = dl.y > 0.0f ? dl.x / dl.y : 0.0f;
        Do = make_float4(Xo, Xo, So, So);
#pragma unroll
        for (int i = 0; i < NB; i++) st.set_aq(i, bin(i) < a.Q ? (float)(a.roots[bin(i)] * (double)bo) : 0.0f);
    }
    __device__ __forceinline__ float origin_X(int) const { return Do.x; }
    __device__ __forceinline__ float origin_S(int) const { return Do.z; }
    __device__ __forceinline__ float empty_psi(const SweepK &k, int i) const {
        return kSqrt2 * planck_k(k, nu_g * (1.0f + st.aq(i) * (float)(1.0 / kC)));
    }
    static __device__ __forceinline__ void put(float4 *rl, int s, const float2 (&x)[G]) {
#pragma unroll
        for (int k = 0; k < G; k++) rl[k * kRing + s] = make_float4(x[k].x, x[k].x, x[k].y, x[k].y);
    }
    __device__ __forceinline__ void first(const SweepK &k, const float4 A, const float4 *rl, float v) {
        first_point<NB>(k, st, A, rl[grp * kRing], nu_g, v);
    }
    template <bool FLOOR>
    __device__ __forceinline__ void step(const SweepK &k, const float4 A, const float4 *rl, int j, const float2 q) {
        step_point<NB, FLOOR>(k, st, A, rl[grp * kRing + j], q);
    }
    __device__ __forceinline__ void origin(const SweepK &k, const float4 Ao, const float2 q) {
        step_point<NB>(k, st, Ao, Do, q);
    }
    __device__ __forceinline__ void results(float (&pi)[NB], float (&ps)[NB], float (&dt)[NB]) const {
        bin_results<NB>(st, pi, ps, dt);
    }
};

// Result i: bin i / G of the lane, line i % G.
template <int G_, int NB_>
struct LineLanes {
    static constexpr int G = G_, NB = NB_, NBL = NB / G, H = G / 2, NP = NBL * H, kRingLines = H;
    static_assert(G % 2 == 0 && NB % G == 0, "whole line pairs");
    float a_q[NBL];
    float2 chi_p[NP], S_p[NP], d_p[NP], Phi[NP], iota[NP], psi[NP];   // pair b H + h: bin b, lines 2h and 2h + 1
    const float *nu;        // GHz, of the warp's lines
    int lines;              // lines of the group that exist
    float4 Do[H];           // the origin's (X0, X1, S0, S1) per line pair

    __device__ __forceinline__ int line(int i) const { return i % G; }
    __device__ __forceinline__ int bin(int i) const { return (threadIdx.x & 31) + 32 * (i / G); }
    __device__ __forceinline__ float aq(int i) const { return a_q[i / G]; }
    __device__ __forceinline__ float nu_of(int k) const { return nu[k < lines ? k : lines - 1]; }
    __device__ __forceinline__ void init(const MixArgs &a, int64_t o, int l0, float bo, float ibo) {
        nu = a.nu_ghz + l0;
        lines = min(G, a.L - l0);
#pragma unroll
        for (int b = 0; b < NBL; b++) {
            const int q = bin(b * G);
            a_q[b] = q < a.Q ? (float)(a.roots[q] * (double)bo) : 0.0f;
        }
        float X[G], S[G];
#pragma unroll
        for (int k = 0; k < G; k++) {
            const float2 dl = reinterpret_cast<const float2 *>(a.line)[o * a.L + l0 + (k < lines ? k : lines - 1)];
            X[k] = fmaxf(dl.y, 0.0f) * (ibo * a.inv_chi_min);   // in units of chi_min
            S[k] = dl.y > 0.0f ? dl.x / dl.y : 0.0f;
        }
#pragma unroll
        for (int h = 0; h < H; h++) Do[h] = make_float4(X[2 * h], X[2 * h + 1], S[2 * h], S[2 * h + 1]);
    }
    __device__ __forceinline__ float origin_X(int i) const { return (i & 1) ? Do[(i % G) >> 1].y : Do[(i % G) >> 1].x; }
    __device__ __forceinline__ float origin_S(int i) const { return (i & 1) ? Do[(i % G) >> 1].w : Do[(i % G) >> 1].z; }
    __device__ __forceinline__ float empty_psi(const SweepK &k, int i) const {
        return kSqrt2 * planck_k(k, nu_of(line(i)) * (1.0f + aq(i) * (float)(1.0 / kC)));
    }
    static __device__ __forceinline__ void put(float4 *rl, int s, const float2 (&x)[G]) {
#pragma unroll
        for (int h = 0; h < H; h++)
            rl[h * kRing + s] = make_float4(x[2 * h].x, x[2 * h + 1].x, x[2 * h].y, x[2 * h + 1].y);
    }
    // 2^(-x'^2) of every bin of the lane
    __device__ __forceinline__ void profile(const float4 A, float (&e)[NBL]) const {
        if constexpr (NBL % 2 == 0) {
#pragma unroll
            for (int b = 0; b < NBL; b += 2) {
                const float2 x = __ffma2_rn(make_float2(a_q[b], a_q[b + 1]), make_float2(A.x, A.y), make_float2(A.z, A.w));
                const float2 xx = __fmul2_rn(x, x);
                e[b] = ex2f(-xx.x);
                e[b + 1] = ex2f(-xx.y);
            }
        } else {
#pragma unroll
            for (int b = 0; b < NBL; b++) {
                const float x = fmaf(a_q[b], A.x, A.z);
                e[b] = ex2f(-x * x);
            }
        }
    }
    __device__ __forceinline__ void first(const SweepK &k, const float4 A, const float4 *rl, float v) {
        float e[NBL];
        profile(A, e);
        const float dop = 1.0f - v * (float)(1.0 / kC);
#pragma unroll
        for (int b = 0; b < NBL; b++)
#pragma unroll
            for (int h = 0; h < H; h++) {
                const int p = b * H + h;
                const float4 D = rl[h * kRing];
                const float2 chil = __fmul2_rn(make_float2(D.x, D.y), make_float2(e[b], e[b]));
                chi_p[p] = make_float2(fmaxf(chil.x, 1.0f), fmaxf(chil.y, 1.0f));
                S_p[p] = __fmul2_rn(make_float2(D.z, D.w), make_float2(fminf(chil.x, 1.0f), fminf(chil.y, 1.0f)));
                Phi[p] = make_float2(kSqrt2, kSqrt2);
                iota[p] = make_float2(1.0f, 1.0f);
                d_p[p] = make_float2(0.0f, 0.0f);
                const float sh = (1.0f + a_q[b] * (float)(1.0 / kC)) * dop;
                psi[p] = make_float2(kSqrt2 * planck_k(k, nu_of(2 * h) * sh), kSqrt2 * planck_k(k, nu_of(2 * h + 1) * sh));
            }
    }
    template <bool FLOOR>
    __device__ __forceinline__ void row(const SweepK &k, int p, const float4 D, float e, const float2 q) {
        const float2 chil = __fmul2_rn(make_float2(D.x, D.y), make_float2(e, e));
        const float2 chi = make_float2(fmaxf(chil.x, 1.0f), fmaxf(chil.y, 1.0f));
        const float2 Sx = __fmul2_rn(make_float2(D.z, D.w), make_float2(fminf(chil.x, 1.0f), fminf(chil.y, 1.0f)));
        const float2 d0 = __fmul2_rn(__fadd2_rn(chi_p[p], chi), q);
        const float2 dl = FLOOR ? make_float2(fmaxf(d0.x, k.dmin), fmaxf(d0.y, k.dmin)) : d0;
        const float2 sm = __fadd2_rn(d_p[p], dl);
        Phi[p] = __ffma2_rn(Phi[p], iota[p], sm);
        const float2 den = __ffma2_rn(dl, Phi[p], make_float2(1.0f, 1.0f));
        iota[p] = make_float2(rcpf(den.x), rcpf(den.y));
        psi[p] = __fmul2_rn(__ffma2_rn(sm, S_p[p], psi[p]), iota[p]);
        d_p[p] = dl;
        chi_p[p] = chi;
        S_p[p] = Sx;
    }
    template <bool FLOOR>
    __device__ __forceinline__ void step(const SweepK &k, const float4 A, const float4 *rl, int j, const float2 q) {
        float e[NBL];
        profile(A, e);
#pragma unroll
        for (int h = 0; h < H; h++) {
            const float4 D = rl[h * kRing + j];
#pragma unroll
            for (int b = 0; b < NBL; b++) row<FLOOR>(k, b * H + h, D, e[b], q);
        }
    }
    __device__ __forceinline__ void origin(const SweepK &k, const float4 Ao, const float2 q) {
        float e[NBL];
        profile(Ao, e);
#pragma unroll
        for (int h = 0; h < H; h++)
#pragma unroll
            for (int b = 0; b < NBL; b++) row<true>(k, b * H + h, Do[h], e[b], q);
    }
    __device__ __forceinline__ void results(float (&pi)[NB], float (&ps)[NB], float (&dt)[NB]) const {
#pragma unroll
        for (int b = 0; b < NBL; b++)
#pragma unroll
            for (int h = 0; h < H; h++) {
                const int p = b * H + h, i = b * G + 2 * h;
                const float2 pp = __fmul2_rn(Phi[p], iota[p]);
                pi[i] = pp.x; pi[i + 1] = pp.y;
                ps[i] = psi[p].x; ps[i + 1] = psi[p].y;
                dt[i] = d_p[p].x; dt[i + 1] = d_p[p].y;
            }
    }
};

// Sweeps half-ray r from its far end to the origin; returns per bin (Phi^ iota, psi^,
// delta) of the row next to the origin, or the empty-half values (sqrt 2, sqrt 2 I_o, 0).
// `pre` says that buffer bf already holds (or is receiving) the first window of r; on
// return it says the same of rnext (the half-ray swept next, -1 for none).
//
// Far points. A point is "far" for the warp when every bin of the warp lies so far in the
// wings of every line of its group that the opacity is floored there: X 2^(-x'^2) <
// chi_min over the warp's range of a_q (x' is monotonic in a_q, so the smallest |x'| is at
// an end of the range or zero). A point whose own and two previous points are all far
// changes the state by O(max(chi_min ds, dtau_min)) only and is left out; rows that
// involve a non-floored interval are still computed exactly. Most far points are left out
// before they are staged, a whole element at a time: each lane tests one element of the
// window (|x'| bounded from below by the ends of its velocity range over the larger width,
// X from above by the larger opacity over the smaller width), and only the first two points
// of a run of far elements are kept. The points of the remaining elements are numbered by a
// prefix sum over the window, staged 32 at a time, tested one by one, and written to the
// ring without gaps, so that the sweep is the same unrolled loop whether points are left
// out or not. Measured, launch of the best shape, every point staged and left out one by one
// -> this: clumpy cloud (50k points, 48 rays, 4 x 31 bins, 69 % of the points far) 11.72 ->
// 9.06 ms; disc (32k points, 192 rays, 19 x 63, 7 % far) 203.3 -> 197.0 ms.
template <typename Lay>
__device__ __forceinline__ void sweep_half(const MixArgs &a, const SweepK &k, int64_t o, int l0, int r, int rnext,
                                           const float4 Ao, Ring &rg, float4 *rl, ElemWin<Lay::G> &w, int &bf,
                                           bool &pre, Lay &lay, float (&pi)[Lay::NB], float (&ps)[Lay::NB],
                                           float (&dt)[Lay::NB], float aq_lo, float aq_hi, int &npts) {
    constexpr int G = Lay::G, NB = Lay::NB;
    const int lane = threadIdx.x & 31;
    const int64_t off = a.ray_off[o * a.R + r];
    const int len = (int)(a.ray_off[o * a.R + r + 1] - off);
    int64_t offn = 0;
    int lenn = 0;
    if (rnext >= 0) {
        offn = a.ray_off[o * a.R + rnext];
        lenn = (int)(a.ray_off[o * a.R + rnext + 1] - offn);
    }
    if (len == 0) {   // an empty half is never prefetched, so `pre` is false here
#pragma unroll
        for (int i = 0; i < NB; i++) {
            pi[i] = kSqrt2;
            ps[i] = lay.empty_psi(k, i);
            dt[i] = 0.0f;
        }
        return;
    }
    if (!pre) {
        win_records<G>(a, off, len - 1, (int32_t)o, w, bf);
        cp_async_wait_all();
        win_gathers<G>(a, l0, w, bf);
    }
    pre = false;
    bool first = true;
    unsigned far1 = 0, far2 = 0;   // whether the last two kept points are far
    int run = 0;                   // far points (at most 2) right before the window
    float qc = 0.0f;               // q' of the last element of the previous window
    int top = len - 1;             // element in window slot 0
    for (;; top -= kWin - 1) {
        cp_async_wait_all();
        __syncwarp();
        // the next window: the following 31 elements of this half-ray, else (this window
        // reaches element 0) the start of the next one
        const bool last_window = top < kWin - 1;
        const bool issue = !last_window || lenn > 0;
        if (!last_window) win_records<G>(a, off, top - (kWin - 1), (int32_t)o, w, bf ^ 1);
        else if (issue) win_records<G>(a, offn, lenn - 1, (int32_t)o, w, bf ^ 1);
        if (last_window) pre = issue;
        bool pending = issue;      // gathers of the next window still to be issued
        // ---- elements: lane i tests the element of slot i (slot 31 only precedes slot 30)
        const bool el = lane < kWin - 1 && lane <= top;
        const int x1 = w.x1[bf][lane], x0 = __shfl_down_sync(0xffffffffu, x1, 1);
        const int np = el ? x1 - x0 : 0;
        const float q = a.qscale * w.ds[bf][lane] * rcpf((float)max(np, 1));
        w.ds[bf][lane] = q;        // the slot's path length becomes its points' q'
        bool near = el;
        if (a.skip) {
            const float2 vb = w.vb[bf][lane];
            float cm = 0.0f;
#pragma unroll
            for (int kk = 0; kk < G; kk++) cm = fmaxf(cm, w.ln[bf][kk][lane].y);
            cm = fmaxf(cm, __shfl_down_sync(0xffffffffu, cm, 1));
            const float v0 = __shfl_down_sync(0xffffffffu, vb.x, 1), b0 = __shfl_down_sync(0xffffffffu, vb.y, 1);
            const float vlo = fminf(vb.x, v0), vhi = fmaxf(vb.x, v0);
            // a_q (1 - v/c) - v falls with v
            const float nlo = aq_lo - vhi * fmaf(aq_lo, (float)(1.0 / kC), 1.0f);
            const float nhi = aq_hi - vlo * fmaf(aq_hi, (float)(1.0 / kC), 1.0f);
            const float xm = fmaxf(fmaxf(nlo, -nhi), 0.0f) * (kSqrtLog2e * rcpf(fmaxf(vb.y, b0)));
            near = el && !(cm * a.inv_chi_min * rcpf(fminf(vb.y, b0)) * ex2f(-xm * xm) < 1.0f);
        }
        const unsigned nearm = __ballot_sync(0xffffffffu, near), onem = __ballot_sync(0xffffffffu, np == 1);
        // far points (at most 2) right before slot i, and the points kept of the slot
        int before = run;
        if (lane >= 1) {
            if ((nearm >> (lane - 1)) & 1u) before = 0;
            else if (!((onem >> (lane - 1)) & 1u)) before = 2;
            else before = lane >= 2 ? (((nearm >> (lane - 2)) & 1u) ? 1 : 2) : min(run + 1, 2);
        }
        const int keep = near ? np : min(np, 2 - before);
        run = __shfl_sync(0xffffffffu, before, kWin - 1);
        int end = keep;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, end, d);
            if (lane >= d) end += y;
        }
        const int start = end - keep, total = __shfl_sync(0xffffffffu, end, 31);
        const unsigned kept = __ballot_sync(0xffffffffu, keep > 0);
        if (keep > 0) rg.own[__popc(kept & ((1u << lane) - 1u))] = make_int4(lane, x1 - 1 + start, x0, np);
        __syncwarp();
        // ---- points, 32 at a time
        for (int c0 = 0; c0 < total; c0 += kRing) {
            const int cnt = min(kRing, total - c0);
            // element of each lane's point: the one before the first with a later start
            const int n0 = __popc(__ballot_sync(0xffffffffu, keep > 0 && start <= c0));
            const unsigned starts = __reduce_or_sync(
                0xffffffffu, (keep > 0 && start > c0 && start < c0 + 32) ? (1u << (start - c0)) : 0u);
            const int4 own = rg.own[n0 - 1 + __popc(starts & (0xffffffffu >> (31 - lane)))];
            bool far = false;
            float qin = 0.0f;
            PointGeo p{};
            float2 lines[G];
            if (lane < cnt) {
                const int i = own.x, j = own.y - (c0 + lane) - own.z + 1;
                p = point_geometry<G>(w, bf, i, j, own.w);
                qin = j < own.w ? w.ds[bf][i] : (i > 0 ? w.ds[bf][i - 1] : qc);
                const float Xmax = point_lines<G>(a, w, bf, i, p, lines);
                const float xlo = aq_lo * p.gz - p.gy, xhi = aq_hi * p.gz - p.gy;
                const float xm = xlo > 0.0f ? xlo : (xhi < 0.0f ? -xhi : 0.0f);
                far = a.skip && Xmax * ex2f(-xm * xm) < 1.0f;
            }
            const unsigned all = cnt == 32 ? 0xffffffffu : ((1u << cnt) - 1u);
            const unsigned fm = __ballot_sync(0xffffffffu, far);
            unsigned proc = ~(fm & ((fm << 1) | far1) & ((fm << 2) | (far1 << 1) | far2)) & all;
            if (first) proc |= 1u;   // the far end
            if (cnt >= 2) {
                far1 = (fm >> (cnt - 1)) & 1u;
                far2 = (fm >> (cnt - 2)) & 1u;
            } else {
                far2 = far1;
                far1 = fm & 1u;
            }
            const int m = __popc(proc);
            const bool mine = (proc >> lane) & 1u;
            if (mine) {
                const int s = __popc(proc & ((1u << lane) - 1u));
                rg.a[s] = make_float4(p.gz, p.gz, -p.gy, -p.gy);
                rg.q[s] = make_float2(qin, qin);
                Lay::put(rl, s, lines);
            }
            __syncwarp();
            npts += m;
            int j = 0;
            if (first) {
                const float4 A = rg.a[0];
                const float vfar = -A.z / (A.x - A.z * (float)(1.0 / kC));   // v = (v pz)/pz
                lay.first(k, A, rl, vfar);
                j = 1;
            }
            // A refill whose intervals all have q' >= q_nofloor sweeps without the dtau floor.
            const bool floor_needed =
                __any_sync(0xffffffffu, mine && qin < a.q_nofloor && !(first && lane == 0));
            first = false;
            auto dense = [&](auto floor_tag, int jend) {
#pragma unroll 4
                for (; j < jend; j++) lay.template step<decltype(floor_tag)::value>(k, rg.a[j], rl, j, rg.q[j]);
            };
            // two segments, with the gathers of the next window issued between them (one
            // copy of each loop body)
            const int mid = m < 16 ? m : 16;
#pragma unroll 1
            for (int seg = 0; seg < 2; seg++) {
                if (floor_needed) dense(std::true_type{}, seg ? m : mid);
                else dense(std::false_type{}, seg ? m : mid);
                if (seg == 0 && pending) {
                    cp_async_wait_all();
                    win_gathers<G>(a, l0, w, bf ^ 1);
                    pending = false;
                }
            }
            __syncwarp();
        }
        if (pending) {   // a window without points to sweep
            cp_async_wait_all();
            win_gathers<G>(a, l0, w, bf ^ 1);
        }
        qc = __shfl_sync(0xffffffffu, q, last_window ? top : kWin - 2);
        if (last_window) break;
        bf ^= 1;
    }
    if (pre) bf ^= 1;   // the next half-ray's first window sits in the other buffer
    lay.origin(k, Ao, make_float2(qc, qc));
    npts++;
    lay.results(pi, ps, dt);
}

// Per-lane, per-bin values that live across the ray pairs (slot [.][i][lane]): the pair
// sums and the backward half's result while the forward half is swept. Held in shared
// memory so that the sweeps keep their registers for the recursion.
template <int NB>
struct PairSmem {
    float acc[3][NB][32];                       // sums over pairs of Lambda*, u - Lambda* S, 1 - Lambda*
    float pi[NB][32], ps[NB][32], dt[NB][32];   // backward half: (Phi^ iota, psi^, delta)
};

// One work item: origin o, lines l0 .. l0+G-1, all ray pairs, all bins (one warp).
template <typename Lay>
__device__ __forceinline__ void solve_item(const MixArgs &a, int64_t o, int l0, Ring &rg, float4 *rl,
                                           ElemWin<Lay::G> &w, PairSmem<Lay::NB> &ps) {
    constexpr int G = Lay::G, NB = Lay::NB;
    const int lane = threadIdx.x & 31;
    const int Q = a.Q;
    const float bo = a.b[o];
    const float ibo = 1.0f / bo;
    // ring entry of the origin (v = 0 there): a = (g_z, g_z, -0, -0)
    const float gzo = kSqrtLog2e * ibo;
    const float4 Ao = make_float4(gzo, gzo, -0.0f, -0.0f);
    const SweepK k{a.delta_min, a.planck_a, a.planck_b};
    Lay lay;
    lay.init(a, o, l0, bo, ibo);
    // range of a_q over the whole warp (all lanes, all bins)
    float aq_lo = 1e30f, aq_hi = -1e30f;
#pragma unroll
    for (int i = 0; i < NB; i++) {
        ps.acc[0][i][lane] = ps.acc[1][i][lane] = ps.acc[2][i][lane] = 0.0f;
        if (lay.bin(i) < Q) { aq_lo = fminf(aq_lo, lay.aq(i)); aq_hi = fmaxf(aq_hi, lay.aq(i)); }
    }
    for (int d = 16; d; d >>= 1) {
        aq_lo = fminf(aq_lo, __shfl_xor_sync(0xffffffffu, aq_lo, d));
        aq_hi = fmaxf(aq_hi, __shfl_xor_sync(0xffffffffu, aq_hi, d));
    }
    int bf = 0;
    bool pre = false;
    int npts = 0;   // points swept (warp-uniform), for the executed-work count
    for (int p = 0; p < a.P; p++) {
        const int rb = a.pb[p], rf = a.pf[p];
        const int rn = p + 1 < a.P ? a.pb[p + 1] : -1;
        float pif[NB], psf[NB], dtf[NB];
#pragma unroll 1
        for (int h = 0; h < 2; h++) {   // backward half, then forward half (one code copy)
            sweep_half<Lay>(a, k, o, l0, h ? rf : rb, h ? rn : rf, Ao, rg, rl, w, bf, pre, lay, pif, psf, dtf, aq_lo,
                            aq_hi, npts);
            if (h == 0) {
#pragma unroll
                for (int i = 0; i < NB; i++) {
                    ps.pi[i][lane] = pif[i];
                    ps.ps[i][lane] = psf[i];
                    ps.dt[i][lane] = dtf[i];
                }
            }
        }
#pragma unroll
        for (int i = 0; i < NB; i++) {
            const float pib = ps.pi[i][lane], psb = ps.ps[i][lane], dtb = ps.dt[i][lane];
            float lam, uml, oml;
            if (dtb == 0.0f && dtf[i] == 0.0f) {   // isolated origin: both halves empty
                lam = 0.0f; uml = psb * (float)(1.0 / 1.4142135623730951); oml = 1.0f;
            } else {
                // sigma (Phi iota) = Phi^ iota / (delta_- + delta_+), sigma psi = psi^ / (delta_- + delta_+)
                const float sig = rcpf(dtb + dtf[i]);
                const float pi2 = sig * (pib + pif[i]);
                lam = rcpf(1.0f + pi2);
                uml = (psb + psf[i]) * (sig * lam);
                oml = pi2 * lam;
            }
            ps.acc[0][i][lane] += lam;
            ps.acc[1][i][lane] += uml;
            ps.acc[2][i][lane] += oml;
        }
    }
    cp_async_wait_all();
    if (a.work && lane == 0) {
        const int lines = min(G, a.L - l0);
        atomicAdd(a.work, (unsigned long long)npts * (unsigned long long)(lines * Q));
    }
    // The origin's line opacity and floored source in a bin are the same for every pair: u =
    // Lambda* S + (u - Lambda* S) and the line's shares of opacity and emission enter after the
    // sums over pairs. v: u, Lambda, J_eff and 1 - Lambda of result i.
    const double invP = 1.0 / a.P;
    auto values = [&](int i, float (&v)[4]) {
        const float xo = lay.aq(i) * gzo, Xo = lay.origin_X(i), So = lay.origin_S(i);
        const float chilo = Xo * ex2f(-xo * xo);
        const float chio = fmaxf(chilo, 1.0f), ichi = rcpf(chio);
        const float Sov = So * fminf(chilo, 1.0f);
        const float lam = ps.acc[0][i][lane], uml = ps.acc[1][i][lane], oml = ps.acc[2][i][lane];
        v[0] = uml + lam * Sov;
        v[1] = lam * (chilo * ichi);
        v[2] = uml + lam * ((Sov * chio - chilo * So) * ichi);
        v[3] = oml + lam * ((chio - chilo) * ichi);
        if (a.Jnu && lay.bin(i) < Q && l0 + lay.line(i) < a.L)
            a.Jnu[(o * a.L + l0 + lay.line(i)) * Q + lay.bin(i)] = (double)v[0] * invP * (double)kI0;
    };
    // weighted sums over each line's bins in FP64, in a fixed order
    if constexpr (Lay::kRingLines == G) {
        // a line per lane group: a shuffle tree within the group
        constexpr int LPG = 32 / G;
        double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int i = 0; i < NB; i++) {
            float v[4];
            values(i, v);
            const double wq = lay.bin(i) < Q ? a.weights[lay.bin(i)] : 0.0;
#pragma unroll
            for (int kk = 0; kk < 4; kk++) s[kk] += wq * (double)v[kk];
        }
#pragma unroll
        for (int kk = 0; kk < 4; kk++)
            for (int d = LPG / 2; d; d >>= 1) s[kk] += __shfl_down_sync(0xffffffffu, s[kk], d);
        const int l = l0 + lay.line(0);
        if (lane % LPG == 0 && l < a.L) {
            a.J[o * a.L + l] = s[0] * invP * (double)kI0;
            a.Lout[o * a.L + l] = s[1] * invP;
            a.Jeff[o * a.L + l] = s[2] * invP * (double)kI0;
            a.Lc[o * a.L + l] = s[3] * invP;
        }
    } else {
        // every lane has every line: 4 G sums over the warp, halving the number of sums a lane
        // carries with each step of the exchange (4 G additions in place of 20 G)
        constexpr int M = 4 * G;
        double s[M];
#pragma unroll
        for (int t = 0; t < M; t++) s[t] = 0.0;
#pragma unroll
        for (int i = 0; i < NB; i++) {
            float v[4];
            values(i, v);
            const double wq = lay.bin(i) < Q ? a.weights[lay.bin(i)] : 0.0;
#pragma unroll
            for (int kk = 0; kk < 4; kk++) s[4 * (i % G) + kk] += wq * (double)v[kk];
        }
        int m = M;
#pragma unroll
        for (int d = 16; d; d >>= 1) {
            if (m > 1) {
                m >>= 1;
                const bool up = lane & d;
#pragma unroll
                for (int t = 0; t < M / 2; t++)
                    if (t < m) {
                        const double keep = up ? s[t + m] : s[t], give = up ? s[t] : s[t + m];
                        s[t] = keep + __shfl_xor_sync(0xffffffffu, give, d);
                    }
            } else {
                s[0] += __shfl_xor_sync(0xffffffffu, s[0], d);
            }
        }
        const int t = lane / (32 / M), l = l0 + t / 4, kk = t % 4;   // (M <= 32)
        if (lane % (32 / M) == 0 && l < a.L) {
            double *dst = kk == 0 ? a.J : (kk == 1 ? a.Lout : (kk == 2 ? a.Jeff : a.Lc));
            dst[o * a.L + l] = s[0] * invP * (kk % 2 == 0 ? (double)kI0 : 1.0);
        }
    }
}

// The layout of a shape: lines on every lane where the bins fill whole warps.
template <int G, int NB, bool LINES>
struct LayoutOf {
    using type = BinLanes<G, NB>;
};
template <int G, int NB>
struct LayoutOf<G, NB, true> {
    using type = LineLanes<G, NB>;
};

template <int G, int NB, int MINB, int W, bool LINES>
__global__ void __launch_bounds__(32 * W, MINB) k_feautrier_warp(MixArgs a) {
    using Lay = typename LayoutOf<G, NB, LINES>::type;
    __shared__ Ring rgs[W];
    __shared__ float4 rls[W][Lay::kRingLines * kRing];
    __shared__ ElemWin<G> ews[W];
    __shared__ PairSmem<NB> pss[W];
    const int warp = threadIdx.x >> 5;
    const int ngroups = (a.L + G - 1) / G;
    const int64_t item = (int64_t)blockIdx.x * W + warp;
    if (item >= a.n * ngroups) return;
    const int64_t o = item / ngroups;
    const int l0 = (int)(item - o * ngroups) * G;
    solve_item<Lay>(a, o, l0, rgs[warp], rls[warp], ews[warp], pss[warp]);
}

// Persistent variant over a batch of models: every warp takes work items (model, origin,
// line group) from a queue ordered by decreasing cost until the queue is empty. The
// per-model arguments are copied once per item into the warp's shared-memory slot.
struct BatchItem {
    int32_t model;
    int32_t local;   // origin * L + first line of the warp's line group
};

template <int G, int NB, int MINB, int W, bool LINES>
__global__ void __launch_bounds__(32 * W, MINB)
k_feautrier_batch(const MixArgs *__restrict__ models, const BatchItem *__restrict__ items, int64_t n_items,
                  unsigned long long *counter, const int32_t *__restrict__ active, int32_t skip) {
    using Lay = typename LayoutOf<G, NB, LINES>::type;
    __shared__ Ring rgs[W];
    __shared__ float4 rls[W][Lay::kRingLines * kRing];
    __shared__ ElemWin<G> ews[W];
    __shared__ PairSmem<NB> pss[W];
    __shared__ MixArgs sa[W];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (;;) {
        unsigned long long idx = 0;
        if (lane == 0) idx = atomicAdd(counter, 1ull);
        idx = __shfl_sync(0xffffffffu, idx, 0);
        if (idx >= (unsigned long long)n_items) break;
        const BatchItem it = items[idx];
        if (!active[it.model]) continue;
        __syncwarp();
        if (lane == 0) {
            sa[warp] = models[it.model];
            sa[warp].skip = skip;
        }
        __syncwarp();
        const MixArgs &a = sa[warp];
        const int64_t o = it.local / a.L;
        const int l0 = (int)(it.local - o * a.L);
        solve_item<Lay>(a, o, l0, rgs[warp], rls[warp], ews[warp], pss[warp]);
    }
}

// Launch variants of the warp kernel: (lines per warp, bins per lane, min blocks per SM,
// far-wing skipping, warps per block).
struct WarpVariant {
    int G, NB, MINB;
    bool skip;
    int W;
    void (*fn)(MixArgs);
    void (*batch)(const MixArgs *, const BatchItem *, int64_t, unsigned long long *, const int32_t *, int32_t);
};
// (the shapes whose NB/G bins per lane and line fill 32-bin rounds take LineLanes)
#define MG_VARIANT_L(G, NB, M, S, W, L) \
    {G, NB, M, S, W, k_feautrier_warp<G, NB, M, W, L>, k_feautrier_batch<G, NB, M, W, L>}
#define MG_VARIANT_W(G, NB, M, S, W) MG_VARIANT_L(G, NB, M, S, W, ((G) % 2 == 0 && (NB) % (G) == 0))
#define MG_VARIANT(G, NB, M, S) MG_VARIANT_W(G, NB, M, S, kWarps2)
const WarpVariant kWarpVariants[] = {
    // with far-wing skipping
    MG_VARIANT(1, 1, 8, true), MG_VARIANT(1, 1, 10, true), MG_VARIANT(2, 2, 4, true), MG_VARIANT(2, 2, 5, true),
    MG_VARIANT(2, 2, 6, true), MG_VARIANT(1, 2, 4, true), MG_VARIANT(1, 2, 6, true), MG_VARIANT(1, 4, 3, true),
    MG_VARIANT(1, 4, 4, true), MG_VARIANT(2, 4, 3, true), MG_VARIANT(2, 4, 4, true), MG_VARIANT(4, 4, 3, true),
    MG_VARIANT(4, 4, 4, true),
    // the same shapes without skipping (every point swept)
    MG_VARIANT(1, 1, 8, false), MG_VARIANT(1, 1, 10, false), MG_VARIANT(2, 2, 4, false), MG_VARIANT(2, 2, 5, false),
    MG_VARIANT(2, 2, 6, false), MG_VARIANT(1, 2, 4, false), MG_VARIANT(1, 2, 6, false), MG_VARIANT(1, 4, 3, false),
    MG_VARIANT(1, 4, 4, false), MG_VARIANT(2, 4, 3, false), MG_VARIANT(2, 4, 4, false), MG_VARIANT(4, 4, 3, false),
    MG_VARIANT(4, 4, 4, false),
    // two lines x four bins per lane at 5 and 6 blocks per SM (95 and 80 registers, a few
    // spilled words) for more warps in flight on lines with 33-64 bins
    MG_VARIANT(2, 4, 5, false), MG_VARIANT(2, 4, 6, false),
    // eight bins per lane (four independent bin pairs per lane) at four lines per warp,
    // for lines with 33-64 bins; three warps per block keep the static shared memory
    // below 48 KB
    MG_VARIANT_W(4, 8, 3, false, 3), MG_VARIANT_W(4, 8, 4, false, 3), MG_VARIANT_W(4, 8, 3, true, 3),
    MG_VARIANT_W(4, 8, 4, true, 3),
    // shapes for few and for odd numbers of bins: up to 16 (two or four lines per warp), 17-24
    // and 33-48 bins per line
    MG_VARIANT(2, 1, 8, true), MG_VARIANT(2, 1, 8, false), MG_VARIANT(4, 2, 5, true), MG_VARIANT(4, 2, 5, false),
    MG_VARIANT(4, 3, 4, true), MG_VARIANT(4, 3, 4, false), MG_VARIANT_W(4, 6, 4, true, 3),
    MG_VARIANT_W(4, 6, 4, false, 3),
};
#undef MG_VARIANT
#undef MG_VARIANT_W
#undef MG_VARIANT_L
constexpr int kNumWarpVariants = sizeof(kWarpVariants) / sizeof(kWarpVariants[0]);

// Far-wing skipping leaves out the floored intervals of far points. Each changes the
// sweep by O(max(chi_min ds, dtau_min)), below FP32 resolution only while the optical depth
// that the floors give a whole ray pair is; otherwise (a large floor) the variant's
// non-skipping twin runs instead. The point after a left-out one must be near the floor as well,
// which the velocity-step rule sees to: with steps of up to two widths its opacity is below
// chi_min exp(4 x' - 4) = 3e11 chi_min at x' = 7.6 (a line 1e25 times the floor), 3e-6 over 1e13 m.
// Where dshift_frac allows larger steps every point is swept (J per bin was off by 3e-3 at 30).
bool skip_allowed(const mg_ctx *ctx) { return mg_floor_depth(ctx) < 1e-7 && ctx->opt.dshift_frac <= 2.0; }

int no_skip_twin(int v) {
    const WarpVariant &w = kWarpVariants[v];
    for (int u = 0; u < kNumWarpVariants; u++) {
        const WarpVariant &x = kWarpVariants[u];
        if (!x.skip && x.G == w.G && x.NB == w.NB && x.MINB == w.MINB && x.W == w.W) return u;
    }
    return v;
}

int effective_variant(const mg_ctx *ctx, int v) {
    if (v < 0 || v >= kNumWarpVariants || !kWarpVariants[v].skip || skip_allowed(ctx)) return v;
    return no_skip_twin(v);
}

bool variant_valid(int v, int L, int Q) {
    if (v < 0 || v >= kNumWarpVariants) return false;
    const WarpVariant &w = kWarpVariants[v];
    if (w.G > L) return false;
    // the smallest number of bins per lane that holds the line among 1, 2, 4, 8 (and 3, 6
    // between them)
    const int less = w.NB == 1 ? 0 : (w.NB == 3 ? 2 : (w.NB == 6 ? 4 : w.NB / 2));
    return Q <= w.NB * (32 / w.G) && Q > less * (32 / w.G);
}

}  // namespace

static LineArgs line_args(const mg_ctx *c) {
    return LineArgs{c->n, c->n_lines, c->n_lev, c->d_pops, c->d_lines, c->d_line, c->d_linef, c->d_scal};
}

int mg_launch_line_data_mixed(mg_ctx *ctx) {
    const int64_t m = ctx->n * ctx->n_lines;
    MgTimed t(ctx, "line_data");
    LineBatch b{};
    b.m[0] = line_args(ctx);
    k_line_data_f32<<<(unsigned)((m + 255) / 256), 256, 0, ctx->stream>>>(b);
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

// Line data of every model of a batch: one launch per 48 models (a launch each left 5 us of
// mostly empty GPU per model and iteration). The counters are cleared first, those of the
// population update too when one follows.
int mg_launch_line_data_batch(mg_ctx *const *models, int count, bool reset_update, cudaStream_t stream) {
    for (int i0 = 0; i0 < count; i0 += 256) {
        ScalBatch b{};
        const int k = std::min(256, count - i0);
        for (int i = 0; i < k; i++) b.scal[i] = models[i0 + i]->d_scal;
        k_clear_words<<<1, 256, 0, stream>>>(b, k, reset_update ? 1 : 0);
    }
    for (int i0 = 0; i0 < count; i0 += kLineBatch) {
        LineBatch b{};
        const int k = std::min(kLineBatch, count - i0);
        int64_t mmax = 0;
        for (int i = 0; i < k; i++) {
            b.m[i] = line_args(models[i0 + i]);
            mmax = std::max(mmax, b.m[i].n * b.m[i].L);
        }
        k_line_data_f32<<<dim3((unsigned)((mmax + 255) / 256), k), 256, 0, stream>>>(b);
    }
    return cudaGetLastError() == cudaSuccess ? MG_OK : MG_ERR_CUDA;
}


static void fill_args(mg_ctx *ctx, MixArgs &a) {
    const int L = ctx->n_lines, Q = ctx->Q;
    a.n = ctx->n; a.R = ctx->R; a.P = ctx->P; a.L = L; a.Q = Q;
    a.pf = ctx->d_pf; a.pb = ctx->d_pb; a.ray_off = ctx->d_ray_off; a.cells = ctx->d_cells; a.xcum = ctx->d_xcum;
    a.ds = ctx->d_dsf; a.vpar = ctx->d_vparf; a.b = ctx->d_bf; a.line = ctx->d_linef;
    a.nu_ghz = ctx->d_lconst + L;
    a.roots = ctx->d_roots; a.weights = ctx->d_weights; a.ovl_off = ctx->d_ovl_off; a.ovl = ctx->d_ovl;
    a.chi_min = (float)ctx->opt.chi_min; a.dtau_min = (float)ctx->opt.dtau_min;
    a.inv_chi_min = (float)(1.0 / ctx->opt.chi_min);
    // Every floored opacity is >= 1 in units of chi_min, so an interval with
    // q' >= q_nofloor has delta = dtau/sqrt 2 = (chi'_prev + chi') q' >= delta_min: the floor
    // cannot bind there.
    a.delta_min = (float)(ctx->opt.dtau_min / 1.4142135623730951);
    a.q_nofloor = std::nextafter((float)(ctx->opt.dtau_min / 2.0) * 1.000001f, INFINITY);
    a.qscale = (float)(ctx->opt.chi_min * (double)kInvSqrt8);
    a.planck_a = (float)(2.0 * kH * 1e27 / (kC * kC) / (double)kI0);
    a.planck_b = (float)(kH * 1e9 / (kKB * ctx->opt.T_cmb));
    a.J = ctx->d_J; a.Lout = ctx->d_L; a.Jeff = ctx->d_Jeff; a.Lc = ctx->d_Lc;
    a.Jnu = ctx->opt.spectrum ? ctx->d_Jnu : nullptr;
    a.kmax = (int32_t)ctx->max_pair_len;
    a.err = ctx->d_err;
    a.work = ctx->opt.profile ? ctx->d_scal + 7 : nullptr;   // executed updates, profiling runs only
    bool overlap = false;
    for (int l = 0; l < L; l++) overlap |= (ctx->h_ovl_off[l + 1] - ctx->h_ovl_off[l]) > 1;
    a.overlap = overlap;
}

static int launch_mixed(mg_ctx *ctx, int variant) {
    const int L = ctx->n_lines, Q = ctx->Q;
    bool overlap = false;
    for (int l = 0; l < L; l++) overlap |= (ctx->h_ovl_off[l + 1] - ctx->h_ovl_off[l]) > 1;
    MixArgs a{};
    fill_args(ctx, a);
    a.kmax = (int32_t)ctx->max_pair_len;
    a.overlap = overlap;
    a.err = ctx->d_err;
    size_t smem = mixed_acc_offset(a.kmax, L) + 16 * (size_t)L * Q;
    if ((overlap || Q > 128) && smem > 227 * 1024) {
        return mg_fail(ctx, MG_ERR_CAPACITY, "mixed formal solve: longest ray pair does not fit in shared memory");
    }
    int threads = 32 * std::min(L, 8);
    if (overlap) variant = -1;
    MG_CUDA(cudaMemsetAsync(ctx->d_err, 0, 4, ctx->stream));
    if (overlap) {
        MG_CUDA(cudaFuncSetAttribute(k_feautrier_mixed<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        MgTimed t(ctx, "feautrier_mixed");
        k_feautrier_mixed<true><<<(unsigned)ctx->n, threads, smem, ctx->stream>>>(a);
    } else if (variant >= 0 && variant < kNumWarpVariants) {
        const WarpVariant &wv = kWarpVariants[effective_variant(ctx, variant)];
        a.skip = wv.skip;
        const int64_t items = ctx->n * ((L + wv.G - 1) / wv.G);
        const unsigned grid = (unsigned)((items + wv.W - 1) / wv.W);
        MgTimed t(ctx, "feautrier_mixed");
        wv.fn<<<grid, 32 * wv.W, 0, ctx->stream>>>(a);
    } else {
        MG_CUDA(cudaFuncSetAttribute(k_feautrier_mixed<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        MgTimed t(ctx, "feautrier_mixed");
        k_feautrier_mixed<false><<<(unsigned)ctx->n, threads, smem, ctx->stream>>>(a);
    }
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

// Default launch variant for a model. A warp's time grows with its bins per lane and has a
// share that does not (staging, windows, pair ends): measured per line on a disc of 31 bins
// 1.62 ms at 1 line x 1 bin, 1.03 ms at 2 x 2 and 0.80 ms at 4 x 4, and with 63 bins 13.6 ms,
// 10.1 ms and 9.0 ms at 1 x 2, 2 x 4 and 4 x 8: within a tenth of proportional to NB +
// 1.6 per group in all six. The default takes the shape with the smallest ceil(L/G) (NB +
// 1.6): 4 lines x 4 bins (8 for 33-64 bins) for most numbers of lines, two lines per warp
// where four would leave half of the last warp idle (5, 6 lines). Among equal shapes the
// first of the list, the fastest number of blocks per SM.
static int default_variant(int L, int Q) {
    const int order[] = {12, 31, 34, 36, 38, 3, 10, 32, 0, 6, 8};
    int best = -1;
    float cost = 1e30f;
    for (int v : order) {
        if (!variant_valid(v, L, Q)) continue;
        const float c = (float)((L + kWarpVariants[v].G - 1) / kWarpVariants[v].G) * (kWarpVariants[v].NB + 1.6f);
        if (c < cost) {
            cost = c;
            best = v;
        }
    }
    return best;
}

int mg_launch_feautrier_mixed(mg_ctx *ctx) {
    int v = ctx->mixed_variant;
    if (!variant_valid(v, ctx->n_lines, ctx->Q)) v = default_variant(ctx->n_lines, ctx->Q);
    return launch_mixed(ctx, v);
}

// Autotuner: times one formal-solve launch of every valid variant on the loaded model
// (CUDA events on the context's stream, best of `reps`) and keeps the fastest.
int mg_autotune_mixed(mg_ctx *ctx, int reps, int *best, double *best_ms, int *n_tried) {
    const int L = ctx->n_lines, Q = ctx->Q;
    cudaEvent_t e0, e1;
    MG_CUDA(cudaEventCreate(&e0));
    MG_CUDA(cudaEventCreate(&e1));
    int bv = -1, tried = 0;
    float bms = 1e30f;
    const int saved_profile = ctx->opt.profile;
    ctx->opt.profile = 0;
    for (int v = 0; v < kNumWarpVariants; v++) {
        if (!variant_valid(v, L, Q) || effective_variant(ctx, v) != v) continue;
        tried++;
        float vbest = 1e30f;
        for (int r = 0; r < reps + 1; r++) {
            cudaEventRecord(e0, ctx->stream);
            int rc = launch_mixed(ctx, v);
            cudaEventRecord(e1, ctx->stream);
            if (rc) { ctx->opt.profile = saved_profile; return rc; }
            cudaEventSynchronize(e1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (r > 0 && ms < vbest) vbest = ms;   // first launch warms up
        }
        if (vbest < bms) { bms = vbest; bv = v; }
    }
    ctx->opt.profile = saved_profile;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (bv >= 0) ctx->mixed_variant = bv;
    if (best) *best = bv;
    if (best_ms) *best_ms = bms;
    if (n_tried) *n_tried = tried;
    return MG_OK;
}

// ---------------------------------------------------------------- batch helpers
size_t mg_mixargs_size() { return sizeof(MixArgs); }

int mg_fill_mixargs(mg_ctx *ctx, void *out) {
    MixArgs a{};
    fill_args(ctx, a);
    if (a.overlap) return mg_fail(ctx, MG_ERR_ARG, "batch: models with overlapping lines are not batched");
    std::memcpy(out, &a, sizeof(a));
    return MG_OK;
}

int mg_variant_count() { return kNumWarpVariants; }
int mg_variant_valid(int v, int L, int Q) { return variant_valid(v, L, Q) ? 1 : 0; }
int mg_variant_effective(const mg_ctx *ctx, int v) { return effective_variant(ctx, v); }
int mg_variant_minb(int v) { return (v >= 0 && v < kNumWarpVariants) ? kWarpVariants[v].MINB : 0; }
int mg_variant_g(int v) { return (v >= 0 && v < kNumWarpVariants) ? kWarpVariants[v].G : 1; }
int mg_variant_default(int L, int Q) { return default_variant(L, Q); }

int mg_batch_launch(int v, int grid, const void *d_args, const void *d_items, int64_t n_items,
                    unsigned long long *counter, const int32_t *active, cudaStream_t stream) {
    if (v < 0 || v >= kNumWarpVariants) return MG_ERR_ARG;
    kWarpVariants[v].batch<<<grid, 32 * kWarpVariants[v].W, 0, stream>>>(static_cast<const MixArgs *>(d_args),
                                                               static_cast<const BatchItem *>(d_items), n_items,
                                                               counter, active, kWarpVariants[v].skip);
    return cudaGetLastError() == cudaSuccess ? MG_OK : MG_ERR_CUDA;
}
