// The FP64 formal solve for lines that do not overlap (included by solve.cu).
//
// One CTA per origin. Its warps share the bins of the point (32 consecutive bins of the
// flattened (line, bin) list per warp) and, when there are few bins, the ray pairs; each
// warp sweeps its pairs through a private ring of staged points and needs no CTA barrier
// until the final sums.
//
// What bounds it. A warp-wide FP64 instruction occupies an SM sub-partition's FP64 pipe for
// 64-80 cycles (0.50 T DFMA/s), so FP64 instructions are the cost and everything else is
// nearly free. Per point and bin the sweep needs 5 of them:
//   x' = a_q g_z - g_y;  P = t Q + P;  R = (t S_prev) Q + R (2);  Q = dtau P + Q.
// - The recursion is homogeneous: with Phi iota = P/Q and psi = R/Q the point update of
//   k_feautrier64 needs no reciprocal, and every term stays a sum of non-negative
//   numbers. (P, Q, R) are scaled by 2^-256 when Q exceeds 2^256.
// - The profile exponential, the line opacity, the floors, delta = dtau/2 = (chi_prev + chi) h
//   with h = ds/4, and t = delta_prev + delta run on the integer pipe (posfp.cuh); so do the
//   divisions of the staging.
// - S = eta/chi of a line does not depend on the bin: one division per staged point.
// - A point whose own and two previous points are far (opacity below chi_min and emission
//   below chi_min times the least intensity, note_source) changes the sweep by O(max(chi_min ds, dtau_min))
//   and is left out while the optical depth that the two floors give a whole ray pair (chi_min
//   times the longest path through the model, dtau_min per interval) is below 1e-14 (`skip`):
//   whole elements before they are staged, points far in every bin of the warp before they
//   reach the ring, and the rest bin by bin, each lane sweeping its own points.
//
// The general kernel k_feautrier64 (a bin sums several lines) takes, per point and bin, an
// exponential (16 DFMA), two divisions (8 each), four interpolations and ~15 further
// operations, and sweeps every point. Measured, one ALI step, general kernel -> this one:
// clumpy cloud of 1500 points, 48 rays, 4 x 31 bins 174.9 -> 8.3 ms (11.1 ms with 8 FP64
// operations per point and bin, warp-wide far points and every point staged), FP64 pipe active
// in 74 % of the cycles; with the band ALO (600 points) 124.8 -> 5.8 ms; spherical cloud of 200
// shells 1.64 -> 0.35 ms; scattering on a 200-point cloud, to a change of 1e-10, 7.1 -> 1.5 ms.
namespace {

constexpr float kLog2e64 = 1.4426950408889634f;

// Larger of two non-negative doubles, on their bits.
__device__ __forceinline__ double pos_max(double a, double b) {
    return __double_as_longlong(a) > __double_as_longlong(b) ? a : b;
}

// Per-warp shared memory: an element window (as in the FP32 kernel: slot i holds element
// top - i, slot 31 only precedes slot 30; element -1 is the origin) and the ring of points.
struct Warp64 {
    int32_t *x1, *cell;          // (x1[32]: points of the half-ray)
    double *v, *b, *ds, *rn;     // (ds: h of the element's intervals; rn: 1 / its points)
    int4 *own;                   // per element with points to sweep: (slot, first point + its position, x0, points)
    double2 *ln;                 // [nl][32] (eta, chi)
    double *gz, *ngy, *h;        // ring: x' = a_q gz + ngy; h of the interval from the previous point
    uint64_t *Xm, *Ym;           // [nl][32] line opacity X and floored source Y = eta/chi_min at line centre
    int32_t *Xe, *Ye;            //   (exponents; Ye holds 8 e + flags: 1 for Y < 0, 2 for X < 0 or NaN, 4
                                 //   for an emissivity that is not finite; S is NaN then)
    double *S;                   // [nl][32]
    float4 *tt;                  // [nl][32]: (g_z, -g_y, |x'| beyond which the line is far, -) in FP32
    double *N;                   // ring: profile normalisation without 1/nu (band terms)
    int32_t *rx;                 // ring: point index (band terms)
    double *w, *xs;              // ring: weight, scattering opacity
    int32_t *ca, *cb;            // ring: cells (scattering)
    double *mac;                 // [32][2 B]
    int32_t *ic;                 // [nl] exponent of the least intensity at the line, rounded down (note_source)
};

__host__ __device__ inline size_t warp64_bytes(int nl, int B, bool sca) {
    return (size_t)32 * (12 + 32 + 16 + 16 * nl + 24 + 32 * nl + 4 + 16 * nl) + (B ? 32 * (8 + 8 + 16 * B) : 0) + (sca ? 32 * 24 : 0);
}

__device__ __forceinline__ Warp64 carve64(unsigned char *p, int nl, int B, bool sca) {
    Warp64 w{};
    auto take = [&](size_t bytes) { unsigned char *q = p; p += 32 * bytes; return q; };
    w.ln = reinterpret_cast<double2 *>(take(16 * nl));
    w.tt = reinterpret_cast<float4 *>(take(16 * nl));
    w.own = reinterpret_cast<int4 *>(take(16));
    w.rn = reinterpret_cast<double *>(take(8));
    w.v = reinterpret_cast<double *>(take(8));
    w.b = reinterpret_cast<double *>(take(8));
    w.ds = reinterpret_cast<double *>(take(8));
    w.gz = reinterpret_cast<double *>(take(8));
    w.ngy = reinterpret_cast<double *>(take(8));
    w.h = reinterpret_cast<double *>(take(8));
    w.Xm = reinterpret_cast<uint64_t *>(take(8 * nl));
    w.Ym = reinterpret_cast<uint64_t *>(take(8 * nl));
    w.S = reinterpret_cast<double *>(take(8 * nl));
    w.Xe = reinterpret_cast<int32_t *>(take(4 * nl));
    w.Ye = reinterpret_cast<int32_t *>(take(4 * nl));
    w.x1 = reinterpret_cast<int32_t *>(take(8));
    w.cell = reinterpret_cast<int32_t *>(take(4));
    w.ic = reinterpret_cast<int32_t *>(take(4));
    if (B) {
        w.N = reinterpret_cast<double *>(take(8));
        w.mac = reinterpret_cast<double *>(take(16 * B));
        w.rx = reinterpret_cast<int32_t *>(take(8));
    }
    if (sca) {
        w.w = reinterpret_cast<double *>(take(8));
        w.xs = reinterpret_cast<double *>(take(8));
        w.ca = reinterpret_cast<int32_t *>(take(4));
        w.cb = reinterpret_cast<int32_t *>(take(4));
    }
    return w;
}

struct Sweep64 {
    SolveArgs s;
    int32_t nc;              // warps' bin chunks: ceil(L Q / 32)
    int32_t nl;              // lines a chunk can touch
    int32_t kl;              // chunks a line can touch (band terms)
    int32_t skip;
    int32_t wide;            // neighbouring points may differ by more than a third of a width in velocity
    int32_t duo;             // the two halves of a pair go to two warps
    int32_t split;           // CTAs per origin, each with its share of the ray pairs
    double *part;            // split > 1: [n][split][F][4 + B] sums of each CTA
    double dmin;             // dtau_min
    PosFp half_dmin, cmin;   // dtau_min / 2 and chi_min
    double inv_chi_min;
    int64_t o0, nb;          // origins of this launch: from o0, at most nb
    double *Mpart;           // band terms of these origins: [kl][nb][L][R][B] unsummed over chunks
};

// Doubles of scratch for unsummed band terms (1 GiB). A launch covers the origins whose terms
// fit: two to five times the terms themselves would be 35 GB for 200k points, 19 lines x 63 bins and
// 192 rays at B = 2. (Those take 33 launches of 6.1k CTAs, 20 waves each.)
constexpr int64_t kBandScratch = (1ll << 30) / sizeof(double);

// One bin's sweep state and (band terms) its last two rows.
struct Bin64 {
    double P, Q, R, S;
    PosFp chi, d;
    double ph, oth;                    // profile and other sources' emissivity of the previous point
    double t1, q1, r1, ph1, ot1;       // last row: t, Q and R before it, and its far point's values
    double t2, q2, r2, ph2, ot2;
    PosFp ch1, ch2;
};

template <int B>
__device__ __forceinline__ void row64(Bin64 &z, double h, double dmin, const PosFp &half_dmin, const PosFp &chi) {
    PosFp d = pos_mul(pos_add(z.chi, chi), pos_from(h));
    double dtau = pos_pack(d.m, d.e + 1);
    if (__double_as_longlong(dtau) < __double_as_longlong(dmin)) {
        dtau = dmin;
        d = half_dmin;
    }
    const PosFp sp = pos_add(z.d, d);
    const double s = pos_pack(sp.m, sp.e);
    if constexpr (B > 0) {
        z.t2 = z.t1; z.q2 = z.q1; z.r2 = z.r1; z.ph2 = z.ph1; z.ot2 = z.ot1; z.ch2 = z.ch1;
        z.t1 = s; z.q1 = z.Q; z.r1 = z.R; z.ph1 = z.ph; z.ot1 = z.oth; z.ch1 = z.chi;
    }
    z.P = fma(s, z.Q, z.P);
    z.R = fma(s * z.S, z.Q, z.R);
    z.Q = fma(dtau, z.P, z.Q);
    z.d = d;
    // (a loop, so that no predicated FP64 instructions are issued in every row)
#pragma unroll 1
    while (__double2hiint(z.Q) >= (1023 + 256) << 20 && __double2hiint(z.Q) < 0x7ff << 20) {
        z.P *= 0x1p-256; z.Q *= 0x1p-256; z.R *= 0x1p-256;
        if constexpr (B > 0) { z.q1 *= 0x1p-256; z.r1 *= 0x1p-256; z.q2 *= 0x1p-256; z.r2 *= 0x1p-256; }
    }
}

// A magnitude with the flags of its Ye: negative (1), NaN in place of what is not finite (4).
__device__ __forceinline__ double flagged64(double v, int ye) {
    return __hiloint2double((__double2hiint(v) | ((ye & 4) ? 0x7ff80000 : 0)) ^ (ye << 31), __double2loint(v));
}

// Position of a comoving offset between the roots: segment and fraction.
__device__ __forceinline__ void bracket64(const double *x, int Q, double r, int &lo, double &t) {
    lo = 0;
    t = 0.0;
    if (Q == 1 || r <= x[0]) return;
    if (r >= x[Q - 1]) {
        lo = Q - 2;
        t = 1.0;
        return;
    }
    int hi = Q - 1;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (x[mid] <= r) lo = mid;
        else hi = mid;
    }
    t = (r - x[lo]) / (x[lo + 1] - x[lo]);
}

// chi_sca J of line l at a point: interpolated between its cells and their bins.
__device__ __forceinline__ double scattered64(const SolveArgs &a, const double *roots, int l, double x, double w,
                                              double xs, int ca, int cb) {
    int lo;
    double t;
    bracket64(roots, a.Q, x, lo, t);
    const int hi = a.Q == 1 ? lo : lo + 1;
    const double *Ja = a.Jsca + ((size_t)ca * a.L + l) * a.Q, *Jb = a.Jsca + ((size_t)cb * a.L + l) * a.Q;
    const double a0 = Ja[lo], a1 = Ja[hi], b0 = Jb[lo], b1 = Jb[hi];
    const double ja = t == 1.0 ? a1 : a0 + t * (a1 - a0), jb = t == 1.0 ? b1 : b0 + t * (b1 - b0);
    return xs * ((1.0 - w) * ja + w * jb);
}

// Bound of log2(e) x'^2 beyond which line k of the warp is far between slots i and i + 1 of the
// window, for widths with 1/b < 2^eb: its opacity X exp(-x'^2) is below chi_min and its
// emissivity below chi_min times the least intensity (binary exponents, rounded to the safe
// side): X = c ib (c/sqrt pi)/nu < 2^ec 2^eb 2^28/nu.
__device__ __forceinline__ float line_bound64(const Warp64 &W, int k, int i, int eb, int chi_min_e) {
    const double2 p0 = W.ln[32 * k + i + 1], p1 = W.ln[32 * k + i];
    const int ech = max(__double2hiint(p0.y), __double2hiint(p1.y));   // (negative: below every positive)
    const int eet = max(__double2hiint(p0.x) & 0x7fffffff, __double2hiint(p1.x) & 0x7fffffff);
    if (max(ech, eet) >= 0x7ff00000) return INFINITY;                  // (infinite or NaN: never far)
    return (float)(max(max(ech >> 20, (eet >> 20) - W.ic[k]) - 1022, -100000) + eb - chi_min_e);
}

// Sweeps half-ray r of origin o to the row next to the origin; returns false for an
// empty half. aq: the lane's a_q; lw its line within the warp's nl lines from l0.
template <int B, bool SCAT>
__device__ __forceinline__ bool sweep_half64(const Sweep64 &A, const Warp64 &W, const uint64_t *tab,
                                             const double *roots, int64_t o, int r, int l0, int nl, int lw, double aq,
                                             double nu_o, const PosFp &chi_o, float aq_lo, float aq_hi, int chi_min_e,
                                             Bin64 &z, int &rows) {
    const SolveArgs &a = A.s;
    const int lane = threadIdx.x & 31;
    const int64_t off = a.ray_off[o * a.R + r];
    const int len = (int)(a.ray_off[o * a.R + r + 1] - off);
    rows = 0;
    if (len == 0) return false;
    int top = len - 1;
    bool first = true;
    unsigned far1 = 0, far2 = 0, bin_far1 = 0, bin_far2 = 0;
    int run = 0;             // far points (at most 2) right before the window
    const float aqf = (float)aq;
    double hc = 0.0;         // h of the last element of the previous window
    const uint64_t *Xm = W.Xm + 32 * lw, *Ym = W.Ym + 32 * lw;
    const int32_t *Xe = W.Xe + 32 * lw, *Ye = W.Ye + 32 * lw;
    const double *Sr = W.S + 32 * lw;
    double inu = 0.0;
    if constexpr (B > 0) inu = 1.0 / a.lc[l0 + lw].nu;
    z.P = 1.0;
    z.Q = 1.0;
    z.d = PosFp{0, -(1 << 20)};
    for (;; top -= 31) {
        __syncwarp();
        const bool last_window = top < 31;
        const bool el = lane < 31 && lane <= top;
        int np = 0, x0 = 0;
        double hel = 0.0;
        bool near = el;
        {
            const int e = top - lane;
            const bool in = e >= 0;
            const int64_t k = off + (in ? e : 0);
            const int32_t c = in ? a.cells[k] : (int32_t)o;
            const int x1 = in ? a.xcum[k] : 0;
            const double v = in ? a.vpar[k] : 0.0, bb = a.b[c], dse = in ? a.ds[k] : 0.0;
            W.x1[lane] = x1;
            W.cell[lane] = c;
            W.v[lane] = v;
            W.b[lane] = bb;
            const double2 *lc = reinterpret_cast<const double2 *>(a.line) + (int64_t)c * a.L + l0;
            for (int i = 0; i < nl; i++) W.ln[32 * i + lane] = lc[i];
            if (first && lane == 0) W.x1[32] = x1;   // points of the half-ray
            x0 = __shfl_down_sync(0xffffffffu, x1, 1);
            np = el ? x1 - x0 : 0;
            const double rn = np > 1 ? pos_pack(pos_rcp(pos_from((double)np))) : 1.0;
            hel = dse * rn * 0.25;
            W.rn[lane] = rn;
            W.ds[lane] = hel;        // h of the element's intervals
            __syncwarp();
            // the far test of a whole element: |x'| bounded from below by the ends of its
            // velocity range over the larger width, the lines' bounds from above with the smaller
            if (A.skip) {
                const float vf = (float)v, bf = (float)bb;
                const float v0 = __shfl_down_sync(0xffffffffu, vf, 1), b0 = __shfl_down_sync(0xffffffffu, bf, 1);
                const float vlo = fminf(vf, v0), vhi = fmaxf(vf, v0);
                const float nlo = aq_lo - vhi * fmaf(aq_lo, (float)(1.0 / kC), 1.0f);
                const float nhi = aq_hi - vlo * fmaf(aq_hi, (float)(1.0 / kC), 1.0f);
                const float err = 1e-6f * (fmaxf(fabsf(aq_lo), fabsf(aq_hi)) + fmaxf(fabsf(vlo), fabsf(vhi)));
                const float xm = fmaxf(fmaxf(nlo, -nhi) - err, 0.0f) / fmaxf(bf, b0);
                const int eb = -ilogbf(fminf(bf, b0));               // 1/b <= 2^eb
                float bound = 0.0f;
                if (el)
                    for (int k2 = 0; k2 < nl; k2++) bound = fmaxf(bound, line_bound64(W, k2, lane, eb, chi_min_e));
                near = el && !(0.999f * kLog2e64 * xm * xm > bound && fabsf(vf) + fabsf(v0) < INFINITY);
                if (B > 0) near = near || (el && x0 < 3);
                if constexpr (SCAT) near = near || (el && (a.chi_sca[W.cell[lane]] != 0.0 || a.chi_sca[W.cell[lane + 1]] != 0.0));
            }
        }
        if (first) rows = W.x1[32];
        // points kept: all of near elements, the first two of a run of far ones (as in the FP32
        // kernel), numbered by a prefix sum
        const unsigned nearm = __ballot_sync(0xffffffffu, near), onem = __ballot_sync(0xffffffffu, np == 1);
        int before = run;
        if (lane >= 1) {
            if ((nearm >> (lane - 1)) & 1u) before = 0;
            else if (!((onem >> (lane - 1)) & 1u)) before = 2;
            else before = lane >= 2 ? (((nearm >> (lane - 2)) & 1u) ? 1 : 2) : min(run + 1, 2);
        }
        const int keep = near ? np : min(np, 2 - before);
        run = __shfl_sync(0xffffffffu, before, 31);
        int end = keep;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, end, d);
            if (lane >= d) end += y;
        }
        const int start = end - keep, total = __shfl_sync(0xffffffffu, end, 31);
        const unsigned kept = __ballot_sync(0xffffffffu, keep > 0);
        if (keep > 0) W.own[__popc(kept & ((1u << lane) - 1u))] = make_int4(lane, W.x1[lane] - 1 + start, x0, np);
        __syncwarp();
        for (int c0 = 0; c0 < total; c0 += 32) {
        const int cnt = min(32, total - c0);
        const int n0 = __popc(__ballot_sync(0xffffffffu, keep > 0 && start <= c0));
        const unsigned starts =
            __reduce_or_sync(0xffffffffu, (keep > 0 && start > c0 && start < c0 + 32) ? (1u << (start - c0)) : 0u);
        const int4 own = W.own[n0 - 1 + __popc(starts & (0xffffffffu >> (31 - lane)))];
        const int i = own.x, x = own.y - (c0 + lane);
        bool far = false;
        double hin = 0.0, gz = 0.0, gy = 0.0, ibk = 0.0, w = 0.0;
        float xerr = 0.0f, shrink = 1.0f, step = 0.0f;
        int eb = 0;
        if (lane < cnt) {
            const int j = x - own.z + 1;
            w = j == own.w ? 1.0 : (double)j * W.rn[i];
            const double w0 = 1.0 - w;
            const double v = w0 * W.v[i + 1] + w * W.v[i];
            const double bp = w0 * W.b[i + 1] + w * W.b[i];
            ibk = pos_pack(pos_rcp(pos_from(bp)));
            hin = j < own.w ? W.ds[i] : (i > 0 ? W.ds[i - 1] : hc);
            gy = v * ibk;
            gz = ibk - gy * (1.0 / kC);
            eb = (int)((__double2hiint(ibk) >> 20) & 0x7ff) - 1022;
            if (A.skip) {
                float bound = 0.0f;      // (far needs x'^2 > 0)
                for (int k = 0; k < nl; k++) bound = fmaxf(bound, line_bound64(W, k, i, eb, chi_min_e));
                const float gzf = (float)gz, gyf = (float)gy;
                const float ylo = aq_lo * gzf, yhi = aq_hi * gzf;
                xerr = 1e-6f * (fabsf(ylo) + fabsf(yhi) + fabsf(gyf));
                const float xlo = ylo - gyf, xhi = yhi - gyf;
                // (with the larger width of the element's ends, so that the next point, up to the
                // inner cell itself, is at the floor too: its opacity is in the line's bound)
                const float bmax = fmaxf((float)W.b[i], (float)W.b[i + 1]);
                shrink = 0.999999f * (float)bp / bmax;
                // the next point's velocity differs by `step` widths: within a third, the default, it
                // stays below 200 chi_min there (exp(2 x' / 3) at x' = 7.6)
                if (A.wide) step = 1.000001f * fabsf((float)(W.v[i] - W.v[i + 1])) * (float)W.rn[i] / bmax;
                const float xm = fmaxf(fmaxf((xlo > 0.0f ? xlo : (xhi < 0.0f ? -xhi : 0.0f)) - xerr, 0.0f) * shrink - step, 0.0f);
                far = 0.999f * kLog2e64 * xm * xm > bound;
                if (B > 0) far = far && x >= 3;
                if constexpr (SCAT) far = far && a.chi_sca[W.cell[i]] == 0.0 && a.chi_sca[W.cell[i + 1]] == 0.0;
            }
        }
        const unsigned valid = cnt == 32 ? 0xffffffffu : ((1u << cnt) - 1u);
        const unsigned fm = __ballot_sync(0xffffffffu, far) & valid;
        unsigned proc = ~(fm & ((fm << 1) | far1) & ((fm << 2) | (far1 << 1) | far2)) & valid;
        if (first) proc |= 1u;
        if (cnt >= 2) {
            far1 = (fm >> (cnt - 1)) & 1u;
            far2 = (fm >> (cnt - 2)) & 1u;
        } else {
            far2 = far1;
            far1 = fm & 1u;
        }
        if ((proc >> lane) & 1u) {
            const int j = __popc(proc & ((1u << lane) - 1u));
            W.gz[j] = gz;
            W.ngy[j] = -gy;
            W.h[j] = hin;
            bool scatters = false, beside = false;   // (beside: this point or the next may scatter)
            if constexpr (SCAT) {
                const int32_t ca = W.cell[i + 1], cb = W.cell[i];
                const double xa = a.chi_sca[ca], xb = a.chi_sca[cb], xs = (1.0 - w) * xa + w * xb;
                W.w[j] = w;
                W.xs[j] = xs;
                W.ca[j] = ca;
                W.cb[j] = cb;
                scatters = xs != 0.0;
                beside = xa != 0.0 || xb != 0.0;
            }
            for (int k = 0; k < nl; k++) {
                W.tt[32 * k + j] = make_float4(
                    (float)gz, -(float)gy, A.skip && !beside ? (sqrtf(1.001f / kLog2e64 * fmaxf(line_bound64(W, k, i, eb, chi_min_e), 0.0f)) + step) / shrink + xerr : INFINITY,
                    0.0f);
                const double2 p0 = W.ln[32 * k + i + 1], p1 = W.ln[32 * k + i];
                const double et = (1.0 - w) * p0.x + w * p1.x, ch = (1.0 - w) * p0.y + w * p1.y;
                const double nrm = a.lc[l0 + k].pnorm * ibk;      // c/(nu sqrt pi) / b
                // (a negative opacity alone ends at the floor; scattering opacity adds to it first)
                const PosFp X = ch > 0.0 || scatters ? pos_from(ch * nrm) : PosFp{0, 0};
                const PosFp Y = pos_from(et * nrm * A.inv_chi_min);
                W.Xm[32 * k + j] = X.m;
                W.Xe[32 * k + j] = X.e;
                W.Ym[32 * k + j] = Y.m;
                const bool bad = not_finite(et) || not_finite(gy);
                W.Ye[32 * k + j] = 8 * Y.e + (et < 0.0 ? 1 : 0) + (SCAT && !(ch >= 0.0) ? 2 : 0) + (bad ? 4 : 0);
                double S = 0.0;
                if (ch > 0.0) {
                    S = pos_pack(pos_mul(pos_from(et), pos_rcp(pos_from(ch))));
                    if (et < 0.0) S = -S;
                    if (not_finite(ch)) S = nan64();
                }
                if (bad) S = nan64();
                W.S[32 * k + j] = S;
            }
            if constexpr (B > 0) {
                W.N[j] = ibk * (kC / kSqrtPi);
                W.rx[j] = x;
            }
        }
        __syncwarp();
        // Each lane sweeps the points that its own bin sees: the far test and the rule of three
        // points once more per bin, as bits over the ring. The loop runs as often as the
        // busiest lane needs.
        const int nr = __popc(proc);
        const unsigned ring = nr == 32 ? 0xffffffffu : ((1u << nr) - 1u);
        unsigned todo = ring;
        if (A.skip) {
            unsigned fb = 0;
#pragma unroll 8
            for (int j = 0; j < nr; j++) {
                const float4 t4 = W.tt[32 * lw + j];
                if (fabsf(fmaf(aqf, t4.x, t4.y)) > t4.z) fb |= 1u << j;
            }
            todo = ~(fb & ((fb << 1) | bin_far1) & ((fb << 2) | (bin_far1 << 1) | bin_far2)) & ring;
            if (first) todo |= 1u;
            if constexpr (B > 0)
                for (int j = 0; j < nr; j++)
                    if (W.rx[j] < 3) todo |= 1u << j;
            if (nr >= 2) {
                bin_far1 = (fb >> (nr - 1)) & 1u;
                bin_far2 = (fb >> (nr - 2)) & 1u;
            } else if (nr == 1) {
                bin_far2 = bin_far1;
                bin_far1 = fb & 1u;
            }
        }
        while (__any_sync(0xffffffffu, todo != 0)) {
            if (!todo) continue;
            const int j = __ffs(todo) - 1;
            todo &= todo - 1;
            const double gzj = W.gz[j], ngyj = W.ngy[j];
            double xp = fma(aq, gzj, ngyj);
            const double xr = xp;
            if ((__double2hiint(xp) & 0x7fffffff) >= 0x404a0000) xp = 52.0;   // exp(-52^2) is zero
            int n;
            const uint64_t e = exp_neg_sq(xp, tab, n);
            // X e: significands in units of 2^-63, e in [2^62, 2^63]
            PosFp chi = pos_norm(mulhi_near(Xm[j], e), Xe[j] + 1 - n);
            double S = Sr[j], oth = 0.0;
            const double xs = SCAT ? W.xs[j] : 0.0;
            if (SCAT && xs != 0.0) {
                oth = scattered64(a, roots, l0 + lw, xr, W.w[j], xs, W.ca[j], W.cb[j]);
                const int ye = Ye[j];
                const double cl = pos_pack(chi.m, chi.e);
                const double c = __hiloint2double(__double2hiint(cl) ^ ((ye & 2) << 30), __double2loint(cl)) + xs;
                chi = pos_from(pos_max(c, a.chi_min));   // (a negative sum is below it as bits too)
                // line emissivity: Y chi_min e
                double et = pos_pack(mulhi_near(Ym[j], e), (ye >> 3) + 1 - n) * a.chi_min;
                et = flagged64(et, ye);
                S = (et + oth) * pos_pack(pos_rcp(chi));
            } else if (chi.m == 0 || chi.e < A.cmin.e || (chi.e == A.cmin.e && chi.m < A.cmin.m)) {
                chi = A.cmin;
                const int ye = Ye[j];
                S = pos_pack(mulhi_near(Ym[j], e), (ye >> 3) + 1 - n);
                S = flagged64(S, ye);
            }
            if (first && j == 0) {
                // the far end: the boundary row starts from Phi iota = 1, psi = I, delta = 0
                const double pz = gzj - ngyj * (1.0 / kC);   // gz + gy/c
                z.R = planck_d(nu_o * (1.0 + ngyj / pz * (1.0 / kC)), a.T_cmb);
            } else {
                row64<B>(z, W.h[j], A.dmin, A.half_dmin, chi);
            }
            z.chi = chi;
            z.S = S;
            if constexpr (B > 0) {
                z.oth = oth;
                if (W.rx[j] < 2) {
                    const PosFp N = pos_from(W.N[j] * inu);
                    z.ph = pos_pack(mulhi_near(N.m, e), N.e + 1 - n);
                }
            }
        }
        first = false;
        __syncwarp();
        }
        hc = __shfl_sync(0xffffffffu, hel, last_window ? top : 30);
        if (last_window) break;
    }
    row64<B>(z, hc, A.dmin, A.half_dmin, chi_o);   // the origin
    return true;
}

// Barrier of the two warps of a unit (named barriers 1 .. 8).
__device__ __forceinline__ void pair_barrier(int id) {
    asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}

template <int B, bool SCAT>
__global__ void __launch_bounds__(512) k_feautrier64w(Sweep64 A) {
    extern __shared__ __align__(16) unsigned char smem64[];
    constexpr int NA = 4 + B;
    const SolveArgs &a = A.s;
    const int L = a.L, Q = a.Q, F = L * Q;
    // a unit is a warp, or two warps that sweep one half of each pair each
    const int nu = (blockDim.x >> 5) >> A.duo, warp = threadIdx.x >> 5, unit = warp >> A.duo, lane = threadIdx.x & 31;
    const int half = A.duo ? warp & 1 : 2;
    const int ob = blockIdx.x / A.split, share = blockIdx.x - ob * A.split;
    int64_t o = B > 0 ? A.o0 + ob : ob;   // (only band terms need several launches)
    if (a.olist) {
        if ((int)blockIdx.x >= *a.ocount) return;
        o = a.olist[blockIdx.x];
    }
    uint64_t *tab = reinterpret_cast<uint64_t *>(smem64);
    double *roots = reinterpret_cast<double *>(tab + 256);       // scattering: the roots
    double *acc_all = roots + (SCAT ? Q : 0);                    // [G][F][NA]
    const int G = a.groups;
    const size_t wb = warp64_bytes(A.nl, B, SCAT);
    unsigned char *wbase = reinterpret_cast<unsigned char *>(acc_all + (size_t)G * F * NA);
    wbase += (16 - ((uintptr_t)wbase & 15)) & 15;
    const Warp64 W = carve64(wbase + warp * wb, A.nl, B, SCAT);
    constexpr int NX = 4 + 8 * (B > 0);                          // values handed from one half to the other
    double *xch = reinterpret_cast<double *>(wbase + (blockDim.x >> 5) * wb) + (size_t)unit * 32 * NX + lane;
    for (int t = threadIdx.x; t < 256; t += blockDim.x) tab[t] = kExp2Table.t[t];
    if (SCAT)
        for (int t = threadIdx.x; t < Q; t += blockDim.x) roots[t] = a.roots[t];
    __syncthreads();
    const double bo = a.b[o], ibo = 1.0 / bo, invP = 1.0 / a.P;
    const int g = G > 1 ? unit / A.nc : 0;
    double *acc = acc_all + (size_t)g * F * NA;
    for (int c = G > 1 ? unit % A.nc : unit; c < A.nc; c += G > 1 ? A.nc : nu) {
        const int f = min(32 * c + lane, F - 1);
        const int l = f / Q, q = f - l * Q;
        const int l0 = 32 * c / Q, nl = min(32 * c + 31, F - 1) / Q - l0 + 1;
        const double aq = a.roots[q] * bo;
        const double k1 = 1.0 + aq / kC;
        const double nu_o = a.lc[l].nu * k1;
        float aq_lo = (float)aq, aq_hi = (float)aq;
        float nu_lo = (float)a.lc[l].nu;
        for (int d = 16; d; d >>= 1) {
            aq_lo = fminf(aq_lo, __shfl_xor_sync(0xffffffffu, aq_lo, d));
            aq_hi = fmaxf(aq_hi, __shfl_xor_sync(0xffffffffu, aq_hi, d));
            nu_lo = fminf(nu_lo, __shfl_xor_sync(0xffffffffu, nu_lo, d));
        }
        // floor test (see the staging): exponents of chi_min nu / 2^28 and of the least intensity,
        // rounded down
        __syncwarp();
        if (lane < nl) W.ic[lane] = least_exponent(ilogb(planck_d(a.lc[l0 + lane].nu, a.T_cmb)), a.least[l0 + lane]);
        const int chi_min_e = ilogb(a.chi_min) + ilogbf(nu_lo) - 28 - 1;
        // the origin's opacity and source in this bin
        const double x0 = aq * ibo;
        const double phi = exp(-x0 * x0) * (a.lc[l].pnorm * ibo);
        const double etal = a.line[(o * L + l) * 2] * phi, chil = a.line[(o * L + l) * 2 + 1] * phi;
        double eta = etal, chi = chil;
        if constexpr (SCAT) {
            const double xs = a.chi_sca[o];
            if (xs != 0.0) {
                chi += xs;
                eta += scattered64(a, roots, l, x0, 0.0, xs, (int)o, (int)o);
            }
        }
        chi = fmax(chi, a.chi_min);
        const PosFp chi_pf = pos_from(chi);
        const double ichi = 1.0 / chi;
        const double So = eta * ichi;
        const double own = chil * ichi, rest = (chi - chil) * ichi, oth = (eta - etal) * ichi;
        double s_u = 0.0, s_l = 0.0, s_e = 0.0, s_c = 0.0, s_b[2] = {0.0, 0.0};
        for (int p = share + g * A.split; p < a.P; p += G * A.split) {
            const int rf = a.pf[p], rb = a.pb[p];
            Bin64 z{};
            // per half: Phi iota, psi, delta, whether it has rows, and the band terms
            // (g, r, phi/chi, other sources) of the last two rows
            double va[NX], vb[NX];
#pragma unroll 1
            for (int side = half == 1 ? 1 : 0; side < (half == 0 ? 1 : 2); side++) {
                int rows = 0;
                const bool full = sweep_half64<B, SCAT>(A, W, tab, roots, o, side ? rf : rb, l0, nl, l - l0, aq, nu_o,
                                                        chi_pf, aq_lo, aq_hi, chi_min_e, z, rows);
                double v[NX];
                v[3] = full;
                if (full) {
                    const double iq = 1.0 / z.Q;
                    v[0] = z.P * iq;
                    v[1] = z.R * iq;
                    v[2] = pos_pack(z.d.m, z.d.e);
                    if constexpr (B > 0) {
                        // psi after the last row is g_1 S_m + g_2 S_{m-1} + r_2 with
                        // iota_k = Q before / Q after: g_1 = t Q_in/Q_out, r_1 = R_in/Q_out
                        const double ic1 = pos_pack(pos_rcp(z.ch1));
                        v[4] = z.t1 * z.q1 * iq;
                        v[6] = z.r1 * iq;
                        v[8] = z.ph1 * ic1;
                        v[10] = z.ot1 * ic1;
                        v[5] = 0.0;
                        v[7] = v[6];
                        v[9] = v[11] = 0.0;
                        if (rows >= 2) {
                            const double ic2 = pos_pack(pos_rcp(z.ch2));
                            v[5] = z.t2 * z.q2 * iq;
                            v[7] = z.r2 * iq;
                            v[9] = z.ph2 * ic2;
                            v[11] = z.ot2 * ic2;
                        }
                    }
                } else {
                    v[0] = 1.0;
                    v[1] = planck_d(nu_o, a.T_cmb);
                    v[2] = 0.0;
                    if constexpr (B > 0) {
                        v[4] = v[5] = v[8] = v[9] = v[10] = v[11] = 0.0;
                        v[6] = v[7] = v[1];
                    }
                }
                if (half == 0) {        // hand over to the other warp
#pragma unroll
                    for (int k = 0; k < NX; k++) xch[32 * k] = v[k];
                    continue;
                }
                if (side == 0) {
#pragma unroll
                    for (int k = 0; k < NX; k++) va[k] = v[k];
                } else {
#pragma unroll
                    for (int k = 0; k < NX; k++) vb[k] = v[k];
                }
            }
            if (half != 2) {                // the other half has been written, and read
                pair_barrier(1 + unit);
                if (half == 1) {
#pragma unroll
                    for (int k = 0; k < NX; k++) va[k] = xch[32 * k];
                }
                pair_barrier(1 + unit);
                if (half == 0) continue;
            }
            const bool any = va[3] + vb[3] != 0.0;
            const double pi[2] = {va[0], vb[0]}, ps[2] = {va[1], vb[1]}, dl[2] = {va[2], vb[2]};
            double gg[2][2], rr[2][2], hh[2][2], so[2][2];
            if constexpr (B > 0) {
#pragma unroll
                for (int j = 0; j < 2; j++) {
                    gg[0][j] = va[4 + j]; rr[0][j] = va[6 + j]; hh[0][j] = va[8 + j]; so[0][j] = va[10 + j];
                    gg[1][j] = vb[4 + j]; rr[1][j] = vb[6 + j]; hh[1][j] = vb[8 + j]; so[1][j] = vb[10 + j];
                }
            }
            double u, lam, uml, oml, jb[2] = {0.0, 0.0}, sD = 0.0;
            if (!any) {
                const double I = planck_d(nu_o, a.T_cmb);
                u = I; lam = 0.0; uml = I; oml = 1.0;
                jb[0] = jb[1] = I;
            } else {
                // sigma = 2/(dtau_- + dtau_+)
                const double sig = 1.0 / (dl[0] + dl[1]);
                const double pi2 = sig * (pi[0] + pi[1]);
                const double iD = 1.0 / (1.0 + pi2);
                lam = iD;
                uml = sig * (ps[0] + ps[1]) * iD;
                oml = pi2 * iD;
                u = So * iD + uml;
                sD = sig * iD;
                if constexpr (B > 0) {
                    jb[0] = sD * (gg[0][0] * so[0][0] + rr[0][0] + gg[1][0] * so[1][0] + rr[1][0]);
                    if constexpr (B > 1)
                        jb[1] = sD * (gg[0][0] * so[0][0] + gg[0][1] * so[0][1] + rr[0][1] + gg[1][0] * so[1][0] +
                                      gg[1][1] * so[1][1] + rr[1][1]);
                }
            }
            const double lo = lam * oth;
            s_u += u;
            s_l += lam * own;
            s_e += uml + lo;
            s_c += oml + lam * rest;
            for (int j = 0; j < B; j++) s_b[j] += jb[j] + lo;
            if constexpr (B > 0) {
                // coupling terms of the band points: weighted sums over the chunk's bins of
                // each line, in lane order
                const double wq = 32 * c + lane < F ? a.weights[q] : 0.0;
                __syncwarp();
                for (int j = 0; j < B; j++) {
                    W.mac[lane * 2 * B + j] = any ? wq * (sD * gg[0][j] * hh[0][j]) : 0.0;
                    W.mac[lane * 2 * B + B + j] = any ? wq * (sD * gg[1][j] * hh[1][j]) : 0.0;
                }
                __syncwarp();
                for (int tk = lane; tk < 2 * B * nl; tk += 32) {
                    const int k = tk / (2 * B), sj = tk - k * 2 * B, ll = l0 + k;
                    const int f0 = max(ll * Q, 32 * c), f1 = min(min((ll + 1) * Q, 32 * c + 32), F);
                    double s = 0.0;
                    for (int ff = f0; ff < f1; ff++) s += W.mac[(ff - 32 * c) * 2 * B + sj];
                    const int side = sj / B, j = sj - side * B, part = c - ll * Q / 32;
                    A.Mpart[((((size_t)part * A.nb + ob) * L + ll) * a.R + (side ? rf : rb)) * B + j] = s;
                }
                __syncwarp();
            }
        }
        if (half != 0 && 32 * c + lane < F) {
            acc[NA * f + 0] = s_u;
            acc[NA * f + 1] = s_l;
            acc[NA * f + 2] = s_e;
            acc[NA * f + 3] = s_c;
            for (int j = 0; j < B; j++) acc[NA * f + 4 + j] = s_b[j];
        }
    }
    __syncthreads();
    if (A.split > 1) {   // k_sums64 adds the shares and the bins
        double *dst = A.part + ((size_t)o * A.split + share) * F * NA;
        for (int t = threadIdx.x; t < F * NA; t += blockDim.x) {
            double v = acc_all[t];
            for (int gg = 1; gg < G; gg++) v += acc_all[(size_t)gg * NA * F + t];
            dst[t] = v;
        }
        return;
    }
    for (int tt = threadIdx.x; tt < NA * L; tt += blockDim.x) {
        const int l = tt / NA, k = tt - l * NA;
        double s = 0.0;
        for (int q = 0; q < Q; q++) {
            double v = acc_all[NA * (l * Q + q) + k];
            for (int gg = 1; gg < G; gg++) v += acc_all[(size_t)gg * NA * F + NA * (l * Q + q) + k];
            s += a.weights[q] * v;
        }
        s *= invP;
        double *dst = k == 0 ? a.J : (k == 1 ? a.Lout : (k == 2 ? a.Jeff : (k == 3 ? a.Lc : a.Jeffb + (size_t)(k - 4) * a.n * L)));
        dst[o * L + l] = s;
    }
    if (a.Jnu)
        for (int f = threadIdx.x; f < F; f += blockDim.x) {
            double v = acc_all[NA * f];
            for (int gg = 1; gg < G; gg++) v += acc_all[(size_t)gg * NA * F + NA * f];
            a.Jnu[o * F + f] = v * invP;
        }
}

// Sums of an origin whose ray pairs were shared among CTAs: one warp per (origin, line), the
// shares in order, the bins over the lanes and a shuffle tree.
template <int NA>
__global__ void __launch_bounds__(128) k_sums64(SolveArgs a, int split, const double *__restrict__ part) {
    const int lane = threadIdx.x & 31, L = a.L, Q = a.Q, F = L * Q;
    const int64_t ol = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (ol >= a.n * L) return;
    const int64_t o = ol / L;
    const int l = (int)(ol - o * L);
    const double invP = 1.0 / a.P;
    double s[NA];
#pragma unroll
    for (int k = 0; k < NA; k++) s[k] = 0.0;
    for (int q = lane; q < Q; q += 32) {
        const double *p = part + ((size_t)o * split * F + l * Q + q) * NA;
        double v[NA];
#pragma unroll
        for (int k = 0; k < NA; k++) v[k] = p[k];
        for (int sh = 1; sh < split; sh++)
#pragma unroll
            for (int k = 0; k < NA; k++) v[k] += p[(size_t)sh * F * NA + k];
        if (a.Jnu) a.Jnu[o * F + l * Q + q] = v[0] * invP;
        const double w = a.weights[q];
#pragma unroll
        for (int k = 0; k < NA; k++) s[k] += w * v[k];
    }
#pragma unroll
    for (int k = 0; k < NA; k++) {
        for (int d = 16; d; d >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], d);
        if (lane == 0) {
            double *dst = k == 0 ? a.J : (k == 1 ? a.Lout : (k == 2 ? a.Jeff : (k == 3 ? a.Lc : a.Jeffb + (size_t)(k - 4) * a.n * L)));
            dst[ol] = s[k] * invP;
        }
    }
}

// Coupling terms of a launch's origins (m of them): the sum over each line's chunks, times
// chi_int(o)/P.
__global__ void k_band_terms64(Sweep64 A, int64_t m, int L, int R, int B) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = A.nb * L * R * B;
    if (t >= m) return;
    const int64_t ol = A.o0 * L + t / (R * B);
    const int l = (int)(ol % L), Q = A.s.Q;
    const int np = (l * Q + Q - 1) / 32 - l * Q / 32 + 1;
    double s = 0.0;
    for (int k = 0; k < np; k++) s += A.Mpart[k * stride + t];
    A.s.Mb[A.o0 * L * R * B + t] = s * (1.0 / A.s.P) * A.s.line[2 * ol + 1];
}

}  // namespace
