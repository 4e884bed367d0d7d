// The FP64 formal solve for lines that do not overlap (included by solve.cu).
//
// One CTA per origin. Its warps share the bins of the point (32 consecutive bins of the
// flattened (line, bin) list per warp) and, when there are few bins, the ray pairs; each
// warp sweeps its pairs through a private ring of staged points and needs no CTA barrier
// until the final sums.
//
// What bounds it. A warp-wide FP64 instruction occupies an SM sub-partition's FP64 pipe for
// about 80 cycles (0.50 T DFMA/s), so FP64 instructions are the cost and everything else
// is nearly free. Per point and bin the sweep needs 8 of them:
//   x' = a_q g_z - g_y;  delta = (chi_prev + chi) h (2);  s = delta_prev + delta;
//   P = s Q + P;  R = (s S_prev) Q + R (2);  Q = delta P + Q.
// - The recursion is homogeneous: with Phi iota = P/Q and psi = R/Q the point update of
//   k_feautrier64 needs no reciprocal, and every term stays a sum of non-negative
//   numbers. (P, Q, R) are scaled by 2^-256 when Q exceeds 2^256. delta, P, R carry the factors 1/sqrt 2, sqrt 2, sqrt 2 of the FP32
//   kernel, so that no factor 1/2 is left.
// - The profile exponential, the line opacity and the floors run on the integer pipe
//   (posfp.cuh); so do the divisions of the staging.
// - S = eta/chi of a line does not depend on the bin: one division per staged point.
// - A point whose own and two previous points are far (opacity below chi_min and emission
//   below chi_min times the boundary intensity in every bin of the warp) changes the sweep
//   by O(chi_min ds) and is left out while chi_min times the longest path through the
//   model stays below 1e-14 (`skip`).
//
// The general kernel k_feautrier64 (a bin sums several lines) takes, per point and bin, an
// exponential (16 DFMA), two divisions (8 each), four interpolations and ~15 further
// operations, and sweeps every point. Measured, one ALI step, general kernel -> this one:
// clumpy cloud of 1500 points, 48 rays, 4 x 31 bins 174.9 -> 11.1 ms (with 69 % of the
// points far); with the band ALO (600 points) 124.8 -> 6.6 ms; spherical cloud of 200 shells
// (nothing far, latency of few warps) 1.64 -> 0.45 ms; one scattering pass of a 200-point
// cloud 7.1 -> 1.9 ms.
namespace {

constexpr double kSqrtLog2e64 = 1.2011224087864497947;
constexpr double kSqrt2_64 = 1.4142135623730950488;

// Larger of two non-negative doubles, on their bits.
__device__ __forceinline__ double pos_max(double a, double b) {
    return __double_as_longlong(a) > __double_as_longlong(b) ? a : b;
}

// Per-warp shared memory: an element window (as in the FP32 kernel: slot i holds element
// top - i, slot 31 only precedes slot 30; element -1 is the origin) and the ring of points.
struct Warp64 {
    int32_t *x1, *cell;
    double *v, *b, *ds;
    double2 *ln;                 // [nl][32] (eta, chi)
    double *gz, *ngy, *h;        // ring: x' = a_q gz + ngy; h of the interval from the previous point
    uint64_t *Xm, *Ym;           // [nl][32] line opacity X and floored source Y = eta/chi_min at line centre
    int32_t *Xe, *Ye;            //   (exponents; Ye holds 2 e + sign)
    double *S;                   // [nl][32]
    double *N;                   // ring: profile normalisation without 1/nu (band terms)
    int32_t *rx;                 // ring: point index (band terms)
    double *w, *xs;              // ring: weight, scattering opacity
    int32_t *ca, *cb;            // ring: cells (scattering)
    double *mac;                 // [32][2 B]
    int32_t *ic;                 // [nl] exponent of the boundary intensity at the line, rounded down
};

__host__ __device__ inline size_t warp64_bytes(int nl, int B, bool sca) {
    return (size_t)32 * (8 + 24 + 16 * nl + 24 + 32 * nl + 4) + (B ? 32 * (8 + 8 + 16 * B) : 0) + (sca ? 32 * 24 : 0);
}

__device__ __forceinline__ Warp64 carve64(unsigned char *p, int nl, int B, bool sca) {
    Warp64 w{};
    auto take = [&](size_t bytes) { unsigned char *q = p; p += 32 * bytes; return q; };
    w.ln = reinterpret_cast<double2 *>(take(16 * nl));
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
    w.x1 = reinterpret_cast<int32_t *>(take(4));
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
    double dmin;             // dtau_min / sqrt 2
    double inv_chi_min;
    double *Mpart;           // band terms: [kl][n][L][R][B] unsummed over chunks
};

// One bin's sweep state and (band terms) its last two rows.
struct Bin64 {
    double P, Q, R, chi, S, d;
    double ph, oth;                    // profile and other sources' emissivity of the previous point
    double t1, q1, r1, ph1, ot1, ch1;  // last row: s, Q and R before it, and its far point's values
    double t2, q2, r2, ph2, ot2, ch2;
};

template <int B>
__device__ __forceinline__ void row64(Bin64 &z, double h, double dmin, double chi) {
    const double dl = pos_max((z.chi + chi) * h, dmin);
    const double s = z.d + dl;
    if constexpr (B > 0) {
        z.t2 = z.t1; z.q2 = z.q1; z.r2 = z.r1; z.ph2 = z.ph1; z.ot2 = z.ot1; z.ch2 = z.ch1;
        z.t1 = s; z.q1 = z.Q; z.r1 = z.R; z.ph1 = z.ph; z.ot1 = z.oth; z.ch1 = z.chi;
    }
    z.P = fma(s, z.Q, z.P);
    z.R = fma(s * z.S, z.Q, z.R);
    z.Q = fma(dl, z.P, z.Q);
    z.d = dl;
    // (a loop, so that no predicated FP64 instructions are issued in every row)
#pragma unroll 1
    while (__double2hiint(z.Q) >= (1023 + 256) << 20 && __double2hiint(z.Q) < 0x7ff << 20) {
        z.P *= 0x1p-256; z.Q *= 0x1p-256; z.R *= 0x1p-256;
        if constexpr (B > 0) { z.q1 *= 0x1p-256; z.r1 *= 0x1p-256; z.q2 *= 0x1p-256; z.r2 *= 0x1p-256; }
    }
}

// Position of a comoving offset between the (scaled) roots: segment and fraction.
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

// Sweeps half-ray r of origin o to the row next to the origin; returns false for an
// empty half. aq: the lane's a_q; lw its line within the warp's nl lines from l0.
template <int B, bool SCAT>
__device__ __forceinline__ bool sweep_half64(const Sweep64 &A, const Warp64 &W, const uint64_t *tab,
                                             const double *roots, int64_t o, int r, int l0, int nl, int lw, double aq,
                                             double nu_o, double chi_o, float aq_lo, float aq_hi, int chi_min_e,
                                             Bin64 &z, int &rows) {
    const SolveArgs &a = A.s;
    const int lane = threadIdx.x & 31;
    const int64_t off = a.ray_off[o * a.R + r];
    const int len = (int)(a.ray_off[o * a.R + r + 1] - off);
    rows = 0;
    if (len == 0) return false;
    int top = len - 1, xnext = -1;
    bool first = true, fresh = true;
    unsigned far1 = 0, far2 = 0;
    double hprev = 0.0;      // h of the last point of the previous refill
    const uint64_t *Xm = W.Xm + 32 * lw, *Ym = W.Ym + 32 * lw;
    const int32_t *Xe = W.Xe + 32 * lw, *Ye = W.Ye + 32 * lw;
    const double *Sr = W.S + 32 * lw;
    double inu = 0.0;
    if constexpr (B > 0) inu = 1.0 / a.lc[l0 + lw].nu;
    z.P = kSqrt2_64;
    z.Q = 1.0;
    z.d = 0.0;
    do {
        __syncwarp();
        if (fresh) {
            const int e = top - lane;
            const bool in = e >= 0;
            const int64_t k = off + (in ? e : 0);
            const int32_t c = in ? a.cells[k] : (int32_t)o;
            W.x1[lane] = in ? a.xcum[k] : 0;
            W.cell[lane] = c;
            W.v[lane] = in ? a.vpar[k] : 0.0;
            W.ds[lane] = in ? a.ds[k] : 0.0;
            W.b[lane] = a.b[c];
            const double2 *lc = reinterpret_cast<const double2 *>(a.line) + (int64_t)c * a.L + l0;
            for (int i = 0; i < nl; i++) W.ln[32 * i + lane] = lc[i];
            __syncwarp();
            if (first) {
                xnext = W.x1[0] - 1;
                rows = xnext + 1;
            }
            fresh = false;
        }
        // owner slot of each lane's point (see the FP32 kernel)
        const int pos = xnext - W.x1[lane] + 1;
        const bool slot_ok = lane < 31 && top - lane >= 0;
        const int n0 = __popc(__ballot_sync(0xffffffffu, slot_ok && pos <= 0));
        const unsigned starts = __reduce_or_sync(0xffffffffu, (slot_ok && pos > 0 && pos < 32) ? (1u << pos) : 0u);
        const int i = n0 - 1 + __popc(starts & (0xffffffffu >> (31 - lane)));
        const int xw = W.x1[31];
        const int cnt = min(32, xnext - xw + 1);
        const int x = xnext - lane;
        bool far = false;
        double hcur = 0.0, gz = 0.0, gy = 0.0, ibk = 0.0, w = 0.0;
        if (lane < cnt) {
            const int x0 = W.x1[i + 1], ns = W.x1[i] - x0;
            const double rn = ns == 1 ? 1.0 : pos_pack(pos_rcp(pos_from((double)ns)));
            w = x - x0 + 1 == ns ? 1.0 : (double)(x - x0 + 1) * rn;
            const double v = (1.0 - w) * W.v[i + 1] + w * W.v[i];
            ibk = pos_pack(pos_rcp(pos_from((1.0 - w) * W.b[i + 1] + w * W.b[i])));
            hcur = W.ds[i] * rn * (0.25 * kSqrt2_64);
            const double pz = kSqrtLog2e64 * ibk;
            gy = v * pz;
            gz = pz - gy * (1.0 / kC);
        }
        if (A.skip) {
            // far: over the bins' range of a_q the largest line opacity is below chi_min and the
            // largest line emissivity below chi_min times the boundary intensity (binary
            // exponents, rounded to the safe side)
            if (lane < cnt) {
                int emax = -100000;
                for (int k = 0; k < nl; k++) {
                    const double2 p0 = W.ln[32 * k + i + 1], p1 = W.ln[32 * k + i];
                    const int ech = max(__double2hiint(p0.y), __double2hiint(p1.y));   // (negative: below every positive)
                    const int eet = max(__double2hiint(p0.x) & 0x7fffffff, __double2hiint(p1.x) & 0x7fffffff);
                    emax = max(emax, max(ech >> 20, (eet >> 20) - W.ic[k]) - 1022);
                }
                // X = c ib (c/sqrt pi)/nu < 2^emax 2^eb 2^28/nu
                const int eb = (int)((__double2hiint(ibk) >> 20) & 0x7ff) - 1022;
                const float gzf = (float)gz, gyf = (float)gy;
                const float ylo = aq_lo * gzf, yhi = aq_hi * gzf;
                const float xlo = ylo - gyf, xhi = yhi - gyf;
                const float xm = (xlo > 0.0f ? xlo : (xhi < 0.0f ? -xhi : 0.0f)) -
                                 1e-6f * (fabsf(ylo) + fabsf(yhi) + fabsf(gyf));
                far = xm > 0.0f && (float)(emax + eb - chi_min_e) < 0.999f * xm * xm;
                if constexpr (SCAT) far = far && a.chi_sca[W.cell[i]] == 0.0 && a.chi_sca[W.cell[i + 1]] == 0.0;
            }
        }
        const unsigned valid = cnt == 32 ? 0xffffffffu : ((1u << cnt) - 1u);
        const unsigned fm = __ballot_sync(0xffffffffu, far) & valid;
        const unsigned f1 = (fm << 1) | far1, f2 = (fm << 2) | (far1 << 1) | far2;
        unsigned proc = ~(fm & f1 & f2) & valid;
        if (first) proc |= 1u;
        if (B > 0 && xnext - cnt < 2) {   // the rows next to the origin are always kept
            const int j0 = max(0, xnext - 2);
            proc |= (j0 < 32 ? 0xffffffffu << j0 : 0u) & valid;
        }
        if (cnt >= 2) {
            far1 = (fm >> (cnt - 1)) & 1u;
            far2 = (fm >> (cnt - 2)) & 1u;
        } else {
            far2 = far1;
            far1 = fm & 1u;
        }
        double hin = __shfl_up_sync(0xffffffffu, hcur, 1);
        if (lane == 0) hin = hprev;
        hprev = __shfl_sync(0xffffffffu, hcur, cnt - 1);
        if ((proc >> lane) & 1u) {
            const int j = __popc(proc & ((1u << lane) - 1u));
            W.gz[j] = gz;
            W.ngy[j] = -gy;
            W.h[j] = hin;
            for (int k = 0; k < nl; k++) {
                const double2 p0 = W.ln[32 * k + i + 1], p1 = W.ln[32 * k + i];
                const double et = (1.0 - w) * p0.x + w * p1.x, ch = (1.0 - w) * p0.y + w * p1.y;
                const double nrm = a.lc[l0 + k].pnorm * ibk;      // c/(nu sqrt pi) / b
                const PosFp X = ch > 0.0 ? pos_from(ch * nrm) : PosFp{0, 0};
                const PosFp Y = pos_from(et * nrm * A.inv_chi_min);
                W.Xm[32 * k + j] = X.m;
                W.Xe[32 * k + j] = X.e;
                W.Ym[32 * k + j] = Y.m;
                W.Ye[32 * k + j] = 2 * Y.e + (et < 0.0 ? 1 : 0);
                double S = 0.0;
                if (ch > 0.0) {
                    S = pos_pack(pos_mul(pos_from(et), pos_rcp(pos_from(ch))));
                    if (et < 0.0) S = -S;
                }
                W.S[32 * k + j] = S;
            }
            if constexpr (B > 0) {
                W.N[j] = ibk * (kC / kSqrtPi);
                W.rx[j] = x;
            }
            if constexpr (SCAT) {
                const int32_t ca = W.cell[i + 1], cb = W.cell[i];
                W.w[j] = w;
                W.xs[j] = (1.0 - w) * a.chi_sca[ca] + w * a.chi_sca[cb];
                W.ca[j] = ca;
                W.cb[j] = cb;
            }
        }
        __syncwarp();
        const int np = __popc(proc);
        for (int j = 0; j < np; j++) {
            const double gzj = W.gz[j], ngyj = W.ngy[j];
            double xp = fma(aq, gzj, ngyj);
            const double xr = xp;
            if ((__double2hiint(xp) & 0x7fffffff) >= 0x404f8000) xp = 63.0;   // 2^(-63^2) is zero
            int n;
            const uint64_t e = exp2_neg_sq(xp, tab, n);
            // X e: significands in units of 2^-63, e in [2^62, 2^63]
            double chi = pos_pack(__umul64hi(Xm[j], e), Xe[j] + 1 - n);
            double S = Sr[j], oth = 0.0;
            const double xs = SCAT ? W.xs[j] : 0.0;
            if (SCAT && xs != 0.0) {   // (the same for the whole warp)
                oth = scattered64(a, roots, l0 + lw, xr, W.w[j], xs, W.ca[j], W.cb[j]);
                chi = pos_max(chi + xs, a.chi_min);
                // line emissivity: Y chi_min e
                const int ye = Ye[j];
                double et = pos_pack(__umul64hi(Ym[j], e), (ye >> 1) + 1 - n) * a.chi_min;
                if (ye & 1) et = -et;
                S = (et + oth) * pos_pack(pos_rcp(pos_from(chi)));
            } else if (__double_as_longlong(chi) < __double_as_longlong(a.chi_min)) {
                chi = a.chi_min;
                const int ye = Ye[j];
                S = pos_pack(__umul64hi(Ym[j], e), (ye >> 1) + 1 - n);
                if (ye & 1) S = -S;
            }
            if (first && j == 0) {
                // the far end: the boundary row starts from Phi iota = 1, psi = I, delta = 0
                const double pz = gzj - ngyj * (1.0 / kC);   // gz + gy/c
                z.R = kSqrt2_64 * planck_d(nu_o * (1.0 + ngyj / pz * (1.0 / kC)), a.T_cmb);
            } else {
                row64<B>(z, W.h[j], A.dmin, chi);
            }
            z.chi = chi;
            z.S = S;
            if constexpr (B > 0) {
                z.oth = oth;
                if (W.rx[j] < 2) {
                    const PosFp N = pos_from(W.N[j] * inu);
                    z.ph = pos_pack(__umul64hi(N.m, e), N.e + 1 - n);
                }
            }
        }
        first = false;
        xnext -= cnt;
        if (xnext >= 0 && xnext < xw) {
            top -= 31;
            fresh = true;
        }
    } while (xnext >= 0);
    row64<B>(z, hprev, A.dmin, chi_o);   // the origin
    return true;
}

template <int B, bool SCAT>
__global__ void __launch_bounds__(512) k_feautrier64w(Sweep64 A) {
    extern __shared__ __align__(16) unsigned char smem64[];
    constexpr int NA = 4 + B;
    const SolveArgs &a = A.s;
    const int L = a.L, Q = a.Q, F = L * Q;
    const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int64_t o = blockIdx.x;
    if (a.olist) {
        if ((int)blockIdx.x >= *a.ocount) return;
        o = a.olist[blockIdx.x];
    }
    uint64_t *tab = reinterpret_cast<uint64_t *>(smem64);
    double *roots = reinterpret_cast<double *>(tab + 256);       // scattering: roots sqrt(log2 e)
    double *acc_all = roots + (SCAT ? Q : 0);                    // [G][F][NA]
    const int G = a.groups;
    const size_t wb = warp64_bytes(A.nl, B, SCAT);
    unsigned char *wbase = reinterpret_cast<unsigned char *>(acc_all + (size_t)G * F * NA);
    wbase += (16 - ((uintptr_t)wbase & 15)) & 15;
    const Warp64 W = carve64(wbase + warp * wb, A.nl, B, SCAT);
    for (int t = threadIdx.x; t < 256; t += blockDim.x) tab[t] = kExp2Table.t[t];
    if (SCAT)
        for (int t = threadIdx.x; t < Q; t += blockDim.x) roots[t] = a.roots[t] * kSqrtLog2e64;
    __syncthreads();
    const double bo = a.b[o], ibo = 1.0 / bo, invP = 1.0 / a.P;
    const int g = G > 1 ? warp / A.nc : 0;
    double *acc = acc_all + (size_t)g * F * NA;
    for (int c = G > 1 ? warp % A.nc : warp; c < A.nc; c += G > 1 ? A.nc : nw) {
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
        // floor test (see the staging): exponents of chi_min nu / 2^28 and of the boundary
        // intensity, rounded down
        __syncwarp();
        if (lane < nl) W.ic[lane] = ilogb(planck_d(a.lc[l0 + lane].nu, a.T_cmb));
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
                eta += scattered64(a, roots, l, x0 * kSqrtLog2e64, 0.0, xs, (int)o, (int)o);
            }
        }
        chi = fmax(chi, a.chi_min);
        const double ichi = 1.0 / chi;
        const double So = eta * ichi;
        const double own = chil * ichi, rest = (chi - chil) * ichi, oth = (eta - etal) * ichi;
        double s_u = 0.0, s_l = 0.0, s_e = 0.0, s_c = 0.0, s_b[2] = {0.0, 0.0};
        for (int p = g; p < a.P; p += G) {
            const int rf = a.pf[p], rb = a.pb[p];
            Bin64 z{};
            double pi[2], ps[2], dl[2], gg[2][2], rr[2][2], hh[2][2], so[2][2];
            bool any = false;
#pragma unroll 1
            for (int side = 0; side < 2; side++) {
                int rows = 0;
                const bool full = sweep_half64<B, SCAT>(A, W, tab, roots, o, side ? rf : rb, l0, nl, l - l0, aq, nu_o,
                                                        chi, aq_lo, aq_hi, chi_min_e, z, rows);
                double pis, pss, dls;
                double g1[2] = {0.0, 0.0}, r1[2], h1[2] = {0.0, 0.0}, o1[2] = {0.0, 0.0};
                if (full) {
                    any = true;
                    const double iq = 1.0 / z.Q;
                    pis = z.P * iq;
                    pss = z.R * iq;
                    dls = z.d;
                    if constexpr (B > 0) {
                        // psi after the last row is g_1 S_m + g_2 S_{m-1} + r_2 with
                        // iota_k = Q before / Q after: g_1 = s Q_in/Q_out, r_1 = R_in/Q_out
                        g1[0] = z.t1 * z.q1 * iq;
                        r1[0] = z.r1 * iq;
                        h1[0] = z.ph1 / z.ch1;
                        o1[0] = z.ot1 / z.ch1;
                        r1[1] = r1[0];
                        if (rows >= 2) {
                            g1[1] = z.t2 * z.q2 * iq;
                            r1[1] = z.r2 * iq;
                            h1[1] = z.ph2 / z.ch2;
                            o1[1] = z.ot2 / z.ch2;
                        }
                    }
                } else {
                    pis = kSqrt2_64;
                    pss = kSqrt2_64 * planck_d(nu_o, a.T_cmb);
                    dls = 0.0;
                    r1[0] = r1[1] = pss;
                }
                if (side == 0) {
                    pi[0] = pis; ps[0] = pss; dl[0] = dls;
                    if constexpr (B > 0)
                        for (int j = 0; j < 2; j++) { gg[0][j] = g1[j]; rr[0][j] = r1[j]; hh[0][j] = h1[j]; so[0][j] = o1[j]; }
                } else {
                    pi[1] = pis; ps[1] = pss; dl[1] = dls;
                    if constexpr (B > 0)
                        for (int j = 0; j < 2; j++) { gg[1][j] = g1[j]; rr[1][j] = r1[j]; hh[1][j] = h1[j]; so[1][j] = o1[j]; }
                }
            }
            double u, lam, uml, oml, jb[2] = {0.0, 0.0}, sD = 0.0;
            if (!any) {
                const double I = planck_d(nu_o, a.T_cmb);
                u = I; lam = 0.0; uml = I; oml = 1.0;
                jb[0] = jb[1] = I;
            } else {
                // sigma (Phi iota) = Phi^ iota/(delta_- + delta_+), sigma psi = psi^/(delta_- + delta_+)
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
                    A.Mpart[((((size_t)part * a.n + o) * L + ll) * a.R + (side ? rf : rb)) * B + j] = s;
                }
                __syncwarp();
            }
        }
        if (32 * c + lane < F) {
            acc[NA * f + 0] = s_u;
            acc[NA * f + 1] = s_l;
            acc[NA * f + 2] = s_e;
            acc[NA * f + 3] = s_c;
            for (int j = 0; j < B; j++) acc[NA * f + 4 + j] = s_b[j];
        }
    }
    __syncthreads();
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

// Coupling terms: the sum over each line's chunks, times chi_int(o)/P.
__global__ void k_band_terms64(int64_t n, int L, int R, int B, int Q, double invP, const double *part,
                               const double *line, double *M) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, m = n * L * R * B;
    if (t >= m) return;
    const int64_t ol = t / (R * B);
    const int l = (int)(ol % L);
    const int np = (l * Q + Q - 1) / 32 - l * Q / 32 + 1;
    double s = 0.0;
    for (int k = 0; k < np; k++) s += part[k * m + t];
    M[t] = s * invP * line[2 * ol + 1];
}

}  // namespace
