// Image kernels for up to four lines in reach of the channels (included by solve.cu after the
// general kernel k_image64).
//
// One CTA per origin, one thread per channel. The pair's points are staged in shared memory,
// one thread per point, up to 512 at a time, and every thread carries its channel through
// them.
//
// A point matters to the channels within a few widths of its velocity only: channels that
// span tens of widths leave each of them a small share of the points (a fifth on the discs).
// Each thread therefore lists, as bits over the staged points, those whose opacity is above
// the floor (or whose emission is above the floor's times the least intensity, note_source) in its
// channel, with the points next to them, and walks through its own list; the warp runs as
// long as its busiest channel. (Over 32 points at a time that saves nothing: they span ten
// widths, the reach of a channel, and keep some lane busy at each of them.) An interval between two points below that changes the
// intensity by O(max(chi_min ds, dtau_min)) of itself; the lists are used while
// the optical depth of the two floors over a whole pair stays below 1e-14.
//
// FP64. The FP64 pipe (64-80 cycles per warp instruction) bounds it: per listed point x',
// (chi_prev + chi) h (2) and the linear-source step (3) are FP64; the exponentials, the
// step's weights (a reciprocal, or their Taylor series below dtau = 2^-7) and the floors run
// on the integer pipe. The general kernel takes three exponentials, two divisions and ~30
// further operations at every point. 10k-point clumpy cloud, 41 channels, one image: general
// kernel 37.5 ms, every point with this arithmetic 5.1 ms, lists 1.3 ms.
namespace {

constexpr int kImgCap = 512;   // points staged at a time, at most

// The FP32 kernel has opacities and emissivities in units of 1/kImgUnit and lengths in units of
// kImgUnit (a power of two: the same bits), so that floors down to 1e-50 are normal FP32 numbers,
// whose reciprocals are finite. Below that the floor is the smallest such number.
constexpr float kImgUnit = 0x1p40f;

// Shared memory: per staged point and line, then the channels' lists.
template <int NOV>
struct ImgStage64 {
    float4 *tt;                  // [NOV][cap] (gz, ngy, |x'| beyond which the line is far, its margin per |u|)
    double *h;                   // [cap] half the path length from the point before
    double *gz, *ngy, *S;        // [NOV][cap] x' = u gz + ngy
    uint64_t *Xm, *Ym;           // opacity, and emissivity over chi_min, at line centre
    int32_t *Xe, *Ye;            // exponents (Xe: e for a single line, else 2 e + 1 for X < 0 or NaN; Ye: 4 e + flags:
                                 //   1 for Y < 0, 2 for an emissivity that is not finite, in place of the source in S)
    uint32_t *todo;              // [cap/32][threads]
    static __host__ __device__ size_t bytes(int cap, int threads) {
        return (size_t)cap * (8 + NOV * (16 + 24 + 16 + 8)) + (size_t)cap / 32 * threads * 4;
    }
    __device__ ImgStage64(unsigned char *p, int cap) {
        auto take = [&](size_t n) { unsigned char *q = p; p += n * cap; return q; };
        tt = reinterpret_cast<float4 *>(take(16 * NOV));
        h = reinterpret_cast<double *>(take(8));
        gz = reinterpret_cast<double *>(take(8 * NOV));
        ngy = reinterpret_cast<double *>(take(8 * NOV));
        S = reinterpret_cast<double *>(take(8 * NOV));
        Xm = reinterpret_cast<uint64_t *>(take(8 * NOV));
        Ym = reinterpret_cast<uint64_t *>(take(8 * NOV));
        Xe = reinterpret_cast<int32_t *>(take(4 * NOV));
        Ye = reinterpret_cast<int32_t *>(take(4 * NOV));
        todo = reinterpret_cast<uint32_t *>(p);
    }
};

// FP32: per pair of points (2p, 2p + 1), as operand pairs of packed arithmetic.
constexpr int kImgPairs = 64;
template <int NOV>
struct ImgStage32 {
    float4 g[NOV][kImgPairs];    // (gz, gz, ngy, ngy): x' = u gz + ngy
    float4 x[NOV][kImgPairs];    // (eta, eta, chi, chi)
    float4 y[kImgPairs];         // (1/b, 1/b, h, h)
};

// Lists a channel's points of a staged chunk of cnt (from `nearby(j)`, whether point j is near):
// near points and the points next to them; near1: whether the point before the chunk is near
// (updated). The chunk's first point of the pair and its last, which stands in for the
// look-ahead into the next chunk, are always listed. One bit per point, word w at todo[w * stride].
template <typename F>
__device__ __forceinline__ void img_list(uint32_t *todo, int stride, int cnt, bool first, unsigned &near1, F nearby) {
    unsigned prev = 0;           // near bits of the word before, not yet stored
    unsigned carry = near1;
    const int nw = (cnt + 31) >> 5;
    for (int w = 0; w <= nw; w++) {
        unsigned nr = 0;
        if (w < nw) {
            const int m = min(32, cnt - 32 * w);
#pragma unroll 8
            for (int j = 0; j < m; j++)
                if (nearby(32 * w + j)) nr |= 1u << j;
        }
        if (w > 0) {
            unsigned t = prev | (prev << 1) | carry | (prev >> 1) | (nr << 31);
            const int m = min(32, cnt - 32 * (w - 1));
            if (first && w == 1) t |= 1u;
            if (w == nw) {
                t |= 1u << (m - 1);
                near1 = (prev >> (m - 1)) & 1u;
            }
            todo[(w - 1) * stride] = m == 32 ? t : t & ((1u << m) - 1u);
            carry = prev >> 31;
        }
        prev = nr;
    }
}

// Point k of the pair: half, index x on it (0 = nearest the origin), element, cells.
struct ImgPoint {
    int x, e, j, np;      // sub-point j of np of element e
    int32_t p, c;
    int64_t off;
    float sgn;            // of the half's velocities
};
__device__ __forceinline__ ImgPoint img_point(const SolveArgs &s, int64_t o, int64_t ofb, int64_t ofl, int lb, int lf,
                                              int Kb, int k) {
    ImgPoint q{};
    if (k == Kb) {
        q.x = -1;
        q.p = q.c = (int32_t)o;
        return q;
    }
    const bool back = k < Kb;
    q.x = back ? Kb - 1 - k : k - Kb - 1;
    q.off = back ? ofb : ofl;
    q.sgn = back ? -1.0f : 1.0f;
    int lo = 0, hi = (back ? lb : lf) - 1;   // the first element that ends beyond x
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (s.xcum[q.off + mid] > q.x) hi = mid;
        else lo = mid + 1;
    }
    q.e = lo;
    const int x0 = lo ? s.xcum[q.off + lo - 1] : 0;
    q.np = s.xcum[q.off + lo] - x0;
    q.j = q.x - x0 + 1;
    q.c = s.cells[q.off + lo];
    q.p = lo ? s.cells[q.off + lo - 1] : (int32_t)o;
    return q;
}

// Element and its number of points behind the interval from point k - 1 to point k (the path
// length belongs to the point farther from the origin).
__device__ __forceinline__ int64_t img_interval(const SolveArgs &s, const ImgPoint &q, int64_t ofb, int k, int Kb,
                                                int &np) {
    int64_t at;
    if (k == Kb) {                      // from the nearest point of the backward half
        np = s.xcum[ofb];
        return ofb;
    }
    at = q.off + q.e;
    np = q.np;
    if (k < Kb && q.j == q.np) {        // the previous point is the next element's first
        np = s.xcum[at + 1] - s.xcum[at];
        at++;
    }
    return at;
}

// 1/n, n a positive integer
__device__ __forceinline__ double img_rn(int n) { return n > 1 ? pos_pack(pos_rcp(pos_from((double)n))) : 1.0; }

// Weights of the linear-source step over d = dtau: I -> e I + wa S_a + wb S_b with e = exp(-d),
// alpha = (1 - e)/d, wa = alpha - e, wb = 1 - alpha, in units of 2^-63 fixed point (1 - e and
// its quotient by d keep 2^-60), from the Taylor series below d = 2^-7.
__device__ __forceinline__ void ls_weights64(const PosFp &d, const uint64_t *tab, double &e, double &wa, double &wb) {
    if (d.e >= 7 - 63) {                // d >= 2^7: e is below 2^-184
        const PosFp al = pos_rcp(d);    // alpha = (1 - e)/d, wa = alpha - e
        e = 0.0;
        if (d.e < 10 - 63) {
            int n;
            const uint64_t s = exp_neg(d, tab, n);
            e = pos_pack(pos_norm(s, -63 - n).m, pos_norm(s, -63 - n).e);
        }
        wa = pos_pack(al);
        wb = 1.0 - wa;
        return;
    }
    int n;
    const uint64_t s = exp_neg(d, tab, n);
    e = pos_pack(s, -63 - n);
    if (d.e < -7 - 63) {                // d < 2^-7: y = d in units of 2^-71
        const int sh = -(d.e + 71);     // m 2^e = y 2^-71
        const uint64_t y = sh < 64 ? d.m >> sh : 0;
        // wb/d = 1/2 - d (1/6 - d (1/24 - d (1/120 - d (1/720 - d/5040)))),
        // wa/d = 1/2 - d (1/3 - d (1/8 - d (1/30 - d (1/144 - d/840)))), in units of 2^-64
        constexpr uint64_t one = ~0ull;
        auto by = [&](uint64_t c) { return mulhi_near(c, y) >> 7; };
        const uint64_t gb =
            (1ull << 63) - by(one / 6 - by(one / 24 - by(one / 120 - by(one / 720 - by(one / 5040)))));
        const uint64_t ga = (1ull << 63) - by(one / 3 - by(one / 8 - by(one / 30 - by(one / 144 - by(one / 840)))));
        wb = pos_pack(pos_mul(d, pos_norm(gb, -64)));
        wa = pos_pack(pos_mul(d, pos_norm(ga, -64)));
        return;
    }
    const uint64_t E = n < 64 ? s >> n : 0, om = (1ull << 63) - E;     // e, 1 - e in units of 2^-63
    const int z = __clzll(om);
    const PosFp al = pos_mul(PosFp{om << z, -63 - z}, pos_rcp(d));
    // alpha < 1 in units of 2^-63
    const int sa = -63 - al.e;
    const uint64_t af = sa < 64 ? al.m >> sa : 0;
    const uint64_t a1 = af < E ? 0 : af - E, b1 = (1ull << 63) - (af >> 63 ? (1ull << 63) : af);
    const int za = __clzll(a1 | 1), zb = __clzll(b1 | 1);
    wa = pos_pack(a1 << za, -63 - za);
    wb = pos_pack(b1 << zb, -63 - zb);
}

template <int NOV>
__global__ void __launch_bounds__(256) k_image64_lines(ImageArgs a, int skip, int cap) {
    extern __shared__ __align__(16) unsigned char img_smem[];
    __shared__ uint64_t tab[256];
    __shared__ double far_w;             // velocity at the far end
    const ImgStage64<NOV> T(img_smem, cap);
    const SolveArgs &s = a.s;
    const int64_t o = blockIdx.x;
    const double *vo = a.vel + 3 * o;
    for (int t = threadIdx.x; t < 256; t += blockDim.x) tab[t] = kExp2Table.t[t];
    const double nvo = a.n0 * vo[0] + a.n1 * vo[1] + a.n2 * vo[2];
    const int64_t ofb = s.ray_off[o * s.R + a.rb], ofl = s.ray_off[o * s.R + a.rf];
    const int lb = (int)(s.ray_off[o * s.R + a.rb + 1] - ofb);
    const int lf = (int)(s.ray_off[o * s.R + a.rf + 1] - ofl);
    const int Kb = lb ? s.xcum[ofb + lb - 1] : 0;
    const int K = Kb + 1 + (lf ? s.xcum[ofl + lf - 1] : 0);
    if (K > s.kmax) {
        if (threadIdx.x == 0) atomicOr(s.err, 2);
        return;
    }
    const double inv_chi_min = 1.0 / s.chi_min;
    const PosFp cmin = pos_from(s.chi_min);
    int ic = 2048;                       // exponent of the least intensity over the lines in reach
#pragma unroll
    for (int i = 0; i < NOV; i++) ic = min(ic, least_exponent(a.lf[i].ic, s.least[a.lf[i].l2]));
    constexpr double kCsp = kC / kSqrtPi;
    for (int c0 = 0; c0 < a.n_ch; c0 += blockDim.x) {
        const int c = c0 + threadIdx.x;
        const double u = a.u[min(c, a.n_ch - 1)];
        const float uf = (float)u;
        double I = 0.0, S_prev = 0.0;
        PosFp chi_prev{0, -(1 << 20)};
        unsigned near1 = 0;                  // whether the point before is near
        uint32_t *todo = T.todo + threadIdx.x;
        for (int k0 = 0; k0 < K; k0 += cap) {
            const int cnt = min(cap, K - k0);
            __syncthreads();
            for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
                const int k = k0 + t;
                const ImgPoint q = img_point(s, o, ofb, ofl, lb, lf, Kb, k);
                double wt = 0.0, w = nvo, ib;
                if (q.x < 0) {
                    ib = pos_pack(pos_rcp(pos_from(s.b[o])));
                } else {
                    wt = q.j == q.np ? 1.0 : (double)q.j * img_rn(q.np);
                    const double pv = q.e ? s.vpar[q.off + q.e - 1] : 0.0;
                    w += (double)q.sgn * ((1.0 - wt) * pv + wt * s.vpar[q.off + q.e]);
                    ib = pos_pack(pos_rcp(pos_from((1.0 - wt) * s.b[q.p] + wt * s.b[q.c])));
                }
                int np = 1;
                const int64_t at = k ? img_interval(s, q, ofb, k, Kb, np) : 0;
                T.h[t] = k ? 0.5 * s.ds[at] * img_rn(np) : 0.0;
                if (!k) far_w = w;
                const double gy = w * ib, gz = ib - gy * (1.0 / kC);
                const int eb = ((__double2hiint(ib) >> 20) & 0x7ff) - 1022;
#pragma unroll
                for (int i = 0; i < NOV; i++) {
                    const Overlap ov = a.ov[i];
                    const double2 p0 = reinterpret_cast<const double2 *>(s.line)[(int64_t)q.p * s.L + ov.l2];
                    const double2 p1 = reinterpret_cast<const double2 *>(s.line)[(int64_t)q.c * s.L + ov.l2];
                    const double et = (1.0 - wt) * p0.x + wt * p1.x, ch = (1.0 - wt) * p0.y + wt * p1.y;
                    const double nrm = ov.inv_nu2 * ib * kCsp;
                    // (a negative opacity alone ends at the floor; several lines add up first)
                    const PosFp X = NOV > 1 ? pos_from(fabs(ch * nrm))
                                            : (ch > 0.0 ? pos_from(ch * nrm) : PosFp{0, -(1 << 20)});
                    const PosFp Y = pos_from(et * nrm * inv_chi_min);
                    // x' = (dnl + rat (u (1 - w/c) - w)) / b
                    const double gzl = ov.rat * gz, ngl = ov.dnl * ib - ov.rat * gy;
                    T.gz[i * cap + t] = gzl;
                    T.ngy[i * cap + t] = ngl;
                    T.Xm[i * cap + t] = X.m;
                    T.Xe[i * cap + t] = NOV > 1 ? 2 * X.e + (ch >= 0.0 ? 0 : 1) : X.e;
                    T.Ym[i * cap + t] = Y.m;
                    const bool bad = not_finite(et) || not_finite(gy);
                    T.Ye[i * cap + t] = 4 * Y.e + (et < 0.0 ? 1 : 0) + (bad ? 2 : 0);
                    double S = 0.0;
                    if (ch > 0.0) {
                        S = pos_pack(pos_mul(pos_from(et), pos_rcp(pos_from(ch))));
                        if (et < 0.0) S = -S;
                    }
                    if (bad) S = nan64();
                    T.S[i * cap + t] = S;
                    const int sgn = NOV > 1 ? 0x7fffffff : -1;   // (alone, a negative opacity is below every other)
                    const int ech = max(__double2hiint(p0.y) & sgn, __double2hiint(p1.y) & sgn) >> 20;
                    const int eet = max(__double2hiint(p0.x) & 0x7fffffff, __double2hiint(p1.x) & 0x7fffffff) >> 20;
                    const float bound = max(ech, eet) >= 0x7ff   // (infinite or NaN: never far)
                                            ? INFINITY
                                            : (float)(max(max(ech, eet - ic) - 1022, -100000) + eb - a.lf[i].cm);
                    T.tt[i * cap + t] = make_float4((float)gzl, (float)ngl,
                                             skip ? sqrtf(1.001f / kLog2e64 * fmaxf(bound, 0.0f)) +
                                                        1e-6f * fabsf((float)ngl)
                                                  : INFINITY,
                                             1e-6f * (float)gzl);
                }
            }
            __syncthreads();
            const int nw = (cnt + 31) >> 5;
            int wd = 0;
            uint32_t bits = 0;
            if (skip) {
                img_list(todo, blockDim.x, cnt, k0 == 0, near1, [&](int j) {
                    bool near = false;
#pragma unroll
                    for (int i = 0; i < NOV; i++) {
                        const float4 t4 = T.tt[i * cap + j];
                        near = near || !(fabsf(fmaf(uf, t4.x, t4.y)) > fmaf(fabsf(uf), t4.w, t4.z));
                    }
                    return near;
                });
                bits = todo[0];
            } else {
                bits = cnt >= 32 ? 0xffffffffu : (1u << cnt) - 1u;
            }
            // the next listed point of each channel, until every channel of the warp is through
            for (;;) {
                while (!bits && ++wd < nw)
                    bits = skip ? todo[wd * blockDim.x]
                                : (cnt - 32 * wd >= 32 ? 0xffffffffu : (1u << (cnt - 32 * wd)) - 1u);
                if (!__any_sync(0xffffffffu, bits != 0)) break;
                if (bits) {
                    const int j = 32 * wd + __ffs(bits) - 1;
                    bits &= bits - 1;
                    PosFp chi{0, -(1 << 20)};
                    double Sk = 0.0, eta = 0.0, chis = 0.0;
#pragma unroll
                    for (int i = 0; i < NOV; i++) {
                        double x = fma(u, T.gz[i * cap + j], T.ngy[i * cap + j]);
                        const int xh = __double2hiint(x) & 0x7fffffff;
                        if (xh >= 0x404a0000) x = 52.0;                       // exp(-52^2) is zero
                        const bool out = xh > 0x403b5025 && xh <= 0x7ff00000;   // x^2 > 746: outside the profile
                        int n;
                        const uint64_t e = exp_neg_sq(x, tab, n);
                        const int xe = T.Xe[i * cap + j];
                        const PosFp ci = pos_norm(mulhi_near(T.Xm[i * cap + j], e), (NOV > 1 ? xe >> 1 : xe) + 1 - n);
                        const int ye = T.Ye[i * cap + j];
                        if (NOV == 1) {
                            chi = ci;
                            Sk = T.S[i * cap + j];
                            if (chi.m == 0 || chi.e < cmin.e || (chi.e == cmin.e && chi.m < cmin.m)) {
                                chi = cmin;
                                Sk = pos_pack(mulhi_near(T.Ym[i * cap + j], e), (ye >> 2) + 1 - n);
                                if (ye & 3) Sk = ye & 2 ? (out ? 0.0 : T.S[i * cap + j]) : -Sk;
                            }
                        } else {
                            // (the emissivity in units of chi_min)
                            double ei = pos_pack(mulhi_near(T.Ym[i * cap + j], e), (ye >> 2) + 1 - n);
                            if (ye & 3) ei = ye & 2 ? (out ? 0.0 : T.S[i * cap + j]) : -ei;
                            eta += ei;
                            double cd = out ? 0.0 : pos_pack(ci);
                            if (xe & 1) cd = -cd;
                            chis += cd;
                        }
                    }
                    if (NOV > 1) {
                        chis = pos_max(chis, s.chi_min);   // (a negative sum is below it as bits too)
                        chi = pos_from(chis);
                        Sk = eta * s.chi_min * pos_pack(pos_rcp(chi));
                    }
                    if (k0 + j == 0) {
                        I = planck_d(a.nu_l * (1.0 + u / kC) * (1.0 - far_w / kC), s.T_cmb);
                    } else {
                        PosFp d = pos_mul(pos_add(chi_prev, chi), pos_from(T.h[j]));
                        if (__double_as_longlong(pos_pack(d)) < __double_as_longlong(s.dtau_min)) d = pos_from(s.dtau_min);
                        double e, wa, wb;
                        ls_weights64(d, tab, e, wa, wb);
                        I = fma(wb, Sk, fma(wa, S_prev, e * I));
                    }
                    chi_prev = chi;
                    S_prev = Sk;
                }
            }
        }
        if (c < a.n_ch) a.I[o * a.n_ch + c] = I;
    }
}

// FP32 (mixed-precision contexts), from the FP32 ray store, widths and line data. Here the
// issue rate bounds it (two ex2 and two rcp per point and channel, ~25 instructions), and walking
// lists costs more than it saves: every channel goes through every point, two points at a
// time in packed FP32x2 arithmetic; only the intensity itself is a chain (three FMAs a
// point). The first point of the pair and one that fills up the last pair have dtau = 0,
// which leaves the intensity as it is. The linear-source weights use their Taylor series below
// dtau = 0.05 (4 terms: relative error below 2e-8 there), where 1 - alpha would cancel.
// 20k-point disc, 63 channels: 386 us with one point at a time and a thread per element in the
// staging, 445 us with lists, 212 us now.
template <int NOV>
__global__ void __launch_bounds__(256) k_image32_lines(ImageArgs a) {
    __shared__ ImgStage32<NOV> T;
    __shared__ float far_w;              // velocity at the far end
    const SolveArgs &s = a.s;
    const int64_t o = blockIdx.x;
    const double *vo = a.vel + 3 * o;
    const float chi_min = a.chi_min32, dtau_min = a.dtau_min32;
    const float nvo = a.nf[0] * (float)vo[0] + a.nf[1] * (float)vo[1] + a.nf[2] * (float)vo[2];
    const int64_t ofb = s.ray_off[o * s.R + a.rb], ofl = s.ray_off[o * s.R + a.rf];
    const int lb = (int)(s.ray_off[o * s.R + a.rb + 1] - ofb);
    const int lf = (int)(s.ray_off[o * s.R + a.rf + 1] - ofl);
    const int Kb = lb ? s.xcum[ofb + lb - 1] : 0;
    const int K = Kb + 1 + (lf ? s.xcum[ofl + lf - 1] : 0);
    if (K > s.kmax) {
        if (threadIdx.x == 0) atomicOr(s.err, 2);
        return;
    }
    constexpr float kic = (float)(1.0 / kC), ks = 1.2011224087864498f, kL2e = 1.4426950408889634f;
    auto ex2 = [](float v) {
        float e;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(v));
        return e;
    };
    auto rcp = [](float v) {
        float e;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(v));
        return e;
    };
    auto two = [](float v) { return make_float2(v, v); };
    for (int c0 = 0; c0 < a.n_ch; c0 += blockDim.x) {
        const int c = c0 + threadIdx.x;
        const float u = (float)a.u[min(c, a.n_ch - 1)];
        const float2 u2 = two(u);
        float I = 0.0f, chi_prev = 0.0f, S_prev = 0.0f;
        for (int k0 = 0; k0 < K; k0 += 2 * kImgPairs) {
            const int cnt = min(2 * kImgPairs, K - k0), np2 = (cnt + 1) >> 1;
            __syncthreads();
            for (int t = threadIdx.x; t < 2 * np2; t += blockDim.x) {
                const int k = k0 + t, pr = t >> 1, odd = t & 1;
                float h = 0.0f, ib = 0.0f;
                if (k < K) {
                    const ImgPoint q = img_point(s, o, ofb, ofl, lb, lf, Kb, k);
                    float wt = 0.0f, w = nvo, b;
                    if (q.x < 0) {
                        b = a.bf[o];
                    } else {
                        // (at the element's own cell, j = np, this can fall one rounding short of 1, so
                        // that a neighbour 1e7 times denser shows through at that point)
                        wt = (float)q.j * (1.0f / (float)q.np);
                        const float pv = q.e ? a.vparf[q.off + q.e - 1] : 0.0f;
                        w += q.sgn * ((1.0f - wt) * pv + wt * a.vparf[q.off + q.e]);
                        b = (1.0f - wt) * a.bf[q.p] + wt * a.bf[q.c];
                    }
                    if (k) {
                        int np;
                        const int64_t at = img_interval(s, q, ofb, k, Kb, np);
                        h = __fdividef((0.5f / kImgUnit) * a.dsf[at], (float)np);
                    } else {
                        far_w = w;
                    }
                    ib = 1.0f / b;
                    const float pz = ks * ib, gy = w * pz, gz = pz - gy * kic;
#pragma unroll
                    for (int i = 0; i < NOV; i++) {
                        const float2 p0 = reinterpret_cast<const float2 *>(a.linef)[(int64_t)q.p * s.L + a.lf[i].l2];
                        const float2 p1 = reinterpret_cast<const float2 *>(a.linef)[(int64_t)q.c * s.L + a.lf[i].l2];
                        float *g = &T.g[i][pr].x + odd, *x = &T.x[i][pr].x + odd;
                        g[0] = a.lf[i].rat * gz;
                        g[2] = a.lf[i].dnl * pz - a.lf[i].rat * gy;
                        x[0] = (1.0f - wt) * p0.x + wt * p1.x;
                        x[2] = (1.0f - wt) * p0.y + wt * p1.y;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < NOV; i++) {
                        float *g = &T.g[i][pr].x + odd, *x = &T.x[i][pr].x + odd;
                        g[0] = g[2] = x[0] = x[2] = 0.0f;
                    }
                }
                float *y = &T.y[pr].x + odd;
                y[0] = ib;
                y[2] = h;
            }
            __syncthreads();
            if (k0 == 0) I = planck_f((float)a.nu_l * (1.0f + u * kic) * (1.0f - far_w * kic), (float)s.T_cmb);
#pragma unroll 2
            for (int j = 0; j < np2; j++) {
                const float4 y = T.y[j];
                float2 chi = two(0.0f), S = two(0.0f);
#pragma unroll
                for (int i = 0; i < NOV; i++) {
                    const float4 g = T.g[i][j], xs = T.x[i][j];
                    const float2 x = __ffma2_rn(u2, make_float2(g.x, g.y), make_float2(g.z, g.w));
                    const float2 xx = __fmul2_rn(x, x);
                    const float2 e = make_float2(ex2(-xx.x), ex2(-xx.y));
                    const float2 phi = __fmul2_rn(e, __fmul2_rn(make_float2(y.x, y.y), two(a.lf[i].nrm)));
                    S = __ffma2_rn(make_float2(xs.x, xs.y), phi, S);         // (the emissivity)
                    chi = __ffma2_rn(make_float2(xs.z, xs.w), phi, chi);
                }
                chi = make_float2(fmaxf(chi.x, chi_min), fmaxf(chi.y, chi_min));
                S = __fmul2_rn(S, make_float2(rcp(chi.x), rcp(chi.y)));
                float2 d = __fmul2_rn(__fadd2_rn(make_float2(chi_prev, chi.x), chi), make_float2(y.z, y.w));
                // (no floor at the first point of the pair and where a last point is missing)
                d.x = fmaxf(d.x, k0 + j ? dtau_min : 0.0f);
                d.y = fmaxf(d.y, k0 + 2 * j + 1 < K ? dtau_min : 0.0f);
                const float2 nd = __fmul2_rn(d, two(-1.0f));
                const float2 dl = __fmul2_rn(nd, two(kL2e));
                const float2 e = make_float2(ex2(dl.x), ex2(dl.y));
                const float2 al = __fmul2_rn(__ffma2_rn(e, two(-1.0f), two(1.0f)), make_float2(rcp(d.x), rcp(d.y)));
                float2 wb = __ffma2_rn(nd, two(1.0f / 120.0f), two(1.0f / 24.0f));
                float2 wa = __ffma2_rn(nd, two(1.0f / 30.0f), two(1.0f / 8.0f));
                wb = __ffma2_rn(nd, wb, two(1.0f / 6.0f));
                wa = __ffma2_rn(nd, wa, two(1.0f / 3.0f));
                wb = __fmul2_rn(d, __ffma2_rn(nd, wb, two(0.5f)));
                wa = __fmul2_rn(d, __ffma2_rn(nd, wa, two(0.5f)));
                const float2 ab = __ffma2_rn(al, two(-1.0f), two(1.0f)), aa = __ffma2_rn(e, two(-1.0f), al);
                wb = make_float2(d.x < 0.05f ? wb.x : ab.x, d.y < 0.05f ? wb.y : ab.y);
                wa = make_float2(d.x < 0.05f ? wa.x : aa.x, d.y < 0.05f ? wa.y : aa.y);
                I = fmaf(e.x, I, fmaf(wa.x, S_prev, wb.x * S.x));
                I = fmaf(e.y, I, fmaf(wa.y, S.x, wb.y * S.y));
                chi_prev = chi.y;
                S_prev = S.y;
            }
        }
        if (c < a.n_ch) a.I[o * a.n_ch + c] = (double)I;
    }
}

// Sky-plane coordinates of every point.
__global__ void k_image_xy(ImageArgs a) {
    const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= a.s.n) return;
    const double *xo = a.pos + 3 * o;
    a.xy[2 * o] = xo[0] * a.e1[0] + xo[1] * a.e1[1] + xo[2] * a.e1[2];
    a.xy[2 * o + 1] = xo[0] * a.e2[0] + xo[1] * a.e2[1] + xo[2] * a.e2[2];
}

}  // namespace
