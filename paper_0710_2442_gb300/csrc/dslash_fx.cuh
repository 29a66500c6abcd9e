// dslash_fx.cuh -- the FP64 hopping term (Sec. 5, Eq. 3) on the integer pipe
// (block fixed point, fx.cuh).
//
// What bounds the FP64 stencil (hop_kernel): 846 FP64 instructions per site, which
// GB300 issues at two lanes per SM and clock.  1648 us on 32^3 x 64, where the bytes
// take 237 us; on 8^4 the 32 blocks that a thread per site makes leave most SMs idle
// and take 34 us.  Two kernels, by the number of sites (kFxSiteMin):
//
//  hop_kernel_fx1, large lattices.  Neighbours and links are read in fixed point:
//  the field is converted once (fx_pack_kernel) instead of in each of the eight hops that
//  read a site, the links when they are packed, and the Schur operator's intermediate
//  field never leaves that form.  Two threads per site, one per half-spin row, sum
//  the eight hops in 64-bit integers, with the next hop's words copied ahead.  About 180 instructions
//  a thread and hop.  No unit is saturated (16^3 x 32: issue 37 %, DRAM 49 %, L1 48 %, FP64 34 %
//  busy): bound by the latency of the copies at 16 warps an SM, at 0.7 to 0.75 of the HBM time of what it
//  reads.  A hop without the conversion (24^3 x 48 / 32^3 x 64): FP64 stencil 552 / 1648 us, here 114 / 333 us
//  (111 / 329 before the guard of fx.cuh); with the conversion in every hop 166 / 512 us; with one thread
//  per site and both rows (24 sums, 168 registers) 124 / 353 us.
//
//  hop_kernel_fx, small lattices.  A block works on 32 consecutive sites of one parity
//  with W warps; lane = site, and the eight hops are dealt out to the warps, so the
//  loads stay coalesced and a warp's control flow is uniform.  A hop converts the
//  neighbour's components (and the link, if it comes as doubles) to fixed point,
//  projects, multiplies, and leaves its half spinor as 64-bit integers in shared memory with one
//  exponent per half-spin row.  After one barrier warp s adds up spin s: the
//  eight hops aligned to their largest exponent, rounded to FP64 once.  8^4: 6.6 us (a call's
//  34 us on the FP64 stencil), 12^4: 11 us (37).
//
//  Both do a site over in FP64 where it is out of range or below the guard (fx_redo).  A lattice all of
//  whose sites are takes 991 us on 24^3 x 48, 57 us on 12^4 and 25 us on 8^4 (FP64 stencil 552, 37 and 34 us);
//  a lone site makes its block about 2 us longer.
#pragma once

#include "dslash_impl.cuh"
#include "fx.cuh"

namespace wl {

// A field of 16-byte words: word k of index i at p + 16 (i site_step + k word_step).
// The index is the half-site index, or the full site's (by_site).
struct FxField {
    char* p;
    long long pstep;  // bytes to the parity-1 block (0: one block, or by_site)
    long long rstep;  // bytes to the next right-hand side
    int site_step, word_step;
    int by_site;
};
// Links: word e of link (parity, mu) of index i at
// p + 16 (parity par_step + mu mu_step + i site_step + e word_step).
struct FxLinks {
    const char* p;
    long long par_step;
    long long mu_step;
    int site_step, word_step;
    int by_site;
};

struct FxParams {
    FxField out, in, x;
    FxField nat;  // the input as doubles, for sites done over in FP64 (p null: in, fixed point with some doubles)
    FxLinks u;    // the links the kernel reads: doubles, or fixed point (FXL)
    FxLinks un;   // the same links as doubles, for those sites
    int un_recon;  // of 12 or 18 reals
    Geom g;
    int nrhs, skip_stride, out_parity, full, xpay, dag;
    int scaled;  // a != 1 (without xpay)
    double a;
    RedArgs red;
    const int* skip;
};

__device__ __forceinline__ const uint4* fx_at(const FxField& f, int par, int k, int s) {
    return reinterpret_cast<const uint4*>(f.p + (par ? f.pstep : 0) + k * f.rstep) +
           (long long)(f.by_site ? s : s >> 1) * f.site_step;
}
__device__ __forceinline__ const uint4* fx_link_at(const FxLinks& u, int par, int mu, int s) {
    return reinterpret_cast<const uint4*>(u.p) + (par ? u.par_step : 0) + (long long)mu * u.mu_step +
           (long long)(u.by_site ? s : s >> 1) * u.site_step;
}

// The neighbour of site s (coordinates c) in hop j = 2 mu + (0 forward, 1 backward).
__device__ __forceinline__ int fx_neighbour(const Geom& g, const int c[4], int s, int j, bool& wrap) {
    const int mu = j >> 1;
    const int L = g.L[mu];
    const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
    const int smu = mu == 0 ? 1 : mu == 1 ? g.L[0] : mu == 2 ? g.L[0] * g.L[1] : g.L[0] * g.L[1] * g.L[2];
    if ((j & 1) == 0) {
        wrap = cm == L - 1;
        return wrap ? s - (L - 1) * smu : s + smu;
    }
    wrap = cm == 0;
    return wrap ? s + (L - 1) * smu : s - smu;
}

__device__ __forceinline__ unsigned fx_max2(unsigned m, const uint4& d) { return max(m, max(d.y << 1, d.w << 1)); }
__device__ __forceinline__ unsigned fx_nonzero(const uint4& d) { return d.x | d.y << 1 | d.z | d.w << 1; }

// Half-spin row r of the projected neighbour, in units of its own largest
// exponent, which is returned (0: out of range; kFxZero: both spins are zero).  The projector's partner spin
// comes in with factor sigma, times i for IMAG; the row comes times sg = +-1.
constexpr int kFxZero = kFxEmin - 1;
template <bool IMAG>
__device__ __forceinline__ int fx_project(const uint4* psi, int ws, int r, int partner, int sigma, int sg,
                                          FxCplx h[3]) {
    uint4 p[3], q[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        p[c] = __ldg(psi + (long long)(r * 3 + c) * ws);
        q[c] = __ldg(psi + (long long)(partner * 3 + c) * ws);
    }
    unsigned m = 0;
#pragma unroll
    for (int c = 0; c < 3; c++) m = fx_max2(fx_max2(m, p[c]), q[c]);
    int e = (int)(m >> 21);
    if (e < kFxEmin || e > kFxEmax) {
        unsigned nz = 0;
#pragma unroll
        for (int c = 0; c < 3; c++) nz |= fx_nonzero(p[c]) | fx_nonzero(q[c]);
        e = nz ? 0 : kFxZero;
    }
    const unsigned ew = fx_scale_word(e + kFxOffSpinor);
    const int sre = sg * (IMAG ? -sigma : sigma), sim = sg * sigma;  // i q = (-q.im, q.re)
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const unsigned ah = IMAG ? q[c].w : q[c].y, al = IMAG ? q[c].z : q[c].x;
        const unsigned bh = IMAG ? q[c].y : q[c].w, bl = IMAG ? q[c].x : q[c].z;
        const FxMag pr = fx_mag(p[c].y, p[c].x, fx_shift(ew, p[c].y << 1));
        const FxMag pi = fx_mag(p[c].w, p[c].z, fx_shift(ew, p[c].w << 1));
        const FxMag a = fx_mag(ah, al, fx_shift(ew, ah << 1)), b = fx_mag(bh, bl, fx_shift(ew, bh << 1));
        const int spr = fx_sign(p[c].y, sg), spi = fx_sign(p[c].w, sg), sa = fx_sign(ah, sre), sb = fx_sign(bh, sim);
        h[c].re = FxReal{a.h * sa + pr.h * spr, a.l * sa + pr.l * spr};
        h[c].im = FxReal{b.h * sb + pi.h * spi, b.l * sb + pi.l * spi};
    }
    return e;
}

// w_i = sum_k u_k h_k, or with x, y in place of -Im h and Re h
__device__ __forceinline__ longlong2 fx_row(const FxCplx u[3], const FxCplx h[3], const FxReal x[3], const FxReal y[3]) {
    FxAcc re = fx_zero(), im = fx_zero();
#pragma unroll
    for (int k = 0; k < 3; k++) {
        fx_mac(re, u[k].re, h[k].re);
        fx_mac(re, u[k].im, x[k]);
        fx_mac(im, u[k].re, h[k].im);
        fx_mac(im, u[k].im, y[k]);
    }
    return make_longlong2(fx_sum(re), fx_sum(im));
}
// h times the boundary phase (pr, pi).
inline __device__ __noinline__ void fx_phase3(double pr, double pi, FxCplx* h) {
    const FxCplx eta{fx_link((unsigned)__double2hiint(pr), (unsigned)__double2loint(pr)),
                     fx_link((unsigned)__double2hiint(pi), (unsigned)__double2loint(pi))};
#pragma unroll
    for (int q = 0; q < 3; q++) h[q] = fx_phase(eta, h[q]);
}
__device__ __forceinline__ void fx_wrap(double pr, double pi, FxCplx (&h)[3]) {
    if (pi == 0.0) {  // +1 or -1
        if (pr < 0.0) {
#pragma unroll
            for (int q = 0; q < 3; q++) h[q] = FxCplx{fx_neg(h[q].re), fx_neg(h[q].im)};
        }
    } else {
        FxCplx t[3];
#pragma unroll
        for (int q = 0; q < 3; q++) t[q] = h[q];
        fx_phase3(pr, pi, t);
#pragma unroll
        for (int q = 0; q < 3; q++) h[q] = t[q];
    }
}

// Shared memory of a tile: the hops' half spinors [hop][row][colour][lane],
// their exponents [hop][row][lane] and the lanes to be done over in FP64, whose
// products take the place of w.
struct FxTile {
    longlong2 w[8][2][3][32];
    int e[8][2][32];
    int bad[32];
};

// Hop j of one site; a backward hop reads the link transposed and conjugated.  What is
// stored is w in x and y, -w in z and t: fx_spin cuts the contributions off at 2^-56 where it
// aligns them, and with these signs each output component adds four and subtracts four of
// the eight, so that what is cut off has no mean (rounding them instead: 12^4 Schur 24.3 -> 25.9 us).
template <bool FXL>
__device__ __forceinline__ void fx_hop(const FxParams& P, FxTile& T, int j, int p, int k, const int c[4], int s,
                                       int lane) {
    const int mu = j >> 1;
    const bool fwd = (j & 1) == 0;
    bool wrap;
    const int sn = fx_neighbour(P.g, c, s, j, wrap);
    const uint4* psi = fx_at(P.in, 1 - p, k, sn);
    const uint4* lk = fwd ? fx_link_at(P.u, p, mu, s) : fx_link_at(P.u, 1 - p, mu, sn);
    const int S = fwd != (P.dag != 0) ? 1 : -1, sg = mu < 2 ? 1 : -1, f = fwd ? 1 : -1;
    // (1 - S g_mu) psi, row r (project() in dslash_impl.cuh)
    auto project = [&](int r, FxCplx (&h)[3]) {
        const int e = mu == 0 || mu == 2
                          ? fx_project<true>(psi, P.in.word_step, r, (mu == 0) == (r == 0) ? 3 : 2,
                                             mu == 2 && r == 1 ? S : -S, sg, h)
                          : fx_project<false>(psi, P.in.word_step, r, (mu == 1) == (r == 0) ? 3 : 2,
                                              mu == 1 && r == 0 ? S : -S, sg, h);
        if (wrap) fx_wrap(P.g.ph[mu][0], f * P.g.ph[mu][1], h);
        T.e[j][r][lane] = e;
        return e == 0;
    };
    const int ws = P.u.word_step;
    bool bad = false;
    if constexpr (FXL) {
        // row i of U or of U^T: the transposition is in the word index
        const int wi = fwd ? 3 : 1, wk = fwd ? 1 : 3;
#pragma unroll 1
        for (int r = 0; r < 2; r++) {
            FxCplx h[3];
            FxReal x[3], y[3];
            bad |= project(r, h);
#pragma unroll
            for (int q = 0; q < 3; q++) {
                x[q] = FxReal{h[q].im.h * -f, h[q].im.l * -f};
                y[q] = FxReal{h[q].re.h * f, h[q].re.l * f};
            }
#pragma unroll
            for (int i = 0; i < 3; i++) {
                FxCplx u[3];
#pragma unroll
                for (int q = 0; q < 3; q++) {
                    const uint4 d = __ldg(lk + (long long)(i * wi + q * wk) * ws);
                    u[q] = FxCplx{FxReal{(int)d.x, (int)d.y}, FxReal{(int)d.z, (int)d.w}};
                }
                if (i == 0) bad |= (unsigned)u[0].re.h == kFxBadLink;
                T.w[j][r][i][lane] = fx_row(u, h, x, y);
            }
        }
    } else {
        FxCplx h[2][3];
        FxReal x[2][3], y[2][3];
#pragma unroll
        for (int r = 0; r < 2; r++) {
            bad |= project(r, h[r]);
#pragma unroll
            for (int q = 0; q < 3; q++) {
                x[r][q] = fx_neg(h[r][q].im);
                y[r][q] = h[r][q].re;
            }
        }
        unsigned mx = 0;
        const int wi = fwd ? 3 : 1, wk = fwd ? 1 : 3;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            FxCplx u[3];
#pragma unroll
            for (int q = 0; q < 3; q++) {
                const uint4 d = __ldg(lk + (long long)(i * wi + q * wk) * ws);
                mx = fx_max2(mx, d);
                u[q] = FxCplx{fx_link(d.y, d.x, 1), fx_link(d.w, d.z, f)};
            }
#pragma unroll
            for (int r = 0; r < 2; r++) T.w[j][r][i][lane] = fx_row(u, h[r], x[r], y[r]);
        }
        bad |= mx > kFxLinkHi;
    }
    if (bad) T.bad[lane] = 1;
}

// N colours from C0 on of output spin SPIN: the eight hops' contributions (expand()
// in dslash_impl.cuh) aligned to their largest exponent; returns whether a component is below
// the guard (fx.cuh).  The sums become doubles with integer instructions
// (INT) where a block is one of several on an SM: 12^4 F64 Schur 24.7 -> 24.0 us; one block of
// eight warps on an SM is as fast or faster with the FP64 additions (8^4 hop, before the guard: 6.42 against 6.49 us).
template <int SPIN, bool INT, int N>
__device__ __forceinline__ bool fx_spin(const FxTile& T, int c0, int dag, int lane, double2 (&v)[N]) {
    constexpr bool lower = SPIN >= 2;
    // half-spin row of hop direction mu: SPIN itself, or for spin 2 rows 1, 1, 0, 0 and for spin 3 rows 0, 0, 1, 1
    auto row = [](int j) { return lower ? ((SPIN == 2) == (j < 4) ? 1 : 0) : SPIN; };
    int e[8], top = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        e[j] = T.e[j][row(j)][lane];
        top = max(top, e[j]);
    }
#pragma unroll
    for (int j = 0; j < 8; j++) e[j] = min(top - e[j], kFxMaxShift);
    const int k2 = top + 1 - 1023 - 56;
    const FxBias bias = fx_bias(k2);
    bool below = false;
#pragma unroll
    for (int c = 0; c < N; c++) {
        long long re = 0, im = 0;
        unsigned nr = 0, ni = 0;
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const longlong2 w = T.w[j][row(j)][c0 + c][lane];
            const long long x = fx_align(w.x, e[j]), y = fx_align(w.y, e[j]);
            // upper: w.  Lower, with S = +1 forward and -1 backward: S i w (x), spin 2: -S w (y),
            // S i w (z), -S w (t); spin 3: S i w, S w, -S i w, -S w.  In z and t the stored one is -w.
            const int mu = j >> 1;
            const bool bwd = (j & 1) != 0, times_i = lower && (mu == 0 || mu == 2);
            const bool flip = (mu >= 2) != (lower && (bwd != (mu == 3 || (mu == 1 && SPIN == 2) || (mu == 2 && SPIN == 3))));
            if (times_i) {  // i (x + i y)
                re = flip ? re + y : re - y;
                im = flip ? im - x : im + x;
                nr = fx_modulus(y, nr);
                ni = fx_modulus(x, ni);
            } else {
                re = flip ? re - x : re + x;
                im = flip ? im - y : im + y;
                nr = fx_modulus(x, nr);
                ni = fx_modulus(y, ni);
            }
        }
        below = below || min(nr, ni) < kFxGuard << 16;
        if (lower && dag) {
            re = -re;
            im = -im;
        }
        v[c] = INT ? make_double2(fx_double_int(re, k2), fx_double_int(im, k2))
                   : make_double2(fx_double(re, bias), fx_double(im, bias));
    }
    return below && top != kFxZero;
}

template <bool INT, int N>
__device__ __forceinline__ bool fx_spin_of(const FxTile& T, int spin, int c0, int dag, int lane, double2 (&v)[N]) {
    switch (spin) {
        case 0: return fx_spin<0, INT>(T, c0, dag, lane, v);
        case 1: return fx_spin<1, INT>(T, c0, dag, lane, v);
        case 2: return fx_spin<2, INT>(T, c0, dag, lane, v);
        default: return fx_spin<3, INT>(T, c0, dag, lane, v);
    }
}

// v = a v, or x + a v, of N words from word0 on, and out = v.  Branches, not
// predicated instructions: the FP64 pipe takes 64 cycles for either.
template <int N>
__device__ __forceinline__ void fx_finish(const FxParams& P, uint4* out, const uint4* x, int word0, double2 (&v)[N]) {
    if (P.xpay) {
        double2 xv[N];
#pragma unroll
        for (int q = 0; q < N; q++)
            xv[q] = __ldg(reinterpret_cast<const double2*>(x) + (long long)(word0 + q) * P.x.word_step);
#pragma unroll
        for (int q = 0; q < N; q++) v[q] = make_double2(fma(P.a, v[q].x, xv[q].x), fma(P.a, v[q].y, xv[q].y));
    } else if (P.scaled) {
#pragma unroll
        for (int q = 0; q < N; q++) v[q] = make_double2(v[q].x * P.a, v[q].y * P.a);
    }
    double2* o = reinterpret_cast<double2*>(out);
#pragma unroll
    for (int q = 0; q < N; q++) {
        if (P.nrhs > 1) __stcs(o + (long long)(word0 + q) * P.out.word_step, v[q]);
        else o[(long long)(word0 + q) * P.out.word_step] = v[q];
    }
}

template <int N>
__device__ __forceinline__ double fx_norm(const double2 (&v)[N]) {
    double n = 0.0;
#pragma unroll
    for (int q = 0; q < N; q++) n += v[q].x * v[q].x + v[q].y * v[q].y;
    return n;
}

__device__ __forceinline__ const int* fx_exponents(const char* f, long long stride) {
    return reinterpret_cast<const int*>(f + 192 * stride);
}
__device__ __forceinline__ int* fx_exponents(char* f, long long stride) { return reinterpret_cast<int*>(f + 192 * stride); }
constexpr int kFxExpMask = 0xFFF;  // of a word of them; bits 12 to 15: the spins with a nonzero component

__device__ __forceinline__ double fx_flip(double v, int neg) {
    return __hiloint2double(__double2hiint(v) ^ neg << 31, __double2loint(v));
}

// Two sites, h of lanes 0 to 15 and h of lanes 16 to 31, in FP64, output included where mine;
// returns this thread's share of its squared modulus.  All lanes of a warp call it; w: three rows of 32 words
// of the warp's own, ws apart.  Sixteen lanes a site, one per hop and half-spin row, and then one per output
// component for the sum, with the FP64 stencil's operations in its order.  A lone
// site takes 54 FP64 instructions of 64 cycles in a row this way, one on a thread of its own 850.
inline __device__ __noinline__ double fx_redo(const FxParams& P, double2* w, int ws, int p, int k, int h, bool mine, int outfx) {
    const int lane = threadIdx.x & 31, l = lane & 15, j = l >> 1, r = l & 1, mu = j >> 1;
    const bool fwd = (j & 1) == 0;
    int c[4], s;
    site_of_half(h, p, P.g, c, s);
    {
        bool wrap;
        const int sn = fx_neighbour(P.g, c, s, j, wrap);
        const int partner = mu < 2 ? 3 - r : 2 + r;
        const int S = fwd != (P.dag != 0) ? 1 : -1, imag = mu == 0 || mu == 2;
        const int neg = ((mu == 2 && r == 1) || (mu == 1 && r == 0) ? S : -S) < 0;
        cpx<double> u[3][3], a[3];
        const FxField& f = P.nat.p ? P.nat : P.in;
        const uint4* psi = fx_at(f, 1 - p, k, sn);
        const int e = P.nat.p ? 0 : fx_exponents(reinterpret_cast<const char*>(fx_at(f, 1 - p, k, 0)), P.g.stride)[sn >> 1] & kFxExpMask;
        const double scale = __hiloint2double((e - 57) << 20, 0);  // 2^(e + 1 - 1023 - 58), if e != 0
        auto load = [&](int q) {
            const uint4 d = __ldg(psi + (long long)q * f.word_step);
            if (e == 0) return cpx<double>{__hiloint2double((int)d.y, (int)d.x), __hiloint2double((int)d.w, (int)d.z)};
            return cpx<double>{__ll2double_rn((long long)(int)d.x * (kFxLow + 1LL) + (int)d.y) * scale,
                               __ll2double_rn((long long)(int)d.z * (kFxLow + 1LL) + (int)d.w) * scale};
        };
        const double2* lk = reinterpret_cast<const double2*>(fwd ? fx_link_at(P.un, p, mu, s) : fx_link_at(P.un, 1 - p, mu, sn));
#pragma unroll
        for (int q = 0; q < 9; q++)
            if (q < P.un_recon / 2) {
                const double2 d = __ldg(lk + (long long)q * P.un.word_step);
                u[q / 3][q % 3] = {d.x, d.y};
            }
        if (P.un_recon == 12) recon_row2(u);
#pragma unroll
        for (int q = 0; q < 3; q++) {  // (1 - S g_mu) psi, row r (project() in dslash_impl.cuh)
            const cpx<double> x = load(3 * r + q), y = load(3 * partner + q);
            a[q] = {x.re + fx_flip(imag ? y.im : y.re, imag ? 1 - neg : neg), x.im + fx_flip(imag ? y.re : y.im, neg)};
        }
        if (wrap) {
            const cpx<double> eta = {P.g.ph[mu][0], fwd ? P.g.ph[mu][1] : -P.g.ph[mu][1]};
#pragma unroll
            for (int q = 0; q < 3; q++) a[q] = cmul(eta, a[q]);
        }
        if (!fwd) {  // U^dag
#pragma unroll
            for (int i = 0; i < 3; i++)
#pragma unroll
                for (int q = 0; q <= i; q++) {
                    const cpx<double> t = cconj(u[i][q]);
                    u[i][q] = cconj(u[q][i]);
                    u[q][i] = t;
                }
        }
#pragma unroll
        for (int i = 0; i < 3; i++) {
            cpx<double> t = cmul(u[i][0], a[0]);
            t = cfma(u[i][1], a[1], t);
            t = cfma(u[i][2], a[2], t);
            w[ws * i + lane] = make_double2(t.re, t.im);
        }
    }
    __syncwarp();
    double n2 = 0.0;
    if (mine && l < 12) {
        const int spin = l / 3, lower = spin >= 2;
        double2 v[1];
#pragma unroll
        for (int q = 0; q < 8; q++) {  // expand() in dslash_impl.cuh
            const int m = q >> 1, row = lower ? (spin == 2) == (m < 2) : spin;
            const double2 t = w[ws * (l - 3 * spin) + (lane & 16) + 2 * q + row];
            const int i = lower && (m == 0 || m == 2);
            const int neg = lower && (((q & 1) != 0) != (P.dag != 0)) != (m == 3 || (m == 1 && spin == 2) || (m == 2 && spin == 3));
            const double2 x = make_double2(fx_flip(i ? t.y : t.x, i ? 1 - neg : neg), fx_flip(i ? t.x : t.y, neg));
            v[0] = q ? make_double2(v[0].x + x.x, v[0].y + x.y) : x;
        }
        if (outfx) {
            char* out = P.out.p + (P.full ? p * P.out.pstep : 0) + k * P.out.rstep;
            reinterpret_cast<double2*>(out)[h + (long long)l * P.g.stride] = v[0];
            if (l == 0) fx_exponents(out, P.g.stride)[h] = 0;
        } else {
            fx_finish(P, const_cast<uint4*>(fx_at(P.out, p, k, s)), P.xpay ? fx_at(P.x, p, k, s) : nullptr, l, v);
            n2 = fx_norm(v);
        }
    }
    __syncwarp();
    return n2;
}
// The sites h0 + i of the bits i of m (the same for all lanes), of every `step` pairs the one numbered `turn`.
__device__ __forceinline__ double fx_redo_sites(const FxParams& P, double2* w, int ws, int p, int k, int h0, unsigned m,
                                                int turn, int step, int outfx) {
    double n2 = 0.0;
    for (; m; turn--) {
        const int a = __ffs(m) - 1;
        m &= m - 1;
        const int b = m ? __ffs(m) - 1 : -1;
        m &= m - 1;
        if (turn) continue;
        turn = step;
        const bool second = threadIdx.x & 16;
        n2 += fx_redo(P, w, ws, p, k, h0 + (second && b >= 0 ? b : a), !second || b >= 0, outfx);
    }
    return n2;
}

// ---------------------------------------------------------------------------
// Fields and links in fixed point, for the kernel below: each is converted once
// instead of in each of the eight hops that read it.  A spinor field has 12 rows
// of 16-byte words (re.h, re.l, im.h, im.l; v = h 2^29 + l) and a row of exponents, one per site, with its
// nonzero spins; a site that does not fit has exponent 0 and holds its doubles.  Links: nine rows
// per (parity, mu) as for doubles; a link that does not fit is marked in its first
// word (kFxBadLink) and read from the doubles.
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ long long fx_field_bytes(long long stride) { return 196 * stride; }

// Converts doubles (src; half-site index i, parity par) to a fixed-point field.
static __global__ void __launch_bounds__(128) fx_pack_kernel(FxField src, char* dst, long long pstep, long long rstep,
                                                             int nrhs, int par0, int npar, Geom g, const int* skip,
                                                             int skip_stride) {
    const int k = blockIdx.x % nrhs, sb = blockIdx.x / nrhs;
    const int par = npar == 2 ? (int)blockIdx.y : par0;
    const int i = sb * blockDim.x + threadIdx.x;
    pdl_wait();
    if (i >= g.Vh || (skip && __ldcg(skip + (size_t)k * skip_stride))) return;
    int s = 2 * i;
    if (src.by_site) {
        int c[4];
        site_of_half(i, par, g, c, s);
    }
    const uint4* in = reinterpret_cast<const uint4*>(src.p + (par && npar == 2 ? src.pstep : 0) + k * src.rstep) +
                      (long long)(src.by_site ? s : i) * src.site_step;
    char* f = dst + (npar == 2 ? par * pstep : 0) + k * rstep;
    uint4 d[12];
    unsigned m = 0, spins = 0;
#pragma unroll
    for (int q = 0; q < 12; q++) {
        d[q] = __ldg(in + (long long)q * src.word_step);
        m = fx_max2(m, d[q]);
        if (fx_nonzero(d[q])) spins |= 1u << (q / 3);
    }
    int e = (int)(m >> 21);
    if (e < kFxEmin || e > kFxEmax) e = spins ? 0 : kFxEmin;
    if (e) {
        const unsigned ew = fx_scale_word(e + kFxOffSpinor);
#pragma unroll
        for (int q = 0; q < 12; q++) {
            const FxMag a = fx_mag(d[q].y, d[q].x, fx_shift(ew, d[q].y << 1));
            const FxMag b = fx_mag(d[q].w, d[q].z, fx_shift(ew, d[q].w << 1));
            const int sa = fx_sign(d[q].y, 1), sb2 = fx_sign(d[q].w, 1);
            d[q] = make_uint4((unsigned)(a.h * sa), (unsigned)(a.l * sa), (unsigned)(b.h * sb2), (unsigned)(b.l * sb2));
        }
    }
    uint4* o = reinterpret_cast<uint4*>(f) + i;
#pragma unroll
    for (int q = 0; q < 12; q++) o[(long long)q * g.stride] = d[q];
    fx_exponents(f, g.stride)[i] = e ? e | (int)(spins << 12) : 0;
    pdl_trigger();
}

// a += SG i^I w.
template <int I, int SG>
__device__ __forceinline__ void fx_add(long long (&a)[2], long long wr, long long wi) {
    const long long x = I ? wi : wr, y = I ? wr : wi;  // i (x + i y) = -y + i x
    a[0] = (I ? -SG : SG) > 0 ? a[0] + x : a[0] - x;
    a[1] = SG > 0 ? a[1] + y : a[1] - y;
}
__device__ __forceinline__ void fx_negate_if(long long (&a)[3][2], int neg) {
    const long long m = -(long long)neg;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int z = 0; z < 2; z++) a[i][z] = (a[i][z] ^ m) - m;
}

// A block's shared memory.  Copies ahead (cp.async), so that the loads in flight hold
// no registers: a thread's six words of its neighbour, filled again as soon as they are projected,
// and the nine words of a hop's link and of the next one's, shared by the site's two
// threads; and the site's neighbours (hop 2 mu + dir: half-site index, wrap in the top bit; exponent).
template <int TB>
struct FxSlots {
    uint4 s[6][TB];
    uint4 l[2][9][TB / 2];
    int2 nb[8][TB / 2];
};
__device__ __forceinline__ void fx_copy(uint4* dst, const uint4* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void fx_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void fx_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Spin r and its partner in direction MU (3 - r or 2 + r) of neighbour hn.
template <int MU, int TB>
__device__ __forceinline__ void fx_issue_spinor(FxSlots<TB>& T, const char* in, int hn, int r, int stride) {
    const uint4* src = reinterpret_cast<const uint4*>(in) + hn;
    const uint4* ps = src + (long long)(3 * r) * stride;
    const uint4* qs = src + (long long)(MU < 2 ? 9 - 3 * r : 6 + 3 * r) * stride;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        fx_copy(&T.s[c][threadIdx.x], ps + (long long)c * stride);
        fx_copy(&T.s[3 + c][threadIdx.x], qs + (long long)c * stride);
    }
    fx_commit();
}
// Words 0-4 (r = 0) or 5-8 of link i of a block.
template <int TB>
__device__ __forceinline__ void fx_issue_link(uint4 (&T)[9][TB / 2], const char* gauge, int blk, int i, int r, int sl,
                                              int stride) {
    const uint4* src = reinterpret_cast<const uint4*>(gauge) + (long long)(blk * 9 + 5 * r) * stride + i;
    uint4* dst = &T[5 * r][sl];
#pragma unroll
    for (int q = 0; q < 4; q++) fx_copy(dst + q * (TB / 2), src + (long long)q * stride);
    if (r == 0) fx_copy(dst + 4 * (TB / 2), src + 4LL * stride);
    fx_commit();
}

// Row r of the neighbour's projection in direction MU: psi_r + sigma i^(imag) psi_partner.
template <int MU, int TB>
__device__ __forceinline__ void fx_take_row(const FxSlots<TB>& T, int sigma, FxCplx (&h)[3]) {
    constexpr bool imag = MU == 0 || MU == 2;
    const int sa = imag ? -sigma : sigma;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const uint4 p = T.s[c][threadIdx.x], q = T.s[3 + c][threadIdx.x];
        // i q = (-q.im, q.re)
        const int ah = (int)(imag ? q.z : q.x), al = (int)(imag ? q.w : q.y);
        const int bh = (int)(imag ? q.x : q.z), bl = (int)(imag ? q.y : q.w);
        h[c].re = FxReal{ah * sa + (int)p.x, al * sa + (int)p.y};
        h[c].im = FxReal{bh * sigma + (int)p.z, bl * sigma + (int)p.w};
    }
}

// The sums of one of a site's two threads (r = 0, 1), with the scale at 2^56: spin r
// (up), and the parts of the lower spins that come from row r: lo[0] from the x and y
// directions, for spin 3 - r, and lo[1] from z and t, for spin 2 + r.
struct FxSums {
    long long up[3][2], lo[2][3][2];
    unsigned n[3][2], k[4][3];  // the guard's moduli of the current direction, and each direction's counts (re, im)
};

// The order of the hops: y, x, z, t, backward before forward (see hop_kernel_fx1).
constexpr int fx_order_mu(int n) { return n < 2 ? 1 : n < 4 ? 0 : n < 6 ? 2 : 3; }

// What the threads of a site have in common.
struct FxTurn {
    int h, top, r, sl, p, S;  // S: the projectors' sign of forward hops
};

// Hop number N of that order into the sums; the copies of its neighbour and its link
// are on their way, and those of the next one are issued.  The lower spins take S
// times the upper ones' image, S = 1 forward and -1 backward here.
template <int N, int TB>
__device__ __forceinline__ bool fx_turn_hop(const FxParams& P, FxSlots<TB>& T, FxSums& A, const FxTurn& t, const char* in) {
    constexpr int MU = fx_order_mu(N), NX = fx_order_mu(N < 7 ? N + 1 : 7);
    constexpr bool bwd = (N & 1) == 0, imag = MU == 0 || MU == 2;
    const int2 nb = T.nb[2 * MU + (bwd ? 1 : 0)][t.sl];
    __syncwarp();  // both threads are done with the last hop's link
    int nhn = 0;
    if constexpr (N < 7) {
        nhn = T.nb[2 * NX + (bwd ? 0 : 1)][t.sl].x & 0x7FFFFFFF;
        fx_issue_link<TB>(T.l[(N + 1) & 1], P.u.p, (bwd ? t.p : 1 - t.p) * 4 + NX, bwd ? t.h : nhn, t.r, t.sl, P.g.stride);
    } else {
        fx_commit();
    }
    fx_wait<1>();  // all but that link
    __syncwarp();
    FxCplx h[3];
    const int sigma = (MU == 1 && t.r == 0) || (MU == 2 && t.r == 1) ? t.S : -t.S;
    fx_take_row<MU>(T, bwd ? -sigma : sigma, h);
    if constexpr (N < 7) fx_issue_spinor<NX>(T, in, nhn, t.r, P.g.stride);
    if (nb.x < 0) fx_wrap(P.g.ph[MU][0], bwd ? -P.g.ph[MU][1] : P.g.ph[MU][1], h);
    const int d = min(t.top - nb.y, kFxMaxShift);
    const long long half = fx_half(d);
    FxReal neg[3];  // forward U h: Ur hr - Ui hi, Ur hi + Ui hr; backward U^dag h: Ur hr + Ui hi, Ur hi - Ui hr
#pragma unroll
    for (int k = 0; k < 3; k++) neg[k] = fx_neg(bwd ? h[k].re : h[k].im);
    bool bad = false;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        FxAcc re = fx_zero(half), im = fx_zero(half);
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const uint4 w = T.l[N & 1][bwd ? k * 3 + i : i * 3 + k][t.sl];
            if (i == 0 && k == 0) bad = w.x == kFxBadLink;
            const FxReal ur{(int)w.x, (int)w.y}, ui{(int)w.z, (int)w.w};
            fx_mac(re, ur, h[k].re);
            fx_mac(im, ur, h[k].im);
            fx_mac(re, ui, bwd ? h[k].im : neg[k]);
            fx_mac(im, ui, bwd ? neg[k] : h[k].re);
        }
        const long long wr = fx_align(fx_sum(re), d), wi = fx_align(fx_sum(im), d);
        A.up[i][0] += wr;
        A.up[i][1] += wi;
        // lower spins: x: i w1, i w0; y: -w1, w0 (spin 2, spin 3); z: i w0, -i w1; t: -w0, -w1;
        // the minus of row 1 in y and z is put in by fx_negate_if
        fx_add<imag ? 1 : 0, bwd == (MU == 3) ? 1 : -1>(A.lo[MU >> 1][i], wr, wi);
        A.n[i][0] = fx_modulus(wr, bwd ? 0 : A.n[i][0]);
        A.n[i][1] = fx_modulus(wi, bwd ? 0 : A.n[i][1]);
        if (!bwd) A.k[MU][i] = fx_count(A.n[i][0], A.n[i][1]);
    }
    return bad;
}

// One site on two threads, lanes l and l + 16 of a warp, one per half-spin row: a
// thread keeps 18 64-bit sums instead of the 24 of a thread with both rows, and half of
// the half spinor.  Output: doubles, or a fixed-point field (OUTFX; out.p in
// that form, no xpay or scale).  The block's sites are h0 and the next ones, a thread past the end runs site 0 and
// stores nothing; returns the sites of its warp that are to be done over (bits 0 to 15).
struct FxDone {
    double n2;  // this thread's share of the output's squared modulus (RED)
    unsigned redo;
};
template <bool OUTFX, bool RED, int TB>
__device__ __forceinline__ FxDone fx_sites(const FxParams& P, FxSlots<TB>& T, const char* in, int p, int k, int h0) {
    const Geom& g = P.g;
    FxTurn t;
    t.r = threadIdx.x >> 4 & 1;
    t.sl = (threadIdx.x >> 5) * 16 + (threadIdx.x & 15);
    t.S = P.dag ? -1 : 1;
    t.p = p;
    double nrm = 0.0;
    const bool ok = h0 + t.sl < g.Vh;
    const int h = ok ? h0 + t.sl : 0, r = t.r;
    t.h = h;
    bool bad;
    int spins;  // nonzero ones of the neighbours: bits 0 to 3 in x and y, 4 to 7 in z and t
    __syncwarp();
    {
        // thread r: the forward (0) or backward (1) neighbours
        const int* ex = fx_exponents(in, g.stride);
        int c[4], s, top = 0, low = 1 << 30;
        spins = 0;
        site_of_half(h, p, g, c, s);
#pragma unroll
        for (int mu = 0; mu < 4; mu++) {
            const int smu = mu == 0 ? 1 : mu == 1 ? g.L[0] : mu == 2 ? g.L[0] * g.L[1] : g.L[0] * g.L[1] * g.L[2];
            const bool w = c[mu] == (r ? 0 : g.L[mu] - 1);
            const int step = r ? -smu : smu;
            const int hn = (w ? s - step * (g.L[mu] - 1) : s + step) >> 1;
            const int ew = __ldg(ex + hn), e = ew & kFxExpMask;
            spins |= ew >> 12 << (mu < 2 ? 0 : 4);
            top = max(top, e);
            low = min(low, e);
            T.nb[2 * mu + r][t.sl] = make_int2(hn | (w ? (int)0x80000000 : 0), e);
        }
        t.top = max(top, __shfl_xor_sync(0xffffffffu, top, 16));
        bad = min(low, __shfl_xor_sync(0xffffffffu, low, 16)) == 0;
        spins |= __shfl_xor_sync(0xffffffffu, spins, 16);
    }
    __syncwarp();
    {
        const int hn = T.nb[3][t.sl].x & 0x7FFFFFFF;
        fx_issue_link<TB>(T.l[0], P.u.p, (1 - p) * 4 + 1, hn, r, t.sl, g.stride);
        fx_issue_spinor<1>(T, in, hn, r, g.stride);
    }
    FxSums A;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int z = 0; z < 2; z++) A.up[i][z] = A.lo[0][i][z] = A.lo[1][i][z] = 0;
    bad |= fx_turn_hop<0>(P, T, A, t, in);
    bad |= fx_turn_hop<1>(P, T, A, t, in);
    fx_negate_if(A.lo[0], r);
    bad |= fx_turn_hop<2>(P, T, A, t, in);
    bad |= fx_turn_hop<3>(P, T, A, t, in);
    bad |= fx_turn_hop<4>(P, T, A, t, in);
    bad |= fx_turn_hop<5>(P, T, A, t, in);
    fx_negate_if(A.lo[1], r);
    bad |= fx_turn_hop<6>(P, T, A, t, in);
    bad |= fx_turn_hop<7>(P, T, A, t, in);
    const int top = t.top;
    // spin 3 - r: this thread's x and y part, the other's z and t part
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int z = 0; z < 2; z++) A.lo[0][i][z] += __shfl_xor_sync(0xffffffffu, A.lo[1][i][z], 16);
    if (P.dag) fx_negate_if(A.lo[0], 1);
    {
        // the guard, but for a spin to which only zeros contribute (row q: spin q, and 3 - q in x and y, 2 + q in z and t)
        bool up = false, lo = false;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const unsigned zt = fx_swap(A.k[2][i]) + A.k[3][i], zt1 = __shfl_xor_sync(0xffffffffu, zt, 16);
            up = up || fx_below(A.k[0][i] + A.k[1][i] + A.k[2][i] + A.k[3][i]);
            lo = lo || fx_below(fx_swap(A.k[0][i]) + A.k[1][i] + zt1);
        }
        const int xy = (1 << r | 8 >> r) & spins, zt = (1 << r | 4 << r) & spins >> 4, zt1 = (2 >> r | 8 >> r) & spins >> 4;
        bad = bad || (up && (xy | zt)) || (lo && (xy | zt1));
        const int bad2 = __shfl_xor_sync(0xffffffffu, (int)bad, 16);
        bad = bad || bad2;
    }
    if constexpr (OUTFX) {
        // to 58 bits below the largest component: shift right by sr, left if negative
        unsigned long long mu = 0, ml = 0;
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int z = 0; z < 2; z++) {
                mu |= (unsigned long long)(A.up[i][z] ^ (A.up[i][z] >> 63));
                ml |= (unsigned long long)(A.lo[0][i][z] ^ (A.lo[0][i][z] >> 63));
            }
        unsigned long long m = mu | ml;
        m |= __shfl_xor_sync(0xffffffffu, m, 16);
        int nz = (mu ? 1 << r : 0) | (ml ? 8 >> r : 0);
        nz |= __shfl_xor_sync(0xffffffffu, nz, 16);
        const int sr = m ? 6 - __clzll((long long)m) : 0;
        const int eo = m ? top + 2 + sr : kFxEmin;
        bad = bad || eo < kFxEmin || eo > kFxEmax;
        if (ok && !bad) {
            const long long half = sr > 0 ? 1LL << (sr - 1) : 0;
            char* out = P.out.p + (P.full ? p * P.out.pstep : 0) + k * P.out.rstep;
            uint4* ob = reinterpret_cast<uint4*>(out) + h;
#pragma unroll
            for (int q = 0; q < 6; q++) {
                long long v[2];
#pragma unroll
                for (int z = 0; z < 2; z++) {
                    v[z] = q < 3 ? A.up[q][z] : A.lo[0][q - 3][z];
                    v[z] = sr > 0 ? (v[z] + half) >> sr : v[z] << -sr;
                }
                ob[(long long)(q < 3 ? 3 * r + q : 6 - 3 * r + q) * g.stride] =
                    make_uint4((unsigned)(v[0] >> kFxLimb), (unsigned)v[0] & kFxLow, (unsigned)(v[1] >> kFxLimb),
                               (unsigned)v[1] & kFxLow);
            }
            if (r == 0) fx_exponents(out, g.stride)[h] = eo | nz << 12;
        }
    } else if (ok && !bad) {
        const FxBias b = fx_bias(top + 1 - 1023 - 56);
        int c[4], s;
        site_of_half(h, p, g, c, s);
        uint4* out = const_cast<uint4*>(fx_at(P.out, p, k, s));
        const uint4* x = P.xpay ? fx_at(P.x, p, k, s) : nullptr;
        double2 v[3];
#pragma unroll
        for (int i = 0; i < 3; i++) v[i] = make_double2(fx_double(A.up[i][0], b), fx_double(A.up[i][1], b));
        fx_finish(P, out, x, 3 * r, v);
        if (RED) nrm += fx_norm(v);
#pragma unroll
        for (int i = 0; i < 3; i++) v[i] = make_double2(fx_double(A.lo[0][i][0], b), fx_double(A.lo[0][i][1], b));
        fx_finish(P, out, x, 9 - 3 * r, v);
        if (RED) nrm += fx_norm(v);
    }
    return FxDone{nrm, __ballot_sync(0xffffffffu, ok && bad) & 0xFFFFu};
}

template <bool OUTFX, bool RED, int TB, int MINB>
__global__ void __launch_bounds__(TB, MINB) hop_kernel_fx1(const __grid_constant__ FxParams P) {
    extern __shared__ __align__(16) unsigned char fx_smem[];
    FxSlots<TB>& T = *reinterpret_cast<FxSlots<TB>*>(fx_smem);
    constexpr int SITES = TB / 2;
    const int k = blockIdx.x % P.nrhs;
    const int sb = blockIdx.x / P.nrhs;
    const int nb = gridDim.x / P.nrhs;
    const int p = P.full ? (int)blockIdx.y : P.out_parity;
    pdl_wait();
    if (P.skip && __ldcg(P.skip + (size_t)k * P.skip_stride)) return;
    const char* in = P.in.p + (P.full && p == 0 ? P.in.pstep : 0) + k * P.in.rstep;
    const int warp = threadIdx.x >> 5;
    double2* w = reinterpret_cast<double2*>(&T.s[0][32 * warp]);  // the warp's columns, all of whose copies have arrived
    double nrm = 0.0;
    if constexpr (RED) {
        // Turns, and then the sites to be done over: a call to fx_redo in the loop costs it 40
        // registers' spills, a call for the turn 28 % of the hop's time.
        unsigned short* redo = reinterpret_cast<unsigned short*>(fx_smem + sizeof(FxSlots<TB>)) + warp;  // [turn][warp]
        int n = 0;
        unsigned any = 0;
        for (int h0 = sb * SITES; h0 < P.g.Vh; h0 += nb * SITES, n++) {
            const FxDone d = fx_sites<OUTFX, RED>(P, T, in, p, k, h0);
            nrm += d.n2;
            any |= d.redo;
            if ((threadIdx.x & 31) == 0) redo[n * (TB / 32)] = (unsigned short)d.redo;
        }
        __syncwarp();
        if (any)
            for (int i = 0; i < n; i++)
                nrm += fx_redo_sites(P, w, TB, p, k, (sb + i * nb) * SITES + 16 * warp, redo[i * (TB / 32)], 0, 1, OUTFX);
    } else {  // the grid covers the sites
        const FxDone d = fx_sites<OUTFX, RED>(P, T, in, p, k, sb * SITES);
        if (d.redo) fx_redo_sites(P, w, TB, p, k, sb * SITES + 16 * warp, d.redo, 0, 1, OUTFX);
    }
    pdl_trigger();
    if (RED) grid_reduce(nrm, P.red, k, nb * gridDim.y, sb + nb * blockIdx.y);
}

// Up to 32 sites, h0 to end, of parity p and right-hand side k, by a block of W warps; adds
// this thread's share of the output's squared modulus to nrm (RED) and returns the sites that are to be
// done over (fx_tile_redo), the same to all threads.  A barrier has to come before the tile is used again.
template <bool FXL, bool RED, int W>
__device__ __forceinline__ unsigned fx_tile(const FxParams& P, FxTile& T, int p, int k, int h0, int end, double& nrm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int h = h0 + lane;
    const bool ok = h < end;
    int c[4], s;
    site_of_half(ok ? h : 0, p, P.g, c, s);
    if (warp == 0) T.bad[lane] = 0;
    __syncthreads();
#pragma unroll 1
    for (int j = warp; j < 8; j += W) fx_hop<FXL>(P, T, j, p, k, c, s, lane);
    __syncthreads();
    const int spin = warp & 3;
    double2 va[W == 8 ? 2 : 3], vb[1];  // warps 4 to 7: the third colour
    const bool below = warp < 4 ? fx_spin_of<W == 4>(T, spin, 0, P.dag, lane, va) : fx_spin_of<W == 4>(T, spin, 2, P.dag, lane, vb);
    if (below) T.bad[lane] = 1;
    // with RED a site that is done over must not be in the sum; else it is stored twice (x is
    // never the output), which puts the stores before the barrier: 8^4 hop 6.70 -> 6.64 us
    if (RED) __syncthreads();
    if (ok && !(RED && T.bad[lane])) {
        uint4* out = const_cast<uint4*>(fx_at(P.out, p, k, s));
        const uint4* x = P.xpay ? fx_at(P.x, p, k, s) : nullptr;
        if (warp < 4) {
            fx_finish(P, out, x, spin * 3, va);
            if (RED) nrm += fx_norm(va);
        } else {
            fx_finish(P, out, x, spin * 3 + 2, vb);
            if (RED) nrm += fx_norm(vb);
        }
    }
    if (!RED) __syncthreads();
    return __ballot_sync(0xffffffffu, ok && T.bad[lane]);
}
template <int W>
__device__ __forceinline__ double fx_tile_redo(const FxParams& P, FxTile& T, int p, int k, int h0, unsigned redo) {
    const int warp = threadIdx.x >> 5;
    return fx_redo_sites(P, reinterpret_cast<double2*>(T.w) + 96 * warp, 32, p, k, h0, redo, warp, W, 0);
}

// Grid: blockIdx.x = tile * nrhs + rhs, tiles of 32 sites; blockIdx.y = output
// parity of a full launch.  W warps, 4 or 8.
template <bool FXL, bool RED, int W, int MINB>
__global__ void __launch_bounds__(32 * W, MINB) hop_kernel_fx(const __grid_constant__ FxParams P) {
    __shared__ FxTile T;
    const int k = blockIdx.x % P.nrhs;
    const int sb = blockIdx.x / P.nrhs;
    const int nb = gridDim.x / P.nrhs;
    const int p = P.full ? (int)blockIdx.y : P.out_parity;
    pdl_wait();
    if (P.skip && __ldcg(P.skip + (size_t)k * P.skip_stride)) return;
    double nrm = 0.0;
    for (int h0 = sb * 32; h0 < P.g.Vh; h0 += nb * 32) {
        const unsigned redo = fx_tile<FXL, RED, W>(P, T, p, k, h0, P.g.Vh, nrm);
        if (redo) {
            const double n2 = fx_tile_redo<W>(P, T, p, k, h0, redo);
            if (RED) nrm += n2;
        }
        if (!RED) break;  // the grid covers the sites
        __syncthreads();
    }
    pdl_trigger();
    if (RED) grid_reduce(nrm, P.red, k, nb * gridDim.y, sb + nb * blockIdx.y);
}

}  // namespace wl
