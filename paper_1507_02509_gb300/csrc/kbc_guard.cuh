// FP64 re-evaluation of the guard's nodes for float storage.
//
// A node whose entropic denominator rho <dh|dh> is at or below the guard is
// collided in double and rounded once to float.  The stored bits of that
// computation are what counts, and for most nodes they can be had without the
// FP64 pipe (64 cycles per warp instruction, about 220 instructions a node):
//
// * In moment space the cancellations that make the node delicate are between
//   sums of the nine floats and products of the conserved moments.  The sums
//   are formed exactly, as 64-bit integers; the products rho u u in
//   pairs of floats (48 bits).  What remains, the six moments of df, is small
//   and known to 48 bits or to 2^-43 rho u^2.
// * Split, scalar products and gamma* follow in single precision, the products
//   of the central split in pairs of floats, and a bound on the
//   total error of each result decides whether its rounding to float is
//   settled (Ziv's test).  Where it is not, the node is queued and collided
//   in double as before.
//
// About 1250 instructions a node; 11 to 20% of the nodes of a shear layer
// (1024^2, B and A, guard 1e-16) go on to the double collision.
#pragma once

#include "kbc_kernels.cuh"

namespace kbc {

// d exactly as integers in the unit 2^(e - 180), e the biased exponent of the
// largest; false when the values do not fit (see FixedSums).
__device__ __forceinline__ bool fixed_values(const float (&d)[9], long long (&v)[9], int& e)
{
    unsigned top = 0u;
#pragma unroll
    for (int i = 0; i < 9; ++i) top = max(top, __float_as_uint(d[i]) & 0x7fffffffu);
    e = (int)(top >> 23);
    bool ok = e >= 64 && e <= 127;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const unsigned b = __float_as_uint(d[i]);
        const int ei = (int)((b >> 23) & 0xffu);
        const int sh = 30 - (e - ei);
        const int m = (int)((b & 0x7fffffu) | 0x800000u);
        const bool zero = (b << 1) == 0u;
        ok &= zero || (sh >= 0 && ei != 0);
        const int sm = zero ? 0 : ((int)b < 0 ? -m : m);
        v[i] = (long long)sm * (long long)(1 << (sh & 31));
    }
    return ok;
}

// |X| < 2^60 in units of 2^(e - 180) as three floats, exactly
__device__ __forceinline__ void three_floats(long long X, int e, float& t2, float& t1, float& t0)
{
    t2 = (float)(int)(X >> 36) * __uint_as_float((unsigned)(e - 17) << 23);
    t1 = (float)(int)((X >> 12) & 0xffffff) * __uint_as_float((unsigned)(e - 41) << 23);
    t0 = (float)(int)(X & 0xfff) * __uint_as_float((unsigned)(e - 53) << 23);
}
__device__ __forceinline__ FF<Lf> fixed_ff(long long X, int e)
{
    float t2, t1, t0;
    three_floats(X, e, t2, t1, t0);
    const FF<Lf> s = two_sum(Lf(t2), Lf(t1));
    return two_sum(s.h, s.l + Lf(t0));
}
// X - 3 p (n3 = -3) or X - p (n3 = -1)
__device__ __forceinline__ FF<Lf> fixed_minus(long long X, int e, FF<Lf> p, float n3)
{
    const Lf c(n3), ph = c * p.h;
    return fixed_ff(X, e) + FF<Lf>(ph, fmaL(c, p.l, fmaL(c, p.h, -ph)));
}

// -2 beta as a pair of floats and -(1 - 2 beta)
struct GuardParams {
    float n2b_h, n2b_l, nb;
    int settle;  // whether to try collide_settled
};

// Up to this guard most nodes of a flow are settled in single precision (1024^2
// shear layer, 856 k nodes at 1e-13: 348 -> 101 us a step for B, 167 -> 50
// for C); at 1e-9 and above few are, and trying costs up to a fifth.
constexpr double kGuardSettle = 1e-12;

// Post-collision floats of one node; false when the rounding of one is not
// settled.  u = 2^-24 is the unit roundoff of float below.
template <int VAR>
__device__ __forceinline__ bool collide_settled(const float (&d)[9], const GuardParams& p, float (&out)[9])
{
    using F = FF<Lf>;
    long long v[9];
    int e;
    bool ok = fixed_values(d, v, e);
    if (!ok) return false;
    const F third(Lf(ff_hi(1.0 / 3.0)), Lf(ff_lo(1.0 / 3.0))), ninth(Lf(ff_hi(1.0 / 9.0)), Lf(ff_lo(1.0 / 9.0)));
    // exact moments of d (a power of a, then of b)
    const long long s08 = v[0] + v[8], s26 = v[2] + v[6], a08 = v[8] - v[0], a26 = v[2] - v[6];
    const long long s35 = v[3] + v[5], a35 = v[5] - v[3], s17 = v[1] + v[7], a17 = v[7] - v[1];
    const long long m22 = s08 + s26, m12 = a08 + a26, m21 = a08 - a26;
    const F jx = fixed_ff(m12 + a35, e), jy = fixed_ff(m21 + a17, e);
    const F drho = fixed_ff(m22 + s35 + s17 + v[4], e);
    // 1 / rho: y (1 + r + r^2) with y the single-precision reciprocal
    F rho = two_sum(Lf(1.0f), drho.h);
    rho = two_sum(rho.h, rho.l + drho.l);
    const Lf y = rcp_fast(rho.h);
    const Lf r = fmaL(-rho.l, y, fmaL(-rho.h, y, Lf(1.0f)));
    const F irho = fast_two_sum(y, y * fmaL(r, r, r));
    const F ux = jx * irho, uy = jy * irho;
    const F mxx = jx * ux, myy = jy * uy, mxy = jx * uy;  // rho u u
    // moments of df = d - (f^eq - W): the equilibrium's are drho/3 + mxx (20),
    // mxy (11), jy/3 (21), drho/9 + (mxx + myy)/3 (22)
    const F M20 = fixed_minus(2 * (m22 + s35) - (s17 + v[4]), e, mxx, -3.0f) * third;
    const F M02 = fixed_minus(2 * (m22 + s17) - (s35 + v[4]), e, myy, -3.0f) * third;
    const F M11 = fixed_minus(s08 - s26, e, mxy, -1.0f);
    const F M21 = fixed_ff(2 * m21 - a17, e) * third;
    const F M12 = fixed_ff(2 * m12 - a35, e) * third;
    const F M22 = fixed_minus(8 * m22 - (s35 + s17 + v[4]), e, mxx + myy, -3.0f) * ninth;
    // split (see collide): second moments c of ds, its third and fourth ones S,
    // the moments H of dh
    F c20, c02;
    Lf h2(0.0f);  // H20 = H02
    if constexpr (VAR == kA || VAR == kC) {
        c20 = M20;
        c02 = M02;
    } else {
        c20 = scale(M20 - M02, 0.5f);
        c02 = -c20;
        h2 = scale(M20 + M02, 0.5f).h;
    }
    Lf s21(0.0f), s12(0.0f), s22(0.0f), h21 = M21.h, h12 = M12.h, h22 = M22.h;
    if constexpr (VAR == kA || VAR == kB) {
        const F S21 = uy * c20 + scale(ux * M11, 2.0f), S12 = ux * c02 + scale(uy * M11, 2.0f);
        const F S22 = uy * S21 + ux * S12;
        s21 = S21.h;
        s12 = S12.h;
        s22 = S22.h;
        h21 = (M21 - S21).h;
        h12 = (M12 - S12).h;
        h22 = (M22 - S22).h;
    }
    // populations with moments (n20, n02, n11, n21, n12, n22) and no mass or momentum
    auto populations = [](Lf n20, Lf n02, Lf n11, Lf n21, Lf n12, Lf n22, Lf (&f)[9]) {
        const Lf x2 = Lf(0.5f) * (n20 - n22), y2 = Lf(0.5f) * (n02 - n22);
        const Lf a = Lf(0.25f) * (n22 + n11), b = Lf(0.25f) * (n22 - n11);
        const Lf cp = Lf(0.25f) * (n12 + n21), cm = Lf(0.25f) * (n12 - n21);
        f[4] = n22 - (n20 + n02);
        f[5] = fmaL(Lf(-0.5f), n12, x2);
        f[3] = fmaL(Lf(0.5f), n12, x2);
        f[7] = fmaL(Lf(-0.5f), n21, y2);
        f[1] = fmaL(Lf(0.5f), n21, y2);
        f[8] = a + cp;
        f[0] = a - cp;
        f[2] = b + cm;
        f[6] = b - cm;
    };
    Lf dh[9], ds[9];
    populations(h2, h2, Lf(0.0f), h21, h12, h22, dh);
    populations(c20.h, c02.h, M11.h, s21, s12, s22, ds);
    // Scalar products weighted by w = rho / f^eq = (1 - P / (1 + P)) / W.  Under
    // 1 / W the Hermite moments are orthogonal, and ds and dh share few of
    // them, so <ds|dh> is far below |ds| |dh|: its part under 1 / W is taken
    // from the moments, only the rest, of order u, from the populations.
    const Lf nusq = Lf(-1.5f) * square_sum(ux.h, uy.h), sxy = ux.h + uy.h, dxy = ux.h - uy.h;
    Lf P[9];
    P[0] = eq_poly<0>(ux.h, uy.h, sxy, dxy, nusq);
    P[1] = eq_poly<1>(ux.h, uy.h, sxy, dxy, nusq);
    P[2] = eq_poly<2>(ux.h, uy.h, sxy, dxy, nusq);
    P[3] = eq_poly<3>(ux.h, uy.h, sxy, dxy, nusq);
    P[4] = nusq;
    P[5] = eq_poly<5>(ux.h, uy.h, sxy, dxy, nusq);
    P[6] = eq_poly<6>(ux.h, uy.h, sxy, dxy, nusq);
    P[7] = eq_poly<7>(ux.h, uy.h, sxy, dxy, nusq);
    P[8] = eq_poly<8>(ux.h, uy.h, sxy, dxy, nusq);
    Lf s1(0.0f), hh(0.0f);
    float Q = 0.0f, H1 = 0.0f, S1 = 0.0f;  // sums of magnitudes for the bound
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const float c = wclass(i) == 0 ? 0.25f : wclass(i) == 1 ? 0.5f : 1.0f;
        const Lf w = rcp_fast(fmaL(Lf((float)wgt(i)), P[i], Lf((float)wgt(i))));
        const Lf t = dh[i] * w, st = ds[i] * t;
        s1 = fmaL(st, P[i], s1);
        hh = fmaL(dh[i], t, hh);
        Q += fabsf(st.v);
        H1 = __fmaf_rn(c, fabsf(t.v), H1);
        S1 = __fmaf_rn(c, fabsf(ds[i].v * w.v), S1);
    }
    // second moments: the traceless part of ds meets the trace of dh (B, D), or
    // dh has none (A, C): no term.  H22' = H22 - (H20 + H02) / 3.
    const Lf third1(-1.0f / 3.0f);
    const Lf g22 = fmaL(third1, h2 + h2, h22);
    const Lf f22 = (VAR == kA || VAR == kC) ? fmaL(third1, c20.h + c02.h, s22) : s22;
    const Lf s0a = s21 * h21, s0b = s12 * h12, s0c = f22 * g22;
    const Lf sh = fmaL(Lf(13.5f), s0a + s0b, fmaL(Lf(20.25f), s0c, -s1));
    const Lf R = ratio(sh, hh), nb(p.nb);
    const Lf nch = fmaL(nb, R, nb);
    // Error bound.  delta: the moments of df.  1 / rho is a pair to 2^-46, u to
    // 2^-44.3, a product rho u u to 2^-43.6 (M22 holds a third of two of them,
    // the third moments hold none and are far more exact), and the double
    // computation that this stands for adds 2^-50 of the largest value.  The
    // split adds um < 0.3 times delta to third and um^2 to fourth moments, so
    // that the populations made of the moments are off by at most 3 delta,
    // times 1/4 and 1/2 on the diagonals and axes (at rest three moments enter
    // whole, of which M22 with a third).  us, uh: rounding of ds and dh formed
    // from their moments.  The sums' own rounding is 14 u of their magnitudes:
    // nine additions, two products and three for the weight, where
    // |P / (1 + P)| <= pm.  <ds|dh>'s part under 1 / W moves with the errors of
    // f22 and g22, below 1.7 delta (20.25 of it, 35), and with those of the
    // third moments, below 2 um delta (13.5 of it 27 um; 60 um is taken).
    const float u = 0x1p-24f;
    const float delta = 0x1p-43f * (mxx.h.v + myy.h.v) + __uint_as_float((unsigned)(e - 49) << 23);
    const float um = fabsf(ux.h.v) + fabsf(uy.h.v), pm = 1.5f * (3.0f * um + 6.0f * um * um);
    const float third_s = fabsf(s21.v) + fabsf(s12.v), third_h = fabsf(h21.v) + fabsf(h12.v);
    const float us = 3.0f * u * (fabsf(c20.h.v) + fabsf(c02.h.v) + fabsf(M11.h.v) + third_s + fabsf(s22.v));
    const float uh = 3.0f * u * (2.0f * fabsf(h2.v) + third_h + fabsf(h22.v));
    const float esh = 14.0f * u * (pm * Q + 13.5f * (fabsf(s0a.v) + fabsf(s0b.v)) + 20.25f * fabsf(s0c.v)) +
                      pm * (H1 * (3.0f * delta + us) + S1 * (3.0f * delta + uh)) +
                      delta * (35.0f * (fabsf(f22.v) + fabsf(g22.v)) + 60.0f * um * (third_s + third_h));
    const float ehh = 14.0f * u * hh.v + (6.0f * delta + 2.0f * uh) * H1;
    const float aR = fabsf(R.v), anb = fabsf(p.nb) * 1.01f, a2b = -p.n2b_h * 1.01f;
    const float dR = anb * (esh + aR * ehh) * __fdividef(1.01f, hh.v);
    const float flat = a2b * (3.0f * delta + us + uh) + anb * (1.0f + aR) * (3.0f * delta + uh);
    // where the constants hold: moderate density and speed
    ok = hh.v > 1e-30f && rho.h.v > 0.5f && rho.h.v < 2.0f && um < 0.3f;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const float c = wclass(i) == 0 ? 0.25f : wclass(i) == 1 ? 0.5f : 1.0f;
        const Lf df = ds[i] + dh[i];
        const Lf corr = fmaL(nch, dh[i], fmaL(Lf(p.n2b_h), df, Lf(p.n2b_l) * df));
        const float ah = fabsf(dh[i].v);
        const float err = ah * dR + c * flat + 4.0f * u * (a2b * fabsf(df.v) + fabsf(nch.v) * ah);
        round_sure(d[i], corr.v, err, out[i], ok);
    }
    return ok;
}

// One block of 16 warps per SM.  A list of up to 128 nodes per block is
// collided in double at once: one warp per scheduler, whose 220 instructions
// of 64 cycles are the shortest time a double collision takes (7 us).  A
// longer one is dealt out in pieces of 32 entries, first over the blocks, then
// over their warps, so that lists of any length and nodes of either kind, which
// lie together, come evenly to the SMs; each warp works through its own pieces
// and leaves the nodes that are not settled at the beginning of them, and after
// one block barrier the block collides those in double.  A warp that settles
// fewer than a quarter leaves its other pieces as they are.
// 1024^2, float B, us a step with every node in double and an atomic addition
// per lane that reports one, with a stretch of the list per block, and now:
// shear layer at 200 steps 151, 45, 39; a vortex with 27 k nodes 29, 50, 28; at
// rest, where nothing is settled, 471, 488, 449.
constexpr int kGuardBlock = 512;
constexpr int kGuardWarps = kGuardBlock / 32;
constexpr int kGuardDirect = 128;

template <int VAR>
__global__ void __launch_bounds__(kGuardBlock, 1)
step_guard(const float* __restrict__ src, float* __restrict__ dst, StepArgs a, GuardParams gp)
{
    // per warp: entries left, and those of them at the beginning of its
    // pieces; the others are all from the piece `from` on
    __shared__ int left[kGuardWarps], kept_of[kGuardWarps], from_of[kGuardWarps];
    chain_enter();
    const int recorded = ld_count(a.fix_count + a.fix_slot);
    const int count = recorded < a.nx * a.ny ? recorded : a.nx * a.ny;
    if (count == 0) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, blocks = (int)gridDim.x;
    // the nine pulled populations of node n
    auto pull = [&](int n, float (&f)[9]) {
        const int y = (int)((unsigned)n / (unsigned)a.nx), x = n - y * a.nx;
        const int ym = pull_row(y - 1, a), yp = pull_row(y + 1, a);
        const int xl = x == 0 ? a.nx - 1 : x - 1, xr = x + 1 == a.nx ? 0 : x + 1;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int sy = vb(i) == 1 ? ym : (vb(i) == -1 ? yp : y);
            const int sx = va(i) == 1 ? xl : (va(i) == -1 ? xr : x);
            f[i] = ld_field(src + (long long)i * a.plane + (long long)sy * a.nx + sx);
        }
    };
    // place in the list of entry q of warp w's pieces
    auto place = [&](int w, int q) {
        return (((long long)(q >> 5) * kGuardWarps + w) * blocks + blockIdx.x) * 32 + (q & 31);
    };
    const bool direct = !gp.settle || count <= blocks * kGuardDirect;
    int m;
    if (direct) {
        m = (count - (int)blockIdx.x + blocks - 1) / blocks;
    } else {
        // the warp's entries: whole pieces but for the list's last one
        const int pieces = (count - 1) / 32 + 1, first = warp * blocks + (int)blockIdx.x;
        const int own = first < pieces ? (pieces - 1 - first) / (kGuardWarps * blocks) + 1 : 0;
        int mine = own * 32;
        if (own > 0 && place(warp, mine - 1) >= count) mine = mine - 32 + (count & 31);
        int kept = 0, k0 = 0;
        for (; k0 < mine && 4 * kept <= 3 * k0; k0 += 32) {
            bool open = k0 + lane < mine;
            int n = 0;
            if (open) {
                n = ld_count(a.fix_list + place(warp, k0 + lane));
                float f[9], out[9];
                pull(n, f);
                open = !collide_settled<VAR>(f, gp, out);
                if (!open) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) dst[(long long)i * a.plane + n] = out[i];
                }
            }
            // every lane has read its entry before entries it may overwrite
            const unsigned vote = __ballot_sync(0xffffffffu, open);
            if (open) a.fix_list[place(warp, kept + __popc(vote & ((1u << lane) - 1u)))] = n;
            kept += __popc(vote);
        }
        if (lane == 0) {
            left[warp] = kept + (k0 < mine ? mine - k0 : 0);
            kept_of[warp] = kept;
            from_of[warp] = k0;
        }
        __syncthreads();  // orders the block's list entries as well
        m = 0;
#pragma unroll
        for (int w = 0; w < kGuardWarps; ++w) m += left[w];
    }
    for (int k = threadIdx.x; k < m; k += kGuardBlock) {
        long long t = (long long)k * blocks + blockIdx.x;
        if (!direct) {
            int w = 0, q = k;
            while (q >= left[w]) q -= left[w++];
            t = place(w, q < kept_of[w] ? q : q - kept_of[w] + from_of[w]);
        }
        const int n = ld_count(a.fix_list + t);
        float f[9];
        pull(n, f);
        double g[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = (double)f[i];
        CollideParams<double> q = a.pd;
        q.guard = 0.0;
        double rho;
        bool hit;
        collide_node<VAR>(g, q, rho, hit);
#pragma unroll
        for (int i = 0; i < 9; ++i) dst[(long long)i * a.plane + n] = CodecF32::from_f64(g[i], i, a.cs);
    }
}

}  // namespace kbc
