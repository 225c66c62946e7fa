// vans_pair.cuh -- the D2Q9 update of two adjacent cells at once in packed FP32
// (fma.rn.f32x2), shared by the kernels that hold the state on chip (kinds 8, 9).
// Every operation is written out as a rounded multiply-add, addition or
// multiplication, so that nothing is left to the compiler's contraction: all
// kernels that call collide_pair get the same bits.
#pragma once

#include "vans_device.cuh"

namespace vans {

using f2 = float2;

__device__ __forceinline__ f2 bc(float v) { return make_float2(v, v); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 sub2(f2 a, f2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ f2 neg2(f2 a) { return make_float2(-a.x, -a.y); }

__device__ __forceinline__ float rcp_ftz(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// the hardware estimates with one Newton-Raphson step each, as rcp_nr and
// sqrt_nr (vans_device.cuh); sqrt2 takes x > 0, normal
__device__ __forceinline__ f2 rcp2(f2 x) {
    const f2 r = make_float2(rcp_ftz(x.x), rcp_ftz(x.y));
    return fma2(r, fma2(neg2(x), r, bc(1.f)), r);
}
__device__ __forceinline__ f2 sqrt2(f2 x) {
    const f2 y = make_float2(rsqrt_ftz(x.x), rsqrt_ftz(x.y));
    const f2 s = mul2(x, y);
    return fma2(mul2(y, bc(0.5f)), fma2(neg2(s), s, x), s);
}

// What a cell's update needs of the porosity, formed once per row and launch:
// eps, Hc = cs^2 grad eps / eps + g, the drag coefficients and w_i (eps - eps~_i).
// Thirteen pairs: six 16-byte words and an 8-byte one per lane.
struct Por {
    f2 e0, hx, hy, al, be;
    f2 wd[9];              // wd[0] unused
};

// pair of cells (x, x+1) with the neighbours on either side: values at x-1 .. x+2
struct Row {
    float l;
    f2 c;
    float r;
    __device__ f2 left() const { return make_float2(l, c.x); }
    __device__ f2 right() const { return make_float2(c.y, r); }
};

__device__ __forceinline__ Row with_neighbours(f2 c) {
    Row o;
    o.c = c;
    o.l = __shfl_up_sync(VANS_FULL, c.y, 1);
    o.r = __shfl_down_sync(VANS_FULL, c.x, 1);
    return o;
}

// values one column to the left (s < 0: what a population moving +x pulls) or
// right of each cell of the pair
__device__ __forceinline__ f2 from_left(f2 c) {
    return make_float2(__shfl_up_sync(VANS_FULL, c.y, 1), c.x);
}
__device__ __forceinline__ f2 from_right(f2 c) {
    return make_float2(c.y, __shfl_down_sync(VANS_FULL, c.x, 1));
}

// direction order: 0 (0,0), 1 (1,0), 2 (0,1), 3 (-1,0), 4 (0,-1), 5 (1,1),
// 6 (-1,1), 7 (-1,-1), 8 (1,-1); m, z, p: the porosity rows y-1, y, y+1
__device__ __forceinline__ void porosity_terms(const VDom &d, const Row &m, const Row &z, const Row &p,
                                               bool lo_wall, bool hi_wall, Por &o) {
    const f2 e0 = z.c;
    f2 et[9];
    et[1] = z.right();
    et[3] = z.left();
    et[2] = p.c;
    et[5] = p.right();
    et[6] = p.left();
    et[4] = m.c;
    et[8] = m.right();
    et[7] = m.left();
    if (hi_wall) et[2] = et[5] = et[6] = e0;     // past a wall: eps(x)
    if (lo_wall) et[4] = et[7] = et[8] = e0;
    const f2 d1 = sub2(et[1], et[3]), d2 = sub2(et[2], et[4]);
    const f2 d5 = sub2(et[5], et[7]), d8 = sub2(et[8], et[6]);
    // grad eps = (4 d1 + d5 + d8, 4 d2 + d5 - d8) / 12
    const f2 gx = fma2(d1, bc(4.f), add2(d5, d8)), gy = fma2(d2, bc(4.f), sub2(d5, d8));
    const f2 inv = make_float2(rcp_nr(e0.x), rcp_nr(e0.y));
    const f2 inv36 = mul2(inv, bc(1.f / 36.f));
    o.e0 = e0;
    o.hx = fma2(gx, inv36, bc(d.g[0]));
    o.hy = fma2(gy, inv36, bc(d.g[1]));
    // the drag law (drag of vans_device.cuh) for the pair
    if (d.k_mode == 0) {
        const f2 om = sub2(bc(1.f), e0);
        o.al = mul2(mul2(mul2(om, bc(d.ca)), om), inv);
        o.be = mul2(om, bc(d.cb));
    } else {
        const f2 ee = mul2(e0, e0);
        o.al = mul2(ee, bc(d.ca));
        o.be = mul2(d.k_mode == 1 ? mul2(ee, e0)
                                  : mul2(e0, sqrt2(make_float2(fmaxf(e0.x, 1e-36f), fmaxf(e0.y, 1e-36f)))),
                    bc(d.cb));
    }
    if (d.drag_mode == 0) o.al = bc(0.f);
    if (d.drag_mode != 2) o.be = bc(0.f);
#pragma unroll
    for (int i = 1; i < 9; ++i) o.wd[i] = mul2(sub2(e0, et[i]), bc(Lat<9>::w(i)));
}

// One update of a pair of cells: the final LBE in deviation form (macro and
// collide of vans_device.cuh), with M = 2m, so that u = M / D, and
// t = p grad eps + R g = R Hc.  With q = omega R u + ct V the odd part of
// f^eq + P_i + F_i is 3 e.q and, with g = q - omega R u / 2, the even part
// 9 (e.u)(e.g) - 3 u.g.  The momentum a cell gains is (1 - omega) j + q = j + V
// only if ct + omega/2 = 1: near rest j = -V/2 is large (the pressure term
// p grad eps, which the lattice takes back), so a rounding of 3e-8 in that sum
// is a spurious force; ct is therefore 1 - omega/2, exact in FP32 for omega >= 1
// (tau <= 1) and off by up to 2^-25 below, and both constants enter unscaled (scaled
// by 3 and rounded again, the velocity was 2 to 3 times further from 64 bits at
// tau = 0.55 .. 0.6).  For tau of 1.05 to 8, carrying that rest of ct as well moved the
// velocity no closer to 64 bits, at rest or flowing, and took 2 % longer: there the
// error is that of the single-step kinds.
struct PairMoments {
    f2 dl, R, ux, uy;
};

__device__ __forceinline__ void collide_pair(const VDom &d, const f2 h[9], const Por &P, f2 o[9],
                                             PairMoments *mom = nullptr) {
    const f2 dl = add2(add2(add2(add2(h[1], h[3]), add2(h[2], h[4])),
                            add2(add2(h[5], h[7]), add2(h[6], h[8]))), h[0]);
    const f2 R = add2(P.e0, dl);
    const f2 d1 = sub2(h[1], h[3]), d2 = sub2(h[2], h[4]);
    const f2 d5 = sub2(h[5], h[7]), d8 = sub2(h[8], h[6]);
    const f2 jx = add2(d1, add2(d5, d8)), jy = add2(d2, sub2(d5, d8));
    const f2 tx = mul2(R, P.hx), ty = mul2(R, P.hy);
    const f2 Mx = fma2(bc(2.f), jx, tx), My = fma2(bc(2.f), jy, ty);
    const f2 m2 = fma2(Mx, Mx, mul2(My, My));
    // |M|; the floor keeps the root finite at rest and is far below any effect
    const f2 M = sqrt2(make_float2(fmaxf(m2.x, 1e-36f), fmaxf(m2.y, 1e-36f)));
    const f2 a = fma2(bc(0.5f), P.al, R);
    const f2 s = rcp2(add2(a, sqrt2(fma2(P.be, M, mul2(a, a)))));
    const f2 ux = mul2(Mx, s), uy = mul2(My, s);
    if (mom) *mom = PairMoments{dl, R, ux, uy};
    const f2 kd = neg2(fma2(P.be, mul2(M, s), P.al));
    const f2 Vx = fma2(kd, ux, tx), Vy = fma2(kd, uy, ty);
    const float om = d.omega;
    const f2 ct = bc(1.f - 0.5f * om), om1 = bc(1.f - om);
    const f2 omR = mul2(R, bc(om)), hR = mul2(omR, bc(-0.5f));
    const f2 qx = fma2(omR, ux, mul2(ct, Vx)), qy = fma2(omR, uy, mul2(ct, Vy));
    const f2 gx = fma2(hR, ux, qx), gy = fma2(hR, uy, qy);
    const f2 xx = mul2(ux, gx), yy = mul2(uy, gy), xy = fma2(ux, gy, mul2(uy, gx));
    const f2 ug = add2(xx, yy);
    const f2 c = fma2(bc(-3.f), ug, mul2(bc(om), dl));
    o[0] = fma2(om1, h[0], mul2(bc(Lat<9>::w(0)), c));
    auto pair = [&](int i, int j, f2 even, f2 q) {
        const f2 w = bc(Lat<9>::w(i));
        o[i] = fma2(w, fma2(bc(3.f), q, even), fma2(om1, h[i], P.wd[i]));
        o[j] = fma2(w, fma2(bc(-3.f), q, even), fma2(om1, h[j], P.wd[j]));
    };
    pair(1, 3, fma2(bc(9.f), xx, c), qx);
    pair(2, 4, fma2(bc(9.f), yy, c), qy);
    const f2 b = fma2(bc(9.f), ug, c);
    pair(5, 7, fma2(bc(9.f), xy, b), add2(qx, qy));
    pair(8, 6, fma2(bc(-9.f), xy, b), sub2(qx, qy));
}

}  // namespace vans
