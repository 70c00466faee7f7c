// The synthesis and derivatives of me_device.cuh at two wavelength points at
// once: lambda_point() with every operation on a packed pair of FP32 numbers.
// Each half takes exactly the operations of the scalar code (signs are moved
// where that is exact, because the packed instructions take no negated
// operand), so a point's values are the same bits either way.
#pragma once

#include "me_device.cuh"

namespace vfisv {

// lambda_point() at the offsets x: `out` gets the same calls with pairs.
template <bool DERIV, class Out>
__device__ __forceinline__ void lambda_pair(const Weideman& W, const PixK& P, f2 x, Out& out) {
  const f2 half = f2_dup(-0.5f), two = f2_dup(2.0f);
  const f2 up = f2_fma(x, f2_dup(P.invD), f2_dup(-P.uv));
  const f2 ub = f2_add(up, f2_dup(P.uB)), ur = f2_sub(up, f2_dup(P.uB));
  f2 Hp, Fp, Hb, Fb, Hr, Fr;
  faddeeva_pair(W, up, P.a, Hp, Fp);
  faddeeva_pair(W, ub, P.a, Hb, Fb);
  faddeeva_pair(W, ur, P.a, Hr, Fr);
  const f2 Hsum = f2_add(Hb, Hr), Hdif = f2_sub(Hr, Hb);
  const f2 Fsum = f2_add(Fb, Fr), Fdif = f2_sub(Fr, Fb);
  const f2 hL = f2_fma(half, Hsum, Hp), fL = f2_fma(half, Fsum, Fp);
  const f2 c1 = f2_dup(P.c1), c2 = f2_dup(P.c2), c4 = f2_dup(P.c4);
  const f2 eI = f2_fma(c1, Hp, f2_fma(c2, Hsum, f2_dup(1.0f)));
  const f2 eL = f2_mul(c1, hL), eV = f2_mul(c4, Hdif);
  const f2 rL = f2_mul(c1, fL), rV = f2_mul(c4, Fdif);
  const f2 eI2 = f2_mul(eI, eI);
  const f2 Pi = f2_fma(eL, rL, f2_mul(eV, rV));
  const f2 rr = f2_fma(rL, rL, f2_mul(rV, rV));
  const f2 g = f2_add(f2_sub(eI2, f2_fma(eL, eL, f2_mul(eV, eV))), rr);
  const f2 nPi = f2_neg(Pi);
  const f2 iD = f2_rcp_fast(f2_fma(eI2, g, f2_mul(nPi, Pi)));
  const f2 niD = f2_neg(iD);
  const f2 NI = f2_mul(eI, f2_add(eI2, rr));
  const f2 NQ = f2_fma(eI2, eL, f2_mul(rL, Pi));
  const f2 nu = f2_fma(eL, rV, f2_mul(f2_neg(eV), rL));
  const f2 NU = f2_mul(eI, nu);
  const f2 NV = f2_fma(eI2, eV, f2_mul(rV, Pi));
  const f2 yI = f2_mul(NI, iD), yQ = f2_mul(NQ, niD), yU = f2_mul(NU, niD), yV = f2_mul(NV, niD);
  out.unit(yI, yQ, yU, yV);
  if constexpr (DERIV) {
    const f2 a2 = f2_dup(2.0f * P.a), ks = f2_dup(-kTwoInvSqrtPi);
    const f2 up2 = f2_mul(two, up), ub2 = f2_mul(two, ub), ur2 = f2_mul(two, ur);
    const f2 alp = f2_fma(a2, Hp, f2_fma(up2, Fp, ks));
    const f2 alb = f2_fma(a2, Hb, f2_fma(ub2, Fb, ks));
    const f2 alr = f2_fma(a2, Hr, f2_fma(ur2, Fr, ks));
    const f2 bep = f2_fma(a2, Fp, f2_mul(f2_neg(up2), Hp));
    const f2 beb = f2_fma(a2, Fb, f2_mul(f2_neg(ub2), Hb));
    const f2 ber = f2_fma(a2, Fr, f2_mul(f2_neg(ur2), Hr));
    const f2 e2 = f2_mul(two, eI);
    const f2 dDe = f2_mul(e2, f2_add(eI2, g));
    const f2 ntwo = f2_dup(-2.0f);
    const f2 dDq = f2_mul(ntwo, NQ), dDv = f2_mul(ntwo, NV);
    const f2 dDr = f2_mul(two, f2_fma(eI2, rL, f2_mul(nPi, eL)));
    const f2 dDt = f2_mul(two, f2_fma(eI2, rV, f2_mul(nPi, eV)));
    const f2 gIL = f2_mul(f2_dup(P.g1), hL), gV = f2_mul(f2_dup(P.g2), Hdif);
    const f2 gRL = f2_mul(f2_dup(P.g1), fL), gRV = f2_mul(f2_dup(P.g2), Fdif);
    out.scale(iD);
    const f2 nc3 = f2_dup(-P.c3);
    const f2 eI1 = f2_sub(eI, f2_dup(1.0f));
    auto stokes = [&](int S, f2 pe, f2 pq, f2 pv, f2 pr, f2 pt) {
      const f2 peq = f2_add(pe, pq);
      const f2 SHp = f2_mul(peq, c1);
      const f2 tH = f2_fma(pe, c2, f2_mul(pq, nc3));
      const f2 SHb = f2_fma(f2_neg(pv), c4, tH), SHr = f2_fma(pv, c4, tH);
      const f2 SFp = f2_mul(pr, c1);
      const f2 tF = f2_mul(pr, nc3);
      const f2 SFb = f2_fma(f2_neg(pt), c4, tF), SFr = f2_fma(pt, c4, tF);
      const f2 Gp = f2_fma(SHp, bep, f2_mul(f2_neg(SFp), alp));
      const f2 Gb = f2_fma(SHb, beb, f2_mul(f2_neg(SFb), alb));
      const f2 Gr = f2_fma(SHr, ber, f2_mul(f2_neg(SFr), alr));
      const f2 vB = f2_sub(Gb, Gr);
      const f2 vG = f2_fma(peq, gIL, f2_fma(pv, gV, f2_fma(pr, gRL, f2_mul(pt, gRV))));
      const f2 vE = f2_fma(pe, eI1, f2_fma(pq, eL, f2_fma(pv, eV, f2_fma(pr, rL, f2_mul(pt, rV)))));
      const f2 vD = f2_fma(up, Gp, f2_fma(ub, Gb, f2_mul(ur, Gr)));
      const f2 vA = f2_fma(SHp, alp, f2_fma(SFp, bep, f2_fma(SHb, alb, f2_fma(SFb, beb,
                    f2_fma(SHr, alr, f2_mul(SFr, ber))))));
      const f2 vV = f2_add(f2_add(Gp, Gb), Gr);
      out.rows(S, vB, vG, vE, vD, vA, vV);
    };
    const f2 nyI = f2_neg(yI), nyQ = f2_neg(yQ), nyU = f2_neg(yU), nyV = f2_neg(yV);
    const f2 ne2 = f2_neg(e2), nrL = f2_neg(rL), nrV = f2_neg(rV), neI = f2_neg(eI);
    stokes(0, f2_fma(nyI, dDe, f2_fma(f2_dup(3.0f), eI2, rr)), f2_mul(nyI, dDq),
           f2_mul(nyI, dDv), f2_fma(nyI, dDr, f2_mul(e2, rL)), f2_fma(nyI, dDt, f2_mul(e2, rV)));
    stokes(1, f2_fma(nyQ, dDe, f2_mul(ne2, eL)),
           f2_fma(nyQ, dDq, f2_neg(f2_fma(rL, rL, eI2))), f2_fma(nyQ, dDv, f2_mul(nrL, rV)),
           f2_fma(nyQ, dDr, f2_neg(f2_fma(rL, eL, Pi))), f2_fma(nyQ, dDt, f2_mul(nrL, eV)));
    stokes(2, f2_fma(nyU, dDe, f2_neg(nu)), f2_fma(nyU, dDq, f2_mul(neI, rV)),
           f2_fma(nyU, dDv, f2_mul(eI, rL)), f2_fma(nyU, dDr, f2_mul(eI, eV)),
           f2_fma(nyU, dDt, f2_mul(neI, eL)));
    stokes(3, f2_fma(nyV, dDe, f2_mul(ne2, eV)), f2_fma(nyV, dDq, f2_mul(nrV, rL)),
           f2_fma(nyV, dDv, f2_neg(f2_fma(rV, rV, eI2))), f2_fma(nyV, dDr, f2_mul(nrV, eL)),
           f2_fma(nyV, dDt, f2_neg(f2_fma(rV, eV, Pi))));
  }
}

}  // namespace vfisv
