// pair_node.cuh -- the per-node part of the step (moments, force, collision)
// for one or two x-neighbouring nodes at a time (included by lbm_kernels.cuh
// inside namespace ctulbm).
//
// N says how many: Pair32 or One64.  A value of the nodes is one N::V (float2 or
// double).  In FP32 every operation on whole pairs is one
// packed FP32x2 instruction (sm_100+) and every shared-memory access of a pair one
// 8-byte access, so a pair costs little more issue slots than a node does.
struct Pair32 {
  using T = float;
  using V = float2;
  static constexpr int W = 2;
  static __device__ __forceinline__ V dup(T v) { return make_float2(v, v); }
  static __device__ __forceinline__ V make(T a, T b) { return make_float2(a, b); }
  static __device__ __forceinline__ V recip(V v) { return make_float2(rcp(v.x), rcp(v.y)); }
};
struct One64 {
  using T = double;
  using V = double;
  static constexpr int W = 1;
  static __device__ __forceinline__ V dup(T v) { return v; }
  static __device__ __forceinline__ V recip(V v) { return rcp(v); }
};

// The constants of the collision phase.
template <typename N>
struct NodeConst {
  using T = typename N::T;
  using V = typename N::V;
  V gw1, gw2, gw3, gw4, kw[6];
  V om, ps, p00, p10, pg, p20, p30;
  V lo, hi, nlo, nhi, lo2, hi2;
  V w[3];
  __device__ explicit NodeConst(const StepArgs<typename N::T>& P)
      : gw1(N::dup(P.gw1)), gw2(N::dup(P.gw2)), gw3(N::dup(-P.gw3)), gw4(N::dup(-P.gw4)), om(N::dup(P.omega)),
        ps(N::dup(P.ps)), p00(N::dup(P.p00)), p10(N::dup(P.p10)), pg(N::dup(P.pg)), p20(N::dup(P.p20)),
        p30(N::dup(P.p30)), lo(N::dup(P.xlo)), hi(N::dup(P.xhi)), nlo(N::dup(-P.xlo)), nhi(N::dup(-P.xhi)),
        lo2(N::dup(P.lo2)), hi2(N::dup(P.hi2)) {
#pragma unroll
    for (int i = 0; i < 6; ++i) kw[i] = N::dup(P.kw[i]);
    for (int i = 0; i < 3; ++i) w[i] = N::dup(P.w[i]);
  }
};

// Rows of the moment rings around a pair: columns (c-2, c-1), (c, c+1), (c+2, c+3).
template <typename V>
struct Row6 {
  V l, m, r;
};
template <typename V, typename T>
__device__ __forceinline__ Row6<V> row6(const T* p) {
  return {*reinterpret_cast<const V*>(p - 2), *reinterpret_cast<const V*>(p),
          *reinterpret_cast<const V*>(p + 2)};
}
template <typename V>
__device__ __forceinline__ Row6<V> sub_rows(const Row6<V>& a, const Row6<V>& b) {
  return {sub2(a.l, b.l), sub2(a.m, b.m), sub2(a.r, b.r)};
}

// dt g / ds at two nodes (Eq. eder) from the moment rings; ph[b + 2], dq[b + 2]
// point at the pair's column in the ring row of lattice row + b, b = -2 .. 2.
//  * grad(p^i - p^w): the fourth-order 5x5 gradient (4 D_h - D_2h)/3 of the
//    isotropic 3x3 gradient D_h at spacings ds and 2 ds;
//  * kappa grad(lap rho*): D_h of the isotropic 9-point Laplacian, the two
//    composed into one 5x5 stencil on rho* - rho_ref (the Laplacian of a
//    constant vanishes).
// Every sum is of differences across the node (the density's large constant part
// cancels before anything is added), from the nearest to the farthest.
template <typename N>
__device__ __forceinline__ void pair_force(const NodeConst<N>& C, const typename N::T* const (&ph)[5],
                                           const typename N::T* const (&dq)[5], typename N::V ir,
                                           typename N::V& gx,
                                           typename N::V& gy,
                                           typename N::V& drho) {
  using T = typename N::T;
  using V = typename N::V;
  V px, py, lx, ly;
  if constexpr (N::W == 2) {
  // rows c - 2 .. c + 2: differences one and two columns apart, and between rows
  const auto d1x = [](const Row6<V>& r) { return N::make(r.m.y - r.l.y, r.r.x - r.m.x); };
  const auto d2x = [](const Row6<V>& r) { return sub2(r.r, r.l); };
  const auto sum1 = [](const Row6<V>& d) { return N::make(d.m.y + d.l.y, d.r.x + d.m.x); };
  const auto sum2 = [](const Row6<V>& d) { return add2(d.r, d.l); };
  {
    const Row6<V> t0 = row6<V>(ph[2]), up = row6<V>(ph[3]), dn = row6<V>(ph[1]);
    const Row6<V> up2 = row6<V>(ph[4]), dn2 = row6<V>(ph[0]);
    const V w1 = C.gw1, w2 = C.gw2, w3 = C.gw3, w4 = C.gw4;  // (w3 and w4 negated)
    px = fma2(w1, d1x(t0), fma2(w2, add2(d1x(up), d1x(dn)),
              fma2(w3, d2x(t0), mul2(w4, add2(d2x(up2), d2x(dn2))))));
    const Row6<V> d1 = sub_rows(up, dn), d2 = sub_rows(up2, dn2);
    py = fma2(w1, d1.m, fma2(w2, sum1(d1), fma2(w3, d2.m, mul2(w4, sum2(d2)))));
  }
  {
    const Row6<V> t0 = row6<V>(dq[2]), up = row6<V>(dq[3]), dn = row6<V>(dq[1]);
    drho = t0.m;
    const Row6<V> up2 = row6<V>(dq[4]), dn2 = row6<V>(dq[0]);
    const V k0 = C.kw[0], k1 = C.kw[1], k2 = C.kw[2], k3 = C.kw[3], k4 = C.kw[4], k5 = C.kw[5];
    lx = fma2(k0, d1x(t0), fma2(k1, add2(d1x(up), d1x(dn)), fma2(k2, add2(d1x(up2), d1x(dn2)),
         fma2(k3, d2x(t0), fma2(k4, add2(d2x(up), d2x(dn)), mul2(k5, add2(d2x(up2), d2x(dn2))))))));
    const Row6<V> d1 = sub_rows(up, dn), d2 = sub_rows(up2, dn2);
    ly = fma2(k0, d1.m, fma2(k1, sum1(d1), fma2(k2, sum2(d1),
         fma2(k3, d2.m, fma2(k4, sum1(d2), mul2(k5, sum2(d2)))))));
  }
  } else {
    // one node: columns c - 2 .. c + 2 of five rows
    const auto diff = [](T a, T b) { return a - b; };
    {
      const T* const(&p)[5] = ph;
      const T x1 = diff(p[2][1], p[2][-1]), x2 = diff(p[2][2], p[2][-2]);
      const T xd1 = diff(p[3][1] + p[1][1], p[3][-1] + p[1][-1]);
      const T xd2 = diff(p[4][2] + p[0][2], p[4][-2] + p[0][-2]);
      px = fma(C.gw1, x1, C.gw2 * xd1) + fma(C.gw3, x2, C.gw4 * xd2);
      const T y1 = diff(p[3][0], p[1][0]), y2 = diff(p[4][0], p[0][0]);
      const T yd1 = diff(p[3][1], p[1][1]) + diff(p[3][-1], p[1][-1]);
      const T yd2 = diff(p[4][2], p[0][2]) + diff(p[4][-2], p[0][-2]);
      py = fma(C.gw1, y1, C.gw2 * yd1) + fma(C.gw3, y2, C.gw4 * yd2);
    }
    {
      const T* const(&p)[5] = dq;
      drho = p[2][0];
      const auto dx = [&](int a, int b) { return (p[2 + b][a] + p[2 - b][a]) - (p[2 + b][-a] + p[2 - b][-a]); };
      const auto dy = [&](int a, int b) { return (p[2 + b][a] - p[2 - b][a]) + (p[2 + b][-a] - p[2 - b][-a]); };
      lx = fma(C.kw[0], diff(p[2][1], p[2][-1]), fma(C.kw[1], dx(1, 1), C.kw[2] * dx(1, 2))) +
           fma(C.kw[3], diff(p[2][2], p[2][-2]), fma(C.kw[4], dx(2, 1), C.kw[5] * dx(2, 2)));
      ly = fma(C.kw[0], diff(p[3][0], p[1][0]), fma(C.kw[1], dy(1, 1), C.kw[2] * dy(2, 1))) +
           fma(C.kw[3], diff(p[4][0], p[0][0]), fma(C.kw[4], dy(1, 2), C.kw[5] * dy(2, 2)));
    }
  }
  gx = fma2(ir, px, lx);
  gy = fma2(ir, py, ly);
}

// Sums over the four sign patterns of each velocity group: d = sum f, sx and sy
// = sums with the signs of xi_x and xi_y, t = with their product.
template <typename V>
struct GroupSums {
  V d[4], sx[4], sy[4], t[4];
};
template <typename V, bool T_TOO, typename Load>
__device__ __forceinline__ GroupSums<V> group_sums(Load f) {
  GroupSums<V> g;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const V f0 = f(4 * m), f1 = f(4 * m + 1), f2 = f(4 * m + 2), f3 = f(4 * m + 3);
    const V p = add2(f0, f2), q = add2(f1, f3), a = sub2(f0, f2), b = sub2(f1, f3);
    g.d[m] = add2(p, q);
    g.sx[m] = sub2(a, b);
    g.sy[m] = add2(a, b);
    if constexpr (T_TOO) g.t[m] = sub2(p, q);
  }
  return g;
}

// rho* - rho_ref, u* and p^i - p^w = rho T - [rho T/(1 - b rho) - a rho^2]
// (Eqs. eder, evdw) of two nodes; f(k) loads velocity k of the pair.
template <typename N, typename Load>
__device__ __forceinline__ void pair_moments(const StepArgs<typename N::T>& P, Load f,
                                             typename N::V& dr,
                                             typename N::V& ux,
                                             typename N::V& uy,
                                             typename N::V& phi) {
  using T = typename N::T;
  using V = typename N::V;
  const GroupSums<V> g = group_sums<V, false>(f);
  dr = add2(add2(g.d[0], g.d[1]), add2(g.d[2], g.d[3]));
  const V rho = add2(N::dup(P.rho_ref), dr);
  const V ir = N::recip(rho);
  const V lo = N::dup(P.xlo), hi = N::dup(P.xhi);
  ux = mul2(fma2(lo, add2(g.sx[0], g.sx[2]), mul2(hi, add2(g.sx[1], g.sx[3]))), ir);
  uy = mul2(fma2(lo, add2(g.sy[0], g.sy[1]), mul2(hi, add2(g.sy[2], g.sy[3]))), ir);
  const V rT = mul2(rho, N::dup(P.Tt));
  const V den = fma2(N::dup(P.b), rho, N::dup(T(-1)));  // -(1 - b rho)
  const V q = N::recip(den);
  phi = fma2(mul2(N::dup(P.a), rho), rho, fma2(rT, q, rT));
}

// u* alone (rho* known).
template <typename N, typename Load>
__device__ __forceinline__ void pair_velocity(const NodeConst<N>& C, Load f,
                                              typename N::V ir,
                                              typename N::V& ux,
                                              typename N::V& uy) {
  using T = typename N::T;
  using V = typename N::V;
  V sx[4], sy[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const V a = sub2(f(4 * m), f(4 * m + 2)), b = sub2(f(4 * m + 1), f(4 * m + 3));
    sx[m] = sub2(a, b);
    sy[m] = add2(a, b);
  }
  ux = mul2(fma2(C.lo, add2(sx[0], sx[2]), mul2(C.hi, add2(sx[1], sx[3]))), ir);
  uy = mul2(fma2(C.lo, add2(sy[0], sy[1]), mul2(C.hi, add2(sy[2], sy[3]))), ir);
}

// The collision as a polynomial in the velocity components.  With x = xi_x,
// y = xi_y, (u, v) = u*, (g, h) = dt g, w = dt/tau, s = (T - 1)/2:
//   [w f^eq + dt F_k - w w_k rho_ref] / (w_k rho)
//     = sum_{m+n<=3} c_mn x^m y^n
// (Eqs. herfeq, herforce: xi.u = x u + y v and xi.g = x g + y h expanded), and
// f^{n+1} = (1 - w) f* + w_k rho sum c_mn x^m y^n.  The velocities are the
// products of x, y in {+-lo, +-hi}, so the polynomial is evaluated by its even
// and odd parts in y, then in x: 50 operations for the 16 values (the form in
// xi.u and xi.g of each velocity takes 112).
template <typename V>
struct Poly {
  V c00, c10, c01, c20, c11, c02, c30, c21, c12, c03;
};

template <typename N>
__device__ __forceinline__ Poly<typename N::V> collision_poly(
    const NodeConst<N>& C, typename N::V drho, typename N::V ir,
    typename N::V u, typename N::V v, typename N::V g,
    typename N::V h) {
  using T = typename N::T;
  using V = typename N::V;
  const V om = C.om, s = C.ps;
  const V a = fma2(om, u, g), b = fma2(om, v, h);  // w u + dt g
  const V hu = mul2(mul2(N::dup(T(0.5)), u), u), hv = mul2(mul2(N::dup(T(0.5)), v), v), uv = mul2(u, v);
  const V k = add2(hu, hv);                 // u^2 / 2
  const V gu = fma2(g, u, mul2(h, v));      // dt g.u
  const V su = add2(s, hu), sv = add2(s, hv);
  Poly<V> p;
  p.c00 = sub2(fma2(om, sub2(mul2(drho, ir), k), C.p00), gu);
  const V K = sub2(sub2(C.p10, mul2(om, k)), gu), G = sub2(C.pg, k);
  p.c10 = fma2(K, u, mul2(G, g));
  p.c01 = fma2(K, v, mul2(G, h));
  p.c20 = fma2(om, hu, fma2(u, g, C.p20));
  p.c02 = fma2(om, hv, fma2(v, h, C.p20));
  p.c11 = fma2(v, a, mul2(u, h));
  p.c30 = fma2(C.p30, mul2(hu, u), mul2(a, su));
  p.c03 = fma2(C.p30, mul2(hv, v), mul2(b, sv));
  p.c21 = fma2(b, su, mul2(g, uv));
  p.c12 = fma2(a, sv, mul2(h, uv));
  return p;
}

// Calls put(k, value) with the polynomial's value at velocity k, k = 0 .. 15.
template <typename N, typename V, typename Put>
__device__ __forceinline__ void poly_each(const NodeConst<N>& C, const Poly<V>& p, Put put) {
#pragma unroll
  for (int iy = 0; iy < 2; ++iy) {
    const V y = iy ? C.hi : C.lo, ny = iy ? C.nhi : C.nlo, y2 = iy ? C.hi2 : C.lo2;
    const V e0 = fma2(p.c02, y2, p.c00), o0 = fma2(p.c03, y2, p.c01), e1 = fma2(p.c12, y2, p.c10);
#pragma unroll
    for (int sy = 0; sy < 2; ++sy) {
      const V yy = sy ? ny : y;
      const V a0 = fma2(yy, o0, e0), a1 = fma2(yy, p.c11, e1), a2 = fma2(yy, p.c21, p.c20);
#pragma unroll
      for (int ix = 0; ix < 2; ++ix) {
        const V x = ix ? C.hi : C.lo, nx = ix ? C.nhi : C.nlo, x2 = ix ? C.hi2 : C.lo2;
        const V e = fma2(a2, x2, a0), o = fma2(p.c30, x2, a1);
        const int k = 4 * (2 * iy + ix);  // signs in a group: (+,+), (-,+), (-,-), (+,-)
        put(k + (sy ? 3 : 0), fma2(x, o, e));
        put(k + (sy ? 2 : 1), fma2(nx, o, e));
      }
    }
  }
}

// Eq. (ereg) inside the collision: f* is replaced by f^eq + w [H2:A2/2 + H3:A3/6],
// A_n = sum f^neq xi^n, which is a polynomial in (x, y) as well; it joins the
// collision's with the factor 1 - w, and f^{n+1} = w_k * (the sum) needs f*
// only through its second and third moments.  p comes in as collision_poly's
// and leaves as the polynomial of f^{n+1} / w_k (s1 = 1 - w, rw = rho, see pair_collide).
template <typename N, typename Load>
__device__ __forceinline__ void regularised_poly(const StepArgs<typename N::T>& P, Load f,
                                                 Poly<typename N::V>& p,
                                                 typename N::V drho,
                                                 typename N::V rho,
                                                 typename N::V u,
                                                 typename N::V v,
                                                 typename N::V s1,
                                                 typename N::V rw) {
  using T = typename N::T;
  using V = typename N::V;
  const GroupSums<V> q = group_sums<V, true>(f);
  const T lo = P.xlo, hi = P.xhi, l2 = P.lo2, h2 = P.hi2;
  auto comb = [&](T a, V x, T b, V y) { return fma2(N::dup(a), x, mul2(N::dup(b), y)); };
  const V mxx = comb(l2, add2(q.d[0], q.d[2]), h2, add2(q.d[1], q.d[3]));
  const V myy = comb(l2, add2(q.d[0], q.d[1]), h2, add2(q.d[2], q.d[3]));
  const V mxy = fma2(N::dup(lo * hi), add2(q.t[1], q.t[2]), comb(l2, q.t[0], h2, q.t[3]));
  const V mxxx = comb(lo * l2, add2(q.sx[0], q.sx[2]), hi * h2, add2(q.sx[1], q.sx[3]));
  const V myyy = comb(lo * l2, add2(q.sy[0], q.sy[1]), hi * h2, add2(q.sy[2], q.sy[3]));
  const V mxxy = add2(comb(lo * l2, q.sy[0], hi * h2, q.sy[3]), comb(lo * h2, q.sy[1], hi * l2, q.sy[2]));
  const V mxyy = add2(comb(lo * l2, q.sx[0], hi * h2, q.sx[3]), comb(hi * l2, q.sx[1], lo * h2, q.sx[2]));
  const V Tt = N::dup(P.Tt), ref = N::dup(P.rho_ref), half = N::dup(T(0.5)), sixth = N::dup(T(1) / T(6));
  const V uu = mul2(u, u), vv = mul2(v, v), uv = mul2(u, v);
  const V Axx = sub2(add2(mxx, ref), mul2(rho, add2(uu, Tt)));
  const V Ayy = sub2(add2(myy, ref), mul2(rho, add2(vv, Tt)));
  const V Axy = sub2(mxy, mul2(rho, uv));
  const V T3 = N::dup(T(3) * P.Tt);
  const V ru = mul2(rho, u), rv = mul2(rho, v);
  const V Axxx = sub2(mxxx, mul2(ru, add2(uu, T3))), Ayyy = sub2(myyy, mul2(rv, add2(vv, T3)));
  const V Axxy = sub2(mxxy, mul2(rv, add2(uu, Tt))), Axyy = sub2(mxyy, mul2(ru, add2(vv, Tt)));
  // f^eq / w - rho_ref = drho + rho (P - 1), P - 1 in powers of x, y
  const V s = N::dup(P.ps), hu = mul2(half, uu), hv = mul2(half, vv);
  const V k = add2(hu, hv), su = add2(hu, s), sv = add2(hv, s);
  const V q10 = sub2(N::dup(T(1) - T(4) * P.ps), k);
  const V third = N::dup(T(1) / T(3));
  Poly<V> r;
  r.c00 = sub2(sub2(drho, mul2(rho, add2(k, N::dup(T(2) * P.ps)))), mul2(half, add2(Axx, Ayy)));
  r.c10 = sub2(mul2(ru, q10), mul2(half, add2(Axxx, Axyy)));
  r.c01 = sub2(mul2(rv, q10), mul2(half, add2(Ayyy, Axxy)));
  r.c20 = fma2(rho, su, mul2(half, Axx));
  r.c02 = fma2(rho, sv, mul2(half, Ayy));
  r.c11 = fma2(rho, uv, Axy);
  r.c30 = fma2(ru, fma2(third, hu, s), mul2(sixth, Axxx));
  r.c03 = fma2(rv, fma2(third, hv, s), mul2(sixth, Ayyy));
  r.c21 = fma2(rv, su, mul2(half, Axxy));
  r.c12 = fma2(ru, sv, mul2(half, Axyy));
  auto join = [&](V& c, V d) { c = fma2(s1, d, mul2(rw, c)); };
  join(p.c00, r.c00);
  join(p.c10, r.c10);
  join(p.c01, r.c01);
  join(p.c20, r.c20);
  join(p.c11, r.c11);
  join(p.c02, r.c02);
  join(p.c30, r.c30);
  join(p.c21, r.c21);
  join(p.c12, r.c12);
  join(p.c03, r.c03);
}

// The plain collision in FP32, by velocity groups: with cu = xi.u, D = dt xi.g,
// w = dt/tau, A = (T - 1)(xi^2 - 2)/2, B = (T - 1)(xi^2 - 4)/2, e = 1 - u^2/2,
//   [w f^eq + dt F_k - w w_k rho_ref] / (w_k rho) = E + O,
//   E = w/2 cu^2 + D cu + w (rho - rho_ref)/rho + w (e - 1) - dt g.u + w A,
//   O = cu [w/6 cu^2 + w e - dt g.u + w B] + D [cu^2/2 + e - T + 1 + A],
// and the opposite velocity is E - O.  Each operation and its order is part of the
// result: an FP32 step returns the same bits in every kernel, whatever the launch,
// and FP16 storage would turn another order into flipped roundings of f.  As the
// polynomial below it is a quarter fewer instructions for the pair (6144^2 1076
// us per step against 1107, 4096^2 FP16 504 against 530), but the density at a
// vapour node then drifts from the FP64 step's by 1.4e-6 of its value in 100
// steps where this form gives 6e-8 (sheared bubble, 1024 x 512).
template <typename Load, typename Put>
__device__ __forceinline__ void group_collide(const StepArgs<float>& P, const NodeConst<Pair32>& C, Load f,
                                              Put put, float2 drho, float2 rho, float2 ir, float2 u,
                                              float2 v, float2 g, float2 h) {
  const float2 half = dup2(0.5f), one = dup2(1.0f), s1 = dup2(P.one_m_omega);
  const float2 e = fma2(dup2(-0.5f), fma2(u, u, mul2(v, v)), one);
  const float2 gu = fma2(g, u, mul2(h, v));
  const float2 p0 = sub2(fma2(C.om, sub2(e, one), mul2(mul2(C.om, drho), ir)), gu);
  const float2 p1 = add2(sub2(e, dup2(P.Tt)), one);
  const float2 p2 = fma2(C.om, e, make_float2(-gu.x, -gu.y));
#pragma unroll
  for (int iy = 0; iy < 2; ++iy) {
    const float2 Y = iy ? C.hi : C.lo;
#pragma unroll
    for (int ix = 0; ix < 2; ++ix) {
      const float2 X = ix ? C.hi : C.lo, xu = mul2(X, u), xg = mul2(X, g);
      const float2 nxu = make_float2(-xu.x, -xu.y), nxg = make_float2(-xg.x, -xg.y);
      const ClassConst& cl = P.cls[ix + iy];
      const float2 P0 = add2(p0, dup2(cl.omA)), P1 = add2(p1, dup2(cl.A)), K = add2(p2, dup2(cl.omB));
      const float2 sw = mul2(C.w[ix + iy], rho), nsw = mul2(make_float2(-C.w[ix + iy].x, -C.w[ix + iy].y), rho);
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const int k = 4 * (2 * iy + ix) + m;  // signs in a group: (+,+), (-,+), (-,-), (+,-)
        const float2 cu = fma2(Y, v, m ? nxu : xu), D = fma2(Y, h, m ? nxg : xg);
        const float2 c2 = mul2(cu, cu);
        const float2 E = fma2(c2, dup2(P.om2), fma2(cu, D, P0));
        const float2 O = fma2(cu, fma2(c2, dup2(P.om6), K), mul2(D, fma2(c2, half, P1)));
        const float2 Q = mul2(sw, E);
        put(k, fma2(s1, f(k), fma2(sw, O, Q)));
        put(k + 2, fma2(s1, f(k + 2), fma2(nsw, O, Q)));
      }
    }
  }
}

// Collision of two nodes: f(k) loads f*_k, put(k, value) receives f^{n+1}_k.
// The density reservoir (Sec. III A) multiplies the result by s: the stored
// deviation becomes s f' + w rho_ref (s - 1), which is the same expression with
// the factors s1 = s (1 - w) and rw = s rho and a constant term: cr = rho_ref
// (s - 1) / rw (rw = rho_ext to rounding), or rho_ref (s - 1) itself for the
// regularised collision.
template <typename N, bool REGU, typename Load, typename Put>
__device__ __forceinline__ void pair_collide(const StepArgs<typename N::T>& P, const NodeConst<N>& C, Load f,
                                             Put put,
                                             typename N::V drho,
                                             typename N::V rho,
                                             typename N::V ir,
                                             typename N::V u,
                                             typename N::V v,
                                             typename N::V g,
                                             typename N::V h,
                                             typename N::V s1,
                                             typename N::V rw,
                                             typename N::V cr) {
  using T = typename N::T;
  using V = typename N::V;
  Poly<V> p = collision_poly<N>(C, drho, ir, u, v, g, h);
  if constexpr (REGU) {
    regularised_poly<N>(P, f, p, drho, rho, u, v, s1, rw);
    p.c00 = add2(p.c00, cr);
    poly_each(C, p, [&](int k, V q) {
      const int grp = k >> 2;
      put(k, mul2(C.w[grp == 0 ? 0 : (grp == 3 ? 2 : 1)], q));
    });
  } else {
    p.c00 = add2(p.c00, cr);
    const V sw[3] = {mul2(C.w[0], rw), mul2(C.w[1], rw), mul2(C.w[2], rw)};
    poly_each(C, p, [&](int k, V q) {
      const int grp = k >> 2;
      put(k, fma2(s1, f(k), mul2(sw[grp == 0 ? 0 : (grp == 3 ? 2 : 1)], q)));
    });
  }
}
