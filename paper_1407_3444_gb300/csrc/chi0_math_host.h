// chi0_math_host.h -- host builds of chi0_math.cuh alone (the CPU tests): the same integrals in forms no
// kernel runs, for comparison.  The two carvings as branching code on sorted vertices (the recipes of
// chi0_math.cuh must tile the same region), the per-frequency evaluation of a piece with the series length
// from its convergence ratio, and the delta term as cubic B-splines per vertex.
#pragma once

namespace chi0dev {

template <typename T> constexpr float kLog2Tol = sizeof(T) == 8 ? -56.4727f : -25.5754f;  // log2(Num<T>::tol)

// the shared table where it applies, else the per-vertex table
template <typename T> inline T inv_sum_fast(const T x[4], const T f[4]) {
  T r;
  if (inv_sum_shared(x, f, r)) return r;
  return inv_sum_table(x, f);
}

// sum_j f_j (1/V) int_S lambda_j / X, sorted knots x (FP64 or FP32 throughout)
template <typename T> inline T inv_sum(const T x[4], const T f[4]) {
  if (series_ok(x, T(Num<T>::kappa))) return series_sum(x, f);
  return inv_sum_fast(x, f);
}

// FP32 evaluation of queued knots: the long series where it converges, else the table
inline float inv_sum_long(const float x[4], const float f[4]) {
  if (series_ok(x, Num<float>::kappa_long)) return series_sum(x, f);
  return inv_sum_fast(x, f);
}

// mixed precision, all branches in one place
inline float inv_sum_mixed(const float d[4], const float f[4], float tau, int *fp64) {
  if (series_ok(d, Num<float>::kappa)) return series_sum(d, f);
  float x[4];
  if (!mixed_knots(x, d, tau)) return inv_sum_long(x, f);
  ++*fp64;
  double xd[4] = {x[0], x[1], x[2], x[3]}, fd[4] = {f[0], f[1], f[2], f[3]};
  return (float)inv_sum_table(xd, fd);
}

// own-series terms for convergence ratio rho (rho^kk <= tol), at most K
template <typename T> inline int own_terms(int K, T rho) {
  if (!(rho > T(0))) return K > 0 ? 1 : 0;
  const float need = __fdividef(kLog2Tol<T>, __log2f((float)rho));  // rho^need = tol
  const int kk = 2 + (int)need;
  return kk < K ? kk : K;
}

// (1/(c - w)) sum_{k<K} a_k z^k with z = c/(c - w), truncated where rho^k < tol
template <typename T> inline T far_eval(const T *a, int K, T c, T w, T rho) {
  return far_eval_k(a, own_terms(K, rho), c, w);
}

// Normalised cubic B-spline density M(w; t0..t4) (integral 1) by the de Boor-Cox
// recursion for M-splines; sorted knots, half-open support.
template <typename T> inline T mspline5(const T t[5], T w) {
  T M[4];
  for (int i = 0; i < 4; ++i)
    M[i] = (t[i] <= w && w < t[i + 1]) ? T(1) / (t[i + 1] - t[i]) : T(0);
  for (int k = 2; k <= 4; ++k) {
    for (int i = 0; i + k <= 4; ++i) {
      const T den = t[i + k] - t[i];
      M[i] = den > T(0) ? T(k) * ((w - t[i]) * M[i] + (t[i + k] - w) * M[i + 1]) / (T(k - 1) * den)
                        : T(0);
    }
  }
  return M[0];
}

// sum_j f_j (1/V) int_S lambda_j delta(w - D) = (1/4) sum_j f_j M(w; d, d_j), sorted d
template <typename T> inline T delta_sum(const T d[4], const T f[4], T w) {
  if (!(w > d[0] && w < d[3])) return T(0);
  T acc = T(0);
  for (int jj = 0; jj < 4; ++jj) {
    T t5[5];
    for (int l = 0; l < 5; ++l) t5[l] = l <= jj ? d[l] : d[l - 1];
    acc += f[jj] * mspline5(t5, w);
  }
  return T(0.25) * acc;
}

// ------------------------------------------------------------------------------------
// carving (Sec. II, Fig. 1): keep the part of a tetrahedron where the key is negative.
// WHICH = 0: key = a (first carving, occupied states); WHICH = 1: key = -b (second
// carving, empty states at k+q).  Each piece is emitted with its volume relative to the
// cut tetrahedron, from the cut fractions along the edges.
// ------------------------------------------------------------------------------------
// vertex: a = e^m_k - eF, D = e^n_{k+q} - e^m_k (b = a + D), f = |M|^2; D is its own
// linear attribute so it is exactly 0 wherever the corner data make it 0
template <typename T> struct Vt {
  T a, D, f;
};

template <typename T> inline Vt<T> vmix(const Vt<T> &P, const Vt<T> &Q, T t) {
  const T s = T(1) - t;
  return Vt<T>{s * P.a + t * Q.a, s * P.D + t * Q.D, s * P.f + t * Q.f};
}

template <int WHICH, typename T> inline T vkey(const Vt<T> &v) {
  return WHICH == 0 ? v.a : -(v.a + v.D);
}

// point where the key vanishes on edge P (key < 0) - Q (key >= 0); returns the fraction
template <int WHICH, typename T>
inline Vt<T> vcut(const Vt<T> &P, const Vt<T> &Q, T &frac) {
  const T kp = vkey<WHICH>(P), kq = vkey<WHICH>(Q);
  frac = quot(kp, kp - kq);
  Vt<T> R = vmix(P, Q, frac);
  if (WHICH == 0) R.a = T(0);  // on the first cut plane; the second cut is the last one
  return R;
}

template <int WHICH, typename T> inline void vswap(Vt<T> &x, Vt<T> &y) {
  if (vkey<WHICH>(y) < vkey<WHICH>(x)) {
    Vt<T> t = x; x = y; y = t;
  }
}

// Piece idx of one cut (keep key < 0) and the number of pieces (0, 1 or 3); r = volume of
// the piece relative to the input tetrahedron, from the cut fractions along the edges.
// Pieces are built on demand so that only one of them is live at a time.
template <int WHICH, typename T>
inline int cut_piece(const Vt<T> in[4], int idx, Vt<T> P[4], T &r) {
  Vt<T> S[4] = {in[0], in[1], in[2], in[3]};
  vswap<WHICH>(S[0], S[1]);
  vswap<WHICH>(S[2], S[3]);
  vswap<WHICH>(S[0], S[2]);
  vswap<WHICH>(S[1], S[3]);
  vswap<WHICH>(S[1], S[2]);
  const int nneg = (vkey<WHICH>(S[0]) < T(0)) + (vkey<WHICH>(S[1]) < T(0)) +
                   (vkey<WHICH>(S[2]) < T(0)) + (vkey<WHICH>(S[3]) < T(0));
  if (nneg == 0) return 0;
  if (nneg == 4) {
    for (int i = 0; i < 4; ++i) P[i] = S[i];
    r = T(1);
    return 1;
  }
  if (nneg == 1) {  // corner tetrahedron at S0: volume t1 t2 t3
    T t1, t2, t3;
    P[0] = S[0];
    P[1] = vcut<WHICH>(S[0], S[1], t1);
    P[2] = vcut<WHICH>(S[0], S[2], t2);
    P[3] = vcut<WHICH>(S[0], S[3], t3);
    r = t1 * t2 * t3;
    return 1;
  }
  if (nneg == 2) {  // prism (S0, P02, P03) - (S1, P12, P13)
    T u0, v0, u1, v1;
    const Vt<T> P02 = vcut<WHICH>(S[0], S[2], u0), P03 = vcut<WHICH>(S[0], S[3], v0);
    const Vt<T> P12 = vcut<WHICH>(S[1], S[2], u1), P13 = vcut<WHICH>(S[1], S[3], v1);
    if (idx == 0) {
      P[0] = S[0]; P[1] = P02; P[2] = P03; P[3] = S[1];
      r = u0 * v0;
    } else if (idx == 1) {
      P[0] = P02; P[1] = P03; P[2] = S[1]; P[3] = P12;
      r = v0 * (T(1) - u0) * u1;
    } else {
      P[0] = P03; P[1] = S[1]; P[2] = P12; P[3] = P13;
      r = (T(1) - v0) * u1 * v1;
    }
    return 3;
  }
  // nneg == 3: tetrahedron minus the corner at S3: prism (S0,S1,S2) - (P03,P13,P23)
  T s0, s1, s2;
  const Vt<T> P03 = vcut<WHICH>(S[0], S[3], s0), P13 = vcut<WHICH>(S[1], S[3], s1),
              P23 = vcut<WHICH>(S[2], S[3], s2);
  if (idx == 0) {
    P[0] = S[0]; P[1] = S[1]; P[2] = S[2]; P[3] = P03;
    r = s0;
  } else if (idx == 1) {
    P[0] = S[1]; P[1] = S[2]; P[2] = P03; P[3] = P13;
    r = (T(1) - s0) * s1;
  } else {
    P[0] = S[2]; P[1] = P03; P[2] = P13; P[3] = P23;
    r = (T(1) - s0) * (T(1) - s1) * s2;
  }
  return 3;
}

// Both carvings of one (tetrahedron, band pair): emit(vol_ratio, d[4], f[4]) for every
// final tetrahedron (d = b - a >= 0, unsorted).  Rolled loops: one copy of the emitted
// body, one live piece per level.
template <typename T, typename Emit>
inline void carve2(const T a[4], const T b[4], const T f[4], Emit &&emit) {
  const T amax = fmax(fmax(a[0], a[1]), fmax(a[2], a[3]));
  const T bmin = fmin(fmin(b[0], b[1]), fmin(b[2], b[3]));
  if (amax < T(0) && bmin > T(0)) {  // occupied at k and empty at k+q everywhere: no cut
    T d[4] = {b[0] - a[0], b[1] - a[1], b[2] - a[2], b[3] - a[3]};
    T ff[4] = {f[0], f[1], f[2], f[3]};
    emit(T(1), d, ff);
    return;
  }
  Vt<T> V[4];
  for (int i = 0; i < 4; ++i) V[i] = Vt<T>{a[i], b[i] - a[i], f[i]};
  for (int i1 = 0; i1 < 3; ++i1) {
    Vt<T> P[4];
    T r1 = T(0);
    const int n1 = cut_piece<0>(V, i1, P, r1);
    if (i1 >= n1) break;
    if (r1 <= T(0)) continue;
    for (int i2 = 0; i2 < 3; ++i2) {
      Vt<T> Qv[4];
      T r2 = T(0);
      const int n2 = cut_piece<1>(P, i2, Qv, r2);
      if (i2 >= n2) break;
      const T r = r1 * r2;
      if (r <= T(0)) continue;
      T d[4], ff[4];
      for (int i = 0; i < 4; ++i) {
        const T dd = Qv[i].D;
        d[i] = dd > T(0) ? dd : T(0);
        ff[i] = Qv[i].f;
      }
      emit(r, d, ff);
    }
  }
}


// Carving with the D attribute as an offset: every vertex carries e = D - D0 for one
// reference value D0 per band pair (passed as koff = D0 rounded to T), so that knots near a
// frequency w can be formed as (D0 - w) + e without the rounding of D0 itself.  First cut on a, second on b = a + koff + e; the emitted
// pieces carry offsets e (clamped to D >= 0).
template <typename T, typename Emit>
inline void carve2_off(const T a[4], const T e[4], T koff, const T f[4], Emit &&emit) {
  const T amax = fmax(fmax(a[0], a[1]), fmax(a[2], a[3]));
  const T bmin = fmin(fmin(a[0] + koff + e[0], a[1] + koff + e[1]), fmin(a[2] + koff + e[2], a[3] + koff + e[3]));
  if (amax < T(0) && bmin > T(0)) {
    T ee[4] = {e[0], e[1], e[2], e[3]};
    T ff[4] = {f[0], f[1], f[2], f[3]};
    emit(T(1), ee, ff);
    return;
  }
  Vt<T> V[4];
  for (int i = 0; i < 4; ++i) V[i] = Vt<T>{a[i], e[i], f[i]};
  for (int i1 = 0; i1 < 3; ++i1) {
    Vt<T> P[4];
    T r1 = T(0);
    const int n1 = cut_piece<0>(V, i1, P, r1);
    if (i1 >= n1) break;
    if (r1 <= T(0)) continue;
    for (int i = 0; i < 4; ++i) P[i].a += koff;  // second-cut key -(a + e) is now -b
    for (int i2 = 0; i2 < 3; ++i2) {
      Vt<T> Qv[4];
      T r2 = T(0);
      const int n2 = cut_piece<1>(P, i2, Qv, r2);
      if (i2 >= n2) break;
      const T r = r1 * r2;
      if (r <= T(0)) continue;
      T ee[4], ff[4];
      for (int i = 0; i < 4; ++i) {
        ee[i] = Qv[i].D > -koff ? Qv[i].D : -koff;
        ff[i] = Qv[i].f;
      }
      emit(r, ee, ff);
    }
  }
}

}  // namespace chi0dev
