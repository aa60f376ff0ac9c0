// Device parts shared by the chain, gradient and state kernels of locally controlled systems
// (kernels_local.cu): the step operator of one qubit, its factorisation, and the row rotations.
//
// A control system is "local" when the drift is diagonal and every control operator is a sum of
// one-qubit operators, H_k = sum_i h_ki (x/y controls of single spins, global x/y fields, z
// controls).  Every table operator of term k (Eq. redoform) is then a tensor product of 2 x 2
// operators u_ki, and so is the product of a step's control factors:
//     E_{K-1} ... E_0 = V_{n-1} (x) ... (x) V_0,   V_i = prod_k u_ki  (2 x 2, in the order of k).
// Applying V_i to a state pairs row r with row r ^ 2^i only: n pairwise rotations instead of K*d
// dense N x N products.  Each V_i is factored into real rotations between phases,
//     V_i = diag(1, x_i) [[c_i, -s_i], [s_i, c_i]] diag(y0_i, y1_i),
// and the phases of all qubits, the drift, a step-opening diagonal and the trailing phases of the
// step before are one diagonal,
//     Delta_n = (tensor_i diag(y0_i(n), y1_i(n))) D P_n (tensor_i diag(1, x_i(n-1))),
// so a step costs 4 operations per entry for Delta_n and 4 per entry and qubit (a 2 x 2 complex
// operator would take 8 per entry and qubit).  Delta_M closes the chain (the last step's x_i).
// Both are kept as their difference from the identity, c - 1 and Delta - 1, and applied as
// v + (c - 1) v - s w and v + (Delta - 1) v (as many operations): a step is near the identity, and a
// c or Delta rounded beside 1 would change the norm by up to 3e-8 in FP32, at every step alike when
// the drive is steady (N = 1024, one global control: 7e-6 of <Z> after 200 steps, now 1e-6).
#pragma once
#include "redo_internal.cuh"

namespace redo {

constexpr int kLocFirst = 0x40000000;   // loc_k flag: the first pair that reads term k (counts bad levels)

template <typename R> __device__ __forceinline__ cplx<R> cmul(cplx<R> a, cplx<R> b) {
  return cmake<R>(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}
template <typename R> __device__ __forceinline__ cplx<R> cmul_conj(cplx<R> a, cplx<R> b) {   // a conj(b)
  return cmake<R>(fma(a.x, b.x, a.y * b.y), fma(a.y, b.x, -(a.x * b.y)));
}

// Powers of two that keep FP32 sums of products in range whatever the length of the vectors and
// targets that they come from: the exponent of a value (clamped so that a few of them add up within
// FP64), 2^e, and the exponent of the larger part.  Scaling by them rounds nothing.
__device__ __forceinline__ int exp_of(double x) {
  const int e = (int)((__double_as_longlong(x) >> 52) & 0x7ff) - 1023;
  return e < -200 ? -200 : (e > 200 ? 200 : e);
}
__device__ __forceinline__ int exp_of(double2 z) { return max(exp_of(z.x), exp_of(z.y)); }
__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }
// x 2^-e by its exponent (an FP64 product is 64 cycles of a warp): 0 below the normal range, infinite above
__device__ __forceinline__ double down2(double x, int e) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  if (ex == 0x7ff || e == 0) return x;
  if (ex - e >= 0x7ff && ex > 0) return __hiloint2double((hi & (int)0x80000000) | 0x7ff00000, 0);
  return ex == 0 || ex - e <= 0 ? 0.0 : __hiloint2double(hi - (int)((unsigned)e << 20), __double2loint(x));
}

// One-qubit tables of a local system: pairs (term k, qubit i) in order of qubit, then term.
template <typename R>
struct LocTab {
  const int32_t* ptr;        // [n + 1] pairs of qubit i
  const int32_t* k;          // [pairs] term | operator set << 8 (| kLocFirst)
  const cplx<R>* u;          // [sets][d][base][4] digit operators, row-major 2 x 2
  int d, base, K;
  int64_t levels;
  int64_t* status;
  int bad_weight;            // dense factors that one level index selects (digits)
};

template <typename R> struct Mat2 { cplx<R> a, b, c, e; };   // [[a, b], [c, e]]

template <typename R> __device__ __forceinline__ Mat2<R> mat2_mul(const Mat2<R>& u, const Mat2<R>& v) {
  Mat2<R> o;
  o.a = cmul<R>(u.a, v.a); cfma<R>(o.a, u.b, v.c);
  o.b = cmul<R>(u.a, v.b); cfma<R>(o.b, u.b, v.e);
  o.c = cmul<R>(u.c, v.a); cfma<R>(o.c, u.e, v.c);
  o.e = cmul<R>(u.c, v.b); cfma<R>(o.e, u.e, v.e);
  return o;
}

template <typename R> __device__ __forceinline__ Mat2<R> loc_load(const LocTab<R>& t, int64_t entry) {
  const cplx<R>* u = t.u + entry * 4;
  Mat2<R> m;
  if constexpr (sizeof(R) == 4) {
    const float4 x = __ldg(reinterpret_cast<const float4*>(u)), y = __ldg(reinterpret_cast<const float4*>(u) + 1);
    m.a = make_float2(x.x, x.y); m.b = make_float2(x.z, x.w);
    m.c = make_float2(y.x, y.y); m.e = make_float2(y.z, y.w);
  } else {
    m.a = __ldg(u); m.b = __ldg(u + 1); m.c = __ldg(u + 2); m.e = __ldg(u + 3);
  }
  return m;
}

// u_ki (kf: its entry of LocTab::k) at level index qv: the product of its digit operators
template <typename R> __device__ __forceinline__ Mat2<R> loc_term(const LocTab<R>& t, int kf, int32_t qv) {
  const int set = (kf & ~kLocFirst) >> 8;
  Mat2<R> m = loc_load(t, (int64_t)set * t.d * t.base + qv % t.base);
  for (int j = 1; j < t.d; ++j) {
    qv /= t.base;
    m = mat2_mul<R>(loc_load(t, ((int64_t)set * t.d + j) * t.base + qv % t.base), m);
  }
  return m;
}

template <typename R>
__device__ __forceinline__ int32_t loc_level(const LocTab<R>& t, const int32_t* qrow, int kf, bool count) {
  int32_t qv = qrow[kf & 0xff];
  if (qv < 0 || qv >= t.levels) {
    if (count && (kf & kLocFirst) && t.status)
      atomicAdd((unsigned long long*)&t.status[REDO_STATUS_BADINDEX], (unsigned long long)t.bad_weight);
    qv = 0;
  }
  return qv;
}

// V_i of one step (qrow: the step's K level indices)
template <typename R>
__device__ __forceinline__ Mat2<R> loc_step(const LocTab<R>& t, const int32_t* qrow, int i, bool count) {
  Mat2<R> v;
  v.a = v.e = cmake<R>(R(1), R(0));
  v.b = v.c = cmake<R>(R(0), R(0));
  const int p0 = t.ptr[i], p1 = t.ptr[i + 1];
  for (int p = p0; p < p1; ++p) {
    const int kf = t.k[p];
    const Mat2<R> u = loc_term<R>(t, kf, loc_level<R>(t, qrow, kf, count));
    v = p == p0 ? u : mat2_mul<R>(u, v);
  }
  return v;
}

// Factorisation of V_i.  The phases are kept so that they add: complex numbers in FP64, and in FP32
// angles in turns of 2^-32 (1.5e-9 rad), whose sums are exact and wrap by themselves.  (FP32 complex
// phases would be rounded to 3e-8 rad each, the same for every qubit under a global control: the
// error of tau over 600 steps was twice that of the dense FP32 chain.)
template <typename R> struct PhaseOf { using T = cplx<R>; };
template <> struct PhaseOf<float> { using T = int32_t; };
template <typename R> using phase_t = typename PhaseOf<R>::T;

constexpr double kTurn64 = 6.283185307179586476925 / 4294967296.0;
constexpr float kTurn = (float)kTurn64, kTurnLo = (float)(kTurn64 - (double)kTurn);   // 2 pi 2^-32
constexpr float kPerTurn = 683565275.576431f;           // 2^32 / (2 pi)

// e^{i t}: the quadrant from the integer's top bits, sine and cosine of the rest (|a| <= pi/4),
// corrected for what its float conversion dropped.  M1: e^{i t} - 1.
template <bool M1> __device__ __forceinline__ float2 phasor(int32_t t) {
  const int32_t k = (int32_t)((uint32_t)t + 0x20000000u) >> 30;
  const int32_t res = (int32_t)((uint32_t)t - ((uint32_t)k << 30));
  const float fh = (float)res;
  const float a = fh * kTurn;
  const float d = fmaf(fh, kTurnLo, fmaf((float)(res - (int32_t)fh), kTurn, fmaf(fh, kTurn, -a)));
  float s, c;
  sincosf(a, &s, &c);
  const float s1 = fmaf(d, c, s), c1 = fmaf(-d, s, c);
  float re = (k & 1) ? -s1 : c1, im = (k & 1) ? c1 : s1;
  if (k & 2) {
    re = -re;
    im = -im;
  }
  if (M1) re = k == 0 ? -s1 * s1 / (1.f + c1) : re - 1.f;
  return make_float2(re, im);
}

// the angle of z in turns: atan2f, then one refinement against the phasor it gives
__device__ __forceinline__ int32_t turns_of(float2 z) {
  const int32_t t = (int32_t)(uint32_t)(long long)rintf(atan2f(z.y, z.x) * kPerTurn);
  const float2 p = phasor<false>(t);
  const float re = fmaf(z.x, p.x, z.y * p.y), im = fmaf(z.y, p.x, -(z.x * p.y));
  return re > 0.f ? (int32_t)((uint32_t)t + (uint32_t)(int32_t)rintf(im / re * kPerTurn)) : t;
}

// FP32 systems of up to four qubits are factored as
//     V_i = diag(x0_i, x1_i) [[c_i, -conj(s_i)], [s_i, c_i]],   s_i complex, y0 = y1 = 1,
// instead: every part is then near the identity when the controls' angles are small, and a step
// rounds once per qubit beside the state's entries (v + t with a small t) where the real rotations
// between O(1) phases round twice and once more for each phase.  It costs 8 operations per entry and
// qubit, not 4; with few rows to average over, the chain's error is 0.6 times as large (N = 4, 790
// steps: 1.4e-6 -> 8e-7 of the gradient), no larger than the dense FP32 products'.  (FP32 propagations
// of one-qubit controls take it at every N: local_chain_form.)  FP64 keeps the real rotations: against
// extended precision (U, 400 steps) they are 3e-15 to 4e-15 off at N = 4, 8 and 16, the dense products 8e-15 to
// 1.8e-14: those apply the same rounded exp(-i dt H0) at every step.
__host__ __device__ constexpr bool loc_near(bool dbl, int N) { return !dbl && N <= 16; }

// c1 = c - 1; s = (s, sy), sy = 0 in the real form; x0 = 1 in the real form
template <typename R> struct Euler { phase_t<R> y0, y1, x0, x; R c1, s, sy; };

// The phases of a vanishing entry are free; x comes from the larger of the two entries that
// determine it, so every entry of V_i is reproduced to rounding.
template <typename R, bool NEAR> __device__ __forceinline__ Euler<R> loc_factor(const Mat2<R>& v) {
  Euler<R> o;
  const R c2 = fma(v.a.x, v.a.x, v.a.y * v.a.y), s2 = fma(v.b.x, v.b.x, v.b.y * v.b.y);
  const R c = sqrt(c2), s = sqrt(s2);
  // (c, s) scaled to c^2 + s^2 = 1 (the residual is exact under fma, so the scaling has no bias), then
  // c - 1 = -s^2 / (1 + c) without cancellation
  const R res = R(0.5) * fma(-s, s, fma(-c, c, R(1)));
  o.s = fma(res, s, s);
  o.sy = R(0);
  o.c1 = -(o.s * o.s) / (R(1) + fma(res, c, c));
  if constexpr (NEAR) {
    o.y0 = o.y1 = 0;
    o.x = c > 0.f ? turns_of(v.e) : 0;
    const float2 q = phasor<false>(o.x);
    const float2 w = cmul_conj<float>(v.c, q);           // s e^{...}: V10 conj(x1)
    o.x0 = c >= s ? turns_of(v.a) : turns_of(cmul<float>(make_float2(-v.b.x, -v.b.y), w));
    const float wn = sqrtf(fmaf(w.x, w.x, w.y * w.y)), f = wn > 0.f ? o.s / wn : 0.f;
    o.s = w.x * f;
    o.sy = w.y * f;
  } else if constexpr (sizeof(R) == 4) {
    // diag(1, e^{iA}) V diag(1, e^{-iA}) has a real entry -s: y1 = e^{iA} cancels in the diagonal
    o.y0 = turns_of(v.a);
    o.y1 = s > 0.f ? turns_of(make_float2(-v.b.x, -v.b.y)) : 0;
    o.x0 = 0;
    o.x = (int32_t)(c >= s ? (uint32_t)turns_of(v.e) - (uint32_t)o.y1 : (uint32_t)turns_of(v.c) - (uint32_t)o.y0);
  } else {
    o.y0 = c > R(0) ? cmake<R>(v.a.x / c, v.a.y / c) : cmake<R>(R(1), R(0));
    o.y1 = s > R(0) ? cmake<R>(-v.b.x / s, -v.b.y / s) : cmake<R>(R(1), R(0));
    o.x0 = cmake<R>(R(1), R(0));
    const cplx<R> w = c >= s ? cmul_conj<R>(v.e, o.y1) : cmul_conj<R>(v.c, o.y0);
    const R wn = sqrt(fma(w.x, w.x, w.y * w.y));
    o.x = wn > R(0) ? cmake<R>(w.x / wn, w.y / wn) : cmake<R>(R(1), R(0));
  }
  return o;
}

// v + d v, and v + conj(d) v.  NEAR: the small part summed first, one rounding beside v.
template <typename R, bool NEAR = false> __device__ __forceinline__ cplx<R> plus_mul(cplx<R> v, cplx<R> d) {
  if constexpr (NEAR) return cmake<R>(v.x + fma(-d.y, v.y, d.x * v.x), v.y + fma(d.y, v.x, d.x * v.y));
  return cmake<R>(fma(-d.y, v.y, fma(d.x, v.x, v.x)), fma(d.y, v.x, fma(d.x, v.y, v.y)));
}
template <typename R, bool NEAR = false> __device__ __forceinline__ cplx<R> plus_mul_conj(cplx<R> v, cplx<R> d) {
  return plus_mul<R, NEAR>(v, cmake<R>(d.x, -d.y));
}
// v + (c1 v + (s + i t) o); t is ignored in the real form
template <typename R, bool NEAR> __device__ __forceinline__ cplx<R> rot_one(cplx<R> v, cplx<R> o, R c1, R s, R t) {
  if constexpr (NEAR)
    return cmake<R>(v.x + fma(-t, o.y, fma(s, o.x, c1 * v.x)), v.y + fma(t, o.x, fma(s, o.y, c1 * v.y)));
  return cmake<R>(fma(s, o.x, fma(c1, v.x, v.x)), fma(s, o.y, fma(c1, v.y, v.y)));
}

// Layout of one column (N rows) over G = N / E lanes, E entries each: lane part l holds rows
// l E + e, so the low qubits pair registers of one lane and the high ones pair lanes.  Lanes of
// the same part are adjacent (C = 32 / G columns a warp), and a diagonal is stored as
// [E/2][G][2] (loc_pos), so a lane reads two of its entries at once and the parts read one line.
template <int N> struct Log2 { static constexpr int v = 1 + Log2<N / 2>::v; };
template <> struct Log2<1> { static constexpr int v = 0; };

__host__ __device__ __forceinline__ int loc_pos(int r, int E, int G) {   // E >= 2
  const int l = r / E, e = r - l * E;
  return ((e >> 1) * G + l) * 2 + (e & 1);
}

template <typename R, int N, int E, bool NR = loc_near(sizeof(R) == 8, N)> struct LocCol {
  static constexpr bool NEAR = NR;
  static constexpr int G = N / E, C = 32 / G, NQ = Log2<N>::v, EB = Log2<E>::v;
  static constexpr int CS = NQ * (NEAR ? 2 : 1);     // (c - 1, s) of every qubit, then (sy, 0)
  static_assert(G * E == N && G <= 32, "column layout");

  // v <- Delta v (or conj(Delta) v), d holding Delta - 1
  template <bool CONJ> static __device__ __forceinline__ void diag(cplx<R> (&v)[E], const cplx<R>* d, int l) {
#pragma unroll
    for (int e = 0; e < E; e += 2) {
      cplx<R> a, b;
      if constexpr (sizeof(R) == 4) {
        const float4 p = __ldg(reinterpret_cast<const float4*>(d) + (e >> 1) * G + l);
        a = make_float2(p.x, p.y);
        b = make_float2(p.z, p.w);
      } else {
        a = __ldg(d + ((e >> 1) * G + l) * 2);
        b = __ldg(d + ((e >> 1) * G + l) * 2 + 1);
      }
      v[e] = CONJ ? plus_mul_conj<R, NEAR>(v[e], a) : plus_mul<R, NEAR>(v[e], a);
      v[e + 1] = CONJ ? plus_mul_conj<R, NEAR>(v[e + 1], b) : plus_mul<R, NEAR>(v[e + 1], b);
    }
  }
  // its entries alone, for a later step
  static __device__ __forceinline__ void load_diag(cplx<R> (&o)[E], const cplx<R>* d, int l) {
#pragma unroll
    for (int e = 0; e < E; e += 2) {
      if constexpr (sizeof(R) == 4) {
        const float4 p = __ldg(reinterpret_cast<const float4*>(d) + (e >> 1) * G + l);
        o[e] = make_float2(p.x, p.y);
        o[e + 1] = make_float2(p.z, p.w);
      } else {
        o[e] = __ldg(d + ((e >> 1) * G + l) * 2);
        o[e + 1] = __ldg(d + ((e >> 1) * G + l) * 2 + 1);
      }
    }
  }
  static __device__ __forceinline__ cplx<R> swap(cplx<R> v, int lane_mask) {
    return cmake<R>(__shfl_xor_sync(0xffffffffu, v.x, lane_mask), __shfl_xor_sync(0xffffffffu, v.y, lane_mask));
  }
  // rotations of every qubit, [[c, -conj(s)], [s, c]] on the pair (bit 0, bit 1)
  static __device__ __forceinline__ void rotate(cplx<R> (&v)[E], const cplx<R> (&cs)[CS], int l) {
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const R c = cs[i].x, s = cs[i].y, t = NEAR ? cs[CS - NQ + i].x : R(0);
      if (i < EB) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if (e & (1 << i)) continue;
          const cplx<R> a = v[e], b = v[e | (1 << i)];
          v[e] = rot_one<R, NEAR>(a, b, c, -s, t);
          v[e | (1 << i)] = rot_one<R, NEAR>(b, a, c, s, t);
        }
      } else {
        const int m = 1 << (i - EB);
        const R sg = (l & m) ? s : -s;
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = rot_one<R, NEAR>(v[e], swap(v[e], m * C), c, sg, t);
      }
    }
  }
  static __device__ __forceinline__ void load_cs(cplx<R> (&cs)[CS], const cplx<R>* p) {
#pragma unroll
    for (int i = 0; i < CS; ++i) cs[i] = __ldg(p + i);
  }
  // The three Bloch sums of every qubit,
  //   X = Im Tr(X_i P R), Y = Im Tr(Y_i P R), Z = Im Tr(Z_i P R)
  // over this lane's entries of a column p of P and the matching row w of R, then the qubit's
  // rotation undone on both (p <- rot^dag p, w <- w rot).  A partial trace over the other qubits
  // does not change when those are rotated, so each qubit is traced just before its own undo.
  static __device__ __forceinline__ void trace_undo(cplx<R> (&p)[E], cplx<R> (&w)[E], const cplx<R> (&cs)[CS],
                                                    int l, R* bl) {
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const R c = cs[i].x, s = cs[i].y, t = NEAR ? cs[CS - NQ + i].x : R(0);
      R bx = R(0), by = R(0), bz = R(0);
      if (i < EB) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if (e & (1 << i)) continue;
          const int f = e | (1 << i);
          const cplx<R> pa = p[e], pb = p[f], wa = w[e], wb = w[f];
          bx = fma(pb.x, wa.y, bx); bx = fma(pb.y, wa.x, bx);
          bx = fma(pa.x, wb.y, bx); bx = fma(pa.y, wb.x, bx);
          by = fma(-pb.x, wa.x, by); by = fma(pb.y, wa.y, by);
          by = fma(pa.x, wb.x, by); by = fma(-pa.y, wb.y, by);
          bz = fma(pa.x, wa.y, bz); bz = fma(pa.y, wa.x, bz);
          bz = fma(-pb.x, wb.y, bz); bz = fma(-pb.y, wb.x, bz);
          p[e] = rot_one<R, NEAR>(pa, pb, c, s, -t);
          p[f] = rot_one<R, NEAR>(pb, pa, c, -s, -t);
          w[e] = rot_one<R, NEAR>(wa, wb, c, s, t);
          w[f] = rot_one<R, NEAR>(wb, wa, c, -s, t);
        }
      } else {
        const int m = 1 << (i - EB);
        const bool up = (l & m) != 0;
        const R sg = up ? -s : s;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const cplx<R> po = swap(p[e], m * C), wo = swap(w[e], m * C);
          bx = fma(po.x, w[e].y, bx); bx = fma(po.y, w[e].x, bx);
          by = fma(po.x, w[e].x, by); by = fma(-po.y, w[e].y, by);
          bz = fma(p[e].x, w[e].y, bz); bz = fma(p[e].y, w[e].x, bz);
          p[e] = rot_one<R, NEAR>(p[e], po, c, sg, -t);
          w[e] = rot_one<R, NEAR>(w[e], wo, c, sg, t);
        }
        if (!up) by = -by;
        if (up) bz = -bz;
      }
      bl[3 * i] = bx;
      bl[3 * i + 1] = by;
      bl[3 * i + 2] = bz;
    }
  }
};

// Sum of each of NV values over groups of W adjacent lanes.  W = 32: halving exchange (P - 1 + few
// shuffles for P = 16 or 32 padded values); the lane's value index is returned (-1: holds none) and
// its sum left in v[0].
template <typename R, int NV> struct WarpSums {
  static constexpr int P = NV <= 8 ? 8 : (NV <= 16 ? 16 : 32);
  static __device__ __forceinline__ int full(R (&v)[P], int lane) {
    int idx = 0, off = 16;
#pragma unroll
    for (int m = P / 2; m >= 1; m >>= 1) {
      const bool up = (lane & off) != 0;
#pragma unroll
      for (int j = 0; j < m; ++j) {
        const R send = up ? v[j] : v[j + m], keep = up ? v[j + m] : v[j];
        v[j] = keep + __shfl_xor_sync(0xffffffffu, send, off);
      }
      if (up) idx += m;
      off >>= 1;
    }
    bool own = true;
#pragma unroll
    for (; off >= 1; off >>= 1) {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
      if (lane & off) own = false;
    }
    return own && idx < NV ? idx : -1;
  }
};

}  // namespace redo
