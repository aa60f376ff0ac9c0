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

// One-qubit tables of a local system: pairs (term k, qubit i) in order of qubit, then term.
template <typename R>
struct LocTab {
  const int32_t* ptr;        // [n + 1] pairs of qubit i
  const int32_t* k;          // [pairs] term (| kLocFirst)
  const cplx<R>* u;          // [pairs][d][base][4] digit operators, row-major 2 x 2
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

// u_ki at level index qv: the product of its digit operators
template <typename R> __device__ __forceinline__ Mat2<R> loc_term(const LocTab<R>& t, int pair, int32_t qv) {
  Mat2<R> m = loc_load(t, (int64_t)pair * t.d * t.base + qv % t.base);
  for (int j = 1; j < t.d; ++j) {
    qv /= t.base;
    m = mat2_mul<R>(loc_load(t, ((int64_t)pair * t.d + j) * t.base + qv % t.base), m);
  }
  return m;
}

template <typename R>
__device__ __forceinline__ int32_t loc_level(const LocTab<R>& t, const int32_t* qrow, int kf, bool count) {
  int32_t qv = qrow[kf & ~kLocFirst];
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
    const Mat2<R> u = loc_term<R>(t, p, loc_level<R>(t, qrow, t.k[p], count));
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
// corrected for what its float conversion dropped
__device__ __forceinline__ float2 phasor(int32_t t) {
  const int32_t k = (int32_t)((uint32_t)t + 0x20000000u) >> 30;
  const int32_t res = (int32_t)((uint32_t)t - ((uint32_t)k << 30));
  const float fh = (float)res;
  const float a = fh * kTurn;
  const float d = fmaf(fh, kTurnLo, fmaf((float)(res - (int32_t)fh), kTurn, fmaf(fh, kTurn, -a)));
  float s, c;
  sincosf(a, &s, &c);
  const float s1 = fmaf(d, c, s), c1 = fmaf(-d, s, c);
  const float re = (k & 1) ? -s1 : c1, im = (k & 1) ? c1 : s1;
  return (k & 2) ? make_float2(-re, -im) : make_float2(re, im);
}

// the angle of z in turns: atan2f, then one refinement against the phasor it gives
__device__ __forceinline__ int32_t turns_of(float2 z) {
  const int32_t t = (int32_t)(uint32_t)(long long)rintf(atan2f(z.y, z.x) * kPerTurn);
  const float2 p = phasor(t);
  const float re = fmaf(z.x, p.x, z.y * p.y), im = fmaf(z.y, p.x, -(z.x * p.y));
  return re > 0.f ? (int32_t)((uint32_t)t + (uint32_t)(int32_t)rintf(im / re * kPerTurn)) : t;
}

template <typename R> struct Euler { phase_t<R> y0, y1, x; R c, s; };

// The phases of a vanishing entry are free; x comes from the larger of the two entries that
// determine it, so every entry of V_i is reproduced to rounding.
template <typename R> __device__ __forceinline__ Euler<R> loc_factor(const Mat2<R>& v) {
  Euler<R> o;
  const R c2 = fma(v.a.x, v.a.x, v.a.y * v.a.y), s2 = fma(v.b.x, v.b.x, v.b.y * v.b.y);
  const R c = sqrt(c2), s = sqrt(s2);
  if constexpr (sizeof(R) == 4) {
    // diag(1, e^{iA}) V diag(1, e^{-iA}) has a real entry -s: y1 = e^{iA} cancels in the diagonal
    o.y0 = turns_of(v.a);
    o.y1 = s > 0.f ? turns_of(make_float2(-v.b.x, -v.b.y)) : 0;
    o.x = (int32_t)(c >= s ? (uint32_t)turns_of(v.e) - (uint32_t)o.y1 : (uint32_t)turns_of(v.c) - (uint32_t)o.y0);
  } else {
    o.y0 = c > R(0) ? cmake<R>(v.a.x / c, v.a.y / c) : cmake<R>(R(1), R(0));
    o.y1 = s > R(0) ? cmake<R>(-v.b.x / s, -v.b.y / s) : cmake<R>(R(1), R(0));
    const cplx<R> w = c >= s ? cmul_conj<R>(v.e, o.y1) : cmul_conj<R>(v.c, o.y0);
    const R wn = sqrt(fma(w.x, w.x, w.y * w.y));
    o.x = wn > R(0) ? cmake<R>(w.x / wn, w.y / wn) : cmake<R>(R(1), R(0));
  }
  // c^2 + s^2 = 1 to the last bit: the residual is exact under fma, so the correction has no bias
  // (dividing by sqrt(c2 + s2), whose spacing is uneven around 1, gained 5e-8 of norm per FP32 step)
  const R res = R(0.5) * fma(-s, s, fma(-c, c, R(1)));
  o.c = fma(res, c, c);
  o.s = fma(res, s, s);
  return o;
}

// Layout of one column (N rows) over G = N / E lanes, E entries each: lane part l holds rows
// l E + e, so the low qubits pair registers of one lane and the high ones pair lanes.  Lanes of
// the same part are adjacent (C = 32 / G columns a warp), and a diagonal is stored as
// [E/2][G][2] (loc_pos), so a lane reads two of its entries at once and the parts read one line.
template <int N> struct Log2 { static constexpr int v = 1 + Log2<N / 2>::v; };
template <> struct Log2<1> { static constexpr int v = 0; };

__host__ __device__ __forceinline__ int loc_pos(int r, int E, int G) {
  const int l = r / E, e = r - l * E;
  return E == 1 ? l : ((e >> 1) * G + l) * 2 + (e & 1);
}

template <typename R, int N, int E> struct LocCol {
  static constexpr int G = N / E, C = 32 / G, NQ = Log2<N>::v, EB = Log2<E>::v;
  static_assert(G * E == N && G <= 32, "column layout");

  // v <- Delta v (or conj(Delta) v)
  template <bool CONJ> static __device__ __forceinline__ void diag(cplx<R> (&v)[E], const cplx<R>* d, int l) {
    if constexpr (E == 1) {
      const cplx<R> a = __ldg(d + l);
      v[0] = CONJ ? cmul_conj<R>(v[0], a) : cmul<R>(v[0], a);
    } else {
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
        v[e] = CONJ ? cmul_conj<R>(v[e], a) : cmul<R>(v[e], a);
        v[e + 1] = CONJ ? cmul_conj<R>(v[e + 1], b) : cmul<R>(v[e + 1], b);
      }
    }
  }
  static __device__ __forceinline__ cplx<R> swap(cplx<R> v, int lane_mask) {
    return cmake<R>(__shfl_xor_sync(0xffffffffu, v.x, lane_mask), __shfl_xor_sync(0xffffffffu, v.y, lane_mask));
  }
  // (c, s) real rotations of every qubit, [[c, -s], [s, c]] on the pair (bit 0, bit 1)
  static __device__ __forceinline__ void rotate(cplx<R> (&v)[E], const cplx<R> (&cs)[NQ], int l) {
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const R c = cs[i].x, s = cs[i].y;
      if (i < EB) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if (e & (1 << i)) continue;
          const cplx<R> a = v[e], b = v[e | (1 << i)];
          v[e] = cmake<R>(fma(-s, b.x, c * a.x), fma(-s, b.y, c * a.y));
          v[e | (1 << i)] = cmake<R>(fma(s, a.x, c * b.x), fma(s, a.y, c * b.y));
        }
      } else {
        const int m = 1 << (i - EB);
        const R sg = (l & m) ? s : -s;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const cplx<R> o = swap(v[e], m * C);
          v[e] = cmake<R>(fma(sg, o.x, c * v[e].x), fma(sg, o.y, c * v[e].y));
        }
      }
    }
  }
  static __device__ __forceinline__ void load_cs(cplx<R> (&cs)[NQ], const cplx<R>* p) {
#pragma unroll
    for (int i = 0; i < NQ; ++i) cs[i] = __ldg(p + i);
  }
  // The three Bloch sums of every qubit,
  //   X = Im Tr(X_i P R), Y = Im Tr(Y_i P R), Z = Im Tr(Z_i P R)
  // over this lane's entries of a column p of P and the matching row w of R, then the qubit's
  // rotation undone on both (p <- rot^T p, w <- rot^T w).  A partial trace over the other qubits
  // does not change when those are rotated, so each qubit is traced just before its own undo.
  static __device__ __forceinline__ void trace_undo(cplx<R> (&p)[E], cplx<R> (&w)[E], const cplx<R> (&cs)[NQ],
                                                    int l, R* bl) {
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const R c = cs[i].x, s = cs[i].y;
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
          p[e] = cmake<R>(fma(s, pb.x, c * pa.x), fma(s, pb.y, c * pa.y));
          p[f] = cmake<R>(fma(-s, pa.x, c * pb.x), fma(-s, pa.y, c * pb.y));
          w[e] = cmake<R>(fma(s, wb.x, c * wa.x), fma(s, wb.y, c * wa.y));
          w[f] = cmake<R>(fma(-s, wa.x, c * wb.x), fma(-s, wa.y, c * wb.y));
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
          p[e] = cmake<R>(fma(sg, po.x, c * p[e].x), fma(sg, po.y, c * p[e].y));
          w[e] = cmake<R>(fma(sg, wo.x, c * w[e].x), fma(sg, wo.y, c * w[e].y));
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
