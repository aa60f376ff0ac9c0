// Chains, gradients and state sweeps of locally controlled systems (local_ops.cuh), N <= 1024.
// (Section II processes 1 and 2: the discrete operators and their products, here on the 2 x 2
// parts whose tensor product the N x N table operator is; Section III: chain, GRAPE gradient, state
// transfer; Section IV: observables along the chain.)
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "local_ops.cuh"

namespace redo {

// ============================================================================
// Detection and one-qubit tables (at table build)
// ============================================================================

// Digit operators u[set][j][c] = exp(-i dt theta h) of a 2 x 2 Hermitian h = a0 I + v.sigma:
// exp(-i t a0) (cos(t |v|) I - i sin(t |v|) / |v| v.sigma), theta as in the dense table; rep[set] is a
// pair with these operators.
__global__ void loc_table_kernel(const double2* __restrict__ h, const int32_t* __restrict__ k,
                                 const int32_t* __restrict__ rep, int sets, int d, int base, double dt,
                                 const double* __restrict__ lo, const double* __restrict__ delta,
                                 double2* __restrict__ u64, float2* __restrict__ u32) {
  const int64_t total = (int64_t)sets * d * base;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(e % base), j = (int)((e / base) % d), p = rep[e / ((int64_t)base * d)];
    const int kk = k[p] & 0xff;
    double bj = 1.0;
    for (int i = 0; i < j; ++i) bj *= (double)base;
    const double th = j == 0 ? __dadd_rn(lo[kk], __dmul_rn((double)c, delta[kk])) : __dmul_rn((double)c * bj, delta[kk]);
    const double2 *hp = h + 4 * p;
    const double a0 = 0.5 * (hp[0].x + hp[3].x), vz = 0.5 * (hp[0].x - hp[3].x), vx = hp[1].x, vy = -hp[1].y;
    const double t = dt * th, v = sqrt(vx * vx + vy * vy + vz * vz);
    double sn, cs, s0, c0;
    sincos(t * v, &sn, &cs);
    sincos(t * a0, &s0, &c0);
    const double f = v > 0.0 ? sn / v : 0.0;
    // cos I - i f (v.sigma), times exp(-i t a0) = c0 - i s0
    const double2 m[4] = {make_double2(cs, -f * vz), make_double2(-f * vy, -f * vx), make_double2(f * vy, -f * vx),
                          make_double2(cs, f * vz)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double2 o = make_double2(m[i].x * c0 + m[i].y * s0, m[i].y * c0 - m[i].x * s0);
      u64[e * 4 + i] = o;
      u32[e * 4 + i] = make_float2((float)o.x, (float)o.y);
    }
  }
}

// Splits H (row-major N x N, host) into one-qubit terms h[i] (2 x 2); false when it has others.
static bool split_local(const double* H, int N, int n, double2* h) {
  auto at = [&](int r, int c) { return make_double2(H[2 * ((size_t)r * N + c)], H[2 * ((size_t)r * N + c) + 1]); };
  double mx = 0.0;
  for (size_t i = 0; i < (size_t)2 * N * N; ++i) mx = std::fmax(mx, std::fabs(H[i]));
  const double tol = 8 * 2.3e-16 * mx;             // rounding of sums of the same terms
  auto close = [&](double2 a, double2 b) { return std::fabs(a.x - b.x) <= tol && std::fabs(a.y - b.y) <= tol; };
  const double2 d0 = at(0, 0);
  for (int i = 0; i < n; ++i) {
    const int m = 1 << i;
    h[4 * i] = i == 0 ? make_double2(d0.x, 0.0) : make_double2(0.0, 0.0);
    h[4 * i + 3] = make_double2(h[4 * i].x + at(m, m).x - d0.x, 0.0);
    h[4 * i + 1] = at(0, m);
    h[4 * i + 2] = make_double2(h[4 * i + 1].x, -h[4 * i + 1].y);
  }
  for (int r = 0; r < N; ++r) {
    double2 dr = make_double2(0.0, 0.0);
    for (int i = 0; i < n; ++i) {
      const int b = (r >> i) & 1;
      dr.x += h[4 * i + 3 * b].x;
      if (!close(at(r, r ^ (1 << i)), h[4 * i + 1 + b])) return false;
    }
    if (!close(at(r, r), dr)) return false;
    for (int c = 0; c < N; ++c) {
      const int m = r ^ c;
      if ((m & (m - 1)) != 0) {                    // more than one qubit flipped
        const double2 v = at(r, c);
        if (std::fabs(v.x) > tol || std::fabs(v.y) > tol) return false;
      }
    }
  }
  return true;
}

// h: host copies of H0 then H_0 .. H_{K-1}.  Leaves o.on false for any other system.
void local_detect(redo_table* t, const std::vector<double>& h, TableArena& ar, LocalParts& o) {
  if (!t->h0_diagonal) return;
  const int N = t->N, K = t->K;
  int n = 0;
  while ((1 << n) < N) ++n;
  const size_t n2 = (size_t)N * N;
  std::vector<double2> hk((size_t)K * n * 4);
  for (int k = 0; k < K; ++k)
    if (!split_local(h.data() + 2 * n2 * (k + 1), N, n, hk.data() + (size_t)k * n * 4)) return;
  std::vector<int32_t> ptr(n + 1), kk;
  std::vector<double2> hp;
  std::vector<char> seen(K, 0);
  for (int i = 0; i < n; ++i) {
    ptr[i] = (int32_t)kk.size();
    for (int k = 0; k < K; ++k) {
      const double2* m = hk.data() + ((size_t)k * n + i) * 4;
      bool any = false;
      for (int e = 0; e < 4; ++e) any = any || m[e].x != 0.0 || m[e].y != 0.0;
      if (!any) continue;
      kk.push_back(k | (seen[k] ? 0 : kLocFirst));
      seen[k] = 1;
      hp.insert(hp.end(), m, m + 4);
    }
  }
  for (int k = 0; k < K; ++k)
    if (!seen[k]) {                                // H_k = 0: still a term whose level index is checked
      kk.push_back(k | kLocFirst);
      hp.insert(hp.end(), 4, make_double2(0.0, 0.0));
    }
  ptr[n] = (int32_t)kk.size();
  const int pairs = (int)kk.size();
  std::vector<int32_t> kptr(K + 1, 0), kpair;
  for (int k = 0; k < K; ++k) {
    kptr[k] = (int32_t)kpair.size();
    for (int i = 0; i < n; ++i)
      for (int p = ptr[i]; p < ptr[i + 1]; ++p)
        if ((kk[p] & ~kLocFirst) == k) kpair.push_back(p | (i << 20));
  }
  kptr[K] = (int32_t)kpair.size();
  std::vector<float4> D32(N);
  for (int r = 0; r < N; ++r) {
    const double a = t->dt * h[2 * ((size_t)r * N + r)], sh = std::sin(0.5 * a), x = -2.0 * sh * sh, y = -std::sin(a);
    D32[r] = make_float4((float)x, (float)y, (float)(x - (double)(float)x), (float)(y - (double)(float)y));
  }
  // X controls of every qubit, or a global field's part on each, are one set of operators: N = 8 with six
  // controls of 4096 levels keeps 0.8 MB, not 2.4 MB (which fits beside the dense table in one mapping:
  // building the table takes 237 us for two global controls, 264 for six local ones; with an allocation,
  // copy and wait of their own 318 and 305, without one-qubit tables 270 and 299)
  std::vector<int32_t> rep;
  for (int p = 0; p < pairs; ++p) {
    const int k = kk[p] & ~kLocFirst;
    int set = 0;
    for (; set < (int)rep.size(); ++set) {
      const int r = rep[set], kr = kk[r] & 0xff;
      if (std::memcmp(&hp[4 * p], &hp[4 * r], 4 * sizeof(double2)) == 0 && t->lo[k] == t->lo[kr] &&
          t->delta[k] == t->delta[kr])
        break;
    }
    if (set == (int)rep.size()) rep.push_back(p);
    kk[p] |= set << 8;
  }
  std::vector<float2> hp32(hp.size());
  // FP32 operators of entries near 1 whatever the unit of the controls; the gradients make up for it
  for (int k = 0; k < K; ++k) {
    double mx = 0.0;
    for (int e = kptr[k]; e < kptr[k + 1]; ++e)
      for (int c = 0; c < 4; ++c) {
        const double2 v = hp[4 * (kpair[e] & 0xfffff) + c];
        mx = std::fmax(mx, std::fmax(std::fabs(v.x), std::fabs(v.y)));
      }
    const int x = mx > 0.0 ? std::ilogb(mx) : 0;
    kptr.push_back(x);
    for (int e = kptr[k]; e < kptr[k + 1]; ++e)
      for (int c = 0; c < 4; ++c) {
        const size_t i = 4 * (size_t)(kpair[e] & 0xfffff) + c;
        hp32[i] = make_float2((float)std::scalbn(hp[i].x, -x), (float)std::scalbn(hp[i].y, -x));
      }
  }
  // one operator per level (no digit products per step) while the table stays small beside L2
  const bool levels = t->levels <= 65536 && (double)rep.size() * t->levels * 96.0 <= 64e6;
  t->loc_d = levels ? 1 : t->digit_count;
  t->loc_base = levels ? (int)t->levels : t->digit_base;
  t->loc_pairs = pairs;
  o.entries = rep.size() * t->loc_d * t->loc_base;
  o.rep = ar.put(rep.data(), sizeof(int32_t) * rep.size());
  std::vector<double2> D(N);
  for (int r = 0; r < N; ++r) {
    const double a = t->dt * h[2 * ((size_t)r * N + r)];
    const double sh = std::sin(0.5 * a);
    D[r] = make_double2(-2.0 * sh * sh, -std::sin(a));                // exp(-i a) - 1
  }
  o.ptr = ar.put(ptr.data(), sizeof(int32_t) * (n + 1));
  o.k = ar.put(kk.data(), sizeof(int32_t) * pairs);
  o.h = ar.put(hp.data(), sizeof(double2) * 4 * pairs);
  o.h32 = ar.put(hp32.data(), sizeof(float2) * 4 * pairs);
  o.kptr = ar.put(kptr.data(), sizeof(int32_t) * kptr.size());
  o.kpair = ar.put(kpair.data(), sizeof(int32_t) * pairs);
  o.D = ar.put(D.data(), sizeof(double2) * N);
  o.D32 = ar.put(D32.data(), sizeof(float4) * N);
  // the phase axes' one-qubit parts (local_phase_axes) and whether they apply
  const std::vector<double> none((size_t)K * n, 0.0);
  const int32_t off = 0;
  o.wz = ar.put(none.data(), sizeof(double) * none.size());
  o.wz_on = ar.put(&off, sizeof(off));
  o.on = true;
}

void local_room(const redo_table* t, TableArena& ar, LocalParts& o) {
  if (!o.on) return;
  o.u64 = ar.room(sizeof(double2) * 4 * o.entries);
  o.u32 = ar.room(sizeof(float2) * 4 * o.entries);
}

cudaError_t local_build(redo_table* t, const LocalParts& o, char* base, cudaStream_t s) {
  if (!o.on) return cudaSuccess;
  t->loc_ptr = (int32_t*)(base + o.ptr);
  t->loc_k = (int32_t*)(base + o.k);
  t->loc_h = (double2*)(base + o.h);
  t->loc_h32 = (float2*)(base + o.h32);
  t->loc_kptr = (int32_t*)(base + o.kptr);
  t->loc_kpair = (int32_t*)(base + o.kpair);
  t->loc_D64 = (double2*)(base + o.D);
  t->loc_D32 = (float4*)(base + o.D32);
  t->wz = (double*)(base + o.wz);
  t->wz_on = (int32_t*)(base + o.wz_on);
  t->loc_u64 = (double2*)(base + o.u64);
  t->loc_u32 = (float2*)(base + o.u32);
  const size_t blocks = (o.entries + 127) / 128, sets = o.entries / ((size_t)t->loc_d * t->loc_base);
  loc_table_kernel<<<(unsigned)(blocks < 4096 ? blocks : 4096), 128, 0, s>>>(
      t->loc_h, t->loc_k, (const int32_t*)(base + o.rep), (int)sets, t->loc_d, t->loc_base, t->dt, t->d_lo, t->d_delta,
      t->loc_u64, t->loc_u32);
  while ((1 << t->loc) < t->N) ++t->loc;
  return cudaGetLastError();
}

// sz [K][N] (host): their one-qubit parts when each is a sum of those, written over the previous ones
// (a captured call reads them, and whether they apply, where it found them at capture)
cudaError_t local_phase_axes(redo_table* t, const double* sz) {
  if (!t->loc) return cudaSuccess;
  const int N = t->N, K = t->K, n = t->loc;
  std::vector<double> w((size_t)K * n);
  int32_t on = 1;
  for (int k = 0; k < K; ++k) {
    const double* z = sz + (size_t)k * N;
    double mx = 0.0;
    for (int r = 0; r < N; ++r) mx = std::fmax(mx, std::fabs(z[r]));
    for (int i = 0; i < n; ++i) w[(size_t)k * n + i] = 0.5 * (z[0] - z[1 << i]);
    for (int r = 0; r < N; ++r) {
      double v = z[0];
      for (int i = 0; i < n; ++i)
        if ((r >> i) & 1) v -= 2.0 * w[(size_t)k * n + i];
      if (std::fabs(v - z[r]) > 8 * 2.3e-16 * mx) on = 0;
    }
  }
  cudaError_t e = cudaMemcpy(t->wz, w.data(), sizeof(double) * w.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(t->wz_on, &on, sizeof(on), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) t->wz_local = on;
  return e;
}

template <typename R> static LocTab<R> loc_tab(const redo_table* t, int64_t* status) {
  LocTab<R> o;
  o.ptr = t->loc_ptr;
  o.k = t->loc_k;
  o.u = std::is_same<R, double>::value ? (const cplx<R>*)t->loc_u64 : (const cplx<R>*)t->loc_u32;
  o.d = t->loc_d;
  o.base = t->loc_base;
  o.K = t->K;
  o.levels = t->levels;
  o.status = status;
  o.bad_weight = t->digits;
  return o;
}

// ============================================================================
// Step operators of the steps m0 .. m0 + T of every pulse: rotations cs[b][n - m0][i] and diagonals
// Delta[b][n - m0][N], n - m0 <= T (Delta_M closes the chain; a window that ends earlier also gets
// the next step's)
// ============================================================================
// A block takes ts steps: the one-qubit work (a long dependent chain per step and qubit) needs many
// steps in a block to fill its warps, few pulses need many blocks (loc_steps_t).  g (gradients):
// also the step's derivative operators, for every pair (term k, qubit i) the real (gx, gy, gz) of
//     W h_ki W^dag,  W the product of the factors after k on qubit i,
// turned by the trailing phases (the sweep's Bloch sums are taken before those), [step][pair][3].
constexpr int kPrepSteps = 32, kPrepThreads = 256;

template <typename R> __device__ __forceinline__ phase_t<R> no_phase() {
  if constexpr (sizeof(R) == 4) return 0;
  else return cmake<R>(R(1), R(0));
}

// (1 + v)(1 + d) - 1.  FP32 takes d as hi + lo: the drift is the same at every step, so its rounding
// would add up over the chain.  (Kept split: converting FP64 values in the kernel, at the FP64 rate,
// took two thirds of its time.)
template <typename R> struct DiagOf { using T = double2; };
template <> struct DiagOf<float> { using T = float4; };            // hi.x, hi.y, lo.x, lo.y
__device__ __forceinline__ float4 loc_split(double2 d) {
  const float2 h = make_float2((float)d.x, (float)d.y);
  return make_float4(h.x, h.y, (float)(d.x - (double)h.x), (float)(d.y - (double)h.y));
}
__device__ __forceinline__ double2 loc_times(double2 v, double2 d) {
  double2 o = make_double2(v.x + d.x, v.y + d.y);
  cfma<double>(o, v, d);
  return o;
}
__device__ __forceinline__ float2 loc_times(float2 v, float4 d) {
  float2 o = make_float2(v.x + d.x + d.z, v.y + d.y + d.w);
  cfma<float>(o, v, make_float2(d.x, d.y));
  return o;
}

template <typename R>
__device__ __forceinline__ void loc_derivatives(const LocTab<R>& tab, const int32_t* qrow, int i, const Euler<R>& f,
                                                const cplx<R>* __restrict__ h, R* __restrict__ g) {
  cplx<R> x;                                         // conj(x0) x1
  if constexpr (sizeof(R) == 4)
    x = phasor<false>((int32_t)((uint32_t)f.x - (uint32_t)f.x0));
  else
    x = f.x;
  Mat2<R> w;
  w.a = w.e = cmake<R>(R(1), R(0));
  w.b = w.c = cmake<R>(R(0), R(0));
  const int p0 = tab.ptr[i];
  for (int p = tab.ptr[i + 1] - 1; p >= p0; --p) {
    const Mat2<R> hm = {h[4 * p], h[4 * p + 1], h[4 * p + 2], h[4 * p + 3]};
    const Mat2<R> wd = {cmake<R>(w.a.x, -w.a.y), cmake<R>(w.c.x, -w.c.y), cmake<R>(w.b.x, -w.b.y),
                        cmake<R>(w.e.x, -w.e.y)};
    const Mat2<R> gm = mat2_mul<R>(mat2_mul<R>(w, hm), wd);
    const cplx<R> g01 = cmul<R>(gm.b, x);
    g[3 * p] = g01.x;
    g[3 * p + 1] = -g01.y;
    g[3 * p + 2] = R(0.5) * (gm.a.x - gm.e.x);
    if (p > p0) w = mat2_mul<R>(w, loc_term<R>(tab, tab.k[p], loc_level<R>(tab, qrow, tab.k[p], false)));
  }
}

template <typename R, bool NEAR>
__global__ void __launch_bounds__(kPrepThreads)
loc_steps_kernel(LocTab<R> tab, const int32_t* __restrict__ q, int64_t M, int64_t m0, int64_t T, int n, int N, int E,
                 int64_t tiles, int ts, const typename DiagOf<R>::T* __restrict__ D, const double2* __restrict__ pd,
                 int64_t pd_b, int64_t pd_n,
                 cplx<R>* __restrict__ cs, cplx<R>* __restrict__ delta, const cplx<R>* __restrict__ h, int pairs,
                 R* __restrict__ gout) {
  // phases of every (step, qubit); row j is step n0 - 1 + j (the step before the tile gives its x)
  __shared__ phase_t<R> y0[kPrepSteps + 1][10], y1[kPrepSteps + 1][10], xx[kPrepSteps + 1][10],
      x0[kPrepSteps + 1][10];
  const int64_t b = blockIdx.x / tiles;
  const int64_t n0 = m0 + (blockIdx.x - b * tiles) * ts;
  for (int idx = threadIdx.x; idx < (ts + 1) * n; idx += kPrepThreads) {
    const int j = idx / n, i = idx - j * n;
    const int64_t m = n0 - 1 + j;
    Euler<R> f;
    f.y0 = f.y1 = f.x = f.x0 = no_phase<R>();
    if (m >= 0 && m < M && m <= m0 + T) {
      const bool own = j > 0 && m < m0 + T;
      f = loc_factor<R, NEAR>(loc_step<R>(tab, q + (b * M + m) * tab.K, i, own));
      if (own) {
        cplx<R>* o = cs + (b * T + m - m0) * n * (NEAR ? 2 : 1) + i;
        o[0] = cmake<R>(f.c1, f.s);
        if (NEAR) o[n] = cmake<R>(f.sy, R(0));
        if (gout) loc_derivatives<R>(tab, q + (b * M + m) * tab.K, i, f, h, gout + (b * T + m - m0) * pairs * 3);
      }
    }
    y0[j][i] = f.y0;
    y1[j][i] = f.y1;
    xx[j][i] = f.x;
    if (NEAR) x0[j][i] = f.x0;
  }
  __syncthreads();
  const int G = N / E;
  // Delta: a thread takes rows of one step that share their high bits
  const int rows = N < 8 ? N : 8, low = N < 8 ? n : 3;
  for (int idx = threadIdx.x; idx < ts * (N / rows); idx += kPrepThreads) {
    const int j = idx / (N / rows) + 1, r0 = (idx - (j - 1) * (N / rows)) * rows;
    const int64_t m = n0 - 1 + j;
    if (m > m0 + T) continue;
    phase_t<R> hi = no_phase<R>();
    auto of = [&](int i, int up) -> phase_t<R> {
      if constexpr (NEAR) {
        return up ? xx[j - 1][i] : x0[j - 1][i];
      } else if constexpr (sizeof(R) == 4) {
        return up ? (int32_t)((uint32_t)y1[j][i] + (uint32_t)xx[j - 1][i]) : y0[j][i];
      } else {
        return up ? cmul<R>(y1[j][i], xx[j - 1][i]) : y0[j][i];
      }
    };
    auto join = [](phase_t<R> a, phase_t<R> b) -> phase_t<R> {
      if constexpr (sizeof(R) == 4)
        return (int32_t)((uint32_t)a + (uint32_t)b);
      else
        return cmul<R>(a, b);
    };
    for (int i = low; i < n; ++i) hi = join(hi, of(i, (r0 >> i) & 1));
    phase_t<R> lo[3][2];
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (i < low) {
        lo[i][0] = of(i, 0);
        lo[i][1] = of(i, 1);
      }
    cplx<R>* o = delta + (b * (T + 1) + m - m0) * N;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (e >= rows) break;
      phase_t<R> a = hi;
#pragma unroll
      for (int i = 0; i < 3; ++i)
        if (i < low) a = join(a, lo[i][(e >> i) & 1]);
      cplx<R> v;                                     // Delta - 1
      if constexpr (sizeof(R) == 4)
        v = phasor<true>(a);
      else
        v = cmake<R>(a.x - R(1), a.y);
      const int r = r0 + e;
      if (m < M) {
        v = loc_times(v, D[r]);
        if (pd) {
          const double2* at = pd + b * pd_b + m * pd_n + r;
          if constexpr (sizeof(R) == 4)
            v = loc_times(v, pd_n == 0 ? *reinterpret_cast<const float4*>(at) : loc_split(make_double2(at->x - 1.0, at->y)));
          else
            v = loc_times(v, make_double2(at->x - 1.0, at->y));
        }
      }
      // scaled to |Delta| = 1: without it the rounding of the phases changed the chain's norm five
      // times as much
      const R res = R(-0.5) * fma(v.x, v.x, fma(v.y, v.y, R(2) * v.x));
      o[loc_pos(r, E, G)] = cmake<R>(v.x + fma(res, v.x, res), fma(res, v.y, v.y));
    }
  }
}

// ============================================================================
// Chains: segment products S_s = Rot_{n1-1} Delta_{n1-1} ... Rot_{n0} Delta_{n0} (the last segment
// of a pulse also takes Delta_M), a column per G lanes, the whole segment in registers
// ============================================================================
constexpr int kLocThreads = 128;

template <typename R, int N, int E, bool NEAR>
__global__ void __launch_bounds__(kLocThreads)
loc_chain_kernel(const cplx<R>* __restrict__ cs, const cplx<R>* __restrict__ delta, int64_t M, int64_t S, int64_t sps,
                 int64_t chains, cplx<R>* __restrict__ out) {
  using L = LocCol<R, N, E, NEAR>;
  static_assert(L::G == 1 || N >= L::C, "lanes of one warp share a chain when they exchange");
  const int lane = threadIdx.x & 31, l = lane / L::C;
  const int64_t col = ((int64_t)blockIdx.x * (kLocThreads / 32) + (threadIdx.x >> 5)) * L::C + lane % L::C;
  const int64_t g = col / N;
  if (g >= chains) return;
  const int x = (int)(col - g * N);
  const int64_t b = g / S, n0 = (g - b * S) * sps, n1 = n0 + sps < M ? n0 + sps : M;
  cplx<R> v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = cmake<R>(l * E + e == x ? R(1) : R(0), R(0));
  const cplx<R>* d = delta + b * (M + 1) * N;
  const cplx<R>* r = cs + b * M * L::CS;
#pragma unroll 1
  for (int64_t m = n0; m < n1; ++m) {
    cplx<R> c[L::CS];
    L::load_cs(c, r + m * L::CS);
    L::template diag<false>(v, d + m * N, l);
    L::rotate(v, c, l);
  }
  if (n1 == M) L::template diag<false>(v, d + M * N, l);
  cplx<R>* o = out + g * N * N + x;
#pragma unroll
  for (int e = 0; e < E; ++e) o[(int64_t)(l * E + e) * N] = v[e];
}

// Entries a lane holds.  FP32: 32 for chains (64 state registers), 16 for the gradient's two
// vectors.  FP64: the FP64 pipe issues one warp instruction per ~70 cycles and scheduler whatever
// the lane count, so a column is spread over more lanes; small N must fill a warp with one chain.
__host__ __device__ constexpr int loc_entries(bool dbl, int N, bool two) {
  if (dbl) return N <= 4 ? N : (N == 8 ? 2 : (N == 16 || (two && N <= 256) ? 8 : (N <= 512 ? 16 : 32)));
  const int e = two && N <= 512 ? 16 : 32;
  return N < e ? N : e;
}

template <typename R, int N, bool TWO>
static cudaError_t loc_chain_n(const redo_table* t, const ChainPlan& p, int64_t B, bool near, const void* cs,
                               const void* delta, void* out, cudaStream_t s) {
  constexpr int E = loc_entries(sizeof(R) == 8, N, TWO);
  const int64_t fps = (int64_t)t->K * t->digits, chains = B * p.S, sps = p.seg_len / fps;
  const int64_t warps = (chains * N * (N / E) + 31) / 32;
  if (warps == 0) return cudaSuccess;
  auto kern = loc_chain_kernel<R, N, E, loc_near(sizeof(R) == 8, N)>;
  if constexpr (sizeof(R) == 4 && !TWO)
    if (near) kern = loc_chain_kernel<R, N, E, true>;
  kern<<<(unsigned)((warps + 3) / 4), kLocThreads, 0, s>>>(
      (const cplx<R>*)cs, (const cplx<R>*)delta, p.M, p.S, sps > 0 ? sps : 1, chains, (cplx<R>*)out);
  return cudaGetLastError();
}

#define LOC_DISPATCH(FN, ...)                                     \
  switch (t->N) {                                                 \
    case 2: return FN<R, 2, TWO>(__VA_ARGS__);                    \
    case 4: return FN<R, 4, TWO>(__VA_ARGS__);                    \
    case 8: return FN<R, 8, TWO>(__VA_ARGS__);                    \
    case 16: return FN<R, 16, TWO>(__VA_ARGS__);                  \
    case 32: return FN<R, 32, TWO>(__VA_ARGS__);                  \
    case 64: return FN<R, 64, TWO>(__VA_ARGS__);                  \
    case 128: return FN<R, 128, TWO>(__VA_ARGS__);                \
    case 256: return FN<R, 256, TWO>(__VA_ARGS__);                \
    case 512: return FN<R, 512, TWO>(__VA_ARGS__);                \
    case 1024: return FN<R, 1024, TWO>(__VA_ARGS__);              \
    default: return cudaErrorInvalidValue;                        \
  }

template <typename R, bool TWO>
static cudaError_t loc_chain_t(const redo_table* t, const ChainPlan& p, int64_t B, bool near, const void* cs,
                               const void* delta, void* out, cudaStream_t s) {
  LOC_DISPATCH(loc_chain_n, t, p, B, near, cs, delta, out, s)
}

// ============================================================================
// GRAPE gradient: reverse sweep of the segments.  A column x of P and row x of R stay with the
// same lanes, so undoing a step (P <- U^dag P, R <- R U) and the traces are local to them; only
// the Bloch sums Im Tr(sigma_i P R) of every qubit are added over x.  (R is taken times conj(tau), in
// FP32 times 2^-exp_of(tau), which the gradients make up for.)  They hold every control's
// trace: Tr(g P R) for g = sum_i g_i needs the one-qubit partial traces only.  bl receives them as
// [step][part][3n], one part per warp of the chain, added in a fixed order afterwards.
// TZ (amplitude/phase calls): also Tz = Im Tr(S_kz P R) at every step boundary.  gate: the form with
// (TZ) and without the boundary traces both stand in a captured call, and the one that the axes in
// force do not need returns.
// ============================================================================
template <typename R, int N, int E, bool TZ>
__global__ void __launch_bounds__(kLocThreads, E * sizeof(R) <= 64 ? 4 : 2)
loc_sweep_kernel(const cplx<R>* __restrict__ cs, const cplx<R>* __restrict__ delta, int64_t M, int64_t S, int64_t sps,
                 int64_t chains, const cplx<R>* __restrict__ Pck, const cplx<R>* __restrict__ Rck,
                 const double2* __restrict__ tau, R* __restrict__ bl, int K, const R* __restrict__ sz,
                 R* __restrict__ bz, const int32_t* __restrict__ gate) {
  if (gate && (*gate != 0) == TZ) return;
  using L = LocCol<R, N, E>;
  using WS = WarpSums<R, 3 * L::NQ>;
  constexpr int LPC = N * L::G, PARTS = LPC >= 32 ? LPC / 32 : 1, W = LPC >= 32 ? 32 : LPC;
  const int lane = threadIdx.x & 31, l = lane / L::C;
  const int64_t col = ((int64_t)blockIdx.x * (kLocThreads / 32) + (threadIdx.x >> 5)) * L::C + lane % L::C;
  const bool on = col / N < chains;
  const int64_t g = on ? col / N : chains - 1;       // idle lanes follow the last chain, write nothing
  const int x = (int)(col % N);
  const int part = x / L::C;
  const int64_t b = g / S, n0 = (g - b * S) * sps, n1 = n0 + sps < M ? n0 + sps : M;
  const cplx<R>* d = delta + b * (M + 1) * N;
  const cplx<R>* r = cs + b * M * L::CS;
  cplx<R> p[E], w[E];
  {
    double2 tb = tau[b];
    if constexpr (sizeof(R) == 4) {
      const int et = exp_of(tb);
      tb = make_double2(down2(tb.x, et), down2(tb.y, et));
    }
    const cplx<R>* P = Pck + g * N * N + x;
    const cplx<R>* Q = Rck + g * N * N + (int64_t)x * N + l * E;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      p[e] = P[(int64_t)(l * E + e) * N];
      const double qx = (double)Q[e].x, qy = (double)Q[e].y;      // R conj(tau): traces come out as Im alone
      w[e] = cmake<R>((R)(qx * tb.x + qy * tb.y), (R)(qy * tb.x - qx * tb.y));
    }
  }
  // Tr(S_kz P R) = sum_r sz[k][r] (P R)[r][r], this lane's rows
  auto boundary = [&](int64_t n, bool act) {
    if constexpr (TZ) {
      R t[E];
#pragma unroll
      for (int e = 0; e < E; ++e) t[e] = fma(p[e].x, w[e].y, p[e].y * w[e].x);
      for (int k = 0; k < K; ++k) {
        R a = R(0);
#pragma unroll
        for (int e = 0; e < E; ++e) a = fma(__ldg(sz + (int64_t)k * N + l * E + e), t[e], a);
#pragma unroll
        for (int off = W / 2; off >= 1; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        if (act && lane % W == 0) bz[((b * (M + 1) + n) * PARTS + part) * K + k] = a;
      }
    }
  };
  if (n1 == M) {
    L::template diag<true>(p, d + M * N, l);
    L::template diag<false>(w, d + M * N, l);
  }
  boundary(M, on && n1 == M);
  const int len = (int)(n1 - n0);
  const int most = LPC >= 32 ? len : __reduce_max_sync(0xffffffffu, len);   // several chains in a warp
#pragma unroll 1
  for (int t = 0; t < most; ++t) {
    const bool act = on && t < len;
    const int64_t m = t < len ? n1 - 1 - t : n0;
    cplx<R> c[L::CS];
    L::load_cs(c, r + m * L::CS);
    R v[WS::P];
#pragma unroll
    for (int i = 0; i < WS::P; ++i) v[i] = R(0);
    L::trace_undo(p, w, c, l, v);
    R* o = bl + ((b * M + m) * PARTS + part) * (3 * L::NQ);
    if constexpr (W == 32) {
      const int idx = WS::full(v, lane);
      if (act && idx >= 0) o[idx] = v[0];
    } else {
#pragma unroll
      for (int i = 0; i < 3 * L::NQ; ++i) {
#pragma unroll
        for (int off = W / 2; off >= 1; off >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], off);
        if (act && lane % W == 0) o[i] = v[i];
      }
    }
    boundary(m, act);
    L::template diag<true>(p, d + m * N, l);
    L::template diag<false>(w, d + m * N, l);
  }
}

// dF/du_kn = (2 dt / N^2) sum_i (gx X_i + gy Y_i + gz Z_i), a thread per (step, term): its pairs are
// kpair[kptr[k] ..] (pair | qubit << 20), the Bloch sums bl [step][part][3n] or, already added, sums.
// The sums are those of scaled vectors (and operators, by 2^-e) in FP32: times 2^e 2^exp_of(tau[b]), or
// 2^e amp[b].
template <typename R>
__device__ __forceinline__ double loc_scaled(double x, const double2* tau, const double* amp, int64_t b, int e) {
  if (sizeof(R) == 8) return x;
  return amp ? down2(x, -e) * amp[b] : down2(x, -exp_of(tau[b]) - e);
}
// The phase gradients when every S_kz is a sum of one-qubit parts (wz [K][n], half the difference of a
// qubit's two values; the species' S_z are): the change of Z_i over a step's rotation follows from the
// Bloch sums as 2 |s|^2 Z - 2 c (sx X + sy Y), without the boundary traces and the difference of two
// nearly equal ones (N = 64, 16 x 200, FP32: error against 64 bits 2.4e-6 -> 4.7e-7).  Formed beside the
// amplitudes' gradients (PH): a launch of its own was 3 of the 66 us of N = 8, 10 x 41.  (A form apart:
// with the choice at run time the other gradients' took 66 us, not 49, at N = 32, 256 x 500.)
template <typename R> struct LocPhaseOut {
  const cplx<R>* cs;
  const double* wz;
  const int32_t* gate;
  double scale;
  double* gphi;
  int cs_step;               // entries of cs per step: n, or 2n with the rotations' second parts
};
template <typename R, bool PH>
__global__ void loc_grad_kernel(int64_t steps, int K, int n, int pairs, int parts, const int32_t* __restrict__ kptr,
                                const int32_t* __restrict__ kpair, const R* __restrict__ g, const R* __restrict__ bl,
                                const double* __restrict__ sums, int64_t M, int64_t w0, int64_t T, double scale,
                                const double2* __restrict__ tau, const double* __restrict__ amp,
                                double* __restrict__ grad, LocPhaseOut<R> ph) {
  const bool phase = PH && !(ph.gate && *ph.gate == 0);
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < steps * K;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t st = idx / K, b = st / T;
    const int k = (int)(idx - st * K);
    auto bloch = [&](int i, int c) -> double {
      if (sums) return sums[st * 3 * n + 3 * i + c];
      double v = 0.0;
      for (int q = 0; q < parts; ++q) v += (double)bl[(st * parts + q) * 3 * n + 3 * i + c];
      return v;
    };
    double acc = 0.0;
    for (int e = kptr[k]; e < kptr[k + 1]; ++e) {
      const int p = kpair[e] & 0xfffff, i = kpair[e] >> 20;
      const R* gp = g + (st * pairs + p) * 3;
      for (int c = 0; c < 3; ++c) acc += (double)gp[c] * bloch(i, c);
    }
    grad[(b * M + w0 + st - b * T) * K + k] = scale * loc_scaled<R>(acc, tau, amp, b, kptr[K + 1 + k]);
    if (!PH || !phase) continue;
    acc = 0.0;
    for (int i = 0; i < n; ++i) {
      const double w = ph.wz[k * n + i];
      if (w == 0.0) continue;
      const cplx<R>* a = ph.cs + st * ph.cs_step + i;
      const double c = 1.0 + (double)a->x, sx = (double)a->y, sy = ph.cs_step > n ? (double)a[n].x : 0.0;
      acc += w * (2.0 * (sx * sx + sy * sy) * bloch(i, 2) - 2.0 * c * (sx * bloch(i, 0) + sy * bloch(i, 1)));
    }
    ph.gphi[idx] = ph.scale * loc_scaled<R>(acc, tau, amp, b, 0);
  }
}

// Bloch sums over many parts, one block per step
template <typename R>
__global__ void __launch_bounds__(256) loc_sums_kernel(const R* __restrict__ bl, int parts, int nv,
                                                       double* __restrict__ sums) {
  __shared__ double s[8][32];
  const int v = threadIdx.x & 31, sl = threadIdx.x >> 5;
  const R* o = bl + (int64_t)blockIdx.x * parts * nv + v;
  double a = 0.0;
  if (v < nv)
    for (int p = sl; p < parts; p += 8) a += (double)o[(int64_t)p * nv];
  s[sl][v] = a;
  __syncthreads();
  if (sl == 0 && v < nv) {
    for (int i = 1; i < 8; ++i) a += s[i][v];
    sums[(int64_t)blockIdx.x * nv + v] = a;
  }
}

// gphi[b][n][k] = (2 / N^2) (Tz[n+1][k] - Tz[n][k]) (the traces already carry conj(tau))
template <typename R>
__global__ void loc_phase_kernel(const R* __restrict__ bz, int64_t B, int64_t M, int parts, int K, double scale,
                                 const double2* __restrict__ tau, double* __restrict__ gphi,
                                 const int32_t* __restrict__ gate) {
  if (gate && *gate != 0) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < B * M * K; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t bn = i / K, b = bn / M, n = bn - b * M;
    const int k = (int)(i - bn * K);
    double a = 0.0, c = 0.0;
    for (int p = 0; p < parts; ++p) {
      a += (double)bz[((b * (M + 1) + n) * parts + p) * K + k];
      c += (double)bz[((b * (M + 1) + n + 1) * parts + p) * K + k];
    }
    gphi[i] = scale * loc_scaled<R>(c - a, tau, nullptr, b, 0);
  }
}

template <typename R, int N, bool TWO>
static cudaError_t loc_sweep_n(const redo_table* t, const ChainPlan& p, int64_t B, const void* cs, const void* delta,
                               const void* Pck, const void* Rck, const double2* tau, void* bl, void* bz,
                               const int32_t* gate, cudaStream_t s) {
  if constexpr (sizeof(R) == 8 && N > 512) {
    return cudaErrorInvalidValue;                    // not eligible: two columns do not fit the registers
  } else {
  constexpr int E = loc_entries(sizeof(R) == 8, N, true);
  const int64_t fps = (int64_t)t->K * t->digits, chains = B * p.S, sps = p.seg_len / fps;
  const int64_t warps = (chains * N * (N / E) + 31) / 32;
  if (warps == 0) return cudaSuccess;
  auto kern = bz ? loc_sweep_kernel<R, N, E, true> : loc_sweep_kernel<R, N, E, false>;
  kern<<<(unsigned)((warps + 3) / 4), kLocThreads, 0, s>>>(
      (const cplx<R>*)cs, (const cplx<R>*)delta, p.M, p.S, sps, chains, (const cplx<R>*)Pck, (const cplx<R>*)Rck, tau,
      (R*)bl, t->K,
      sizeof(R) == 8 ? (const R*)t->sz64 : (const R*)t->sz32, (R*)bz, gate);
  return cudaGetLastError();
  }
}

template <typename R>
static cudaError_t loc_sweep_t(const redo_table* t, const ChainPlan& p, int64_t B, const void* cs, const void* delta,
                               const void* Pck, const void* Rck, const double2* tau, void* bl, void* bz,
                               const int32_t* gate, cudaStream_t s) {
  constexpr bool TWO = true;
  LOC_DISPATCH(loc_sweep_n, t, p, B, cs, delta, Pck, Rck, tau, bl, bz, gate, s)
}

// ============================================================================
// State sweeps: one column per pulse (Section IV observables, Section III state transfer).  The
// steps of a pulse are serial, so a column is spread over a whole warp (N >= 64) and the next step's
// diagonal and rotations are loaded while the present ones are applied; one warp per block, so that
// a few pulses reach as many SMs.
// ============================================================================
__host__ __device__ constexpr int loc_vec_entries(int N) { return N >= 64 ? N / 32 : 2; }
__host__ __device__ constexpr int loc_sim_entries(int N) { return N > 256 ? 8 : loc_vec_entries(N); }

// a + b exactly as s + e
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float z = s - a;
  e = (a - (s - z)) + (b - z);
}

// This lane's part of sum_r o_r |v_r|^2.  FP32 states keep the FP64 accumulation's accuracy in
// FP32 pairs (products split by fma, sums by two_sum): the FP64 pipe would take longer than the step.
template <int E> __device__ __forceinline__ float2 lane_expect(const float2 (&v)[E], const float2 (&o)[E]) {
  float acc = 0.f, lo = 0.f;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const float h = v[e].x * v[e].x, h2 = v[e].y * v[e].y;
    float s, er;
    two_sum(h, h2, s, er);
    const float l = (fmaf(v[e].x, v[e].x, -h) + fmaf(v[e].y, v[e].y, -h2)) + er;
    const float p = o[e].x * s;
    const float pl = fmaf(o[e].y, s, fmaf(o[e].x, l, fmaf(o[e].x, s, -p)));
    float t;
    two_sum(acc, p, t, er);
    acc = t;
    lo += er + pl;
  }
  return make_float2(acc, lo);
}
template <int E> __device__ __forceinline__ double2 lane_expect(const double2 (&v)[E], const double2 (&o)[E]) {
  double acc = 0.0;
#pragma unroll
  for (int e = 0; e < E; ++e) acc = fma(o[e].x, fma(v[e].x, v[e].x, v[e].y * v[e].y), acc);
  return make_double2(acc, 0.0);
}

// FP32 pairs serve observables and states whose products stay in FP32's range; others (a largest
// weight outside 2^-60 .. 2^60, or a largest entry of psi_0 outside 2^-60 .. 2^30) are summed in
// FP64, with the weights read again.  A pulse's flag tells loc_expect_kernel what its parts hold.  (The
// step loop stands once for each: with the choice inside, a step took 15 % longer.)
template <int E> __device__ __forceinline__ int2 lane_top(const double2* psi, const double* obs) {
  int2 t = make_int2(-200, -200);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    t.x = max(t.x, exp_of(obs[e]));
    t.y = max(t.y, exp_of(psi[e]));
  }
  return t;
}
__device__ __forceinline__ bool outside(int2 t) { return t.x < -60 || t.x > 60 || t.y < -60 || t.y > 30; }
template <int E> __device__ __forceinline__ float2 lane_expect_wide(const float2 (&v)[E], const double* obs) {
  double acc = 0.0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const double x = (double)v[e].x, y = (double)v[e].y;
    acc = fma(obs[e], fma(x, x, y * y), acc);
  }
  return make_float2(__int_as_float(__double2hiint(acc)), __int_as_float(__double2loint(acc)));
}
template <typename R, int E, bool FP64SUM>
__device__ __forceinline__ cplx<R> lane_part(const cplx<R> (&v)[E], const cplx<R> (&o)[E], const double* obs) {
  if constexpr (sizeof(R) == 4 && FP64SUM) return lane_expect_wide<E>(v, obs);
  else return lane_expect<E>(v, o);
}

// The same for N >= 512: a pulse per block of W warps, eight entries a lane (one warp would issue
// 2500 instructions a step, one after another).  The qubits of the warp index pair the same lanes of
// other warps through shared memory; two of them share one exchange, and the buffers alternate so
// that one barrier a step is enough.
template <typename R, int N, bool FP64SUM>
__device__ __forceinline__ void
loc_sim_wide_steps(cplx<R> (*ex)[8][N / 8], const cplx<R>* __restrict__ cs, const cplx<R>* __restrict__ delta, int64_t M,
                   const double2* __restrict__ psi0, int batched, const double* __restrict__ obs,
                   cplx<R>* __restrict__ part) {
  constexpr int E = 8, W = N / 256, LANES = 32 * W, NQ = Log2<N>::v;
  using L = LocCol<R, 256, E>;                       // the qubits within a warp
  const int lane = threadIdx.x & 31, l = threadIdx.x, wp = threadIdx.x >> 5;
  const int64_t b = blockIdx.x;
  const cplx<R>* d = delta + b * (M + 1) * N;
  const cplx<R>* r = cs + b * M * NQ;
  cplx<R>* o = part + b * (M + 1) * LANES + l;
  cplx<R> v[E], w[E], dn[E], cn[NQ];
  auto load = [&](int64_t m) {
#pragma unroll
    for (int e = 0; e < E; e += 2) {
      const cplx<R>* p = d + m * N + ((e >> 1) * LANES + l) * 2;
      if constexpr (sizeof(R) == 4) {
        const float4 q = __ldg(reinterpret_cast<const float4*>(p));
        dn[e] = make_float2(q.x, q.y);
        dn[e + 1] = make_float2(q.z, q.w);
      } else {
        dn[e] = __ldg(p);
        dn[e + 1] = __ldg(p + 1);
      }
    }
#pragma unroll
    for (int i = 0; i < NQ; ++i) cn[i] = __ldg(r + m * NQ + i);
  };
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const double2 z = psi0[(batched ? b * N : 0) + l * E + e];
    v[e] = cmake<R>((R)z.x, (R)z.y);
    const double ov = obs[l * E + e];
    w[e] = cmake<R>((R)ov, (R)(ov - (double)(R)ov));
  }
  o[0] = lane_part<R, E, FP64SUM>(v, w, obs + l * E);
  if (M > 0) load(0);
#pragma unroll 1
  for (int64_t m = 0; m < M; ++m) {
    cplx<R> c[L::NQ];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = plus_mul<R>(v[e], dn[e]);
#pragma unroll
    for (int i = 0; i < L::NQ; ++i) c[i] = cn[i];
    const cplx<R> c8 = cn[8], c9 = cn[NQ - 1];
    load(m + 1 < M ? m + 1 : m);
    L::rotate(v, c, lane);
    cplx<R>(*x)[LANES] = ex[m & 1];
#pragma unroll
    for (int e = 0; e < E; ++e) x[e][l] = v[e];
    __syncthreads();
    const R s8 = (wp & 1) ? c8.y : -c8.y;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      v[e] = rot_one<R, false>(v[e], x[e][l ^ 32], c8.x, s8, R(0));
      if constexpr (W == 4) {
        const cplx<R> p = rot_one<R, false>(x[e][l ^ 64], x[e][l ^ 96], c8.x, s8, R(0));
        v[e] = rot_one<R, false>(v[e], p, c9.x, (wp & 2) ? c9.y : -c9.y, R(0));
      }
    }
    o[(m + 1) * LANES] = lane_part<R, E, FP64SUM>(v, w, obs + l * E);
  }
}
template <typename R, int N>
__global__ void __launch_bounds__(N / 8)
loc_sim_wide_kernel(const cplx<R>* __restrict__ cs, const cplx<R>* __restrict__ delta, int64_t M,
                    const double2* __restrict__ psi0, int batched, const double* __restrict__ obs,
                    cplx<R>* __restrict__ part, int32_t* __restrict__ flags) {
  constexpr int E = 8;
  __shared__ cplx<R> ex[2][E][N / 8];
  if constexpr (sizeof(R) == 4) {
    const int l = threadIdx.x;
    const int2 t = lane_top<E>(psi0 + (batched ? (int64_t)blockIdx.x * N : 0) + l * E, obs + l * E);
    int* top = reinterpret_cast<int*>(ex);           // (free until the first step)
    if (l == 0) top[0] = top[1] = -200;
    __syncthreads();
    const int x = __reduce_max_sync(0xffffffffu, t.x), y = __reduce_max_sync(0xffffffffu, t.y);
    if ((l & 31) == 0) {
      atomicMax(top, x);
      atomicMax(top + 1, y);
    }
    __syncthreads();
    const bool far = outside(make_int2(top[0], top[1]));
    __syncthreads();
    if (l == 0) flags[blockIdx.x] = far;
    if (far) return loc_sim_wide_steps<R, N, true>(ex, cs, delta, M, psi0, batched, obs, part);
  }
  loc_sim_wide_steps<R, N, false>(ex, cs, delta, M, psi0, batched, obs, part);
}

// part[b][n][l]: lane l's part of <O> after n steps
template <typename R, int N, bool FP64SUM>
__device__ __forceinline__ void
loc_sim_steps(const cplx<R>* __restrict__ cs, const cplx<R>* __restrict__ delta, int64_t B, int64_t M,
              const double2* __restrict__ psi0, int batched, const double* __restrict__ obs, cplx<R>* __restrict__ part) {
  constexpr int E = loc_vec_entries(N);
  using L = LocCol<R, N, E>;
  const int lane = threadIdx.x, l = lane / L::C;
  const int64_t b_raw = (int64_t)blockIdx.x * L::C + lane % L::C;
  const bool on = b_raw < B;
  const int64_t b = on ? b_raw : B - 1;              // idle lanes follow the last pulse, write nothing
  const cplx<R>* d = delta + b * (M + 1) * N;
  const cplx<R>* r = cs + b * M * L::CS;
  cplx<R>* o = part + b * (M + 1) * L::G + l;
  cplx<R> v[E], w[E], dn[E], cn[L::CS];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const double2 z = psi0[(batched ? b * N : 0) + l * E + e];
    v[e] = cmake<R>((R)z.x, (R)z.y);
    const double ov = obs[l * E + e];
    w[e] = cmake<R>((R)ov, (R)(ov - (double)(R)ov));
  }
  cplx<R> a = lane_part<R, E, FP64SUM>(v, w, obs + l * E);
  if (on) o[0] = a;
  if (M > 0) {
    L::load_diag(dn, d, l);
    L::load_cs(cn, r);
  }
#pragma unroll 1
  for (int64_t m = 0; m < M; ++m) {
    cplx<R> c[L::CS];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = plus_mul<R, L::NEAR>(v[e], dn[e]);
#pragma unroll
    for (int i = 0; i < L::CS; ++i) c[i] = cn[i];
    const int64_t nx = m + 1 < M ? m + 1 : m;
    L::load_diag(dn, d + nx * N, l);
    L::load_cs(cn, r + nx * L::CS);
    L::rotate(v, c, l);
    a = lane_part<R, E, FP64SUM>(v, w, obs + l * E); // |v|^2: the trailing phases do not enter
    if (on) o[(m + 1) * L::G] = a;
  }
}
// A warp's pulses are summed alike; each one's flag is the warp's.
template <typename R, int N>
__global__ void __launch_bounds__(32)
loc_sim_kernel(const cplx<R>* __restrict__ cs, const cplx<R>* __restrict__ delta, int64_t B, int64_t M,
               const double2* __restrict__ psi0, int batched, const double* __restrict__ obs, cplx<R>* __restrict__ part,
               int32_t* __restrict__ flags) {
  constexpr int E = loc_vec_entries(N);
  using L = LocCol<R, N, E>;
  if constexpr (sizeof(R) == 4) {
    const int lane = threadIdx.x, l = lane / L::C;
    const int64_t b_raw = (int64_t)blockIdx.x * L::C + lane % L::C, b = b_raw < B ? b_raw : B - 1;
    int2 t = lane_top<E>(psi0 + (batched ? b * N : 0) + l * E, obs + l * E);
#pragma unroll
    for (int off = L::C; off < 32; off *= 2)
      t = make_int2(max(t.x, __shfl_xor_sync(0xffffffffu, t.x, off)), max(t.y, __shfl_xor_sync(0xffffffffu, t.y, off)));
    const bool far = __any_sync(0xffffffffu, outside(t));
    if (b_raw < B && l == 0) flags[b] = far;
    if (far) return loc_sim_steps<R, N, true>(cs, delta, B, M, psi0, batched, obs, part);
  }
  loc_sim_steps<R, N, false>(cs, delta, B, M, psi0, batched, obs, part);
}

// expect[i] = sum of its G parts, min(G, 32) lanes an item (per items a pulse)
template <typename R>
__global__ void loc_expect_kernel(const cplx<R>* __restrict__ part, int64_t n, int64_t items, int G,
                                  const int32_t* __restrict__ flags, double* __restrict__ expect) {
  const int w = G < 32 ? G : 32, l = threadIdx.x % w;
  const int64_t per = blockDim.x / w;
  for (int64_t i0 = blockIdx.x * per; i0 < n; i0 += gridDim.x * per) {
    const int64_t i = i0 + threadIdx.x / w;
    double a = 0.0;
    // (a slice's parts are 8 bytes or more of 512 MiB, so i and items hold in 32 bits)
    const bool wide = sizeof(R) == 4 && i < n && flags[(uint32_t)i / (uint32_t)items] != 0;
    for (int q = l; q < G && i < n; q += w) {
      const cplx<R> p = part[i * G + q];
      if constexpr (sizeof(R) == 4)
        a += wide ? __hiloint2double(__float_as_int(p.x), __float_as_int(p.y)) : (double)p.x + (double)p.y;
      else
        a += p.x;
    }
    for (int off = w / 2; off >= 1; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    if (l == 0 && i < n) expect[i] = a;
  }
}

// F_S = |<psi_T|U|psi_0>|^2 and the Bloch sums of its gradient: forward over the steps, then back
// with the state undone and the costate <psi_T| U_M ... carried along (trace_undo).  One launch
// covers the steps [m0, m0 + T): forward (fwd), at the chain's end the overlap, and back (back);
// between launches both vectors rest in st[b][2][N].  FP32 vectors are scaled by powers of two (psi_0
// to entries near 1, the costate likewise), whose product goes to amp[b] for the gradient.
template <typename R, int N>
__global__ void __launch_bounds__(32)
loc_state_kernel(const cplx<R>* __restrict__ cs, const cplx<R>* __restrict__ delta, int64_t B, int64_t M, int64_t m0,
                 int64_t T, int fwd, int back, const double2* __restrict__ psi0, const double2* __restrict__ psiT,
                 int batched, double* __restrict__ F_out, R* __restrict__ bl, cplx<R>* __restrict__ st,
                 double* __restrict__ amp) {
  constexpr int E = loc_vec_entries(N);
  using L = LocCol<R, N, E>;
  using WS = WarpSums<R, 3 * L::NQ>;
  const int lane = threadIdx.x, l = lane / L::C;
  const int64_t b_raw = (int64_t)blockIdx.x * L::C + lane % L::C;
  const bool on = b_raw < B;
  const int64_t b = on ? b_raw : B - 1;              // idle lanes follow the last pulse, write nothing
  const cplx<R>* d = delta + b * (T + 1) * N;
  const cplx<R>* r = cs + b * T * L::CS;
  cplx<R>* sp = st + b * 2 * N + l * E;
  cplx<R> p[E], w[E], dn[E], cn[L::CS];
  // exponent of the largest entry of a vector (this lane's E entries at v)
  auto top = [&](const double2* v) -> int {
    int x = -200;
#pragma unroll
    for (int e = 0; e < E; ++e) x = max(x, exp_of(v[e]));
    if constexpr (L::C == 1) return __reduce_max_sync(0xffffffffu, x);
#pragma unroll
    for (int off = L::C; off < 32; off *= 2) x = max(x, __shfl_xor_sync(0xffffffffu, x, off));
    return x;
  };
  const double2 *z0 = psi0 + (batched ? b * N : 0) + l * E, *zT = psiT + (batched ? b * N : 0) + l * E;
  const int e0 = sizeof(R) == 4 && fwd ? top(z0) : 0;
  if (fwd) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const double2 z = m0 == 0 ? z0[e] : make_double2(0.0, 0.0);
      p[e] = m0 == 0 ? cmake<R>((R)down2(z.x, e0), (R)down2(z.y, e0)) : sp[e];
    }
    L::load_diag(dn, d, l);
    if (T > 0) L::load_cs(cn, r);
#pragma unroll 1
    for (int64_t m = 0; m < T; ++m) {
      cplx<R> c[L::CS];
#pragma unroll
      for (int e = 0; e < E; ++e) p[e] = plus_mul<R, L::NEAR>(p[e], dn[e]);
#pragma unroll
      for (int i = 0; i < L::CS; ++i) c[i] = cn[i];
      L::load_diag(dn, d + (m + 1) * N, l);          // the last one read is the window's closing diagonal
      if (m + 1 < T) L::load_cs(cn, r + (m + 1) * L::CS);
      L::rotate(p, c, l);
    }
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      p[e] = sp[e];
      w[e] = sp[N + e];
    }
  }
  if (fwd && m0 + T == M) {
    double tx = 0.0, ty = 0.0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const double2 z = zT[e];
      const cplx<R> u = plus_mul<R, L::NEAR>(p[e], dn[e]);
      tx = fma(z.x, (double)u.x, tx); tx = fma(z.y, (double)u.y, tx);
      ty = fma(z.x, (double)u.y, ty); ty = fma(-z.y, (double)u.x, ty);
    }
#pragma unroll
    for (int off = L::C; off < 32; off *= 2) {
      tx += __shfl_xor_sync(0xffffffffu, tx, off);
      ty += __shfl_xor_sync(0xffffffffu, ty, off);
    }
    if (F_out && on && l == 0) {
      const double x = down2(tx, -e0), y = down2(ty, -e0);
      F_out[b] = x * x + y * y;
    }
    if constexpr (sizeof(R) == 4) {
      const int eT = top(zT), et = exp_of(make_double2(tx, ty));
      tx = down2(tx, eT + et);
      ty = down2(ty, eT + et);
      if (on && l == 0) amp[b] = pow2(2 * e0 + eT + et);
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
      // conj(psi_T) conj(tau), then the closing diagonal
      const double2 z = zT[e];
      w[e] = plus_mul<R, L::NEAR>(cmake<R>((R)(z.x * tx - z.y * ty), (R)(-z.y * tx - z.x * ty)), dn[e]);
    }
  }
  if (back && T > 0) {
    L::load_diag(dn, d + (T - 1) * N, l);
    L::load_cs(cn, r + (T - 1) * L::CS);
#pragma unroll 1
    for (int64_t m = T - 1; m >= 0; --m) {
      cplx<R> c[L::CS], dc[E];
#pragma unroll
      for (int e = 0; e < E; ++e) dc[e] = dn[e];
#pragma unroll
      for (int i = 0; i < L::CS; ++i) c[i] = cn[i];
      const int64_t nx = m > 0 ? m - 1 : 0;
      L::load_diag(dn, d + nx * N, l);
      L::load_cs(cn, r + nx * L::CS);
      R v[WS::P];
#pragma unroll
      for (int i = 0; i < WS::P; ++i) v[i] = R(0);
      L::trace_undo(p, w, c, l, v);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        p[e] = plus_mul_conj<R, L::NEAR>(p[e], dc[e]);
        w[e] = plus_mul<R, L::NEAR>(w[e], dc[e]);
      }
      R* o = bl + (b * T + m) * (3 * L::NQ);
      if constexpr (L::G == 32) {
        const int idx = WS::full(v, lane);
        if (on && idx >= 0) o[idx] = v[0];
      } else {
#pragma unroll
        for (int i = 0; i < 3 * L::NQ; ++i) {
#pragma unroll
          for (int off = L::C; off < 32; off *= 2) v[i] += __shfl_xor_sync(0xffffffffu, v[i], off);
          if (on && l == 0) o[i] = v[i];
        }
      }
    }
  }
  if (on && T < M) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      sp[e] = p[e];
      if (!fwd || back) sp[N + e] = w[e];
    }
  }
}

// ============================================================================
// Host side: step-operator scratch in slices of pulses, plans, launches
// ============================================================================
// A slice holds the rotations and diagonals of as many pulses as fit kLocSlice bytes, so that long
// batches need bounded scratch; a pulse that does not fit alone keeps the dense path.
constexpr size_t kLocSlice = (size_t)512 << 20;

static size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// parts of the Bloch sums of one step: the warps of a chain
static int loc_parts(const redo_table* t, bool dbl) {
  const int lanes = t->N * (t->N / loc_entries(dbl, t->N, true));
  return lanes >= 32 ? lanes / 32 : 1;
}

// Scratch of nb pulses: diagonals and rotations, then by what is computed (LocalWhat) the Bloch
// sums, the boundary traces or the lanes' parts of the observable.
struct LocScratch {
  void *delta, *cs, *bl, *bz, *g;
  int32_t* flags;                                    // [pulses], observables only
  double* sums;
  size_t total;
};
constexpr size_t kLocSumParts = 8;                   // from here on the parts are added by a kernel of their own
static bool loc_near_of(const redo_table* t, bool dbl, int what) { return what == kLocalChainFine || loc_near(dbl, t->N); }
static LocScratch loc_scratch(const redo_table* t, int64_t nb, int64_t M, int prec, int what, void* base) {
  const size_t el = prec == REDO_FP64 ? sizeof(double) : sizeof(float);
  const bool grad = what == kLocalGrad || what == kLocalPhaseGrad;
  const size_t parts = grad ? (size_t)loc_parts(t, prec == REDO_FP64) : 1;
  const size_t lanes = what == kLocalSim ? (size_t)(t->N / loc_sim_entries(t->N)) : 0;
  LocScratch w;
  char* c = (char*)base;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    void* at = c + off;
    off += up256(bytes);
    return at;
  };
  w.delta = take((size_t)nb * (M + 1) * t->N * 2 * el);
  w.cs = take((size_t)nb * M * t->loc * 2 * el * (loc_near_of(t, prec == REDO_FP64, what) ? 2 : 1));
  w.bl = take(grad ? (size_t)nb * M * parts * 3 * t->loc * el : (size_t)nb * (M + 1) * lanes * 2 * el);
  w.bz = take(what == kLocalPhaseGrad ? (size_t)nb * (M + 1) * parts * t->K * el : 0);
  w.g = grad ? take((size_t)nb * M * t->loc_pairs * 3 * el) : nullptr;
  w.sums = grad && parts >= kLocSumParts ? (double*)take((size_t)nb * M * 3 * t->loc * sizeof(double)) : nullptr;
  w.flags = what == kLocalSim ? (int32_t*)take((size_t)nb * sizeof(int32_t)) : nullptr;
  w.total = off;
  return w;
}

bool local_eligible(const redo_table* t, int64_t M, int prec, int what) {
  if (t->loc == 0) return false;
  if ((what == kLocalGrad || what == kLocalPhaseGrad) && prec == REDO_FP64 && t->N > 512) return false;
  return loc_scratch(t, 1, M, prec, what, nullptr).total <= kLocSlice;
}

// Whether a call gains by it (systems of a few levels; the others always do).  Multiply-adds of a step:
// dense 4 N^3 (a state: 4 N^2) K digits; here 32 a pair, per qubit 230 FP64 operations of square roots
// and divisions (FP32: 500, three angles), 28 a row for the diagonal (FP32: 100, a sine and cosine), and
// 4 + 4n an entry (complex rotations: 6 + 8n).
// FP64, by measurement over B = 1 .. 3000, N = 2 .. 16: while the pulses leave SMs idle a call waits for
// its dependent products and this form is ahead from N = 4 on (N = 4, two controls, 40 x 200: 158 us dense,
// 101 here) and level at N = 2; once they fill the GPU its serial one-qubit work runs at half the rate of
// the dense columns (N = 4, 300 x 100: 126 us dense, 195 here).  A state's dense factors take about 1 us
// each, one after another, its step here 2.5 to 3.5 (300 x 100, N = 4: one control 224 us dense, 265 here,
// two 381 and 258; N = 8: 261 and 351, 435 and 345; N = 16: always ahead).
// FP32: the dense column kernel is bound by its operand reads at about two thirds of this path's rate
// (N = 4, global controls, 1000 x 500: 155 us dense, 234 us here; N = 8: 528 and 315), so plain
// propagations at N = 2, and at N = 4 and 8 with few factors, stay dense; with a step-opening diagonal, for
// gradients and for states this form is level or ahead at every size, and several times more exact.
bool local_pays(const redo_table* t, int64_t B, int prec, int what, bool diag) {
  const double N = t->N, n = t->loc, kd = (double)t->K * t->digits;
  const bool dbl = prec == REDO_FP64, full = B >= t->num_sms;
  const double prep = dbl ? 32.0 * t->loc_pairs + 230.0 * n + 28.0 * N : 40.0 * t->loc_pairs + 500.0 * n + 100.0 * N;
  const double rot = loc_near(dbl, t->N) ? 6 + 8 * n : 4 + 4 * n;
  if (what == kLocalSim) return !dbl || !full || N > 8 || kd > 2;
  if (what == kLocalGrad) return !dbl || diag || N > 2 || !full;
  if (what == kLocalPhaseGrad) return true;
  const double dense = 4.0 * N * N * N * kd + (diag ? 4.0 * N * N : 0.0), here = prep + N * N * rot;
  if (dbl) return N > 2 && (!full || dense > 2.0 * here);
  return diag || 1.5 * dense > here;
}

// Which chain form a call takes.  FP32 products of controls that act on one qubit each have two nonzeros
// a row, so the dense chain rounds twice a product, and the real rotations' error was up to 1.4 times its
// (U, N = 64, 12 controls, 200 steps: 7.9e-7 dense, 1.0e-6); rotations near the identity, twice the
// multiply-adds, give 4.4e-7 (N = 32: 6.3e-7, 9.1e-7, 3.6e-7; N = 128: 5.1e-7, 6.6e-7, 3.1e-7).  256 x
// 2000 at N = 64, re-unitarised: 3.82 ms with the real rotations, 4.96 here, 232 dense.  Split
// FP16 was 5 times less exact (5.5e-6) and takes the real rotations; controls on several qubits at once
// (global fields) have dense rows, whose error was larger (N = 64: 1.7e-6, 1.0e-6 with the real rotations).
int local_chain_form(const redo_table* t, int prec_asked) {
  return prec_asked == REDO_FP32 && t->loc_pairs <= t->K && t->N > 16 ? kLocalChainFine : kLocalChain;
}

static int64_t local_slice(const redo_table* t, int64_t B, int64_t M, int prec, int what) {
  const int64_t n = (int64_t)(kLocSlice / loc_scratch(t, 1, M, prec, what, nullptr).total);
  return n < B ? n : B;
}

size_t local_ops_bytes(const redo_table* t, int64_t B, int64_t M, int prec, int what) {
  return loc_scratch(t, local_slice(t, B, M, prec, what), M, prec, what, nullptr).total;
}

// Segments of whole steps.  Columns of one pulse are independent, so time is cut only as far as the
// columns leave the GPU's schedulers idle (about four warps each), and not below 8 steps: every
// further segment costs a dense product when the segments are multiplied.
ChainPlan plan_chain_local(const redo_table* t, int64_t B, int64_t M, int prec, bool two) {
  const bool dbl = prec == REDO_FP64;
  const int E = loc_entries(dbl, t->N, two);
  const int64_t warps = (B * t->N * (t->N / E) + 31) / 32;
  int64_t S = warps > 0 ? (4 * 4 * (int64_t)t->num_sms + warps - 1) / warps : 1;
  const int64_t min_steps = t->N <= 8 ? 4 : (t->N <= 64 ? 8 : 32);
  if (S > M / min_steps) S = M / min_steps;
  // M / S dependent steps, then 2 sqrt(S) dependent products when the segments are multiplied (in
  // groups): best near S = (M / r)^(2/3), r the time of a product beside that of a step.  One pulse,
  // M = 1e5, N = 8: FP64 2.7 ms with 64 segments, 0.57 ms with 1024 (dense plan 3.1 ms); FP32 3.8 ms with
  // 16, 0.17 ms with 1024 (dense 0.77).  r as measured over M = 500 .. 1e5 (N = 64 FP64: 64 segments are
  // best at every length).  Short FP32 pulses of N <= 16 stay with one combine pass.
  const double r = t->N <= 16 ? 1.0 : (t->N == 32 ? 2.0 : (dbl ? 16.0 : 6.0));
  int64_t most = (int64_t)std::cbrt(((double)M / r) * ((double)M / r));
  if (most > 1024) most = 1024;
  const int64_t least = !dbl && t->N <= 16 ? 16 : 64;
  if (most < least || M < 400) most = least;
  if (S > most) S = most;
  if (S < 1) S = 1;
  return plan_chain_aligned(t, B, M, M > 0 ? (M + S - 1) / S : 1);
}

template <typename R>
static cudaError_t loc_steps_t(const redo_table* t, const int32_t* q, int64_t B, int64_t M, int64_t m0, int64_t T, int E,
                               bool near, const LocalDiag& pd, int64_t b0, const LocScratch& w, int64_t* status,
                               cudaStream_t s) {
  const int ts = B * (T + 1) >= (int64_t)t->num_sms * 8 * kPrepSteps ? kPrepSteps : 8;
  const int64_t tiles = (T + 1 + ts - 1) / ts;
  auto kern = loc_steps_kernel<R, false>;
  if constexpr (sizeof(R) == 4)
    if (near) kern = loc_steps_kernel<R, true>;
  kern<<<(unsigned)(B * tiles), kPrepThreads, 0, s>>>(
      loc_tab<R>(t, status), q + b0 * M * t->K, M, m0, T, t->loc, t->N, E, tiles, ts,
      sizeof(R) == 8 ? (const typename DiagOf<R>::T*)t->loc_D64 : (const typename DiagOf<R>::T*)t->loc_D32,
      pd.p ? pd.p + b0 * pd.sb : nullptr, pd.sb, pd.sn, (cplx<R>*)w.cs,
      (cplx<R>*)w.delta, sizeof(R) == 8 ? (const cplx<R>*)t->loc_h : (const cplx<R>*)t->loc_h32, t->loc_pairs, (R*)w.g);
  return cudaGetLastError();
}

static cudaError_t loc_steps(const redo_table* t, const int32_t* q, int64_t nb, int64_t M, int prec, int what, int E,
                             const LocalDiag& pd, int64_t b0, const LocScratch& w, int64_t* status, cudaStream_t s) {
  const bool near = loc_near_of(t, prec == REDO_FP64, what);
  return prec == REDO_FP64 ? loc_steps_t<double>(t, q, nb, M, 0, M, E, near, pd, b0, w, status, s)
                           : loc_steps_t<float>(t, q, nb, M, 0, M, E, near, pd, b0, w, status, s);
}

cudaError_t launch_local_chain(const redo_table* t, const int32_t* q, const ChainPlan& p, int prec, int what,
                               const LocalDiag& pd, void* ops, void* seg_out, int64_t* status, cudaStream_t s) {
  const bool dbl = prec == REDO_FP64, two = what == kLocalGrad || what == kLocalPhaseGrad;
  const bool near = loc_near_of(t, dbl, what);
  const int64_t slice = local_slice(t, p.B, p.M, prec, what);
  const LocScratch w = loc_scratch(t, slice, p.M, prec, what, ops);
  const int E = loc_entries(dbl, t->N, two);
  const size_t mat = (size_t)t->N * t->N * (dbl ? sizeof(double2) : sizeof(float2));
  for (int64_t b0 = 0; b0 < p.B; b0 += slice) {
    const int64_t nb = b0 + slice < p.B ? slice : p.B - b0;
    cudaError_t e = loc_steps(t, q, nb, p.M, prec, what, E, pd, b0, w, status, s);
    if (e) return e;
    void* out = (char*)seg_out + (size_t)(b0 * p.S) * mat;
    e = dbl ? (two ? loc_chain_t<double, true>(t, p, nb, near, w.cs, w.delta, out, s)
                   : loc_chain_t<double, false>(t, p, nb, near, w.cs, w.delta, out, s))
            : (two ? loc_chain_t<float, true>(t, p, nb, near, w.cs, w.delta, out, s)
                   : loc_chain_t<float, false>(t, p, nb, near, w.cs, w.delta, out, s));
    if (e) return e;
  }
  return cudaSuccess;
}

// Which form of the phase gradient a call launches.  The axes in force decide; a captured call is
// replayed with the axes set by then, so it holds both forms behind the table's device flag (gate).
struct PhaseForm {
  bool sums = true, boundary = false;
  const int32_t* gate = nullptr;
};
static PhaseForm phase_form(const redo_table* t, cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  PhaseForm f;
  if (cudaStreamIsCapturing(s, &st) == cudaSuccess && st == cudaStreamCaptureStatusNone) {
    f.sums = t->wz_local != 0;
    f.boundary = !f.sums;
  } else {
    f.boundary = true;
    f.gate = t->wz_on;
  }
  return f;
}

template <typename R>
static cudaError_t loc_finish_t(const redo_table* t, int64_t B, int64_t M, int64_t m0, int64_t T, int parts, double norm,
                                const LocScratch& w, double* grad, double* gphi, const PhaseForm& f,
                                const double2* tau, const double* amp, cudaStream_t s) {
  const int64_t steps = B * T, gn = steps * t->K, gb = (gn + 127) / 128;
  if (w.sums)
    loc_sums_kernel<R><<<(unsigned)steps, 256, 0, s>>>((const R*)w.bl, parts, 3 * t->loc, w.sums);
  auto kern = gphi && f.sums ? loc_grad_kernel<R, true> : loc_grad_kernel<R, false>;
  kern<<<(unsigned)(gb < 16384 ? gb : 16384), 128, 0, s>>>(
      steps, t->K, t->loc, t->loc_pairs, parts, t->loc_kptr, t->loc_kpair, (const R*)w.g, (const R*)w.bl, w.sums, M, m0,
      T, 2.0 * t->dt / norm, tau, amp, grad,
      LocPhaseOut<R>{(const cplx<R>*)w.cs, t->wz, f.gate, 2.0 / norm, gphi,
                     t->loc * (loc_near(sizeof(R) == 8, t->N) ? 2 : 1)});
  if (gphi && f.boundary) {
    const int64_t n = B * M * t->K, blocks = (n + 255) / 256;
    loc_phase_kernel<R><<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, s>>>((const R*)w.bz, B, M, parts, t->K,
                                                                                  2.0 / norm, tau, gphi, f.gate);
  }
  return cudaGetLastError();
}

// Reverse sweep and gradients of all pulses (what = 2: also the phase gradients gphi).  With more
// than one slice the step operators, overwritten by the later slices, are formed again.
cudaError_t launch_local_grad(const redo_table* t, const int32_t* q, const ChainPlan& p, int prec, int what,
                              const LocalDiag& pd, void* ops, const void* Pck, const void* Rck, const double2* tau,
                              double* grad, double* gphi, int64_t* status, cudaStream_t s) {
  const bool dbl = prec == REDO_FP64;
  const int64_t slice = local_slice(t, p.B, p.M, prec, what);
  const LocScratch w = loc_scratch(t, slice, p.M, prec, what, ops);
  const int E = loc_entries(dbl, t->N, true), parts = loc_parts(t, dbl);
  const size_t mat = (size_t)t->N * t->N * (dbl ? sizeof(double2) : sizeof(float2));
  const double norm = (double)t->N * (double)t->N;
  const PhaseForm f = what == kLocalPhaseGrad ? phase_form(t, s) : PhaseForm{};
  for (int64_t b0 = 0; b0 < p.B; b0 += slice) {
    const int64_t nb = b0 + slice < p.B ? slice : p.B - b0;
    cudaError_t e = cudaSuccess;
    if (slice < p.B && (e = loc_steps(t, q, nb, p.M, prec, what, E, pd, b0, w, status, s))) return e;
    const char* P = (const char*)Pck + (size_t)(b0 * p.S) * mat;
    const char* Q = (const char*)Rck + (size_t)(b0 * p.S) * mat;
    for (int tz = 0; tz < 2; ++tz) {
      if (!(tz ? f.boundary : f.sums)) continue;
      void* bz = tz ? w.bz : nullptr;
      e = dbl ? loc_sweep_t<double>(t, p, nb, w.cs, w.delta, P, Q, tau + b0, w.bl, bz, f.gate, s)
              : loc_sweep_t<float>(t, p, nb, w.cs, w.delta, P, Q, tau + b0, w.bl, bz, f.gate, s);
      if (e) return e;
    }
    const int64_t at = b0 * p.M * t->K;
    double* gp = gphi ? gphi + at : nullptr;
    e = dbl ? loc_finish_t<double>(t, nb, p.M, 0, p.M, parts, norm, w, grad + at, gp, f, tau + b0, nullptr, s)
            : loc_finish_t<float>(t, nb, p.M, 0, p.M, parts, norm, w, grad + at, gp, f, tau + b0, nullptr, s);
    if (e) return e;
  }
  return cudaSuccess;
}

#define LOC_VEC(KERNEL, ...)                                                       \
  switch (t->N) {                                                                 \
    case 2: KERNEL<R, 2><<<blocks, 32, 0, s>>>(__VA_ARGS__); break;               \
    case 4: KERNEL<R, 4><<<blocks, 32, 0, s>>>(__VA_ARGS__); break;               \
    case 8: KERNEL<R, 8><<<blocks, 32, 0, s>>>(__VA_ARGS__); break;               \
    case 16: KERNEL<R, 16><<<blocks, 32, 0, s>>>(__VA_ARGS__); break;             \
    case 32: KERNEL<R, 32><<<blocks, 32, 0, s>>>(__VA_ARGS__); break;             \
    case 64: KERNEL<R, 64><<<blocks, 32, 0, s>>>(__VA_ARGS__); break;             \
    case 128: KERNEL<R, 128><<<blocks, 32, 0, s>>>(__VA_ARGS__); break;           \
    case 256: KERNEL<R, 256><<<blocks, 32, 0, s>>>(__VA_ARGS__); break;           \
    case 512: KERNEL<R, 512><<<blocks, 32, 0, s>>>(__VA_ARGS__); break;           \
    case 1024: KERNEL<R, 1024><<<blocks, 32, 0, s>>>(__VA_ARGS__); break;         \
    default: return cudaErrorInvalidValue;                                        \
  }

template <typename R>
static cudaError_t loc_sim_t(const redo_table* t, int64_t B, int64_t M, const double2* psi0, int batched,
                             const double* obs, const LocScratch& w, double* expect, cudaStream_t s) {
  const int lanes = t->N / loc_sim_entries(t->N), cols = lanes < 32 ? 32 / lanes : 1;
  const unsigned blocks = (unsigned)((B + cols - 1) / cols);
  const cplx<R>*cs = (const cplx<R>*)w.cs, *delta = (const cplx<R>*)w.delta;
  cplx<R>* part = (cplx<R>*)w.bl;
  switch (t->N) {
    case 2: loc_sim_kernel<R, 2><<<blocks, 32, 0, s>>>(cs, delta, B, M, psi0, batched, obs, part, w.flags); break;
    case 4: loc_sim_kernel<R, 4><<<blocks, 32, 0, s>>>(cs, delta, B, M, psi0, batched, obs, part, w.flags); break;
    case 8: loc_sim_kernel<R, 8><<<blocks, 32, 0, s>>>(cs, delta, B, M, psi0, batched, obs, part, w.flags); break;
    case 16: loc_sim_kernel<R, 16><<<blocks, 32, 0, s>>>(cs, delta, B, M, psi0, batched, obs, part, w.flags); break;
    case 32: loc_sim_kernel<R, 32><<<blocks, 32, 0, s>>>(cs, delta, B, M, psi0, batched, obs, part, w.flags); break;
    case 64: loc_sim_kernel<R, 64><<<blocks, 32, 0, s>>>(cs, delta, B, M, psi0, batched, obs, part, w.flags); break;
    case 128: loc_sim_kernel<R, 128><<<blocks, 32, 0, s>>>(cs, delta, B, M, psi0, batched, obs, part, w.flags); break;
    case 256: loc_sim_kernel<R, 256><<<blocks, 32, 0, s>>>(cs, delta, B, M, psi0, batched, obs, part, w.flags); break;
    case 512: loc_sim_wide_kernel<R, 512><<<blocks, 64, 0, s>>>(cs, delta, M, psi0, batched, obs, part, w.flags); break;
    case 1024: loc_sim_wide_kernel<R, 1024><<<blocks, 128, 0, s>>>(cs, delta, M, psi0, batched, obs, part, w.flags); break;
    default: return cudaErrorInvalidValue;
  }
  const int64_t n = B * (M + 1), per = 128 / (lanes < 32 ? lanes : 32), nb = (n + per - 1) / per;
  loc_expect_kernel<R><<<(unsigned)(nb < 4096 ? nb : 4096), 128, 0, s>>>((const cplx<R>*)w.bl, n, M + 1, lanes,
                                                                     w.flags, expect);
  return cudaGetLastError();
}

cudaError_t launch_local_sim(const redo_table* t, const int32_t* q, int64_t B, int64_t M, int prec, const double2* psi0,
                             int batched, const double* obs, double* expect, void* ops, int64_t* status, cudaStream_t s) {
  const int64_t slice = local_slice(t, B, M, prec, kLocalSim);
  const LocScratch w = loc_scratch(t, slice, M, prec, kLocalSim, ops);
  for (int64_t b0 = 0; b0 < B; b0 += slice) {
    const int64_t nb = b0 + slice < B ? slice : B - b0;
    cudaError_t e = loc_steps(t, q, nb, M, prec, kLocalSim, loc_sim_entries(t->N), LocalDiag{nullptr, 0, 0}, b0, w,
                              status, s);
    if (e) return e;
    const double2* p0 = psi0 + (batched ? b0 * t->N : 0);
    double* ex = expect + b0 * (M + 1);
    e = prec == REDO_FP64 ? loc_sim_t<double>(t, nb, M, p0, batched, obs, w, ex, s)
                          : loc_sim_t<float>(t, nb, M, p0, batched, obs, w, ex, s);
    if (e) return e;
  }
  return cudaSuccess;
}

// State-transfer scratch.  Its size may depend on the number of pulses only, so the step operators
// are held for a window of steps (at most 4096, at least 64) of a slice of pulses and the sweep
// goes window by window, forward and then back (most calls have one window).
struct LocStatePlan {
  int64_t pulses, steps;
};
static size_t loc_state_step(const redo_table* t) {              // FP64 bytes of one step of one pulse
  return ((size_t)t->N + 3 * t->loc) * sizeof(double2) + 3 * t->loc_pairs * sizeof(double);
}
static LocStatePlan loc_state_plan(const redo_table* t, int64_t B) {
  const size_t per = loc_state_step(t);
  int64_t pulses = (int64_t)(((size_t)256 << 20) / (64 * per));
  if (pulses > B) pulses = B;
  if (pulses < 1) pulses = 1;
  int64_t steps = (int64_t)(((size_t)64 << 20) / ((size_t)pulses * per));
  if (steps > 4096) steps = 4096;
  if (steps < 64) steps = 64;
  return LocStatePlan{pulses, steps};
}
// delta, rotations, Bloch sums of the window, and the two vectors of every pulse of the slice
static LocScratch loc_state_scratch(const redo_table* t, const LocStatePlan& p, void* base) {
  LocScratch w;
  char* c = (char*)base;
  const size_t nb = (size_t)p.pulses, T = (size_t)p.steps;
  w.delta = c;
  c += up256(nb * (T + 1) * t->N * sizeof(double2));
  w.cs = c;
  c += up256(nb * T * t->loc * sizeof(double2));
  w.bl = c;
  c += up256(nb * T * 3 * t->loc * sizeof(double));
  w.bz = c;
  c += up256(nb * 2 * t->N * sizeof(double2));
  w.g = c;
  c += up256(nb * T * 3 * t->loc_pairs * sizeof(double));
  w.sums = nullptr;
  w.flags = nullptr;
  w.total = (size_t)(c - (char*)base);
  return w;
}

// A bound of loc_state_scratch that never falls with B (the windows are rounded to whole steps): scratch
// asked for a batch serves every smaller one.
size_t local_state_bytes(const redo_table* t, int64_t B) {
  if (t->loc == 0 || B <= 0) return 0;
  const size_t nb = (size_t)loc_state_plan(t, B).pulses, step = nb * loc_state_step(t), cap = (size_t)64 << 20;
  const size_t steps = 64 * step > cap ? 64 * step : (4096 * step < cap ? 4096 * step : cap);
  return up256(steps + nb * t->N * 3 * sizeof(double2) + 5 * 256);
}

template <typename R>
static cudaError_t loc_state_t(const redo_table* t, const int32_t* q, int64_t B, int64_t M, int64_t win,
                               const double2* psi0, const double2* psiT, int batched, double* F_out, double* grad,
                               const LocScratch& w, int64_t* status, cudaStream_t s) {
  const int lanes = t->N / loc_vec_entries(t->N), cols = 32 / lanes;
  const unsigned blocks = (unsigned)((B + cols - 1) / cols);
  const int64_t nw = M > 0 ? (M + win - 1) / win : 1;
  const bool back = grad && M > 0;
  // (sized for FP64 vectors: behind the FP32 ones there is room for their scales)
  double* amp = sizeof(R) == 4 ? (double*)((char*)w.bz + (size_t)B * 2 * t->N * sizeof(cplx<R>)) : nullptr;
  LocScratch fo = w;                                 // forward only: no derivative operators
  fo.g = nullptr;
  // windows 0 .. nw - 1 forward, the last one also back, then nw - 2 .. 0 back
  for (int64_t i = 0; i < (back ? 2 * nw - 1 : nw); ++i) {
    const bool fwd = i < nw;
    const int64_t k = fwd ? i : 2 * nw - 2 - i, m0 = k * win, T = m0 + win < M ? win : M - m0;
    const int bk = back && i >= nw - 1;
    cudaError_t e = loc_steps_t<R>(t, q, B, M, m0, T, loc_vec_entries(t->N), loc_near(sizeof(R) == 8, t->N),
                                   LocalDiag{nullptr, 0, 0}, 0,
                                   bk ? w : fo, fwd ? status : nullptr, s);
    if (e) return e;
    LOC_VEC(loc_state_kernel, (const cplx<R>*)w.cs, (const cplx<R>*)w.delta, B, M, m0, T, fwd, bk, psi0, psiT, batched,
            F_out, (R*)w.bl, (cplx<R>*)w.bz, amp)
    if (bk && (e = loc_finish_t<R>(t, B, M, m0, T, 1, 1.0, w, grad, nullptr, PhaseForm{}, nullptr, amp, s))) return e;
  }
  return cudaGetLastError();
}

cudaError_t launch_local_state(const redo_table* t, const int32_t* q, int64_t B, int64_t M, int prec,
                               const double2* psi0, const double2* psiT, int batched, double* F_out, double* grad,
                               void* ops, int64_t* status, cudaStream_t s) {
  const LocStatePlan p = loc_state_plan(t, B);
  const LocScratch w = loc_state_scratch(t, p, ops);
  for (int64_t b0 = 0; b0 < B; b0 += p.pulses) {
    const int64_t nb = b0 + p.pulses < B ? p.pulses : B - b0, at = b0 * M * t->K, v = batched ? b0 * t->N : 0;
    double *F = F_out ? F_out + b0 : nullptr, *g = grad ? grad + at : nullptr;
    const cudaError_t e =
        prec == REDO_FP64
            ? loc_state_t<double>(t, q + at, nb, M, p.steps, psi0 + v, psiT + v, batched, F, g, w, status, s)
            : loc_state_t<float>(t, q + at, nb, M, p.steps, psi0 + v, psiT + v, batched, F, g, w, status, s);
    if (e) return e;
  }
  return cudaSuccess;
}

}  // namespace redo
