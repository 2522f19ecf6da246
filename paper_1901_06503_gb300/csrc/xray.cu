// xray.cu -- the X-ray transform P of eq. (4) in every horizontal plane, its
// exact transpose P^T (the discrete backprojection X^* of Sec. 3.1) and the
// ramp preconditioner Lambda of Sec. 3.1.
//
// Geometry: the planes have n cells per axis of physical size dx = 2 / nimg
// (nimg = n on the box [-1, 1]^3; n = nimg + 2 pad on a padded wave grid,
// which then spans [-L, L], L = n / nimg); n detectors and Ns = 2 ceil(n /
// sqrt 2) ray samples, both spaced dx.  The index geometry depends on n only;
// dx enters as the sample length and the detector spacing of Lambda.
//
// The geometry is the same in every plane, so both kernels run along z: the
// operand is first copied to a layout with z innermost (k_zlast), the bilinear
// weights of one angle are worked out once into shared-memory lists, and the
// lanes of a warp then apply each weight to 32, 64 or 128 planes at a time.
// What bounds them is thus the multiply-adds and the loads of the operand
// (through L1), no longer the index arithmetic.  Fixed order, no atomics:
// deterministic.
//
// P (ray-driven).  FP32: a ray is walked along its major axis (y where |cos|
// >= |sin|, else x); the weights of all its samples in one row of cells are
// merged into at most four taps.  FP64: sample by sample, with the
// interpolation done in round-to-nearest multiply/add with no contraction, in
// the order of the plain definition, so that indices, weights and sums are
// reproducible bit for bit.
//
// P^T (voxel-driven).  For every angle the samples whose bilinear footprint
// covers a voxel lie within sqrt(2) grid units of it in the rotated (xi, s)
// frame, i.e. at most 3 x 3 candidates; each contributes hat(dx) hat(dy) times
// its row value, which is exactly the bilinear weight P gives that voxel.
//
// Lambda: the linear (non-circular) convolution of a detector row with the odd
// taps t_d = -1/(2 pi^2 d^2 dxi) and t_0 = 1/(8 dxi), as a Toeplitz product: a CTA
// stages 32 rows, 512 inputs at a time, for up to 256 of their outputs.
#include <limits.h>
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <mutex>
#include <type_traits>

#include "internal.cuh"

namespace ffpat {
namespace {

constexpr double kPi = 3.14159265358979323846;

// FP64 ray sample (theta, k, m): lower-left corner and fractions.  Same
// operations, same order as the plain definition; no fused multiply-add.  The
// plane spans [-L, L] in cells of size dx = 2 / nimg (L = n / nimg: 1 on the
// box, larger on a padded wave grid); half = nimg / 2.
__device__ __forceinline__ void sample64(double cs, double sn, int k, int m, int ns, double dx,
                                         double half, double L, int& i0, int& j0, double& fx,
                                         double& fy) {
  const double xi = __dadd_rn(-L, __dmul_rn((double)k + 0.5, dx));
  const double s = __dmul_rn(((double)m + 0.5) - (double)(ns / 2), dx);
  const double x = __dsub_rn(__dmul_rn(xi, cs), __dmul_rn(s, sn));
  const double y = __dadd_rn(__dmul_rn(xi, sn), __dmul_rn(s, cs));
  const double gx = __dsub_rn(__dmul_rn(__dadd_rn(x, L), half), 0.5);
  const double gy = __dsub_rn(__dmul_rn(__dadd_rn(y, L), half), 0.5);
  const double flx = floor(gx), fly = floor(gy);
  i0 = (int)flx;
  j0 = (int)fly;
  fx = __dsub_rn(gx, flx);
  fy = __dsub_rn(gy, fly);
}

// Range [mlo, mhi) of ray samples that can touch the grid (conservative).
__device__ __forceinline__ void ray_range(float cs, float sn, int k, int n, int ns, int& mlo,
                                          int& mhi) {
  const float cN = 0.5f * (float)(n - 1);
  const float u = (float)k + 0.5f - 0.5f * (float)n;
  float vlo = -1e30f, vhi = 1e30f;
  // x = cN + u cs - v sn must lie in (-1, n)
  const float ax = cN + u * cs;
  if (fabsf(sn) > 1e-6f) {
    float a = (ax + 1.0f) / sn, b = (ax - (float)n) / sn;
    vlo = fmaxf(vlo, fminf(a, b));
    vhi = fminf(vhi, fmaxf(a, b));
  } else if (!(ax > -1.5f && ax < (float)n + 0.5f)) {
    vlo = 1.0f;
    vhi = -1.0f;
  }
  // y = cN + u sn + v cs must lie in (-1, n)
  const float ay = cN + u * sn;
  if (fabsf(cs) > 1e-6f) {
    float a = (-1.0f - ay) / cs, b = ((float)n - ay) / cs;
    vlo = fmaxf(vlo, fminf(a, b));
    vhi = fminf(vhi, fmaxf(a, b));
  } else if (!(ay > -1.5f && ay < (float)n + 0.5f)) {
    vlo = 1.0f;
    vhi = -1.0f;
  }
  if (!(vlo <= vhi)) {
    mlo = 0;
    mhi = 0;
    return;
  }
  const float off = 0.5f * (float)ns - 0.5f;
  mlo = max(0, (int)floorf(vlo + off) - 1);
  mhi = min(ns, (int)ceilf(vhi + off) + 2);
  if (mhi < mlo) mhi = mlo;
}

// Programmatic dependent launch: k_zlast lets its consumer start, and the
// consumer waits for k_zlast (its writes visible) before it reads the operand.
__device__ __forceinline__ void launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_for_operand() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ------------------------------------------------- z-innermost operands --
// out[slab][o][i][rl] = in[o so + z sz + i], z = slab rl + r: the volume (o = y,
// i = x) or the data (o = theta, i = xi) with z innermost, in slabs of rl planes
// (zero past the last plane), so that the lanes of a warp read planes side by
// side with aligned vector loads.  32 x 32 tiles through shared memory.
template <typename T>
__global__ void __launch_bounds__(256)
    k_zlast(const T* __restrict__ in, T* __restrict__ out, int nz, int ni, size_t so, size_t sz,
            int rl) {
  __shared__ T t[32][33];
  launch_dependents();  // the consumer works out its first weights meanwhile
  const size_t o = blockIdx.z;
  const int i0 = blockIdx.x * 32, z0 = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int z = z0 + r, i = i0 + threadIdx.x;
    t[r][threadIdx.x] = (z < nz && i < ni) ? in[o * so + (size_t)z * sz + i] : T(0);
  }
  __syncthreads();
  const int z = z0 + threadIdx.x, slab = z / rl;
  const size_t row = ((size_t)slab * gridDim.z + o) * ni;
  if (z >= (nz + rl - 1) / rl * rl) return;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int i = i0 + r;
    if (i < ni) out[(row + i) * rl + z % rl] = t[threadIdx.x][r];
  }
}

// The planes of one lane in a slab of 32 V C planes: C vectors of V neighbours,
// 32 V apart.  Sums go through the packed two-lane FMA of sm_100+ in pairs.
template <int V, int C>
struct ZRow {
  static constexpr int N = V * C, RL = 32 * N;
  float v[N];
  __device__ __forceinline__ void load(const float* q) {  // q: the lane's first plane
#pragma unroll
    for (int c = 0; c < C; ++c) {
      if constexpr (V == 4) {
        const float4 t = __ldg(reinterpret_cast<const float4*>(q + c * 32 * V));
        v[4 * c] = t.x;
        v[4 * c + 1] = t.y;
        v[4 * c + 2] = t.z;
        v[4 * c + 3] = t.w;
      } else if constexpr (V == 2) {
        const float2 t = __ldg(reinterpret_cast<const float2*>(q + c * 32 * V));
        v[2 * c] = t.x;
        v[2 * c + 1] = t.y;
      } else {
        v[c] = __ldg(q + c * 32);
      }
    }
  }
  // the plane of element i within the slab
  static __device__ __forceinline__ int plane(int lane, int i) {
    return i / V * 32 * V + lane * V + i % V;
  }
};

__device__ __forceinline__ float2 ffma2(float w, float2 x, float2 a) {
  unsigned long long r, u, p, q;
  const float2 ww = make_float2(w, w);
  memcpy(&u, &ww, 8);
  memcpy(&p, &x, 8);
  memcpy(&q, &a, 8);
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(u), "l"(p), "l"(q));
  float2 o;
  memcpy(&o, &r, 8);
  return o;
}

// What adding t to s0 (the sum: s1) rounded off; 0 where the sum has overflowed,
// so that it stays infinite.  Exact where |s0| >= |t|, as it is once a sum of one
// sign has two groups; where t is the larger, s1 - s0 is rounded itself.
__device__ __forceinline__ float rounded_off(float t, float s1, float s0) {
  const float e = __fsub_rn(t, __fsub_rn(s1, s0));
  return fabsf(e) < 1e32f ? e : 0.0f;
}

template <int N>
struct ZAcc {
  float2 a[N / 2 + 1];  // pairs; the last one's first lane is the odd plane
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i <= N / 2; ++i) a[i] = make_float2(0.0f, 0.0f);
  }
  __device__ __forceinline__ void fma(float w, const float* v) {
#pragma unroll
    for (int i = 0; i < N / 2; ++i) a[i] = ffma2(w, make_float2(v[2 * i], v[2 * i + 1]), a[i]);
    if constexpr (N % 2) a[N / 2].x = fmaf(w, v[N - 1], a[N / 2].x);
  }
  // adds o and leaves in o what the additions rounded off
  __device__ __forceinline__ void add_carry(ZAcc& o) {
#pragma unroll
    for (int i = 0; i <= N / 2; ++i) {
      const float2 s = make_float2(__fadd_rn(a[i].x, o.a[i].x), __fadd_rn(a[i].y, o.a[i].y));
      o.a[i] = make_float2(rounded_off(o.a[i].x, s.x, a[i].x), rounded_off(o.a[i].y, s.y, a[i].y));
      a[i] = s;
    }
  }
  __device__ __forceinline__ float get(int i) const { return i & 1 ? a[i / 2].y : a[i / 2].x; }
};

// fraction (bits 0 .. 30 of a scale-2^31 fixed-point value) as a float
__device__ __forceinline__ float frac31(long long v) {
  return __uint2float_rn((unsigned)v & 0x7fffffffu) * 0x1p-31f;
}

// --------------------------------------------------------------- P, FP32 --
// The taps of ray k (angle cs, sn in fixed point, 2^30) in row `a` of the
// ray's major axis: weight w[t] = sum over the ray's samples of hat(major
// distance) hat(minor distance) for the cells base .. base + 3 of the minor
// axis.  Samples advance by at least 1/sqrt 2 along the major and at most that
// much along the minor axis, so at most three samples touch the row and their
// corners span at most four cells.  Coordinates are 64-bit fixed point (2^31
// per cell; the steps along a ray are exact), inv = 1 / (major step).
struct RowTaps {
  float w[4];
  int base, count;  // the nonzero taps are among base .. base + count - 1, inside the plane
};
__device__ __forceinline__ RowTaps row_taps(int a, int k, long long CS, long long SN, bool ymajor,
                                            float inv, int n, int ns) {
  const long long u2 = 2LL * k + 1 - n, v0 = 1LL - ns, c2 = (long long)(n - 1) << 30;
  const long long X0 = c2 + u2 * CS - v0 * SN, Y0 = c2 + u2 * SN + v0 * CS;
  const long long A0 = ymajor ? Y0 : X0, B0 = ymajor ? X0 : Y0;
  const long long dA = ymajor ? 2 * CS : -2 * SN, dB = ymajor ? -2 * SN : 2 * CS;
  const long long D0 = ((long long)a << 31) - A0;
  // samples within sqrt 2 of the row's crossing (0.01 covers the float rounding
  // of the crossing; three integers always cover the interval)
  const int m0 = (int)ceilf(__ll2float_rn(D0) * inv - 1.4243f);
  const long long Bm = B0 + m0 * dB;
  RowTaps r;
  r.base = min((int)(Bm >> 31), (int)((Bm + 2 * dB) >> 31));
#pragma unroll
  for (int t = 0; t < 4; ++t) r.w[t] = 0.0f;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const long long D = D0 - (m0 + s) * dA, B = Bm + s * dB;
    float ha = __saturatef(1.0f - fabsf(__int2float_rn((int)(D >> 2)) * 0x1p-29f));
    if ((unsigned)(m0 + s) >= (unsigned)ns) ha = 0.0f;
    const int p = (int)(B >> 31) - r.base;
    const float fb = frac31(B), hi = ha * fb, lo = ha * (1.0f - fb);
#pragma unroll
    for (int t = 0; t < 4; ++t) r.w[t] += p == t ? lo : (p + 1 == t ? hi : 0.0f);
  }
#pragma unroll
  for (int t = 0; t < 4; ++t)
    if ((unsigned)(r.base + t) >= (unsigned)n) r.w[t] = 0.0f;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (r.w[0] == 0.0f) {  // the first tap kept is a nonzero one
      r.w[0] = r.w[1];
      r.w[1] = r.w[2];
      r.w[2] = r.w[3];
      r.w[3] = 0.0f;
      r.base += 1;
    }
  }
  r.count = r.w[3] != 0.0f ? 4 : (r.w[2] != 0.0f ? 3 : (r.w[1] != 0.0f ? 2 : (r.w[0] != 0.0f ? 1 : 0)));
  return r;
}

// P for all planes of a slab at once.  A CTA takes one angle, rg neighbouring
// rays and one slab; a warp owns a ray, or every `split`-th block of kPSum rows
// of it, a lane V C planes.  Row by row of the major axis, the taps of every ray are worked out
// into shared memory (ch rows at a time) and applied to all planes: two
// broadcast shared loads, then two to four taps of C vector loads and V C / 2
// packed FMAs.  Bound by waiting for loads, nothing saturated: at 192^3 and 90
// angles half of them hit L1 (neighbouring rays share cells), 57 % of the issue
// slots and 56 % of L1's throughput are in use.
// 64 registers and 32 warps an SM: half of the loads miss L1 (every cell is new
// to the CTA once), and more warps hid that better than fetching a row ahead
// (192^3, 90 angles: 0.36 ms, against 0.54 with 16 warps and two rows in
// flight).  Per standalone call, 384^3 and 180 angles: 13.0 -> 5.2 ms against
// the plane-by-plane kernel it replaces, 256^3 and 180: 3.7 -> 1.7 ms.
// Sums: per kPSum rows, then over those; what adding a group rounds off starts
// the next one, so that the error of a sum of one sign, where the groups' total is
// the large term, does not grow with N (a smooth volume, relative:
// 150^3 8.3e-8 -> 4.7e-8, 256^3 9.6e-8 -> 3.0e-8; 192^3 and 90 angles, standalone
// call, 541 -> 547 us).
constexpr int kPSum = 8;
constexpr int kPWarps = 16;

template <int T, int V, int C>
__device__ __forceinline__ void ray_taps(const float* q, long long sb, float4 w,
                                         ZAcc<V * C>& c) {
  ZRow<V, C> x[T];
#pragma unroll
  for (int t = 0; t < T; ++t) x[t].load(q + t * sb);
  c.fma(w.x, x[0].v);
  if constexpr (T > 1) c.fma(w.y, x[1].v);
  if constexpr (T > 2) c.fma(w.z, x[2].v);
  if constexpr (T > 3) c.fma(w.w, x[3].v);
}

template <int V, int C>
__global__ void __launch_bounds__(kPWarps * 32, 2)
    k_project_z(const float* __restrict__ pt, float* __restrict__ g,
                const float* __restrict__ sub, const float* __restrict__ mask,
                const int32_t* __restrict__ tabi, int n, int nz, int nth, int ns, int nimg,
                int rg, int ch) {
  constexpr int RL = ZRow<V, C>::RL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int split = blockDim.x / 32 / rg;
  float4* w4 = reinterpret_cast<float4*>(smem_raw);            // [ch][rg]
  int* xb = reinterpret_cast<int*>(w4 + (size_t)ch * rg);       // [ch][rg]: 8 base + count
  float* stage = reinterpret_cast<float*>(smem_raw);           // [split][RL][rg + 1], afterwards
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ray = warp % rg, part = warp / rg;
  const int j = blockIdx.y, k0 = blockIdx.x * rg;
  const int zbase = blockIdx.z * RL;
  const float* __restrict__ pz = pt + (size_t)blockIdx.z * n * n * RL + lane * V;
  const int CSi = tabi[j], SNi = tabi[nth + j];
  const long long CS = CSi, SN = SNi;
  const bool ymajor = abs(CSi) >= abs(SNi);
  const float inv = 1.0f / (float)(ymajor ? 2 * CS : -2 * SN);
  const long long sa = (long long)(ymajor ? n : 1) * RL, sb = (long long)(ymajor ? 1 : n) * RL;
  ZAcc<V * C> total, c;
  total.zero();
  c.zero();
  for (int a0 = 0; a0 < n; a0 += ch) {
    const int rows = min(ch, n - a0);
    __syncthreads();
    for (int e = tid; e < rows * rg; e += blockDim.x) {
      const int k = k0 + e % rg;
      RowTaps t{{0.0f, 0.0f, 0.0f, 0.0f}, 0, 0};
      if (k < n) t = row_taps(a0 + e / rg, k, CS, SN, ymajor, inv, n, ns);
      w4[e] = make_float4(t.w[0], t.w[1], t.w[2], t.w[3]);
      xb[e] = t.base * 8 + t.count;
    }
    if (a0 == 0) wait_for_operand();
    __syncthreads();
#pragma unroll 1
    for (int rs = part * kPSum; rs < rows; rs += split * kPSum) {
      const int re = min(rs + kPSum, rows);
      const float* prow = pz + (a0 + rs) * sa;
#pragma unroll 1
      for (int r = rs; r < re; ++r, prow += sa) {
        const int code = xb[r * rg + ray], cnt = code & 7;
        const float4 w = w4[r * rg + ray];
        const float* q = prow + (code >> 3) * sb;
        if (cnt == 3)
          ray_taps<3, V, C>(q, sb, w, c);
        else if (cnt == 2)
          ray_taps<2, V, C>(q, sb, w, c);
        else if (cnt == 4)
          ray_taps<4, V, C>(q, sb, w, c);
        else if (cnt == 1)
          ray_taps<1, V, C>(q, sb, w, c);
      }
      total.add_carry(c);
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < V * C; ++i)
    stage[(part * RL + ZRow<V, C>::plane(lane, i)) * (rg + 1) + ray] = total.get(i);
  __syncthreads();
  const float scale = 2.0f / (float)nimg;
  for (int e = tid; e < RL * rg; e += blockDim.x) {
    const int r = e % rg, zl = e / rg;
    if (k0 + r >= n || zbase + zl >= nz) continue;
    const size_t o = ((size_t)j * n + zbase + zl) * n + k0 + r;
    float sum = stage[zl * (rg + 1) + r], carry = 0.0f;
    for (int q = 1; q < split; ++q) {
      const float t = stage[(q * RL + zl) * (rg + 1) + r] + carry, s = __fadd_rn(sum, t);
      carry = rounded_off(t, s, sum);
      sum = s;
    }
    float out = scale * sum;
    if (sub) out = out - sub[o];
    if (mask) out = out * mask[o];
    g[o] = out;
  }
}

// --------------------------------------------------------------- P, FP64 --
// The same organisation sample by sample: per sample of a ray the four corner
// weights, the corner cell and which corners lie in the plane go to shared
// memory; every plane then takes four multiplications and four additions in
// the order of the plain definition (corners outside count as zero), bit for
// bit.  Bound by the FP64 pipe: 8 instructions a sample and plane (128^3, 90
// angles: 14.1 -> 3.3 ms; 2.9 ms at the measured FP64 rate).
constexpr int kP64Samples = 32;

template <int V>
__global__ void __launch_bounds__(384)
    k_project_z64(const double* __restrict__ pt, double* __restrict__ g,
                  const double* __restrict__ sub, const double* __restrict__ mask,
                  const double* __restrict__ tab, const float* __restrict__ tabf, int n, int nz,
                  int nth, int ns, int nimg, int zp, int nslab, int rg) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* wlo = reinterpret_cast<double2*>(smem_raw);               // row j0: (x0, x0 + 1)
  double2* whi = wlo + (size_t)kP64Samples * rg;                      // row j0 + 1
  int* at = reinterpret_cast<int*>(whi + (size_t)kP64Samples * rg);   // 16 (j0 n + i0) + corners
  double* stage = reinterpret_cast<double*>(smem_raw);
  __shared__ int s_lo, s_hi;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int slab = warp % nslab, r0 = 2 * (warp / nslab);
  const int j = blockIdx.y, k0 = blockIdx.x * rg;
  const int zbase = blockIdx.z * nslab * 32 * V;
  const int z = zbase + (slab * 32 + lane) * V;
  const double* __restrict__ pz = pt + min(z, zp - V);
  const double cs = tab[j], sn = tab[nth + j];
  const double dx = 2.0 / nimg, half = nimg / 2.0, L = (double)n / nimg;
  if (tid == 0) {
    s_lo = INT_MAX;
    s_hi = 0;
  }
  __syncthreads();
  if (tid < rg && k0 + tid < n) {
    int mlo, mhi;
    ray_range(tabf[j], tabf[nth + j], k0 + tid, n, ns, mlo, mhi);
    if (mlo < mhi) {
      atomicMin(&s_lo, mlo);
      atomicMax(&s_hi, mhi);
    }
  }
  __syncthreads();
  const int lo = s_lo, hi = s_hi;
  wait_for_operand();
  constexpr int kGroup = V == 1 ? 4 : 1;
  double acc0[V], acc1[V];
#pragma unroll
  for (int v = 0; v < V; ++v) acc0[v] = acc1[v] = 0.0;
  for (int ma = lo; ma < hi; ma += kP64Samples) {
    const int ms = min(kP64Samples, hi - ma);
    __syncthreads();
    for (int e = tid; e < ms * rg; e += blockDim.x) {
      const int k = k0 + e % rg;
      int code = 0;
      if (k < n) {
        int i0, j0;
        double fx, fy;
        sample64(cs, sn, k, ma + e / rg, ns, dx, half, L, i0, j0, fx, fy);
        const double ofx = __dsub_rn(1.0, fx), ofy = __dsub_rn(1.0, fy);
        wlo[e] = make_double2(__dmul_rn(ofx, ofy), __dmul_rn(fx, ofy));
        whi[e] = make_double2(__dmul_rn(ofx, fy), __dmul_rn(fx, fy));
        const bool x0 = (unsigned)i0 < (unsigned)n, x1 = (unsigned)(i0 + 1) < (unsigned)n;
        const bool y0 = (unsigned)j0 < (unsigned)n, y1 = (unsigned)(j0 + 1) < (unsigned)n;
        const int in = (x0 && y0 ? 1 : 0) | (x1 && y0 ? 2 : 0) | (x0 && y1 ? 4 : 0) |
                       (x1 && y1 ? 8 : 0);
        if (in) code = (j0 * n + i0) * 16 + in;
      }
      at[e] = code;
    }
    __syncthreads();
    // kGroup samples of both rays at a time: all their loads in flight, then the
    // sums (each ray's samples in order)
    for (int m = 0; m < ms; m += kGroup) {
      double v[kGroup][2][4][V];
      int code[kGroup][2];
#pragma unroll
      for (int q = 0; q < kGroup; ++q)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          code[q][r] = m + q < ms ? at[(m + q) * rg + r0 + r] : 0;
          const double* p = pz + (long long)(code[q][r] >> 4) * zp;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const double* c = p + (k & 1 ? zp : 0) + (k & 2 ? (long long)n * zp : 0LL);
            if constexpr (V == 1) {
              v[q][r][k][0] = code[q][r] & (1 << k) ? __ldg(c) : 0.0;
            } else {
              const double2 t = code[q][r] & (1 << k) ? __ldg(reinterpret_cast<const double2*>(c))
                                                      : make_double2(0.0, 0.0);
              v[q][r][k][0] = t.x;
              v[q][r][k][1] = t.y;
            }
          }
        }
#pragma unroll
      for (int q = 0; q < kGroup; ++q)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          if ((code[q][r] & 15) == 0) continue;  // adds an exact zero
          const int e = (m + q) * rg + r0 + r;
          const double2 wl = wlo[e], wh = whi[e];
          double(&acc)[V] = r == 0 ? acc0 : acc1;
#pragma unroll
          for (int i = 0; i < V; ++i) {
            double b = __dmul_rn(wl.x, v[q][r][0][i]);
            b = __dadd_rn(b, __dmul_rn(wl.y, v[q][r][1][i]));
            b = __dadd_rn(b, __dmul_rn(wh.x, v[q][r][2][i]));
            b = __dadd_rn(b, __dmul_rn(wh.y, v[q][r][3][i]));
            acc[i] = __dadd_rn(acc[i], b);
          }
        }
    }
  }
  __syncthreads();
#pragma unroll
  for (int v = 0; v < V; ++v) {
    double* s = stage + ((slab * 32 + lane) * V + v) * (rg + 1) + r0;
    s[0] = acc0[v];
    s[1] = acc1[v];
  }
  __syncthreads();
  for (int e = tid; e < nslab * 32 * V * rg; e += blockDim.x) {
    const int r = e % rg, zl = e / rg;
    if (k0 + r >= n || zbase + zl >= nz) continue;
    const size_t o = ((size_t)j * n + zbase + zl) * n + k0 + r;
    double out = __dmul_rn(dx, stage[zl * (rg + 1) + r]);
    if (sub) out = out - sub[o];
    if (mask) out = out * mask[o];
    g[o] = out;
  }
}

// ------------------------------------------------------------- P^T, FP32 --
// FP32 hat: 1 - |a| <= 1 always, so clamping to [0, 1] is max(0, .); one
// saturating add on the FMA pipe instead of an add and a min/max on the ALU
__device__ __forceinline__ float hat1f(float a) { return __saturatef(1.0f - fabsf(a)); }

// The weights a voxel gets from angle (cs, sn): its position in the rotated
// frame, kk (detector units) and mm (sample units), in fixed point (2^31; exact
// integer parts, fractions to ~1e-9); the candidate samples are k = kb .. kb + 2
// and m = mb .. mb + 2 around it (|k - kk|, |m - mm| < sqrt 2), each weighted by
// hat(a) hat(b) of its offset in the grid frame.  r[i]: the sum over the samples
// of detector kb + i.
__device__ __forceinline__ int voxel_sums(long long KK, long long MM, float cs, float sn, int ns,
                                          float (&r)[3]) {
  const int KI = (int)(KK >> 31), MI = (int)(MM >> 31);
  const float fk = frac31(KK), fm = frac31(MM);
  const int hk = fk >= 0.5f ? 1 : 0, hm = fm >= 0.5f ? 1 : 0;
  const int mb = MI - 1 + hm;
  const float du0 = (float)(hk - 1) - fk, dv0 = (float)(hm - 1) - fm;
  const float a0 = du0 * cs - dv0 * sn, b0 = du0 * sn + dv0 * cs;
  float mv[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) mv[q] = (unsigned)(mb + q) < (unsigned)ns ? 1.0f : 0.0f;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    r[i] = 0.0f;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float a = a0 + (float)i * cs - (float)q * sn;
      const float b = b0 + (float)i * sn + (float)q * cs;
      r[i] = fmaf(hat1f(a) * hat1f(b), mv[q], r[i]);
    }
  }
  return KI - 1 + hk;
}

constexpr int kBAngles = 8;  // angles of a batch of k_backproject_z

// The sum of voxel (x, y) over the detectors it sees, one plane (gp: its data,
// detectors rl apart), in the order of k_backproject_z.  There the four voxels of a
// block share their detectors, with zero weights, which make NaN of an infinite
// datum that a voxel does not see: a NaN is taken from here instead.
__device__ __noinline__ float voxel_alone(const float* __restrict__ gp, int rl, int x, int y,
                                          const float* __restrict__ tabf,
                                          const int32_t* __restrict__ tabi, int n, int nth,
                                          int ns) {
  const long long X2 = 2 * x - (n - 1), Y2 = 2 * y - (n - 1);
  const long long ck = (long long)(n - 1) << 30, cm = (long long)(ns - 1) << 30;
  float acc = 0.0f;
  const int nb = (nth + kBAngles - 1) / kBAngles;
  for (int a = 0; a < nb * kBAngles; ++a) {
    const int j = a / kBAngles + a % kBAngles * nb;
    if (j >= nth) continue;
    const long long CS = tabi[j], SN = tabi[nth + j];
    float r[3];
    const int kb = voxel_sums(X2 * CS + Y2 * SN + ck, Y2 * CS - X2 * SN + cm, tabf[j],
                              tabf[nth + j], ns, r);
    for (int i = 0; i < 3; ++i)
      if (r[i] != 0.0f && (unsigned)(kb + i) < (unsigned)n)
        acc = fmaf(r[i], gp[((size_t)j * n + kb + i) * rl], acc);
  }
  return acc;
}

// P^T for all planes of a slab at once.  A warp owns a block of 2 x 2 voxels
// and the slab's planes, V C a lane.  Its lanes work out the weights of eight
// angles at a time (a lane: one voxel and angle) into the warp's part of shared
// memory; then, angle by angle, the (at most five) detectors any of the four
// voxels sees are loaded once and applied to all four: C vector loads and 2 V C
// packed FMAs per detector (58 % of the issue slots and 57 % of L1's throughput in
// use at 192^3 and 90 angles, waits for loads the first stall; a voxel alone
// would load three detectors for as many multiply-adds each).  kk of the block
// spans |cos| + |sin| =: s <= sqrt 2 and a voxel's detectors lie within s of its
// kk: 3 s < 4.25 holds at most five.  Per standalone call, 384^3 and 180 angles:
// 14.5 -> 2.6 ms against the plane-by-plane gather it replaces, 192^3 and 90:
// 1.18 -> 0.38 ms.
// A batch of eight angles is spread over all directions: data that change sign
// slowly with the angle (filtered ones) then keep the partial sums, and with them
// the rounding of the long sum, small (256^3, 180 angles of filtered data, error
// against 64 bits 3.1 - 3.6e-7 -> 2.9e-7).  The list holds addresses: stepping a
// pointer through the spread rows took 2 % more (fbp at 192^3 / 90 angles 231 -> 222
// us, 256^3 / 180 779 -> 757 us, 384^3 / 180 2.56 -> 2.49 ms).
constexpr int kBDet = 5;
constexpr int kBTileX = 4, kBTileY = 2;  // blocks of a CTA (8 x 4 voxels), one a warp
// the detectors of a block and angle: address of the first one's planes, and count
// (one 16-byte shared load; as two loads 256^3 took 3 % more)
using BDetectors = ulonglong2;
constexpr size_t kBWarpBytes = kBAngles * (kBDet * 16 + sizeof(BDetectors));

template <int T, int V, int C>
__device__ __forceinline__ void block_taps(const float* q, const float4* w,
                                           ZAcc<V * C> (&acc)[4]) {
  ZRow<V, C> x[T];
#pragma unroll
  for (int t = 0; t < T; ++t) x[t].load(q + t * ZRow<V, C>::RL);
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const float4 u = w[t];
    acc[0].fma(u.x, x[t].v);
    acc[1].fma(u.y, x[t].v);
    acc[2].fma(u.z, x[t].v);
    acc[3].fma(u.w, x[t].v);
  }
}

template <int V, int C>
__global__ void __launch_bounds__(kBTileX* kBTileY * 32, V* C > 8 ? 2 : 3)
    k_backproject_z(const float* __restrict__ gt, float* __restrict__ h,
                    const float* __restrict__ scale, const float* __restrict__ tabf,
                    const int32_t* __restrict__ tabi, int n, int np, int nz, int nth, int ns,
                    int nimg, int tx,
                    float mult) {
  constexpr int RL = ZRow<V, C>::RL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = blockDim.x / 32;
  float4* W = reinterpret_cast<float4*>(smem_raw) + (size_t)warp * kBAngles * kBDet;
  BDetectors* list =
      reinterpret_cast<BDetectors*>(smem_raw + (size_t)warps * kBAngles * kBDet * 16) +
      warp * kBAngles;
  const int ty = warps / tx;  // tx x ty blocks in this CTA
  const int x0 = 2 * (blockIdx.x * tx + warp % tx), y0 = 2 * (blockIdx.y * ty + warp / tx);
  const int zbase = blockIdx.z * RL;
  const long long ck = (long long)(n - 1) << 30, cm = (long long)(ns - 1) << 30;
  // this lane's voxel and angle in the weight pass
  const int vox = lane & 3, al = lane >> 2;
  const long long X2 = 2 * x0 - (n - 1), Y2 = 2 * y0 - (n - 1);
  const long long dx = 2 * (vox & 1), dy = vox & 2;
  ZAcc<V * C> acc[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) acc[v].zero();
  // batch ja: angles ja, ja + nb, ... (see kBAngles)
  const int nb = (nth + kBAngles - 1) / kBAngles;
  for (int ja = 0; ja < nb; ++ja) {
    const int j = min(ja + al * nb, nth - 1);
    const float cs = tabf[j], sn = tabf[nth + j];
    const long long CS = tabi[j], SN = tabi[nth + j];
    const long long KK = X2 * CS + Y2 * SN + ck, MM = Y2 * CS - X2 * SN + cm;
    // the first detector closer than s to the block (SN >= 0)
    int kd = (int)((KK + min(2 * CS, 0LL) - 2 * (llabs(CS) + SN)) >> 31) + 1;
    float r[3], w[kBDet];
    const int p = voxel_sums(KK + dx * CS + dy * SN, MM + dy * CS - dx * SN, cs, sn, ns, r) - kd;
    unsigned on = 0;
#pragma unroll
    for (int d = 0; d < kBDet; ++d) {
      w[d] = p == d ? r[0] : (p + 1 == d ? r[1] : (p + 2 == d ? r[2] : 0.0f));
      if ((unsigned)(kd + d) >= (unsigned)n) w[d] = 0.0f;
      if (w[d] != 0.0f) on |= 1u << d;
    }
    on |= __shfl_xor_sync(0xffffffffu, on, 1);
    on |= __shfl_xor_sync(0xffffffffu, on, 2);
    // the detectors from the first to the last that any voxel sees
    const int first = on ? __ffs(on) - 1 : 0, count = on ? 32 - __clz(on) - first : 0;
    __syncwarp();
    float* wl = reinterpret_cast<float*>(W + al * kBDet) + vox;
#pragma unroll
    for (int d = 0; d < kBDet; ++d)
      if (d >= first) wl[4 * (d - first)] = w[d];
    if (vox == 0)
      list[al] = make_ulonglong2(
          (unsigned long long)(gt + ((size_t)blockIdx.z * nth * n + (long long)(j * n + kd + first)) * RL),
          ja + al * nb < nth ? count : 0);
    if (ja == 0) wait_for_operand();
    __syncwarp();
#pragma unroll 1
    for (int t = 0; t < kBAngles; ++t) {
      const BDetectors det = list[t];
      const unsigned cnt = (unsigned)det.y;
      const float* q = reinterpret_cast<const float*>(det.x) + lane * V;
      const float4* u = W + t * kBDet;
      if (cnt == 4)
        block_taps<4, V, C>(q, u, acc);
      else if (cnt == 3)
        block_taps<3, V, C>(q, u, acc);
      else if (cnt == 5) {
        block_taps<3, V, C>(q, u, acc);
        block_taps<2, V, C>(q + 3 * RL, u + 3, acc);
      } else if (cnt == 2)
        block_taps<2, V, C>(q, u, acc);
      else if (cnt == 1)
        block_taps<1, V, C>(q, u, acc);
    }
  }
  // through shared memory to the planes' rows, 32 planes at a time
  const int sx = 2 * tx, nv = 4 * warps;
  const float f = 2.0f / (float)nimg;
  float* stage = reinterpret_cast<float*>(smem_raw);  // [32 V planes][nv + 1]
  bool nan = false;
#pragma unroll
  for (int c = 0; c < C; ++c) {
    __syncthreads();
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int at = (2 * (warp / tx) + (v >> 1)) * sx + 2 * (warp % tx) + (v & 1);
#pragma unroll
      for (int i = 0; i < V; ++i) stage[(lane * V + i) * (nv + 1) + at] = acc[v].get(c * V + i);
    }
    __syncthreads();
    for (int e = tid; e < nv * 32 * V; e += blockDim.x) {
      const int v = e % nv, zl = e / nv;
      const int x = blockIdx.x * sx + v % sx, y = blockIdx.y * 2 * ty + v / sx;
      const int z = zbase + c * 32 * V + zl;
      if (x >= n || y >= n || z >= nz) continue;
      const size_t o = ((size_t)z * n + y) * np + x;
      float out = f * stage[zl * (nv + 1) + v];
      if (scale) out *= scale[o];
      if (mult != 1.0f) out *= mult;
      h[o] = out;
      nan |= isnan(out);
    }
  }
  if (nan)  // the elements that this thread wrote
    for (int e = tid; e < nv * RL; e += blockDim.x) {
      const int v = e % nv, zl = e / nv;
      const int x = blockIdx.x * sx + v % sx, y = blockIdx.y * 2 * ty + v / sx;
      if (x >= n || y >= n || zbase + zl >= nz) continue;
      const size_t o = ((size_t)(zbase + zl) * n + y) * np + x;
      if (!isnan(h[o])) continue;
      float out = f * voxel_alone(gt + (size_t)blockIdx.z * nth * n * RL + zl, RL, x, y, tabf, tabi,
                                  n, nth, ns);
      if (scale) out *= scale[o];
      if (mult != 1.0f) out *= mult;
      h[o] = out;
    }
}

// ------------------------------------------------------------- P^T, FP64 --
// The same, each voxel of the block with its own three detectors: here the
// FP64 pipe is the bound, so only nonzero weights are applied (2.3 of them a
// voxel and angle on average) and the loads do not matter (128^3, 90 angles:
// 32.9 -> 1.1 ms; 0.8 ms at the measured FP64 rate).
__device__ __forceinline__ double hat1d(double a) {
  const double v = 1.0 - fabs(a);
  return v > 0.0 ? v : 0.0;
}

constexpr int kB64Angles = 32;
constexpr size_t kB64WarpBytes = kB64Angles * (4 * 3 * 8 + 4 * 4);

template <int V>
__global__ void __launch_bounds__(128)
    k_backproject_z64(const double* __restrict__ gt, double* __restrict__ h,
                      const double* __restrict__ scale, const double* __restrict__ tab, int n,
                      int np, int nz, int nth, int ns, int nimg, int zp, int tb, double mult) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* W = reinterpret_cast<double*>(smem_raw) + (size_t)warp * kB64Angles * 12;
  int* info = reinterpret_cast<int*>(smem_raw + (size_t)(blockDim.x / 32) * kB64Angles * 96) +
              warp * kB64Angles * 4;
  const int x0 = 2 * (blockIdx.x * tb + warp % tb), y0 = 2 * (blockIdx.y * tb + warp / tb);
  const int zbase = blockIdx.z * 32 * V;
  const double* __restrict__ gz = gt + min(zbase + lane * V, zp - (V < 2 ? 1 : 2));
  const bool hi_ok = V < 4 || zbase + lane * V + 2 < zp;
  double acc[4][V];
#pragma unroll
  for (int v = 0; v < 4; ++v)
#pragma unroll
    for (int i = 0; i < V; ++i) acc[v][i] = 0.0;
  for (int ja = 0; ja < nth; ja += kB64Angles) {
    __syncwarp();
    if (ja + lane < nth) {
      const double cs = tab[ja + lane], sn = tab[nth + ja + lane];
#pragma unroll(V == 1 ? 2 : 1)
      for (int v = 0; v < 4; ++v) {
        const double X = (x0 + (v & 1)) - 0.5 * (n - 1), Y = (y0 + (v >> 1)) - 0.5 * (n - 1);
        const double kk = fma(X, cs, Y * sn) + 0.5 * (n - 1);
        const double mm = fma(Y, cs, -X * sn) + 0.5 * (ns - 1);
        const double fkk = floor(kk), fmm = floor(mm);
        const double fk = kk - fkk, fm = mm - fmm;
        const int hk = fk >= 0.5 ? 1 : 0, hm = fm >= 0.5 ? 1 : 0;
        const int kb = (int)fkk - 1 + hk, mb = (int)fmm - 1 + hm;
        const double du0 = (double)(hk - 1) - fk, dv0 = (double)(hm - 1) - fm;
        const double a0 = du0 * cs - dv0 * sn, b0 = du0 * sn + dv0 * cs;
        int on = 0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const double ai = a0 + i * cs, bi = b0 + i * sn;
          double w = 0.0;
          if ((unsigned)mb < (unsigned)ns) w += hat1d(ai) * hat1d(bi);
          if ((unsigned)(mb + 1) < (unsigned)ns) w += hat1d(ai - sn) * hat1d(bi + cs);
          if ((unsigned)(mb + 2) < (unsigned)ns) w += hat1d(ai - 2.0 * sn) * hat1d(bi + 2.0 * cs);
          W[(lane * 4 + v) * 3 + i] = w;
          if (w != 0.0 && (unsigned)(kb + i) < (unsigned)n) on |= 1 << i;
        }
        info[lane * 4 + v] = kb * 8 + on;
      }
    }
    if (ja == 0) wait_for_operand();
    __syncwarp();
    const int jn = min(kB64Angles, nth - ja);
    for (int t = 0; t < jn; ++t) {
      const double* row = gz + (long long)(ja + t) * n * zp;
      if constexpr (V == 4) {
        // enough planes a lane to cover the loads' latency
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int on = info[t * 4 + v];
          const double* q = row + (long long)(on >> 3) * zp;
#pragma unroll
          for (int i = 0; i < 3; ++i)
            if (on & (1 << i)) {
              const double w = W[(t * 4 + v) * 3 + i];
              const double2 d = __ldg(reinterpret_cast<const double2*>(q + i * zp));
              acc[v][0] = fma(w, d.x, acc[v][0]);
              acc[v][1] = fma(w, d.y, acc[v][1]);
              if (hi_ok) {
                const double2 e = __ldg(reinterpret_cast<const double2*>(q + i * zp + 2));
                acc[v][2] = fma(w, e.x, acc[v][2]);
                acc[v][3] = fma(w, e.y, acc[v][3]);
              }
            }
        }
      } else {
        // the detectors of NV voxels in flight, then their multiply-adds
        constexpr int NV = V == 1 ? 4 : 2;
#pragma unroll
        for (int v0 = 0; v0 < 4; v0 += NV) {
          double d[NV][3][V];
          int on[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            on[v] = info[t * 4 + v0 + v];
            const double* q = row + (long long)(on[v] >> 3) * zp;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              const bool use = on[v] & (1 << i);
              if constexpr (V == 1) {
                d[v][i][0] = use ? __ldg(q + i * zp) : 0.0;
              } else {
                const double2 a = use ? __ldg(reinterpret_cast<const double2*>(q + i * zp))
                                      : make_double2(0.0, 0.0);
                d[v][i][0] = a.x;
                d[v][i][1] = a.y;
              }
            }
          }
#pragma unroll
          for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int i = 0; i < 3; ++i)
              if (on[v] & (1 << i)) {
                const double w = W[(t * 4 + v0 + v) * 3 + i];
#pragma unroll
                for (int k = 0; k < V; ++k) acc[v0 + v][k] = fma(w, d[v][i][k], acc[v0 + v][k]);
              }
        }
      }
    }
  }
  __syncthreads();
  double* stage = reinterpret_cast<double*>(smem_raw);
  const int side = 2 * tb;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const int vx = 2 * (warp % tb) + (v & 1), vy = 2 * (warp / tb) + (v >> 1);
#pragma unroll
    for (int i = 0; i < V; ++i) stage[(vy * side + vx) * 32 * V + lane * V + i] = acc[v][i];
  }
  __syncthreads();
  for (int e = tid; e < side * side * 32 * V; e += blockDim.x) {
    const int v = e % (side * side), zl = e / (side * side);
    const int x = blockIdx.x * side + v % side, y = blockIdx.y * side + v / side;
    const int z = zbase + zl;
    if (x >= n || y >= n || z >= nz) continue;
    const size_t o = ((size_t)z * n + y) * np + x;
    double out = (2.0 / nimg) * stage[v * 32 * V + zl];
    if (scale) out *= scale[o];
    if (mult != 1.0) out *= mult;
    h[o] = out;
  }
}

// Lambda on rows of n detectors.  Only odd taps (and t_0) are nonzero, so the
// outputs of one parity are a dense Toeplitz product with the inputs of the other:
// n / 2 multiply-adds an output, bound by the FMA pipe.  A CTA stages 32 rows with
// the rows innermost (lane = row); a warp owns kROut outputs of one parity in all
// 32: per input it loads one value a row and one new tap (broadcast; the other
// taps slide through registers) for kROut multiply-adds.  The same kernel in FP64.
// On smooth rows t_0 r_k nearly cancels the nearest taps' sum, so those (|d| <=
// NEAR) are summed apart, outwards from t_0, the two large products without rounding
// them, and the Toeplitz product holds the others (a tenth of t_0 in all with NEAR =
// 3), whose rounding then shows as little.  NEAR is 7 beyond 448 points, where more
// of the others are added (FP32).  Error on smooth rows over that of the sum outwards
// pair by pair: 0.57 at 64, 0.81 at 256, 0.79 at 384, 0.87 at 512, 0.99 at 1024
// points (with rounded products and NEAR = 3 throughout 1.03 - 1.5 from 512 on).
// 384^3 and 180 angles: 1.63 -> 0.40 ms against two inputs and a tap loaded for
// every multiply-add, 256^3 and 180: 0.50 -> 0.122 ms (0.16 with one CTA an SM at
// 127 registers, 0.17 with eight outputs a warp).
constexpr int kROut = 16;
constexpr int kRPitch = 33;  // of a staged input: 32 rows and one word against bank conflicts

// (Lambda row)_k by the odd taps alone.  The Toeplitz product has zeros for taps
// among those of its other parity (|d| <= NEAR), which make NaN of an infinite
// input: an output that is NaN is taken from here, which says whether it is.
template <typename T>
__device__ __noinline__ T ramp_direct(const T* __restrict__ row, int k, int n, int nimg) {
  const double dxi = 2.0 / nimg;
  T v = (T)(1.0 / (8.0 * dxi)) * row[k];
  for (int d = 1; d < n && v == v; d += 2) {
    const T t = (T)(-1.0 / (2.0 * kPi * kPi * (double)d * d * dxi));
    v += t * ((k >= d ? row[k - d] : T(0)) + (k + d < n ? row[k + d] : T(0)));
  }
  return v;
}

// rows of staged inputs: all of them and what the last outputs' nearest taps reach,
// or a piece of jc, or the outputs of a CTA
__host__ __device__ inline int ramp_rows(int n, int jc, int nout, int ctas, int near) {
  const int reach = jc >= n ? ctas * nout : nout;
  return (jc > reach ? jc : reach) + 2 * near;
}

template <typename T, int NEAR>
__global__ void __launch_bounds__(512, sizeof(T) == 4 ? 2 : 1)
    k_ramp(const T* __restrict__ r, T* __restrict__ out, const T* __restrict__ mask, int n,
           int nimg, int rows, int jc) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = blockDim.x / 32;
  const int ko = blockIdx.y * warps * kROut;   // first output of the CTA (a multiple of 32)
  const int nout = warps * kROut;
  const int H = n / 2 + 2 * kROut + nout / 2;  // taps by u, d = 2 u + 1, -H <= u < H
  // staged inputs [ramp_rows][kRPitch], NEAR rows of room before the first
  const int srows = ramp_rows(n, jc, nout, gridDim.y, NEAR);
  T* s = reinterpret_cast<T*>(smem_raw);
  T* ts = s + (size_t)srows * kRPitch;
  const double dxi = 2.0 / nimg;
  for (int i = tid; i < 2 * H; i += blockDim.x) {
    const double d = 2.0 * (i - H) + 1.0;
    ts[i] = fabs(d) > NEAR ? (T)(-1.0 / (2.0 * kPi * kPi * d * d * dxi)) : T(0);
  }
  if (jc >= n)  // zeros around the rows for the nearest taps
    for (int i = tid; i < (srows - n) * 32; i += blockDim.x)
      s[(i / 32 < NEAR ? i / 32 : n + i / 32) * kRPitch + i % 32] = T(0);
  const int row0 = blockIdx.x * 32, live = min(32, rows - row0);
  // outputs k = 2 (q0 + m) + p, inputs j = 2 i + 1 - p, tap u = q0 + m + p - 1 - i
  const int p = warp & 1, q0 = ko / 2 + (warp >> 1) * kROut;
  T acc[kROut];
#pragma unroll
  for (int m = 0; m < kROut; ++m) acc[m] = T(0);
  for (int j0 = 0; j0 < n; j0 += jc) {
    const int len = min(jc, n - j0);
    __syncthreads();
    for (int q = warp; q < 32; q += warps) {
      const T* src = r + (size_t)(row0 + q) * n + j0;
      for (int j = lane; j < len; j += 32) s[(NEAR + j) * kRPitch + q] = q < live ? src[j] : T(0);
    }
    __syncthreads();
    const int ni = (len + p) / 2;
    const T* x = s + (NEAR + 1 - p) * kRPitch + lane;
    const T* t = ts + H + q0 + p - 1 - j0 / 2;  // t[m - i]: the tap of output m, input i
    T w[kROut];  // slot (m - i) mod kROut
#pragma unroll
    for (int m = 1; m < kROut; ++m) w[m] = t[m];
    int i = 0;
    for (; i + kROut <= ni; i += kROut) {
#pragma unroll
      for (int e = 0; e < kROut; ++e) {
        const T v = x[(i + e) * 2 * kRPitch];
        w[(kROut - e) % kROut] = t[-(i + e)];
#pragma unroll
        for (int m = 0; m < kROut; ++m)
          acc[m] = fma(w[(m - e + kROut) % kROut], v, acc[m]);
      }
    }
    for (; i < ni; ++i) {  // the rest, taps from shared memory
      const T v = x[i * 2 * kRPitch];
#pragma unroll
      for (int m = 0; m < kROut; ++m) acc[m] = fma(t[m - i], v, acc[m]);
    }
  }
  // the nearest taps, outwards from t_0, on the rows as staged or, where that was in
  // several pieces, on the inputs around the CTA's outputs staged again
  const T* near = s + (NEAR - (jc < n ? ko : 0)) * kRPitch + lane;  // input j at j kRPitch
  if (jc < n) {
    __syncthreads();
    for (int q = warp; q < 32; q += warps) {
      const T* src = r + (size_t)(row0 + q) * n;
      for (int j = lane; j < nout + 2 * NEAR; j += 32) {
        const int from = ko - NEAR + j;
        s[j * kRPitch + q] = q < live && (unsigned)from < (unsigned)n ? src[from] : T(0);
      }
    }
    __syncthreads();
  }
  const T t0 = (T)(1.0 / (8.0 * dxi));
  T tn[(NEAR + 1) / 2];
#pragma unroll
  for (int e = 0; e < (NEAR + 1) / 2; ++e) {
    const double d = 2.0 * e + 1.0;
    tn[e] = (T)(-1.0 / (2.0 * kPi * kPi * d * d * dxi));
  }
  auto at = [&](int j) -> T { return near[j * kRPitch]; };
#pragma unroll
  for (int m = 0; m < kROut; ++m) {
    const int k = 2 * (q0 + m) + p;
    const T pair = at(k - 1) + at(k + 1);
    T v;
    if constexpr (sizeof(T) == 4) {  // t_0 r_k + t_1 pair, neither product rounded
      const T prod = tn[0] * pair;
      v = fma(t0, at(k), prod) + fma(tn[0], pair, -prod);
    } else {
      v = fma(tn[0], pair, t0 * at(k));
    }
#pragma unroll
    for (int e = 1; e < (NEAR + 1) / 2; ++e)
      v = fma(tn[e], at(k - 2 * e - 1) + at(k + 2 * e + 1), v);
    acc[m] = v + acc[m];
  }
  // through shared memory to the rows
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kROut; ++m)
    s[(2 * ((warp >> 1) * kROut + m) + p) * kRPitch + lane] = acc[m];
  __syncthreads();
  const int kn = min(nout, n - ko);
  for (int q = warp; q < live; q += warps)
    for (int k = lane; k < kn; k += 32) {
      const size_t o = (size_t)(row0 + q) * n + ko + k;
      T v = s[k * kRPitch + q];
      if (v != v) v = ramp_direct(r + (size_t)(row0 + q) * n, ko + k, n, nimg);
      if (mask) v = v * mask[o];
      out[o] = v;
    }
}

__global__ void k_debug_samples(int count, const int32_t* __restrict__ jkm, int32_t* __restrict__ ij,
                                double* __restrict__ f, const double* __restrict__ tab, int n,
                                int nth, int ns, int nimg) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= count) return;
  const int j = jkm[3 * t], k = jkm[3 * t + 1], m = jkm[3 * t + 2];
  if (j < 0 || j >= nth) return;
  int i0, j0;
  double fx, fy;
  sample64(tab[j], tab[nth + j], k, m, ns, 2.0 / nimg, nimg / 2.0, (double)n / nimg, i0, j0, fx,
           fy);
  ij[2 * t] = i0;
  ij[2 * t + 1] = j0;
  f[2 * t] = fx;
  f[2 * t + 1] = fy;
}

}  // namespace

// Planes in a slab of a z-innermost operand, `most` of them at most (or as few as a
// slab can have).  FP64: all of them in one slab, rounded up to 16 bytes.  FP32: 32 V
// C for one of the instantiated (V, C), the one of least time for n planes, slabs x
// the measured cost of a slab (P + P^T at 128^3, 192^3 and 384^3 with every width, in
// units of the 64-plane slab): wider slabs share the weights and addresses among more
// planes, until the last one is mostly idle lanes.
static int slab_planes(int n, size_t esize, size_t most) {
  if (esize == 8) {
    const int all = (n + 1) / 2 * 2;
    if ((size_t)all <= most) return all;
    return most >= 32 ? (int)(most / 32 * 32) : (most >= 2 ? (int)(most / 2 * 2) : kMinPlanes64);
  }
  static const int rl[] = {32, 64, 96, 128, 160, 192, 256, 320, 384};
  static const float cost[] = {0.85f, 1.0f, 1.14f, 1.25f, 1.4f, 1.5f, 1.85f, 2.3f, 2.7f};
  int best = kMinPlanes32;
  float best_cost = 1e30f;
  for (int i = 0; i < 9; ++i) {
    if ((size_t)rl[i] > most) break;
    const float c = cost[i] * (float)((n + rl[i] - 1) / rl[i]);
    if (c < best_cost) {
      best = rl[i];
      best_cost = c;
    }
  }
  return best;
}

// The planes a call takes at a time with `limit` bytes of scratch for `rows` rows of
// planes, and the planes of a slab: whole slabs, the widest choice that fits (the
// narrowest where not even one fits; then the limit is exceeded).
static int planes_at_once(int n, size_t rows, size_t esize, size_t limit, int* rl) {
  const size_t most = limit / (rows * esize);
  *rl = slab_planes(n, esize, most);
  const size_t slabs = (n + *rl - 1) / *rl, fit = most / *rl;
  return slabs <= fit ? n : *rl * (int)(fit < 1 ? 1 : fit);
}
size_t zscratch_bytes(int n, size_t rows, size_t esize, size_t limit) {
  int rl;
  const size_t nz = planes_at_once(n, rows, esize, limit, &rl);
  return rows * ((nz + rl - 1) / rl * (size_t)rl) * esize;
}

template <typename T>
static int launch_zlast(const void* in, void* out, int nz, int ni, int no, size_t so, size_t sz,
                        int rl, cudaStream_t st) {
  const int zn = (nz + rl - 1) / rl * rl;
  const dim3 grid((ni + 31) / 32, (zn + 31) / 32, no);
  k_zlast<T><<<grid, dim3(32, 8), 0, st>>>((const T*)in, (T*)out, nz, ni, so, sz, rl);
  count_launch();
  return check_launch("k_zlast");
}

// the consumer of k_zlast's output: may start before k_zlast has finished
template <typename... KArgs, typename... Args>
static void launch_after_zlast(void (*kern)(KArgs...), dim3 grid, int threads, size_t smem,
                               cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);  // errors: check_launch
  count_launch();
}

// f(V, C) as compile-time constants for a slab of rl planes
template <class Fn>
static void with_slab(int rl, Fn f) {
  switch (rl) {
    case 32: f(std::integral_constant<int, 1>(), std::integral_constant<int, 1>()); break;
    case 64: f(std::integral_constant<int, 2>(), std::integral_constant<int, 1>()); break;
    case 96: f(std::integral_constant<int, 1>(), std::integral_constant<int, 3>()); break;
    case 128: f(std::integral_constant<int, 4>(), std::integral_constant<int, 1>()); break;
    case 160: f(std::integral_constant<int, 1>(), std::integral_constant<int, 5>()); break;
    case 192: f(std::integral_constant<int, 2>(), std::integral_constant<int, 3>()); break;
    case 256: f(std::integral_constant<int, 4>(), std::integral_constant<int, 2>()); break;
    case 320: f(std::integral_constant<int, 2>(), std::integral_constant<int, 5>()); break;
    default: f(std::integral_constant<int, 4>(), std::integral_constant<int, 3>()); break;
  }
}

// FP64: planes per lane, of the widths 1, 2 and 4 up to vmax the one of least
// cost: FP64 instructions, idle lanes included, plus `extra` per slab for what a
// slab repeats (the weights of P^T: about 60 instructions a voxel and angle
// against 2.3 V; P's lists serve all slabs of a CTA); the wider on ties
static int choose_v64(int n, int vmax, float extra) {
  int best = 1;
  float best_cost = 1e30f;
  for (int v = 1; v <= vmax; v *= 2) {
    const float c = ((float)v + extra) * (float)((n + 32 * v - 1) / (32 * v));
    if (c <= best_cost) {
      best = v;
      best_cost = c;
    }
  }
  return best;
}

// planes z0 .. z0 + nz - 1 of P in slabs of rl
static int project_planes(const Plan& pl, const void* p, void* g, const void* sub, const void* mask,
                          void* scratch, int z0, int nz, int rl, cudaStream_t st) {
  const int n = pl.n, slabs = (nz + rl - 1) / rl;
  const size_t so = pl.np, sz = (size_t)n * pl.np;  // p[z][y][x] in rows of np
  const size_t es = pl.esize, row0 = (size_t)z0 * n;
  auto at = [&](const void* q) { return q ? (const char*)q + row0 * es : nullptr; };
  const void* pz = (const char*)p + (size_t)z0 * sz * es;
  if (pl.prec == FFPAT_FP64) {
    const int rc = launch_zlast<double>(pz, scratch, nz, n, n, so, sz, rl, st);
    if (rc != FFPAT_OK) return rc;
    const int V = choose_v64(nz, 2, 0.2f);
    // slabs of 32 V planes, up to four of them in a CTA (they share the sample
    // lists), two rays a warp and at most 12 warps; fewer rays a CTA while the
    // grid would not give every SM two
    const int vs = (nz + 32 * V - 1) / (32 * V), nslab = vs < 4 ? vs : 4;
    int rg = nslab == 1 ? 16 : (nslab == 2 ? 12 : (nslab == 3 ? 8 : 6));
    const int zg = (vs + nslab - 1) / nslab;
    while (rg > 4 && (n + rg - 1) / rg * (long long)pl.nth * zg < 2 * kNumSMs) rg -= 4;
    const size_t list = (size_t)kP64Samples * rg * 36, stage = (size_t)nslab * 32 * V * (rg + 1) * 8;
    launch_after_zlast(V == 2 ? k_project_z64<2> : k_project_z64<1>,
                       dim3((n + rg - 1) / rg, pl.nth, zg), 32 * nslab * (rg / 2),
                       list > stage ? list : stage, st, (const double*)scratch,
                       (double*)at(g), (const double*)at(sub), (const double*)at(mask), pl.tab,
                       pl.tabf, n, nz, pl.nth, pl.ns, pl.nimg, rl, nslab, rg);
    return check_launch("k_project_z64");
  }
  const int rc = launch_zlast<float>(pz, scratch, nz, n, n, so, sz, rl, st);
  if (rc != FFPAT_OK) return rc;
  // 16 warps a CTA: one a ray where the rays fill two CTAs on every SM, else
  // two or four a ray, and longer row blocks between the CTA's barriers (latency
  // is the bound there: 68^3, 17 angles 25 -> 12 us)
  const long long rays = (long long)n * pl.nth * slabs, fill = 2LL * kNumSMs * kPWarps;
  const int split = rays >= fill ? 1 : (2 * rays >= fill ? 2 : 4), rg = kPWarps / split;
  const int ch = split == 1 ? 32 : 128;
  const size_t list = (size_t)ch * rg * 20, stage = (size_t)split * rl * (rg + 1) * 4;
  with_slab(rl, [&](auto V, auto C) {
    launch_after_zlast(k_project_z<V.value, C.value>, dim3((n + rg - 1) / rg, pl.nth, slabs),
                       32 * kPWarps, list > stage ? list : stage, st, (const float*)scratch,
                       (float*)at(g), (const float*)at(sub), (const float*)at(mask), pl.tabi, n, nz,
                       pl.nth, pl.ns, pl.nimg, rg, ch);
  });
  return check_launch("k_project_z");
}

int launch_project(const Plan& pl, const void* p, void* g, const void* sub, cudaStream_t st,
                   const void* mask, Scratch scratch) {
  const size_t rows = (size_t)pl.n * pl.n;
  if (!scratch.p || zscratch_bytes(pl.n, rows, pl.esize, scratch.bytes) > scratch.bytes)
    return report(FFPAT_EINVAL, "launch_project: %zu bytes of scratch", scratch.bytes);
  int rl;
  const int step = planes_at_once(pl.n, rows, pl.esize, scratch.bytes, &rl);
  for (int z0 = 0; z0 < pl.n; z0 += step) {
    const int nz = pl.n - z0 < step ? pl.n - z0 : step;
    const int rc = project_planes(pl, p, g, sub, mask, scratch.p, z0, nz, rl, st);
    if (rc != FFPAT_OK) return rc;
  }
  return FFPAT_OK;
}

// planes z0 .. z0 + nz - 1 of P^T in slabs of rl
static int backproject_planes(const Plan& pl, const void* g, void* h, const void* scale,
                              void* scratch, int z0, int nz, int rl, double mult,
                              cudaStream_t st) {
  const int n = pl.n, slabs = (nz + rl - 1) / rl;
  const size_t nn = (size_t)n * n, es = pl.esize, vol0 = (size_t)z0 * n * pl.np;
  const void* gz = (const char*)g + (size_t)z0 * n * es;
  auto at = [&](const void* q) { return q ? (const char*)q + vol0 * es : nullptr; };
  if (pl.prec == FFPAT_FP64) {
    const int rc = launch_zlast<double>(gz, scratch, nz, n, pl.nth, nn, (size_t)n, rl, st);
    if (rc != FFPAT_OK) return rc;
    const int V = choose_v64(nz, 4, 0.8f), vs = (nz + 32 * V - 1) / (32 * V);
    int tb = 2;  // tb x tb blocks of 2 x 2 voxels a CTA
    if ((long long)((n + 3) / 4) * ((n + 3) / 4) * vs < 2 * kNumSMs) tb = 1;
    const int side = 2 * tb, tiles = (n + side - 1) / side;
    const size_t list = (size_t)tb * tb * kB64WarpBytes, stage = (size_t)side * side * 32 * V * 8;
    launch_after_zlast(
        V == 4 ? k_backproject_z64<4> : (V == 2 ? k_backproject_z64<2> : k_backproject_z64<1>),
        dim3(tiles, tiles, vs), 32 * tb * tb, list > stage ? list : stage, st,
        (const double*)scratch, (double*)at(h), (const double*)at(scale), pl.tab, n, pl.np, nz,
        pl.nth, pl.ns, pl.nimg, rl, tb, mult);
    return check_launch("k_backproject_z64");
  }
  const int rc = launch_zlast<float>(gz, scratch, nz, n, pl.nth, nn, (size_t)n, rl, st);
  if (rc != FFPAT_OK) return rc;
  // blocks of 2 x 2 voxels a CTA: neighbouring blocks share detectors in L1;
  // fewer while the grid would not give every SM two CTAs
  int tx = kBTileX, ty = kBTileY;
  auto ctas = [&] {
    return (long long)((n + 2 * tx - 1) / (2 * tx)) * ((n + 2 * ty - 1) / (2 * ty)) * slabs;
  };
  if (ctas() < 2 * kNumSMs) tx = 2;
  if (ctas() < 2 * kNumSMs) ty = 1;
  if (ctas() < 2 * kNumSMs) tx = 1;
  const size_t list = (size_t)tx * ty * kBWarpBytes;
  with_slab(rl, [&](auto V, auto C) {
    const size_t stage = (size_t)32 * V.value * (4 * tx * ty + 1) * 4;
    launch_after_zlast(k_backproject_z<V.value, C.value>,
                       dim3((n + 2 * tx - 1) / (2 * tx), (n + 2 * ty - 1) / (2 * ty), slabs),
                       32 * tx * ty, list > stage ? list : stage, st, (const float*)scratch,
                       (float*)at(h), (const float*)at(scale), pl.tabf, pl.tabi, n, pl.np, nz,
                       pl.nth, pl.ns, pl.nimg, tx, (float)mult);
  });
  return check_launch("k_backproject_z");
}

int launch_backproject(const Plan& pl, const void* g, void* h, const void* scale, cudaStream_t st,
                       Scratch scratch, double mult) {
  const size_t rows = (size_t)pl.nth * pl.n;
  if (!scratch.p || zscratch_bytes(pl.n, rows, pl.esize, scratch.bytes) > scratch.bytes)
    return report(FFPAT_EINVAL, "launch_backproject: %zu bytes of scratch", scratch.bytes);
  int rl;
  const int step = planes_at_once(pl.n, rows, pl.esize, scratch.bytes, &rl);
  for (int z0 = 0; z0 < pl.n; z0 += step) {
    const int nz = pl.n - z0 < step ? pl.n - z0 : step;
    const int rc = backproject_planes(pl, g, h, scale, scratch.p, z0, nz, rl, mult, st);
    if (rc != FFPAT_OK) return rc;
  }
  return FFPAT_OK;
}

template <typename T, int NEAR>
static int ramp_launch(const Plan& pl, const void* r, void* out, const void* mask,
                       cudaStream_t st) {
  const int n = pl.n, rows = pl.nth * n;
  // pairs of warps (both parities of 2 kROut outputs), up to eight a CTA, spread
  // evenly; 512 inputs staged at a time (all of them up to 512^3)
  const int pairs = (n + 2 * kROut - 1) / (2 * kROut), gy = (pairs + 7) / 8;
  const int warps = 2 * ((pairs + gy - 1) / gy), nout = warps * kROut;
  const int jc = n < 512 ? (n + 1) / 2 * 2 : 512, H = n / 2 + 2 * kROut + nout / 2;
  const size_t smem =
      ((size_t)ramp_rows(n, jc, nout, gy, NEAR) * kRPitch + 2 * (size_t)H) * sizeof(T);
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(k_ramp<T, NEAR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                220 * 1024);
  });
  if (attr != cudaSuccess || smem > 220 * 1024) {
    cudaGetLastError();
    return report(FFPAT_ECUDA, "k_ramp: %zu bytes of shared memory refused", smem);
  }
  k_ramp<T, NEAR><<<dim3((rows + 31) / 32, gy), 32 * warps, smem, st>>>(
      (const T*)r, (T*)out, (const T*)mask, n, pl.nimg, rows, jc);
  count_launch();
  return check_launch("k_ramp");
}

int launch_ramp(const Plan& pl, const void* r, void* out, cudaStream_t st, const void* mask) {
  return pl.prec == FFPAT_FP64 ? ramp_launch<double, 3>(pl, r, out, mask, st)
         : pl.n <= 448         ? ramp_launch<float, 3>(pl, r, out, mask, st)
                               : ramp_launch<float, 7>(pl, r, out, mask, st);
}

int launch_debug_samples(const Plan& pl, int count, const int32_t* jkm, int32_t* ij, double* f,
                         cudaStream_t st) {
  if (count <= 0) return FFPAT_OK;
  k_debug_samples<<<(count + 127) / 128, 128, 0, st>>>(count, jkm, ij, f, pl.tab, pl.n, pl.nth,
                                                      pl.ns, pl.nimg);
  count_launch();
  return check_launch(__func__);
}

}  // namespace ffpat
