// Resident COCG loop (Eq. 4, Section 4): one thread-block cluster solves one Sternheimer
// system from its first to its last iteration, with the direction p and w = (H - sigma) p (and,
// while they fit, r and x) in the shared memory of its blocks.
//
// Why: launched kernel by kernel, an iteration reads and writes every vector through L2 or
// HBM, costs five launches, and once most systems of a batch have retired the launches run
// over a few blocks, bound by latency.  Here a system's iterations need no launch and no
// global traffic but the brick halos of p; systems retire by their cluster ending, and the
// hardware starts the next one in its place.
//
// Layout: the grid is cut into gy x gz bricks of full x rows, one per block.  Per iteration
//   A  p = r + beta p in the brick; p also goes to global memory (L2) for the neighbours;
//      projector sums chi^T p over the brick's entries
//   -- cluster barrier 1 (the x part of the stencil, which needs no halo, runs inside it)
//   B  projector coefficients gathered from the blocks that touch each group (distributed
//      shared memory); z and y parts, diagonal and projector term of w; p^T w
//   -- cluster barrier 2: alpha
//   C  r -= alpha w, x += alpha p; ||r||^2, r^T r
//   -- cluster barrier 3: convergence, beta
// Each part of the stencil runs along one axis: a thread takes a segment of L outputs of one
// grid line, loads the L + 2R inputs once (brick points from shared memory, halo points from
// L2) and accumulates the L sums in registers, so a point costs about three shared-memory
// reads per axis instead of 2R.  FP32 complex values are one 64-bit register pair and all
// their arithmetic is packed (fma.rn.f32x2).
// What bounds it: FP64, the FP64 pipe (1.7 multiply-adds per clock and SM; about 125 per point
// and iteration); FP32, latency -- 16 warps per SM, phases separated by barriers; 41 % of the issue
// slots and 4 TB/s of L2 are used.  Cycles per iteration (with clock reads between the phases):
//                              26^3 FP32, two blocks   26^3 FP64, four   12^3 FP64, sixteen
//   direction and update             10,900                35,000              2,550
//   projector entries, from L2       26,400                86,500                  -
//   x, z and y parts                 29,700               187,000             13,200
//   coefficients                      1,400                 2,000                100
//   sums over the block               2,200                 4,700              2,800
//   the three cluster barriers        4,300                50,300              3,600
//   scalar steps                      4,100                 4,200              3,900
// (26^3 FP64: the bricks of 13 x 13 rows hold unequal numbers of projector entries, and the others
// wait 43,000 cycles for the fullest.)
// Every block of a cluster computes alpha, beta and the status from the same partial sums in
// the same order, so all of them take the same branches; the barriers are the hardware's.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "cocg.cuh"
#include "cocg_resident.cuh"
#include "fused_dev.cuh"

namespace rpa {

namespace {

namespace cg = cooperative_groups;

// ---- one complex value as the unit of arithmetic ----------------------------------------
using u64 = unsigned long long;
struct alignas(16) d2 {
  double re, im;
};
template <typename T>
struct Val;
template <>
struct Val<float> {
  using V = u64;  // (re, im) packed
  using K = u64;  // (k, k)
};
template <>
struct Val<double> {
  using V = d2;
  using K = double;
};

__device__ __forceinline__ u64 mkv(float a, float b) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ d2 mkv(double a, double b) { return d2{a, b}; }
__device__ __forceinline__ void parts(u64 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ void parts(const d2& v, double& a, double& b) {
  a = v.re;
  b = v.im;
}
__device__ __forceinline__ u64 mkk(float k) { return mkv(k, k); }
__device__ __forceinline__ double mkk(double k) { return k; }
// a + k v, k real
__device__ __forceinline__ u64 kfma(u64 a, u64 k, u64 v) {
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(k), "l"(v), "l"(a));
  return r;
}
__device__ __forceinline__ d2 kfma(const d2& a, double k, const d2& v) {
  return d2{fma(k, v.re, a.re), fma(k, v.im, a.im)};
}
__device__ __forceinline__ u64 vadd(u64 a, u64 b) {
  u64 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ d2 vadd(const d2& a, const d2& b) { return d2{a.re + b.re, a.im + b.im}; }
// a + z v for complex z = (zr, zi)
__device__ __forceinline__ u64 cfma(u64 a, float zr, float zi, u64 v) {
  float x, y;
  parts(v, x, y);
  return kfma(kfma(a, mkk(zr), v), mkv(-zi, zi), mkv(y, x));
}
__device__ __forceinline__ d2 cfma(const d2& a, double zr, double zi, const d2& v) {
  return d2{fma(-zi, v.im, fma(zr, v.re, a.re)), fma(zi, v.re, fma(zr, v.im, a.im))};
}
template <typename T>
__device__ __forceinline__ typename Val<T>::V vzero() {
  return mkv((T)0, (T)0);
}
// L2 accesses (data other blocks of the cluster write or read)
__device__ __forceinline__ u64 ldg2(const u64* p) { return __ldcg(p); }
__device__ __forceinline__ d2 ldg2(const d2* p) {
  const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
  return d2{v.x, v.y};
}
__device__ __forceinline__ void stg2(u64* p, u64 v) { __stcg(p, v); }
__device__ __forceinline__ void stg2(d2* p, const d2& v) {
  __stcg(reinterpret_cast<double2*>(p), make_double2(v.re, v.im));
}

template <typename T>
struct Args {
  Stencil<T> st;
  const T* vloc;
  long long nd;
  int ns, nb;
  const double *eps, *omega;
  typename Val<T>::V *x, *r, *p, *p_odd;
  double* sysd;
  int* sysi;
  int maxit, cont;
  int G, gy, gz, cap, pitch, lx, ly, lz, r_res, x_res;
  unsigned mg_pitch, mg_nx;  // exact quotients of values below 2^16 (see quot)
  ResidentProj<T> pj;
};

// The thread's index, read anew: what a phase derives from it is not kept (and spilled) across
// the iteration loop.
__device__ __forceinline__ int tid() {
  int r;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ int quot(int a, unsigned magic) { return (int)__umulhi((unsigned)a, magic); }

// ---- per-system scalars ------------------------------------------------------------------
// The sums over warps and blocks, rho, ||r||^2, its target and the quotients alpha and beta are
// FP64 in both forms, as in the launched iteration.  An FP64 instruction takes 64 cycles of a
// warp whatever its active lanes, so the values that belong together go through one instruction
// in lanes of their own, and what can be read off the bits is.
__device__ __forceinline__ bool finite_bits(double v) {
  return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;
}
__device__ __forceinline__ bool zero_bits(double v) {
  return ((__double2hiint(v) & 0x7fffffff) | __double2loint(v)) == 0;
}
// a <= b for finite values >= 0
__device__ __forceinline__ bool le_bits(double a, double b) {
  return __double_as_longlong(a) <= __double_as_longlong(b);
}
// (ar + i ai) / (br + i bi): the real part in even lanes, the imaginary part in odd ones.  A
// division, not a product with the reciprocal of |b|^2: that of a subnormal |b|^2 overflows.
__device__ __forceinline__ double cdiv_lanes(double ar, double ai, double br, double bi, int lane) {
  const bool im = (lane & 1) != 0;
  const double p = im ? ai : ar, q = im ? -ar : ai;
  return (p * br + q * bi) / (br * br + bi * bi);
}

template <typename T>
struct Brick;
// The block's Brick, at the start of its dynamic shared memory, and its vectors behind it.  All
// of them are found from the array itself: a pointer kept in memory, or passed to a function,
// would lose that it points to shared memory.
template <typename T>
__device__ __forceinline__ Brick<T>& brick();
template <typename T>
__device__ __forceinline__ typename Val<T>::V* smem_vec(int off);

// What the phases of one block share.  The phases are functions of their own that read what they
// need from here, so that nothing lives in registers from phase to phase: with most of the SM's
// memory taken by p and w there is little L1 left, and a spilled register costs an L2 access.
template <typename T>
struct alignas(16) Brick {
  using V = typename Val<T>::V;
  using K = typename Val<T>::K;
  V *xg, *rg, *pg;  // x, r and p of the system in global memory
  int nx, ny, nz, y0, z0, by, bz, pitch, cap, nslot, rank, ng4;
  int px, py, pz;  // periodic axes
  T eps, om, be_r, be_i, al_r, al_i;
  double rho_r, rho_i, rn2, target2;
  int ctl, iters;
  K kc[3 * (kMaxRadius + 1)];  // stencil coefficients per axis
  dacc_t<T> red[32 * 4];
  double slots2[kResMaxCluster * 4], slots3[kResMaxCluster * 4];
  Args<T> a;  // the launch's arguments
  // offsets of the vectors: p at 0, w, r and x (if resident), projector sums and coefficients
  __device__ int off_w() const { return cap; }
  __device__ int off_r() const { return 2 * cap; }
  __device__ int off_x() const { return (2 + a.r_res) * cap; }
  __device__ int off_cps() const { return (2 + a.r_res + a.x_res) * cap; }
  __device__ int off_cpt() const { return off_cps() + ng4; }
  __device__ int* rowoff() const { return reinterpret_cast<int*>(smem_vec<T>(off_cpt() + ng4)); }
};

template <typename T>
__device__ __forceinline__ Brick<T>& brick() {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  return *reinterpret_cast<Brick<T>*>(dyn_smem);
}
template <typename T>
__device__ __forceinline__ typename Val<T>::V* smem_vec(int off) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  return reinterpret_cast<typename Val<T>::V*>(dyn_smem + sizeof(Brick<T>)) + off;
}

// sums of one segment: acc[i] += sum_m c_m (v[i + R - m] + v[i + R + m])
template <typename T, int L, int R>
__device__ __forceinline__ void seg_sums(typename Val<T>::V (&acc)[L],
                                         const typename Val<T>::V (&v)[L + 2 * R],
                                         const typename Val<T>::K (&c)[R + 1]) {
  // the brick's own points first (the middle), then outwards to the halo points, whose loads
  // take longest
#pragma unroll
  for (int jj = 0; jj < L + 2 * R; ++jj) {
    const int o = jj - L;  // 0, 1, 2, ...: R - 1, R + L, R - 2, R + L + 1, ...
    const int j = jj < L ? R + jj : ((o & 1) ? R + L + o / 2 : R - 1 - o / 2);
#pragma unroll
    for (int i = 0; i < L; ++i) {
      const int m = j - R - i;
      if (m != 0 && m >= -R && m <= R) acc[i] = kfma(acc[i], c[m < 0 ? -m : m], v[j]);
    }
  }
}

// Unit u of a warp: its lane's segment and line.  FP32: a warp takes 32 lines of one segment,
// so that the segment's edges are uniform in it.  FP64: segments and lines are dealt to the
// lanes without gaps -- an FP64 instruction occupies its pipe for 64 cycles whatever the number
// of lanes that need it, and a small brick has few lines.
template <typename T>
__device__ __forceinline__ int units_of(int lines, int segs) {
  return sizeof(T) == 8 ? (lines * segs + 31) >> 5 : ((lines + 31) >> 5) * segs;
}
template <typename T>
__device__ __forceinline__ bool unit(int u, int lane, int lines, int segs, int& seg, int& line) {
  if (sizeof(T) == 8) {
    const int v = u * 32 + lane;
    seg = v / lines;
    line = v - seg * lines;
    return seg < segs;
  }
  const int lw = (lines + 31) >> 5;
  seg = u / lw;
  line = (u - seg * lw) * 32 + lane;
  return line < lines;
}
__device__ __forceinline__ int warp_id() { return __shfl_sync(0xffffffffu, tid() >> 5, 0); }

// Segments of L outputs of a line of b points, evenly spread, the first at 0 and the last at
// b - L: outputs that two segments share belong to the second.
struct Segs {
  int n, num, den;
  __device__ Segs(int b, int L) {
    n = (b + L - 1) / L;
    num = b > L ? b - L : 0;
    den = max(n - 1, 1);
  }
  __device__ int start(int s) const { return (s * num + den / 2) / den; }
};

// x part: W = (rows of the brick, lanes over rows)
template <typename T, int L, int R>
__device__ __noinline__ void part_x() {
  const Brick<T>& k = brick<T>();
  using V = typename Val<T>::V;
  typename Val<T>::K c[R + 1];
#pragma unroll
  for (int m = 1; m <= R; ++m) c[m] = k.kc[m];
  const int nx = k.nx, pitch = k.pitch, nrow = k.by * k.bz, per = k.px;
  const Segs sg(nx, L);
  const int units = units_of<T>(nrow, sg.n);
  const V* const P = smem_vec<T>(0);
  V* const W = smem_vec<T>(k.off_w());
  const int lane = tid() & 31, nw = blockDim.x >> 5;
#pragma unroll 1
  for (int u = warp_id(); u < units; u += nw) {
    int seg, row;
    if (!unit<T>(u, lane, nrow, sg.n, seg, row)) continue;
    const int i0 = sg.start(seg), keep = (seg + 1 < sg.n ? sg.start(seg + 1) : nx) - i0;
    const V* const p = P + row * pitch + i0;
    V v[L + 2 * R];
    // R points to the left and to the right: of the row, of its other end, or zeros; wl, wr:
    // how many of them lie beyond the row's ends
    const int wl = max(R - i0, 0), wr = max(i0 + L + R - nx, 0);
    if ((wl == 0 || wl == R) && (wr == 0 || wr == R)) {
      const V* const pl = p + (wl ? nx - R : -R);
      const V* const pr = p + (wr ? L - nx : L);
#pragma unroll
      for (int j = 0; j < R; ++j) {
        v[j] = v[R + L + j] = vzero<T>();
        if (!wl || per) v[j] = pl[j];
        if (!wr || per) v[R + L + j] = pr[j];
      }
    } else {
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const int xl = i0 - R + j, xr = i0 + L + j;
        v[j] = v[R + L + j] = vzero<T>();
        if (xl >= 0 || per) v[j] = p[xl >= 0 ? j - R : j - R + nx];
        if (xr < nx || per) v[R + L + j] = p[xr < nx ? L + j : L + j - nx];
      }
    }
#pragma unroll
    for (int j = 0; j < L; ++j) v[R + j] = p[j];
    V acc[L];
#pragma unroll
    for (int i = 0; i < L; ++i) acc[i] = vzero<T>();
    seg_sums<T, L, R>(acc, v, c);
    V* const w = W + row * pitch + i0;
#pragma unroll
    for (int i = 0; i < L; ++i)
      if (i < keep) w[i] = acc[i];
  }
}

// One axis of the brick: origin o and length b of the brick, extent n of the grid.
struct Axis {
  int o, b, n, per;
};
// N consecutive inputs from brick coordinate q0 of one line (shared memory sp, stride ss;
// global memory gp, stride gs), some of them outside the brick: from the neighbours' bricks
// through global memory, or the brick's own other end where the axis is not cut.
template <typename T, int N>
__device__ __forceinline__ void wing(typename Val<T>::V* v, const typename Val<T>::V* sp, int ss,
                                     const typename Val<T>::V* gp, int gs, int q0, const Axis& x) {
  if (q0 >= 0 && q0 + N <= x.b) {
    const typename Val<T>::V* p = sp + q0 * ss;
#pragma unroll
    for (int j = 0; j < N; ++j, p += ss) v[j] = *p;
    return;
  }
  int g0 = x.o + q0;  // the whole run wraps, or lies outside a Dirichlet axis, or neither
  if (g0 + N <= 0 || g0 >= x.n) {
    if (!x.per) {
#pragma unroll
      for (int j = 0; j < N; ++j) v[j] = vzero<T>();
      return;
    }
    g0 += g0 < 0 ? x.n : -x.n;
  }
  if ((q0 + N <= 0 || q0 >= x.b) && g0 >= 0 && g0 + N <= x.n) {
    if (x.b == x.n) {
      const typename Val<T>::V* p = sp + g0 * ss;
#pragma unroll
      for (int j = 0; j < N; ++j, p += ss) v[j] = *p;
      return;
    }
    if (g0 + N <= x.o || g0 >= x.o + x.b) {
      const typename Val<T>::V* p = gp + (long long)g0 * gs;
#pragma unroll
      for (int j = 0; j < N; ++j, p += gs) v[j] = ldg2(p);
      return;
    }
  }
  // anything else, point by point
#pragma unroll
  for (int j = 0; j < N; ++j) {
    int g = x.o + q0 + j;
    const bool out = g < 0 || g >= x.n;
    g += g < 0 ? x.n : (g >= x.n ? -x.n : 0);
    const int q = g - x.o;
    v[j] = vzero<T>();
    if ((!out || x.per) && g >= 0 && g < x.n)
      v[j] = (q >= 0 && q < x.b) ? sp[q * ss] : ldg2(gp + (long long)g * gs);
  }
}
// the L + 2R inputs of the segment from i0, halo first
template <typename T, int L, int R>
__device__ __forceinline__ void line_load(typename Val<T>::V (&v)[L + 2 * R],
                                          const typename Val<T>::V* sp, int ss,
                                          const typename Val<T>::V* gp, int gs, int i0,
                                          const Axis& x) {
  wing<T, R>(v, sp, ss, gp, gs, i0 - R, x);
  wing<T, R>(v + R + L, sp, ss, gp, gs, i0 + L, x);
  const typename Val<T>::V* p = sp + i0 * ss;
#pragma unroll
  for (int j = 0; j < L; ++j, p += ss) {
    v[R + j] = vzero<T>();
    if (i0 + j < x.b) v[R + j] = *p;
  }
}

// z part: W += (columns of the brick, lanes over x)
template <typename T, int L, int R>
__device__ __noinline__ void part_z() {
  const Brick<T>& k = brick<T>();
  using V = typename Val<T>::V;
  typename Val<T>::K c[R + 1];
#pragma unroll
  for (int m = 1; m <= R; ++m) c[m] = k.kc[2 * (kMaxRadius + 1) + m];
  const int nx = k.nx, by = k.by, pitch = k.pitch, ncol = nx * by;
  const int stride = by * pitch, plane = nx * k.ny;
  const unsigned mg_nx = k.a.mg_nx;
  const Axis ax{k.z0, k.bz, k.nz, k.pz};
  const Segs sg(ax.b, L);
  const int units = units_of<T>(ncol, sg.n);
  const V* const P = smem_vec<T>(0);
  V* const W = smem_vec<T>(k.off_w());
  const V* const pg = k.pg + nx * k.y0;
  const int lane = tid() & 31, nw = blockDim.x >> 5;
#pragma unroll 1
  for (int u = warp_id(); u < units; u += nw) {
    int seg, col;
    if (!unit<T>(u, lane, ncol, sg.n, seg, col)) continue;
    const int i0 = sg.start(seg), keep = (seg + 1 < sg.n ? sg.start(seg + 1) : ax.b) - i0;
    const int yl = quot(col, mg_nx), base = yl * (pitch - nx) + col;  // yl * pitch + x
    V v[L + 2 * R];
    line_load<T, L, R>(v, P + base, stride, pg + col, plane, i0, ax);
    V acc[L];
    V* const w = W + base + i0 * stride;
#pragma unroll
    for (int i = 0; i < L; ++i) {
      acc[i] = vzero<T>();
      if (i < keep) acc[i] = w[i * stride];
    }
    seg_sums<T, L, R>(acc, v, c);
#pragma unroll
    for (int i = 0; i < L; ++i)
      if (i < keep) w[i * stride] = acc[i];
  }
}

// y part, diagonal and the end of w: W += y sums + (c0 + V - sigma) p; sums p^T w
template <typename T, int L, int R>
__device__ __noinline__ cpx<dacc_t<T>> part_y() {
  const Brick<T>& k = brick<T>();
  using V = typename Val<T>::V;
  using D = dacc_t<T>;
  typename Val<T>::K c[R + 1];
#pragma unroll
  for (int m = 1; m <= R; ++m) c[m] = k.kc[kMaxRadius + 1 + m];
  const int nx = k.nx, pitch = k.pitch, ncol = nx * k.bz;
  const int plane = nx * k.ny, zstep = k.by * pitch;
  const unsigned mg_nx = k.a.mg_nx;
  const Axis ax{k.y0, k.by, k.ny, k.py};
  const Segs sg(ax.b, L);
  const int units = units_of<T>(ncol, sg.n);
  const V* const P = smem_vec<T>(0);
  V* const W = smem_vec<T>(k.off_w());
  const V* const pg = k.pg + plane * k.z0;
  const T* const vloc = k.a.vloc + plane * k.z0 + nx * k.y0;
  const T c0 = k.a.st.c0, eps = k.eps, om = k.om;
  V sum = vzero<T>();
  D dre = 0, dim = 0;  // the sum where its type is not T (RPA_DOT_F64)
  const int lane = tid() & 31, nw = blockDim.x >> 5;
#pragma unroll 1
  for (int u = warp_id(); u < units; u += nw) {
    int seg, col;
    if (!unit<T>(u, lane, ncol, sg.n, seg, col)) continue;
    const int i0 = sg.start(seg), keep = (seg + 1 < sg.n ? sg.start(seg + 1) : ax.b) - i0;
    const int zl = quot(col, mg_nx), x = col - zl * nx;
    const int base = zl * zstep + x, gl = zl * plane + x;
    T vl[L];
#pragma unroll
    for (int i = 0; i < L; ++i) {
      vl[i] = (T)0;
      if (i < keep) vl[i] = __ldg(vloc + gl + nx * (i0 + i));
    }
    V v[L + 2 * R];
    line_load<T, L, R>(v, P + base, pitch, pg + gl, nx, i0, ax);
    V acc[L];
    V* const w = W + base + i0 * pitch;
#pragma unroll
    for (int i = 0; i < L; ++i) {
      acc[i] = vzero<T>();
      if (i < keep) acc[i] = w[i * pitch];
    }
    seg_sums<T, L, R>(acc, v, c);
#pragma unroll
    for (int i = 0; i < L; ++i)
      if (i < keep) {
        const V pc = v[i + R];
        // (c0 + V - eps) p - i omega p; in FP32 eps in a term of its own, so that the
        // coefficient is rounded once
        V wv;
        if constexpr (sizeof(T) == 4)
          wv = kfma(cfma(acc[i], c0 + vl[i], -om, pc), mkk(-eps), pc);
        else
          wv = cfma(acc[i], vl[i] + (c0 - eps), -om, pc);
        w[i * pitch] = wv;
        T pr, pi;
        parts(pc, pr, pi);
        if constexpr (std::is_same<D, T>::value) {
          sum = cfma(sum, pr, pi, wv);
        } else {
          T wr, wi;
          parts(wv, wr, wi);
          dre += (D)pr * wr - (D)pi * wi;
          dim += (D)pr * wi + (D)pi * wr;
        }
      }
  }
  if constexpr (!std::is_same<D, T>::value) return mk<D>(dre, dim);
  T sre, sim;
  parts(sum, sre, sim);
  return mk<D>(sre, sim);
}

// Sums of NQ (2 or 4) values over the block; every lane of warp 0 gets them.  Within a warp the
// lanes exchange halves of the values first, so that each adds one value in the end.
template <typename T, int NQ>
__device__ __forceinline__ void block_total(T (&v)[NQ], T* red, double (&out)[NQ]) {
  const int lane = tid() & 31, wid = tid() >> 5, nw = blockDim.x >> 5;
  int o = 16, q = 0;
#pragma unroll
  for (int h = NQ / 2; h >= 1; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
    if (up) q += h;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const T give = up ? v[i] : v[i + h];
      v[i] = (up ? v[i + h] : v[i]) + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  if ((lane & (32 / NQ - 1)) == 0) red[wid * NQ + q] = v[0];
  __syncthreads();
  if (wid == 0) {
    // warp 0 holds value q of warps w, w + 32 / NQ in lane q * (32 / NQ) + w: one addition and
    // one tree for all values together (FP64 additions take 64 cycles of the pipe each)
    constexpr int S = 32 / NQ;
    const int qq = lane / S, w = lane % S;
    double t = w < nw ? (double)red[w * NQ + qq] : 0.0;
    if (nw > S) t += w + S < nw ? (double)red[(w + S) * NQ + qq] : 0.0;
#pragma unroll
    for (int x = S / 2; x > 0; x >>= 1)
      if (x < nw) t += __shfl_xor_sync(0xffffffffu, t, x);
#pragma unroll
    for (int i = 0; i < NQ; ++i) out[i] = __shfl_sync(0xffffffffu, t, i * S);
  }
}

// Sum over the blocks of the cluster: warp 0 puts the block's totals into every block's slots;
// after the barrier warp 0 of each block adds the slots in a fixed tree.
template <int NQ>
__device__ __forceinline__ void post_totals(cg::cluster_group& cl, const double (&v)[NQ],
                                            double* slots, int G, int rank) {
  if ((int)threadIdx.x < G) {
    double* dst = cl.map_shared_rank(slots, threadIdx.x);
#pragma unroll
    for (int q = 0; q < NQ; ++q) dst[rank * 4 + q] = v[q];
  }
}
template <int NQ>
__device__ __forceinline__ void read_totals(const double* slots, int G, double (&v)[NQ]) {
  // value q of blocks r, r + 32 / NQ in lane q * (32 / NQ) + r
  constexpr int S = 32 / NQ;
  const int lane = threadIdx.x & 31, q = lane / S, r = lane % S;
  double t = r < G ? slots[r * 4 + q] : 0.0;
  if (G > S) t += r + S < G ? slots[(r + S) * 4 + q] : 0.0;
  for (int x = 1; x < G && x < S; x <<= 1) t += __shfl_xor_sync(0xffffffffu, t, x);
#pragma unroll
  for (int i = 0; i < NQ; ++i) v[i] = __shfl_sync(0xffffffffu, t, i * S);
}

#define RES_BY_LEN(l, call) \
  switch (l) {              \
    case 1: if constexpr (sizeof(T) == 8) call(1); break; \
    case 2: call(2); break; \
    case 3: if constexpr (sizeof(T) == 8) call(3); break; \
    case 4: call(4); break; \
    case 5: call(5); break; \
    case 6: if constexpr (sizeof(T) == 4) call(6); break; \
    default: if constexpr (sizeof(T) == 4) call(7); break; \
  }

template <typename T>
constexpr int max_threads() {
  return 512;
}


// points of a thread in flight in the pointwise phases
template <typename T>
__host__ __device__ constexpr int batch() {
  return sizeof(T) == 4 ? 4 : 2;
}

// The pointwise and projector phases of an iteration (see the file comment).
// Point i of the brick (rows without their padding): its slot and its grid offset.
__device__ __forceinline__ void locate(int i, unsigned mg_nx, int nx, int pad, const int* rowoff,
                                       int& slot, int& g) {
  const int row = quot(i, mg_nx);
  slot = i + row * pad;
  g = rowoff[row] + i - row * nx;
}

// p = r + beta p; RRES: r in shared memory; SHARE: p also to global memory
template <typename T, bool RRES, bool SHARE>
__device__ __noinline__ void phase_direction() {
  using V = typename Val<T>::V;
  const Brick<T>& k = brick<T>();
  constexpr int U = batch<T>();
  const int T0 = blockDim.x, nx = k.nx, pad = k.pitch - nx, np = k.by * k.bz * nx;
  const unsigned mg = k.a.mg_nx;
  const T be_r = k.be_r, be_i = k.be_i;
  V *const P = smem_vec<T>(0), *const rs = smem_vec<T>(k.off_r()), *const pg = k.pg;
  const V* const rg = k.rg;
  const int* const rowoff = k.rowoff();
  int i0 = tid();
#pragma unroll 1
  for (; i0 + (U - 1) * T0 < np; i0 += U * T0) {
    V rv[U], pv[U];
    int g[U], slot[U];
#pragma unroll
    for (int u = 0; u < U; ++u) locate(i0 + u * T0, mg, nx, pad, rowoff, slot[u], g[u]);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      rv[u] = RRES ? rs[slot[u]] : ldg2(rg + g[u]);
      pv[u] = P[slot[u]];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      pv[u] = cfma(rv[u], be_r, be_i, pv[u]);
      P[slot[u]] = pv[u];
      if (SHARE) stg2(pg + g[u], pv[u]);
    }
  }
#pragma unroll 1
  for (; i0 < np; i0 += T0) {
    int g, slot;
    locate(i0, mg, nx, pad, rowoff, slot, g);
    const V pv = cfma(RRES ? rs[slot] : ldg2(rg + g), be_r, be_i, P[slot]);
    P[slot] = pv;
    if (SHARE) stg2(pg + g, pv);
  }
}

// Projector sums chi^T p over the brick: a warp per record, the partial sums to W (free until
// the x part), then those of each group added in order.  The entries come from L2: all loads
// of a record are issued before the first is used.
template <typename T>
__device__ __noinline__ void phase_proj_sums() {
  const Brick<T>& k = brick<T>();
  const int T0 = blockDim.x, lane = tid() & 31, rank = k.rank, nw = T0 >> 5;
  const typename Val<T>::V* const P = smem_vec<T>(0);
  T* const part = reinterpret_cast<T*>(smem_vec<T>(k.off_w()));
  const int* const rstep = k.a.pj.rstep;
  const unsigned short* const gslot = k.a.pj.gslot + lane;
  const T* const gchi = k.a.pj.gchi + lane * kProjChunk;
  const int q0 = k.a.pj.roff[rank], q1 = k.a.pj.roff[rank + 1];
#pragma unroll 1
  for (int q = q0 + warp_id(); q < q1; q += nw) {
    const int s0 = rstep[q], s1 = rstep[q + 1];
    constexpr int U = res_steps<T>();
    T ch[U][kProjChunk];
    int slot[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      slot[u] = 0;
#pragma unroll
      for (int l = 0; l < kProjChunk; ++l) ch[u][l] = (T)0;
      if (s0 + u < s1) {
        slot[u] = gslot[32 * (s0 + u)];
        load_chi4(gchi + (s0 + u) * (32 * kProjChunk), ch[u]);
      }
    }
    T f[2 * kProjChunk];
#pragma unroll
    for (int l = 0; l < 2 * kProjChunk; ++l) f[l] = (T)0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      T pr, pi;
      parts(P[slot[u]], pr, pi);
#pragma unroll
      for (int l = 0; l < kProjChunk; ++l) {
        f[2 * l] = fma(ch[u][l], pr, f[2 * l]);
        f[2 * l + 1] = fma(ch[u][l], pi, f[2 * l + 1]);
      }
    }
    // lanes exchange halves of the eight sums, so that each adds one in the end
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int o = 16 >> b, h = 4 >> b;
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int i = 0; i < h; ++i) {
        const T give = up ? f[i] : f[i + h];
        f[i] = (up ? f[i + h] : f[i]) + __shfl_xor_sync(0xffffffffu, give, o);
      }
    }
    f[0] += __shfl_xor_sync(0xffffffffu, f[0], 2);
    f[0] += __shfl_xor_sync(0xffffffffu, f[0], 1);
    if ((lane & 3) == 0) part[(q - q0) * 2 * kProjChunk + (lane >> 2)] = f[0];
  }
  __syncthreads();
  const int* const groups = k.a.pj.groups;
  T* const cps = reinterpret_cast<T*>(smem_vec<T>(k.off_cps()));
  const int g0 = k.a.pj.goff[rank], ngl = (k.a.pj.goff[rank + 1] - g0) * 2 * kProjChunk;
#pragma unroll 1
  for (int i = tid(); i < ngl; i += T0) {
    const int q = g0 + i / (2 * kProjChunk), l = i % (2 * kProjChunk);
    const int r1 = groups[3 * q + 2];
    T sum = (T)0;
    for (int r = groups[3 * q + 1]; r < r1; ++r) sum += part[r * 2 * kProjChunk + l];
    cps[groups[3 * q] * 2 * kProjChunk + l] = sum;
  }
  __syncthreads();
}

template <typename T>
__device__ __noinline__ void phase_proj_coef() {
  cg::cluster_group cl = cg::this_cluster();
  const Brick<T>& k = brick<T>();
  const Args<T>& a = k.a;
  const int T0 = blockDim.x;
  using V = typename Val<T>::V;
  // B: projector coefficients of the groups this block touches
  {
    const int ng4 = k.ng4, rank = k.rank, G = a.G;
    V *const cps = smem_vec<T>(k.off_cps()), *const cpt = smem_vec<T>(k.off_cpt());
    const unsigned* const gmask = a.pj.gmask;
    const T* const coef = a.pj.coef;
#pragma unroll 1
    for (int i = tid(); i < ng4; i += T0) {
      const unsigned m = gmask[i / kProjChunk];
      if (!((m >> rank) & 1u)) continue;
      V sum = vzero<T>();
#pragma unroll 4
      for (int q = 0; q < G; ++q)
        if ((m >> q) & 1u) sum = vadd(sum, *cl.map_shared_rank(cps + i, q));
      cpt[i] = kfma(vzero<T>(), mkk(coef[i]), sum);
    }
  }
}

// Projector term W += chi cp, every warp on its own points.
template <typename T>
__device__ __noinline__ void phase_proj_term() {
  const Brick<T>& k = brick<T>();
  constexpr int U = res_steps<T>();
  const int lane = tid() & 31, w = k.rank * (int)(blockDim.x >> 5) + warp_id();
  typename Val<T>::V* const W = smem_vec<T>(k.off_w());
  const typename Val<T>::V* const cpt = smem_vec<T>(k.off_cpt());
  const int s1 = k.a.pj.lwarp[w + 1];
  int s = k.a.pj.lwarp[w];
  const unsigned* const lkey = k.a.pj.lkey + lane;
  const T* const lchi = k.a.pj.lchi + lane * kProjChunk;
#pragma unroll 1
  for (; s < s1; s += U) {
    unsigned key[U];
    T ch[U][kProjChunk];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      key[u] = ~0u;
      if (s + u < s1) {
        key[u] = lkey[32 * (s + u)];
        load_chi4(lchi + (s + u) * (32 * kProjChunk), ch[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      __syncwarp();  // the step before may have written this step's points
      if (key[u] == ~0u) continue;
      const int slot = key[u] & 0xffffu;
      const typename Val<T>::V* const cg4 = cpt + (key[u] >> 16) * kProjChunk;
      T wr, wi, cr, ci;
      parts(W[slot], wr, wi);
#pragma unroll
      for (int j = 0; j < kProjChunk; ++j) {
        parts(cg4[j], cr, ci);
        wr = fma(ch[u][j], cr, wr);
        wi = fma(ch[u][j], ci, wi);
      }
      W[slot] = mkv(wr, wi);
    }
  }
  __syncthreads();
}

// the thread's ||r||^2 and r^T r
template <typename T>
struct Sum3 {
  dacc_t<T> v[3];
};
// r -= alpha w, x += alpha p; RRES, XRES: r and x in shared memory
template <typename T, bool RRES, bool XRES>
__device__ __noinline__ Sum3<T> phase_update() {
  using V = typename Val<T>::V;
  const Brick<T>& k = brick<T>();
  constexpr int U = batch<T>();
  const int T0 = blockDim.x, nx = k.nx, pad = k.pitch - nx, np = k.by * k.bz * nx;
  const unsigned mg = k.a.mg_nx;
  const T al_r = k.al_r, al_i = k.al_i;
  V *const rs = smem_vec<T>(k.off_r()), *const xs = smem_vec<T>(k.off_x()), *const rg = k.rg,
           *const xg = k.xg;
  const V *const P = smem_vec<T>(0), *const W = smem_vec<T>(k.off_w());
  const int* const rowoff = k.rowoff();
  using D = dacc_t<T>;
  D s0 = 0, s1 = 0, s2 = 0;
  auto step = [&](int slot, int g, const V& rv, const V& xv, const V& wv, const V& pv) {
    const V r = cfma(rv, -al_r, -al_i, wv), x = cfma(xv, al_r, al_i, pv);
    if (RRES)
      rs[slot] = r;
    else
      stg2(rg + g, r);
    if (XRES)
      xs[slot] = x;
    else
      stg2(xg + g, x);
    T re, im;
    parts(r, re, im);
    if constexpr (sizeof(T) == 8) {  // three multiply-adds; combined at the end
      s0 = fma(re, re, s0);
      s1 = fma(im, im, s1);
      s2 = fma(re, im, s2);
    } else {
      s0 += (D)re * re + (D)im * im;
      s1 += (D)re * re - (D)im * im;
      s2 += (D)2 * re * im;
    }
  };
  int i0 = tid();
#pragma unroll 1
  for (; i0 + (U - 1) * T0 < np; i0 += U * T0) {
    V rv[U], xv[U], wv[U], pv[U];
    int g[U], slot[U];
#pragma unroll
    for (int u = 0; u < U; ++u) locate(i0 + u * T0, mg, nx, pad, rowoff, slot[u], g[u]);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      xv[u] = XRES ? xs[slot[u]] : ldg2(xg + g[u]);
      rv[u] = RRES ? rs[slot[u]] : ldg2(rg + g[u]);
      wv[u] = W[slot[u]];
      pv[u] = P[slot[u]];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) step(slot[u], g[u], rv[u], xv[u], wv[u], pv[u]);
  }
#pragma unroll 1
  for (; i0 < np; i0 += T0) {
    int g, slot;
    locate(i0, mg, nx, pad, rowoff, slot, g);
    step(slot, g, RRES ? rs[slot] : ldg2(rg + g), XRES ? xs[slot] : ldg2(xg + g), W[slot], P[slot]);
  }
  if constexpr (sizeof(T) == 8) return Sum3<T>{{s0 + s1, s0 - s1, 2 * s2}};
  return Sum3<T>{{s0, s1, s2}};
}

template <typename T, int R>
__global__ void __launch_bounds__(max_threads<T>(), 1) k_cocg_resident(const __grid_constant__ Args<T> arg) {
  using V = typename Val<T>::V;
  cg::cluster_group cl = cg::this_cluster();
  Brick<T>& k = brick<T>();
  const Args<T>& a = k.a;
  {
    const int t = threadIdx.x;
    static_assert(sizeof(Args<T>) % 4 == 0, "copied by words");
    for (int i = t; i < (int)(sizeof(Args<T>) / 4); i += blockDim.x)
      reinterpret_cast<int*>(&k.a)[i] = reinterpret_cast<const int*>(&arg)[i];
    __syncthreads();
    // slow systems first: high states, whose eigenvalue is next to the unoccupied ones
    const int ci = blockIdx.x / a.G;
    const int n = a.ns - 1 - ci / a.nb, b = ci % a.nb, s = b * a.ns + n;
    if (a.sysi[(long long)s * kSysI + kStatus] != kActive) return;  // the whole cluster
    if (t < 3 * (R + 1)) {
      const int ax = t / (R + 1), m = t - ax * (R + 1);
      k.kc[ax * (kMaxRadius + 1) + m] =
          mkk(ax == 0 ? a.st.cx[m] : ax == 1 ? a.st.cy[m] : a.st.cz[m]);
    }
    if (t == 0) {
      const int rank = (int)cl.block_rank();
      const double* sd = a.sysd + (long long)s * kSysD;
      const int ry = rank % a.gy, rz = rank / a.gy;
      k.rank = rank;
      k.nx = a.st.nx;
      k.ny = a.st.ny;
      k.nz = a.st.nz;
      k.y0 = ry * k.ny / a.gy;
      k.z0 = rz * k.nz / a.gz;
      k.by = (ry + 1) * k.ny / a.gy - k.y0;
      k.bz = (rz + 1) * k.nz / a.gz - k.z0;
      k.pitch = a.pitch;
      k.nslot = k.by * k.bz * k.pitch;
      k.px = a.st.bcx == 0;
      k.py = a.st.bcy == 0;
      k.pz = a.st.bcz == 0;
      k.cap = a.cap;
      k.ng4 = a.pj.ngroup * kProjChunk;
      const long long sb = (long long)s * a.nd;
      k.xg = a.x + sb;
      k.rg = a.r + sb;
      k.pg = a.p + sb;
      k.eps = (T)a.eps[n];
      k.om = (T)a.omega[b];
      k.be_r = a.cont ? (T)sd[kBeta] : (T)0;
      k.be_i = a.cont ? (T)sd[kBeta + 1] : (T)0;
      k.rho_r = sd[kRho];
      k.rho_i = sd[kRho + 1];
      k.rn2 = sd[kRnorm] * sd[kRnorm];
      k.target2 = sd[kTarget] * sd[kTarget];
      k.iters = a.sysi[(long long)s * kSysI + kIters];
      k.ctl = kActive;
    }
  }
  __syncthreads();
  const int T0 = blockDim.x;
  {
    int* const rowoff = k.rowoff();
    const int by = k.by, nrow = by * k.bz, nx = k.nx, ny = k.ny, y0 = k.y0, z0 = k.z0;
    for (int i = tid(); i < nrow; i += T0) rowoff[i] = nx * (y0 + i % by + ny * (z0 + i / by));
  }
  __syncthreads();
  {
    const bool keep = k.be_r != (T)0 || k.be_i != (T)0, r_res = a.r_res, x_res = a.x_res;
    V *const P = smem_vec<T>(0), *const W = smem_vec<T>(k.off_w()),
             *const rs = smem_vec<T>(k.off_r()), *const xs = smem_vec<T>(k.off_x());
    const V *const xg = k.xg, *const rg = k.rg, *const pg = k.pg;
    const int* const rowoff = k.rowoff();
    const int nslot = k.nslot, nx = k.nx, pitch = k.pitch;
    const unsigned mg = a.mg_pitch;
#pragma unroll 1
    for (int i = tid(); i < nslot; i += T0) {
      const int row = quot(i, mg), x = i - row * pitch;
      V pv = vzero<T>(), rv = vzero<T>(), xv = vzero<T>();
      if (x < nx) {
        const int g = rowoff[row] + x;
        if (keep) pv = ldg2(pg + g);
        if (r_res) rv = ldg2(rg + g);
        if (x_res) xv = ldg2(xg + g);
      }
      P[i] = pv;
      W[i] = vzero<T>();
      if (r_res) rs[i] = rv;
      if (x_res) xs[i] = xv;
    }
  }
  __syncthreads();
  for (;;) {
    if (a.r_res) {
      if (a.G > 1)
        phase_direction<T, true, true>();
      else
        phase_direction<T, true, false>();
    } else {
      if (a.G > 1)
        phase_direction<T, false, true>();
      else
        phase_direction<T, false, false>();
    }
    __syncthreads();
    if (k.ng4) phase_proj_sums<T>();
    cl.barrier_arrive();
#define RES_X(L) part_x<T, L, R>()
    RES_BY_LEN(a.lx, RES_X)
    cl.barrier_wait();
    if (k.ng4) phase_proj_coef<T>();
    __syncthreads();
#define RES_Z(L) part_z<T, L, R>()
    RES_BY_LEN(a.lz, RES_Z)
    __syncthreads();
    if (k.ng4) phase_proj_term<T>();
    {
      cpx<dacc_t<T>> pw;
#define RES_Y(L) pw = part_y<T, L, R>()
      RES_BY_LEN(a.ly, RES_Y)
      dacc_t<T> sum2[2] = {pw.re, pw.im};
      double tot2[2];
      block_total<dacc_t<T>, 2>(sum2, k.red, tot2);
      if (tid() < 32) post_totals<2>(cl, tot2, k.slots2, a.G, k.rank);
    }
    cl.sync();
    // alpha = rho / (p^T A p)
    if (tid() < 32) {
      double tot2[2];
      read_totals<2>(k.slots2, a.G, tot2);
      const double q = cdiv_lanes(k.rho_r, k.rho_i, tot2[0], tot2[1], tid());
      if (tid() == 1) k.al_i = (T)q;
      if (tid() == 0) {
        k.al_r = (T)q;
        if (k.iters >= a.maxit)
          k.ctl = kMaxit;
        else if ((zero_bits(tot2[0]) && zero_bits(tot2[1])) || !finite_bits(tot2[0]) ||
                 !finite_bits(tot2[1]))
          k.ctl = kBreakdown;
      }
    }
    __syncthreads();
    if (k.ctl != kActive) break;
    {
      const Sum3<T> rr = a.x_res ? phase_update<T, true, true>()
                                 : (a.r_res ? phase_update<T, true, false>()
                                            : phase_update<T, false, false>());
      dacc_t<T> sum3[4] = {rr.v[0], rr.v[1], rr.v[2], 0};
      double tot3[4];
      block_total<dacc_t<T>, 4>(sum3, k.red, tot3);
      if (tid() < 32) post_totals<4>(cl, tot3, k.slots3, a.G, k.rank);
    }
    cl.sync();
    if (tid() < 32) {
      double tot3[4];
      read_totals<4>(k.slots3, a.G, tot3);
      const double q = cdiv_lanes(tot3[1], tot3[2], k.rho_r, k.rho_i, tid());
      __syncwarp();  // every lane has read rho
      if (tid() == 1) k.be_i = (T)q;
      if (tid() == 0) {
        k.be_r = (T)q;
        k.iters += 1;
        k.rn2 = tot3[0];
        if (!finite_bits(tot3[0])) {
          k.ctl = kBreakdown;
        } else if (le_bits(tot3[0], k.target2)) {
          k.ctl = kConverged;  // rho stays that of the residual of the last direction
        } else {
          k.rho_r = tot3[1];
          k.rho_i = tot3[2];
        }
      }
    }
    __syncthreads();
    if (k.ctl != kActive) break;
  }
  // results: x, and the last direction where a continued recurrence looks for it: in p after
  // an even number of iterations of the loop (there already where it is exchanged), else in
  // p_odd
  {
    const int ci = blockIdx.x / a.G;
    const long long s = (long long)(ci % a.nb) * a.ns + (a.ns - 1 - ci / a.nb);
    V* pd = (k.iters - a.sysi[s * kSysI + kIterBase]) & 1 ? a.p_odd : (a.G > 1 ? nullptr : a.p);
    if (pd) pd += s * a.nd;
    const bool x_res = a.x_res;
    const V *const P = smem_vec<T>(0), *const xs = smem_vec<T>(k.off_x());
    V* const xg = k.xg;
    const int* const rowoff = k.rowoff();
    const int np = k.by * k.bz * k.nx, nx = k.nx, pad = k.pitch - nx;
    if (x_res || pd)
#pragma unroll 1
      for (int i = tid(); i < np; i += T0) {
        int slot, g;
        locate(i, a.mg_nx, nx, pad, rowoff, slot, g);
        if (x_res) stg2(xg + g, xs[slot]);
        if (pd) stg2(pd + g, P[slot]);
      }
  }
  if (k.rank == 0 && tid() == 0) {
    const int ci = blockIdx.x / a.G;
    const long long s = (long long)(ci % a.nb) * a.ns + (a.ns - 1 - ci / a.nb);
    double* sd = a.sysd + s * kSysD;
    int* si = a.sysi + s * kSysI;
    sd[kRho] = k.rho_r;
    sd[kRho + 1] = k.rho_i;
    sd[kRnorm] = sqrt(k.rn2);
    si[kIters] = k.iters;
    si[kStatus] = k.ctl;
  }
}

// ---- shapes ----------------------------------------------------------------------------
constexpr int kLens[] = {1, 2, 3, 4, 5, 6, 7};

// segment length of one axis: `lines` lines of `b` points on `warps` warps, N = FP work of an
// output next to the loads of an input
int seg_len(int bmin, int b, int lines, int warps, int R, bool fp64, double* cost) {
  int best = 2;
  *cost = 1e300;
  for (int L : kLens) {
    // a segment lies inside the smallest brick; lengths built: 1 - 5 (FP64), 2, 4 - 7
    if (L > bmin || (fp64 ? L > 5 : L == 1 || L == 3)) continue;
    const long long segs = (b + L - 1) / L;
    const long long w = fp64 ? ((long long)lines * segs + 31) / 32 : (long long)((lines + 31) / 32) * segs;
    const double rounds = (double)((w + warps - 1) / warps);
    // FP64 arithmetic keeps its pipe busy whatever the number of warps: count the warps'
    // instructions; FP32 counts the rounds of the block
    const double c = fp64 ? std::ceil(w / 4.0) * (24.0 * L + 0.5 * (L + 2 * R)) + rounds * 2.0
                          : rounds * (24.0 * L / 2 + 2.0 * (L + 2 * R) + 20.0);
    if (c < *cost) {
      *cost = c;
      best = L;
    }
  }
  return best;
}

template <typename T, int R>
cudaError_t shape_r(int nx, int ny, int nz, int ngroup, int G, ResidentShape* out) {
  *out = ResidentShape();
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int optin = 0;
  e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, k_cocg_resident<T, R>);
  if (e != cudaSuccess) return e;
  const size_t room = (size_t)optin - fa.sharedSizeBytes;
  if (nx < R || ny < R || nz < R || ngroup > 4096) return cudaSuccess;
  ResidentShape best;
  double best_halo = 1e300;
  for (int gz = 1; gz <= G; gz *= 2) {
    const int gy = G / gz;
    if (2 * gy > ny || 2 * gz > nz) continue;  // bricks of two rows at least
    ResidentShape s;
    s.G = G;
    s.gy = gy;
    s.gz = gz;
    s.bym = (ny + gy - 1) / gy;
    s.bzm = (nz + gz - 1) / gz;
    s.pitch = nx | 1;
    const long long cap = (long long)s.bym * s.bzm * s.pitch;
    if (cap >= 65536) continue;
    const size_t vec = sizeof(cpx<T>) * (size_t)cap;
    const size_t fix = sizeof(Brick<T>) + sizeof(cpx<T>) * 2 * (size_t)ngroup * kProjChunk + sizeof(int) * (size_t)(s.bym * s.bzm);
    if (2 * vec + fix > room) continue;
    s.r_res = 3 * vec + fix <= room;
    s.x_res = 4 * vec + fix <= room;
    s.smem = fix + vec * (2 + s.r_res + s.x_res);
    // halo points per brick: those of the axes that are cut
    const double halo = (gy > 1 ? 2.0 * R * s.bzm : 0.0) + (gz > 1 ? 2.0 * R * s.bym : 0.0);
    if (halo < best_halo) {
      best_halo = halo;
      best = s;
    }
  }
  if (!best.G) return cudaSuccess;
  double best_cost = 1e300;
  for (int th = 64; th <= max_threads<T>(); th += 32) {
    double c0, c1, c2;
    const bool f64 = sizeof(T) == 8;
    const int w = th / 32;
    const int lx = seg_len(nx, nx, best.bym * best.bzm, w, R, f64, &c0);
    const int lz = seg_len(nz / best.gz, best.bzm, nx * best.bym, w, R, f64, &c1);
    const int ly = seg_len(ny / best.gy, best.bym, nx * best.bzm, w, R, f64, &c2);
    const double pts = (double)nx * best.bym * best.bzm;
    const double c = c0 + c1 + c2 + (f64 ? 40.0 : 30.0) * std::ceil(pts / th) + 0.5 * w;
    if (c < best_cost) {
      best_cost = c;
      best.threads = th;
      best.lx = lx;
      best.ly = ly;
      best.lz = lz;
    }
  }
  e = cudaFuncSetAttribute(k_cocg_resident<T, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)room);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_cocg_resident<T, R>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)G);
  cfg.blockDim = dim3((unsigned)best.threads);
  cfg.dynamicSmemBytes = best.smem;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)G;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int nc = 0;
  if (cudaOccupancyMaxActiveClusters(&nc, k_cocg_resident<T, R>, &cfg) != cudaSuccess) {
    cudaGetLastError();  // clusters of this size cannot be placed
    nc = 0;
  }
  if (nc < 1) return cudaSuccess;
  best.clusters = nc;
  *out = best;
  return cudaSuccess;
}

// exact floor(a / d) for a < 2^16: ceil(2^32 / d), d < 2^16
unsigned magic_of(int d) { return (unsigned)((0x100000000ULL + (unsigned)d - 1) / (unsigned)d); }

template <typename T, int R>
cudaError_t launch_r(const CocgView<T>& cv, const ResidentShape& sh, const ResidentProj<T>& pj,
                     cpx<T>* p_odd, int maxit, int cont, cudaStream_t s) {
  using V = typename Val<T>::V;
  Args<T> a;
  a.st = cv.st;
  a.vloc = cv.vloc;
  a.nd = cv.nd;
  a.ns = cv.ns;
  a.nb = cv.nsys / cv.ns;
  a.eps = cv.eps;
  a.omega = cv.omega;
  a.x = reinterpret_cast<V*>(cv.x);
  a.r = reinterpret_cast<V*>(cv.r);
  a.p = reinterpret_cast<V*>(cv.p);
  a.p_odd = reinterpret_cast<V*>(p_odd);
  a.sysd = cv.sysd;
  a.sysi = cv.sysi;
  a.maxit = maxit;
  a.cont = cont;
  a.G = sh.G;
  a.gy = sh.gy;
  a.gz = sh.gz;
  a.cap = sh.bym * sh.bzm * sh.pitch;
  a.pitch = sh.pitch;
  a.lx = sh.lx;
  a.ly = sh.ly;
  a.lz = sh.lz;
  a.r_res = sh.r_res;
  a.x_res = sh.x_res;
  a.mg_pitch = magic_of(sh.pitch);
  a.mg_nx = magic_of(cv.st.nx);
  a.pj = pj;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(cv.nsys * sh.G));
  cfg.blockDim = dim3((unsigned)sh.threads);
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)sh.G;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_cocg_resident<T, R>, a);
  note_launch();
  return e;
}

template <typename T>
__global__ void __launch_bounds__(256) k_resident_gather(long long n, const int* __restrict__ e,
                                                         const T* __restrict__ chi,
                                                         T* __restrict__ out) {
  const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  T v[kProjChunk] = {0, 0, 0, 0};
  if (e[i] >= 0) load_chi4(chi + (long long)e[i] * kProjChunk, v);
#pragma unroll
  for (int l = 0; l < kProjChunk; ++l) out[i * kProjChunk + l] = v[l];
}

}  // namespace

template <typename T>
cudaError_t resident_gather(long long n, const int* e, const T* chi, T* out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_resident_gather<T><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, e, chi, out);
  note_launch();
  return cudaGetLastError();
}

bool resident_supported(int R) { return R == 4 || R == 6; }

template <typename T>
cudaError_t resident_shape(int nx, int ny, int nz, int R, int ngroup, int G, ResidentShape* out) {
  return R == 4 ? shape_r<T, 4>(nx, ny, nz, ngroup, G, out)
                : shape_r<T, 6>(nx, ny, nz, ngroup, G, out);
}

template <typename T>
cudaError_t resident_cocg(const CocgView<T>& cv, const ResidentShape& sh,
                          const ResidentProj<T>& pj, cpx<T>* p_odd, int maxit, int cont,
                          cudaStream_t s) {
  return cv.st.R == 4 ? launch_r<T, 4>(cv, sh, pj, p_odd, maxit, cont, s)
                      : launch_r<T, 6>(cv, sh, pj, p_odd, maxit, cont, s);
}

template cudaError_t resident_gather<float>(long long, const int*, const float*, float*, cudaStream_t);
template cudaError_t resident_gather<double>(long long, const int*, const double*, double*,
                                             cudaStream_t);
template cudaError_t resident_shape<float>(int, int, int, int, int, int, ResidentShape*);
template cudaError_t resident_shape<double>(int, int, int, int, int, int, ResidentShape*);
template cudaError_t resident_cocg<float>(const CocgView<float>&, const ResidentShape&,
                                          const ResidentProj<float>&, cpx<float>*, int, int,
                                          cudaStream_t);
template cudaError_t resident_cocg<double>(const CocgView<double>&, const ResidentShape&,
                                           const ResidentProj<double>&, cpx<double>*, int, int,
                                           cudaStream_t);

}  // namespace rpa
