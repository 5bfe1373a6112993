// Smooth particle-mesh Ewald (Essmann et al. 1995; arXiv 2503.07526
// Sec. 5.3 and Appendix B) for the ionic-melt path.  Per step:
//   1. spread: every atom adds q M_n(u_x - k_x) M_n(u_y - k_y) M_n(u_z - k_z)
//      to the n^3 mesh points around it (fixed-point integer atomics, so
//      the sums do not depend on the order of the atoms: 64-bit words at a
//      scale of 2^40 in the mixed form, 128-bit words at 2^80 in FP64);
//   2. forward real-to-complex FFT of the mesh (cuFFT);
//   3. multiply by B(m) C(m) (phi mesh) and by B(m) C(m) h(m) (psi mesh),
//      C(m) = exp(-pi^2 m^2 / alpha^2) / (pi V m^2),
//      h(m) = 2 (1 + pi^2 m^2 / alpha^2) / m^2;
//   4. two inverse FFTs;
//   5. gather: each atom's spline weights, their first and second
//      derivatives read phi (energy, force) and psi (virial).
// Per atom j, with the sums over its n^3 mesh points:
//   E_j = 1/2 ke q_j sum W_j phi,  F_j = -ke q_j (K/L) sum grad_u W_j phi,
//   W_j,ab = delta_ab E_j + ke q_j K^2 / (8 pi^2 L^2) sum d_a d_b W_j psi,
// the last being Appendix B's form of the per-particle reciprocal virial
// (the factor m_a m_b of the k-space virial carried by two derivatives of
// the spline weights).  The self term -ke alpha q_j^2 / sqrt(pi) goes to E_j.
#include <cmath>
#include <complex>
#include <type_traits>
#include <vector>

#include "spme.cuh"

namespace otf {
namespace {

constexpr double kFix = 1099511627776.0;  // 2^40: fixed-point scale of the mixed form's charge mesh
// FP64 form: each mesh point is a 128-bit two's-complement integer (a low
// and a high 64-bit word) counting units of 2^-80 of a charge, so the
// quantisation (2^-81 per added value) is far below FP64 rounding and the
// range (2^47 charges) cannot be reached.
constexpr double kPi = 3.14159265358979323846;

template <typename T>
struct Rec;
template <>
struct Rec<float> {
  using type = float4;
};
template <>
struct Rec<double> {
  using type = dvec4;
};
template <typename T>
struct Cplx;
template <>
struct Cplx<float> {
  using type = cufftComplex;
};
template <>
struct Cplx<double> {
  using type = cufftDoubleComplex;
};

__device__ __forceinline__ long long to_fix(float v) { return __float2ll_rn(v * (float)kFix); }

// Adds v to mesh point idx of a mesh of K3 points: one 64-bit word per point
// (mixed form) or 128 bits per point, low words [0, K3) and high words
// [K3, 2 K3) (FP64).  The 128-bit addend is round(v 2^80) split as
// hi 2^64 + lo with lo in [0, 2^64); the carry out of the low word is the
// unsigned wrap of that add, so every order of the adds gives the same
// integer.
__device__ __forceinline__ void mesh_add(unsigned long long *Q, int64_t idx, int64_t K3, float v) {
  const long long f = to_fix(v);
  if (f != 0) atomicAdd(Q + idx, (unsigned long long)f);
}
__device__ __forceinline__ void mesh_add(unsigned long long *Q, int64_t idx, int64_t K3, double v) {
  if (v == 0.0) return;
  const double t = v * 65536.0;  // v 2^16: the high word's units (exact)
  const double fh = floor(t);
  // t - fh is exact and at most 1 - 2^-53, so its product with 2^64 is at
  // most 2^64 - 2^11 and rounds to an integer below 2^64
  const unsigned long long l = __double2ull_rn((t - fh) * 18446744073709551616.0);
  long long hi = (long long)fh;
  if (l != 0ull) {
    const unsigned long long old = atomicAdd(Q + idx, l);
    if (old + l < old) hi += 1;  // carry
  }
  if (hi != 0) atomicAdd(Q + K3 + idx, (unsigned long long)hi);
}

// The mesh and how a cell row's atoms are cut into CTAs (see plan_chunks).
struct MeshPlan {
  int K;
  double kl;          // K / L
  float kl_h, kl_l;   // the same as a double-float
  int chunk, slots;   // atoms per CTA at a time; CTAs per cell row
  int cap;            // mesh points that the gather's shared tile holds
  int cap_spread;     // words of the spread's shared tile (rows and planes padded, see SpreadPitch)
};

// Mesh coordinates of atom i: base mesh point and fraction per axis, from
// the cell index and the offset from the cell centre.  The base is not wrapped
// into [0, K) (an atom that has left its cell since the last sort may sit just
// outside the box), so that the mesh points of one cell row stay contiguous;
// mesh indices are wrapped where the mesh is read or written.  It is kept
// within a box of the box, so that a non-finite coordinate (which md_step
// reports) cannot index anything.
//
// Mixed form: in double-float arithmetic (~48 bits) instead of FP64: the cell
// centre in mesh units is (2 c + 1) K / (2 nc), split exactly into integer and
// fraction.  The fraction is rounded to FP32 once, as from FP64, except where the
// coordinate is a small negative number, whose high word is rounded when its
// floor comes off (errors 1.33e-8 rms and 4.5e-8 at most, from FP64 1.30e-8 and
// 3.0e-8).  The ~36 FP64 operations per atom took 33 us of each kernel at 512,000 ions.
template <typename T>
__device__ __forceinline__ void mesh_coords(const SpmeAtoms &a, int64_t i, const MeshPlan &g,
                                            const typename Rec<T>::type &r, int (&base)[3], T (&frac)[3]) {
  const int c = a.cpk[i];
  const int cc[3] = {c & 1023, (c >> 10) & 1023, c >> 20};
  if constexpr (std::is_same<T, double>::value) {
    const double off[3] = {r.x, r.y, r.z};
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      const double u = ((cc[ax] + 0.5) * a.edge + off[ax]) * g.kl;
      const double b = floor(u);
      base[ax] = (int)b;
      frac[ax] = u - b;
    }
  } else {
    const float4 l4 = a.rlo[i];
    const float oh[3] = {r.x, r.y, r.z}, ol[3] = {l4.x, l4.y, l4.z};
    const int den = 2 * a.nc;
    const float fd = (float)den;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      const int num = (2 * cc[ax] + 1) * g.K, q = num / den;
      const float rem = (float)(num - q * den);  // below 2^11: exact
      const float h = rem / fd;
      const dfloat u = df_add(dfloat{h, fmaf(-h, fd, rem) / fd}, df_mul(dfloat{oh[ax], ol[ax]}, dfloat{g.kl_h, g.kl_l}));
      float fl = floorf(u.h), f = (u.h - fl) + u.l;
      if (f < 0.f) {
        f += 1.f;
        fl -= 1.f;
      }
      base[ax] = q + (int)fl;
      frac[ax] = f;
    }
  }
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) base[ax] = max(-g.K, min(2 * g.K, base[ax]));
}

// Cardinal B-spline weights m[t] = M_N(w + t), t = 0..N-1, by the
// recursion M_p(x) = (x M_{p-1}(x) + (p - x) M_{p-1}(x - 1)) / (p - 1)
// from M_2; with derivatives, d1[t] = M_{N-1}(w+t) - M_{N-1}(w+t-1) and
// d2[t] = M_{N-2}(w+t) - 2 M_{N-2}(w+t-1) + M_{N-2}(w+t-2).
template <typename T, int N, bool DERIV>
__device__ __forceinline__ void spline(T w, T (&m)[N], T (&d1)[N], T (&d2)[N]) {
  T b[N];
  b[0] = w;
  b[1] = T(1) - w;
#pragma unroll
  for (int k = 2; k < N; ++k) b[k] = T(0);
  T o2[N], o1[N];
  if (N - 2 == 2) {
#pragma unroll
    for (int k = 0; k < N; ++k) o2[k] = b[k];
  }
#pragma unroll
  for (int p = 3; p <= N; ++p) {
    const T inv = T(1) / T(p - 1);
#pragma unroll
    for (int k = p - 1; k >= 0; --k) {
      const T prev = k > 0 ? b[k - 1] : T(0);
      b[k] = ((w + T(k)) * b[k] + (T(p) - w - T(k)) * prev) * inv;
    }
    if (p == N - 2) {
#pragma unroll
      for (int k = 0; k < N; ++k) o2[k] = b[k];
    }
    if (p == N - 1) {
#pragma unroll
      for (int k = 0; k < N; ++k) o1[k] = b[k];
    }
  }
#pragma unroll
  for (int k = 0; k < N; ++k) m[k] = b[k];
  if (DERIV) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      d1[k] = o1[k] - (k > 0 ? o1[k - 1] : T(0));
      d2[k] = o2[k] - T(2) * (k > 0 ? o2[k - 1] : T(0)) + (k > 1 ? o2[k - 2] : T(0));
    }
  }
}

__device__ __forceinline__ int wrap(int v, int K) { return ((v % K) + K) % K; }
// wrap() without the divisions for the usual case v in [-K, 2K) (mesh points
// of atoms at most a cell outside the box), with wrap() as the fallback.
__device__ __forceinline__ int wrap_near(int v, int K) {
  int w = v < 0 ? v + K : v;
  w = w >= K ? w - K : w;
  return (unsigned)w < (unsigned)K ? w : wrap(v, K);
}

constexpr int kRowThreads = 128;       // threads of a spread or gather CTA, and the largest chunk
constexpr int kRowWarps = kRowThreads / 32;
constexpr int kMaxOrder = 8;
constexpr int kSpreadPitch = 3 * kMaxOrder + 1;     // an atom's weights in the spread (odd: no bank conflicts)
constexpr int kGatherPitch = 9 * kMaxOrder + 1;     // an atom's weights and derivatives in the gather
constexpr int kGatherBatch = 8;                     // atoms whose weights a warp of the gather holds
constexpr size_t kMaxTileBytes = 160 * 1024;        // shared memory that a mesh tile may take
constexpr int kMaxTileSide = 128;                   // largest tile side in mesh points

template <typename T>
struct Two;
template <>
struct Two<float> {
  using type = float2;
};
template <>
struct Two<double> {
  using type = double2;
};

// The charge of one atom straight into the wrapped global mesh, at points
// (base - t0, base - t1, base - t2) for t = 0..N-1.
template <typename T, int N>
__device__ void spread_atom(const int (&base)[3], const T (&frac)[3], T q, unsigned long long *dst, int K) {
  const int64_t K3 = (int64_t)K * K * K;
  T wx[N], wy[N], wz[N], d1[N], d2[N];
  spline<T, N, false>(frac[0], wx, d1, d2);
  spline<T, N, false>(frac[1], wy, d1, d2);
  spline<T, N, false>(frac[2], wz, d1, d2);
  int iz[N];
#pragma unroll
  for (int t = 0; t < N; ++t) iz[t] = wrap_near(base[2] - t, K);
  for (int t0 = 0; t0 < N; ++t0) {
    const int ix = wrap_near(base[0] - t0, K);
    const T qx = q * wx[t0];
    for (int t1 = 0; t1 < N; ++t1) {
      const int iy = wrap_near(base[1] - t1, K);
      const T qxy = qx * wy[t1];
      const int64_t row = ((int64_t)ix * K + iy) * K;
#pragma unroll
      for (int t2 = 0; t2 < N; ++t2) mesh_add(dst, row + iz[t2], K3, qxy * wz[t2]);
    }
  }
}

// The tile of one chunk of a cell row: the box of mesh points its atoms
// touch, from the block-wide extremes of their base points.
struct Tile {
  int ox, oy, oz, ex, ey, ez;
  __device__ int64_t vol() const { return (int64_t)ex * ey * ez; }
  __device__ bool fits(int cap) const { return vol() <= cap && max(ex, max(ey, ez)) <= kMaxTileSide; }
};
template <int N>
__device__ __forceinline__ Tile chunk_tile(const int (&base)[3], bool live, int *bmin, int *bmax) {
  if (threadIdx.x < 3) {
    bmin[threadIdx.x] = 0x7fffffff;
    bmax[threadIdx.x] = -0x7fffffff;
  }
  __syncthreads();
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    const int lo = __reduce_min_sync(0xffffffffu, live ? base[ax] : 0x7fffffff);
    const int hi = __reduce_max_sync(0xffffffffu, live ? base[ax] : -0x7fffffff);
    if ((threadIdx.x & 31) == 0) {
      atomicMin(&bmin[ax], lo);
      atomicMax(&bmax[ax], hi);
    }
  }
  __syncthreads();
  Tile t;
  t.ox = bmin[0] - (N - 1);
  t.oy = bmin[1] - (N - 1);
  t.oz = bmin[2] - (N - 1);
  t.ex = bmax[0] - bmin[0] + N;
  t.ey = bmax[1] - bmin[1] + N;
  t.ez = bmax[2] - bmin[2] + N;
  return t;
}

// Mesh offset of every plane, row and point of a tile (wrapped into the box),
// so that a tile point's mesh index is three table reads and two additions.
struct TileTable {
  int x[kMaxTileSide], y[kMaxTileSide], z[kMaxTileSide];
};
__device__ __forceinline__ void fill_table(TileTable &tt, const Tile &t, int K) {
  for (int k = threadIdx.x; k < kMaxTileSide; k += kRowThreads) {
    if (k < t.ex) tt.x[k] = wrap_near(t.ox + k, K) * K * K;
    if (k < t.ey) tt.y[k] = wrap_near(t.oy + k, K) * K;
    if (k < t.ez) tt.z[k] = wrap_near(t.oz + k, K);
  }
}

// Steps an element index k = (lx * ey + ly) * ez + lz of a tile by
// kRowThreads without dividing: consecutive threads take consecutive z.
struct TileWalk {
  int lx, ly, lz, dx, dy, dz;
  __device__ explicit TileWalk(const Tile &t) {
    dz = kRowThreads % t.ez;
    const int qz = kRowThreads / t.ez;
    dy = qz % t.ey;
    dx = qz / t.ey;
    lz = threadIdx.x % t.ez;
    ly = (threadIdx.x / t.ez) % t.ey;
    lx = threadIdx.x / (t.ez * t.ey);
  }
  __device__ __forceinline__ int mesh_index(const TileTable &tt) const { return tt.x[lx] + tt.y[ly] + tt.z[lz]; }
  __device__ __forceinline__ void step(const Tile &t) {
    lz += dz;
    ly += dy;
    lx += dx;
    if (lz >= t.ez) {
      lz -= t.ez;
      ++ly;
    }
    if (ly >= t.ey) {
      ly -= t.ey;
      ++lx;
    }
  }
};

// Copies one value to shared memory without holding a register for it.
__device__ __forceinline__ void copy_async(float *dst, const float *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_async(double *dst, const double *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Row pitch and plane size of the spread's tile.  A warp adds 8 z points of two
// neighbouring rows in two planes four apart: with the pitch a multiple of 8
// words (not of 32) and the plane padded so that four planes lie a quarter or
// half of the 32 banks further, its four runs of eight words fill the banks
// once, wherever they start.
struct SpreadPitch {
  int row, plane;
  __host__ __device__ SpreadPitch(int ey, int ez) {
    row = (ez + 7) & ~7;
    if (row % 32 == 0) row += 8;
    plane = ey * row;  // a multiple of 8
    plane += row % 32 == 16 ? 2 : 4;
  }
};

// Charge spreading: the atoms of a cell row in chunks of g.chunk, one CTA per
// chunk.  The chunk's spline weights (q M_n in x) go to shared memory, an
// (atom, axis) pair per thread; then every warp walks all atoms and adds the
// mesh planes it owns (those with x = its number mod 4, two of an atom's eight)
// into the chunk's shared tile, lanes over eight z, two y and both planes.  A
// tile point has one owner warp, which adds the atoms in order, so no atomic is
// needed inside the tile and the sums do not depend on scheduling.  The tile's
// non-zero points go to the global mesh in fixed point (integer atomics:
// order-independent), consecutive lanes on consecutive z.  A chunk whose tile
// does not fit spreads atom by atom straight into the global mesh.
//
// Against a thread per mesh column that tests every atom of the chunk (a third
// of the tests hit, and its flush walked z in each thread): 440 -> 156 us at
// 512,000 ions (mixed form, 128^3 mesh, order 8), 410 -> 35 us at 1,728 (FP64,
// 32^3).  What is left is the load/store unit (77 %; issue 72 %, mixed form): 256
// warp instructions per atom, half of them the tile additions, a fifth the flush.
template <typename T, int N>
__global__ void __launch_bounds__(kRowThreads) k_spme_spread(SpmeAtoms a, MeshPlan g, unsigned long long *Qi) {
  using R = typename Rec<T>::type;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int2 sb[kRowThreads];  // an atom's last tile point and its x plane there
  __shared__ T sf[kRowThreads][3];
  __shared__ T sq[kRowThreads];
  __shared__ int bmin[3], bmax[3];
  __shared__ TileTable tt;
  T *tile = reinterpret_cast<T *>(smraw);
  T *sw = tile + g.cap_spread;  // [chunk][kSpreadPitch]
  const R *rel = static_cast<const R *>(a.rel);
  const int K = g.K, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t K3 = (int64_t)K * K * K;
  const int z = lane & 7, y = (lane >> 3) & 1, u = lane >> 4;
  const int64_t nwork = (int64_t)a.nc * a.nc * g.slots;
  for (int64_t wk = blockIdx.x; wk < nwork; wk += gridDim.x) {
    const int row = (int)(wk / g.slots), slot = (int)(wk % g.slots);
    const int a0 = a.cellstart[(int64_t)row * a.nc], a1 = a.cellstart[(int64_t)row * a.nc + a.nc];
    for (int c0 = a0 + slot * g.chunk; c0 < a1; c0 += g.slots * g.chunk) {
      const int na = min(g.chunk, a1 - c0);
      const int64_t i = c0 + threadIdx.x;
      const bool live = (int)threadIdx.x < na;
      int base[3] = {0, 0, 0};
      T frac[3] = {T(0), T(0), T(0)};
      T q = T(0);
      if (live) {
        const R r = rel[i];
        mesh_coords<T>(a, i, g, r, base, frac);
        q = (T)r.w;
      }
      const Tile tl = chunk_tile<N>(base, live, bmin, bmax);
      const SpreadPitch sp(tl.ey, tl.ez);
      if (tl.fits(g.cap_spread) && (int64_t)tl.ex * sp.plane <= g.cap_spread) {
        if (live) {
          const int bx = base[0] - tl.ox;
          sb[threadIdx.x] = make_int2(bx * sp.plane + (base[1] - tl.oy) * sp.row + (base[2] - tl.oz), bx);
#pragma unroll
          for (int ax = 0; ax < 3; ++ax) sf[threadIdx.x][ax] = frac[ax];
          sq[threadIdx.x] = q;
        }
        fill_table(tt, tl, K);
        for (int k = threadIdx.x; k < tl.ex * sp.plane; k += kRowThreads) tile[k] = T(0);
        __syncthreads();
        for (int k = threadIdx.x; k < 3 * na; k += kRowThreads) {
          const int ax = k / na, j = k - ax * na;
          T w[N], d1[N], d2[N];
          spline<T, N, false>(sf[j][ax], w, d1, d2);
          const T f = ax == 0 ? sq[j] : T(1);
          T *o = sw + j * kSpreadPitch + ax * kMaxOrder;
#pragma unroll
          for (int t = 0; t < N; ++t) o[t] = f * w[t];
        }
        __syncthreads();
        constexpr int V = N / 2;  // rows per lane
        // the lane's point of an atom, once its last tile point is added
        T *mine = tile - (z < N ? z : 0) - y * sp.row - u * 4 * sp.plane;
        // the next atom's record and weights are read ahead of this one's
        // stores, which the compiler must assume to overlap them
        int2 b;
        T wz, qx, wy[V];
        auto read = [&](int j) {
          const T *wl = sw + j * kSpreadPitch;
          b = sb[j];
          b.y = (b.y - warp) & 3;  // the first of this warp's planes
          b.x -= b.y * sp.plane;
          wz = wl[2 * kMaxOrder + (z < N ? z : 0)];
          qx = wl[min(b.y + 4 * u, kMaxOrder - 1)];
#pragma unroll
          for (int v = 0; v < V; ++v) wy[v] = wl[kMaxOrder + y + 2 * v];
        };
        read(0);
        for (int j = 0; j < na; ++j) {
          T *p = mine + b.x;
          const bool on = z < N && b.y + 4 * u < N;
          const T w = wz;
          T c[V];
#pragma unroll
          for (int v = 0; v < V; ++v) c[v] = qx * wy[v];
          read(min(j + 1, na - 1));
          if (on) {
            T t[V];
#pragma unroll
            for (int v = 0; v < V; ++v) t[v] = p[-2 * v * sp.row];
#pragma unroll
            for (int v = 0; v < V; ++v) p[-2 * v * sp.row] = fma(c[v], w, t[v]);
          }
          __syncwarp();  // the next atom's points may be other lanes'
        }
        __syncthreads();
        TileWalk tw(tl);
        const int vol = (int)tl.vol();
        for (int k = threadIdx.x; k < vol; k += kRowThreads, tw.step(tl))
          mesh_add(Qi, tw.mesh_index(tt), K3, tile[tw.lx * sp.plane + tw.ly * sp.row + tw.lz]);
      } else if (live) {
        spread_atom<T, N>(base, frac, q, Qi, K);
      }
      __syncthreads();  // the tile, the atom tables and the extremes are reused by the next chunk
    }
  }
}

template <typename T>
__global__ void k_spme_unfix(const unsigned long long *Qi, T *Qr, int64_t total) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total; k += (int64_t)gridDim.x * blockDim.x) {
    if constexpr (std::is_same<T, double>::value)  // hi 2^-16 + lo 2^-80
      Qr[k] = (double)(long long)Qi[total + k] * (1.0 / 65536.0) + (double)Qi[k] * 8.271806125530277e-25;
    else
      Qr[k] = (T)((double)(long long)Qi[k] * (1.0 / kFix));
  }
}

// The factors of both convolutions at mode e of the half spectrum
// [K][K][K/2+1]; zero at the origin.
__device__ __forceinline__ double2 conv_factors(int64_t e, int K, const double *bmod, double invL, double pa2,
                                                double cpre) {
  const int kh = K / 2 + 1;
  const int iz = (int)(e % kh);
  const int iy = (int)((e / kh) % K);
  const int ix = (int)(e / ((int64_t)kh * K));
  const double mx = (ix <= K / 2 ? ix : ix - K) * invL;
  const double my = (iy <= K / 2 ? iy : iy - K) * invL;
  const double mz = iz * invL;
  const double m2 = mx * mx + my * my + mz * mz;
  if (m2 == 0.0) return make_double2(0.0, 0.0);
  const double t = pa2 * m2;
  const double bc = bmod[ix] * bmod[iy] * bmod[iz] * exp(-t) / m2 * cpre;
  return make_double2(bc, bc * 2.0 * (1.0 + t) / m2);
}

// The mixed form's factors, rounded once from FP64 when the plan is made: formed
// in FP32 on every step, each carried the rounding of its exponent (3e-7 and
// more of the factor) into every virial alike.
__global__ void k_spme_factors(float2 *fac, int64_t total, int K, const double *bmod, double invL, double pa2,
                               double cpre) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const double2 f = conv_factors(e, K, bmod, invL, pa2, cpre);
    fac[e] = make_float2((float)f.x, (float)f.y);
  }
}

// The two convolutions on the half spectrum.
template <typename T>
__global__ void k_spme_conv(typename Cplx<T>::type *G1, typename Cplx<T>::type *G2, const float2 *fac,
                            const double *bmod, int K, double invL, double pa2, double cpre) {
  const int64_t total = (int64_t)K * K * (K / 2 + 1);
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    typename Two<T>::type f;
    if constexpr (std::is_same<T, double>::value)
      f = conv_factors(e, K, bmod, invL, pa2, cpre);
    else
      f = fac[e];
    typename Cplx<T>::type a = G1[e], b = a;
    a.x *= f.x;
    a.y *= f.x;
    b.x *= f.y;
    b.y *= f.y;
    G1[e] = a;
    G2[e] = b;
  }
}

// The sums of one atom over its mesh points by a group of eight lanes (lane z
// of the group takes the points z of every (x, y)): energy (phi), force (first
// derivatives, phi) and the six virial sums (second derivatives, psi), summed
// axis by axis -- over x into five sums, over y into nine, then the z weights
// give this lane's share of the ten results.  w: the atom's weights and
// derivatives [axis][0..2][kMaxOrder].
//
// The (phi, psi) pairs are multiplied as pairs: two FP32 operations per
// instruction (f32x2) in the mixed form.  That form also takes the pair `mid` of
// one point of the stencil off every point first: the long waves hardly change
// over a stencil, and every force and virial sum holds a derivative weight, whose
// sum is zero, so only their rounding is lost (the energy, whose weights sum to
// one, gets it back).
template <typename T>
struct Pair;
template <>
struct Pair<float> {
  uint64_t v;
  __device__ __forceinline__ static Pair both(float x) {
    Pair p;
    asm("mov.b64 %0, {%1, %1};" : "=l"(p.v) : "f"(x));
    return p;
  }
  __device__ __forceinline__ static Pair of(float2 x) {
    Pair p;
    asm("mov.b64 %0, {%1, %2};" : "=l"(p.v) : "f"(x.x), "f"(x.y));
    return p;
  }
  __device__ __forceinline__ void fma(Pair a, Pair b) {  // this += a b
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(v) : "l"(a.v), "l"(b.v));
  }
  __device__ __forceinline__ void less(Pair a) {  // this -= a
    const Pair m = both(-1.f);
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(v) : "l"(a.v), "l"(m.v));
  }
  __device__ __forceinline__ float2 get() const {
    float2 x;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x.x), "=f"(x.y) : "l"(v));
    return x;
  }
};
template <>
struct Pair<double> {
  double2 v;
  __device__ __forceinline__ static Pair both(double x) { return Pair{make_double2(x, x)}; }
  __device__ __forceinline__ static Pair of(double2 x) { return Pair{x}; }
  __device__ __forceinline__ void fma(Pair a, Pair b) {
    v.x = ::fma(a.v.x, b.v.x, v.x);
    v.y = ::fma(a.v.y, b.v.y, v.y);
  }
  __device__ __forceinline__ void less(Pair a) {
    v.x -= a.v.x;
    v.y -= a.v.y;
  }
  __device__ __forceinline__ double2 get() const { return v; }
};

template <typename T, int N, typename Fetch>
__device__ __forceinline__ void gather_lane(const T *w, int z, Pair<T> mid, Fetch fetch, T (&out)[16]) {
  using P = Pair<T>;
  P wx[N], dx[N];
  T ex[N];
#pragma unroll
  for (int t = 0; t < N; ++t) {
    wx[t] = P::both(w[t]);
    dx[t] = P::both(w[kMaxOrder + t]);
    ex[t] = w[2 * kMaxOrder + t];
  }
  const P zero = P::both(T(0));
  P ww = zero, dw = zero, wd = zero;  // (phi, psi): sums with weights w w, d w, w d of x and y
  T s_ew = T(0), s_dd = T(0), s_we = T(0);
#pragma unroll 2
  for (int t1 = 0; t1 < N; ++t1) {
    P c0 = zero, c1 = zero;
    T s2 = T(0);
#pragma unroll
    for (int t0 = 0; t0 < N; ++t0) {
      P pv = P::of(fetch(t0, t1));
      if (sizeof(T) == 4) pv.less(mid);
      c0.fma(wx[t0], pv);
      c1.fma(dx[t0], pv);
      s2 += ex[t0] * pv.get().y;
    }
    const T wy = w[3 * kMaxOrder + t1], dy = w[4 * kMaxOrder + t1], ey = w[5 * kMaxOrder + t1];
    const P wy2 = P::both(wy), dy2 = P::both(dy);
    ww.fma(wy2, c0);
    dw.fma(wy2, c1);
    wd.fma(dy2, c0);
    s_ew += wy * s2;
    s_dd += dy * c1.get().y;
    s_we += ey * c0.get().y;
  }
  const T p_ww = ww.get().x, s_ww = ww.get().y, p_dw = dw.get().x, s_dw = dw.get().y, p_wd = wd.get().x,
          s_wd = wd.get().y;
  const bool on = z < N;
  const T wz = on ? w[6 * kMaxOrder + z] : T(0), dz = on ? w[7 * kMaxOrder + z] : T(0),
          ez = on ? w[8 * kMaxOrder + z] : T(0);
  out[0] = p_ww * wz;
  out[1] = p_dw * wz;
  out[2] = p_wd * wz;
  out[3] = p_ww * dz;
  out[4] = s_ew * wz;
  out[5] = s_we * wz;
  out[6] = s_ww * ez;
  out[7] = s_dd * wz;
  out[8] = s_dw * dz;
  out[9] = s_wd * dz;
#pragma unroll
  for (int q = 10; q < 16; ++q) out[q] = T(0);
}

// Gather, one CTA per chunk of a cell row (as the spread): the chunk's tile of
// (phi, psi) is staged in shared memory, then each warp takes eight atoms at a
// time: 24 lanes form the weights of their three axes, and groups of eight
// lanes sum the points of one atom each (gather_lane: 5 operations per point
// where the separate ten sums took 14, and 64-byte rows of the tile where a
// thread per atom read 32 unrelated places per load).  At 512,000 ions in the
// mixed form, order 8: 297 -> 220 us; at 1,728 ions in FP64 319 -> 44 us.  Bound
// by the shared-memory pipe (81 %, a third of its wavefronts conflict replays).
template <typename T, int N>
__global__ void __launch_bounds__(kRowThreads, sizeof(T) == 4 ? 5 : 2)
    k_spme_gather(SpmeAtoms a, MeshPlan g, const T *phi, const T *psi, T ke, T kL, T cw, T self, T *F, T *epot, T *W) {
  using R = typename Rec<T>::type;
  using T2 = typename Two<T>::type;
  extern __shared__ __align__(16) unsigned char smraw[];
  T2 *tile = reinterpret_cast<T2 *>(smraw);
  T *sw = reinterpret_cast<T *>(tile + g.cap);  // [warp][kGatherBatch][kGatherPitch]
  __shared__ TileTable tt;
  __shared__ int sb[kRowThreads][3];
  __shared__ T sf[kRowThreads][3];
  __shared__ T sq[kRowThreads];
  __shared__ int bmin[3], bmax[3];
  const R *rel = static_cast<const R *>(a.rel);
  const int64_t n = a.n;
  const int K = g.K, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = lane >> 3, z = lane & 7;
  T *wb = sw + warp * kGatherBatch * kGatherPitch;
  const int64_t nwork = (int64_t)a.nc * a.nc * g.slots;
  for (int64_t wk = blockIdx.x; wk < nwork; wk += gridDim.x) {
    const int row = (int)(wk / g.slots), slot = (int)(wk % g.slots);
    const int a0 = a.cellstart[(int64_t)row * a.nc], a1 = a.cellstart[(int64_t)row * a.nc + a.nc];
    for (int c0 = a0 + slot * g.chunk; c0 < a1; c0 += g.slots * g.chunk) {
      const int na = min(g.chunk, a1 - c0);
      const bool live = (int)threadIdx.x < na;
      int base[3] = {0, 0, 0};
      T frac[3] = {T(0), T(0), T(0)};
      if (live) {
        const R r = rel[c0 + threadIdx.x];
        mesh_coords<T>(a, c0 + threadIdx.x, g, r, base, frac);
        sq[threadIdx.x] = (T)r.w;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
          sb[threadIdx.x][ax] = base[ax];
          sf[threadIdx.x][ax] = frac[ax];
        }
      }
      const Tile tl = chunk_tile<N>(base, live, bmin, bmax);
      const bool tiled = tl.fits(g.cap);
      if (tiled) {
        fill_table(tt, tl, K);
        __syncthreads();
        const int vol = (int)tl.vol();
        TileWalk tw(tl);
        for (int k = threadIdx.x; k < vol; k += kRowThreads, tw.step(tl)) {
          const int m = tw.mesh_index(tt);
          copy_async(&tile[k].x, phi + m);
          copy_async(&tile[k].y, psi + m);
        }
        copy_async_wait();
      }
      __syncthreads();
      for (int b0 = warp * kGatherBatch; b0 < na; b0 += kRowWarps * kGatherBatch) {
        const int nb = min(kGatherBatch, na - b0);
        if (lane < 3 * nb) {
          const int j = lane / 3, ax = lane - 3 * j;
          T m[N], d1[N], d2[N];
          spline<T, N, true>(sf[b0 + j][ax], m, d1, d2);
          T *o = wb + j * kGatherPitch + ax * 3 * kMaxOrder;
#pragma unroll
          for (int t = 0; t < N; ++t) {
            o[t] = m[t];
            o[kMaxOrder + t] = d1[t];
            o[2 * kMaxOrder + t] = d2[t];
          }
        }
        __syncwarp();
        for (int h = 0; h < kGatherBatch; h += 4) {
          if (h >= nb) break;  // uniform over the warp
          const int j = min(h + grp, nb - 1);  // a group past the end repeats the last atom
          const int bx = sb[b0 + j][0], by = sb[b0 + j][1], bz = sb[b0 + j][2] - min(z, N - 1);
          // the lane's two results and what they hold now, read ahead
          const int64_t i = c0 + b0 + j;
          T *r0 = z == 0 ? epot + i : (z == 1 ? F + n + i : W + (2 * z - 4) * n + i);
          T *r1 = z == 0 ? F + i : (z == 1 ? F + 2 * n + i : W + (2 * z - 3) * n + i);
          const bool put = h + grp < nb && z < 5;
          const T v0 = put ? *r0 : T(0), v1 = put ? *r1 : T(0);
          T acc[16];
          T2 mid = {T(0), T(0)};  // (phi, psi) at a point of the stencil that the group's lanes share
          if (tiled) {
            const int plane = tl.ey * tl.ez;
            const T2 *p = tile + (bx - tl.ox) * plane + (by - tl.oy) * tl.ez + (bz - tl.oz);
            if (sizeof(T) == 4) mid = p[min(z, N - 1) - N / 2 - N / 2 * (plane + tl.ez)];
            gather_lane<T, N>(wb + j * kGatherPitch, z, Pair<T>::of(mid),
                              [&](int t0, int t1) { return p[-(t0 * plane + t1 * tl.ez)]; }, acc);
          } else {
            const int iz = wrap_near(bz, K);
            const auto at = [&](int t0, int t1, int mz) {
              const int64_t m = ((int64_t)wrap_near(bx - t0, K) * K + wrap_near(by - t1, K)) * K + mz;
              T2 v;
              v.x = phi[m];
              v.y = psi[m];
              return v;
            };
            if (sizeof(T) == 4) mid = at(N / 2, N / 2, wrap_near(bz + min(z, N - 1) - N / 2, K));
            gather_lane<T, N>(wb + j * kGatherPitch, z, Pair<T>::of(mid),
                              [&](int t0, int t1) { return at(t0, t1, iz); }, acc);
          }
          // the group's sums: lane z ends with values 2 z and 2 z + 1
#pragma unroll
          for (int hh = 8, o = 4; o >= 1; hh >>= 1, o >>= 1) {
            const bool up = (z & o) != 0;
#pragma unroll
            for (int k = 0; k < hh; ++k) {
              const T give = up ? acc[k] : acc[k + hh], keep = up ? acc[k + hh] : acc[k];
              acc[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
          }
          const T q = sq[b0 + j];
          T pot = __shfl_sync(0xffffffffu, acc[0], lane & 24);
          if (sizeof(T) == 4) pot += mid.x;  // the weights sum to one
          const T er = T(0.5) * ke * q * pot;
          if (put) {
            const T fq = -ke * q * kL, wq = cw * q;
            *r0 = v0 + (z == 0 ? er - self * q * q : (z == 1 ? fq * acc[0] : (z < 4 ? er : T(0)) + wq * acc[0]));
            *r1 = v1 + (z < 2 ? fq * acc[1] : (z == 2 ? er : T(0)) + wq * acc[1]);
          }
        }
        __syncwarp();  // the batch's weights are rewritten next
      }
      __syncthreads();
    }
  }
}

// M_n at the integers 1..n-1 (host, FP64), for the b(m) moduli.
std::vector<double> spline_at_integers(int n) {
  std::vector<double> b(n, 0.0);
  b[0] = 0.0;  // M_2 at w = 0: M_2(0) = 0, M_2(1) = 1
  b[1] = 1.0;
  for (int p = 3; p <= n; ++p)
    for (int k = p - 1; k >= 0; --k) b[k] = ((double)k * b[k] + (double)(p - k) * (k > 0 ? b[k - 1] : 0.0)) / (p - 1);
  return b;  // b[k] = M_n(k)
}

int cufft_ok(cufftResult r, const char *what) {
  if (r == CUFFT_SUCCESS) return MD_OK;
  set_error("%s failed (cuFFT error %d)", what, (int)r);
  return MD_ECUDA;
}

int grid_of(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, 152 * 16); }

constexpr size_t kMaxSpmeSmem =
    kMaxTileBytes + std::max(kRowWarps * kGatherBatch * kGatherPitch, kRowThreads * kSpreadPitch) * sizeof(double);
static_assert(kMaxSpmeSmem + 8 * 1024 <= 227 * 1024, "tile, weights and static tables fit one CTA");

// Chunk and tile sizes: the largest chunk of 128, 64 or 32 atoms that still
// gives four CTAs per SM in FP64, one per two SMs in the mixed form, whose
// expected tile of the gather (the cells the chunk spans plus the spline's
// support) fits.  128 atoms share a tile's halo (at 512,000 ions 10 tile points
// are flushed per mesh point, against 17 with 32 atoms); below 78,000 atoms more
// CTAs count for more in FP64, whose pipe they spread the work over.
void plan_chunks(const SpmeAtoms &a, int order, size_t ts, MeshPlan &g) {
  const double cells = (double)a.nc * a.nc * a.nc, apc = a.n / cells, e = a.edge * g.kl;
  double pts = 0.0, words = 0.0;
  for (g.chunk = kRowThreads; g.chunk >= 32; g.chunk /= 2) {
    const double side = std::ceil(e) + order + 1, len = std::ceil(e * std::min<double>(a.nc, g.chunk / apc + 1.0)) + order + 1;
    const SpreadPitch sp((int)side, (int)side);
    pts = side * side * len;
    words = len * sp.plane;
    if (g.chunk == 32 || (a.n >= (int64_t)(ts == 8 ? 608 : 76) * g.chunk && pts * 2 * ts <= kMaxTileBytes / 2)) break;
  }
  g.cap = (int)std::min(pts, (double)(kMaxTileBytes / (2 * ts)));
  g.cap = (g.cap + 3) & ~3;
  if ((size_t)g.cap * 2 * ts > kMaxTileBytes) g.cap -= 4;
  g.cap_spread = (int)std::min(words, (double)(kMaxTileBytes / ts)) & ~3;
  g.slots = std::max(1, (int)std::ceil(apc * a.nc / g.chunk));
}

}  // namespace

int Spme::create(const SpmeParams &p, bool fp64, cudaStream_t st) {
  p_ = p;
  fp64_ = fp64;
  const int K = p.K;
  const int64_t K3 = (int64_t)K * K * K, KH = (int64_t)K * K * (K / 2 + 1);
  const size_t ts = fp64 ? sizeof(double) : sizeof(float);
  // |b(m)|^2 = 1 / |sum_{k=0}^{n-2} M_n(k+1) exp(2 pi i m k / K)|^2
  const std::vector<double> Mk = spline_at_integers(p.order);
  std::vector<double> bm(K);
  for (int m = 0; m < K; ++m) {
    std::complex<double> s(0.0, 0.0);
    for (int k = 0; k <= p.order - 2; ++k) s += Mk[k + 1] * std::polar(1.0, 2.0 * kPi * m * k / K);
    bm[m] = 1.0 / std::norm(s);
  }
  OTF_CUDA(cudaMalloc(&Qi_, sizeof(unsigned long long) * K3 * (fp64 ? 2 : 1)));  // 128-bit points in FP64
  OTF_CUDA(cudaMalloc(&Qr_, ts * K3));
  // both convolved meshes, and their spectra, end to end: one batched inverse
  OTF_CUDA(cudaMalloc(&phi_, 2 * ts * K3));
  psi_ = static_cast<char *>(phi_) + ts * K3;
  OTF_CUDA(cudaMalloc(&G1_, 4 * ts * KH));
  G2_ = static_cast<char *>(G1_) + 2 * ts * KH;
  OTF_CUDA(cudaMalloc(&bmod_, sizeof(double) * K));
  OTF_CUDA(cudaMemcpy(bmod_, bm.data(), sizeof(double) * K, cudaMemcpyHostToDevice));
  if (!fp64) {
    OTF_CUDA(cudaMalloc(&fac_, sizeof(float2) * KH));
    k_spme_factors<<<grid_of(KH), 256, 0, st>>>(fac_, KH, K, bmod_, 1.0 / p.L, kPi * kPi / (p.alpha * p.alpha),
                                                1.0 / (kPi * p.L * p.L * p.L));
    OTF_LAUNCH_CHECK();
  }
  int rc = cufft_ok(cufftPlan3d(&fwd_, K, K, K, fp64 ? CUFFT_D2Z : CUFFT_R2C), "cufftPlan3d (forward)");
  int dims[3] = {K, K, K};
  if (!rc)
    rc = cufft_ok(cufftPlanMany(&inv_, 3, dims, nullptr, 1, 0, nullptr, 1, 0, fp64 ? CUFFT_Z2D : CUFFT_C2R, 2),
                  "cufftPlanMany (inverse)");
  if (rc) return rc;
  plans_ = true;
  rc = cufft_ok(cufftSetStream(fwd_, st), "cufftSetStream");
  if (!rc) rc = cufft_ok(cufftSetStream(inv_, st), "cufftSetStream");
  return rc;
}

void Spme::destroy() {
  if (plans_) {
    cufftDestroy(fwd_);
    cufftDestroy(inv_);
    plans_ = false;
  }
  for (void *q : {(void *)Qi_, Qr_, phi_, G1_, (void *)bmod_, (void *)fac_})
    if (q) cudaFree(q);
  Qi_ = nullptr;
  Qr_ = phi_ = psi_ = G1_ = G2_ = nullptr;
  bmod_ = nullptr;
  fac_ = nullptr;
}

template <typename T>
int Spme::run_t(const SpmeAtoms &a, T *F, T *epot, T *W, cudaStream_t st) {
  const int K = p_.K;
  const int64_t K3 = (int64_t)K * K * K;
  const double kl = K / p_.L;
  // the FFTs follow the caller's stream (a graph may be capturing it)
  int rs = cufft_ok(cufftSetStream(fwd_, st), "cufftSetStream");
  if (!rs) rs = cufft_ok(cufftSetStream(inv_, st), "cufftSetStream");
  if (rs) return rs;
  OTF_CUDA(cudaMemsetAsync(Qi_, 0, sizeof(unsigned long long) * K3 * (fp64_ ? 2 : 1), st));
  if (!a.cellstart || a.nc < 1) {
    set_error("spme: the cell list is missing");
    return MD_EINVAL;
  }
  MeshPlan g;
  g.K = K;
  g.kl = kl;
  const dfloat kd = df_from_double(kl);
  g.kl_h = kd.h;
  g.kl_l = kd.l;
  plan_chunks(a, p_.order, sizeof(T), g);
  const int grid = (int)std::min<int64_t>((int64_t)a.nc * a.nc * g.slots, 152 * 64);
  const size_t spread_smem = ((size_t)g.cap_spread + (size_t)g.chunk * kSpreadPitch) * sizeof(T);
  const size_t gather_smem = ((size_t)2 * g.cap + (size_t)kRowWarps * kGatherBatch * kGatherPitch) * sizeof(T);
  if (!attr_) {
    for (const void *f : {(const void *)k_spme_spread<T, 4>, (const void *)k_spme_spread<T, 6>,
                          (const void *)k_spme_spread<T, 8>, (const void *)k_spme_gather<T, 4>,
                          (const void *)k_spme_gather<T, 6>, (const void *)k_spme_gather<T, 8>})
      OTF_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSpmeSmem));
    attr_ = true;
  }
  switch (p_.order) {
    case 4:
      k_spme_spread<T, 4><<<grid, kRowThreads, spread_smem, st>>>(a, g, Qi_);
      break;
    case 6:
      k_spme_spread<T, 6><<<grid, kRowThreads, spread_smem, st>>>(a, g, Qi_);
      break;
    default:
      k_spme_spread<T, 8><<<grid, kRowThreads, spread_smem, st>>>(a, g, Qi_);
  }
  k_spme_unfix<T><<<grid_of(K3), 256, 0, st>>>(Qi_, static_cast<T *>(Qr_), K3);
  OTF_LAUNCH_CHECK();
  using C = typename Cplx<T>::type;
  int rc;
  if constexpr (std::is_same<T, double>::value)
    rc = cufft_ok(cufftExecD2Z(fwd_, static_cast<double *>(Qr_), static_cast<C *>(G1_)), "cufftExecD2Z");
  else
    rc = cufft_ok(cufftExecR2C(fwd_, static_cast<float *>(Qr_), static_cast<C *>(G1_)), "cufftExecR2C");
  if (rc) return rc;
  const double V = p_.L * p_.L * p_.L;
  k_spme_conv<T><<<grid_of((int64_t)K * K * (K / 2 + 1)), 256, 0, st>>>(
      static_cast<C *>(G1_), static_cast<C *>(G2_), fac_, bmod_, K, 1.0 / p_.L, kPi * kPi / (p_.alpha * p_.alpha),
      1.0 / (kPi * V));
  OTF_LAUNCH_CHECK();
  if constexpr (std::is_same<T, double>::value) {
    rc = cufft_ok(cufftExecZ2D(inv_, static_cast<C *>(G1_), static_cast<double *>(phi_)), "cufftExecZ2D");
  } else {
    rc = cufft_ok(cufftExecC2R(inv_, static_cast<C *>(G1_), static_cast<float *>(phi_)), "cufftExecC2R");
  }
  if (rc) return rc;
  const T ke = (T)p_.ke, kL = (T)kl, cw = (T)(p_.ke * kl * kl / (8.0 * kPi * kPi)),
          self = (T)(p_.ke * p_.alpha / std::sqrt(kPi));
  const T *phi = static_cast<const T *>(phi_), *psi = static_cast<const T *>(psi_);
  switch (p_.order) {
    case 4:
      k_spme_gather<T, 4><<<grid, kRowThreads, gather_smem, st>>>(a, g, phi, psi, ke, kL, cw, self, F, epot, W);
      break;
    case 6:
      k_spme_gather<T, 6><<<grid, kRowThreads, gather_smem, st>>>(a, g, phi, psi, ke, kL, cw, self, F, epot, W);
      break;
    default:
      k_spme_gather<T, 8><<<grid, kRowThreads, gather_smem, st>>>(a, g, phi, psi, ke, kL, cw, self, F, epot, W);
  }
  OTF_LAUNCH_CHECK();
  return MD_OK;
}

int Spme::run(const SpmeAtoms &a, void *F, void *epot, void *W, cudaStream_t st) {
  if (fp64_)
    return run_t<double>(a, static_cast<double *>(F), static_cast<double *>(epot), static_cast<double *>(W), st);
  return run_t<float>(a, static_cast<float *>(F), static_cast<float *>(epot), static_cast<float *>(W), st);
}

}  // namespace otf
