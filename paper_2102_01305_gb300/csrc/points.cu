// Stand-alone immersed-boundary transfers on an arbitrary point cloud: the
// interpolation of Eq. 17 and the spreading of Eq. 15 on device arrays,
// without the implicit solve.
//
// Both run on a plan of the cloud that every call forms anew: points binned
// by the tile of PT_X x PT_Y x PT_Z cells (2D: PT_X2 x PT_Y2) that holds
// their first stencil node, and in bin order one record (first nodes, point
// index) and the twelve delta weights per point.  The interpolation reads
// the points in that order, so neighbouring warps touch neighbouring cells;
// the spreading gives one block to every output tile, which gathers the
// points of the bins around it.  The results do not depend on the order of
// the points inside a bin: an interpolation is one point's own sum, and the
// spreading adds 64-bit integers.
#include <algorithm>

#include "ib_stencil.cuh"

namespace ibl {
namespace {

constexpr double PT_FIX_SCALE = 70368744177664.0;   // 2^46
constexpr double PT_FIX_LIMIT = 9.0e18 / PT_FIX_SCALE;
constexpr int PT_BAD_STENCIL = 1;
constexpr int PT_BAD_RANGE = 2;

// Bins and output tiles: 1024 cells, whose spreading sums (33 bytes a cell in 3D
// with the padding) and candidate list take 38 KB, five 256-thread blocks on an
// SM.  A point is visited by
// every tile that its 4-node stencil reaches, 2.2 on average at 16 x 8 x 8.
constexpr int PT_X = 16, PT_Y = 8, PT_Z = 8;
constexpr int PT_X2 = 32, PT_Y2 = 32;
constexpr int PT_CELLS = 1024;
constexpr int PT_THREADS = 256;
constexpr int PT_LIST = 512;   // candidates of a tile looked at before the ones that reach it are added
// Points around one tile above which a single block would hold up the whole
// spreading (about 0.3 ms): such tiles are left to k_pt_spread_heavy.
constexpr int PT_HEAVY = 16384;

// Row and plane strides of a tile's sums in shared memory: with 20 and 176
// words (2D: 36) the eight stencil rows of four nodes that a warp adds at once
// (4 in y, 2 in z) fall into 32 different banks.
template <int D> struct PtTile {
  static constexpr int X = D == 3 ? PT_X : PT_X2;
  static constexpr int Y = D == 3 ? PT_Y : PT_Y2;
  static constexpr int Z = D == 3 ? PT_Z : 1;
  static constexpr int ROW = X + 4;
  static constexpr int PLANE = D == 3 ? 176 : ROW * Y;
  static constexpr int WORDS = PLANE * Z;
};

struct PtGeo {
  int D;
  int n[3];
  int per[3];
  int nt[3];     // tiles per axis
  int tiles;
};

__device__ __forceinline__ int wrap_once(int v, int n) { return v >= n ? v - n : v; }

// ---------------------------------------------------------------- the plan
template <int D>
__device__ __forceinline__ int bin_of(const PtGeo& g, const int b[3]) {
  using T = PtTile<D>;
  const int tz = D == 3 ? b[2] / T::Z : 0;
  return (tz * g.nt[1] + b[1] / T::Y) * g.nt[0] + b[0] / T::X;
}

// Bin and rank within the bin of every point.
template <int D>
__global__ void k_pt_bin(int m, const double* __restrict__ X, PtGeo g, int* __restrict__ cnt, int2* __restrict__ slot) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= m) return;
  int b[3] = {0, 0, 0};
  for (int a = 0; a < D; ++a) {
    long long t;
    first_node(X[3LL * l + a], g.n[a], g.per[a] != 0, b[a], t);
  }
  const int bin = bin_of<D>(g, b);
  slot[l] = make_int2(bin, atomicAdd(&cnt[bin], 1));
}

// Exclusive scan of n counters, 4096 per block of 1024 threads: a block adds
// up the counters before its own range itself (coalesced, from L2; 64 KB for
// a 256^3 grid), so no second pass waits on it.  off[n] receives the total.
constexpr int SCAN_ITEMS = 4096;
__global__ void __launch_bounds__(1024) k_pt_scan(int n, const int* __restrict__ cnt, int* __restrict__ off) {
  __shared__ int wsum[32], wpre[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int b0 = blockIdx.x * SCAN_ITEMS;
  int before = 0;
  for (int i = threadIdx.x; i < b0; i += 1024) before += cnt[i];
  for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
  const int i0 = b0 + 4 * threadIdx.x;
  int c[4], s = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    c[k] = i0 + k < n ? cnt[i0 + k] : 0;
    s += c[k];
  }
  int v = s;
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  if (lane == 31) wsum[w] = v;
  if (lane == 0) wpre[w] = before;
  __syncthreads();
  if (w == 0) {
    int x = wsum[lane], y = wpre[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += t;
    }
    for (int o = 16; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
    wsum[lane] = x;
    wpre[lane] = y;
  }
  __syncthreads();
  int run = wpre[0] + (w > 0 ? wsum[w - 1] : 0) + v - s;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (i0 + k < n) off[i0 + k] = run;
    run += c[k];
    if (i0 + k == n - 1) off[n] = run;
  }
}

// Records and weights in bin order (slot == nullptr: in the given order), and
// for the spreading V_l ds_l 2^46 as double-floats.  rec = (first nodes, point);
// a point whose stencil fails gets first node -1 and is left out later.
// EXACT64: the weights from the FP64 formula (interpolation in FP64 contexts),
// else in integers, which err by less.
template <int D, bool EXACT64>
__global__ void k_pt_records(int m, const double* __restrict__ X, PtGeo g, const int2* __restrict__ slot,
                             const int* __restrict__ off, int4* __restrict__ rec, df* __restrict__ wts,
                             const double* __restrict__ V, const double* __restrict__ ds, df* __restrict__ vd,
                             int* flag) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= m) return;
  int pos = l;
  if (slot) {
    const int2 s = slot[l];
    pos = off[s.x] + s.y;
  }
  int b[3] = {0, 0, 0};
  bool ok = true;
  float4* wo = reinterpret_cast<float4*>(wts + 12LL * pos);
  for (int a = 0; a < 3; ++a) {
    df w[4] = {df_make(1.f, 0.f), df_make(0.f, 0.f), df_make(0.f, 0.f), df_make(0.f, 0.f)};
    if (a < D) {
      const double x = X[3LL * l + a];
      ok = axis_stencil<EXACT64>(x, g.n[a], g.per[a] != 0, b[a], w) && ok;
    }
    wo[2 * a] = make_float4(w[0].hi, w[0].lo, w[1].hi, w[1].lo);
    wo[2 * a + 1] = make_float4(w[2].hi, w[2].lo, w[3].hi, w[3].lo);
  }
  rec[pos] = make_int4(ok ? b[0] : -1, b[1], b[2], l);
  if (!ok) atomicOr(flag, PT_BAD_STENCIL);
  if (V) {
    const double dl = ds[l];
    for (int c = 0; c < D; ++c) vd[3LL * pos + c] = df_from_double(V[(long long)D * l + c] * dl * PT_FIX_SCALE);
  }
}

// ---------------------------------------------------------------- interpolation
// drho and u* of one node, four values side by side.
template <class R> struct __align__(4 * sizeof(R)) Mom4 {
  R v[4];
};
__device__ __forceinline__ Mom4<float> load_mom(const Mom4<float>* p) {
  const float4 f = *reinterpret_cast<const float4*>(p);
  Mom4<float> m;
  m.v[0] = f.x; m.v[1] = f.y; m.v[2] = f.z; m.v[3] = f.w;
  return m;
}
__device__ __forceinline__ Mom4<double> load_mom(const Mom4<double>* p) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  Mom4<double> m;
  m.v[0] = a.x; m.v[1] = a.y; m.v[2] = b.x; m.v[3] = b.y;
  return m;
}
__device__ __forceinline__ void acc_term(dfacc& a, df q, float v) { acc_fma_f(a, q, v); }
__device__ __forceinline__ void acc_term(dfacc& a, df q, double v) { acc_fma(a, q, df_from_double(v)); }

// One point by four lanes, lane i = threadIdx.x % 4 taking the stencil's x
// node i: the sum over the rows of w_y w_z (drho, u*) in double-float, times
// w_x, then the four lanes in a fixed order.  node(j, k) gives the lane's
// node of row (j, k).  Four lanes rather than a warp a point: the
// double-float butterfly over 32 lanes cost more than the terms it added (1e6
// points on 256^3: 1140 us, now 191).  rho = 1 + the sum of drho (the weights sum
// to one).
template <int D, class R, class F>
__device__ __forceinline__ void interpolate_four(const df* __restrict__ w, F node, df out[4]) {
  const int i = threadIdx.x & 3;
  df wy[4], wz[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    wy[k] = w[4 + k];
    if (D == 3) wz[k] = w[8 + k];
  }
  const df wx = w[i];
  dfacc acc[4] = {acc_zero(), acc_zero(), acc_zero(), acc_zero()};
#pragma unroll
  for (int k = 0; k < (D == 3 ? 4 : 1); ++k) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const Mom4<R> v = node(j, k);
      const df q = D == 3 ? df_mul(wy[j], wz[k]) : wy[j];
#pragma unroll
      for (int c = 0; c < 4; ++c) acc_term(acc[c], q, v.v[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) out[c] = df_warp_sum(df_mul(wx, acc_value(acc[c])), 4);
  out[0] = df_add(df_make(1.f, 0.f), out[0]);
}

// Lane 3 writes rho, lane c < D component c of u*.
template <int D>
__device__ __forceinline__ void write_point(const df v[4], int l, double* __restrict__ U, double* __restrict__ rho_out) {
  const int i = threadIdx.x & 3;
  if (i == 3) {
    if (rho_out) rho_out[l] = df_to_double(v[0]);
  } else if (i < D) {
    U[(long long)D * l + i] = df_to_double(i == 0 ? v[1] : (i == 1 ? v[2] : v[3]));
  }
}

// Small clouds: a block forms the moments of its points' nodes (512 nodes,
// two a thread) in shared memory and then sums 8 points (2D: 32).  Bound by the
// scattered pulls, 16 bytes of a 64-byte DRAM access (1e4 points on 256^3: 72 us,
// DRAM 65 % busy; 90 us with a warp a point).
constexpr int DIRECT_NODES = 512;
template <int Q, class T, bool PULL>
__global__ void __launch_bounds__(256) k_points_interpolate(int m, const int4* __restrict__ rec, const df* __restrict__ wts,
                                                            const T* __restrict__ src, FluidParams<typename Store<T>::R> p,
                                                            PtGeo g, double* __restrict__ U, double* __restrict__ rho_out) {
  using R = typename Store<T>::R;
  constexpr int D = Lat<Q>::D, NN = D == 3 ? 64 : 16, PTS = DIRECT_NODES / NN;
  __shared__ Mom4<R> sm[DIRECT_NODES];
  const int p0 = blockIdx.x * PTS;
#pragma unroll
  for (int h = 0; h < DIRECT_NODES / 256; ++h) {
    const int e = h * 256 + threadIdx.x, pt = p0 + e / NN, k = e % NN;
    if (pt >= m) continue;
    const int4 r = rec[pt];
    if (r.x < 0) continue;
    const int x = wrap_once(r.x + (k & 3), g.n[0]), y = wrap_once(r.y + ((k >> 2) & 3), g.n[1]);
    const int z = D == 3 ? wrap_once(r.z + (k >> 4), g.n[2]) : 0;
    R drho, u[3];
    node_moments<Q, T, PULL>(src, x, y, z, p, drho, u);
    sm[e].v[0] = drho;
    sm[e].v[1] = u[0];
    sm[e].v[2] = u[1];
    sm[e].v[3] = u[2];
  }
  __syncthreads();
  if (threadIdx.x >= 4 * PTS) return;
  const int q = threadIdx.x >> 2, pt = p0 + q;
  const bool live = pt < m && rec[pt < m ? pt : 0].x >= 0;   // whole groups of four; every lane shuffles
  const Mom4<R>* row = sm + q * NN + (threadIdx.x & 3);
  df v[4];
  interpolate_four<D, R>(wts + 12LL * (pt < m ? pt : 0), [&](int j, int k) { return row[(k * 4 + j) * 4]; }, v);
  if (live) write_point<D>(v, rec[pt].w, U, rho_out);
}

// Clouds with at least as many stencil nodes as cells: every cell's moments
// once (the same node moments, so the same bits) into 4 N values, then the
// points read 16 bytes a node.  The moments' pass is bound by HBM: 218 us for
// 256^3 FP32 cells, 1.54 GB (721 us with gather_q's face tests per direction).
template <int Q, class T, bool PULL>
__global__ void __launch_bounds__(256) k_cell_moments(const T* __restrict__ src, FluidParams<typename Store<T>::R> p,
                                                      Mom4<typename Store<T>::R>* __restrict__ mom) {
  using R = typename Store<T>::R;
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z;
  if (x >= p.nx || y >= p.ny) return;
  Mom4<R> o;
  R u[3];
  node_moments<Q, T, PULL>(src, x, y, z, p, o.v[0], u);
  o.v[1] = u[0];
  o.v[2] = u[1];
  o.v[3] = u[2];
  mom[((long long)z * p.ny + y) * p.nx + x] = o;
}

template <int D, class R>
__global__ void __launch_bounds__(256) k_points_interpolate_cached(int m, const int4* __restrict__ rec,
                                                                   const df* __restrict__ wts,
                                                                   const Mom4<R>* __restrict__ mom, PtGeo g,
                                                                   double* __restrict__ U, double* __restrict__ rho_out) {
  const int pt = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 2);
  // lanes past the end repeat the last point and write nothing (every lane shuffles)
  const int pc = min(pt, m - 1);
  const int4 r = rec[pc];
  const bool live = pt < m && r.x >= 0;
  int b[3] = {r.x < 0 ? 0 : r.x, r.y, r.z};
  const int x = wrap_once(b[0] + (threadIdx.x & 3), g.n[0]);
  int yo[4], zo[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    yo[k] = wrap_once(b[1] + k, g.n[1]) * g.n[0] + x;
    zo[k] = D == 3 ? wrap_once(b[2] + k, g.n[2]) * g.n[1] * g.n[0] : 0;
  }
  df v[4];
  interpolate_four<D, R>(wts + 12LL * pc, [&](int j, int k) { return load_mom(mom + (zo[k] + yo[j])); }, v);
  if (live) write_point<D>(v, r.w, U, rho_out);
}

// ---------------------------------------------------------------- spreading
// A double-float in units of 2^-46 (the plan scales V ds) as an integer, its
// parts rounded separately (error <= 1 unit).  Conversions to 64-bit integers
// are as slow as FP64 arithmetic, so below 2^53 units hi is cut at 2^23 first:
// hi = A 2^23 + r with A from one 32-bit conversion, and r (|r| <= 2^22) is
// rounded by adding 1.5 2^23; the integer is that of the whole conversion,
// since A 2^23 is even.
constexpr float PT_SMALL = 0x1p53f, PT_FIX_MAXF = 0x1p62f;
__device__ __forceinline__ long long small_fixed(df v) {
  const int a = __float2int_rn(__fmul_rn(v.hi, 0x1p-23f));
  const float r = fmaf((float)a, -0x1p23f, v.hi);   // exact: a has at most 24 significant bits
  const int b = __float_as_int(__fadd_rn(r, 0x1.8p23f)) - __float_as_int(0x1.8p23f);
  const int c = __float2int_rn(v.lo);               // |lo| <= 2^28
  return ((long long)a << 23) + (long long)(b + c);
}
__device__ __forceinline__ bool to_fixed(df v, long long& out) {
  if (!(fabsf(v.hi) < (float)(PT_FIX_LIMIT * PT_FIX_SCALE))) return false;
  out = fabsf(v.hi) < PT_SMALL ? small_fixed(v) : __float2ll_rn(v.hi) + __float2ll_rn(v.lo);
  return true;
}

// A sum in fixed point as the nearest double, (double)a 2^-46, in integer
// arithmetic (the conversion instruction bounded the former pass: 213 us for
// 3 x 256^3 values).
__device__ __forceinline__ double from_fixed(unsigned long long a) {
  if (a == 0) return 0.0;
  const unsigned long long sign = a & 0x8000000000000000ull;
  const unsigned long long mag = sign ? 0ull - a : a;
  const int lz = __clzll((long long)mag);
  const unsigned long long m = mag << lz;
  unsigned long long q = m >> 11;
  const unsigned rem = (unsigned)(m & 0x7ff);
  q += (rem > 0x400 || (rem == 0x400 && (q & 1))) ? 1 : 0;
  // the leading bit of q carries into the exponent field
  const unsigned long long e = (unsigned long long)(1023 + 63 - 46 - 1 - lz);
  return __longlong_as_double((long long)(sign | ((e << 52) + q)));
}

// 64-bit sum in two shared-memory words: the low word's old value gives the carry.
__device__ __forceinline__ void shared_add64(unsigned* lo, unsigned* hi, long long v) {
  const unsigned vl = (unsigned)v;
  const unsigned old = atomicAdd(lo, vl);
  const unsigned vh = (unsigned)((unsigned long long)v >> 32) + (old + vl < old ? 1u : 0u);
  atomicAdd(hi, vh);
}

// Which of the stencil's four nodes b .. b + 3 on one axis lie in the tile
// [o, o + ext), as their first local coordinate and a bit per node; wrapped:
// the nodes beyond the axis's end, which a periodic axis puts at 0, 1, 2 (only
// the first tile can hold those).
__device__ __forceinline__ int axis_nodes(int b, int n, int o, int ext, bool wrapped, int& local) {
  local = wrapped ? b - n : b - o;
  int mk = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    mk |= (unsigned)(local + k) < (unsigned)ext && (b + k >= n) == wrapped ? 1 << k : 0;
  return mk;
}

// du(x) = sum_l V_l ds_l D(x - X_l) (Eq. 15) on one output tile: the points
// whose first node lies in the tile or in the three nodes below it on an axis
// are in the bins around it (two an axis; three where a periodic axis ends in
// a tile narrower than a stencil).  The block lists the candidates that reach
// the tile, then its warps take the list's entries in turn (without the list
// the warps that held the tile's own bin did all the work: 1257 us at 1e6
// points on 256^3, half of it in barriers): lane (i, j, k) of 4 x 4 x 2 adds
// node (i, j, k) and then (i, j, k + 2) into shared-memory sums.  The tile is
// written once, as doubles.  The former kernels added every term to global memory
// and cleared and converted the whole array in passes of their own.  Bound by
// the double-float products and conversions of the terms (1e6 points on
// 256^3: 644 us, where the three former passes took 1420); with few points by the
// output's write (1e4 points: 121 us for 403 MB, 300 before).
template <int D>
__global__ void __launch_bounds__(PT_THREADS) k_pt_spread_tiles(const int4* __restrict__ rec, const df* __restrict__ wts,
                                                                const df* __restrict__ vd, const int* __restrict__ off,
                                                                PtGeo g, long long N, double* __restrict__ out,
                                                                bool vec2, unsigned char* __restrict__ heavy, int* __restrict__ any_heavy,
                                                                int* flag) {
  using TL = PtTile<D>;
  __shared__ __align__(16) unsigned lo[D * TL::WORDS], hi[D * TL::WORDS];
  __shared__ int start[27], pre[28], listed;
  __shared__ int2 list[PT_LIST];
  const int tile = blockIdx.x;
  const int t3[3] = {tile % g.nt[0], (tile / g.nt[0]) % g.nt[1], tile / (g.nt[0] * g.nt[1])};
  const int ext[3] = {TL::X, TL::Y, TL::Z};
  const int o[3] = {t3[0] * TL::X, t3[1] * TL::Y, t3[2] * TL::Z};
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid < 32) {
    // candidate bins: own, the one below, and on a periodic axis's first tile
    // one more if the last tile holds fewer than three nodes
    int cnt = 0;
    if (lane < 27) {
      const int c[3] = {lane % 3, (lane / 3) % 3, lane / 9};
      int bt[3] = {0, 0, 0};
      bool ok = true;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (a >= D) {
          ok = ok && c[a] == 0;
          continue;
        }
        int t = t3[a] - c[a];
        if (c[a] == 2 && (t3[a] != 0 || g.n[a] - (g.nt[a] - 1) * ext[a] >= 3)) ok = false;
        if (t < 0) {
          if (g.per[a] && g.nt[a] > c[a]) t += g.nt[a];
          else ok = false;
        }
        bt[a] = t;
      }
      if (ok) {
        const int bin = (bt[2] * g.nt[1] + bt[1]) * g.nt[0] + bt[0];
        start[lane] = off[bin];
        cnt = off[bin + 1] - off[bin];
      } else {
        start[lane] = 0;
      }
    }
    int v = cnt;
    for (int s = 1; s < 32; s <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, v, s);
      if (lane >= s) v += t;
    }
    if (lane < 27) pre[lane] = v - cnt;
    if (lane == 26) pre[27] = v;
  }
  __syncthreads();
  const int total = pre[27];
  const bool is_heavy = total > PT_HEAVY;
  if (tid == 0) {
    heavy[tile] = is_heavy ? 1 : 0;
    if (is_heavy) *any_heavy = 1;
  }
  bool work = false;   // whether any point reaches the tile
  if (total > 0 && !is_heavy) {
    for (int i = tid; i < D * TL::WORDS / 4; i += PT_THREADS) {
      reinterpret_cast<uint4*>(lo)[i] = make_uint4(0u, 0u, 0u, 0u);
      reinterpret_cast<uint4*>(hi)[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    // the wrapped parts of stencils only reach an axis's first tile
    int wraps = 0;
#pragma unroll
    for (int a = 0; a < D; ++a)
      if (g.per[a] && t3[a] == 0) wraps |= 1 << a;
    for (int img = 0; img <= wraps; ++img) {   // bit a: the part wrapped on axis a
      if (img & ~wraps) continue;
      for (int c0 = 0; c0 < total; c0 += PT_LIST) {
        if (tid == 0) listed = 0;
        __syncthreads();
#pragma unroll
        for (int h = 0; h < PT_LIST / PT_THREADS; ++h) {
          const int ci = c0 + h * PT_THREADS + tid;
          bool take = false;
          int2 entry = make_int2(0, 0);
          if (ci < total) {
            int b = 0;
            while (ci >= pre[b + 1]) ++b;
            entry.x = start[b] + ci - pre[b];
            const int4 r = rec[entry.x];
            int l[3], mz = 1;
            const int mx = axis_nodes(r.x, g.n[0], o[0], TL::X, img & 1, l[0]);
            const int my = axis_nodes(r.y, g.n[1], o[1], TL::Y, img >> 1 & 1, l[1]);
            if (D == 3) mz = axis_nodes(r.z, g.n[2], o[2], TL::Z, img >> 2 & 1, l[2]);
            else l[2] = 0;
            take = r.x >= 0 && mx && my && mz;
            // local coordinates are -3 .. 31
            entry.y = mx | my << 4 | mz << 8 | (l[0] + 3) << 12 | (l[1] + 3) << 18 | (l[2] + 3) << 24;
          }
          const unsigned bal = __ballot_sync(0xffffffffu, take);
          int at = 0;
          if (lane == 0 && bal) at = atomicAdd(&listed, __popc(bal));
          at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & ((1u << lane) - 1));
          if (take) list[at] = entry;
        }
        __syncthreads();
        const int count = listed;
        work = work || count > 0;
        const int i = lane & 3, j = (lane >> 2) & 3, kh = lane >> 4;
        for (int q = tid >> 5; q < count; q += PT_THREADS / 32) {
          const int2 en = list[q];
          if (!((en.y >> i) & (en.y >> (4 + j)) & 1)) continue;
          const df* w = wts + 12LL * en.x;
          const df wxy = df_mul(w[i], w[4 + j]);
          df v[D];
#pragma unroll
          for (int c = 0; c < D; ++c) v[c] = vd[3LL * en.x + c];
          const int cell0 = ((en.y >> 18 & 63) - 3 + j) * TL::ROW + (en.y >> 12 & 63) - 3 + i;
#pragma unroll
          for (int kk = 0; kk < (D == 3 ? 2 : 1); ++kk) {
            const int k = D == 3 ? 2 * kk + kh : 0;
            if (D == 2 && kh) continue;
            if (!(en.y >> (8 + k) & 1)) continue;
            df wt = wxy;
            int cell = cell0;
            if (D == 3) {
              wt = df_mul(wxy, w[8 + k]);
              cell += ((en.y >> 24 & 63) - 3 + k) * TL::PLANE;
            }
            df t[D];
            float big = 0.f;
#pragma unroll
            for (int c = 0; c < D; ++c) {
              t[c] = df_mul(wt, v[c]);
              big = c == 0 ? fabsf(t[c].hi) : fmaxf(big, fabsf(t[c].hi));
            }
            // (fmaxf drops a NaN beside a number: the sum does not)
            if (big < PT_SMALL && t[0].hi + t[1].hi + t[D - 1].hi < PT_FIX_MAXF) {
#pragma unroll
              for (int c = 0; c < D; ++c)
                shared_add64(lo + c * TL::WORDS + cell, hi + c * TL::WORDS + cell, small_fixed(t[c]));
            } else {
              for (int c = 0; c < D; ++c) {
                long long fx;
                if (!to_fixed(t[c], fx)) atomicOr(flag, PT_BAD_RANGE);
                else shared_add64(lo + c * TL::WORDS + cell, hi + c * TL::WORDS + cell, fx);
              }
            }
          }
        }
        __syncthreads();
      }
    }
  }
  // two x-adjacent cells a thread, one 16-byte store where both exist and are aligned
  for (int e = 2 * tid; e < PT_CELLS; e += 2 * PT_THREADS) {
    const int ex = e % TL::X, ey = (e / TL::X) % TL::Y, ez = e / (TL::X * TL::Y);
    const int x = o[0] + ex, y = o[1] + ey, z = o[2] + ez;
    if (x >= g.n[0] || y >= g.n[1] || z >= g.n[2]) continue;
    const long long cell = ((long long)z * g.n[1] + y) * g.n[0] + x;
#pragma unroll
    for (int c = 0; c < D; ++c) {
      const int w = c * TL::WORDS + ez * TL::PLANE + ey * TL::ROW + ex;
      double a = 0.0, b = 0.0;
      if (work) {
        const uint2 l2 = *reinterpret_cast<const uint2*>(lo + w), h2 = *reinterpret_cast<const uint2*>(hi + w);
        if (l2.x | l2.y | h2.x | h2.y) {
          a = from_fixed((unsigned long long)h2.x << 32 | l2.x);
          b = from_fixed((unsigned long long)h2.y << 32 | l2.y);
        }
      }
      double* d = out + c * N + cell;
      if (vec2) {
        *reinterpret_cast<double2*>(d) = make_double2(a, b);
      } else {
        d[0] = a;
        if (x + 1 < g.n[0]) d[1] = b;
      }
    }
  }
}

// Tiles with more than PT_HEAVY candidates (clouds packed into a few tiles),
// which the tile kernel left zero: all points are swept by the whole grid, the
// terms that fall into such a tile added to the output in place as 64-bit
// integers, and k_pt_heavy_convert turns those tiles into doubles.  Both
// return at once when there is no such tile.
template <int D>
__global__ void k_pt_spread_heavy(int m, const int4* __restrict__ rec, const df* __restrict__ wts,
                                  const df* __restrict__ vd, PtGeo g, long long N, unsigned long long* __restrict__ acc,
                                  const unsigned char* __restrict__ heavy, const int* __restrict__ any_heavy, int* flag) {
  if (!*any_heavy) return;
  const int lane = threadIdx.x & 31;
  constexpr int NN = D == 3 ? 64 : 16;
  const int warps = gridDim.x * (blockDim.x >> 5);
  for (int pos = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; pos < m; pos += warps) {
    const int4 r = rec[pos];
    if (r.x < 0) continue;
    const df* w = wts + 12LL * pos;
    for (int k = lane; k < NN; k += 32) {
      int b[3] = {wrap_once(r.x + (k & 3), g.n[0]), wrap_once(r.y + ((k >> 2) & 3), g.n[1]),
                  D == 3 ? wrap_once(r.z + (k >> 4), g.n[2]) : 0};
      if (!heavy[bin_of<D>(g, b)]) continue;
      df wt = df_mul(w[k & 3], w[4 + ((k >> 2) & 3)]);
      if (D == 3) wt = df_mul(wt, w[8 + (k >> 4)]);
      const long long cell = ((long long)b[2] * g.n[1] + b[1]) * g.n[0] + b[0];
      for (int c = 0; c < D; ++c) {
        long long fx;
        if (!to_fixed(df_mul(wt, vd[3LL * pos + c]), fx)) {
          atomicOr(flag, PT_BAD_RANGE);
          continue;
        }
        atomicAdd(acc + c * N + cell, (unsigned long long)fx);
      }
    }
  }
}

template <int D>
__global__ void k_pt_heavy_convert(PtGeo g, long long N, unsigned long long* __restrict__ acc,
                                   const unsigned char* __restrict__ heavy, const int* __restrict__ any_heavy) {
  if (!*any_heavy) return;
  using TL = PtTile<D>;
  for (int tile = blockIdx.x; tile < g.tiles; tile += gridDim.x) {
    if (!heavy[tile]) continue;
    const int o[3] = {tile % g.nt[0] * TL::X, (tile / g.nt[0]) % g.nt[1] * TL::Y, tile / (g.nt[0] * g.nt[1]) * TL::Z};
    for (int e = threadIdx.x; e < PT_CELLS; e += blockDim.x) {
      const int x = o[0] + e % TL::X, y = o[1] + (e / TL::X) % TL::Y, z = o[2] + e / (TL::X * TL::Y);
      if (x >= g.n[0] || y >= g.n[1] || z >= g.n[2]) continue;
      const long long cell = ((long long)z * g.n[1] + y) * g.n[0] + x;
      for (int c = 0; c < D; ++c) reinterpret_cast<double*>(acc)[c * N + cell] = from_fixed(acc[c * N + cell]);
    }
  }
}

// ---------------------------------------------------------------- host side
PtGeo pt_geo(const ibl_ctx* c) {
  PtGeo g;
  g.D = c->D;
  g.n[0] = c->nx;
  g.n[1] = c->ny;
  g.n[2] = c->nz;
  const int t3[3] = {PT_X, PT_Y, PT_Z}, t2[3] = {PT_X2, PT_Y2, 1};
  for (int a = 0; a < 3; ++a) {
    const int t = c->D == 3 ? t3[a] : t2[a];
    g.per[a] = c->bc[2 * a] == IBL_PERIODIC;
    g.nt[a] = (g.n[a] + t - 1) / t;
  }
  g.tiles = g.nt[0] * g.nt[1] * g.nt[2];
  return g;
}

// The cloud's plan in the context's scratch (grown on demand).
struct PtPlan {
  const int4* rec;
  const df* wts;
  const df* vd;
  const int* off;
};

template <class P>
cudaError_t grow(P*& ptr, size_t bytes) {
  if (ptr) cudaFree(ptr);
  ptr = nullptr;
  return cudaMalloc(reinterpret_cast<void**>(&ptr), bytes);
}

cudaError_t point_scratch(ibl_ctx* c, int m, int tiles) {
  cudaError_t e = cudaSuccess;
  if (c->pt_cap < (size_t)m) {
    c->pt_cap = 0;
    const size_t n = (size_t)m;
    e = grow(c->d_pt_slot, sizeof(int2) * n);
    if (e == cudaSuccess) e = grow(c->d_pt_rec, sizeof(int4) * n);
    if (e == cudaSuccess) e = grow(c->d_pt_wts, sizeof(df) * 12 * n);
    if (e == cudaSuccess) e = grow(c->d_pt_vd, sizeof(df) * 3 * n);
    if (e != cudaSuccess) return e;
    c->pt_cap = n;
  }
  if (!c->d_pt_off) {
    // counters (tiles), offsets (tiles + 1), the heavy flag, the tiles' heavy marks
    e = grow(c->d_pt_off, sizeof(int) * (2 * (size_t)tiles + 2) + (size_t)tiles);
  }
  return e;
}

template <int D>
cudaError_t point_plan(ibl_ctx* c, int m, const double* X, const double* V, const double* ds, bool sorted, bool exact64,
                       PtPlan& plan) {
  const PtGeo g = pt_geo(c);
  cudaError_t e = point_scratch(c, m, g.tiles);
  if (e != cudaSuccess) return e;
  int* cnt = static_cast<int*>(c->d_pt_off);
  int* off = cnt + g.tiles + 1;
  int2* slot = static_cast<int2*>(c->d_pt_slot);
  const unsigned pb = (unsigned)((m + 255) / 256);
  if (sorted) {
    e = cudaMemsetAsync(cnt, 0, sizeof(int) * ((size_t)g.tiles + 1), c->stream);   // counters and the heavy flag
    if (e != cudaSuccess) return e;
    k_pt_bin<D><<<pb, 256, 0, c->stream>>>(m, X, g, cnt, slot);
    k_pt_scan<<<(unsigned)((g.tiles + SCAN_ITEMS - 1) / SCAN_ITEMS), 1024, 0, c->stream>>>(g.tiles, cnt, off);
    c->launches += 2;
  }
  int4* rec = static_cast<int4*>(c->d_pt_rec);
  df* wts = static_cast<df*>(c->d_pt_wts);
  df* vd = static_cast<df*>(c->d_pt_vd);
  if (exact64)
    k_pt_records<D, true><<<pb, 256, 0, c->stream>>>(m, X, g, sorted ? slot : nullptr, off, rec, wts, V, ds, vd,
                                                     c->d_status + 1);
  else
    k_pt_records<D, false><<<pb, 256, 0, c->stream>>>(m, X, g, sorted ? slot : nullptr, off, rec, wts, V, ds, vd,
                                                      c->d_status + 1);
  c->launches++;
  plan.rec = rec;
  plan.wts = wts;
  plan.vd = vd;
  plan.off = off;
  return cudaGetLastError();
}

// Clouds whose stencils cover less than an eighth of the grid keep the given
// order in the interpolation: they share too few nodes for the binning to pay.
constexpr long long SORT_COVER = 8;

template <int Q, class T>
cudaError_t interpolate_points(ibl_ctx* c, int m, const double* X, double* U, double* rho) {
  using R = typename Store<T>::R;
  constexpr int D = Lat<Q>::D, NN = D == 3 ? 64 : 16;
  FluidParams<R> p{};
  p.nx = c->nx;
  p.ny = c->ny;
  p.nz = c->nz;
  p.N = c->N;
  for (int i = 0; i < 6; ++i) p.bc[i] = c->bc[i];
  for (int a = 0; a < 3; ++a) {
    p.u_in[a] = (R)c->u_in[a];
    p.G[a] = (R)c->G[a];
  }
  p.rho_out = (R)c->rho_out;
  p.tg = c->tg;
  p.status = c->d_status;
  const T* src = (const T*)c->f[c->cur];
  const PtGeo g = pt_geo(c);
  const bool moments_first = (long long)m * NN >= c->N;
  PtPlan plan;
  cudaError_t e = point_plan<D>(c, m, X, nullptr, nullptr, (long long)m * NN * SORT_COVER >= c->N, sizeof(T) == 8, plan);
  if (e != cudaSuccess) return e;
  if (moments_first) {
    const size_t bytes = sizeof(Mom4<R>) * (size_t)c->N;
    if (c->pt_mom_bytes < bytes) {
      c->pt_mom_bytes = 0;
      e = grow(c->d_pt_mom, bytes);
      if (e != cudaSuccess) return e;
      c->pt_mom_bytes = bytes;
    }
    Mom4<R>* mom = static_cast<Mom4<R>*>(c->d_pt_mom);
    const dim3 cb(64, 4, 1), cg((c->nx + 63) / 64, (c->ny + 3) / 4, c->nz);
    if (c->poststream) k_cell_moments<Q, T, false><<<cg, cb, 0, c->stream>>>(src, p, mom);
    else k_cell_moments<Q, T, true><<<cg, cb, 0, c->stream>>>(src, p, mom);
    k_points_interpolate_cached<D, R><<<(unsigned)((4LL * m + 255) / 256), 256, 0, c->stream>>>(m, plan.rec, plan.wts,
                                                                                              mom, g, U, rho);
    c->launches += 2;
    return cudaGetLastError();
  }
  const unsigned blocks = (unsigned)((m + DIRECT_NODES / NN - 1) / (DIRECT_NODES / NN));
  if (c->poststream)
    k_points_interpolate<Q, T, false><<<blocks, 256, 0, c->stream>>>(m, plan.rec, plan.wts, src, p, g, U, rho);
  else
    k_points_interpolate<Q, T, true><<<blocks, 256, 0, c->stream>>>(m, plan.rec, plan.wts, src, p, g, U, rho);
  c->launches++;
  return cudaGetLastError();
}

template <int Q>
cudaError_t interpolate_points_q(ibl_ctx* c, int m, const double* X, double* U, double* rho) {
  switch (c->prec) {
    case IBL_FP64: return interpolate_points<Q, double>(c, m, X, U, rho);
    case IBL_FP32: return interpolate_points<Q, float>(c, m, X, U, rho);
    case IBL_FP16DEV: return interpolate_points<Q, __half>(c, m, X, U, rho);
    default: return interpolate_points<Q, __nv_bfloat16>(c, m, X, U, rho);
  }
}

template <int D>
cudaError_t spread_points(ibl_ctx* c, int m, const double* X, const double* V, const double* ds, double* out) {
  if (m == 0) return cudaMemsetAsync(out, 0, sizeof(double) * (size_t)D * (size_t)c->N, c->stream);
  const PtGeo g = pt_geo(c);
  PtPlan plan;
  cudaError_t e = point_plan<D>(c, m, X, V, ds, true, false, plan);
  if (e != cudaSuccess) return e;
  int* any_heavy = static_cast<int*>(c->d_pt_off) + g.tiles;
  unsigned char* heavy = reinterpret_cast<unsigned char*>(static_cast<int*>(c->d_pt_off) + 2 * (size_t)g.tiles + 2);
  const bool vec2 = c->nx % 2 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0;
  k_pt_spread_tiles<D><<<(unsigned)g.tiles, PT_THREADS, 0, c->stream>>>(plan.rec, plan.wts, plan.vd, plan.off, g, c->N,
                                                                       out, vec2, heavy, any_heavy, c->d_status + 1);
  c->launches++;
  if (m > PT_HEAVY) {
    unsigned long long* acc = reinterpret_cast<unsigned long long*>(out);
    k_pt_spread_heavy<D><<<num_sms() * 8, 256, 0, c->stream>>>(m, plan.rec, plan.wts, plan.vd, g, c->N, acc, heavy,
                                                             any_heavy, c->d_status + 1);
    k_pt_heavy_convert<D><<<num_sms() * 2, 256, 0, c->stream>>>(g, c->N, acc, heavy, any_heavy);
    c->launches += 2;
  }
  return cudaGetLastError();
}

bool axes_ok(const ibl_ctx* c) {
  const int n[3] = {c->nx, c->ny, c->nz};
  for (int a = 0; a < c->D; ++a)
    if (n[a] < 8) return false;
  return true;
}

// Status of an enqueued point operator: one blocking copy of both words (the
// steps' status bits and the operator's flag) waits for the stream and brings
// everything that the call reports; a set bit is folded in by the usual route.
ibl_status finish(ibl_ctx* c, cudaError_t e, const char* what) {
  int st[2] = {0, 0};
  if (e == cudaSuccess) e = to_host(c, st, c->d_status, sizeof(st));
  if (e == cudaSuccess && st[1]) e = cudaMemsetAsync(c->d_status + 1, 0, sizeof(int), c->stream);
  if (e != cudaSuccess) return cuda_check(c, e, what);
  const ibl_status s = st[0] || c->sticky ? sync_and_collect(c) : IBL_OK;
  if (s != IBL_OK && s != IBL_ENOTCONV) return s;
  if (st[1] & PT_BAD_STENCIL) return fail(c, IBL_EINVAL, "a point's stencil leaves a bounded axis (or is not finite)");
  if (st[1] & PT_BAD_RANGE) return fail(c, IBL_EINVAL, "|V ds| exceeds the fixed-point range of the spreading");
  return s;
}

}  // namespace
}  // namespace ibl

using namespace ibl;

extern "C" {

ibl_status ibl_interpolate_points(ibl_ctx* c, int32_t m, const double* d_X, double* d_U, double* d_rho) {
  if (!c) return IBL_EINVAL;
  if (m < 0 || (m > 0 && (!d_X || !d_U))) return fail(c, IBL_EINVAL, "ibl_interpolate_points: bad arguments");
  if (!axes_ok(c)) return fail(c, IBL_EINVAL, "axes carrying points need at least 8 nodes");
  if (!c->initialised) return fail(c, IBL_ESTATE, "fluid not initialised");
  if (m == 0 || c->sticky) {   // nothing to do, or an error that an earlier call has reported
    const ibl_status s = sync_and_collect(c);
    if (m == 0 || (s != IBL_OK && s != IBL_ENOTCONV)) return s;
  }
  const cudaError_t e = c->Q == 9 ? interpolate_points_q<9>(c, m, d_X, d_U, d_rho)
                                  : interpolate_points_q<19>(c, m, d_X, d_U, d_rho);
  return finish(c, e, "ibl_interpolate_points");
}

ibl_status ibl_spread_points(ibl_ctx* c, int32_t m, const double* d_X, const double* d_V, const double* d_ds,
                             double* d_out) {
  if (!c) return IBL_EINVAL;
  if (m < 0 || !d_out || (m > 0 && (!d_X || !d_V || !d_ds)))
    return fail(c, IBL_EINVAL, "ibl_spread_points: bad arguments");
  if (!axes_ok(c)) return fail(c, IBL_EINVAL, "axes carrying points need at least 8 nodes");
  if (c->sticky) {
    const ibl_status s = sync_and_collect(c);
    if (s != IBL_OK && s != IBL_ENOTCONV) return s;
  }
  const cudaError_t e = c->D == 2 ? spread_points<2>(c, m, d_X, d_V, d_ds, d_out)
                                  : spread_points<3>(c, m, d_X, d_V, d_ds, d_out);
  return finish(c, e, "ibl_spread_points");
}

}  // extern "C"
