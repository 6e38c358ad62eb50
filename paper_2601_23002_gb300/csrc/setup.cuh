// Per-cell setup kernels: ion structure factor and local pseudopotential,
// Ewald ion-ion energy, the nonlocal kernel table K(|G|), S_ei shell sums.
#pragma once
#include "common.cuh"
#include "passes.cuh"

namespace ofdft {

// ---------------------------------------------------------------------------
// Structure factor on the half spectrum.  Phases factorise per axis:
// exp(-i G.R) = e_x(m_x) e_y(m_y) e_z(m_z) with e_d(m) = exp(-2 pi i m R_d / L);
// ph[(I*3 + d)*n + k] holds them (k in FFT order): FP64 values, in FP32 plans as pairs
// of floats (48 bits); pt the same rounded to the plan's type (FP64 plans: ph itself).
// One sine and cosine per |m|, the negative m by conjugation; one warp per (ion, axis).
// FP32 plans: its lanes evaluate e(0..15) and e(16 k), k = 0..15 (one FP64 sine and
// cosine each; 65 of them per axis at 128^3 kept the FP64 pipe busy for 13 us with 300
// ions), and e(16 k + l) = e(16 k) e(l), 3e-16 off, below the pairs' 2e-15.  FP64 plans
// evaluate every m (1e-16).
template <typename T> struct Phase;
template <> struct Phase<double> {
  using type = double2;
  static __device__ __forceinline__ double2 make(double c, double s) { return make_double2(c, s); }
  static __device__ __forceinline__ double2 conj(double2 e) { return make_double2(e.x, -e.y); }
};
template <> struct Phase<float> {
  using type = float4;                   // cos, sin, and their remainders
  static __device__ __forceinline__ float4 make(double c, double s) {
    const float ch = (float)c, sh = (float)s;
    return make_float4(ch, sh, (float)(c - (double)ch), (float)(s - (double)sh));
  }
  static __device__ __forceinline__ float4 conj(float4 e) { return make_float4(e.x, -e.y, e.z, -e.w); }
};
template <typename T> struct alignas(16) Quad { T a, b, c, d; };
// The row products P = e_x e_y and M = e_x e_y*: (Re P, Im P, Re M, Im M), each rounded
// to the plan's type once.  FP32: exact products of the leading floats (their remainders
// by fma) and of leading with trailing ones, two-sums: 1e-14 before the rounding, in 48
// FP32 operations (four FP64 products and sums per row and ion took 35 us of the FP64
// pipe for 300 ions on 128^3).
static __device__ __forceinline__ Quad<double> row_products(double2 x, double2 y, double z) {
  const double xr = x.x * z, xi = x.y * z;
  return Quad<double>{xr * y.x - xi * y.y, xr * y.y + xi * y.x, xr * y.x + xi * y.y, xi * y.x - xr * y.y};
}
static __device__ __forceinline__ float pair_sum(float2 a, float2 b) {
  const float s = a.x + b.x, t = s - a.x;
  return s + ((a.x - (s - t)) + (b.x - t) + (a.y + b.y));
}
static __device__ __forceinline__ Quad<float> row_products(float4 x, float4 y, float z) {
  const float2 xr = make_float2(x.x, x.z), xi = make_float2(x.y, x.w), yr = make_float2(y.x, y.z), yi = make_float2(y.y, y.w);
  const float2 rr = wide_mul(xr, yr), ii = wide_mul(xi, yi), ri = wide_mul(xr, yi), ir = wide_mul(xi, yr);
  const float2 mi = make_float2(-ii.x, -ii.y), mri = make_float2(-ri.x, -ri.y);
  return Quad<float>{z * pair_sum(rr, mi), z * pair_sum(ri, ir), z * pair_sum(rr, ii), z * pair_sum(ir, mri)};
}
template <typename T>
__device__ __forceinline__ void phases_part(const double* __restrict__ pos, int n_ion, int n, double L,
                                            typename Phase<T>::type* __restrict__ ph, cplx<T>* __restrict__ pt, int block,
                                            int blocks) {
  const int h = n / 2 + 1, lane = threadIdx.x & 31;
  const int per = blockDim.x >> 5;
  for (int q = block * per + (threadIdx.x >> 5); q < n_ion * 3; q += blocks * per) {
    double f = pos[q] / L;
    f -= floor(f);                       // wrap into [0, 1)
    // exp(-2 pi i m f), m f reduced modulo 1 before the trig call
    auto phase = [&](int m, double& s, double& c) {
      double mf = (double)m * f;
      mf -= rint(mf);
      sincospi(-2.0 * mf, &s, &c);
    };
    auto put = [&](int k, double c, double s) {
      ph[(size_t)q * n + k] = Phase<T>::make(c, s);
      if constexpr (sizeof(T) == 4) pt[(size_t)q * n + k] = mk<T>((T)c, (T)s);
    };
    double s0 = 0, c0 = 0;
    if constexpr (sizeof(T) == 4) phase(lane < 16 ? lane : (lane - 16) * 16, s0, c0);
    for (int mb = 0; mb < h; mb += 32) {
      const int m = mb + lane;
      double c, s;
      if constexpr (sizeof(T) == 4) {
        const int k = min(m >> 4, 15), l = m - 16 * k;     // m <= 256: l = 16 only with k = 15
        const int ll = l < 16 ? l : 17;
        const double ck = __shfl_sync(0xffffffffu, c0, 16 + k), sk = __shfl_sync(0xffffffffu, s0, 16 + k);
        const double cl = __shfl_sync(0xffffffffu, c0, ll & 31), sl = __shfl_sync(0xffffffffu, s0, ll & 31);
        c = cl; s = sl;
        if (k > 0) { c = ck * cl - sk * sl; s = ck * sl + sk * cl; }
      }
      if (m >= h) continue;
      if constexpr (sizeof(T) == 8) phase(m, s, c);
      if (2 * m < n) put(m, c, s);
      if (m > 0) put(n - m, c, -s);          // m = n/2 of even n is stored as -n/2
    }
  }
}

// S(G) = sum_I w_I exp(-i G.R_I) as a real matrix product over the ions.  With
// P = e_x(a) e_y(b) and M = e_x(a) e_y(b)*, a, b >= 0, and e_z = C + i D the four
// rows (+-a, +-b) are
//   P e_z, P* e_z:  (sum Pr C -+ sum Pi D) + i (sum Pr D +- sum Pi C)
// and the same with M: eight real sums give four complex entries, two
// multiply-adds per entry and ion.  (One product per entry and lane, with the
// phase products re-read from shared memory for each, took 492 us for 300 ions
// on the full 128^3 half spectrum; the FP32 pipe needs 17 us for these sums.)
// A thread owns TR row pairs (a, b) and TC kz; the ions go in chunks of CH whose
// row products and kz phases are staged in shared memory, so a chunk's step
// reads TR + TC/2 16-byte groups for 8 TR TC multiply-adds.  The row products are
// rounded to the plan's type once (row_products).  Two stages: the next
// chunk's kz phases are copied asynchronously and its row phases loaded before
// the current chunk's sums, one barrier per chunk.
// rows: (a, b) list, or nullptr for all 0 <= a, b <= n/2.
// zw: weights (nullptr: 1).  Outputs (any may be null): S, S2 (a second copy),
// SZ = zs S, V_loc = f.x SZ, and per block the Ewald reciprocal sum
// sum w f.y |SZ|^2 over the entries of rows with |G|^2 <= g2rows:
//   f = (v~(G)/Omega per unit charge, (2 pi/Omega) exp(-G^2/(4 eta^2))/G^2) by m^2,
// tabulated once per plan.  FP32 plans hold the first as two floats, so that V_loc
// is the FP32 rounding of the exact product without FP64 conversions and products.
// The Ewald sum loses nothing to FP32 from weight to sum, which FP32 plans carry as pairs
// of floats (48 bits; FP64 products and sums took 6 us for 300 ions on 128^3): it enters F
// directly, and its size (thousands of hartree in a large cell) is far above that of its changes.
// grid: (row tiles, kz tiles); CT threads along kz.
template <typename T> struct SfEntry;
template <> struct alignas(16) SfEntry<float> {
  float v, vlo, e, elo;
  static SfEntry make(double a, double b) {
    return {(float)a, (float)(a - (double)(float)a), (float)b, (float)(b - (double)(float)b)};
  }
  __device__ __forceinline__ float2 weight(float w) const { return make_float2(w * e, w * elo); }   // w = 1, 2
  __device__ __forceinline__ float vloc(float z) const { return fmaf(v, z, vlo * z); }
};
template <> struct alignas(16) SfEntry<double> {
  double v, e;
  static SfEntry make(double a, double b) { return {a, b}; }
  __device__ __forceinline__ double weight(double w) const { return w * e; }
  __device__ __forceinline__ double vloc(double z) const { return v * z; }
};
template <typename T> struct StructOut {
  cplx<T>*S, *S2, *SZ, *vloc;
  double zs;
  const SfEntry<T>* sf_tab;
  double m2rows;              // vloc and the Ewald sum: rows with a^2 + b^2 <= m2rows
  double* ew;
  // when set, the last block writes res[0] = sum of ew, res[1] = sum of the
  // nreal real-space partials
  double* res;
  const double* real; int nreal;
  unsigned int* counter;
};
template <typename T> struct StructCH { static constexpr int v = sizeof(T) == 4 ? 16 : 8; };   // ions per chunk
// rows a lane of the staging holds: a block has at most 32 of these rows
__host__ __device__ constexpr int struct_nr(int TR, int TC) { return TR * TC == 4 ? 2 : 1; }
// kz tiles and threads along kz (at most 64) for nh columns, TC to a thread
constexpr int struct_ctiles(int nh, int TC) { return (nh + TC * 64 - 1) / (TC * 64); }
constexpr int struct_ct(int nh, int TC) { return (nh + TC * struct_ctiles(nh, TC) - 1) / (TC * struct_ctiles(nh, TC)); }
template <typename T, int TR, int TC, int NT>
constexpr size_t struct_smem(int CT) {
  return 2 * (size_t)StructCH<T>::v * ((size_t)CT * TC * sizeof(cplx<T>) + (size_t)(NT / CT) * TR * sizeof(Quad<T>));
}
template <typename T, int TR, int TC, int NT>
__global__ void __launch_bounds__(NT) k_struct(const typename Phase<T>::type* __restrict__ ph, const cplx<T>* __restrict__ pt,
                                               const double* __restrict__ zw, int n_ion, int n,
                                               const int2* __restrict__ rows, int nrows, int CT, StructOut<T> o) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  constexpr int CH = StructCH<T>::v;
  const int h = n / 2, nh = h + 1;
  const int RB = NT / CT, RT = RB * TR, CC = CT * TC;    // row threads, rows and columns of the block
  Quad<T>* sr = reinterpret_cast<Quad<T>*>(smem_raw);    // [2][CH][RT]
  cplx<T>* se = reinterpret_cast<cplx<T>*>(sr + (size_t)2 * CH * RT);   // [2][CH][CC]
  const int tid = threadIdx.x, ct = tid % CT, rt = tid / CT;
  const bool act = rt < RB;
  const int col0 = blockIdx.y * CC;
  auto row_of = [&](int r, int& a, int& b) {
    if (rows) { const int2 v = rows[r]; a = v.x; b = v.y; }
    else { a = r / nh; b = r - a * nh; }
  };
  T acc[TR][TC][8];
#pragma unroll
  for (int i = 0; i < TR; ++i)
#pragma unroll
    for (int j = 0; j < TC; ++j)
#pragma unroll
      for (int k = 0; k < 8; ++k) acc[i][j][k] = 0;
  // Staging.  kz phases: the block's columns of an ion's z row by its warps in
  // turn (columns past nh stay zero).  Row products: a warp per ion as well, its
  // lanes over the block's rows; lane l holds row l of the block (l < RT <= 32 NR).
  constexpr int NW = NT / 32, NR = struct_nr(TR, TC);
  const int lane = tid & 31, wid = tid >> 5;
  int ra[NR], rb[NR];                                    // this lane's rows (a < 0: none)
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int l = lane + 32 * u, r = blockIdx.x * RT + l;
    ra[u] = -1; rb[u] = 0;
    if (l < RT && r < nrows) row_of(r, ra[u], rb[u]);
  }
  for (int q = tid; q < 2 * CH * CC; q += NT) se[q] = mk<T>((T)0, (T)0);
  __syncthreads();
  const int ncol = min(CC, nh - col0);
  auto stage_z = [&](int I0, int buf) {
    for (int c = wid; c < CH && I0 + c < n_ion; c += NW) {
      const cplx<T>* p = pt + ((size_t)(I0 + c) * 3 + 2) * n + col0;
      cplx<T>* d = se + ((size_t)buf * CH + c) * CC;
      for (int k = lane; k < ncol; k += 32) cp_async_c(d + k, p + k, true);
    }
    cp_async_commit();
  };
  constexpr int CW = (CH + NW - 1) / NW;                 // ions per warp and chunk
  using Ph = typename Phase<T>::type;
  Ph vx[CW][NR], vy[CW][NR];
  auto load_rows = [&](int I0) {
#pragma unroll
    for (int w = 0; w < CW; ++w) {
      const int I = I0 + wid + NW * w;
      if (wid + NW * w >= CH || I >= n_ion) continue;
      const Ph* p = ph + (size_t)I * 3 * n;
#pragma unroll
      for (int u = 0; u < NR; ++u)
        if (ra[u] >= 0) { vx[w][u] = p[ra[u]]; vy[w][u] = p[n + rb[u]]; }
    }
  };
  auto store_rows = [&](int I0, int buf) {
#pragma unroll
    for (int w = 0; w < CW; ++w) {
      const int c = wid + NW * w, I = I0 + c;
      if (c >= CH || I >= n_ion) continue;
      const T z = zw ? (T)zw[I] : (T)1;
#pragma unroll
      for (int u = 0; u < NR; ++u) {
        if (ra[u] < 0) continue;
        // (index n/2 holds -n/2)
        sr[((size_t)buf * CH + c) * RT + lane + 32 * u] =
            row_products(2 * ra[u] == n ? Phase<T>::conj(vx[w][u]) : vx[w][u],
                         2 * rb[u] == n ? Phase<T>::conj(vy[w][u]) : vy[w][u], z);
      }
    }
  };
  stage_z(0, 0);
  load_rows(0);
  store_rows(0, 0);
  cp_async_wait<0>();
  __syncthreads();
  for (int I0 = 0, buf = 0; I0 < n_ion; I0 += CH, buf ^= 1) {
    const int cnt = min(CH, n_ion - I0);
    const bool more = I0 + CH < n_ion;
    if (more) { stage_z(I0 + CH, buf ^ 1); load_rows(I0 + CH); }
    if (act) {
      const Quad<T>* pr = sr + (size_t)buf * CH * RT + rt;
      const cplx<T>* pe = se + (size_t)buf * CH * CC + ct;
#pragma unroll 2
      for (int c = 0; c < cnt; ++c) {
        Quad<T> p[TR];
        cplx<T> e[TC];
#pragma unroll
        for (int i = 0; i < TR; ++i) p[i] = pr[c * RT + RB * i];
#pragma unroll
        for (int j = 0; j < TC; ++j) e[j] = pe[c * CC + CT * j];
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
          for (int j = 0; j < TC; ++j) {
            T(&x)[8] = acc[i][j];
            x[0] = fma(p[i].a, e[j].x, x[0]); x[1] = fma(p[i].b, e[j].y, x[1]);
            x[2] = fma(p[i].a, e[j].y, x[2]); x[3] = fma(p[i].b, e[j].x, x[3]);
            x[4] = fma(p[i].c, e[j].x, x[4]); x[5] = fma(p[i].d, e[j].y, x[5]);
            x[6] = fma(p[i].c, e[j].y, x[6]); x[7] = fma(p[i].d, e[j].x, x[7]);
          }
      }
    }
    if (more) { store_rows(I0 + CH, buf ^ 1); cp_async_wait<0>(); }
    __syncthreads();
  }
  using V = typename TreeVal<T>::type;
  V ewa{};
#pragma unroll
  for (int i = 0; i < TR; ++i) {
    const int r = blockIdx.x * RT + rt + RB * i;
    if (!act || r >= nrows) continue;
    int a, b;
    row_of(r, a, b);
    const bool pa = 2 * a < n, ma = a > 0, pb = 2 * b < n, mb = b > 0;
    const bool inside = (double)(a * a + b * b) <= o.m2rows;
#pragma unroll
    for (int j = 0; j < TC; ++j) {
      const int kz = col0 + ct + CT * j;
      if (kz >= nh) continue;
      const T(&x)[8] = acc[i][j];
      SfEntry<T> f{};
      if (inside) f = o.sf_tab[a * a + b * b + kz * kz];
      V sz2{};
      auto put = [&](int kx, int ky, T re, T im) {
        const size_t at = ((size_t)kx * n + ky) * nh + kz;
        const cplx<T> s = mk<T>(re, im);
        if (o.S) o.S[at] = s;
        if (o.S2) o.S2[at] = s;
        if (o.SZ) {
          const T z = (T)o.zs;
          const cplx<T> sz = mk<T>(z * re, z * im);
          o.SZ[at] = sz;
          if (inside) {
            o.vloc[at] = mk<T>(f.vloc(sz.x), f.vloc(sz.y));
            sz2 = tree_add(sz2, wide_dot(sz, sz));
          } else {
            o.vloc[at] = mk<T>((T)0, (T)0);
          }
        }
      };
      if (pa && pb) put(a, b, x[0] - x[1], x[2] + x[3]);
      if (ma && mb) put(n - a, n - b, x[0] + x[1], x[2] - x[3]);
      if (pa && mb) put(a, n - b, x[4] - x[5], x[6] + x[7]);
      if (ma && pb) put(n - a, b, x[4] + x[5], x[6] - x[7]);
      ewa = tree_add(ewa, wide_mul(f.weight(kz == 0 || 2 * kz == n ? (T)1 : (T)2), sz2));
    }
  }
  double v[1] = {tree_get(ewa)}, out[1];
  block_sum<1>(v, red, out);
  if (tid == 0) o.ew[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = out[0];
  const int nb = gridDim.x * gridDim.y;
  if (o.res && arrive_last(o.counter, nb)) {
    double t2[2] = {0, 0}, t[2];
    for (int i = tid; i < nb; i += NT) t2[0] += __ldcg(o.ew + i);
    for (int i = tid; i < o.nreal; i += NT) t2[1] += o.real[i];
    __shared__ double red2[64];
    block_sum<2>(t2, red2, t);
    if (tid == 0) { o.res[0] = t[0]; o.res[1] = t[1]; *o.counter = 0u; }
  }
}

// ---------------------------------------------------------------------------
// Ewald: real-space sum over ion pairs and lattice images within rcut.  Each
// pair is taken once: ion I with I + d (mod n_ion), d = 0 .. n_ion/2 (d = 0, an
// ion with its own images, and d = n_ion/2 of an even count, met from both ends,
// count half).  Displacements are at minimum image (|x| <= L/2 per axis), so an
// image shift by |a| cells lies at least (|a| - 1/2) L away and the images
// |a| <= nimg = ceil(rcut/L + 1/2) - 1 per axis are all: none but the pair itself
// once L >= 2 rcut.  (Shifts of +-1 were walked for every pair: 27 times the
// distances, 152 us for 300 ions in a 28-bohr cell.)  A block walks its share of
// the (pair, image) combinations blockDim at a time, screens them in FP32 with a
// margin, compacts the ones that may be inside rcut into shared memory (warp
// ballots and a block prefix, in combination order), and only these, on dense
// warps, are measured and evaluated in FP64 (partial[block]; fixed order).

// The minimum image of a separation x: x less L times the nearest integer to x / L,
// found in FP32 where x is good to 3e-4 bohr there (|x| < 4e3), else in FP64.
// Screening (FP32) and evaluation (FP64) use the same integer, so a pair at half a
// cell has one and the same image a = 0.
static __device__ __forceinline__ bool near_origin(double x) { return fabsf((float)x) < 4e3f; }
static __device__ __forceinline__ float min_image_f(double x, double L, float Lf, float iL) {
  const float xf = (float)x;
  return near_origin(x) ? fmaf(-Lf, rintf(xf * iL), xf) : (float)(x - L * rint(x / L));
}
// the separation at image a in FP64
static __device__ __forceinline__ double at_image(double x, double L, float iL, int a) {
  return near_origin(x) ? x + L * (double)(a - rintf((float)x * iL)) : x - L * rint(x / L) + L * (double)a;
}
// The squared distance in FP32 at image (a, b, c), each axis good to 1e-3 bohr.
static __device__ __forceinline__ bool maybe_inside(const double* p, const double* q, double L, float Lf, float iL,
                                                    int a, int b, int c, float rc2m) {
  const int im[3] = {a, b, c};
  float r2 = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float u = min_image_f(p[d] - q[d], L, Lf, iL) + (float)im[d] * Lf;
    r2 += u * u;
  }
  return r2 < rc2m;
}
// the displacement at that image in FP64
static __device__ __forceinline__ double3 displacement(const double* p, const double* q, double L, float iL, int a,
                                                       int b, int c) {
  return make_double3(at_image(p[0] - q[0], L, iL, a), at_image(p[1] - q[1], L, iL, b), at_image(p[2] - q[2], L, iL, c));
}
// Slots, in thread order, of the threads with `in` among blockDim <= 256; the
// count in total.  Between two block barriers.
static __device__ __forceinline__ int compact_slot(bool in, int* wcount, int* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned bal = __ballot_sync(0xffffffffu, in);
  if (lane == 0) wcount[wid] = __popc(bal);
  __syncthreads();
  int base = 0, tot = 0;
  for (int w = 0; w < nw; ++w) { if (w == wid) base = tot; tot += wcount[w]; }
  *total = tot;
  return base + __popc(bal & ((1u << lane) - 1u));
}

static __device__ __forceinline__ void ewald_real_part(const double* __restrict__ pos, const double* __restrict__ Z,
                                                       int n_ion, double L, double eta, double rcut, int nimg,
                                                       double* __restrict__ partial, int block, int blocks) {
  __shared__ double red[32];
  __shared__ int list[256], wcount[8];
  const int side = 2 * nimg + 1;
  const int nim3 = side * side * side;
  const int nd = n_ion / 2 + 1;
  const long tot = (long)n_ion * nd * nim3;
  const long per = (tot + blocks - 1) / blocks;
  const long q0 = (long)block * per, q1 = min(tot, q0 + per);
  const double rc2 = rcut * rcut;
  const float rc2m = (float)((rcut + 4e-3) * (rcut + 4e-3)), Lf = (float)L, iLf = 1.0f / Lf;
  auto decode = [&](long q, int& I, int& J, int& d, int& a, int& b, int& c) {
    const long p = q / nim3;
    const int im = (int)(q - p * nim3);
    I = (int)(p / nd); d = (int)(p - (long)I * nd);
    J = I + d < n_ion ? I + d : I + d - n_ion;
    a = im / (side * side) - nimg; b = (im / side) % side - nimg; c = im % side - nimg;
  };
  double acc = 0;
  int I, J, d, a, b, c;
  for (long base = q0; base < q1; base += blockDim.x) {
    const long q = base + threadIdx.x;
    bool in = false;
    if (q < q1) {
      decode(q, I, J, d, a, b, c);
      in = maybe_inside(pos + I * 3, pos + J * 3, L, Lf, iLf, a, b, c, rc2m);
    }
    int total;
    const int slot = compact_slot(in, wcount, &total);
    if (in) list[slot] = threadIdx.x;
    __syncthreads();
    if ((int)threadIdx.x < total) {
      decode(base + list[threadIdx.x], I, J, d, a, b, c);
      const double3 x = displacement(pos + I * 3, pos + J * 3, L, iLf, a, b, c);
      const double r2 = x.x * x.x + x.y * x.y + x.z * x.z;
      if (r2 > 1e-24 && r2 < rc2) {
        const double r = sqrt(r2);
        acc += Z[I] * Z[J] * (d == 0 || 2 * d == n_ion ? 0.5 : 1.0) * erfc(eta * r) / r;
      }
    }
    __syncthreads();
  }
  double v[1] = {acc}, out[1];
  block_sum<1>(v, red, out);
  if (threadIdx.x == 0) partial[block] = out[0];
}

// What depends on the positions alone, in one launch: blocks 0 .. ne - 1 the
// Ewald real-space sum, the others the phases (independent chains of FP64
// latency that overlap).
template <typename T>
__global__ void __launch_bounds__(256) k_ions(const double* __restrict__ pos, const double* __restrict__ Z, int n_ion,
                                              int n, double L, typename Phase<T>::type* __restrict__ ph,
                                              cplx<T>* __restrict__ pt, double eta, double rcut, int nimg, int ne,
                                              double* __restrict__ partial) {
  if ((int)blockIdx.x < ne) ewald_real_part(pos, Z, n_ion, L, eta, rcut, nimg, partial, blockIdx.x, ne);
  else phases_part<T>(pos, n_ion, n, L, ph, pt, blockIdx.x - ne, gridDim.x - ne);
}

// ---------------------------------------------------------------------------
// Nonlocal kernel table.  One thread per integer m^2 in [0, nm2).
//   chi0(q;T) = -1/(pi^2 q) int_0^kmax k f(k) ln|(2k+q)/(2k-q)| dk
// with f(k) = 1/(1 + exp((k^2/2 - mu0)/T)).  The 4k/q part of the logarithm
// integrates to 4 pi^2 nbar / q exactly, so only the excess over it is
// integrated (no cancellation when -1/chi0 is compared with q^2/(4 nbar)).
// On the panel holding the logarithmic singularity c = q/2 the integrand is
// written with g(k) = k f(k) as g [ln(2k+q) - 4k/q] - (g - g(c)) ln|2k-q| plus
// g(c) int ln|2k-q| in closed form, and graded geometrically toward c; panel
// widths stay below pi T / k_F so the Fermi edge is resolved.
//   K(q) = [-1/chi0 - dmu0/dn - q^2/(4 nbar)] / (2 a^2 nbar^(2a-2)),  K(0) = 0.
struct KernArgs {
  double L, nbar, T, mu0, dmudn, alpha;
  int nm2;
};

static __device__ __forceinline__ double occ_fd(double k, double mu0, double T) {
  const double u = (0.5 * k * k - mu0) / T;
  if (u > 0) { const double e = exp(-u); return e / (1.0 + e); }
  return 1.0 / (1.0 + exp(u));
}

// 10-point Gauss-Legendre on [-1, 1]
static __device__ __constant__ double c_glx[10] = {
    -0.97390652851717172008, -0.86506336668898451073, -0.67940956829902440623, -0.43339539412924719080,
    -0.14887433898163121088, 0.14887433898163121088, 0.43339539412924719080, 0.67940956829902440623,
    0.86506336668898451073, 0.97390652851717172008};
static __device__ __constant__ double c_glw[10] = {
    0.06667134430868813759, 0.14945134915058059315, 0.21908636251598204400, 0.26926671930999635509,
    0.29552422172787993740, 0.29552422172787993740, 0.26926671930999635509, 0.21908636251598204400,
    0.14945134915058059315, 0.06667134430868813759};

// Gauss-Legendre on [a, b] of g(k) [ln|(2k+q)/(2k-q)| - 4k/q], for panels that
// do not contain q/2: x = 2k/q, 2 (atanh x - x) below 1, ln((x+1)/(x-1)) - 2x above.
static __device__ double lind_panel_plain(double a, double b, double q, double mu0, double T) {
  const double h = 0.5 * (b - a), m = 0.5 * (b + a);
  double s = 0;
#pragma unroll
  for (int j = 0; j < 10; ++j) {
    const double k = m + h * c_glx[j];
    const double x = 2.0 * k / q;
    const double e = x < 1.0 ? 2.0 * (atanh(x) - x) : log((x + 1.0) / (x - 1.0)) - 2.0 * x;
    s += c_glw[j] * k * occ_fd(k, mu0, T) * e;
  }
  return s * h;
}

// Same integrand near q/2, written g [ln(2k+q) - 4k/q] - (g - g(c)) ln|2k - q|
// (the g(c) ln|2k - q| part is added in closed form by the caller).
static __device__ double lind_panel_split(double a, double b, double q, double c, double gc, double mu0,
                                          double T) {
  const double h = 0.5 * (b - a), m = 0.5 * (b + a);
  double s = 0;
#pragma unroll
  for (int j = 0; j < 10; ++j) {
    const double k = m + h * c_glx[j];
    const double g = k * occ_fd(k, mu0, T);
    const double d = fabs(2.0 * k - q);
    double v = g * (log(2.0 * k + q) - 4.0 * k / q);
    if (d > 0) v -= (g - gc) * log(d);
    s += c_glw[j] * v;
  }
  return s * h;
}

// One warp per m^2 (kKernWarps warps per block): the lanes take the plain
// panels and the graded levels in turn, and the lane sums are added by a
// fixed shuffle tree, so the result does not depend on the launch.  (One
// thread per m^2 left a small grid's table to a few hundred threads, each
// integrating thousands of panels: 5.6 ms at 16^3.)
constexpr int kKernWarps = 4;
static __global__ void __launch_bounds__(32 * kKernWarps) k_kernel_table(KernArgs a, double* __restrict__ Kout) {
  const int lane = threadIdx.x & 31;
  const int m2 = blockIdx.x * kKernWarps + (threadIdx.x >> 5);
  if (m2 >= a.nm2) return;                            // whole warps leave together
  if (m2 == 0) { if (lane == 0) Kout[0] = 0.0; return; }
  const double q = 2.0 * kPi / a.L * sqrt((double)m2);
  const double T = a.T, mu0 = a.mu0;
  const double kmax = sqrt(2.0 * fmax(mu0 + 45.0 * T, 45.0 * T));
  const double kedge = mu0 > 0 ? sqrt(2.0 * mu0) : sqrt(2.0 * T);
  double hmax = fmin(kmax / 16.0, 0.5 * kPi * T / fmax(kedge, sqrt(2.0 * T)));
  const int npan = min(4096, (int)ceil(kmax / hmax));
  const double h = kmax / npan;     // plain panel width
  const double c = 0.5 * q;
  const double gc = c * occ_fd(c, mu0, T);
  // closed form of int ln|2k - q| dk: (1/2) [u ln|u| - u], u = 2k - q
  auto F = [](double u) { return u == 0 ? 0.0 : u * log(fabs(u)) - u; };
  double part = 0;   // this lane's share of int_0^kmax k f(k) [ln|(2k+q)/(2k-q)| - 4k/q] dk
  // graded region [ga, gb] around c (at least 2 panel widths on each side, so
  // that every plain panel stays >= 2h away from the singularity)
  const bool sing = c < kmax + 2.0 * h;
  const double ga = sing ? fmax(0.0, c - 2.0 * h) : kmax;
  const double gb = sing ? fmin(kmax, c + 2.0 * h) : kmax;
  // plain panels on [0, ga] and [gb, kmax]
  auto plain = [&](double a0, double b0) {
    if (b0 <= a0) return;
    const int np = max(1, (int)ceil((b0 - a0) / h));
    const double hh = (b0 - a0) / np;
    for (int p = lane; p < np; p += 32) part += lind_panel_plain(a0 + p * hh, a0 + (p + 1) * hh, q, mu0, T);
  };
  plain(0.0, ga);
  plain(gb, kmax);
  if (sing && gb > ga) {
    // split at c (if inside), grade geometrically toward c from both ends:
    // level l covers [cl - w 2^-l, cl - w 2^-(l+1)] on the left (w = cl - ga)
    // and [cl + w' 2^-(l+1), cl + w' 2^-l] on the right (w' = gb - cl), down
    // to widths of 1e-15 (c + h), at most 48 levels a side
    const double cl = fmin(fmax(c, ga), gb);
    const double wl = cl - ga, wr = gb - cl, wmin = 1e-15 * (c + h);
    for (int lev = lane; lev < 96; lev += 32) {
      const bool left = lev < 48;
      const int l = left ? lev : lev - 48;
      const double w = (left ? wl : wr) * ldexp(1.0, -l);
      if (!(w > wmin)) continue;
      if (left) part += lind_panel_split(cl - w, cl - 0.5 * w, q, c, gc, mu0, T);
      else part += lind_panel_split(cl + 0.5 * w, cl + w, q, c, gc, mu0, T);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if (lane != 0) return;
  double integral = part;
  if (sing && gb > ga) integral -= gc * 0.5 * (F(2.0 * gb - q) - F(2.0 * ga - q));
  // chi0 = -(4 nbar / q^2)(1 + eps);  -1/chi0 - q^2/(4 nbar) = -(q^2/(4 nbar)) eps / (1 + eps)
  const double eps = integral * q / (4.0 * kPi * kPi * a.nbar);
  const double resp_excess = -q * q / (4.0 * a.nbar) * eps / (1.0 + eps);
  const double denom = 2.0 * a.alpha * a.alpha * pow(a.nbar, 2.0 * a.alpha - 2.0);
  Kout[m2] = (resp_excess - a.dmudn) / denom;
}

// Launch shape of k_kernel_table for nm2 entries.
inline int kernel_table_blocks(int nm2) { return (nm2 + kKernWarps - 1) / kKernWarps; }

// I_{-1/2}(eta) = int_0^inf 2 / (1 + exp(t^2 - eta)) dt at the mean density,
// FP64: 400 panels of 10-point Gauss-Legendre, one panel per thread (one
// block of kMeanThreads), summed by a fixed tree.
constexpr int kMeanThreads = 512;
static __global__ void __launch_bounds__(kMeanThreads) k_mean_density(double y, double T, double* out) {
  __shared__ double red[kMeanThreads];
  double eta, p;
  fd_eta_p(y, eta, p);
  const double tmax = sqrt(fmax(eta, 0.0) + 60.0);
  const int npan = 400;
  const double h = tmax / npan;
  double s = 0;
  for (int i = threadIdx.x; i < npan; i += blockDim.x) {
    const double a = i * h, m = a + 0.5 * h;
    for (int j = 0; j < 10; ++j) {
      const double t = m + 0.5 * h * c_glx[j];
      const double u = t * t - eta;
      const double f = u > 0 ? exp(-u) / (1.0 + exp(-u)) : 1.0 / (1.0 + exp(u));
      s += c_glw[j] * 2.0 * f;
    }
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x >> 1; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x != 0) return;
  const double im = red[0] * 0.5 * h;
  out[0] = eta;
  out[1] = T * eta;                                                      // mu0
  out[2] = 2.0 * kPi * kPi / (1.4142135623730950488 * sqrt(T) * im);     // dmu0/dn
  out[3] = im;
}

// ---------------------------------------------------------------------------
// Structure-factor shells: block s sums over the half-spectrum entries of
// shell s (CSR lists built on the host; entry kx | ky << 10 | kz << 20, w =
// Hermitian weight), FP64, fixed order.  out[3 s] = sum w Re[n~ S*] scale,
// out[3 s + 1] = sum w |S|^2, out[3 s + 2] = sum w (pinned host memory).
template <typename T>
__global__ void __launch_bounds__(256) k_sei_shells(const cplx<T>* __restrict__ nt, SpecView view,
                                                    const cplx<T>* __restrict__ S, const int* __restrict__ ptr,
                                                    const int* __restrict__ idx, const float* __restrict__ wgt,
                                                    double scale, double* __restrict__ out) {
  __shared__ double red[3 * 32];
  const int s = blockIdx.x, n = view.n, nh = n / 2 + 1;
  double acc[3] = {0, 0, 0};
  for (int e = ptr[s] + threadIdx.x; e < ptr[s + 1]; e += blockDim.x) {
    const int q = idx[e], kx = q & 1023, ky = (q >> 10) & 1023, kz = q >> 20;
    const cplx<T> a = nt[view.at(kx, ky, kz)], b = S[((size_t)kx * n + ky) * nh + kz];
    const double w = (double)wgt[e];
    acc[0] += w * ((double)a.x * (double)b.x + (double)a.y * (double)b.y) * scale;
    acc[1] += w * ((double)b.x * (double)b.x + (double)b.y * (double)b.y);
    acc[2] += w;
  }
  double o[3];
  block_sum<3>(acc, red, o);
  if (threadIdx.x == 0) { out[3 * s] = o[0]; out[3 * s + 1] = o[1]; out[3 * s + 2] = o[2]; }
}

}  // namespace ofdft

namespace ofdft {

// ---------------------------------------------------------------------------
// Hellmann-Feynman forces at a given density (same derivation as the energy:
// at fixed n the ions enter only through E_loc and the Ewald energy).
//   F_I = -Z_I sum_G Im[qq(G) e_I(G)] G  +  Ewald real-space part,
//   e_I(G) = exp(-i G.R_I),  qq(G) = w(G) conj(vfac(G) n~(G) + efac(G) A(G)),
//   A(G) = sum_J Z_J exp(-i G.R_J),  vfac = -4 pi exp(-G^2 rc^2/4)/G^2 (per unit Z),
//   efac = (4 pi / Omega) exp(-G^2/(4 eta^2))/G^2,
// over 0 < |G|^2 within the local and Ewald cutoffs (half spectrum with
// Hermitian weight w = 2, or 1 on the kz = 0 and n/2 planes), the G set and
// signed m of k_struct, so the forces are the exact derivative of the energy the
// evaluation computes.
//
// The G are taken as row pairs (a, b), a, b >= 0, of four rows (+-a, +-b) each
// (see k_struct), rows[] sorted by a^2 + b^2; a tile of 32 pairs shares its
// largest kz.  qq in the order [tile][kz][half][lane] of float4 / 2 double2
// (half 0: rows (+a,+b), (-a,-b); half 1: (+a,-b), (-a,+b)), zero where a row or
// kz is outside; tile t starts at kz offset tk[t] and has tk[t + 1] - tk[t] kz.

// one thread per (tile, kz, lane): the four rows' qq
template <typename T>
__global__ void k_forces_q(const cplx<T>* __restrict__ nt, SpecView view, const cplx<T>* __restrict__ SZ,
                           const int2* __restrict__ rows, int nrows, const int* __restrict__ tk, int ntile,
                           const double2* __restrict__ gf, int m2max, int n, double invN, Quad<T>* __restrict__ qq) {
  const int nh = n / 2 + 1;
  const int lane = threadIdx.x & 31;
  const int tot = tk[ntile];
  for (int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < tot; g += (gridDim.x * blockDim.x) >> 5) {
    // the tile of this kz slot (uniform per warp)
    int lo = 0, hi = ntile;
    while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (tk[mid] <= g) lo = mid; else hi = mid; }
    const int kz = g - tk[lo], r = lo * 32 + lane;
    Quad<T> q0{0, 0, 0, 0}, q1{0, 0, 0, 0};
    if (r < nrows) {
      const int2 ab = rows[r];
      const int a = ab.x, b = ab.y, m2 = a * a + b * b + kz * kz;
      if (m2 > 0 && m2 <= m2max) {
        const double2 f = gf[m2];                        // (vfac, efac)
        const double w = (kz == 0 || 2 * kz == n) ? 1.0 : 2.0;
        auto one = [&](int kx, int ky, T& re, T& im) {
          const cplx<T> v = nt[view.at(kx, ky, kz)], A = SZ[((size_t)kx * n + ky) * nh + kz];
          re = (T)(w * (f.x * (double)v.x * invN + f.y * (double)A.x));
          im = (T)(-w * (f.x * (double)v.y * invN + f.y * (double)A.y));   // w conj(Q)
        };
        const bool pa = 2 * a < n, ma = a > 0, pb = 2 * b < n, mb = b > 0;
        if (pa && pb) one(a, b, q0.a, q0.b);
        if (ma && mb) one(n - a, n - b, q0.c, q0.d);
        if (pa && mb) one(a, n - b, q1.a, q1.b);
        if (ma && pb) one(n - a, b, q1.c, q1.d);
      }
    }
    qq[((size_t)g * 2) * 32 + lane] = q0;
    qq[((size_t)g * 2 + 1) * 32 + lane] = q1;
  }
}

// Ewald real-space force on ion I = block / nsplit from the share
// block % nsplit of its (J, image) terms, FP64, into part[block * 3
// ..] (k_sum_force_parts adds the shares in a fixed order).  Images and
// compaction of the in-range terms as in ewald_real_part.
struct EwaldForceArgs {
  const double *pos, *Z;
  double L, eta, rcut;
  int nimg, nsplit;
  double* part;
};
static __device__ __forceinline__ void ewald_force_part(const EwaldForceArgs& w, int n_ion, int block) {
  __shared__ double red[3 * 32];
  __shared__ int list[256], wcount[8];
  const int I = block / w.nsplit, sh = block % w.nsplit;
  const int side = 2 * w.nimg + 1;
  const int nim3 = side * side * side;
  const long tot = (long)n_ion * nim3;
  const long per = (tot + w.nsplit - 1) / w.nsplit;
  const long q0 = (long)sh * per, q1 = min(tot, q0 + per);
  const double rc2 = w.rcut * w.rcut;
  const double c2 = 2.0 * w.eta / 1.7724538509055160273;   // 2 eta / sqrt(pi)
  const float rc2m = (float)((w.rcut + 4e-3) * (w.rcut + 4e-3)), Lf = (float)w.L, iLf = 1.0f / Lf;
  auto decode = [&](long q, int& J, int& a, int& b, int& c) {
    J = (int)(q / nim3);
    const int im = (int)(q - (long)J * nim3);
    a = im / (side * side) - w.nimg; b = (im / side) % side - w.nimg; c = im % side - w.nimg;
  };
  const double* pI = w.pos + I * 3;
  double f[3] = {0, 0, 0};
  int J, a, b, c;
  for (long base = q0; base < q1; base += blockDim.x) {
    const long q = base + threadIdx.x;
    bool in = false;
    if (q < q1) {
      decode(q, J, a, b, c);
      in = maybe_inside(pI, w.pos + J * 3, w.L, Lf, iLf, a, b, c, rc2m);
    }
    int total;
    const int slot = compact_slot(in, wcount, &total);
    if (in) list[slot] = threadIdx.x;
    __syncthreads();
    if ((int)threadIdx.x < total) {
      decode(base + list[threadIdx.x], J, a, b, c);
      const double3 x = displacement(pI, w.pos + J * 3, w.L, iLf, a, b, c);
      const double rr = x.x * x.x + x.y * x.y + x.z * x.z;
      if (rr > 1e-24 && rr < rc2) {
        const double r = sqrt(rr);
        const double s = w.Z[I] * w.Z[J] * (erfc(w.eta * r) / rr + c2 * exp(-w.eta * w.eta * rr) / r) / r;
        f[0] += s * x.x; f[1] += s * x.y; f[2] += s * x.z;
      }
    }
    __syncthreads();
  }
  double o[3];
  block_sum<3>(f, red, o);
  if (threadIdx.x == 0) {
    double* part = w.part + (size_t)block * 3;
    part[0] = o[0]; part[1] = o[1]; part[2] = o[2];
  }
}

// Block: one tile of 32 row pairs (a lane each) and NW TI ions (TI per warp).
// Along kz (from the tile's largest down) a lane sums U = sum qq e_z and V = sum m_z qq e_z
// for its four rows: KF kz at a time as running sums (V by adding U after every step), which
// then go into sums without loss (U, and V + kz U).  In FP32, KF = 2, 21 operations per G
// and ion (34 for every term without loss): the rounding of these sums and products
// leaves (4.4, 4.4, 3.9)e-9 hartree/bohr on three ions in 27 bohr, compensated sums of
// single terms with FP32 products (11.8, 11.6, 4.5)e-9, sums running over the whole column
// (13.5, 11.8, 7.0)e-9.  Against the tile's qq (registers, read once per TI ions) and the ions' e_z (broadcast
// from shared memory); then Im[P U] etc. times (a, b) and Im[P V], summed over the lanes.
// (A gather of three phases and two complex products per
// G and ion took 186 us for 128 ions at 108^3.)  part[tile][ion][3], FP64, without the factor -Z_I 2 pi / L.
// grid.x: ntile tiles times ny ion groups, then n_ion nsplit blocks of the
// Ewald real-space part, which overlap with them.
constexpr int kForceWarps = 4;
template <typename T, int TI>
__global__ void __launch_bounds__(32 * kForceWarps) k_forces_g(const Quad<T>* __restrict__ qq, const int2* __restrict__ rows,
                                                               int nrows, const int* __restrict__ tk,
                                                               const typename Phase<T>::type* __restrict__ ph,
                                                               const cplx<T>* __restrict__ pt, int n_ion, int n,
                                                               double* __restrict__ part, int ntile, int ny,
                                                               EwaldForceArgs ewald) {
  constexpr int NI = kForceWarps * TI, KC = 32;
  __shared__ cplx<T> se[KC][NI];
  if ((int)blockIdx.x >= ntile * ny) {
    ewald_force_part(ewald, n_ion, blockIdx.x - ntile * ny);
    return;
  }
  const int tile = blockIdx.x % ntile, I0 = blockIdx.x / ntile * NI;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int k0 = tk[tile], nk = tk[tile + 1] - k0;
  using V = typename TreeVal<T>::type;                   // FP64, or pairs of floats
  constexpr int KF = sizeof(T) == 4 ? 2 : 16;
  V Ux[TI][4], Uy[TI][4], Vx[TI][4], Vy[TI][4];
  cplx<T> u[TI][4], v[TI][4];
#pragma unroll
  for (int i = 0; i < TI; ++i)
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      Ux[i][s] = Uy[i][s] = Vx[i][s] = Vy[i][s] = V{};
      u[i][s] = v[i][s] = mk<T>((T)0, (T)0);
    }
  for (int kt = nk; kt > 0; kt -= KC) {                  // chunks [kb, kt), the small terms first
    const int kb = max(0, kt - KC);
    __syncthreads();
    for (int q = threadIdx.x; q < (kt - kb) * NI; q += 32 * kForceWarps) {
      const int i = q / (kt - kb), k = q - i * (kt - kb);
      se[k][i] = I0 + i < n_ion ? pt[((size_t)(I0 + i) * 3 + 2) * n + kb + k] : mk<T>((T)0, (T)0);
    }
    __syncthreads();
    for (int k = kt - 1; k >= kb; --k) {
      const Quad<T> q0 = qq[((size_t)(k0 + k) * 2) * 32 + lane], q1 = qq[((size_t)(k0 + k) * 2 + 1) * 32 + lane];
#pragma unroll
      for (int i = 0; i < TI; ++i) {
        const cplx<T> e = se[k - kb][warp * TI + i];
        const cplx<T> q[4] = {mk<T>(q0.a, q0.b), mk<T>(q0.c, q0.d), mk<T>(q1.a, q1.b), mk<T>(q1.c, q1.d)};
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          u[i][s].x = fma(q[s].x, e.x, fma(-q[s].y, e.y, u[i][s].x));
          u[i][s].y = fma(q[s].x, e.y, fma(q[s].y, e.x, u[i][s].y));
        }
        if (2 * k == n) {                                // (the first step) kz = n/2 is -n/2
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            wide_acc(Vx[i][s], mul_rn((T)-n, u[i][s].x)); wide_acc(Vy[i][s], mul_rn((T)-n, u[i][s].y));
          }
        }
        if (k % KF != 0) {
#pragma unroll
          for (int s = 0; s < 4; ++s) { v[i][s].x += u[i][s].x; v[i][s].y += u[i][s].y; }
        } else {
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            wide_acc(Ux[i][s], u[i][s].x); wide_acc(Uy[i][s], u[i][s].y);
            wide_acc(Vx[i][s], fma((T)k, u[i][s].x, v[i][s].x)); wide_acc(Vy[i][s], fma((T)k, u[i][s].y, v[i][s].y));
            u[i][s] = v[i][s] = mk<T>((T)0, (T)0);
          }
        }
      }
    }
  }
  const int r = tile * 32 + lane;
  const int2 ab = rows[min(r, nrows - 1)];               // (lanes past the end hold zeros)
  const int a = ab.x, b = ab.y;
#pragma unroll
  for (int i = 0; i < TI; ++i) {
    const int I = I0 + warp * TI + i;
    if (I >= n_ion) break;                               // the whole warp
    const typename Phase<T>::type* p = ph + (size_t)I * 3 * n;
    const auto ex = p[a], ey = p[n + b];
    const Quad<T> pm = row_products(2 * a == n ? Phase<T>::conj(ex) : ex, 2 * b == n ? Phase<T>::conj(ey) : ey, (T)1);
    // Im[P u] and Im[P* u] of the column sums
    V w[4], z[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const T re = s < 2 ? pm.a : pm.c, im = s == 0 ? pm.b : s == 1 ? -pm.b : s == 2 ? pm.d : -pm.d;
      const T sg = s & 1 ? (T)-1 : (T)1;                 // rows (-a, -b), (-a, +b): minus in the x component
      w[s] = wide_mul(sg, tree_add(wide_mul(re, Uy[i][s]), wide_mul(im, Ux[i][s])));
      z[s] = tree_add(wide_mul(re, Vy[i][s]), wide_mul(im, Vx[i][s]));
    }
    const V p01 = tree_add(w[0], w[1]), p23 = tree_add(w[2], w[3]);
    V f[3] = {wide_mul((T)a, tree_add(p01, p23)), wide_mul((T)b, tree_add(p01, wide_mul((T)-1, p23))),
              tree_add(tree_add(z[0], z[1]), tree_add(z[2], z[3]))};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) f[d] = tree_add(f[d], shfl_xor_v(f[d], o));
      if (lane == 0) part[((size_t)tile * n_ion + I) * 3 + d] = tree_get(f[d]);
    }
  }
}

// The force component t = 3 I + d: -Z_I tp times the G-space sums gpart[tile][I][d]
// of the ntile tiles, plus the real-space shares part[(I nsplit + s) 3 + d].  One
// warp per component: lanes take the tiles and shares in turn, the lane sums are
// added by a fixed tree.
static __global__ void k_sum_force_parts(const double* __restrict__ gpart, int ntile, const double* __restrict__ Z,
                                         double tp, const double* __restrict__ part, int n_ion, int nsplit,
                                         double* __restrict__ out) {
  const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (t >= n_ion * 3) return;
  const int I = t / 3, d = t - I * 3;
  double g = 0, s = 0;
  for (int k = lane; k < ntile; k += 32) g += gpart[(size_t)k * n_ion * 3 + t];
  for (int k = lane; k < nsplit; k += 32) s += part[((size_t)I * nsplit + k) * 3 + d];
  s = warp_sum(s - Z[I] * tp * g);
  if (lane == 0) out[t] = s;
}

}  // namespace ofdft

namespace ofdft {

// ---------------------------------------------------------------------------
// Pressure P = -dF/dOmega under a homogeneous dilation (L, R_I -> lambda L,
// lambda R_I; n -> n / lambda^3; fixed T).  The local functionals contribute
// (1/Omega) int (n v - f): for TF that is n T p(y), for LDA xc n (v_xc - e_xc).
// partial[block][2] = (sum n T p, sum n (v_xc - e_xc)) over the grid; the last
// block adds them into out[0..1].
template <typename T>
__global__ void __launch_bounds__(256) k_pressure_r(const T* __restrict__ rho, size_t N, T cy, T Te, int terms,
                                                    double* __restrict__ partial, int fd64, double cy_d,
                                                    unsigned int* counter, double* out) {
  __shared__ typename TreeVal<T>::type scr[2 * 257];
  Acc<T> acc[2];
  const T nmin = (T)kNmin;
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < N; q += (size_t)gridDim.x * blockDim.x) {
    const T nval = rho[q];
    const T nf = fmax(nval, nmin);
    if (terms & 1) {
      if (sizeof(T) == 4 && fd64) {          // FP64 inversion, as in the evaluation
        double eta, p;
        fd_eta_p((double)nf * cy_d, eta, p);
        acc[0].add((T)((double)nf * (double)Te * p));
      } else {
        T eta, p;
        fd_eta_p(nf * cy, eta, p);
        acc[0].add(nf * Te * p);
      }
    }
    if (terms & 8) {
      T exc, vxc;
      pz81(nf, exc, vxc);
      acc[1].add(nval * (vxc - exc));
    }
  }
  block_sum_tree<2, T>(acc, 2, partial + (size_t)blockIdx.x * 2, scr);
  if (arrive_last(counter)) {
    block_sum_columns(partial, gridDim.x, 2, out, nullptr);
    if (threadIdx.x == 0) *counter = 0u;
  }
}

// G-space sums over the half spectrum (Hermitian weight w) of the unnormalised
// transforms nt (n), wt (n^a) and pt (sqrt n), any of them null; V_loc and the
// transforms in the view's layout:
//   0: sum w Re[n~* V_loc] c(G),  c = 3 at G = 0, 1 - G^2 rc^2/2 else (entries with
//      |G|^2 <= g2cut, as in the energy)
//   1: sum w |(n^a)~|^2 pnl(m^2),  pnl = (3 - 6a) K + dK/dlambda
//   2: sum w 4 pi |n~|^2 / G^2      3: sum w G^2 |(sqrt n)~|^2
// with the spectra scaled by the power of two sc instead of 1 / N.  A warp takes a row
// of the layout at a time.  0 and 1 (terms that cancel in the total) from the tables
// tab[m^2] = (pnl, c) to the sums in FP64, which FP32 plans carry as pairs of floats (48
// bits; FP64 products and sums took 200 of 573 us at 256^3); 2 and 3 as the evaluation's
// energies: products in the plan's precision, compensated sums.  m2cut: |G|^2 <= g2cut.
// The last block adds the blocks' partial[block][4] into out[].
template <typename T> struct PressureTab;
template <> struct PressureTab<double> {
  double pnl, c;
  static PressureTab make(double p, double c) { return {p, c}; }
};
template <> struct alignas(16) PressureTab<float> {
  float2 pnl, c;
  static float2 split(double v) { return make_float2((float)v, (float)(v - (double)(float)v)); }
  static PressureTab make(double p, double c) { return {split(p), split(c)}; }
};
template <typename T>
__global__ void __launch_bounds__(256) k_pressure_g(const cplx<T>* __restrict__ nt, const cplx<T>* __restrict__ wt,
                                                    const cplx<T>* __restrict__ pt, SpecView view,
                                                    const cplx<T>* __restrict__ vloc, const T* __restrict__ cou,
                                                    const PressureTab<T>* __restrict__ tab, T tp2, int m2cut, T sc,
                                                    double* __restrict__ partial, unsigned int* counter,
                                                    double* __restrict__ out) {
  using V = typename TreeVal<T>::type;
  __shared__ V scr[4 * 257];
  const int n = view.n, nh = n / 2 + 1;
  const int len = view.planes ? n : nh, rows = view.planes ? nh * n : n * n;
  const int lane = threadIdx.x & 31;
  auto sgn = [&](int k) { return k <= (n - 1) / 2 ? k : k - n; };
  V loc{}, nl{};
  Acc<T> har, vw;
  for (int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < rows; r += (gridDim.x * blockDim.x) >> 5) {
    const int a = r / n, b = r - a * n;
    // plane layout: row (kz = a, px = b) over py; tiled: row (kx = a, ky = b) over kz
    const int m0 = view.planes ? sgn(view.rev ? view.rev[b] : b) : sgn(a);
    const int m1 = view.planes ? 0 : sgn(b);
    for (int c = lane; c < len; c += 32) {
      const int kz = view.planes ? a : c;
      const int my = view.planes ? sgn(view.rev ? view.rev[c] : c) : m1;
      const int m2 = m0 * m0 + my * my + kz * kz;
      const T w = (kz == 0 || 2 * kz == n) ? (T)1 : (T)2;
      const size_t q = (size_t)r * len + c;
      if (nt) {
        const cplx<T> f = cscale(nt[q], sc);
        har.add(w * cou[m2] * (f.x * f.x + f.y * f.y));
        if (vloc && m2 <= m2cut) loc = tree_add(loc, wide_mul(wide_dot(cscale(f, w), vloc[q]), tab[m2].c));
      }
      if (wt) {
        const cplx<T> f = cscale(wt[q], sc);
        nl = tree_add(nl, wide_mul(wide_dot(cscale(f, w), f), tab[m2].pnl));
      }
      if (pt) {
        const cplx<T> f = cscale(pt[q], sc);
        vw.add(w * (tp2 * (T)m2) * (f.x * f.x + f.y * f.y));
      }
    }
  }
  V* col = scr + threadIdx.x;
  const int pitch = blockDim.x + 1;
  col[0] = loc; col[pitch] = nl; col[2 * pitch] = tree_put(har); col[3 * pitch] = tree_put(vw);
  block_tree_core(4, scr);
  if (threadIdx.x < 4) partial[(size_t)blockIdx.x * 4 + threadIdx.x] = tree_get(scr[threadIdx.x * pitch]);
  if (arrive_last(counter)) {
    block_sum_columns(partial, gridDim.x, 4, out, nullptr);
    if (threadIdx.x == 0) *counter = 0u;
  }
}

}  // namespace ofdft

namespace ofdft {

// The energies of a density evaluation (mode 0) from its raw sums raw[0..11]
// (see finalize_eval), written to e[0..10] in the order of ofdft_energies:
// F_TF, E_vW, E_NL, E_H, E_loc, E_xc, E_ion, F_total, N_e, mu, residual.
// One thread; the same arithmetic as the host's finish for mode 0.
static __global__ void k_finish_energies(const double* __restrict__ raw, double dV, double E_ion, int merged,
                                         double* __restrict__ e) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double E_H = raw[0], E_loc = raw[1], E_NL = raw[2], E_vW = raw[3];
  const double F_TF = raw[4] * dV, E_xc = raw[5] * dV, vn = raw[6] * dV + (merged ? E_NL : 0.0);
  const double gg = raw[8] * dV, gpsi = raw[9] * dV, ne = raw[10] * dV;
  const double mu = (vn + E_vW) / ne;
  const double r2 = (gg - 2.0 * mu * gpsi + mu * mu * ne) / ne;
  e[0] = F_TF; e[1] = E_vW; e[2] = E_NL; e[3] = E_H; e[4] = E_loc; e[5] = E_xc; e[6] = E_ion;
  e[7] = F_TF + E_vW + E_NL + E_H + E_loc + E_xc + E_ion;
  e[8] = ne; e[9] = mu; e[10] = sqrt(fmax(r2, 0.0));
}

}  // namespace ofdft
