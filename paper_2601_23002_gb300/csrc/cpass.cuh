// The passes of the plane path with the grid size known at compile time
// (2,3,5-smooth n from 24 to 160, FP32 to 250): the z passes and the plane pass of
// one evaluation, or of one preconditioning pass.
//
// What bounds the generic passes (k_zfwd, k_plane, k_zinv_epi) on these grids is
// neither memory (the spectra stay in L2) nor arithmetic but instructions and
// barriers: index arithmetic with run-time sizes, staging copies and a trip
// through shared memory per field and stage took 390 + 505 + 684 instructions
// per grid point at 75^3 (two fields), issued at 1.6 per cycle, and the plane
// pass of a small grid left most SMs idle.  Here every size, stride and radix is
// a constant; the first stage reads its inputs from memory into registers, the
// G-space terms sit between the last forward and the first inverse stage in
// registers, the last inverse stage stores to memory; all fields of a z pass go
// through each stage together (three barriers instead of a dozen); and the plane
// of a small grid, or one too large for a block, is spread over a cluster of up to
// five blocks.  One evaluation with its call, before and now: FP32 75^3 92 -> 48 us,
// 128^3 143 -> 87; FP64 45^3 193 -> 96.
//
// The FP32 transforms up to 160 keep the generic passes' radices (the same search,
// evaluated at compile time), twiddles and operation order, so a potential differs
// by how the compiler contracts a product at most: the rounding of the psi transform,
// amplified by G^2, is the largest error of an FP32 potential.  FP64 takes the radices
// that suit its pipe (dfac).
#pragma once
#include <initializer_list>
#include <cooperative_groups.h>
#include "passes.cuh"

namespace ofdft {

// ---------------------------------------------------------------------------
// Radices at compile time: the first factorisation with the fewest passes in
// the order of factor_radices, and that of factor_radices_balanced.
struct CFac { int c; int r[4]; };
constexpr int kCand[10] = {16, 12, 10, 9, 8, 6, 5, 4, 3, 2};
constexpr bool is_cand(int n) {
  for (int c : kCand) if (c == n) return true;
  return false;
}
// the k-th (k = 0 first) factorisation into three at most; bal: the smallest largest radix
constexpr CFac cfac(int n, bool bal) {
  CFac best{0, {0, 0, 0, 0}};
  int bmax = 1 << 30;
  if (is_cand(n)) return CFac{1, {n, 0, 0, 0}};
  for (int a : kCand) {
    if (n % a) continue;
    const int b = n / a;
    if (!is_cand(b)) continue;
    const int mx = a > b ? a : b;
    if (!bal) return CFac{2, {a, b, 0, 0}};
    if (mx < bmax) { bmax = mx; best = CFac{2, {a, b, 0, 0}}; }
  }
  if (best.c) return best;
  for (int a : kCand) {
    if (n % a) continue;
    for (int b : kCand) {
      if ((n / a) % b) continue;
      const int d = n / a / b;
      if (!is_cand(d)) continue;
      int mx = a > b ? a : b;
      if (d > mx) mx = d;
      if (!bal) return CFac{3, {a, b, d, 0}};
      if (mx < bmax) { bmax = mx; best = CFac{3, {a, b, d, 0}}; }
    }
  }
  return best;
}
constexpr int cdiv(int a, int b) { return (a + b - 1) / b; }

// FP64 plans choose their radices by time instead: one FP64 instruction of a warp
// takes its SM quarter's pipe 64 cycles whatever the number of active lanes, so a
// stage of `items` butterflies of radix R costs ceil(warps / 4) times the
// butterfly's instructions.  Large radices leave that pipe to one warp on small
// grids (30^3: radix 10 on 24 lanes, 140 instructions = 4.3 us per stage).
// Evaluation, all passes: 24^3 84 -> 53 us, 30^3 73 -> 60, 32^3 101 -> 55, 45^3 105 ->
// 94, 96^3 480 -> 449, 120^3 1018 -> 987, 128^3 unchanged (the same radices win).
constexpr int dcost(int r) {      // FP64 instructions of a butterfly and its twiddles
  return r == 2 ? 8 : r == 3 ? 22 : r == 4 ? 28 : r == 5 ? 50 : r == 6 ? 64 : r == 8 ? 84 : r == 9 ? 130
         : r == 10 ? 140 : r == 12 ? 155 : 230;
}
// `points` of the block in lines of `len`, nb blocks sharing an SM; per stage 24
// more for its barriers and latency and the round trip through shared memory (8
// cycles for 32 points): 128^3 keeps 8 x 16 (465 us; 4 x 4 x 8: 473)
constexpr long dstage(int points, int r, int nb) {
  return (long)cdiv(nb * cdiv(points / r, 32), 4) * dcost(r) + 24 + nb * points / 256;
}
constexpr long dtime(const CFac& f, int points, int nb) {
  long t = 0;
  for (int i = 0; i < f.c; ++i) t += dstage(points, f.r[i], nb);
  return t;
}
constexpr CFac dfac(int n, int points, int nb) {
  CFac best{0, {0, 0, 0, 0}};
  long tb = 1L << 60;
  auto look = [&](const CFac& f) {
    const long t = dtime(f, points, nb);
    if (t < tb) { tb = t; best = f; }
  };
  if (is_cand(n)) look(CFac{1, {n, 0, 0, 0}});
  for (int i = 9; i >= 0; --i) {
    const int a = kCand[i];
    if (n % a) continue;
    if (is_cand(n / a)) look(CFac{2, {a, n / a, 0, 0}});
    for (int j = i; j >= 0; --j) {
      const int b = kCand[j];
      if ((n / a) % b || !is_cand(n / a / b) || n / a / b < b) continue;
      look(CFac{3, {a, b, n / a / b, 0}});
    }
  }
  return best;
}
constexpr int least(int a, int b) { return a < b ? a : b; }
// threads for `items` items, at most `most`, in as few and as full rounds as possible
constexpr int fit_threads(int items, int most, int least) {
  const int rounds = cdiv(items, most);
  int nt = cdiv(cdiv(items, rounds), 32) * 32;
  return nt < least ? least : nt;
}

// Rows per block of the z passes: 8 up to 50^3 and 16 above.  In FP64 another count
// (even: whole sectors of a spectrum's run) where it leaves the busiest SM 5% less to
// do: the blocks run in about one wave, ceil(blocks / 152) on an SM, and the pass takes
// as long as the warps' worth of points on a quarter's FP64 pipe (plus a quarter of one
// a block).  Both z passes: 54^3 87 -> 65 us with 20 rows, 72^3 151 -> 126 with 18,
// 100^3 349 -> 292 with 22.  The same count in FP32 changed nothing beyond 2% either
// way up to 90^3 (latency, not work, fills those passes).
constexpr long z_load(int n, int r) {
  const int nb = cdiv(cdiv(n * n, r), 152);
  return 4L * cdiv(nb * cdiv(r * n, 32), 4) + nb;
}
constexpr int z_rows(int n, bool d) {
  int best = n <= 50 ? 8 : 16;
  if (!d) return best;
  long tb = z_load(n, best) * 95 / 100;
  // at least a tile schedule's 8; above 108 points more than 16 leave one block an SM
  for (int r = 8; r <= (n <= 108 ? 24 : 16); r += 2) {
    const long t = z_load(n, r);
    if (t <= tb) { tb = t; best = r; }
  }
  return best;
}

// z passes: rows per block, transform length (half for even n, full for odd n:
// two rows per transform), radices, threads, pitches.
// D: FP64.
template <int N, bool D> struct CZ {
  static constexpr bool ODD = N & 1;
  static constexpr int H = N / 2, NH = H + 1;
  static constexpr int R = z_rows(N, D);
  static constexpr int L = ODD ? N : H;
  static constexpr int LINES = ODD ? R / 2 : R;         // transforms per block and field
  static constexpr int GRID = cdiv(N * N, R);
  static constexpr CFac F = D ? dfac(L, 2 * LINES * L, cdiv(GRID, 152) < 2 ? 1 : 2) : cfac(L, !ODD);
  static constexpr int F0 = F.r[0], F1 = F.c >= 2 ? F.r[1] : 1, F2 = F.c == 3 ? F.r[2] : 1;
  static constexpr int NT = N <= 50 && R * N <= 400 ? 128 : 256;
  // element e of a line sits at e + e / F0 (even F0: the first stage writes
  // with stride F0); odd pitch, so that lines differ in bank
  static __host__ __device__ constexpr int pad(int e) { return (F0 & 1) ? e : e + e / F0; }
  static constexpr int XP = (pad(L - 1) + 1) | 1;
  static constexpr int SP = (ODD ? (N + 1) / 2 : NH) | 1;   // spectrum row pitch (odd n: two rows hold a line of L <= 2 SP)
  static constexpr int BP = (ODD ? 2 : 1) * SP;             // the same region as lines: pitch
};

// ---------------------------------------------------------------------------
// Block sums of 8 per-thread values without a tree of barriers: each warp
// halves columns and lanes together (lane bits 4..2 choose the column, 7
// additions), two more steps finish the warp, one barrier, and the first warp
// adds the warps' sums.  Fixed order.  Floats as (hi, lo) pairs (tree_add).

// scr: [warps][8]; dst[c] (c < ncol) by thread c of the first warp.  Begins
// with a barrier (scr may alias data still being read); no barrier at the end.
template <typename V>
__device__ __forceinline__ void block_sum8(V (&v)[8], V* scr, V* dst, int ncol) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  V w4[4], w2[2], w1;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool hi = lane & 16;
    const V keep = hi ? v[i + 4] : v[i], send = hi ? v[i] : v[i + 4];
    w4[i] = tree_add(keep, shfl_xor_v(send, 16));
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const bool hi = lane & 8;
    const V keep = hi ? w4[i + 2] : w4[i], send = hi ? w4[i] : w4[i + 2];
    w2[i] = tree_add(keep, shfl_xor_v(send, 8));
  }
  {
    const bool hi = lane & 4;
    const V keep = hi ? w2[1] : w2[0], send = hi ? w2[0] : w2[1];
    w1 = tree_add(keep, shfl_xor_v(send, 4));
  }
  w1 = tree_add(w1, shfl_xor_v(w1, 2));
  w1 = tree_add(w1, shfl_xor_v(w1, 1));
  const int col = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
  __syncthreads();
  if ((lane & 3) == 0) scr[wid * 8 + col] = w1;
  __syncthreads();
  if (wid == 0) {
    const int c = lane & 7;
    V s{};
    for (int w = lane >> 3; w < nw; w += 4) s = tree_add(s, scr[w * 8 + c]);
    s = tree_add(s, shfl_xor_v(s, 8));
    s = tree_add(s, shfl_xor_v(s, 16));
    if (lane < ncol) dst[lane] = s;
  }
}
template <typename T> __device__ __forceinline__ typename TreeVal<T>::type short_val(const AccShort<T>& a) {
  if constexpr (sizeof(T) == 4) return make_float2(a.s, 0.0f);
  else return a.s;
}

// finalize_eval with block_sum8: by the last block of the epilogue.
template <typename T>
static __device__ void finalize_eval8(const FinArgs<T>& f, typename TreeVal<T>::type* scr) {
  using V = typename TreeVal<T>::type;
  __shared__ V tot[16];
  const int nt = blockDim.x;
  V g[8], e[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) { g[q] = V{}; e[q] = V{}; }
  for (int b = threadIdx.x; b < f.ng; b += nt) {
#pragma unroll
    for (int q = 0; q < 4; ++q) g[q] = tree_add(g[q], __ldcg(f.pg + (size_t)b * 4 + q));
  }
  for (int b0 = threadIdx.x; b0 < f.ne; b0 += 4 * nt) {
    V x[4][8];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int b = b0 + u * nt;
#pragma unroll
      for (int q = 0; q < 8; ++q) x[u][q] = b < f.ne ? __ldcg(f.pe + (size_t)b * 8 + q) : V{};
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int q = 0; q < 8; ++q) e[q] = tree_add(e[q], x[u][q]);
  }
  block_sum8(e, scr, tot + 4, 8);
  block_sum8(g, scr, tot, 4);
  __syncthreads();
  if (threadIdx.x < 12) f.out[threadIdx.x] = tree_get(tot[threadIdx.x]);
}

// ---------------------------------------------------------------------------
// The stages of a z pass after the first, in shared memory, all lines of the
// block at once: data in xa (padded), the result as natural elements (cz_get):
// element e of a line at xa[line XP + pad(e)] for one or two stages and at
// xb[line BP + e] for three.  Ends with a barrier.
template <typename T, int N, int DIR>
__device__ __forceinline__ void cz_stages(cplx<T>* xa, cplx<T>* xb, int lines, const cplx<T>* __restrict__ tw) {
  using Z = CZ<N, sizeof(T) == 8>;
  constexpr int L = Z::L, F0 = Z::F0, F1 = Z::F1, F2 = Z::F2;
  if constexpr (Z::F.c == 1) {
    return;
  } else if constexpr (Z::F.c == 2) {
    for (int it = threadIdx.x; it < lines * F0; it += Z::NT) {
      const int ln = it / F0, j = it - ln * F0;
      cplx<T>* x = xa + ln * Z::XP;
      cplx<T> v[F1];
#pragma unroll
      for (int r = 0; r < F1; ++r) v[r] = x[Z::pad(r * F0) + j];
#pragma unroll
      for (int r = 1; r < F1; ++r) {
        cplx<T> w = tw[j * r];
        if (DIR > 0) w.y = -w.y;
        v[r] = cmul(v[r], w);
      }
      Codelet<cplx<T>, F1, DIR>::run(v);
#pragma unroll
      for (int r = 0; r < F1; ++r) x[Z::pad(r * F0) + j] = v[r];
    }
    __syncthreads();
  } else {
    constexpr int M1 = L / F1, M2 = L / F2;
    for (int it = threadIdx.x; it < lines * M1; it += Z::NT) {
      const int ln = it / M1, j = it - ln * M1;
      const cplx<T>* x = xa + ln * Z::XP;
      cplx<T> v[F1];
#pragma unroll
      for (int r = 0; r < F1; ++r) v[r] = x[Z::pad(j + r * M1)];
      const int jq = j / F0, k = j - jq * F0;
#pragma unroll
      for (int r = 1; r < F1; ++r) {
        cplx<T> w = tw[k * r * F2];
        if (DIR > 0) w.y = -w.y;
        v[r] = cmul(v[r], w);
      }
      Codelet<cplx<T>, F1, DIR>::run(v);
      cplx<T>* y = xb + ln * Z::BP + jq * F0 * F1 + k;
#pragma unroll
      for (int r = 0; r < F1; ++r) y[r * F0] = v[r];
    }
    __syncthreads();
    for (int it = threadIdx.x; it < lines * M2; it += Z::NT) {
      const int ln = it / M2, j = it - ln * M2;
      cplx<T>* y = xb + ln * Z::BP + j;
      cplx<T> v[F2];
#pragma unroll
      for (int r = 0; r < F2; ++r) v[r] = y[r * M2];
#pragma unroll
      for (int r = 1; r < F2; ++r) {
        cplx<T> w = tw[j * r];
        if (DIR > 0) w.y = -w.y;
        v[r] = cmul(v[r], w);
      }
      Codelet<cplx<T>, F2, DIR>::run(v);
#pragma unroll
      for (int r = 0; r < F2; ++r) y[r * M2] = v[r];
    }
    __syncthreads();
  }
}
template <typename T, int N>
__device__ __forceinline__ cplx<T> cz_get(const cplx<T>* xa, const cplx<T>* xb, int ln, int e) {
  using Z = CZ<N, sizeof(T) == 8>;
  if constexpr (Z::F.c <= 2) return xa[ln * Z::XP + Z::pad(e)];
  else return xb[ln * Z::BP + e];
}

// The active fields' indices and spectra by selection: a parameter array indexed
// at run time would be copied to local memory.
template <typename T> struct CField {
  int i0, i1, i2;
  cplx<T>*s0, *s1, *s2;
  __device__ __forceinline__ explicit CField(const Spectra<T>& sp) : i0(sp.idx[0]), i1(sp.idx[1]), i2(sp.idx[2]) {
    s0 = pick(sp, i0); s1 = pick(sp, i1); s2 = pick(sp, i2);
  }
  static __device__ __forceinline__ cplx<T>* pick(const Spectra<T>& sp, int i) {
    return i == 0 ? sp.s[0] : i == 1 ? sp.s[1] : sp.s[2];
  }
  __device__ __forceinline__ int id(int f) const { return f == 0 ? i0 : f == 1 ? i1 : i2; }
  __device__ __forceinline__ cplx<T>* spec(int f) const { return f == 0 ? s0 : f == 1 ? s1 : s2; }
};

// shared memory: tw[L] | twn[NH] | xa[nf][LINES][XP] | xb[nf][LINES][BP] (three
// stages) | FP64: sq[R][N] reals
template <typename T, int N> __host__ __device__ constexpr size_t czfwd_bytes(int nf) {
  using Z = CZ<N, sizeof(T) == 8>;
  return ((size_t)Z::L + Z::NH + (size_t)nf * Z::LINES * (Z::XP + (Z::F.c == 3 ? Z::BP : 0))) * sizeof(cplx<T>) +
         (sizeof(T) == 8 ? (size_t)Z::R * N * sizeof(T) : 0);
}
// Forward z pass: prologue (n, n^a, psi from rho or from psi + t d) and the
// real-to-complex transform of R rows of every active field, plane layout.
template <typename T, int N>
__global__ void __launch_bounds__(CZ<N, sizeof(T) == 8>::NT, (sizeof(T) == 4 ? 1024 : 512) / CZ<N, sizeof(T) == 8>::NT)
k_zfwd_c(ProArgs<T> a, Spectra<T> sp, const cplx<T>* __restrict__ tw_l, const cplx<T>* __restrict__ tw_n) {
  using Z = CZ<N, sizeof(T) == 8>;
  using C = cplx<T>;
  constexpr int R = Z::R, L = Z::L, H = Z::H, NH = Z::NH, F0 = Z::F0, M0 = L / F0, NN = N * N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* twn = tw + L;
  C* xa = twn + NH;
  C* xb = xa + sp.nact * Z::LINES * Z::XP;
  const CField<T> fl_(sp);
  const int row0 = blockIdx.x * R;
  const int rows = min(R, NN - row0);
  const int lines = Z::ODD ? (rows + 1) >> 1 : rows;
  for (int q = threadIdx.x; q < L + NH; q += Z::NT) tw[q] = q < L ? tw_l[q] : tw_n[q - L];
  dependency_wait();
  const T* src = (a.mode == 0 ? a.rho : a.psi) + (size_t)row0 * N;
  const bool has_d = a.mode != 0 && a.d != nullptr;
  const T* dsrc = has_d ? a.d + (size_t)row0 * N : src;
  const T tstep = a.dsc ? (T)a.dsc[2] : a.t;
  const T scale = a.dsc ? (T)a.dsc[0] : a.scale, alpha = a.alpha, nmin = (T)kNmin;
  const T shift = a.dsc ? (T)a.dsc[1] : a.psi_shift;
  // the field's value from the density (mode 0) or psi_t
  auto val = [&](int fid, T x) -> T {
    if (fid == 2) {
      if (a.mode == 0) x = sqrt(fmax(x, (T)0));
      return x - shift;
    }
    const T nv = a.mode == 0 ? x : scale * x * x;
    return fid == 0 ? nv : pow_t<T>(fmax(nv, nmin), alpha);
  };
  // FP64 and a given density: psi = sqrt(rho) by all threads first (about 20 FP64
  // instructions a point; in stage 0 the threads of the psi field alone would take
  // 2 F0 each; 45^3: 23.4 -> 16.8 us with the radices)
  T* sq = reinterpret_cast<T*>(xb + (Z::F.c == 3 ? sp.nact * Z::LINES * Z::BP : 0));
  const bool pre = sizeof(T) == 8 && a.mode == 0 && (fl_.id(sp.nact - 1) == 2);
  if (pre) {
    for (int q = threadIdx.x; q < rows * N; q += Z::NT) sq[q] = val(2, src[q]);
    __syncthreads();
  }
  // stage 0: the line's elements j + s M0 from memory, radix F0
  for (int it = threadIdx.x; it < sp.nact * Z::LINES * M0; it += Z::NT) {
    const int fl = it / M0, j = it - fl * M0;
    const int f = fl / Z::LINES, ln = fl - f * Z::LINES;
    if (ln >= lines) continue;
    const int fid = fl_.id(f);
    C v[F0];
    if constexpr (Z::ODD) {
      const bool two = 2 * ln + 1 < rows;
      const bool ready = pre && fid == 2;
      const T* p0 = (ready ? sq : src) + 2 * ln * N + j;
      const T* d0 = dsrc + 2 * ln * N + j;
#pragma unroll
      for (int s = 0; s < F0; ++s) v[s] = mk<T>(p0[s * M0], two ? p0[N + s * M0] : (T)0);
      if (has_d) {
#pragma unroll
        for (int s = 0; s < F0; ++s) {
          v[s].x = v[s].x + tstep * d0[s * M0];
          if (two) v[s].y = v[s].y + tstep * d0[N + s * M0];
        }
      }
      if (!ready) {
#pragma unroll
        for (int s = 0; s < F0; ++s) v[s] = mk<T>(val(fid, v[s].x), two ? val(fid, v[s].y) : (T)0);
      }
    } else {
      const bool ready = pre && fid == 2;
      const C* p0 = reinterpret_cast<const C*>((ready ? sq : src) + ln * N) + j;
      const C* d0 = reinterpret_cast<const C*>(dsrc + ln * N) + j;
#pragma unroll
      for (int s = 0; s < F0; ++s) v[s] = p0[s * M0];
      if (has_d) {
#pragma unroll
        for (int s = 0; s < F0; ++s) {
          const C d = d0[s * M0];
          v[s].x = v[s].x + tstep * d.x; v[s].y = v[s].y + tstep * d.y;
        }
      }
      if (!ready) {
#pragma unroll
        for (int s = 0; s < F0; ++s) v[s] = mk<T>(val(fid, v[s].x), val(fid, v[s].y));
      }
    }
    Codelet<C, F0, -1>::run(v);
    C* x = xa + fl * Z::XP + Z::pad(j * F0);
#pragma unroll
    for (int s = 0; s < F0; ++s) x[s] = v[s];
  }
  __syncthreads();
  cz_stages<T, N, -1>(xa, xb, sp.nact * Z::LINES, tw);
  // the rows' half spectra; consecutive threads take consecutive rows of one kz
  if constexpr (Z::ODD) {
    for (int q = threadIdx.x; q < sp.nact * NH * R; q += Z::NT) {
      const int fk = q / R, r = q - fk * R;
      const int f = fk / NH, k = fk - f * NH;
      if (r >= rows || k >= a.nkz) continue;
      C o;
      // X_a[k] = (Z[k] + Z*[n-k]) / 2, X_b[k] = -i (Z[k] - Z*[n-k]) / 2
      const int ln = f * Z::LINES + (r >> 1);
      const C zk = cz_get<T, N>(xa, xb, ln, k);
      const C zc = cconj(cz_get<T, N>(xa, xb, ln, k == 0 ? 0 : N - k));
      if ((r & 1) == 0) {
        o = mk<T>((T)0.5 * (zk.x + zc.x), (T)0.5 * (zk.y + zc.y));
      } else {
        const C dd = csub(zk, zc);
        o = mk<T>((T)0.5 * dd.y, (T)-0.5 * dd.x);
      }
      fl_.spec(f)[(size_t)k * NN + row0 + r] = o;
    }
  } else {
    // X[k] = (Z[k] + Z*[h-k])/2 - (i/2) W^k (Z[k] - Z*[h-k]),  k = 0..h; k and h - k
    // together: the sums and the product of one are the conjugates of the other's
    // (FP64 128^3 177 -> 162 us, two fields without the inverse at 72^3 42 -> 40)
    constexpr int HP = H / 2 + 1;
    for (int q = threadIdx.x; q < sp.nact * HP * R; q += Z::NT) {
      const int fk = q / R, r = q - fk * R;
      const int f = fk / HP, k = fk - f * HP;
      if (r >= rows || k >= a.nkz) continue;
      const int ln = f * Z::LINES + r;
      const C zk = cz_get<T, N>(xa, xb, ln, k);
      const C zc = cconj(cz_get<T, N>(xa, xb, ln, k == 0 ? 0 : H - k));
      const C e = cadd(zk, zc);
      const C wo = cmul(twn[k], csub(zk, zc));
      C* out = fl_.spec(f) + row0 + r;
      out[(size_t)k * NN] = mk<T>((T)0.5 * (e.x + wo.y), (T)0.5 * (e.y - wo.x));
      if (2 * k != H && H - k < a.nkz)
        out[(size_t)(H - k) * NN] = mk<T>((T)0.5 * (e.x - wo.y), (T)-0.5 * (e.y + wo.x));
    }
  }
}

// shared memory: tw[L] | twn[NH] | stg[nf][R][SP] | xa[nf][LINES][XP]
template <typename T, int N> __host__ __device__ constexpr size_t czinv_bytes(int nf) {
  using Z = CZ<N, sizeof(T) == 8>;
  const size_t b = ((size_t)Z::L + Z::NH + (size_t)nf * (Z::R * Z::SP + Z::LINES * Z::XP)) * sizeof(cplx<T>);
  const size_t s = (size_t)(Z::NT / 32) * 8 * 8;
  return b > s ? b : s;
}
// Inverse z pass: complex-to-real transform of R rows of every active field
// (plane layout) and the pointwise functional (KIND 0, 1, 2: see EpiPoint), or
// the preconditioning pass's output (KIND 3: mode 3).
template <typename T, int N, int KIND>
__global__ void __launch_bounds__(CZ<N, sizeof(T) == 8>::NT, (sizeof(T) == 4 ? 1024 : 512) / CZ<N, sizeof(T) == 8>::NT)
k_zinv_c(Spectra<T> sp, EpiArgs<T> a, const cplx<T>* __restrict__ tw_l, const cplx<T>* __restrict__ tw_n) {
  using Z = CZ<N, sizeof(T) == 8>;
  using C = cplx<T>;
  constexpr int R = Z::R, L = Z::L, H = Z::H, NH = Z::NH, F0 = Z::F0, M0 = L / F0, NN = N * N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* twn = tw + L;
  C* stg = twn + NH;
  C* xa = stg + sp.nact * R * Z::SP;
  const CField<T> fl_(sp);
  const int row0 = blockIdx.x * R;
  const int rows = min(R, NN - row0);
  const size_t off = (size_t)row0 * N;
  for (int q = threadIdx.x; q < L + NH; q += Z::NT) tw[q] = q < L ? tw_l[q] : tw_n[q - L];
  dependency_wait();
  for (int q = threadIdx.x; q < sp.nact * NH * R; q += Z::NT) {
    const int fk = q / R, r = q - fk * R;
    const int f = fk / NH, k = fk - f * NH;
    if (r < rows) cp_async_c(stg + (f * R + r) * Z::SP + k, fl_.spec(f) + (size_t)k * NN + row0 + r, true);
  }
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  // stage 0: Z at j + s M0 from the staged spectra, radix F0
  for (int it = threadIdx.x; it < sp.nact * Z::LINES * M0; it += Z::NT) {
    const int fl = it / M0, j = it - fl * M0;
    C v[F0];
    if constexpr (Z::ODD) {
      // Z[k] = A[k] + i B[k], rows 2 ln and 2 ln + 1, A[n-k] = A*[k] (the
      // imaginary parts at k = 0 dropped)
      const int f = fl / Z::LINES, ln = fl - f * Z::LINES;
      const C* in = stg + (f * R + 2 * ln) * Z::SP;
      const bool two = 2 * ln + 1 < rows;
#pragma unroll
      for (int s = 0; s < F0; ++s) {
        const int k = j + s * M0;
        const bool lo = k < NH;
        const int kk = lo ? k : N - k;
        C A = in[kk];
        C B = two ? in[Z::SP + kk] : mk<T>((T)0, (T)0);
        if (k == 0) { A.y = 0; B.y = 0; }
        if (!lo) { A.y = -A.y; B.y = -B.y; }
        v[s] = mk<T>(A.x - B.y, A.y + B.x);
      }
    } else {
      // Z[k] = (X[k] + X*[h-k]) + i W^-k (X[k] - X*[h-k])
      const C* in = stg + fl * Z::SP;
#pragma unroll
      for (int s = 0; s < F0; ++s) {
        const int k = j + s * M0;
        const C xk = in[k];
        const C xc = cconj(in[H - k]);
        const C e = cadd(xk, xc);
        const C o = cmul(cconj(twn[k]), csub(xk, xc));
        v[s] = mk<T>(e.x - o.y, e.y + o.x);
      }
    }
    Codelet<C, F0, +1>::run(v);
    C* x = xa + fl * Z::XP + Z::pad(j * F0);
#pragma unroll
    for (int s = 0; s < F0; ++s) x[s] = v[s];
  }
  __syncthreads();                                       // (the staged spectra are free)
  cz_stages<T, N, +1>(xa, stg, sp.nact * Z::LINES, tw);
  // real value i of row r, field slot f: component i % 2 of element i / 2 (even
  // n) or the row's component of element i (odd n)
  const T* xr = reinterpret_cast<const T*>(Z::F.c <= 2 ? xa : stg);
  auto real_at = [&](int f, int r, int i) -> T {
    constexpr int PT = Z::F.c <= 2 ? Z::XP : Z::BP;
    const int ln = f * Z::LINES + (Z::ODD ? r >> 1 : r), e = Z::ODD ? i : i >> 1, c = (Z::ODD ? r : i) & 1;
    return xr[2 * (ln * PT + (Z::F.c <= 2 ? Z::pad(e) : e)) + c];
  };
  // (r, i) of the thread's points tid, tid + NT, ...
  int r = threadIdx.x / N, i = threadIdx.x - r * N;
  auto step = [&]() {
    i += Z::NT % N; r += Z::NT / N;
    if (Z::NT % N != 0 && i >= N) { i -= N; ++r; }
  };
  if constexpr (KIND == 3) {
#pragma unroll 2
    for (int q = threadIdx.x; q < rows * N; q += Z::NT, step()) {
      const T v = real_at(0, r, i);
      a.out[off + q] = v;
      if (a.pyout) a.pyout[off + q] = v - a.pold[off + q];
    }
    return;
  } else {
  // the slot of each field, -1: not active
  int slot[3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    slot[k] = (sp.nact > 0 && fl_.i0 == k) ? 0 : (sp.nact > 1 && fl_.i1 == k) ? 1 : (sp.nact > 2 && fl_.i2 == k) ? 2 : -1;
  const EpiPoint<T, KIND> ep(sp, a);
  AccShort<T> acc[8];
  const bool with_d = KIND == 1 || (KIND == 0 && a.mode == 1);
  const T* src = (EpiPoint<T, KIND>::mode(a) == 0 ? a.rho : a.psi) + off;
  const T* dsrc = with_d ? a.d + off : src;
#pragma unroll 2
  for (int q = threadIdx.x; q < rows * N; q += Z::NT, step()) {
    const T x = src[q], d = with_d ? dsrc[q] : (T)0;
    if constexpr (KIND != 0)                             // slots 0 (n) and 1 (psi)
      ep.point(a, x, d, real_at(0, r, i), (T)0, real_at(1, r, i), off + q, acc);
    else
      ep.point(a, x, d, slot[0] >= 0 ? real_at(slot[0], r, i) : (T)0, slot[1] >= 0 ? real_at(slot[1], r, i) : (T)0,
               slot[2] >= 0 ? real_at(slot[2], r, i) : (T)0, off + q, acc);
  }
  using V = typename TreeVal<T>::type;
  V v[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) v[c] = short_val<T>(acc[c]);
  V* scr = reinterpret_cast<V*>(smem_raw);
  block_sum8(v, scr, a.partials + (size_t)blockIdx.x * 8, 8);
  if (arrive_last(a.counter)) {
    finalize_eval8<T>(a.fin, scr);
    if (threadIdx.x == 0) *a.counter = 0u;
  }
  }
}

// ---------------------------------------------------------------------------
// Plane pass on clusters of CL blocks: y and x transforms, G-space terms and
// the inverses of one kz plane of one field.  Block c of the cluster holds the
// rows ROWS c .. of the plane (as k_plane's shared-memory plane, pitch N + 1).
// CL = 1: columns in place.  CL > 1: block c transforms the columns COLS c ..;
// the first stage along x reads its rows from the cluster's blocks through
// distributed shared memory into a column buffer of its own, the last inverse
// stage writes the rows back; two cluster barriers in all.

// Shared memory of a plane pass (bytes) and, in FP64, the cluster size and radices
// by dtime: CL of 1, 2, 4 for nf fields, ROWS lines a block, cdiv(planes CL, 152)
// blocks on an SM (32^3: 16 x 2 -> 2 x 4 x 4, 38 -> 18 us a pass;
// 96^3: 16 x 6 -> 8 x 12, 225 -> 194).
constexpr size_t cp_bytes(int n, int cl, int csize) {
  const int rows = cdiv(n, cl);
  return ((size_t)rows * (n | 1) + (cl == 1 ? 0 : (size_t)n * (rows | 1)) + n) * csize;
}
constexpr long cp_time64(int n, int cl, int nf, const CFac& f) {
  if (cp_bytes(n, cl, 16) > (size_t)225 * 1024) return 1L << 60;
  return dtime(f, cdiv(n, cl) * n, cdiv(nf * (n / 2 + 1) * cl, 152));
}
constexpr CFac cp_fac64(int n) {
  CFac best{0, {0, 0, 0, 0}};
  long tb = 1L << 61;
  for (int cl : {1, 2, 4}) {
    const CFac f = dfac(n, cdiv(n, cl) * n, cdiv(2 * (n / 2 + 1) * cl, 152));
    const long t = cp_time64(n, cl, 2, f);
    if (f.c >= 2 && t < tb) { tb = t; best = f; }
  }
  return best;
}
template <typename T, int N> constexpr CFac cp_fac() { return sizeof(T) == 4 ? cfac(N, false) : cp_fac64(N); }
template <typename T, int N, int CL> struct CP {
  static constexpr CFac F = cp_fac<T, N>();
  static constexpr int NP = F.c, F0 = F.r[0], F1 = F.r[1], F2 = NP == 3 ? F.r[2] : 1;
  static constexpr int ROWS = cdiv(N, CL), P = N | 1;        // odd pitch: rows and columns free of bank conflicts
  static constexpr int CPT = CL == 1 ? P : (ROWS | 1);       // column buffer pitch
  static constexpr int NH = N / 2 + 1;
  static constexpr size_t BYTES = cp_bytes(N, CL, sizeof(cplx<T>));
  // FP64: blocks of a plane that share an SM (two fields, and what its memory takes)
  static constexpr int SHARE = sizeof(T) == 4 ? 1 : least(cdiv(2 * NH * CL, 152), (int)((size_t)227 * 1024 / (BYTES + 1024)));
  // radix 16 takes more than the 64 registers of a 1024-thread block; blocks that
  // share an SM in FP64 take at most 288 threads, so that their registers do not keep
  // them apart (108^3: 279 us with 256, 382 with 512)
  static constexpr int NT = fit_threads(ROWS * (N / F0), sizeof(T) == 4 && F0 < 16 ? 1024 : SHARE > 1 ? 288 : 512, 128);
  static constexpr int MIN_BLOCKS = SHARE > 1 ? least(SHARE, 512 / NT) : 1;
};

// One in-place butterfly with its twiddles (ip_stage's arithmetic).
template <typename T, int N, int R, int DIR, int LSUB>
__device__ __forceinline__ void cp_bfly(cplx<T> (&v)[R], int j, const cplx<T>* __restrict__ tw) {
  constexpr int m = LSUB / R, tstep = N / LSUB;
  if constexpr (DIR > 0 && m > 1) {
#pragma unroll
    for (int r = 1; r < R; ++r) {
      cplx<T> w = tw[j * r * tstep];
      w.y = -w.y;
      v[r] = cmul(v[r], w);
    }
  }
  Codelet<cplx<T>, R, DIR>::run(v);
  if constexpr (DIR < 0 && m > 1) {
#pragma unroll
    for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tw[j * r * tstep]);
  }
}

// A stage along the rows held by the block, in shared memory.
template <typename T, int N, int CL, int R, int DIR, int LSUB>
__device__ __forceinline__ void cp_rows(cplx<T>* a, int nr, const cplx<T>* __restrict__ tw) {
  using Q = CP<T, N, CL>;
  constexpr int m = LSUB / R, PER = N / R;
  for (int it = threadIdx.x; it < Q::ROWS * PER; it += Q::NT) {
    int ln, t;
    if constexpr (m >= 16) { ln = it / PER; t = it - ln * PER; }
    else { t = it / Q::ROWS; ln = it - t * Q::ROWS; }
    if (ln >= nr) continue;
    const int b = t / m, j = t - b * m;
    cplx<T>* x = a + ln * Q::P + b * LSUB + j;
    cplx<T> v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = x[r * m];
    cp_bfly<T, N, R, DIR, LSUB>(v, j, tw);
#pragma unroll
    for (int r = 0; r < R; ++r) x[r * m] = v[r];
  }
  __syncthreads();
}
// A stage along the block's columns, in the column buffer.
template <typename T, int N, int CL, int R, int DIR, int LSUB>
__device__ __forceinline__ void cp_cols(cplx<T>* b0, int nc, const cplx<T>* __restrict__ tw) {
  using Q = CP<T, N, CL>;
  constexpr int m = LSUB / R, PER = N / R;
  for (int it = threadIdx.x; it < Q::ROWS * PER; it += Q::NT) {
    const int t = it / Q::ROWS, col = it - t * Q::ROWS;
    if (col >= nc) continue;
    const int b = t / m, j = t - b * m;
    cplx<T>* x = b0 + (b * LSUB + j) * Q::CPT + col;
    cplx<T> v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = x[r * m * Q::CPT];
    cp_bfly<T, N, R, DIR, LSUB>(v, j, tw);
#pragma unroll
    for (int r = 0; r < R; ++r) x[r * m * Q::CPT] = v[r];
  }
  __syncthreads();
}

template <typename T, int N, int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(CP<T, N, CL>::NT, CP<T, N, CL>::MIN_BLOCKS)
k_plane_c(Spectra<T> sp, GArgs<T> g, const cplx<T>* __restrict__ tw_g) {
  namespace cg = cooperative_groups;
  using Q = CP<T, N, CL>;
  using C = cplx<T>;
  constexpr int F0 = Q::F0, F1 = Q::F1, F2 = Q::F2, P = Q::P, NN = N * N, M0 = N / F0;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* a = reinterpret_cast<C*>(smem_raw);
  C* bc = CL == 1 ? a : a + Q::ROWS * P;
  C* tw = (CL == 1 ? a + Q::ROWS * P : bc + N * Q::CPT);
  const int c = CL == 1 ? 0 : (int)(blockIdx.x % CL);
  const int kz = blockIdx.x / CL;
  const int row0 = c * Q::ROWS;                          // first row, and first column, of this block
  const int nr = min(Q::ROWS, N - row0);
  const int fid = blockIdx.y == 0 ? sp.idx[0] : blockIdx.y == 1 ? sp.idx[1] : sp.idx[2];
  C* gpl = CField<T>::pick(sp, fid) + (size_t)kz * NN + (size_t)row0 * N;
  for (int q = threadIdx.x; q < N; q += Q::NT) tw[q] = tw_g[q];
  __syncthreads();
  dependency_wait();
  // along ky: stage 0 from memory
  for (int it = threadIdx.x; it < Q::ROWS * M0; it += Q::NT) {
    const int ln = it / M0, j = it - ln * M0;
    if (ln >= nr) continue;
    const C* x = gpl + ln * N + j;
    C v[F0];
#pragma unroll
    for (int r = 0; r < F0; ++r) v[r] = __ldcg(x + r * M0);
    cp_bfly<T, N, F0, -1, N>(v, j, tw);
    C* y = a + ln * P + j;
#pragma unroll
    for (int r = 0; r < F0; ++r) y[r * M0] = v[r];
  }
  __syncthreads();
  cp_rows<T, N, CL, F1, -1, M0>(a, nr, tw);
  if constexpr (Q::NP == 3) cp_rows<T, N, CL, F2, -1, F2>(a, nr, tw);
  // along kx
  if constexpr (CL == 1) {
    cp_cols<T, N, CL, F0, -1, N>(a, N, tw);
  } else {
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    for (int it = threadIdx.x; it < Q::ROWS * M0; it += Q::NT) {
      const int j = it / Q::ROWS, col = it - j * Q::ROWS;
      if (col >= nr) continue;
      C v[F0];
#pragma unroll
      for (int r = 0; r < F0; ++r) {
        const int row = j + r * M0, o = row / Q::ROWS;
        v[r] = cl.map_shared_rank(a, o)[(row - o * Q::ROWS) * P + row0 + col];
      }
      cp_bfly<T, N, F0, -1, N>(v, j, tw);
      C* y = bc + j * Q::CPT + col;
#pragma unroll
      for (int r = 0; r < F0; ++r) y[r * M0 * Q::CPT] = v[r];
    }
    __syncthreads();
  }
  if constexpr (Q::NP == 3) cp_cols<T, N, CL, F1, -1, M0>(bc, nr, tw);
  // last forward stage, G-space terms, first inverse stage, in registers
  constexpr int RL = Q::NP == 3 ? F2 : F1;               // position b RL + r
  const T tp2 = g.tp2, invN = g.invN, Om = g.Om, halfOm = g.halfOm, g2cut = g.g2cut_loc;
  const bool with_loc = fid == 0 && g.vloc != nullptr;
  const T w = (kz == 0 || 2 * kz == N) ? (T)1 : (T)2;
  const C* vpl = with_loc ? g.vloc + (size_t)kz * NN : nullptr;
  // frequency at a position of the in-place transforms
  auto freq = [](int p) {
    const int k0 = p / M0, rest = p - k0 * M0;
    if constexpr (Q::NP == 2) return k0 + F0 * rest;
    else { const int k1 = rest / F2; return k0 + F0 * k1 + F0 * F1 * (rest - k1 * F2); }
  };
  auto sgn = [](int k) { return k <= (N - 1) / 2 ? k : k - N; };
  AccShort<T> e0, e1;                                    // (E_H, E_loc) or (E_NL, E_vW), before the factors
  for (int it = threadIdx.x; it < Q::ROWS * (N / RL); it += Q::NT) {
    const int b = it / Q::ROWS, col = it - b * Q::ROWS;
    if (col >= nr) continue;
    C* x = bc + b * RL * Q::CPT + col;
    C v[RL];
#pragma unroll
    for (int r = 0; r < RL; ++r) v[r] = x[r * Q::CPT];
    Codelet<C, RL, -1>::run(v);
    if (g.forward) {
      // (every block of the cluster has read its rows: they can be overwritten)
      C* y = CField<T>::pick(sp, fid) + (size_t)kz * NN + b * RL * N + row0 + col;
#pragma unroll
      for (int r = 0; r < RL; ++r) y[r * N] = v[r];
      continue;
    }
    const int py = row0 + col, my = sgn(freq(py));
    const int mk2 = my * my + kz * kz;
    const int kx0 = freq(b * RL);
    constexpr int KS = N / RL;                           // frequency step of the last stage
#pragma unroll
    for (int r = 0; r < RL; ++r) {
      const int mx = sgn(kx0 + KS * r);
      const int m2 = mx * mx + mk2;
      const T vr = v[r].x * invN, vi = v[r].y * invN;    // f~(G)
      const T a2 = vr * vr + vi * vi;
      if (fid == 0) {
        T orr = 0, oi = 0;
        if (g.hartree && m2 > 0) {
          const T cc = __ldg(g.cou + m2);                // 4 pi / G^2
          e0.add(cc * a2);
          orr = cc * vr; oi = cc * vi;
        }
        if (with_loc && tp2 * (T)m2 <= g2cut) {          // zero beyond the cutoff
          const C vl = __ldg(vpl + (b * RL + r) * N + py);
          e1.add(vr * vl.x + vi * vl.y);
          orr += vl.x; oi += vl.y;
        }
        v[r] = mk<T>(orr, oi);
      } else if (fid == 1) {
        const T k = __ldg(g.K + m2);
        e0.add(k * a2);
        v[r] = mk<T>(k * vr, k * vi);
      } else if (g.prec != nullptr) {
        const T pg = __ldg(g.prec + m2);
        v[r] = mk<T>(pg * vr, pg * vi);
      } else {
        const T G2 = tp2 * (T)m2;
        e1.add(G2 * a2);
        if (sp.merged) {
          const T k = __ldg(g.K + m2);
          e0.add(k * a2);
          const T cc = k + (T)0.5 * G2;
          v[r] = mk<T>(cc * vr, cc * vi);
        } else {
          v[r] = mk<T>(G2 * vr, G2 * vi);
        }
      }
    }
    Codelet<C, RL, +1>::run(v);
#pragma unroll
    for (int r = 0; r < RL; ++r) x[r * Q::CPT] = v[r];
  }
  if (g.forward) {
    if constexpr (CL > 1) cg::this_cluster().sync();     // other blocks may still read this one's rows
    return;
  }
  __syncthreads();
  // inverse along kx
  if constexpr (Q::NP == 3) cp_cols<T, N, CL, F1, 1, M0>(bc, nr, tw);
  if constexpr (CL == 1) {
    cp_cols<T, N, CL, F0, 1, N>(a, N, tw);
  } else {
    cg::cluster_group cl = cg::this_cluster();
    for (int it = threadIdx.x; it < Q::ROWS * M0; it += Q::NT) {
      const int j = it / Q::ROWS, col = it - j * Q::ROWS;
      if (col >= nr) continue;
      const C* y = bc + j * Q::CPT + col;
      C v[F0];
#pragma unroll
      for (int r = 0; r < F0; ++r) v[r] = y[r * M0 * Q::CPT];
      cp_bfly<T, N, F0, 1, N>(v, j, tw);
#pragma unroll
      for (int r = 0; r < F0; ++r) {
        const int row = j + r * M0, o = row / Q::ROWS;
        cl.map_shared_rank(a, o)[(row - o * Q::ROWS) * P + row0 + col] = v[r];
      }
    }
    cl.sync();                                           // (no remote access after this)
  }
  // inverse along ky: the last stage to memory
  if constexpr (Q::NP == 3) cp_rows<T, N, CL, F2, 1, F2>(a, nr, tw);
  cp_rows<T, N, CL, F1, 1, M0>(a, nr, tw);
  for (int it = threadIdx.x; it < Q::ROWS * M0; it += Q::NT) {
    const int ln = it / M0, j = it - ln * M0;
    if (ln >= nr) continue;
    const C* y = a + ln * P + j;
    C v[F0];
#pragma unroll
    for (int r = 0; r < F0; ++r) v[r] = y[r * M0];
    cp_bfly<T, N, F0, 1, N>(v, j, tw);
    C* x = gpl + ln * N + j;
#pragma unroll
    for (int r = 0; r < F0; ++r) x[r * M0] = v[r];
  }
  if (g.prec != nullptr) return;                         // (the whole grid alike: no sums)
  using V = typename TreeVal<T>::type;
  AccShort<T> acc[4];
  if (fid == 0) { acc[0].s = w * halfOm * e0.s; acc[1].s = w * Om * e1.s; }
  else { acc[2].s = w * Om * e0.s; acc[3].s = w * halfOm * e1.s; }
  V v8[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v8[q] = q < 4 ? short_val<T>(acc[q]) : V{};
  const size_t bi = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
  block_sum8(v8, reinterpret_cast<V*>(smem_raw), g.partials + bi * 4, 4);
}

// ---------------------------------------------------------------------------
// The kernels of one grid size: function pointers and launch shapes, or
// nothing when n has none (see cpass_kernels).
template <typename T> struct CPass {
  using ZF = void (*)(ProArgs<T>, Spectra<T>, const cplx<T>*, const cplx<T>*);
  using ZI = void (*)(Spectra<T>, EpiArgs<T>, const cplx<T>*, const cplx<T>*);
  using PL = void (*)(Spectra<T>, GArgs<T>, const cplx<T>*);
  int n, rows, zthreads, zgrid;
  CFac fz, fp;
  ZF zfwd; ZI zinv[4];                  // zinv by KIND
  size_t zf_bytes[4], zi_bytes[4];      // by number of fields
  // the plane pass with one field, and with more
  struct { PL kern; int cl, threads; size_t bytes; } pl[2];
};

// Cluster size for nf fields.  FP32 (bound by latency and barriers): clusters
// only where they fit about one wave of the 152 SMs (75^3, 76 planes: 17.9 ->
// 13.8 us with 2; 108^3, 110 planes: 22.0 -> 30 us with 4, since the remote rows
// cost more than the shorter stages save), or where single blocks need a second
// wave (160^3, 162 planes: 93 -> 64 us with 5).  Above 160 a plane takes several
// blocks: 4 up to 200 (200^3: 147 us, 165 with 5), then 5 (216^3: 207, 213 with 4;
// 240^3: 296, 379 with 8); the tiled chain took 264 us at 200^3, 332 at 216^3.  FP64: the
// least dtime of 1, 2 and 4 (two fields, before the radices were chosen with it: 96^3
// 277 us with 1, 224 with 4; 45^3 69 with 1, 43 with 2, 36 to 46 with 3 to 8).
template <typename T, int N> constexpr int cp_cluster(int nf) {
  const int planes = nf * (N / 2 + 1);
  if (sizeof(T) == 4)
    return planes * 4 <= 168 ? 4 : planes * 2 <= 168 ? 2 : planes <= 152 && N <= 160 ? 1 : N > 160 && N <= 200 ? 4 : 5;
  int best = 1;
  for (int cl : {2, 4})
    if (cp_time64(N, cl, nf, cp_fac64(N)) < cp_time64(N, best, nf, cp_fac64(N))) best = cl;
  return cp_bytes(N, best, 16) <= (size_t)225 * 1024 ? best : 0;
}

template <typename T, int N> CPass<T> make_cpass() {
  using Z = CZ<N, sizeof(T) == 8>;
  CPass<T> p{};
  p.n = N; p.rows = Z::R; p.zthreads = Z::NT; p.zgrid = Z::GRID;
  p.fz = Z::F; p.fp = cp_fac<T, N>();
  p.zfwd = k_zfwd_c<T, N>;
  p.zinv[0] = k_zinv_c<T, N, 0>; p.zinv[1] = k_zinv_c<T, N, 1>;
  p.zinv[2] = k_zinv_c<T, N, 2>; p.zinv[3] = k_zinv_c<T, N, 3>;
  for (int f = 0; f < 4; ++f) { p.zf_bytes[f] = czfwd_bytes<T, N>(f); p.zi_bytes[f] = czinv_bytes<T, N>(f); }
  constexpr int c1 = cp_cluster<T, N>(1), c2 = cp_cluster<T, N>(2);
  if constexpr (c1 > 0) { p.pl[0].kern = k_plane_c<T, N, c1>; p.pl[0].cl = c1; p.pl[0].threads = CP<T, N, c1>::NT; p.pl[0].bytes = CP<T, N, c1>::BYTES; }
  if constexpr (c2 > 0) { p.pl[1].kern = k_plane_c<T, N, c2>; p.pl[1].cl = c2; p.pl[1].threads = CP<T, N, c2>::NT; p.pl[1].bytes = CP<T, N, c2>::BYTES; }
  return p;
}

// nullptr when the grid has no compile-time passes
template <typename T> const CPass<T>* cpass_kernels(int n);

}  // namespace ofdft
