// Slab kernel for any tube length n3: one CTA per mode-1 index i1, the mode-3
// transforms as register-tiled products with the DFT matrix of Eq. (bar BA-k) /
// Eq. (barAAk), folded by its symmetries.
//
// Folding.  With theta = 2 pi / n3 and c, s = cos, sin(theta k l):
//   inverse  x_l, x_{n3-l} = C -+ D,  C = sum_k Re X_k c,  D = sum_k Im X_k s,
//   forward  X_k = (sum_l e_l c, -sum_l o_l s),  e, o_l = x_l +- x_{n3-l},
// so a pair of rows (l, n3 - l) costs one product with (c, s).  For even
// n3 = 2M the rows M - l, M + l have the same products up to the parity of k
// (c -> (-1)^k c, s -> -(-1)^k s): the inverse keeps one sum over the even and
// one over the odd slices and gets four rows from them, and the forward folds
// the four rows into one pair for the even and one for the odd slices.  Per
// tube and direction n3^2/2 multiply-adds (odd n3) or n3^2/4 (even) in place of
// n3^2, and the sums are half as long.
//
// Pairs.  A value (re, im), a coefficient (c, s) and an accumulator (C, D) are
// pairs, so FP32 uses the packed fma.rn.f32x2 with no shuffling.  The slab is
// kept as pairs too: slot p of a tube holds (x_p, x_{n3-p}) (slot 0: x_0 and,
// for even n3, x_{n3/2}), laid out [slot][tube] with an odd number of tubes per
// slot: the transforms read 32 consecutive tubes of a slot and the W-step 32
// consecutive rows of a tube, both without bank conflicts.
//
// Tiles.  An SM returns 128 bytes a clock from shared memory, so a pair that a
// lane reads has to feed several products: a lane computes TL rows (inverse, one
// parity of slices at a time) or slices (forward) of four tubes, 8 (TL + 4) bytes
// for 4 TL products; two groups of 16 lanes take neighbouring TL columns of 64
// tubes (FP64: 32 lanes, one tube each).  tc_init times TL = 2 and 4 (a larger
// tile has fewer loads per product, a smaller one fills the warps of small slabs).
// The even and odd sums of a row pair are parked in the slab and unfolded in a
// pass of their own, which also places G.
//
// Staging.  The coefficients of one direction, and the spectrum of as many 64-tube
// groups as fit (all of them for most sizes) are copied to shared memory by
// cp.async, so the transforms read nothing but shared memory: with the
// spectrum and the coefficients read through L1 and G inside the item's
// epilogue the inverse took 72K cycles of a 925 x 153 x 92 CTA against 28K for
// the forward one.  Sizes whose slab leaves no room for a stage take the
// unstaged form (STAGED = false).
//
// The modes are those of k_slab.
#pragma once

namespace tc {

// Threads per CTA: kSlabGThreads where one CTA fills an SM, kSlabGHalf where two
// slabs fit.  FP32: 32 warps of 64 registers on an SM either way (16 of 128
// before: the kernel waits on shared memory and barriers, issue active 38%;
// 925 x 153 x 92: 162 -> 150 us).  FP64 values take two registers each.
template <typename T>
constexpr int kSlabGThreads = sizeof(T) == 8 ? 256 : 1024;
template <typename T>
constexpr int kSlabGHalf = sizeof(T) == 8 ? 256 : 512;
// A warp's item: kLW lanes side by side along the tubes with kTT tubes each (kLW
// apart), and 32 / kLW groups of lanes with TL columns of the product each.  FP64
// takes one tube per lane: no product is worth a half-empty warp there.
template <typename T>
constexpr int kLW = sizeof(T) == 8 ? 32 : 16;
template <typename T>
constexpr int kTT = sizeof(T) == 8 ? 1 : 4;
template <typename T>
constexpr int kLG = 32 / kLW<T>;
template <typename T>
constexpr int kGTubes = kLW<T> * kTT<T>;  // tubes of an item
constexpr int kFoldPad = 16;              // columns of the tables, padded: a multiple of kLG TL
constexpr int kSlabGMaxN3 = 512;      // the tables grow as n3^2

// Pairs of T with packed arithmetic.
template <typename T>
struct Pk;
template <>
struct Pk<float> {
  typedef unsigned long long V;
  __device__ __forceinline__ static V mk(float a, float b) {
    V v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
    return v;
  }
  __device__ __forceinline__ static cx<float> un(V v) {
    cx<float> r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.re), "=f"(r.im) : "l"(v));
    return r;
  }
  __device__ __forceinline__ static V ldg(const cx<float>* p) {
    return __ldg(reinterpret_cast<const unsigned long long*>(p));
  }
  __device__ __forceinline__ static V lds(const cx<float>* p) { return *reinterpret_cast<const unsigned long long*>(p); }
  // two consecutive coefficients (16-byte aligned), from shared or global memory
  template <bool SH>
  __device__ __forceinline__ static void ld2(const cx<float>* p, V& a, V& b) {
    const ulonglong2 v = SH ? *reinterpret_cast<const ulonglong2*>(p) : __ldg(reinterpret_cast<const ulonglong2*>(p));
    a = v.x;
    b = v.y;
  }
  __device__ __forceinline__ static void fma(V& a, V x, V y) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a) : "l"(x), "l"(y));
  }
  __device__ __forceinline__ static V add(V x, V y) {
    V v;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(x), "l"(y));
    return v;
  }
};
template <>
struct Pk<double> {
  typedef cx<double> V;
  __device__ __forceinline__ static V mk(double a, double b) { return V{a, b}; }
  __device__ __forceinline__ static cx<double> un(V v) { return v; }
  __device__ __forceinline__ static V ldg(const cx<double>* p) { return ldg_cx(p); }
  __device__ __forceinline__ static V lds(const cx<double>* p) { return *p; }
  template <bool SH>
  __device__ __forceinline__ static void ld2(const cx<double>* p, V& a, V& b) {
    a = SH ? p[0] : ldg_cx(p);
    b = SH ? p[1] : ldg_cx(p + 1);
  }
  __device__ __forceinline__ static void fma(V& a, V x, V y) {
    a.re = ::fma(x.re, y.re, a.re);
    a.im = ::fma(x.im, y.im, a.im);
  }
  __device__ __forceinline__ static V add(V x, V y) { return x + y; }
};

// Sizes of the folded transform of length n3.
struct FoldDims {
  int even, M, h;      // n3 = 2M, or n3 = 2h + 1
  int np;              // pair slots of a tube
  int nl, nlp;         // rows l of the inverse (the others follow), padded
  int kmax;            // slices 1 .. kmax of the inverse loop
  int nke, nkep, nkt;  // even slices (all slices for odd n3), padded; columns of the forward table
  int lmax;            // rows 1 .. lmax of the forward loop
};
__host__ __device__ inline FoldDims fold_dims(int n3) {
  FoldDims f{};
  auto pad = [](int n) { return (n + kFoldPad - 1) / kFoldPad * kFoldPad; };
  f.even = (n3 % 2) == 0;
  f.M = n3 / 2;
  f.h = (n3 - 1) / 2;
  f.np = (n3 + 1) / 2;
  f.nl = f.even ? f.M / 2 + 1 : f.h + 1;
  f.nlp = pad(f.nl);
  f.kmax = f.even ? f.M - 1 : f.h;
  f.nke = f.even ? f.M / 2 + 1 : f.h + 1;
  f.nkep = pad(f.nke);
  f.nkt = f.even ? f.nkep + pad((f.M + 1) / 2) : f.nkep;
  f.lmax = f.even ? (f.M - 1) / 2 : f.h;
  return f;
}
// Complex entries of the two tables: inverse [kmax + 1][nlp], forward [lmax + 1][nkt].
__host__ __device__ inline size_t fold_table_entries(int n3) {
  const FoldDims f = fold_dims(n3);
  return (size_t)(f.kmax + 1) * f.nlp + (size_t)(f.lmax + 1) * f.nkt;
}
// Slice of column q of the forward table (even slices first for even n3), or
// one past the last slice for padding.
__host__ __device__ inline int fold_slice(const FoldDims& f, int n3, int q) {
  int k;
  if (!f.even) k = q;
  else if (q < f.nkep) k = (q < f.nke) ? 2 * q : n3;
  else k = 2 * (q - f.nkep) + 1;
  const int S = n3 / 2 + 1;
  return k < S ? k : S;
}

// The tables, from twg[m] = exp(-2 pi i m / n3) (FP64 cos and sin rounded to T).
template <typename T>
__global__ void k_fold_tables(cx<T>* __restrict__ tab, const cx<T>* __restrict__ twg, int n3) {
  const FoldDims f = fold_dims(n3);
  const size_t ni = (size_t)(f.kmax + 1) * f.nlp, tot = fold_table_entries(n3);
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < tot; e += (size_t)gridDim.x * blockDim.x) {
    int k, l;
    bool live;
    if (e < ni) {
      k = (int)(e / f.nlp);
      l = (int)(e % f.nlp);
      live = l < f.nl;
    } else {
      const size_t o = e - ni;
      l = (int)(o / f.nkt);
      k = fold_slice(f, n3, (int)(o % f.nkt));
      live = k < n3 / 2 + 1;
    }
    cx<T> v = {T(0), T(0)};
    if (live) {
      const cx<T> w = twg[((long long)k * l) % n3];
      v = cx<T>{w.re, -w.im};
    }
    tab[e] = v;
  }
}

struct SlabGLayout {
  size_t wtab, red, msk, tab, pairs, stage, total;
};
// Tubes per slot of the slab: odd, so that consecutive slots start in other banks.
__host__ __device__ inline int slab_g_stride(int n2) { return n2 | 1; }
// Row pitch of a stage of sg groups (whole groups: the lanes past n2 read what is
// there and store nothing).
template <typename T>
__host__ __device__ inline int slab_g_width(int sg) { return sg * kGTubes<T>; }
// sg: 64-tube groups per stage (0: unstaged).
template <typename T>
__host__ __device__ inline SlabGLayout slab_g_layout(int n2, int n3, int sg) {
  SlabGLayout L{};
  const FoldDims f = fold_dims(n3);
  size_t off = 0;
  L.wtab = off;
  off = align_up(off + sizeof(T) * 6 * (size_t)n2, 16);
  L.red = off;
  off = align_up(off + sizeof(double) * 2 * 32, 16);
  L.msk = off;
  off = align_up(off + sizeof(uint32_t) * (size_t)n3 * ((n2 + 31) / 32), 16);
  L.tab = off;
  if (sg > 0) {
    const size_t ni = (size_t)(f.kmax + 1) * f.nlp, nf = (size_t)(f.lmax + 1) * f.nkt;
    off = align_up(off + sizeof(cx<T>) * (ni > nf ? ni : nf), 16);
  }
  L.pairs = off;
  // (the last slot's lanes past n2 read up to a group further)
  off = align_up(off + sizeof(cx<T>) * ((size_t)((n3 + 1) / 2) * slab_g_stride(n2) + kGTubes<T>), 16);
  L.stage = off;
  off = align_up(off + sizeof(cx<T>) * (size_t)(n3 / 2 + 1) * slab_g_width<T>(sg), 16);
  L.total = off;
  return L;
}

// Launch shape of the folded-transform slab kernels: two CTAs of kSlabGHalf threads on
// an SM where the slab, the coefficients and a stage of one group fit half of
// its shared memory, else one with twice the threads; as many groups per stage
// as fit; unstaged where even one does not.  False where the slab itself does
// not fit (k_slab keeps it in global memory).
struct SlabGPlan {
  int threads, sg;
  size_t smem;
};
template <typename T>
inline bool slab_g_plan(int n2, int n3, int optin, SlabGPlan& pl) {
  // (the W-step has a thread per segment of a row)
  if (n3 > kSlabGMaxN3 || (n2 + kWSeg<T> - 1) / kWSeg<T> > 256) return false;
  const int ngr = (n2 + kGTubes<T> - 1) / kGTubes<T>;
  const size_t half = (size_t)(optin + kStaticSmemReserve + 1024) / 2 - 1024;  // 1 KB per CTA is the system's
  for (int pass = 0; pass < 2; ++pass) {
    const size_t room = pass == 0 ? half : (size_t)optin;
    for (int sg = ngr; sg >= 1; --sg) {
      const size_t b = slab_g_layout<T>(n2, n3, sg).total;
      if (b <= room) {
        pl = SlabGPlan{pass == 0 ? kSlabGHalf<T> : kSlabGThreads<T>, sg, b};
        return true;
      }
    }
  }
  pl = SlabGPlan{kSlabGThreads<T>, 0, slab_g_layout<T>(n2, n3, 0).total};
  return pl.smem <= (size_t)optin;
}

// Items of the inverse transform per group of kGTubes tubes with TL = 4 columns a lane.
template <typename T>
inline int fold_items(int n3) {
  const FoldDims f = fold_dims(n3);
  return (f.even ? 2 : 1) * ((f.nl + 4 * kLG<T> - 1) / (4 * kLG<T>));
}
// Tile where none is timed: TL = 2, twice the items, where the CTA has a warp for each
// of them (us per iteration of tc_complete_static, TL = 4 and 2: 16 x 48 x 9 FP64 53.0, 50.9,
// 30 x 90 x 9 FP32 44.3, 42.8; with more items than warps 60 x 90 x 14 FP64 77.4, 79.9).
template <typename T>
inline int fold_tile(int n2, int n3, int threads) {
  return 64 * fold_items<T>(n3) * ((n2 + kGTubes<T> - 1) / kGTubes<T>) <= threads ? 2 : 4;
}
// Whether tc_init times the tiles.  In FP64 the pipe is the bound at either, so where
// one item at TL = 4 is the whole transform of its tubes (odd n3 up to 7) TL = 2
// spreads it over more lanes' warps and there is nothing to choose.
template <typename T>
inline bool fold_timed(int n3) {
  return sizeof(T) == 4 || fold_items<T>(n3) > 1;
}

// Row l of the q-th row in slab order (slot by slot), 0 <= q < n3, and the
// position of row l in the slab, in units of T.
__device__ __forceinline__ int slab_g_row(bool even, int n3, int q) {
  if (even) {
    const int p = q >> 1;
    return (q & 1) ? (p == 0 ? n3 >> 1 : n3 - p) : p;
  }
  if (q == 0) return 0;
  const int p = (q + 1) >> 1;
  return (q & 1) ? p : n3 - p;
}
__device__ __forceinline__ int slab_g_off(bool even, int n3, int l, int np2) {
  const int m = n3 >> 1;
  if (even && l == m) return 1;
  return (l <= m) ? 2 * np2 * l : 2 * np2 * (n3 - l) + 1;
}

// acc[i][j] += sum over n rows of x(tube j) * tab[i]: the pair matrix and the
// table advance by dx and dc pairs per row, tube j is kLW j pairs on.  (Running
// pointers and one base per operand: with a clamped pointer per tube and indexed
// rows the loop had ten integer instructions to its sixteen products.)
template <typename T, int TL, bool SH>
__device__ __forceinline__ void fold_product(typename Pk<T>::V (&acc)[TL][kTT<T>], const cx<T>* __restrict__ tab, int dc,
                                             const cx<T>* __restrict__ x, int dx, int n) {
  using P = Pk<T>;
  using V = typename P::V;
#pragma unroll 2
  for (int q = 0; q < n; ++q, x += dx, tab += dc) {
    V v[kTT<T>];
#pragma unroll
    for (int j = 0; j < kTT<T>; ++j) v[j] = P::lds(x + kLW<T> * j);
#pragma unroll
    for (int i = 0; i < TL; i += 2) {
      V c0, c1;
      P::template ld2<SH>(tab + i, c0, c1);
#pragma unroll
      for (int j = 0; j < kTT<T>; ++j) {
        P::fma(acc[i][j], v[j], c0);
        P::fma(acc[i + 1][j], v[j], c1);
      }
    }
  }
}

// One item of the inverse transform: the sums (C, D) over the slices of parity
// par (all slices for odd n3) at rows l0 .. l0 + TL - 1, slices 0 and n3/2 with
// weight 1/2.
// x: the lane's first tube in the staged spectrum [k][ldx].
template <typename T, int TL, bool EVEN>
__device__ __forceinline__ void fold_inverse(const FoldDims& f, const cx<T>* __restrict__ tab, int l0, int par,
                                             const cx<T>* __restrict__ x, int ldx,
                                             typename Pk<T>::V (&acc)[TL][kTT<T>]) {
  using P = Pk<T>;
#pragma unroll
  for (int j = 0; j < kTT<T>; ++j) {
    const T x0 = (!EVEN || par == 0) ? T(0.5) * x[kLW<T> * j].re : T(0);
    const T xm = (EVEN && (f.M & 1) == par) ? T(0.5) * x[f.M * ldx + kLW<T> * j].re : T(0);
#pragma unroll
    for (int i = 0; i < TL; ++i) acc[i][j] = P::mk(((l0 + i) & 1) ? x0 - xm : x0 + xm, T(0));
  }
  const int k0 = EVEN ? 2 - par : 1, step = EVEN ? 2 : 1;
  fold_product<T, TL, true>(acc, tab + l0 + k0 * f.nlp, step * f.nlp, x + k0 * ldx, step * ldx,
                            (f.kmax - k0 + step) / step);
}
// The same from the stored spectrum in global memory (tube j of the lane at z[j],
// rows n2 apart, plus r[j] where ADD) and the tables there.
template <typename T, int TL, bool EVEN, bool ADD>
__device__ __forceinline__ void fold_inverse_global(const FoldDims& f, const cx<T>* __restrict__ tab, int l0, int par,
                                                    const cx<T>* const (&z)[kTT<T>], const cx<T>* const (&r)[kTT<T>],
                                                    int n2, typename Pk<T>::V (&acc)[TL][kTT<T>]) {
  using P = Pk<T>;
  using V = typename P::V;
  auto load = [&](int k, int j) -> V {
    const size_t o = (size_t)k * n2;
    return ADD ? P::add(P::ldg(z[j] + o), P::ldg(r[j] + o)) : P::ldg(z[j] + o);
  };
#pragma unroll
  for (int j = 0; j < kTT<T>; ++j) {
    const T x0 = (!EVEN || par == 0) ? T(0.5) * P::un(load(0, j)).re : T(0);
    const T xm = (EVEN && (f.M & 1) == par) ? T(0.5) * P::un(load(f.M, j)).re : T(0);
#pragma unroll
    for (int i = 0; i < TL; ++i) acc[i][j] = P::mk(((l0 + i) & 1) ? x0 - xm : x0 + xm, T(0));
  }
#pragma unroll 2
  for (int k = EVEN ? 2 - par : 1; k <= f.kmax; k += EVEN ? 2 : 1) {
    V x[kTT<T>];
#pragma unroll
    for (int j = 0; j < kTT<T>; ++j) x[j] = load(k, j);
#pragma unroll
    for (int i = 0; i < TL; i += 2) {
      V c0, c1;
      P::template ld2<false>(tab + l0 + k * f.nlp + i, c0, c1);
#pragma unroll
      for (int j = 0; j < kTT<T>; ++j) {
        P::fma(acc[i][j], x[j], c0);
        P::fma(acc[i + 1][j], x[j], c1);
      }
    }
  }
}

// Where the sums of row l and parity par go in the slab until all are there: the
// even slices' to slot l, the odd ones' to slot M - l; rows 0 and M/2, whose
// sums have one component each, share a slot.
// (live: one bit per tube of the lane)
template <typename T, bool EVEN>
__device__ __forceinline__ void fold_park(const FoldDims& f, cx<T>* col, int np2, int l, int par, uint32_t live,
                                          const typename Pk<T>::V (&v)[kTT<T>]) {
  if (EVEN && (l == 0 || 2 * l == f.M)) {
    T* at = reinterpret_cast<T*>(col + l * np2) + par;
    const bool re = par == 0 || l == 0;
#pragma unroll
    for (int j = 0; j < kTT<T>; ++j) {
      const cx<T> a = Pk<T>::un(v[j]);
      if ((live >> j) & 1u) at[2 * kLW<T> * j] = re ? a.re : a.im;
    }
  } else {
    cx<T>* at = col + (EVEN && par ? f.M - l : l) * np2;
#pragma unroll
    for (int j = 0; j < kTT<T>; ++j)
      if ((live >> j) & 1u) at[kLW<T> * j] = Pk<T>::un(v[j]);
  }
}

// One item of the forward transform: columns q0 .. q0 + TL - 1 of the forward
// table (slices of one parity for even n3) of the item's tubes, from the folded
// slab.  acc receives (sum e c, sum o s).
template <typename T, int TL, bool EVEN, bool SH>
__device__ __forceinline__ void fold_forward(const FoldDims& f, const cx<T>* __restrict__ tab, int q0,
                                             const cx<T>* __restrict__ col, int np2,
                                             typename Pk<T>::V (&acc)[TL][kTT<T>]) {
  using P = Pk<T>;
  const bool oddk = EVEN && q0 >= f.nkep;
  const int kk0 = oddk ? q0 - f.nkep : q0;  // k = 2 (kk0 + i) + oddk for even n3
#pragma unroll
  for (int j = 0; j < kTT<T>; ++j) {
    const cx<T> s0 = col[kLW<T> * j];
    const T x0 = EVEN && oddk ? s0.im : s0.re;
    // row M/2: e cos(pi k / 2) on even slices, o sin(pi k / 2) on odd ones
    const cx<T> sm = (EVEN && (f.M & 1) == 0) ? col[(f.M / 2) * np2 + kLW<T> * j] : cx<T>{T(0), T(0)};
    const T a = oddk ? T(0) : sm.re, b = oddk ? sm.im : T(0);
#pragma unroll
    for (int i = 0; i < TL; ++i) {
      const bool neg = (kk0 + i) & 1;
      acc[i][j] = P::mk(neg ? x0 - a : x0 + a, neg ? -b : b);
    }
  }
  // slot l holds the even fold, slot M - l the odd one
  const cx<T>* x = col + (oddk ? f.M - 1 : 1) * np2;
  fold_product<T, TL, SH>(acc, tab + q0 + f.nkt, f.nkt, x, oddk ? -np2 : np2, f.lmax);
}

template <typename T, int MODE, int TL, bool EVEN, bool STAGED, bool GENERAL>
__device__ __forceinline__ void slab_g_impl(const Dev<T>& d, T* __restrict__ Wout, int flags, int init,
                                            unsigned char* smem) {
  using P = Pk<T>;
  using V = typename P::V;
  const int i1 = blockIdx.x;
  const int n1 = d.n1, n2 = d.n2, n3 = d.n3, S = n3 / 2 + 1, mw = d.mw;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  const FoldDims f = fold_dims(n3);
  const int sg = STAGED ? d.fold_sg : 0;
  const SlabGLayout lay = slab_g_layout<T>(n2, n3, sg);
  const int np2 = slab_g_stride(n2);
  T* wtab = reinterpret_cast<T*>(smem + lay.wtab);
  double* red = reinterpret_cast<double*>(smem + lay.red);
  uint32_t* msk = reinterpret_cast<uint32_t*>(smem + lay.msk);  // rows in slab order
  cx<T>* tab = reinterpret_cast<cx<T>*>(smem + lay.tab);
  cx<T>* pairs = reinterpret_cast<cx<T>*>(smem + lay.pairs);
  cx<T>* stg = reinterpret_cast<cx<T>*>(smem + lay.stage);
  T* spat = reinterpret_cast<T*>(pairs);
  const int ni = (f.kmax + 1) * f.nlp, nf = (f.lmax + 1) * f.nkt;
  const cx<T>* tabf = STAGED ? tab : d.fold + ni;
  const cx<T>* zrow = d.Zt + (size_t)i1 * S * n2;
  const cx<T>* rrow = d.Rt + (size_t)i1 * S * n2;
  const T* Gi = d.G + (size_t)i1 * n2 * n3;
  const uint32_t* Mi = d.mask + (size_t)i1 * n3 * mw;
  const bool wsolve = (MODE == MODE_ITER) && !init && d.rho2 != T(0);
  const T zfac = init ? T(0) : ((d.rho2 == T(0)) ? T(1) / (T(1) + d.mu) : T(1));
  constexpr bool NEED_G = (MODE == MODE_ITER || MODE == MODE_GRAD);

  // ---- masks, W-step table, coefficients, G into its place in the slab ---------------------
  // (rows 2 and 3 of the table are read in FP64 only; FP32 keeps the excess ratios
  // in their place)
  constexpr bool HEX_SH = GENERAL && sizeof(T) == 4;
  if (wsolve)
    for (int j = tid; j < 6 * n2; j += nt) wtab[j] = HEX_SH && j >= 2 * n2 && j < 4 * n2 ? d.wexc[j - 2 * n2] : d.winv[j];
  if (MODE != MODE_W)
    for (int e = tid; e < n3 * mw; e += nt) {
      const int q = e / mw;
      msk[e] = __ldg(Mi + (size_t)slab_g_row(EVEN, n3, q) * mw + (e - q * mw));
    }
  if (STAGED)
    for (int e = tid; e < ni; e += nt) cp_async_elem(tab + e, d.fold + e);
  if (NEED_G)  // G, wanted after the inverse transform, on its way to L2
    for (int e = 128 / (int)sizeof(T) * tid; e < n3 * n2; e += 128 / (int)sizeof(T) * nt) asm volatile("prefetch.global.L2 [%0];" ::"l"(Gi + e));

  // ---- inverse transform: the sums of every row pair, parked in the slab -------------------
  const int ngr = (n2 + kGTubes<T> - 1) / kGTubes<T>;
  const int gstage = STAGED ? sg : ngr;
  const int width = slab_g_width<T>(gstage);  // tubes of a full stage, its row stride
  constexpr int LC = kLG<T> * TL;                 // columns of a warp's item
  const int lt = lane & (kLW<T> - 1), lg = lane / kLW<T>;
  SqSum<T> gsum;
  for (int g0 = 0; g0 < ngr; g0 += gstage) {
    const int gn = min(gstage, ngr - g0);
    if (STAGED) {
      const int t0 = g0 * kGTubes<T>, tn = min(gn * kGTubes<T>, n2 - t0);
      if (g0 > 0) __syncthreads();  // the stage is read no more
      for (int k = wid; k < S; k += nw) {
        const cx<T>* zs = (MODE == MODE_R ? rrow : zrow) + (size_t)k * n2 + t0;
        const cx<T>* rs = rrow + (size_t)k * n2 + t0;
        for (int t = lane; t < tn; t += 32) {
          if (MODE == MODE_W) stg[k * width + t] = ldg_cx(zs + t) + ldg_cx(rs + t);
          else cp_async_elem(stg + k * width + t, zs + t);
        }
      }
    }
    cp_async_wait_all();
    __syncthreads();
    const int ntile = (f.nl + LC - 1) / LC, npar = EVEN ? 2 : 1;
    for (int e = wid; e < npar * ntile * gn; e += nw) {
      const int gl = e / (npar * ntile), rest = e - gl * npar * ntile, par = rest & (npar - 1);
      const int g = g0 + gl, l0 = (rest / npar) * LC + lg * TL;
      const int t0 = g * kGTubes<T> + lt;
      uint32_t live = 0;
#pragma unroll
      for (int j = 0; j < kTT<T>; ++j) live |= (uint32_t)(t0 + kLW<T> * j < n2) << j;
      V acc[TL][kTT<T>];
      if constexpr (STAGED) {
        fold_inverse<T, TL, EVEN>(f, tab, l0, par, stg + t0 - g0 * kGTubes<T>, width, acc);
      } else {
        const cx<T>* zc[kTT<T>];
        const cx<T>* rc[kTT<T>];
#pragma unroll
        for (int j = 0; j < kTT<T>; ++j) {
          const int tq = min(t0 + kLW<T> * j, n2 - 1);
          zc[j] = (MODE == MODE_R ? rrow : zrow) + tq;
          rc[j] = rrow + tq;
        }
        fold_inverse_global<T, TL, EVEN, MODE == MODE_W>(f, d.fold, l0, par, zc, rc, n2, acc);
      }
#pragma unroll
      for (int i = 0; i < TL; ++i) {
        if (l0 + i >= f.nl) break;
        fold_park<T, EVEN>(f, pairs + t0, np2, l0 + i, par, live, acc[i]);
      }
    }
  }
  __syncthreads();
  // ---- the rows from the sums; v = G on the mask, Z elsewhere (MODE_GRAD: Z - G on the
  // mask, 0 elsewhere) ------------------------------------------------------------------------
  {
    const T fac = (T(2) / T(n3)) * (MODE == MODE_ITER ? zfac : T(1));
    // (two warps share a slot, 32 tubes in turn)
    const int nun = EVEN ? f.M / 2 + 1 : f.h + 1;
    for (int e = wid; e < 2 * nun; e += nw) {
      const int l = e >> 1;
      // slots of the item and their rows: slot l = rows (l, r1), slot M - l = rows (r2, r3)
      const bool two = EVEN && l > 0 && 2 * l != f.M;
      const int r1 = EVEN ? (l == 0 ? f.M : n3 - l) : (l == 0 ? 0 : n3 - l);
      const int q0 = EVEN ? 2 * l : (l == 0 ? 0 : 2 * l - 1), q2 = two ? 2 * (f.M - l) : q0;
      const uint32_t *m0 = msk + q0 * mw, *m2 = msk + q2 * mw;
      const int first = (EVEN || l > 0) ? mw : 0;  // the second row's words
      const T *g0 = Gi + l * n2, *g1 = Gi + r1 * n2, *g2 = Gi + (two ? f.M - l : l) * n2, *g3 = Gi + (two ? f.M + l : l) * n2;
      cx<T>*c0 = pairs + l * np2, *c2 = pairs + (two ? f.M - l : l) * np2;
#pragma unroll 2
      for (int t = 32 * (e & 1) + lane; t < n2; t += 64) {
        T gv[4] = {};
        uint32_t w[4] = {};
        if (NEED_G) {
          const int blk = t >> 5;
          gv[0] = __ldg(g0 + t), gv[1] = __ldg(g1 + t);
          w[0] = m0[blk], w[1] = m0[first + blk];
          if (EVEN) {
            gv[2] = __ldg(g2 + t), gv[3] = __ldg(g3 + t);
            w[2] = m2[blk], w[3] = m2[mw + blk];
          }
        }
        T x[4];
        const cx<T> a = c0[t];
        if (EVEN) {
          const cx<T> b = c2[t];
          const T cs = a.re + b.re, ds = a.im + b.im, cd = a.re - b.re, dd = a.im - b.im;
          x[0] = two ? cs - ds : (l == 0 ? a.re + a.im : a.re - a.im);
          x[1] = two ? cs + ds : (l == 0 ? a.re - a.im : a.re + a.im);
          x[2] = cd + dd, x[3] = cd - dd;
        } else {
          x[0] = l == 0 ? a.re : a.re - a.im;
          x[1] = l == 0 ? T(0) : a.re + a.im;
          x[2] = x[3] = T(0);
        }
#pragma unroll
        for (int q = 0; q < (EVEN ? 4 : 2); ++q) {
          x[q] *= fac;
          const bool ob = (w[q] >> lane) & 1u;
          if (MODE == MODE_ITER) x[q] = ob ? gv[q] : x[q];
          if (MODE == MODE_GRAD) {
            x[q] = ob ? x[q] - gv[q] : T(0);
            if ((q < 2 && (EVEN || q == 0 || l > 0)) || two) gsum.add(x[q]);
          }
        }
        c0[t] = cx<T>{x[0], x[1]};
        if (two) c2[t] = cx<T>{x[2], x[3]};
      }
    }
  }
  __syncthreads();
  if (MODE == MODE_GRAD) {
    double g = gsum.total(), unused = 0.0;
    block_sum2(g, unused, red);
    if (sq_again<T>(g, gsum.nonzero())) {
      SqSum64 g64;
      for (int l = wid; l < n3; l += nw)
        for (int t = lane; t < n2; t += 32) g64.add(spat[slab_g_off(EVEN, n3, l, np2) + 2 * t]);
      g = g64.s;
      block_sum2(g, unused, red);
    }
    if (tid == 0) d.part[(size_t)i1 * 4] = g;
  }

  // ---- read-back modes: partial sums, optional copy of W ----------------------------------
  if (MODE == MODE_W || MODE == MODE_R) {
    const bool sums = MODE == MODE_R || !(flags & SLAB_NOSUM);
    if (MODE == MODE_W && Wout)
      for (int q = wid; q < n3; q += nw) {
        const int l = slab_g_row(EVEN, n3, q);
        const T* row = spat + slab_g_off(EVEN, n3, l, np2);
        for (int t = lane; t < n2; t += 32) {
          if (flags & SLAB_WROWS) Wout[((size_t)i1 * n3 + l) * n2 + t] = row[2 * t];
          else Wout[(size_t)i1 + (size_t)n1 * ((size_t)t + (size_t)n2 * l)] = row[2 * t];
        }
      }
    if (!sums) return;
    auto walk = [&](auto& sa, auto& sb) {
      for (int q = wid; q < n3; q += nw) {
        const T* row = spat + slab_g_off(EVEN, n3, slab_g_row(EVEN, n3, q), np2);
        for (int t = lane; t < n2; t += 32) {
          const T v = row[2 * t];
          sa.add(v);
          if (MODE == MODE_W) {
            if (t + 1 < n2) sb.add_diff(v, row[2 * (t + 1)]);
          } else {
            if ((msk[q * mw + (t >> 5)] >> lane) & 1u) sb.add(v);
          }
        }
      }
    };
    SqSum<T> sa, sb;
    walk(sa, sb);
    double a = sa.total(), b = sb.total();
    block_sum2(a, b, red);
    const bool again_a = sq_again<T>(a, sa.nonzero()), again_b = sq_again<T>(b, sb.nonzero());
    if (again_a || again_b) {
      SqSum64 a64, b64;
      walk(a64, b64);
      a = a64.s, b = b64.s;
      block_sum2(a, b, red);
    }
    if (tid == 0) {
      const int o = (MODE == MODE_W) ? 2 : 0;
      d.part[(size_t)i1 * 4 + o] = a;
      d.part[(size_t)i1 * 4 + o + 1] = b;
    }
    return;
  }
  if (STAGED && EVEN)  // the forward coefficients (odd n3: the same table)
    for (int e = tid; e < nf; e += nt) cp_async_elem(tab + e, d.fold + ni + e);

  // ---- W-step -------------------------------------------------------------------------------
  if (wsolve) {
    auto col_of = [&](int q) { return spat + slab_g_off(EVEN, n3, slab_g_row(EVEN, n3, q), np2); };
    wstep_segments<T, kWSeg<T>, GENERAL>(col_of, 2, msk, n3, n2, d.rho2, wtab, HEX_SH ? wtab + 2 * n2 : d.wexc);
  }

  // ---- fold -----------------------------------------------------------------------------------
  {
    const int nfold = EVEN ? f.M / 2 + 1 : f.h + 1;
    for (int l = wid; l < nfold; l += nw)
      for (int t = lane; t < n2; t += 32) {
        cx<T>* cp = pairs + t;
        const cx<T> a = cp[l * np2];
        if (EVEN && l > 0 && 2 * l != f.M) {
          const cx<T> b = cp[(f.M - l) * np2];
          const T ea = a.re + a.im, oa = a.re - a.im, eb = b.re + b.im, ob = b.re - b.im;
          cp[l * np2] = cx<T>{ea + eb, oa - ob};
          cp[(f.M - l) * np2] = cx<T>{ea - eb, oa + ob};
        } else if (EVEN || l > 0) {
          cp[l * np2] = cx<T>{a.re + a.im, a.re - a.im};
        }
      }
  }
  cp_async_wait_all();
  __syncthreads();

  // ---- forward transform, R~ = W~ - Z~ -----------------------------------------------------------
  const bool track = (MODE == MODE_ITER) && !init && d.dZt != nullptr;
  const bool zstaged = STAGED && gstage >= ngr;  // the whole spectrum is still staged
  double dw2 = 0.0;
  {
    const int nte = (f.nke + LC - 1) / LC;                                  // tiles of even (all) slices
    const int ntile = nte + (EVEN ? ((f.M + 1) / 2 + LC - 1) / LC : 0);
    cx<T>* rt = d.Rt + (size_t)i1 * S * n2;
    const cx<T>* dz = track ? d.dZt + (size_t)i1 * S * n2 : nullptr;
    // the change of W~ (FP64) in a loop of its own: as a predicated part of the
    // plain one its instructions took their issue slots of the FP64 pipe (one in
    // 60 clocks per scheduler) in every iteration
    auto tiles = [&](auto tr) {
      constexpr bool TRACK = decltype(tr)::value;
      for (int e = wid; e < ntile * ngr; e += nw) {
        const int g = e / ntile, it = e - g * ntile;
        const int q0 = ((it < nte) ? it * LC : f.nkep + (it - nte) * LC) + lg * TL;
        const int t0 = g * kGTubes<T> + lt;
        V acc[TL][kTT<T>];
        fold_forward<T, TL, EVEN, STAGED>(f, tabf, q0, pairs + t0, np2, acc);
        int k = EVEN ? (it < nte ? 2 * q0 : 2 * (q0 - f.nkep) + 1) : q0;
        int o = k * n2 + t0;
        const int dk = EVEN ? 2 : 1;
#pragma unroll
        for (int i = 0; i < TL; ++i, k += dk, o += dk * n2) {
          if (k >= S) break;
          const bool real = k == 0 || 2 * k == n3;
          cx<T> zv[kTT<T>];
          if (MODE != MODE_GRAD) {
#pragma unroll
            for (int j = 0; j < kTT<T>; ++j)
              if (t0 + kLW<T> * j < n2) {
                if (STAGED && zstaged) zv[j] = stg[k * width + t0 + kLW<T> * j];
                else zv[j] = ldg_cx(zrow + o + kLW<T> * j);
              }
          }
#pragma unroll
          for (int j = 0; j < kTT<T>; ++j) {
            if (t0 + kLW<T> * j >= n2) break;
            const cx<T> a = P::un(acc[i][j]);
            cx<T> x = {a.re, real ? T(0) : -a.im};
            if (MODE != MODE_GRAD) x = x - zv[j];
            if constexpr (TRACK) dw2 += dw_term(x, rt[o + kLW<T> * j], dz[o + kLW<T> * j], k, n3);
            rt[o + kLW<T> * j] = x;
          }
        }
      }
    };
    if (track) tiles(BoolC<true>{});
    else tiles(BoolC<false>{});
  }
  if (track) {
    double unused = 0.0;
    block_sum2(dw2, unused, red);
    if (tid == 0) d.part_dw[i1] = dw2;
  }
}

// ---------------------------------------------------------------------------
// Transforms of the factors with the same products: kGTubes tubes per CTA, the
// tubes and the coefficients staged in shared memory.  A factor is U = n r tubes,
// contiguous for every l (and, in the spectrum [S][r][n], for every k); with
// transposed = 1 (Y: spatial order s fastest) tube u of the spectrum is
// u = s n + i and of the spatial side s + r i.
//   k_fold_dft   real [n3][U] -> half spectrum [S][U]
//   k_fold_idft  half spectrum -> real, 1 / n3 included
// One thread per tube and four outputs before (k_factor_dft, k_factor_idft, which
// keep the lengths whose tables do not fit and the exact order of Engine::strict_):
// 80 + 51 and 88 + 65 us for both factors of 529 x 288 x 168, r = 16, against
// 27 + 23 and 18 + 14 here.
// ---------------------------------------------------------------------------
constexpr int kFoldThreads = 512;
constexpr int kFoldTL = 2;  // 22 items of the forward transform at n3 = 168 for 16 warps

// Shared bytes: table, then the folded pairs (forward) or the spectrum (inverse).
template <typename T>
__host__ __device__ inline size_t fold_dft_smem(int n3) {
  const FoldDims f = fold_dims(n3);
  const size_t ni = (size_t)(f.kmax + 1) * f.nlp, nf = (size_t)(f.lmax + 1) * f.nkt;
  return ((ni > nf ? ni : nf) + (size_t)(n3 / 2 + 1) * (kGTubes<T> + 1)) * sizeof(cx<T>);
}
template <typename T>
inline bool fold_dft_fits(int n3, int optin) {
  return n3 <= kSlabGMaxN3 && fold_dft_smem<T>(n3) <= (size_t)optin;
}

template <typename T, bool EVEN>
__device__ __forceinline__ void fold_dft_impl(const T* __restrict__ in, cx<T>* __restrict__ out,
                                              const cx<T>* __restrict__ fold, int n, int r, int n3, int transposed,
                                              unsigned char* smem) {
  constexpr int TL = kFoldTL, W = kGTubes<T>, LD = W + 1, LC = kLG<T> * TL;
  using P = Pk<T>;
  const FoldDims f = fold_dims(n3);
  const int ni = (f.kmax + 1) * f.nlp, nf = (f.lmax + 1) * f.nkt, S = n3 / 2 + 1;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  cx<T>* tab = reinterpret_cast<cx<T>*>(smem);
  cx<T>* pairs = tab + (ni > nf ? ni : nf);
  const size_t U = (size_t)n * r, u0 = (size_t)blockIdx.x * W;
  const int tn = (int)(U - u0 < (size_t)W ? U - u0 : (size_t)W);
  for (int e = tid; e < nf; e += blockDim.x) tab[e] = fold[ni + e];
  // the rows folded as in the slab kernel
  const int nfold = EVEN ? f.M / 2 + 1 : f.h + 1;
  for (int l = wid; l < nfold; l += nw)
    for (int t = lane; t < tn; t += 32) {
      const T* x = in + u0 + t;
      auto row = [&](int q) { return x[(size_t)q * U]; };
      if (EVEN && l > 0 && 2 * l != f.M) {
        const T a = row(l), b = row(n3 - l), c = row(f.M - l), e = row(f.M + l);
        const T ea = a + b, oa = a - b, eb = c + e, ob = c - e;
        pairs[l * LD + t] = cx<T>{ea + eb, oa - ob};
        pairs[(f.M - l) * LD + t] = cx<T>{ea - eb, oa + ob};
      } else if (EVEN) {
        const T a = row(l), b = row(l == 0 ? f.M : n3 - l);
        pairs[l * LD + t] = cx<T>{a + b, a - b};
      } else {
        const T a = row(l), b = l > 0 ? row(n3 - l) : T(0);
        pairs[l * LD + t] = l > 0 ? cx<T>{a + b, a - b} : cx<T>{a, T(0)};
      }
    }
  __syncthreads();
  const int lt = lane & (kLW<T> - 1), lg = lane / kLW<T>;
  const int nte = (f.nke + LC - 1) / LC, ntile = nte + (EVEN ? ((f.M + 1) / 2 + LC - 1) / LC : 0);
  for (int it = wid; it < ntile; it += nw) {
    const int q0 = ((it < nte) ? it * LC : f.nkep + (it - nte) * LC) + lg * TL;
    typename P::V acc[TL][kTT<T>];
    fold_forward<T, TL, EVEN, true>(f, tab, q0, pairs + lt, LD, acc);
#pragma unroll
    for (int i = 0; i < TL; ++i) {
      const int k = EVEN ? (it < nte ? 2 * (q0 + i) : 2 * (q0 - f.nkep + i) + 1) : q0 + i;
      if (k >= S) break;
#pragma unroll
      for (int j = 0; j < kTT<T>; ++j) {
        const int t = kLW<T> * j + lt;
        if (t >= tn) continue;
        const size_t u = u0 + t, o = transposed ? (u % r) * n + u / r : u;
        const cx<T> a = P::un(acc[i][j]);
        out[(size_t)k * U + o] = cx<T>{a.re, (k == 0 || 2 * k == n3) ? T(0) : -a.im};
      }
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(kFoldThreads) k_fold_dft(const T* __restrict__ in, cx<T>* __restrict__ out,
                                                           const cx<T>* __restrict__ fold, int n, int r, int n3,
                                                           int transposed) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (n3 & 1) fold_dft_impl<T, false>(in, out, fold, n, r, n3, transposed, smem);
  else fold_dft_impl<T, true>(in, out, fold, n, r, n3, transposed, smem);
}

template <typename T, bool EVEN>
__device__ __forceinline__ void fold_idft_impl(const cx<T>* __restrict__ in, T* __restrict__ out,
                                               const cx<T>* __restrict__ fold, int n, int r, int n3, int transposed,
                                               unsigned char* smem) {
  constexpr int TL = kFoldTL, W = kGTubes<T>, LC = kLG<T> * TL;
  using P = Pk<T>;
  const FoldDims f = fold_dims(n3);
  const int ni = (f.kmax + 1) * f.nlp, nf = (f.lmax + 1) * f.nkt, S = n3 / 2 + 1;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  cx<T>* tab = reinterpret_cast<cx<T>*>(smem);
  cx<T>* spec = tab + (ni > nf ? ni : nf);  // [S][W]
  const size_t U = (size_t)n * r, u0 = (size_t)blockIdx.x * W;
  const int tn = (int)(U - u0 < (size_t)W ? U - u0 : (size_t)W);
  for (int e = tid; e < ni; e += blockDim.x) cp_async_elem(tab + e, fold + e);
  for (int k = wid; k < S; k += nw)
    for (int t = lane; t < tn; t += 32) cp_async_elem(spec + k * W + t, in + (size_t)k * U + u0 + t);
  cp_async_wait_all();
  __syncthreads();
  const T scale = T(2) / T(n3);
  const int lt = lane & (kLW<T> - 1), lg = lane / kLW<T>;
  for (int lb = wid * LC; lb < f.nl; lb += nw * LC) {
    const int l0 = lb + lg * TL;
    typename P::V E[TL][kTT<T>], O[TL][kTT<T>];
    fold_inverse<T, TL, EVEN>(f, tab, l0, 0, spec + lt, W, E);
    if (EVEN) fold_inverse<T, TL, EVEN>(f, tab, l0, 1, spec + lt, W, O);
#pragma unroll
    for (int i = 0; i < TL; ++i) {
      const int l = l0 + i;
      if (l >= f.nl) break;
#pragma unroll
      for (int j = 0; j < kTT<T>; ++j) {
        const int t = kLW<T> * j + lt;
        if (t >= tn) continue;
        const size_t u = u0 + t, o = transposed ? (u % n) * r + u / n : u;
        auto put = [&](int q, T v) { out[(size_t)q * U + o] = v * scale; };
        const cx<T> a = P::un(E[i][j]);
        if constexpr (EVEN) {
          const cx<T> b = P::un(O[i][j]);
          const T cs = a.re + b.re, ds = a.im + b.im, cd = a.re - b.re, dd = a.im - b.im;
          put(l, cs - ds);
          if (l > 0) put(n3 - l, cs + ds);
          if (l == 0) put(f.M, cd);
          else if (2 * l != f.M) {
            put(f.M - l, cd + dd);
            put(f.M + l, cd - dd);
          }
        } else {
          put(l, a.re - a.im);
          if (l > 0) put(n3 - l, a.re + a.im);
        }
      }
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(kFoldThreads) k_fold_idft(const cx<T>* __restrict__ in, T* __restrict__ out,
                                                            const cx<T>* __restrict__ fold, int n, int r, int n3,
                                                            int transposed) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (n3 & 1) fold_idft_impl<T, false>(in, out, fold, n, r, n3, transposed, smem);
  else fold_idft_impl<T, true>(in, out, fold, n, r, n3, transposed, smem);
}

// GENERAL (MODE_ITER): the W-step of long runs and strong smoothing (see
// wstep_segments), chosen by the engine; as a branch of one kernel it cost the plain
// form 5% (925 x 153 x 92: 150 -> 160 us, in spills).
template <typename T, int MODE, int TL, bool STAGED, bool GENERAL = false>
__global__ void __launch_bounds__(kSlabGThreads<T>, GENERAL && sizeof(T) == 8 ? 2 : 1) k_slab_g(Dev<T> d, T* __restrict__ Wout, int flags, int init) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (MODE == MODE_ITER && !init && converged(d)) return;
  if ((d.n3 & 1) == 0) slab_g_impl<T, MODE, TL, true, STAGED, GENERAL>(d, Wout, flags, init, smem);
  else slab_g_impl<T, MODE, TL, false, STAGED, GENERAL>(d, Wout, flags, init, smem);
}

}  // namespace tc
