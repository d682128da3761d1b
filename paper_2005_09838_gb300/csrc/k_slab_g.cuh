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
// Tiles.  A warp computes TL rows (inverse) or slices (forward) of 64 tubes
// (two per lane; FP64: 32): each pair that is read feeds TL products and each
// coefficient two.  tc_init times TL = 2, 4, 8 (a larger tile has fewer loads
// per product, a smaller one fills the warps of small slabs).
//
// Staging.  The coefficients of one direction, the spectrum of as many 64-tube
// groups as fit (all of them for most sizes) and G are copied to shared memory
// by cp.async, so the transforms read nothing but shared memory: with the
// spectrum and the coefficients read through L1 and G inside the item's
// epilogue the inverse took 72K cycles of a 925 x 153 x 92 CTA against 28K for
// the forward one.  G goes straight to its place in the slab and the inverse
// stores only the missing entries.  Sizes whose slab leaves no room for the
// stages take the unstaged form (STAGED = false).
//
// The modes are those of k_slab.
#pragma once

namespace tc {

// Threads per CTA at most: 512 leave 128 registers a thread (FP64 values take
// two each, so half as many threads).
template <typename T>
constexpr int kSlabGThreads = sizeof(T) == 8 ? 256 : 512;
// Tubes per lane (FP64: one, no product is worth a half-empty warp there) and per item.
template <typename T>
constexpr int kTT = sizeof(T) == 8 ? 1 : 2;
template <typename T>
constexpr int kGTubes = 32 * kTT<T>;
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
  int nl, nlp;         // rows l of the inverse (the others follow), padded to 8
  int kmax;            // slices 1 .. kmax of the inverse loop
  int nke, nkep, nkt;  // even slices (all slices for odd n3), padded to 8; columns of the forward table
  int lmax;            // rows 1 .. lmax of the forward loop
};
__host__ __device__ inline FoldDims fold_dims(int n3) {
  FoldDims f{};
  f.even = (n3 % 2) == 0;
  f.M = n3 / 2;
  f.h = (n3 - 1) / 2;
  f.np = (n3 + 1) / 2;
  f.nl = f.even ? f.M / 2 + 1 : f.h + 1;
  f.nlp = (f.nl + 7) / 8 * 8;
  f.kmax = f.even ? f.M - 1 : f.h;
  f.nke = f.even ? f.M / 2 + 1 : f.h + 1;
  f.nkep = (f.nke + 7) / 8 * 8;
  f.nkt = f.even ? f.nkep + ((f.M + 1) / 2 + 7) / 8 * 8 : f.nkep;
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
// Tubes of a stage of sg groups.
template <typename T>
__host__ __device__ inline int slab_g_width(int n2, int sg) { return sg * kGTubes<T> < n2 ? sg * kGTubes<T> : n2; }
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
  off = align_up(off + sizeof(cx<T>) * (size_t)((n3 + 1) / 2) * slab_g_stride(n2), 16);
  L.stage = off;
  off = align_up(off + sizeof(cx<T>) * (size_t)(n3 / 2 + 1) * slab_g_width<T>(n2, sg), 16);
  L.total = off;
  return L;
}

// Launch shape of the folded-transform slab kernels: two CTAs of 256 threads on
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
        pl = SlabGPlan{pass == 0 ? 256 : kSlabGThreads<T>, sg, b};
        return true;
      }
    }
  }
  pl = SlabGPlan{kSlabGThreads<T>, 0, slab_g_layout<T>(n2, n3, 0).total};
  return pl.smem <= (size_t)optin;
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

// One item of the inverse transform: rows l0 .. l0 + TL - 1 (and those that
// follow from them) of kGTubes<T> tubes.  load(k, j) gives the spectrum pair of
// slice k in tube j of the lane; E, O receive the sums over even and odd
// slices (all slices in E for odd n3), slices 0 and n3/2 included with weight 1/2.
template <typename T, int TL, bool EVEN, bool SH, typename LoadFn>
__device__ __forceinline__ void fold_inverse(const FoldDims& f, const cx<T>* __restrict__ tab, int l0, LoadFn load,
                                             typename Pk<T>::V (&E)[TL][kTT<T>],
                                             typename Pk<T>::V (&O)[EVEN ? TL : 1][kTT<T>]) {
  using P = Pk<T>;
  using V = typename P::V;
#pragma unroll
  for (int j = 0; j < kTT<T>; ++j) {
    const V x0 = P::mk(T(0.5) * P::un(load(0, j)).re, T(0));
#pragma unroll
    for (int i = 0; i < TL; ++i) E[i][j] = x0;
    if constexpr (EVEN) {
      const T xm = T(0.5) * P::un(load(f.M, j)).re;
      const bool modd = f.M & 1;
#pragma unroll
      for (int i = 0; i < TL; ++i) {
        const V a = P::mk(((l0 + i) & 1) ? -xm : xm, T(0));
        O[i][j] = modd ? a : P::mk(T(0), T(0));
        if (!modd) E[i][j] = P::add(E[i][j], a);
      }
    }
  }
  const cx<T>* tl = tab + l0;
  auto step = [&](int k, const V (&x)[kTT<T>], V (&acc)[TL][kTT<T>]) {
    const cx<T>* tk = tl + (size_t)k * f.nlp;
#pragma unroll
    for (int i = 0; i < TL; i += 2) {
      V c0, c1;
      P::template ld2<SH>(tk + i, c0, c1);
#pragma unroll
      for (int j = 0; j < kTT<T>; ++j) {
        P::fma(acc[i][j], x[j], c0);
        P::fma(acc[i + 1][j], x[j], c1);
      }
    }
  };
  auto acc_of = [&](int odd) -> V(&)[TL][kTT<T>] {
    if constexpr (EVEN) {
      if (odd) return O;
    }
    return E;
  };
  constexpr int U = 4;  // slices whose loads are in flight together (even: parity fixed per position)
  V xn[U][kTT<T>];
  int k = 1;
  const int kend = 1 + f.kmax / U * U;
  if (k < kend) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int j = 0; j < kTT<T>; ++j) xn[u][j] = load(k + u, j);
  }
  for (; k < kend; k += U) {
    V x[U][kTT<T>];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int j = 0; j < kTT<T>; ++j) x[u][j] = xn[u][j];
    if (k + U < kend) {
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int j = 0; j < kTT<T>; ++j) xn[u][j] = load(k + U + u, j);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) step(k + u, x[u], acc_of((u + 1) & 1));
  }
#pragma unroll
  for (int u = 0; u < U - 1; ++u) {
    if (k + u <= f.kmax) {
      V x[kTT<T>];
#pragma unroll
      for (int j = 0; j < kTT<T>; ++j) x[j] = load(k + u, j);
      step(k + u, x, acc_of((u + 1) & 1));
    }
  }
}

// One item of the forward transform: columns q0 .. q0 + TL - 1 of the forward
// table (slices of one parity for even n3) of kGTubes<T> tubes, from the folded
// slab.  acc receives (sum e c, sum o s).
template <typename T, int TL, bool EVEN, bool SH>
__device__ __forceinline__ void fold_forward(const FoldDims& f, const cx<T>* __restrict__ tab, int q0,
                                             const cx<T>* const (&col)[kTT<T>], int np2,
                                             typename Pk<T>::V (&acc)[TL][kTT<T>]) {
  using P = Pk<T>;
  using V = typename P::V;
  const bool oddk = EVEN && q0 >= f.nkep;
  const int kk0 = oddk ? q0 - f.nkep : q0;  // k = 2 (kk0 + i) + oddk for even n3
#pragma unroll
  for (int j = 0; j < kTT<T>; ++j) {
    const cx<T> s0 = col[j][0];
    const V a0 = P::mk(EVEN && oddk ? s0.im : s0.re, T(0));
#pragma unroll
    for (int i = 0; i < TL; ++i) acc[i][j] = a0;
    if (EVEN && (f.M & 1) == 0) {
      // row M/2: e cos(pi k / 2) on even slices, o sin(pi k / 2) on odd ones
      const cx<T> sm = col[j][(size_t)(f.M / 2) * np2];
#pragma unroll
      for (int i = 0; i < TL; ++i) {
        const bool neg = (kk0 + i) & 1;
        const T a = neg ? -sm.re : sm.re, b = neg ? -sm.im : sm.im;
        acc[i][j] = P::add(acc[i][j], oddk ? P::mk(T(0), b) : P::mk(a, T(0)));
      }
    }
  }
  // slot l holds the even fold, slot M - l the odd one
  const int sl = oddk ? f.M : 0, sd = oddk ? -1 : 1;
  const cx<T>* tq = tab + q0;
#pragma unroll 4
  for (int l = 1; l <= f.lmax; ++l) {
    V x[kTT<T>];
    const int so = (sl + sd * l) * np2;
#pragma unroll
    for (int j = 0; j < kTT<T>; ++j) x[j] = P::lds(col[j] + so);
    const cx<T>* tk = tq + (size_t)l * f.nkt;
#pragma unroll
    for (int i = 0; i < TL; i += 2) {
      V c0, c1;
      P::template ld2<SH>(tk + i, c0, c1);
#pragma unroll
      for (int j = 0; j < kTT<T>; ++j) {
        P::fma(acc[i][j], x[j], c0);
        P::fma(acc[i + 1][j], x[j], c1);
      }
    }
  }
}

template <typename T, int MODE, int TL, bool EVEN, bool STAGED>
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
  const cx<T>* tabi = STAGED ? tab : d.fold;
  const cx<T>* tabf = STAGED ? tab : d.fold + ni;
  const cx<T>* zrow = d.Zt + (size_t)i1 * S * n2;
  const cx<T>* rrow = d.Rt + (size_t)i1 * S * n2;
  const T* Gi = d.G + (size_t)i1 * n2 * n3;
  const uint32_t* Mi = d.mask + (size_t)i1 * n3 * mw;
  const bool wsolve = (MODE == MODE_ITER) && !init && d.rho2 != T(0);
  const T zfac = init ? T(0) : ((d.rho2 == T(0)) ? T(1) / (T(1) + d.mu) : T(1));
  constexpr bool NEED_G = (MODE == MODE_ITER || MODE == MODE_GRAD);

  // ---- masks, W-step table, coefficients, G into its place in the slab ---------------------
  if (wsolve)
    for (int j = tid; j < 6 * n2; j += nt) wtab[j] = d.winv[j];
  if (MODE != MODE_W)
    for (int e = tid; e < n3 * mw; e += nt) {
      const int q = e / mw;
      msk[e] = __ldg(Mi + (size_t)slab_g_row(EVEN, n3, q) * mw + (e - q * mw));
    }
  if (STAGED)
    for (int e = tid; e < ni; e += nt) cp_async_elem(tab + e, d.fold + e);
  if (NEED_G)
    for (int l = wid; l < n3; l += nw) {
      T* row = spat + slab_g_off(EVEN, n3, l, np2);
      for (int t = lane; t < n2; t += 32) cp_async_elem(row + 2 * t, Gi + (size_t)l * n2 + t);
    }

  // ---- inverse transform; v = G on the mask, Z elsewhere (MODE_GRAD: Z - G on the
  // mask, 0 elsewhere) --------------------------------------------------------------------
  const int ngr = (n2 + kGTubes<T> - 1) / kGTubes<T>;
  const int gstage = STAGED ? sg : ngr;
  const int width = slab_g_width<T>(n2, gstage);  // tubes of a full stage, its row stride
  const T scale = T(2) / T(n3);
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
    const int ntile = (f.nl + TL - 1) / TL;
    for (int e = wid; e < ntile * gn; e += nw) {
      const int gl = e / ntile, g = g0 + gl, l0 = (e - gl * ntile) * TL;
      int t[kTT<T>];
      const cx<T>* zc[kTT<T>];
      const cx<T>* rc[kTT<T>];
#pragma unroll
      for (int j = 0; j < kTT<T>; ++j) {
        t[j] = g * kGTubes<T> + 32 * j + lane;
        const int tq = min(t[j], n2 - 1);
        zc[j] = STAGED ? stg + (tq - g0 * kGTubes<T>) : zrow + tq;
        rc[j] = rrow + tq;
      }
      auto load = [&](int k, int j) -> V {
        if (STAGED) return P::lds(zc[j] + k * width);
        const size_t o = (size_t)k * n2;
        if (MODE == MODE_W) return P::add(P::ldg(zc[j] + o), P::ldg(rc[j] + o));
        return P::ldg((MODE == MODE_R ? rc[j] : zc[j]) + o);
      };
      V E[TL][kTT<T>], O[EVEN ? TL : 1][kTT<T>];
      fold_inverse<T, TL, EVEN, STAGED>(f, tabi, l0, load, E, O);
      // value of the row at slab index q (row order), half h of slot p, tube j
      auto put = [&](T x, int q, T* at, int j) {
        x *= scale;
        const bool live = t[j] < n2;
        if (NEED_G) {
          const uint32_t w = (g * kTT<T> + j < mw) ? msk[q * mw + g * kTT<T> + j] : 0u;
          const bool ob = (w >> lane) & 1u;
          if (MODE == MODE_ITER) {
            if (live && !ob) *at = x * zfac;
          } else if (live) {
            x = ob ? x - *at : T(0);
            gsum.add(x);
            *at = x;
          }
        } else if (live) {
          *at = x;
        }
      };
#pragma unroll
      for (int i = 0; i < TL; ++i) {
        const int l = l0 + i;
        if (l >= f.nl) break;
#pragma unroll
        for (int j = 0; j < kTT<T>; ++j) {
          T* cp = spat + 2 * (l * np2 + t[j]);
          if constexpr (EVEN) {
            const cx<T> a = P::un(E[i][j]), b = P::un(O[i][j]);
            const T cs = a.re + b.re, ds = a.im + b.im, cd = a.re - b.re, dd = a.im - b.im;
            if (l == 0) {
              put(cs, 0, cp, j);
              put(cd, 1, cp + 1, j);
            } else {
              put(cs - ds, 2 * l, cp, j);
              put(cs + ds, 2 * l + 1, cp + 1, j);
              if (2 * l != f.M) {
                T* cm = spat + 2 * ((f.M - l) * np2 + t[j]);
                put(cd + dd, 2 * (f.M - l), cm, j);
                put(cd - dd, 2 * (f.M - l) + 1, cm + 1, j);
              }
            }
          } else {
            const cx<T> a = P::un(E[i][j]);
            if (l == 0) {
              put(a.re, 0, cp, j);
            } else {
              put(a.re - a.im, 2 * l - 1, cp, j);
              put(a.re + a.im, 2 * l, cp + 1, j);
            }
          }
        }
      }
    }
  }
  __syncthreads();

  // ---- read-back modes: partial sums, optional copy of W ----------------------------------
  if (MODE == MODE_W || MODE == MODE_R) {
    const bool sums = MODE == MODE_R || !(flags & SLAB_NOSUM);
    SqSum<T> sa, sb;
    for (int q = wid; q < n3; q += nw) {
      const int l = slab_g_row(EVEN, n3, q);
      const T* row = spat + slab_g_off(EVEN, n3, l, np2);
      for (int t = lane; t < n2; t += 32) {
        const T v = row[2 * t];
        if (sums) sa.add(v);
        if (MODE == MODE_W) {
          if (sums && t + 1 < n2) sb.add_diff(v, row[2 * (t + 1)]);
          if (Wout) {
            if (flags & SLAB_WROWS) Wout[((size_t)i1 * n3 + l) * n2 + t] = v;
            else Wout[(size_t)i1 + (size_t)n1 * ((size_t)t + (size_t)n2 * l)] = v;
          }
        } else {
          if ((msk[q * mw + (t >> 5)] >> lane) & 1u) sb.add(v);
        }
      }
    }
    if (!sums) return;
    double a = sa.total(), b = sb.total();
    block_sum2(a, b, red);
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
  if (wsolve)
    wstep_segments<T>([&](int q) { return spat + slab_g_off(EVEN, n3, slab_g_row(EVEN, n3, q), np2); }, 2, msk, n3, n2,
                   d.rho2, wtab);

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
    const int nte = (f.nke + TL - 1) / TL;                                  // tiles of even (all) slices
    const int ntile = nte + (EVEN ? ((f.M + 1) / 2 + TL - 1) / TL : 0);
    cx<T>* rt = d.Rt + (size_t)i1 * S * n2;
    const cx<T>* dz = track ? d.dZt + (size_t)i1 * S * n2 : nullptr;
    // the change of W~ (FP64) in a loop of its own: as a predicated part of the
    // plain one its instructions took their issue slots of the FP64 pipe (one in
    // 60 clocks per scheduler) in every iteration
    auto tiles = [&](auto tr) {
      constexpr bool TRACK = decltype(tr)::value;
      for (int e = wid; e < ntile * ngr; e += nw) {
        const int g = e / ntile, it = e - g * ntile;
        const int q0 = (it < nte) ? it * TL : f.nkep + (it - nte) * TL;
        int t[kTT<T>];
        const cx<T>* col[kTT<T>];
#pragma unroll
        for (int j = 0; j < kTT<T>; ++j) {
          t[j] = g * kGTubes<T> + 32 * j + lane;
          col[j] = pairs + min(t[j], n2 - 1);
        }
        V acc[TL][kTT<T>];
        fold_forward<T, TL, EVEN, STAGED>(f, tabf, q0, col, np2, acc);
#pragma unroll
        for (int i = 0; i < TL; ++i) {
          const int k = EVEN ? (it < nte ? 2 * (q0 + i) : 2 * (q0 - f.nkep + i) + 1) : q0 + i;
          if (k >= S) break;
#pragma unroll
          for (int j = 0; j < kTT<T>; ++j) {
            if (t[j] >= n2) continue;
            const int o = k * n2 + t[j];
            const cx<T> a = P::un(acc[i][j]);
            cx<T> x = {a.re, (k == 0 || 2 * k == n3) ? T(0) : -a.im};
            if (MODE != MODE_GRAD) x = x - (zstaged ? stg[o] : ldg_cx(zrow + o));
            if constexpr (TRACK) dw2 += dw_term(x, rt[o], dz[o], k, n3);
            rt[o] = x;
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
  if (MODE == MODE_GRAD) {
    double g = gsum.total(), unused = 0.0;
    block_sum2(g, unused, red);
    if (tid == 0) d.part[(size_t)i1 * 4] = g;
  }
}

template <typename T, int MODE, int TL, bool STAGED>
__global__ void __launch_bounds__(kSlabGThreads<T>, 1) k_slab_g(Dev<T> d, T* __restrict__ Wout, int flags, int init) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (MODE == MODE_ITER && !init && converged(d)) return;
  if ((d.n3 & 1) == 0) slab_g_impl<T, MODE, TL, true, STAGED>(d, Wout, flags, init, smem);
  else slab_g_impl<T, MODE, TL, false, STAGED>(d, Wout, flags, init, smem);
}

}  // namespace tc
