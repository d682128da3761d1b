// FP32 slice contractions of larger ranks as register-tiled complex products:
//   k_qcon_f  Q_k = R~_k Y~_k^H    (rows of 64, all r columns, summed over n2)
//   k_dcon_f  D_k = X~'_k^H R~_k   (all r rows, 64 columns, partial sums over n1)
//   k_zsyn_f  Z~_k = X~'_k Y~'_k   (64 x 64 tiles)
// A thread holds 4 x 4 complex accumulators: per step 64 multiply-adds for 64
// bytes read from shared memory, the ratio at which the 128 bytes per clock that
// an SM returns from shared memory and its FP32 lanes finish together.  Operands
// come by cp.async, two stages deep where the sum is long.  Where 4 x 4 tiles of
// an r x 64 output do not fill the CTA's 128 threads (r <= 16), groups of threads
// share the tile and split the sum.
//
// The kernels they replace (k_qcon, and k_ystep doing D, the update and Z~ on
// one column tile) read each operand from shared memory for one or two products
// and held all of X~' per CTA: at r > 8 one CTA per SM, 364 us for the Y-step of
// 601 x 253 x 86, r = 15.
#pragma once

namespace tc {

constexpr int kGmThreads = 128;
constexpr int kGmTile = 64;   // rows (Q, Z~) and columns (D, Z~) of a tile
constexpr int kGmKC = 16;     // rows of R~ per stage of k_dcon_f
constexpr int kGmKQ = 32;     // columns of R~ per stage of k_qcon_f

template <int RP>
struct GmGroups {
  static constexpr int SG = RP / 4;                       // groups of four columns / rows s
  static constexpr int KG = kGmThreads / (16 * SG);       // thread groups that split the sum
};

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// four consecutive complex values (16-byte aligned)
__device__ __forceinline__ void lds_cx4(const cx<float>* p, cx<float> (&v)[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 2);
  v[0] = {a.x, a.y};
  v[1] = {a.z, a.w};
  v[2] = {b.x, b.y};
  v[3] = {b.z, b.w};
}

__device__ __forceinline__ void lds_cx4(const cx<double>* p, cx<double> (&v)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = p[q];
}

// Sums of the KG thread groups, into group 0 (fixed order); red: KG - 1 tiles.
// pairs: the accumulators are (value, rounding errors) pairs.
template <int KG>
__device__ __forceinline__ void group_sum(cx<float> (&acc)[4][4], cx<float>* red, int g, int t, int nt, bool pairs) {
  if constexpr (KG > 1) {
    __syncthreads();
    if (g > 0)
#pragma unroll
      for (int e = 0; e < 16; ++e) red[((g - 1) * 16 + e) * nt + t] = acc[e / 4][e % 4];
    __syncthreads();
    if (g == 0)
#pragma unroll
      for (int q = 1; q < KG; ++q)
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          cx<float>& a = acc[e / 4][e % 4];
          const cx<float> b = red[((q - 1) * 16 + e) * nt + t];
          if (pairs) pair_add(a.re, a.im, b.re, b.im);
          else a = a + b;
        }
  }
}

// ---- D = X~'^H R~: grid (S, ceil(n2/64), ksplit), partial sums over ranges of n1 ------------
template <int RP>
__host__ __device__ constexpr size_t dcon_f_smem() {
  return 2 * (size_t)kGmKC * (kGmTile + RP) * sizeof(cx<float>);
}

// Columns j0 .. j0 + 63 of the partial D of slice k over the z-th of ks ranges of
// rows, by 128 threads (tid) with dcon_f_smem<RP>() bytes; every thread of the
// block calls it with the same range.
//
// STRIDED: partial w of eight sums the rows i = w mod 8 in increasing order, as the
// warps of the fused k_ystep do (bit for bit: see Engine::strict_, r <= 8); the thread
// groups take a partial each in place of sharing one, and z counts the CTAs.
//
// Real slices (with d.dpairs): the factors and the residual are real, and D is formed as a
// compensated sum, (value, rounding errors) in the (re, im) fields.  D of the DC
// slice is the one sum of the iteration whose rounding matters: it is added to
// Dg Y~ of nearly the same size, and G^+ multiplies what is left of both by the
// condition number of the DC Gram.  Rounded to FP32 it alone gave 1.5e-5 of the
// 1.5e-5 error of X~ and 2.6e-5 of the 2.7e-5 of Y~ after five iterations on
// 529 x 96 x 112, r = 32; every other sum and stored array together 6e-6.
constexpr int kDStride = 8;  // partials of the strided form
template <int RP, bool STRIDED>
__device__ __forceinline__ void dcon_f_tile(const Dev<float>& d, int k, int j0, int z, int ks, unsigned char* smem,
                                            int tid) {
  constexpr int SG = GmGroups<RP>::SG, KG = GmGroups<RP>::KG, NTG = 16 * SG;
  const int n1 = d.n1, n2 = d.n2, r = d.r, S = d.S;
  const bool real = (k == 0 || 2 * k == d.n3) && d.dpairs;
  const int per = (n1 + ks - 1) / ks;
  // staged rows ib .. ie - 1; the strided form counts them from 0: kDStride / KG
  // CTAs share n1 rows, KG of them at a time
  const int ib = STRIDED ? 0 : min(z * per, n1), ie = STRIDED ? (n1 + kDStride - 1) / kDStride * KG : min(ib + per, n1);
  auto row_of = [&](int q) { return STRIDED ? kDStride * (q / KG) + z * KG + q % KG : q; };
  cx<float>* Rs = reinterpret_cast<cx<float>*>(smem);        // [2][KC][64]
  cx<float>* Xs = Rs + 2 * kGmKC * kGmTile;                  // [2][KC][RP]
  const int cl = tid & 15, sgi = (tid >> 4) % SG, g = tid / NTG;
  const int ncol = min(kGmTile, n2 - j0);
  const size_t rs = (size_t)S * n2;
  const cx<float>* Rb = d.Rt + (size_t)k * n2 + j0;
  const cx<float>* Xb = d.Xt + (size_t)k * r * n1;
  const bool vec = (n2 & 1) == 0;  // rows of R~ start on 16 bytes
  if (r < RP)
    for (int e = tid; e < 2 * kGmKC * RP; e += kGmThreads)
      if (e % RP >= r) Xs[e] = cx<float>{0.f, 0.f};
  auto rows_in = [&](int i0) {  // rows of the stage at i0 that exist
    int nk = min(kGmKC, ie - i0);
    if (STRIDED)
      while (nk > 0 && row_of(i0 + nk - 1) >= n1) --nk;
    return nk;
  };
  auto stage = [&](int b, int i0) {
    const int nk = rows_in(i0);
    cx<float>* rd = Rs + b * kGmKC * kGmTile;
    cx<float>* xd = Xs + b * kGmKC * RP;
    if (vec) {
      for (int e = tid; e < nk * (kGmTile / 2); e += kGmThreads) {
        const int q = e / (kGmTile / 2), c = 2 * (e % (kGmTile / 2));
        if (c < ncol) cp_async16(rd + q * kGmTile + c, Rb + (size_t)row_of(i0 + q) * rs + c);
      }
    } else {
      for (int e = tid; e < nk * kGmTile; e += kGmThreads) {
        const int q = e / kGmTile, c = e % kGmTile;
        if (c < ncol) cp_async_elem(rd + q * kGmTile + c, Rb + (size_t)row_of(i0 + q) * rs + c);
      }
    }
    for (int e = tid; e < r * kGmKC; e += kGmThreads) {
      const int s = e / kGmKC, q = e % kGmKC;
      if (q < nk) cp_async_elem(xd + q * RP + s, Xb + (size_t)s * n1 + row_of(i0 + q));
    }
    cp_async_commit();
  };
  cx<float> acc[4][4];  // [column][s]
#pragma unroll
  for (int e = 0; e < 16; ++e) acc[e / 4][e % 4] = cx<float>{0.f, 0.f};
  if (ib < ie) stage(0, ib);
  int b = 0;
  for (int i0 = ib; i0 < ie; i0 += kGmKC, b ^= 1) {
    if (i0 + kGmKC < ie) {
      stage(b ^ 1, i0 + kGmKC);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const cx<float>* rd = Rs + b * kGmKC * kGmTile + cl;
    const cx<float>* xd = Xs + b * kGmKC * RP + 4 * sgi;
    const int nk = rows_in(i0);
    if (!STRIDED && real) {
      // four rows in plain FP32, then one error-free addition: the roundings that
      // count are those against the whole sum
      for (int q = g; q < nk; q += 4 * KG) {
        float p4[4][4];
#pragma unroll
        for (int e = 0; e < 16; ++e) p4[e / 4][e % 4] = 0.f;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const int row = q + w * KG;
          if (row < nk) {
            cx<float> x[4];
            lds_cx4(xd + row * RP, x);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const float v = rd[row * kGmTile + 16 * c].re;
#pragma unroll
              for (int p = 0; p < 4; ++p) p4[c][p] = fmaf(x[p].re, v, p4[c][p]);
            }
          }
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) pair_add(acc[e / 4][e % 4].re, acc[e / 4][e % 4].im, p4[e / 4][e % 4], 0.f);
      }
    } else {
#pragma unroll 4
      for (int q = g; q < nk; q += KG) {
        cx<float> x[4], v[4];
        lds_cx4(xd + q * RP, x);
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = rd[q * kGmTile + 16 * c];
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int p = 0; p < 4; ++p) cfmaconj(acc[c][p], x[p], v[c]);
      }
    }
    __syncthreads();
  }
  int zp = z;  // partial written
  if constexpr (STRIDED) {
    zp = z * KG + g;
  } else {
    group_sum<KG>(acc, Rs, g, tid % NTG, NTG, real);
    if (g > 0) return;
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int s = 4 * sgi + p;
    if (s >= r) break;
    cx<float>* o = d.Dpart + (((size_t)k * d.ksplit + zp) * r + s) * n2 + j0;
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (cl + 16 * c < ncol) o[cl + 16 * c] = acc[c][p];
  }
}

template <int RP, bool STRIDED = false>
__global__ void __launch_bounds__(kGmThreads) k_dcon_f(Dev<float> d) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (converged(d)) return;
  dcon_f_tile<RP, STRIDED>(d, blockIdx.x, blockIdx.y * kGmTile, blockIdx.z, gridDim.z, smem, threadIdx.x);
}

inline int dcon_f_groups(int rp) { return rp == 8 ? GmGroups<8>::KG : rp == 16 ? GmGroups<16>::KG : GmGroups<32>::KG; }

// Splits of n1: about four CTAs of k_dcon_f per SM, at least 32 rows each.
inline int dcon_f_split(int S, int n1, int n2, int nsm) {
  const int base = S * ((n2 + kGmTile - 1) / kGmTile), want = (4 * nsm + base - 1) / base, most = (n1 + 31) / 32;
  return want < 1 ? 1 : want < most ? want : most;
}

// ---- Q = R~ Y~^H: grid (S, ceil(n1/64)) ---------------------------------------------------------
constexpr int kGmLdQ = kGmKQ + 1;  // odd row pitch: sixteen rows read distinct banks
template <int RP>
__host__ __device__ constexpr size_t qcon_f_smem() {
  return align_up(2 * (size_t)kGmTile * kGmLdQ * sizeof(cx<float>), 16) + 2 * (size_t)kGmKQ * RP * sizeof(cx<float>);
}

template <int RP>
__global__ void __launch_bounds__(kGmThreads) k_qcon_f(Dev<float> d, cx<float>* __restrict__ Qout) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (converged(d)) return;
  constexpr int SG = GmGroups<RP>::SG, KG = GmGroups<RP>::KG, NTG = 16 * SG;
  const int k = blockIdx.x, i0 = blockIdx.y * kGmTile;
  const int n1 = d.n1, n2 = d.n2, r = d.r, S = d.S, tid = threadIdx.x;
  cx<float>* Rs = reinterpret_cast<cx<float>*>(smem);                                     // [2][64][LdQ]
  cx<float>* Ys = reinterpret_cast<cx<float>*>(smem + align_up(2 * (size_t)kGmTile * kGmLdQ * sizeof(cx<float>), 16));
  const int rl = tid & 15, sgi = (tid >> 4) % SG, g = tid / NTG;
  const int nrow = min(kGmTile, n1 - i0);
  const size_t rs = (size_t)S * n2;
  const cx<float>* Rb = d.Rt + (size_t)i0 * rs + (size_t)k * n2;
  const cx<float>* Yb = d.Yt + (size_t)k * r * n2;
  if (r < RP)
    for (int e = tid; e < 2 * kGmKQ * RP; e += kGmThreads)
      if (e % RP >= r) Ys[e] = cx<float>{0.f, 0.f};
  auto stage = [&](int b, int j0) {
    const int nk = min(kGmKQ, n2 - j0), c = tid % kGmKQ;
    cx<float>* rd = Rs + b * kGmTile * kGmLdQ;
    cx<float>* yd = Ys + b * kGmKQ * RP;
    if (c < nk) {
      for (int q = tid / kGmKQ; q < nrow; q += kGmThreads / kGmKQ)
        cp_async_elem(rd + q * kGmLdQ + c, Rb + (size_t)q * rs + j0 + c);
      for (int s = tid / kGmKQ; s < r; s += kGmThreads / kGmKQ)
        cp_async_elem(yd + c * RP + s, Yb + (size_t)s * n2 + j0 + c);
    }
    cp_async_commit();
  };
  cx<float> acc[4][4];  // [row][s]
#pragma unroll
  for (int e = 0; e < 16; ++e) acc[e / 4][e % 4] = cx<float>{0.f, 0.f};
  stage(0, 0);
  int b = 0;
  for (int j0 = 0; j0 < n2; j0 += kGmKQ, b ^= 1) {
    if (j0 + kGmKQ < n2) {
      stage(b ^ 1, j0 + kGmKQ);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const cx<float>* rd = Rs + b * kGmTile * kGmLdQ + rl * kGmLdQ;
    const cx<float>* yd = Ys + b * kGmKQ * RP + 4 * sgi;
    const int nk = min(kGmKQ, n2 - j0);
#pragma unroll 4
    for (int q = g; q < nk; q += KG) {
      cx<float> y[4], v[4];
      lds_cx4(yd + q * RP, y);
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = rd[16 * c * kGmLdQ + q];
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int p = 0; p < 4; ++p) cfmac(acc[c][p], v[c], y[p]);
    }
    __syncthreads();
  }
  group_sum<KG>(acc, Rs, g, tid % NTG, NTG, false);
  if (g > 0) return;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int s = 4 * sgi + p;
    if (s >= r) break;
    cx<float>* o = Qout + ((size_t)k * r + s) * n1 + i0;
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (rl + 16 * c < nrow) o[rl + 16 * c] = acc[c][p];
  }
}

// ---- Q = R~ Y~^H with the lanes along the columns: grid (S, ceil(n1/32)), 256 threads.
// A warp forms 4 rows x 8 columns of Q, each lane summing the columns j = lane mod
// 32 in increasing order and the lanes added pairwise (distance 16, 8, .., 1): the
// order of k_qcon, bit for bit, at 12 loads for 32 complex products where k_qcon
// has 33 (529 x 96 x 112, r = 32: 53 -> 41 us).
constexpr int kQlRows = 4, kQlCols = 8;
template <int RP>
__global__ void __launch_bounds__(256, 2) k_qcon_l(Dev<float> d, cx<float>* __restrict__ Qout) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (converged(d)) return;
  constexpr int NS = RP / kQlCols, NR = 8 / NS;  // warps along s, along the rows
  const int k = blockIdx.x, n1 = d.n1, n2 = d.n2, r = d.r, S = d.S;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  cx<float>* Ys = reinterpret_cast<cx<float>*>(smem);  // [r][n2]
  const cx<float>* Y = d.Yt + (size_t)k * r * n2;
  for (int e = tid; e < r * n2; e += 256) cp_async_elem(Ys + e, Y + e);
  cp_async_wait_all();
  __syncthreads();
  const int s0 = (wid % NS) * kQlCols;
  if (s0 >= r) return;
  for (int ii = (wid / NS) * kQlRows; ii < 32; ii += NR * kQlRows) {
    const int i0 = blockIdx.y * 32 + ii;
    if (i0 >= n1) break;
    const cx<float>* row[kQlRows];
#pragma unroll
    for (int q = 0; q < kQlRows; ++q) row[q] = d.Rt + ((size_t)min(i0 + q, n1 - 1) * S + k) * n2;
    cx<float> acc[kQlRows][kQlCols], nx[kQlRows];
#pragma unroll
    for (int q = 0; q < kQlRows; ++q) {
      nx[q] = lane < n2 ? ldg_cx(row[q] + lane) : cx<float>{0.f, 0.f};
#pragma unroll
      for (int s = 0; s < kQlCols; ++s) acc[q][s] = cx<float>{0.f, 0.f};
    }
    for (int j = lane; j < n2; j += 32) {
      cx<float> v[kQlRows];
#pragma unroll
      for (int q = 0; q < kQlRows; ++q) {
        v[q] = nx[q];
        if (j + 32 < n2) nx[q] = ldg_cx(row[q] + j + 32);
      }
      const cx<float>* yj = Ys + s0 * n2 + j;
#pragma unroll
      for (int s = 0; s < kQlCols; ++s) {
        const cx<float> y = yj[min(s, r - 1 - s0) * n2];
#pragma unroll
        for (int q = 0; q < kQlRows; ++q) cfmac(acc[q][s], v[q], y);
      }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < kQlRows; ++q) {
      float f[2 * kQlCols];
#pragma unroll
      for (int s = 0; s < kQlCols; ++s) {
        f[2 * s] = acc[q][s].re;
        f[2 * s + 1] = acc[q][s].im;
      }
      const float tot = warp_reduce_scatter<float, 2 * kQlCols>(f);
      const int idx = lane >> 1, s = s0 + idx / 2;
      if ((lane & 1) == 0 && s < r && i0 + q < n1)
        reinterpret_cast<float*>(Qout + ((size_t)k * r + s) * n1 + i0 + q)[idx & 1] = tot;
    }
  }
}

// ---- Z~ = X~'Y~': grid (S, ceil(n1/64), ceil(n2/64)), 256 threads -------------------------------
constexpr int kGmZThreads = 256;
template <typename T>
inline size_t zsyn_f_smem(int r) {
  return 2 * (size_t)r * kGmTile * sizeof(cx<T>);
}

template <typename T>
__global__ void __launch_bounds__(kGmZThreads) k_zsyn_f(Dev<T> d) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (converged(d)) return;
  const int k = blockIdx.x, i0 = blockIdx.y * kGmTile, j0 = blockIdx.z * kGmTile;
  const int n1 = d.n1, n2 = d.n2, r = d.r, S = d.S, tid = threadIdx.x;
  cx<T>* Xs = reinterpret_cast<cx<T>*>(smem);  // [r][64]
  cx<T>* Ys = Xs + r * kGmTile;                    // [r][64]
  const int nrow = min(kGmTile, n1 - i0), ncol = min(kGmTile, n2 - j0);
  const cx<T>* Xb = d.Xt + (size_t)k * r * n1 + i0;
  const cx<T>* Yb = d.Yt + (size_t)k * r * n2 + j0;
  for (int e = tid; e < r * kGmTile; e += kGmZThreads) {
    const int s = e / kGmTile, c = e % kGmTile;
    if (c < nrow) cp_async_elem(Xs + e, Xb + (size_t)s * n1 + c);
    if (c < ncol) cp_async_elem(Ys + e, Yb + (size_t)s * n2 + c);
  }
  cp_async_wait_all();
  __syncthreads();
  const int tx = tid & 15, ty = tid >> 4;
  cx<T> acc[4][4];  // [row][column]
#pragma unroll
  for (int e = 0; e < 16; ++e) acc[e / 4][e % 4] = cx<T>{T(0), T(0)};
#pragma unroll 4
  for (int s = 0; s < r; ++s) {
    cx<T> x[4], y[4];
    lds_cx4(Xs + s * kGmTile + 4 * ty, x);
#pragma unroll
    for (int c = 0; c < 4; ++c) y[c] = Ys[s * kGmTile + tx + 16 * c];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int c = 0; c < 4; ++c) cfma(acc[p][c], x[p], y[c]);
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    if (4 * ty + p >= nrow) break;
    const size_t o = ((size_t)(i0 + 4 * ty + p) * S + k) * n2 + j0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int j = tx + 16 * c;
      if (j < ncol) {
        if (d.dZt) d.dZt[o + j] = acc[p][c] - d.Zt[o + j];  // for the stopping test
        d.Zt[o + j] = acc[p][c];
      }
    }
  }
}

// Sum of the ksplit partials of D (the differentiation form's X~^H R~), real
// slices from their pairs.
template <typename T>
__global__ void __launch_bounds__(256) k_dsum(Dev<T> d, cx<T>* __restrict__ out) {
  const int rn = d.r * d.n2, k = blockIdx.y;
  const bool real = k == 0 || 2 * k == d.n3;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < rn; e += gridDim.x * blockDim.x) {
    const cx<T>* p = d.Dpart + (size_t)k * d.ksplit * rn + e;
    cx<T> v = p[0];
    for (int z = 1; z < d.ksplit; ++z) {
      const cx<T> q = p[(size_t)z * rn];
      if (real) pair_add(v.re, v.im, q.re, q.im);
      else v = v + q;
    }
    if (real) v = cx<T>{v.re + v.im, T(0)};  // (value, rounding errors) pairs
    out[(size_t)k * rn + e] = v;
  }
}

}  // namespace tc
