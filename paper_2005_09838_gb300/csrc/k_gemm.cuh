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
template <int KG>
__device__ __forceinline__ void group_sum(cx<float> (&acc)[4][4], cx<float>* red, int g, int t, int nt) {
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
        for (int e = 0; e < 16; ++e) acc[e / 4][e % 4] = acc[e / 4][e % 4] + red[((q - 1) * 16 + e) * nt + t];
  }
}

// ---- D = X~'^H R~: grid (S, ceil(n2/64), ksplit), partial sums over ranges of n1 ------------
template <int RP>
__host__ __device__ constexpr size_t dcon_f_smem() {
  return 2 * (size_t)kGmKC * (kGmTile + RP) * sizeof(cx<float>);
}

template <int RP>
__global__ void __launch_bounds__(kGmThreads) k_dcon_f(Dev<float> d) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (converged(d)) return;
  constexpr int SG = GmGroups<RP>::SG, KG = GmGroups<RP>::KG, NTG = 16 * SG;
  const int k = blockIdx.x, j0 = blockIdx.y * kGmTile, z = blockIdx.z, ks = gridDim.z;
  const int n1 = d.n1, n2 = d.n2, r = d.r, S = d.S, tid = threadIdx.x;
  const int per = (n1 + ks - 1) / ks, ib = min(z * per, n1), ie = min(ib + per, n1);
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
  auto stage = [&](int b, int i0) {
    const int nk = min(kGmKC, ie - i0);
    cx<float>* rd = Rs + b * kGmKC * kGmTile;
    cx<float>* xd = Xs + b * kGmKC * RP;
    if (vec) {
      for (int e = tid; e < nk * (kGmTile / 2); e += kGmThreads) {
        const int q = e / (kGmTile / 2), c = 2 * (e % (kGmTile / 2));
        if (c < ncol) cp_async16(rd + q * kGmTile + c, Rb + (size_t)(i0 + q) * rs + c);
      }
    } else {
      for (int e = tid; e < nk * kGmTile; e += kGmThreads) {
        const int q = e / kGmTile, c = e % kGmTile;
        if (c < ncol) cp_async_elem(rd + q * kGmTile + c, Rb + (size_t)(i0 + q) * rs + c);
      }
    }
    for (int e = tid; e < r * kGmKC; e += kGmThreads) {
      const int s = e / kGmKC, q = e % kGmKC;
      if (q < nk) cp_async_elem(xd + q * RP + s, Xb + (size_t)s * n1 + i0 + q);
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
    const int nk = min(kGmKC, ie - i0);
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
    __syncthreads();
  }
  group_sum<KG>(acc, Rs, g, tid % NTG, NTG);
  if (g > 0) return;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int s = 4 * sgi + p;
    if (s >= r) break;
    cx<float>* o = d.Dpart + (((size_t)k * ks + z) * r + s) * n2 + j0;
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (cl + 16 * c < ncol) o[cl + 16 * c] = acc[c][p];
  }
}

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
  group_sum<KG>(acc, Rs, g, tid % NTG, NTG);
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
// slices with a zero imaginary part.
template <typename T>
__global__ void __launch_bounds__(256) k_dsum(Dev<T> d, cx<T>* __restrict__ out) {
  const int rn = d.r * d.n2, k = blockIdx.y;
  const bool real = k == 0 || 2 * k == d.n3;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < rn; e += gridDim.x * blockDim.x) {
    const cx<T>* p = d.Dpart + (size_t)k * d.ksplit * rn + e;
    cx<T> v = p[0];
    for (int z = 1; z < d.ksplit; ++z) v = v + p[(size_t)z * rn];
    if (real) v.im = T(0);
    out[(size_t)k * rn + e] = v;
  }
}

}  // namespace tc
