// Differentiation form: the adjoint of the masked t-product loss of the factor
// model,
//   L(X, Y) = 1/2 ||P_Omega(X*Y - G)||_F^2 + rho1/2 ||H unfold(X*Y, 1)||_F^2
// (the factor terms of f0, Eq. (TETP-optim), with W held at G on the mask).
// With E = P_Omega(Z - G) + rho1 (H^T H) x_1 Z, Z = X*Y, the gradients are the
// t-products dL/dX = E * Y^* and dL/dY = X^* * E (conjugate transpose of
// Sec. 2), i.e. per slice of the half spectrum
//   dL/dX~_k = E~_k Y~_k^H,  dL/dY~_k = X~_k^H E~_k,
// E~_k = R~_k + rho1 H^T H Z~_k with R~ = DFT(P_Omega(Z - G)) from the slab
// kernel (MODE_GRAD) and the rho1 part added in place by k_grad_rho1; the
// inverse mode-3 DFT brings the gradients back to the spatial factors.  FP32 ranks above 4 take the tiled
// contractions of k_gemm.cuh, the others those below.
#pragma once

namespace tc {

// D = X~^H R~ per slice (r x n2), over a tile of 32 columns: grid
// (S, ceil(n2/32)); warp w accumulates rows i = w, w + 8, ...
template <typename T, int RP>
__global__ void __launch_bounds__(kYThreads) k_dcon(Dev<T> d, cx<T>* __restrict__ Dout) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int k = blockIdx.x;
  const int j0 = blockIdx.y * 32;
  const int n1 = d.n1, n2 = d.n2, r = d.r, S = d.S;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  cx<T>* red = reinterpret_cast<cx<T>*>(smem);  // [nw][RP][32]
  const cx<T>* Xg = d.Xt + (size_t)k * r * n1;
  const cx<T>* Xs = Xg;                         // [r][n1], staged when it fits
  if (!d.yx_global) {
    cx<T>* xs = red + nw * RP * 32;
    for (int e = tid; e < r * n1; e += blockDim.x) xs[e] = Xg[e];
    Xs = xs;
  }
  __syncthreads();
  const int j = j0 + lane;
  cx<T> acc[RP];
#pragma unroll
  for (int s = 0; s < RP; ++s) acc[s] = cx<T>{T(0), T(0)};
  if (j < n2) {
    int i = wid;
    for (; i + 3 * nw < n1; i += 4 * nw) {
      cx<T> v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = ldg_cx(d.Rt + ((size_t)(i + q * nw) * S + k) * n2 + j);
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int s = 0; s < RP; ++s)
          if (s < r) cfmaconj(acc[s], Xs[(size_t)s * n1 + i + q * nw], v[q]);
    }
    for (; i < n1; i += nw) {
      const cx<T> v = ldg_cx(d.Rt + ((size_t)i * S + k) * n2 + j);
#pragma unroll
      for (int s = 0; s < RP; ++s)
        if (s < r) cfmaconj(acc[s], Xs[(size_t)s * n1 + i], v);
    }
  }
#pragma unroll
  for (int s = 0; s < RP; ++s) red[(wid * RP + s) * 32 + lane] = acc[s];
  __syncthreads();
  const bool realslice = (k == 0) || (2 * k == d.n3);
  for (int e = tid; e < r * 32; e += blockDim.x) {
    const int s = e >> 5, c = e & 31;
    if (j0 + c >= n2) continue;
    cx<T> v = {T(0), T(0)};
    for (int w = 0; w < nw; ++w) v = v + red[(w * RP + s) * 32 + c];
    if (realslice) v.im = T(0);
    Dout[((size_t)k * r + s) * n2 + j0 + c] = v;
  }
}

template <typename T>
__host__ inline size_t dcon_smem_bytes(int n1, int r, int rp, bool x_in_smem = true) {
  return ((size_t)(kYThreads / 32) * rp * 32 + (x_in_smem ? (size_t)r * n1 : 0)) * sizeof(cx<T>);
}

// rho1 terms in one pass over Z~: R~ += rho1 H^T H Z~ (with WRITE), so that the
// contractions R~Y~^H and X~^H R~ that follow give the whole gradient, and the
// sum ||H Z~_k||^2 of the loss (part_k, as k_rho1_term).  (H^T H z)_i = deg_i z_i
// - z_{i-1} - z_{i+1} along mode 1.  Grid (S, kRhoChunks): a thread walks down
// one column of its chunk of rows with the row above and below in registers, so
// Z~ is read once and R~ once and written once (312 MB at 529 x 288 x 168; as two
// kernels, one of them a thread per entry reading three rows, 31 + 70 us).
template <typename T, bool WRITE>
__global__ void __launch_bounds__(256) k_grad_rho1(Dev<T> d) {
  __shared__ double part[8];
  const int k = blockIdx.x, ch = blockIdx.y;
  const int n1 = d.n1, n2 = d.n2;
  const size_t rs = (size_t)d.S * n2;
  const cx<T>* Z = d.Zt + (size_t)k * n2;
  cx<T>* R = d.Rt + (size_t)k * n2;
  const bool real = k == 0 || 2 * k == d.n3;
  const T rho1 = d.rho1;
  const int per = (n1 + kRhoChunks - 1) / kRhoChunks, i0 = min(ch * per, n1), i1 = min(i0 + per, n1);
  T s = T(0), c = T(0);  // (dot2, as in k_rho1_term)
  constexpr int U = 4;  // rows in flight
  for (int j = threadIdx.x; j < n2 && i0 < i1; j += blockDim.x) {
    cx<T> cur = Z[(size_t)i0 * rs + j];
    cx<T> up = {T(0), T(0)};  // z_i - z_{i-1}
    if (i0 > 0) up = cur - Z[(size_t)(i0 - 1) * rs + j];
    for (int i = i0; i < i1; i += U) {
      cx<T> nx[U], rv[U];
#pragma unroll
      for (int q = 0; q < U; ++q) {
        if (i + q < i1 && i + q + 1 < n1) nx[q] = Z[(size_t)(i + q + 1) * rs + j];
        if (WRITE && i + q < i1) rv[q] = R[(size_t)(i + q) * rs + j];
      }
#pragma unroll
      for (int q = 0; q < U; ++q) {
        if (i + q >= i1) break;
        cx<T> dn = {T(0), T(0)};  // z_{i+1} - z_i
        if (i + q + 1 < n1) {
          dn = nx[q] - cur;
          dot2(s, c, dn.re, dn.re);
          dot2(s, c, dn.im, dn.im);
        }
        if (WRITE) {
          const cx<T> h = up - dn;
          R[(size_t)(i + q) * rs + j] = cx<T>{fma(h.re, rho1, rv[q].re), real ? T(0) : fma(h.im, rho1, rv[q].im)};
        }
        up = dn;
        cur = nx[q];
      }
    }
  }
  const double tot = warp_sum((double)s + (double)c);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) part[wid] = tot;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += part[w];
    d.part_k[(size_t)k * kRhoChunks + ch] = sum;
  }
}

}  // namespace tc
