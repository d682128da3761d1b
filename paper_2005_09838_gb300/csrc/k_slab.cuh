// Slab kernel of the TCTF2R iteration: one CTA per mode-1 index i1 (one OD
// pair).  The spatial slab (i1, :, :) lives in shared memory, tube-major with
// an odd stride (conflict-free for tube-per-thread and row-per-thread access).
//
//   phase A  inverse mode-3 DFT (Eq. (barAAk)) of every tube of Z~ = X~Y~
//            (step 3; the half spectrum is written by the Y-step kernel);
//            the slab receives v = G on the mask and Z elsewhere
//   phase B  W-step of every row (i1, :, i3) (step 4, Eq. (subquKKT))
//   phase C  forward mode-3 DFT of every tube of W (step 7, Eq. (bar BA-k));
//            the residual spectrum R~ = W~ - Z~ is stored
#pragma once

namespace tc {

enum SlabMode : int { MODE_ITER = 0, MODE_W = 1, MODE_R = 2, MODE_GRAD = 3 };

// Launch flags of the slab kernels: the slab lives in shared memory (else in
// d.scratch; k_slab only), and MODE_W writes Wout in the row-major order
// [i1][i3][i2] (one CTA then writes whole rows; k_unpack brings it to the
// caller's column-major order; not k_slab) instead of the column-major one.
// SLAB_NOSUM: MODE_W forms no sums.
enum SlabFlag : int { SLAB_IN_SMEM = 1, SLAB_WROWS = 2, SLAB_NOSUM = 4 };

// Threads per CTA.
constexpr int kSlabThreads = 256;
// Rows (inverse) or slices (forward) per item of the generic transform by
// default; every tile gives the same sums in the same order, and tc_init times
// 2 and 4 where this kernel runs the iteration.  It runs where k_slab_g does
// not hold the slab in shared memory, and for TC_BF16: the split operands of
// its contractions keep 16 bits, so any other rounding of the transform
// comes back as other BF16 rounding errors in the factors (3e-5 of Y~ after
// five iterations on 435 x 205 x 34, r = 28, as large as the form's error).
constexpr int kTL = 4;

// Odd stride between tubes in the slab (n3 values per tube).
__host__ __device__ inline int slab_stride(int n3) { return n3 | 1; }

struct SlabLayout {
  size_t wtab, red, msk, stw, tw, spec, spat, total;  // byte offsets and total shared bytes
  size_t slab_bytes;                         // bytes of the slab buffers per CTA
};

template <typename T>
__host__ __device__ inline SlabLayout slab_layout(int n2, int n3, bool slabs_in_smem) {
  SlabLayout L{};
  const int S = n3 / 2 + 1;
  size_t off = 0;
  L.wtab = off;
  off = align_up(off + sizeof(T) * 6 * n2, 16);
  L.red = off;
  off = align_up(off + sizeof(double) * 4 * 32, 16);
  L.msk = off;  // row-major mask bits: [n3][ceil(n2/32)]
  off = align_up(off + sizeof(uint32_t) * (size_t)n3 * ((n2 + 31) / 32), 16);
  L.stw = off;  // per row and mask word: start of the run of missing entries entering the word
  off = align_up(off + sizeof(int) * (size_t)n3 * ((n2 + 31) / 32), 16);
  L.tw = off;  // generic transform: the n3 twiddles exp(-2 pi i m / n3)
  off = align_up(off + sizeof(cx<T>) * (size_t)n3, 16);
  const size_t spec_bytes = align_up(sizeof(cx<T>) * (size_t)S * n2, 16);
  const size_t spat_bytes = align_up(sizeof(T) * (size_t)n2 * slab_stride(n3), 16);
  L.slab_bytes = spec_bytes + spat_bytes;
  if (slabs_in_smem) {
    L.spec = off;
    L.spat = off + spec_bytes;
    off += spec_bytes + spat_bytes;
  } else {
    L.spec = 0;
    L.spat = spec_bytes;
  }
  L.total = off;
  return L;
}

// ---------------------------------------------------------------------------
// W-step of one row (i1, :, i3) (Eq. (subquKKT), Eq. (Wkiom)).
//
// For a missing j, (W K_{mu rho2})_j = Z_j with K_{mu rho2} = (1+mu) I +
// rho2 K^T K (tridiagonal); W_j = G_j on the mask (identity rows).  On entry
// the row holds v_j = G_j on the mask and Z_j elsewhere; the observed
// neighbours of a missing entry enter through the elimination itself.  The
// LU pivots of a run of missing entries depend only on the position p in the
// run, on whether the run starts at j = 0 and on whether j is the last entry
// of the row (the first and last entries have one neighbour), so their
// inverses come from a table and each sweep is a single fused multiply-add
// chain:
//   forward   d_j = a_j d_{j-1} + b_j,   a_j = rho2 inv_j,  b_j = v_j inv_j
//   backward  w_j = c_j w_{j+1} + d_j,   c_j = rho2 inv_j (0 at j = n2-1)
// with a_j = c_j = 0, b_j = v_j at observed entries.  On return the row
// holds W.  row[j] is at col[j * LP].  The row is processed one mask word
// (32 entries) at a time: the entries are read into registers first and the
// table indices come from the mask bits, so only the multiply-add chain stays
// on the critical path.  The run start entering each word is saved by the
// forward sweep for the backward one.
//
// wtab: [6][n2] inv1, inv0 (runs starting at j = 0 / j > 0), c1 = rho2 inv1,
//       c0 = rho2 inv0, e1, e0 (inverse pivot when the run ends at j = n2-1)
// rowm: the row's mask bits along j (word j / 32, bit j % 32)
// rowst: per-word run starts (written here)
// ---------------------------------------------------------------------------
// Fills the [6][n2] W-step table of wstep_sweeps in FP64, rounded to T.
// Pivots of a run of missing entries by position p: the first has diagonal
// 1 + mu + rho2 (run at j = 0, one neighbour) or 1 + mu + 2 rho2; each later
// one subtracts rho2^2 times the previous inverse pivot; at j = n2 - 1 the
// diagonal loses one rho2 (one neighbour).
template <typename T>
__host__ __device__ inline void wstep_tables(T* w, int n2, double mu, double rho2) {
  const double first[2] = {1.0 + mu + rho2 * (n2 > 1 ? 1.0 : 0.0), 1.0 + mu + 2.0 * rho2};
  const double last[2] = {first[0], 1.0 + mu + rho2};
  for (int b = 0; b < 2; ++b) {  // b = 0: run starting at j = 0; b = 1: j > 0
    double prev = 0.0;
    for (int q = 0; q < n2; ++q) {
      const double sub = (q > 0) ? rho2 * rho2 * prev : 0.0;
      const double inv = 1.0 / (((q > 0) ? 1.0 + mu + 2.0 * rho2 : first[b]) - sub);
      const double inv_last = 1.0 / (last[b] - sub);
      w[(size_t)b * n2 + q] = (T)inv;
      w[(size_t)(2 + b) * n2 + q] = (T)(rho2 * inv);
      w[(size_t)(4 + b) * n2 + q] = (T)inv_last;
      prev = inv;
    }
  }
}

// Excess ratios of the same pivots, h = 1 - rho2 inv = g / (rho2 + g) with the
// excess g = 1 / inv - rho2 of a pivot, [2][n2] by position in the run (run start
// as in wstep_tables).  g follows g_q = 1 + mu + rho2 g_{q-1} / (rho2 + g_{q-1}):
// no subtraction, so h keeps its digits however close to 1 rho2 inv is.
template <typename T>
__host__ __device__ inline void wstep_excess(T* h, int n2, double mu, double rho2) {
  const double first[2] = {1.0 + mu, 1.0 + mu + rho2};
  for (int b = 0; b < 2; ++b) {
    double prev = 0.0;
    for (int q = 0; q < n2; ++q) {
      const double g = (q > 0) ? 1.0 + mu + rho2 * prev : first[b];
      prev = g / (rho2 + g);
      h[(size_t)b * n2 + q] = (T)prev;
    }
  }
}

// One mask word (32 entries, fewer in the last word) of the forward sweep.
// The table index of entry j is inv-table + (j - rs), rs the start of the run
// holding j: from the mask bits below j (rs = 32 w + 32 - clz(below)) or,
// when there are none in this word, the run start st_w entering the word, so
// every index is known without the recurrence; the recurrence itself is one
// fused multiply-add per entry (a_j = 0, b_j = v_j at observed entries).
// LAST: the word holds j = n2 - 1 (the e-table pivot there).
template <typename T, bool FULL, bool LAST>
__device__ __forceinline__ void wstep_fwd_word(T* __restrict__ col, int LP, uint32_t mw, int w, int qn, int st_w,
                                               int n2, T rho2, const T* __restrict__ wtab, T& d) {
  const int base = 32 * w;
  const int cw = ((st_w == 0) ? 0 : n2) + base - st_w;  // index base of entries without bits below
  T v[32];
#pragma unroll
  for (int q = 0; q < 32; ++q)
    if (FULL || q < qn) v[q] = col[(base + q) * LP];
#pragma unroll
  for (int q = 0; q < 32; ++q) {
    if (FULL || q < qn) {
      const bool ob = (mw >> q) & 1u;
      const uint32_t below = mw & ((1u << q) - 1u);
      int idx = below ? (n2 - 32 + q + __clz(below)) : (cw + q);
      if (LAST && base + q == n2 - 1) idx += 4 * n2;
      const T inv = wtab[idx];
      d = fma(ob ? T(0) : rho2 * inv, d, ob ? v[q] : v[q] * inv);
      v[q] = d;
    }
  }
#pragma unroll
  for (int q = 0; q < 32; ++q)
    if (FULL || q < qn) col[(base + q) * LP] = v[q];
}

// One mask word of the backward sweep: c_j = rho2 inv_j at table index
// 2 n2 + (forward index), 0 at observed entries and at j = n2 - 1 (observed
// slots already hold G).
template <typename T, bool FULL, bool LAST>
__device__ __forceinline__ void wstep_bwd_word(T* __restrict__ col, int LP, uint32_t mw, int w, int qn, int st_w,
                                               int n2, const T* __restrict__ wtab, T& wn) {
  const int base = 32 * w;
  const int cw = ((st_w == 0) ? 2 * n2 : 3 * n2) + base - st_w;
  T v[32];
#pragma unroll
  for (int q = 0; q < 32; ++q)
    if (FULL || q < qn) v[q] = col[(base + q) * LP];
#pragma unroll
  for (int q = 31; q >= 0; --q) {
    if (FULL || q < qn) {
      const bool ob = (mw >> q) & 1u;
      const uint32_t below = mw & ((1u << q) - 1u);
      const int idx = below ? (3 * n2 - 32 + q + __clz(below)) : (cw + q);
      const T c = wtab[idx];
      const bool zero = ob || (LAST && base + q == n2 - 1);
      wn = fma(zero ? T(0) : c, wn, v[q]);
      v[q] = wn;
    }
  }
#pragma unroll
  for (int q = 0; q < 32; ++q)
    if (FULL || q < qn) col[(base + q) * LP] = v[q];
}

template <typename T>
__device__ void wstep_sweeps(T* __restrict__ col, int LP, const uint32_t* __restrict__ rowm, int* __restrict__ rowst,
                             int n2, T rho2, const T* __restrict__ wtab) {
  const int words = (n2 + 31) >> 5;
  const int ql = n2 - 32 * (words - 1);  // entries in the last word
  // ---- forward: d_j = a_j d_{j-1} + b_j --------------------------------------
  T d = T(0);
  int st = 0;  // start of the run of missing entries entering the word
  for (int w = 0; w < words - 1; ++w) {
    const uint32_t mw = rowm[w];
    rowst[w] = st;
    wstep_fwd_word<T, true, false>(col, LP, mw, w, 32, st, n2, rho2, wtab, d);
    if (mw) st = 32 * w + 32 - __clz(mw);
  }
  {
    const int w = words - 1;
    rowst[w] = st;
    if (ql == 32) wstep_fwd_word<T, true, true>(col, LP, rowm[w], w, 32, st, n2, rho2, wtab, d);
    else wstep_fwd_word<T, false, true>(col, LP, rowm[w], w, ql, st, n2, rho2, wtab, d);
  }
  // ---- backward: w_j = c_j w_{j+1} + d_j ---------------------------------------
  T wn = T(0);
  {
    const int w = words - 1;
    if (ql == 32) wstep_bwd_word<T, true, true>(col, LP, rowm[w], w, 32, rowst[w], n2, wtab, wn);
    else wstep_bwd_word<T, false, true>(col, LP, rowm[w], w, ql, rowst[w], n2, wtab, wn);
  }
  for (int w = words - 2; w >= 0; --w)
    wstep_bwd_word<T, true, false>(col, LP, rowm[w], w, 32, rowst[w], n2, wtab, wn);
}

// ---------------------------------------------------------------------------
// The same W-step with each row split into nseg segments of whole mask words,
// one thread per (row, segment): a block-wide call that takes three barriers.
// Both recurrences restart at every observed entry (there a_j = 0 and c_j = 0:
// the value is G), and the backward one also at j = n2 - 1.  So the value
// entering a segment follows from the entries between the last restart and
// the segment boundary, and each thread recomputes it with the very operations
// the sequential sweep would apply (results are bit-identical to
// wstep_sweeps): forward, from the last observed entry before the segment (or
// j = 0); backward, from the first observed entry at or after the segment's
// end (or j = n2 - 1).  The carries are formed before the values they read
// are overwritten.
//   item: this thread's (row, segment) index, row = item % nrows, segment =
//         item / nrows; items >= nrows * nseg only join the barriers
//   col(l): the row's first entry; rows are strided by LP along j
// SEQ: a row with a run of missing words over more than half of it is left to
// its first thread and the sequential sweeps: the carries of its segments walk the
// run at twice their cost per entry (slab kernel with a tenth of the rows missing:
// 32 x 2000 x 12 FP64 1046 -> 713 us, 702 with all rows sequential; 150 x 205 x 34
// BF16 61 -> 55; with 85 registers to a thread the sweeps spill: 435 x 205 x 34
// 108 -> 115, so not there).
// ---------------------------------------------------------------------------
template <typename T, bool SEQ, typename ColFn>
__device__ void wstep_sweeps_seg(ColFn col_of, int LP, const uint32_t* __restrict__ msk, int* __restrict__ stw,
                                 int nrows, int nseg, int item, int n2, T rho2, const T* __restrict__ wtab) {
  const int words = (n2 + 31) >> 5;
  const int ql = n2 - 32 * (words - 1);  // entries in the last word
  const int wps = (words + nseg - 1) / nseg;
  const bool active = item < nrows * nseg;
  const int l = active ? item % nrows : 0, sg = active ? item / nrows : 0;
  const int w0 = min(sg * wps, words), w1 = min(w0 + wps, words);
  T* col = col_of(l);
  const uint32_t* rowm = msk + (size_t)l * ((n2 + 31) >> 5);
  int* rowst = stw + (size_t)l * ((n2 + 31) >> 5);
  bool seq = false;
  if (SEQ && nseg > 1 && active) {
    for (int w = 0, run = 0; w < words; ++w) {
      run = rowm[w] ? 0 : run + 1;
      seq |= 2 * run > words;
    }
    if (seq && sg == 0) wstep_sweeps<T>(col, LP, rowm, rowst, n2, rho2, wtab);
  }
  const bool work = active && w0 < w1 && !seq;
  auto bit = [&](int j) { return (rowm[j >> 5] >> (j & 31)) & 1u; };

  // ---- forward carry: d_{j0 - 1} and the run start entering word w0 -------------------
  T d = T(0);
  int st = 0;
  if (work && w0 > 0) {
    for (int w = w0 - 1; w >= 0; --w) {
      const uint32_t mw = rowm[w];
      if (mw) {
        st = 32 * w + 32 - __clz(mw);
        break;
      }
    }
    const int j0 = 32 * w0;
    if (st > 0) d = col[(size_t)(st - 1) * LP];  // observed: the recurrence restarts at G
    for (int j = st; j < j0; ++j) {             // the run of missing entries up to the boundary
      const T inv = wtab[((st == 0) ? 0 : n2) + (j - st)];
      d = fma(rho2 * inv, d, col[(size_t)j * LP] * inv);
    }
  }
  __syncthreads();
  // ---- forward sweep of the segment -----------------------------------------------------
  if (work) {
    for (int w = w0; w < w1; ++w) {
      const uint32_t mw = rowm[w];
      rowst[w] = st;
      if (w < words - 1) wstep_fwd_word<T, true, false>(col, LP, mw, w, 32, st, n2, rho2, wtab, d);
      else if (ql == 32) wstep_fwd_word<T, true, true>(col, LP, mw, w, 32, st, n2, rho2, wtab, d);
      else wstep_fwd_word<T, false, true>(col, LP, mw, w, ql, st, n2, rho2, wtab, d);
      if (mw) st = 32 * w + 32 - __clz(mw);
    }
  }
  __syncthreads();
  // ---- backward carry: w_{j1}, j1 = 32 w1, from the first restart at or after it --------
  T wn = T(0);
  if (work && w1 < words) {
    const int j1 = 32 * w1;
    int k = j1;
    while (k < n2 - 1 && !bit(k)) ++k;
    wn = col[(size_t)k * LP];  // w_k = d_k at a restart
    for (int j = k - 1; j >= j1; --j) {
      const int w = j >> 5, q = j & 31;
      const uint32_t below = rowm[w] & ((1u << q) - 1u);
      const int rs = below ? 32 * w + 32 - __clz(below) : rowst[w];
      const T c = wtab[2 * n2 + ((rs == 0) ? 0 : n2) + (j - rs)];
      wn = fma(c, wn, col[(size_t)j * LP]);
    }
  }
  __syncthreads();
  // ---- backward sweep of the segment ----------------------------------------------------
  if (work) {
    for (int w = w1 - 1; w >= w0; --w) {
      if (w < words - 1) wstep_bwd_word<T, true, false>(col, LP, rowm[w], w, 32, rowst[w], n2, wtab, wn);
      else if (ql == 32) wstep_bwd_word<T, true, true>(col, LP, rowm[w], w, 32, rowst[w], n2, wtab, wn);
      else wstep_bwd_word<T, false, true>(col, LP, rowm[w], w, ql, rowst[w], n2, wtab, wn);
    }
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// W-step with every segment of a row (kWSeg entries, fewer in the last one) solved
// on its own by one thread, from the slab's values v (G on the mask, Z elsewhere)
// as they were before any segment was solved; the caller stores the results once
// all segments of the row have read.  Inside the segment the sweeps are those of
// wstep_sweeps, with the values and the backward coefficients in registers.
//   Left:  d_{base-1} of a run that enters the segment, by the forward
//          recurrence from the run's start.
//   Right: a run that goes on past the segment is eliminated from its other end,
//          w_j = e w_{j-1} + f (pivots by the distance from that end: the same
//          table), so the segment's last entry is (d + c f) / (1 - c e).  c and
//          e tend to 1 as rho2 grows, so from c e = 1/2 on 1 - c e is formed from the
//          excess ratios of the two pivots, h_c + c h_e: the difference loses the digits
//          (FP32, a row of 100 missing entries, mu = 1e-3: 6e-4 of W at rho2 = 1e6
//          and 3e-2 at 1e8, against 2e-7 and 4e-7 of the sequential sweeps).
// Both walk the run's entries, a few for scattered observations.  In a run of
// kWLong entries or more (a row or day without data) every segment that lies in
// it whole first leaves its part of the two recurrences, d -> a d + b, in its own
// slots of the slab (its values are in registers), and the walks take a segment
// per step: a row of n2 missing entries costs each of its threads some n2 / kWSeg
// steps, where walking the entries cost them n2 (slab kernel with a tenth of the
// rows missing: 60 x 144 x 30 FP64 194 -> 92 us, 32 x 3000 x 10 FP32 272 -> 84; with
// none 70 and 48).
// The further barrier, the values held across it and the excess ratios are the
// GENERAL form, 5% of the slab kernel where no run is long.  The engine takes it
// where rho2 asks for it (wstep_strong) or at least a quarter of the slabs have a
// run of kWChoice entries, which masks with 10% or more observed at random don't
// (FP32; FP64, where a step is the dearer, has it earlier).
// Fewer than half the instructions of the two sweeps over shared memory (no
// second pass over the values, the table and the mask).  FP32 segments of 16 keep
// the thread within 64 registers; in FP64, where a warp instruction holds its scheduler's pipe for
// 60 clocks however few lanes take part, shorter ones fill the lanes (121 x 144 x 7:
// 7 rows are 7 lanes as rows, 126 as segments of 8).
// ---------------------------------------------------------------------------
template <typename T>
constexpr int kWSeg = sizeof(T) == 8 ? 8 : 16;
template <typename T>
constexpr int kWLong = 4 * kWSeg<T>;
template <typename T>
constexpr int kWChoice = sizeof(T) == 8 ? 64 : 192;

// Start of the run of missing entries that reaches entry `base` from the left, and
// end (one past its last entry) of the one that reaches entry j1 - 1 from the right.
__device__ __forceinline__ int run_start(const uint32_t* __restrict__ rowm, int base, uint32_t word) {
  int u = base >> 5;  // (word = rowm[u])
  uint32_t m = word & ((1u << (base & 31)) - 1u);
  while (m == 0u && u > 0) m = rowm[--u];
  return m ? 32 * u + 32 - __clz(m) : 0;
}
__device__ __forceinline__ int run_end(const uint32_t* __restrict__ rowm, int words, int j1, int n2) {
  int u = j1 >> 5;
  uint32_t m = rowm[u] & (0xffffffffu << (j1 & 31));
  while (m == 0u && u + 1 < words) m = rowm[++u];
  return m ? 32 * u + __ffs(m) - 1 : n2;
}

// A whole segment inside a long run: the forward recurrence over it as d -> a d + b
// in its first two slots, the one from the run's other end in the next two.
template <typename T, int SEG>
__device__ __forceinline__ void wstep_publish(T* __restrict__ col, int LP, int base, int st, int k, int n2, T rho2,
                                              const T* __restrict__ wtab, const T (&v)[SEG]) {
  const T* tf = wtab + (st == 0 ? 0 : n2) + base - st;
  const T* tr = wtab + (k < n2 ? n2 : 0) + k - 1 - base;
  T a = T(1), b = T(0), e = T(1), f = T(0);
#pragma unroll
  for (int q = 0; q < SEG; ++q) {
    const T inv = tf[q], c = rho2 * inv;
    a *= c;
    b = fma(c, b, v[q] * inv);
  }
#pragma unroll
  for (int q = SEG - 1; q >= 0; --q) {
    const T inv = tr[-q], c = rho2 * inv;
    e *= c;
    f = fma(c, f, v[q] * inv);
  }
  T* o = col + base * LP;
  o[0] = a;
  o[LP] = b;
  o[2 * LP] = e;
  o[3 * LP] = f;
}

// Whether c e can reach 1/2: the largest coefficient is that of a run's first entry
// at the row's start, rho2 / (1 + mu + rho2), whose square is below 4/9 up to here.
inline bool wstep_strong(double mu, double rho2) { return rho2 > 2.0 * (1.0 + mu); }
// GENERAL: the whole segments of long runs have published theirs; any rho2.
template <typename T, int SEG, bool FULL, bool LAST, bool GENERAL>
__device__ __forceinline__ void wstep_segment(const T* __restrict__ col, int LP, const uint32_t* __restrict__ rowm,
                                              int words, int segs, int sgm, int qn, int n2, T rho2,
                                              const T* __restrict__ wtab, const T* __restrict__ hex, T (&v)[SEG]) {
  const int base = SEG * sgm, j1 = base + SEG;
  const uint32_t word = rowm[base >> 5], mw = word >> (base & 31);
  const uint32_t mb = mw & ((1u << SEG) - 1u);  // (bits past n2 are 0)
  int st = 0;  // start of the run of missing entries that enters the segment
  T d = T(0);
  if (base > 0) {
    st = run_start(rowm, base, word);
    if (!(mw & 1u)) {
      if (st > 0) d = col[(st - 1) * LP];
      const T* tb = wtab + (st == 0 ? 0 : n2);
      int jf = base;  // entries up to here, then segments
      if (GENERAL && base - st >= SEG) {
        const int k = mb ? base + __ffs(mb) - 1 : (LAST ? n2 : run_end(rowm, words, j1, n2));
        if (k - st >= kWLong<T>) jf = (st + SEG - 1) / SEG * SEG;
      }
      for (int j = st; j < jf; ++j) {
        const T inv = tb[j - st];
        d = fma(rho2 * inv, d, col[j * LP] * inv);
      }
      if (GENERAL)
        for (int j = jf; j < base; j += SEG) d = fma(col[j * LP], d, col[(j + 1) * LP]);
    }
  }
  // table position of the entry: one further per missing entry, the start of the
  // second table after an observed one
  const T* tp = wtab + ((st == 0) ? 0 : n2) + base - st;
  const T* const t1 = wtab + n2;
  T c[SEG];
#pragma unroll
  for (int q = 0; q < SEG; ++q) {
    if (FULL || q < qn) {
      const bool ob = (mw >> q) & 1u;
      const bool end = LAST && base + q == n2 - 1;
      const T inv = end ? tp[4 * n2] : *tp;
      // rho2 inv from its table in FP64, whose pipe is the scarce one
      const T a = (sizeof(T) == 8 && !end) ? tp[2 * n2] : rho2 * inv;
      d = fma(ob ? T(0) : a, d, ob ? v[q] : v[q] * inv);
      v[q] = d;
      c[q] = (ob || end) ? T(0) : a;
      tp = ob ? t1 : tp + 1;
    }
  }
  T wn = T(0);
  if (!LAST && !((mw >> (SEG - 1)) & 1u)) {
    const int k = run_end(rowm, words, j1, n2);  // next observed entry, or the row's end
    T x = (k < n2) ? col[k * LP] : T(0), e = T(0);
    const int tb = k < n2 ? n2 : 0;
    int jl = j1;  // entries down to here, then segments
    if (GENERAL && k - j1 >= SEG) {
      const int s0 = mb ? base + 32 - __clz(mb) : st;
      if (k - s0 >= kWLong<T>) jl = max(j1, min(k / SEG, segs - 1) * SEG);
    }
    for (int j = k - 1; j >= jl; --j) {
      const T inv = wtab[tb + k - 1 - j];
      e = rho2 * inv;
      x = fma(e, x, col[j * LP] * inv);
    }
    if (GENERAL)
      for (int j = jl - SEG; j >= j1; j -= SEG) x = fma(col[(j + 2) * LP], x, col[(j + 3) * LP]);
    wn = fma(c[SEG - 1], x, v[SEG - 1]);
    if (k > j1) {
      const int p1 = tb + k - 1 - j1;
      if (GENERAL) e = rho2 * wtab[p1];
      const T ce = c[SEG - 1] * e;
      // (tp is one past the position of the segment's last entry)
      wn *= rcp_refined(!GENERAL || ce < T(0.5) ? fma(-c[SEG - 1], e, T(1))
                                                : fma(c[SEG - 1], hex[p1], hex[tp - 1 - wtab]));
    }
    v[SEG - 1] = wn;
    c[SEG - 1] = T(0);
  }
#pragma unroll
  for (int q = SEG - 1; q >= 0; --q)
    if (FULL || q < qn) {
      wn = fma(c[q], wn, v[q]);
      v[q] = wn;
    }
}

// W-step of every row of the slab: a thread per (row, segment), as many whole
// rows at a time as the block has threads for; rows at col_of(q) (stride LP
// along j), their mask words at msk + q words; hex: [2][n2] excess ratios
// (wstep_excess; read in the GENERAL form only).  Ends with a barrier.
template <typename T, int SEG, bool GENERAL, typename ColFn>
__device__ __forceinline__ void wstep_segments(ColFn col_of, int LP, const uint32_t* __restrict__ msk, int nrows, int n2,
                                               T rho2, const T* __restrict__ wtab, const T* __restrict__ hex) {
  const int words = (n2 + 31) >> 5, segs = (n2 + SEG - 1) / SEG, ql = n2 - SEG * (segs - 1);
  const int rpr = blockDim.x / segs;  // rows per round (the block has at least segs threads)
  const int row = threadIdx.x % rpr, w = threadIdx.x / rpr;
  for (int r0 = 0; r0 < nrows; r0 += rpr) {
    const bool work = w < segs && r0 + row < nrows;
    const uint32_t* rowm = msk + (size_t)(r0 + row) * words;
    T v[SEG];
    T* col = nullptr;
    if (work) {
      col = col_of(r0 + row);
      const T* cb = col + SEG * w * LP;
      if (w < segs - 1) {
#pragma unroll
        for (int q = 0; q < SEG; ++q) v[q] = cb[q * LP];
      } else {
#pragma unroll
        for (int q = 0; q < SEG; ++q)
          if (q < ql) v[q] = cb[q * LP];
      }
    }
    if constexpr (GENERAL) {
      const int base = SEG * w;
      const uint32_t word = work ? rowm[base >> 5] : 0u;
      if (work && w < segs - 1 && ((word >> (base & 31)) & ((1u << SEG) - 1u)) == 0u) {
        const int st = run_start(rowm, base, word), k = run_end(rowm, words, base + SEG, n2);
        if (k - st >= kWLong<T>) wstep_publish<T, SEG>(col, LP, base, st, k, n2, rho2, wtab, v);
      }
      __syncthreads();
    }
    if (work) {
      if (w < segs - 1)
        wstep_segment<T, SEG, true, false, GENERAL>(col, LP, rowm, words, segs, w, SEG, n2, rho2, wtab, hex, v);
      else wstep_segment<T, SEG, false, true, GENERAL>(col, LP, rowm, words, segs, w, ql, n2, rho2, wtab, hex, v);
    }
    __syncthreads();
    if (work) {
      const int qn = (w < segs - 1) ? SEG : ql;
      T* cb = col + SEG * w * LP;
      if (qn == SEG) {
#pragma unroll
        for (int q = 0; q < SEG; ++q) cb[q * LP] = v[q];
      } else {
#pragma unroll
        for (int q = 0; q < SEG; ++q)
          if (q < qn) cb[q * LP] = v[q];
      }
    }
  }
  __syncthreads();
}

// Weighted |W~^{l+1} - W~^l|^2 of one half-spectrum entry: W~ = Z~ + R~, so the
// change is (R~new - R~old) + (Z~new - Z~old); weight 1 for the real slices
// (k = 0 and, for even n3, k = n3/2), 2 for the others (their mirror).
template <typename T>
__device__ __forceinline__ double dw_term(cx<T> rnew, cx<T> rold, cx<T> dz, int k, int n3) {
  const double a = (double)rnew.re - (double)rold.re + (double)dz.re;
  const double b = (double)rnew.im - (double)rold.im + (double)dz.im;
  return ((k == 0 || 2 * k == n3) ? 1.0 : 2.0) * (a * a + b * b);
}

// ---------------------------------------------------------------------------
// MODE_ITER: phases A, B, C (init != 0: W = P_Omega(G), the initial point, in
//            place of the W-step).
// MODE_W   : W = iDFT(Z~ + R~); optional copy to Wout (column-major), partial
//            sums ||W||^2 and ||K unfold(W,2)||^2.
// MODE_R   : R = iDFT(R~); partial sums ||R||^2 and ||P_Omega R||^2.
// Layouts used here: G row-major [i1][n3][n2] and mask words row-major
// [i1][n3][ceil(n2/32)] (written by k_pack), copied to shared memory.
// ---------------------------------------------------------------------------
// NB: CTAs per SM to leave registers for, as many as the slab's shared memory
// and the grid allow (the sweeps alone take 255 registers, one CTA of 8 warps per SM;
// at 85 and three CTAs the iteration of 435 x 205 x 34 went from 223 to 180 us, but
// with fewer slabs than that the smaller budget only costs: 64 x 600 x 112 FP32
// 767 -> 806 us, 300 x 205 x 34 BF16 145 -> 161).
template <typename T, int MODE, int TL = kTL, int NB = 1>
__global__ void __launch_bounds__(kSlabThreads, NB)
    k_slab(Dev<T> d, T* __restrict__ Wout, int flags, int init) {
  const int slabs_in_smem = flags & SLAB_IN_SMEM;
  extern __shared__ __align__(16) unsigned char smem[];
  const int i1 = blockIdx.x;
  const int n1 = d.n1, n2 = d.n2;
  const int n3 = d.n3;
  const int S = n3 / 2 + 1;
  const int LP = slab_stride(n3);
  const int tid = threadIdx.x, nt = blockDim.x;
  if (MODE == MODE_ITER && !init && converged(d)) return;
  const SlabLayout lay = slab_layout<T>(n2, n3, slabs_in_smem != 0);
  T* wtab = reinterpret_cast<T*>(smem + lay.wtab);
  double* red = reinterpret_cast<double*>(smem + lay.red);
  uint32_t* msk = reinterpret_cast<uint32_t*>(smem + lay.msk);
  int* stw = reinterpret_cast<int*>(smem + lay.stw);
  unsigned char* slab_base =
      slabs_in_smem ? smem : reinterpret_cast<unsigned char*>(d.scratch) + (size_t)i1 * lay.slab_bytes;
  cx<T>* spec = reinterpret_cast<cx<T>*>(slab_base + lay.spec);
  T* spat = reinterpret_cast<T*>(slab_base + lay.spat);
  const cx<T>* zrow = d.Zt + (size_t)i1 * S * n2;
  const cx<T>* rrow = d.Rt + (size_t)i1 * S * n2;
  const T* Gi = d.G + (size_t)i1 * n2 * n3;
  const int mwords = d.mw;
  const uint32_t* Mi = d.mask + (size_t)i1 * n3 * mwords;
  const bool wsolve = (MODE == MODE_ITER) && !init && d.rho2 != T(0);
  const T zfac = init ? T(0) : ((d.rho2 == T(0)) ? T(1) / (T(1) + d.mu) : T(1));

  if (wsolve)
    for (int j = tid; j < 6 * n2; j += nt) wtab[j] = d.winv[j];
  if (MODE != MODE_W) {
    for (int j = tid; j < n3 * mwords; j += nt) msk[j] = __ldg(Mi + j);
    __syncthreads();
  }

  // ---- phase A: inverse transform of each tube; v = G on the mask ------------
  // (MODE_GRAD: v = Z - G on the mask, 0 elsewhere; gsum = ||v||^2)
  SqSum<T> gsum;
  {
    // the half spectrum of the slab ([k][n2], as stored) and the twiddles
    cx<T>* tw = reinterpret_cast<cx<T>*>(smem + lay.tw);
    for (int m = tid; m < n3; m += nt) tw[m] = d.twg[m];
    for (int e = tid; e < S * n2; e += nt) {
      cx<T> v;
      if (MODE == MODE_ITER || MODE == MODE_GRAD) v = zrow[e];
      else if (MODE == MODE_W) v = zrow[e] + rrow[e];
      else v = rrow[e];
      spec[e] = v;
    }
    __syncthreads();
    // Eq. (barAAk) for any n3, as a product of the spectrum with the DFT matrix:
    // x_l = (1/n3) (X_0 + 2 sum_{k=1}^{kmax} Re(X_k conj(w_{kl})) [+ (-1)^l X_{n3/2}]),
    // w_m = exp(-2 pi i m / n3), for items of one tube and TL consecutive rows l,
    // tube index fastest (a warp reads one slice of 32 tubes and shares the
    // twiddles)
    const bool even = (n3 % 2) == 0;
    const int kmax = even ? S - 2 : S - 1;
    const T inv = T(1) / T(n3);
    const int nlb = (n3 + TL - 1) / TL;
    for (int e = tid; e < nlb * n2; e += nt) {
      const int lb = e / n2, t = e - lb * n2, l0 = lb * TL;
      T acc[TL];
      const T s0 = spec[t].re;
#pragma unroll
      for (int j = 0; j < TL; ++j) acc[j] = s0;
      int base = 0;  // k l0 mod n3
      for (int k = 1; k <= kmax; ++k) {
        base += l0;
        if (base >= n3) base -= n3;
        const cx<T> v = spec[(size_t)k * n2 + t];
        int idx = base;  // k (l0 + j) mod n3
#pragma unroll
        for (int j = 0; j < TL; ++j) {
          const cx<T> w = tw[idx];
          acc[j] += T(2) * (v.re * w.re + v.im * w.im);
          idx += k;
          if (idx >= n3) idx -= n3;
        }
      }
      const T sn = even ? spec[(size_t)(S - 1) * n2 + t].re : T(0);
      T* col = spat + (size_t)t * LP;
#pragma unroll
      for (int j = 0; j < TL; ++j) {
        const int l = l0 + j;
        if (l >= n3) break;
        T a = acc[j];
        if (even) a += (l & 1) ? -sn : sn;
        T x = a * inv;
        if (MODE == MODE_ITER) {
          const bool ob = (msk[l * mwords + (t >> 5)] >> (t & 31)) & 1u;
          x = ob ? __ldg(Gi + (size_t)l * n2 + t) : x * zfac;
        } else if (MODE == MODE_GRAD) {
          const bool ob = (msk[l * mwords + (t >> 5)] >> (t & 31)) & 1u;
          x = ob ? x - __ldg(Gi + (size_t)l * n2 + t) : T(0);
          gsum.add(x);
        }
        col[l] = x;
      }
    }
  }
  __syncthreads();
  if (MODE == MODE_GRAD) {
    double g = gsum.total(), unused = 0.0;
    block_sum2(g, unused, red);
    if (sq_again<T>(g, gsum.nonzero())) {
      SqSum64 g64;
      for (int e = tid; e < n2 * n3; e += nt) g64.add(spat[(e / n3) * LP + e % n3]);
      g = g64.s;
      block_sum2(g, unused, red);
    }
    if (tid == 0) d.part[(size_t)i1 * 4] = g;
  }

  // ---- phase B: rows ------------------------------------------------------
  if (MODE == MODE_W || MODE == MODE_R) {
    const bool sums = MODE == MODE_R || !(flags & SLAB_NOSUM);
    if (MODE == MODE_W && Wout)
      for (int e = tid; e < n2 * n3; e += nt) {
        const int j = e / n3, l = e - j * n3;
        Wout[(size_t)i1 + (size_t)n1 * ((size_t)j + (size_t)n2 * l)] = spat[j * LP + l];
      }
    if (!sums) return;
    auto walk = [&](auto& sa, auto& sb) {
      for (int e = tid; e < n2 * n3; e += nt) {
        const int j = e / n3, l = e - j * n3;
        const T v = spat[j * LP + l];
        sa.add(v);
        if (MODE == MODE_W) {
          if (j + 1 < n2) sb.add_diff(v, spat[(j + 1) * LP + l]);
        } else {
          if ((msk[l * mwords + (j >> 5)] >> (j & 31)) & 1u) sb.add(v);
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
  if (wsolve) {
    if (n3 <= nt) {  // every thread one (row, segment)
      wstep_sweeps_seg<T, (NB <= 2)>([&](int l) { return spat + l; }, LP, msk, stw, n3, nt / n3, tid, n2, d.rho2, wtab);
    } else {
      for (int l = tid; l < n3; l += nt)
        wstep_sweeps<T>(spat + l, LP, msk + l * mwords, stw + l * mwords, n2, d.rho2, wtab);
      __syncthreads();
    }
  }

  // ---- phase C: forward transform, R~ = W~ - Z~ ------------------------------
  const bool track = (MODE == MODE_ITER) && !init && d.dZt != nullptr;
  double dw2 = 0.0;
  {
    // Eq. (bar BA-k) for any n3, as a product of the slab with the DFT matrix:
    // X_k = sum_l x_l w_{kl} for k < S, for items of one tube and TL consecutive
    // slices k, tube index fastest
    const cx<T>* tw = reinterpret_cast<const cx<T>*>(smem + lay.tw);
    const int nkb = (S + TL - 1) / TL;
    // the change of W~ (FP64) in a loop of its own: predicated into the plain one,
    // its instructions would take their issue slots of the FP64 pipe all the same
    auto slices = [&](auto tr) {
      constexpr bool TRACK = decltype(tr)::value;
      for (int e = tid; e < nkb * n2; e += nt) {
        const int kb = e / n2, t = e - kb * n2, k0 = kb * TL;
        cx<T> acc[TL];
#pragma unroll
        for (int j = 0; j < TL; ++j) acc[j] = cx<T>{T(0), T(0)};
        int idx[TL], inc[TL];  // (k0 + j) l mod n3, advanced by (k0 + j) mod n3 (< n3)
#pragma unroll
        for (int j = 0; j < TL; ++j) {
          idx[j] = 0;
          inc[j] = (k0 + j) % n3;
        }
        const T* col = spat + (size_t)t * LP;
        for (int l = 0; l < n3; ++l) {
          const T x = col[l];
#pragma unroll
          for (int j = 0; j < TL; ++j) {
            const cx<T> w = tw[idx[j]];
            acc[j].re += x * w.re;
            acc[j].im += x * w.im;
            idx[j] += inc[j];
            if (idx[j] >= n3) idx[j] -= n3;
          }
        }
        const size_t o = (size_t)i1 * S * n2 + t;
#pragma unroll
        for (int j = 0; j < TL; ++j) {
          const int k = k0 + j;
          if (k >= S) break;
          cx<T> a = acc[j];
          if (k == 0 || (2 * k == n3)) a.im = T(0);
          const size_t ok = o + (size_t)k * n2;
          const cx<T> rn = (MODE == MODE_GRAD) ? a : a - zrow[(size_t)k * n2 + t];
          if constexpr (TRACK) dw2 += dw_term(rn, d.Rt[ok], d.dZt[ok], k, n3);
          d.Rt[ok] = rn;
        }
      }
    };
    if (track) slices(BoolC<true>{});
    else slices(BoolC<false>{});
  }
  if (track) {
    double unused = 0.0;
    block_sum2(dw2, unused, red);
    if (tid == 0) d.part_dw[i1] = dw2;
  }
}

}  // namespace tc
