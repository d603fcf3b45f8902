// select.cu -- greedy ensemble selection on the device (Sec. 3.5 "Greedy
// ensembling").  Each iteration scores every unused candidate c as the
// ensemble S + {c}, picks the best (lowest index on ties), and stops when the
// best addition does not strictly improve the current score.  The running sum
// S of the selected candidates' predictions is fp64; the ensemble value of a
// row, (S + p_c) * (1 / (n + 1)), is rounded to fp32; each row's loss /
// squared-error term is then taken in fp32, and terms are summed to about
// 2^-45 relative in a fixed order.  Accuracy decisions (the argmax, or above
// 1/2) are those of the fp64 ensemble values.
//
// fp64 runs at about 1/64 of the fp32 rate on this part: with an fp64 value
// per row, candidate and iteration the fp64 pipe is what bounds a selection.
// So the ensemble value is carried as an unevaluated sum of two fp32 numbers
// (to 2^-46 of its operands), and S is split into two once per iteration.
// Accuracy takes the fp64 expression itself wherever two decisions are
// closer than the fp32 arithmetic can tell.
//
// One iteration is two launches: the score kernel, whose last block to finish
// makes the pick, and k_sel_add, which brings S up to date.
#include "kernels.cuh"
#include "two_float.cuh"

namespace tp {

constexpr int kSelThreads = 256;
constexpr int kSelRowsPerThread = 4;
constexpr int kSelRowsPerBlock = kSelThreads * kSelRowsPerThread;
constexpr int kSelGroup = 8;      // candidates per block of the score kernel

// state words: n, done, last pick, blocks done | selected[m_ens] | used[P].
// Bit 0 of used[c] says that c is excluded or selected; the bits above it
// count the finished row blocks of the candidate group that starts at c.
enum { kStN = 0, kStDone = 1, kStLast = 2, kStTicket = 3, kStHdr = 4 };
constexpr int kScoreAuc = 3;      // TP_SCORE_AUC
constexpr int kAucThreads = 1024;
enum SelKind { kSelLoss = 0, kSelSquare = 1, kSelHitBinary = 2, kSelHitMulti = 3 };

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ------------------------------------------------- two-float ensemble values
struct EnsInv {
  double inv;       // 1 / (n + 1)
  float hi, lo;     // the same as a sum of two fp32 numbers
};
// what follows the current score in SelectScratch::cur
struct SelTail {
  EnsInv iv;        // of the next ensemble size
  uint32_t cnt[2];  // ROC-AUC: positives and negatives placed
};
__device__ __forceinline__ SelTail* sel_tail(double* cur) { return reinterpret_cast<SelTail*>(cur + 1); }
__device__ __forceinline__ EnsInv ens_inv(int n) {
  EnsInv v;
  v.inv = 1.0 / (double)(n + 1);
  v.hi = (float)v.inv;
  v.lo = (float)(v.inv - (double)v.hi);
  return v;
}
// S as two fp32 numbers: read, or (SPLIT = 0: where S2 found no room) taken
// apart where it is used.  A template, because a run-time choice is compiled
// into fp64 conversions that run either way.
template <int SPLIT>
__device__ __forceinline__ float2 ens_sum(const double* S, const float2* S2, int64_t j);
__device__ __forceinline__ float2 split2(double s) {
  const float h = (float)s;
  return make_float2(h, (float)(s - (double)h));
}

template <>
__device__ __forceinline__ float2 ens_sum<1>(const double*, const float2* S2, int64_t j) { return S2[j]; }
template <>
__device__ __forceinline__ float2 ens_sum<0>(const double* S, const float2*, int64_t j) { return split2(S[j]); }

// (h, l): h + l = (S + q) / (n + 1) to 2^-46 of (|S| + |q|) / (n + 1)
__device__ __forceinline__ void ens_two(float2 s, float q, const EnsInv& v, float& h, float& l) {
  const float t = __fadd_rn(s.x, q);
  const float b = __fsub_rn(t, s.x);
  const float e = __fadd_rn(__fadd_rn(__fsub_rn(s.x, __fsub_rn(t, b)), __fsub_rn(q, b)), s.y);
  h = __fmul_rn(t, v.hi);
  l = __fmaf_rn(e, v.hi, __fmaf_rn(t, v.lo, __fmaf_rn(t, v.hi, -h)));
}

// The ensemble value rounded to fp32.  A sum of a few fp32 numbers over
// n + 1 is often exactly half way between two fp32 numbers, where fp64
// rounds to even: the low part is first rounded to multiples of 2^-44 of the
// value's power of two, which removes its own error there.  The result is
// fp64's rounding but for values within 2^-45 of such a point without lying
// on it.  Values that are not finite are ens_value's caller's to handle, and
// so are sums S + q below kEnsTiny (n + 1) other than zero: 2^-46 of them
// lies below fp32's smallest number, 2^-149.
constexpr float kEnsTiny = 7.8886091e-31f;   // 2^-100
__device__ __forceinline__ float ens_value(float2 s, float q, const EnsInv& v) {
  float h, l;
  ens_two(s, q, v, h, l);
  const float p2 = __uint_as_float(__float_as_uint(h) & 0x7f800000u);
  const float m = __fmul_rn(p2, 7.1525574e-07f);   // 1.5 2^-21: sums with it round to 2^-44 p2
  return __fadd_rn(h, __fsub_rn(__fadd_rn(l, m), m));
}

// the fp64 expression itself; out of line, so that it is a branch and not
// predicated fp64 work of every row
__device__ __noinline__ float ens_exact(const double* S, float q, double inv) { return (float)((*S + (double)q) * inv); }

__global__ void k_sel_init(double* __restrict__ S, float2* __restrict__ S2, int64_t n_S, int32_t* __restrict__ state,
                           int32_t n_state, double* __restrict__ cur, const uint8_t* __restrict__ excl, int32_t m_ens) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n_S; e += (int64_t)gridDim.x * blockDim.x) {
    S[e] = 0.0;
    if (S2) S2[e] = make_float2(0.f, 0.f);
  }
  if (blockIdx.x == 0) {
    const int used0 = kStHdr + m_ens;  // used[c] starts as excl[c]
    for (int e = threadIdx.x; e < n_state; e += blockDim.x)
      state[e] = e == kStLast ? -1 : (excl != nullptr && e >= used0) ? (excl[e - used0] != 0) : 0;
    if (threadIdx.x == 0) {
      cur[0] = __longlong_as_double(0x7ff0000000000000LL);  // +inf
      SelTail* tail = sel_tail(cur);
      tail->iv = ens_inv(0);
      tail->cnt[0] = tail->cnt[1] = 0;
    }
  }
}

// The pick of one iteration, by the last block to finish: scores[c * stride]
// of the unused candidates, lowest index on ties.
template <int THREADS>
__device__ void sel_pick(const double* scores, int32_t P, int64_t stride, int32_t* state, double* cur, int32_t m_ens,
                         double* solo) {
  __shared__ double sb[THREADS / 32];
  __shared__ int sc_[THREADS / 32];
  int32_t* used = state + kStHdr + m_ens;
  const double inf = __longlong_as_double(0x7ff0000000000000LL);
  double best = inf;
  int best_c = -1;
  for (int c = threadIdx.x; c < P; c += THREADS) {
    const int u = __ldcg(used + c);
    if (u > 1) used[c] = u & 1;   // the group counts of this iteration
    const double sc = (u & 1) ? __longlong_as_double(0x7ff8000000000000LL) : __ldcg(scores + (int64_t)c * stride);
    if (solo) solo[c] = sc;
    if (sc < best) { best = sc; best_c = c; }   // ascending c per thread: lowest index wins ties
  }
  auto merge = [&](double ob, int oc) {
    if (oc >= 0 && (best_c < 0 || ob < best || (ob == best && oc < best_c))) { best = ob; best_c = oc; }
  };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oc = __shfl_xor_sync(0xffffffffu, best_c, o);
    merge(ob, oc);
  }
  if ((threadIdx.x & 31) == 0) {
    sb[threadIdx.x >> 5] = best;
    sc_[threadIdx.x >> 5] = best_c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < THREADS / 32; ++w) merge(sb[w], sc_[w]);
    const int n = state[kStN];
    if (best_c < 0 || (n > 0 && !(best < cur[0]))) {
      state[kStDone] = 1;
      state[kStLast] = -1;
    } else {
      state[kStHdr + n] = best_c;
      used[best_c] = 1;
      state[kStN] = n + 1;
      state[kStLast] = best_c;
      cur[0] = best;
      sel_tail(cur)->iv = ens_inv(n + 1);
      if (n + 1 >= m_ens) state[kStDone] = 1;
    }
    state[kStTicket] = 0;
  }
}

// ------------------------------------------- loss, squared error, accuracy
// The value a row's term reads from candidate c: vals[c * cand_stride + b *
// row_stride + k], k the row's label where by_label (cross-entropy reads the
// true class only), else 0.
struct SelVals {
  const float* vals;
  int64_t cand_stride;
  int32_t row_stride, by_label;
};

// comp[c, b] = preds[c, b, y[b]]: the only value the cross-entropy of row b
// ever reads, so that an iteration streams N floats per candidate instead of
// N rows (select_enqueue, for more than one iteration).  An invalid label's
// entry is never used.
__global__ void __launch_bounds__(kSelThreads) k_sel_compact(const float* __restrict__ preds,
                                                             const int32_t* __restrict__ y, int64_t N, int32_t d_out,
                                                             float* __restrict__ comp) {
  pdl_trigger();
  pdl_wait();
  const int64_t c = blockIdx.y, r0 = (int64_t)blockIdx.x * kSelRowsPerBlock;
#pragma unroll
  for (int q = 0; q < kSelRowsPerThread; ++q) {
    const int64_t b = r0 + q * kSelThreads + threadIdx.x;
    if (b >= N) continue;
    const int k = y[b];
    comp[c * N + b] = k >= 0 && k < d_out ? __ldcs(preds + (c * N + b) * d_out + k) : 0.f;
  }
}

template <int KIND>
__device__ __forceinline__ float sel_term(float e, float yf, bool positive, bool valid) {
  if constexpr (KIND == kSelSquare) {
    const float d = e - yf;
    return d * d;
  } else {
    e = fminf(fmaxf(e, 1e-7f), 1.0f - 1e-7f);
    e = positive ? e : 1.0f - e;   // one logarithm, not a choice of two
    return valid ? -logf(e) : __int_as_float(0x7fc00000);  // invalid label: NaN score
  }
}

// Whether row `b` of candidate matrix q [d_out] is classified right by the
// ensemble: argmax (first of equals) of (S_k + q_k) inv in fp64.
__device__ bool sel_hit_exact(const double* s, const float* q, int32_t d_out, double inv, int yv) {
  int pred = 0;
  double best = (s[0] + (double)q[0]) * inv;
  for (int c = 1; c < d_out; ++c) {
    const double e = (s[c] + (double)q[c]) * inv;
    if (e > best) { best = e; pred = c; }
  }
  return pred == yv;
}

// Partial scores of up to kSelGroup candidates over 1024 rows, whose S is read
// once for the group.  Bound by instruction issue (2.4 per cycle and SM: the
// logarithm, the two-float value and sum).  96 candidates x 100k rows x 10
// classes: 39 us per iteration and 58 us once for k_sel_compact, against 110
// us with fp64 values and the label's sector re-read from HBM each time.
// Groups of 8: the sums of a group stay in registers and its eight warps make
// one warp per candidate at the end.  Multiclass accuracy keeps S as fp32 in
// shared memory and compares fp32 sums; a row whose two best classes are
// within 2^-20 of each other is decided in fp64.
template <int KIND, int SPLIT>
__global__ void __launch_bounds__(kSelThreads) k_sel_score(const double* __restrict__ S,
                                                           const float2* __restrict__ S2, SelVals V,
                                                           const void* __restrict__ y, int64_t N, int32_t d_out,
                                                           int32_t score, int32_t* state, double* partial,
                                                           int32_t n_blk, int32_t P, int32_t m_ens, double* cur,
                                                           double* solo) {
  pdl_trigger();
  pdl_wait();
  if (state[kStDone]) return;
  const int c0 = blockIdx.y * kSelGroup, nc = min(kSelGroup, P - c0);
  int32_t* used = state + kStHdr + m_ens;
  const EnsInv iv = sel_tail(cur)->iv;
  const int64_t r0 = (int64_t)blockIdx.x * kSelRowsPerBlock;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ float2 wsum[kSelGroup][kSelThreads / 32];
  __shared__ double dsum[kSelThreads / 32];
  __shared__ int use_s[kSelGroup];
  if (tid < kSelGroup) use_s[tid] = tid < nc && !(__ldcg(used + c0 + tid) & 1);
  __syncthreads();
  float ah[kSelGroup], al[kSelGroup];
#pragma unroll
  for (int g = 0; g < kSelGroup; ++g) ah[g] = al[g] = 0.f;

  if constexpr (KIND == kSelHitMulti) {
    extern __shared__ float Sf[];   // [d_out][256]: S of 256 rows in fp32
    for (int q = 0; q < kSelRowsPerThread; ++q) {
      const int64_t rb = r0 + q * kSelThreads;
      if (rb >= N) break;           // block-uniform
      const int rows = (int)min((int64_t)kSelThreads, N - rb);
      __syncthreads();
      for (int e = tid; e < rows * d_out; e += kSelThreads) {
        const int r = e / d_out, k = e - r * d_out;
        Sf[k * kSelThreads + r] = (float)S[rb * d_out + e];
      }
      __syncthreads();
      if (tid < rows) {
        const int64_t b = rb + tid;
        const int yv = ((const int32_t*)y)[b];
        for (int g = 0; g < nc; ++g) {
          if (!use_s[g]) continue;
          const float* qv = V.vals + (int64_t)(c0 + g) * V.cand_stride + b * d_out;
          float best = Sf[tid] + qv[0], second = -INFINITY, top = fabsf(Sf[tid]) + fabsf(qv[0]);
          int pred = 0;
          for (int k = 1; k < d_out; ++k) {
            const float s = Sf[k * kSelThreads + tid], v = qv[k];
            const float e = s + v;
            top = fmaxf(top, fabsf(s) + fabsf(v));
            if (e > best) {
              second = best;
              best = e;
              pred = k;
            } else {
              second = fmaxf(second, e);
            }
          }
          // a NaN or an infinity makes the comparison false
          const bool sure = best - second > top * 9.5367432e-07f && top < 1e37f && top > 1e-30f;
          const bool hit = sure ? pred == yv : sel_hit_exact(S + b * d_out, qv, d_out, iv.inv, yv);
#pragma unroll
          for (int g2 = 0; g2 < kSelGroup; ++g2)
            if (g2 == g) ah[g2] += hit ? 1.f : 0.f;   // at most 4 per thread: exact
        }
      }
    }
  } else {
    float2 s2[kSelRowsPerThread];
    float yf[kSelRowsPerThread];
    bool pos[kSelRowsPerThread], val[kSelRowsPerThread], in[kSelRowsPerThread];
    int64_t off[kSelRowsPerThread];
#pragma unroll
    for (int q = 0; q < kSelRowsPerThread; ++q) {
      const int64_t b = r0 + q * kSelThreads + tid;
      in[q] = b < N;
      const int64_t bb = in[q] ? b : 0;
      s2[q] = ens_sum<SPLIT>(S, S2, bb);
      yf[q] = 0.f;
      pos[q] = true;
      val[q] = true;
      off[q] = bb * V.row_stride;
      if constexpr (KIND == kSelSquare) {
        yf[q] = ((const float*)y)[bb];
      } else {
        const int yv = ((const int32_t*)y)[bb];
        if (KIND == kSelLoss && d_out > 1) {
          val[q] = yv >= 0 && yv < d_out;
          if (V.by_label && val[q]) off[q] += yv;
        } else {
          pos[q] = yv == 1;
          if (KIND == kSelHitBinary) val[q] = yv == 0 || yv == 1;   // any other label is never hit
        }
      }
    }
#pragma unroll
    for (int g = 0; g < kSelGroup; ++g) {
      if (g >= nc || !use_s[g]) continue;
      const float* vp = V.vals + (int64_t)(c0 + g) * V.cand_stride;
      float v[kSelRowsPerThread];
#pragma unroll
      for (int q = 0; q < kSelRowsPerThread; ++q) v[q] = in[q] ? __ldg(vp + off[q]) : 0.f;
#pragma unroll
      for (int q = 0; q < kSelRowsPerThread; ++q) {
        if (!in[q]) continue;
        if constexpr (KIND == kSelHitBinary) {
          float h, l;
          ens_two(s2[q], v[q], iv, h, l);
          const float d = __fadd_rn(__fsub_rn(h, 0.5f), l);   // the subtraction is exact near 1/2
          bool yes = d > 0.f;
          const float m = (fabsf(s2[q].x) + fabsf(v[q])) * iv.hi;
          if (!(fabsf(d) > m * 2.2737368e-13f + 1e-30f) || !(m < 1e37f))
            yes = (S[r0 + q * kSelThreads + tid] + (double)v[q]) * iv.inv > 0.5;
          ah[g] += val[q] && yes == pos[q] ? 1.f : 0.f;
        } else {
          // (values below kEnsTiny need no care here: cross-entropy clips at
          // 1e-7, and a square does not feel 2^-24 of them)
          float e = ens_value(s2[q], v[q], iv);
          if (!(fabsf(e) < 1e36f)) e = ens_exact(S + r0 + q * kSelThreads + tid, v[q], iv.inv);
          two_add(ah[g], al[g], sel_term<KIND>(e, yf[q], pos[q], val[q]));
        }
      }
    }
  }

  // Sum over the block (two_merge is symmetric, so that equal candidates get
  // equal sums wherever they stand in a group): halving exchanges leave lane l with candidate
  // (l >> 2) & 7 of the warp's two-float sums (a whole warp's sum costs 9
  // exchanges of pairs instead of 40), then the warps in order.
  {
    int width = kSelGroup;
#pragma unroll
    for (int o = 16; o >= 4; o >>= 1) {
      width >>= 1;
      const bool up = lane & o;
#pragma unroll
      for (int g = 0; g < kSelGroup / 2; ++g) {
        if (g >= width) break;
        const float sh = up ? ah[g] : ah[g + width], sl = up ? al[g] : al[g + width];
        const float rh = __shfl_xor_sync(0xffffffffu, sh, o), rl = __shfl_xor_sync(0xffffffffu, sl, o);
        if (up) {
          ah[g] = ah[g + width];
          al[g] = al[g + width];
        }
        two_merge(ah[g], al[g], rh, rl);
      }
    }
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) {
      const float rh = __shfl_xor_sync(0xffffffffu, ah[0], o), rl = __shfl_xor_sync(0xffffffffu, al[0], o);
      two_merge(ah[0], al[0], rh, rl);
    }
    if ((lane & 3) == 0) wsum[lane >> 2][warp] = make_float2(ah[0], al[0]);
  }
  __shared__ double bsum[kSelGroup];
  __syncthreads();
  if (tid < kSelGroup) {
    float2 s = wsum[tid][0];
    for (int w = 1; w < kSelThreads / 32; ++w) two_merge(s.x, s.y, wsum[tid][w].x, wsum[tid][w].y);
    bsum[tid] = isfinite(s.x) ? (double)s.x + (double)s.y : (double)s.x;
  }
  __syncthreads();
  if constexpr (KIND == kSelSquare) {
    // squared errors can overflow an fp32 sum where fp64 does not: such a
    // candidate's block is summed again in fp64
    for (int g = 0; g < nc; ++g) {
      if (!use_s[g] || isfinite(bsum[g])) continue;   // block-uniform
      double acc = 0.0;
      for (int q = 0; q < kSelRowsPerThread; ++q) {
        const int64_t b = r0 + q * kSelThreads + tid;
        if (b >= N) continue;
        const float v = V.vals[(int64_t)(c0 + g) * V.cand_stride + b * V.row_stride];
        const float d = (float)((S[b] + (double)v) * iv.inv) - ((const float*)y)[b];
        acc += (double)(d * d);
      }
      acc = warp_sum_d(acc);
      __syncthreads();
      if (lane == 0) dsum[warp] = acc;
      __syncthreads();
      if (tid == 0) {
        double s = 0.0;
        for (int w = 0; w < kSelThreads / 32; ++w) s += dsum[w];
        bsum[g] = s;
      }
      __syncthreads();
    }
  }
  if (tid < nc && use_s[tid]) partial[(int64_t)(c0 + tid) * n_blk + blockIdx.x] = bsum[tid];

  // the group's last block adds the row blocks of its candidates (fixed
  // order), the last group makes the pick
  __shared__ int last_s;
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    last_s = (atomicAdd(used + c0, 2) >> 1) == n_blk - 1;
  }
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  static_assert(kSelThreads / 32 == kSelGroup, "a warp per candidate");
  if (warp < nc && use_s[warp]) {
    double* pc = partial + (int64_t)(c0 + warp) * n_blk;
    double s = 0.0;
    for (int b = lane; b < n_blk; b += 32) s += __ldcg(pc + b);
    s = warp_sum_d(s);
    const double mean = s / (double)N;
    __syncwarp();
    if (lane == 0) pc[0] = score == 1 ? -mean : (score == 2 ? sqrt(mean) : mean);
  }
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    last_s = atomicAdd(state + kStTicket, 1) == (int)gridDim.y - 1;
  }
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  sel_pick<kSelThreads>(partial, P, n_blk, state, cur, m_ens, solo);
}

// S += the last pick's values ([N] for the label's or the only value, [N,
// d_out] for multiclass accuracy); S2 (if kept): S as two fp32 numbers
__global__ void k_sel_add(double* __restrict__ S, float2* __restrict__ S2, SelVals V, const void* __restrict__ y, int64_t n_S, int32_t d_out,
                          const int32_t* __restrict__ state) {
  pdl_trigger();
  pdl_wait();
  const int c = state[kStLast];
  if (state[kStDone] || c < 0) return;
  const float* p = V.vals + (int64_t)c * V.cand_stride;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n_S; e += (int64_t)gridDim.x * blockDim.x) {
    int64_t o = e * V.row_stride;
    if (V.by_label) {
      const int k = ((const int32_t*)y)[e];
      if (k >= 0 && k < d_out) o += k;
    }
    const double v = S[e] + (double)p[o];
    S[e] = v;
    if (S2) S2[e] = split2(v);
  }
}

// ------------------------------------------------------------------ ROC-AUC
// The score of candidate c is minus the ROC-AUC of the ensemble values
// rounded to fp32, ties counted 1/2: AUC = U / (n_pos n_neg), 2 U = sum over
// (positive, negative) pairs of 2 [key_pos > key_neg] + [equal], on
// order-preserving integer keys.  U needs no sort of all rows, only for every
// row of the larger class its place among the keys of the smaller class:
//   1. the smaller class's values are counted into up to 32768 buckets by a
//      monotone fp32 map (v - lo) scale, lo and hi from the candidates' own
//      value ranges, so that buckets follow the order of the keys;
//   2. their keys are placed bucket by bucket in shared memory;
//   3. each row of the larger class finds its bucket: the keys before it are
//      smaller, those after it larger, and the few inside are compared.
// One block per candidate; with the rows laid out by class beforehand
// (k_auc_perm, k_auc_permute) every pass reads whole segments.  Where a
// bucket holds more than kAucBucketMax keys (heavy ties), a value is not
// finite, sums fall below kEnsTiny (n + 1), or N is tiny, the smaller class is
// sorted by a 4-pass radix sort and the larger one searches it: any input.
// The counts are integers, so neither path's order of work shows in the
// result.  Measured (266 candidates x 60k rows, balanced classes): 99 us per
// iteration, in two waves of one block per SM (the buckets and keys take 184
// KB).  A selection of 32 members takes 3.8 ms; with a full stable sort of every
// candidate and mid-ranks by binary search, in fp64 values, 46 ms.  With all
// values in 17 groups of ties 17 against 33 ms, a third of them at 0 and a
// third at 1 7.5 against 46 ms, 86 % of them at 0 23 against 45 ms.
constexpr int kAucBucketMax = 192;
constexpr int kAucMinRows = 16;
constexpr int kAucSmemMax = 220 * 1024;
constexpr int kAucSortSmem = (32 * 256 + 3 * 256) * 4;

__device__ __forceinline__ uint32_t auc_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float auc_value(uint32_t key) {
  return __uint_as_float((key & 0x80000000u) ? key ^ 0x80000000u : ~key);
}

// perm: positives from the front, negatives from the back (the order within a
// class is free); cnt counts the rows placed
__global__ void __launch_bounds__(256) k_auc_perm(const int32_t* __restrict__ y, int64_t N, uint32_t* __restrict__ perm,
                                                  double* cur) {
  pdl_trigger();
  pdl_wait();
  uint32_t* cnt = sel_tail(cur)->cnt;
  const int64_t b = (int64_t)blockIdx.x * 256 + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool in = b < N, p = in && y[b] == 1;
  const uint32_t mp = __ballot_sync(0xffffffffu, p), mn = __ballot_sync(0xffffffffu, in && !p);
  uint32_t bp = 0, bn = 0;
  if (lane == 0) {
    bp = atomicAdd(cnt, __popc(mp));
    bn = atomicAdd(cnt + 1, __popc(mn));
  }
  bp = __shfl_sync(0xffffffffu, bp, 0);
  bn = __shfl_sync(0xffffffffu, bn, 0);
  const uint32_t below = (1u << lane) - 1u;
  if (p) perm[bp + __popc(mp & below)] = (uint32_t)b;
  else if (in) perm[N - 1 - (bn + __popc(mn & below))] = (uint32_t)b;
}

// pm[c, j] = preds[c, perm[j]], the range of the candidate's values (an empty
// one, lo > hi, when a value is not finite), and whether it has any below
// 2^-50 other than zero.  Values without such are multiples of 2^-74, and so
// are their sums: averages of up to 2^26 of them are zero or not below kEnsTiny.
__global__ void __launch_bounds__(kAucThreads) k_auc_permute(const float* __restrict__ preds,
                                                             const uint32_t* __restrict__ perm, int64_t N,
                                                             float* __restrict__ pm, float* __restrict__ range) {
  pdl_trigger();
  pdl_wait();
  const float* p = preds + (int64_t)blockIdx.x * N;
  float* o = pm + (int64_t)blockIdx.x * N;
  float lo = INFINITY, hi = -INFINITY;
  bool bad = false, small = false;
#pragma unroll 4
  for (int64_t j = threadIdx.x; j < N; j += kAucThreads) {
    const float v = p[perm[j]];
    o[j] = v;
    lo = fminf(lo, v);
    hi = fmaxf(hi, v);
    bad |= !(fabsf(v) < 1e36f);
    small |= v != 0.f && fabsf(v) < 8.8817842e-16f;   // 2^-50
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, s));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, s));
  }
  __shared__ float slo[32], shi[32];
  if ((threadIdx.x & 31) == 0) {
    slo[threadIdx.x >> 5] = lo;
    shi[threadIdx.x >> 5] = hi;
  }
  const bool any = __syncthreads_or(bad), any_small = __syncthreads_or(small);
  if (threadIdx.x == 0 && range) {
    for (int w = 1; w < kAucThreads / 32; ++w) {
      slo[0] = fminf(slo[0], slo[w]);
      shi[0] = fmaxf(shi[0], shi[w]);
    }
    range[3 * blockIdx.x] = any ? INFINITY : slo[0];
    range[3 * blockIdx.x + 1] = any ? -INFINITY : shi[0];
    range[3 * blockIdx.x + 2] = any_small ? 1.f : 0.f;
  }
}

// fp32 ensemble value of row j of a candidate (rows ordered by class)
template <int SPLIT>
struct AucEns {
  const double* S;
  const float2* S2;
  const float* p;
  EnsInv iv;
  __device__ __forceinline__ float operator()(uint32_t j) const {
    return ens_value(ens_sum<SPLIT>(S, S2, j), p[j], iv);
  }
  __device__ __forceinline__ float sum(int64_t j) const { return __fadd_rn(ens_sum<SPLIT>(S, S2, j).x, p[j]); }
  __device__ __forceinline__ float exact(uint32_t j) const { return ens_exact(S + j, p[j], iv.inv); }
};

__device__ __forceinline__ int64_t auc_block_sum(int64_t v, int64_t* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  int64_t s = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < kAucThreads / 32; ++w) s += red[w];
  return s;   // thread 0's
}

// Ascending 4-pass LSD radix sort of k0[0 .. n) by one block (8-bit digits;
// within a 1024-key tile a key's place among equal digits comes from its
// warp's match mask and the warps before it); k1: a second buffer.  The
// result is in k0.  sm: kAucSortSmem bytes.
__device__ __noinline__ void auc_sort(uint32_t* k0, uint32_t* k1, int64_t n, uint32_t* sm) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t(*wcnt)[256] = reinterpret_cast<uint32_t(*)[256]>(sm);
  uint32_t* hist = sm + 32 * 256;
  uint32_t* base = hist + 256;
  uint32_t* tot = base + 256;
  for (int e = tid; e < 32 * 256; e += kAucThreads) sm[e] = 0;
  __syncthreads();
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 8 * pass;
    const uint32_t* src = (pass & 1) ? k1 : k0;
    uint32_t* dst = (pass & 1) ? k0 : k1;
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
    for (int64_t b = tid; b < n; b += kAucThreads) atomicAdd(&hist[(src[b] >> shift) & 255u], 1u);
    __syncthreads();
    if (tid == 0) {
      uint32_t run = 0;
      for (int d = 0; d < 256; ++d) {
        base[d] = run;
        run += hist[d];
      }
    }
    __syncthreads();
    for (int64_t t0 = 0; t0 < n; t0 += kAucThreads) {
      const int64_t b = t0 + tid;
      const bool valid = b < n;
      const uint32_t key = valid ? src[b] : 0u;
      const int d = valid ? (int)((key >> shift) & 255u) : 256;
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      const int rank = __popc(peers & ((1u << lane) - 1u));
      if (valid && rank == 0) wcnt[warp][d] = __popc(peers);
      __syncthreads();
      if (tid < 256) {   // per digit: exclusive prefix over warps, then the tile's total
        uint32_t run = 0;
        for (int w = 0; w < 32; ++w) {
          const uint32_t v = wcnt[w][tid];
          wcnt[w][tid] = run;
          run += v;
        }
        tot[tid] = run;
      }
      __syncthreads();
      if (valid) dst[base[d] + wcnt[warp][d] + (uint32_t)rank] = key;
      __syncthreads();
      if (tid < 256) {
        base[tid] += tot[tid];
        for (int w = 0; w < 32; ++w) wcnt[w][tid] = 0;
      }
      __syncthreads();
    }
  }
}

// STAGED: a row of the smaller class is valued once; its key and its place in
// its bucket wait in the sort buffers (L2) for the buckets' starts.  Counters
// and starts are 16-bit, so twice the buckets fit; needs the smaller class
// below 2^16 and its keys in shared memory.  Else the values are computed
// twice and the counters are 32-bit.
template <int SPLIT, int STAGED>
__global__ void __launch_bounds__(kAucThreads, 1) k_sel_auc(const double* __restrict__ S,
                                                            const float2* __restrict__ S2,
                                                            const float* __restrict__ pm, int64_t N, int32_t* state,
                                                            double* partial, int32_t n_blk, int32_t P, int32_t m_ens,
                                                            double* cur, double* solo,
                                                            const float* __restrict__ range, uint32_t* srt,
                                                            int32_t nb, int32_t key_cap) {
  pdl_trigger();
  pdl_wait();
  if (state[kStDone]) return;
  extern __shared__ __align__(16) uint32_t auc_sm[];
  const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ int64_t red[kAucThreads / 32];
  __shared__ uint32_t wtot[kAucThreads / 32];
  __shared__ float rng_s[3];
  __shared__ int last_s;
  if (!(__ldcg(state + kStHdr + m_ens + c) & 1)) {   // block-uniform
    AucEns<SPLIT> ens;
    ens.S = S;
    ens.S2 = S2;
    ens.p = pm + (int64_t)c * N;
    ens.iv = sel_tail(cur)->iv;
    const uint32_t n_pos = sel_tail(cur)->cnt[0], n_neg = (uint32_t)N - n_pos;   // rows are numbered in 32 bits
    const bool few_pos = n_pos <= n_neg;
    const uint32_t few0 = few_pos ? 0u : n_pos, n_few = few_pos ? n_pos : n_neg;      // the smaller class
    const uint32_t many0 = few_pos ? n_pos : 0u, n_many = few_pos ? n_neg : n_pos;
    // this thread's rows of the larger class, counted: a row number may lie
    // within one stride of 2^32
    const uint32_t my_many = (uint32_t)tid < n_many ? (n_many - 1 - tid) / kAucThreads + 1 : 0;
    uint32_t* const k0 = srt + (int64_t)c * 2 * (N / 2);
    uint32_t* const k1 = k0 + N / 2;
    if (warp == 0) {   // the ensemble's value range: the mean of the members' ranges
      float lo = 0.f, hi = -1.f, small = 0.f;   // empty: values taken in fp64, no buckets
      if (N >= kAucMinRows) {
        hi = 0.f;
        const int n = state[kStN];
        for (int k = lane; k <= n; k += 32) {
          const int e = k < n ? state[kStHdr + k] : c;
          lo += range[3 * e];
          hi += range[3 * e + 1];
          small += range[3 * e + 2];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          lo += __shfl_xor_sync(0xffffffffu, lo, o);
          hi += __shfl_xor_sync(0xffffffffu, hi, o);
          small += __shfl_xor_sync(0xffffffffu, small, o);
        }
      }
      if (lane == 0) {
        rng_s[0] = lo * ens.iv.hi;
        rng_s[1] = hi * ens.iv.hi;
        rng_s[2] = small;
      }
    }
    __syncthreads();
    const float lo = rng_s[0], hi = rng_s[1];
    // an empty range (few rows, or a value that is not finite) or sums that overflow: no buckets
    bool plain = hi >= lo && fabsf(lo) < 1e36f && fabsf(hi) < 1e36f;
    if (plain && rng_s[2] > 0.f) {   // block-uniform: a look for sums that ens_value does not take
      const float limit = kEnsTiny * (float)(state[kStN] + 1);
      bool tiny = false;
      for (int64_t j = tid; j < N; j += kAucThreads) {
        const float t = ens.sum(j);
        tiny |= t != 0.f && fabsf(t) < limit;
      }
      plain = !__syncthreads_or(tiny);
    }
    bool buckets = plain;
    float scale = 0.f;
    if (buckets) {
      scale = (float)nb / (hi - lo);
      if (!(scale < 1e36f)) scale = 0.f;
    }
    auto bucket = [&](float v) {   // monotone: fp32 subtraction, product, truncation and clamp all are
      const int b = (int)__fmul_rn(__fsub_rn(v, lo), scale);
      return min(max(b, 0), nb - 1);
    };
    int64_t u2 = 0;   // twice the pairs a positive wins
    if (buckets) {
      uint32_t* hist = auc_sm;   // STAGED: two 16-bit counters per word
      const int words = STAGED ? nb / 2 : nb;
      uint32_t* keys = STAGED || n_few <= key_cap ? auc_sm + words : k0;
      uint8_t* place = reinterpret_cast<uint8_t*>(k0);   // STAGED: a key's place in its bucket
      for (int e = tid; e < words; e += kAucThreads) hist[e] = 0;
      __syncthreads();
#pragma unroll 4
      for (uint32_t i = tid; i < n_few; i += kAucThreads) {
        const float v = ens(few0 + i);
        const int b = bucket(v);
        if constexpr (STAGED) {
          const int sh = 16 * (b & 1);
          const uint32_t at = (atomicAdd(&hist[b >> 1], 1u << sh) >> sh) & 0xffffu;
          k1[i] = auc_key(v);
          place[i] = (uint8_t)min(at, 255u);   // a fuller bucket sends the candidate to the sort
        } else {
          atomicAdd(&hist[b], 1u);
        }
      }
      __syncthreads();
      // exclusive prefix, a run of words per warp, 32 at a time, and the
      // fullest bucket
      const int seg = words / 32, w0 = warp * seg;   // words: a power of two from 128 on
      uint32_t sum = 0, most = 0;
      for (int e = lane; e < seg; e += 32) {
        const uint32_t x = hist[w0 + e];
        const uint32_t c0 = STAGED ? x & 0xffffu : x, c1 = STAGED ? x >> 16 : 0u;
        sum += c0 + c1;
        most = max(most, max(c0, c1));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if (lane == 0) wtot[warp] = sum;
      buckets = !__syncthreads_or(most > (uint32_t)kAucBucketMax);
      if (buckets) {
        uint32_t run = 0;
        for (int w = 0; w < warp; ++w) run += wtot[w];
        for (int e0 = 0; e0 < seg; e0 += 32) {
          const bool in = e0 + lane < seg;
          const uint32_t x = in ? hist[w0 + e0 + lane] : 0u;
          const uint32_t c0 = STAGED ? x & 0xffffu : x, c1 = STAGED ? x >> 16 : 0u;
          uint32_t inc = c0 + c1;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
          }
          const uint32_t first = run + inc - (c0 + c1);
          if (in) hist[w0 + e0 + lane] = STAGED ? first | (first + c0) << 16 : first;
          run += __shfl_sync(0xffffffffu, inc, 31);
        }
        __syncthreads();
        const uint16_t* start = reinterpret_cast<const uint16_t*>(hist);
#pragma unroll 4
        for (uint32_t i = tid; i < n_few; i += kAucThreads) {
          if constexpr (STAGED) {
            const uint32_t key = k1[i];   // this thread's own of the first pass
            keys[start[bucket(auc_value(key))] + place[i]] = key;
          } else {   // placing a key moves its bucket's start on to the next bucket's
            const float v = ens(few0 + i);
            keys[atomicAdd(&hist[bucket(v)], 1u)] = auc_key(v);
          }
        }
        __syncthreads();
#pragma unroll 4
        for (uint32_t i = many0 + tid, left = my_many; left > 0; --left, i += kAucThreads) {
          const float v = ens(i);
          const uint32_t key = auc_key(v);
          const int b = bucket(v);
          const uint32_t s0 = STAGED ? (uint32_t)start[b] : b ? hist[b - 1] : 0u;
          const uint32_t s1 = STAGED ? (b + 1 < nb ? (uint32_t)start[b + 1] : n_few) : hist[b];
          // twice the keys below, plus the equal ones: [k < key] + [k <= key]
          uint32_t twice = 2 * s0;
          for (uint32_t t = s0; t < s1; ++t) {
            const uint32_t k = keys[t];
            twice += (k < key) + (k <= key);
          }
          u2 += few_pos ? 2u * n_few - twice : twice;   // below 2^32: n_few <= N / 2
        }
      }
      __syncthreads();
    }
    if (!buckets) {
      for (uint32_t i = tid; i < n_few; i += kAucThreads)
        k0[i] = auc_key(plain ? ens(few0 + i) : ens.exact(few0 + i));
      __syncthreads();
      auc_sort(k0, k1, n_few, auc_sm);
      __syncthreads();
      for (uint32_t i = many0 + tid, left = my_many; left > 0; --left, i += kAucThreads) {
        const uint32_t key = auc_key(plain ? ens(i) : ens.exact(i));
        uint32_t a = 0, z = n_few;                  // keys below this one
        while (a < z) {
          const uint32_t mid = (a + z) >> 1;
          if (k0[mid] < key) a = mid + 1; else z = mid;
        }
        const uint32_t less = a;
        z = n_few;                             // keys up to and equal to it
        while (a < z) {
          const uint32_t mid = (a + z) >> 1;
          if (k0[mid] <= key) a = mid + 1; else z = mid;
        }
        const uint32_t eq = a - less;
        u2 += 2 * (int64_t)(few_pos ? n_few - less - eq : less) + eq;
      }
    }
    u2 = auc_block_sum(u2, red);
    if (tid == 0) {
      double auc = __longlong_as_double(0x7ff8000000000000LL);
      if (n_pos > 0 && n_neg > 0) auc = 0.5 * (double)u2 / ((double)n_pos * (double)n_neg);
      partial[(int64_t)c * n_blk] = -auc;
    }
  }
  if (tid == 0) {
    __threadfence();
    last_s = atomicAdd(state + kStTicket, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  sel_pick<kAucThreads>(partial, P, n_blk, state, cur, m_ens, solo);
}

// ------------------------------------------------------------------ scratch
int64_t select_scratch_bytes(int32_t P, int64_t N, int32_t d_out, int32_t m_ens, int32_t score) {
  const int64_t n_blk = ceil_div(N, kSelRowsPerBlock);
  int64_t bytes = round_up(N * d_out * 8, 256) + round_up((int64_t)P * n_blk * 8, 256) + 256 +
                  round_up((int64_t)(kStHdr + m_ens + P) * 4, 256);
  if (score == kScoreAuc) bytes += round_up((int64_t)P * 2 * N * 4, 256) + round_up((int64_t)P * 2 * N, 256);
  return bytes;
}

// Optional scratch that makes the iterations cheaper, a buffer of its own:
// cross-entropy's compact label values where more than one iteration may read
// them (a pass over the predictions), S2 where it does not fit beside S.
int64_t select_extra_bytes(int32_t P, int64_t N, int32_t d_out, int32_t m_ens, int32_t score) {
  if (score == kScoreAuc || (score == 1 && d_out > 1)) return 0;
  if (d_out > 1) return m_ens > 1 ? (int64_t)P * N * 4 : 0;
  return N * 8;
}
void select_attach(SelectScratch& s, void* extra, int32_t d_out) {
  if (d_out > 1) s.comp = (float*)extra;
  else if (extra) s.S2 = (float2*)extra;
}

// ROC-AUC, in the 10 P N bytes after the state: the permuted predictions
// (4 P N), the value ranges (12 P), the sort buffers (2 of N / 2 keys per
// candidate: up to 4 P N) and, where it fits behind them, S2 (8 N); the row
// permutation (4 N) lies in the sort buffers, which are not in use yet.
// Below kAucMinRows rows the ranges are left out (they would not fit beside
// one or two rows).  Multiclass cross-entropy sums one value per row, so S2
// fits beside S.
SelectScratch select_carve(void* base, int32_t P, int64_t N, int32_t d_out, int32_t m_ens, int32_t score) {
  const int64_t n_blk = ceil_div(N, kSelRowsPerBlock);
  char* p = (char*)base;
  SelectScratch s;
  s.S = (double*)p;
  p += round_up(N * d_out * 8, 256);
  s.partial = (double*)p;
  p += round_up((int64_t)P * n_blk * 8, 256);
  s.cur = (double*)p;
  p += 256;
  s.state = (int32_t*)p;
  p += round_up((int64_t)(kStHdr + m_ens + P) * 4, 256);
  s.comp = nullptr;
  s.S2 = score == 0 && d_out > 1 ? (float2*)(s.S + N) : nullptr;
  s.pm = s.range = nullptr;
  s.srt = nullptr;
  s.perm = nullptr;
  if (score == kScoreAuc) {
    char* q = p;
    s.pm = (float*)q;
    q += (int64_t)P * N * 4;
    if (N >= kAucMinRows) {
      s.range = (float*)q;
      q += (int64_t)P * 12;
    }
    s.srt = (uint32_t*)q;
    q += (int64_t)P * 8 * (N / 2);
    const int64_t at = round_up(q - p, 8);
    if (N >= kAucMinRows && at + 8 * N <= (int64_t)P * 10 * N) s.S2 = (float2*)(p + at);
    // (a single candidate with an odd N: two keys short of the permutation, so the end, where no S2 fits)
    s.perm = (int64_t)P * 8 * (N / 2) >= 4 * N ? s.srt
                                               : (uint32_t*)(p + ((int64_t)P * 10 * N - 4 * N) / 4 * 4);
  }
  return s;
}

void select_prepare() {
  cudaFuncSetAttribute(k_sel_auc<0, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAucSmemMax);
  cudaFuncSetAttribute(k_sel_auc<1, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAucSmemMax);
  cudaFuncSetAttribute(k_sel_auc<0, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAucSmemMax);
  cudaFuncSetAttribute(k_sel_auc<1, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAucSmemMax);
}

// Enqueue the whole selection (m_ens iterations) on `st`; no host sync.
// Returns the number of the state words to copy back (header + selection).
int select_enqueue(cudaStream_t st, const SelectScratch& s, const float* preds, int32_t P, int64_t N,
                   int32_t d_out, const void* y, int32_t task, int32_t score, int32_t m_ens,
                   const uint8_t* excl, double* solo, int64_t* launches) {
  const int32_t n_blk = (int32_t)ceil_div(N, kSelRowsPerBlock);
  const int32_t n_state = kStHdr + m_ens + P;
  const bool multi_hit = score == 1 && task == 1;
  const int64_t n_S = multi_hit ? N * d_out : N;
  const unsigned add_blocks = (unsigned)std::min<int64_t>(ceil_div(n_S, 256), 152 * 8);
  k_sel_init<<<add_blocks, 256, 0, st>>>(s.S, s.S2, n_S, s.state, n_state, s.cur, excl, m_ens);
  int64_t nl = 1;
  if (score == kScoreAuc) {
    select_prepare();
    launch_pdl(k_auc_perm, dim3((unsigned)ceil_div(N, 256)), dim3(256), 0, st, (const int32_t*)y, N, s.perm,
               s.cur);
    launch_pdl(k_auc_permute, dim3(P), dim3(kAucThreads), 0, st, preds, (const uint32_t*)s.perm, N, s.pm, s.range);
    nl += 2;
    // staged: about one key of the smaller class per bucket; else about two,
    // and as many of its keys in shared memory as fit beside the buckets (the
    // others stay in the sort buffer)
    int nb = 256;
    while (nb < 32768 && nb * 2 < N) nb *= 2;
    const bool staged = N / 2 < 65536 && nb * 2 + (N / 2) * 4 <= kAucSmemMax;
    if (!staged) nb = 16384;
    const int64_t words = staged ? nb / 2 : nb;
    const int64_t key_cap = std::min<int64_t>(N / 2, kAucSmemMax / 4 - words);
    const size_t smem = std::max<size_t>(kAucSortSmem, (size_t)(words + key_cap) * 4);
    auto kernel = staged ? (s.S2 ? k_sel_auc<1, 1> : k_sel_auc<0, 1>) : (s.S2 ? k_sel_auc<1, 0> : k_sel_auc<0, 0>);
    for (int it = 0; it < m_ens; ++it) {
      launch_pdl(kernel, dim3(P), dim3(kAucThreads), smem, st, (const double*)s.S, (const float2*)s.S2, (const float*)s.pm,
                 N, s.state, s.partial, n_blk, P, m_ens, s.cur, it == 0 ? solo : (double*)nullptr, (const float*)s.range, s.srt, nb,
                 (int32_t)key_cap);
      launch_pdl(k_sel_add, dim3(add_blocks), dim3(256), 0, st, s.S, s.S2, SelVals{s.pm, N, 1, 0}, y, N, 1,
                 (const int32_t*)s.state);
      nl += 2;
    }
    if (launches) *launches += nl;
    return kStHdr + m_ens;
  }
  SelVals V{preds, N * d_out, multi_hit ? 1 : d_out, score == 0 && d_out > 1 ? 1 : 0};
  if (s.comp != nullptr && V.by_label) {
    launch_pdl(k_sel_compact, dim3((unsigned)n_blk, P), dim3(kSelThreads), 0, st, preds, (const int32_t*)y, N, d_out,
               s.comp);
    V = SelVals{s.comp, N, 1, 0};
    ++nl;
  }
  const dim3 grid((unsigned)n_blk, (unsigned)ceil_div(P, kSelGroup));
  for (int it = 0; it < m_ens; ++it) {
    double* so = it == 0 ? solo : nullptr;
    auto go = [&](auto kernel, size_t smem) {
      launch_pdl(kernel, grid, dim3(kSelThreads), smem, st, (const double*)s.S, (const float2*)s.S2, V, y, N, d_out, score, s.state,
                 s.partial, n_blk, P, m_ens, s.cur, so);
    };
    const bool split = s.S2 != nullptr;
    if (multi_hit) go(k_sel_score<kSelHitMulti, 0>, (size_t)d_out * kSelThreads * 4);
    else if (score == 1) go(split ? k_sel_score<kSelHitBinary, 1> : k_sel_score<kSelHitBinary, 0>, 0);
    else if (task == 2) go(split ? k_sel_score<kSelSquare, 1> : k_sel_score<kSelSquare, 0>, 0);
    else go(split ? k_sel_score<kSelLoss, 1> : k_sel_score<kSelLoss, 0>, 0);
    launch_pdl(k_sel_add, dim3(add_blocks), dim3(256), 0, st, s.S, s.S2, V, y, n_S, d_out,
               (const int32_t*)s.state);
    nl += 2;
  }
  if (launches) *launches += nl;
  return kStHdr + m_ens;
}

}  // namespace tp
