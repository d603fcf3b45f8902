// kernels.cu -- element-wise, reduction and CUDA-core matrix kernels of the
// packed training step (gather, CUDA-core grouped GEMM, head + loss + head
// AdamW, AdamW, init, predict head, mask dump).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "kernels.cuh"
#include "loss.cuh"
#include "two_float.cuh"

namespace tp {

// ------------------------------------------------------------------ gather
// Four values at once: 8-byte bf16 / 16-byte fp32 stores.
__device__ __forceinline__ void store4(__nv_bfloat16* p, float4 v) {
  uint2 u;
  __nv_bfloat162* b = reinterpret_cast<__nv_bfloat162*>(&u);
  b[0] = __floats2bfloat162_rn(v.x, v.y);
  b[1] = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(p) = u;
}
__device__ __forceinline__ void store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

// Eight columns of one class of a head-weight image (HeadSplit): thread t of
// all, eight per (chunk, class).
__device__ __forceinline__ void head_split(const HeadSplit& hs, int t) {
  const int per = hs.cp * 8, k = t / per;
  if (k >= hs.n) return;
  const HeadSplitJob jb = hs.jobs[k];
  const int c = (t - k * per) >> 3, g8 = t & 7, col = jb.col0 + 8 * g8;
  float e[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) e[j] = 0.f;
  if (c < hs.d_out && col < jb.w) {   // widths are multiples of 16
    const float4* p = reinterpret_cast<const float4*>(hs.params + jb.w_off + (int64_t)c * jb.w + col);
    const float4 a = p[0], b = p[1];
    e[0] = a.x; e[1] = a.y; e[2] = a.z; e[3] = a.w; e[4] = b.x; e[5] = b.y; e[6] = b.z; e[7] = b.w;
  }
  // A part is the rest rounded to bf16; past bf16's largest number it is cut
  // off (rounding would make it infinite), and an infinity leaves no rest
  // (infinity less itself is not a number, which every class would then take).
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    uint4 u;
    uint32_t* o = reinterpret_cast<uint32_t*>(&u);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float f = __bfloat162float(__float2bfloat16_rn(e[j]));
      if (isinf(f)) f = __uint_as_float(__float_as_uint(e[j]) & 0xFFFF0000u);
      e[j] = isinf(f) ? 0.f : e[j] - f;
      const uint32_t b = __float_as_uint(f) >> 16;
      o[j >> 1] = j & 1 ? o[j >> 1] | b << 16 : b;
    }
    const int row = q * hs.cp + c;
    *reinterpret_cast<uint4*>(hs.out + jb.out_off + row * 128 + ((g8 ^ (row & 7)) << 4)) = u;
  }
}

// xb[b, k] = X[idx[b], k] for b < B, k < d_in; zero for the rest of the first
// d_in_pad columns of rows < B_pad (column d_in_pad holds the constant 1).
// Grid: ceil(B_pad / 8) blocks of 8 warps, a row per warp.
// Block 0 also advances the step count of every active member and stores the
// AdamW bias corrections 1 - beta^t of the new step (when `advance`); the
// grid clears `zero[0 .. n_zero)` (the GEMMs' row-block completion counters).
// stacked != 0 (a batch per member, Sec. 3.6): blockIdx.y is an active
// member's index, whose rows are idx[member * B ..] and whose batch matrix
// starts xb_stride elements after the previous member's.
template <typename T>
__global__ void k_gather(const float* __restrict__ X, const int32_t* __restrict__ idx,
                         int32_t B, int32_t B_pad, int32_t d_in, int32_t d_in_pad, int32_t ldx, T* __restrict__ xb,
                         int32_t advance, int32_t* __restrict__ t_dev, float2* __restrict__ bias_corr,
                         const int32_t* __restrict__ active_ids, int32_t n_active, float ln_beta1,
                         float ln_beta2, int32_t* __restrict__ zero, int32_t n_zero, int32_t stacked,
                         int64_t xb_stride, HeadSplit hs, int32_t row_blocks) {
  pdl_trigger();
  pdl_wait();
  if ((int)blockIdx.x >= row_blocks) {   // blocks past the batch's: the head weights' parts
    if (blockIdx.y == 0) head_split(hs, ((int)blockIdx.x - row_blocks) * (int)blockDim.x + (int)threadIdx.x);
    return;
  }
  if (stacked) {
    const int member = active_ids[blockIdx.y];
    if (idx) idx += (int64_t)member * B;
    xb += (int64_t)member * xb_stride;
  }
  if (blockIdx.y == 0)
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n_zero; e += row_blocks * blockDim.x) zero[e] = 0;
  if (advance && blockIdx.x == 0 && blockIdx.y == 0) {
    for (int a = threadIdx.x; a < n_active; a += blockDim.x) {
      int i = active_ids[a];
      int t = t_dev[i] + 1;
      t_dev[i] = t;
      // Adam's bias corrections 1 - beta^t = -expm1(t ln beta), in fp32 to
      // about 1e-7 relative (fp64 runs at a small fraction of the fp32 rate)
      bias_corr[i] = make_float2(-expm1f((float)t * ln_beta1), -expm1f((float)t * ln_beta2));
    }
  }
  // one warp per batch row: float4 reads of the source row when it is
  // 16-byte aligned, four converted values written at once
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x * (blockDim.x >> 5) + warp;
  if (b >= B_pad) return;
  T* dst = xb + (int64_t)b * ldx;
  const bool live = b < B;
  const int64_t row = live ? (idx ? (int64_t)idx[b] : (int64_t)b) : 0;
  const float* src = X + row * d_in;
  int k0 = 0;
  if (live && (d_in & 3) == 0 && ((uintptr_t)src & 15) == 0) {
    const float4* s4 = reinterpret_cast<const float4*>(src);
    for (int c = lane; c < (d_in >> 2); c += 32) {
      store4(dst + 4 * c, __ldg(s4 + c));
    }
    k0 = d_in;
  }
  for (int k = k0 + lane; k < d_in_pad; k += 32) dst[k] = Elem<T>::from_f(live && k < d_in ? src[k] : 0.f);
}

// Column `col` of the first `rows` rows := 1 (xb and every act matrix, once).
template <typename T>
__global__ void k_fill_ones(const OnesJob* __restrict__ jobs, T* __restrict__ xb, T* __restrict__ act,
                            T* __restrict__ ex) {
  const OnesJob jb = jobs[blockIdx.x];
  T* base = (jb.arena == 0 ? xb : jb.arena == 1 ? act : ex) + jb.off;
  for (int r = threadIdx.x; r < jb.rows; r += blockDim.x) base[(int64_t)r * jb.ld + jb.col] = Elem<T>::from_f(1.f);
}

// ------------------------------------------------------- CUDA-core GEMM
// fp32 products: one BM x BN output tile per block, TM x TN outputs per
// thread, k-slabs of BK in two shared-memory buffers (the next slab's loads
// are in flight in registers while this one's products run).  Each output
// accumulates its k terms in increasing k order with fused multiply-adds, so
// the tile shape does not show in the result.  Bound by the fp32 pipe: the
// products are packed pairs (fma.rn.f32x2: two independent multiply-adds per
// lane and instruction), which leaves issue slots for the shared-memory reads.
// 128 x 64 with 8 x 8 per thread at 168 registers (three blocks per SM) keeps
// the fma pipe 72 % busy at 3 shared-memory wavefronts per read; capping the
// registers at 128 for a fourth block was 11 % slower, 128 x 128 tiles of 256
// threads 5 %.  Smaller tiles, for launches short of blocks, take slabs of 32:
// half the barriers and load latencies on a block's k loop.  The medium pack
// (32 members of 128..1024 columns, batch 500) takes 1.27 ms of products per
// step, 43 TFLOP/s; one 64 x 64 tile per block with unpaired products and no
// slab in flight took 3.34 ms.
// Loads are float4 along the operand's contiguous direction: every pitch, offset and
// column origin is a multiple of 4 elements.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// Four outputs of row r, columns c0 .. c0 + 3 (c0 < N a multiple of 4).
__device__ __forceinline__ void simt_store4(const GemmArgs<float>& g, const GemmProblem& P, const MemberDev& md,
                                            uint32_t step, int r, int c0, float4 v) {
  if (P.kind >= kNsGram) {  // Newton-Schulz: alpha acc + beta aux (N a multiple of 8)
    const float al = P.kind == kNsPoly ? kNsC : 1.f;
    const float be = P.kind == kNsPoly ? kNsB : (P.kind == kNsApply ? kNsA : 0.f);
    float4 o = make_float4(al * v.x, al * v.y, al * v.z, al * v.w);
    if (P.kind != kNsGram) {
      const float4 x = *reinterpret_cast<const float4*>(g.ns + P.aux_off + (int64_t)r * P.ld_aux + c0);
      o.x += be * x.x;
      o.y += be * x.y;
      o.z += be * x.z;
      o.w += be * x.w;
    }
    *reinterpret_cast<float4*>(g.ns + P.c_off + (int64_t)r * P.ldc + c0) = o;
  } else if (P.kind == kFwd) {  // N = w, a multiple of 16
    const uint32_t keep = g.train ? keep_bits4(g.seed, (uint32_t)P.member, (uint32_t)P.layer, step, (uint32_t)r,
                                               (uint32_t)(c0 >> 2), md.drop_T)
                                  : 0xFu;
    const float sc = g.train ? md.scale : 1.f;
    const float4 b = *reinterpret_cast<const float4*>(g.params + P.aux_off + c0);
    const float z[4] = {v.x + b.x, v.y + b.y, v.z + b.z, v.w + b.w};
    float o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) o[j] = ((keep >> j) & 1u) ? (z[j] > 0.f ? z[j] : 0.f) * sc : 0.f;
    *reinterpret_cast<float4*>(g.act + P.c_off + (int64_t)r * P.ldc + c0) = make_float4(o[0], o[1], o[2], o[3]);
  } else if (P.kind == kDgrad) {  // N = w (the first layer's input gradient: no mask, aux_off < 0)
    float4 o = v;
    if (P.aux_off >= 0) {
      const float4 h = *reinterpret_cast<const float4*>(g.act + P.aux_off + (int64_t)r * P.ld_aux + c0);
      o.x = h.x > 0.f ? v.x * md.scale : 0.f;
      o.y = h.y > 0.f ? v.y * md.scale : 0.f;
      o.z = h.z > 0.f ? v.z * md.scale : 0.f;
      o.w = h.w > 0.f ? v.w * md.scale : 0.f;
    }
    *reinterpret_cast<float4*>(g.dz + P.c_off + (int64_t)r * P.ldc + c0) = o;
  } else {  // weight gradient, N = in_pad, a multiple of 8
    *reinterpret_cast<float4*>(g.grads + P.c_off + (int64_t)r * P.ldc + c0) = v;
  }
}

template <int BM, int BN, int TM, int TN, int BK>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), BM == 128 ? 3 : 4) k_gemm_simt(GemmArgs<float> g, int32_t tile_base) {
  constexpr int NT = (BM / TM) * (BN / TN), TX = BN / TN;
  constexpr int LA = BM * BK / 4 / NT, LB = BN * BK / 4 / NT;   // float4 loads per thread and slab
  constexpr int PA = BM + 4, PB = BN + 4;
  constexpr int GM = TM / 4, GN = TN / 4;                       // groups of 4 rows / columns per thread
  constexpr int SM = BM / GM, SN = BN / GN;                     // distance between a thread's groups
  const GemmTile t = g.tiles[tile_base + blockIdx.x];   // the work list changes only while the stream is idle
  const GemmProblem P = g.probs[t.prob];
  pdl_wait();
  const int M = P.M ? P.M : g.B_pad;
  const int N = P.N;
  const int K = P.K ? P.K : g.B_pad;
  if (t.m0 >= M) return;
  const uint32_t step = g.step;
  auto base = [&](int src) {
    return src == kSrcXb ? g.xb : src == kSrcAct ? g.act : src == kSrcDz ? g.dz : src == kSrcWq ? g.wq
                                                                : src == kSrcNs ? g.ns : g.ex;
  };
  // stacked batches: the member's own batch matrix
  const int64_t xs = (int64_t)P.member * g.xb_stride;
  const float* A = base(P.a_src) + P.a_off + (P.a_src == kSrcXb ? xs : 0);
  const float* Bm = base(P.b_src) + P.b_off + (P.b_src == kSrcXb ? xs : 0);
  // contiguous along k (K-major) or along the output rows / columns
  const bool a_k = P.kind != kWgrad;
  const bool b_k = P.kind == kFwd || P.kind == kNsGram || P.kind == kNsPoly;
  __shared__ __align__(16) float As[2][BK][PA];
  __shared__ __align__(16) float Bs[2][BK][PB];
  const int tid = threadIdx.x;
  float4 ra[LA], rb[LB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < LA; ++q) {
      const int e = tid + q * NT;
      const int r = a_k ? e / (BK / 4) : 4 * (e % (BM / 4)), kk = a_k ? 4 * (e % (BK / 4)) : e / (BM / 4);
      const int gr = t.m0 + r, gk = k0 + kk;
      ra[q] = gr < M && gk < K
                  ? __ldg(reinterpret_cast<const float4*>(A + (a_k ? (int64_t)gr * P.lda + gk : (int64_t)gk * P.lda + gr)))
                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int q = 0; q < LB; ++q) {
      const int e = tid + q * NT;
      const int c = b_k ? e / (BK / 4) : 4 * (e % (BN / 4)), kk = b_k ? 4 * (e % (BK / 4)) : e / (BN / 4);
      const int gc = t.n0 + c, gk = k0 + kk;
      rb[q] = gc < N && gk < K
                  ? __ldg(reinterpret_cast<const float4*>(Bm + (b_k ? (int64_t)gc * P.ldb + gk : (int64_t)gk * P.ldb + gc)))
                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto stage = [&](int buf) {
#pragma unroll
    for (int q = 0; q < LA; ++q) {
      const int e = tid + q * NT;
      if (a_k) {
        const int r = e / (BK / 4), kk = 4 * (e % (BK / 4));
        As[buf][kk][r] = ra[q].x;
        As[buf][kk + 1][r] = ra[q].y;
        As[buf][kk + 2][r] = ra[q].z;
        As[buf][kk + 3][r] = ra[q].w;
      } else {
        *reinterpret_cast<float4*>(&As[buf][e / (BM / 4)][4 * (e % (BM / 4))]) = ra[q];
      }
    }
#pragma unroll
    for (int q = 0; q < LB; ++q) {
      const int e = tid + q * NT;
      if (b_k) {
        const int c = e / (BK / 4), kk = 4 * (e % (BK / 4));
        Bs[buf][kk][c] = rb[q].x;
        Bs[buf][kk + 1][c] = rb[q].y;
        Bs[buf][kk + 2][c] = rb[q].z;
        Bs[buf][kk + 3][c] = rb[q].w;
      } else {
        *reinterpret_cast<float4*>(&Bs[buf][e / (BN / 4)][4 * (e % (BN / 4))]) = rb[q];
      }
    }
  };
  uint64_t acc[TM][TN / 2];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;
  const int tx = tid % TX, ty = tid / TX;
  // Weight gradients: the tiles of column 0 also add up dZ's columns, a row
  // of theirs per thread, into the bias gradient.  (As a last column of ones
  // in B it cost a column tile of its own where in_pad is a multiple of 64.)
  const bool bias = P.kind == kWgrad && t.n0 == 0 && tid < BM;
  float bsum = 0.f;
  fetch(0);
  stage(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += BK, buf ^= 1) {
    if (k0 + BK < K) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[TM];
      uint64_t b[TN / 2];
#pragma unroll
      for (int i = 0; i < GM; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(&As[buf][kk][i * SM + 4 * ty]);
        a[4 * i] = v.x;
        a[4 * i + 1] = v.y;
        a[4 * i + 2] = v.z;
        a[4 * i + 3] = v.w;
      }
#pragma unroll
      for (int j = 0; j < GN; ++j) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][j * SN + 4 * tx]);
        b[2 * j] = v.x;
        b[2 * j + 1] = v.y;
      }
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const uint64_t aa = pack2(a[i], a[i]);
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) fma2(acc[i][j], aa, b[j]);
      }
    }
    if (bias)
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) bsum += As[buf][kk][tid];
    if (k0 + BK < K) {
      stage(buf ^ 1);   // last read one slab ago, before the barrier below
      __syncthreads();
    }
  }
  // The next launch's blocks may take their places now.  From the start of a
  // small grid on, they crowded onto the SMs that this one left idle: eight
  // small members, 140 us per step against 103 us (112 us without dependent
  // launches).
  pdl_trigger();
  if (bias && t.m0 + tid < M) g.grads[P.aux_off + t.m0 + tid] = bsum;
  const MemberDev md = g.mem[P.member];
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int r = t.m0 + (i / 4) * SM + 4 * ty + (i & 3);
    if (r >= M) continue;
#pragma unroll
    for (int j = 0; j < GN; ++j) {
      const int c0 = t.n0 + j * SN + 4 * tx;
      if (c0 >= N) continue;
      const float2 lo = unpack2(acc[i][2 * j]), hi = unpack2(acc[i][2 * j + 1]);
      simt_store4(g, P, md, step, r, c0, make_float4(lo.x, lo.y, hi.x, hi.y));
    }
  }
}

// ---------------------------------------------------------- vector helpers
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 8 consecutive values as floats (16-byte bf16 / 2 x 16-byte fp32 loads).
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&h)[8]) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  const __nv_bfloat16* b = reinterpret_cast<const __nv_bfloat16*>(&u);
#pragma unroll
  for (int k = 0; k < 8; ++k) h[k] = __bfloat162float(b[k]);
}
__device__ __forceinline__ void load8(const float* p, float (&h)[8]) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  h[0] = a.x; h[1] = a.y; h[2] = a.z; h[3] = a.w; h[4] = b.x; h[5] = b.y; h[6] = b.z; h[7] = b.w;
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float (&v)[8]) {
  uint4 u;
  __nv_bfloat162* b = reinterpret_cast<__nv_bfloat162*>(&u);
#pragma unroll
  for (int k = 0; k < 4; ++k) b[k] = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
  *reinterpret_cast<uint4*>(p) = u;
}
__device__ __forceinline__ void store8(float* p, const float (&v)[8]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}

// ------------------------------------------------------------- head + loss
// Values of G consecutive columns as floats, and back.
template <int G>
__device__ __forceinline__ void loadG(const __nv_bfloat16* p, float (&h)[G]) {
  if constexpr (G == 8) {
    load8(p, h);
  } else if constexpr (G == 4) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    const __nv_bfloat16* b = reinterpret_cast<const __nv_bfloat16*>(&u);
#pragma unroll
    for (int k = 0; k < 4; ++k) h[k] = __bfloat162float(b[k]);
  } else if constexpr (G == 2) {
    const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
    h[0] = f.x;
    h[1] = f.y;
  } else {
    h[0] = __bfloat162float(*p);
  }
}
template <int G>
__device__ __forceinline__ void loadG(const float* p, float (&h)[G]) {
  if constexpr (G == 8) {
    load8(p, h);
  } else if constexpr (G == 4) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    h[0] = a.x; h[1] = a.y; h[2] = a.z; h[3] = a.w;
  } else if constexpr (G == 2) {
    const float2 a = *reinterpret_cast<const float2*>(p);
    h[0] = a.x; h[1] = a.y;
  } else {
    h[0] = *p;
  }
}
template <int G>
__device__ __forceinline__ void storeG(__nv_bfloat16* p, const float (&v)[G]) {
  if constexpr (G == 8) {
    store8(p, v);
  } else if constexpr (G == 4) {
    uint2 u;
    __nv_bfloat162* b = reinterpret_cast<__nv_bfloat162*>(&u);
    b[0] = __floats2bfloat162_rn(v[0], v[1]);
    b[1] = __floats2bfloat162_rn(v[2], v[3]);
    *reinterpret_cast<uint2*>(p) = u;
  } else if constexpr (G == 2) {
    *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(v[0], v[1]);
  } else {
    *p = __float2bfloat16_rn(v[0]);
  }
}
template <int G>
__device__ __forceinline__ void storeG(float* p, const float (&v)[G]) {
  if constexpr (G == 8) {
    store8(p, v);
  } else if constexpr (G == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else if constexpr (G == 2) {
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  } else {
    *p = v[0];
  }
}

// G consecutive elements of T loaded with one vector load and converted to
// float when used, so that several rows' loads can be in flight at once.
template <typename T, int G>
struct RawG;
template <int G>
struct RawG<__nv_bfloat16, G> {
  using V = std::conditional_t<G == 8, uint4, std::conditional_t<G == 4, uint2,
                               std::conditional_t<G == 2, uint32_t, unsigned short>>>;
  V v;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { v = *reinterpret_cast<const V*>(p); }
  __device__ __forceinline__ void to_float(float (&h)[G]) const {
    const __nv_bfloat16* b = reinterpret_cast<const __nv_bfloat16*>(&v);
#pragma unroll
    for (int k = 0; k < G; ++k) h[k] = __bfloat162float(b[k]);
  }
};
template <int G>
struct RawG<float, G> {
  float v[G];
  __device__ __forceinline__ void load(const float* p) { loadG<G>(p, v); }
  __device__ __forceinline__ void to_float(float (&h)[G]) const {
#pragma unroll
    for (int k = 0; k < G; ++k) h[k] = v[k];
  }
};

// The logit pass of a head block (128 rows of one member, 8 warps of 16
// rows).  LPR lanes share a row (the smallest power of two >= the row's
// 8-column groups, at most 32; lanes walk the groups with 16-byte loads) and
// a warp's 32 / LPR lane groups take different rows, R rows per group at a
// time, so that every head-weight load serves R rows.  After the call the
// group's lane 0 holds the R rows' logits (bias added); `rl0` is the block-
// local index of the group's first row and `live` whether the group has
// rows in this pass.  Returns the number of passes.
template <typename T, int DO, int R>
struct HeadLogits {
  static constexpr int kRowsPerWarp = kHeadRows / 8;
  int lpr, groups, grp, gl;
  __device__ __forceinline__ HeadLogits(int w, int lane) {
    const int ng = w >> 3;
    lpr = 1;
    while (lpr < ng && lpr < 32) lpr <<= 1;
    groups = min(32 / lpr, kRowsPerWarp / R);
    grp = lane / lpr;
    gl = lane % lpr;
  }
  __device__ __forceinline__ int step() const { return groups * R; }
  // rows rl0 .. rl0 + R - 1 (block-local) of H (block origin), head weights Wh [d_out, w]
  __device__ __forceinline__ void run(const T* __restrict__ H, int ldh, const float* __restrict__ Wh,
                                      const float* __restrict__ bh, int w, int d_out,
                                      int rl0, bool live, float (&acc)[R][DO]) const {
#pragma unroll
    for (int q = 0; q < R; ++q)
#pragma unroll
      for (int c = 0; c < DO; ++c) acc[q][c] = 0.f;
    if (live) {
      // two-deep register pipeline over the column groups: the next group's
      // rows are in flight while this group's products run
      const int ng = w >> 3;
      RawG<T, 8> cur[R], nxt[R];
      if (gl < ng)
#pragma unroll
        for (int q = 0; q < R; ++q) cur[q].load(H + (int64_t)(rl0 + q) * ldh + 8 * gl);
      for (int gi = gl; gi < ng; gi += lpr) {
        if (gi + lpr < ng)
#pragma unroll
          for (int q = 0; q < R; ++q) nxt[q].load(H + (int64_t)(rl0 + q) * ldh + 8 * (gi + lpr));
        float h[R][8];
#pragma unroll
        for (int q = 0; q < R; ++q) cur[q].to_float(h[q]);
#pragma unroll
        for (int c = 0; c < DO; ++c) {
          if (c < d_out) {
            float w8[8];
            load8(Wh + (int64_t)c * w + 8 * gi, w8);
#pragma unroll
            for (int q = 0; q < R; ++q)
#pragma unroll
              for (int k = 0; k < 8; ++k) acc[q][c] = fmaf(h[q][k], w8[k], acc[q][c]);
          }
        }
#pragma unroll
        for (int q = 0; q < R; ++q) cur[q] = nxt[q];
      }
    }
    // sum over the group's lanes (every lane of the warp takes part)
    for (int o = lpr >> 1; o > 0; o >>= 1)
#pragma unroll
      for (int q = 0; q < R; ++q)
#pragma unroll
        for (int c = 0; c < DO; ++c)
          if (c < d_out) acc[q][c] += __shfl_xor_sync(0xffffffffu, acc[q][c], o);
#pragma unroll
    for (int q = 0; q < R; ++q)
#pragma unroll
      for (int c = 0; c < DO; ++c)
        if (c < d_out) acc[q][c] += bh[c];
  }
};

// Sum of a value of every row of the block (p[r * stride]), by one warp; the
// same bits in every lane.  With the labels asked for early (row_label): eight
// small members 316.3 -> 314.9 us per eight steps, 256 narrow ones 3034 -> 3021
// us per sixteen, sixteen wide ones 1919 -> 1909 us per step, against one thread
// adding the 64 rows in order.
__device__ __forceinline__ float rows_sum(const float* p, int stride, int lane) {
  static_assert(kHeadRows == 64, "two rows per lane");
  float v = p[lane * stride] + p[(lane + 32) * stride];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One block per (member, 128-row block), 256 threads.
//   1. logits, per-row loss and dlogits (HeadLogits; the group's lane 0 takes
//      the loss of its rows) into shared memory;
//   2. the gradient pass: a thread owns G = head_cols(DO) columns and keeps
//      their head weights and partial weight gradients in registers while it
//      walks its rows in order: dZ of the last hidden layer
//      = (dlogits W_h) * [H > 0] / (1 - p), and dW_h += dlogits^T H.  Narrow
//      heads split the rows into jb.split sets, added in order in shared
//      memory, so that every block writes one partial.
// One output: three blocks per SM (80 registers a thread, no spills; the
// kernel waits on memory, 64 to 68 us per wide step for three against two).
template <typename T, int DO>
__global__ void __launch_bounds__(256, DO == 1 ? 3 : 2) k_head(HeadArgs<T> g) {
  constexpr int R = DO <= 4 ? 4 : 2;
  constexpr int G = head_cols(DO);
  constexpr int DOP = DO == 1 ? 1 : (DO + 3) & ~3;  // padded row of dlogits in shared memory
  pdl_trigger();
  const HeadJob jb = g.jobs[blockIdx.x];   // the work list changes only while the stream is idle
  const int r0 = jb.blk * kHeadRows;
  const MemberDev md = g.mem[jb.member];
  pdl_wait();
  if (r0 >= g.B_pad) return;
  const int w = md.w, d_out = g.d_out, ldh = jb.h_ld;
  const T* __restrict__ H = g.act + jb.h_off + (int64_t)r0 * ldh;
  const float* __restrict__ Wh = g.params + jb.w_off;
  const float* __restrict__ bh = g.params + jb.b_off;
  __shared__ __align__(16) float dlog[kHeadRows][DOP];
  __shared__ float lrow[kHeadRows];
  __shared__ __align__(16) float red[256 * G * DO];  // row-set partials when the rows are split
  constexpr bool kColSums = std::is_same_v<T, __nv_bfloat16>;  // dZ column sums (tensor-core mode only)
  __shared__ __align__(16) float redz[kColSums ? 256 * G : 4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float invB = 1.f / (float)g.B;
  const int32_t* idx = g.idx ? g.idx + (int64_t)jb.member * g.idx_stride : nullptr;

  const HeadLogits<T, DO, R> hl(w, lane);
  for (int p0 = 0; p0 < HeadLogits<T, DO, R>::kRowsPerWarp; p0 += hl.step()) {
    const int rl0 = warp * HeadLogits<T, DO, R>::kRowsPerWarp + p0 + hl.grp * R;
    const bool live = hl.grp < hl.groups;
    const int rq = r0 + rl0 + hl.gl;   // this lane's first row
    const uint32_t label0 = live && hl.gl < R && rq < g.B ? row_label(g.y, idx, rq) : 0u;
    float acc[R][DO];
    hl.run(H, ldh, Wh, bh, w, d_out, rl0, live, acc);
    // the group's lanes take its R rows in turn (every lane holds the sums)
    for (int q = hl.gl; live && q < R; q += hl.lpr) {
      float z[DO];
#pragma unroll
      for (int c = 0; c < DO; ++c) z[c] = acc[0][c];
#pragma unroll
      for (int qq = 1; qq < R; ++qq)
        if (q == qq)
#pragma unroll
          for (int c = 0; c < DO; ++c) z[c] = acc[qq][c];
      const int r = r0 + rl0 + q;
      float dl[DO];
      float loss = 0.f;
#pragma unroll
      for (int c = 0; c < DO; ++c) dl[c] = 0.f;
      if (r < g.B) {
        loss = row_loss<DO>(g.task, d_out, z, q == hl.gl ? label0 : row_label(g.y, idx, r), invB, dl);
        float* lg = g.logits + ((int64_t)jb.member * g.B_cap + r) * d_out;
#pragma unroll
        for (int c = 0; c < DO; ++c)
          if (c < d_out) lg[c] = z[c];
      }
#pragma unroll
      for (int c = 0; c < DOP; ++c) dlog[rl0 + q][c] = c < DO ? dl[c < DO ? c : 0] : 0.f;
      lrow[rl0 + q] = loss;
    }
  }
  __syncthreads();

  const int n_cg = w / G;
  const int S = jb.split;
  const int rows_per_set = kHeadRows / S;
  T* __restrict__ dZ = g.dz + jb.dz_off + (int64_t)r0 * w;
  float* part = g.head_part + jb.part_off;
  float* dbp = kColSums && g.dbp && jb.colsum ? g.dbp + jb.dz_off / 32 + (int64_t)jb.blk * w : nullptr;
  for (int u = threadIdx.x; u < n_cg * S; u += blockDim.x) {
    const int cg = u % n_cg, set = u / n_cg;
    const int col = G * cg;
    float Wr[DO][G], a[DO][G], cz[G];
#pragma unroll
    for (int k = 0; k < G; ++k) cz[k] = 0.f;
#pragma unroll
    for (int c = 0; c < DO; ++c) {
      if (c < d_out) loadG<G>(Wh + (int64_t)c * w + col, Wr[c]);
      else {
#pragma unroll
        for (int k = 0; k < G; ++k) Wr[c][k] = 0.f;
      }
#pragma unroll
      for (int k = 0; k < G; ++k) a[c][k] = 0.f;
    }
    const int rb = set * rows_per_set;
    // rows in batches of U (rows_per_set is a multiple of 8): the batch's
    // loads are all issued before its products
    constexpr int U = G * DO >= 32 ? 4 : 8;
    for (int rb0 = rb; rb0 < rb + rows_per_set; rb0 += U) {
      RawG<T, G> raw[U];
#pragma unroll
      for (int u2 = 0; u2 < U; ++u2) raw[u2].load(H + (int64_t)(rb0 + u2) * ldh + col);
#pragma unroll
      for (int u2 = 0; u2 < U; ++u2) {
      const int rr = rb0 + u2;
      float h[G], s[G];
      raw[u2].to_float(h);
      float dl[DOP];
      if constexpr (DOP % 4 == 0) {
#pragma unroll
        for (int c = 0; c < DOP; c += 4) {
          const float4 v = *reinterpret_cast<const float4*>(&dlog[rr][c]);
          dl[c] = v.x; dl[c + 1] = v.y; dl[c + 2] = v.z; dl[c + 3] = v.w;
        }
      } else {
#pragma unroll
        for (int c = 0; c < DOP; ++c) dl[c] = dlog[rr][c];
      }
#pragma unroll
      for (int k = 0; k < G; ++k) s[k] = 0.f;
#pragma unroll
      for (int c = 0; c < DO; ++c)
#pragma unroll
        for (int k = 0; k < G; ++k) {
          s[k] = fmaf(dl[c], Wr[c][k], s[k]);
          a[c][k] = fmaf(dl[c], h[k], a[c][k]);
        }
#pragma unroll
      for (int k = 0; k < G; ++k) {
        s[k] = h[k] > 0.f ? s[k] * md.scale : 0.f;
        if constexpr (kColSums)
          if (dbp) cz[k] += __bfloat162float(__float2bfloat16_rn(s[k]));  // dZ as stored
      }
      storeG<G>(dZ + (int64_t)rr * w + col, s);
      }
    }
    if (S == 1) {
#pragma unroll
      for (int c = 0; c < DO; ++c)
        if (c < d_out) storeG<G>(part + (int64_t)c * w + col, a[c]);
      if (dbp) storeG<G>(dbp + col, cz);
    } else {  // n_cg * S <= 256: one (column group, row set) per thread
#pragma unroll
      for (int c = 0; c < DO; ++c)
        if (c < d_out) storeG<G>(&red[((set * DO + c) * n_cg + cg) * G], a[c]);
      if constexpr (kColSums) storeG<G>(&redz[(set * n_cg + cg) * G], cz);
    }
  }
  if (S > 1) {  // the block's partial: row sets added in order
    __syncthreads();
    for (int e = threadIdx.x; e < d_out * w; e += blockDim.x) {
      const int c = e / w, k = e - c * w;
      const int cg = k / G, kk = k - cg * G;
      float v = 0.f;
      for (int set = 0; set < S; ++set) v += red[((set * DO + c) * n_cg + cg) * G + kk];
      part[e] = v;
    }
    if (dbp)
      for (int e = threadIdx.x; e < w; e += blockDim.x) {
        const int cg = e / G, kk = e - cg * G;
        float v = 0.f;
        for (int set = 0; set < S; ++set) v += redz[(set * n_cg + cg) * G + kk];
        dbp[e] = v;
      }
  }
  // bias and loss partials of the block
  for (int c = warp; c <= d_out; c += 8) {
    const float v = c < d_out ? rows_sum(&dlog[0][c], DOP, lane) : rows_sum(lrow, 1, lane);
    if (lane == 0) (c < d_out ? part[(int64_t)d_out * w + c] : g.loss_part[(int64_t)jb.member * g.n_blk_cap + jb.blk]) = v;
  }
}

constexpr int kStageWarps = 8;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ----------------------------------- one-output head + loss, staged (bf16)
// The same work as k_head for a one-output member up to 512 wide on one 64-row
// block in bf16 mode, with the block's H_L rows (one bulk copy per row) and the head weights (one
// bulk copy) staged in shared memory, so that H is read from HBM once and
// both passes run from shared memory:
//   1. logits: warp v takes the 8-column groups v, v + 8, ... and lane l rows
//      l and l + 32 (16-byte loads; the row pitch is 16 bytes past a
//      multiple of 128, so the eight rows of a quarter-warp fall in distinct
//      banks), with the head weights read warp-uniformly (broadcast); the
//      eight warps' partial logits are added in warp order through shared
//      memory, and one thread per row takes its loss and dlogit;
//   2. gradients: a thread owns 4 consecutive columns of a row set and walks
//      its rows: dZ = dlogit W_h [H > 0] / (1 - p) stored in bf16, dW_h
//      partials in registers; row sets (narrow members) are added in order
//      through shared memory.
// Shared memory: H [64][pitch] | W_h [w] | partial logits [8][64] |
// dlogits [64] | row losses [64] | mbarrier.
__global__ void __launch_bounds__(256) k_head_stage(HeadArgs<__nv_bfloat16> g) {
  // no early trigger: the next kernels' CTAs (the backward GEMM's hold most
  // of an SM's shared memory) must not park beside these blocks
  const HeadJob jb = g.jobs[blockIdx.x];   // the work list changes only while the stream is idle
  const int r0 = jb.blk * kHeadRows;
  const MemberDev md = g.mem[jb.member];
  pdl_wait();
  if (r0 >= g.B_pad) return;
  const int w = md.w, ldh = jb.h_ld;
  const int pitch = head_stage_pitch(w);
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* Hs = smem;
  float* Ws = reinterpret_cast<float*>(smem + (int64_t)kHeadRows * pitch);      // [w]
  float* zpart = Ws + w;                                                        // [8][64]
  float* dlog = zpart + kStageWarps * kHeadRows;                               // [64]
  float* lrow = dlog + kHeadRows;                                               // [64]
  uint64_t* bar = reinterpret_cast<uint64_t*>(lrow + kHeadRows + 2);            // 8-byte aligned
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const __nv_bfloat16* __restrict__ H = g.act + jb.h_off + (int64_t)r0 * ldh;
  const float* __restrict__ Wg = g.params + jb.w_off;
  const uint32_t row_bytes = (uint32_t)w * 2u;
  const uint32_t w_bytes = (uint32_t)w * 4u;

  // this thread's row of the loss: its label comes while the copies are in flight
  const bool has_row = threadIdx.x < kHeadRows && r0 + (int)threadIdx.x < g.B;
  const int32_t* idx = g.idx ? g.idx + (int64_t)jb.member * g.idx_stride : nullptr;
  uint32_t label = 0;

  // stage the 64 rows and the head weights (warp 0 issues the bulk copies)
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  if (warp == 0) {
    if (lane == 0) {
      asm volatile("fence.proxy.async.global;" ::: "memory");
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                   "r"(row_bytes * (uint32_t)kHeadRows + w_bytes)
                   : "memory");
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
              smem_addr(Ws)),
          "l"(Wg), "r"(w_bytes), "r"(smem_addr(bar))
          : "memory");
    }
    __syncwarp();
    for (int r = lane; r < kHeadRows; r += 32)
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
              smem_addr(Hs + (int64_t)r * pitch)),
          "l"(H + (int64_t)r * ldh), "r"(row_bytes), "r"(smem_addr(bar))
          : "memory");
  }
  if (has_row) label = row_label(g.y, idx, r0 + threadIdx.x);
  {  // bounded wait for the copies (2 s); on expiry record site 20 and leave
    uint32_t ok = 0;
    uint64_t t0 = 0;
    for (int it = 0;; ++it) {
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}\n"
          : "=r"(ok)
          : "r"(smem_addr(bar))
          : "memory");
      if (ok) break;
      uint64_t t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (it == 0) {
        t0 = t;
      } else if (t - t0 > 2000000000ull) {
        if (g.err) atomicCAS(g.err, 0, 20);
        return;
      }
    }
  }

  // 1. logits
  {
    float acc[2] = {0.f, 0.f};
    const int ng = w >> 3;
#pragma unroll 2
    for (int gi = warp; gi < ng; gi += kStageWarps) {
      float h[2][8];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const uint4 v = *reinterpret_cast<const uint4*>(Hs + (int64_t)(lane + 32 * q) * pitch + 16 * gi);
        const __nv_bfloat16* b = reinterpret_cast<const __nv_bfloat16*>(&v);
#pragma unroll
        for (int k = 0; k < 8; ++k) h[q][k] = __bfloat162float(b[k]);
      }
      const float4 wa = *reinterpret_cast<const float4*>(Ws + 8 * gi);
      const float4 wb = *reinterpret_cast<const float4*>(Ws + 8 * gi + 4);
      const float w8[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[q] = fmaf(h[q][k], w8[k], acc[q]);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) zpart[warp * kHeadRows + lane + 32 * q] = acc[q];
  }
  __syncthreads();
  if (threadIdx.x < kHeadRows) {
    const int rl = threadIdx.x, r = r0 + rl;
    float v = 0.f;
    for (int v8 = 0; v8 < kStageWarps; ++v8) v += zpart[v8 * kHeadRows + rl];
    const float z[1] = {v + g.params[jb.b_off]};
    float dl[1] = {0.f}, loss = 0.f;
    if (has_row) {
      loss = row_loss<1>(g.task, 1, z, label, 1.f / (float)g.B, dl);
      g.logits[(int64_t)jb.member * g.B_cap + r] = z[0];
    }
    dlog[rl] = dl[0];
    lrow[rl] = loss;
  }
  __syncthreads();

  // 2. dZ of the last hidden layer and the head-weight gradient partial
  const int n_cg = w >> 2;
  const int S = head_stage_split(w);
  const int rows_per_set = kHeadRows / S;
  __nv_bfloat16* __restrict__ dZ = g.dz + jb.dz_off + (int64_t)r0 * w;
  float* part = g.head_part + jb.part_off;
  float* dbp = g.dbp && jb.colsum ? g.dbp + jb.dz_off / 32 + (int64_t)jb.blk * w : nullptr;
  float a[4] = {0.f, 0.f, 0.f, 0.f}, cz[4] = {0.f, 0.f, 0.f, 0.f};
  int cg = 0, set = 0;
  for (int u = threadIdx.x; u < n_cg * S; u += blockDim.x) {
    cg = u % n_cg;
    set = u / n_cg;
    const int col = 4 * cg;
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = cz[k] = 0.f;
    const float4 wv = *reinterpret_cast<const float4*>(Ws + col);
    const float Wr[4] = {wv.x, wv.y, wv.z, wv.w};
    const int rb = set * rows_per_set;
#pragma unroll 4
    for (int rr = rb; rr < rb + rows_per_set; ++rr) {
      const uint2 hv = *reinterpret_cast<const uint2*>(Hs + (int64_t)rr * pitch + 2 * col);
      const __nv_bfloat16* hb = reinterpret_cast<const __nv_bfloat16*>(&hv);
      float h[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) h[k] = __bfloat162float(hb[k]);
      const float dl = dlog[rr];
#pragma unroll
      for (int k = 0; k < 4; ++k) a[k] = fmaf(dl, h[k], a[k]);
      __align__(8) __nv_bfloat16 o[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        o[k] = __float2bfloat16_rn(h[k] > 0.f ? fmaf(dl, Wr[k], 0.f) * md.scale : 0.f);
        if (dbp) cz[k] += __bfloat162float(o[k]);  // dZ as stored
      }
      *reinterpret_cast<uint2*>(dZ + (int64_t)rr * w + col) = *reinterpret_cast<const uint2*>(o);
    }
    if (S == 1) {
      *reinterpret_cast<float4*>(part + col) = make_float4(a[0], a[1], a[2], a[3]);
      if (dbp) *reinterpret_cast<float4*>(dbp + col) = make_float4(cz[0], cz[1], cz[2], cz[3]);
    }
  }
  if (S > 1) {  // one (column group, row set) per thread; sets added in order (the H area is free now)
    __syncthreads();
    float* red = reinterpret_cast<float*>(Hs);   // [S][w], then [S][w] of dZ column sums:
    float* redz = red + (int64_t)S * w;          // 2 S w <= 16 w floats fit in 64 rows of H
    if (threadIdx.x < n_cg * S) {
      *reinterpret_cast<float4*>(red + (int64_t)set * w + 4 * cg) = make_float4(a[0], a[1], a[2], a[3]);
      *reinterpret_cast<float4*>(redz + (int64_t)set * w + 4 * cg) = make_float4(cz[0], cz[1], cz[2], cz[3]);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < w; e += blockDim.x) {
      float v = 0.f;
      for (int st = 0; st < S; ++st) v += red[(int64_t)st * w + e];
      part[e] = v;
    }
    if (dbp)
      for (int e = threadIdx.x; e < w; e += blockDim.x) {
        float v = 0.f;
        for (int st = 0; st < S; ++st) v += redz[(int64_t)st * w + e];
        dbp[e] = v;
      }
  }
  pdl_trigger();
  // bias and loss partials of the block
  if (warp < 2) {
    const float v = rows_sum(warp == 0 ? dlog : lrow, 1, lane);
    if (lane == 0) (warp == 0 ? part[w] : g.loss_part[(int64_t)jb.member * g.n_blk_cap + jb.blk]) = v;
  }
}

// ------------------------------------------ one-output head, one pass (bf16)
// The head of a one-output task (binary or regression) for one member on one
// 64-row block, with H_L read once.  The block's 256 threads form S = 256 / T
// row sets of T threads (T = w / 8 rounded up to a power of two, at least
// 32); thread t of a set owns the 8-column group t, keeps its head weights
// and its partial weight gradient in registers, and walks the set's rows
// kOneRows at a time with the next rows' 16-byte loads in flight:
//   1. partial logits of the rows, summed over the warp by shuffles and over
//      the set's warps in warp order through shared memory, bias added; one
//      thread per row takes its loss and dlogit;
//   2. dZ of the last hidden layer = dlogit W_h [H > 0] / (1 - p) stored in
//      bf16, and dW_h += dlogit H.
// The sets' partials are added in set order, so each block writes one
// partial of dW_h, db_h and the loss, the layout k_head
// writes for k_head_reduce, and (dbp) the column sums of its dZ rows.
// Widths up to 2048.
constexpr int kOneRows = 8;

__global__ void __launch_bounds__(256, 2) k_head_one(HeadArgs<__nv_bfloat16> g) {
  pdl_trigger();
  const HeadJob jb = g.jobs[blockIdx.x];   // the work list changes only while the stream is idle
  const int r0 = jb.blk * kHeadRows;
  const MemberDev md = g.mem[jb.member];
  pdl_wait();
  if (r0 >= g.B_pad) return;
  const int w = md.w, ldh = jb.h_ld, ng = w >> 3;
  int T = 32;
  while (T < ng) T <<= 1;
  const int S = 256 / T, set = threadIdx.x / T, t = threadIdx.x % T;
  const int rows_set = kHeadRows / S, n_steps = rows_set / kOneRows, wpset = T >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool has = t < ng;
  const int col = 8 * t;
  __shared__ float zp[8][kOneRows];
  __shared__ float dls[8][kOneRows];
  __shared__ float dlrow[kHeadRows], lrow[kHeadRows];
  __shared__ uint32_t ysm[kHeadRows];
  __shared__ __align__(16) float red[8 * 256];  // [S][w]: S * w <= 8 * T * S = 2048
  __shared__ __align__(16) float redz[8 * 256]; // the same for the column sums of dZ
  const __nv_bfloat16* __restrict__ H = g.act + jb.h_off + (int64_t)(r0 + set * rows_set) * ldh + col;
  __nv_bfloat16* __restrict__ dZ = g.dz + jb.dz_off + (int64_t)(r0 + set * rows_set) * w + col;
  const float bias = g.params[jb.b_off];
  const float invB = 1.f / (float)g.B;
  const int32_t* idx = g.idx ? g.idx + (int64_t)jb.member * g.idx_stride : nullptr;
  float Wr[8], a[8], cz[8];
  if (has) load8(g.params + jb.w_off + col, Wr);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    if (!has) Wr[k] = 0.f;
    a[k] = 0.f;
    cz[k] = 0.f;
  }
  uint4 cur[kOneRows], nxt[kOneRows];
#pragma unroll
  for (int u = 0; u < kOneRows; ++u) {
    cur[u] = has ? *reinterpret_cast<const uint4*>(H + (int64_t)u * ldh) : make_uint4(0u, 0u, 0u, 0u);
    nxt[u] = make_uint4(0u, 0u, 0u, 0u);
  }
  // the rows' labels, while the first rows are in flight (read after the
  // first step's barrier)
  uint32_t label = 0;
  if (threadIdx.x < kHeadRows && r0 + (int)threadIdx.x < g.B) label = row_label(g.y, idx, r0 + threadIdx.x);
  for (int st = 0; st < n_steps; ++st) {
    if (has && st + 1 < n_steps)
#pragma unroll
      for (int u = 0; u < kOneRows; ++u)
        nxt[u] = *reinterpret_cast<const uint4*>(H + (int64_t)((st + 1) * kOneRows + u) * ldh);
    // 1. logits of the set's kOneRows rows
    float p[kOneRows];
#pragma unroll
    for (int u = 0; u < kOneRows; ++u) {
      const __nv_bfloat16* b = reinterpret_cast<const __nv_bfloat16*>(&cur[u]);
      float s = 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k) s = fmaf(__bfloat162float(b[k]), Wr[k], s);
      p[u] = s;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < kOneRows; ++u) p[u] += __shfl_xor_sync(0xffffffffu, p[u], o);
    if (lane == 0)
#pragma unroll
      for (int u = 0; u < kOneRows; ++u) zp[warp][u] = p[u];
    if (st == 0 && threadIdx.x < kHeadRows) ysm[threadIdx.x] = label;
    __syncthreads();
    if (threadIdx.x < S * kOneRows) {
      const int s2 = threadIdx.x / kOneRows, u = threadIdx.x % kOneRows;
      float zz[1] = {0.f};
      for (int v = 0; v < wpset; ++v) zz[0] += zp[s2 * wpset + v][u];
      zz[0] += bias;
      const int rl = s2 * rows_set + st * kOneRows + u, r = r0 + rl;
      float dl[1] = {0.f}, loss = 0.f;
      if (r < g.B) {
        loss = row_loss<1>(g.task, 1, zz, ysm[rl], invB, dl);
        g.logits[(int64_t)jb.member * g.B_cap + r] = zz[0];
      }
      dls[s2][u] = dl[0];
      dlrow[rl] = dl[0];
      lrow[rl] = loss;
    }
    __syncthreads();
    // 2. dZ of the last hidden layer and the weight-gradient partial
#pragma unroll
    for (int u = 0; u < kOneRows; ++u) {
      const float dl = dls[set][u];
      const __nv_bfloat16* b = reinterpret_cast<const __nv_bfloat16*>(&cur[u]);
      float o[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float h = __bfloat162float(b[k]);
        o[k] = h > 0.f ? (dl * Wr[k]) * md.scale : 0.f;
        a[k] = fmaf(dl, h, a[k]);
      }
      uint4 pz;
      __nv_bfloat162* pb = reinterpret_cast<__nv_bfloat162*>(&pz);
#pragma unroll
      for (int k = 0; k < 4; ++k) pb[k] = __floats2bfloat162_rn(o[2 * k], o[2 * k + 1]);
      if (has) *reinterpret_cast<uint4*>(dZ + (int64_t)(st * kOneRows + u) * w) = pz;
      if (jb.colsum) {  // column sums of dZ as stored
        const uint32_t* pw = reinterpret_cast<const uint32_t*>(&pz);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          cz[2 * k] += __uint_as_float(pw[k] << 16);
          cz[2 * k + 1] += __uint_as_float(pw[k] & 0xFFFF0000u);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kOneRows; ++u) cur[u] = nxt[u];
  }
  float* part = g.head_part + jb.part_off;
  float* dbp = g.dbp && jb.colsum ? g.dbp + jb.dz_off / 32 + (int64_t)jb.blk * w : nullptr;
  if (S == 1) {
    if (has) {
      store8(part + col, a);
      if (dbp) store8(dbp + col, cz);
    }
  } else {  // the sets' partials added in set order
    if (has) {
      store8(red + set * w + col, a);
      store8(redz + set * w + col, cz);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < w; e += blockDim.x) {
      float v = 0.f, vz = 0.f;
      for (int s2 = 0; s2 < S; ++s2) {
        v += red[s2 * w + e];
        vz += redz[s2 * w + e];
      }
      part[e] = v;
      if (dbp) dbp[e] = vz;
    }
  }
  // bias and loss partials of the block
  if (warp < 2) {
    const float v = rows_sum(warp == 0 ? dlrow : lrow, 1, lane);
    if (lane == 0) (warp == 0 ? part[w] : g.loss_part[(int64_t)jb.member * g.n_blk_cap + jb.blk]) = v;
  }
}

// Sum the per-block head partials (fixed order) into the head gradients and
// the per-member mean loss; in update mode apply the member's AdamW to the
// head parameters directly (the gradients are not stored).  Grid: member x
// chunks of 256 head parameters; inactive members report NaN.
__global__ void k_head_reduce(HeadReduceArgs g) {
  pdl_trigger();
  pdl_wait();
  const int i = blockIdx.x;
  const HeadReduceJob jb = g.jobs[i];
  const int n_blk = g.B_pad / g.blk_rows;
  if (!g.active[i]) {
    float* lo = g.loss_out;
    if (blockIdx.y == 0 && threadIdx.x == 0 && lo) lo[i] = __int_as_float(0x7fc00000);
    return;
  }
  const int w = jb.w, d_out = g.d_out;
  const int e0 = blockIdx.y * blockDim.x;
  if (e0 >= d_out * w + d_out) return;
  const int64_t stride = g.part_stride[i];
  float lr = 0.f, wdw = 0.f, wdb = 0.f, ib1 = 1.f, ib2 = 1.f;
  if (g.update) {
    const MemberDev md = g.adam.mem[i];
    const float2 bc = g.adam.bias_corr[i];
    lr = md.lr;
    wdw = md.wd;
    wdb = g.adam.wd_on_bias ? md.wd : 0.f;
    ib1 = 1.f / bc.x;
    ib2 = 1.f / bc.y;
  }
  for (int e = e0 + threadIdx.x; e < min(e0 + (int)blockDim.x, d_out * w + d_out); e += blockDim.x) {
    float s = 0.f;
#pragma unroll 8
    for (int b = 0; b < n_blk; ++b) s += g.head_part[jb.part_off + b * stride + e];
    const bool is_b = e >= d_out * w;
    const int64_t o = is_b ? jb.gb_off + (e - d_out * w) : jb.gw_off + e;
    if (g.update) {
      float p = g.adam.params[o], m = g.adam.m[o], v = g.adam.v[o];
      adamw_elem(p, m, v, s, lr, is_b ? wdb : wdw, g.adam.beta1, g.adam.beta2, g.adam.eps, ib1, ib2);
      g.adam.params[o] = p;
      g.adam.m[o] = m;
      g.adam.v[o] = v;
      if (g.adam.wq_out) g.adam.wq_out[o] = __float2bfloat16_rn(p);
    } else {
      g.grads[o] = s;
    }
  }
  if (blockIdx.y == 0 && threadIdx.x == 0) {
    float s = 0.f;
    for (int b = 0; b < n_blk; ++b) s += g.loss_part[(int64_t)i * g.n_blk_cap + b];
    const float loss = s / (float)g.B;
    float* lo = g.loss_out;
    if (lo) lo[i] = loss;
    g.loss_last[i] = loss;
  }
}

// ------------------------------------------------------------------ AdamW
// Stand-alone AdamW over chunks of the arena (unless AdamW is fused into the
// weight-gradient epilogue), with the member's lr and wd and its step's bias
// corrections; float4 body, scalar tail.  In bf16 mode the same threads
// first fill the dropout mask arena for the next step.
// Head chunks (the first n_head in the list) take their gradients from the
// head kernel's per-block partials, added in block order, and store them;
// the bias chunk's block also takes the member's mean loss.  This is
// k_head_reduce's work without its launch (5 to 11 us on the step's chain;
// eight small members 56 -> 50 us per step together with 1024-element chunks).
// At the copy rate; 48 registers leave five blocks per SM, which is best.  Bound
// to six (40 registers, 20 bytes spilled) a whole pass of the large pack takes
// 2015 us against 2004, of the wide one 1924 against 1914, of the narrow one
// the same; to seven (32, 68 bytes) 3 % more, to four (57) 2 %; two float4 in
// flight per thread 0.3 % more at five blocks and 2.3 % at four.
__global__ void __launch_bounds__(256) k_adamw(AdamArgs g) {
  pdl_trigger();
  // the work lists change only while the stream is idle: read before the wait
  const Chunk ch = g.chunks[blockIdx.x];
  const Segment s = g.segs[ch.seg];
  const MemberDev md = g.mem[s.member];
  pdl_wait();
  const float2 bc = g.bias_corr[s.member];
  const float lr = md.lr;
  const float wd = (s.is_bias && !g.wd_on_bias) ? 0.f : md.wd;
  const float b1 = g.beta1, b2 = g.beta2, eps = g.eps;
  const float ib1 = 1.f / bc.x, ib2 = 1.f / bc.y;
  if ((int)blockIdx.x < g.n_head) {   // block-uniform
    const HeadPartials& hp = g.head;
    const int n_blk = hp.B_pad / hp.blk_rows;
    const int64_t stride = hp.part_stride[s.member];
    const int32_t e0 = (int32_t)(ch.off - s.off) + (s.is_bias ? hp.d_out * hp.jobs[s.member].w : 0);
    const float* part = hp.part + hp.jobs[s.member].part_off + e0;
    for (int e = threadIdx.x; e < ch.len; e += blockDim.x) {
      float gr = 0.f;
#pragma unroll 8
      for (int b = 0; b < n_blk; ++b) gr += part[b * stride + e];
      const int64_t o = ch.off + e;
      float p = g.params[o], m = g.m[o], v = g.v[o];
      adamw_elem(p, m, v, gr, lr, wd, b1, b2, eps, ib1, ib2);
      g.grads[o] = gr;
      g.params[o] = p;
      g.m[o] = m;
      g.v[o] = v;
      if (g.wq) g.wq[o] = __float2bfloat16_rn(p);
    }
    if (s.is_bias && threadIdx.x == 0) {
      float sum = 0.f;
#pragma unroll 8
      for (int b = 0; b < n_blk; ++b) sum += hp.loss_part[(int64_t)s.member * hp.n_blk_cap + b];
      const float loss = sum / (float)hp.B;
      float* lo = hp.loss_out;
      if (lo) lo[s.member] = loss;
      hp.loss_last[s.member] = loss;
    }
    if (blockIdx.x == 0) {   // inactive members report NaN
      float* lo = hp.loss_out;
      for (int i = threadIdx.x; lo && i < hp.m; i += blockDim.x)
        if (!hp.active[i]) lo[i] = __int_as_float(0x7fc00000);
    }
    fill_masks(g.mg, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x);
    return;
  }
  const int n4 = ch.len >> 2;  // chunk offsets are multiples of 4 elements
  float4* P4 = reinterpret_cast<float4*>(g.params + ch.off);
  const float4* G4 = reinterpret_cast<const float4*>(g.grads + ch.off);
  float4* M4 = reinterpret_cast<float4*>(g.m + ch.off);
  float4* V4 = reinterpret_cast<float4*>(g.v + ch.off);
  for (int e = threadIdx.x; e < n4; e += blockDim.x) {
    float4 p = P4[e], m = M4[e], v = V4[e];
    const float4 gr = __ldcs(G4 + e);
    adamw_elem(p.x, m.x, v.x, gr.x, lr, wd, b1, b2, eps, ib1, ib2);
    adamw_elem(p.y, m.y, v.y, gr.y, lr, wd, b1, b2, eps, ib1, ib2);
    adamw_elem(p.z, m.z, v.z, gr.z, lr, wd, b1, b2, eps, ib1, ib2);
    adamw_elem(p.w, m.w, v.w, gr.w, lr, wd, b1, b2, eps, ib1, ib2);
    P4[e] = p;
    M4[e] = m;
    V4[e] = v;
    if (g.wq) {
      __nv_bfloat162 lo = __floats2bfloat162_rn(p.x, p.y), hi = __floats2bfloat162_rn(p.z, p.w);
      uint2 u;
      u.x = *reinterpret_cast<uint32_t*>(&lo);
      u.y = *reinterpret_cast<uint32_t*>(&hi);
      *reinterpret_cast<uint2*>(g.wq + ch.off + 4 * e) = u;
    }
  }
  for (int e = 4 * n4 + threadIdx.x; e < ch.len; e += blockDim.x) {
    const int64_t o = ch.off + e;
    float p = g.params[o], m = g.m[o], v = g.v[o];
    adamw_elem(p, m, v, g.grads[o], lr, wd, b1, b2, eps, ib1, ib2);
    g.params[o] = p;
    g.m[o] = m;
    g.v[o] = v;
    if (g.wq) g.wq[o] = __float2bfloat16_rn(p);
  }
  // the next step's dropout masks: ALU work that other blocks' HBM streaming
  // overlaps (after this block's own stores have left, so that it does not
  // delay them)
  fill_masks(g.mg, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x);
}

// ------------------------------------------------------------------- init
// Element of the padded arena -> the element index within the layer
// (weights row-major unpadded, then biases) -> Philox word -> U(-b, b), fp32.
__global__ void k_init(InitArgs g) {
  const Chunk ch = g.chunks[blockIdx.x];
  const Segment s = g.segs[ch.seg];
  for (int e = threadIdx.x; e < ch.len; e += blockDim.x) {
    const int64_t o = ch.off + e;
    const int64_t local = o - s.off;
    float val = 0.f;
    bool real = true;
    uint32_t idx;
    if (s.is_bias) {
      idx = (uint32_t)(s.w_elems + local);
    } else {
      const int64_t row = local / s.cols_pad, col = local % s.cols_pad;
      real = col < s.cols;
      idx = (uint32_t)(row * s.cols + col);
    }
    if (real) {
      U4 r4 = philox10(idx >> 2, 0u, 0u, (1u << 28) | ((uint32_t)s.member << 4) | (uint32_t)s.layer,
                       (uint32_t)g.seed, (uint32_t)(g.seed >> 32));
      const uint32_t q = idx & 3u;
      const uint32_t r = q == 0 ? r4.x : q == 1 ? r4.y : q == 2 ? r4.z : r4.w;
      const double u = ((double)(r >> 8) + 0.5) * 5.9604644775390625e-08;  // 2^-24
      const double bound = 1.0 / sqrt((double)s.fan_in);
      val = (float)((2.0 * u - 1.0) * bound);
    }
    g.params[o] = val;
    g.grads[o] = 0.f;
    g.m[o] = 0.f;
    g.v[o] = 0.f;
    if (g.wq0) {
      g.wq0[o] = __float2bfloat16_rn(val);
      g.wq1[o] = __float2bfloat16_rn(val);
    }
  }
}

// bf16 copies of the whole arena (after pack_set_params / pack_set_active).
__global__ void k_refresh_wq(const float* __restrict__ p, __nv_bfloat16* __restrict__ wq0,
                             __nv_bfloat16* __restrict__ wq1, int64_t n) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const __nv_bfloat16 b = __float2bfloat16_rn(p[e]);
    wq0[e] = b;
    wq1[e] = b;
  }
}

// ----------------------------------------------------------- predict head
// Forward-only head: probabilities (softmax / sigmoid) or values into
// out[member, n0 + r, :] for r < rows.
template <typename T, int DO>
__global__ void __launch_bounds__(256) k_predict_head(PredictHeadArgs<T> g) {
  constexpr int R = DO <= 10 ? 4 : 2;
  const HeadJob jb = g.jobs[blockIdx.x];   // the work list changes only while the stream is idle
  const int r0 = jb.blk * kHeadRows;
  const MemberDev md = g.mem[jb.member];
  pdl_wait();
  if (r0 >= g.rows) return;
  const int w = md.w, d_out = g.d_out, ldh = jb.h_ld;
  const T* H = g.act + jb.h_off + (int64_t)r0 * ldh;
  const float* Wh = g.params + jb.w_off;
  const float* bh = g.params + jb.b_off;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const HeadLogits<T, DO, R> hl(w, lane);
  for (int p0 = 0; p0 < HeadLogits<T, DO, R>::kRowsPerWarp; p0 += hl.step()) {
    const int rl0 = warp * HeadLogits<T, DO, R>::kRowsPerWarp + p0 + hl.grp * R;
    const bool live = hl.grp < hl.groups && r0 + rl0 < g.rows;
    float acc[R][DO];
    hl.run(H, ldh, Wh, bh, w, d_out, rl0, live, acc);
    if (!live) continue;
    // the group's lanes write its R rows in turn
    for (int q = hl.gl; q < R; q += hl.lpr) {
      const int r = r0 + rl0 + q;
      if (r >= g.rows) break;
      float z[DO];
#pragma unroll
      for (int c = 0; c < DO; ++c) z[c] = acc[0][c];
#pragma unroll
      for (int qq = 1; qq < R; ++qq)
        if (q == qq)
#pragma unroll
          for (int c = 0; c < DO; ++c) z[c] = acc[qq][c];
      float* o = g.out + ((int64_t)jb.member * g.N + g.n0 + r) * d_out;
      if (g.task == 1) {
        float mx = z[0];
#pragma unroll
        for (int c = 1; c < DO; ++c) if (c < d_out) mx = fmaxf(mx, z[c]);
        float sum = 0.f;
#pragma unroll
        for (int c = 0; c < DO; ++c) if (c < d_out) sum += expf(z[c] - mx);
        const float inv = 1.f / sum;
#pragma unroll
        for (int c = 0; c < DO; ++c)
          if (c < d_out) o[c] = expf(z[c] - mx) * inv;
      } else {
        o[0] = g.task == 0 ? 1.f / (1.f + expf(-z[0])) : z[0];
      }
    }
  }
}

// ------------------------------------------------------------- mask dump
__global__ void k_debug_masks(uint8_t* __restrict__ out, int32_t B, int32_t w, uint64_t seed,
                              uint32_t member, uint32_t layer, uint32_t step, uint32_t T) {
  const int64_t n4 = (int64_t)B * (w / 4);
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n4; e += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(e / (w / 4)), c4 = (int)(e % (w / 4));
    const uint32_t k = keep_bits4(seed, member, layer, step, (uint32_t)r, (uint32_t)c4, T);
#pragma unroll
    for (int q = 0; q < 4; ++q) out[(int64_t)r * w + c4 * 4 + q] = (uint8_t)((k >> q) & 1u);
  }
}

// ------------------------------------------------------------- Philox words
// in [n, 6]: counter c0..c3 then key k0, k1; out [n, 4]: the four words.
__global__ void k_debug_philox(const uint32_t* __restrict__ in, uint32_t* __restrict__ out, int32_t n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t* c = in + (int64_t)i * 6;
  const U4 r = philox10(c[0], c[1], c[2], c[3], c[4], c[5]);
  uint32_t* o = out + (int64_t)i * 4;
  o[0] = r.x;
  o[1] = r.y;
  o[2] = r.z;
  o[3] = r.w;
}

// ------------------------------------------------------------- launchers
template <typename T>
void launch_gather(cudaStream_t st, const float* X, const int32_t* idx, int B, int B_pad,
                   int d_in, int d_in_pad, int ldx, T* xb, int advance, int32_t* t_dev, float2* bias_corr,
                   const int32_t* active_ids, int n_active, float beta1, float beta2, int* zero, int n_zero,
                   int stacked, int64_t xb_stride, const HeadSplit& hs) {
  const int rows = std::max(1, (int)ceil_div(B_pad, 8));  // 8 rows (warps) per block
  const int blocks = rows + (int)ceil_div((int64_t)hs.n * hs.cp * 8, 256);
  const unsigned gy = stacked ? (unsigned)std::max(n_active, 1) : 1u;
  const float ln_b1 = (float)std::log((double)beta1), ln_b2 = (float)std::log((double)beta2);
  launch_pdl(k_gather<T>, dim3(blocks, gy), dim3(256), 0, st, X, idx, B, B_pad, d_in, d_in_pad, ldx, xb, advance,
             t_dev, bias_corr, active_ids, n_active, ln_b1, ln_b2, zero, n_zero, stacked, xb_stride, hs, rows);
}

template <typename T>
void launch_fill_ones(cudaStream_t st, const OnesJob* jobs, int n_jobs, T* xb, T* act, T* ex) {
  if (n_jobs > 0) k_fill_ones<T><<<n_jobs, 256, 0, st>>>(jobs, xb, act, ex);
}

void launch_gemm_simt(cudaStream_t st, const GemmArgs<float>& g, const SimtRange& r) {
  if (r.count <= 0) return;
  if (r.bm == 128) launch_pdl(k_gemm_simt<128, 64, 8, 8, 16>, dim3(r.count), dim3(128), 0, st, g, r.first);
  else if (r.bm == 64) launch_pdl(k_gemm_simt<64, 64, 8, 4, 32>, dim3(r.count), dim3(128), 0, st, g, r.first);
  else if (r.bn == 64) launch_pdl(k_gemm_simt<32, 64, 4, 4, 32>, dim3(r.count), dim3(128), 0, st, g, r.first);
  else launch_pdl(k_gemm_simt<32, 32, 4, 4, 32>, dim3(r.count), dim3(64), 0, st, g, r.first);
}

void head_stage_prepare() {
  cudaFuncSetAttribute(k_head_stage, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)head_stage_smem(kHeadStageMaxW));
}

template <typename T>
void launch_head(cudaStream_t st, const HeadArgs<T>& g, int n_jobs) {
  if (n_jobs <= 0) return;
  if constexpr (std::is_same_v<T, __nv_bfloat16>) {
    // one output (more: launch_head_tc).  The one-pass kernel for members wider
    // than 512 (the staged block would run one per SM), or at most one block
    // per SM (eight small members 322 us per eight steps against 333 us staged;
    // 256 narrow members, 1024 blocks, 3123 against 3030 us)
    if (g.w_max <= 2048 && (g.w_max > kHeadStageMaxW || n_jobs <= 152))
      launch_pdl(k_head_one, dim3(n_jobs), dim3(256), 0, st, g);
    else if (g.w_max <= kHeadStageMaxW)
      launch_pdl(k_head_stage, dim3(n_jobs), dim3(256), (size_t)head_stage_smem(g.w_max), st, g);
    else
      launch_pdl(k_head<T, 1>, dim3(n_jobs), dim3(256), 0, st, g);
  } else {
    switch (head_bucket(g.d_out)) {
      case 1: launch_pdl(k_head<T, 1>, dim3(n_jobs), dim3(256), 0, st, g); break;
      case 2: launch_pdl(k_head<T, 2>, dim3(n_jobs), dim3(256), 0, st, g); break;
      case 4: launch_pdl(k_head<T, 4>, dim3(n_jobs), dim3(256), 0, st, g); break;
      case 8: launch_pdl(k_head<T, 8>, dim3(n_jobs), dim3(256), 0, st, g); break;
      case 10: launch_pdl(k_head<T, 10>, dim3(n_jobs), dim3(256), 0, st, g); break;
      case 16: launch_pdl(k_head<T, 16>, dim3(n_jobs), dim3(256), 0, st, g); break;
      default: launch_pdl(k_head<T, kMaxDout>, dim3(n_jobs), dim3(256), 0, st, g); break;
    }
  }
}

void launch_head_reduce(cudaStream_t st, const HeadReduceArgs& g, int m, int max_elems) {
  launch_pdl(k_head_reduce, dim3(m, (unsigned)ceil_div(max_elems, 256)), dim3(256), 0, st, g);
}

void launch_adamw(cudaStream_t st, const AdamArgs& g, int n_chunks) {
  if (n_chunks > 0) launch_pdl(k_adamw, dim3(n_chunks), dim3(256), 0, st, g);
}

void launch_init(cudaStream_t st, const InitArgs& g, int n_chunks) {
  if (n_chunks > 0) k_init<<<n_chunks, 256, 0, st>>>(g);
}

// ---------------------------------------------------- periodic embeddings
// E_i[b, q] (q = j d + k) = alpha_q f_q(x_bj) + beta_q with f_0(x) = x and
// f_k(x) = cos(w_j,k-1 x + b_j,k-1).  Both kernels tile a member's columns
// in groups of 64 (a lane takes two neighbours: each thread keeps its columns'
// features, components and parameters in registers, and moves E and dE in
// pairs) and spread the rows over the block's 8 warps.  Bound by issue, most
// of it the cosine.  32 members with d_emb 8..32 of 64 features, 512 rows (42
// MB of E): forward 36 us, backward 50 us; one column per lane with x loaded
// per element, the library's cosf / sincosf and fp64 sums took 57 and 93 us.
// (The own sine and cosine alone, without x staged, left them at 45 and 102.)
constexpr int kEmbRows = 128;  // rows per forward block
constexpr int kEmbRowsB = 64;  // rows at a time of a backward block
constexpr int kEmbCols = 64;   // columns per block

// sin u and cos u to about an ulp of fp32 for |u| <= 1e5: u less the nearest
// multiple n of pi/2, taken out as three fp32 numbers with fused multiply-adds
// (Cody and Waite 1980), then the Taylor polynomials on |r| <= pi/4 (first
// terms left out: r^11 / 11! < 2e-9, r^12 / 12! < 2e-10) and the quadrant's
// choice and sign.  n comes out of the low bits of a sum with 1.5 2^23, which
// avoids the conversion unit.  Larger |u| and values that are not finite take
// the library's functions.
__device__ __forceinline__ void sincos_small(float u, float& sn, float& cs) {
  const float big = fmaf(u, 0.636619772f, 12582912.f);
  const int k = __float_as_int(big);
  const float n = big - 12582912.f;
  float r = fmaf(n, -1.57079637f, u);     // fp32(pi/2)
  r = fmaf(n, 4.37113883e-8f, r);         // pi/2 less that, fp32
  r = fmaf(n, 1.71512451e-15f, r);        // and the rest
  const float r2 = r * r;
  float p = fmaf(r2, 2.75573192e-6f, -1.98412698e-4f);   // 1/9!, -1/7!
  p = fmaf(p, r2, 8.33333333e-3f);                        // 1/5!
  p = fmaf(p, r2, -1.66666667e-1f);                       // -1/3!
  const float s = fmaf(r * r2, p, r);
  float c = fmaf(r2, -2.75573192e-7f, 2.48015873e-5f);    // -1/10!, 1/8!
  c = fmaf(c, r2, -1.38888889e-3f);                       // -1/6!
  c = fmaf(c, r2, 4.16666667e-2f);                        // 1/4!
  c = fmaf(c, r2, -0.5f);
  c = fmaf(c, r2, 1.f);
  const float a = (k & 1) ? c : s, b = (k & 1) ? s : c;
  sn = __int_as_float(__float_as_int(a) ^ ((k & 2) << 30));
  cs = __int_as_float(__float_as_int(b) ^ (((k + 1) & 2) << 30));
}
__device__ __noinline__ float2 sincos_any(float u) {
  float2 r;
  sincosf(u, &r.x, &r.y);
  return r;
}
__device__ __forceinline__ void emb_sincos(float u, float& sn, float& cs) {
  sincos_small(u, sn, cs);
  if (!(fabsf(u) <= 1e5f)) {
    const float2 r = sincos_any(u);
    sn = r.x;
    cs = r.y;
  }
}

struct EmbCol {
  int j, k;
  float w, b, alpha, beta;
};

__device__ __forceinline__ EmbCol emb_col(const EmbMember& em, const float* params, int d_in, int q) {
  const int d = em.d, dm = d - 1;
  const float* w = params + em.p_off;
  const float* bb = w + (int64_t)d_in * dm;
  const float* al = bb + (int64_t)d_in * dm;
  const float* be = al + (int64_t)d_in * d;
  EmbCol c;
  c.j = q / d;
  c.k = q - c.j * d;
  c.alpha = al[q];
  c.beta = be[q];
  c.w = c.k ? w[c.j * dm + c.k - 1] : 0.f;
  c.b = c.k ? bb[c.j * dm + c.k - 1] : 0.f;
  return c;
}

__device__ __forceinline__ void store2(__nv_bfloat16* p, float a, float b) {
  *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(a, b);
}
__device__ __forceinline__ void store2(float* p, float a, float b) { *reinterpret_cast<float2*>(p) = make_float2(a, b); }

// The x values of ROWS rows from b0 (from B on: 0) and features j0 .. j0 +
// nf - 1, a thread per row and every 256 / ROWS-th feature: [feature][row], so
// that a warp's reads of one row at its lanes' features are broadcasts or fall
// in distinct banks.  Loading them a group of rows at a time keeps the
// dependent loads (row index, then value) of 256 threads in flight; taken
// element by element they were what the backward kernel waited for.
template <int ROWS>
using EmbX = float[kEmbCols][ROWS + 1];
template <int ROWS>
__device__ __forceinline__ void emb_stage_x(EmbX<ROWS>& xs, const float* X, const int32_t* idx, int B, int d_in, int b0,
                                            int j0, int nf) {
  const int r = threadIdx.x & (ROWS - 1), b = b0 + r;
  const float* x = X + (b < B ? (idx ? (int64_t)idx[b] : (int64_t)b) : 0) * d_in + j0;
  for (int f = threadIdx.x / ROWS; f < nf; f += 256 / ROWS) xs[f][r] = b < B ? x[f] : 0.f;
}

// Forward: block (64-column group, 128-row group, active member); rows >= B
// and the pad columns up to in0_pad (a multiple of 8) are written as zero.
template <typename T>
__global__ void __launch_bounds__(256) k_emb_fwd(EmbArgs<T> a) {
  pdl_trigger();
  pdl_wait();
  const int member = a.active_ids[blockIdx.z];
  const EmbMember em = a.em[member];
  const int qb = blockIdx.x * kEmbCols, q = qb + 2 * (threadIdx.x & 31);
  if (qb >= em.in0_pad) return;   // block-uniform
  __shared__ EmbX<kEmbRows> xs;
  const float* X = a.X;
  const int32_t* idx = a.idx;
  if (idx) idx += (int64_t)member * a.idx_stride;
  const int j0 = min(qb, em.in0 - 1) / em.d, b0 = blockIdx.y * kEmbRows;
  emb_stage_x<kEmbRows>(xs, X, idx, a.B, a.d_in, b0, j0, min(qb + kEmbCols - 1, em.in0 - 1) / em.d - j0 + 1);
  EmbCol c[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) c[u] = q + u < em.in0 ? emb_col(em, a.params, a.d_in, q + u) : EmbCol{j0, 0, 0.f, 0.f, 0.f, 0.f};
  __syncthreads();
  if (q >= em.in0_pad) return;
  const int ld = em.in0_pad + kOnesCols, r0 = threadIdx.x >> 5;
  T* E = a.ex + em.e_off + q + (int64_t)(b0 + r0) * ld;
  const float* x0 = xs[c[0].j - j0];
  const float* x1 = xs[c[1].j - j0];
#pragma unroll 4
  for (int i = 0; i < kEmbRows / 8; ++i) {
    const int r = r0 + 8 * i;
    if (b0 + r >= a.B_pad) break;
    const float xv[2] = {x0[r], x1[r]};
    float e[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      float sn, cs;
      emb_sincos(fmaf(c[u].w, xv[u], c[u].b), sn, cs);
      e[u] = fmaf(c[u].alpha, c[u].k == 0 ? xv[u] : cs, c[u].beta);
      if (b0 + r >= a.B) e[u] = 0.f;
    }
    store2(E + (int64_t)(8 * i) * ld, e[0], e[1]);
  }
}

// Backward: block (64-column group, active member), warp r takes rows r,
// r + 8, ...; with dE = the first layer's input gradient,
//   d alpha_q = sum_b dE f_q,  d beta_q = sum_b dE,
//   d w = -alpha_q sum_b dE sin(u) x,  d b = -alpha_q sum_b dE sin(u)
// (u = w x + b, cosine components).  Each thread sums 32 of its rows in fp32
// and adds that partial to a two-float sum; the 8 warps' sums are added in
// warp order.
template <typename T>
__global__ void __launch_bounds__(256, 4) k_emb_bwd(EmbArgs<T> a) {
  pdl_trigger();
  pdl_wait();
  const int member = a.active_ids[blockIdx.y];
  const EmbMember em = a.em[member];
  const int qb = blockIdx.x * kEmbCols;
  if (qb >= em.in0) return;   // block-uniform
  __shared__ EmbX<kEmbRowsB> xs;
  __shared__ float2 red[8][8][32];   // [column of the pair, sum][warp][lane]: each thread's running sums
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int q0 = qb + 2 * lane;
  const int qc = min(q0, em.in0_pad - 2);             // in-range pair for the loads of idle lanes
  const float* X = a.X;
  const int32_t* idx = a.idx;
  if (idx) idx += (int64_t)member * a.idx_stride;
  const int j0 = qb / em.d, nf = min(qb + kEmbCols - 1, em.in0 - 1) / em.d - j0 + 1;
  EmbCol c[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) c[u] = emb_col(em, a.params, a.d_in, min(qc + u, em.in0 - 1));
  const T* dE = a.dz + em.de_off + qc + (int64_t)wp * em.in0_pad;
  const float* x0 = xs[c[0].j - j0];
  const float* x1 = xs[c[1].j - j0];
#pragma unroll
  for (int t = 0; t < 8; ++t) red[t][wp][lane] = make_float2(0.f, 0.f);
  float p[2][4];   // alpha, beta, w, b
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int t = 0; t < 4; ++t) p[u][t] = 0.f;
  for (int b0 = 0; b0 < a.B; b0 += kEmbRowsB, dE += (int64_t)kEmbRowsB * em.in0_pad) {
    // the group's rows of dE (rows up to B_pad exist), in flight over the staging
    RawG<T, 2> raw[kEmbRowsB / 8];
#pragma unroll
    for (int i = 0; i < kEmbRowsB / 8; ++i) raw[i].load(dE + (int64_t)(8 * i) * em.in0_pad);
    __syncthreads();   // the previous group's values have been read
    emb_stage_x<kEmbRowsB>(xs, X, idx, a.B, a.d_in, b0, j0, nf);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kEmbRowsB / 8; ++i) {
      const int r = wp + 8 * i;
      float g[2];
      raw[i].to_float(g);
      const float xv[2] = {x0[r], x1[r]};
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (b0 + r >= a.B) g[u] = 0.f;
        float sn, cs;
        emb_sincos(fmaf(c[u].w, xv[u], c[u].b), sn, cs);
        const float gs = g[u] * sn;
        p[u][0] = fmaf(g[u], c[u].k == 0 ? xv[u] : cs, p[u][0]);
        p[u][1] += g[u];
        p[u][2] = fmaf(gs, xv[u], p[u][2]);
        p[u][3] += gs;
      }
    }
    if ((b0 / kEmbRowsB) % 4 == 3 || b0 + kEmbRowsB >= a.B) {
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          float2 v = red[4 * u + t][wp][lane];
          two_add(v.x, v.y, p[u][t]);
          red[4 * u + t][wp][lane] = v;
          p[u][t] = 0.f;
        }
    }
  }
  __syncthreads();
  // warp v takes sum v & 3 of the pair's column v >> 2
  const int u = wp >> 2, t = wp & 3, q = q0 + u;
  if (q >= em.in0) return;
  float2 s = red[wp][0][lane];
#pragma unroll
  for (int r = 1; r < 8; ++r) two_merge(s.x, s.y, red[wp][r][lane].x, red[wp][r][lane].y);
  // a sum that overflowed or met a NaN: its first part alone says so
  const double sum = isfinite(s.x) ? (double)s.x + (double)s.y : (double)s.x;
  const EmbCol cc = u ? c[1] : c[0];
  const int d = em.d, dm = d - 1;
  float* gw = a.grads + em.p_off;
  float* gb = gw + (int64_t)a.d_in * dm;
  float* ga = gb + (int64_t)a.d_in * dm;
  float* gbt = ga + (int64_t)a.d_in * d;
  if (t == 0) ga[q] = (float)sum;
  else if (t == 1) gbt[q] = (float)sum;
  else if (cc.k) (t == 2 ? gw : gb)[cc.j * dm + cc.k - 1] = (float)(-(double)cc.alpha * sum);
}

template <typename T>
void launch_emb_fwd(cudaStream_t st, const EmbArgs<T>& a, int n_active, int cols_max) {
  if (n_active > 0 && a.B_pad > 0)
    launch_pdl(k_emb_fwd<T>, dim3((unsigned)ceil_div(cols_max, kEmbCols), (unsigned)ceil_div(a.B_pad, kEmbRows),
                                  (unsigned)n_active), dim3(256), 0, st, a);
}
template <typename T>
void launch_emb_bwd(cudaStream_t st, const EmbArgs<T>& a, int n_active, int cols_max) {
  if (n_active > 0)
    launch_pdl(k_emb_bwd<T>, dim3((unsigned)ceil_div(cols_max, kEmbCols), (unsigned)n_active), dim3(256), 0, st, a);
}

// ------------------------------------------------------------------ Muon
// One block of 256 threads per chunk of a Muon matrix (row-major [rows,
// cols] in the arena): kMuonChunk consecutive elements, or for a transposed
// matrix a 32 x 128 tile of W (muon_chunks).  Widths are multiples of 16 and
// padded input widths multiples of 8, and arena blocks start 32-element
// aligned, so 4 consecutive elements of a chunk share a row and start at a
// 16-byte boundary: the kernels move float4 and 4-element vectors, each
// thread kMuonV of them, all loads first.  The per-element arithmetic is
// fp32; doubles appear only in the partial sums (GB300's FP64 rate is a
// small fraction of its FP32 rate).
constexpr int kMuonV = kMuonChunk / 4 / 256;
static_assert(kMuonChunk % 1024 == 0, "a Muon chunk is a whole number of float4 per thread");

template <typename T>
struct MuonChunk {
  MuonMat mt;
  int mat;     // its index in the matrix list
  int e0, n4;  // flat chunk: its first element within the matrix and its float4 count
  int i0, j0;  // tile of a transposed matrix: its first row and column of W
  __device__ __forceinline__ MuonChunk(const MuonArgs<T>& a, int blk) {
    mat = a.chunk_mat[blk];
    mt = a.mats[mat];
    const int k = blk - mt.chunk0;
    if (!mt.tr) {
      e0 = k * kMuonChunk;
      n4 = (min(e0 + kMuonChunk, mt.rows * mt.cols) - e0) >> 2;
      i0 = j0 = 0;
    } else {
      const int tpr = (mt.cols + kMuonTileC - 1) / kMuonTileC;
      i0 = (k / tpr) * kMuonTileR;
      j0 = (k % tpr) * kMuonTileC;
      e0 = n4 = 0;
    }
  }
  // Element offset in W (from w_off) of this chunk's float4 q (0 <= q <
  // kMuonChunk / 4), or -1 outside the matrix.  Tiles: row q / 32, columns
  // 4 (q % 32) .. + 3 of the tile, so a warp reads 512 contiguous bytes.
  __device__ __forceinline__ int w_elem(int q) const {
    if (!mt.tr) return q < n4 ? e0 + 4 * q : -1;
    const int row = i0 + (q >> 5), col = j0 + 4 * (q & 31);
    return row < mt.rows && col < mt.cols ? row * mt.cols + col : -1;
  }
  // Tiles: piece p (0 <= p < kMuonChunk / 4) of X's rows -- row j0 + p / 8,
  // columns i0 + 4 (p % 8) .. + 3, i.e. W's column j0 + p / 8 at its rows
  // i0 + 4 (p % 8) .. + 3 -- as an element offset in X, or -1 outside.
  __device__ __forceinline__ int x_piece(int p) const {
    const int j = j0 + (p >> 3), i = i0 + 4 * (p & 7);
    return j < mt.cols && i < mt.rows ? j * mt.c + i : -1;
  }
};

__device__ __forceinline__ float4 load4f(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4f(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// A tile's X values staged in shared memory as [tile row][tile column] of W
// (pitch kMuonTileC + 2: the column reads of x_piece order touch distinct
// banks).
template <typename T>
using MuonStage = T[kMuonTileR][kMuonTileC + 2];

// the momentum update of one element; returns U's element
__device__ __forceinline__ float muon_mom(float g, float& m, float mu) {
  m = mu * m + (1.f - mu) * g;
  return (1.f - mu) * g + mu * m;
}

// 1 / max(|U|_F, 1e-7) of a matrix from its chunks' sums of squares, by one
// warp in a fixed order (lane j sums chunks j, j + 32, ...; then a butterfly):
// the same value wherever it is computed.
__device__ __forceinline__ float muon_inv_norm(const double* part, int chunk0, int n_chunks, int lane) {
  double ss = 0.0;
  for (int k = lane; k < n_chunks; k += 32) ss += __ldcg(part + chunk0 + k);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  return (float)(1.0 / fmax(sqrt(ss), 1e-7));
}

// momentum M <- mu M + (1 - mu) G; U = (1 - mu) G + mu M; the chunk's sum of
// squares of U (fp32 per thread, then fp64 in a fixed-order tree).  Also
// clears the counters of the Newton-Schulz launch that follows.  x0_fused:
// U is also written as X0 (a transposed matrix's tile through shared memory,
// as whole row segments of X), and the last chunk of a matrix to finish
// stores the matrix's scale.
template <typename T>
__global__ void __launch_bounds__(256) k_muon_momentum(MuonArgs<T> a) {
  pdl_trigger();
  pdl_wait();
  for (int i = blockIdx.x * 256 + threadIdx.x; i < a.n_ns_cnt; i += gridDim.x * 256) a.ns_cnt[i] = 0;
  const MuonChunk<T> ck(a, blockIdx.x);
  const float mu = a.mu;
  const float* G = a.grads + ck.mt.w_off;
  float* M = a.mom + ck.mt.w_off;
  T* X = a.ns + ck.mt.x_off[0];
  __shared__ MuonStage<T> st;
  float4 g[kMuonV], m[kMuonV];
  int ev[kMuonV];
#pragma unroll
  for (int k = 0; k < kMuonV; ++k) {
    ev[k] = ck.w_elem(threadIdx.x + 256 * k);
    if (ev[k] >= 0) {
      g[k] = *reinterpret_cast<const float4*>(G + ev[k]);
      m[k] = *reinterpret_cast<const float4*>(M + ev[k]);
    }
  }
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < kMuonV; ++k) {
    if (ev[k] < 0) continue;
    const float u0 = muon_mom(g[k].x, m[k].x, mu), u1 = muon_mom(g[k].y, m[k].y, mu);
    const float u2 = muon_mom(g[k].z, m[k].z, mu), u3 = muon_mom(g[k].w, m[k].w, mu);
    *reinterpret_cast<float4*>(M + ev[k]) = m[k];
    ss = fmaf(u0, u0, ss);
    ss = fmaf(u1, u1, ss);
    ss = fmaf(u2, u2, ss);
    ss = fmaf(u3, u3, ss);
    if (a.x0_fused) {
      if (!ck.mt.tr) {
        store4(X + ev[k], make_float4(u0, u1, u2, u3));
      } else {
        const int q = threadIdx.x + 256 * k, r = q >> 5, c = 4 * (q & 31);
        st[r][c] = Elem<T>::from_f(u0);
        st[r][c + 1] = Elem<T>::from_f(u1);
        st[r][c + 2] = Elem<T>::from_f(u2);
        st[r][c + 3] = Elem<T>::from_f(u3);
      }
    }
  }
  if (a.x0_fused && ck.mt.tr) {  // block-uniform
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kMuonV; ++k) {
      const int p = threadIdx.x + 256 * k, xo = ck.x_piece(p);
      if (xo < 0) continue;
      const int jj = p >> 3, i4 = 4 * (p & 7);
      store4(X + xo, make_float4(Elem<T>::to_f(st[i4][jj]), Elem<T>::to_f(st[i4 + 1][jj]),
                                 Elem<T>::to_f(st[i4 + 2][jj]), Elem<T>::to_f(st[i4 + 3][jj])));
    }
  }
  double s = (double)ss;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ double red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  __shared__ int last;
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    a.part[blockIdx.x] = t;
    if (a.x0_fused) {
      __threadfence();  // the partial before the arrival
      last = atomicAdd(a.mat_done + ck.mat, 1) == ck.mt.n_chunks - 1;
    }
  }
  if (!a.x0_fused) return;
  __syncthreads();
  if (last && threadIdx.x < 32) {
    __threadfence();  // every arrival before the partials' reads
    const float inv = muon_inv_norm(a.part, ck.mt.chunk0, ck.mt.n_chunks, threadIdx.x);
    if (threadIdx.x == 0) {
      a.ns_scale[ck.mat] = inv;
      a.mat_done[ck.mat] = 0;
    }
  }
}

// X0 = U / max(||U||_F, 1e-7), transposed when rows > cols (element by
// element: this pass serves the fp32 mode).  Chunks in reverse order: the
// momentum pass's last chunks are still in L2.
template <typename T>
__global__ void __launch_bounds__(256) k_muon_x0(MuonArgs<T> a) {
  pdl_trigger();
  pdl_wait();
  const MuonChunk<T> ck(a, gridDim.x - 1 - blockIdx.x);
  __shared__ float inv_s;
  if (threadIdx.x < 32) {  // the matrix's norm from its chunks' partials, one warp
    const float inv = muon_inv_norm(a.part, ck.mt.chunk0, ck.mt.n_chunks, threadIdx.x);
    if (threadIdx.x == 0) inv_s = inv;
  }
  const float mu = a.mu;
  const float* G = a.grads + ck.mt.w_off;
  const float* M = a.mom + ck.mt.w_off;
  float4 g[kMuonV], m[kMuonV];
  int ev[kMuonV];
#pragma unroll
  for (int k = 0; k < kMuonV; ++k) {
    ev[k] = ck.w_elem(threadIdx.x + 256 * k);
    if (ev[k] >= 0) {
      g[k] = __ldcs(reinterpret_cast<const float4*>(G + ev[k]));
      m[k] = *reinterpret_cast<const float4*>(M + ev[k]);
    }
  }
  __syncthreads();
  const float inv = inv_s;
  T* X = a.ns + ck.mt.x_off[0];
#pragma unroll
  for (int k = 0; k < kMuonV; ++k) {
    const int e = ev[k];
    if (e < 0) continue;
    const float4 u = make_float4(((1.f - mu) * g[k].x + mu * m[k].x) * inv, ((1.f - mu) * g[k].y + mu * m[k].y) * inv,
                                 ((1.f - mu) * g[k].z + mu * m[k].z) * inv, ((1.f - mu) * g[k].w + mu * m[k].w) * inv);
    if (!ck.mt.tr) {
      store4(X + e, u);
    } else {  // the 4 elements share a row i of W: entries (j .. j + 3, i) of X
      const int i = e / ck.mt.cols, j = e - i * ck.mt.cols;
      const int x0 = j * ck.mt.c + i;
      X[x0] = Elem<T>::from_f(u.x);
      X[x0 + ck.mt.c] = Elem<T>::from_f(u.y);
      X[x0 + 2 * ck.mt.c] = Elem<T>::from_f(u.z);
      X[x0 + 3 * ck.mt.c] = Elem<T>::from_f(u.w);
    }
  }
}

// W <- W - lr wd W; W <- W - lr scale O, O = the final X (transposed back: a
// transposed matrix's tile reads whole row segments of X into shared memory)
template <typename T>
__global__ void __launch_bounds__(256) k_muon_apply(MuonArgs<T> a) {
  pdl_trigger();
  pdl_wait();
  const MuonChunk<T> ck(a, blockIdx.x);
  const float lr = ck.mt.lr, wd = a.mem[ck.mt.member].wd, sc = ck.mt.scale;
  const T* X = a.ns + (a.x_final ? ck.mt.x_off[1] : ck.mt.x_off[0]);  // no runtime index into the record
  float* P = a.params + ck.mt.w_off;
  __shared__ MuonStage<T> st;
  if (ck.mt.tr) {  // block-uniform
#pragma unroll
    for (int k = 0; k < kMuonV; ++k) {
      const int p = threadIdx.x + 256 * k, xo = ck.x_piece(p);
      if (xo < 0) continue;
      const float4 v = load4f(X + xo);
      const int jj = p >> 3, i4 = 4 * (p & 7);
      st[i4][jj] = Elem<T>::from_f(v.x);
      st[i4 + 1][jj] = Elem<T>::from_f(v.y);
      st[i4 + 2][jj] = Elem<T>::from_f(v.z);
      st[i4 + 3][jj] = Elem<T>::from_f(v.w);
    }
    __syncthreads();
  }
  float4 p[kMuonV], x[kMuonV];
  int ev[kMuonV];
#pragma unroll
  for (int k = 0; k < kMuonV; ++k) {
    const int q = threadIdx.x + 256 * k, r = q >> 5, c = 4 * (q & 31);
    ev[k] = ck.w_elem(q);
    p[k] = x[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (ev[k] >= 0) {
      p[k] = *reinterpret_cast<const float4*>(P + ev[k]);
      x[k] = ck.mt.tr ? make_float4(Elem<T>::to_f(st[r][c]), Elem<T>::to_f(st[r][c + 1]),
                                    Elem<T>::to_f(st[r][c + 2]), Elem<T>::to_f(st[r][c + 3]))
                      : load4f(X + ev[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < kMuonV; ++k) {
    if (ev[k] < 0) continue;
    float4 q = p[k];
    q.x = q.x - lr * wd * q.x;
    q.y = q.y - lr * wd * q.y;
    q.z = q.z - lr * wd * q.z;
    q.w = q.w - lr * wd * q.w;
    q.x = q.x - lr * sc * x[k].x;
    q.y = q.y - lr * sc * x[k].y;
    q.z = q.z - lr * sc * x[k].z;
    q.w = q.w - lr * sc * x[k].w;
    *reinterpret_cast<float4*>(P + ev[k]) = q;
    if (a.wq_out) store4(a.wq_out + ck.mt.w_off + ev[k], q);
  }
  // the next step's dropout masks, as in k_adamw: this pass has the threads
  // (under Muon, AdamW's few blocks took 123 us for the large workload's)
  fill_masks(a.mg, (int64_t)blockIdx.x * 256 + threadIdx.x, (int64_t)gridDim.x * 256);
}

template <typename T>
void launch_muon(cudaStream_t st, const MuonArgs<T>& a, int n_chunks, int phase) {
  if (n_chunks <= 0) return;
  if (phase == 0) launch_pdl(k_muon_momentum<T>, dim3(n_chunks), dim3(256), 0, st, a);
  else if (phase == 1) launch_pdl(k_muon_x0<T>, dim3(n_chunks), dim3(256), 0, st, a);
  else launch_pdl(k_muon_apply<T>, dim3(n_chunks), dim3(256), 0, st, a);
}

__global__ void __launch_bounds__(256) k_masks(MaskGen mg) {
  pdl_trigger();
  pdl_wait();
  fill_masks(mg, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x);
}

void launch_masks(cudaStream_t st, const MaskGen& mg) {
  const int64_t total = (int64_t)mg.n_chunks * mg.rows;
  if (total <= 0) return;
  launch_pdl(k_masks, dim3((unsigned)std::min<int64_t>(ceil_div(total, 256), 152 * 8)), dim3(256), 0, st, mg);
}

// A member's run copied out.  Bound by HBM for wide members (8 bytes per
// element) and by the launch for narrow ones.  Dependent launches overlap
// their set-up, copies by the runtime do not, and one float4 per thread makes
// the shortest kernel: 256 members of 45 k elements 2.5 us each (3.8 at four
// per thread, 5.7 without dependent launches); two steps of 64 members and
// their snapshots 2361 us with the runtime's copies, 2040 us so.
__global__ void __launch_bounds__(256) k_copy(float* __restrict__ dst, const float* __restrict__ src, int64_t n) {
  pdl_wait();
  pdl_trigger();
  const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x, step = (int64_t)gridDim.x * 256;
  int64_t done = 0;
  if (((uintptr_t)dst & 15) == 0) {   // a caller's buffer may start anywhere
    const int64_t n4 = n >> 2;
#pragma unroll 4
    for (int64_t e = t; e < n4; e += step)
      reinterpret_cast<float4*>(dst)[e] = reinterpret_cast<const float4*>(src)[e];
    done = 4 * n4;
  }
#pragma unroll 4
  for (int64_t e = done + t; e < n; e += step) dst[e] = src[e];
}

void launch_copy(cudaStream_t st, float* dst, const float* src, int64_t n) {
  launch_pdl(k_copy, dim3((unsigned)std::min<int64_t>(ceil_div(n, 1024), 152 * 8)), dim3(256), 0, st, dst, src, n);
}

void launch_refresh_wq(cudaStream_t st, const float* p, __nv_bfloat16* wq0, __nv_bfloat16* wq1, int64_t n) {
  k_refresh_wq<<<152 * 4, 256, 0, st>>>(p, wq0, wq1, n);
}

template <typename T>
void launch_predict_head(cudaStream_t st, const PredictHeadArgs<T>& g, int n_jobs) {
  if (n_jobs <= 0) return;
  if constexpr (std::is_same_v<T, __nv_bfloat16>) {
    launch_pdl(k_predict_head<T, 1>, dim3(n_jobs), dim3(256), 0, st, g);   // more outputs: launch_head_tc
  } else {
    switch (head_bucket(g.d_out)) {
      case 1: launch_pdl(k_predict_head<T, 1>, dim3(n_jobs), dim3(256), 0, st, g); break;
      case 2: launch_pdl(k_predict_head<T, 2>, dim3(n_jobs), dim3(256), 0, st, g); break;
      case 4: launch_pdl(k_predict_head<T, 4>, dim3(n_jobs), dim3(256), 0, st, g); break;
      case 8: launch_pdl(k_predict_head<T, 8>, dim3(n_jobs), dim3(256), 0, st, g); break;
      case 10: launch_pdl(k_predict_head<T, 10>, dim3(n_jobs), dim3(256), 0, st, g); break;
      case 16: launch_pdl(k_predict_head<T, 16>, dim3(n_jobs), dim3(256), 0, st, g); break;
      default: launch_pdl(k_predict_head<T, kMaxDout>, dim3(n_jobs), dim3(256), 0, st, g); break;
    }
  }
}

void launch_debug_masks(cudaStream_t st, uint8_t* out, int B, int w, uint64_t seed, uint32_t member,
                        uint32_t layer, uint32_t step, uint32_t T) {
  k_debug_masks<<<64, 256, 0, st>>>(out, B, w, seed, member, layer, step, T);
}

void launch_debug_philox(cudaStream_t st, const uint32_t* in, uint32_t* out, int n) {
  k_debug_philox<<<(int)ceil_div(n, 128), 128, 0, st>>>(in, out, n);
}

#define TP_INSTANTIATE(T)                                                                              \
  template void launch_gather<T>(cudaStream_t, const float*, const int32_t*, int, int, int, int,                 \
                                 int, T*, int, int32_t*, float2*, const int32_t*, int, float, float,    \
                                 int*, int, int, int64_t, const HeadSplit&);                            \
  template void launch_fill_ones<T>(cudaStream_t, const OnesJob*, int, T*, T*, T*);                    \
  template void launch_head<T>(cudaStream_t, const HeadArgs<T>&, int);                                 \
  template void launch_predict_head<T>(cudaStream_t, const PredictHeadArgs<T>&, int);           \
  template void launch_muon<T>(cudaStream_t, const MuonArgs<T>&, int, int);                      \
  template void launch_emb_fwd<T>(cudaStream_t, const EmbArgs<T>&, int, int);                     \
  template void launch_emb_bwd<T>(cudaStream_t, const EmbArgs<T>&, int, int);

TP_INSTANTIATE(float)
TP_INSTANTIATE(__nv_bfloat16)

}  // namespace tp
