// head_tc.cu -- the multiclass head on the tensor cores (bf16 mode).
//
// One CTA takes one member on one 128-row block of its last hidden layer's
// activations H [128, w].  In 128-column steps H streams through shared memory
// by TMA twice (prediction: once), the second time from L2:
//   1. logits   Z = H W_h^T           (tcgen05, M = 128 rows, N = classes)
//      then per row the loss and D = d(mean loss)/dZ, or the probabilities;
//   2. per step dH = D W_h, masked by H > 0 and scaled, is the step's part of
//      dZ_L (written over H in shared memory and stored by TMA), and
//      dW_h^T = H^T D (M = 128 columns, N = classes) the block's partial.
// The head weights and D are fp32.  Each enters as three bf16 numbers whose
// sum it is (24 bits), so every product of two parts is exact: Z and dW_h are
// sums of three products, dH of the six with a weight above 2^-24.  The
// accumulators do not round to nearest (a chain of n instructions ends about
// n 10^-8 of its value off), so Z takes an accumulator per 64 columns and dW_h
// one per 64 rows, four instructions each, which are added up in fp32 registers
// (dH is rounded to bf16 at once).  Distance from the exact sums (norm-wise), logits / dW_h, ten
// classes: 256..1024 columns, 1024 rows 7.4e-8 / 8.4e-8 (as fp32 multiply-adds
// 1.3e-7 / 7.6e-8, in one chain 4.4e-7 / 4.6e-7); 2048 columns and rows 9.9e-8 /
// 9.9e-8 (1.3e-7 / 9.4e-8, 1.4e-6 / 9.6e-7).
// The weights' parts are laid out by k_gather as the 128-byte-swizzled image
// [3 CP classes][64 columns] per 64-column chunk; the same image serves product
// 1 K-major and product 2 MN-major, and likewise D (rows of 3 CP classes) and H
// serve both majors from one copy.
//
// Bound by the passes over H and dZ (4 w bytes per row from HBM or L2, H once
// more from L2) and the per-element epilogue of dZ; the products are a few
// per cent of the tensor rate.  64 members of 256..1024 columns, 1024 rows, ten
// classes: 54 us per launch (168 MB of H and dZ), against 143 us for the same
// sums in fp32 multiply-adds with a 64-row block's H in shared memory;
// prediction, 8192 rows: 136 us (671 MB of H, 4.9 TB/s) against 772 us (one
// chain per sum took 53 and 132 us).  128
// rows and two 44 KB stages let two CTAs (256 TMEM columns each) share an SM
// up to 16 classes, so one CTA's loads and products fill the other's epilogue.
#include "kernels.cuh"
#include "loss.cuh"
#include "tc_ptx.cuh"

namespace tp {
namespace {

constexpr int kHtBox = 64 * 128 * 2;       // 128 rows x 64 columns of H, 128-byte swizzled
constexpr int kHtStages = 2;
constexpr int kHtEpi = 8;                  // epilogue warps of the training kernel
constexpr uint64_t kHtWaitNs = 2000000000ull;

template <int CP>
struct HtGeo {
  static constexpr int kN = 3 * CP;                       // MMA columns of the classes' parts
  static constexpr int kWChunk = kN * 128;                // weights of one 64-column chunk
  static constexpr int kStage = 2 * kHtBox + 2 * kWChunk;
  static constexpr int kD = (kN + 63) / 64 * kHtBox;      // D [128, 3 CP]
  // TMEM, in accumulators of kN columns kAcc apart: Z of (step parity, 64-column
  // half) at 2 parity + half; then dW_h of the two 64-row halves, and dH
  static constexpr uint32_t kAcc = CP == 16 ? 64 : 128, kDh = 2 * kAcc, kTmemCols = 4 * kAcc;
};
struct HtTail {
  uint64_t full[kHtStages], empty[kHtStages], rel[kHtStages];
  uint64_t half[kHtStages][2];             // the epilogue warps of a 64-column half have written it
  uint64_t z_full[2], z_free[2], d_ready, t_full, t_free, done;
  uint32_t tmem_base;
  int abort;
  float loss[4], db[4][32];                // per 32-row group: loss and class sums of D
  float colsum[kHtStages][4][128];         // per 32-row group: column sums of dZ as stored
};
template <int CP, bool TRAIN>
constexpr int ht_smem() {
  return kHtStages * HtGeo<CP>::kStage + (TRAIN ? HtGeo<CP>::kD : 0) + (int)sizeof(HtTail) + 1024;
}
static_assert(ht_smem<32, true>() <= 232448, "shared memory per CTA");
static_assert(2 * (ht_smem<16, true>() + 1024) <= 233472, "two CTAs per SM");

template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&v)[N]);
template <>
__device__ __forceinline__ void tmem_ld<32>(uint32_t taddr, uint32_t (&v)[32]) { tmem_ld32(taddr, v); }
template <>
__device__ __forceinline__ void tmem_ld<16>(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
template <>
__device__ __forceinline__ void tmem_ld<8>(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// The sum of the three parts' products for N classes from column c0 (parts CP
// columns apart) in one accumulator, or in the two from taddr on, the smallest
// part first.
template <int CP, int N>
__device__ __forceinline__ void tmem_sum3(uint32_t taddr, int c0, bool both, float (&z)[N]) {
#pragma unroll
  for (int p = 2; p >= 0; --p) {
    uint32_t v[N];
    tmem_ld<N>(taddr + p * CP + c0, v);
#pragma unroll
    for (int c = 0; c < N; ++c) z[c] = p == 2 ? __uint_as_float(v[c]) : z[c] + __uint_as_float(v[c]);
    if (both) {
      tmem_ld<N>(taddr + HtGeo<CP>::kAcc + p * CP + c0, v);
#pragma unroll
      for (int c = 0; c < N; ++c) z[c] += __uint_as_float(v[c]);
    }
  }
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
      "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(map), "r"(src),
               "r"(x), "r"(y)
               : "memory");
}
// this thread's shared-memory writes before later async-proxy reads (MMA, TMA)
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

template <int CP, bool TRAIN>
__global__ void __launch_bounds__(TRAIN ? 96 + 32 * kHtEpi : 192, CP == 16 ? 2 : 1) k_head_tc(const HeadTcArgs g) {
  using G = HtGeo<CP>;
  const HeadTcJob jb = g.jobs[blockIdx.x];
  const int r0 = jb.blk * kRowTile;
  if (r0 >= g.B_pad) return;
  extern __shared__ uint8_t ht_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)ht_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* Ds = smem + kHtStages * G::kStage;
  HtTail* tl = (HtTail*)(Ds + (TRAIN ? G::kD : 0));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int w = jb.w, nst = (w + 127) >> 7;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kHtStages; ++s) {
      mbar_init(&tl->full[s], 1);
      mbar_init(&tl->empty[s], 1);
      mbar_init(&tl->rel[s], 1);
      mbar_init(&tl->half[s][0], 4);
      mbar_init(&tl->half[s][1], 4);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&tl->z_full[s], 1);
      mbar_init(&tl->z_free[s], 4);
    }
    mbar_init(&tl->d_ready, 4);
    mbar_init(&tl->t_full, 1);
    mbar_init(&tl->t_free, kHtEpi);
    mbar_init(&tl->done, 1);
    tl->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  constexpr uint32_t kCols = G::kTmemCols;
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tl->tmem_base)),
                 "r"(kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();   // the set-up above overlaps the previous kernel
  const uint32_t tmem = tl->tmem_base;
  volatile int* abort_flag = &tl->abort;

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      fence_proxy_async_global();
      const CUtensorMap* map = g.maps + jb.map_h;
      const int total = TRAIN ? 2 * nst : nst;
      int it = 0;
      for (; it < total; ++it) {
        const int s = it & 1, step = it < nst ? it : it - nst;
        if (it >= kHtStages) {
          const int prev = it - kHtStages;   // the stage's previous step: the MMAs' or the storer's to free
          const int first = nst + ((nst ^ s) & 1);
          const bool got = prev < nst ? mbar_wait(&tl->empty[s], (prev >> 1) & 1, abort_flag, g.err, kHtWaitNs, 21)
                                      : mbar_wait(&tl->rel[s], ((prev - first) >> 1) & 1, abort_flag, g.err,
                                                  2 * kHtWaitNs, 22);
          if (!got) break;
        }
        const int nb = w - 128 * step > 64 ? 2 : 1;
        uint8_t* st = smem + s * G::kStage;
        mbar_expect_tx(&tl->full[s], (uint32_t)nb * (kHtBox + G::kWChunk));
        for (int b = 0; b < nb; ++b)
          tma_load_2d(smem_u32(st + b * kHtBox), map, &tl->full[s], 128 * step + 64 * b, r0);
        bulk_load(smem_u32(st + 2 * kHtBox), g.wsplit + jb.wsplit_off + (int64_t)2 * step * G::kWChunk,
                  (uint32_t)nb * G::kWChunk, &tl->full[s]);
      }
      // every copy has landed before the CTA leaves
      for (int k = max(0, it - kHtStages); k < it; ++k) {
        int dummy_abort = 0;
        mbar_wait(&tl->full[k & 1], (k >> 1) & 1, &dummy_abort, g.err, kHtWaitNs, 23);
      }
    }
  } else if (warp == 1) {
    // ----------------------------------------------------------------- MMA
    if (lane == 0) {
      const uint32_t s0 = smem_u32(smem), d0 = smem_u32(Ds);
      bool ok = true;
      const uint32_t id_z = instr_desc(128, G::kN, 0, 0);
      for (int step = 0; ok && step < nst; ++step) {
        const int s = step & 1;
        if (!mbar_wait(&tl->full[s], (step >> 1) & 1, abort_flag, g.err, 2 * kHtWaitNs, 24) ||
            (step >= 2 && !mbar_wait(&tl->z_free[s], ((step >> 1) - 1) & 1, abort_flag, g.err, 4 * kHtWaitNs, 26))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t h = s0 + s * G::kStage, wp = h + 2 * kHtBox;
        const int nk = min(128, w - 128 * step) >> 4;
        for (int k = 0; k < nk; ++k)
          umma_bf16<1>(tmem + (2 * s + (k >> 2)) * G::kAcc, smem_desc(h + (k >> 2) * kHtBox + 32 * (k & 3), 16, 1024),
                       smem_desc(wp + (k >> 2) * G::kWChunk + 32 * (k & 3), 16, 1024), id_z, k & 3);
        umma_commit<1>(&tl->empty[s]);
        umma_commit<1>(&tl->z_full[s]);
      }
      if constexpr (TRAIN) {
        if (ok) ok = mbar_wait(&tl->d_ready, 0, abort_flag, g.err, 4 * kHtWaitNs, 25);
        const uint32_t id_w = instr_desc(128, G::kN, 1, 1);
        for (int step = 0; ok && step < nst; ++step) {
          const int it = nst + step, s = it & 1;
          if (!mbar_wait(&tl->full[s], (it >> 1) & 1, abort_flag, g.err, 2 * kHtWaitNs, 24) ||
              (step && !mbar_wait(&tl->t_free, (step - 1) & 1, abort_flag, g.err, 4 * kHtWaitNs, 26))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t h = s0 + s * G::kStage, wp = h + 2 * kHtBox;
          const uint32_t id_h = instr_desc(128, min(128, w - 128 * step), 0, 1);
          // dH: parts (of D, of the weights), the smallest products first;
          // K = 16 classes per instruction
          uint32_t acc = 0;
          constexpr int kG = CP / 16;
#pragma unroll
          for (int q = 0; q < 6; ++q) {
            const int pd = q == 0 ? 2 : q == 1 || q == 3 ? 1 : 0, pw = q == 2 ? 2 : q == 1 || q == 4 ? 1 : 0;
#pragma unroll
            for (int c = 0; c < kG; ++c) {
              const int gd = pd * kG + c, gw = pw * kG + c;
              umma_bf16<1>(tmem + G::kDh, smem_desc(d0 + (gd >> 2) * kHtBox + 32 * (gd & 3), 16, 1024),
                           smem_desc(wp + 2048 * gw, G::kWChunk, 1024), id_h, acc);
              acc = 1;
            }
          }
          // dW_h^T of the step's columns: K = the 128 rows, each half for itself
          for (int k = 0; k < 8; ++k)
            umma_bf16<1>(tmem + (k >> 2) * G::kAcc, smem_desc(h + 2048 * k, kHtBox, 1024),
                         smem_desc(d0 + 2048 * k, kHtBox, 1024), id_w, k & 3);
          umma_commit<1>(&tl->t_full);
        }
      }
      umma_commit<1>(&tl->done);   // all MMAs this thread issued are over before TMEM is freed
      int dummy_abort = 0;
      mbar_wait(&tl->done, 0, &dummy_abort, g.err, kHtWaitNs, 27);
    }
  } else if (warp < 2 + (TRAIN ? kHtEpi : 4)) {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3, half = (warp - 2) >> 2;
    const int rl = 32 * q + lane, r = r0 + rl;
    const uint32_t tq = tmem + ((uint32_t)(32 * q) << 16);
    const int d_out = g.d_out;
    bool ok = true;
    if (half == 0) {
      uint32_t label = 0;
      if constexpr (TRAIN)
        if (r < g.B) label = row_label(g.y, g.idx ? g.idx + (int64_t)jb.member * g.idx_stride : nullptr, r);
      float z[CP];
#pragma unroll
      for (int c = 0; c < CP; ++c) z[c] = 0.f;
      for (int step = 0; ok && step < nst; ++step) {   // each step's products, added in fp32
        const int s = step & 1;
        ok = mbar_wait(&tl->z_full[s], (step >> 1) & 1, abort_flag, g.err, 4 * kHtWaitNs, 28);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        float zs[CP];
        tmem_sum3<CP, CP>(tq + 2 * s * G::kAcc, 0, w - 128 * step > 64, zs);
#pragma unroll
        for (int c = 0; c < CP; ++c) z[c] += zs[c];
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_relaxed(&tl->z_free[s]);   // the loads above have completed
      }
      if (ok) {
        const float* bh = g.params + jb.b_off;
#pragma unroll
        for (int c = 0; c < CP; ++c)
          if (c < d_out) z[c] += __ldg(bh + c);
        if constexpr (!TRAIN) {
          if (r < g.B) {   // probabilities (a multiclass head)
            float mx = z[0];
#pragma unroll
            for (int c = 1; c < CP; ++c)
              if (c < d_out) mx = fmaxf(mx, z[c]);
            float sum = 0.f;
#pragma unroll
            for (int c = 0; c < CP; ++c)
              if (c < d_out) {
                z[c] = expf(z[c] - mx);
                sum += z[c];
              }
            const float inv = 1.f / sum;
            float* o = g.out + ((int64_t)jb.member * g.N + g.n0 + r) * d_out;
#pragma unroll
            for (int c = 0; c < CP; ++c)
              if (c < d_out) o[c] = z[c] * inv;
          }
        } else {
          float dl[CP];
          float loss = 0.f;
#pragma unroll
          for (int c = 0; c < CP; ++c) dl[c] = 0.f;
          if (r < g.B) {
            loss = row_loss<CP>(g.task, d_out, z, label, 1.f / (float)g.B, dl);
            float* lg = g.logits + ((int64_t)jb.member * g.B_cap + r) * d_out;
#pragma unroll
            for (int c = 0; c < CP; ++c)
              if (c < d_out) lg[c] = z[c];
          }
          // D's row: three parts of CP classes, in 16-byte groups of eight
#pragma unroll
          for (int gr = 0; gr < CP / 8; ++gr) {
            float e[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) e[k] = dl[8 * gr + k];
#pragma unroll
            for (int p = 0; p < 3; ++p) {
              uint32_t pk[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                pk[k] = pack_bf16x2(e[2 * k], e[2 * k + 1]);
                e[2 * k] -= __uint_as_float(pk[k] << 16);
                e[2 * k + 1] -= __uint_as_float(pk[k] & 0xFFFF0000u);
              }
              const int c16 = (p * CP + 8 * gr) >> 3;   // 16-byte group within the row of 3 CP classes
              *reinterpret_cast<uint4*>(Ds + (c16 >> 3) * kHtBox + rl * 128 + (((c16 & 7) ^ (rl & 7)) << 4)) =
                  make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
          }
          fence_proxy_async_smem();
          // the 32 rows' loss and class sums (bias gradient)
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
          float cs[32];
#pragma unroll
          for (int c = 0; c < 32; ++c) cs[c] = c < CP ? dl[c < CP ? c : 0] : 0.f;
          tl->db[q][lane] = colsum32(cs, lane);
          if (lane == 0) tl->loss[q] = loss;
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&tl->d_ready);
        }
      }
    }
    if constexpr (TRAIN) {
      const float scale = g.mem[jb.member].scale;
      float* part = g.head_part + jb.part_off;
      for (int step = 0; ok && step < nst; ++step) {
        const int it = nst + step, s = it & 1;
        const int ncols = min(128, w - 128 * step);
        ok = mbar_wait(&tl->t_full, step & 1, abort_flag, g.err, 4 * kHtWaitNs, 28) &&
             mbar_wait(&tl->full[s], (it >> 1) & 1, abort_flag, g.err, kHtWaitNs, 28);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        uint8_t* hrow = smem + s * G::kStage + half * kHtBox + rl * 128;
#pragma unroll 1
        for (int ci = 0; ci < 2; ++ci) {
          const int c = 64 * half + 32 * ci;
          if (c >= ncols) break;   // warp-uniform
          uint32_t v[32];
          tmem_ld32(tq + G::kDh + c, v);
#pragma unroll
          for (int sg = 0; sg < 4; ++sg) {
            uint4* slot = reinterpret_cast<uint4*>(hrow + (((4 * ci + sg) ^ (rl & 7)) << 4));
            const uint4 hv = *slot;
            const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w};
            uint32_t pk[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float h0 = __uint_as_float(hw[e] << 16), h1 = __uint_as_float(hw[e] & 0xFFFF0000u);
              pk[e] = pack_bf16x2(h0 > 0.f ? __uint_as_float(v[8 * sg + 2 * e]) * scale : 0.f,
                                  h1 > 0.f ? __uint_as_float(v[8 * sg + 2 * e + 1]) * scale : 0.f);
            }
            *slot = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            if (jb.colsum) {
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                v[8 * sg + 2 * e] = pk[e] << 16;
                v[8 * sg + 2 * e + 1] = pk[e] & 0xFFFF0000u;
              }
            }
          }
          if (jb.colsum) {   // column sums of dZ as stored over the warp's 32 rows
            float x[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) x[e] = __uint_as_float(v[e]);
            tl->colsum[s][q][c + lane] = colsum32(x, lane);
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tl->half[s][half]);
        // dW_h of column 128 step + rl, this half's classes
        {
          float dw[CP / 2];
          tmem_sum3<CP, CP / 2>(tq, half * (CP / 2), true, dw);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_relaxed(&tl->t_free);   // the loads above have completed
          if (rl < ncols) {
#pragma unroll
            for (int c = 0; c < CP / 2; ++c) {
              const int cc = half * (CP / 2) + c;
              if (cc < d_out) part[(int64_t)cc * w + 128 * step + rl] = dw[c];
            }
          }
        }
      }
    }
  } else {
    // -------------------------------------------------------------- storer
    // Per step, once both halves are written: dZ's boxes leave by TMA (the
    // map clips columns past the width) and the stage is free.
    if constexpr (TRAIN) {
      float* part = g.head_part + jb.part_off;
      bool ok = __all_sync(0xffffffffu, mbar_wait(&tl->d_ready, 0, abort_flag, g.err, 8 * kHtWaitNs, 25));
      if (ok) {   // the block's bias gradient and loss, 32-row groups in order
        if (lane < g.d_out)
          part[(int64_t)g.d_out * w + lane] = ((tl->db[0][lane] + tl->db[1][lane]) + tl->db[2][lane]) + tl->db[3][lane];
        if (lane == 0)
          g.loss_part[(int64_t)jb.member * g.n_blk_cap + jb.blk] =
              ((tl->loss[0] + tl->loss[1]) + tl->loss[2]) + tl->loss[3];
      }
      const CUtensorMap* map = g.maps + jb.map_dz;
      for (int step = 0; ok && step < nst; ++step) {
        const int it = nst + step, s = it & 1;
        const int first = nst + ((nst ^ s) & 1);
        const uint32_t par = ((it - first) >> 1) & 1;
        const int ncols = min(128, w - 128 * step);
        ok = mbar_wait(&tl->half[s][0], par, abort_flag, g.err, 8 * kHtWaitNs, 29) &&
             mbar_wait(&tl->half[s][1], par, abort_flag, g.err, 8 * kHtWaitNs, 29);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        if (lane == 0) {
          const uint32_t st = smem_u32(smem + s * G::kStage);
          tma_store_2d(map, st, 128 * step, r0);
          if (ncols > 64) tma_store_2d(map, st + kHtBox, 128 * step + 64, r0);
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        if (jb.colsum && g.dbp) {   // partials of 64 rows: pairs of the 32-row sums
          float* dbp = g.dbp + jb.dz_off / 32 + (int64_t)(2 * jb.blk) * w + 128 * step;
          for (int c = lane; c < ncols; c += 32) {
            dbp[c] = tl->colsum[s][0][c] + tl->colsum[s][1][c];
            dbp[w + c] = tl->colsum[s][2][c] + tl->colsum[s][3][c];
          }
        }
        __syncwarp();
        if (lane == 0) {
          asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          mbar_arrive(&tl->rel[s]);
        }
      }
      if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
  }

  pdl_trigger();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

}  // namespace

int64_t head_tc_chunk_bytes(int d_out) { return d_out <= 16 ? HtGeo<16>::kWChunk : HtGeo<32>::kWChunk; }

void head_tc_prepare() {
  cudaFuncSetAttribute(k_head_tc<16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ht_smem<16, true>());
  cudaFuncSetAttribute(k_head_tc<32, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ht_smem<32, true>());
  cudaFuncSetAttribute(k_head_tc<16, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, ht_smem<16, false>());
  cudaFuncSetAttribute(k_head_tc<32, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, ht_smem<32, false>());
}

void launch_head_tc(cudaStream_t st, const HeadTcArgs& g, int n_jobs, bool train) {
  if (n_jobs <= 0) return;
  const bool few = g.d_out <= 16;
  if (train) {
    if (few) launch_pdl(k_head_tc<16, true>, dim3(n_jobs), dim3(96 + 32 * kHtEpi), ht_smem<16, true>(), st, g);
    else launch_pdl(k_head_tc<32, true>, dim3(n_jobs), dim3(96 + 32 * kHtEpi), ht_smem<32, true>(), st, g);
  } else {
    if (few) launch_pdl(k_head_tc<16, false>, dim3(n_jobs), dim3(192), ht_smem<16, false>(), st, g);
    else launch_pdl(k_head_tc<32, false>, dim3(n_jobs), dim3(192), ht_smem<32, false>(), st, g);
  }
}

}  // namespace tp
