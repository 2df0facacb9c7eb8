// The warm-start network on the tensor cores.  A tile of 128 samples goes
// through all layers in one CTA: its activations never leave the SM (bf16, the
// MMA's A operand, 64 KB of shared memory), the weights stream in from L2 in
// 16 KB chunks, sums are FP32 in TMEM, and bias, tanh (or its derivative) and
// the rounding to bf16 are the epilogue.
//   forward   A = features, W_1 .. W_5          -> outputs (and H_l for a gradient)
//   backward  A = dY, W_5^T .. W_2^T            -> D_4 .. D_1 and their column sums
//   weights   dW_l = H_{l-1}^T D_l, K = samples -> one partial per CTA, added in order
// What bounds it: the 1024 tanhf of a sample, about 40 instructions each; the
// products are a tenth of that time and run beside the other CTA's tanh (two
// CTAs per SM).
#include "mlp_umma.cuh"
#include "umma_core.cuh"

namespace nedmft {

using namespace umma;

namespace {

constexpr int kRows = 128;             // samples per tile
constexpr int kChunkK = 32;            // k per weight chunk
constexpr int kChunk = 256 * kChunkK;  // bf16 elements (16 KB): 256 rows x 32 k
constexpr int kFwdChunks = 26;         // 1 (W_1, k padded to 32) + 3 x 8 + 1 (W_5: 16 rows x 256 k)
constexpr int kBwdChunks = 25;         // 1 (W_5^T, k padded to 16 of 32) + 3 x 8
constexpr int kAct = kRows * kMlpHid;  // elements of an activation image (64 KB)
constexpr int kEpiWarps = 16;
constexpr int kThreads = 64 + 32 * kEpiWarps;

// element offset in an image of R rows x (8 cores) k, 8 x 8 core matrices of
// 128 bytes, k-adjacent cores next to each other
__host__ __device__ __forceinline__ int img_off(int r, int k, int cores) {
  return ((r >> 3) * cores + (k >> 3)) * 64 + (r & 7) * 8 + (k & 7);
}

// ------------------------------------------------------------------ weights

// Chunk blockIdx.x of the forward (< 26) or backward images; a thread takes eight
// consecutive k of one row, a 16-byte core-matrix row, four CTAs per chunk (22 us
// on 51 CTAs with one element at a time).
constexpr int kPackSplit = 4;
__global__ void __launch_bounds__(256) mlp_pack_kernel(const float* __restrict__ params,
                                                       __nv_bfloat16* __restrict__ img) {
  const int c = blockIdx.x, u = blockIdx.y * 256 + threadIdx.x;  // unit of the chunk's 1024
  __nv_bfloat16* out = img + (size_t)c * kChunk;
  int off;
  float v[8];
  auto at = [&](bool inside, size_t o) { return inside ? params[o] : 0.f; };
  if (c == kFwdChunks - 1) {  // W_5: rows o < 2 (of 16), k = i
    const int r = u & 15, k = 8 * (u >> 4);
    if (k >= kMlpHid) return;
    off = img_off(r, k, 32);
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = at(r < kMlpOut, mlp_w_off(4) + (size_t)(k + q) * kMlpOut + r);
  } else if (c < kFwdChunks) {  // rows o, k = i: consecutive threads, consecutive outputs of a row of W
    const int l = c == 0 ? 0 : 1 + (c - 1) / 8, k0 = c == 0 ? 0 : 32 * ((c - 1) % 8);
    const int r = u & 255, k = 8 * (u >> 8);
    off = img_off(r, k, 4);
#pragma unroll
    for (int q = 0; q < 8; ++q)
      v[q] = at(k0 + k + q < (l == 0 ? kMlpIn : kMlpHid), mlp_w_off(l) + (size_t)(k0 + k + q) * kMlpHid + r);
  } else {
    const int d = c - kFwdChunks, r = u >> 2, k = 8 * (u & 3);
    off = img_off(r, k, 4);
    if (d == 0) {  // W_5^T: rows i, k = o
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = at(k + q < kMlpOut, mlp_w_off(4) + (size_t)r * kMlpOut + k + q);
    } else {  // rows i, k = o
      const int l = 3 - (d - 1) / 8, k0 = 32 * ((d - 1) % 8);
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = params[mlp_w_off(l) + (size_t)r * kMlpHid + k0 + k + q];
    }
  }
  uint32_t w[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const __nv_bfloat162 h = __halves2bfloat162(__float2bfloat16_rn(v[2 * q]), __float2bfloat16_rn(v[2 * q + 1]));
    w[q] = *reinterpret_cast<const uint32_t*>(&h);
  }
  *reinterpret_cast<uint4*>(out + off) = make_uint4(w[0], w[1], w[2], w[3]);
}

// ------------------------------------------------------------------ forward and backward

struct MlpBars {
  uint64_t full[8], empty[8], a_ready, d_full, drain;
  uint32_t tmem_slot;
  int abort;
  float col[4][kMlpHid];  // column sums of a tile's four row quarters (backward)
  double loss[4];
};
constexpr int kActBytes = kAct * 2, kChunkBytes = kChunk * 2;
constexpr size_t mlp_smem(int stages) { return kActBytes + (size_t)stages * kChunkBytes + sizeof(MlpBars) + 1024; }

struct MlpParams {
  const float* params;
  const __nv_bfloat16* wimg;  // the pass's chunks
  MlpInput in;
  size_t n;
  int tiles, stages;
  // forward
  float* y;
  bool accumulate, first;
  float scale;
  // gradient: activations FP32, [tile][layer][column / 4][row][4], and bf16 images
  float* h32;
  __nv_bfloat16 *himg, *ximg, *dimg, *dyimg;
  const float* target;
  float inv;
  double* loss_part;
  float* colsum;  // [tile][layer][256], the output layer's two in [tile][4]
  int* status;
};

__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
        "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// shared -> global bulk copy, tracked by bulk groups
__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ uint32_t bf16_pair(float a, float b) {
  const __nv_bfloat162 h = __halves2bfloat162(__float2bfloat16_rn(a), __float2bfloat16_rn(b));
  return *reinterpret_cast<const uint32_t*>(&h);
}
// feature f of sample s, the pair (a, b) when features come from a contour
__device__ __forceinline__ float feature(const MlpInput& in, size_t s, int a, int b, int f) {
  if (in.x) return in.x[s * kMlpIn + f];
  if (f == 0) return in.u;
  if (f == 1) return in.e;
  if (f == 2) return in.rel[s];
  if (f < 9) return in.row[a * 6 + f - 3];
  if (f < 15) return in.row[b * 6 + f - 9];
  return f == 15 ? (a >= b ? 1.f : 0.f) : in.dt;
}
// the same answer on every one of the epilogue's threads
__device__ __forceinline__ bool epi_all(bool x) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 6, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)x), "n"(32 * kEpiWarps)
      : "memory");
  return r != 0;
}

// Persistent over tiles.  Warp 0 streams the pass's weight chunks through
// p.stages buffers, warp 1 issues the products of a layer once its A operand is
// there, the 16 epilogue warps (four per TMEM lane quarter, 64 columns each)
// write the next layer's A operand over it.
template <bool BWD, int MINB>
__global__ void __launch_bounds__(kThreads, MINB) mlp_tile_kernel(const __grid_constant__ MlpParams p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* act = smem;
  unsigned char* ring = smem + kActBytes;
  MlpBars& bars = *reinterpret_cast<MlpBars*>(ring + (size_t)p.stages * kChunkBytes);
  volatile int* abort_flag = &bars.abort;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  constexpr int kChunks = BWD ? kBwdChunks : kFwdChunks;
  constexpr int kSteps = BWD ? 4 : 5;  // products of a tile
  constexpr uint32_t kCols = 256;
  if (t == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&bars.full[s], 1);
      mbar_init(&bars.empty[s], 1);
    }
    mbar_init(&bars.a_ready, kEpiWarps);
    mbar_init(&bars.d_full, 1);
    mbar_init(&bars.drain, 1);
    bars.abort = 0;
    fence_barrier_init();
  }
  if (warp == 0) tmem_alloc(&bars.tmem_slot, kCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars.tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < p.tiles && ok; tile += gridDim.x)
        for (int c = 0; c < kChunks; ++c, ++it) {
          const int s = it % p.stages, round = it / p.stages;
          if (round > 0 && !mbar_wait(&bars.empty[s], (round - 1) & 1, abort_flag)) {
            ok = false;
            break;
          }
          const uint32_t bytes = !BWD && c == kChunks - 1 ? 16 * 256 * 2 : kChunkBytes;
          mbar_arrive_expect_tx(&bars.full[s], bytes);
          bulk_g2s(ring + (size_t)s * kChunkBytes, p.wimg + (size_t)c * kChunk, bytes, &bars.full[s]);
        }
      // no copy may be in flight when the CTA leaves
      for (int k = it > p.stages ? it - p.stages : 0; k < it; ++k)
        drain_wait(&bars.full[k % p.stages], (k / p.stages) & 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int it = 0, layer_no = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < p.tiles && ok; tile += gridDim.x)
        for (int l = 0; l < kSteps && ok; ++l, ++layer_no) {
          if (!(ok = mbar_wait(&bars.a_ready, layer_no & 1, abort_flag))) break;
          tc_fence_after();
          bool stored = false;
          if (p.h32 && l > 0) {  // the A operand, H_l or D_(5-l), is also a weight gradient's operand
            __nv_bfloat16* img = (BWD ? p.dimg : p.himg) + ((size_t)tile * 4 + (BWD ? 4 - l : l - 1)) * kAct;
            bulk_s2g(img, act, kActBytes);
            bulk_commit();
            stored = true;
          }
          const bool out_layer = !BWD && l == 4;
          const int nch = l == 0 || out_layer ? 1 : 8;
          for (int c = 0; c < nch; ++c, ++it) {
            const int s = it % p.stages;
            if (!(ok = mbar_wait(&bars.full[s], (it / p.stages) & 1, abort_flag))) break;
            tc_fence_after();
            const uint32_t a = smem_u32(act), b = smem_u32(ring + (size_t)s * kChunkBytes);
            if (out_layer) {
              for (int kk = 0; kk < 16; ++kk)
                mma_bf16(tmem, smem_desc(a + kk * 256, 128, 4096), smem_desc(b + kk * 256, 128, 4096),
                         idesc_bf16(128, 16), kk > 0 ? 1u : 0u);
            } else {
              const int ksteps = BWD && l == 0 ? 1 : 2;
              for (int kk = 0; kk < ksteps; ++kk)
                mma_bf16(tmem, smem_desc(a + c * 512 + kk * 256, 128, 4096), smem_desc(b + kk * 256, 128, 512),
                         idesc_bf16(128, 256), c > 0 || kk > 0 ? 1u : 0u);
            }
            mma_commit(&bars.empty[s]);
          }
          if (stored) bulk_wait_read();  // before the epilogue writes over the operand
          if (ok) mma_commit(&bars.d_full);
        }
      mma_commit(&bars.drain);
      drain_wait(&bars.drain, 0);
      if (p.h32) bulk_wait_all();
    }
  } else {
    const int quarter = warp & 3, part = (warp - 2) >> 2;
    const int r = quarter * 32 + lane;  // row of the tile
    const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16);
    auto a_done = [&]() {  // this warp's part of the A operand is written, its part of the accumulator read
      tc_fence_before();
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars.a_ready);
    };
    int step_no = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < p.tiles && ok; tile += gridDim.x) {
      const size_t s = (size_t)tile * kRows + r;
      const bool live = s < p.n;
      if constexpr (!BWD) {  // features, k = 8 part .. 8 part + 7 of 32
        float f[8];
        int pa = 0, pb = 0;
        if (p.in.nc > 0) {
          pa = (int)(s / (unsigned)p.in.nc);
          pb = (int)(s - (size_t)pa * p.in.nc);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) f[q] = live && 8 * part + q < kMlpIn ? feature(p.in, s, pa, pb, 8 * part + q) : 0.f;
        const uint4 v = make_uint4(bf16_pair(f[0], f[1]), bf16_pair(f[2], f[3]), bf16_pair(f[4], f[5]),
                                   bf16_pair(f[6], f[7]));
        *reinterpret_cast<uint4*>(act + 2 * img_off(r, 8 * part, 32)) = v;
        if (p.ximg) *reinterpret_cast<uint4*>(p.ximg + (size_t)tile * kRows * 32 + img_off(r, 8 * part, 4)) = v;
      } else if (part < 2) {  // dY = 2 (Y - T) / count, k = 0, 1 of 16
        uint4 v = make_uint4(0, 0, 0, 0);
        if (part == 0) {
          float d[2] = {0.f, 0.f};
          double sq = 0.0;
          if (live) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const float e = p.y[s * 2 + q] - p.target[s * 2 + q];
              d[q] = 2.f * e * p.inv;
              sq += (double)e * e;
            }
          }
          v.x = bf16_pair(d[0], d[1]);
          for (int o = 16; o > 0; o >>= 1) {
            d[0] += __shfl_xor_sync(0xffffffffu, d[0], o);
            d[1] += __shfl_xor_sync(0xffffffffu, d[1], o);
            sq += __shfl_xor_sync(0xffffffffu, sq, o);
          }
          if (lane == 0) {
            p.loss_part[(size_t)tile * 4 + quarter] = sq;
            p.colsum[((size_t)tile * 5 + 4) * kMlpHid + 2 * quarter] = d[0];
            p.colsum[((size_t)tile * 5 + 4) * kMlpHid + 2 * quarter + 1] = d[1];
          }
        }
        *reinterpret_cast<uint4*>(act + 2 * img_off(r, 8 * part, 32)) = v;
        *reinterpret_cast<uint4*>(p.dyimg + (size_t)tile * kRows * 16 + img_off(r, 8 * part, 2)) = v;
      }
      a_done();
      for (int l = 0; l < kSteps; ++l, ++step_no) {
        ok = __all_sync(0xffffffffu, mbar_wait(&bars.d_full, step_no & 1, abort_flag));
        if constexpr (BWD) ok = epi_all(ok);  // its barriers below need every warp
        if (!ok) break;
        tc_fence_after();
        if (!BWD && l == 4) {  // the two outputs
          if (part == 0) {
            float v[16];
            tmem_ld16(trow, v);
            tc_fence_before();
            if (live) {
              const float* bias = p.params + mlp_w_off(5) - kMlpOut;
#pragma unroll
              for (int q = 0; q < kMlpOut; ++q) {
                float o = v[q] + bias[q];
                float* dst = p.y + s * kMlpOut + q;
                if (p.accumulate) o = (p.first ? 0.f : *dst) + p.scale * o;
                *dst = o;
              }
            }
          }
          ++step_no;
          break;  // the next tile's features follow (every product has read the operand)
        }
        const int hl = BWD ? 3 - l : l;  // the hidden layer this epilogue makes (H_hl or D_hl), 0-based
        const float* bias = p.params + mlp_w_off(hl) + (size_t)(hl == 0 ? kMlpIn : kMlpHid) * kMlpHid;
        float* h32 = p.h32 ? p.h32 + ((size_t)tile * 4 + hl) * kAct : nullptr;
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          const int col = 64 * part + 16 * c;
          float v[16];
          tmem_ld16(trow + col, v);
#pragma unroll
          for (int q = 0; q < 16; q += 4) {
            if constexpr (!BWD) {
#pragma unroll
              for (int u = 0; u < 4; ++u) v[q + u] = tanhf(v[q + u] + bias[col + q + u]);
              if (h32)
                *reinterpret_cast<float4*>(h32 + ((size_t)((col + q) >> 2) * kRows + r) * 4) =
                    make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
            } else {
              const float4 h = *reinterpret_cast<const float4*>(h32 + ((size_t)((col + q) >> 2) * kRows + r) * 4);
              v[q] *= 1.f - h.x * h.x;
              v[q + 1] *= 1.f - h.y * h.y;
              v[q + 2] *= 1.f - h.z * h.z;
              v[q + 3] *= 1.f - h.w * h.w;
            }
          }
          if (BWD && !live) {
#pragma unroll
            for (int q = 0; q < 16; ++q) v[q] = 0.f;
          }
#pragma unroll
          for (int q = 0; q < 16; q += 8)
            *reinterpret_cast<uint4*>(act + 2 * img_off(r, col + q, 32)) =
                make_uint4(bf16_pair(v[q], v[q + 1]), bf16_pair(v[q + 2], v[q + 3]), bf16_pair(v[q + 4], v[q + 5]),
                           bf16_pair(v[q + 6], v[q + 7]));
          if constexpr (BWD) {
            // column sums over the warp's rows: halve the columns a lane holds, four
            // times, then add the lane pair; lane 2 q (and 2 q + 1) ends with column q
#pragma unroll
            for (int w = 8, bit = 16; w >= 1; w >>= 1, bit >>= 1)
#pragma unroll
              for (int q = 0; q < 8; ++q)
                if (q < w) {
                  const bool up = lane & bit;
                  const float mine = up ? v[q + w] : v[q], other = up ? v[q] : v[q + w];
                  v[q] = mine + __shfl_xor_sync(0xffffffffu, other, bit);
                }
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
            if ((lane & 1) == 0) bars.col[quarter][col + (lane >> 1)] = v[0];
          }
        }
        if (!BWD || l < kSteps - 1) a_done();  // D_1 is no product's operand
        else tc_fence_before();
        if constexpr (BWD) {
          // the four quarters' sums of the same 64 columns are added by the first quarter's warp
          asm volatile("bar.sync %0, 128;" ::"r"(1 + part) : "memory");
          if (quarter == 0)
            for (int q = lane; q < 64; q += 32) {
              const int col = 64 * part + q;
              p.colsum[((size_t)tile * 5 + hl) * kMlpHid + col] =
                  (bars.col[0][col] + bars.col[1][col]) + (bars.col[2][col] + bars.col[3][col]);
            }
          asm volatile("bar.sync %0, 128;" ::"r"(1 + part) : "memory");
        }
      }
      if (BWD && ok) {
        // D_1's image goes out once every warp has written it
        asm volatile("bar.sync 5, %0;" ::"n"(32 * kEpiWarps) : "memory");
        for (int e = t - 64; e < kActBytes / 16; e += 32 * kEpiWarps)
          reinterpret_cast<uint4*>(p.dimg + (size_t)tile * 4 * kAct)[e] = reinterpret_cast<const uint4*>(act)[e];
        asm volatile("bar.sync 5, %0;" ::"n"(32 * kEpiWarps) : "memory");
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kCols);
  }
  if (t == 0 && bars.abort && p.status) atomicCAS(p.status, 0, DS_TIMEOUT);
}

// ------------------------------------------------------------------ weight gradients

// dW of layer blockIdx.y over the tiles of split blockIdx.x, K = samples: the
// stored images are MN-major operands as they are (their 8 x 8 cores hold eight
// samples of eight features).  A (M = 256, two MMAs of 128 rows) is D_l, for
// the output layer H_4; B is H_{l-1}, the features or dY.  Half tiles of 64
// samples through three buffers.
constexpr int kHalf = 64;
constexpr int kDwStages = 3;
constexpr int kDwThreads = 64 + 256;
struct DwBars {
  uint64_t full[kDwStages], empty[kDwStages], done;
  uint32_t tmem_slot;
  int abort;
};
constexpr int kDwStageBytes = 2 * kHalf * kMlpHid * 2;  // 32 KB of A, at most 32 KB of B
constexpr size_t kDwSmem = (size_t)kDwStages * kDwStageBytes + sizeof(DwBars) + 1024;

__device__ __forceinline__ uint32_t idesc_mn(int n) { return idesc_bf16(128, n) | (1u << 15) | (1u << 16); }

__global__ void __launch_bounds__(kDwThreads, 1)
    mlp_dw_kernel(const __nv_bfloat16* __restrict__ himg, const __nv_bfloat16* __restrict__ ximg,
                  const __nv_bfloat16* __restrict__ dimg, const __nv_bfloat16* __restrict__ dyimg, int tiles,
                  float* __restrict__ partial, int* status) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  DwBars& bars = *reinterpret_cast<DwBars*>(smem + (size_t)kDwStages * kDwStageBytes);
  volatile int* abort_flag = &bars.abort;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int layer = blockIdx.y, split = blockIdx.x;
  const int t0 = (int)((long long)split * tiles / gridDim.x), t1 = (int)((long long)(split + 1) * tiles / gridDim.x);
  const int halves = 2 * (t1 - t0);
  const int N = layer == 0 ? 32 : layer == 4 ? 16 : kMlpHid;
  if (t == 0) {
    for (int s = 0; s < kDwStages; ++s) {
      mbar_init(&bars.full[s], 1);
      mbar_init(&bars.empty[s], 1);
    }
    mbar_init(&bars.done, 1);
    bars.abort = 0;
    fence_barrier_init();
  }
  if (warp == 0) tmem_alloc(&bars.tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars.tmem_slot;
  if (warp == 0) {
    if (lane == 0) {
      int k = 0;
      for (; k < halves; ++k) {
        const int s = k % kDwStages, round = k / kDwStages;
        if (round > 0 && !mbar_wait(&bars.empty[s], (round - 1) & 1, abort_flag)) break;
        const size_t tile = t0 + (k >> 1);
        const int h = k & 1;
        const __nv_bfloat16* a =
            (layer == 4 ? himg + (tile * 4 + 3) * kAct : dimg + (tile * 4 + layer) * kAct) + h * kHalf * kMlpHid;
        const __nv_bfloat16* b = layer == 0   ? ximg + tile * kRows * 32 + h * kHalf * 32
                                 : layer == 4 ? dyimg + tile * kRows * 16 + h * kHalf * 16
                                              : himg + (tile * 4 + layer - 1) * kAct + h * kHalf * kMlpHid;
        const uint32_t ab = kHalf * kMlpHid * 2, bb = kHalf * N * 2;
        unsigned char* st = smem + (size_t)s * kDwStageBytes;
        mbar_arrive_expect_tx(&bars.full[s], ab + bb);
        bulk_g2s(st, a, ab, &bars.full[s]);
        bulk_g2s(st + kDwStageBytes / 2, b, bb, &bars.full[s]);
      }
      for (int q = k > kDwStages ? k - kDwStages : 0; q < k; ++q)
        drain_wait(&bars.full[q % kDwStages], (q / kDwStages) & 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t bk = (uint32_t)N * 16;  // bytes between K-adjacent cores of B (eight samples)
      for (int k = 0; k < halves; ++k) {
        const int s = k % kDwStages;
        if (!mbar_wait(&bars.full[s], (k / kDwStages) & 1, abort_flag)) break;
        tc_fence_after();
        const uint32_t a = smem_u32(smem + (size_t)s * kDwStageBytes), b = a + kDwStageBytes / 2;
        for (int mh = 0; mh < 2; ++mh)
          for (int kk = 0; kk < kHalf / 16; ++kk)
            mma_bf16(tmem + (uint32_t)(mh * N), smem_desc(a + mh * 2048 + kk * 2 * 4096, 4096, 128),
                     smem_desc(b + kk * 2 * bk, bk, 128), idesc_mn(N), k > 0 || kk > 0 ? 1u : 0u);
        mma_commit(&bars.empty[s]);
      }
      mma_commit(&bars.done);
      drain_wait(&bars.done, 0);
    }
  } else {
    bool ok = __all_sync(0xffffffffu, mbar_wait(&bars.done, 0, abort_flag));
    if (!ok) drain_wait(&bars.done, 0);
    tc_fence_after();
    if (ok) {
      const int quarter = warp & 3, mh = (warp - 2) >> 2;
      const int row = mh * 128 + quarter * 32 + lane;
      const int n_out = layer == 0 ? kMlpIn : layer == 4 ? kMlpOut : kMlpHid;
      float* out = partial + (size_t)split * mlp_w_off(kMlpLayers) + mlp_w_off(layer);
      for (int c = 0; c < N; c += 16) {
        float v[16];
        tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(mh * N + c), v);
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (c + q < n_out) out[layer == 4 ? (size_t)row * kMlpOut + c + q : (size_t)(c + q) * kMlpHid + row] = v[q];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (t == 0 && bars.abort && status) atomicCAS(status, 0, DS_TIMEOUT);
}

// grad = the splits' weight gradients, and the tiles' column sums for the biases, added in order; the loss.
__global__ void __launch_bounds__(256) mlp_finish_kernel(const float* __restrict__ partial, int splits,
                                                         const float* __restrict__ colsum, int tiles,
                                                         const double* __restrict__ loss_part, double inv,
                                                         float* __restrict__ grad, float* __restrict__ loss) {
  constexpr int kParams = (int)mlp_w_off(kMlpLayers);
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e < kParams) {
    int l = 0;
#pragma unroll
    for (int q = 1; q < kMlpLayers; ++q)
      if (e >= (int)mlp_w_off(q)) l = q;
    const int width = l == kMlpLayers - 1 ? kMlpOut : kMlpHid;
    const int w = (l == 0 ? kMlpIn : kMlpHid) * width;
    const int at = e - (int)mlp_w_off(l);
    float x = 0.f;
    if (at < w) {
#pragma unroll 8
      for (int s = 0; s < splits; ++s) x += partial[(size_t)s * kParams + e];
    } else if (l < kMlpLayers - 1) {
#pragma unroll 8
      for (int tl = 0; tl < tiles; ++tl) x += colsum[((size_t)tl * 5 + l) * kMlpHid + at - w];
    } else {
#pragma unroll 4
      for (int tl = 0; tl < tiles; ++tl) {
        const float* c = colsum + ((size_t)tl * 5 + 4) * kMlpHid + at - w;
        x += (c[0] + c[2]) + (c[4] + c[6]);
      }
    }
    grad[e] = x;
  }
  if (blockIdx.x == gridDim.x - 1) {  // the loss: threads in strides, then a tree
    __shared__ double red[256];
    double sum = 0.0;
    for (int k = threadIdx.x; k < 4 * tiles; k += 256) sum += loss_part[k];
    red[threadIdx.x] = sum;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
      if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
      __syncthreads();
    }
    if (threadIdx.x == 0) *loss = (float)(red[0] * inv);
  }
}

constexpr int kMaxSplits = 30;  // 5 layers x 30 splits cover the 152 SMs

struct GradLayout {
  size_t wimg, h32, himg, ximg, dimg, dyimg, y, loss, colsum, partial, total;
  int tiles, splits;
};
GradLayout grad_layout(int n) {
  GradLayout L;
  L.tiles = (n + kRows - 1) / kRows;
  L.splits = L.tiles < kMaxSplits ? L.tiles : kMaxSplits;
  const size_t t = L.tiles;
  L.wimg = align256(2 * (size_t)kChunk * (kFwdChunks + kBwdChunks));
  L.h32 = align256(sizeof(float) * t * 4 * kAct);
  L.himg = align256(2 * t * 4 * kAct);
  L.ximg = align256(2 * t * kRows * 32);
  L.dimg = L.himg;
  L.dyimg = align256(2 * t * kRows * 16);
  L.y = align256(sizeof(float) * t * kRows * kMlpOut);
  L.loss = align256(sizeof(double) * t * 4);
  L.colsum = align256(sizeof(float) * t * 5 * kMlpHid);
  L.partial = align256(sizeof(float) * mlp_w_off(kMlpLayers) * L.splits);
  L.total = L.wimg + L.h32 + L.himg + L.ximg + L.dimg + L.dyimg + L.y + L.loss + L.colsum + L.partial;
  return L;
}

// A CTA per SM with eight weight buffers while every tile has an SM to itself,
// else two per SM with two buffers each: one's products and loads run beside
// the other's tanh.
template <bool BWD>
int launch_tiles(MlpParams& p, cudaStream_t st) {
  int sms = 0;
  if (int rc = device_sm_count(&sms)) return rc;
  if (p.tiles <= sms) {
    p.stages = 8;
    const int smem = (int)mlp_smem(8);
    if (int rc = ensure_dyn_smem(reinterpret_cast<const void*>(mlp_tile_kernel<BWD, 1>), smem)) return rc;
    mlp_tile_kernel<BWD, 1><<<p.tiles, kThreads, smem, st>>>(p);
  } else {
    p.stages = 2;
    const int smem = (int)mlp_smem(2);
    if (int rc = ensure_dyn_smem(reinterpret_cast<const void*>(mlp_tile_kernel<BWD, 2>), smem)) return rc;
    mlp_tile_kernel<BWD, 2><<<p.tiles < 2 * sms ? p.tiles : 2 * sms, kThreads, smem, st>>>(p);
  }
  NED_LAUNCH_CHECK("mlp_tile_kernel");
  return NEDMFT_OK;
}

}  // namespace

size_t mlp_forward_scratch() { return align256(2 * (size_t)kChunk * (kFwdChunks + kBwdChunks)); }
size_t mlp_grad_scratch(int n) { return grad_layout(n).total; }

int mlp_set_wait_ns(uint64_t ns, cudaStream_t st) {
  NED_CUDA(cudaMemcpyToSymbolAsync(umma::g_wait_ns, &ns, sizeof(ns), 0, cudaMemcpyHostToDevice, st));
  NED_CUDA(cudaStreamSynchronize(st));
  return NEDMFT_OK;
}

int mlp_forward(const float* params, const MlpInput& in, size_t n, float* y, bool accumulate, bool first, float scale,
                bool pack, char* scratch, cudaStream_t st) {
  __nv_bfloat16* wimg = reinterpret_cast<__nv_bfloat16*>(scratch);
  if (pack) {
    mlp_pack_kernel<<<dim3(kFwdChunks, kPackSplit), 256, 0, st>>>(params, wimg);
    NED_LAUNCH_CHECK("mlp_pack_kernel");
  }
  MlpParams p{};
  p.params = params;
  p.wimg = wimg;
  p.in = in;
  p.n = n;
  p.tiles = (int)((n + kRows - 1) / kRows);
  p.y = y;
  p.accumulate = accumulate;
  p.first = first;
  p.scale = scale;
  p.status = device_status_ptr();
  return launch_tiles<false>(p, st);
}

int mlp_gradient(const float* params, const float* x, const float* target, int n, float* grad, float* loss,
                 char* scratch, cudaStream_t st) {
  const GradLayout L = grad_layout(n);
  char* q = scratch;
  auto take = [&](size_t bytes) {
    char* r = q;
    q += bytes;
    return r;
  };
  __nv_bfloat16* wimg = reinterpret_cast<__nv_bfloat16*>(take(L.wimg));
  MlpParams p{};
  p.params = params;
  p.in.x = x;
  p.n = (size_t)n;
  p.tiles = L.tiles;
  p.h32 = reinterpret_cast<float*>(take(L.h32));
  p.himg = reinterpret_cast<__nv_bfloat16*>(take(L.himg));
  p.ximg = reinterpret_cast<__nv_bfloat16*>(take(L.ximg));
  p.dimg = reinterpret_cast<__nv_bfloat16*>(take(L.dimg));
  p.dyimg = reinterpret_cast<__nv_bfloat16*>(take(L.dyimg));
  p.y = reinterpret_cast<float*>(take(L.y));
  p.loss_part = reinterpret_cast<double*>(take(L.loss));
  p.colsum = reinterpret_cast<float*>(take(L.colsum));
  float* partial = reinterpret_cast<float*>(take(L.partial));
  p.target = target;
  p.inv = 1.f / (float)((size_t)n * kMlpOut);
  p.status = device_status_ptr();
  mlp_pack_kernel<<<dim3(kFwdChunks + kBwdChunks, kPackSplit), 256, 0, st>>>(params, wimg);
  NED_LAUNCH_CHECK("mlp_pack_kernel");
  p.wimg = wimg;
  if (int rc = launch_tiles<false>(p, st)) return rc;
  p.wimg = wimg + (size_t)kFwdChunks * kChunk;
  if (int rc = launch_tiles<true>(p, st)) return rc;
  if (int rc = ensure_dyn_smem(reinterpret_cast<const void*>(mlp_dw_kernel), (int)kDwSmem)) return rc;
  mlp_dw_kernel<<<dim3(L.splits, kMlpLayers), kDwThreads, kDwSmem, st>>>(p.himg, p.ximg, p.dimg, p.dyimg, L.tiles,
                                                                         partial, p.status);
  NED_LAUNCH_CHECK("mlp_dw_kernel");
  const int blocks = (int)((mlp_w_off(kMlpLayers) + 255) / 256);
  mlp_finish_kernel<<<blocks, 256, 0, st>>>(partial, L.splits, p.colsum, L.tiles, p.loss_part,
                                            1.0 / (double)((size_t)n * kMlpOut), grad, loss);
  NED_LAUNCH_CHECK("mlp_finish_kernel");
  return NEDMFT_OK;
}

}  // namespace nedmft
