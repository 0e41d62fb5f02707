// kp_mlp_tc.cuh -- the network's inference on the fifth-generation tensor
// cores: all three layers of a 128-row tile in one kernel, weights and hidden
// activations on chip.
#pragma once

#include "kp_mlp.cuh"
#include "kp_tc.cuh"

namespace kp {
namespace tc {

// ---------------------------------------------------------------------------
// weights as the tensor cores read them
// ---------------------------------------------------------------------------

// A hidden layer's weights W[n][k] in the order a CTA copies them to shared
// memory, so that an untiled bulk copy brings the operand in its final form:
// W2 as four K chunks of 64 (rows n of 128 bytes, 128-byte swizzle: 16-byte
// piece c of row n at c ^ (n & 7)), then W1 (rows of 64 bytes, 64-byte
// swizzle: piece c at c ^ ((n >> 1) & 3)).
constexpr int WT_CHUNK = MLP_H * 64;                 // elements of one W2 chunk
constexpr int WT_W1 = MLP_H * MLP_H;                 // W1 after W2
constexpr int WT_ELEMS = MLP_H * MLP_H + MLP_H * MLP_IN;

__host__ __device__ __forceinline__ int wt_index_w2(int n, int k) {
  const int c = (k & 63) >> 3;
  return (k >> 6) * WT_CHUNK + n * 64 + ((c ^ (n & 7)) << 3) + (k & 7);
}

__host__ __device__ __forceinline__ int wt_index_w1(int n, int k) {
  const int c = k >> 3;
  return WT_W1 + n * MLP_IN + ((c ^ ((n >> 1) & 3)) << 3) + (k & 7);
}

// Shared-memory matrix descriptor of a K-major tile of 64-byte rows with the
// 64-byte swizzle: 8-row groups 512 bytes apart.
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t addr) {
  uint64_t d = (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void fence_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes,
                                          uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

// Waits (bounded) as mbar_wait; gives up at once when another thread of the
// block has given up (*fail).
__device__ __forceinline__ bool mbar_wait_or(uint32_t bar, uint32_t parity, uint64_t limit_ns,
                                             int* fail, int site) {
  // the device clock is read only once the wait has become a long one (a
  // read of it takes longer than most waits here)
  uint64_t t0 = 0;
  for (uint32_t i = 0;; ++i) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if ((i & 63u) == 63u) {
      if (*((volatile int*)fail) != 0) return false;
      if (t0 == 0) t0 = now_ns();
      if (now_ns() - t0 > limit_ns) {
        *((volatile int*)fail) = site;
        return false;
      }
    }
  }
}

// 16 lanes x 32 columns of tensor memory in the accumulator layout of
// mma.sync: block b of 8 columns in r[4 b ..]: (row g, columns 2t, 2t + 1),
// then (row g + 8, the same columns), g = lane / 4, t = lane % 4.  Not
// waited for (tmem_wait_ld).
__device__ __forceinline__ void tmem_ld_16x256_x4(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}

// Waits for the calling thread's tensor-memory loads; the loaded registers
// pass through, so that no use moves above the wait.
template <int N>
__device__ __forceinline__ void tmem_wait_ld(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < N; ++i) asm volatile("" : "+r"(r[i]));
}

__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ void sts128(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w)
               : "memory");
}

// Two accumulators plus two biases, rounded to BF16, negative and NaN to 0.
__device__ __forceinline__ uint32_t bias_relu_bf16(uint32_t a, uint32_t b, float2 bias) {
  float x, y;  // one packed addition (two correctly rounded FP32 sums)
  asm("{\n .reg .b64 p, q;\n mov.b64 p, {%2, %3};\n mov.b64 q, {%4, %5};\n"
      " add.rn.f32x2 p, p, q;\n mov.b64 {%0, %1}, p;\n}"
      : "=f"(x), "=f"(y)
      : "r"(a), "r"(b), "f"(bias.x), "f"(bias.y));
  const __nv_bfloat162 v = __floats2bfloat162_rn(x, y);
  const __nv_bfloat162 r = __hmax2(v, __floats2bfloat162_rn(0.0f, 0.0f));
  return *reinterpret_cast<const uint32_t*>(&r);
}

// ---------------------------------------------------------------------------
// inference
// ---------------------------------------------------------------------------

constexpr int FT_ROWS = 128;           // rows of a tile: one tcgen05 M
constexpr int FT_G1 = 4, FT_G2 = 8;    // warps of epilogue 1 and of epilogue 2
constexpr int FT_THREADS = 32 * (FT_G1 + FT_G2 + 1);  // and one that issues
constexpr uint32_t FT_W2 = 0, FT_H = FT_W2 + 4 * MLP_H * 128, FT_W1 = FT_H + 4 * FT_ROWS * 128,
                   FT_X = FT_W1 + MLP_H * 64, FT_END = FT_X + FT_ROWS * 64;
constexpr int FT_SMEM = (int)FT_END + 1024;  // + room to align to 1 KB

struct FtArgs {
  const __nv_bfloat16* wt;  // W2, W1 in operand order (wt_index_*)
  const __nv_bfloat16* W3;  // row-major [8][256]
  const float *b1, *b2, *b3;
  const float* x;           // [M][32]
  float* out;               // [M][8]: mean, log_std
  int M, vec;               // vec: x and out allow 16- and 8-byte accesses
  int* err;
  unsigned long long wait_ns;
};

// Inputs 16 part .. 16 part + 15 of a row (zeros past the last row).
__device__ __forceinline__ void ft_load_x(const FtArgs& a, int row, int part, float* v) {
  const float* src = a.x + (size_t)row * MLP_IN + 16 * part;
  if (row >= a.M) {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = 0.0f;
  } else if (a.vec) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 f = __ldg(reinterpret_cast<const float4*>(src) + q);
      v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __ldg(src + i);
  }
}

// One persistent CTA per SM walks 128-row tiles.  Shared memory: both hidden
// layers' weights for the CTA's life, the tile's inputs and its first hidden
// activations (BF16 operands); tensor memory: the two layers' accumulators
// (256 columns each).  The last warp issues the tensor instructions; two
// groups of warps make the two epilogues, so that they run beside each other
// and beside layer 2, which then waits only for the first 64 columns:
//   1  warps 0-3 (rows 32 w ..): bias, ReLU, BF16 into the operand of layer 2,
//      which starts on each 64 columns (a K chunk) as soon as they are there;
//   2  warps 4-11 (rows 32 (w % 4) .., columns 128 half ..): bias, ReLU, BF16
//      as A fragments of mma.sync, which multiplies them by the 8-column
//      output layer without a round trip through memory; the two halves of a
//      row are added in shared memory; then tanh and the clamp.  They also
//      bring in the inputs of the next tile.
// Accumulators are read in the fragment layout of mma.sync, so that a thread
// needs the biases of few columns and keeps them in registers: shared memory
// is left to the tensor pipe, which takes 96 of its 128 B a clock.
//
// Measured (GB300): 262,145 rows in 42.5 us (0.93 PFLOP/s, 49 % of the measured
// bf16 rate) against 326 us for a kernel of one 32-row tile a block on mma.sync,
// which fetched every weight fragment from L2 for each tile; 33 rows 8.2
// against 10.3 us a call.  A tile takes about 5,000 clocks where its products
// need 2,300: the chain accumulator -> epilogue 1 -> first chunk -> layer 2 is
// what is left, and layer 2 runs at two thirds of its rate beside the
// epilogues' shared-memory and tensor-memory traffic.  Arrangements measured
// slower on the same rows: one group of 8 or 16 warps for both epilogues (54
// us), layer 2 in two halves of 128 columns (its operands then take all of the
// shared-memory bandwidth, 54 us), row-per-thread loads with the biases in
// shared memory (51 us).
__global__ void __launch_bounds__(FT_THREADS, 1) kp_mlp_forward_tc_kernel(FtArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t b_w1, b_w2[4], b_x, b_d1, b_h[4], b_d2, b_e2;
  __shared__ __align__(8) float s_part[2][FT_ROWS][MLP_OUT];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_fail;
  const uint32_t base = (saddr(smem_raw) + 1023u) & ~1023u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_tiles = (a.M + FT_ROWS - 1) / FT_ROWS;
  const int stride = (int)gridDim.x;
  if (tid == 32 * (FT_G1 + FT_G2)) {
    mbar_init(saddr(&b_w1), 1);
    mbar_init(saddr(&b_x), FT_G2);
    mbar_init(saddr(&b_d1), 1);
    for (int c = 0; c < 4; ++c) {
      mbar_init(saddr(&b_w2[c]), 1);
      mbar_init(saddr(&b_h[c]), FT_G1);
    }
    mbar_init(saddr(&b_d2), 1);
    mbar_init(saddr(&b_e2), FT_G2);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async();
    mbar_expect_tx(saddr(&b_w1), MLP_H * 64);
    bulk_load(base + FT_W1, a.wt + WT_W1, MLP_H * 64, saddr(&b_w1));
    for (int c = 0; c < 4; ++c) {
      mbar_expect_tx(saddr(&b_w2[c]), MLP_H * 128);
      bulk_load(base + FT_W2 + c * MLP_H * 128, a.wt + c * WT_CHUNK, MLP_H * 128, saddr(&b_w2[c]));
    }
  }
  if (warp == FT_G1 + FT_G2) {
    __syncwarp();
    tmem_alloc(saddr(&tmem_slot), 512);
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;
  // One arrival a warp.
  auto arrive = [&](uint64_t* bar) {
    fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(saddr(bar));
  };
  // After a wait that gave up the epilogues run on to their end (the waits
  // left return at once) without storing.
  auto wait = [&](uint64_t* bar, uint32_t parity, int site) {
    const bool ok = mbar_wait_or(saddr(bar), parity, a.wait_ns, &s_fail, site);
    __syncwarp(__activemask());
    fence_after();
    return ok;
  };

  if (warp == FT_G1 + FT_G2) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16_f32(FT_ROWS, MLP_H);
      auto layer1 = [&]() {
#pragma unroll
        for (int k = 0; k < 2; ++k)
          mma_bf16(tmem, sdesc_sw64(base + FT_X + 32 * k), sdesc_sw64(base + FT_W1 + 32 * k), idesc,
                   k != 0 ? 1u : 0u);
        mma_commit(saddr(&b_d1));
      };
      bool ok = wait(&b_w1, 0, 10) && wait(&b_x, 0, 11);
      if (ok) layer1();
      uint32_t ph = 0;
      for (int t = blockIdx.x; ok && t < n_tiles; t += stride, ph ^= 1u) {
        const bool first = t == (int)blockIdx.x, more = t + stride < n_tiles;
        if (!first) ok = wait(&b_e2, ph ^ 1u, 12);
        for (int c = 0; c < 4 && ok; ++c) {
          ok = (!first || wait(&b_w2[c], 0, 13)) && wait(&b_h[c], ph, 14);
          if (!ok) break;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_bf16(tmem + MLP_H, sdesc_sw128(base + FT_H + c * FT_ROWS * 128 + 32 * k),
                     sdesc_sw128(base + FT_W2 + c * MLP_H * 128 + 32 * k), idesc,
                     (c | k) != 0 ? 1u : 0u);
        }
        if (ok) mma_commit(saddr(&b_d2));
        if (ok && more) {
          ok = wait(&b_x, ph ^ 1u, 15);
          if (ok) layer1();
        }
      }
      // the weights' copies have landed before the block's memory goes
      for (int c = 0; c < 4; ++c) mbar_wait(saddr(&b_w2[c]), 0, a.wait_ns);
    }
    __syncwarp();
  } else if (warp < FT_G1) {
    const int g = lane >> 2, tq = lane & 3;
    const uint32_t tl = tmem + ((uint32_t)(32 * warp) << 16);
    // this thread's word of row 32 warp + g, piece 0 (pieces at piece ^ (row & 7))
    const uint32_t hrow = base + FT_H + (uint32_t)((32 * warp + g) * 128 + (g << 4) + 4 * tq);
    float2 bias[32];  // of columns 8 b + 2 tq, + 1
#pragma unroll
    for (int b = 0; b < 32; ++b) bias[b] = *reinterpret_cast<const float2*>(a.b1 + 8 * b + 2 * tq);
    uint32_t ph = 0;
    for (int t = blockIdx.x; t < n_tiles; t += stride, ph ^= 1u) {
      wait(&b_d1, ph, 20);
      if (t != (int)blockIdx.x) wait(&b_d2, ph ^ 1u, 21);  // the operand's last reader
      uint32_t r[2][16];
      // unit u: columns 32 (u / 2) .., rows 16 (u % 2) ..; the next unit's
      // load runs beside this one's arithmetic
      tmem_ld_16x256_x4(tl, r[0]);
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        tmem_wait_ld<16>(r[u & 1]);
        if (u < 15)
          tmem_ld_16x256_x4(tl + (uint32_t)(32 * ((u + 1) >> 1)) + ((uint32_t)(16 * ((u + 1) & 1)) << 16),
                            r[(u + 1) & 1]);
        const int c = u >> 2;
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            // row 32 warp + 16 (u % 2) + 8 h + g, 16-byte piece 4 (u / 2 % 2) + e
            const uint32_t* rr = r[u & 1] + 4 * e + 2 * h;
            sts32((hrow ^ (uint32_t)((4 * ((u >> 1) & 1) + e) << 4)) +
                      (uint32_t)(c * FT_ROWS * 128 + (16 * (u & 1) + 8 * h) * 128),
                  bias_relu_bf16(rr[0], rr[1], bias[4 * (u >> 1) + e]));
          }
        if ((u & 3) == 3) {
          fence_async();
          arrive(&b_h[c]);
        }
      }
    }
  } else {
    const int q = warp & 3, half = (warp - FT_G1) >> 2, g = lane >> 2, tq = lane & 3;
    const int xr = (tid - 32 * FT_G1) >> 1, xp = tid & 1;  // input row and part of this thread
    const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(MLP_H + 128 * half);
    float2 bias[16];    // of columns 128 half + 8 b + 2 tq, + 1
    uint32_t w3[8][2];  // the output layer's fragments of columns 128 half + 16 s
#pragma unroll
    for (int b = 0; b < 16; ++b)
      bias[b] = *reinterpret_cast<const float2*>(a.b2 + 128 * half + 8 * b + 2 * tq);
#pragma unroll
    for (int s = 0; s < 8; ++s) frag_b(a.W3, MLP_H, 0, 128 * half + 16 * s, w3[s]);
    const float b3a = a.b3[2 * tq], b3b = a.b3[2 * tq + 1];
    float xv[16];
    auto stage_x = [&]() {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int c = 2 * xp + i;
        sts128(base + FT_X + (uint32_t)(xr * 64 + ((c ^ ((xr >> 1) & 3)) << 4)),
               pack_bf16(xv[8 * i], xv[8 * i + 1]), pack_bf16(xv[8 * i + 2], xv[8 * i + 3]),
               pack_bf16(xv[8 * i + 4], xv[8 * i + 5]), pack_bf16(xv[8 * i + 6], xv[8 * i + 7]));
      }
      fence_async();
      arrive(&b_x);
    };
    ft_load_x(a, (int)blockIdx.x * FT_ROWS + xr, xp, xv);
    stage_x();
    if ((int)blockIdx.x + stride < n_tiles)
      ft_load_x(a, ((int)blockIdx.x + stride) * FT_ROWS + xr, xp, xv);
    uint32_t ph = 0;
    for (int t = blockIdx.x; t < n_tiles; t += stride, ph ^= 1u) {
      if (t + stride < n_tiles) {
        wait(&b_d1, ph, 22);  // layer 1 has read this tile's inputs
        stage_x();
        if (t + 2 * stride < n_tiles) ft_load_x(a, (t + 2 * stride) * FT_ROWS + xr, xp, xv);
      }
      wait(&b_d2, ph, 23);
      float o[2][4];
      uint32_t r[2][16];
      tmem_ld_16x256_x4(tl, r[0]);
#pragma unroll
      for (int u = 0; u < 8; ++u) {  // rows 16 (u / 4) .., columns 32 (u % 4) ..
        const int m = u >> 2;
        tmem_wait_ld<16>(r[u & 1]);
        if (u < 7)
          tmem_ld_16x256_x4(tl + (uint32_t)(32 * ((u + 1) & 3)) + ((uint32_t)(16 * ((u + 1) >> 2)) << 16),
                            r[(u + 1) & 1]);
        else
          arrive(&b_e2);
        if ((u & 3) == 0) o[m][0] = o[m][1] = o[m][2] = o[m][3] = 0.0f;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          uint32_t f[4];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const uint32_t* rr = r[u & 1] + 4 * (2 * s + e);
            const float2 b = bias[4 * (u & 3) + 2 * s + e];
            f[2 * e] = bias_relu_bf16(rr[0], rr[1], b);
            f[2 * e + 1] = bias_relu_bf16(rr[2], rr[3], b);
          }
          mma_bf16_16816(o[m], f, w3[2 * (u & 3) + s]);
        }
      }
      // each half finishes the 16-row block of its number: it hands the other
      // block's sums to its partner and takes the partner's (two buffers: a
      // warp writes tile t + 2's only after its partner has read tile t's)
      float* part = &s_part[ph][0][0];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float* give = half == 0 ? o[1] : o[0];
        *reinterpret_cast<float2*>(part + (32 * q + 16 * (half ^ 1) + 8 * e + g) * MLP_OUT + 2 * tq) =
            make_float2(give[2 * e], give[2 * e + 1]);
      }
      asm volatile("bar.sync %0, 64;" ::"r"(1 + q) : "memory");
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int rl = 32 * q + 16 * half + 8 * e + g;
        const float2 s = *reinterpret_cast<const float2*>(part + rl * MLP_OUT + 2 * tq);
        const float* own = half == 0 ? o[0] : o[1];
        float v0 = (b3a + own[2 * e]) + s.x, v1 = (b3b + own[2 * e + 1]) + s.y;
        if (tq < 2) {
          v0 = tanhf(v0);
          v1 = tanhf(v1);
        } else {
          v0 = fminf(fmaxf(v0, MLP_LOGSTD_MIN), MLP_LOGSTD_MAX);
          v1 = fminf(fmaxf(v1, MLP_LOGSTD_MIN), MLP_LOGSTD_MAX);
        }
        const int row = t * FT_ROWS + rl;
        if (row < a.M && *((volatile int*)&s_fail) == 0) {
          float* dst = a.out + (size_t)row * MLP_OUT + 2 * tq;
          if (a.vec) {
            *reinterpret_cast<float2*>(dst) = make_float2(v0, v1);
          } else {
            dst[0] = v0;
            dst[1] = v1;
          }
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == FT_G1 + FT_G2) {
    fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (tid == 0 && s_fail) atomicExch(a.err, 200 + s_fail);
}

}  // namespace tc
}  // namespace kp
