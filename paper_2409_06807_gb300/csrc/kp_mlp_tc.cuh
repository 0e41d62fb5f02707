// kp_mlp_tc.cuh -- the network's inference and training on the fifth-generation
// tensor cores: all layers of a 128-row tile in one kernel, forward and
// backward, weights and hidden activations on chip.
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

// 8 consecutive 32-bit columns of the calling thread's TMEM lane (waited for).
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
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
  int hold;                 // test hook: no product after the first ones is issued
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
// which fetched every weight fragment from L2 for each tile; 33 rows 8.2 to 9.8
// us a call over runs against 10.3 to 10.6.  A tile takes about 5,000 clocks where its products
// need 2,300: the chain accumulator -> epilogue 1 -> first chunk -> layer 2 is
// what is left, and layer 2 runs at two thirds of its rate beside the
// epilogues' shared-memory and tensor-memory traffic.  Arrangements measured
// slower on the same rows: one group of 8 or 16 warps for both epilogues (54
// us), layer 2 in two halves of 128 columns (its operands then take all of the
// shared-memory bandwidth, 54 us), row-per-thread loads with the biases in
// shared memory (51 us).
__global__ void __launch_bounds__(FT_THREADS, 1) kp_mlp_forward_tc_kernel(FtArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t b_w1, b_w2[4], b_x, b_d1, b_h[4], b_d2, b_e2, b_end;
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
    mbar_init(saddr(&b_end), 1);
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
  // left return at once), and the rows that are still to come are NaN: the
  // caller has no status to ask, and must not take what the output held before
  // for a result.
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
      if (a.hold) ok = wait(&b_d2, 0, 16);  // (nothing is committed to it)
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
        if (*((volatile int*)&s_fail) != 0) v0 = v1 = __int_as_float(0x7fffffff);
        if (row < a.M) {
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
    if (lane == 0 && s_fail) {
      // a wait gave up: products and the weights' copies may be in flight, and
      // they end before the block's memories go
      mma_commit(saddr(&b_end));
      mbar_wait(saddr(&b_end), 0, a.wait_ns);
      mbar_wait(saddr(&b_w1), 0, a.wait_ns);
      for (int c = 0; c < 4; ++c) mbar_wait(saddr(&b_w2[c]), 0, a.wait_ns);
    }
    __syncwarp();
    fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (tid == 0 && s_fail) atomicExch(a.err, 200 + s_fail);
}

// ---------------------------------------------------------------------------
// training: forward, backward and optimiser
// ---------------------------------------------------------------------------

// flat parameter vector (FP32), row-major: W1 b1 W2 b2 W3 b3
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + MLP_H * MLP_IN, OFF_W2 = OFF_B1 + MLP_H,
              OFF_B2 = OFF_W2 + MLP_H * MLP_H, OFF_W3 = OFF_B2 + MLP_H,
              OFF_B3 = OFF_W3 + MLP_OUT * MLP_H, N_PARAMS = OFF_B3 + MLP_OUT;

// A CTA's share of a mini-batch's gradient: groups of four parameters, then its
// share of the loss.  At most ST_MAX_SLOTS CTAs work on tiles.  The groups of
// dW1 and dW2 are in the order in which the warps hold them in tensor memory
// (a lane a row, a warp's 32 lanes' groups together), so that a warp writes 512
// contiguous bytes at a time: written in rows, where a warp's store touches 16
// to 32 lines, the two halves of dW2 took 15,000 of a step's 57,000 clocks.
constexpr int SLOT = N_PARAMS + 4, ST_MAX_SLOTS = 152;

// Group of dW1 rows 32 (4 tile + q) + lane, columns 4 j ..
__device__ __forceinline__ int slot_group_w1(int tile, int q, int j, int lane) {
  return ((tile * 4 + q) * 8 + j) * 32 + lane;
}

// Group of dW2 rows 128 tile + 32 (warp % 4) + lane, columns 64 (warp / 4) +
// 32 u + 4 j ..
__device__ __forceinline__ int slot_group_w2(int tile, int warp, int u, int j, int lane) {
  return OFF_W2 / 4 + (((tile * 16 + warp) * 2 + u) * 8 + j) * 32 + lane;
}

// First parameter of a slot's group.
__device__ __forceinline__ int slot_param(int gr) {
  if (gr < OFF_B1 / 4) return ((gr >> 8) * 32 + (gr & 31)) * MLP_IN + 4 * ((gr >> 5) & 7);
  if (gr >= OFF_W2 / 4 && gr < OFF_B2 / 4) {
    const int e = gr - OFF_W2 / 4, lane = e & 31, j = (e >> 5) & 7, u = (e >> 8) & 1,
              warp = (e >> 9) & 15, tile = e >> 13;
    return OFF_W2 + (128 * tile + 32 * (warp & 3) + lane) * MLP_H + 64 * (warp >> 2) + 32 * u + 4 * j;
  }
  return 4 * gr;
}

// Parameters i .. i + 3 (i a multiple of 4) rounded to BF16 into the copies
// the kernels read: the hidden layers' weights in tensor-core operand order
// (wt) and in the fragment order of the planner's loop kernel (wf); the output
// layer's row-major (w3) and in fragment order.
__device__ __forceinline__ void store_weights(int i, float4 p, __nv_bfloat16* w3, __nv_bfloat16* wf,
                                              __nv_bfloat16* wt) {
  const uint32_t lo = pack_bf16(p.x, p.y), hi = pack_bf16(p.z, p.w);
  auto put = [&](__nv_bfloat16* row, __nv_bfloat16* f0, __nv_bfloat16* f2) {
    *reinterpret_cast<uint2*>(row) = make_uint2(lo, hi);
    *reinterpret_cast<uint32_t*>(f0) = lo;
    *reinterpret_cast<uint32_t*>(f2) = hi;
  };
  if (i < OFF_B1) {
    const int n = i / MLP_IN, k = i % MLP_IN;
    put(wt + wt_index_w1(n, k), wf + frag_index_hidden(n, k, MLP_IN),
        wf + frag_index_hidden(n, k + 2, MLP_IN));
  } else if (i >= OFF_W2 && i < OFF_B2) {
    const int n = (i - OFF_W2) / MLP_H, k = (i - OFF_W2) % MLP_H;
    __nv_bfloat16* f = wf + MLP_H * MLP_IN;
    put(wt + wt_index_w2(n, k), f + frag_index_hidden(n, k, MLP_H), f + frag_index_hidden(n, k + 2, MLP_H));
  } else if (i >= OFF_W3 && i < OFF_B3) {
    const int n = (i - OFF_W3) / MLP_H, k = (i - OFF_W3) % MLP_H;
    __nv_bfloat16* f = wf + MLP_H * MLP_IN + MLP_H * MLP_H;
    put(w3 + (i - OFF_W3), f + frag_index_out(n, k), f + frag_index_out(n, k + 2));
  }
}

// Sum over the slots of a group, in slot order (read past L1: other SMs wrote
// them).
__device__ __forceinline__ float4 slot_sum(const float* slots, int n, int gr) {
  const float4* g = reinterpret_cast<const float4*>(slots) + gr;
  float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  for (int k0 = 0; k0 < n; k0 += 16) {  // sixteen loads in flight, the last ones too
    float4 v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k)
      v[k] = k0 + k < n ? __ldcg(g + (size_t)(k0 + k) * (SLOT / 4)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      s.x += v[k].x;
      s.y += v[k].y;
      s.z += v[k].z;
      s.w += v[k].w;
    }
  }
  return s;
}

struct AdamArgs {
  float *p, *m, *v;
  const float* slots;
  int n_slots;
  __nv_bfloat16 *w3, *wf, *wt;
  float lr;
};

// One Adam step (beta 0.9 / 0.999, eps 1e-8) on the parameters of a slot group;
// c1, c2 = 1 - beta^step.
__device__ __forceinline__ void adam_update(const AdamArgs& a, int gr, float c1, float c2) {
  const int i = slot_param(gr);
  const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
  float4 p = *reinterpret_cast<const float4*>(a.p + i), m = *reinterpret_cast<const float4*>(a.m + i),
         v = *reinterpret_cast<const float4*>(a.v + i);
  const float4 g = slot_sum(a.slots, a.n_slots, gr);
  auto one = [&](float& pi, float& mi, float& vi, float gi) {
    mi = beta1 * mi + (1.0f - beta1) * gi;
    vi = beta2 * vi + (1.0f - beta2) * gi * gi;
    pi = pi - a.lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  };
  one(p.x, m.x, v.x, g.x);
  one(p.y, m.y, v.y, g.y);
  one(p.z, m.z, v.z, g.z);
  one(p.w, m.w, v.w, g.w);
  *reinterpret_cast<float4*>(a.p + i) = p;
  *reinterpret_cast<float4*>(a.m + i) = m;
  *reinterpret_cast<float4*>(a.v + i) = v;
  store_weights(i, p, a.w3, a.wf, a.wt);
}

__device__ __forceinline__ void adam_corrections(int step, float* c1, float* c2) {
  *c1 = 1.0f - powf(0.9f, (float)step);
  *c2 = 1.0f - powf(0.999f, (float)step);
}

constexpr int ST_THREADS = 512;
// shared memory: h1 (first the inputs and W1), h2 then dh2 (first two chunks
// of W2), two chunks of W2 then dh1, the transposed inputs with a block of
// ones, the transposed output gradient, W3 twice, the output gradient split
// into three BF16 parts
constexpr uint32_t ST_H1 = 0, ST_G = 65536, ST_W = 131072, ST_XT = 196608, ST_DT = ST_XT + 2 * 6144,
                   ST_W3 = ST_DT + 2 * 2048, ST_DA = ST_W3 + 4 * 2048, ST_END = ST_DA + 8192;
constexpr int ST_SMEM = (int)ST_END + 1024;
constexpr uint32_t ST_X = ST_H1, ST_W1 = ST_H1 + 16384;  // before h1 is written
constexpr uint32_t ST_B1 = ST_DA, ST_B2 = ST_DA + 1024;   // before the split gradient is

struct StepArgs {
  const float *x, *t;      // [rows][32], [rows][4]
  const int32_t* perm;     // row behind each row of the batches (null: itself)
  int M;                   // rows of a mini-batch
  int64_t steps;           // mini-batches: rows s M .. of the order
  int epoch;               // 1: an Adam step after each (cooperative launch)
  int step0;               // Adam steps taken before
  AdamArgs adam;           // parameters, BF16 copies, the slots
  float* slots;            // each CTA's share of the gradient, written
  float* loss_sum;         // epoch: sum over its mini-batches, 0 at launch
  uint32_t* bar;           // epoch: grid barrier word, 0 at launch
  int* err;
  unsigned long long wait_ns;
  int hold;                // test hook: a wait for what is not yet asked for
};

// kind::f16 descriptor with the operands' majors (1: M or N contiguous).
__host__ __device__ constexpr uint32_t idesc_majors(int M, int N, int a_mn, int b_mn) {
  return idesc_bf16_f32(M, N) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16);
}

// Descriptor of a 128-byte-swizzled operand whose M or N index is contiguous:
// 64 of them in a 128-byte row, rows along K; 8-row groups 1024 bytes apart,
// the next 64 of M or N 'next' bytes on.
__device__ __forceinline__ uint64_t sdesc_mn128(uint32_t addr, uint32_t next) {
  uint64_t d = (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)(next >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

__device__ __forceinline__ void sts16(uint32_t addr, __nv_bfloat16 v) {
  asm volatile("st.shared.b16 [%0], %1;" ::"r"(addr), "h"(*reinterpret_cast<const uint16_t*>(&v))
               : "memory");
}

// 16 bytes of a slot: written by the CTA's first tile of a mini-batch, added to
// by its later ones.
__device__ __forceinline__ void slot_put4(float* p, const uint32_t* r, bool add) {
  float4 v = make_float4(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]),
                         __uint_as_float(r[3]));
  if (add) {
    const float4 o = *reinterpret_cast<const float4*>(p);
    v = make_float4(o.x + v.x, o.y + v.y, o.z + v.z, o.w + v.w);
  }
  *reinterpret_cast<float4*>(p) = v;
}

__device__ __forceinline__ void slot_put(float* p, float v, bool add) { *p = add ? *p + v : v; }

// The two BF16 halves of v kept where those of h are not zero (h is the
// output of a ReLU: positive or zero).
__device__ __forceinline__ uint32_t keep_active(uint32_t v, uint32_t h) {
  const uint32_t lo = (h & 0x00007fffu) ? 0x0000ffffu : 0u, hi = (h & 0x7fff0000u) ? 0xffff0000u : 0u;
  return v & (lo | hi);
}

// Waits (bounded, one thread) until all CTAs of the launch have arrived 'n'
// times; false when the wait or another CTA gave up.  What the CTAs wrote
// before their arrivals is visible to generic and bulk-copy reads after it.
__device__ __forceinline__ bool grid_arrive_wait(uint32_t* bar, uint32_t n, const int* err,
                                                 uint64_t limit_ns) {
  __threadfence();
  atomicAdd(bar, 1u);
  uint64_t t0 = 0;
  for (uint32_t i = 1;; ++i) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
    if ((int32_t)(v - n) >= 0) break;
    if ((i & 63u) == 0) {
      if (*((const volatile int*)err) != 0) return false;
      if (t0 == 0) t0 = now_ns();
      if (now_ns() - t0 > limit_ns) return false;
    }
  }
  asm volatile("fence.proxy.async;" ::: "memory");
  return true;
}

// Forward, loss and backward of 128-row tiles, every product on the tensor
// cores, nothing of a tile in global memory but its inputs and its gradient
// contributions; in an epoch (a cooperative launch of at most one CTA per SM)
// every mini-batch ends with a grid barrier, each CTA's share of the Adam step
// and another barrier, so the whole epoch is one launch.  The phases of a tile
// (X the inputs, D the gradient of the eight outputs; thread = row 32 (w % 4) +
// lane and columns 64 (w / 4) ..):
//   h1 = relu(X W1' + b1), h2 = relu(h1 W2' + b2), raw = h2 W3' + b3; the
//   loss and D (FP32);
//   dW3 += D' h2;  dh2 = (D W3) where h2 > 0, D entering as three BF16 parts
//   whose sum is the FP32 value (their products with W3 are exact);
//   dh1 = (dh2 W2) where h1 > 0;  dW2 += dh2' h1;  dW1 += dh1' X; db2 and db1
//   as products with a block of ones.
// The transposed operands are the same shared-memory tiles read with their
// other index contiguous, so nothing is transposed.  W2 is brought in twice,
// half of it only once (its first half survives the forward pass).  Rows past
// M have inputs 0, activations 0 and D 0.
//
// Every CTA writes its share of the gradient to a slot of its own, and the
// optimiser adds the slots up in slot order: additions in L2 by 32 CTAs took
// 17,000 of a step's 57,000 clocks (L2 added 120 values a clock), and the
// result now has the same bits every time.
//
// A mini-batch of 4096 is 32 tiles, so a step is one tile's chain (21,000
// clocks: nine products, forward and backward, in six rounds, each round behind
// the epilogue of the one before), 9,000 for the slot's 305 KB, 5,000 for the
// optimiser's share and 6,000 in the two barriers: 25 us of the launch (GB300).
// Epochs of 16 steps of 4,096 rows, whole calls with the parameter read-back
// (50 us): 1,333 us as 15 launches a step (row-major and transposed activations
// in global memory, split-K products), 561 us as two launches a step with this
// pass, 460 us now.
__global__ void __launch_bounds__(ST_THREADS, 1) kp_mlp_train_kernel(StepArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t b_w1, b_w2[4], b_mma, b_c, b_t0, b_r, b_end;
  __shared__ float s_red[4][MLP_NQ][3];  // sums over a warp's rows: loss, both gradients
  __shared__ float s_b3[MLP_OUT];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_fail;
  const uint32_t base = (saddr(smem_raw) + 1023u) & ~1023u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q = warp & 3, qt = warp >> 2;
  if (tid == 0) {
    mbar_init(saddr(&b_w1), 1);
    for (int c = 0; c < 4; ++c) mbar_init(saddr(&b_w2[c]), 1);
    mbar_init(saddr(&b_mma), 1);
    mbar_init(saddr(&b_c), 1);
    mbar_init(saddr(&b_r), 1);
    mbar_init(saddr(&b_t0), 1);
    mbar_init(saddr(&b_end), 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    tmem_alloc(saddr(&tmem_slot), 512);
  }
  // the parts of the operands that stay: ones (rows 32..47 of the transposed
  // inputs), zeros (rows 8..15 of the transposed output gradient)
  if (tid < 256) {
    const uint32_t one2 = 0x3F803F80u;
    sts128(base + ST_XT + (uint32_t)((tid >> 7) * 6144 + 4096 + (tid & 127) * 16), one2, one2, one2, one2);
  } else if (tid < 384) {
    const int e = tid - 256;
    sts128(base + ST_DT + (uint32_t)((e >> 6) * 2048 + 1024 + (e & 63) * 16), 0, 0, 0, 0);
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16);
  const int r = 32 * q + lane;
  // this row's piece 0 of a 128-byte-row tile (piece c at c ^ (r & 7))
  const uint32_t hoff = (uint32_t)(r * 128 + ((r & 7) << 4) + qt * 16384);
  const uint32_t A0 = tmem, B0 = tmem + 256;  // the two halves of tensor memory
  const float* par = a.adam.p;
  float* g = a.slots + (size_t)blockIdx.x * SLOT;
  uint32_t ph = 0, ph_t = 0;  // parities: of b_mma, and of the once-a-tile barriers
  auto wait = [&](uint64_t* bar, uint32_t parity, int site) {
    mbar_wait_or(saddr(bar), parity, a.wait_ns, &s_fail, site);
  };
  auto failed1 = [&]() { return *((volatile int*)&s_fail) != 0; };
  auto failed = [&]() { return __any_sync(0xffffffffu, failed1()) != 0; };  // the warp agrees
  auto wait_mma = [&](int site) {  // all threads: the products committed last are there
    __syncwarp();
    wait(&b_mma, ph, site);
    ph ^= 1u;
    __syncwarp();
    fence_after();
  };
  auto publish = [&]() {  // shared-memory operands written, accumulators read
    fence_async();
    fence_before();
    __syncthreads();
    fence_after();
  };
  // bias, ReLU, BF16 of this thread's 64 columns of an accumulator into a tile
  auto activate = [&](uint32_t acc, uint32_t tile, uint32_t bias, bool live) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      uint32_t v[32];
      const int c0 = 64 * qt + 32 * u;
      tmem_ld32(acc + (uint32_t)c0, v);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint4 ba = lds128(base + bias + (uint32_t)(4 * (c0 + 8 * j)));
        const uint4 bb = lds128(base + bias + (uint32_t)(4 * (c0 + 8 * j + 4)));
        auto two = [](uint32_t x, uint32_t y) {
          return make_float2(__uint_as_float(x), __uint_as_float(y));
        };
        const uint32_t* vv = v + 8 * j;
        const uint32_t w0 = bias_relu_bf16(vv[0], vv[1], two(ba.x, ba.y)),
                       w1 = bias_relu_bf16(vv[2], vv[3], two(ba.z, ba.w)),
                       w2 = bias_relu_bf16(vv[4], vv[5], two(bb.x, bb.y)),
                       w3 = bias_relu_bf16(vv[6], vv[7], two(bb.z, bb.w));
        sts128(base + tile + (hoff ^ (uint32_t)((4 * u + j) << 4)), live ? w0 : 0u, live ? w1 : 0u,
               live ? w2 : 0u, live ? w3 : 0u);
      }
    }
  };
  // BF16 of this thread's 64 columns of an accumulator where the activations
  // in tile 'act' are not zero, into 'tile' (which may be 'act')
  auto mask = [&](uint32_t acc, uint32_t act, uint32_t tile) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      uint32_t v[32];
      tmem_ld32(acc + (uint32_t)(64 * qt + 32 * u), v);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t off = hoff ^ (uint32_t)((4 * u + j) << 4);
        const uint4 h = lds128(base + act + off);
        const float* f = reinterpret_cast<const float*>(v + 8 * j);
        sts128(base + tile + off, keep_active(pack_bf16(f[0], f[1]), h.x),
               keep_active(pack_bf16(f[2], f[3]), h.y), keep_active(pack_bf16(f[4], f[5]), h.z),
               keep_active(pack_bf16(f[6], f[7]), h.w));
      }
    }
  };
  // half 'tile' of dW2 (128 rows) from an accumulator into the slot
  auto put_dw2 = [&](uint32_t acc, int tile, bool add) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      uint32_t v[32];
      tmem_ld32(acc + (uint32_t)(64 * qt + 32 * u), v);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        slot_put4(g + 4 * slot_group_w2(tile, warp, u, j, lane), v + 4 * j, add);
    }
  };
  constexpr uint32_t ID_FWD = idesc_majors(128, 256, 0, 0), ID_RAW = idesc_majors(128, 16, 0, 0),
                     ID_DW3 = idesc_majors(128, 16, 1, 0), ID_DH2 = idesc_majors(128, 256, 0, 1),
                     ID_DH1 = idesc_majors(128, 128, 0, 1), ID_DW2 = idesc_majors(128, 256, 1, 1),
                     ID_DW1 = idesc_majors(128, 48, 1, 0);

  const int n_tiles = (a.M + 127) / 128;
  uint32_t arrivals = 0;
  bool in_tile = false;  // a wait of the last tile gave up
  for (int64_t s = 0; s < a.steps; ++s) {
    for (int tile = blockIdx.x; tile < n_tiles; tile += (int)gridDim.x, ph_t ^= 1u) {
      const int row0 = tile * 128;
      const bool live = row0 + r < a.M, add = tile != (int)blockIdx.x;
      auto source_row = [&](int row) {  // row of x and t behind row 'row' of the batch
        const int64_t i = s * a.M + row;
        return a.perm ? (size_t)a.perm[i] : (size_t)i;
      };
      if (tid == 0) {
        // (the last tile's reads of these buffers are over; its generic
        // writes to them come before the copies)
        fence_async();
        mbar_expect_tx(saddr(&b_w1), MLP_H * 64);
        bulk_load(base + ST_W1, a.adam.wt + WT_W1, MLP_H * 64, saddr(&b_w1));
        for (int c = 0; c < 4; ++c) {
          mbar_expect_tx(saddr(&b_w2[c]), MLP_H * 128);
          bulk_load(base + (c < 2 ? ST_W + c * 32768 : ST_G + (c - 2) * 32768),
                    a.adam.wt + c * WT_CHUNK, MLP_H * 128, saddr(&b_w2[c]));
        }
      }
      {
        // inputs: thread = row tid / 4 and 8 columns
        const int xr = tid >> 2, part = tid & 3;
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 0.0f;
        if (row0 + xr < a.M) {
          const float* src = a.x + source_row(row0 + xr) * MLP_IN + 8 * part;
          if (((uintptr_t)src & 15u) == 0) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const float4 f = __ldg(reinterpret_cast<const float4*>(src) + i);
              v[4 * i] = f.x; v[4 * i + 1] = f.y; v[4 * i + 2] = f.z; v[4 * i + 3] = f.w;
            }
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __ldg(src + i);
          }
        }
        sts128(base + ST_X + (uint32_t)(xr * 64 + ((part ^ ((xr >> 1) & 3)) << 4)), pack_bf16(v[0], v[1]),
               pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
#pragma unroll
        for (int i = 0; i < 8; ++i)
          sts16(base + ST_XT + (uint32_t)((xr >> 6) * 6144 + (8 * part + i) * 128 +
                                          ((((xr & 63) >> 3) ^ i) << 4) + (xr & 7) * 2),
                __float2bfloat16_rn(v[i]));
      }
      {
        // W3 twice, the biases (read past L1: the last step's optimiser ran
        // on other SMs too)
        const int c = tid >> 7, copy = (tid >> 6) & 1, n = (tid >> 3) & 7, j = tid & 7;
        const uint4 w = __ldcg(reinterpret_cast<const uint4*>(a.adam.w3 + n * MLP_H + 64 * c + 8 * j));
        sts128(base + ST_W3 + (uint32_t)(c * 2048 + copy * 1024 + n * 128 + ((j ^ n) << 4)), w.x, w.y, w.z,
               w.w);
        const float b = __ldcg(par + (tid < MLP_H ? OFF_B1 + tid : OFF_B2 + tid - MLP_H));
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(base + ST_B1 + 4 * tid), "f"(b) : "memory");
        if (tid < MLP_OUT) s_b3[tid] = __ldcg(par + OFF_B3 + tid);
      }
      // target qt of row r
      const float tv = live ? __ldg(a.t + source_row(row0 + r) * MLP_NQ + qt) : 0.0f;
      publish();

      // ---- forward
      if (tid == 0) {
        if (a.hold) wait(&b_r, ph_t, 41);  // (W2's second copy starts below)
        wait(&b_w1, ph_t, 30);
        fence_after();
#pragma unroll
        for (int k = 0; k < 2; ++k)
          mma_bf16(A0, sdesc_sw64(base + ST_X + 32 * k), sdesc_sw64(base + ST_W1 + 32 * k), ID_FWD,
                   k != 0 ? 1u : 0u);
        mma_commit(saddr(&b_mma));
      }
      wait_mma(31);
      activate(tl, ST_H1, ST_B1, live);
      publish();
      if (tid == 0) {
        for (int c = 0; c < 4; ++c) {
          wait(&b_w2[c], ph_t, 32);
          const uint32_t w = base + (c < 2 ? ST_W + c * 32768 : ST_G + (c - 2) * 32768);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_bf16(B0, sdesc_sw128(base + ST_H1 + c * 16384 + 32 * k), sdesc_sw128(w + 32 * k), ID_FWD,
                     (c | k) != 0 ? 1u : 0u);
        }
        mma_commit(saddr(&b_mma));
      }
      wait_mma(33);
      activate(tl + 256, ST_G, ST_B2, live);
      publish();
      if (tid == 0) {
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_bf16(A0, sdesc_sw128(base + ST_G + c * 16384 + 32 * k),
                     sdesc_sw128(base + ST_W3 + c * 2048 + 32 * k), ID_RAW, (c | k) != 0 ? 1u : 0u);
        mma_commit(saddr(&b_mma));
      }
      wait_mma(34);

      // ---- loss and the outputs' gradient: a thread a row and output pair
      // (mean qt, log standard deviation qt)
      {
        uint32_t raw[8];
        tmem_ld8(tl, raw);
        const float inv_m = 1.0f / (float)a.M;
        const float rm = __uint_as_float(qt == 0 ? raw[0] : qt == 1 ? raw[1] : qt == 2 ? raw[2] : raw[3]);
        const float rs = __uint_as_float(qt == 0 ? raw[4] : qt == 1 ? raw[5] : qt == 2 ? raw[6] : raw[7]);
        const float mu = tanhf(rm + s_b3[qt]);
        const float lr = rs + s_b3[MLP_NQ + qt];
        const bool clamped = lr < MLP_LOGSTD_MIN || lr > MLP_LOGSTD_MAX;
        const float ls = fminf(fmaxf(lr, MLP_LOGSTD_MIN), MLP_LOGSTD_MAX);
        const float is = expf(-ls);
        const float z = (tv - mu) * is;
        float sum[3] = {live ? ls + 0.5f * z * z : 0.0f,
                        live ? -z * is * (1.0f - mu * mu) * inv_m : 0.0f,
                        live && !clamped ? (1.0f - z * z) * inv_m : 0.0f};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int n = qt + MLP_NQ * i;
          const float d = sum[1 + i];
          // three BF16 parts of the value: rounding, then what is left, twice
          // (nothing of an infinite one: infinity minus infinity would be NaN;
          // what would round to infinity, only for the first part's weight, is
          // cut to BF16's largest number)
          const __nv_bfloat16 pd = __float2bfloat16_rn(d);
          const bool over = __hisinf(pd) != 0;
          const __nv_bfloat16 p0 = over ? __float2bfloat16_rz(d) : pd;
          const float r1 = over && isinf(d) ? 0.0f : d - __bfloat162float(p0);
          const __nv_bfloat16 p1 = __float2bfloat16_rn(r1);
          const __nv_bfloat16 p2 = __float2bfloat16_rn(r1 - __bfloat162float(p1));
          sts16(base + ST_DT + (uint32_t)((r >> 6) * 2048 + n * 128 + ((((r & 63) >> 3) ^ n) << 4) +
                                          (r & 7) * 2),
                pd);
          const uint32_t da = base + ST_DA + (uint32_t)(r * 64 + 2 * n), sw = (uint32_t)((r >> 1) & 3);
          sts16(da + ((0u ^ sw) << 4), p0);
          sts16(da + ((1u ^ sw) << 4), p1);
          sts16(da + ((2u ^ sw) << 4), p2);
          sts16(da + ((3u ^ sw) << 4), __float2bfloat16_rn(0.0f));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int i = 0; i < 3; ++i) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
        if (lane == 0)
#pragma unroll
          for (int i = 0; i < 3; ++i) s_red[q][qt][i] = sum[i];
      }
      publish();

      // ---- backward
      if (tid == 0) {
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int k = 0; k < 8; ++k)
            mma_bf16(A0 + 16 + 16 * m, sdesc_mn128(base + ST_G + m * 32768 + k * 2048, 16384),
                     sdesc_sw128(base + ST_DT + (k >> 2) * 2048 + (k & 3) * 32), ID_DW3, k != 0 ? 1u : 0u);
#pragma unroll
        for (int k = 0; k < 2; ++k)  // both K groups of W3's tile hold W3: parts 0 and 1, then 2 and zeros
          mma_bf16(B0, sdesc_sw64(base + ST_DA + 32 * k), sdesc_mn128(base + ST_W3, 2048), ID_DH2,
                   k != 0 ? 1u : 0u);
        mma_commit(saddr(&b_mma));
      }
      if (tid >= 64 && tid < 64 + MLP_OUT + 1) {  // db3 and the loss from the warps' sums
        const int n = tid - 64;
        float sum = 0.0f;
        for (int w = 0; w < 4; ++w) {
          if (n < MLP_OUT) {
            sum += s_red[w][n & 3][1 + (n >> 2)];
          } else {
            for (int i = 0; i < MLP_NQ; ++i) sum += s_red[w][i][0];
          }
        }
        slot_put(g + (n < MLP_OUT ? OFF_B3 + n : N_PARAMS), n < MLP_OUT ? sum : sum / (float)a.M, add);
      }
      wait_mma(35);
      mask(tl + 256, ST_G, ST_G);
      if (qt < 2) {
        uint32_t v[8];
        tmem_ld8(tl + 16 + 16 * qt, v);
#pragma unroll
        for (int n = 0; n < MLP_OUT; ++n)
          slot_put(g + OFF_W3 + n * MLP_H + 128 * qt + r, __uint_as_float(v[n]), add);
      }
      publish();
      if (tid == 0) {
        auto dh1_half = [&](int c) {  // 128 columns: two chunks of W2
#pragma unroll
          for (int k = 0; k < 16; ++k)
            mma_bf16(A0 + 128 * c, sdesc_sw128(base + ST_G + (k >> 2) * 16384 + (k & 3) * 32),
                     sdesc_mn128(base + ST_W + k * 2048, 32768), ID_DH1, k != 0 ? 1u : 0u);
        };
        dh1_half(0);
        mma_commit(saddr(&b_c));
#pragma unroll
        for (int k = 0; k < 8; ++k)
          mma_bf16(B0, sdesc_mn128(base + ST_G + k * 2048, 16384),
                   sdesc_mn128(base + ST_H1 + k * 2048, 16384), ID_DW2, k != 0 ? 1u : 0u);
        wait(&b_c, ph_t, 36);
        mbar_expect_tx(saddr(&b_r), 2 * MLP_H * 128);
        for (int c = 0; c < 2; ++c)
          bulk_load(base + ST_W + c * 32768, a.adam.wt + (2 + c) * WT_CHUNK, MLP_H * 128, saddr(&b_r));
        wait(&b_r, ph_t, 37);
        dh1_half(1);
        mma_commit(saddr(&b_mma));
      }
      wait_mma(39);
      mask(tl, ST_H1, ST_W);
      publish();
      if (tid == 0) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
          mma_bf16(A0, sdesc_mn128(base + ST_G + 32768 + k * 2048, 16384),
                   sdesc_mn128(base + ST_H1 + k * 2048, 16384), ID_DW2, k != 0 ? 1u : 0u);
        mma_commit(saddr(&b_t0));
      }
      __syncwarp();
      put_dw2(tl + 256, 0, add);  // beside the second half's products
      publish();
      if (tid == 0) {
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint32_t xt = base + ST_XT + (k >> 2) * 6144 + (k & 3) * 32;
            mma_bf16(B0 + 48 * m, sdesc_mn128(base + ST_W + m * 32768 + k * 2048, 16384), sdesc_sw128(xt),
                     ID_DW1, k != 0 ? 1u : 0u);
            mma_bf16(B0 + 96 + 16 * m, sdesc_mn128(base + ST_G + m * 32768 + k * 2048, 16384),
                     sdesc_sw128(xt + 4096), ID_DW3, k != 0 ? 1u : 0u);
          }
        mma_commit(saddr(&b_mma));
      }
      __syncwarp();
      wait(&b_t0, ph_t, 38);
      __syncwarp();
      fence_after();
      put_dw2(tl, 1, add);
      wait_mma(40);
      {
        const int o = 128 * (qt & 1) + r;
        uint32_t v[8];
        if (qt < 2) {
#pragma unroll
          for (int j = 0; j < 8; j += 2) {
            tmem_ld8(tl + 256 + 48 * qt + (uint32_t)(4 * j), v);
            slot_put4(g + 4 * slot_group_w1(qt, q, j, lane), v, add);
            slot_put4(g + 4 * slot_group_w1(qt, q, j + 1, lane), v + 4, add);
          }
          tmem_ld8(tl + 256 + 48 * qt + 32, v);
          slot_put(g + OFF_B1 + o, __uint_as_float(v[0]), add);
        } else {
          tmem_ld8(tl + 256 + 96 + 16 * (qt - 2), v);
          slot_put(g + OFF_B2 + o, __uint_as_float(v[0]), add);
        }
      }
      fence_before();
      __syncthreads();
      fence_after();
      // a wait gave up: no further tile, and the barriers stay at this tile's
      // phases (every thread sees the flag: the next one to set it would wait
      // behind the next tile's first __syncthreads)
      in_tile = failed();
      if (in_tile) break;
    }
    if (!a.epoch) break;
    // ---- optimiser: every tile's gradient is in; this CTA's share of the
    // parameters; then the next mini-batch may read them
    __syncthreads();
    arrivals += gridDim.x;
    if (tid == 0 && (failed1() || !grid_arrive_wait(a.bar, arrivals, a.err, a.wait_ns))) {
      if (!failed1()) s_fail = 50;
      atomicExch(a.err, 100 + s_fail);  // the other CTAs' barrier waits see it
    }
    __syncthreads();
    if (failed()) break;
    float c1, c2;
    adam_corrections((int)(a.step0 + s + 1), &c1, &c2);
    // groups of four parameters, the loss after them; a warp's groups are
    // consecutive, the warps of all CTAs take turns
    for (int i = ((int)blockIdx.x + (int)gridDim.x * warp) * 32 + lane; i <= N_PARAMS / 4;
         i += (int)gridDim.x * ST_THREADS) {
      if (i < N_PARAMS / 4)
        adam_update(a.adam, i, c1, c2);
      else
        *a.loss_sum += slot_sum(a.adam.slots, a.adam.n_slots, i).x;
    }
    asm volatile("fence.proxy.async;" ::: "memory");  // the BF16 copies are read by bulk copies
    __syncthreads();
    arrivals += gridDim.x;
    if (tid == 0 && !grid_arrive_wait(a.bar, arrivals, a.err, a.wait_ns)) {
      s_fail = 51;
      atomicExch(a.err, 100 + s_fail);
    }
    __syncthreads();
    if (failed()) break;
  }
  fence_before();
  __syncthreads();
  if (warp == 0) {
    if (lane == 0 && s_fail) {
      if (in_tile) {
        // the tile's products and copies may be in flight, and they end before
        // the block's memories go (a block whose grid barrier gave up, or that
        // had no tile, has none)
        mma_commit(saddr(&b_end));
        mbar_wait(saddr(&b_end), 0, a.wait_ns);
        mbar_wait(saddr(&b_w1), ph_t, a.wait_ns);
        for (int c = 0; c < 4; ++c) mbar_wait(saddr(&b_w2[c]), ph_t, a.wait_ns);
        mbar_wait(saddr(&b_r), ph_t, a.wait_ns);
      }
      atomicExch(a.err, 100 + s_fail);
    }
    __syncwarp();
    fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace tc
}  // namespace kp
