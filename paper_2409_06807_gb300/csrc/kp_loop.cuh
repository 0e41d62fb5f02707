// kp_loop.cuh -- the Kino-PAX loop as one persistent cooperative kernel, plus
// the small reset / import / trajectory kernels.  Instantiated once per
// system by kp_sys_*.cu.
//
// One pass of the loop body (Algorithm 1) runs as four grid phases separated
// by bounded grid barriers, with no host involvement:
//   E  Propagate (Algorithm 2): lanes carry one sample (V_E position, j)
//      each and are refilled from a grid-wide key counter; draw u and k,
//      integrate k steps in FP32 registers, check each step against the
//      state box and the obstacle boxes staged in shared memory, bin the
//      end (or first invalid) state, count n_valid / n_invalid, claim newly
//      reached sub-regions (smallest sample key wins), keep the end state
//      of a sample that may still be accepted.
//   A  accept decisions (representative or P_accept draw), accepted keys
//      compacted per warp in key order; before it, on the warps with a region
//      chunk (a block's first, which takes no keys):
//   S  Score per region (Eq. 3-4, FP64, rounded exactly as written) and
//      the pairwise partial sum of each aligned region chunk (Eq. 5's sum).
//   N  a warp of each block takes the sum of Eq. 5 from the partial sums while
//      the block appends its own accepted samples (Algorithm 4, to T and V_E)
//      at their key-order node ids, from the kept end states, with the goal
//      test; then one selection draw per old node against P_accept of its
//      region, from the region's score (Algorithm 4, V_E <-> V_O), per-block
//      V_E counts, and on the warps with a region chunk, T: the integer
//      accept threshold per region, for the next pass.
//   L  V_E list in ascending node id, lambda for the next pass (Eq. 6),
//      stop decision.
// With a network attached (learned proposal) a phase F before E evaluates
// it on every V_E node.
#pragma once

#include <cstddef>
#include <cstdint>

#include "kp_device.cuh"
#include "kp_mlp.cuh"

#ifndef KP_MIN_BLOCKS
#define KP_MIN_BLOCKS 1
#endif

namespace kp {

// Sets a kernel's limit of dynamic shared memory to what the device has beside
// the kernel's static shared memory, whatever this context or server needs of
// it: the limit is one for all of them, and the one configured last must not
// lower it below what another one's launch takes.
inline cudaError_t raise_shared_limit(const void* kernel, size_t smem) {
  constexpr int kStaticShared = 1280;  // LoopShared and the barrier's words fit it
  int dev = 0, most = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  most -= kStaticShared;
  if (smem > (size_t)most) most = (int)smem;  // refused by the next call if it is too much
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

// (KP_BLOCK, the most threads of a block, is set by the including file)
constexpr int KP_WARPS = KP_BLOCK / 32;
static_assert(KP_WARPS <= 32 && KP_BLOCK % KP_MLP_GROUP == 0, "warps fit a lane each, groups are whole");

struct LoopShared {
  union {
    // the expand phase's five counters, a value a warp
    unsigned long long cnt[5][KP_WARPS];
    struct {
      // a value a warp: the counts a block prefix adds up, the tile counts of
      // the V_E list (two tiles in turn)
      uint32_t pre[KP_WARPS], tot[KP_WARPS];
      uint32_t tile[2][KP_WARPS];
      // accepted samples of this block, from the accept phase to the node-set
      // phase: warp w compacted acc_n[w] keys at acc_key[acc_a[w]...], which
      // are the block's accepted samples acc_off[w] .. acc_off[w] + acc_n[w] - 1
      int acc_a[KP_WARPS], acc_n[KP_WARPS], acc_off[KP_WARPS];
      int acc_tot;
    };
  };
  uint64_t mbar;
  int flag;
  int bcast[2];
  ScoreSum score;  // of the pass
  int goal, err;         // the pass's goal node and error word, read in phase L
  int32_t phase_ns[12];  // per-pass phase timers (block 0, thread 0)
};
static_assert(sizeof(LoopShared) <= 1200, "see raise_shared_limit");

// Stage the obstacle blob (boxes and broad-phase grid) into shared memory
// with bulk asynchronous copies (TMA engine) completing on one mbarrier.
// Returns false on a wait timeout.
__device__ __forceinline__ bool stage_boxes(const KParams& P, float4* sbox, LoopShared& sh) {
  const uint32_t bytes = (uint32_t)P.blob_bytes;  // multiple of 16
  if (bytes == 0) return true;
  const uint32_t mb = (uint32_t)__cvta_generic_to_shared(&sh.mbar);
  const uint32_t dst0 = (uint32_t)__cvta_generic_to_shared(sbox);
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb) : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes)
                 : "memory");
    const uint32_t piece = 16384u;  // several copies of <= 16 KB each
    for (uint32_t off = 0; off < bytes; off += piece) {
      const uint32_t n = bytes - off < piece ? bytes - off : piece;  // multiple of 16
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
          "[%3];" ::"r"(dst0 + off),
          "l"(reinterpret_cast<const char*>(P.boxes) + off), "r"(n), "r"(mb)
          : "memory");
    }
    // bounded wait for phase 0 of the mbarrier
    int ok = 0;
    const uint64_t t0 = global_ns();
    for (uint32_t spin = 0;; ++spin) {
      uint32_t done;
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n"
          " selp.u32 %0, 1, 0, p;\n}"
          : "=r"(done)
          : "r"(mb)
          : "memory");
      if (done) { ok = 1; break; }
      if (global_ns() - t0 > P.wait_ns) break;
    }
    if (!ok) {
      raise_error(P.ctl, KP_DEV_ERR_TIMEOUT, 1);
      // wait once more, again bounded, for the copies still in flight
      const uint64_t t1 = global_ns();
      for (;;) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n"
            " selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(mb)
            : "memory");
        if (done || global_ns() - t1 > P.wait_ns) break;
      }
    }
    // invalidate the object so that a later staging (the server stages one
    // blob per query) initialises a fresh mbarrier
    if (ok) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(mb) : "memory");
    sh.flag = ok;
  }
  __syncthreads();
  return sh.flag != 0;
}

__device__ __forceinline__ int eq6_lambda(int t_e, int n_tree, int n_ve, int lambda_max) {
  if (n_ve <= 0) return lambda_max;
  int room = t_e - n_tree;
  if (room < 0) room = 0;
  const int lam = room / n_ve;
  return lam < lambda_max ? lam : lambda_max;
}

// Node chunk [v0, v1) of this block over n nodes.
__device__ __forceinline__ void chunk_of(const Team& T, int n, int* c0, int* c1) {
  const int per = (n + T.nb - 1) / T.nb;
  const long long a = (long long)T.b * per;
  *c0 = (int)(a < n ? a : n);
  *c1 = (int)(a + per < n ? a + per : n);
}

// Sum of one value per warp of the block, by every warp (a lane a value).
__device__ __forceinline__ uint32_t warp_total(const uint32_t* v) {
  const uint32_t lane = threadIdx.x & 31u;
  return __reduce_add_sync(0xffffffffu, lane < (blockDim.x >> 5) ? v[lane] : 0u);
}

// The same over the warps before this one.
__device__ __forceinline__ uint32_t warp_before(const uint32_t* v) {
  const uint32_t lane = threadIdx.x & 31u;
  return __reduce_add_sync(0xffffffffu, lane < (threadIdx.x >> 5) ? v[lane] : 0u);
}

// Sum of blk[0..nb) and of blk[0..b) (counts of at most 2^28 in all): a
// reduction per warp, one block barrier, then every thread adds the warps'
// sums.  The shared values are free again after the block's next barrier.
// 'publish' runs before the barrier: what it writes is read after it.
struct Nothing {
  __device__ __forceinline__ void operator()() const {}
};

template <class F = Nothing>
__device__ __forceinline__ void block_prefix(const Team& T, const uint32_t* blk, LoopShared& sh,
                                             uint32_t* before, uint32_t* total, F publish = F()) {
  uint32_t pre = 0, tot = 0;
  for (int i = threadIdx.x; i < T.nb; i += blockDim.x) {
    const uint32_t c = __ldcg(blk + i);
    tot += c;
    if (i < T.b) pre += c;
  }
  pre = __reduce_add_sync(0xffffffffu, pre);
  tot = __reduce_add_sync(0xffffffffu, tot);
  if ((threadIdx.x & 31u) == 0) {
    sh.pre[threadIdx.x >> 5] = pre;
    sh.tot[threadIdx.x >> 5] = tot;
  }
  publish();
  __syncthreads();
  *before = warp_total(sh.pre);
  *total = warp_total(sh.tot);
}

// Nodes of a block's chunk are visited in tiles of blockDim.x: node v0 +
// tile * blockDim.x + threadIdx.x, so that a warp's loads and stores of the
// per-node arrays are coalesced.

// Block sum of one count per thread (at most 2^31 in all), for thread 0.
__device__ __forceinline__ uint32_t block_sum(uint32_t c, LoopShared& sh) {
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31u) == 0) sh.pre[threadIdx.x >> 5] = c;
  __syncthreads();
  return warp_total(sh.pre);
}

// Phase N': count V_E members of this block's node chunk (no draws) and
// publish the count.
__device__ __forceinline__ void count_ve(const KParams& P, const Team& T, int n, LoopShared& sh) {
  int v0, v1;
  chunk_of(T, n, &v0, &v1);
  int c = 0;
  for (int v = v0 + (int)threadIdx.x; v < v1; v += (int)blockDim.x)
    c += P.in_ve[KP_IDX(P, v, P.t_e, 1)] ? 1 : 0;
  const uint32_t tot = block_sum((uint32_t)c, sh);
  if (threadIdx.x == 0) P.blk_b[KP_IDX(P, T.b, KP_MAX_GRID, 2)] = tot;
}

// Phase L: write the V_E list (ascending node id) from the per-block counts:
// the block's offset is the sum of the counts before it; inside the chunk
// each tile is compacted in node order (warp ballots, then the warps'
// counts in order).  Returns |V_E|.
// goal_now, err_now: thread 0's reads of those words, for the block (sh.goal,
// sh.err); they and the first tile's flags are fetched beside the counts.
__device__ __forceinline__ int write_ve(const KParams& P, const Team& T, int n, LoopShared& sh,
                                        int goal_now = 0, int err_now = 0) {
  int v0, v1;
  chunk_of(T, n, &v0, &v1);
  auto member = [&](int v) { return v < v1 && P.in_ve[KP_IDX(P, v, P.t_e, 3)]; };
  bool first = member(v0 + (int)threadIdx.x);
  uint32_t off, total;
  block_prefix(T, P.blk_b, sh, &off, &total, [&]() {
    if (threadIdx.x == 0) {
      sh.goal = goal_now;
      sh.err = err_now;
    }
  });
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
  int base = (int)off, buf = 0;
  for (int t0 = v0; t0 < v1; t0 += (int)blockDim.x, buf ^= 1) {
    const int v = t0 + (int)threadIdx.x;
    const bool m = t0 == v0 ? first : member(v);
    const uint32_t bal = __ballot_sync(0xffffffffu, m);
    // the other buffer's readers are past this barrier before it is written
    if (lane == 0) sh.tile[buf][w] = (uint32_t)__popc(bal);
    __syncthreads();
    const int before = (int)warp_before(sh.tile[buf]), tile = (int)warp_total(sh.tile[buf]);
    if (m) P.ve[KP_IDX(P, base + before + __popc(bal & ((1u << lane) - 1u)), P.t_e, 4)] = v;
    base += tile;
  }
  return (int)total;
}

// ---------------------------------------------------------------------------
// learned proposal: node features and the network (6D systems)
// ---------------------------------------------------------------------------

// Features 2q and 2q+1 (q = 0..15) of node v under the current region
// tables; the 32 features are: bounded state entries mapped to [-1, 1], an
// unbounded one wrapped to [-pi, pi) and divided by pi; goal minus
// position; Cov / n'; FreeVol / vol; log(1 + n_valid); log(1 + n_invalid);
// P_accept of the node's region and of its six face neighbours in the
// position grid (0 outside, and 0 under the kd-tree decomposition); zeros
// from feature 20 on.
__device__ __forceinline__ float state_feature(const KParams& P, int i, float x) {
  if (P.feat_scale[i] > 0.0f) return (x - P.x_lo[i]) * P.feat_scale[i] - 1.0f;
  const float y = x - 6.28318530717958648f * floorf((x + 3.14159265358979324f) *
                                                    0.159154943091895336f);
  return y * 0.318309886183790672f;
}

// What a feature pair is computed from.  Fetched without branches, every lane
// the same fields (the sixteen lanes of a node read the same addresses but for
// states and thresholds): behind a branch a pair's loads would wait for the
// ones before it.
struct FeatureInput {
  float s0, s1;           // state entries
  uint32_t nv, ni, cov;   // region counts
  uint64_t t0, t1;        // thresholds, 0 outside the grid
};

__device__ __forceinline__ FeatureInput feature_input(const KParams& P, int v, int q) {
  FeatureInput in;
  const int r = P.region[v];
  // q < 3: entries 2q, 2q + 1; q = 3: 0, 1; q = 4: 2
  const int d0 = q < 3 ? 2 * q : q == 3 ? 0 : 2, d1 = q < 3 ? 2 * q + 1 : 1;
  in.s0 = P.st[(size_t)d0 * P.t_e + v];
  in.s1 = P.st[(size_t)d1 * P.t_e + v];
  in.nv = P.n_valid[r];
  in.ni = P.n_invalid[r];
  in.cov = P.cov[r];
  // q = 6: the region's threshold second; q = 7, 8, 9: those of its
  // neighbours along axis q - 7 (none for kd-tree regions)
  const bool axis = q >= 7 && q < 10 && !P.fso;
  const int g = q == 7 ? P.grid[0] : q == 8 ? P.grid[1] : P.grid[2];
  const int stride = q == 7 ? 1 : q == 8 ? P.grid[0] : P.grid[0] * P.grid[1];
  const int c = (r / stride) % g;
  const bool has0 = axis && c > 0, has1 = (axis && c < g - 1) || q == 6;
  const uint64_t t0 = P.thr[has0 ? r - stride : r], t1 = P.thr[has1 && axis ? r + stride : r];
  in.t0 = has0 ? t0 : 0ull;
  in.t1 = has1 ? t1 : 0ull;
  return in;
}

__device__ __forceinline__ void node_feature_pair(const KParams& P, int q, const FeatureInput& in,
                                                  float* f2) {
  const float nv = (float)in.nv, ni = (float)in.ni, dl = (float)P.delta;
  // thresholds first; zeros where a pair has none
  f2[0] = (float)in.t0 * 2.3283064365386963e-10f;
  f2[1] = (float)in.t1 * 2.3283064365386963e-10f;
  if (q < 3) {
    f2[0] = state_feature(P, 2 * q, in.s0);
    f2[1] = state_feature(P, 2 * q + 1, in.s1);
  } else if (q == 3) {
    f2[0] = P.goal_c[0] - in.s0;
    f2[1] = P.goal_c[1] - in.s1;
  } else if (q < 7) {
    const float ratio = (q == 4 ? (float)in.cov : dl + nv) / (q == 4 ? (float)P.n_sub_per : dl + nv + ni);
    const float lg = log1pf(q == 5 ? nv : ni);
    f2[0] = q == 4 ? P.goal_c[2] - in.s0 : q == 5 ? ratio : lg;
    if (q < 6) f2[1] = q == 4 ? ratio : lg;
  }
}

// One network tile.  Not inlined: it runs a few times per pass, and as a call
// it gets the register budget of the loop kernel to itself instead of sharing
// it with the loop state live around it.  What it needs is passed by value: a
// field read through a reference to the kernel's parameters is a load from
// memory here, not from the constant bank.
template <bool STAGED>
static __device__ __noinline__ void network_tile(MlpWeights w, const uint4* W2,
                                                 const __nv_bfloat16* sX, __nv_bfloat16* sH,
                                                 float* heads, int row0, int rows) {
  mlp_tile_forward<MLP_LOOP_TILE / 16, STAGED>(w, W2, sX, sH, heads, row0, rows);
}

// Phase F: features of every V_E position (kept for the harvest) and, with
// a network attached, its outputs, in tiles of 32 positions per group of 256
// threads; 16 threads share the features of one position.  The chain of loads
// bounds it: a pass has at most a few tiles a group.  The second layer's weights
// (128 KB, which every tile reads) are staged in shared memory where they
// fit.  Measured at the last pass of a 200-box forest query (35,000 positions,
// three tiles a group): 45 us with a branch a feature pair, parameters read
// through a reference and the weights fetched from L2, 26 us as it is; one tile
// 18,000 and 11,700 clocks (features 8,700 -> 5,000, second layer 5,200 ->
// 2,900; with three groups an SM, mma.sync's rate bounds that layer at 2,000).
// Fetching the next tile's lines into L1 ahead made a launch 2 % slower.
__device__ __forceinline__ void phase_features(const KParams& P, const Team& T, int n_ve,
                                               unsigned char* mtile, const uint4* staged) {
  const int group = (int)threadIdx.x / KP_MLP_GROUP, groups = P.mlp_groups;
  if (group >= groups) return;  // (no room for their tiles)
  const int tid = (int)threadIdx.x % KP_MLP_GROUP;
  __nv_bfloat16* sX = reinterpret_cast<__nv_bfloat16*>(mtile + group * MLP_LOOP_TILE_SMEM);
  __nv_bfloat16* sH = sX + MLP_LOOP_TILE * MLP_XS;
  const int n_tiles = (n_ve + MLP_LOOP_TILE - 1) / MLP_LOOP_TILE;
  constexpr int ROUNDS = MLP_LOOP_TILE / 16;  // 16 rows x 16 feature pairs per round
  const int q = tid & 15;
  for (int tile = T.b + T.nb * group; tile < n_tiles; tile += T.nb * groups) {
    const int p0 = tile * MLP_LOOP_TILE;
    const int rows = n_ve - p0 < MLP_LOOP_TILE ? n_ve - p0 : MLP_LOOP_TILE;
    FeatureInput in[ROUNDS];
    int v[ROUNDS];
#pragma unroll
    for (int rr = 0; rr < ROUNDS; ++rr) {
      const int row = rr * 16 + (tid >> 4);
      v[rr] = P.ve[p0 + (row < rows ? row : 0)];
    }
#pragma unroll
    for (int rr = 0; rr < ROUNDS; ++rr) in[rr] = feature_input(P, v[rr], q);
#pragma unroll
    for (int rr = 0; rr < ROUNDS; ++rr) {
      const int row = rr * 16 + (tid >> 4);
      float f2[2];
      node_feature_pair(P, q, in[rr], f2);
      const uint32_t v2 = row < rows ? pack_bf16(f2[0], f2[1]) : 0u;
      *reinterpret_cast<uint32_t*>(sX + row * MLP_XS + 2 * q) = v2;
      if (row < rows) *reinterpret_cast<uint32_t*>(P.feat + (size_t)(p0 + row) * 32 + 2 * q) = v2;
    }
    // the next tile's inputs and hidden rows are written after this tile's last
    // and the next one's first barrier: every thread is past its reads by then
    if (P.mix_thr) {
      MlpWeights w;
      w.W1 = reinterpret_cast<const __nv_bfloat16*>(P.mlp_W1);
      w.b1 = P.mlp_b1;
      w.b2 = P.mlp_b2;
      w.W3 = reinterpret_cast<const __nv_bfloat16*>(P.mlp_W3);
      w.b3 = P.mlp_b3;
      if (P.mlp_w2_off > 0)
        network_tile<true>(w, staged, sX, sH, P.net_heads, p0, rows);
      else
        network_tile<false>(w, reinterpret_cast<const uint4*>(P.mlp_W2), sX, sH, P.net_heads, p0, rows);
    }
  }
}

// Standard normals z[0..3] from four Philox words (Box-Muller, pairs of
// words: radius from the first, angle from the second).
__device__ __forceinline__ void box_muller4(uint4 w, float* z) {
  const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int pr = 0; pr < 2; ++pr) {
    const float r1 = (float)((ws[2 * pr] >> 8) + 1u) * 5.9604644775390625e-08f;  // (0, 1]
    const float r2 = (float)(ws[2 * pr + 1] >> 8) * 5.9604644775390625e-08f;     // [0, 1)
    const float rad = sqrtf(-2.0f * logf(r1));
    float s, c;
    sincospif(2.0f * r2, &s, &c);
    z[2 * pr] = rad * c;
    z[2 * pr + 1] = rad * s;
  }
}

// The draw of sample key (V_E position p = key / lam of node v, j = key - p
// lam) in pass it (Algorithm 2: random control in U, random duration).
// Counter (it, node, j, purpose): purpose 0 the control words (kept in wr),
// purpose 1 (duration, accept word, selector); with a network attached and the
// selector below the mix threshold, the control comes from the node's Gaussian
// with normals from purpose 3 (the duration keeps the uniform draw).
// The expand phase and the node-set phase (which appends accepted samples
// by their keys) both draw through this function, so both see the same
// numbers.
template <int SYS>
__device__ __forceinline__ void draw_controls(const KParams& P, uint32_t it, int key, int v,
                                              const KeyDiv& kd, float* u, int* k, uint32_t* wacc,
                                              uint32_t* wr) {
  constexpr int N = System<SYS>::N;
  const int p = kd.quot(key);
  const int j = key - p * kd.lam;
  const uint4 w0 = philox4x32_10(make_uint4(it, (uint32_t)v, (uint32_t)j, 0u), P.seed_lo, P.seed_hi);
  const uint4 w1 = philox4x32_10(make_uint4(it, (uint32_t)v, (uint32_t)j, 1u), P.seed_lo, P.seed_hi);
  wr[0] = w0.x; wr[1] = w0.y; wr[2] = w0.z; wr[3] = w0.w;
#pragma unroll
  for (int d = 0; d < N; ++d) u[d] = __fmaf_rn(P.u_scale[d], unit24(wr[d]), P.u_lo[d]);
  *k = P.k_min + (int)__umulhi(w1.x, P.k_span);
  if (w1.z < P.mix_thr) {
    // learned draw from the node's Gaussian (normals: purpose 3)
    const uint4 w3 = philox4x32_10(make_uint4(it, (uint32_t)v, (uint32_t)j, 3u), P.seed_lo, P.seed_hi);
    const float4* heads = reinterpret_cast<const float4*>(P.net_heads + (size_t)p * MLP_OUT);
    const float4 m4 = heads[0], s4 = heads[1];
    const float mean[4] = {m4.x, m4.y, m4.z, m4.w}, sd[4] = {s4.x, s4.y, s4.z, s4.w};
    float z[4], q[4];
    box_muller4(w3, z);
#pragma unroll
    for (int d = 0; d < N; ++d) q[d] = fminf(fmaxf(__fmaf_rn(sd[d], z[d], mean[d]), -1.0f), 1.0f);
#pragma unroll
    for (int d = 0; d < N; ++d)
      u[d] = __fmaf_rn(P.u_scale[d], __fmul_rn(__fadd_rn(q[d], 1.0f), 0.5f), P.u_lo[d]);
  }
  *wacc = w1.y;
}

// The draw of sample 'key' and its parent's state (the start of the
// segment).
template <int SYS>
__device__ __forceinline__ void draw_sample(const KParams& P, uint32_t it, int key, int v,
                                            const KeyDiv& kd, float* x, float* u, int* k,
                                            uint32_t* wacc, uint32_t* wr) {
  constexpr int D = System<SYS>::D;
#pragma unroll
  for (int d = 0; d < D; ++d) x[d] = P.st[(size_t)d * P.t_e + v];
  draw_controls<SYS>(P, it, key, v, kd, u, k, wacc, wr);
}

// Phase E: Algorithm 2 for every sample key in [0, S).
//
// Lanes integrate step by step and are refilled as they finish: a warp
// takes keys in batches from a grid-wide counter, every lane carries one
// sample (k steps, or fewer when a step is invalid), and when enough lanes
// of the warp have finished they are finalised (binning, counters, claim,
// flags) and given new keys together, so that the divergent finalise /
// start-up work is shared by many lanes and no lane idles while a long
// sample runs next to it.  Every sample's arithmetic depends on its key
// alone, so the result does not depend on which lane ran it.
// keys a warp takes from the grid counter at most (256: 0.5 % of a launch with a
// large frontier faster than 128, 64 1.5 % slower)
constexpr int KP_KEY_BATCH = 256;

// A warp whose time ran out gives up its lanes' samples, the keys it has taken
// and those that no warp has taken (whoever asks for more finds none): their
// flags say that nothing came of them.  The accept phase reads every key's flags,
// and the barrier before it stops only blocks that wait for long.  (Every warp
// looking at the error word there cost a pass 0.1 to 0.6 us, a call of 20 passes
// 1.1 %; this costs 0 to 0.3 %, a call, so that the loop's registers stay.)
static __device__ __noinline__ void give_up_keys(const KParams& P, int key, int pool_next, int pool_end,
                                             int static_end, int S) {
  const int lane = (int)(threadIdx.x & 31u);
  auto clear = [&](int q) { P.flags[KP_IDX(P, q, P.t_e, 11)] = 0; };
  if (key >= 0) clear(key);
  for (int q = pool_next + lane; q < pool_end; q += 32) clear(q);
  int rest = S;
  if (lane == 0 && static_end < S)
    rest = static_end + atomicMax(&P.ctl->work_next, S - static_end);
  rest = __shfl_sync(0xffffffffu, rest, 0);
  for (int q = rest + lane; q < S; q += 32) clear(q);
}

template <int SYS, bool LOG>
__device__ __forceinline__ void phase_expand(const KParams& P, const Team& T,
                                             const unsigned char* sblob, uint32_t it, const KeyDiv& kd,
                                             int S, LoopShared& sh) {
  using Sys = System<SYS>;
  constexpr int D = Sys::D, N = Sys::N;
  const float4* sbox = reinterpret_cast<const float4*>(sblob);
  const uint16_t* sstart = reinterpret_cast<const uint16_t*>(sblob + P.bp_start_off);
  const uint16_t* sids = reinterpret_cast<const uint16_t*>(sblob + P.bp_ids_off);
  const uint8_t* sclear = P.bp_clear_off >= 0 ? sblob + P.bp_clear_off : nullptr;
  const uint32_t FULL = 0xffffffffu;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t lt = (1u << lane) - 1u;

  // per-thread counts of one pass: a thread runs at most 2^28 / 256 keys of
  // at most 255 steps each, so 32 bits hold them; n_refill counts the keys
  // a lane starts after its first one, n_batch (lane 0) the batches its
  // warp takes from the grid counter
  uint32_t n_steps = 0, n_hull = 0, n_box = 0, n_refill = 0, n_batch = 0;
  bool ran = false;
  // lane state: the sample being integrated
  int key = -1, v = 0, k = 0, i = 0, fail = 0;
  bool busy = false;  // a sample in flight (a finished one keeps its key)
  float x[D], u[N];
  uint32_t wacc = 0, wr[4] = {0, 0, 0, 0};
  // warp state (uniform): the current batch of keys.  The first batch of
  // every warp is fixed by the warp's index (keys [gw b0, (gw + 1) b0), the
  // size the live sizing below gives at the start of a pass), so no warp
  // queues on the counter to start; later batches come from the counter,
  // offset past the statically handed-out keys.
  const int n_warps = T.nb * (int)(blockDim.x >> 5);
  // The warps are numbered across the blocks first, so that a pass of fewer
  // batches than warps spreads over all SMs (block by block, a small pass filled
  // some SMs and left the others idle: 0.9 to 1.7 % of a launch).
  const int gw = T.b + T.nb * (int)(threadIdx.x >> 5);
  int b0 = S / (2 * n_warps);
  b0 = b0 < Sys::FIRST_BATCH_MIN ? Sys::FIRST_BATCH_MIN : (b0 > KP_KEY_BATCH ? KP_KEY_BATCH : b0);
  const int static_end = n_warps * b0 < S ? n_warps * b0 : S;
  int pool_next = gw * b0 < S ? gw * b0 : S;
  int pool_end = pool_next + b0 < S ? pool_next + b0 : S;
  bool exhausted = S <= 0;
  int refill_at = exhausted ? 32 : Sys::REFILL_MIN;
  // bound on the phase's device time, checked warp-uniformly at every
  // refill (a sample runs at most 255 steps, so refills are at most 255
  // iterations apart)
  const uint64_t t_phase = global_ns();

  for (;;) {
    // finished lanes are finalised together: REFILL_MIN of them while keys
    // remain (they are refilled at once), and once the pass's keys are all
    // handed out, only when every lane has finished, so that the warp's
    // last samples cost one finalise instead of one per finishing step
    const uint32_t m_free = __ballot_sync(FULL, !busy);
    if (__popc(m_free) >= refill_at) {
      const uint64_t now = __shfl_sync(FULL, global_ns(), 0);
      if (now - t_phase > P.wait_ns) {
        if (lane == 0) raise_error(P.ctl, KP_DEV_ERR_TIMEOUT, 30);
        give_up_keys(P, key, pool_next, pool_end, static_end, S);
        break;
      }
      // Finalise and refill together: what each needs from memory is issued
      // side by side, two round trips to L2 in a row (three when the warp
      // needs a batch of keys) where one after the other took four to six
      // (0.5 to 1 % of a launch: the other warps hide most of a round trip).
      // ---- first round trip -----------------------------------------------
      // the pool's keys for the free lanes (and their nodes), and, when it
      // holds too few, the counter's value
      const bool fin = key >= 0 && !busy;
      const int rank = __popc(m_free & lt), avail = pool_end - pool_next;
      const int short_by = __popc(m_free) - avail;
      const bool take = !exhausted && short_by > 0;
      int next = -1, next_v = 0, cur = 0;
      if (!busy && rank < avail) {
        next = pool_next + rank;
        next_v = P.ve[KP_IDX(P, kd.quot(next), P.t_e, 5)];
      }
      pool_next = short_by > 0 ? pool_end : pool_next + __popc(m_free);
      if (take && lane == 0 && static_end < S) cur = *((volatile int*)&P.ctl->work_next);
      // the finished lanes' bins: whether the sub-region was visited, its
      // claim so far, the region's threshold
      int r = 0, s = 0;
      uint32_t claimed = 0;
      uint64_t thr = 0;
      bool cont = false;
      const bool valid = fin && fail == 0;
      if (fin) {
        // steps run, and hull tests (every step but one that left the
        // state box)
        n_steps += (uint32_t)i;
        n_hull += (uint32_t)(fail < 0 ? i - 1 : i);
        bin_state<SYS>(x, P, &r, &s, sblob);
        if (valid) {
          r = KP_IDX(P, r, P.R, 7);
          s = KP_IDX(P, s, (long long)P.R * P.n_sub_per, 8);
          key = KP_IDX(P, key, P.t_e, 9);
          cont = P.visited[s] == 0;
          claimed = __ldcg(P.claim + s);
          thr = P.thr[r];
        }
      }
      // ---- second round trip ----------------------------------------------
      // the claim, unless a smaller key is there already (it is lost then)
      const bool bern = valid && (uint64_t)wacc < thr;
      const bool may_win = cont && claimed > (uint32_t)key;
      uint32_t prev = 0;
      if (may_win) prev = atomicMin(&P.claim[s], (uint32_t)key);
      // the first claimant of a sub-region knows it is newly reached: it will
      // get exactly one representative in region r (before the draw where its
      // twelve states leave no registers to keep the answer: 0.5 % of a
      // quadrotor query; after it 0.8 % of a Dubins one)
      auto new_region = [&]() {
        if (prev == 0xffffffffu) {
          atomicAdd(&P.cov[r], 1u);
          P.avail[r] = 1;
        }
      };
      // batches shrink towards the end of the pass so that warps run out of
      // work together
      // (at the very end a warp takes only what its idle lanes can start
      // now, so no warp is left with a second round of samples)
      // (the batch is sized from the counter's current value: a warp that
      // last took keys long ago must not size it from a stale position and
      // leave with a large batch just before the end)
      int base = S;
      if (take && lane == 0 && static_end < S) {
        int want = (S - static_end - cur) / (Sys::GUIDED_DIV * n_warps);
        want = want < short_by ? short_by : (want > KP_KEY_BATCH ? KP_KEY_BATCH : want);
        base = static_end + atomicAdd(&P.ctl->work_next, want);
        base = base < S ? base : S;
        n_batch += base < S ? 1u : 0u;
        pool_end = base + want < S ? base + want : S;
      }
      if (fin) {
        atomicAdd((valid ? P.n_valid : P.n_invalid) + KP_IDX(P, r, P.R, 10), 1u);
        // a sample that may still be accepted (a contender not yet beaten,
        // or past its draw) keeps its end state for the append, and a
        // contender its sub-region for the claim check
        if (cont) P.cs[key] = s;
        if (may_win || bern) {
          float4* row = reinterpret_cast<float4*>(P.xs + (size_t)key * kp_xs_stride(D));
#pragma unroll
          for (int q = 0; q < kp_xs_stride(D) / 4; ++q)
            row[q] = make_float4(4 * q < D ? x[4 * q] : 0.0f, 4 * q + 1 < D ? x[4 * q + 1] : 0.0f,
                                 4 * q + 2 < D ? x[4 * q + 2] : 0.0f,
                                 4 * q + 3 < D ? x[4 * q + 3] : 0.0f);
        }
        if (bern) P.avail[r] = 1;
        P.flags[KP_IDX(P, key, P.t_e, 11)] = (uint8_t)(valid ? KP_F_VALID | (cont ? KP_F_CONTENDER : 0u) |
                                                                   (bern ? KP_F_BERN : 0u)
                                                             : 0u);
        if (LOG && key < P.log.capacity) {
          P.log.node[key] = v;
          P.log.k[key] = k;
#pragma unroll
          for (int d = 0; d < 4; ++d) P.log.uraw[4 * (size_t)key + d] = wr[d];
          P.log.fail_step[key] = fail < 0 ? -fail : fail;
          P.log.region[key] = r;
          P.log.sub[key] = s;
#pragma unroll
          for (int d = 0; d < 12; ++d) P.log.state[12 * (size_t)key + d] = d < D ? x[d] : 0.0f;
        }
        key = -1;
      }
      if (take) {
        base = __shfl_sync(FULL, base, 0);
        pool_end = __shfl_sync(FULL, pool_end, 0);
        pool_next = base;
        if (key < 0 && rank >= avail && rank - avail < pool_end - base) {
          next = base + rank - avail;
          next_v = P.ve[KP_IDX(P, kd.quot(next), P.t_e, 5)];
        }
        // (a batch covers the free lanes unless the keys end)
        if (pool_end - base >= short_by) {
          pool_next = base + short_by;
        } else {
          pool_next = pool_end = S;
          exhausted = true;
          refill_at = 32;
        }
      }
      if (D == 12) new_region();
      if (next >= 0) {
        key = next;
        n_refill += ran ? 1u : 0u;
        ran = true;
        v = KP_IDX(P, next_v, P.t_e, 6);
        draw_sample<SYS>(P, it, key, v, kd, x, u, &k, &wacc, wr);
        Sys::prepare(u, P);
        i = 0;
        fail = 0;
        busy = true;
      }
      if (D != 12) new_region();
      if (!__any_sync(FULL, busy)) break;
    }
    // ---- one integrator step (PropagateODE) and its validity check --------
    if (busy) {
      const float px = x[0], py = x[1], pz = x[2];
      Sys::step(x, u, P.dt, P);
      ++i;
      const bool inbox = in_state_box<Sys>(x, P);
      busy = inbox && i < k;
      fail = inbox ? 0 : -i;  // negative: the end state left the state box
      if (inbox) {
        const float p0[3] = {px, py, pz};
        if (hull_hits_grid(P, sbox, sstart, sids, sclear, p0, x, &n_box)) {
          fail = i;
          busy = false;
        }
      }
    }
  }
  // a sum per warp, then one thread a counter adds the warps' sums (the team
  // barrier that follows frees the shared values)
  const uint32_t mine[5] = {n_steps, n_hull, n_box, n_batch, n_refill};
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    const unsigned long long s = warp_sum_wide(mine[c]);
    if (lane == 0) sh.cnt[c][threadIdx.x >> 5] = s;
  }
  __syncthreads();
  if (threadIdx.x < 5) {
    unsigned long long s = 0;
#pragma unroll 4
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh.cnt[threadIdx.x][w];
    static_assert(offsetof(KCtl, tot_refills) == offsetof(KCtl, tot_steps) + 32, "counters in order");
    if (s) atomicAdd(&P.ctl->tot_steps + threadIdx.x, s);
  }
}

// Contiguous key range [a, b) of warp w >= 1 inside the block's chunk
// [c0, c1) (warp 0 runs the region estimates and gets none).
__device__ __forceinline__ void warp_range(int c0, int c1, int* a, int* b) {
  const int nw = (int)(blockDim.x >> 5) - 1;
  const int w = (int)(threadIdx.x >> 5) - 1;
  if (w < 0) {
    *a = *b = c0;
    return;
  }
  const int per = (c1 - c0 + nw - 1) / nw;
  const long long lo = (long long)c0 + (long long)w * per;
  *a = (int)(lo < c1 ? lo : c1);
  *b = (int)(lo + per < c1 ? lo + per : c1);
}

// Phase A (warps 1..): accept decisions of this block's key chunk.  Each
// warp walks its own key range in tiles of 32 x KP_ACC_KPL keys (lane l
// takes keys t0 + 32q + l: every load is coalesced), with the loads of a
// tile's flags, contenders' sub-regions and their claims issued together,
// and compacts its accepted keys (claim winners marked in bit 31) in key
// order at the start of its range in acc_key.  Phase S comes before it, on the
// warps with a region chunk.  Publishes the block's accepted count, adds the
// valid count to the pass, and leaves where each warp's accepted keys are, and
// their offsets among the block's, in shared memory for the node-set phase.
constexpr int KP_ACC_KPL = 8;

__device__ __forceinline__ void phase_scores(const KParams& P, const Team& T, int nch);

template <bool LOG>
__device__ __forceinline__ void phase_accept(const KParams& P, const Team& T, int S, int nch,
                                             LoopShared& sh) {
  phase_scores(P, T, nch);
  const uint32_t FULL = 0xffffffffu;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t lt = (1u << lane) - 1u;
  int k0, k1, a, b;
  chunk_of(T, S, &k0, &k1);
  warp_range(k0, k1, &a, &b);
  int n_acc = 0;
  uint32_t n_valid = 0;
  for (int t0 = a; t0 < b; t0 += 32 * KP_ACC_KPL) {
    uint32_t f[KP_ACC_KPL], c[KP_ACC_KPL];
    int s[KP_ACC_KPL];
#pragma unroll
    for (int q = 0; q < KP_ACC_KPL; ++q) {
      const int key = t0 + 32 * q + (int)lane;
      f[q] = key < b ? P.flags[key] : 0u;
    }
#pragma unroll
    for (int q = 0; q < KP_ACC_KPL; ++q)
      s[q] = (f[q] & KP_F_CONTENDER) ? P.cs[KP_IDX(P, t0 + 32 * q + (int)lane, P.t_e, 12)] : 0;
#pragma unroll
    for (int q = 0; q < KP_ACC_KPL; ++q)
      c[q] = (f[q] & KP_F_CONTENDER)
                 ? P.claim[KP_IDX(P, s[q], (long long)P.R * P.n_sub_per, 13)]
                 : 0u;
#pragma unroll
    for (int q = 0; q < KP_ACC_KPL; ++q) {
      const int key = t0 + 32 * q + (int)lane;
      const bool valid = (f[q] & KP_F_VALID) != 0;
      n_valid += valid ? 1u : 0u;
      const bool win = (f[q] & KP_F_CONTENDER) && c[q] == (uint32_t)key;
      const bool acc = valid && (win || (f[q] & KP_F_BERN));
      const uint32_t m = __ballot_sync(FULL, acc);
      if (acc)
        P.acc_key[KP_IDX(P, a + n_acc + __popc(m & lt), P.t_e, 14)] =
            (uint32_t)key | (win ? 0x80000000u : 0u);
      n_acc += __popc(m);
      if (LOG && key < b && key < P.log.capacity)
        P.log.flags[key] =
            (uint8_t)(f[q] | (win ? KP_F_WINNER : 0u) | (acc ? KP_F_ACCEPTED : 0u));
    }
  }
  // warp counts -> offsets in key order (warps own ascending ranges)
  const int w = (int)(threadIdx.x >> 5);
  n_valid = __reduce_add_sync(FULL, n_valid);
  if (lane == 0) {
    sh.pre[w] = (uint32_t)n_acc;
    sh.tot[w] = n_valid;
  }
  __syncthreads();
  const int off = (int)warp_before(sh.pre), block_acc = (int)warp_total(sh.pre);
  const uint32_t bv = warp_total(sh.tot);
  if (lane == 0) {
    sh.acc_a[w] = a;
    sh.acc_n[w] = n_acc;
    sh.acc_off[w] = off;
  }
  if (threadIdx.x == 0) {
    sh.acc_tot = block_acc;
    if (T.b == 0) P.ctl->work_next = 0;  // the expand phase is over
    P.blk_a[KP_IDX(P, T.b, KP_MAX_GRID, 15)] = (uint32_t)block_acc;
    if (bv) atomicAdd(&P.ctl->it_valid, bv);
  }
}

// Pairwise (bottom-up, the same tree as recursive halving) sum of n values, n a
// power of two at most 32 KP_TREE_PER_LANE, by one warp in registers: lane l
// loads the m = max(n / 32, 1) values l m .. l m + m - 1 through load(i), adds
// the tree's levels of stride below m in place, and the levels of stride m,
// 2m, ... across lanes by shuffles (left operand the lower index).  Every lane
// gets the sum.
constexpr int KP_TREE_PER_LANE = 8;

// The levels across the first 'lanes' lanes (a power of two).
__device__ __forceinline__ double warp_tree_lanes(double sum, int lanes) {
  const int lane = (int)(threadIdx.x & 31u);
  for (int d = 1; d < lanes; d <<= 1) {
    const double o = __shfl_down_sync(0xffffffffu, sum, d);
    if ((lane & (2 * d - 1)) == 0) sum = __dadd_rn(sum, o);
  }
  return __shfl_sync(0xffffffffu, sum, 0);
}

template <class L>
__device__ __forceinline__ double warp_tree_sum(int n, L load) {
  const int lane = (int)(threadIdx.x & 31u);
  const int m = n >= 32 ? n >> 5 : 1;
  double v[KP_TREE_PER_LANE];
#pragma unroll
  for (int q = 0; q < KP_TREE_PER_LANE; ++q) {
    const int i = lane * m + q;
    v[q] = q < m && i < n ? load(i) : 0.0;
  }
#pragma unroll
  for (int st = 1; st < KP_TREE_PER_LANE; st <<= 1)
#pragma unroll
    for (int q = 0; q + st < KP_TREE_PER_LANE; q += 2 * st)
      if (st < m) v[q] = __dadd_rn(v[q], v[q + st]);
  return warp_tree_lanes(v[0], n / m);
}

// Region chunks of the score sums: nch of them (a power of two, at most 256),
// chunk c the work of warp c / blocks of block c % blocks (then of the same
// warp again, were there more chunks than warps).
template <class F>
__device__ __forceinline__ void for_own_chunks(const Team& T, int nch, F body) {
  for (int c = T.b + T.nb * (int)(threadIdx.x >> 5); c < nch; c += T.nb * (int)(blockDim.x >> 5)) body(c);
}

// Phase S: Eq. 3-4 for a warp's region chunk and the chunk's pairwise partial
// sum (published by the grid barrier that ends the phase).  Lane l takes the
// chunk's m = max(ch / 32, 1) regions from l m on and adds their scores up as
// they come: level k of the tree waits in left[k] for its right half.  Most
// decompositions have chunks of 32 (a region a lane): FP64 divisions are long
// chains here (about two FP64 operations a clock and SM), and one warp that
// took all of a 512-region chunk, as a small team has, held the pass up by 16
// of them.  Every operation is an explicitly rounded IEEE double operation in
// the order
// FreeVol = ((delta + nv) vol) / ((delta + nv) + ni),
// f4 = (FreeVol FreeVol)(FreeVol FreeVol),
// Score = f4 / ((1 + Cov)(1 + (nv + ni)(nv + ni))).
__device__ __forceinline__ void phase_scores(const KParams& P, const Team& T, int nch) {
  const int lane = (int)(threadIdx.x & 31u);
  const int ch = P.R_pad / nch;
  const int m = ch >= 32 ? ch >> 5 : 1;  // below 2^12: R is at most 2^24
  for_own_chunks(T, nch, [&](int c) {
    double left[12], sum = 0.0;
#pragma unroll 1
    for (int q = 0; q < m; ++q) {
      const int r = c * ch + lane * m + q;
      double sc = 0.0;
      if (lane < ch && r < P.R) {
        // every input is loaded at once; the counts' sum is exact as an
        // integer, so its conversion is the double sum
        const uint32_t cv = P.n_valid[r], ci = P.n_invalid[r], cc = P.cov[r];
        const bool avail = P.avail[r] != 0;
        const double vol = P.region_vol ? P.region_vol[r] : P.vol;
        if (avail) {
          const double nv = (double)cv, ni = (double)ci;
          const double na = (double)((unsigned long long)cv + ci);
          const double dn = __dadd_rn(P.delta, nv);
          const double den = __dmul_rn(__dadd_rn(1.0, (double)cc), __dadd_rn(1.0, __dmul_rn(na, na)));
          const double fv = __ddiv_rn(__dmul_rn(dn, vol), __dadd_rn(dn, ni));
          const double f2 = __dmul_rn(fv, fv);
          sc = __ddiv_rn(__dmul_rn(f2, f2), den);
        }
        P.score[r] = avail ? sc : KP_NO_SCORE;  // P_accept = 1
      }
      int k = 0;
      for (; (q >> k) & 1; ++k) sc = __dadd_rn(left[k], sc);
      if (k < 12) left[k] = sc;
      sum = sc;
    }
    const double part = warp_tree_lanes(sum, ch < 32 ? ch : 32);
    if (lane == 0) P.chunk_sum[KP_IDX(P, c, KP_MAX_GRID, 16)] = part;
  });
}

// The sum of Eq. 5 from the chunks' partial sums, by the calling warp, for the
// block: sh.score.
__device__ __forceinline__ void sum_scores(const KParams& P, const Team& T, int nch, LoopShared& sh) {
  const double sum = warp_tree_sum(nch, [&](int i) { return __ldcg(P.chunk_sum + i); });
  if ((threadIdx.x & 31u) == 0) {
    sh.score = score_sum_of(sum, P.eps);
    if (T.b == 0) P.ctl->score_sum = sum;
  }
}

// Phase T: the thresholds of the warp's region chunks, for the next expand phase.
__device__ __forceinline__ void phase_thresholds(const KParams& P, const Team& T, int nch,
                                                 const LoopShared& sh) {
  const int ch = P.R_pad / nch;
  for_own_chunks(T, nch, [&](int c) {
    for (int r = c * ch + (int)(threadIdx.x & 31u); r < (c + 1) * ch && r < P.R; r += 32)
      P.thr[r] = accept_threshold(P.score[r], sh.score.sum, sh.score.inv, P.eps);
  });
}

// Accepted sample j of this block: its key, bit 31 set for a claim winner.  The
// warp that holds it is the last one whose offset is at most j (warps without
// samples have their successor's offset).
__device__ __forceinline__ uint32_t accepted_key(const KParams& P, const LoopShared& sh, int j) {
  int w = 0;
#pragma unroll
  for (int s = 16; s > 0; s >>= 1)
    if (w + s < (int)(blockDim.x >> 5) && sh.acc_off[w + s] <= j) w += s;
  return P.acc_key[KP_IDX(P, sh.acc_a[w] + (j - sh.acc_off[w]), P.t_e, 17)];
}

// Materialises this block's accepted samples as the nodes id0 .. id0 +
// acc_tot - 1 (id0 = t_old + the accepted samples of the blocks before it:
// node ids follow the sample keys).  Every accepted sample takes the end
// state the expand phase kept for it, its parent, control and duration
// from its key (the same draw), and its region and sub-region; visited and
// the goal test (closed ball on position; the smallest new goal node wins)
// follow.  Thread j of the block takes the block's samples j, j +
// blockDim.x, ... (e: sample threadIdx.x's accepted_key, fetched by the
// caller beside its own loads); consecutive threads write consecutive nodes.
// With the sample log on, the sample is also re-derived from its key (the
// same integrator steps, explicitly rounded, so the same numbers) and must
// match the kept and the logged state bit for bit.
template <int SYS, bool LOG>
__device__ __forceinline__ void materialise(const KParams& P, uint32_t it, int id0, const KeyDiv& kd,
                                            const LoopShared& sh, const unsigned char* sblob,
                                            uint32_t e) {
  using Sys = System<SYS>;
  constexpr int D = Sys::D, N = Sys::N;
  for (int j = (int)threadIdx.x; j < sh.acc_tot; j += (int)blockDim.x) {
    if (j != (int)threadIdx.x) e = accepted_key(P, sh, j);
    const int key = KP_IDX(P, (int)(e & 0x7fffffffu), P.t_e, 18);
    const int id = KP_IDX(P, id0 + j, P.t_e, 19);
    float x[D], u[N];
    int k;
    uint32_t wacc, wr[4];
    const int v = KP_IDX(P, P.ve[KP_IDX(P, kd.quot(key), P.t_e, 5)], P.t_e, 6);
    draw_controls<SYS>(P, it, key, v, kd, u, &k, &wacc, wr);
    {
      const float4* row = reinterpret_cast<const float4*>(P.xs + (size_t)key * kp_xs_stride(D));
#pragma unroll
      for (int q = 0; q < (D + 3) / 4; ++q) {
        const float4 c = row[q];
        if (4 * q < D) x[4 * q] = c.x;
        if (4 * q + 1 < D) x[4 * q + 1] = c.y;
        if (4 * q + 2 < D) x[4 * q + 2] = c.z;
        if (4 * q + 3 < D) x[4 * q + 3] = c.w;
      }
    }
    int r, s;
    bin_state<SYS>(x, P, &r, &s, sblob);
    r = KP_IDX(P, r, P.R, 20);
    s = KP_IDX(P, s, (long long)P.R * P.n_sub_per, 21);
#pragma unroll
    for (int d = 0; d < D; ++d) P.st[(size_t)d * P.t_e + id] = x[d];
#pragma unroll
    for (int d = 0; d < N; ++d) P.ctrl[(size_t)d * P.t_e + id] = u[d];
    P.steps[id] = (uint8_t)k;
    P.parent[id] = v;
    P.region[id] = r;
    P.node_sub[id] = s;
    P.in_ve[id] = 1;
    P.visited[s] = 1;
    const float dx = __fsub_rn(x[0], P.goal_c[0]), dy = __fsub_rn(x[1], P.goal_c[1]),
                dz = __fsub_rn(x[2], P.goal_c[2]);
    const bool goal = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx))) <= P.goal_r2;
    if (goal) atomicMin(&P.ctl->goal_node, id);
    if (P.hv_cap > 0 && (e & 0x80000000u)) {
      // training pair: the parent's features and this sample's draw
      const uint32_t h = atomicAdd(P.hv_count, 1u);
      if (h < (uint32_t)P.hv_cap) {
        const __nv_bfloat16* fr =
            reinterpret_cast<const __nv_bfloat16*>(P.feat) + (size_t)kd.quot(key) * 32;
        for (int c = 0; c < 32; ++c) P.hv_feat[(size_t)h * 32 + c] = __bfloat162float(fr[c]);
#pragma unroll
        for (int d = 0; d < 3; ++d)
          P.hv_target[(size_t)h * 4 + d] = 2.0f * (u[d] - P.u_lo[d]) / P.u_scale[d] - 1.0f;
        P.hv_target[(size_t)h * 4 + 3] =
            P.k_span > 1 ? 2.0f * (float)(k - P.k_min) / (float)(P.k_span - 1) - 1.0f : 0.0f;
      }
    }
    if (LOG && key < P.log.capacity) {
      if (goal) P.log.flags[key] |= (uint8_t)KP_F_GOAL;
      float y[D];
#pragma unroll
      for (int d = 0; d < D; ++d) y[d] = P.st[(size_t)d * P.t_e + v];
      Sys::prepare(u, P);  // (the node's controls are written above)
      for (int st = 0; st < k; ++st) Sys::step(y, u, P.dt, P);
      bool same = P.log.region[key] == r && P.log.sub[key] == s;
#pragma unroll
      for (int d = 0; d < D; ++d)
        same = same && __float_as_uint(P.log.state[12 * (size_t)key + d]) == __float_as_uint(x[d]) &&
               __float_as_uint(y[d]) == __float_as_uint(x[d]);
      if (!same) raise_error(P.ctl, KP_DEV_ERR_REPLAY, 40);
    }
  }
}

// Phase N: Algorithm 4 node sets, one draw per old node (counter: it, v, 0,
// purpose 2) against the threshold of its region; new nodes are in V_E.
// Publishes the block chunk's V_E count; returns in *n_new the number of
// accepted samples of the pass (the new nodes).
// Order inside the phase: a warp sums the scores while the others append the
// block's accepted samples (ids from t_old, in key order); then the block makes
// its draws, each with the threshold of its node's region worked out from the
// region's score, and last the warps with a region chunk write its thresholds
// for the next pass.  (With the table written first, every block waited for the
// chunks' sums, divisions and a count of the chunks done: 3,900 to 6,100 clocks and
// 1,500 more.)  New nodes are counted as V_E members without reading their sets.
template <int SYS, bool LOG>
__device__ __forceinline__ void phase_nodesets(const KParams& P, const Team& T, uint32_t it,
                                               int t_old, const KeyDiv& kd, LoopShared& sh, int* n_new,
                                               const unsigned char* sblob) {
  const int nch = P.nch;
  uint32_t acc_before, acc_total;
  const uint32_t e0 = (int)threadIdx.x < sh.acc_tot ? accepted_key(P, sh, (int)threadIdx.x) : 0u;
  block_prefix(T, P.blk_a, sh, &acc_before, &acc_total);
  if ((threadIdx.x >> 5) == (blockDim.x >> 5) - 1) sum_scores(P, T, nch, sh);
  *n_new = (int)acc_total;
  const int t_new = t_old + (int)acc_total;
  materialise<SYS, LOG>(P, it, t_old + (int)acc_before, kd, sh, sblob, e0);
  // old nodes of the chunk: two tiles at a time, their region and score loads
  // issued together (the first two tiles' before the wait for the sum)
  int v0, v1;
  chunk_of(T, t_new, &v0, &v1);
  const int o1 = v1 < t_old ? v1 : t_old;
  const int stride = (int)blockDim.x;
  double sq[2];
  auto scores = [&](int t0) {
    int rq[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int v = t0 + q * stride + (int)threadIdx.x;
      rq[q] = v < o1 ? KP_IDX(P, __ldcg(P.region + KP_IDX(P, v, P.t_e, 22)), P.R, 23) : 0;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
      sq[q] = t0 + q * stride + (int)threadIdx.x < o1 ? __ldcg(P.score + rq[q]) : 0.0;
  };
  scores(v0);
  __syncthreads();
  int c = 0;
  for (int t0 = v0; t0 < o1; t0 += 2 * stride) {
    if (t0 != v0) scores(t0);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int v = t0 + q * stride + (int)threadIdx.x;
      if (v < o1) {
        const uint4 w = philox4x32_10(make_uint4(it, (uint32_t)v, 0u, 2u), P.seed_lo, P.seed_hi);
        const int e = draw_accepted(w.x, sq[q], sh.score, P.eps) ? 1 : 0;
        P.in_ve[v] = (uint8_t)e;
        c += e;
      }
    }
  }
  phase_thresholds(P, T, nch, sh);
  // new nodes are V_E members (their flags are set by the blocks that
  // appended them, so they are counted, not read)
  const int new0 = v0 > t_old ? v0 : t_old;
  const uint32_t tot = block_sum((uint32_t)c, sh) + (uint32_t)(v1 > new0 ? v1 - new0 : 0);
  if (threadIdx.x == 0) P.blk_b[KP_IDX(P, T.b, KP_MAX_GRID, 24)] = tot;
}

// The loop of one query (Algorithm 1 body, repeated) run by a team of
// blocks, with the query's obstacle blob already in shared memory.  Stops
// when a goal node is appended, Eq. 6 gives lambda = 0, or the pass or time
// budget is spent.  Returns false when a bounded wait expired.
template <int SYS, bool LOG>
__device__ __forceinline__ bool run_loop(const KParams& P, const Team& T, unsigned char* smem,
                                         LoopShared& sh, int max_iters, uint64_t max_ns) {
  KCtl* ctl = P.ctl;
  const uint64_t t_start = global_ns();
  if (T.b == 0 && threadIdx.x == 0) {
    ctl->it_valid = 0;
    ctl->stop = 0;
    ctl->n_run = 0;
    ctl->work_next = 0;
  }
  // the loop state, read once per block
  // the second layer's weights of an attached network, for every pass
  uint4* staged = reinterpret_cast<uint4*>(smem + P.mlp_w2_off);
  if (P.mlp_w2_off > 0)
    for (int i = (int)threadIdx.x; i < MLP_W2_SMEM / 16; i += (int)blockDim.x)
      staged[staged_index(i)] = __ldg(reinterpret_cast<const uint4*>(P.mlp_W2) + i);
  if (threadIdx.x == 0) {
    sh.bcast[0] = ctl->n_nodes;
    sh.bcast[1] = ctl->iteration;
  }
  __syncthreads();
  int n_tree = sh.bcast[0];
  uint32_t it = (uint32_t)sh.bcast[1];
  const int nch = P.nch;

  // V_E list from the stored node sets
  count_ve(P, T, n_tree, sh);
  if (!team_sync(T, ctl, P.wait_ns, 10)) return false;
  int n_ve = write_ve(P, T, n_tree, sh);
  if (!team_sync(T, ctl, P.wait_ns, 11)) return false;
  int lam = eq6_lambda(P.t_e, n_tree, n_ve, P.lambda_max);
  if (n_ve > 0 && lam == 0) {
    if (T.b == 0 && threadIdx.x == 0) {
      ctl->state = KP_DEV_FULL;
      ctl->n_ve = n_ve;
    }
    return true;
  }

  int run = 0;
  // block 0 stamps the device clock between phases and barriers
  const bool timer = T.b == 0 && threadIdx.x == 0;
  uint64_t t_mark = timer ? global_ns() : 0;
  int32_t* phase_ns = sh.phase_ns;
  int32_t prev_wait = 0;
  auto stamp = [&](int ph) {
    if (timer) {
      const uint64_t now = global_ns();
      phase_ns[ph] = (int32_t)(now - t_mark);
      t_mark = now;
    }
  };
  unsigned char* mtile = smem + P.blob_bytes + P.sd_bytes;
  for (;;) {
    if (P.features_on) {
      phase_features(P, T, n_ve, mtile, staged);
      stamp(3);
      if (!team_sync(T, ctl, P.wait_ns, 19)) return false;
      stamp(6);
    } else if (timer) {
      phase_ns[3] = phase_ns[6] = 0;
    }
    const int S = n_ve > 0 ? n_ve * lam : 0;
    const KeyDiv kd(lam);
    phase_expand<SYS, LOG>(P, T, smem, it, kd, S, sh);
    stamp(0);
    if (!team_sync(T, ctl, P.wait_ns, 20)) return false;
    stamp(1);
    phase_accept<LOG>(P, T, S, nch, sh);
    stamp(2);
    if (!team_sync(T, ctl, P.wait_ns, 21)) return false;
    stamp(4);
    if (timer) phase_ns[5] = phase_ns[7] = 0;
    const int t_old = n_tree;
    int n_acc;
    phase_nodesets<SYS, LOG>(P, T, it, t_old, kd, sh, &n_acc, smem);
    n_tree = t_old + n_acc;
    stamp(8);
    if (!team_sync(T, ctl, P.wait_ns, 23)) return false;
    stamp(9);
    const int ve_prev = n_ve, lam_prev = lam;
    // the pass's goal node and any error raised before the barrier above:
    // every block reads the same words, beside the counts of the V_E list
    int goal_now = 0, err_now = 0;
    if (threadIdx.x == 0) {
      goal_now = *((volatile int*)&ctl->goal_node);
      err_now = *((volatile int*)&ctl->err);
    }
    n_ve = write_ve(P, T, n_tree, sh, goal_now, err_now);
    lam = eq6_lambda(P.t_e, n_tree, n_ve, P.lambda_max);
    ++run;
    const int goal = sh.goal;
    if (sh.err != 0) return false;
    const bool solved = goal != KP_NO_GOAL;
    const bool full = n_ve > 0 && lam == 0;
    int stop = solved || full || run >= max_iters ? 1 : 0;
    if (T.b == 0 && threadIdx.x == 0) {
      if (run <= P.stats_cap && P.stats) {
        KStats s;
        s.iteration = (int)it;
        s.n_ve = ve_prev;
        s.lambda = lam_prev;
        s.n_samples = S;
        s.n_valid = (int)*((volatile uint32_t*)&ctl->it_valid);
        s.n_accepted = n_acc;
        s.n_nodes = n_tree;
        s.goal_node = solved ? goal : -1;
        phase_ns[10] = (int32_t)(global_ns() - t_mark);
        phase_ns[11] = prev_wait;
        for (int q = 0; q < 12; ++q) s.phase_ns[q] = phase_ns[q];
        P.stats[run - 1] = s;
      }
      ctl->it_valid = 0;
      ctl->tot_samples += (unsigned long long)S;
      ctl->state = solved ? KP_DEV_SOLVED : (full ? KP_DEV_FULL : KP_DEV_RUNNING);
      // a time limit ends the loop by block 0's clock
      if (max_ns > 0) ctl->stop = stop || global_ns() - t_start >= max_ns ? 1 : 0;
    }
    ++it;
    const uint64_t t_l = timer ? global_ns() : 0;
    if (!team_sync(T, ctl, P.wait_ns, 24, max_ns > 0 ? &ctl->stop : nullptr, &stop)) return false;
    if (timer) {
      t_mark = global_ns();
      prev_wait = (int32_t)(t_mark - t_l);  // reported with the next pass
    }
    if (stop) break;
  }
  if (T.b == 0 && threadIdx.x == 0) {
    ctl->n_nodes = n_tree;
    ctl->n_ve = n_ve;
    ctl->iteration = (int)it;
    ctl->n_run = run;
  }
  return true;
}

// n bytes at p set to the 16-byte pattern v, by 16-byte stores (every table
// slice of the arena starts on 256 bytes and is padded to a multiple of
// 256, so the last store stays inside the slice).
__device__ __forceinline__ void fill_slice(void* p, size_t n, uint4 v, size_t tid, size_t nth) {
  uint4* q = reinterpret_cast<uint4*>(p);
  const size_t n16 = (n + 15) / 16;
  for (size_t i = tid; i < n16; i += nth) q[i] = v;
}

template <int SYS>
__device__ void init_root(const KParams& P, const RootState& root, bool box_free);

// Whether the root's position lies in no obstacle box (closed boxes, the
// test the hull check makes with a hull of one point), by the whole block:
// thread t tests boxes t, t + blockDim.x, ...  Every thread of the block
// calls it and gets the answer.
__device__ __forceinline__ bool root_box_free(const KParams& P, const RootState& root) {
  const float4* gb = reinterpret_cast<const float4*>(P.boxes);
  const float px = root.x[0], py = root.x[1], pz = root.x[2];
  bool hit = false;
  for (int b = (int)threadIdx.x; b < P.n_boxes_pad; b += (int)blockDim.x) {
    const float4 bl = gb[2 * b], bh = gb[2 * b + 1];
    hit |= (px <= bh.x) & (bl.x <= px) & (py <= bh.y) & (bl.y <= py) & (pz <= bh.z) &
           (bl.z <= pz);
  }
  return __syncthreads_or(hit) == 0;
}

// The region and sub-region tables of Algorithm 1's initialisation, cleared
// by the whole team: visited 0, claims 2^32 - 1, counters 0, R_avail empty,
// P_accept = 1 as the threshold 2^32.
__device__ __forceinline__ void clear_tables(const KParams& P, size_t tid, size_t nth) {
  const size_t R = (size_t)P.R, n_sub = R * (size_t)P.n_sub_per;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  fill_slice(P.visited, n_sub, zero, tid, nth);
  fill_slice(P.claim, n_sub * 4, make_uint4(~0u, ~0u, ~0u, ~0u), tid, nth);
  fill_slice(P.n_valid, R * 4, zero, tid, nth);
  fill_slice(P.n_invalid, R * 4, zero, tid, nth);
  fill_slice(P.cov, R * 4, zero, tid, nth);
  fill_slice(P.avail, R, zero, tid, nth);
  fill_slice(P.thr, R * 8, make_uint4(0u, 1u, 0u, 1u), tid, nth);  // 2^32 each
}

// Algorithm 1's initialisation inside the loop launch: the team clears the
// tables, then block 0 writes the root (which also clears the control
// block's error word, so neither barrier here reads it).
template <int SYS>
__device__ __forceinline__ bool reset_in_launch(const KParams& P, const Team& T,
                                                const RootState& root) {
  clear_tables(P, (size_t)T.b * blockDim.x + threadIdx.x, (size_t)T.nb * blockDim.x);
  const bool box_free = T.b == 0 ? root_box_free(P, root) : false;
  if (!team_sync(T, P.ctl, P.wait_ns, 50, nullptr, nullptr, false)) return false;
  if (T.b == 0 && threadIdx.x == 0) init_root<SYS>(P, root, box_free);
  return team_sync(T, P.ctl, P.wait_ns, 51, nullptr, nullptr, false);
}

// Root-to-goal chain into P.traj rows (state 12, control 4, steps), root
// first; ctl->n_edges its length, -1 without a goal node (rows are written
// for at most KP_TRAJ_ROWS edges).  Run by every thread of one block:
// thread 0 walks the chain once from the goal and keeps the node ids in
// ids[0 .. cap), then the block writes the rows in parallel; a chain longer
// than cap is written by thread 0 on a second walk.
template <int SYS>
__device__ void extract_chain_block(const KParams& P, int* ids, int cap) {
  constexpr int D = System<SYS>::D, N = System<SYS>::N;
  KCtl* ctl = P.ctl;
  __shared__ int s_len;
  if (threadIdx.x == 0) {
    const int g = ctl->goal_node;
    int len = -1;
    if (g != KP_NO_GOAL && g >= 0 && g < P.t_e) {
      len = 0;
      for (int v = g; v > 0 && len <= P.t_e; v = P.parent[v]) {
        if (len < cap) ids[len] = v;
        ++len;
      }
    }
    ctl->n_edges = len;
    s_len = len;
  }
  __syncthreads();
  const int len = s_len;
  if (len <= 0 || len > KP_TRAJ_ROWS) return;
  auto write_row = [&](int row, int v) {
    float* out = P.traj + (size_t)row * 17;
#pragma unroll
    for (int i = 0; i < 12; ++i) out[i] = i < D ? P.st[(size_t)i * P.t_e + v] : 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) out[12 + i] = i < N ? P.ctrl[(size_t)i * P.t_e + v] : 0.0f;
    out[16] = (float)P.steps[v];
  };
  if (len <= cap) {
    for (int e = (int)threadIdx.x; e < len; e += (int)blockDim.x) write_row(len - 1 - e, ids[e]);
  } else if (threadIdx.x == 0) {
    int row = len - 1;
    for (int v = ctl->goal_node; v > 0 && row >= 0; v = P.parent[v], --row) write_row(row, v);
  }
}

// Single-query launch: the whole grid is one team.  mode: KP_LOOP_RESET
// runs Algorithm 1's initialisation from 'root' first, KP_LOOP_EXTRACT
// writes the root-to-goal chain after the passes (block 0, the ids kept in
// the dynamic shared memory the passes no longer use).
template <int SYS, bool LOG>
__global__ void __launch_bounds__(KP_BLOCK, KP_MIN_BLOCKS)
    kp_loop_kernel(KParams P, int max_iters, uint64_t max_ns, RootState root, int mode) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ LoopShared sh;
  KCtl* ctl = P.ctl;
  const Team T{(int)blockIdx.x, (int)gridDim.x, &ctl->bar};
  if ((mode & KP_LOOP_RESET) && !reset_in_launch<SYS>(P, T, root)) return;
  if (ctl->state == KP_DEV_RUNNING) {
    if (!stage_boxes(P, reinterpret_cast<float4*>(smem), sh)) return;
    if (!run_loop<SYS, LOG>(P, T, smem, sh, max_iters, max_ns)) return;
  } else if (blockIdx.x == 0 && threadIdx.x == 0) {
    ctl->n_run = 0;
  }
  if ((mode & KP_LOOP_EXTRACT) && blockIdx.x == 0) {
    __syncthreads();
    int cap = (int)(((size_t)P.blob_bytes + (size_t)P.sd_bytes) / 4);
    if (P.extract_cap > 0 && P.extract_cap < cap) cap = P.extract_cap;
    extract_chain_block<SYS>(P, reinterpret_cast<int*>(smem), cap);
  }
}

// Root of a query (thread 0): x_init checked (state box; box_free: no
// obstacle box contains it, root_box_free) and binned; tree, decomposition
// and control block set to Algorithm 1, initialisation.  Thresholds and
// cleared tables are the caller's.
template <int SYS>
__device__ void init_root(const KParams& P, const RootState& root, bool box_free) {
  using Sys = System<SYS>;
  constexpr int D = Sys::D;
  KCtl* ctl = P.ctl;
  float x[D];
  for (int i = 0; i < D; ++i) x[i] = root.x[i];
  bool ok = in_state_box<Sys>(x, P) && box_free;
  ctl->n_run = 0;
  ctl->stop = 0;
  ctl->it_valid = 0;
  ctl->err = 0;
  ctl->err_where = 0;
  ctl->iteration = 0;
  ctl->n_edges = 0;
  ctl->tot_samples = 0;
  ctl->tot_steps = 0;
  ctl->tot_hull = 0;
  ctl->tot_box_tests = 0;
  ctl->tot_batches = 0;
  ctl->tot_refills = 0;
  ctl->work_next = 0;
  if (!ok) {
    ctl->state = KP_DEV_BAD_ROOT;
    ctl->n_nodes = 0;
    ctl->n_ve = 0;
    ctl->goal_node = KP_NO_GOAL;
    return;
  }
  int r, s;
  bin_state<SYS>(x, P, &r, &s);
  for (int i = 0; i < D; ++i) P.st[(size_t)i * P.t_e] = x[i];
  for (int i = 0; i < Sys::N; ++i) P.ctrl[(size_t)i * P.t_e] = 0.0f;
  P.parent[0] = -1;
  P.steps[0] = 0;
  P.region[0] = r;
  P.node_sub[0] = s;
  P.in_ve[0] = 1;
  P.visited[s] = 1;
  P.cov[r] = 1;
  P.avail[r] = 1;
  ctl->n_nodes = 1;
  ctl->n_ve = 1;
  const float dx = x[0] - P.goal_c[0], dy = x[1] - P.goal_c[1], dz = x[2] - P.goal_c[2];
  const bool in_goal = dx * dx + dy * dy + dz * dz <= P.goal_r2;
  ctl->goal_node = in_goal ? 0 : KP_NO_GOAL;
  ctl->state = in_goal ? KP_DEV_SOLVED : KP_DEV_RUNNING;
}

// Algorithm 1, initialisation, as a launch of its own (kp_reset; a query does
// it inside its loop launch): every block clears its share of the tables
// (clear_tables); the last block to finish (a counter taken after a fence)
// writes the root, so the root's table entries come after every clear.
template <int SYS>
__global__ void kp_reset_kernel(KParams P, RootState root) {
  clear_tables(P, (size_t)blockIdx.x * blockDim.x + threadIdx.x, (size_t)gridDim.x * blockDim.x);
  __shared__ int last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(&P.ctl->reset_done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  const bool box_free = root_box_free(P, root);
  if (threadIdx.x != 0) return;
  __threadfence();
  P.ctl->reset_done = 0;
  P.ctl->bar = 0;
  init_root<SYS>(P, root, box_free);
}

}  // namespace kp
