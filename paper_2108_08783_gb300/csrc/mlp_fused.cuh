// Whole-network kernels of the warm-start MLP for hidden widths up to 256
// (two 128-row accumulator tiles) and n_in, n_out <= 16: the forward pass in
// one launch, and a training step in three (forward + back-propagation,
// weight gradients, optimiser).  Included by mlp.cu inside its namespace.
//
// Activations are held transposed: a tile of NB batch rows is the N extent of
// every MMA and the layer's output features are its M extent, so a thread of
// the epilogue owns one feature (its bias is one register) and writes 8
// consecutive batch rows of it as one 16-byte store, without bank conflicts.
// Every operand image is made of 8 x 8 core matrices of 128 contiguous bytes
// (no swizzle), and each image serves two contractions by the descriptor's
// transpose bits and strides alone:
//   weights W_l, core (cg, rg) holding 8 rows (out features) of 8 columns (in
//     features), column groups outermost: K-major A of the forward product
//     (M = rows, K = columns) and MN-major A of the input error (M = columns,
//     K = rows); any run of columns is one contiguous block;
//   activations h_l and errors delta_l, core (fg, ng) holding 8 features of 8
//     batch rows: MN-major B of the products above (N = rows, K = features)
//     and K-major A or B of the weight gradient (K = batch rows).
// The contractions run over K in the same 16-wide steps as k_gemm does, and
// the epilogues round the same quantities, so the results are the same bits.
#pragma once

constexpr int kFusedWidth = 256;
constexpr int kFusedLayers = 16;
constexpr int kFwdRows = 128;        // batch rows of a forward tile, at most
constexpr int kTrainRows = 64;       // batch rows of a training tile, at most
constexpr int kCoreBytes = 128;

__host__ __device__ constexpr int pad16(int v) { return (v + 15) & ~15; }

struct FusedLayer {
  int32_t rows, cols;    // W_l is [rows][cols]
  int32_t rg, cg;        // 8-groups of the padded rows and columns (even)
  uint32_t pack;         // byte offset of the layer's image in the packed weights
  uint32_t b_off;        // offset of b_l in the parameter vector
  uint32_t w_off;        // offset of W_l in the parameter vector
};

struct FusedNet {
  FusedLayer l[kFusedLayers];
  int32_t n_layers, n_in, n_out;
  const unsigned char* wpack;
  const float* theta;  // biases
  int* err;
};

// ---------------------------------------------------------------- primitives

__device__ __forceinline__ void mbar_init_n(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void copy_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(saddr(dst)),
      "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(saddr(bar))
      : "memory");
}
__device__ __forceinline__ void copy_s2g(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                   __cvta_generic_to_global(dst)),
               "r"(saddr(src)), "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void copies_read() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void copies_done() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ void fence_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          saddr(bar))
      : "memory");
}
__device__ __forceinline__ void tc_alloc(uint32_t* where, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   saddr(where)),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_free(uint32_t tmem, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols)
               : "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc ? 1u : 0u)
      : "memory");
}
// The loads are collective (.sync.aligned): the warp is brought together first,
// as loops issue them after branches by lane.
__device__ __forceinline__ void tc_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
      "%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Matrix descriptor of an unswizzled image: k_stride (leading byte offset)
// between core matrices along K, mn_stride (stride byte offset) along M or N.
__device__ __forceinline__ uint64_t core_desc(uint32_t addr, uint32_t k_stride, uint32_t mn_stride) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(k_stride >> 4) << 16) |
         ((uint64_t)(mn_stride >> 4) << 32) | ((uint64_t)1 << 46);
}
// Instruction descriptor of a 128 x n x 16 bf16 MMA with FP32 accumulation;
// ta, tb: A, B stored MN-major.
__device__ __forceinline__ uint32_t mma_desc(int n, bool ta, bool tb) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((ta ? 1u : 0u) << 15) | ((tb ? 1u : 0u) << 16) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
// Two floats rounded to bfloat16 (to nearest even), lo in the low half.
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  uint32_t w;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w) : "f"(hi), "f"(lo));
  return w;
}
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// A tile's inputs as an image (2 feature groups, nb / 8 row groups): x rounded
// to bfloat16, zero for features >= n_in and rows >= valid.
__device__ __forceinline__ void stage_inputs(unsigned char* image, const float* x, int64_t row0,
                                             int valid, int n_in, int nb, int tid, int threads) {
  for (int e = tid; e < nb * 16; e += threads) {
    const int n = e >> 4, k = e & 15;
    const float v = (n < valid && k < n_in) ? __ldg(x + (row0 + n) * n_in + k) : 0.0f;
    *reinterpret_cast<bf16*>(image + (k >> 3) * nb * 16 + (n >> 3) * kCoreBytes + (k & 7) * 16 +
                             (n & 7) * 2) = __float2bfloat16_rn(v);
  }
}

// --------------------------------------------------------------- forward pass
// y = network(x) for n rows.  A CTA takes tiles of nb <= 128 rows through all
// layers: the activations stay in shared memory (64 KB, overwritten in place
// once a layer's MMAs have read them), the packed weights stream from L2
// through a ring of 16 KB stages (32 input features of the layer's rows each, one
// bulk copy: 32 copies of 512 bytes a stage held the products back to half rate).
// Warps 0-7 are the epilogue, warp 8 fills the ring, one lane of warp 9 issues
// the MMAs.  Its epilogues bound it (50 M tanhf for 65,536 rows of the 4 x 256
// network), by latency as much as by instructions: 56 % of the issue slots are
// used at 30 % of the warps, 4.5 stalls an issue wait for a tensor-memory or
// global load (each warp has one load of 8 columns in flight), and a tanh of half
// the instructions gained nothing.  So two CTAs share an SM (2 x 112 KB of shared
// memory, 2 x 256 accumulator columns): one's products run under the other's
// epilogue.  nb is chosen so that the tiles fill whole rounds of 2 CTAs per SM.
// 65,536 rows of the 4 x 256 network: 219 us layer by layer, 59 us so; the
// pass of a warm start of 926,000 sites (227 chunks of 4,096 rows before, about
// 20 ms): 0.72 ms, at 2.4 warp instructions a cycle and SM.
constexpr int kFwdStages = 3;
constexpr int kStageBytes = 32 * 4 * kCoreBytes;  // 256 rows x 32 columns
constexpr int kFwdEpiWarps = 8;  // 8 or 16 (16 measured no faster)
constexpr int kFwdThreads = (kFwdEpiWarps + 2) * 32;
constexpr uint32_t kFwdTmem = 256;
constexpr int kFwdSmem = 32 * (kFwdRows / 8) * kCoreBytes + kFwdStages * kStageBytes + 128;

struct FwdBars {
  uint64_t full[kFwdStages], empty[kFwdStages], acc, ready;
  uint32_t tmem;
};

__global__ void __launch_bounds__(kFwdThreads, 2)
    k_mlp_forward(const __grid_constant__ FusedNet net, const float* x, int64_t n, int nb, float* y) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* act = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~(uintptr_t)127);
  unsigned char* ring = act + 32 * (kFwdRows / 8) * kCoreBytes;
  __shared__ __align__(8) FwdBars s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == kFwdEpiWarps + 1) tc_alloc(&s.tmem, kFwdTmem);
  if (tid == 0) {
    for (int i = 0; i < kFwdStages; ++i) {
      mbar_init_n(&s.full[i], 1);
      mbar_init_n(&s.empty[i], 1);
    }
    mbar_init_n(&s.acc, 1);
    mbar_init_n(&s.ready, kFwdEpiWarps * 32);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = s.tmem;
  const int64_t tiles = (n + nb - 1) / nb;
  const uint32_t kstr = (uint32_t)nb * 16;  // feature-group stride of the activations

  if (warp == kFwdEpiWarps) {
    // ring producer: chunks of 4 column groups of every layer of every tile
    uint32_t it = 0;
    bool ok = true;
    for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x)
      for (int l = 0; l < net.n_layers && ok; ++l) {
        const FusedLayer& L = net.l[l];
        for (int c = 0; c < L.cg; c += 4, ++it) {
          const uint32_t st = it % kFwdStages, use = it / kFwdStages;
          if (use > 0 && !__all_sync(0xffffffffu, mbar_wait(&s.empty[st], (use - 1) & 1u))) {
            ok = false;
            break;
          }
          const uint32_t bytes = (uint32_t)(min(4, L.cg - c) * L.rg) * kCoreBytes;
          if (lane == 0) {
            mbar_expect(&s.full[st], bytes);
            copy_g2s(ring + st * kStageBytes, net.wpack + L.pack + (uint32_t)(c * L.rg) * kCoreBytes,
                     bytes, &s.full[st]);
          }
        }
      }
    if (!ok) {
      if (lane == 0) atomicOr(net.err, 1);
      // copies in flight get one more (bounded) chance to land
      for (int i = 0; i < kFwdStages; ++i) mbar_wait(&s.full[i], 0);
    }
  } else if (warp == kFwdEpiWarps + 1) {
    if (lane == 0) {
      uint32_t it = 0, step = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x)
        for (int l = 0; l < net.n_layers && ok; ++l, ++step) {
          const FusedLayer& L = net.l[l];
          const int mt = (L.rg + 15) / 16;
          const uint32_t idesc = mma_desc(nb, false, true);
          const uint32_t rstr = (uint32_t)L.rg * kCoreBytes;  // column-group stride
          ok = mbar_wait(&s.ready, step & 1u);
          tc_after();
          for (int c = 0; c < L.cg && ok; c += 4, ++it) {
            const uint32_t st = it % kFwdStages;
            ok = mbar_wait(&s.full[st], (it / kFwdStages) & 1u);
            if (!ok) break;
            const uint32_t a0 = saddr(ring + st * kStageBytes);
            for (int m = 0; m < mt; ++m)
              for (int k = 0; k < 4 && c + k < L.cg; k += 2)
                tc_mma(tmem + (uint32_t)(m * nb),
                       core_desc(a0 + (uint32_t)(m * 16) * kCoreBytes + k * rstr, rstr, kCoreBytes),
                       core_desc(saddr(act) + (uint32_t)(c + k) * kstr, kstr, kCoreBytes), idesc,
                       c + k > 0);
            tc_commit(&s.empty[st]);
          }
          if (ok) tc_commit(&s.acc);
        }
      if (!ok) atomicOr(net.err, 1);
    }
    __syncwarp();
  } else {
    constexpr int kRowsets = kFwdEpiWarps / 4;  // warps of each 32-feature row set
    const int q = warp & 3, set = warp >> 2;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    uint32_t step = 0;
    bool ok = true;
    for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      const int64_t row0 = t * nb;
      const int valid = (int)(n - row0 < nb ? n - row0 : nb);
      stage_inputs(act, x, row0, valid, net.n_in, nb, tid, kFwdEpiWarps * 32);
      fence_async();
      tc_before();
      mbar_arrive(&s.ready);
      for (int l = 0; l < net.n_layers; ++l, ++step) {
        const FusedLayer& L = net.l[l];
        const bool last = l + 1 == net.n_layers;
        // two accumulator tiles: half of the row sets each, and the 8-row column
        // groups dealt out among the warps of a row set
        const bool two = L.rg > 16;
        const int part = two ? set >> 1 : set, parts = two ? kRowsets / 2 : kRowsets;
        const int f = (two ? (set & 1) * 128 : 0) + q * 32 + lane;
        const float bias = f < L.rows ? __ldg(net.theta + L.b_off + f) : 0.0f;
        if (!__all_sync(0xffffffffu, mbar_wait(&s.acc, step & 1u))) {
          ok = false;
          break;
        }
        tc_after();
        const uint32_t base = lane_addr + (two ? (uint32_t)((set & 1) * nb) : 0u);
        if (last) {
          if (q == 0)
            for (int c0 = part * 8; c0 < nb; c0 += parts * 8) {
              float v[8];
              tc_ld8(base + c0, v);
              if (lane < net.n_out) {
                float* o = y + (row0 + c0) * net.n_out + lane;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                  if (c0 + j < valid) o[j * net.n_out] = v[j] + bias;
              }
            }
        } else {
          const bool keep = f < L.rg * 8;  // features the next layer reads
          unsigned char* row = act + (f >> 3) * kstr + (f & 7) * 16;
          for (int c0 = part * 8; c0 < nb; c0 += parts * 8) {
            float v[8];
            tc_ld8(base + c0, v);
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
              w[j] = bf16_pair(tanhf(v[2 * j] + bias), tanhf(v[2 * j + 1] + bias));
            // predicated, not skipped: lanes that went ahead would be waited for at
            // the next load (61.4 us for 65,536 rows with a branch here, 59.4 so)
            if (keep)
              *reinterpret_cast<uint4*>(row + (c0 >> 3) * kCoreBytes) =
                  make_uint4(w[0], w[1], w[2], w[3]);
          }
          fence_async();
          tc_before();
          mbar_arrive(&s.ready);
        }
      }
    }
    if (!ok && lane == 0) atomicOr(net.err, 1);
  }
  tc_before();
  __syncthreads();
  if (warp == kFwdEpiWarps + 1) {
    tc_after();
    tc_free(tmem, kFwdTmem);
  }
}

// ------------------------------------------------- forward + back-propagation
// One CTA per SM takes tiles of nb <= 64 batch rows through the network and
// back.  All activations of the tile stay in shared memory, and the error of a
// hidden layer replaces its activations in place; a layer's whole weight image
// (<= 128 KB) is copied in once its predecessor's MMAs are done, under the
// epilogue.  The images of activations and errors also leave for device memory
// as bulk copies, as the operands of k_mlp_wgrad.  Small tiles (32 rows for a
// batch of 4,096) spread the tanhf over all SMs: what bounds a step at the
// study's batch is the chain of 2 n_layers - 1 dependent products.  A training
// step of 4,096 rows of the 4 x 256 network, all kernels: 1,134 us layer by
// layer, 45 us so (this kernel 22, the weight gradients 12, the optimiser 8).
constexpr int kTrainEpiWarps = 16;
constexpr int kTrainThreads = (kTrainEpiWarps + 2) * 32;
constexpr uint32_t kTrainTmem = 128;

struct TrainArgs {
  FusedNet net;
  const float* x;
  const float* t;
  int64_t n;
  int32_t nb;
  int32_t w_bytes;          // weight buffer
  float scale;              // 2 / count
  double inv_count;
  unsigned char* h[kFusedLayers];  // images of h_l, tile after tile
  unsigned char* d[kFusedLayers];  // images of delta_l
  double* loss_part;        // [tiles][4]
};

// Waits see a phase by its parity only, so no barrier may run two phases ahead
// of a thread that waits on it.  `ready` (a product's operand is staged) and
// `acc` (it is computed) alternate; delta_0, which no product follows, has a
// barrier of its own: on `ready` the next tile's inputs could complete a second
// phase before the product warp had seen the first, and it would wait for ever.
struct TrainBars {
  uint64_t w_full, acc, ready, tail;
  uint32_t tmem;
};

__global__ void __launch_bounds__(kTrainThreads, 1)
    k_mlp_train(const __grid_constant__ TrainArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const FusedNet& net = a.net;
  const int nb = a.nb, NL = net.n_layers;
  const uint32_t kstr = (uint32_t)nb * 16;
  unsigned char* wbuf = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~(uintptr_t)127);
  // images: x, then h_1 .. h_{L-1} (later delta_0 .. delta_{L-2}), then delta_{L-1}
  unsigned char* const img0 = wbuf + a.w_bytes;
  const uint32_t hidden = (uint32_t)net.l[0].rg * kstr;  // every hidden layer has the same width
  auto image = [&](int l) { return l == 0 ? img0 : img0 + 2 * kstr + (uint32_t)(l - 1) * hidden; };
  __shared__ __align__(8) TrainBars s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == kTrainEpiWarps) tc_alloc(&s.tmem, kTrainTmem);
  if (tid == 0) {
    mbar_init_n(&s.w_full, 1);
    mbar_init_n(&s.acc, 1);
    mbar_init_n(&s.ready, kTrainEpiWarps * 32);
    mbar_init_n(&s.tail, kTrainEpiWarps * 32);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = s.tmem;
  const int64_t tiles = (a.n + nb - 1) / nb;
  const int ops = 2 * NL - 1;  // products of a tile: forward 0 .. L-1, back L-1 .. 1

  if (warp == kTrainEpiWarps) {
    // weights: op g needs layer g (forward) or 2 L - 1 - g (back); the first
    // product of the way back uses the layer already there
    if (lane == 0) {
      bool ok = true;
      uint32_t done = 0;  // products issued and waited for
      for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x)
        for (int g = 0; g < ops && ok; ++g, ++done) {
          // the previous product has read the buffer
          if (done > 0 && !mbar_wait(&s.acc, (done - 1) & 1u)) {
            ok = false;
            break;
          }
          if (g == NL) {  // the layer is there: keeps the product and this loop in step
            mbar_arrive(&s.w_full);
            continue;
          }
          const FusedLayer& L = net.l[g < NL ? g : 2 * NL - 1 - g];
          const uint32_t bytes = (uint32_t)(L.rg * L.cg) * kCoreBytes;
          mbar_expect(&s.w_full, bytes);
          for (uint32_t o = 0; o < bytes; o += 16384)
            copy_g2s(wbuf + o, net.wpack + L.pack + o, min(16384u, bytes - o), &s.w_full);
        }
      if (!ok) atomicOr(net.err, 1);
    }
    __syncwarp();
  } else if (warp == kTrainEpiWarps + 1) {
    if (lane == 0) {
      bool ok = true;
      uint32_t rd = 0, wf = 0, tl = 0;
      for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        for (int g = 0; g < ops; ++g) {
          ok = mbar_wait(&s.ready, rd++ & 1u) && mbar_wait(&s.w_full, wf++ & 1u);
          if (!ok) break;
          tc_after();
          // images leaving earlier have been read before this product's
          // epilogue overwrites one of them
          if (g == 0 || g >= NL) copies_read();
          const bool fwd = g < NL;
          const int l = fwd ? g : 2 * NL - 1 - g;
          const FusedLayer& L = net.l[l];
          unsigned char* b = fwd ? image(l) : image(l + 1);
          const uint32_t bytes = (uint32_t)(fwd ? L.cg : L.rg) * kstr;
          const int mt = ((fwd ? L.rg : L.cg) + 15) / 16, ks = fwd ? L.cg : L.rg;
          const uint32_t rstr = (uint32_t)L.rg * kCoreBytes;  // column-group stride
          const uint32_t idesc = mma_desc(nb, !fwd, true);
          for (int m = 0; m < mt; ++m)
            for (int k = 0; k < ks; k += 2) {
              const uint64_t ad =
                  fwd ? core_desc(saddr(wbuf) + (uint32_t)(m * 16) * kCoreBytes + k * rstr, rstr,
                                  kCoreBytes)
                      : core_desc(saddr(wbuf) + (uint32_t)(m * 16) * rstr + k * kCoreBytes,
                                  kCoreBytes, rstr);
              tc_mma(tmem + (uint32_t)(m * nb), ad, core_desc(saddr(b) + k * kstr, kstr, kCoreBytes),
                     idesc, k > 0);
            }
          tc_commit(&s.acc);
          copy_s2g((fwd ? a.h[l] : a.d[l]) + t * bytes, b, bytes);
        }
        // delta_0, ready after the last product's epilogue
        if (ok) ok = mbar_wait(&s.tail, tl++ & 1u);
        if (ok) {
          const uint32_t bytes = (uint32_t)net.l[0].rg * kstr;
          copy_s2g(a.d[0] + t * bytes, image(1), bytes);
        }
      }
      copies_done();
      if (!ok) atomicOr(net.err, 1);
    }
    __syncwarp();
  } else {
    const int q = warp & 3, quarter = warp >> 2;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    uint32_t step = 0;
    bool ok = true;
    auto wait_acc = [&]() {
      ok = __all_sync(0xffffffffu, mbar_wait(&s.acc, step & 1u));
      ++step;
      tc_after();
      return ok;
    };
    auto publish = [&](uint64_t* bar) {
      fence_async();
      tc_before();
      mbar_arrive(bar);
    };
    for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      const int64_t row0 = t * nb;
      const int valid = (int)(a.n - row0 < nb ? a.n - row0 : nb);
      stage_inputs(image(0), a.x, row0, valid, net.n_in, nb, tid, kTrainEpiWarps * 32);
      publish(&s.ready);
      // hidden layers: two accumulator tiles, two warps of 8-row column groups
      // each (one tile: four)
      const bool two = net.l[0].rg > 16;
      const int f = (two ? (quarter & 1) * 128 : 0) + q * 32 + lane;
      const int part = two ? quarter >> 1 : quarter, parts = two ? 2 : 4;
      const bool keep = f < net.l[0].rg * 8;
      const uint32_t base = lane_addr + (two ? (uint32_t)((quarter & 1) * nb) : 0u);
      const uint32_t at = (uint32_t)(f >> 3) * kstr + (f & 7) * 16;
      for (int l = 0; l + 1 < NL && ok; ++l) {
        const float bias = f < net.l[l].rows ? __ldg(net.theta + net.l[l].b_off + f) : 0.0f;
        if (!wait_acc()) break;
        unsigned char* row = image(l + 1) + at;
        for (int c = part; c < nb / 8; c += parts) {
          float v[8];
          tc_ld8(base + c * 8, v);
          if (!keep) continue;
          uint32_t w[4];
#pragma unroll
          for (int j = 0; j < 4; ++j)
            w[j] = bf16_pair(tanhf(v[2 * j] + bias), tanhf(v[2 * j + 1] + bias));
          *reinterpret_cast<uint4*>(row + c * kCoreBytes) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        publish(&s.ready);
      }
      if (!ok) break;
      // output layer: y, the loss and its error delta_{L-1} = 2 (y - t) / count
      {
        const FusedLayer& L = net.l[NL - 1];
        const bool mine = q == 0 && lane < L.rows;
        const float bias = mine ? __ldg(net.theta + L.b_off + lane) : 0.0f;
        float tt[2][8];  // nb / 8 <= 8 column groups over four warps
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int r = (quarter + 4 * i) * 8 + j;
            tt[i][j] = (mine && r < valid) ? __ldg(a.t + (row0 + r) * net.n_out + lane) : 0.0f;
          }
        if (!wait_acc()) break;
        if (q == 0) {
          float sum = 0.0f;
          unsigned char* out = image(NL) + (lane >> 3) * kstr + (lane & 7) * 16;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int c = quarter + 4 * i;
            if (c >= nb / 8) break;  // warp-uniform
            float v[8], e[8];
            tc_ld8(lane_addr + c * 8, v);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              e[j] = (mine && c * 8 + j < valid) ? (v[j] + bias) - tt[i][j] : 0.0f;
              sum += e[j] * e[j];
            }
            if (lane < 16) {
              uint32_t w[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) w[j] = bf16_pair(a.scale * e[2 * j], a.scale * e[2 * j + 1]);
              *reinterpret_cast<uint4*>(out + c * kCoreBytes) = make_uint4(w[0], w[1], w[2], w[3]);
            }
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
          if (lane == 0) a.loss_part[t * 4 + quarter] = (double)sum * a.inv_count;
        }
        publish(&s.ready);
      }
      // way back: delta_{l-1} = (delta_l W_l)(1 - h_l^2) over h_l
      for (int l = NL - 1; l >= 1 && ok; --l) {
        if (!wait_acc()) break;
        unsigned char* row = image(l) + at;
        for (int c = part; c < nb / 8; c += parts) {
          float v[8];
          tc_ld8(base + c * 8, v);
          if (!keep) continue;
          uint4* p = reinterpret_cast<uint4*>(row + c * kCoreBytes);
          const uint4 hw = *p;
          const uint32_t h[4] = {hw.x, hw.y, hw.z, hw.w};
          uint32_t w[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float h0 = bf16_lo(h[j]), h1 = bf16_hi(h[j]);
            w[j] = bf16_pair(v[2 * j] * (1.0f - h0 * h0), v[2 * j + 1] * (1.0f - h1 * h1));
          }
          *p = make_uint4(w[0], w[1], w[2], w[3]);
        }
        publish(l > 1 ? &s.ready : &s.tail);
      }
    }
    if (!ok && lane == 0) atomicOr(net.err, 1);
  }
  tc_before();
  __syncthreads();
  if (warp == kTrainEpiWarps) {
    tc_after();
    tc_free(tmem, kTrainTmem);
  }
}

// ------------------------------------------------------------ weight gradients
// Partial gradients of split blockIdx.y (a run of the training tiles) for one
// 128-feature block of one layer (blockIdx.x): dW_l = delta_l^T h_l with the
// batch as the contraction, A = 128 features of delta_l and B = all of h_l
// (the output layer, with at most 16 rows, the other way round), and the
// bias gradient as FP32 sums of delta_l.  The operand images come tile by tile
// through a ring of bulk copies.  Each partial is written by one CTA, and the
// optimiser adds the splits in order: no atomics, the same gradient every run.
constexpr int kGradEpiWarps = 8;
constexpr int kGradThreads = (kGradEpiWarps + 2) * 32;
constexpr uint32_t kGradTmem = 256;
constexpr int kGradMaxStages = 8;
constexpr int kGradRing = 96 * 1024;  // two CTAs per SM

struct GradArgs {
  FusedNet net;
  const unsigned char* h[kFusedLayers];
  const unsigned char* d[kFusedLayers];
  int64_t tiles;
  int32_t nb, splits, blocks;  // blocks: 128-feature blocks per layer
  int32_t stages;
  float* part;               // [splits][part_stride]
  int64_t part_stride;       // n_params rounded up to 4: rows stay 16-byte aligned
};

struct GradBars {
  uint64_t full[kGradMaxStages], empty[kGradMaxStages], acc;
  uint32_t tmem;
};

__global__ void __launch_bounds__(kGradThreads, 2) k_mlp_wgrad(const __grid_constant__ GradArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* ring = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~(uintptr_t)127);
  __shared__ __align__(8) GradBars s;
  const FusedNet& net = a.net;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int l = blockIdx.x / a.blocks, m = blockIdx.x % a.blocks;
  const bool last = l + 1 == net.n_layers;
  const FusedLayer& L = net.l[l];
  const uint32_t kstr = (uint32_t)a.nb * 16;
  // A: 16 feature groups from group 16 m of an image of ga groups; B: gb groups
  const int ga = last ? L.cg : L.rg, gb = last ? L.rg : L.cg;
  const unsigned char* ga_p = last ? a.h[l] : a.d[l];
  const unsigned char* gb_p = last ? a.d[l] : a.h[l];
  const int na = min(16, ga - 16 * m);
  if (na <= 0) return;  // block-uniform, before any barrier
  const uint32_t a_bytes = (uint32_t)na * kstr, b_bytes = (uint32_t)gb * kstr;
  const uint32_t stage_bytes = 48u * kstr, b_at = 16u * kstr;
  const int64_t t0 = a.tiles * blockIdx.y / a.splits, t1 = a.tiles * (blockIdx.y + 1) / a.splits;
  const int nst = a.stages;
  if (warp == kGradEpiWarps + 1) tc_alloc(&s.tmem, kGradTmem);
  if (tid == 0) {
    for (int i = 0; i < nst; ++i) {
      mbar_init_n(&s.full[i], 1);
      mbar_init_n(&s.empty[i], 1 + 128);
    }
    mbar_init_n(&s.acc, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = s.tmem;
  float* part = a.part + blockIdx.y * a.part_stride;
  bool ok = true;
  if (warp == kGradEpiWarps) {
    if (lane == 0) {
      for (int64_t t = t0; t < t1; ++t) {
        const uint32_t it = (uint32_t)(t - t0), st = it % nst;
        if (it >= (uint32_t)nst && !mbar_wait(&s.empty[st], (it / nst - 1) & 1u)) {
          ok = false;
          break;
        }
        unsigned char* p = ring + st * stage_bytes;
        mbar_expect(&s.full[st], a_bytes + b_bytes);
        copy_g2s(p, ga_p + (t * ga + 16 * m) * kstr, a_bytes, &s.full[st]);
        copy_g2s(p + b_at, gb_p + t * gb * kstr, b_bytes, &s.full[st]);
      }
      if (!ok) {
        atomicOr(net.err, 1);
        for (int i = 0; i < nst; ++i) mbar_wait(&s.full[i], 0);
      }
    }
    __syncwarp();
  } else if (warp == kGradEpiWarps + 1) {
    if (lane == 0) {
      const uint32_t idesc = mma_desc(gb * 8, false, false);
      for (int64_t t = t0; t < t1; ++t) {
        const uint32_t it = (uint32_t)(t - t0), st = it % nst;
        if (!mbar_wait(&s.full[st], (it / nst) & 1u)) {
          ok = false;
          break;
        }
        const uint32_t p = saddr(ring + st * stage_bytes);
        for (int k = 0; k < a.nb / 8; k += 2)
          tc_mma(tmem, core_desc(p + k * kCoreBytes, kCoreBytes, kstr),
                 core_desc(p + b_at + k * kCoreBytes, kCoreBytes, kstr), idesc, it > 0 || k > 0);
        tc_commit(&s.empty[st]);
      }
      if (ok) tc_commit(&s.acc);
      else atomicOr(net.err, 1);
    }
    __syncwarp();
  } else {
    if (warp < 4) {
      // bias gradient: thread f adds the errors of feature f of the block (the
      // output layer: of output f, in the first block)
      const int f = tid;
      const bool mine = last ? (m == 0 && f < L.rows) : (m * 128 + f < L.rows);
      float sum = 0.0f;
      for (int64_t t = t0; t < t1; ++t) {
        const uint32_t it = (uint32_t)(t - t0), st = it % nst;
        ok = ok && mbar_wait(&s.full[st], (it / nst) & 1u);
        if (!ok) break;
        if (mine) {
          const unsigned char* p =
              ring + st * stage_bytes + (last ? b_at : 0u) + (f >> 3) * kstr + (f & 7) * 16;
          for (int c = 0; c < a.nb / 8; ++c) {
            const uint4 w = *reinterpret_cast<const uint4*>(p + c * kCoreBytes);
            sum += ((bf16_lo(w.x) + bf16_hi(w.x)) + (bf16_lo(w.y) + bf16_hi(w.y))) +
                   ((bf16_lo(w.z) + bf16_hi(w.z)) + (bf16_lo(w.w) + bf16_hi(w.w)));
          }
        }
        mbar_arrive(&s.empty[st]);
      }
      if (mine) part[L.b_off + (last ? f : m * 128 + f)] = sum;
    }
    __syncwarp();
    ok = __all_sync(0xffffffffu, ok && mbar_wait(&s.acc, 0));
    tc_after();
    if (ok) {
      const int f = m * 128 + (warp & 3) * 32 + lane;  // accumulator row = feature of A
      const uint32_t base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
      for (int c0 = (warp >> 2) * 16; c0 < gb * 8; c0 += 32) {
        float v[16];
        tc_ld16(base + c0, v);
        if (last) {
          if (f < L.cols)
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (c0 + j < L.rows) part[L.w_off + (int64_t)(c0 + j) * L.cols + f] = v[j];
        } else if (f < L.rows) {
          float* o = part + L.w_off + (int64_t)f * L.cols + c0;
          if (c0 + 16 <= L.cols && ((uintptr_t)o & 15u) == 0) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              reinterpret_cast<float4*>(o)[j] =
                  make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (c0 + j < L.cols) o[j] = v[j];
          }
        }
      }
    } else if (lane == 0) {
      atomicOr(net.err, 1);
    }
  }
  tc_before();
  __syncthreads();
  if (warp == kGradEpiWarps + 1) {
    tc_after();
    tc_free(tmem, kGradTmem);
  }
}

// Sum of a parameter's partial gradients, in the order of the splits.
__device__ __forceinline__ float grad_of(const float* part, int splits, int64_t stride, int64_t i) {
  float g = 0.0f;
#pragma unroll 8
  for (int k = 0; k < splits; ++k) g += __ldg(part + k * stride + i);
  return g;
}
// The loss from its per-tile parts, in a fixed order, by one warp.
__device__ __forceinline__ void loss_of(const double* part, int64_t n, double* loss) {
  double v = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += 32) v += part[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (threadIdx.x == 0) *loss = v;
}

__global__ void k_grad_sum(const float* part, int splits, int64_t stride, int64_t n, const double* loss_part,
                           int64_t n_loss, float* grad, double* loss) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) grad[i] = grad_of(part, splits, stride, i);
  if (blockIdx.x == 0 && threadIdx.x < 32) loss_of(loss_part, n_loss, loss);
}

// k_adam on the summed partial gradients; also writes the packed weights
// (pmap: byte offset of a weight in the images, -1 for a bias).
__global__ void k_adam_fused(float* th, const float* part, int splits, int64_t stride, float* m, float* v,
                             bf16* w16, const int32_t* pmap, unsigned char* wpack, int64_t n,
                             float lr, float b1, float b2, float eps, float c1, float c2,
                             const double* loss_part, int64_t n_loss, double* loss) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (blockIdx.x == 0 && threadIdx.x < 32) loss_of(loss_part, n_loss, loss);
  if (i >= n) return;
  const float gi = grad_of(part, splits, stride, i);
  const float mi = b1 * m[i] + (1.0f - b1) * gi;
  const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float t = th[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
  th[i] = t;
  const bf16 w = __float2bfloat16_rn(t);
  w16[i] = w;
  const int32_t q = pmap[i];
  if (q >= 0) *reinterpret_cast<bf16*>(wpack + q) = w;
}

// The packed weights from the bfloat16 parameters.
__global__ void k_pack(const bf16* w16, const int32_t* pmap, unsigned char* wpack, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && pmap[i] >= 0) *reinterpret_cast<bf16*>(wpack + pmap[i]) = w16[i];
}

// The parameters rounded to bfloat16, as a vector and packed: one launch of
// lbm_mlp_set_params (two took 4 us longer).
__global__ void k_round_pack(const float* th, bf16* w16, const int32_t* pmap, unsigned char* wpack,
                             int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const bf16 w = __float2bfloat16_rn(th[i]);
  w16[i] = w;
  const int32_t q = pmap[i];
  if (q >= 0) *reinterpret_cast<bf16*>(wpack + q) = w;
}
