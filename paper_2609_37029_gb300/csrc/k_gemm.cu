// Weight-streaming projection GEMM on the 5th-generation tensor cores (sm_103a).
//
// Every dense projection of the drafter -- boundary fusion (Sec. 2.2), the
// q/k/v, output, gate/up and down projections of each draft layer and the
// frozen LM head (Sec. 2.3) -- has a small token count M = C*B (or C) and a
// large weight: Y[m][n] = sum_k X[m][k] W[n][k].
//
// What bounds it: the weights' HBM stream, closely followed at 256 tokens by the
// tensor cores (an MMA of 128 tokens x N weights x 16 takes N / 2 cycles).  So
// that nothing else does, tokens are on the UMMA M axis (one or two accumulators of up
// to 128) and weight rows on its N axis, up to 256 of them: a k-block is 64 KB of
// loads and 256 x 256 outputs, where a tile of 128 weight rows loaded 48 KB for half
// of them and left twice as many k-blocks to wait for and commit.  N comes in
// steps of 16, so the tile width is chosen for the number of SMs (choose_width)
// and not the other way round.  Measured against that 128-row kernel (two or three CTAs an
// SM): gate/up at 256 tokens 51 -> 38 us, LM head 242 -> 224, at 16 tokens 204 -> 175
// (7.1 TB/s); 512 x 17408 x 5120 66 -> 57; the Qwen3-8B round 1046 -> 973 us.
//
//   warp 0      TMA producer of weight tiles, one k-block a stage of a ring
//   warp 10     the same for activation tiles, in a ring of its own: those come
//               from L2 in half the time, so they take fewer stages and leave
//               the shared memory to weights in flight (LM head, 256 tokens:
//               236 -> 224 us).  Up to 128 tokens the tiles are small and warp
//               0 loads them into the weights' stages: short launches end
//               0.5 us earlier
//   warp 1      TMEM allocation and the tcgen05.mma issue (one lane of a
//               uniform warp: its instructions set the issue rate)
//   warps 2-9   epilogue, two groups of four warps (one a token tile; one
//               every other chunk of a single tile): tcgen05.ld of 32 features of
//               a token row a thread, staged in shared memory (128-byte
//               swizzle) and written by TMA tensor stores; SwiGLU needs no
//               exchange, a thread holds a token's gate and up columns
//
// Grid: one CTA per work item (weight tile x token group x k split), or one per
// SM walking the items where they make more than a wave: its ring streams
// across item boundaries, so the next item's weights arrive under this one's
// epilogue.
//
// Launched as a programmatic dependent: before the preceding kernel finishes,
// the producer already streams this launch's weights (the weight halves of the
// first stages); activation loads wait for it.  Split-K partials are summed in
// split order by the consuming kernel, so results are deterministic and no CTA
// waits on another.  An output's sum runs over k in order inside one
// accumulator: neither tile width nor token tiling changes its bits.  Every
// mbarrier wait is bounded and records LSP_DEV_TIMEOUT instead of spinning
// forever.
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "lsp_internal.h"

namespace lsp {

template <typename T> struct GemmType;
template <> struct GemmType<bf16> {
  static constexpr int BK = 64;   // one 128-byte swizzle row of bf16
  static constexpr int UK = 16;   // K of one kind::f16 MMA
  static constexpr uint32_t FMT = 1;
};
template <> struct GemmType<float> {
  static constexpr int BK = 32;   // one 128-byte swizzle row of fp32 (read as tf32)
  static constexpr int UK = 8;    // K of one kind::tf32 MMA
  static constexpr uint32_t FMT = 2;
};

constexpr int kTileTok = 128;          // UMMA M: token rows of one accumulator
constexpr int kChunk = 32;             // output features of one staged store (128 bytes of fp32)
constexpr uint32_t kChunkBytes = kTileTok * 128;
constexpr int kEpiGroup = 128;         // threads of one epilogue group (named barrier 1 + group)
constexpr int kXWarp = 10;             // activation producer
constexpr int kMaxStages = 8;
static_assert(kGemmThreads == 96 + 2 * kEpiGroup, "warp 0 weights, warp 1 MMA, two epilogue groups, warp 10 activations");

// Instruction descriptor: fp32 accumulate, A/B format `fmt`, both K-major,
// N = n, M = 128.
__device__ __forceinline__ uint32_t make_idesc(int n, uint32_t fmt) {
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTileTok >> 4) << 24);
}

__device__ __forceinline__ void st_shared4(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}

// Bounded wait that also ends when another role has given up.
__device__ __forceinline__ bool gemm_wait(uint32_t bar, uint32_t parity, volatile int* stop, unsigned* err) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 31u) == 0) {
      if (*stop) return false;
      if (global_ns() - t0 > kWaitLimitNs) {
        set_err(err, LSP_DEV_TIMEOUT);
        *stop = 1;
        return false;
      }
    }
  }
}

// A work item: weight rows [row0, row0 + width) of segment `seg`, token rows
// from tok0, k-blocks [kb0, kb0 + nk) of split `split`; output column col0.
struct GemmItem {
  int seg, row0, cols, col0, tok0, split, kb0, nk;
};
__device__ __forceinline__ GemmItem gemm_item(const GemmParams& p, int item) {
  GemmItem w;
  const int per = p.n_tiles * p.tok_groups;
  w.split = item / per;
  const int r = item - w.split * per, tile = r / p.tok_groups;   // the groups of a tile are adjacent: it is shared through L2
  w.tok0 = (r - tile * p.tok_groups) * p.m_pad;
  w.seg = p.nseg > 2 && tile >= p.seg_tile0[2] ? 2 : p.nseg > 1 && tile >= p.seg_tile0[1] ? 1 : 0;
  w.row0 = (tile - p.seg_tile0[w.seg]) * p.width;
  w.cols = min(p.width, p.seg_rows[w.seg] - w.row0);
  w.col0 = p.seg_col0[w.seg] + w.row0;
  w.kb0 = (int)((long long)w.split * p.kblocks / p.splits);
  w.nk = (int)((long long)(w.split + 1) * p.kblocks / p.splits) - w.kb0;
  return w;
}

// fp32 output (final or one split's partial) of one accumulator, in chunks of
// 32 features, thread = token row.  A chunk is written to a staging buffer of
// the group (stg, nbuf of them; n counts the group's chunks) and stored by
// one thread.  Token rows past M and features past N fall outside the output
// view; a segment's last tile stops at its `cols`.
__device__ __forceinline__ void epilogue_f32(const GemmParams& p, const CUtensorMap* to, uint8_t* stg, int nbuf, int& n,
                                             uint32_t acc, const GemmItem& w, int tok0, int c_first, int c_step, int row,
                                             int bar) {
  const bool issuer = row == 0;
  const uint64_t pol_part = policy_evict_last();
  for (int c = c_first * kChunk; c < w.cols; c += c_step * kChunk, ++n) {
    float v[32];
    tmem_ld32(acc + (uint32_t)c, v);
    uint8_t* buf = stg + (size_t)(n % nbuf) * kChunkBytes;
    if (n >= nbuf && p.tma_out) {                       // the buffer's last store has read it
      if (issuer) {
        if (nbuf >= 4) bulk_wait_read<3>();
        else if (nbuf >= 2) bulk_wait_read<1>();
        else bulk_wait_read<0>();
      }
      named_bar(bar, kEpiGroup);
    }
    const uint32_t r = smem_u32(buf) + (uint32_t)row * 128u;
    if (row < p.tile_tok) {
#pragma unroll
      for (int q = 0; q < 8; ++q)
        st_shared4(r + (uint32_t)((q ^ (row & 7)) << 4), __float_as_uint(v[4 * q]), __float_as_uint(v[4 * q + 1]),
                   __float_as_uint(v[4 * q + 2]), __float_as_uint(v[4 * q + 3]));
    }
    if (p.tma_out) {
      fence_proxy_async_smem();
      named_bar(bar, kEpiGroup);
      if (issuer && tok0 < p.M) {
        if (p.mode == EPI_PARTIAL)   // read once more, by the consumer: kept in L2 past the weight stream
          tma_store_3d_hint(to, smem_u32(buf), w.col0 + c, tok0, w.split, pol_part);
        else
          tma_store_3d(to, smem_u32(buf), w.col0 + c, tok0, w.split);
      }
      if (issuer) bulk_commit();
    } else {
      // no tensor map describes Y (its row pitch or address is no multiple of
      // 16 bytes): the group's four warps take the tile's rows in turn, lanes along the
      // features.  (A warp's own 32 rows each left three of them idle at 16 tokens.)
      named_bar(bar, kEpiGroup);
      const int lane = row & 31, f = w.col0 + c + lane, rows = min(p.tile_tok, p.M - tok0);
      float* y = static_cast<float*>(p.Y) + (p.mode == EPI_PARTIAL ? (size_t)w.split * p.M * p.ldy : 0) + (size_t)tok0 * p.ldy + f;
      for (int i0 = row >> 5; i0 < rows; i0 += 16) {
        float x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + 4 * u;                       // (a row past the tile is in the buffer all the same)
          x[u] = *reinterpret_cast<const float*>(buf + (size_t)(i & (kTileTok - 1)) * 128 + (((lane >> 2) ^ (i & 7)) << 4) + (lane & 3) * 4);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i0 + 4 * u < rows && f < p.N) y[(size_t)(i0 + 4 * u) * p.ldy] = x[u];
      }
      if (nbuf == 1) named_bar(bar, kEpiGroup);           // (else the next chunk's barrier frees this buffer)
    }
  }
}

// The same for an output that no tensor map describes (its row pitch or address is no
// multiple of 16 bytes), where a CTA has one item and its ring is idle: `cb` features of
// every token row are staged where they lie against a 16-byte boundary in the output, and a
// thread a row copies the part between the boundaries in bulk.  Stores of registers
// pass about 32 bytes a cycle and SM: 206 x 30561 x 416 takes 14.6 us, 17.6 with them (11.4 by
// tensor map at N = 30560), 300 x 5001 x 2048 17.5 and 19.1.
__device__ __forceinline__ void epilogue_rows(const GemmParams& p, uint8_t* smem, uint32_t acc, const GemmItem& w, int cb, int tile,
                                              int c_first, int c_step, int row, int thread) {
  const int pitch = cb + 4;                             // floats; rows begin on 16 bytes
  const size_t out0 = (p.mode == EPI_PARTIAL ? (size_t)w.split * p.M * p.ldy : 0) + (size_t)w.tok0 * p.ldy + w.col0;
  float* stage = reinterpret_cast<float*>(smem);
  auto shift = [&](int r, int c) {                      // floats of row r, feature c past a 16-byte boundary
    return (int)((reinterpret_cast<uintptr_t>(static_cast<float*>(p.Y) + out0 + (size_t)r * p.ldy + c) >> 2) & 3);
  };
  for (int c0 = 0; c0 < w.cols; c0 += cb) {
    const int n = min(min(cb, w.cols - c0), p.N - w.col0 - c0);
    const int r0 = tile * p.tile_tok + row;
    float* dst = stage + (size_t)r0 * pitch + shift(r0, c0);
    for (int c = c_first * kChunk; c < min(cb, w.cols - c0); c += c_step * kChunk) {
      float v[32];
      tmem_ld32(acc + (uint32_t)(c0 + c), v);
      if (row < p.tile_tok) {
#pragma unroll
        for (int e = 0; e < 32; ++e) dst[c + e] = v[e];
      }
    }
    fence_proxy_async_smem();
    named_bar(3, 2 * kEpiGroup);
    if (thread < min(p.m_pad, p.M - w.tok0) && n > 0) {
      float* y = static_cast<float*>(p.Y) + out0 + (size_t)thread * p.ldy + c0;
      const int a = shift(thread, c0), head = min((4 - a) & 3, n), mid = (n - head) & ~3;
      const float* src = stage + (size_t)thread * pitch + a;
      if (mid > 0) bulk_store(y + head, smem_u32(src + head), (uint32_t)mid * 4u);
      bulk_commit();
      for (int i = 0; i < head; ++i) y[i] = src[i];
      for (int i = head + mid; i < n; ++i) y[i] = src[i];
      bulk_wait_read<0>();                              // the rows are staged again, or the CTA ends
    }
    if (c0 + cb < w.cols) named_bar(3, 2 * kEpiGroup);
  }
}

// silu(gate) * up of a token row, eight features at a time, into the row of the
// staged [token][width / 2] tile.  The fast exponential and division keep the
// chain short (their relative error is far below the bf16 rounding of the
// result).  The widths are odd multiples of eight features, so the rows'
// 16-byte stores spread over the banks without swizzling.
template <typename T>
__device__ __forceinline__ void swiglu_row(uint32_t acc, uint32_t dst, int fw, int first, int step, bool on) {
  for (int c = first * 8; c < fw; c += step * 8) {
    float g[8], u[8], y[8];
    tmem_ld8(acc + (uint32_t)c, g);
    tmem_ld8(acc + (uint32_t)(fw + c), u);
    tmem_ld_wait(g);
    tmem_ld_wait(u);
#pragma unroll
    for (int e = 0; e < 8; ++e) y[e] = __fdividef(g[e], 1.0f + __expf(-g[e])) * u[e];
    if (on) {
      if constexpr (sizeof(T) == 2) {
        st_shared4(dst + (uint32_t)c * 2u, pack_bf16(y[0], y[1]), pack_bf16(y[2], y[3]), pack_bf16(y[4], y[5]),
                   pack_bf16(y[6], y[7]));
      } else {
        const uint32_t a = dst + (uint32_t)c * 4u;
        st_shared4(a, __float_as_uint(y[0]), __float_as_uint(y[1]), __float_as_uint(y[2]), __float_as_uint(y[3]));
        st_shared4(a + 16u, __float_as_uint(y[4]), __float_as_uint(y[5]), __float_as_uint(y[6]), __float_as_uint(y[7]));
      }
    }
    __syncwarp();
  }
}

// kTwoRings: activations in a ring of their own (more than 128 tokens), else
// in the weights' stages.
template <typename T, bool kTwoRings>
__global__ void __launch_bounds__(kTwoRings ? kGemmThreads : kGemmThreads - 32, 2)
    gemm_kernel(const __grid_constant__ CUtensorMap ta0, const __grid_constant__ CUtensorMap ta1,
                const __grid_constant__ CUtensorMap ta2, const __grid_constant__ CUtensorMap tb,
                const __grid_constant__ CUtensorMap to, const __grid_constant__ GemmParams p) {
  using G = GemmType<T>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const int SW = p.w_stages, SX = kTwoRings ? p.x_stages : p.w_stages;
  const uint32_t x_bytes = (uint32_t)p.m_pad * 128u, w_bytes = (uint32_t)p.width * 128u;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.off_bar);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 4 * kMaxStages + 5);
  volatile int* stop = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = warp_index();
  const int lane = threadIdx.x & 31;
  const uint32_t bar0 = smem_u32(bars), x0 = smem_u32(smem), w0 = x0 + (uint32_t)SX * x_bytes;
  auto wfull = [&](int s) { return bar0 + 8u * s; };
  auto wempty = [&](int s) { return bar0 + 8u * (kMaxStages + s); };
  auto xfull = [&](int s) { return bar0 + 8u * (2 * kMaxStages + s); };
  auto xempty = [&](int s) { return bar0 + 8u * (3 * kMaxStages + s); };
  auto acc_full = [&](int a) { return bar0 + 8u * (4 * kMaxStages + a); };
  auto acc_empty = [&](int a) { return bar0 + 8u * (4 * kMaxStages + 2 + a); };
  const uint32_t end_bar = bar0 + 8u * (4 * kMaxStages + 4);

  // one barrier a thread of warp 2: each takes its arrivals (the accumulators' empty
  // barriers one a warp of the epilogue, every other one a single one)
  if (warp == 2) {
    for (int i = lane; i < 4 * kMaxStages + 5; i += 32)
      mbar_init(bar0 + 8u * i, i == 4 * kMaxStages + 2 || i == 4 * kMaxStages + 3 ? 2 * kEpiGroup / 32 : 1);
    if (lane == 0) stop[0] = stop[1] = 0;
    fence_barrier_init();
  }
  if (threadIdx.x == 0) {
    tma_prefetch_desc(&ta0);
    tma_prefetch_desc(&tb);
    if (p.tma_out) tma_prefetch_desc(&to);
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), (uint32_t)p.tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (!p.late_trigger) griddep_launch();
  const uint32_t tmem_base = uniform(*tmem_slot);

  if (warp == 0) {
    // ------------------------------------------------------------ weight producer
    // a weight tile read by one CTA goes first; shared by token groups, it stays
    const uint64_t pol = p.tok_groups > 1 ? policy_evict_normal() : policy_evict_first();
    const uint64_t pol_x = policy_evict_last();
    const uint32_t bytes = w_bytes + (kTwoRings ? 0u : x_bytes);
    auto load_w = [&](const GemmItem& w, int i, int s) {
      const int kx = (w.kb0 + i) * G::BK;
      const uint32_t dst = w0 + (uint32_t)s * w_bytes;
      mbar_expect_tx(wfull(s), bytes);
      if (p.mode == EPI_SWIGLU) {                  // the tile's gate rows, then the matching up rows
        tma_load_2d(dst, &ta0, wfull(s), kx, w.row0 / 2, pol);
        tma_load_2d(dst + w_bytes / 2, &ta1, wfull(s), kx, w.row0 / 2, pol);
      } else {
        tma_load_2d(dst, w.seg == 0 ? &ta0 : (w.seg == 1 ? &ta1 : &ta2), wfull(s), kx, w.row0, pol);
      }
    };
    auto load_x = [&](const GemmItem& w, int i, int s) {
      tma_load_2d(x0 + (uint32_t)s * x_bytes, &tb, wfull(s), (w.kb0 + i) * G::BK, w.tok0, pol_x);
    };
    int s = 0, issued = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x) {
      const GemmItem w = gemm_item(p, item);
      int i = 0;
      if (!kTwoRings && issued == 0) {
        // the first stages' weights go out before the preceding kernel is done: they do not depend on it
        const int pre = min(SW, w.nk);
        for (; i < pre; ++i) {
          if (elect_one()) load_w(w, i, i);
          __syncwarp();
        }
        griddep_wait();
        if (p.late_trigger) griddep_launch();
        for (i = 0; i < pre; ++i) {
          if (elect_one()) load_x(w, i, i);
          __syncwarp();
        }
        issued = pre;
        s = pre % SW;
        ph = (uint32_t)(pre / SW) & 1u;
      }
      for (; i < w.nk; ++i) {
        if (issued >= SW && !gemm_wait(wempty(s), ph ^ 1u, stop, p.err)) { ok = false; break; }
        if (elect_one()) {
          load_w(w, i, s);
          if (!kTwoRings) load_x(w, i, s);
        }
        __syncwarp();
        ++issued;
        if (++s == SW) { s = 0; ph ^= 1u; }
      }
    }
    // every load has landed before the CTA's shared memory goes away
    for (int i = max(0, issued - SW); i < issued; ++i) mbar_wait(wfull(i % SW), (uint32_t)(i / SW) & 1u, p.err);
  } else if (kTwoRings && warp == kXWarp) {
    // ------------------------------------------------------------ activation producer
    const uint64_t pol = policy_evict_last();
    griddep_wait();                         // activations come from the preceding kernel
    // A late trigger lets the next kernel start only once every kernel before
    // this one has completed (it may then read their outputs before its own
    // wait, as the attention does with the view state).
    if (p.late_trigger) griddep_launch();
    int s = 0, issued = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x) {
      const GemmItem w = gemm_item(p, item);
      for (int i = 0; i < w.nk; ++i) {
        if (issued >= SX && !gemm_wait(xempty(s), ph ^ 1u, stop, p.err)) { ok = false; break; }
        if (elect_one()) {
          mbar_expect_tx(xfull(s), x_bytes);
          tma_load_2d(x0 + (uint32_t)s * x_bytes, &tb, xfull(s), (w.kb0 + i) * G::BK, w.tok0, pol);
        }
        __syncwarp();
        ++issued;
        if (++s == SX) { s = 0; ph ^= 1u; }
      }
    }
    for (int i = max(0, issued - SX); i < issued; ++i) mbar_wait(xfull(i % SX), (uint32_t)(i / SX) & 1u, p.err);
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issue
    // The whole warp walks the k-blocks and one lane issues: descriptors formed
    // once per stage and stepped by the byte offset >> 4 in their address field
    // (offsets stay inside the stage, so the field never carries), stage and
    // phase by counters, everything uniform (see elect_one).  The MMAs of a
    // k-block issue in 200 cycles a token tile instead of 500.
    const uint32_t idesc = make_idesc(p.width, G::FMT);
    const bool two = p.tok_tiles == 2;
    const uint64_t xd1 = (uint64_t)((p.tile_tok * 128) >> 4);
    int s = 0, sx = 0, n = 0;
    uint32_t ph = 0, phx = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x, ++n) {
      const GemmItem w = gemm_item(p, item);
      const int a = n % p.n_acc;
      if (n >= p.n_acc) ok = gemm_wait(acc_empty(a), (uint32_t)(n / p.n_acc - 1) & 1u, stop, p.err);
      tc_fence_after();
      const uint32_t d0 = tmem_base + (uint32_t)(a * p.acc_cols), d1 = d0 + (uint32_t)p.tile_cols;
      bool ready = false;
      for (int i = 0; i < w.nk; ++i) {
        if (!ready) ok = (!kTwoRings || gemm_wait(xfull(sx), phx, stop, p.err)) && gemm_wait(wfull(s), ph, stop, p.err);
        if (!ok) break;
        const uint64_t xd = sdesc_sw128(x0 + (uint32_t)sx * x_bytes), wd = sdesc_sw128(w0 + (uint32_t)s * w_bytes);
        auto tile = [&](uint32_t d, uint64_t x) {
#pragma unroll
          for (int kk = 0; kk < G::BK / G::UK; ++kk) {
            const uint32_t keep = (i > 0 || kk > 0) ? 1u : 0u;
            if constexpr (sizeof(T) == 2) umma_f16(d, x + (uint64_t)(2 * kk), wd + (uint64_t)(2 * kk), idesc, keep);
            else umma_tf32(d, x + (uint64_t)(2 * kk), wd + (uint64_t)(2 * kk), idesc, keep);
          }
        };
        const int s1 = s + 1 == SW ? 0 : s + 1, sx1 = sx + 1 == SX ? 0 : sx + 1;
        const uint32_t ph1 = s1 ? ph : ph ^ 1u, phx1 = sx1 ? phx : phx ^ 1u;
        if (elect_one()) {
          tile(d0, xd);
          if (two) tile(d1, xd + xd1);
        }
        __syncwarp();
        // is the next k-block here already?  (asked while these MMAs are queued: a
        // wait that succeeds at once still takes about 80 cycles)
        const bool rx = !kTwoRings || mbar_test_wait(xfull(sx1), phx1), rw = mbar_test_wait(wfull(s1), ph1);
        if (elect_one()) {
          umma_commit(wempty(s));
          if (kTwoRings) umma_commit(xempty(sx));
        }
        __syncwarp();
        ready = rx && rw;
        s = s1; ph = ph1;
        sx = sx1; phx = phx1;
      }
      if (elect_one()) umma_commit(acc_full(a));
      __syncwarp();
    }
    if (!ok) {                              // no MMA outlives the CTA's shared memory and TMEM
      if (elect_one()) umma_commit(end_bar);
      __syncwarp();
      mbar_wait(end_bar, 0, p.err);
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int grp = (warp - 2) >> 2, q = warp & 3, row = q * 32 + lane;
    const bool two = p.tok_tiles == 2;
    uint8_t* stg = smem + p.off_stg + (size_t)grp * p.n_stg * kChunkBytes;
    griddep_wait();
    int n = 0, chunks = 0;
    for (int item = blockIdx.x; item < p.items; item += gridDim.x, ++n) {
      const GemmItem w = gemm_item(p, item);
      const int a = n % p.n_acc;
      gemm_wait(acc_full(a), (uint32_t)(n / p.n_acc) & 1u, stop, p.err);
      tc_fence_after();
      // one thread's view of `stop` (which another role may set at any time), so
      // that every warp of a barrier takes the same branch
      named_bar(3, 2 * kEpiGroup);
      if (warp == 2 && lane == 0) stop[1] = *stop;
      named_bar(3, 2 * kEpiGroup);
      if (stop[1]) break;
      const int t = two ? grp : 0;
      const uint32_t acc = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(a * p.acc_cols + t * p.tile_cols);
      if (p.mode == EPI_SWIGLU) {
        // (one item a CTA: the ring is idle once its MMAs are done)
        const int fw = p.width / 2;
        uint8_t* tile = smem + (size_t)t * p.stg_tile;
        swiglu_row<T>(acc, smem_u32(tile) + (uint32_t)(row * fw) * (uint32_t)sizeof(T), fw, two ? 0 : grp, two ? 1 : 2,
                      row < p.tile_tok);
        fence_proxy_async_smem();
        named_bar(3, 2 * kEpiGroup);
        const int tok = w.tok0 + t * p.tile_tok;
        if (row == 0 && (two || grp == 0) && tok < p.M) {
          tma_store_3d(&to, smem_u32(tile), w.row0 / 2, tok, 0);
          bulk_commit();
        }
      } else if (p.row_cols > 0) {
        epilogue_rows(p, smem, acc, w, p.row_cols, t, two ? 0 : grp, two ? 1 : 2, row, grp * kEpiGroup + row);
      } else {
        epilogue_f32(p, &to, stg, p.n_stg, chunks, acc, w, w.tok0 + t * p.tile_tok, two ? 0 : grp, two ? 1 : 2, row, 1 + grp);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty(a));
    }
    if (row == 0) bulk_wait_read<0>();                          // staging smem is released at exit
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
  }
}

// y[i] = part[0][i] + part[1][i] + ... in split order.  Every split's load of a
// thread is in flight at once (a loop of dependent loads paid the L2 latency for
// each split: 3.5 us more at 7 x 4096 outputs and 9 splits), four outputs a thread where
// the split stride keeps float4 alignment.
template <typename V>
__device__ __forceinline__ V add_vec(const V& a, const V& b);
template <>
__device__ __forceinline__ float add_vec(const float& a, const float& b) { return a + b; }
template <>
__device__ __forceinline__ float4 add_vec(const float4& a, const float4& b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

template <typename V>
__global__ void __launch_bounds__(256) sum_partials_kernel(const V* __restrict__ part, int splits, size_t n, V* __restrict__ y) {
  griddep_launch();
  griddep_wait();
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    V acc = part[i];
    for (int s0 = 1; s0 < splits; s0 += 8) {
      V v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (s0 + u < splits) v[u] = __ldcs(part + (size_t)(s0 + u) * n + i);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (s0 + u < splits) acc = add_vec(acc, v[u]);
    }
    y[i] = acc;
  }
}

// ====================================================================== host

static PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
static std::once_flag g_encode_once;

static PFN_cuTensorMapEncodeTiled_v12000 encoder() {
  std::call_once(g_encode_once, [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  });
  return g_encode;
}

// 2-D K-major map: rows x K elements, box (BK, box_rows), 128-byte swizzle.
static int make_map(CUtensorMap* m, int dtype, const void* ptr, int K, int rows, int box_rows) {
  auto enc = encoder();
  if (!enc) return LSP_ERR_UNSUPPORTED;
  const int es = dtype == LSP_DTYPE_BF16 ? 2 : 4;
  const int bk = 128 / es;
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)K * es};
  cuuint32_t box[2] = {(cuuint32_t)bk, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, dtype == LSP_DTYPE_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                              : CU_TENSOR_MAP_DATA_TYPE_TFLOAT32,
                   2, const_cast<void*>(ptr), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? LSP_OK : LSP_ERR_CUDA;
}

int tmap_2d_bf16_sw128(CUtensorMap* m, const void* ptr, uint64_t inner, uint64_t rows, uint64_t row_bytes,
                       uint32_t box_inner, uint32_t box_rows) {
  auto enc = encoder();
  if (!enc) return LSP_ERR_UNSUPPORTED;
  if (((uintptr_t)ptr & 15) || (row_bytes % 16) || box_inner * 2 > 128 || box_rows < 1 || box_rows > 256)
    return LSP_ERR_SHAPE;
  cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)row_bytes};
  cuuint32_t box[2] = {box_inner, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? LSP_OK : LSP_ERR_CUDA;
}

// [splits][M][N] view of the output (row stride ldy) for TMA stores of
// box (cols features, tok tokens, 1 split); swizzled: 128-byte rows staged with
// the 128-byte swizzle, else rows as they are.
static int make_out_map(CUtensorMap* m, bool f32, bool swizzled, const void* Y, int N, int M, int splits, int ldy,
                        int cols, int tok) {
  auto enc = encoder();
  if (!enc) return LSP_ERR_UNSUPPORTED;
  const int es = f32 ? 4 : 2;
  if (((uintptr_t)Y & 15) || ((size_t)ldy * es) % 16) return LSP_ERR_SHAPE;
  cuuint64_t dims[3] = {(cuuint64_t)N, (cuuint64_t)M, (cuuint64_t)splits};
  cuuint64_t strides[2] = {(cuuint64_t)ldy * es, (cuuint64_t)M * ldy * es};
  cuuint32_t box[3] = {(cuuint32_t)cols, (cuuint32_t)tok, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(m, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
                   const_cast<void*>(Y), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   swizzled ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? LSP_OK : LSP_ERR_CUDA;
}

static constexpr int kSmemBudget = 227 * 1024;

int gemm_tiles(int mode, const int* seg_rows, int nseg) {
  if (mode == EPI_SWIGLU) return (seg_rows[0] + 63) / 64;
  int t = 0;
  for (int i = 0; i < nseg; ++i) t += (seg_rows[i] + kTileRows - 1) / kTileRows;
  return t;
}

int gemm_kblocks(int K, int dtype) {
  const int bk = dtype == LSP_DTYPE_BF16 ? 64 : 32;
  return (K + bk - 1) / bk;
}

static void token_tiling(int M, int* bn, int* ntt) {
  *ntt = (M + 255) / 256;
  int per = (M + *ntt - 1) / *ntt;
  *bn = std::max(16, (per + 15) / 16 * 16);
}

int gemm_group_rows(int M, int G) {
  int bn, ntt;
  token_tiling((M + G - 1) / G, &bn, &ntt);
  return bn * ntt;
}


// ---- split-K factor.  The k ranges decide the order of the fp32 sums, so their
// rule is fixed: it is the cost model of a kernel with one 128-row weight tile
// a CTA (16 KB of weights a stage; two or three CTAs an SM where their rings and
// accumulators fit), which gives the short projections enough CTAs for this
// one as well.
constexpr int kSplitTileBytes = kTileRows * 128;

static bool two_per_sm_fits(int m_pad) {
  const int stage_bytes = kSplitTileBytes + m_pad * 128;
  return 2 * stage_bytes + 2048 <= kSmemBudget / 2 && 2 * m_pad <= 512;
}

constexpr int kSmemPerSm = 228 * 1024;
static bool three_per_sm_fits(int m_pad, int groups) {
  if (groups < 2) return false;
  int cols = 32;
  while (cols < m_pad) cols *= 2;
  const int stage_bytes = kSplitTileBytes + m_pad * 128;
  return 3 * (2 * stage_bytes + 1280 + 1024) <= kSmemPerSm && 3 * cols <= 512;
}

// Token groups of the model: two above 256 tokens, and for a gate/up projection
// whose tiles fill at least one wave of one CTA per SM but less than one of two.
static int token_groups(int M, int mode, int n_tiles, int num_sms) {
  const int g = (M > 256 || (mode == EPI_SWIGLU && M >= 128 && n_tiles <= 2 * num_sms && n_tiles >= num_sms)) ? 2 : 1;
  if (g == 1) return 1;
  int bn, ntt;
  token_tiling((M + g - 1) / g, &bn, &ntt);
  return (g - 1) * bn * ntt < M ? g : 1;     // every group holds at least one token row
}

// In units of one k-block of one of two co-resident CTAs (~0.8 us at M = 256):
// waves x (k-blocks per CTA + fixed per-CTA cost) + the cost of combining the
// splits (per_split_cost per split: the consumer's re-read of fp32 partials
// from L2).  A lone CTA on an SM moves a k-block in 0.53 of that time.
constexpr double kLoneCtaCost = 0.53;

int gemm_auto_splits(int n_ctas, int kblocks, int num_sms, double per_split_cost, int max_splits,
                     int occ_max) {
  double best = 1e30;
  int splits = 1;
  for (int s = 1; s <= std::min(max_splits, kblocks); ++s) {
    const long long ctas = (long long)n_ctas * s;
    const int occ = (occ_max >= 3 && ctas >= 2LL * num_sms) ? 3
                    : (occ_max >= 2 && ctas * 4 >= (long long)num_sms * 5) ? 2 : 1;
    const long long slots = (long long)occ * num_sms;
    const long long waves = (ctas + slots - 1) / slots;
    const double per = (double)((kblocks + s - 1) / s) * (occ > 1 ? 1.0 : kLoneCtaCost) + 2.0;
    const double cost = (double)waves * per + (s > 1 ? per_split_cost * s : 0.0);
    if (cost < best - 1e-9) { best = cost; splits = s; }
  }
  return splits;
}

// Consumer cost of one M x N fp32 partial read back from L2 (~5 TB/s), in the
// model's k-block units (~1.56 us).
double gemm_partial_cost(int M, int N) { return (double)M * N * 4.0 / 5e12 / 1.56e-6; }

void gemm_choose(int dtype, int M, int K, int n_tiles, int mode, int num_sms, int* splits, int* groups) {
  const int G = token_groups(M, mode, n_tiles, num_sms);
  if (groups) *groups = G;
  int bn, ntt;
  token_tiling((M + G - 1) / G, &bn, &ntt);
  const int m_pad = bn * ntt;
  const int kblocks = gemm_kblocks(K, dtype);
  const int n_ctas = n_tiles * G;
  const int occ_max = three_per_sm_fits(m_pad, G) ? 3 : two_per_sm_fits(m_pad) ? 2 : 1;
  if (*splits <= 0)
    *splits = mode == EPI_PARTIAL
                  ? gemm_auto_splits(n_ctas, kblocks, num_sms, gemm_partial_cost(M, n_tiles * kTileRows), 16, occ_max)
                  : 1;
  *splits = std::max(1, std::min(*splits, kblocks));
}


// ---- tiling of a launch: weight rows per tile, and how CTAs walk the items
struct Tiling {
  int width, tiles, w_stages, x_stages, persistent;
};

static constexpr int kBarBytes = 384;

// Bytes an epilogue keeps for itself where CTAs walk several items (two
// groups, one chunk buffer each); with one item it stages in the idle rings.
static constexpr int kStgBytes = 2 * (int)kChunkBytes;

// Stages in the shared memory left.  Up to 128 tokens a stage holds both tiles;
// above, activations take 3 stages (2 where weights would get fewer than 4).
static void ring_stages(int width, int m_pad, bool persistent, int* w, int* x) {
  const int room = (kSmemBudget - 1024 - kBarBytes - (persistent ? kStgBytes : 0)) / 128;
  if (m_pad <= kTileTok) {
    *w = *x = std::min(kMaxStages, room / (width + m_pad));
    return;
  }
  for (*x = 3; *x > 2 && (room - *x * m_pad) / width < 4; --*x) {}
  *w = std::min(kMaxStages, (room - *x * m_pad) / width);
}

// Time of one launch in ns for a tile width, from what was measured on the
// GB300.  A k-block takes the longest of: the SM's intake (115 B/ns), its share
// of HBM (6.4 KB/ns over all CTAs), its MMAs (width / 2 cycles, at least 50, for
// each of four steps and each token tile) with 150 cycles of waits and commits,
// and the round trip of a stage (2 us) over the weight stages.  A CTA costs
// about 2 us to start; writing an item out takes 0.7 us and 0.35 us a 32-feature
// chunk (a burst of all CTAs), under the next item's MMAs where a walk has two accumulator
// sets, partly exposed where it has one.  A walk that stores from registers takes 2.2 us
// and, from 85 tokens on, longer a chunk (22 x 10875 x 3344 in 6 splits: 20.8 -> 18.1 us by the width
// that this chooses).
static double tiling_cost(int width, int m_pad, int tok_tiles, int kblocks, long long items, int num_sms, int stages,
                          bool persistent, bool mapped) {
  const double in = (width + m_pad) * 128.0 / 115.0;
  const double hbm = width * 128.0 * (double)std::min<long long>(items, num_sms) / 6400.0;
  const double mma = (tok_tiles * 4 * std::max(width / 2, 50) + 150) / 1.9, trip = 2000.0 / stages;
  const double kb = kblocks * std::max(std::max(in, hbm), std::max(mma, trip));
  const double waves = (double)((items + num_sms - 1) / num_sms);
  const double out = mapped || !persistent ? 700.0 + 11.0 * width : 2200.0 + std::max(11.0, 0.13 * m_pad) * width;
  if (!persistent) return waves * (kb + 2000.0 + out);
  const bool two_sets = 2 * tok_tiles * ((width + 31) / 32 * 32) <= 512;
  return (two_sets ? waves * std::max(kb, out) : waves * kb + (waves - 1) * 0.6 * out) + 2000.0 + out;
}

// The tile width with the least modelled time: multiples of 32 up to 256 weight
// rows (a chunk of the epilogue is 32), for gate/up twice an odd multiple of
// eight features.  CTAs walk the items where these make more than one wave.
static Tiling choose_width(int mode, const int* seg_rows, int nseg, int m_pad, int tok_tiles, int groups, int splits,
                           int kblocks, int num_sms, bool mapped) {
  Tiling best = {};
  double cost = 1e30;
  const bool gu = mode == EPI_SWIGLU;
  const int kb = (kblocks + splits - 1) / splits;
  for (int width = gu ? 16 : 32; width <= 256; width += 32) {
    int tiles = 0;
    for (int i = 0; i < (gu ? 1 : nseg); ++i) tiles += (seg_rows[i] + (gu ? width / 2 : width) - 1) / (gu ? width / 2 : width);
    const long long items = (long long)tiles * groups * splits;
    const bool persistent = !gu && items > num_sms;
    int ws, xs;
    ring_stages(width, m_pad, persistent, &ws, &xs);
    if (ws < 2) continue;
    const double c = tiling_cost(width, m_pad, tok_tiles, kb, items, num_sms, ws, persistent, mapped);
    if (c < cost - 1e-9) {
      cost = c;
      best = {width, tiles, ws, xs, persistent};
    }
  }
  return best;
}

int gemm_layout(GemmParams* pp, size_t* smem, int* ctas, int dtype, int M, int K, const int* seg_rows, int nseg, int mode,
                int num_sms, int splits, bool mapped) {
  if (M < 1 || M > 512 || K < 1 || nseg < 1 || nseg > 3) return LSP_ERR_SHAPE;
  const bool gu = mode == EPI_SWIGLU;
  if (gu && nseg != 2) return LSP_ERR_SHAPE;
  const int es = dtype == LSP_DTYPE_BF16 ? 2 : 4;
  if ((K * es) % 16) return LSP_ERR_SHAPE;
  for (int i = 0; i + 1 < nseg && !gu; ++i)
    if (seg_rows[i] % kTileRows) return LSP_ERR_SHAPE;
  GemmParams& p = *pp;
  p = GemmParams{};
  p.M = M;
  p.K = K;
  p.mode = mode;
  p.nseg = gu ? 1 : nseg;
  p.kblocks = gemm_kblocks(K, dtype);
  gemm_choose(dtype, M, K, gemm_tiles(mode, seg_rows, nseg), mode, num_sms, &splits);
  if (splits > 1 && mode != EPI_PARTIAL) return LSP_ERR_SHAPE;
  p.splits = splits;
  // up to 256 tokens a CTA, in one or two accumulators of at most 128
  p.tok_groups = M > 256 ? 2 : 1;
  p.m_pad = ((M + p.tok_groups - 1) / p.tok_groups + 15) / 16 * 16;
  p.tok_tiles = p.m_pad > kTileTok ? 2 : 1;
  p.tile_tok = p.m_pad / p.tok_tiles;
  const Tiling t = choose_width(mode, seg_rows, nseg, p.m_pad, p.tok_tiles, p.tok_groups, splits, p.kblocks, num_sms, mapped);
  if (t.w_stages < 2) return LSP_ERR_SHAPE;
  p.width = t.width;
  p.n_tiles = t.tiles;
  p.w_stages = t.w_stages;
  p.x_stages = t.x_stages;
  p.items = t.tiles * p.tok_groups * splits;
  for (int i = 0, tile = 0; i < p.nseg; ++i) {
    p.seg_tile0[i] = tile;
    p.seg_rows[i] = gu ? 2 * seg_rows[i] : seg_rows[i];
    p.seg_col0[i] = p.N;
    tile += (p.seg_rows[i] + p.width - 1) / p.width;
    p.N += seg_rows[i];
  }
  // accumulators: one set of tok_tiles x width columns, or two where a walk over
  // several items can alternate between them
  p.tile_cols = (p.width + 31) / 32 * 32;
  p.acc_cols = p.tok_tiles * p.tile_cols;
  p.n_acc = t.persistent && 2 * p.acc_cols <= 512 ? 2 : 1;
  p.tmem_cols = 32;
  while (p.tmem_cols < p.n_acc * p.acc_cols) p.tmem_cols *= 2;
  // shared memory: activation ring | weight ring | staging of a walk | barriers;
  // an accumulator of fewer than 128 tokens reads past its activation tile
  // (lanes nobody looks at), into the weight ring or what follows
  const int ring = (p.w_stages * p.width + p.x_stages * p.m_pad) * 128;
  p.off_stg = t.persistent ? ring : 0;
  p.n_stg = t.persistent ? 1 : std::max(1, std::min(4, ring / kStgBytes));
  p.stg_tile = (p.tile_tok * (p.width / 2) * es + 127) / 128 * 128;
  if (gu && p.tok_tiles * p.stg_tile > ring) return LSP_ERR_SHAPE;
  p.off_bar = std::max(ring + (t.persistent ? kStgBytes : 0), (p.x_stages * p.m_pad - p.tile_tok + kTileTok) * 128);
  if (!gu && !t.persistent) p.off_bar = std::max(p.off_bar, p.n_stg * kStgBytes);
  // (copies of narrow tiles' rows cost more than the registers' stores: width 32, 500 x 2001 x
  // 300 9.8 us against 9.2; 64, one accumulator, 64 x 3001 x 4096 11.1 and 10.2, but two, 250 x 9001 x
  // 512, 8.3 and 8.8; 96, 300 x 5001 x 2048, 16.6 and 17.5)
  if (!gu && !mapped && !t.persistent && p.width >= (p.tok_tiles == 2 ? 64 : 96))
    p.row_cols = std::min(p.width, (ring / (4 * p.m_pad) - 4) / kChunk * kChunk);
  *smem = (size_t)p.off_bar + kBarBytes + 1024;
  if (*smem > (size_t)kSmemBudget) return LSP_ERR_SHAPE;
  *ctas = t.persistent ? num_sms : p.items;
  return LSP_OK;
}

int gemm_plan(GemmOp* op, int dtype, const void* X, int M, int K, const void* const* W,
              const int* seg_rows, int nseg, int mode, void* Y, int ldy, unsigned* err,
              int num_sms, int splits) {
  const bool gu = mode == EPI_SWIGLU;
  const bool mapped = ((reinterpret_cast<uintptr_t>(Y) | (uintptr_t)ldy * 4u) & 15) == 0;   // (fp32 outputs)
  GemmParams& p = op->p;
  int ctas = 0, rc;
  if ((rc = gemm_layout(&p, &op->smem, &ctas, dtype, M, K, seg_rows, nseg, mode, num_sms, splits, mapped)) != LSP_OK) return rc;
  op->grid = dim3((unsigned)ctas, 1, 1);
  op->dtype = dtype;
  p.Y = Y;
  p.ldy = ldy;
  p.err = err;
  const int box = gu ? p.width / 2 : p.width;
  for (int i = 0; i < 3; ++i) {
    if (i >= nseg) op->a[i] = op->a[0];      // unused placeholder (an encoding takes the host 0.2 us)
    else if ((rc = make_map(&op->a[i], dtype, W[i], K, seg_rows[i], box)) != LSP_OK) return rc;
  }
  if ((rc = make_map(&op->b, dtype, X, K, M, p.m_pad)) != LSP_OK) return rc;
  // TMA-store epilogue when the output view can be described (else per-thread stores)
  if (gu) {
    if ((rc = make_out_map(&op->out, dtype == LSP_DTYPE_F32, false, Y, p.N, M, 1, ldy, p.width / 2, p.tile_tok)) != LSP_OK)
      return rc;
    p.tma_out = 1;
  } else {
    p.tma_out = make_out_map(&op->out, true, true, Y, p.N, M, p.splits, ldy, kChunk, p.tile_tok) == LSP_OK;
    if (!p.tma_out) op->out = op->b;       // unused placeholder
  }
  return LSP_OK;
}

template <typename T, bool kTwoRings>
static int launch_t(const GemmOp* op, cudaStream_t s) {
  static SmemOptIn once;
  if (smem_opt_in(once, gemm_kernel<T, kTwoRings>, kSmemBudget) != cudaSuccess) return LSP_ERR_CUDA;
  const cudaError_t e = launch_pdl(gemm_kernel<T, kTwoRings>, op->grid, dim3(kTwoRings ? kGemmThreads : kGemmThreads - 32),
                                   op->smem, s, op->a[0], op->a[1], op->a[2], op->b, op->out, op->p);
  return e == cudaSuccess ? LSP_OK : LSP_ERR_CUDA;
}

int gemm_launch(const GemmOp* op, cudaStream_t s) {
  const bool two = op->p.tok_tiles == 2;
  if (op->dtype == LSP_DTYPE_BF16) return two ? launch_t<bf16, true>(op, s) : launch_t<bf16, false>(op, s);
  return two ? launch_t<float, true>(op, s) : launch_t<float, false>(op, s);
}

int launch_sum_partials(const float* part, int splits, size_t n, float* y, cudaStream_t s) {
  const bool vec = n % 4 == 0 && (((uintptr_t)part | (uintptr_t)y) & 15) == 0;
  const size_t m = vec ? n / 4 : n;
  const dim3 blocks((unsigned)std::min<size_t>((m + 255) / 256, 4096));
  const cudaError_t e = vec ? launch_pdl(sum_partials_kernel<float4>, blocks, dim3(256), 0, s,
                                         reinterpret_cast<const float4*>(part), splits, m, reinterpret_cast<float4*>(y))
                            : launch_pdl(sum_partials_kernel<float>, blocks, dim3(256), 0, s, part, splits, m, y);
  return e == cudaSuccess ? LSP_OK : LSP_ERR_CUDA;
}

}  // namespace lsp
