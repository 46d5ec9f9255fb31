// Folding long runs of prefix rows into the interface on the tcgen05 tensor
// cores (Sec. 2.2, Eq. global-summary, App. A.2): lsp_prefill (one request's
// whole prefix, Fig. 3) and lsp_view_update calls whose row capacity is a
// chunk of a prefix rather than one round's accepted tokens.  bf16 storage,
// head dim 128, at most 16 summary queries a head and 8 query heads a KV head.
//
// For every tapped layer l and query head h the new rows' statistics are
//     s_j = g_r . k_j / sqrt(d),  eta_N = log sum_j exp(s_j),
//     m_N = sum_j exp(s_j - eta_N) v_j,
// merged with the stored (eta_A, m_A) by Eq. summary-update (a prefill merges
// with the empty prefix).  A unit is one (request, layer, KV head): its
// queries are the 16 REP rows of the KV head's REP query heads (R padded to
// 16), its keys the request's new rows in blocks of 128.
//
// What bounds it: the K/V rows, read once from HBM.  The arithmetic is small
// for tcgen05 (about 0.4 of the time the rows take to arrive at REP = 4) but
// was the bound on mma.sync, one warp a query head.
//
// fold_tc_kernel, one CTA per SM, an equal share of the 128-row blocks of all
// units each (a share may end one unit and begin the next, so no last wave is
// left over whatever the row counts are):
//   warp 8      TMA producer: K and V blocks (32 KB each, 128-byte swizzle)
//               through a ring of four or five slots: at least 64 KB of loads
//               in flight an SM, what HBM's latency asks for
//   warp 9      TMEM allocation and MMA issue.  S^T = K G^T: keys on the 128
//               lanes, queries on N, two buffers, so the next block's scores
//               run under this block's softmax.  O^T += V^T P^T: dims on the
//               lanes, V as the MN-major A operand straight from its rows, P
//               as the MN-major B operand.  Both operands of P V take the
//               layout their producer writes, so nothing is transposed.
//   warps 0-7   softmax: a thread owns one key (TMEM lane) and half of the
//               queries, P = 2^((s - ref) log2(e) / sqrt(d)) is written as a
//               bf16 high part and one or two bf16 remainders (two MMAs, ~16
//               significant bits, or three, ~24: see fold_parts), and the sums
//               stay in registers.
//   warps 10-11 the window ring and the boundary rows; the softmax warps join
//               them when their blocks are done
//
// The reference ref of each query is not the running maximum: bf16 and fp32
// share their exponent range, so P keeps its precision under any reference
// near the maximum.  ref is the maximum over the first block, and is raised
// only when a score passes it by 24 in base-2 units (one compare a score and
// one barrier a block instead of a maximum across the 128 lanes for every
// query and block).  The accumulator is drained into registers every
// kFlushBlocks blocks and when ref moves, and the remainders' MMAs of a block go
// first: tcgen05 accumulation drops low bits.  Relative error of m against 64
// bits at 131072 / 2048 / 1999 rows: 2.8e-6 / 4.9e-7 / 2.3e-6 with 8 blocks and
// the parts in turn, 2.1e-6 / 4.0e-7 / 2.1e-6 with 2 or 1 and the remainders
// first (the mma.sync kernel this replaces: 4.6e-6 / 8.3e-7 / 2.0e-6); the call of
// 131072 rows takes 450.6, 452.1 and 453.9 us with 8, 2 and 1 (460 with the
// parts in turn).  (With three parts the 1999 rows leave 4.9e-7.)
//
// fold_merge_kernel merges a unit's pieces (one per CTA share that touches
// it) and the stored state, in share order: deterministic.
//
// Measured (GB300, Qwen3-8B heads, 5 layers, in a graph): lsp_prefill of 131072
// rows (2.68 GB) 738 us with the mma.sync kernel, 399 us now with the merge (6.7
// TB/s, the copy bandwidth), of 1999 rows 44 -> 23 us; lsp_view_update of 2048 rows
// 231 -> 22 us for one request, 421 -> 162 us for 16.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "lsp_internal.h"

namespace lsp {
namespace {

constexpr int kFoldD = 128;                  // head dim
constexpr int kFoldKeys = 128;               // keys per block (UMMA M)
constexpr int kFoldSoftmax = 256;            // softmax threads (8 warps)
constexpr int kFoldCopy = 64;                // threads that copy the window (2 warps)
constexpr int kFoldThreads = kFoldSoftmax + 64 + kFoldCopy;
constexpr int kFoldSlot = kFoldKeys * 256;   // bytes of one K or V block
constexpr int kFoldRec = 16 + 16 * kFoldD;   // floats per (piece, query head): eta[16], m[16][d]
constexpr int kFlushBlocks = 2;
constexpr float kRefSlack = 24.f;            // log2 units a score may pass its reference by
constexpr int kFoldMaxC = 64;
constexpr int kCopyBatch = 4;                // window vectors a copying lane has in flight (K and V each)
constexpr int kFoldMaxSlots = 5;
constexpr int kFoldSmall = 128;              // rows of a prefill up to which it takes fold_small_kernel

struct FoldLayout {
  int slots;
  uint32_t off_p, off_ring, off_misc, bytes;
};

// bytes: G [2][16 REP][128 B], P in parts [64-query blocks][128][128 B],
// the ring, then references, scales, block counts, rows and slots, barriers
__host__ __device__ constexpr FoldLayout fold_layout(int rep, int parts) {
  FoldLayout L{};
  const int nb = (16 * rep + 63) / 64;
  L.off_p = (uint32_t)rep * 4096u;
  L.off_ring = L.off_p + (uint32_t)(parts * nb) * 16384u;
  const uint32_t misc = 2u * 16u * (uint32_t)rep * 4u + 272u + 2u * kFoldMaxC * 4u + 160u;
  const int fit = (int)((227u * 1024u - 1024u - misc - L.off_ring) / (uint32_t)kFoldSlot);
  const int most = parts == 2 ? kFoldMaxSlots : kFoldMaxSlots - 1;   // (three: room for CTAs of the merge to wait in)
  L.slots = fit < most ? fit : most;
  L.off_misc = L.off_ring + (uint32_t)L.slots * kFoldSlot;
  L.bytes = L.off_misc + misc + 1024u;
  return L;
}
static_assert(fold_layout(8, 2).slots >= 4 && fold_layout(4, 3).slots == 4, "K and V of two blocks fit the ring");
static_assert(fold_layout(8, 3).slots >= 3, "K and V of a block and the next K fit the ring");

__host__ __device__ constexpr uint32_t fold_tmem_cols(int rep) {
  uint32_t c = 32;
  while (c < 48u * (uint32_t)rep) c *= 2;    // two score buffers and the output, 16 rep columns each
  return c;
}

// MN-major operand with 128-byte swizzling: 64 contiguous elements per 128-B
// row, 8 rows of K per 1024-B group, `lbo` bytes between 64-element blocks.
__device__ __forceinline__ uint64_t fold_desc_mn(uint32_t saddr, uint32_t lbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)(1024u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// kind::f16, bf16 A and B, fp32 D, M = 128, N = n; `mn`: A and B MN-major.
__device__ __forceinline__ uint32_t fold_idesc(int n, bool mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? (3u << 15) : 0u) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(kFoldKeys >> 4) << 24);
}

template <int N>
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, float (&v)[N]) {
  static_assert(N % 8 == 0, "columns come in eights");
#pragma unroll
  for (int c = 0; c < N; c += 8) tmem_ld8(taddr + (uint32_t)c, v + c);
  tmem_ld_wait(v);
}

__device__ __forceinline__ float fold_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void st_v4(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}

// Wait that gives up after kWaitLimitNs (recorded), or as soon as another
// role of the CTA has given up: every loop below still runs to its end then.
__device__ __forceinline__ bool fold_wait(uint32_t bar, uint32_t parity, volatile int* stop, unsigned* err) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 15u) == 0) {
      if (*stop) return false;
      if (global_ns() - t0 > kWaitLimitNs) {
        set_err(err, LSP_DEV_TIMEOUT);
        *stop = 1;
        return false;
      }
    }
  }
}

__device__ __forceinline__ bool softmax_any(bool x) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.or.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}"
      : "=r"(r)
      : "r"((uint32_t)x), "n"(kFoldSoftmax)
      : "memory");
  return r != 0;
}

// The warp's max or sum over its 32 lanes of eight columns: lane L gets column
// L & 7 (nine shuffles instead of five for each column).
template <bool kMax>
__device__ __forceinline__ float reduce8(const float* x, int lane) {
  auto op = [](float a, float b) { return kMax ? fmaxf(a, b) : a + b; };
  float y[4], z[2];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float send = (lane & 4) ? x[k] : x[k + 4], keep = (lane & 4) ? x[k + 4] : x[k];
    y[k] = op(keep, __shfl_xor_sync(0xffffffffu, send, 4));
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float send = (lane & 2) ? y[k] : y[k + 2], keep = (lane & 2) ? y[k + 2] : y[k];
    z[k] = op(keep, __shfl_xor_sync(0xffffffffu, send, 2));
  }
  const float send = (lane & 1) ? z[0] : z[1], keep = (lane & 1) ? z[1] : z[0];
  float r = op(keep, __shfl_xor_sync(0xffffffffu, send, 1));
  r = op(r, __shfl_xor_sync(0xffffffffu, r, 8));
  return op(r, __shfl_xor_sync(0xffffffffu, r, 16));
}

// Accepted rows of request i of this call (0 where the count is out of range).
__device__ __forceinline__ int fold_rows(const FoldParams& p, int i) {
  const int n = p.acc ? p.acc[i] : p.rows;
  return n < 0 || n > p.rows ? 0 : n;
}

// pre[i] = blocks per unit of requests 0 .. i-1 (one warp; nreq <= 64).
__device__ __forceinline__ void fold_prefix(const FoldParams& p, int* pre, int lane) {
  auto nblk = [&](int i) { return i < p.nreq && p.R > 0 ? (fold_rows(p, i) + kFoldKeys - 1) / kFoldKeys : 0; };
  const int a = nblk(2 * lane), b = nblk(2 * lane + 1);
  int s = a + b;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += v;
  }
  pre[2 * lane] = s - a - b;
  pre[2 * lane + 1] = s - b;
  if (lane == 31) pre[kFoldMaxC] = s;
}

// CTAs that get blocks: every share holds at least one (1 when there are none).
__device__ __forceinline__ long long fold_shares(long long total, unsigned grid) {
  return max(1ll, min(total, (long long)grid));
}

// The piece of a CTA's share [f, f_end) that begins at flattened block f: the
// blocks of all units in order (request, layer x KV head, block).
struct FoldPiece {
  int req, lg, blk, n, unit;       // n blocks from block blk of unit = req * LG + lg
};
__device__ __forceinline__ FoldPiece fold_piece(const int* pre, int nreq, int LG, int f, int f_end) {
  FoldPiece q;
  int i = 0;
  while (i + 1 < nreq && f >= pre[i + 1] * LG) ++i;
  const int nb = pre[i + 1] - pre[i], r = f - pre[i] * LG;
  q.req = i;
  q.lg = r / nb;
  q.blk = r - q.lg * nb;
  q.n = min(nb - q.blk, f_end - f);
  q.unit = i * LG + q.lg;
  return q;
}

// Window ring (row q of the prefix in slot q mod W): a warp copies the chunks of
// kCopyBatch x 32 vectors that next() names.  The walk goes over `longest` rows of every
// (request, layer), the most that any request has for its window, and skips what lies past
// a request's own (over W rows it took 6 us more at 16 requests of one row each, W = 256).
template <typename F>
__device__ __forceinline__ void fold_copy_window(const FoldParams& p, int longest, const int* srows, const int* sslot, int lane, F next) {
  const int vpr = p.nkv * (kFoldD / 8), span = longest * vpr;   // 16-byte vectors of a row (all KV heads), of the rows walked
  const int items = p.nreq * p.L * span;
  for (;;) {
    const long long first = next() * (kCopyBatch * 32);
    if (first >= items) break;
    const int k0 = (int)first + lane;
    uint4 xk[kCopyBatch], xv[kCopyBatch];
    size_t dst[kCopyBatch];
    bool on[kCopyBatch];
#pragma unroll
    for (int u = 0; u < kCopyBatch; ++u) {
      const int k = k0 + u * 32, ul = k / span, w = k - ul * span, r = w / vpr, v = w - r * vpr;
      const int i = ul / p.L, l = ul - i * p.L;
      on[u] = k < items && r < min(srows[i], p.W);
      if (on[u]) {
        const int n = srows[i];
        int slot = sslot[i] + r;
        if (slot >= p.W) slot -= p.W;
        dst[u] = ((((size_t)(p.b0 + i) * p.L + l) * p.nkv + (v >> 4)) * p.W + slot) * kFoldD + (size_t)(v & 15) * 8;
        const size_t src = (((size_t)ul * p.rows + (n - min(n, p.W)) + r) * vpr + v) * 8;
        xk[u] = *reinterpret_cast<const uint4*>(static_cast<const bf16*>(p.k) + src);
        xv[u] = *reinterpret_cast<const uint4*>(static_cast<const bf16*>(p.v) + src);
      }
    }
#pragma unroll
    for (int u = 0; u < kCopyBatch; ++u)
      if (on[u]) {
        *reinterpret_cast<uint4*>(static_cast<bf16*>(p.win_k) + dst[u]) = xk[u];
        *reinterpret_cast<uint4*>(static_cast<bf16*>(p.win_v) + dst[u]) = xv[u];
      }
  }
}

// Boundary rows: the (request, layer) pairs first, first + step, .. by nthr threads.
__device__ __forceinline__ void fold_copy_boundary(const FoldParams& p, const int* srows, int first, int step, int t, int nthr) {
  for (int ul = first; ul < p.nreq * p.L; ul += step) {
    const int i = ul / p.L, n = srows[i];
    if (n == 0) continue;
    const bf16* hin = static_cast<const bf16*>(p.hid) + ((size_t)ul * p.h_rows + (p.h_rows == 1 ? 0 : n - 1)) * p.H;
    bf16* hout = static_cast<bf16*>(p.h) + ((size_t)p.b0 * p.L + ul) * p.H;
    for (int k = t * 8; k < p.H; k += nthr * 8) *reinterpret_cast<uint4*>(hout + k) = *reinterpret_cast<const uint4*>(hin + k);
  }
}

// The summary over at most kFoldSmall rows, of one layer l and query head h, by a CTA of
// 256 threads: scores, weights and values in shared memory, products with mma.sync,
// weights in three parts (see fold_parts).  What bounds it is latency: one round trip
// for K, V and G and three barriers.
constexpr int kSmallLd = kFoldD + 8, kSmallPLd = kFoldSmall + 8, kSmallSLd = kFoldSmall + 4;
struct alignas(16) SmallSmem {
  bf16 k[kFoldSmall * kSmallLd], v[kFoldSmall * kSmallLd];
  union {
    bf16 g[16 * kSmallLd];
    bf16 p[3][16 * kSmallPLd];
  };
  float s[16 * kSmallSLd];
  float sum[16];
};

__device__ __forceinline__ void fold_small(const FoldParams& p, SmallSmem& sm, int l, int h) {
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31, r = tid >> 4, c = tid & 15, n = p.rows;
  const size_t row = (size_t)p.nkv * kFoldD, in = (size_t)l * n * row + (size_t)(h / (p.nq / p.nkv)) * kFoldD;
  const size_t q0 = (((size_t)p.b0 * p.L + l) * p.nq + h) * p.R;
  const bf16* k = static_cast<const bf16*>(p.k) + in;
  const bf16* v = static_cast<const bf16*>(p.v) + in;
  const bf16* G = static_cast<const bf16*>(p.G) + ((size_t)l * p.nq + h) * p.R * kFoldD;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  uint4 xk[kFoldSmall / 16], xv[kFoldSmall / 16];
#pragma unroll
  for (int u = 0; u < kFoldSmall / 16; ++u) {
    const int j = r + u * 16;
    xk[u] = j < n ? *reinterpret_cast<const uint4*>(k + j * row + c * 8) : zero;
    xv[u] = j < n ? *reinterpret_cast<const uint4*>(v + j * row + c * 8) : zero;
  }
  const uint4 xg = r < p.R ? *reinterpret_cast<const uint4*>(G + r * kFoldD + c * 8) : zero;
#pragma unroll
  for (int u = 0; u < kFoldSmall / 16; ++u) {
    *reinterpret_cast<uint4*>(sm.k + (r + u * 16) * kSmallLd + c * 8) = xk[u];
    *reinterpret_cast<uint4*>(sm.v + (r + u * 16) * kSmallLd + c * 8) = xv[u];
  }
  *reinterpret_cast<uint4*>(sm.g + r * kSmallLd + c * 8) = xg;
  __syncthreads();
  const int g = lane >> 2;
  for (int j0 = 8 * warp; j0 < n; j0 += 64) {                 // scores of eight keys
    float sc[4] = {};
#pragma unroll
    for (int kk = 0; kk < kFoldD; kk += 32) {
      uint32_t b[4], a[4];
      ldsm_x4(b, sm.k + (j0 + (lane & 7)) * kSmallLd + kk + (lane >> 3) * 8);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        ldsm_x4(a, sm.g + (lane & 15) * kSmallLd + kk + e * 16 + (lane >> 4) * 8);
        mma_bf16(sc, a, b[2 * e], b[2 * e + 1]);
      }
    }
    float* o = sm.s + g * kSmallSLd + j0 + 2 * (lane & 3);
    *reinterpret_cast<float2*>(o) = make_float2(sc[0], sc[1]);
    *reinterpret_cast<float2*>(o + 8 * kSmallSLd) = make_float2(sc[2], sc[3]);
  }
  __syncthreads();
  const float isd = rsqrtf((float)kFoldD), sl2 = 1.4426950408889634f * isd;
  float x[kFoldSmall / 16], mx = -INFINITY, sum = 0.f;
#pragma unroll
  for (int u = 0; u < kFoldSmall / 16; ++u) {
    x[u] = c + 16 * u < n ? sm.s[r * kSmallSLd + c + 16 * u] : -INFINITY;
    mx = fmaxf(mx, x[u]);
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (mx == -INFINITY) mx = 0.f;                              // no finite score
#pragma unroll
  for (int u = 0; u < kFoldSmall / 16; ++u) {
    x[u] = exp2f((x[u] - mx) * sl2);
    sum += x[u];
#pragma unroll
    for (int part = 0; part < 3; ++part) {                    // (g has been read)
      const bf16 y = __float2bfloat16_rn(x[u]);
      sm.p[part][r * kSmallPLd + c + 16 * u] = y;
      x[u] -= __bfloat162float(y);
    }
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (c == 0) {
    sm.sum[r] = sum;
    if (r < p.R) p.eta[q0 + r] = mx * isd + logf(sum);
  }
  __syncthreads();
  float o[2][4] = {};                                         // rows g and g + 8, dims 16 warp + 8 t + 2 (lane & 3) and the next
#pragma unroll
  for (int ks = 0; ks < kFoldSmall / 16; ++ks) {
    if (16 * ks >= n) break;
    uint32_t b[4], a[4];
    ldsm_x4_t(b, sm.v + (16 * ks + (lane & 15)) * kSmallLd + warp * 16 + (lane >> 4) * 8);
#pragma unroll
    for (int part = 2; part >= 0; --part) {
      ldsm_x4(a, sm.p[part] + (lane & 15) * kSmallPLd + 16 * ks + (lane >> 4) * 8);
      mma_bf16(o[0], a, b[0], b[1]);
      mma_bf16(o[1], a, b[2], b[3]);
    }
  }
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    const int q = g + 8 * hh;
    if (q >= p.R) continue;
    const float inv = 1.0f / sm.sum[q];
#pragma unroll
    for (int t = 0; t < 2; ++t)
      *reinterpret_cast<float2*>(p.m + (q0 + q) * kFoldD + warp * 16 + 8 * t + 2 * (lane & 3)) =
          make_float2(o[t][2 * hh] * inv, o[t][2 * hh + 1] * inv);
  }
}

// A prefill of at most kFoldSmall rows: CTA (layer, query head), then `ncopy` CTAs that copy
// the window and the boundary rows; CTA 0 sets t (a prefill reads none).  The two kernels
// below pay 11 to 14 us for tensor memory, records and the merge whatever the rows are,
// more than the mma.sync kernels before them.  Device time in us (those, the two below, this
// one): 5 layers of 32 heads 7.1, 13.8, 3.9 at 1 row, 11.8, 14.0, 5.5 at 84, 13.8, 13.6, 6.5 at 128;
// 3 layers of 8 heads 9.1, 11.0, 4.3 at 128 rows.
__global__ void __launch_bounds__(256) fold_small_kernel(const FoldParams p, const int ncopy) {
  extern __shared__ __align__(16) uint8_t small_raw[];
  griddep_launch();
  griddep_wait();
  const int nsum = (int)gridDim.x - ncopy;
  if (blockIdx.x == 0 && threadIdx.x == 0) p.t[p.b0] = p.rows;
  if ((int)blockIdx.x < nsum) {
    if (p.R > 0)
      fold_small(p, *reinterpret_cast<SmallSmem*>(small_raw), (int)blockIdx.x / p.nq, (int)blockIdx.x % p.nq);
    return;
  }
  int* srows = reinterpret_cast<int*>(small_raw);
  int* sslot = srows + 1;
  const int cta = (int)blockIdx.x - nsum, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = min(p.rows, p.W);
  if (threadIdx.x == 0) {
    srows[0] = p.rows;
    sslot[0] = p.W > 0 ? (p.rows - nw) % p.W : 0;
  }
  __syncthreads();
  long long chunk = (long long)cta * 8 + warp;
  fold_copy_window(p, nw, srows, sslot, lane, [&] {
    const long long c = chunk;
    chunk += (long long)ncopy * 8;
    return c;
  });
  if (p.h) fold_copy_boundary(p, srows, cta, ncopy, threadIdx.x, 256);
}

template <int REP, int PARTS>
__global__ void __launch_bounds__(kFoldThreads, 1)
    fold_tc_kernel(const __grid_constant__ CUtensorMap mk, const __grid_constant__ CUtensorMap mv, const FoldParams p) {
  constexpr int Q = 16 * REP, QH = 8 * REP;               // queries; a softmax thread's share of them
  constexpr int CW = REP <= 5 ? QH : (REP == 7 ? 8 : 16); // score columns a thread holds at a time
  constexpr FoldLayout L = fold_layout(REP, PARTS);
  constexpr int NS = L.slots, NB = (Q + 63) / 64;
  extern __shared__ uint8_t fsm_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(fsm_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const uint32_t s_g = smem_u32(sm), s_p = s_g + L.off_p, s_ring = s_g + L.off_ring;
  float* sref = reinterpret_cast<float*>(sm + L.off_misc);   // reference of each query
  float* sscale = sref + Q;                                  // factor of a reference that moved; at a piece's end 1 / sum
  float* sinv = sscale;
  int* pre = reinterpret_cast<int*>(sscale + Q);             // [65]
  int* srows = pre + 68;                                     // new rows of each request
  int* sslot = srows + kFoldMaxC;                            // and its first window slot
  uint64_t* bars = reinterpret_cast<uint64_t*>(sslot + kFoldMaxC);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 2 * kFoldMaxSlots + 8);
  volatile int* stop = reinterpret_cast<volatile int*>(tslot + 1);
  volatile int* sfresh = stop + 1;
  int* scopy = reinterpret_cast<int*>(tslot + 3);            // next chunk of the window copy
  float* exch = reinterpret_cast<float*>(sm + L.off_p);      // [4][Q] between warps, while P is idle
  const uint32_t bar0 = smem_u32(bars);
  auto b_full = [&](int s) { return bar0 + 8u * (uint32_t)s; };
  auto b_empty = [&](int s) { return bar0 + 8u * (uint32_t)(kFoldMaxSlots + s); };
  auto b_sfull = [&](int s) { return bar0 + 8u * (uint32_t)(2 * kFoldMaxSlots + s); };
  auto b_sempty = [&](int s) { return bar0 + 8u * (uint32_t)(2 * kFoldMaxSlots + 2 + s); };
  const uint32_t b_p = bar0 + 8u * (2 * kFoldMaxSlots + 4), b_pv = b_p + 8, b_g = b_p + 16, b_end = b_p + 24;

  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(b_full(s), 1);
      mbar_init(b_empty(s), 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(b_sfull(s), 1);
      mbar_init(b_sempty(s), kFoldSoftmax / 32);
    }
    mbar_init(b_p, kFoldSoftmax / 32);
    mbar_init(b_pv, 1);
    mbar_init(b_g, kFoldSoftmax / 32);
    mbar_init(b_end, 1);
    *stop = 0;
    *scopy = 0;
    fence_barrier_init();
    tma_prefetch_desc(&mk);
    tma_prefetch_desc(&mv);
  }
  if (warp == 9) tmem_alloc(smem_u32(tslot), fold_tmem_cols(REP));
  griddep_launch();
  griddep_wait();
  if (warp == 0) fold_prefix(p, pre, lane);
  if (warp == 1)
    for (int i = lane; i < p.nreq; i += 32) {
      const int n = fold_rows(p, i);
      srows[i] = n;
      sslot[i] = p.W > 0 ? (int)(((p.replace ? 0 : p.t[p.b0 + i]) + n - min(n, p.W)) % p.W) : 0;
    }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = uniform(*tslot), t_o = tmem + 2u * Q;
  const int LG = p.L * p.nkv;
  const long long total = (long long)pre[kFoldMaxC] * LG;
  const long long nshare = fold_shares(total, gridDim.x);
  const int f0 = (int)min(total, total * blockIdx.x / nshare), f1 = (int)min(total, total * (blockIdx.x + 1) / nshare);

  if (warp == 8) {
    // ------------------------------------------------------------ TMA producer
    const uint64_t pol = policy_evict_first();
    int q = 0;                                            // ring position: K and V of a block in turn
    bool ok = true;
    for (int f = f0; f < f1 && ok;) {
      const FoldPiece pc = fold_piece(pre, p.nreq, LG, f, f1);
      const int l = pc.lg / p.nkv, x = (pc.lg % p.nkv) * kFoldD;
      const int y0 = (pc.req * p.L + l) * p.rows + pc.blk * kFoldKeys;
      for (int i = 0; i < pc.n && ok; ++i)
        for (int kv = 0; kv < 2; ++kv, ++q) {
          const int s = q % NS;
          if (q >= NS && !fold_wait(b_empty(s), (uint32_t)(q / NS - 1) & 1u, stop, p.err)) { ok = false; break; }
          if (elect_one()) {
            mbar_expect_tx(b_full(s), kFoldSlot);
            const uint32_t dst = s_ring + (uint32_t)s * kFoldSlot;
            const CUtensorMap* mp = kv ? &mv : &mk;
            tma_load_2d(dst, mp, b_full(s), x, y0 + i * kFoldKeys, pol);
            tma_load_2d(dst + kFoldSlot / 2, mp, b_full(s), x + 64, y0 + i * kFoldKeys, pol);
          }
          __syncwarp();
        }
      f += pc.n;
    }
    // every load has landed before the CTA's shared memory goes away
    for (int i = max(0, q - NS); i < q; ++i) mbar_wait(b_full(i % NS), (uint32_t)(i / NS) & 1u, p.err);
  } else if (warp == 9) {
    // ------------------------------------------------------------ MMA issue
    const uint32_t id_s = fold_idesc(Q, false), id_o = fold_idesc(Q, true);
    int n = 0, piece = 0;                                 // block and piece of this CTA
    bool ok = true;
    auto scores = [&](int nn) {
      const int s = (2 * nn) % NS, buf = nn & 1;
      ok = ok && fold_wait(b_full(s), (uint32_t)(2 * nn / NS) & 1u, stop, p.err);
      if (nn >= 2) ok = ok && fold_wait(b_sempty(buf), (uint32_t)(nn / 2 - 1) & 1u, stop, p.err);
      if (!ok) return;
      tc_fence_after();
      const uint32_t sk = s_ring + (uint32_t)s * kFoldSlot;
      if (elect_one()) {
#pragma unroll
        for (int ks = 0; ks < kFoldD / 16; ++ks) {
          const uint32_t kb = (uint32_t)(ks >> 2), in = (uint32_t)(ks & 3) * 32u;
          umma_f16(tmem + (uint32_t)(buf * Q), sdesc_sw128(sk + kb * (kFoldSlot / 2) + in),
                   sdesc_sw128(s_g + kb * (uint32_t)(Q * 128) + in), id_s, ks > 0 ? 1u : 0u);
        }
        umma_commit(b_empty(s));
        umma_commit(b_sfull(buf));
      }
      __syncwarp();
    };
    for (int f = f0; f < f1; ++piece) {
      const FoldPiece pc = fold_piece(pre, p.nreq, LG, f, f1);
      ok = ok && fold_wait(b_g, (uint32_t)piece & 1u, stop, p.err);
      scores(n);
      for (int i = 0; i < pc.n; ++i, ++n) {
        if (i + 1 < pc.n) scores(n + 1);
        const int s = (2 * n + 1) % NS;
        ok = ok && fold_wait(b_full(s), (uint32_t)((2 * n + 1) / NS) & 1u, stop, p.err);
        ok = ok && fold_wait(b_p, (uint32_t)n & 1u, stop, p.err);
        if (!ok) continue;
        tc_fence_after();
        const uint32_t sv = s_ring + (uint32_t)s * kFoldSlot;
        const uint32_t keep = uniform(*sfresh ? 0u : 1u);   // fresh: the accumulator was drained
        if (elect_one()) {
          // remainders first: the accumulator is small while they are added, so the
          // bits that each MMA's addition drops are theirs
#pragma unroll
          for (int part = PARTS - 1; part >= 0; --part) {
#pragma unroll
            for (int ks = 0; ks < kFoldKeys / 16; ++ks)
              umma_f16(t_o, fold_desc_mn(sv + (uint32_t)ks * 2048u, kFoldSlot / 2),
                       fold_desc_mn(s_p + (uint32_t)(part * NB * 16384) + (uint32_t)ks * 2048u, 16384u), id_o,
                       part < PARTS - 1 || ks > 0 ? 1u : keep);
          }
          umma_commit(b_empty(s));
          umma_commit(b_pv);
        }
        __syncwarp();
      }
      f += pc.n;
    }
    if (elect_one()) umma_commit(b_end);                  // no MMA outlives the CTA's TMEM
    __syncwarp();
    mbar_wait(b_end, 0, p.err);
  } else if (warp < 8) {
    // ------------------------------------------------------------ softmax
    const int quad = warp & 3, half = warp >> 2;
    const int j = quad * 32 + lane;                       // key of the block (S), dim of the head (O)
    const uint32_t tl = (uint32_t)(quad * 32) << 16;
    const int c0 = half * QH;                             // first of this thread's queries
    const float isd = rsqrtf((float)kFoldD), sl2 = 1.4426950408889634f * isd;
    const uint32_t prow = s_p + (uint32_t)(j >> 3) * 1024u + (uint32_t)(j & 7) * 128u;
    auto bar = [] { named_bar(1, kFoldSoftmax); };
    // the queries' maxima (kMax) or sums over the block's 128 keys into out(query, value)
    auto across = [&](auto is_max, const float* x, int cbase, int n) {
#pragma unroll
      for (int c = 0; c < n; c += 8) {
        const float r = reduce8<decltype(is_max)::value>(x + c, lane);
        if (lane < 8) exch[quad * Q + cbase + c + lane] = r;
      }
    };

    auto load_g = [&](int lg) {
      const int l = lg / p.nkv, g = lg % p.nkv;
      const bf16* G = static_cast<const bf16*>(p.G) + ((size_t)l * p.nq + (size_t)g * REP) * p.R * kFoldD;
      uint4 v[REP];                                       // every load before the first store
#pragma unroll
      for (int u = 0; u < REP; ++u) {
        const int i = tid + u * kFoldSoftmax, row = i >> 4, c8 = i & 15, hh = row >> 4, r = row & 15;
        v[u] = make_uint4(0u, 0u, 0u, 0u);
        if (r < p.R) v[u] = *reinterpret_cast<const uint4*>(G + ((size_t)hh * p.R + r) * kFoldD + c8 * 8);
      }
#pragma unroll
      for (int u = 0; u < REP; ++u) {
        const int i = tid + u * kFoldSoftmax, row = i >> 4, c8 = i & 15;
        st_v4(s_g + (uint32_t)((c8 >> 3) * (Q * 128) + (row >> 3) * 1024 + (row & 7) * 128 + (((c8 & 7) ^ (row & 7)) << 4)),
              v[u].x, v[u].y, v[u].z, v[u].w);
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(b_g);
    };
    if (f0 < f1) load_g(fold_piece(pre, p.nreq, LG, f0, f1).lg);

    int n = 0;
    bool first_piece = true;
    for (int f = f0; f < f1;) {
      const FoldPiece pc = fold_piece(pre, p.nreq, LG, f, f1);
      if (!first_piece) load_g(pc.lg);                    // every score MMA of the last piece has completed
      first_piece = false;
      const int nrows = fold_rows(p, pc.req);
      float acc[QH], sum[QH];
#pragma unroll
      for (int c = 0; c < QH; ++c) acc[c] = sum[c] = 0.f;
      int since = 0;                                      // blocks in the accumulator
      auto drain = [&] {
        tc_fence_after();
        float o[CW];
#pragma unroll
        for (int cc = 0; cc < QH; cc += CW) {
          tmem_ld_cols(t_o + tl + (uint32_t)(c0 + cc), o);
#pragma unroll
          for (int c = 0; c < CW; ++c) acc[cc + c] += o[c];
        }
      };
      for (int i = 0; i < pc.n; ++i, ++n) {
        const int buf = n & 1;
        const int nvalid = nrows - (pc.blk + i) * kFoldKeys;   // rows of this block (may exceed 128)
        const bool valid = j < nvalid;
        fold_wait(b_sfull(buf), (uint32_t)(n >> 1) & 1u, stop, p.err);
        tc_fence_after();
        const uint32_t ts = tmem + tl + (uint32_t)(buf * Q + c0);
        float s[CW];
        auto load = [&](int cc) {
          tmem_ld_cols(ts + (uint32_t)cc, s);
          if (!valid) {
#pragma unroll
            for (int c = 0; c < CW; ++c) s[c] = -INFINITY;
          }
        };
        // does a score pass its reference by more than the slack?
        bool move = i == 0;
        if (i == 0) {
          if (CW == QH) load(0);
        } else {
          float mx = -INFINITY;
#pragma unroll
          for (int cc = 0; cc < QH; cc += CW) {
            load(cc);
#pragma unroll
            for (int c = 0; c < CW; c += 4) {
              const float4 r = *reinterpret_cast<const float4*>(sref + c0 + cc + c);
              mx = fmaxf(mx, fmaxf(fmaxf(s[c] - r.x, s[c + 1] - r.y), fmaxf(s[c + 2] - r.z, s[c + 3] - r.w)));
            }
          }
          move = softmax_any(mx * sl2 > kRefSlack);
          // P and the accumulator are free once the previous block's MMAs are done
          if (CW != QH || move || since == kFlushBlocks) fold_wait(b_pv, (uint32_t)(n - 1) & 1u, stop, p.err);
          if (move || since == kFlushBlocks) {
            drain();
            since = 0;
          }
        }
        if (move) {
#pragma unroll
          for (int cc = 0; cc < QH; cc += CW) {
            if (CW != QH) load(cc);
            across(std::true_type{}, s, c0 + cc, CW);
          }
          bar();
          if (tid < Q) {
            float m = fmaxf(fmaxf(exch[tid], exch[Q + tid]), fmaxf(exch[2 * Q + tid], exch[3 * Q + tid]));
            if (m == -INFINITY) m = 0.f;                  // no finite score yet
            const float old = i == 0 ? m : sref[tid];
            m = fmaxf(m, old);
            sscale[tid] = fold_ex2((old - m) * sl2);
            sref[tid] = m;
          }
          bar();
          if (i > 0) {
#pragma unroll
            for (int c = 0; c < QH; ++c) {
              const float a = sscale[c0 + c];
              acc[c] *= a;
              sum[c] *= a;
            }
          }
        }
        // P in PARTS bf16 parts, each the rounded rest of those before, eight queries a
        // 16-byte store; where a thread holds all its scores, P is formed under the
        // previous block's MMAs and waits for them only here
        auto weights = [&](int cc, int c, uint32_t (&w)[PARTS][4]) {
          const float4 ra = *reinterpret_cast<const float4*>(sref + c0 + cc + c);
          const float4 rb = *reinterpret_cast<const float4*>(sref + c0 + cc + c + 4);
          const float r[8] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w};
#pragma unroll
          for (int e = 0; e < 8; e += 2) {
            const float x0 = fold_ex2((s[c + e] - r[e]) * sl2), x1 = fold_ex2((s[c + e + 1] - r[e + 1]) * sl2);
            sum[cc + c + e] += x0;
            sum[cc + c + e + 1] += x1;
            float y0 = x0, y1 = x1;
#pragma unroll
            for (int part = 0; part < PARTS; ++part) {
              const uint32_t h = pack_bf16(y0, y1);
              w[part][e >> 1] = h;
              y0 -= __uint_as_float(h << 16);
              y1 -= __uint_as_float(h & 0xffff0000u);
            }
          }
        };
        auto store_p = [&](int col, const uint32_t (&w)[PARTS][4]) {
          const uint32_t a = prow + (uint32_t)(col >> 6) * 16384u + (uint32_t)((((col & 63) >> 3) ^ (j & 7)) << 4);
#pragma unroll
          for (int part = 0; part < PARTS; ++part)
            st_v4(a + (uint32_t)(part * NB * 16384), w[part][0], w[part][1], w[part][2], w[part][3]);
        };
        if constexpr (CW == QH) {
          uint32_t w[QH / 8][PARTS][4];
#pragma unroll
          for (int c = 0; c < QH; c += 8) weights(0, c, w[c / 8]);
          if (i > 0) fold_wait(b_pv, (uint32_t)(n - 1) & 1u, stop, p.err);
#pragma unroll
          for (int c = 0; c < QH; c += 8) store_p(c0 + c, w[c / 8]);
        } else {
#pragma unroll
          for (int cc = 0; cc < QH; cc += CW) {
            load(cc);
#pragma unroll
            for (int c = 0; c < CW; c += 8) {
              uint32_t w[PARTS][4];
              weights(cc, c, w);
              store_p(c0 + cc + c, w);
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(b_sempty(buf));
        if (nvalid < kFoldKeys) {
          // the unit's ragged end: rows past it may hold anything, and 0 x V has to stay 0
          const int vs = (2 * n + 1) % NS;
          fold_wait(b_full(vs), (uint32_t)((2 * n + 1) / NS) & 1u, stop, p.err);
          if (!valid) {
            const uint32_t a = s_ring + (uint32_t)vs * kFoldSlot + (uint32_t)half * (kFoldSlot / 2) + (uint32_t)j * 128u;
#pragma unroll
            for (int c = 0; c < 8; ++c) st_v4(a + (uint32_t)c * 16u, 0u, 0u, 0u, 0u);
          }
        }
        fence_proxy_async_smem();
        if (tid == 0) *sfresh = since == 0;
        ++since;
        __syncwarp();
        if (lane == 0) mbar_arrive(b_p);
      }
      // ---- the piece's (eta, m) of every query
      fold_wait(b_pv, (uint32_t)(n - 1) & 1u, stop, p.err);
      drain();
      tc_fence_before();
      across(std::false_type{}, sum, c0, QH);
      bar();
      float* rec = p.ws + (size_t)((int)blockIdx.x + pc.unit) * REP * kFoldRec;
      if (tid < Q) {
        const float t = (exch[tid] + exch[Q + tid]) + (exch[2 * Q + tid] + exch[3 * Q + tid]);
        sinv[tid] = 1.0f / t;
        rec[(tid >> 4) * kFoldRec + (tid & 15)] = sref[tid] * isd + logf(t);
      }
      bar();
#pragma unroll
      for (int c = 0; c < QH; ++c) {
        const int col = c0 + c;
        rec[(col >> 4) * kFoldRec + 16 + (col & 15) * kFoldD + j] = acc[c] * sinv[col];
      }
      f += pc.n;
    }
  }

  // ---- window ring and boundary rows: warps 10 and 11 from the start, and the softmax
  // warps once their blocks are done (a long fold hides the copy under its blocks, in
  // a short one it is most of the work), a chunk of the CTA's share at a time
  if (warp < 8 || warp >= 10) {
    if (p.acc && blockIdx.x == 0 && warp == 10)
      for (int i = lane; i < p.nreq; i += 32)
        if (p.acc[i] < 0 || p.acc[i] > p.rows) set_err(p.err, LSP_DEV_BAD_DELTA);
    const int n0 = lane < p.nreq ? srows[lane] : 0, n1 = lane + 32 < p.nreq ? srows[lane + 32] : 0;
    const int longest = min(__reduce_max_sync(0xffffffffu, max(n0, n1)), p.W);
    fold_copy_window(p, longest, srows, sslot, lane, [&] {
      const int c = lane == 0 ? atomicAdd(scopy, 1) : 0;
      return (long long)__shfl_sync(0xffffffffu, c, 0) * gridDim.x + blockIdx.x;
    });
    if (p.h && warp >= 10) fold_copy_boundary(p, srows, (int)blockIdx.x, (int)gridDim.x, tid - (kFoldSoftmax + 64), kFoldCopy);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tmem, fold_tmem_cols(REP));
  }
}

// One CTA per (request, layer, query head): 16 rows x 16 groups of 8 dims.
// The pieces' weights come from one pass over their eta, so their values are
// all in flight at once (a chain of two-way merges waited for each in turn).
// CTA 0 also advances t.
constexpr int kMergeBatch = 4;

__global__ void __launch_bounds__(256) fold_merge_kernel(const FoldParams p, const int grid) {
  __shared__ int pre[kFoldMaxC + 1];
  griddep_launch();
  griddep_wait();
  if (threadIdx.x < 32) fold_prefix(p, pre, threadIdx.x);
  __syncthreads();
  if (blockIdx.x == 0 && (int)threadIdx.x < p.nreq) {
    const int n = fold_rows(p, threadIdx.x);
    int64_t* t = p.t + p.b0 + threadIdx.x;
    if (p.replace) *t = n;
    else if (n > 0) *t += n;
  }
  const int i = blockIdx.x / (p.L * p.nq), lh = blockIdx.x % (p.L * p.nq);
  const int l = lh / p.nq, h = lh % p.nq;
  const int rep = p.nq / p.nkv, lg = l * p.nkv + h / rep, hh = h % rep;
  const int r = threadIdx.x >> 4, c0 = (threadIdx.x & 15) * 8;
  const int nb = pre[i + 1] - pre[i];
  if (r >= p.R || nb == 0) return;
  const long long LG = (long long)p.L * p.nkv, total = pre[kFoldMaxC] * LG;
  const long long f0 = pre[i] * LG + (long long)lg * nb, nshare = fold_shares(total, grid);
  const int s0 = (int)(((f0 + 1) * nshare - 1) / total), s1 = (int)(((f0 + nb) * nshare - 1) / total);
  const int unit = i * (int)LG + lg;
  auto rec = [&](int s) { return p.ws + ((size_t)(s + unit) * rep + hh) * kFoldRec; };
  const size_t q = (((size_t)(p.b0 + i) * p.L + l) * p.nq + h) * p.R + r;
  float* mo = p.m + q * kFoldD + c0;
  const float ea = p.replace ? -INFINITY : p.eta[q];
  float mx = ea;
  for (int s = s0; s <= s1; ++s) mx = fmaxf(mx, __ldcg(rec(s) + r));
  float w = 0.f, m[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) m[e] = 0.f;
  auto add = [&](float wt, const float4& a, const float4& b) {
    w += wt;
    const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int e = 0; e < 8; ++e) m[e] = fmaf(wt, v[e], m[e]);
  };
  if (!p.replace) add(expf(ea - mx), *reinterpret_cast<const float4*>(mo), *reinterpret_cast<const float4*>(mo + 4));
  for (int s = s0; s <= s1; s += kMergeBatch) {
    float4 a[kMergeBatch], b[kMergeBatch];
    float e[kMergeBatch];
#pragma unroll
    for (int u = 0; u < kMergeBatch; ++u)
      if (s + u <= s1) {
        const float* x = rec(s + u);
        e[u] = __ldcg(x + r);
        a[u] = __ldcg(reinterpret_cast<const float4*>(x + 16 + r * kFoldD + c0));
        b[u] = __ldcg(reinterpret_cast<const float4*>(x + 16 + r * kFoldD + c0 + 4));
      }
#pragma unroll
    for (int u = 0; u < kMergeBatch; ++u)
      if (s + u <= s1) add(expf(e[u] - mx), a[u], b[u]);
  }
  const float inv = 1.0f / w;
  *reinterpret_cast<float4*>(mo) = make_float4(m[0] * inv, m[1] * inv, m[2] * inv, m[3] * inv);
  *reinterpret_cast<float4*>(mo + 4) = make_float4(m[4] * inv, m[5] * inv, m[6] * inv, m[7] * inv);
  // this query's eta is read by its 16 threads, all of one half-warp, above
  __syncwarp(0xffffu << ((threadIdx.x & 16) ? 16 : 0));
  if ((threadIdx.x & 15) == 0) p.eta[q] = mx + logf(w);
}

template <int REP, int PARTS>
int launch_rep(const FoldParams& p, const CUtensorMap& mk, const CUtensorMap& mv, int grid, cudaStream_t s) {
  constexpr FoldLayout L = fold_layout(REP, PARTS);
  static_assert(L.bytes <= 227 * 1024, "one CTA's shared memory");
  static SmemOptIn once;
  if (smem_opt_in(once, fold_tc_kernel<REP, PARTS>, L.bytes) != cudaSuccess) return LSP_ERR_CUDA;
  return launch_pdl(fold_tc_kernel<REP, PARTS>, dim3(grid), dim3(kFoldThreads), L.bytes, s, mk, mv, p) == cudaSuccess
             ? LSP_OK
             : LSP_ERR_CUDA;
}

// Parts of P.  Two leave 2^-18 on a weight, 2.0e-6 on m against 64 bits whatever the
// length, three 1e-7 at 100 rows to 6e-7 at 60000.  Three are taken where two would be
// less exact than the kernel that the call took without this one: view updates whose
// 8 to 128 queries a KV head are no multiple of 16 (fp32 FMA: 6.2e-7 at 1126 rows, 40 queries,
// where two parts leave 2.1e-6 and three 5.1e-7), and folds so short that the mma.sync
// kernels' own two parts were their only error (prefill of 421, 1999, 4096, 60000 rows: 2.03e-6,
// 2.08e-6, 2.29e-6, 3.1e-6; update of 100, 200 rows: 1.79e-6, 1.96e-6).  Their cost, device
// time in us: 38.6 -> 41.8 at 40 queries and 4 x 1024 rows, prefill of 512 rows 15.1 -> 14.7,
// 2048 20.9 -> 22.0, 4096 28.5 -> 31.4 (the ring is one slot shorter, so that CTAs of the merge
// can wait on the SMs); prefill of 60000 rows it would be 124 -> 141.
int fold_parts(const FoldParams& p) {
  const bool fma = !p.replace && (p.nq / p.nkv * p.R) % 16 != 0;
  return fma || p.rows <= (p.replace ? 4096 : 256) ? 3 : 2;
}

template <int REP>
int launch_parts(const FoldParams& p, const CUtensorMap& mk, const CUtensorMap& mv, int grid, cudaStream_t s) {
  return fold_parts(p) == 3 ? launch_rep<REP, 3>(p, mk, mv, grid, s) : launch_rep<REP, 2>(p, mk, mv, grid, s);
}

}  // namespace

bool fold_supported(int dtype, int d, int R, int nq, int nkv) {
  return dtype == LSP_DTYPE_BF16 && d == kFoldD && R >= 0 && R <= 16 && nq / nkv <= 8;
}

// One record per query head for each (share, unit) pair a walk over the
// flattened blocks meets: at most one more than the shares for each unit.
size_t fold_ws_floats(int C, int L, int nq, int nkv, int num_sms) {
  return ((size_t)num_sms + (size_t)C * L * nkv) * (nq / nkv) * kFoldRec;
}

int launch_fold(const FoldParams& p, int num_sms, cudaStream_t s) {
  if (p.rows < 1 || p.nreq < 1 || p.nreq > kFoldMaxC || !p.ws) return LSP_ERR_UNSUPPORTED;
  if (p.H % 8) return LSP_ERR_SHAPE;
  // what the tensor maps refuse, also where none is made
  if ((reinterpret_cast<uintptr_t>(p.k) | reinterpret_cast<uintptr_t>(p.v)) & 15) return LSP_ERR_SHAPE;
  if (p.replace && p.rows <= kFoldSmall) {
    const int items = std::min(p.rows, p.W) * p.L * p.nkv * (kFoldD / 8);
    const int ncopy = std::max(p.L, (items + 8 * kCopyBatch * 32 - 1) / (8 * kCopyBatch * 32));
    constexpr size_t smem = sizeof(SmallSmem);
    static SmemOptIn once;
    if (smem_opt_in(once, fold_small_kernel, smem) != cudaSuccess) return LSP_ERR_CUDA;
    return launch_pdl(fold_small_kernel, dim3(p.L * p.nq + ncopy), dim3(256), smem, s, p, ncopy) == cudaSuccess ? LSP_OK
                                                                                                               : LSP_ERR_CUDA;
  }
  CUtensorMap mk, mv;
  const uint64_t rows = (uint64_t)p.nreq * p.L * p.rows, pitch = (uint64_t)p.nkv * kFoldD;
  int rc;
  if ((rc = tmap_2d_bf16_sw128(&mk, p.k, pitch, rows, pitch * 2, 64, kFoldKeys)) != LSP_OK) return rc;
  if ((rc = tmap_2d_bf16_sw128(&mv, p.v, pitch, rows, pitch * 2, 64, kFoldKeys)) != LSP_OK) return rc;
  // one CTA per SM, fewer when the capacity holds fewer blocks
  const long long blocks = (long long)p.nreq * p.L * p.nkv * ((p.rows + kFoldKeys - 1) / kFoldKeys);
  const int grid = (int)std::max(1ll, std::min((long long)num_sms, blocks));
  switch (p.nq / p.nkv) {
    case 1: rc = launch_parts<1>(p, mk, mv, grid, s); break;
    case 2: rc = launch_parts<2>(p, mk, mv, grid, s); break;
    case 3: rc = launch_parts<3>(p, mk, mv, grid, s); break;
    case 4: rc = launch_parts<4>(p, mk, mv, grid, s); break;
    case 5: rc = launch_parts<5>(p, mk, mv, grid, s); break;
    case 6: rc = launch_parts<6>(p, mk, mv, grid, s); break;
    case 7: rc = launch_parts<7>(p, mk, mv, grid, s); break;
    case 8: rc = launch_parts<8>(p, mk, mv, grid, s); break;
    default: return LSP_ERR_UNSUPPORTED;
  }
  if (rc != LSP_OK) return rc;
  return launch_pdl(fold_merge_kernel, dim3(p.nreq * p.L * p.nq), dim3(256), 0, s, p, grid) == cudaSuccess ? LSP_OK
                                                                                                           : LSP_ERR_CUDA;
}

}  // namespace lsp
