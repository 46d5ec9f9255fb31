// Markov correction + sequential proposal sampling (Eq. markov,
// Eq. proposal-factorization):  for i = 1..B in order,
//     z_i = z_i^(0) + W_c E_c(y_{i-1}),   y_0 = a,
//     y_i = argmax_v z_i[v]                      (temperature 0, greedy)
//     y_i = argmax_v (z_i[v] / T + g_{b,i,v})    (T > 0, Gumbel-max == sampling softmax(z_i / T))
// with g = -log(-log u) from Philox4x32-10 (Salmon et al., SC'11).
//
// Two kernels compute the same thing.
//
// sample_persistent_kernel (bf16, C <= 16, rc in {32, 64}, vocabulary slice
// fits shared memory): one cooperative launch for all B steps, one CTA per SM
// (32 CTAs for a small vocabulary).
// Each CTA owns a contiguous slice of 32-row vocabulary tiles and keeps its
// W_c rows resident in shared memory for the whole launch.  The requests form one
// or two groups of eight, which sixteen compute warps take in turn: the
// correction as mma.sync tiles with the vocabulary on M and the group's requests on N, base
// logits, noise, a running argmax.  A control warp of each group exchanges the
// CTA's best (value, index) with the other CTAs, learns y_i and gathers
// E_c(y_i) for the next step, and an I/O warp moves the corrected logits out and
// the next ones in, while the compute warps draw the next step's noise and score
// the other group.  The k index of the contraction is permuted
// identically in both operands so that each lane's operand words are
// contiguous in shared memory, and the vocabulary rows are permuted so that
// each lane's accumulators are four consecutive vocabulary entries of two requests (one
// Philox call, one float4 of logits each).
//
// sample_step_kernel (every other shape): one launch per step i: every CTA
// first finishes step i-1's argmax from the per-CTA partials (so y_{i-1} is
// known everywhere), gathers E_c(y_{i-1}) of all C requests into shared
// memory, then sweeps its share of 16-row vocabulary tiles: the correction
// W_c[v0:v0+16] E_c^T is one mma.sync tile per warp (bf16 in, fp32
// accumulate; fp32 storage uses FMA), the corrected logits are read/written
// as float4, one Philox call feeds four vocabulary entries, and a per-lane
// running argmax (ties to the lowest index) is reduced to one partial per CTA
// and request.  A last tiny launch resolves y_B.
#include <algorithm>

#include "common.cuh"
#include "lsp_internal.h"

namespace lsp {

constexpr int kSampThreads = 256;
constexpr int kSampWarps = kSampThreads / 32;
constexpr int kMaxC = 64;
constexpr int kMaxPartialsPerLane = 16;    // sampler grids of up to 512 CTAs


__device__ __forceinline__ bool better(float v, int i, float bv, int bi) {
  return v > bv || (v == bv && i < bi);
}

__device__ __forceinline__ void mma_bf16_s(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9},"
      " {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// argmax over the previous step's per-CTA partials of request b (one warp);
// partials are laid out [buf][b][block] so the lanes read consecutive blocks.
__device__ __forceinline__ int resolve_prev(const SampleParams& p, int buf, int b, int lane) {
  float bv = -INFINITY;
  int bi = 0x7fffffff;
  const float* pv = p.part_val + ((size_t)buf * p.C + b) * p.nblk;
  const int* pi = p.part_idx + ((size_t)buf * p.C + b) * p.nblk;
  // every load in flight before the first compare (nblk <= 32 * kMaxPartialsPerLane)
  float v[kMaxPartialsPerLane];
  int ix[kMaxPartialsPerLane];
#pragma unroll
  for (int k = 0; k < kMaxPartialsPerLane; ++k) {
    const int g = lane + 32 * k;
    v[k] = g < p.nblk ? pv[g] : -INFINITY;
    ix[k] = g < p.nblk ? pi[g] : 0x7fffffff;
  }
#pragma unroll
  for (int k = 0; k < kMaxPartialsPerLane; ++k)
    if (better(v[k], ix[k], bv, bi)) { bv = v[k]; bi = ix[k]; }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (better(ov, oi, bv, bi)) { bv = ov; bi = oi; }
  }
  return bi;
}

// KG = ceil(4 * C / 32): groups of four vocabulary entries each lane handles per tile.
template <typename T, int KG>
__global__ void __launch_bounds__(kSampThreads, 2) sample_step_kernel(const SampleParams p, const int step) {
  extern __shared__ __align__(16) uint8_t ssm_raw[];
  const int C = p.C, rc = p.rc;
  const int C8 = (C + 7) / 8 * 8;
  const int lde = rc + 8;                                   // padded row (elements)
  int* yprev = reinterpret_cast<int*>(ssm_raw);             // [kMaxC]
  float* red_v = reinterpret_cast<float*>(yprev + kMaxC);   // [warps][C]
  int* red_i = reinterpret_cast<int*>(red_v + kSampWarps * kMaxC);
  float* corr_s = reinterpret_cast<float*>(red_i + kSampWarps * kMaxC);   // [warps][C][17]
  T* e_s = reinterpret_cast<T*>(corr_s + kSampWarps * kMaxC * 17);        // [C8][lde]
  // per-warp double buffer of the 16 W_c rows of the current / next tile (bf16 path)
  bf16* wbuf = reinterpret_cast<bf16*>(e_s + (size_t)kMaxC * lde) + (size_t)(threadIdx.x >> 5) * 2 * 16 * lde;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  griddep_launch();
  griddep_wait();

  // ---- y_{i-1} for every request
  if (step == 0) {
    for (int b = tid; b < C; b += kSampThreads) {
      int y = p.prev[(size_t)b * p.prev_stride];
      if (y < 0 || y >= p.V) {
        if (blockIdx.x == 0) set_err(p.err, LSP_DEV_BAD_TOKEN);
        y = 0;
      }
      yprev[b] = y;
    }
  } else {
    for (int b = warp; b < C; b += kSampWarps) {
      const int y = resolve_prev(p, (step - 1) & 1, b, lane);
      if (lane == 0) {
        yprev[b] = y;
        if (blockIdx.x == 0) p.out_tokens[(size_t)b * p.B + step - 1] = y;
      }
    }
  }
  __syncthreads();
  // ---- E_c(y_{i-1}) rows
  const T* Ec = static_cast<const T*>(p.Ec);
  for (int idx = tid; idx < C8 * rc; idx += kSampThreads) {
    const int b = idx / rc, r = idx % rc;
    e_s[b * lde + r] = b < C ? Ec[(size_t)yprev[b] * rc + r] : from_f<T>(0.f);
  }
  __syncthreads();

  const T* Wc = static_cast<const T*>(p.Wc);
  const uint2 key = make_uint2((uint32_t)p.seed, (uint32_t)(p.seed >> 32));
  const bool sample = p.temperature > 0.f;
  const float inv_temp = sample ? 1.0f / p.temperature : 1.0f;   // exact for T = 1
  float* cw = corr_s + (size_t)warp * kMaxC * 17;
  float bv[KG];
  int bi[KG];
#pragma unroll
  for (int k = 0; k < KG; ++k) { bv[k] = -INFINITY; bi[k] = 0x7fffffff; }

  const int ntiles = p.V / 16;
  const int stride = gridDim.x * kSampWarps;
  auto zoff = [&](int tile, int k) {
    const int gi = lane + 32 * k;
    return ((size_t)(gi >> 2) * p.B + step) * p.V + tile * 16 + 4 * (gi & 3);
  };
  float4 zc[KG], zn[KG];
  int tile = blockIdx.x * kSampWarps + warp;
  // the 16 W_c rows of a tile -> this warp's buffer `buf` (16-byte cp.async chunks)
  auto stage_wc = [&](int t, int buf) {
    if constexpr (sizeof(T) == 2) {
      if (t < ntiles) {
        const int chunks = 16 * rc / 8;
        for (int c = lane; c < chunks; c += 32) {
          const int r = c / (rc / 8), e = (c % (rc / 8)) * 8;
          const bf16* src = reinterpret_cast<const bf16*>(Wc) + (size_t)(t * 16 + r) * rc + e;
          bf16* dst = wbuf + (size_t)buf * 16 * lde + (size_t)r * lde + e;
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
  };
  stage_wc(tile, 0);
#pragma unroll
  for (int k = 0; k < KG; ++k)
    if (tile < ntiles && lane + 32 * k < 4 * C) zc[k] = *reinterpret_cast<const float4*>(p.src + zoff(tile, k));
  int cur = 0;
  for (; tile < ntiles; tile += stride, cur ^= 1) {
    const int next = tile + stride;
    stage_wc(next, cur ^ 1);
#pragma unroll
    for (int k = 0; k < KG; ++k)
      if (next < ntiles && lane + 32 * k < 4 * C) zn[k] = *reinterpret_cast<const float4*>(p.src + zoff(next, k));
    const int v0 = tile * 16;
    // correction W_c[v0:v0+16] . E_c(y)^T for all requests -> cw[b][v]
    if constexpr (sizeof(T) == 2) {
      asm volatile("cp.async.wait_group 1;" ::: "memory");   // this tile's rows have landed
      __syncwarp();
      const bf16* es = reinterpret_cast<const bf16*>(e_s);
      const bf16* wr = wbuf + (size_t)cur * 16 * lde + (size_t)(lane >> 2) * lde + (lane & 3) * 2;
      float acc[KG][4];                                     // KG = ceil(C / 8) n-tiles of 8 requests
#pragma unroll
      for (int nt = 0; nt < KG; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
      for (int kk = 0; kk < rc / 16; ++kk) {
        uint32_t a[4];
        a[0] = *reinterpret_cast<const uint32_t*>(wr + kk * 16);
        a[1] = *reinterpret_cast<const uint32_t*>(wr + 8 * lde + kk * 16);
        a[2] = *reinterpret_cast<const uint32_t*>(wr + kk * 16 + 8);
        a[3] = *reinterpret_cast<const uint32_t*>(wr + 8 * lde + kk * 16 + 8);
#pragma unroll
        for (int nt = 0; nt < KG; ++nt) {
          const bf16* er = es + (size_t)(nt * 8 + (lane >> 2)) * lde + (lane & 3) * 2 + kk * 16;
          mma_bf16_s(acc[nt], a, *reinterpret_cast<const uint32_t*>(er),
                     *reinterpret_cast<const uint32_t*>(er + 8));
        }
      }
#pragma unroll
      for (int nt = 0; nt < KG; ++nt) {
        const int bcol = nt * 8 + (lane & 3) * 2, vr = lane >> 2;
        if (bcol < C) { cw[bcol * 17 + vr] = acc[nt][0]; cw[bcol * 17 + vr + 8] = acc[nt][2]; }
        if (bcol + 1 < C) { cw[(bcol + 1) * 17 + vr] = acc[nt][1]; cw[(bcol + 1) * 17 + vr + 8] = acc[nt][3]; }
      }
    } else {
      for (int idx = lane; idx < 16 * C; idx += 32) {
        const int v = idx & 15, b = idx >> 4;
        const T* wrow = Wc + (size_t)(v0 + v) * rc;
        const T* er = e_s + (size_t)b * lde;
        float acc = 0.f;
        for (int r = 0; r < rc; ++r) acc = fmaf(to_f(wrow[r]), to_f(er[r]), acc);
        cw[b * 17 + v] = acc;
      }
    }
    __syncwarp();
    // corrected logits, noise and running argmax: lane handles groups of 4 entries
#pragma unroll
    for (int k = 0; k < KG; ++k) {
      const int gi = lane + 32 * k;
      if (gi < 4 * C) {
        const int b = gi >> 2, vq = gi & 3;
        const int v = v0 + 4 * vq;
        float4 z = zc[k];
        z.x += cw[b * 17 + 4 * vq + 0];
        z.y += cw[b * 17 + 4 * vq + 1];
        z.z += cw[b * 17 + 4 * vq + 2];
        z.w += cw[b * 17 + 4 * vq + 3];
        if (p.dst) *reinterpret_cast<float4*>(p.dst + zoff(tile, k)) = z;
        float sc[4] = {z.x, z.y, z.z, z.w};
        if (sample) {
          const uint4 x = philox4x32_10(make_uint4((uint32_t)(v >> 2), (uint32_t)step, (uint32_t)(p.b0 + b), p.round), key);
          sc[0] = sc[0] * inv_temp + gumbel_of(x.x);
          sc[1] = sc[1] * inv_temp + gumbel_of(x.y);
          sc[2] = sc[2] * inv_temp + gumbel_of(x.z);
          sc[3] = sc[3] * inv_temp + gumbel_of(x.w);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (better(sc[e], v + e, bv[k], bi[k])) { bv[k] = sc[e]; bi[k] = v + e; }
      }
    }
    __syncwarp();                                           // wbuf[cur] is refilled next iteration
#pragma unroll
    for (int k = 0; k < KG; ++k) zc[k] = zn[k];
  }
  if constexpr (sizeof(T) == 2) asm volatile("cp.async.wait_all;" ::: "memory");

  // ---- per-CTA partial argmax of every request
#pragma unroll
  for (int k = 0; k < KG; ++k) {
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, bv[k], o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi[k], o);
      if (better(ov, oi, bv[k], bi[k])) { bv[k] = ov; bi[k] = oi; }
    }
    const int b = (lane >> 2) + 8 * k;
    if ((lane & 3) == 0 && b < C) {
      red_v[warp * kMaxC + b] = bv[k];
      red_i[warp * kMaxC + b] = bi[k];
    }
  }
  __syncthreads();
  for (int b = tid; b < C; b += kSampThreads) {
    float v = red_v[b];
    int i = red_i[b];
    for (int w = 1; w < kSampWarps; ++w)
      if (better(red_v[w * kMaxC + b], red_i[w * kMaxC + b], v, i)) {
        v = red_v[w * kMaxC + b];
        i = red_i[w * kMaxC + b];
      }
    const size_t o = ((size_t)(step & 1) * C + b) * p.nblk + blockIdx.x;
    p.part_val[o] = v;
    p.part_idx[o] = i;
  }
}

// ------------------------------------------------------------------ persistent kernel
constexpr int kPWarps = 16;                          // compute warps
// A vocabulary of few tiles goes to 32 CTAs, and every CTA reads all keys itself, a lane a
// CTA: one hop through L2 instead of two, and fewer words to poll.  Beyond, all SMs and
// leaders.  The lines are where both take about the same time (us, B = 8, 32 CTAs against
// 152): one group of requests, C = 8, 23.2 and 26.8 at V = 6400, 25.1 and 26.7 at 9984, 26.9 and
// 27.2 at 16000 (T = 0; T = 1: 29.1 and 27.3); two, C = 16, 25.1 and 29.1 at 4096, 27.1 and 29.4 at 8000,
// 31.4 and 29.4 at 16000 (T = 1: 35.5 and 30.8).
constexpr int kPFewCtas = 32;
__host__ __device__ constexpr int few_pairs(int groups) { return kPFewCtas * (groups == 1 ? 10 : 8); }
constexpr int kPMaxGroups = 2;                       // request groups of eight
constexpr int kPPairsPerWarp = 2;
constexpr int kPMaxPairs = kPWarps * kPPairsPerWarp; // 32-row vocabulary tiles a CTA: 1024 rows
constexpr int kPGroup = 8;                           // requests of a group (mma N)
constexpr int kPMaxC = kPGroup * kPMaxGroups;
constexpr int kIdxBits = 20, kTagBits = 12;          // low half of an exchanged key: ~index, step tag
constexpr int kAnsCopies = 4;                        // copies of the answers
constexpr int kLineWords = 16;                       // 64-bit words of a 128-byte line
constexpr int kLeadBatch = 5;                        // slots a leader's lane has in flight (152 CTAs in one go)
// named barriers of the compute warps with one more warp: 1 + group, a step's keys (-> control); 3 + group,
// E_c(y) (control ->); 5 + group, a step's corrected rows (-> I/O)
constexpr int kPBar = (kPWarps + 1) * 32;
// Floats between two requests' logits rows in shared memory: 16 bytes of padding
// put the four requests that lanes read together on different banks.
__host__ __device__ inline int z_pitch(int tpc) { return tpc * 32 + 4; }

// Order-preserving 64-bit key of (value, index): a larger value wins, equal
// values go to the lower index; -0 ranks as +0.
__device__ __forceinline__ unsigned long long arg_key(float v, int i) {
  uint32_t u = __float_as_uint(v);
  if (u == 0x80000000u) u = 0u;
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  return ((unsigned long long)u << 32) | (uint32_t)~(uint32_t)i;
}

__device__ __forceinline__ unsigned long long max_u64(unsigned long long a, unsigned long long b) {
  return a > b ? a : b;
}

// The warp's largest key, in every lane: the value half, then the index half of
// the lanes that hold it.
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long k) {
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32) == hi ? (unsigned)k : 0u);
  return ((unsigned long long)hi << 32) | lo;
}

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Four words of a 32-byte sector at once (each one of them relaxed).
__device__ __forceinline__ void ld_relaxed_4xu64(const unsigned long long* p, unsigned long long* v) {
  asm volatile("ld.relaxed.gpu.global.v4.u64 {%0, %1, %2, %3}, [%4];"
               : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3])
               : "l"(p)
               : "memory");
}

__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void named_arrive(int id, int count) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// Control warp: E_c rows of the group's current tokens (lane r < C holds y_r)
// into Es, 16-byte chunk c of row r stored at chunk c ^ (r & 1).
template <int CH>
__device__ __forceinline__ void gather_e(const bf16* Ec, int y, int C, int rc, uint8_t* Es, int lane) {
  uint4 v[(kPGroup * CH + 31) / 32];
#pragma unroll
  for (int i0 = 0; i0 < kPGroup * CH; i0 += 32) {
    const int i = i0 + lane, r = i / CH, c = i % CH;
    const int yr = __shfl_sync(0xffffffffu, y, r & 31);
    if (r < C) v[i0 / 32] = *reinterpret_cast<const uint4*>(Ec + (size_t)yr * rc + c * 8);
  }
#pragma unroll
  for (int i0 = 0; i0 < kPGroup * CH; i0 += 32) {
    const int i = i0 + lane, r = i / CH, c = i % CH;
    if (r < C) *reinterpret_cast<uint4*>(Es + r * (CH * 16) + ((c ^ (r & 1)) * 16)) = v[i0 / 32];
  }
}

// Where row r of the W_c slice sits: rows r and r + 4, which neighbouring lane
// groups read together, are adjacent (and swizzled against each other).
__device__ __forceinline__ int wc_pos(int r) { return (r & ~7) + 2 * (r & 3) + ((r >> 2) & 1); }

// KS = rc / 16 k-steps of the m16n8k16 contraction; NG groups of up to eight
// requests: 16 compute warps, then a control warp and an I/O warp a group (20 warps:
// 96 registers a thread).
template <int KS, int NG>
__global__ void __launch_bounds__((kPWarps + 4) * 32, 1)
    sample_persistent_kernel(const SampleParams p, const int npairs) {
  constexpr int RB = KS * 32;        // bytes of one W_c / E_c row
  constexpr int CH = RB / 16;        // 16-byte chunks per row
  constexpr int TCH = KS / 2;        // chunks of one lane's k range
  constexpr int kThreads = (kPWarps + 2 * NG) * 32;
  extern __shared__ __align__(128) uint8_t psm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nblk = gridDim.x;
  const int t_begin = (int)(((long long)blockIdx.x * npairs) / nblk);
  const int cnt = (int)(((long long)(blockIdx.x + 1) * npairs) / nblk) - t_begin;
  const int tpc = (npairs + nblk - 1) / nblk;
  const int zpitch = z_pitch(tpc);                                      // floats
  uint8_t* Ws = psm;                                                    // [tpc*32][RB]
  float* Zs = reinterpret_cast<float*>(psm + (size_t)tpc * 32 * RB);    // [NG][8][zpitch]
  uint8_t* Es = reinterpret_cast<uint8_t*>(Zs + (size_t)NG * kPGroup * zpitch);              // [NG][8][RB]
  unsigned long long* red = reinterpret_cast<unsigned long long*>(Es + NG * kPGroup * RB);   // [NG][warps][8]
  unsigned long long* zbar = red + NG * kPWarps * kPGroup;                        // [NG] the group's logits have landed
  const bf16* Wc = static_cast<const bf16*>(p.Wc);
  const bf16* Ec = static_cast<const bf16*>(p.Ec);
  const int C = p.C, B = p.B, V = p.V, rc = p.rc;
  const bool sample = p.temperature > 0.f;
  const float inv_temp = sample ? 1.0f / p.temperature : 1.0f;
  const uint2 key = make_uint2((uint32_t)p.seed, (uint32_t)(p.seed >> 32));
  const int g = lane >> 2, q = lane & 3;                               // mma group / thread in group

  // ---- prologue: W_c slice, zero E rows, y_0, E_c(y_0)
  for (int i = tid; i < cnt * 32 * CH; i += kThreads) {
    const int r = i / CH, c = i % CH, pos = wc_pos(r);
    if (t_begin * 32 + r < V) cp_async16(Ws + pos * RB + ((c ^ (pos & 1)) * 16), Wc + (size_t)(t_begin * 32 + r) * rc + c * 8);
  }
  for (int i = tid; i < NG * kPGroup * RB / 16; i += kThreads)
    reinterpret_cast<uint4*>(Es)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    for (int h = 0; h < NG; ++h) mbar_init(smem_u32(zbar + h), 1);
    fence_barrier_init();
  }
  // E_c rows are gathered at random every step: keep the table in L2 (this CTA's share)
  if (tid == kPWarps * 32) {
    const size_t bytes = (size_t)V * rc * 2;
    const size_t share = (bytes / nblk + 4095) / 4096 * 4096;
    const size_t lo = share * blockIdx.x, hi = lo + share < bytes ? lo + share : bytes;
    const uint64_t pol = policy_evict_last();
    for (size_t o = lo; o < hi; o += 4096) {
      const uint32_t n = (uint32_t)(hi - o < 4096 ? hi - o : 4096);
      asm volatile("cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;" ::"l"(
                       reinterpret_cast<const char*>(Ec) + o),
                   "r"(n), "l"(pol)
                   : "memory");
    }
  }

  // A lane's four vocabulary entries of local tile lt start at v_of(lt); its
  // requests of group h are 8 h + 2 q + e, e = 0, 1.
  auto v_of = [&](int lt) { return (t_begin + lt) * 32 + 4 * g; };
  float gn[kPPairsPerWarp][NG][2][4];      // noise of the step about to be scored
  auto draw_noise_tile = [&](int s, int j, int lt, int h) {
    const int v = v_of(lt);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (e == 1 && h * kPGroup + 1 >= C) break;                        // one request in the group
      const uint4 x = philox4x32_10(make_uint4((uint32_t)(v >> 2), (uint32_t)s, (uint32_t)(p.b0 + h * kPGroup + 2 * q + e), p.round), key);
      gn[j][h][e][0] = gumbel_of(x.x);
      gn[j][h][e][1] = gumbel_of(x.y);
      gn[j][h][e][2] = gumbel_of(x.z);
      gn[j][h][e][3] = gumbel_of(x.w);
    }
  };
#pragma unroll
  for (int j = 0; j < kPPairsPerWarp; ++j)
#pragma unroll
    for (int h = 0; h < NG; ++h)
#pragma unroll
      for (int e = 0; e < 2; ++e) gn[j][h][e][0] = gn[j][h][e][1] = gn[j][h][e][2] = gn[j][h][e][3] = 0.f;

  const bool control = warp >= kPWarps && warp < kPWarps + NG;
  const int grp = warp < kPWarps ? 0 : (warp - kPWarps) % NG;           // control and I/O warps: their group
  const int Cg = min(kPGroup, C - grp * kPGroup);
  int y = 0;                                                            // control warps: y of request `lane`
  unsigned epoch = 0;
  if (control) {
    epoch = *reinterpret_cast<volatile unsigned*>(p.sync);              // before any CTA can end
    if (lane < Cg) {
      y = p.prev[(size_t)(grp * kPGroup + lane) * p.prev_stride];
      if (y < 0 || y >= V) {
        if (blockIdx.x == 0) set_err(p.err, LSP_DEV_BAD_TOKEN);
        y = 0;
      }
    }
  }
  __syncthreads();                                                      // E rows zeroed, barriers ready
  if (control) gather_e<CH>(Ec, y, Cg, rc, Es + grp * kPGroup * RB, lane);
  // this CTA's slice of a logits row
  const size_t first = (size_t)t_begin * 32;
  const uint32_t zrow = (uint32_t)(min((size_t)cnt * 32, (size_t)V - first) * sizeof(float));
  // I/O warp: rows of step s into the group's buffer (lane r: its request's row)
  auto load_rows = [&](int s) {
    const uint32_t bar = smem_u32(zbar + grp);
    if (lane == 0) mbar_expect_tx(bar, zrow * (uint32_t)Cg);
    __syncwarp();
    if (lane < Cg)
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                       smem_u32(Zs + (size_t)(grp * kPGroup + lane) * zpitch)),
                   "l"(p.src + ((size_t)(grp * kPGroup + lane) * B + s) * V + first), "r"(zrow), "r"(bar)
                   : "memory");
  };
  if (warp >= kPWarps + NG) load_rows(0);
  if (warp < kPWarps && sample) {
#pragma unroll
    for (int j = 0; j < kPPairsPerWarp; ++j)
#pragma unroll
      for (int h = 0; h < NG; ++h)
        if (warp + kPWarps * j < cnt) draw_noise_tile(0, j, warp + kPWarps * j, h);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();                                                      // W_c slice and E_c(y_0) visible

  if (warp < kPWarps) {
    // ================= compute warps: the groups in turn, so that one group's
    // exchange and logits traffic run under the other's scoring and noise.  Every
    // role passes the same barriers in every step, whatever happens: a control warp
    // that gives up waiting goes on without the exchange, so no warp is ever left
    // at a barrier that another has not reached.
    for (int s = 0; s < B; ++s) {
      const bool more = s + 1 < B;
#pragma unroll
      for (int h = 0; h < NG; ++h) {
        if (s > 0) named_bar(3 + h, kPBar);
        // B operand: E_c(y) row g of the group over this lane's k range
        uint32_t eb[2 * KS];
#pragma unroll
        for (int c = 0; c < TCH; ++c) {
          const uint4 u = *reinterpret_cast<const uint4*>(Es + (h * kPGroup + g) * RB + (((TCH * q + c) ^ (g & 1)) * 16));
          eb[4 * c] = u.x; eb[4 * c + 1] = u.y; eb[4 * c + 2] = u.z; eb[4 * c + 3] = u.w;
        }
        mbar_wait(smem_u32(zbar + h), (uint32_t)s & 1u, p.err);         // z_s landed
        float bv[2] = {-INFINITY, -INFINITY};
        int bi[2] = {v_of(warp), v_of(warp)};
#pragma unroll
        for (int j = 0; j < kPPairsPerWarp; ++j) {
          const int lt = warp + kPWarps * j;
          if (lt >= cnt) break;                                         // warp-uniform
          const int v = v_of(lt);
          // row g (+ 8) of m-tile t is vocabulary row 4 g + 2 t (+ 1): a lane's
          // accumulators are four consecutive entries of two requests
          float acc[2][4];
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            uint32_t w0[2 * KS], w1[2 * KS];
            const int pos = lt * 32 + (g >> 1) * 8 + 4 * t + (g & 1);
#pragma unroll
            for (int c = 0; c < TCH; ++c) {
              const int pc = ((TCH * q + c) ^ (g & 1)) * 16;
              const uint4 u0 = *reinterpret_cast<const uint4*>(Ws + pos * RB + pc);
              const uint4 u1 = *reinterpret_cast<const uint4*>(Ws + (pos + 2) * RB + pc);
              w0[4 * c] = u0.x; w0[4 * c + 1] = u0.y; w0[4 * c + 2] = u0.z; w0[4 * c + 3] = u0.w;
              w1[4 * c] = u1.x; w1[4 * c + 1] = u1.y; w1[4 * c + 2] = u1.z; w1[4 * c + 3] = u1.w;
            }
            acc[t][0] = acc[t][1] = acc[t][2] = acc[t][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
              const uint32_t a[4] = {w0[2 * ks], w1[2 * ks], w0[2 * ks + 1], w1[2 * ks + 1]};
              mma_bf16_s(acc[t], a, eb[2 * ks], eb[2 * ks + 1]);
            }
          }
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            float4* zp = reinterpret_cast<float4*>(Zs + (size_t)(h * kPGroup + 2 * q + e) * zpitch + lt * 32 + 4 * g);
            const float4 z = *zp;
            float zc[4] = {z.x + acc[0][e], z.y + acc[0][2 + e], z.z + acc[1][e], z.w + acc[1][2 + e]};
            if (p.dst) *zp = make_float4(zc[0], zc[1], zc[2], zc[3]);   // the I/O warp stores the row
            if (sample) {
#pragma unroll
              for (int i = 0; i < 4; ++i) zc[i] = zc[i] * inv_temp + gn[j][h][e][i];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (zc[i] > bv[e] && v < V) { bv[e] = zc[i]; bi[e] = v + i; }
          }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          unsigned long long k = warp < cnt && bi[e] < V ? arg_key(bv[e], bi[e]) : 0ull;
          k = max_u64(k, __shfl_xor_sync(0xffffffffu, k, 4));
          k = max_u64(k, __shfl_xor_sync(0xffffffffu, k, 8));
          k = max_u64(k, __shfl_xor_sync(0xffffffffu, k, 16));
          if (g == 0) red[(h * kPWarps + warp) * kPGroup + 2 * q + e] = k;
        }
        named_arrive(1 + h, kPBar);
        fence_proxy_async_smem();                                       // the row buffers go to the async proxy
        named_arrive(5 + h, kPBar);
        if (more && sample) {
#pragma unroll
          for (int j = 0; j < kPPairsPerWarp; ++j)
            if (warp + kPWarps * j < cnt) draw_noise_tile(s + 1, j, warp + kPWarps * j, h);
        }
      }
    }
    return;
  }

  if (warp >= kPWarps + NG) {
    // ================= I/O warp of group grp: the corrected rows out and the next
    // ones in by bulk copies, a row a lane, so that no compute warp waits on
    // the memory system (their vector stores and loads took 2.6 us a step at
    // 16 requests, the bandwidth's time, with nothing under them)
    for (int s = 0; s < B; ++s) {
      named_bar(5 + grp, kPBar);
      if (lane < Cg && p.dst) {
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                         p.dst + ((size_t)(grp * kPGroup + lane) * B + s) * V + first),
                     "r"(smem_u32(Zs + (size_t)(grp * kPGroup + lane) * zpitch)), "r"(zrow)
                     : "memory");
        bulk_commit();
        bulk_wait_read<0>();
      }
      __syncwarp();
      if (s + 1 < B) load_rows(s + 1);
    }
    return;
  }

  // ================= control warp of group grp
  // The exchange carries its own evidence: a CTA's best (value, index) of a
  // request is one 64-bit word with the step's tag in its low bits, written with a
  // plain store into the CTA's slot.  The request's leader (CTA r leads request r,
  // round robin where there are fewer CTAs) reads its slots until all tags are the step's,
  // and answers with a tagged word that every CTA reads: no counter, no
  // fence and no atomic, so the words do not queue behind the step's logits
  // traffic (the atomic key, release add and count of before: 3.6 + 1.3 us a step at
  // T = 1).  Each answer has a 128-byte line of its own, in kAnsCopies copies that the
  // CTAs share: answers of several leaders in one line, which every CTA polls, are stored
  // one after the other wherever the line's home is the far die (C = 16, V = 151936, B = 8
  // T = 0: 49 or 68 us by the page that the workspace had got, now 50 on any).
  // Slots alternate between two sets: a CTA writes step s + 2 only after
  // the answer of step s + 1, which its leader gives after reading step s (without
  // leaders: after every CTA's word of step s + 1).
  // Tags go on from launch to launch (the epoch word), so nothing is cleared.
  unsigned long long* answers = p.slots;                                // [2][kAnsCopies][kPMaxC], a line each
  constexpr unsigned long long kTagMask = (1ull << kTagBits) - 1;
  const int r0 = grp * kPGroup;
  const bool direct = nblk <= kPFewCtas;
  // direct: a CTA's words lie together, in a 32-byte sector up to four requests and a line
  // of their own beyond: one store and one or two loads for all requests.  (As rows of a
  // request, 16 CTAs a line: 23 or 29 us by the page at C = 8, V = 8000, B = 8, 23 now.)
  const int cw = Cg <= 4 ? 4 : kLineWords;
  bool ok = true;                                                       // false: a wait has given up
  for (int s = 0; s < B; ++s) {
    const unsigned long long tag = (unsigned long long)(epoch + s + 1) & kTagMask;
    unsigned long long* slots = p.slots + 2 * kAnsCopies * kPMaxC * kLineWords + (size_t)(s & 1) * C * nblk;   // [request][CTA]
    unsigned long long* lines = p.slots + (size_t)((s & 1) * kPMaxGroups + grp) * kPFewCtas * kLineWords;   // direct: [CTA][cw]
    unsigned long long* ans = answers + (s & 1) * kAnsCopies * kPMaxC * kLineWords;
    const bool last = s + 1 == B;
    named_bar(1 + grp, kPBar);
    if (!ok) {                                                          // nothing is published any more; the others' waits end too
      if (!last) named_arrive(3 + grp, kPBar);
      continue;
    }
    if (lane < Cg) {
      unsigned long long k = 0ull;
#pragma unroll
      for (int w = 0; w < kPWarps; ++w) k = max_u64(k, red[(grp * kPWarps + w) * kPGroup + lane]);
      st_relaxed_u64(direct ? lines + (int)blockIdx.x * cw + lane : slots + (size_t)(r0 + lane) * nblk + blockIdx.x,
                     (k & 0xffffffff00000000ull) | ((k & ((1ull << kIdxBits) - 1)) << kTagBits) | tag);
    }
    __syncwarp();
    unsigned long long k = tag;                                         // lane r: the best key of request r0 + r
    if (direct) {
      // ---- few CTAs: one lane a CTA, all requests at once, no leader
      const bool writes = (int)blockIdx.x < Cg || nblk < Cg;            // (block 0 writes in both groups)
      if (!last || writes) {
        unsigned long long v[kPGroup];
        const unsigned long long* w = lines + min(lane, nblk - 1) * cw;
        auto poll = [&](auto load) {
          const uint64_t t0 = global_ns();
          for (uint32_t it = 1;; ++it) {
            bool all = true;
            load();
#pragma unroll
            for (int u = 0; u < kPGroup; ++u) {
              if (u >= Cg) v[u] = tag;
              all = all && (v[u] & kTagMask) == tag;
            }
            if (__all_sync(0xffffffffu, all)) return true;
            if ((it & 63u) == 0 && __any_sync(0xffffffffu, global_ns() - t0 > kWaitLimitNs)) return false;
          }
        };
        ok = Cg <= 4 ? poll([&] { ld_relaxed_4xu64(w, v); })
                     : poll([&] { ld_relaxed_4xu64(w, v); ld_relaxed_4xu64(w + 4, v + 4); });
#pragma unroll
        for (int u = 0; u < kPGroup; ++u) {
          const unsigned long long best = warp_max_key(v[u]);
          if (lane == u) k = best;
        }
        if (ok && lane < Cg && lane % nblk == (int)blockIdx.x) {
          const int t = (int)(~(uint32_t)(k >> kTagBits) & ((1u << kIdxBits) - 1));
          p.out_tokens[(size_t)(r0 + lane) * B + s] = t < V ? t : 0;
        }
      }
    } else {
      // ---- leader: the best of all CTAs
      for (int r = r0 + ((int)blockIdx.x - r0 % nblk + nblk) % nblk; r < r0 + Cg && ok; r += nblk) {
        unsigned long long best = 0ull;
        for (int c0 = 0; c0 < nblk && ok; c0 += 32 * kLeadBatch) {
          unsigned long long k[kLeadBatch];
          const uint64_t t0 = global_ns();
          for (uint32_t it = 1;; ++it) {
            bool all = true;
#pragma unroll
            for (int u = 0; u < kLeadBatch; ++u) {
              const int c = c0 + u * 32 + lane;
              k[u] = c < nblk ? ld_relaxed_u64(slots + (size_t)r * nblk + c) : tag;
            }
#pragma unroll
            for (int u = 0; u < kLeadBatch; ++u) all = all && (k[u] & kTagMask) == tag;
            if (__all_sync(0xffffffffu, all)) break;
            if ((it & 63u) == 0 && __any_sync(0xffffffffu, global_ns() - t0 > kWaitLimitNs)) { ok = false; break; }
          }
#pragma unroll
          for (int u = 0; u < kLeadBatch; ++u) best = max_u64(best, k[u]);
        }
        best = warp_max_key(best);
        if (ok && lane < kAnsCopies) st_relaxed_u64(ans + (lane * kPMaxC + r) * kLineWords, best);
        if (ok && lane == 0) {
          const int t = (int)(~(uint32_t)(best >> kTagBits) & ((1u << kIdxBits) - 1));
          p.out_tokens[(size_t)r * B + s] = t < V ? t : 0;
        }
      }
      // ---- everyone: the answers
      if (ok && !last) {
        const uint64_t t0 = global_ns();
        for (uint32_t it = 1;; ++it) {
          if (lane < Cg) k = ld_relaxed_u64(ans + (((int)blockIdx.x % kAnsCopies) * kPMaxC + r0 + lane) * kLineWords);
          if (__all_sync(0xffffffffu, (k & kTagMask) == tag)) break;
          if ((it & 63u) == 0 && __any_sync(0xffffffffu, global_ns() - t0 > kWaitLimitNs)) { ok = false; break; }
        }
      }
    }
    if (!ok && lane == 0) set_err(p.err, LSP_DEV_TIMEOUT);
    if (last) break;
    if (ok) {
      y = (int)(~(uint32_t)(k >> kTagBits) & ((1u << kIdxBits) - 1));
      if (y >= V) y = 0;                                                // (no entry of the row compared)
      gather_e<CH>(Ec, y, Cg, rc, Es + grp * kPGroup * RB, lane);
    }
    __syncwarp();
    named_arrive(3 + grp, kPBar);
  }
  // every CTA has read the epoch before its first keys, and those have arrived here
  if (ok && blockIdx.x == 0 && grp == 0 && lane == 0) *reinterpret_cast<volatile unsigned*>(p.sync) = epoch + (unsigned)B;
}

// ------------------------------------------------------------------ persistent kernel, fp32 storage
// One cooperative launch for all B steps with fp32 W_c / E_c (the fp32
// reference shape): CTA k owns 16-row vocabulary tiles [t_begin, t_begin +
// cnt) and keeps their W_c rows resident in shared memory (a float4 of padding puts
// the rows that lanes read together on different banks).  A warp takes its
// requests through all steps on its own: its lanes form z = z^(0) + W_c[v] .
// E_c(y) (fp32 FMA) over the slice, write the corrected logits, add the noise and
// keep a running argmax; the CTA's best goes into its slot as one tagged word,
// the warp reads the slots of all CTAs until they carry the step's tag (as in
// the bf16 loop), and gathers E_c(y_i) for the next step.  No barrier after the
// start, and one hop through L2 instead of atomic key, release add, count and key
// (tiny round: 27 -> 17 us for 8 steps).
constexpr int kPfThreads = 256;

__global__ void __launch_bounds__(kPfThreads, 1)
    sample_persistent_f32_kernel(const SampleParams p, const int ntiles, const int pad) {
  extern __shared__ __align__(16) float pfs[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = kPfThreads / 32;
  const int nblk = gridDim.x;
  const int t_begin = (int)(((long long)blockIdx.x * ntiles) / nblk);
  const int cnt = (int)(((long long)(blockIdx.x + 1) * ntiles) / nblk) - t_begin;
  const int C = p.C, B = p.B, V = p.V, rc = p.rc, wp = rc + pad;
  const int v0 = t_begin * 16, nv = cnt * 16;
  float* Ws = pfs;                                  // [nv][wp]
  float* Es = Ws + (size_t)nv * wp;                 // [C][rc]
  const float* Wc = static_cast<const float*>(p.Wc);
  const float* Ec = static_cast<const float*>(p.Ec);
  const bool sample = p.temperature > 0.f;
  const float inv_temp = sample ? 1.0f / p.temperature : 1.0f;
  const uint2 key = make_uint2((uint32_t)p.seed, (uint32_t)(p.seed >> 32));
  constexpr unsigned long long kTagMask = (1ull << kTagBits) - 1;

  const unsigned epoch = *reinterpret_cast<volatile unsigned*>(p.sync);
  const int r4 = rc / 4;
  for (int i = tid; i < nv * r4; i += kPfThreads)
    *reinterpret_cast<float4*>(Ws + (size_t)(i / r4) * wp + 4 * (i % r4)) = reinterpret_cast<const float4*>(Wc + (size_t)v0 * rc)[i];
  for (int c = warp; c < C; c += nw) {
    int y = p.prev[(size_t)c * p.prev_stride];
    if (y < 0 || y >= V) {
      if (blockIdx.x == 0 && lane == 0) set_err(p.err, LSP_DEV_BAD_TOKEN);
      y = 0;
    }
    for (int i = lane; i < rc; i += 32) Es[c * rc + i] = Ec[(size_t)y * rc + i];
  }
  __syncthreads();                                  // W_c is here, and every warp has read the epoch
  for (int s = 0; s < B; ++s) {
    const unsigned long long tag = (unsigned long long)(epoch + s + 1) & kTagMask;
    unsigned long long* slots = p.slots + (size_t)(s & 1) * C * nblk;   // [request][CTA]
    for (int c = warp; c < C; c += nw) {
      const float* zr = p.src + ((size_t)c * B + s) * V;
      float bv = -INFINITY;
      int bi = 0x7fffffff;
      for (int v = v0 + lane; v < v0 + nv; v += 32) {
        const float z0 = zr[v];
        const float* w = Ws + (size_t)(v - v0) * wp;
        const float* e = Es + (size_t)c * rc;
        float corr = 0.f;
#pragma unroll 4
        for (int r = 0; r < rc; r += 4) {
          const float4 a = *reinterpret_cast<const float4*>(w + r), b = *reinterpret_cast<const float4*>(e + r);
          corr = fmaf(a.x, b.x, corr);
          corr = fmaf(a.y, b.y, corr);
          corr = fmaf(a.z, b.z, corr);
          corr = fmaf(a.w, b.w, corr);
        }
        const float z = z0 + corr;
        if (p.dst) p.dst[((size_t)c * B + s) * V + v] = z;
        float sc = z;
        if (sample) {
          const uint4 x = philox4x32_10(make_uint4((uint32_t)(v >> 2), (uint32_t)s, (uint32_t)(p.b0 + c), p.round), key);
          const uint32_t wd = (v & 3) == 0 ? x.x : (v & 3) == 1 ? x.y : (v & 3) == 2 ? x.z : x.w;
          sc = z * inv_temp + gumbel_of(wd);
        }
        if (better(sc, v, bv, bi)) { bv = sc; bi = v; }
      }
      const unsigned long long k = warp_max_key(bi != 0x7fffffff ? arg_key(bv, bi) : 0ull);
      if (lane == 0)
        st_relaxed_u64(slots + (size_t)c * nblk + blockIdx.x,
                       (k & 0xffffffff00000000ull) | ((k & ((1ull << kIdxBits) - 1)) << kTagBits) | tag);
    }
    const bool last = s + 1 == B;
    if (last && blockIdx.x != 0) return;            // only CTA 0 needs y_B
    for (int c = warp; c < C; c += nw) {
      unsigned long long best = 0ull;
      for (int c0 = 0; c0 < nblk; c0 += 32 * kLeadBatch) {
        unsigned long long k[kLeadBatch];
        const uint64_t t0 = global_ns();
        for (uint32_t it = 1;; ++it) {
          bool all = true;
#pragma unroll
          for (int u = 0; u < kLeadBatch; ++u) {
            const int b = c0 + u * 32 + lane;
            k[u] = tag;
            if (b < nblk) k[u] = ld_relaxed_u64(slots + (size_t)c * nblk + b);
          }
#pragma unroll
          for (int u = 0; u < kLeadBatch; ++u) all = all && (k[u] & kTagMask) == tag;
          if (__all_sync(0xffffffffu, all)) break;
          if ((it & 63u) == 0 && __any_sync(0xffffffffu, global_ns() - t0 > kWaitLimitNs)) {
            if (lane == 0) set_err(p.err, LSP_DEV_TIMEOUT);
            return;                                 // (the other warps wait for no one but the CTAs' slots)
          }
        }
#pragma unroll
        for (int u = 0; u < kLeadBatch; ++u) best = max_u64(best, k[u]);
      }
      best = warp_max_key(best);
      int y = (int)(~(uint32_t)(best >> kTagBits) & ((1u << kIdxBits) - 1));
      if (y >= V) y = 0;                            // (no entry of the row compared)
      if (blockIdx.x == 0 && lane == 0) p.out_tokens[(size_t)c * B + s] = y;
      if (!last)
        for (int i = lane; i < rc; i += 32) Es[c * rc + i] = Ec[(size_t)y * rc + i];
    }
    __syncwarp();
  }
  // CTA 0's first warp has read every CTA's last keys of request 0: all of them have read the epoch
  if (blockIdx.x == 0 && tid == 0) *reinterpret_cast<volatile unsigned*>(p.sync) = epoch + (unsigned)B;
}

__global__ void __launch_bounds__(kSampThreads) sample_final_kernel(const SampleParams p) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  griddep_launch();
  griddep_wait();
  for (int b = warp; b < p.C; b += kSampWarps) {
    const int y = resolve_prev(p, (p.B - 1) & 1, b, lane);
    if (lane == 0) p.out_tokens[(size_t)b * p.B + p.B - 1] = y;
  }
}

__global__ void philox_words_kernel(uint64_t seed, uint32_t round, uint32_t b, uint32_t i,
                                    uint32_t* out, int count) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= count) return;
  const uint4 x = philox4x32_10(make_uint4((uint32_t)(n >> 2), i, b, round),
                                make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
  const int w = n & 3;
  out[n] = w == 0 ? x.x : w == 1 ? x.y : w == 2 ? x.z : x.w;
}

int sample_blocks(int num_sms) { return std::min(2 * num_sms, 32 * kMaxPartialsPerLane); }

static size_t sample_smem(int rc, int es) {
  return kMaxC * sizeof(int) + 2 * kSampWarps * kMaxC * sizeof(float) +
         (size_t)kSampWarps * kMaxC * 17 * sizeof(float) + (size_t)kMaxC * (rc + 8) * es +
         (size_t)kSampWarps * 2 * 16 * (rc + 8) * 2;
}

template <typename T, int KG>
static cudaError_t launch_step(const SampleParams& p, int step, size_t smem, cudaStream_t s) {
  static SmemOptIn once;
  const cudaError_t e = smem_opt_in(once, sample_step_kernel<T, KG>, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(sample_step_kernel<T, KG>, dim3(p.nblk), dim3(kSampThreads), smem, s, p, step);
}

// The bf16 loop's exchange: two sets of answers (copies x requests) and of (request, CTA) key slots.
size_t sample_slot_bytes(int C, int num_sms) {
  static_assert(kPMaxGroups * kPFewCtas <= kAnsCopies * kPMaxC, "without leaders the words take the answers' room");
  return (size_t)2 * (kAnsCopies * kPMaxC * kLineWords + std::min(C, kPMaxC) * num_sms) * sizeof(unsigned long long);
}

// The loops' epoch word.  (Kept at its size: lsp_sample_noalloc's documented need counts it.)
size_t sample_sync_bytes(int B) {
  return ((size_t)B * kPMaxC * 16 * sizeof(unsigned long long) + (size_t)B * sizeof(unsigned) + 255) / 256 * 256;
}

// The bf16 loop's vocabulary tiles, CTAs and shared memory.
struct PersistentPlan {
  int npairs, nblk, tpc, groups;
  size_t smem;
};
static PersistentPlan persistent_plan(const SampleParams& p) {
  PersistentPlan q;
  q.npairs = (p.V + 31) / 32;
  q.groups = p.C > kPGroup ? 2 : 1;
  q.nblk = std::min(std::min(p.num_sms, q.npairs), q.npairs <= few_pairs(q.groups) ? kPFewCtas : q.npairs);
  q.tpc = (q.npairs + q.nblk - 1) / q.nblk;
  const size_t rb = (size_t)p.rc * 2;
  q.smem = (size_t)q.tpc * 32 * rb + (size_t)q.groups * kPGroup * (z_pitch(q.tpc) * sizeof(float) + rb) +
           (size_t)q.groups * (kPWarps * kPGroup + 1) * sizeof(unsigned long long);
  return q;
}

template <int KS, int NG>
static int launch_persistent(const SampleParams& p, cudaStream_t s) {
  const PersistentPlan q = persistent_plan(p);
  const int threads = (kPWarps + 2 * NG) * 32;
  static SmemOptIn once;
  if (smem_opt_in(once, sample_persistent_kernel<KS, NG>, q.smem) != cudaSuccess) return LSP_ERR_CUDA;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sample_persistent_kernel<KS, NG>, threads, q.smem) !=
      cudaSuccess)
    return LSP_ERR_CUDA;
  if (per_sm < 1) return LSP_ERR_SHAPE;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(q.nblk);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = q.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr_c[1];
  attr_c[0].id = cudaLaunchAttributeCooperative;       // every CTA resident: the step waits are safe
  attr_c[0].val.cooperative = 1;
  cfg.attrs = attr_c;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, sample_persistent_kernel<KS, NG>, p, q.npairs) == cudaSuccess ? LSP_OK : LSP_ERR_CUDA;
}

static int launch_persistent_any(const SampleParams& p, cudaStream_t s) {
  if (p.C > kPGroup) return p.rc == 32 ? launch_persistent<2, 2>(p, s) : launch_persistent<4, 2>(p, s);
  return p.rc == 32 ? launch_persistent<2, 1>(p, s) : launch_persistent<4, 1>(p, s);
}

// The persistent kernel's shape limits (anything else takes the per-step kernel).
static size_t persistent_f32_smem(int tpc, int rc, int pad) {
  return ((size_t)tpc * 16 * (rc + pad) + kPMaxC * rc) * sizeof(float);
}
// Floats between two W_c rows: a vector, or none where only that fits (slices that fit
// without padding had become B + 1 launches: V = 240000, rc = 32).
constexpr size_t kPfSmem = 220 * 1024;
static int persistent_f32_pad(int tpc, int rc) { return persistent_f32_smem(tpc, rc, 4) <= kPfSmem ? 4 : 0; }

static bool coop_ok() {
  int dev = 0, coop = 0;
  return cudaGetDevice(&dev) == cudaSuccess &&
         cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop != 0;
}

// fp32 storage: the whole B-step loop in one cooperative launch when the W_c
// slice of a CTA fits shared memory.
static bool persistent_f32_ok(const SampleParams& p, int dtype) {
  if (dtype != LSP_DTYPE_F32 || p.C > kPMaxC || !p.sync || !p.slots || p.num_sms < 1 || p.rc % 4) return false;
  if (p.V > (1 << kIdxBits) || 2 * p.B + 2 > (1 << kTagBits)) return false;
  const int ntiles = p.V / 16;
  const int nblk = std::min(p.num_sms, ntiles);
  const int tpc = (ntiles + nblk - 1) / nblk;
  return persistent_f32_smem(tpc, p.rc, persistent_f32_pad(tpc, p.rc)) <= kPfSmem && coop_ok();
}

static int launch_persistent_f32(const SampleParams& p, cudaStream_t s) {
  const int ntiles = p.V / 16;
  const int nblk = std::min(p.num_sms, ntiles);
  const int tpc = (ntiles + nblk - 1) / nblk;
  const int pad = persistent_f32_pad(tpc, p.rc);
  const size_t smem = persistent_f32_smem(tpc, p.rc, pad);
  static SmemOptIn once;
  if (smem_opt_in(once, sample_persistent_f32_kernel, smem) != cudaSuccess) return LSP_ERR_CUDA;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sample_persistent_f32_kernel, kPfThreads,
                                                    smem) != cudaSuccess)
    return LSP_ERR_CUDA;
  if (per_sm < 1) return LSP_ERR_SHAPE;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nblk);
  cfg.blockDim = dim3(kPfThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr_c[1];
  attr_c[0].id = cudaLaunchAttributeCooperative;       // every CTA resident: the step waits are safe
  attr_c[0].val.cooperative = 1;
  cfg.attrs = attr_c;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, sample_persistent_f32_kernel, p, ntiles, pad) == cudaSuccess ? LSP_OK
                                                                                         : LSP_ERR_CUDA;
}

static bool persistent_ok(const SampleParams& p, int dtype) {
  if (dtype != LSP_DTYPE_BF16 || p.C > kPMaxC || (p.rc != 32 && p.rc != 64) || !p.sync || !p.slots || p.num_sms < 1)
    return false;
  const PersistentPlan q = persistent_plan(p);
  if (q.tpc > kPMaxPairs || q.smem > 227 * 1024 || p.V > (1 << kIdxBits) || 2 * p.B + 2 > (1 << kTagBits)) return false;
  return coop_ok();
}

// More than kPMaxC requests: the requests' proposal chains are independent,
// so the one-launch loop runs once per group of up to kPMaxC requests
// whenever every group fits it (the Philox counter keeps the global request
// index, so the draws are those of one launch over all requests); the
// per-step kernel covers all C otherwise.
static SampleParams request_group(const SampleParams& p, int g0) {
  SampleParams q = p;
  q.C = std::min(kPMaxC, p.C - g0);
  q.src = p.src + (size_t)g0 * p.B * p.V;
  if (p.dst) q.dst = p.dst + (size_t)g0 * p.B * p.V;
  q.prev = p.prev + (size_t)g0 * p.prev_stride;
  q.out_tokens = p.out_tokens + (size_t)g0 * p.B;
  q.b0 = p.b0 + g0;
  return q;
}

static int persistent_groups(const SampleParams& p, int dtype) {
  if (p.C <= kPMaxC) return persistent_ok(p, dtype) || persistent_f32_ok(p, dtype) ? 1 : 0;
  for (int g0 = 0; g0 < p.C; g0 += kPMaxC) {
    const SampleParams q = request_group(p, g0);
    if (!persistent_ok(q, dtype) && !persistent_f32_ok(q, dtype)) return 0;
  }
  return (p.C + kPMaxC - 1) / kPMaxC;
}

int sample_launches(const SampleParams& p, int dtype) {
  const int groups = persistent_groups(p, dtype);
  return groups > 0 ? groups : p.B + 1;
}

int launch_sample(const SampleParams& p, int dtype, cudaStream_t s) {
  if (p.C > kMaxC || p.V % 16 || p.rc % 16 || p.rc > 256) return LSP_ERR_SHAPE;
  // float4 / 16-byte accesses to the logits and the correction tables
  if ((reinterpret_cast<uintptr_t>(p.src) | reinterpret_cast<uintptr_t>(p.dst) |
       reinterpret_cast<uintptr_t>(p.Ec) | reinterpret_cast<uintptr_t>(p.Wc)) & 15)
    return LSP_ERR_ARG;
  if (persistent_groups(p, dtype) > 0) {
    for (int g0 = 0; g0 < p.C; g0 += kPMaxC) {
      const SampleParams q = request_group(p, g0);
      const int rc = persistent_ok(q, dtype) ? launch_persistent_any(q, s) : launch_persistent_f32(q, s);
      if (rc != LSP_OK) return rc;
    }
    return LSP_OK;
  }

  if (p.nblk > 32 * kMaxPartialsPerLane) return LSP_ERR_SHAPE;
  const int es = dtype == LSP_DTYPE_BF16 ? 2 : 4;
  const size_t smem = sample_smem(p.rc, es);
  if (smem > 227 * 1024) return LSP_ERR_SHAPE;

  const int kg = (4 * p.C + 31) / 32;
  for (int step = 0; step < p.B; ++step) {
    cudaError_t e;
    if (dtype == LSP_DTYPE_BF16)
      e = kg <= 1 ? launch_step<bf16, 1>(p, step, smem, s)
        : kg <= 2 ? launch_step<bf16, 2>(p, step, smem, s)
        : kg <= 4 ? launch_step<bf16, 4>(p, step, smem, s)
                  : launch_step<bf16, 8>(p, step, smem, s);
    else
      e = kg <= 1 ? launch_step<float, 1>(p, step, smem, s)
        : kg <= 2 ? launch_step<float, 2>(p, step, smem, s)
        : kg <= 4 ? launch_step<float, 4>(p, step, smem, s)
                  : launch_step<float, 8>(p, step, smem, s);
    if (e != cudaSuccess) return LSP_ERR_CUDA;
  }
  if (launch_pdl(sample_final_kernel, dim3(1), dim3(kSampThreads), 0, s, p) != cudaSuccess)
    return LSP_ERR_CUDA;
  return LSP_OK;
}

int launch_philox_words(uint64_t seed, uint32_t round, uint32_t b, uint32_t i, uint32_t* out,
                        int count, cudaStream_t s) {
  if (count <= 0) return LSP_OK;
  philox_words_kernel<<<(count + 255) / 256, 256, 0, s>>>(seed, round, b, i, out, count);
  return cudaGetLastError() == cudaSuccess ? LSP_OK : LSP_ERR_CUDA;
}

}  // namespace lsp
