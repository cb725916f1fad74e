// Decode attention over a caller-owned cache image, with no allocation anywhere.
//
// Some users of this library are not allowed to allocate device memory: a serving process that
// carved its whole memory budget into a fixed arena at start-up, a plugin running inside someone
// else's allocator policy, or code that is called while a CUDA stream is being captured (where
// cudaMalloc is illegal).  lq_cache_create cannot serve them, because it allocates the stores and the
// split-K workspace.  This entry point takes the two stores as plain device arrays in the canonical
// image format of include/lq.h (wherever the caller keeps them) and keeps its only scratch -- the
// split-K partial results -- in a fixed array that is part of the library image itself.
//
// The arithmetic is plain fp32: x^ = zero + code * scale in one fma, fp32 dot products and sums.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "../../include/lq.h"

namespace {

constexpr int kD = 128;
constexpr int kMaxR = 8;
constexpr int kStaticMaxRecords = 8192;  // (batch row, query head, split) partials that fit the scratch
constexpr int kRecordFloats = kD + 2;    // o[128], m, l
constexpr int kWarps = 4;
constexpr int kStages = 3;
constexpr int kTile = 32;    // quantised tokens a warp takes at a time (a key group of 64 is two such tiles)
constexpr int kFpUnit = 8;   // bf16 rows a warp takes at a time
constexpr int kCtasPerSm = 3;
constexpr int kQuantCost = 4;  // cost of a tile in fp units, by instruction count
constexpr int kMergeThreads = 512;
constexpr uint32_t kFull = 0xFFFFFFFFu;

// Split-K scratch.  Every GPU that loads the library holds these 4.06 MiB until the process exits.
// In host code this name is only a handle for cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) float g_static_partials[kStaticMaxRecords * kRecordFloats];

struct ImageArgs {
  int Hq, Hkv, G, n_fp, S;
  int head_blocks;  // CTAs that share a (b, kv) pair's stores, each with up to R of its query heads
  long long n_quant;
  const uint8_t *fp_k, *fp_v, *k_codes, *v_codes, *k_scale, *k_zero, *v_scale, *v_zero;
  const __nv_bfloat16* q;
  float scale_log2;
  float* partials;
  float* out;
};

// ---- two fp32 lanes per instruction (fma.rn.f32x2: both halves are ordinary IEEE operations) -----------------------
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ uint32_t lds_u16(uint32_t a) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ float lds_bf16(uint32_t a) { return __uint_as_float(lds_u16(a) << 16); }
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint4 lds_u128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
// N consecutive float pairs (16-byte aligned when N is even, 8 otherwise)
template <int N>
__device__ __forceinline__ void lds_pairs(uint32_t a, uint64_t (&v)[N]) {
  if (N == 1) {
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v[0]) : "r"(a));
  } else {
#pragma unroll
    for (int i = 0; i < N; i += 2)
      asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(v[i]), "=l"(v[(i + 1) % N]) : "r"(a + 8 * i));
  }
}
__device__ __forceinline__ void sts_pair(uint32_t a, float lo, float hi) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(lo), "f"(hi) : "memory");
}
__device__ __forceinline__ float bf16lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// Code i of either half of a word, masked in place, is the fp32 subnormal code * 2^(BITS i - 149): no conversion.  One
// exact multiplication by 2^(127 - BITS i) turns it into code * 2^-22, for which x^ * 2^-22 = fma(., scale, zero * 2^-22)
// rounds exactly as fma(code, scale, zero) does, down to |x^| of about 2^-104, where the scaled result becomes subnormal
// (its error is then at most 2^-128 in units of x^).
constexpr float kCodeUnit = 0x1p-22f;
template <int BITS>
__device__ __forceinline__ uint64_t code_pair(uint32_t w, uint32_t whi, int i) {
  const uint32_t mask = ((1u << BITS) - 1u) << (BITS * i);
  const float f = __uint_as_float(static_cast<uint32_t>(254 - BITS * i) << 23);  // 2^(127 - BITS i)
  return mul2(pack2(__uint_as_float(w & mask), __uint_as_float(whi & mask)), pack2(f, f));
}

// n bytes (a multiple of 16) from global to shared memory by one warp
template <bool ALIGNED>
__device__ __forceinline__ void copy_in(uint32_t dst, const uint8_t* src, int n, int lane, int first) {
  if (ALIGNED) {
    for (int i = 16 * ((lane - first) & 31); i < n; i += 512)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i), "l"(src + i) : "memory");
  } else {
    for (int i = lane; i < n; i += 32) {
      const uint32_t x = src[i];
      asm volatile("st.shared.u8 [%0], %1;" ::"r"(dst + i), "r"(x) : "memory");
    }
  }
}

template <int BITS>
struct Geo {
  static constexpr int kTok = kD * BITS / 8;   // code bytes of a token
  static constexpr int kCpw = 32 / BITS;       // codes per word
  static constexpr int kCph = 16 / BITS;       // codes per half word
  static constexpr int kCols = kD / kCpw;      // words per token = lanes that share a token in p.v
  static constexpr int kSub = 32 / kCols;      // tokens a warp works on at a time in p.v
  // stage: K codes, V codes, K scale, K zero, V scale, V zero; or 8 K rows and 8 V rows
  static constexpr int kV = kTile * kTok, kKs = 2 * kV, kKz = kKs + 256, kVs = kKz + 256, kVz = kVs + 256;
  static constexpr int kStage = kVz + 256 > 4096 ? kVz + 256 : 4096;
};

// shared memory: [stages of every warp][q, two arrangements][K parameters of every warp][p of every warp]
template <int BITS, int R>
struct Smem {
  static constexpr int kQ = kWarps * kStages * Geo<BITS>::kStage;
  static constexpr int kQf = kQ + 64 * R * 8;
  static constexpr int kKp = kQf + 64 * R * 8;
  static constexpr int kP = kKp + kWarps * 1024;
  static constexpr int kBytes = kP + kWarps * kTile * R * 8;
};

// What bounds it: fp32 instruction issue (per token and KV head 2 * 128 * R multiply-adds and 2 * 128 dequantisations
// against 96 bytes), so everything is arranged to keep those at one instruction per pair of values.  One warp takes
// kTile quantised tokens (or kFpUnit bf16 rows) at a time through its own ring of kStages cp.async stages and keeps its
// own online-softmax state, so warps never wait for one another before the end.
//   q.k  lane = (token mod 8, quarter of the channels), four tokens per lane: one shared load of the key parameters and
//        of q serves 4 tokens x R heads.  The pairs are the codes i of the two halves of a word (equal position).
//   p.v  lane = (word of a token's codes, one of kSub tokens): 16 R or 8 R accumulators per lane, nothing to exchange
//        until the end.
// The reference maximum moves only when a score exceeds it by more than 8, found by one vote per tile.
// ALIGNED: every array starts on a 16-byte boundary (all rows and groups are multiples of 16 bytes, so only the start
// can spoil it) and is fetched by 16-byte asynchronous copies; otherwise byte by byte, the arrays need no alignment.
// Measured (B = 4, 32/8 heads, 4096 tokens, 17.8 MB): a call 717 -> 23 us; of these the kernel about 18, with the
// schedulers issuing on 45 % of the cycles (three CTAs of 168 registers per SM, two to three tiles per warp).  Distance
// from 64-bit arithmetic 1.3e-6 -> 5e-7 of the result (more and shorter partial sums).
template <int BITS, int R, bool ALIGNED>
__global__ void __launch_bounds__(kWarps * 32, kCtasPerSm) lq_image_split_kernel(ImageArgs a) {
  using Ge = Geo<BITS>;
  using Sm = Smem<BITS, R>;
  constexpr int kCph = Ge::kCph, kSub = Ge::kSub, kPer = kTile / kSub;
  extern __shared__ __align__(128) uint8_t smem[];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = a.Hq / a.Hkv;
  const int s = blockIdx.x % a.S;
  const int hb = (blockIdx.x / a.S) % a.head_blocks;
  const long long pair = blockIdx.x / (static_cast<long long>(a.S) * a.head_blocks);
  const int b = static_cast<int>(pair / a.Hkv), kv = static_cast<int>(pair % a.Hkv);
  const int h0 = hb * r / a.head_blocks, nh = (hb + 1) * r / a.head_blocks - h0;  // this CTA's heads of the pair
  const long long head0 = static_cast<long long>(b) * a.Hq + kv * r + h0;
  const uint32_t sm = smem_u32(smem);

  // q times the score scale, in two arrangements of pairs, [pair][channel quarter][head]: the halves of a code word
  // (channels c, c + kCph), and neighbouring channels for the bf16 rows.  Heads beyond nh are zero.
  for (int i = threadIdx.x; i < 64 * R; i += kWarps * 32) {
    const int h = i % R, cq = (i / R) & 3, pi = i / (4 * R);
    const int c0 = 32 * cq + (pi / kCph) * Ge::kCpw + pi % kCph, f0 = 32 * cq + 2 * pi;
    float x0 = 0.f, x1 = 0.f, y0 = 0.f, y1 = 0.f;
    if (h < nh) {
      const __nv_bfloat16* q = a.q + (head0 + h) * kD;
      x0 = __bfloat162float(q[c0]) * a.scale_log2;
      x1 = __bfloat162float(q[c0 + kCph]) * a.scale_log2;
      y0 = __bfloat162float(q[f0]) * a.scale_log2;
      y1 = __bfloat162float(q[f0 + 1]) * a.scale_log2;
    }
    sts_pair(sm + Sm::kQ + 8 * i, x0, x1);
    sts_pair(sm + Sm::kQf + 8 * i, y0, y1);
  }
  __syncthreads();

  // items of the pair: fp units, then tiles, cut into equal ranges of a cost line over all its warps
  const int n_fpu = (a.n_fp + kFpUnit - 1) / kFpUnit;
  const long long n_tiles = a.n_quant / kTile;
  const long long cost = n_fpu + kQuantCost * n_tiles;
  const auto cut = [&](long long k) -> long long {
    const long long pos = k * cost / (static_cast<long long>(a.S) * kWarps);
    return pos < n_fpu ? pos : n_fpu + (pos - n_fpu + kQuantCost / 2) / kQuantCost;
  };
  const long long first = cut(s * kWarps + warp), last = cut(s * kWarps + warp + 1);

  const uint32_t stage0 = sm + warp * kStages * Ge::kStage;
  const int ng = kD / a.G, vbytes = 2 * ng * kTile;  // value groups of a token; bytes of a tile's value scales
  const auto load = [&](long long it, int st) {
    const uint32_t dst = stage0 + st * Ge::kStage;
    if (it < n_fpu) {
      const int row = lane >> 2, t = static_cast<int>(it) * kFpUnit + row;
      const long long off = (pair * a.n_fp + t) * (2 * kD);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        // 16-byte chunk c of a row is stored where the 8 lanes of a shared-load phase meet 8 different bank groups
        const int c = 4 * j + (lane & 3);
        const uint32_t d = dst + row * 256 + ((c ^ (c >> 3) ^ ((row & 1) << 1)) << 4);
#pragma unroll
        for (int kvh = 0; kvh < 2; ++kvh) {
          const uint8_t* src = (kvh ? a.fp_v : a.fp_k) + off + 16 * c;
          if (ALIGNED) {
            const int n = t < a.n_fp ? 16 : 0;  // rows behind the end are filled with zeros
            if (n == 0) src = kvh ? a.fp_v : a.fp_k;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d + 2048 * kvh), "l"(src), "r"(n) : "memory");
          } else {
            for (int i = 0; i < 16; ++i) {
              const uint32_t x = t < a.n_fp ? src[i] : 0;
              asm volatile("st.shared.u8 [%0], %1;" ::"r"(d + 2048 * kvh + i), "r"(x) : "memory");
            }
          }
        }
      }
    } else {
      const long long tq = (it - n_fpu) * kTile;  // first token of the tile
      const long long row = pair * a.n_quant + tq, grp = pair * (a.n_quant / a.G) + tq / a.G;
      copy_in<ALIGNED>(dst, a.k_codes + row * Ge::kTok, kTile * Ge::kTok, lane, 0);
      copy_in<ALIGNED>(dst + Ge::kV, a.v_codes + row * Ge::kTok, kTile * Ge::kTok, lane, 0);
      copy_in<ALIGNED>(dst + Ge::kKs, a.k_scale + grp * (2 * kD), 256, lane, 0);
      copy_in<ALIGNED>(dst + Ge::kKz, a.k_zero + grp * (2 * kD), 256, lane, 16);
      copy_in<ALIGNED>(dst + Ge::kVs, a.v_scale + row * (2 * ng), vbytes, lane, 0);
      copy_in<ALIGNED>(dst + Ge::kVz, a.v_zero + row * (2 * ng), vbytes, lane, 16);
    }
  };

  const int tk = lane >> 2, cq = lane & 3;               // q.k: token mod 8, channel quarter
  const int sub = lane / Ge::kCols, col = lane % Ge::kCols;  // p.v: token mod kSub, code word
  const int vg = col * Ge::kCpw / a.G;                    // value group of this lane's word
  const uint32_t kp = sm + Sm::kKp + warp * 1024, sp = sm + Sm::kP + warp * (kTile * R * 8);
  uint64_t o[R][kCph];  // (channels i, i + kCph of this lane's word) of sum_t p_t v_t
  float m[R], l[R];     // reference maximum; this lane's share of the denominator
#pragma unroll
  for (int h = 0; h < R; ++h) {
    m[h] = -INFINITY;
    l[h] = 0.f;
#pragma unroll
    for (int i = 0; i < kCph; ++i) o[h][i] = 0ull;
  }

  // softmax of this lane's token (sc[h], valid: the lane holds one); leaves (p, p) * unit per token and head at sp
  const auto softmax = [&](float (&sc)[R], bool valid, int token, float unit) {
    bool up = false;
#pragma unroll
    for (int h = 0; h < R; ++h) {
      if (!valid) sc[h] = -INFINITY;
      up |= sc[h] > m[h] + 8.f;  // m = -inf at first
    }
    if (__any_sync(kFull, up)) {
#pragma unroll
      for (int h = 0; h < R; ++h) {
        float mx = sc[h];
#pragma unroll
        for (int x = 16; x; x >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, x));
        const float mn = fmaxf(m[h], mx);
        const float corr = m[h] == -INFINITY ? 0.f : exp2f(m[h] - mn);
        m[h] = mn;
        l[h] *= corr;
        const uint64_t c2 = pack2(corr, corr);
#pragma unroll
        for (int i = 0; i < kCph; ++i) o[h][i] = mul2(o[h][i], c2);
      }
    }
#pragma unroll
    for (int h = 0; h < R; ++h) {
      const float p = sc[h] == -INFINITY ? 0.f : exp2f(sc[h] - m[h]);  // (m is -inf as long as every score is)
      l[h] += p;
      if (valid) sts_pair(sp + (token * R + h) * 8, p * unit, p * unit);
    }
    __syncwarp();
  };

#pragma unroll
  for (int st = 0; st < kStages - 1; ++st) {
    if (first + st < last) load(first + st, st);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  int st = 0;
#pragma unroll 1
  for (long long it = first; it < last; ++it) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncwarp();  // the other lanes' copies have landed too, and everybody is done with the stage loaded next
    if (it + kStages - 1 < last) load(it + kStages - 1, st == 0 ? kStages - 1 : st - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const uint32_t base = stage0 + st * Ge::kStage;
    st = st == kStages - 1 ? 0 : st + 1;
    if (it < n_fpu) {
      // ---- kFpUnit bf16 rows ----
      uint64_t acc[R];
#pragma unroll
      for (int h = 0; h < R; ++h) acc[h] = 0ull;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = 4 * cq + j;
        const uint4 x = lds_u128(base + tk * 256 + ((c ^ (c >> 3) ^ ((tk & 1) << 1)) << 4));
        const uint32_t xw[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          uint64_t q2[R];
          lds_pairs<R>(sm + Sm::kQf + ((4 * j + k) * 4 + cq) * (8 * R), q2);
          const uint64_t k2 = pack2(bf16lo(xw[k]), bf16hi(xw[k]));
#pragma unroll
          for (int h = 0; h < R; ++h) acc[h] = fma2(k2, q2[h], acc[h]);
        }
      }
      float sc[R];
#pragma unroll
      for (int h = 0; h < R; ++h) {
        float lo, hi;
        unpack2(acc[h], lo, hi);
        sc[h] = lo + hi;
        sc[h] += __shfl_xor_sync(kFull, sc[h], 1);
        sc[h] += __shfl_xor_sync(kFull, sc[h], 2);
      }
      const int nv = min(kFpUnit, a.n_fp - static_cast<int>(it) * kFpUnit);
      if (cq == 0 && tk >= nv) {  // no row here: its p meets rows of zeros
#pragma unroll
        for (int h = 0; h < R; ++h) sts_pair(sp + (tk * R + h) * 8, 0.f, 0.f);
      }
      softmax(sc, cq == 0 && tk < nv, tk, kCodeUnit);
#pragma unroll
      for (int i = 0; i < kFpUnit / kSub; ++i) {
        const int t = kSub * i + sub;
        uint64_t p2[R];
        lds_pairs<R>(sp + t * (8 * R), p2);
        float v[2 * kCph];
#pragma unroll
        for (int j = 0; j < kCph / 4; ++j) {
          const int c = col * (kCph / 4) + j;
          const uint4 x = lds_u128(base + 2048 + t * 256 + ((c ^ (c >> 3) ^ ((t & 1) << 1)) << 4));
          const uint32_t xw[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            v[8 * j + 2 * k] = bf16lo(xw[k]);
            v[8 * j + 2 * k + 1] = bf16hi(xw[k]);
          }
        }
#pragma unroll
        for (int k = 0; k < kCph; ++k) {
          const uint64_t v2 = pack2(v[k], v[k + kCph]);
#pragma unroll
          for (int h = 0; h < R; ++h) o[h][k] = fma2(v2, p2[h], o[h][k]);
        }
      }
    } else {
      // ---- kTile quantised tokens ----
#pragma unroll
      for (int e = lane; e < 64; e += 32) {  // (scale, scale, zero, zero) of the channel pairs, as q is arranged
        const int pi = e >> 2, c0 = 32 * (e & 3) + (pi / kCph) * Ge::kCpw + pi % kCph;
        const float s0 = lds_bf16(base + Ge::kKs + 2 * c0), s1 = lds_bf16(base + Ge::kKs + 2 * (c0 + kCph));
        const float z0 = lds_bf16(base + Ge::kKz + 2 * c0), z1 = lds_bf16(base + Ge::kKz + 2 * (c0 + kCph));
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(kp + 16 * e), "f"(s0), "f"(s1),
                     "f"(z0 * kCodeUnit), "f"(z1 * kCodeUnit)
                     : "memory");
      }
      __syncwarp();
      uint64_t acc[4][R];
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int h = 0; h < R; ++h) acc[t][h] = 0ull;
#pragma unroll
      for (int w = 0; w < 32 / Ge::kCpw; ++w) {
        uint32_t x[4], xh[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          x[t] = lds_u32(base + (8 * t + tk) * Ge::kTok + cq * (Ge::kTok / 4) + 4 * w);
          xh[t] = x[t] >> 16;
        }
#pragma unroll
        for (int i = 0; i < kCph; ++i) {
          const int pi = w * kCph + i;
          uint64_t q2[R], sz[2];
          lds_pairs<2>(kp + 16 * (4 * pi + cq), sz);
          lds_pairs<R>(sm + Sm::kQ + (4 * pi + cq) * (8 * R), q2);
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const uint64_t k2 = fma2(code_pair<BITS>(x[t], xh[t], i), sz[0], sz[1]);
#pragma unroll
            for (int h = 0; h < R; ++h) acc[t][h] = fma2(k2, q2[h], acc[t][h]);
          }
        }
      }
      // sums over the channel quarters: afterwards the lane holds token 8 cq + tk
      float sc[R];
#pragma unroll
      for (int h = 0; h < R; ++h) {
        float f[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          float lo, hi;
          unpack2(acc[t][h], lo, hi);
          f[t] = lo + hi;
        }
        const bool up2 = cq & 2, up1 = cq & 1;
        float k0 = up2 ? f[2] : f[0], k1 = up2 ? f[3] : f[1];
        k0 += __shfl_xor_sync(kFull, up2 ? f[0] : f[2], 2);
        k1 += __shfl_xor_sync(kFull, up2 ? f[1] : f[3], 2);
        sc[h] = (up1 ? k1 : k0) + __shfl_xor_sync(kFull, up1 ? k0 : k1, 1);
        sc[h] *= 1.f / kCodeUnit;
      }
      softmax(sc, true, 8 * cq + tk, 1.f);
#pragma unroll 2
      for (int i = 0; i < kPer; ++i) {
        const int t = kSub * i + sub;
        uint64_t p2[R];
        lds_pairs<R>(sp + t * (8 * R), p2);
        const uint32_t x = lds_u32(base + Ge::kV + t * Ge::kTok + 4 * col), xh = x >> 16;
        const float vs = lds_bf16(base + Ge::kVs + 2 * (t * ng + vg));
        const float vz = lds_bf16(base + Ge::kVz + 2 * (t * ng + vg)) * kCodeUnit;
        const uint64_t vs2 = pack2(vs, vs), vz2 = pack2(vz, vz);
#pragma unroll
        for (int k = 0; k < kCph; ++k) {
          const uint64_t v2 = fma2(code_pair<BITS>(x, xh, k), vs2, vz2);
#pragma unroll
          for (int h = 0; h < R; ++h) o[h][k] = fma2(v2, p2[h], o[h][k]);
        }
      }
    }
    __syncwarp();  // sp and kp are free again
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // ---- sums over the kSub token subsets by a folding exchange: lane (sub, col) ends with its share of word col ----
  constexpr int kVals = 2 * kCph * R;
  float val[kVals];  // [head][i][half]
#pragma unroll
  for (int h = 0; h < R; ++h)
#pragma unroll
    for (int i = 0; i < kCph; ++i) unpack2(o[h][i], val[(h * kCph + i) * 2], val[(h * kCph + i) * 2 + 1]);
  int base = 0;
#pragma unroll
  for (int step = 0, x = 16, n = kVals / 2; (1 << step) < kSub; ++step, x >>= 1, n >>= 1) {
    const bool upper = lane & x;
    base += upper ? n : 0;
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const float send = upper ? val[k] : val[k + n], keep = upper ? val[k + n] : val[k];
      val[k] = keep + __shfl_xor_sync(kFull, send, x);
    }
  }
  __syncthreads();  // every warp is done with its stages
  float* wo = reinterpret_cast<float*>(smem);  // [warp][R][kD], still times kCodeUnit: room for sums near the range's end
  float* wml = wo + kWarps * R * kD;           // [warp][R][2]
#pragma unroll
  for (int k = 0; k < kVals / kSub; ++k) {
    const int f = base + k, half = f & 1, i = (f >> 1) % kCph, h = f / (2 * kCph);
    wo[(warp * R + h) * kD + col * Ge::kCpw + half * kCph + i] = val[k];
  }
#pragma unroll
  for (int h = 0; h < R; ++h) {
#pragma unroll
    for (int x = 16; x; x >>= 1) l[h] += __shfl_xor_sync(kFull, l[h], x);
    if (lane == 0) {
      wml[2 * (warp * R + h)] = m[h];
      wml[2 * (warp * R + h) + 1] = l[h];
    }
  }
  __syncthreads();
  const int d = threadIdx.x;
  for (int h = 0; h < nh; ++h) {
    float M = -INFINITY, L = 0.f, acc = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w)
      if (!(wml[2 * (w * R + h) + 1] == 0.f)) M = fmaxf(M, wml[2 * (w * R + h)]);
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float lw = wml[2 * (w * R + h) + 1];
      if (lw == 0.f) continue;  // a warp without tokens
      const float f = exp2f(wml[2 * (w * R + h)] - M);
      L = fmaf(lw, f, L);
      acc = fmaf(wo[(w * R + h) * kD + d], f, acc);
    }
    if (a.S == 1) {
      a.out[(head0 + h) * kD + d] = acc / L * (1.f / kCodeUnit);
    } else {
      // every record of this call is written here before the merge reads it: nothing in the scratch has to start at
      // zero, and whatever the previous call left behind is simply overwritten
      float* rec = a.partials + ((head0 + h) * a.S + s) * kRecordFloats;
      rec[d] = acc;
      if (d == 0) { rec[kD] = M; rec[kD + 1] = L; }
    }
  }
}

// One CTA per query head; a quarter of the threads per quarter of the records.  Latency is all there is: the first
// kMergeAhead records of every thread are fetched before the weights are known.
__global__ void __launch_bounds__(kMergeThreads) lq_image_merge_kernel(ImageArgs a) {
  extern __shared__ float sw[];  // [S] weights
  __shared__ float red[kMergeThreads / 32], redl[kMergeThreads / 32], part[kMergeThreads];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const long long bh = blockIdx.x;
  const int tid = threadIdx.x, d = tid % kD, quarter = tid / kD;
  const float* rec0 = a.partials + bh * a.S * kRecordFloats;
  constexpr int kQuarters = kMergeThreads / kD, kMergeAhead = 8;
  float v[kMergeAhead];
#pragma unroll
  for (int i = 0; i < kMergeAhead; ++i) {
    const int s = quarter + kQuarters * i;
    v[i] = s < a.S ? __ldcg(rec0 + s * kRecordFloats + d) : 0.f;
  }
  // (m, l) of one record per thread: there are fewer records than threads
  float ms = -INFINITY, ls = 0.f;
  if (tid < a.S) {
    ms = __ldcg(rec0 + tid * kRecordFloats + kD);
    ls = __ldcg(rec0 + tid * kRecordFloats + kD + 1);
  }
  float M = ls == 0.f ? -INFINITY : ms;
#pragma unroll
  for (int x = 16; x; x >>= 1) M = fmaxf(M, __shfl_xor_sync(kFull, M, x));
  if (tid % 32 == 0) red[tid / 32] = M;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kMergeThreads / 32; ++w) M = fmaxf(M, red[w]);
  const float wt = ls == 0.f ? 0.f : exp2f(ms - M);
  if (tid < a.S) sw[tid] = wt;
  float L = ls == 0.f ? 0.f : ls * wt, o = 0.f;
#pragma unroll
  for (int x = 16; x; x >>= 1) L += __shfl_xor_sync(kFull, L, x);
  if (tid % 32 == 0) redl[tid / 32] = L;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kMergeAhead; ++i) {
    const int s = quarter + kQuarters * i;
    const float w = s < a.S ? sw[s] : 0.f;
    if (w != 0.f) o = fmaf(v[i], w, o);  // (without a token its sums may not even be finite)
  }
#pragma unroll 8
  for (int s = quarter + kQuarters * kMergeAhead; s < a.S; s += kQuarters) {
    const float x = __ldcg(rec0 + s * kRecordFloats + d), w = sw[s];
    if (w != 0.f) o = fmaf(x, w, o);
  }
  part[tid] = o;
  __syncthreads();
  if (quarter == 0) {
    L = 0.f;
    o = 0.f;
#pragma unroll
    for (int w = 0; w < kMergeThreads / 32; ++w) L += redl[w];
#pragma unroll
    for (int w = 0; w < kQuarters; ++w) o += part[w * kD + d];
    a.out[bh * kD + d] = o / L * (1.f / kCodeUnit);
  }
}

struct Variant {
  void (*kernel)(ImageArgs);
  int smem;
};
template <int BITS, int R, bool ALIGNED>
constexpr Variant kVariant = {lq_image_split_kernel<BITS, R, ALIGNED>, Smem<BITS, R>::kBytes};
const Variant kVariants[2][2][3] = {  // [4-bit codes][aligned][1, 2, up to 4 heads]
    {{kVariant<2, 1, false>, kVariant<2, 2, false>, kVariant<2, 4, false>},
     {kVariant<2, 1, true>, kVariant<2, 2, true>, kVariant<2, 4, true>}},
    {{kVariant<4, 1, false>, kVariant<4, 2, false>, kVariant<4, 4, false>},
     {kVariant<4, 1, true>, kVariant<4, 2, true>, kVariant<4, 4, true>}}};

// Both kernels take the programmatic launch (their first instruction waits for everything before them): it hides the
// launch of the merge behind the split kernel.
cudaError_t launch(void (*kernel)(ImageArgs), const ImageArgs& a, unsigned grid, unsigned threads, size_t smem, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

// device address of the scratch, looked up once per device (index = CUDA device ordinal)
float* g_partials_ptr[64] = {};
int g_sm_count[64] = {};

}  // namespace

extern "C" lq_status_t lq_decode_attn_image_static(const lq_device_image_t* img, const void* q, float sm_scale,
                                                   float* out, void* stream) {
  if (!img || !q || !out) return LQ_ERR_INVALID_ARG;
  if (img->batch < 1 || img->n_q_heads < 1 || img->n_kv_heads < 1 || img->n_q_heads % img->n_kv_heads ||
      img->n_fp < 0 || img->n_quant < 0 || img->n_fp + img->n_quant < 1)
    return LQ_ERR_INVALID_ARG;
  if (img->bits != 2 && img->bits != 4) return LQ_ERR_INVALID_ARG;
  if (img->head_dim != kD || (img->group != 32 && img->group != 64) || img->n_q_heads / img->n_kv_heads > kMaxR ||
      img->n_quant % img->group)
    return LQ_ERR_UNSUPPORTED;
  if ((img->n_fp > 0 && (!img->fp_k || !img->fp_v)) ||
      (img->n_quant > 0 && (!img->k_codes || !img->v_codes || !img->k_scale || !img->k_zero || !img->v_scale || !img->v_zero)))
    return LQ_ERR_INVALID_ARG;

  const long long heads = static_cast<long long>(img->batch) * img->n_q_heads;
  if (heads > kStaticMaxRecords) return LQ_ERR_CAPACITY;

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LQ_ERR_CUDA;
  if (!g_partials_ptr[dev]) {
    // first call on this device: resolve the device address of the scratch (the host-side name of a
    // __device__ array is not one).  Not legal during stream capture, hence "call once before".
    float* p = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_static_partials) != cudaSuccess || !p) {
      cudaGetLastError();
      return LQ_ERR_CUDA;
    }
    bool ok = cudaDeviceGetAttribute(&g_sm_count[dev], cudaDevAttrMultiProcessorCount, dev) == cudaSuccess;
    // every variant is prepared now, so that a later call may be captured whichever one it takes
    for (const auto& width : kVariants)
      for (const auto& align : width)
        for (const Variant& v : align)
          ok = ok && cudaFuncSetAttribute(v.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, v.smem) == cudaSuccess;
    cudaFuncAttributes attr;
    ok = ok && cudaFuncGetAttributes(&attr, lq_image_merge_kernel) == cudaSuccess;
    if (!ok) {
      cudaGetLastError();
      return LQ_ERR_CUDA;
    }
    g_partials_ptr[dev] = p;
  }

  // At most 4 heads per CTA (64 accumulators a lane): more query heads per KV head share the stores between CTAs, whose
  // second reading comes from L2.  Splits: one resident wave of CTAs, at least two items per warp (a warp with one has
  // nothing to overlap its load with), and never more records than the scratch holds.
  const int r = img->n_q_heads / img->n_kv_heads;
  const int head_blocks = (r + 3) / 4;
  const long long groups = static_cast<long long>(img->batch) * img->n_kv_heads * head_blocks;
  const long long items = (img->n_fp + kFpUnit - 1) / kFpUnit + img->n_quant / kTile;
  long long S = kCtasPerSm * g_sm_count[dev] / groups;
  S = std::min(S, items / (2 * kWarps));
  S = std::min(S, std::min<long long>(kStaticMaxRecords / heads, kMergeThreads));
  S = std::max(S, 1LL);

  ImageArgs a;
  a.Hq = img->n_q_heads; a.Hkv = img->n_kv_heads; a.G = img->group;
  a.n_fp = img->n_fp; a.n_quant = img->n_quant; a.S = static_cast<int>(S); a.head_blocks = head_blocks;
  const auto bytes = [](const uint16_t* p) { return reinterpret_cast<const uint8_t*>(p); };
  a.fp_k = bytes(img->fp_k); a.fp_v = bytes(img->fp_v); a.k_codes = img->k_codes; a.v_codes = img->v_codes;
  a.k_scale = bytes(img->k_scale); a.k_zero = bytes(img->k_zero); a.v_scale = bytes(img->v_scale); a.v_zero = bytes(img->v_zero);
  a.q = static_cast<const __nv_bfloat16*>(q);
  if (!(sm_scale > 0.f)) sm_scale = 0.08838834764831845f;  // 1/sqrt(128)
  a.scale_log2 = sm_scale * 1.4426950408889634f;
  a.partials = g_partials_ptr[dev];
  a.out = out;
  uintptr_t starts = 0;  // (a null array is one that the call does not read)
  for (const uint8_t* p : {a.fp_k, a.fp_v, a.k_codes, a.v_codes, a.k_scale, a.k_zero, a.v_scale, a.v_zero})
    starts |= reinterpret_cast<uintptr_t>(p);
  const bool aligned = (starts & 15) == 0;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const unsigned grid = static_cast<unsigned>(groups * S);
  const int per_block = (r + head_blocks - 1) / head_blocks;
  const Variant& v = kVariants[img->bits == 4][aligned][per_block == 1 ? 0 : per_block == 2 ? 1 : 2];
  cudaError_t e = launch(v.kernel, a, grid, kWarps * 32, v.smem, st);
  if (e == cudaSuccess && S > 1)
    e = launch(lq_image_merge_kernel, a, static_cast<unsigned>(heads), kMergeThreads, static_cast<size_t>(S) * sizeof(float), st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return LQ_ERR_CUDA;
  }
  return LQ_OK;
}
