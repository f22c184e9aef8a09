// Learned hit proposal: an MLP 14 -> 64 -> 64 -> 1 (ReLU) scoring (predicted candidate, hit)
// pairs, trained on the GPU with these kernels (binary cross-entropy with logits, Adam). The
// network is not in the paper; the features and the pruning rule are described in kfgb.h.
//
// Parameter buffer (FP32): W1[64][14], b1[64], W2[64][64], b2[64], W3[64], b3, then the feature
// normaliser mean[14], sd[14] (KF_MLP_PARAMS weights + 28).
#include <algorithm>

#include "mlp.cuh"
#include "pdl.cuh"
#include "tc.cuh"

namespace kfgb {

// Shared shape of the two kernels: a persistent CTA per SM in groups of 256 threads. A group takes
// tiles of 128 samples, two threads per sample: thread t takes sample t % 128 of the tile and half
// h = t / 128 of its columns. Warps w and w + 4 of a group read the same tensor-memory lanes
// (32 (w % 4) ..), each its half of a 64-column accumulator; every branch around a tensor-memory
// load is uniform within a warp. A tile is a chain of MMAs and CUDA-core steps that wait for one
// another, so the groups of a CTA, on their own barriers, work in each other's waits; they
// share the weights in shared memory. Every operand is three bf16 tiles (hi, mid, lo; tc.cuh).
// Inputs: the 14 standardised features, a one (W1's column for it is b1, so the first MMA adds the
// bias), a zero.
constexpr int kTcM = 128;   // samples per tile (the MMA's M)
constexpr int kTcK1 = 16;   // inputs padded to one MMA K step
constexpr int kOne = kMlpIn;  // the input that is one
constexpr int kGroup = 2 * kTcM;

// Hidden activations as the A operand of the next layer: the parts go to tensor memory, 16 columns
// of a thread's 32 at a time. With A in shared memory every MMA of K = 16 read 4 KB for A and 2 KB
// for B there, 48 cycles of its bandwidth for 32 cycles of tensor work. The columns may be those of
// the accumulator that the activations came from: a thread's hi and mid parts lie in the 32 columns
// that it reads itself (half h: 32 h + 0-15 hi, 32 h + 16-31 mid; lo at 64 + 16 h).
struct Parts {
  uint4 h[4], m[4], l[4];  // 8 columns each
};
__device__ __forceinline__ void split16(const float* v, int q, Parts& p) {
  tc::split8(v, p.h[2 * q], p.m[2 * q], p.l[2 * q]);
  tc::split8(v + 8, p.h[2 * q + 1], p.m[2 * q + 1], p.l[2 * q + 1]);
}
template <bool LO>
__device__ __forceinline__ void parts_to_tmem(uint32_t region, int half, int q, const Parts& p) {
  tc::tmem_st8(region + 32 * half + 8 * q, p.h[2 * q], p.h[2 * q + 1]);
  tc::tmem_st8(region + 32 * half + 16 + 8 * q, p.m[2 * q], p.m[2 * q + 1]);
  if (LO) tc::tmem_st8(region + 64 + 16 * half + 8 * q, p.l[2 * q], p.l[2 * q + 1]);
}
// This thread's parts of columns [32 half, 32 half + 32) into a K-major tile of KT columns, the hi,
// mid and lo parts starting at its column blocks H, M and L.
template <int KT, int H, int M, int L>
__device__ __forceinline__ void parts_to_smem(unsigned char* t0, int row, int half, const Parts& p) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    *reinterpret_cast<uint4*>(t0 + tc::kmajor_off(row, H + 4 * half + c, KT)) = p.h[c];
    *reinterpret_cast<uint4*>(t0 + tc::kmajor_off(row, M + 4 * half + c, KT)) = p.m[c];
    *reinterpret_cast<uint4*>(t0 + tc::kmajor_off(row, L + 4 * half + c, KT)) = p.l[c];
  }
}

// Inference: per tile, standardised inputs -> X tile (128 x 16); D1 = X W1^T in tensor memory; h1 =
// relu(D1) -> the next A operand (in D1's columns; its lo part over the X tile, which the finished
// MMA no longer needs); D2 = H W2^T; logit = b3 + sum_j W3[j] relu(D2[j] + b2[j]) on the CUDA cores.
// Four groups per CTA (1024 threads at 64 registers, all 512 tensor-memory columns). 1,000,003 rows take
// 53 us (192 TFLOP/s of the network's flops, six times that on the tensor cores: 61% of the measured
// bf16 rate), where one chain per CTA, two CTAs per SM, took 115 us. On 4 M rows issue is 59% active and
// the tensor pipe 55%: what is left is a group's chain of barriers, MMA waits and operand stores.
namespace fwd {
constexpr int kGroups = 4;
constexpr uint32_t W1_T = 2048, W2_T = 8192, H_T = 16384, X_T = 4096;  // bytes of one tile
constexpr uint32_t W1 = 0, W2 = W1 + 3 * W1_T, H = W2 + 3 * W2_T, B2 = H + kGroups * H_T, W3 = B2 + 256,
                   MEAN = W3 + 256, SD = MEAN + 64, RS = SD + 64, PART = RS + 64, BAR = PART + kGroups * 512, TMEM = BAR + 8 * kGroups,
                   BYTES = TMEM + 8;
constexpr uint32_t kCols = 128 * kGroups;
static_assert(BYTES + 1024 <= 227 * 1024 && 3 * X_T <= H_T, "shared-memory layout");
}  // namespace fwd

// Loads W1 (64 x 16: 14 inputs, b1, zero) and W2 (64 x 64) as the MMAs' B operands in the K-major
// core-matrix layout, by all threads of the block.
__device__ __forceinline__ void stage_weights_b(const float* __restrict__ params, unsigned char* w1, uint32_t w1_t,
                                                unsigned char* w2, uint32_t w2_t) {
  for (int item = threadIdx.x; item < kMlpHid * 2; item += blockDim.x) {
    const int j = item >> 1, c = item & 1;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int i = 8 * c + e;
      v[e] = i < kMlpIn ? params[kMlpW1 + j * kMlpIn + i] : i == kOne ? params[kMlpB1 + j] : 0.f;
    }
    tc::store8_split(w1, w1_t, tc::kmajor_off(j, c, kTcK1), v);
  }
  for (int item = threadIdx.x; item < kMlpHid * 8; item += blockDim.x) {
    const int o = item >> 3, c = item & 7;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = params[kMlpW2 + o * kMlpHid + 8 * c + e];
    tc::store8_split(w2, w2_t, tc::kmajor_off(o, c, kMlpHid), v);
  }
}

// Raw features [8 h, 8 h + 8) of sample r (zeros past n and past the 14 inputs), loaded ahead of
// their tile.
__device__ __forceinline__ void fetch_half(const float* __restrict__ feats, int r, int n, int half, float2* f) {
  const float2* f2 = reinterpret_cast<const float2*>(feats + static_cast<size_t>(r) * kMlpIn);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = 4 * half + i;
    f[i] = (r < n && k < kMlpIn / 2) ? __ldg(f2 + k) : make_float2(0.f, 0.f);
  }
}

// Normaliser in shared memory, 16 entries each: mean, sd and 1 / sd; the inputs past the 14, fetched as
// zeros, become the one and the zero. Tells whether each sd is within [2^-100, 2^100], where the
// reciprocal form below gives the quotient.
__device__ __forceinline__ bool stage_normaliser(const float* __restrict__ params, float* mean, float* sd, float* rs) {
  const int t = threadIdx.x;
  bool in_range = true;
  if (t < kTcK1) {
    const float s = t < kMlpIn ? params[kMlpSd + t] : 1.f;
    mean[t] = t < kMlpIn ? params[kMlpMean + t] : t == kOne ? -1.f : 0.f;
    sd[t] = s;
    rs[t] = 1.f / s;
    in_range = fabsf(s) >= 7.8886091e-31f && fabsf(s) <= 1.2676506e30f;
  }
  return in_range;
}

// Standardised inputs [8 h, 8 h + 8), split for their tile. The quotient is a / sd from the correctly
// rounded reciprocal r: q = a r, then q + (a - q sd) r with the remainder exact in a fused operation
// (P. W. Markstein, Computation of elementary functions on the IBM RISC System/6000 processor, IBM J.
// Res. Dev. 34, 1990), the bits of the division (a test compares them); divisions were a seventh of the
// forward pass's instructions. A row past n, fetched as zeros, is (0 - mean) / sd in the forward pass, where it meets
// nothing else; in the loss gradient, whose MMAs multiply it by an error of zero, it has to be finite
// whatever the normaliser is, and a mean of zeros is passed for it.
__device__ __forceinline__ void standardise_half(const float2* f, int half, const float* mean, const float* sd,
                                                 const float* rs, bool by_reciprocal, uint4 (&x)[3]) {
  float v[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = 8 * half + 2 * i;
    const float2 m = *reinterpret_cast<const float2*>(mean + k), s = *reinterpret_cast<const float2*>(sd + k);
    const float2 r = *reinterpret_cast<const float2*>(rs + k);
    const uint64_t a = tc::sub2(tc::pack2(f[i].x, f[i].y), tc::pack2(m.x, m.y)), rr = tc::pack2(r.x, r.y);
    if (by_reciprocal) {
      const uint64_t q = tc::mul2(a, rr);
      tc::unpack2(tc::fma2(tc::fma2(q, tc::pack2(-s.x, -s.y), a), rr, q), v[2 * i], v[2 * i + 1]);
    } else {
      float a0, a1;
      tc::unpack2(a, a0, a1);
      v[2 * i] = a0 / s.x;
      v[2 * i + 1] = a1 / s.y;
    }
  }
  tc::split8(v, x[0], x[1], x[2]);
}

// relu(v + b2) of this thread's 16 columns [c, c + 16) (16-byte aligned in shared memory), in place.
__device__ __forceinline__ void relu16(float* v, const float* b2) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 b = reinterpret_cast<const float4*>(b2)[i];
    tc::unpack2(tc::add2(tc::pack2(v[4 * i], v[4 * i + 1]), tc::pack2(b.x, b.y)), v[4 * i], v[4 * i + 1]);
    tc::unpack2(tc::add2(tc::pack2(v[4 * i + 2], v[4 * i + 3]), tc::pack2(b.z, b.w)), v[4 * i + 2], v[4 * i + 3]);
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = fmaxf(v[i], 0.f);
}

// acc += the even and odd terms of sum_j w3[j] v[j] over 16 columns.
__device__ __forceinline__ uint64_t dot16(const float* v, const float* w3, uint64_t acc) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 w = reinterpret_cast<const float4*>(w3)[i];
    acc = tc::fma2(tc::pack2(w.x, w.y), tc::pack2(v[4 * i], v[4 * i + 1]), acc);
    acc = tc::fma2(tc::pack2(w.z, w.w), tc::pack2(v[4 * i + 2], v[4 * i + 3]), acc);
  }
  return acc;
}

// One MMA operand in shared memory: the descriptor of the first of its three tiles, whose size, layout
// and advance per K = 16 step are compile-time constants, so that the thread that issues the MMAs
// adds one constant to the descriptor's low word for each (with descriptors assembled per MMA by a
// thread picked by its index, the loss gradient of 2,000,003 rows took 604 us against 456).
template <uint32_t LBO, uint32_t SBO, uint32_t STEP>
struct Operand {
  uint32_t lo;
  __device__ __forceinline__ explicit Operand(uint32_t base) : lo(static_cast<uint32_t>(tc::smem_desc(base, LBO, SBO))) {}
  // The operand `off` bytes on, at K step k.
  __device__ __forceinline__ uint64_t at(uint32_t off, int k) const {
    constexpr uint64_t hi = (static_cast<uint64_t>(SBO >> 4) << 32) | (1ull << 46);
    return hi | (lo + ((off + STEP * k) >> 4));
  }
};

// K-major operand (tc.cuh layout) of a tile with KT columns.
template <int KT>
__device__ __forceinline__ auto kmajor(uint32_t base) {
  return Operand<128u, KT / 8 * 128u, 256u>(base);
}

// The same tile read MN-major (its rows become K, its columns M or N): 8-column blocks are 128 B
// apart (stride byte offset), 8-row groups KT / 8 * 128 B apart (leading byte offset).
template <int KT>
__device__ __forceinline__ auto mnmajor(uint32_t base) {
  return Operand<KT / 8 * 128u, 128u, 2u * (KT / 8 * 128u)>(base);
}

// D = A B^T over one K = 16 step as the six products of the three-part split, the smallest first
// (lo*hi, hi*lo, mid*mid, mid*hi, hi*mid, hi*hi); the parts of A and B lie AT and BT bytes apart. One
// thread issues, the mbarrier receives the completion. The order costs nothing (the same MMAs) and the
// tensor pipe's rounding of the FP32 accumulator then falls on small sums: with hi*hi first the logits'
// error against FP64 was 7.4e-7 of the largest, with it last, here and over K = 64, it is 1.7e-7.
template <uint32_t AT, uint32_t BT, class OA, class OB>
__device__ __forceinline__ void mma_split16(uint32_t d, const OA& A, const OB& B, uint32_t idesc, uint64_t* bar) {
  constexpr int kPa[6] = {2, 0, 1, 1, 0, 0}, kPb[6] = {0, 2, 1, 0, 1, 0};
  tc::fence_after_sync();
#pragma unroll
  for (int p = 0; p < 6; ++p) tc::mma_bf16(d, A.at(AT * kPa[p], 0), B.at(BT * kPb[p], 0), idesc, p > 0 ? 1u : 0u);
  tc::mma_commit(bar);
}

// D = A B^T over K = 64 with A's parts in tensor memory (columns from region as parts_to_tmem lays
// them), or (LO = false) its lo part, which one of the six products reads, in shared memory. The hi*hi
// products of all four K steps come last.
template <bool LO, uint32_t BT, class OL, class OB>
__device__ __forceinline__ void mma_split_ta(uint32_t d, uint32_t region, const OL& lo, const OB& B, uint32_t idesc,
                                             uint64_t* bar) {
  tc::fence_after_sync();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t ah = region + 32 * (k >> 1) + 8 * (k & 1), am = ah + 16;
    if constexpr (LO) tc::mma_bf16_ta(d, region + 64 + 8 * k, B.at(0, k), idesc, k > 0 ? 1u : 0u);
    else tc::mma_bf16(d, lo.at(0, k), B.at(0, k), idesc, k > 0 ? 1u : 0u);
    tc::mma_bf16_ta(d, ah, B.at(2 * BT, k), idesc, 1u);
    tc::mma_bf16_ta(d, am, B.at(BT, k), idesc, 1u);
    tc::mma_bf16_ta(d, am, B.at(0, k), idesc, 1u);
    tc::mma_bf16_ta(d, ah, B.at(BT, k), idesc, 1u);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) tc::mma_bf16_ta(d, region + 32 * (k >> 1) + 8 * (k & 1), B.at(0, k), idesc, 1u);
  tc::mma_commit(bar);
}

__global__ void __launch_bounds__(fwd::kGroups* kGroup, 1) k_mlp_forward(const float* __restrict__ params,
                                                                         const float* __restrict__ feats, int n,
                                                                         float* __restrict__ logits) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* S = smem_raw + ((1024 - (tc::smem_u32(smem_raw) & 1023)) & 1023);
  const uint32_t sb = tc::smem_u32(S);
  float* b2 = reinterpret_cast<float*>(S + fwd::B2);
  float* w3 = reinterpret_cast<float*>(S + fwd::W3);
  float* mean = reinterpret_cast<float*>(S + fwd::MEAN);
  float* sd = reinterpret_cast<float*>(S + fwd::SD);
  float* rs = reinterpret_cast<float*>(S + fwd::RS);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(S + fwd::TMEM);
  const int gi = threadIdx.x / kGroup, t = threadIdx.x % kGroup;
  const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);  // (uniform, so that the MMAs' operands are too)
  const int row = t & (kTcM - 1), half = t / kTcM;
  float* part = reinterpret_cast<float*>(S + fwd::PART) + gi * kTcM;  // second half's output-layer sums
  uint64_t* bar = reinterpret_cast<uint64_t*>(S + fwd::BAR) + gi;
  const uint32_t h_off = fwd::H + gi * fwd::H_T;  // this group's X tile, then h1's lo part
  const int bid = gi + 1;

  pdl_begin();
  stage_weights_b(params, S + fwd::W1, fwd::W1_T, S + fwd::W2, fwd::W2_T);
  if (threadIdx.x < kMlpHid) {
    b2[threadIdx.x] = params[kMlpB2 + threadIdx.x];
    w3[threadIdx.x] = params[kMlpW3 + threadIdx.x];
  }
  const bool odd_sd = !stage_normaliser(params, mean, sd, rs);
  const float b3 = params[kMlpB3];
  if (threadIdx.x < 32) tc::tmem_alloc(tmem_slot, fwd::kCols);
  if (t == 0) tc::mbar_init(bar, 1);
  tc::fence_proxy_async();
  tc::fence_before_sync();
  const bool by_rs = !__syncthreads_or(odd_sd);
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot, d = tmem + 128u * gi;
  const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16, lane_base = d + lane_off + 32u * half;
  constexpr uint32_t idesc = tc::idesc_bf16_f32(kTcM, kMlpHid);
  uint32_t phase = 0;
  bool ok = true;  // a wait that gives up ends the group's tiles; until then its threads keep in step

  const int n_tiles = (n + kTcM - 1) / kTcM;
  const int tile0 = blockIdx.x + gridDim.x * gi, stride = gridDim.x * fwd::kGroups;
  int tile = tile0;
  // This thread's half of its sample's inputs in the next tile: loaded during the first layer, split
  // during the second.
  float2 fin[4];
  uint4 x[3];
  fetch_half(feats, tile * kTcM + row, n, half, fin);
  standardise_half(fin, half, mean, sd, rs, by_rs, x);
  for (; tile < n_tiles; tile += stride) {
    const int r = tile * kTcM + row;
    tc::store8(S + h_off, fwd::X_T, tc::kmajor_off(row, half, kTcK1), x[0], x[1], x[2]);
    tc::fence_proxy_async();
    tc::bar_sync(bid, kGroup);
    if (warp == 0 && tc::elect_one())
      mma_split16<fwd::X_T, fwd::W1_T>(d, kmajor<kTcK1>(sb + h_off), kmajor<kTcK1>(sb + fwd::W1), idesc, bar);
    if (tile + stride < n_tiles) fetch_half(feats, (tile + stride) * kTcM + row, n, half, fin);
    ok = ok && tc::mbar_wait(bar, phase);
    phase ^= 1u;
    tc::fence_after_sync();
    {  // h1 columns [32 h, 32 h + 32), all read before their accumulator columns are written
      Parts p;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float v[16];
        tc::tmem_ld16(lane_base + 16 * q, v);
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = fmaxf(v[i], 0.f);
        split16(v, q, p);
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) parts_to_tmem<false>(d + lane_off, half, q, p);
#pragma unroll
      for (int c = 0; c < 4; ++c)
        *reinterpret_cast<uint4*>(S + h_off + tc::kmajor_off(row, 4 * half + c, kMlpHid)) = p.l[c];
    }
    tc::tmem_st_wait();
    tc::fence_proxy_async();
    tc::fence_before_sync();
    tc::bar_sync(bid, kGroup);
    if (warp == 0 && tc::elect_one())
      mma_split_ta<false, fwd::W2_T>(d + 64, d, kmajor<kMlpHid>(sb + h_off), kmajor<kMlpHid>(sb + fwd::W2), idesc, bar);
    standardise_half(fin, half, mean, sd, rs, by_rs, x);
    ok = ok && tc::mbar_wait(bar, phase);
    phase ^= 1u;
    tc::fence_after_sync();
    uint64_t acc2 = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float v[16];
      tc::tmem_ld16(lane_base + 64 + 16 * q, v);
      relu16(v, b2 + 32 * half + 16 * q);
      acc2 = dot16(v, w3 + 32 * half + 16 * q, acc2);
    }
    float acc, odd;
    tc::unpack2(acc2, acc, odd);
    acc += odd;
    if (half == 1) part[row] = acc;
    tc::fence_before_sync();
    if (tc::bar_or(bid, kGroup, !ok)) break;
    if (half == 0 && r < n) logits[r] = b3 + acc + part[row];
  }
  if (tile < n_tiles) {
    // A tensor-core wait gave up: this group's remaining samples get NaN logits; the MMA in flight
    // gets one more bounded wait before the tensor memory is released.
    for (; tile < n_tiles; tile += stride) {
      const int r = tile * kTcM + row;
      if (half == 0 && r < n) logits[r] = __int_as_float(0x7fc00000);
    }
    tc::mbar_wait(bar, phase ^ 1u);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (threadIdx.x < 32) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, fwd::kCols);
  }
}

// The finder's A fragments of both hidden layers (layout in mlp.cuh): entry i holds, for row tile
// m and K step s, lane l's four f16x2 words (rows 16 m + l / 4 and + 8, columns 16 s + 2 (l % 4)
// and + 8; zero beyond the 14 inputs of the first layer), hi or scaled lo part.
__global__ void k_mlp_fragments(const float* __restrict__ w, uint4* __restrict__ frag) {
  pdl_begin();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kFragWords; i += gridDim.x * blockDim.x) {
    const int part = i & 1, lane = (i >> 1) % 32;
    int m, s, ld;
    const float* W;
    if (i < kFragL2) {
      m = (i >> 1) / 32;
      s = 0;
      W = w + kMlpW1;
      ld = kMlpIn;
    } else {
      const int j = ((i - kFragL2) >> 1) / 32;
      m = j / 4;
      s = j % 4;
      W = w + kMlpW2;
      ld = kMlpHid;
    }
    const int r = 16 * m + lane / 4, c = 16 * s + 2 * (lane % 4);
    const int rr[4] = {r, r + 8, r, r + 8}, cc[4] = {c, c, c + 8, c + 8};
    unsigned word[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float v0 = cc[q] < ld ? W[rr[q] * ld + cc[q]] : 0.f;
      const float v1 = cc[q] + 1 < ld ? W[rr[q] * ld + cc[q] + 1] : 0.f;
      unsigned h, l;
      split_f16x2(v0, v1, h, l);
      word[q] = part ? l : h;
    }
    frag[i] = make_uint4(word[0], word[1], word[2], word[3]);
  }
}

int launch_mlp_fragments(const float* params, uint4* frag, cudaStream_t st) {
  launch_pdl(k_mlp_fragments, (kFragWords + 255) / 256, 256, 0, st, params, frag);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// The finder's scoring outside the finder: warp w of the grid takes rows 8w .. 8w + 7, lane l the
// features of row 8w + l / 4 in its operand columns, standardised as the finder standardises its
// candidate features and pulls; lanes 0-3 write the logits of rows 8w + 2l, 8w + 2l + 1.
__global__ void k_mlp_finder_scores(const uint4* __restrict__ frag, const float* __restrict__ prm,
                                    const float* __restrict__ feats, int n, float* __restrict__ logits) {
  pdl_begin();
  const int lane = threadIdx.x & 31;
  const long long r0 = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) / 32 * 8;
  if (r0 >= n) return;  // whole warps leave together (r0 is the same for the warp's lanes)
  const long long row = r0 + (lane >> 2);
  const int t = lane & 3;
  const int cols[4] = {2 * t, 2 * t + 1, 2 * t + 8, 2 * t + 9};
  float x[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = cols[q];
    x[q] = (row < n && c < kMlpIn) ? (feats[row * kMlpIn + c] - prm[kMlpMean + c]) / prm[kMlpSd + c] : 0.f;
  }
  const float2 l2 = mlp_logit8(frag, prm, x, lane);
  if (lane < 4) {
    if (r0 + 2 * lane < n) logits[r0 + 2 * lane] = l2.x;
    if (r0 + 2 * lane + 1 < n) logits[r0 + 2 * lane + 1] = l2.y;
  }
}

int launch_mlp_finder_scores(const float* params, const float* feats, int n, float* logits, uint4* frag,
                             cudaStream_t st) {
  if (launch_mlp_fragments(params, frag, st) != 0) return -3;
  if (n == 0) return 0;
  const long long warps = (static_cast<long long>(n) + 7) / 8;
  launch_pdl(k_mlp_finder_scores, static_cast<int>((warps + 7) / 8), 256, 0, st, frag, params, feats, n, logits);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// Loss and gradient on the tensor cores. Per tile of a group:
//   D1 = X W1^T -> h1 = relu(D1);  D2 = H1 W2^T -> z3 = b3 + W3 . relu(D2 + b2),
//   g = (sigmoid(z3) - y), e2 = g W3 [z2 > 0];  D3 = E2 W2 -> e1 = D3 [h1 > 0];
//   Dg2 += E2^T [H1 | X],  Dg1 += E1^T X   (accumulated in tensor memory over all the CTA's tiles),
// Dg2 giving dW2 and (in the column of X's ones) db2, Dg1 dW1 and db1. dW3, db3 and the loss are
// summed in registers.
//
// Two groups per CTA. Shared memory: per group one sample x [h1 mid | h1 hi | x hi | x mid | x lo | h1
// lo] tile (128 x 240; x K-major the A operand of the first MMA, all of it MN-major the B operand of
// the gradient MMAs), one sample x [e hi | e mid | e lo | 0] tile (128 x 256: e2, then e1; MN-major
// the A operand of the gradient MMAs), W1 and W2 in three tiles each (W2 read MN-major is W2^T for
// the third MMA). With the parts side by side one gradient MMA does several of the six products:
// per K = 16 step of dW2, [hi | mid] by [mid, hi, x hi] (M 128, N 144), [lo | 0] by [hi, x hi] (N 80)
// and [hi | mid] by lo (N 64), into accumulators whose rows u and 64 + u, and columns c and 64 + c,
// are added at the end; of dW1, [hi | mid] by [x hi, x mid], [lo | 0] by x hi, [hi | mid] by x lo: half
// the 48 MMAs per layer of six products of M = 64 each (2,000,003 rows 456 -> 415 us). The e tile (two do not fit) is one group's at a time, during its
// gradient MMAs; the other group then runs its layers.
// Tensor memory: per group D1, then h1, then e2 (parts_to_tmem) at 0, D2 then D3 at 96; Dg2 at 320,
// Dg1 at 464.
// 2,000,003 rows take 407 us (140 TFLOP/s of the network's flops), where one group per CTA took 895 us.
// On 4 M rows the tensor pipe is 42% active and issue 38%: the two groups' chains of six MMA round trips
// a tile, one of them holding the e tile. A step's 4,096 rows: the whole step 18 us against 98 us; their tile, prologue and epilogue
// are one chain (the old epilogue added 32 lanes to one shared-memory float, a CAS loop each).
namespace grd {
constexpr int kGroups = 2;
constexpr int kXhK = 240, kEK = 256;                            // columns of the two tiles
constexpr int kHm = 0, kHh = 8, kXh = 16, kXm = 18, kXl = 20, kHl = 22;  // 8-column blocks of the parts
constexpr uint32_t E_T = kTcM * kEK * 2, XH_T = kTcM * kXhK * 2, W1_T = 2048, W2_T = 8192;  // bytes of one tile
constexpr uint32_t E = 0, XH = E + E_T, W2 = XH + kGroups * XH_T, W1 = W2 + 3 * W2_T, B2 = W1 + 3 * W1_T,
                   W3 = B2 + 256, MEAN = W3 + 256, SD = MEAN + 64, RS = SD + 64, NIL = RS + 64, PART = NIL + 64, RED = PART + kGroups * 1024,
                   BAR = RED + 16 * 34 * 4, TMEM = BAR + 16 * kGroups, LOCK = TMEM + 4, USED = LOCK + 4, BYTES = USED + 8;
static_assert(BYTES + 1024 <= 227 * 1024, "shared-memory layout");
constexpr uint32_t kCols = 512, kColD2 = 96, kColG2 = 320, kColG1 = 464;
}  // namespace grd

// Instruction descriptor bits 15 and 16: A, B MN-major.
constexpr uint32_t kAmn = 1u << 15, kBmn = 1u << 16;

// D (+)= E^T B over K = the tile's 128 samples, both MN-major: per K = 16 step [hi | mid] of e by the N1
// columns of B from block B1 on, [lo | 0] by N2 from B2 on (D's columns from C2 on), [hi | mid] by N3
// from B3 on.
template <int C2, int B1, int N1, int B2, int N2, int B3, int N3, class OE, class OB>
__device__ __forceinline__ void mma_grad(uint32_t d, const OE& E, const OB& B, uint64_t* bar, bool accumulate) {
  tc::fence_after_sync();
#pragma unroll
  for (int k = 0; k < kTcM / 16; ++k) {
    tc::mma_bf16(d, E.at(0, k), B.at(128 * B1, k), tc::idesc_bf16_f32(kTcM, N1) | kAmn | kBmn, k > 0 || accumulate);
    tc::mma_bf16(d + C2, E.at(128 * 16, k), B.at(128 * B2, k), tc::idesc_bf16_f32(kTcM, N2) | kAmn | kBmn, 1u);
    tc::mma_bf16(d, E.at(0, k), B.at(128 * B3, k), tc::idesc_bf16_f32(kTcM, N3) | kAmn | kBmn, 1u);
  }
  tc::mma_commit(bar);
}

// Sums of v[i] over the warp's lanes, element i in lane i: five halving exchanges.
__device__ __forceinline__ float warp_sum32(float* v, int lane) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float other = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + o], o);
      v[i] = (up ? v[i + o] : v[i]) + other;
    }
  }
  return v[0];
}

// grad[0 .. 3] += v[0 .. 3], as one 16-byte reduction where the address allows.
__device__ __forceinline__ void add4(float* grad, const float* v) {
  if ((reinterpret_cast<size_t>(grad) & 15) == 0) {
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(grad), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3])
                 : "memory");
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) atomicAdd(grad + i, v[i]);
  }
}

// PROBE: the group that takes tile `fail` treats its second layer's wait there as given up, after it has
// completed (kf_mlp_wait_probe: what a wait that gives up leaves in the outputs).
template <bool PROBE>
__global__ void __launch_bounds__(grd::kGroups* kGroup, 1)
    k_mlp_loss_grad(const float* __restrict__ params, const float* __restrict__ feats, const float* __restrict__ labels,
                    int n, float inv_n, float* __restrict__ grad, float* __restrict__ loss, int fail) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* S = smem_raw + ((1024 - (tc::smem_u32(smem_raw) & 1023)) & 1023);
  const uint32_t sb = tc::smem_u32(S);
  float* b2 = reinterpret_cast<float*>(S + grd::B2);
  float* w3 = reinterpret_cast<float*>(S + grd::W3);
  float* mean = reinterpret_cast<float*>(S + grd::MEAN);
  float* sd = reinterpret_cast<float*>(S + grd::SD);
  float* rs = reinterpret_cast<float*>(S + grd::RS);
  float* nil = reinterpret_cast<float*>(S + grd::NIL);  // [16] zeros
  float* red = reinterpret_cast<float*>(S + grd::RED);  // [16 warps][34]: dW3 of the warp's 32 units, db3, loss
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(S + grd::TMEM);
  int* lock = reinterpret_cast<int*>(S + grd::LOCK);  // 1: the e tile is taken
  int* used = reinterpret_cast<int*>(S + grd::USED);  // 1: the gradient accumulators hold a tile
  const int gi = threadIdx.x / kGroup, t = threadIdx.x % kGroup;
  const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);  // (uniform, so that the MMAs' operands are too)
  const int row = t & (kTcM - 1), half = t / kTcM;
  const int hc = 32 * half;  // this thread's first column of a 64-column accumulator
  float* part = reinterpret_cast<float*>(S + grd::PART) + gi * 2 * kTcM;  // [2][128] output-layer partial sums
  // bar[0]: the layers' MMAs, bar[1]: the gradient MMAs (the first of them is in flight with the third layer's)
  uint64_t* bar = reinterpret_cast<uint64_t*>(S + grd::BAR) + 2 * gi;
  const uint32_t xh = grd::XH + gi * grd::XH_T;
  const int bid = gi + 1;

  pdl_begin();
  stage_weights_b(params, S + grd::W1, grd::W1_T, S + grd::W2, grd::W2_T);
  if (threadIdx.x < kMlpHid) {
    b2[threadIdx.x] = params[kMlpB2 + threadIdx.x];
    w3[threadIdx.x] = params[kMlpW3 + threadIdx.x];
  }
  const bool odd_sd = !stage_normaliser(params, mean, sd, rs);
  if (threadIdx.x < kTcK1) nil[threadIdx.x] = 0.f;
  for (int i = threadIdx.x; i < kTcM * 8; i += blockDim.x)  // the e tile's zero columns
    *reinterpret_cast<uint4*>(S + grd::E + tc::kmajor_off(i >> 3, 24 + (i & 7), grd::kEK)) = make_uint4(0u, 0u, 0u, 0u);
  const float b3 = params[kMlpB3];
  if (threadIdx.x < 32) tc::tmem_alloc(tmem_slot, grd::kCols);
  if (threadIdx.x == 0) *lock = *used = 0;
  if (t == 0) {
    tc::mbar_init(bar, 1);
    tc::mbar_init(bar + 1, 1);
  }
  tc::fence_proxy_async();
  tc::fence_before_sync();
  const bool by_rs = !__syncthreads_or(odd_sd);
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot, d = tmem + 160u * gi;
  const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
  const uint32_t lane_base = d + lane_off + hc;
  constexpr uint32_t id_kk = tc::idesc_bf16_f32(kTcM, kMlpHid);
  const auto e_mn = mnmajor<grd::kEK>(sb + grd::E);
  const auto xh_mn = mnmajor<grd::kXhK>(sb + xh);
  uint32_t phase = 0, gphase = 0;
  bool ok = true, locked = false;
  uint64_t acc3[16];  // dW3 partial sums of this thread's 32 hidden units, in pairs
#pragma unroll
  for (int j = 0; j < 16; ++j) acc3[j] = 0;
  float gsum = 0.f, lsum = 0.f;

  const int n_tiles = (n + kTcM - 1) / kTcM;
  const int stride = gridDim.x * grd::kGroups;
  int tile = blockIdx.x + gridDim.x * gi;
  // This thread's half of its sample's inputs, and the label, in the next tile: loaded and
  // split during the gradient MMAs.
  float2 fin[4];
  uint4 x[3];
  fetch_half(feats, tile * kTcM + row, n, half, fin);
  standardise_half(fin, half, tile * kTcM + row < n ? mean : nil, sd, rs, by_rs, x);
  float yin = tile * kTcM + row < n ? labels[tile * kTcM + row] : 0.f;
  for (; tile < n_tiles; tile += stride) {
    const bool valid = tile * kTcM + row < n;
    tc::store8(S + xh, 128 * (grd::kXm - grd::kXh), tc::kmajor_off(row, grd::kXh + half, grd::kXhK), x[0], x[1], x[2]);
    const float y = yin;
    tc::fence_proxy_async();
    tc::bar_sync(bid, kGroup);
    if (warp == 0 && tc::elect_one())
      mma_split16<128 * (grd::kXm - grd::kXh), grd::W1_T>(d, kmajor<grd::kXhK>(sb + xh + 128 * grd::kXh),
                                                          kmajor<kTcK1>(sb + grd::W1), id_kk, bar);
    ok = ok && tc::mbar_wait(bar, phase);
    phase ^= 1u;
    tc::fence_after_sync();
    // h1 -> columns [hc, hc + 32) of the [h1 | x] tile; mask1 = [h1 > 0]
    unsigned mask1 = 0u;
    {
      Parts p;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float v[16];
        tc::tmem_ld16(lane_base + 16 * q, v);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          v[i] = fmaxf(v[i], 0.f);
          if (v[i] > 0.f) mask1 |= 1u << (16 * q + i);
        }
        split16(v, q, p);
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) parts_to_tmem<true>(d + lane_off, half, q, p);
      parts_to_smem<grd::kXhK, grd::kHh, grd::kHm, grd::kHl>(S + xh, row, half, p);
    }
    tc::tmem_st_wait();
    tc::fence_proxy_async();
    tc::fence_before_sync();
    tc::bar_sync(bid, kGroup);
    if (warp == 0 && tc::elect_one())
      mma_split_ta<true, grd::W2_T>(d + grd::kColD2, d, 0, kmajor<kMlpHid>(sb + grd::W2), id_kk, bar);
    ok = ok && tc::mbar_wait(bar, phase);
    if (PROBE && tile == fail) ok = false;
    phase ^= 1u;
    tc::fence_after_sync();
    {  // logit from the two halves' partial sums
      uint64_t acc2 = 0;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float v[16];
        tc::tmem_ld16(lane_base + grd::kColD2 + 16 * q, v);
        relu16(v, b2 + hc + 16 * q);
        acc2 = dot16(v, w3 + hc + 16 * q, acc2);
      }
      float acc, odd;
      tc::unpack2(acc2, acc, odd);
      part[half * kTcM + row] = acc + odd;
    }
    tc::bar_sync(bid, kGroup);
    const float z3 = b3 + part[row] + part[kTcM + row];
    const float g = valid ? 1.f / (1.f + expf(-z3)) - y : 0.f;
    // e2 columns [hc, hc + 32) and dW3 partial sums; e2 to tensor memory, where h1 was
    Parts p;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float v[16];
      tc::tmem_ld16(lane_base + grd::kColD2 + 16 * q, v);
      relu16(v, b2 + hc + 16 * q);
      const uint64_t gg = tc::pack2(g, g);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        uint64_t& a3 = acc3[8 * q + i];
        a3 = tc::fma2(gg, tc::pack2(v[2 * i], v[2 * i + 1]), a3);
        const float2 w = *reinterpret_cast<const float2*>(w3 + hc + 16 * q + 2 * i);
        float e0, e1;
        tc::unpack2(tc::mul2(gg, tc::pack2(w.x, w.y)), e0, e1);
        v[2 * i] = v[2 * i] > 0.f ? e0 : 0.f;
        v[2 * i + 1] = v[2 * i + 1] > 0.f ? e1 : 0.f;
      }
      split16(v, q, p);
      parts_to_tmem<true>(d + lane_off, half, q, p);
    }
    tc::tmem_st_wait();
    tc::fence_before_sync();
    tc::bar_sync(bid, kGroup);
    // D3 = E2 W2: W2's K-major tile (rows o, columns i) read MN-major is W2^T (n = i, k = o).
    if (warp == 0) {
      if (tc::elect_one())
        mma_split_ta<true, grd::W2_T>(d + grd::kColD2, d, 0, mnmajor<kMlpHid>(sb + grd::W2), id_kk | kBmn, bar);
      __syncwarp();
      if (t == 0 && ok) {  // the e tile: the other group's until its gradient MMAs are done
        const uint64_t t0 = tc::global_ns();
        while (!(locked = atomicCAS(lock, 0, 1) == 0) && tc::global_ns() - t0 < 2000000000ull) __nanosleep(20);
        ok = locked;
        __threadfence_block();
      }
    }
    if (tc::bar_or(bid, kGroup, !ok)) {
      phase ^= 1u;  // the third layer's MMAs are in flight
      break;
    }
    parts_to_smem<grd::kEK, 0, 8, 16>(S + grd::E, row, half, p);
    tc::fence_proxy_async();
    tc::bar_sync(bid, kGroup);
    // Dg2 += E2^T [H1 | X], K = the tile's 128 samples.
    if (warp == 0 && tc::elect_one())
      mma_grad<64, grd::kHm, 144, grd::kHh, 80, grd::kHl, 64>(tmem + grd::kColG2, e_mn, xh_mn, bar + 1, *used != 0);
    if (tile + stride < n_tiles) {
      const int rn = (tile + stride) * kTcM + row;
      fetch_half(feats, rn, n, half, fin);
      yin = rn < n ? labels[rn] : 0.f;
    }
    if (half == 0) {  // under the gradient MMA
      if (valid) lsum += fmaxf(z3, 0.f) - z3 * y + log1pf(expf(-fabsf(z3)));
      gsum += g;
    }
    ok = ok && tc::mbar_wait(bar, phase);
    phase ^= 1u;
    tc::fence_after_sync();
    ok = ok && tc::mbar_wait(bar + 1, gphase);
    gphase ^= 1u;
    tc::fence_after_sync();
    // e1
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float v[16];
      tc::tmem_ld16(lane_base + grd::kColD2 + 16 * q, v);
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = (mask1 >> (16 * q + i)) & 1u ? v[i] : 0.f;
      split16(v, q, p);
    }
    parts_to_smem<grd::kEK, 0, 8, 16>(S + grd::E, row, half, p);
    tc::fence_proxy_async();
    tc::fence_before_sync();
    tc::bar_sync(bid, kGroup);
    // Dg1 += E1^T X
    if (warp == 0 && tc::elect_one())
      mma_grad<0, grd::kXh, 32, grd::kXh, 16, grd::kXl, 16>(tmem + grd::kColG1, e_mn, xh_mn, bar + 1, *used != 0);
    standardise_half(fin, half, (tile + stride) * kTcM + row < n ? mean : nil, sd, rs, by_rs, x);
    ok = ok && tc::mbar_wait(bar + 1, gphase);
    gphase ^= 1u;
    tc::fence_after_sync();
    if (t == 0) {
      *used = 1;
      __threadfence_block();
      atomicExch(lock, 0);
      locked = false;
    }
  }
  if (tc::bar_or(bid, kGroup, !ok)) {
    // A tensor-core wait gave up: the loss becomes NaN and the block adds nothing to the gradient; the
    // MMAs in flight get one more bounded wait before the tensor memory is released.
    if (t == 0) {
      if (locked) atomicExch(lock, 0);
      atomicAdd(loss, __int_as_float(0x7fc00000));
    }
    tc::mbar_wait(bar, phase ^ 1u);
    tc::mbar_wait(bar + 1, gphase ^ 1u);
    gsum = lsum = 0.f;
  }
  // dW3, db3 and the loss: over the warp's samples, then over the eight warps of each half.
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  {
    float v[32];
#pragma unroll
    for (int j = 0; j < 16; ++j) tc::unpack2(acc3[j], v[2 * j], v[2 * j + 1]);
    red[wid * 34 + lane] = warp_sum32(v, lane);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    gsum += __shfl_xor_sync(0xffffffffu, gsum, o);
    lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  }
  if (lane == 0) {
    red[wid * 34 + 32] = gsum;
    red[wid * 34 + 33] = lsum;
  }
  tc::fence_before_sync();
  const bool failed = __syncthreads_or(!ok);
  tc::fence_after_sync();
  if (threadIdx.x < kMlpHid + 2 && !failed) {
    const int j = threadIdx.x;  // dW3[j], db3, loss: warps 0-3 and 8-11 hold units 0-31, the others 32-63
    float v = 0.f;
    for (int w = 0; w < 16; ++w) {
      if (j < kMlpHid) v += ((w >> 2) & 1) == (j >> 5) ? red[w * 34 + (j & 31)] : 0.f;
      else v += red[w * 34 + 32 + j - kMlpHid];
    }
    if (j <= kMlpHid) atomicAdd(grad + (j < kMlpHid ? kMlpW3 + j : kMlpB3), v * inv_n);
    else atomicAdd(loss, v * inv_n);
  }
  // The gradient accumulators: unit u is rows u and 64 + u. Warps w with w % 4 >= 2 hold the latter and
  // pass them through shared memory (where the e tile was); the four pairs of warps of each half take
  // 16 columns of dW2 each, the second also db2, the third dW1 and db1.
  {
    const int rr = 32 * (wid & 3) + lane, u = rr & 63, q = wid >> 2;
    float v[16], w[16];
    float* st = reinterpret_cast<float*>(S + grd::E);  // [5][64][17]
    auto meet = [&](float* z, int k) {
      float* m = st + (k * 64 + u) * 17;
      if (rr >= 64)
#pragma unroll
        for (int i = 0; i < 16; ++i) m[i] = z[i];
      __syncthreads();
      if (rr < 64)
#pragma unroll
        for (int i = 0; i < 16; ++i) z[i] = (z[i] + m[i]) * inv_n;
    };
    const bool any = *used != 0 && !failed;
    if (any) {
      tc::tmem_ld16(tmem + lane_off + grd::kColG2 + 16 * q, v);
      tc::tmem_ld16(tmem + lane_off + grd::kColG2 + 64 + 16 * q, w);
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] += w[i];
      if (q == 1) {
        tc::tmem_ld16(tmem + lane_off + grd::kColG2 + 128, w);
      } else if (q == 2) {
        float w2[16];
        tc::tmem_ld16(tmem + lane_off + grd::kColG1, w);
        tc::tmem_ld16(tmem + lane_off + grd::kColG1 + 16, w2);
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] += w2[i];
      }
    }
    meet(v, q);
    __syncthreads();
    meet(w, q);
    if (any && rr < 64) {
#pragma unroll
      for (int i = 0; i < 4; ++i) add4(grad + kMlpW2 + u * kMlpHid + 16 * q + 4 * i, v + 4 * i);
      if (q == 1) {
        atomicAdd(grad + kMlpB2 + u, w[kOne]);
      } else if (q == 2) {
#pragma unroll
        for (int k = 0; k < kMlpIn; ++k) atomicAdd(grad + kMlpW1 + u * kMlpIn + k, w[k]);
        atomicAdd(grad + kMlpB1 + u, w[kOne]);
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (threadIdx.x < 32) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, grd::kCols);
  }
}

__global__ void k_mlp_zero(float* grad, float* loss) {
  pdl_begin();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < kMlpParams) grad[p] = 0.f;
  else if (p == kMlpParams) *loss = 0.f;
}

// Adam (Kingma and Ba) on the weights; moments m, v; step t >= 1.
__global__ void k_mlp_adam(float* params, const float* grad, float* m, float* v, int t, float lr, float b1, float b2,
                           float eps) {
  pdl_begin();
  const float c1 = 1.f - powf(b1, static_cast<float>(t)), c2 = 1.f - powf(b2, static_cast<float>(t));
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < kMlpParams; p += gridDim.x * blockDim.x) {
    const float g = grad[p];
    const float mp = b1 * m[p] + (1.f - b1) * g;
    const float vp = b2 * v[p] + (1.f - b2) * g * g;
    m[p] = mp;
    v[p] = vp;
    params[p] -= lr * (mp / c1) / (sqrtf(vp / c2) + eps);
  }
}

// Number of SMs of the current device and, once per device, the kernel's shared-memory opt-in.
static int tc_prepare(const void* kernel, int smem, int* sms) {
  static int sm_count[64] = {0};
  static int smem_set[3][64] = {{0}};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -3;
  if (!sm_count[dev] && cudaDeviceGetAttribute(&sm_count[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return -3;
  const int which = kernel == reinterpret_cast<const void*>(k_mlp_forward)            ? 0
                    : kernel == reinterpret_cast<const void*>(k_mlp_loss_grad<false>) ? 1
                                                                                      : 2;
  if (smem > smem_set[which][dev]) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return -3;
    smem_set[which][dev] = smem;
  }
  *sms = sm_count[dev];
  return 0;
}

int launch_mlp_forward(const float* params, const float* feats, int n, float* logits, cudaStream_t st) {
  if (n == 0) return 0;
  const int smem = static_cast<int>(fwd::BYTES) + 1024;
  int sms = 0;
  if (tc_prepare(reinterpret_cast<const void*>(k_mlp_forward), smem, &sms) != 0) return -3;
  const int tiles = (n + kTcM - 1) / kTcM;
  launch_pdl(k_mlp_forward, std::min(tiles, sms), fwd::kGroups * kGroup, smem, st, params, feats, n, logits);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

template <bool PROBE>
static int launch_loss_grad(const float* params, const float* feats, const float* labels, int n, float* grad, float* loss,
                            int fail, cudaStream_t st) {
  const int smem = static_cast<int>(grd::BYTES) + 1024;
  int sms = 0;
  if (tc_prepare(reinterpret_cast<const void*>(k_mlp_loss_grad<PROBE>), smem, &sms) != 0) return -3;
  launch_pdl(k_mlp_zero, (kMlpParams + 256) / 256, 256, 0, st, grad, loss);
  const int tiles = (n + kTcM - 1) / kTcM;
  if (n > 0)
    launch_pdl(k_mlp_loss_grad<PROBE>, std::min(tiles, sms), grd::kGroups * kGroup, smem, st, params, feats, labels, n, 1.f / n,
               grad, loss, fail);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int launch_mlp_loss_grad(const float* params, const float* feats, const float* labels, int n, float* grad, float* loss,
                         cudaStream_t st) {
  return launch_loss_grad<false>(params, feats, labels, n, grad, loss, -1, st);
}

int launch_mlp_wait_probe(const float* params, const float* feats, const float* labels, int n, float* grad, float* loss,
                          int fail, cudaStream_t st) {
  return launch_loss_grad<true>(params, feats, labels, n, grad, loss, fail, st);
}

int launch_mlp_adam(float* params, const float* grad, float* m, float* v, int t, float lr, float b1, float b2, float eps,
                    cudaStream_t st) {
  launch_pdl(k_mlp_adam, (kMlpParams + 255) / 256, 256, 0, st, params, grad, m, v, t, lr, b1, b2, eps);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // namespace kfgb
