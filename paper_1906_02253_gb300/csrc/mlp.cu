// Learned hit proposal: an MLP 14 -> 64 -> 64 -> 1 (ReLU) scoring (predicted candidate, hit)
// pairs, trained on the GPU with these kernels (binary cross-entropy with logits, Adam). The
// network is not in the paper; the features and the pruning rule are described in kfgb.h.
//
// Parameter buffer (FP32): W1[64][14], b1[64], W2[64][64], b2[64], W3[64], b3, then the feature
// normaliser mean[14], sd[14] (KF_MLP_PARAMS weights + 28).
#include <algorithm>

#include "mlp.cuh"
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

// Inference: per tile, standardised inputs -> X tile (128 x 16); D = X W1^T in tensor memory; h1 =
// relu(D) -> H tile (128 x 64, over the X tile, which the finished MMA no longer needs); D = H W2^T;
// logit = b3 + sum_j W3[j] relu(D[j] + b2[j]) on the CUDA cores. Four groups per CTA (1024 threads
// at 64 registers; shared memory for four H tiles and one set of weights): on 1,000,003 rows
// FWD_NOTE
namespace fwd {
constexpr int kGroups = 4;
constexpr uint32_t W1_T = 2048, W2_T = 8192, H_T = 16384, X_T = 4096;  // bytes of one tile
constexpr uint32_t W1 = 0, W2 = W1 + 3 * W1_T, H = W2 + 3 * W2_T, B2 = H + kGroups * 3 * H_T, W3 = B2 + 256,
                   MEAN = W3 + 256, SD = MEAN + 64, PART = SD + 64, BAR = PART + kGroups * 512, TMEM = BAR + 8 * kGroups,
                   BYTES = TMEM + 8;
constexpr uint32_t kCols = 64 * kGroups;
static_assert(BYTES + 1024 <= 227 * 1024 && 3 * X_T <= 3 * H_T, "shared-memory layout");
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

// Standardised inputs [8 h, 8 h + 8) into x[8] (zero past n), the one and the zero.
__device__ __forceinline__ void standardise_half(const float2* f, bool valid, int half, const float* mean,
                                                 const float* sd, float* x) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = 8 * half + 2 * i;
    x[2 * i] = (valid && k < kMlpIn) ? (f[i].x - mean[k]) / sd[k] : 0.f;
    x[2 * i + 1] = (valid && k + 1 < kMlpIn) ? (f[i].y - mean[k + 1]) / sd[k + 1] : 0.f;
  }
  if (half == 1) x[kOne - 8] = 1.f;
}

// This thread's 16 columns [c, c + 16) of sum_j w3[j] relu(v[j] + b2[j]) onto acc (columns 16-byte
// aligned in shared memory).
__device__ __forceinline__ float out_layer16(const float* v, const float* b2, const float* w3, float acc) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 b = reinterpret_cast<const float4*>(b2)[i], w = reinterpret_cast<const float4*>(w3)[i];
    acc = fmaf(w.x, fmaxf(v[4 * i] + b.x, 0.f), acc);
    acc = fmaf(w.y, fmaxf(v[4 * i + 1] + b.y, 0.f), acc);
    acc = fmaf(w.z, fmaxf(v[4 * i + 2] + b.z, 0.f), acc);
    acc = fmaf(w.w, fmaxf(v[4 * i + 3] + b.w, 0.f), acc);
  }
  return acc;
}

// One MMA operand in shared memory: the first of its three tiles (shared-window address), the
// tile size, the descriptor's leading and stride byte offsets, and the byte advance per K = 16 step.
struct Operand {
  uint32_t base, tile, lbo, sbo, step;
};

// K-major operand (tc.cuh layout) of a tile with kt columns, starting at column block c0.
__device__ __forceinline__ Operand kmajor(uint32_t base, uint32_t tile, int kt, int c0 = 0) {
  return Operand{base + 128u * c0, tile, 128u, static_cast<uint32_t>(kt / 8 * 128), 256u};
}

// The same tile read MN-major (its rows become K, its columns M or N): 8-column blocks are 128 B
// apart (stride byte offset), 8-row groups kt / 8 * 128 B apart (leading byte offset).
__device__ __forceinline__ Operand mnmajor(uint32_t base, uint32_t tile, int kt, int c0 = 0) {
  const uint32_t g = static_cast<uint32_t>(kt / 8 * 128);
  return Operand{base + 128u * c0, tile, g, 128u, 2u * g};
}

// D = A B^T over k_steps steps of K = 16 as the six products of the three-part split (hi*hi,
// hi*mid, mid*hi, hi*lo, lo*hi, mid*mid); one thread issues, the mbarrier receives the
// completion; the first product overwrites D unless accumulate is set.
__device__ __forceinline__ void mma_split(uint32_t d, const Operand& A, const Operand& B, int k_steps, uint32_t idesc,
                                          uint64_t* bar, bool accumulate = false) {
  constexpr int kPa[6] = {0, 0, 1, 0, 2, 1}, kPb[6] = {0, 1, 0, 2, 0, 1};
  tc::fence_after_sync();
  for (int k = 0; k < k_steps; ++k) {
#pragma unroll
    for (int p = 0; p < 6; ++p) {
      const uint64_t ad = tc::smem_desc(A.base + A.tile * kPa[p] + A.step * k, A.lbo, A.sbo);
      const uint64_t bd = tc::smem_desc(B.base + B.tile * kPb[p] + B.step * k, B.lbo, B.sbo);
      tc::mma_bf16(d, ad, bd, idesc, (k > 0 || p > 0 || accumulate) ? 1u : 0u);
    }
  }
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
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(S + fwd::TMEM);
  const int gi = threadIdx.x / kGroup, t = threadIdx.x % kGroup, warp = t >> 5, row = t & (kTcM - 1), half = t / kTcM;
  float* part = reinterpret_cast<float*>(S + fwd::PART) + gi * kTcM;  // second half's output-layer sums
  uint64_t* bar = reinterpret_cast<uint64_t*>(S + fwd::BAR) + gi;
  const uint32_t h_off = fwd::H + gi * 3 * fwd::H_T;  // this group's H tile, and X tile before it
  const int bid = gi + 1;

  stage_weights_b(params, S + fwd::W1, fwd::W1_T, S + fwd::W2, fwd::W2_T);
  if (threadIdx.x < kMlpHid) {
    b2[threadIdx.x] = params[kMlpB2 + threadIdx.x];
    w3[threadIdx.x] = params[kMlpW3 + threadIdx.x];
  }
  if (threadIdx.x < kMlpIn) {
    mean[threadIdx.x] = params[kMlpMean + threadIdx.x];
    sd[threadIdx.x] = params[kMlpSd + threadIdx.x];
  }
  const float b3 = params[kMlpB3];
  if (threadIdx.x < 32) tc::tmem_alloc(tmem_slot, fwd::kCols);
  if (t == 0) tc::mbar_init(bar, 1);
  tc::fence_proxy_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot, d = tmem + 64u * gi;
  const uint32_t lane_base = d + (static_cast<uint32_t>((warp & 3) * 32) << 16) + 32u * half;
  constexpr uint32_t idesc = tc::idesc_bf16_f32(kTcM, kMlpHid);
  uint32_t phase = 0;
  bool ok = true;  // a wait that gives up ends the group's tiles; until then its threads keep in step

  const int n_tiles = (n + kTcM - 1) / kTcM;
  const int tile0 = blockIdx.x + gridDim.x * gi, stride = gridDim.x * fwd::kGroups;
  int tile = tile0;
  float2 fin[4];  // this thread's half of the raw features of its sample in the next tile
  fetch_half(feats, tile * kTcM + row, n, half, fin);
  for (; tile < n_tiles; tile += stride) {
    const int r = tile * kTcM + row;
    {
      float x[8];
      standardise_half(fin, r < n, half, mean, sd, x);
      tc::store8_split(S + h_off, fwd::X_T, tc::kmajor_off(row, half, kTcK1), x);
    }
    tc::fence_proxy_async();
    tc::bar_sync(bid, kGroup);
    if (t == 0) mma_split(d, kmajor(sb + h_off, fwd::X_T, kTcK1), kmajor(sb + fwd::W1, fwd::W1_T, kTcK1), 1, idesc, bar);
    if (tile + stride < n_tiles) fetch_half(feats, (tile + stride) * kTcM + row, n, half, fin);  // in flight meanwhile
    ok = ok && tc::mbar_wait(bar, phase);
    phase ^= 1u;
    tc::fence_after_sync();
    // h1 columns [32 h, 32 h + 32) -> the H tile
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float v[16];
      tc::tmem_ld16(lane_base + 16 * q, v);
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = fmaxf(v[i], 0.f);
      tc::store8_split(S + h_off, fwd::H_T, tc::kmajor_off(row, 4 * half + 2 * q, kMlpHid), v);
      tc::store8_split(S + h_off, fwd::H_T, tc::kmajor_off(row, 4 * half + 2 * q + 1, kMlpHid), v + 8);
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    tc::bar_sync(bid, kGroup);
    if (t == 0) mma_split(d, kmajor(sb + h_off, fwd::H_T, kMlpHid), kmajor(sb + fwd::W2, fwd::W2_T, kMlpHid), 4, idesc, bar);
    ok = ok && tc::mbar_wait(bar, phase);
    phase ^= 1u;
    tc::fence_after_sync();
    float acc = 0.f;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float v[16];
      tc::tmem_ld16(lane_base + 16 * q, v);
      acc = out_layer16(v, b2 + 32 * half + 16 * q, w3 + 32 * half + 16 * q, acc);
    }
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
  k_mlp_fragments<<<(kFragWords + 255) / 256, 256, 0, st>>>(params, frag);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// The finder's scoring outside the finder: warp w of the grid takes rows 8w .. 8w + 7, lane l the
// features of row 8w + l / 4 in its operand columns, standardised as the finder standardises its
// candidate features and pulls; lanes 0-3 write the logits of rows 8w + 2l, 8w + 2l + 1.
__global__ void k_mlp_finder_scores(const uint4* __restrict__ frag, const float* __restrict__ prm,
                                    const float* __restrict__ feats, int n, float* __restrict__ logits) {
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
  k_mlp_finder_scores<<<static_cast<unsigned>((warps + 7) / 8), 256, 0, st>>>(frag, params, feats, n, logits);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// Loss and gradient on the tensor cores. Per tile of a group:
//   D1 = X W1^T -> h1 = relu(D1);  D2 = H1 W2^T -> z3 = b3 + W3 . relu(D2 + b2),
//   g = (sigmoid(z3) - y), e2 = g W3 [z2 > 0];  D3 = E2 W2 -> e1 = D3 [h1 > 0];
//   Dg2 += E2^T [H1 | X],  Dg1 += E1^T X   (accumulated in tensor memory over all the CTA's tiles),
// so that Dg2's rows 0-63 hold dW2 (columns 0-63) and db2 (column 64 + 14, X's ones) and Dg1's rows
// 0-63 dW1 (columns 0-13) and db1 (column 14). dW3, db3 and the loss are summed in registers.
//
// Two groups per CTA. Shared memory (bytes; each operand three tiles, hi, mid, lo): each group's
// sample x [h1 | x] tile (128 x 80: the A operand of the first two MMAs, K-major, and the B operand of
// the gradient MMAs, read MN-major), one sample x e tile (128 x 64: e2, then e1; K-major the A
// operand of the third MMA, MN-major of the gradient MMAs), W1 and W2 (W2 read MN-major is W2^T for
// the third MMA). The e tile is one group's at a time, from its e2 until its last MMA; the other
// group then runs its forward layers. A gradient MMA has M = 128 with the tile's 64 columns as
// the first rows; the rest reads what lies behind in shared memory (the next rows' values, at
// the end the [h1 | x] tile) into accumulator rows 64-127, which nothing uses.
// Tensor memory: per group D1 then D3 at 0 and D2 at 64; Dg2 at 256, Dg1 at 336.
// GRD_NOTE
namespace grd {
constexpr int kGroups = 2;
constexpr uint32_t E_T = 16384, XH_T = 20480, W1_T = 2048, W2_T = 8192;  // bytes of one tile
constexpr uint32_t E = 0, XH = E + 3 * E_T, W2 = XH + kGroups * 3 * XH_T, W1 = W2 + 3 * W2_T, B2 = W1 + 3 * W1_T,
                   W3 = B2 + 256, MEAN = W3 + 256, SD = MEAN + 64, PART = SD + 64, RED = PART + kGroups * 1024,
                   BAR = RED + 16 * 34 * 4, TMEM = BAR + 16 * kGroups, LOCK = TMEM + 4, USED = LOCK + 4, BYTES = USED + 8;
static_assert(BYTES + 1024 <= 227 * 1024, "shared-memory layout");
constexpr uint32_t kCols = 512, kColD2 = 64, kColG2 = 256, kColG1 = 336;
constexpr int kXhK = 80, kEK = 64;
}  // namespace grd

// Instruction descriptor bits 15 and 16: A, B MN-major.
constexpr uint32_t kAmn = 1u << 15, kBmn = 1u << 16;

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

__global__ void __launch_bounds__(grd::kGroups* kGroup, 1)
    k_mlp_loss_grad(const float* __restrict__ params, const float* __restrict__ feats, const float* __restrict__ labels,
                    int n, float inv_n, float* __restrict__ grad, float* __restrict__ loss) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* S = smem_raw + ((1024 - (tc::smem_u32(smem_raw) & 1023)) & 1023);
  const uint32_t sb = tc::smem_u32(S);
  float* b2 = reinterpret_cast<float*>(S + grd::B2);
  float* w3 = reinterpret_cast<float*>(S + grd::W3);
  float* mean = reinterpret_cast<float*>(S + grd::MEAN);
  float* sd = reinterpret_cast<float*>(S + grd::SD);
  float* red = reinterpret_cast<float*>(S + grd::RED);  // [16 warps][34]: dW3 of the warp's 32 units, db3, loss
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(S + grd::TMEM);
  int* lock = reinterpret_cast<int*>(S + grd::LOCK);  // 1: the e tile is taken
  int* used = reinterpret_cast<int*>(S + grd::USED);  // 1: the gradient accumulators hold a tile
  const int gi = threadIdx.x / kGroup, t = threadIdx.x % kGroup, warp = t >> 5, row = t & (kTcM - 1), half = t / kTcM;
  const int hc = 32 * half;  // this thread's first column of a 64-column accumulator
  float* part = reinterpret_cast<float*>(S + grd::PART) + gi * 2 * kTcM;  // [2][128] output-layer partial sums
  // bar[0]: the layers' MMAs, bar[1]: the gradient MMAs (the first of them is in flight with the third layer's)
  uint64_t* bar = reinterpret_cast<uint64_t*>(S + grd::BAR) + 2 * gi;
  const uint32_t xh = grd::XH + gi * 3 * grd::XH_T;
  const int bid = gi + 1;

  stage_weights_b(params, S + grd::W1, grd::W1_T, S + grd::W2, grd::W2_T);
  if (threadIdx.x < kMlpHid) {
    b2[threadIdx.x] = params[kMlpB2 + threadIdx.x];
    w3[threadIdx.x] = params[kMlpW3 + threadIdx.x];
  }
  if (threadIdx.x < kMlpIn) {
    mean[threadIdx.x] = params[kMlpMean + threadIdx.x];
    sd[threadIdx.x] = params[kMlpSd + threadIdx.x];
  }
  const float b3 = params[kMlpB3];
  if (threadIdx.x < 32) tc::tmem_alloc(tmem_slot, grd::kCols);
  if (threadIdx.x == 0) *lock = *used = 0;
  if (t == 0) {
    tc::mbar_init(bar, 1);
    tc::mbar_init(bar + 1, 1);
  }
  tc::fence_proxy_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot, d = tmem + 128u * gi;
  const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
  const uint32_t lane_base = d + lane_off + hc;
  constexpr uint32_t id_kk = tc::idesc_bf16_f32(kTcM, kMlpHid);
  constexpr uint32_t id_g2 = tc::idesc_bf16_f32(kTcM, grd::kXhK) | kAmn | kBmn;
  constexpr uint32_t id_g1 = tc::idesc_bf16_f32(kTcM, kTcK1) | kAmn | kBmn;
  const Operand e_k = kmajor(sb + grd::E, grd::E_T, grd::kEK), e_mn = mnmajor(sb + grd::E, grd::E_T, grd::kEK);
  uint32_t phase = 0, gphase = 0;
  bool ok = true, locked = false;
  float acc3[32];  // dW3 partial sums of this thread's 32 hidden units
#pragma unroll
  for (int j = 0; j < 32; ++j) acc3[j] = 0.f;
  float gsum = 0.f, lsum = 0.f;

  const int n_tiles = (n + kTcM - 1) / kTcM;
  const int stride = gridDim.x * grd::kGroups;
  int tile = blockIdx.x + gridDim.x * gi;
  float2 fin[4];  // this thread's half of the raw features, and the label, of its sample in the next tile
  fetch_half(feats, tile * kTcM + row, n, half, fin);
  float yin = tile * kTcM + row < n ? labels[tile * kTcM + row] : 0.f;
  for (; tile < n_tiles; tile += stride) {
    const bool valid = tile * kTcM + row < n;
    {  // inputs -> columns 64-79 of the [h1 | x] tile
      float x[8];
      standardise_half(fin, valid, half, mean, sd, x);
      tc::store8_split(S + xh, grd::XH_T, tc::kmajor_off(row, 8 + half, grd::kXhK), x);
    }
    const float y = yin;
    tc::fence_proxy_async();
    tc::bar_sync(bid, kGroup);
    if (t == 0)
      mma_split(d, kmajor(sb + xh, grd::XH_T, grd::kXhK, 8), kmajor(sb + grd::W1, grd::W1_T, kTcK1), 1, id_kk, bar);
    if (tile + stride < n_tiles) {  // in flight during this tile
      const int rn = (tile + stride) * kTcM + row;
      fetch_half(feats, rn, n, half, fin);
      yin = rn < n ? labels[rn] : 0.f;
    }
    ok = ok && tc::mbar_wait(bar, phase);
    phase ^= 1u;
    tc::fence_after_sync();
    // h1 -> columns [hc, hc + 32) of the [h1 | x] tile; mask1 = [h1 > 0]
    unsigned mask1 = 0u;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float v[16];
      tc::tmem_ld16(lane_base + 16 * q, v);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        v[i] = fmaxf(v[i], 0.f);
        if (v[i] > 0.f) mask1 |= 1u << (16 * q + i);
      }
      tc::store8_split(S + xh, grd::XH_T, tc::kmajor_off(row, 4 * half + 2 * q, grd::kXhK), v);
      tc::store8_split(S + xh, grd::XH_T, tc::kmajor_off(row, 4 * half + 2 * q + 1, grd::kXhK), v + 8);
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    tc::bar_sync(bid, kGroup);
    if (t == 0)
      mma_split(d + grd::kColD2, kmajor(sb + xh, grd::XH_T, grd::kXhK), kmajor(sb + grd::W2, grd::W2_T, kMlpHid), 4, id_kk,
                bar);
    ok = ok && tc::mbar_wait(bar, phase);
    phase ^= 1u;
    tc::fence_after_sync();
    {  // logit from the two halves' partial sums
      float acc = 0.f;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float v[16];
        tc::tmem_ld16(lane_base + grd::kColD2 + 16 * q, v);
        acc = out_layer16(v, b2 + hc + 16 * q, w3 + hc + 16 * q, acc);
      }
      part[half * kTcM + row] = acc;
    }
    if (t == 0 && ok) {  // the e tile: the other group's until its gradient MMAs are done
      const uint64_t t0 = tc::global_ns();
      while (!(locked = atomicCAS(lock, 0, 1) == 0) && tc::global_ns() - t0 < 2000000000ull) __nanosleep(40);
      ok = locked;
      __threadfence_block();
    }
    if (tc::bar_or(bid, kGroup, !ok)) break;
    const float z3 = b3 + part[row] + part[kTcM + row];
    const float g = valid ? 1.f / (1.f + expf(-z3)) - y : 0.f;
    if (half == 0) {
      if (valid) lsum += fmaxf(z3, 0.f) - z3 * y + log1pf(expf(-fabsf(z3)));
      gsum += g;
    }
    // e2 -> columns [hc, hc + 32) of the e tile; dW3 partial sums
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float v[16];
      tc::tmem_ld16(lane_base + grd::kColD2 + 16 * q, v);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 b = reinterpret_cast<const float4*>(b2 + hc + 16 * q)[i];
        const float4 w = reinterpret_cast<const float4*>(w3 + hc + 16 * q)[i];
        const float bb[4] = {b.x, b.y, b.z, b.w}, ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float a2 = fmaxf(v[4 * i + e] + bb[e], 0.f);
          acc3[16 * q + 4 * i + e] = fmaf(g, a2, acc3[16 * q + 4 * i + e]);
          v[4 * i + e] = a2 > 0.f ? g * ww[e] : 0.f;
        }
      }
      tc::store8_split(S + grd::E, grd::E_T, tc::kmajor_off(row, 4 * half + 2 * q, grd::kEK), v);
      tc::store8_split(S + grd::E, grd::E_T, tc::kmajor_off(row, 4 * half + 2 * q + 1, grd::kEK), v + 8);
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    tc::bar_sync(bid, kGroup);
    // D3 = E2 W2: W2's K-major tile (rows o, columns i) read MN-major is W2^T (n = i, k = o). Then
    // Dg2 += E2^T [H1 | X]: both tiles read MN-major, K = the tile's 128 samples.
    if (t == 0) {
      mma_split(d, e_k, mnmajor(sb + grd::W2, grd::W2_T, kMlpHid), 4, id_kk | kBmn, bar);
      mma_split(tmem + grd::kColG2, e_mn, mnmajor(sb + xh, grd::XH_T, grd::kXhK), kTcM / 16, id_g2, bar + 1, *used != 0);
    }
    ok = ok && tc::mbar_wait(bar, phase);
    phase ^= 1u;
    tc::fence_after_sync();
    // e1, split while the gradient MMA still reads e2
    uint4 e1[4][3];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float v[16];
      tc::tmem_ld16(lane_base + 16 * q, v);
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = (mask1 >> (16 * q + i)) & 1u ? v[i] : 0.f;
      tc::split8(v, e1[2 * q][0], e1[2 * q][1], e1[2 * q][2]);
      tc::split8(v + 8, e1[2 * q + 1][0], e1[2 * q + 1][1], e1[2 * q + 1][2]);
    }
    ok = ok && tc::mbar_wait(bar + 1, gphase);
    gphase ^= 1u;
    tc::fence_after_sync();
#pragma unroll
    for (int c = 0; c < 4; ++c)
      tc::store8(S + grd::E, grd::E_T, tc::kmajor_off(row, 4 * half + c, grd::kEK), e1[c][0], e1[c][1], e1[c][2]);
    tc::fence_proxy_async();
    tc::fence_before_sync();
    tc::bar_sync(bid, kGroup);
    // Dg1 += E1^T X
    if (t == 0)
      mma_split(tmem + grd::kColG1, e_mn, mnmajor(sb + xh, grd::XH_T, grd::kXhK, 8), kTcM / 16, id_g1, bar + 1, *used != 0);
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
    // A tensor-core wait gave up: the loss becomes NaN; the MMAs in flight get one more bounded wait
    // before the tensor memory is released.
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
  red[wid * 34 + lane] = warp_sum32(acc3, lane);
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
  __syncthreads();
  tc::fence_after_sync();
  if (threadIdx.x < kMlpHid + 2) {
    const int j = threadIdx.x;  // dW3[j], db3, loss: warps 0-3 and 8-11 hold units 0-31, the others 32-63
    float v = 0.f;
    for (int w = 0; w < 16; ++w) {
      if (j < kMlpHid) v += ((w >> 2) & 1) == (j >> 5) ? red[w * 34 + (j & 31)] : 0.f;
      else v += red[w * 34 + 32 + j - kMlpHid];
    }
    if (j <= kMlpHid) atomicAdd(grad + (j < kMlpHid ? kMlpW3 + j : kMlpB3), v * inv_n);
    else atomicAdd(loss, v * inv_n);
  }
  // The gradient accumulators' rows 0-63 (tensor-memory lanes 0-63, the warps w with w % 4 < 2): the
  // four such pairs of warps take 16 columns of dW2 each; db2 (pair 1), dW1 and db1 (pair 2).
  if (*used && (wid & 3) < 2) {
    const int j = 32 * (wid & 3) + lane, q = wid >> 2;
    float v[16];
    tc::tmem_ld16(tmem + lane_off + grd::kColG2 + 16 * q, v);
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] *= inv_n;
#pragma unroll
    for (int i = 0; i < 4; ++i) add4(grad + kMlpW2 + j * kMlpHid + 16 * q + 4 * i, v + 4 * i);
    if (q == 1) {
      tc::tmem_ld16(tmem + lane_off + grd::kColG2 + 64, v);
      atomicAdd(grad + kMlpB2 + j, v[kOne] * inv_n);
    }
    if (q == 2) {
      tc::tmem_ld16(tmem + lane_off + grd::kColG1, v);
#pragma unroll
      for (int k = 0; k < kMlpIn; ++k) atomicAdd(grad + kMlpW1 + j * kMlpIn + k, v[k] * inv_n);
      atomicAdd(grad + kMlpB1 + j, v[kOne] * inv_n);
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
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < kMlpParams) grad[p] = 0.f;
  else if (p == kMlpParams) *loss = 0.f;
}

// Adam (Kingma and Ba) on the weights; moments m, v; step t >= 1.
__global__ void k_mlp_adam(float* params, const float* grad, float* m, float* v, int t, float lr, float b1, float b2,
                           float eps) {
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
  static int smem_set[2][64] = {{0}};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -3;
  if (!sm_count[dev] && cudaDeviceGetAttribute(&sm_count[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return -3;
  const int which = kernel == reinterpret_cast<const void*>(k_mlp_forward) ? 0 : 1;
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
  k_mlp_forward<<<std::min(tiles, sms), fwd::kGroups * kGroup, smem, st>>>(params, feats, n, logits);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int launch_mlp_loss_grad(const float* params, const float* feats, const float* labels, int n, float* grad, float* loss,
                         cudaStream_t st) {
  const int smem = static_cast<int>(grd::BYTES) + 1024;
  int sms = 0;
  if (tc_prepare(reinterpret_cast<const void*>(k_mlp_loss_grad), smem, &sms) != 0) return -3;
  k_mlp_zero<<<(kMlpParams + 256) / 256, 256, 0, st>>>(grad, loss);
  const int tiles = (n + kTcM - 1) / kTcM;
  if (n > 0)
    k_mlp_loss_grad<<<std::min(tiles, sms), grd::kGroups * kGroup, smem, st>>>(params, feats, labels, n, 1.f / n, grad, loss);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int launch_mlp_adam(float* params, const float* grad, float* m, float* v, int t, float lr, float b1, float b2, float eps,
                    cudaStream_t st) {
  k_mlp_adam<<<(kMlpParams + 255) / 256, 256, 0, st>>>(params, grad, m, v, t, lr, b1, b2, eps);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // namespace kfgb
