// Combinatorial Kalman-filter track finding, host side and plain instances: the seed states,
// launch plans (capacity, block size, adaptive capacity), the allocation-free scratch and the
// dispatch of the compiled instances. The kernel itself is in find_kernel.cuh.
#include "find_kernel.cuh"
#include "pdl.cuh"

namespace kfgb {

// Order of the seeds by direction, for geometries with disks. A track's length and the kind of its
// surfaces follow from |cot theta|: with seeds in index order a warp mixes lanes that head for
// barrel layers with lanes that head for disks, and tracks of 12 surfaces with tracks of 20, so
// both path solvers run for it and its block waits for the longest step. Seeds of a class of
// |cot theta| / (1 + |cot theta|) run together, the central ones (most surfaces) first, so that the
// last seeds are short. 24 classes (finder alone, measured on sorted seeds): 100 barrel + disk
// events 4.57 -> 3.97 ms (8 classes 4.07, fully sorted 3.92, longest last 4.37, sorted in chunks of
// 20 events 4.34), learned 4.38 -> 3.78, field map 1.75 -> 1.34. The order spans the batch, so the longer
// it is the more of the index is read from memory again; the present kernels against index order (a
// workspace without the list), ns a seed on 60, 100, 300 and 600 events: two passes 7.4/8.4, 7.5/8.1,
// 7.7/7.6, 7.7/7.6; one pass 9.4/9.9, 9.7/9.9, 9.9/9.8, 9.9/9.8; learned in two passes 7.0/7.8, 6.7/7.1,
// 6.9/7.2, 6.7/6.7, in one 17.4/18.1, 17.9/18.1, 18.4/18.0, 18.6/18.0; field map 10.8/12.4, 11.2/12.8,
// 11.5/12.3, 11.5/12.3. On barrel layers alone every track crosses all of them and the order of the
// events serves the cache: sorted 10.4 against 9.8 ms, so there the seeds stay in index order.
constexpr int kClasses = 24;
__device__ __forceinline__ int seed_class(float theta) {
  float st, ct;
  sincos_small(theta, st, ct);
  const float u = fabsf(ct);
  return min(max(static_cast<int>(u / (u + fabsf(st)) * kClasses), 0), kClasses - 1);
}

// Seed states, one thread per seed: the circle seed of the three hits and the filter over them
// (update with hit 1, propagate and update through hits 2 and 3). For the finder (FIND) each seed's
// state is one record of kSeedWords words (p[6], C[21], chi2), which its order of seeds reads
// whole; kf_seed_states gets a structure of arrays. chi2 < 0 marks a failed seed, whose track
// outputs are written here.
//
// Geometries without disks take their seeds in index order, but for those that curl within the
// layers, |omega| R > 1.7 with R the outermost radius: the particles that reach the outer layers
// are straighter, so these come from wrong combinations of hits. Their windows are wide, and a
// block that holds one waits for it at every step: where they are 1 in 64 seeds or more they are taken
// first, together, from a list. 218,000 seeds of overlapping modules, 31% of them such: the whole
// pass 3.32 -> 2.96 ms; the other barrel workloads hold next to none (2 in 10,000) and stay in index
// order (looking costs 100 events 0.3%).
constexpr float kCurling = 1.7f;
template <bool FIND>
__global__ void __launch_bounds__(128) k_seed_states(DevGeom G, const __grid_constant__ DevMat M, FindArgs A) {
  pdl_begin();
  const int seed = blockIdx.x * blockDim.x + threadIdx.x;
  const int n = A.n_seeds;
  const bool in = seed < n;
  int ids[3] = {-1, -1, -1}, ev = -1;
  bool removed = false;
  if (in) {
#pragma unroll
    for (int k = 0; k < 3; ++k) ids[k] = A.seed_hits[static_cast<size_t>(k) * n + seed];
    ev = A.seed_event[seed];
    removed = A.seed_keep && A.seed_keep[seed] == 0;
  }
  bool ok = !removed && ids[0] >= 0 && ids[1] >= 0 && ids[2] >= 0 && ev >= 0 && ev < A.n_events;
  Cand c;
  int ss[3] = {0, 0, 0};
  if (ok) {
    float xs[3], ys[3], zs[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float2 h = A.hits[ids[k]];
      ss[k] = A.hit_surface[ids[k]];
      ok = ok && ss[k] >= 0 && ss[k] < G.n_surf;
      if (ok) hit_xyz(G, ss[k], h.x, h.y, xs[k], ys[k], zs[k]);
    }
    ok = ok && seed_from_hits(G, xs, ys, zs, ss[0], c.p, c.C);
  }
  c.chi2 = 0.f;
  for (int k = 0; k < 3 && ok; ++k) {
    if (k > 0) {
      const float w = -kCurvF * start_field(G, c.p) * c.p[3];
      float st, ct, bz;
      sincos_small(c.p[5], st, ct);
      Prop pr;
      ok = path_to_surface(G, ss[k], c.p, w, st, ct, pr) && step_field(G, ss[k], c.p, st, ct, pr, bz);
      ok = ok && apply_propagation(G, M, ss[k], c.p, c.C, pr, st, ct, bz);
      if (!ok) break;
    }
    const float2 h = A.hits[ids[k]];
    c.chi2 += update_exact(G, ss[k], c, h.x, h.y);
  }
  // One predicate for "the finder takes it" and "its outputs are written here": a chi2 that is NaN (a hit
  // with a NaN coordinate) or negative (a covariance that lost its sign in FP32) marks no state.
  ok = ok && c.chi2 >= 0.f;
  // With an order to make: the class of a seed the finder will take (k_order_seeds reads it from
  // above the surface), counted per block and added once.
  int cls = -1;
  if (A.class_count) {
    __shared__ int hist[kClasses];
    if (threadIdx.x < kClasses) hist[threadIdx.x] = 0;
    __syncthreads();
    if (ok) {
      cls = seed_class(c.p[5]);
      atomicAdd(&hist[cls], 1);
    }
    __syncthreads();
    if (threadIdx.x < kClasses && hist[threadIdx.x] > 0) atomicAdd(A.class_count + threadIdx.x, hist[threadIdx.x]);
  }
  int mark = A.class_count ? cls + 1 : 0;
  if (A.front_list) {
    const bool front = ok && fabsf(kCurvF * G.bz * c.p[3]) * G.barrel_r[G.n_barrel - 1] > kCurling;
    const unsigned mask = __ballot_sync(kFull, front);
    if (mask) {
      const int lane = threadIdx.x & 31;
      int at = 0;
      if (lane == __ffs(mask) - 1) at = atomicAdd(A.front_count, __popc(mask));
      at = __shfl_sync(kFull, at, __ffs(mask) - 1) + __popc(mask & ((1u << lane) - 1u));
      if (front && at < n) A.front_list[at] = seed;
    }
    mark = (front ? 1 : 0) | (ok ? 0 : 2);  // passed over in index order
  }
  if (!in) return;
  // (a failed seed has no surface: 255, above every surface's number, so that nothing looks its hits up)
  if (FIND || ok) A.seed_surf[seed] = (ok ? ss[2] : 255) | (mark << 8);
  if constexpr (FIND) {
    float* out = A.seed_state + static_cast<size_t>(seed) * kSeedWords;
    if (ok) {
      const float v[kSeedWords] = {c.p[0], c.p[1], c.p[2], c.p[3], c.p[4], c.p[5], c.C[0], c.C[1], c.C[2], c.C[3],
                                   c.C[4], c.C[5], c.C[6], c.C[7], c.C[8], c.C[9], c.C[10], c.C[11], c.C[12], c.C[13],
                                   c.C[14], c.C[15], c.C[16], c.C[17], c.C[18], c.C[19], c.C[20], c.chi2};
#pragma unroll
      for (int i = 0; i < kSeedWords / 4; ++i)
        reinterpret_cast<float4*>(out)[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    } else {
      out[27] = -1.f;
    }
  } else {
    float* out = A.seed_state + seed;
    if (ok) {
#pragma unroll
      for (int i = 0; i < 6; ++i) out[static_cast<size_t>(i) * n] = c.p[i];
#pragma unroll
      for (int i = 0; i < 21; ++i) out[static_cast<size_t>(6 + i) * n] = c.C[i];
    }
    out[static_cast<size_t>(27) * n] = ok ? c.chi2 : -1.f;
  }
  if (FIND && !ok) {
    const float nanf_ = __int_as_float(0x7fc00000);
    for (int k = 0; k < A.lmax; ++k) A.hits_out[static_cast<size_t>(k) * n + seed] = -1;
    A.nhits_out[seed] = 0;
    A.chi2_out[seed] = nanf_;
    for (int i = 0; i < 6; ++i) A.state_out[static_cast<size_t>(i) * n + seed] = nanf_;
    for (int i = 0; i < 21; ++i) A.cov_out[static_cast<size_t>(i) * n + seed] = nanf_;
    A.status_out[seed] = removed ? 2 : 1;
  }
}

__global__ void k_clear_counters(int* counter, int n) {
  pdl_begin();
  if (static_cast<int>(threadIdx.x) < n) counter[threadIdx.x] = 0;
}

// The list of the seeds by class, from the classes and their counts; nearly in index order within a
// class (a block's seeds together). Leaves the surface alone in seed_surf.
constexpr int kOrderThreads = 512, kOrderSeeds = 4 * kOrderThreads;
__global__ void __launch_bounds__(kOrderThreads) k_order_seeds(FindArgs A, int* __restrict__ cursor, int* __restrict__ list,
                                                               int* __restrict__ live) {
  __shared__ int start[kClasses], hist[kClasses];
  const int n = A.n_seeds, t = threadIdx.x;
  if (t < 32) {
    const int count = t < kClasses ? A.class_count[t] : 0;
    int incl = count;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, o);
      if (t >= o) incl += v;
    }
    if (t < kClasses) {
      start[t] = incl - count;
      hist[t] = 0;
    }
    if (t == 31 && blockIdx.x == 0) *live = incl;
  }
  __syncthreads();
  int cls[4], at[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const long long seed = static_cast<long long>(blockIdx.x) * kOrderSeeds + u * kOrderThreads + t;
    cls[u] = -1;
    if (seed < n) {
      const int w = A.seed_surf[seed];
      A.seed_surf[seed] = w & 255;
      cls[u] = (w >> 8) - 1;
      if (cls[u] >= 0) at[u] = atomicAdd(&hist[cls[u]], 1);
    }
  }
  __syncthreads();
  if (t < kClasses && hist[t] > 0) start[t] += atomicAdd(cursor + t, hist[t]);
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    if (cls[u] < 0) continue;
    const int to = start[cls[u]] + at[u];
    if (to < n) list[to] = static_cast<int>(static_cast<long long>(blockIdx.x) * kOrderSeeds + u * kOrderThreads + t);
  }
}

// The learned instances' launch and occupancy come from find_learned.cu.
#define KF_LEARNED_INSTANCE(KC, FEAT)                                                                    \
  extern template int find_occupancy<KC, true, FEAT>(int, size_t, int*);                                 \
  extern template void find_launch_kernel<KC, true, FEAT>(const DevGeom&, const DevMat&, const FindArgs&, int, \
                                                          int, size_t, cudaStream_t);
KF_LEARNED_INSTANCE(1, 0) KF_LEARNED_INSTANCE(1, kFeatAll) KF_LEARNED_INSTANCE(2, 0) KF_LEARNED_INSTANCE(2, kFeatAll)
KF_LEARNED_INSTANCE(4, 0) KF_LEARNED_INSTANCE(4, kFeatAll) KF_LEARNED_INSTANCE(6, 0) KF_LEARNED_INSTANCE(6, kFeatAll)
KF_LEARNED_INSTANCE(8, 0) KF_LEARNED_INSTANCE(8, kFeatAll) KF_LEARNED_INSTANCE(16, 0) KF_LEARNED_INSTANCE(16, kFeatAll)
#undef KF_LEARNED_INSTANCE

// Compile-time choice of capacity, mode (plain or learned proposal) and instance (plain, one
// option alone, every option), dispatched from the runtime plan.
template <int KC, bool L, int FEAT>
struct FindKernel {
  static constexpr int kc = KC;
  static constexpr bool learned = L;
  static constexpr int feat = FEAT;
};

// The compiled instance that covers the options in use.
static int compiled_features(bool learned, int feat) {
  if (feat == 0) return 0;
  if (learned) return kFeatAll;
  return (feat == kFeatSteer || feat == kFeatMaterial || feat == kFeatField) ? feat : kFeatAll;
}

template <int KC, class F>
static int dispatch_mode(bool learned, int feat, F&& f) {
  if (learned) return feat == 0 ? f(FindKernel<KC, true, 0>{}) : f(FindKernel<KC, true, kFeatAll>{});
  if (feat == 0) return f(FindKernel<KC, false, 0>{});
  if (feat == kFeatSteer) return f(FindKernel<KC, false, kFeatSteer>{});
  if (feat == kFeatMaterial) return f(FindKernel<KC, false, kFeatMaterial>{});
  if (feat == kFeatField) return f(FindKernel<KC, false, kFeatField>{});
  return f(FindKernel<KC, false, kFeatAll>{});
}

template <class F>
static int dispatch_find(int kc, bool learned, int feat, F&& f) {
  switch (kc) {
    case 1: return dispatch_mode<1>(learned, feat, f);
    case 2: return dispatch_mode<2>(learned, feat, f);
    case 4: return dispatch_mode<4>(learned, feat, f);
    case 6: return dispatch_mode<6>(learned, feat, f);
    case 8: return dispatch_mode<8>(learned, feat, f);
    case 16: return dispatch_mode<16>(learned, feat, f);
    default: return KF_ERR_ARG;
  }
}

// ------------------------------------------------------------------------------------------------

static int pick_kc(int need) {
  static const int caps[] = {1, 2, 4, 6, 8, 16};
  for (int c : caps)
    if (c >= need) return c;
  return -1;
}

int plan_find(int n_seeds, const KfFindParams* p, int sms, int features, FindPlan* plan) {
  if (!p || n_seeds < 0 || sms <= 0) return KF_ERR_ARG;
  if (p->k_max < 1 || p->k_max > KF_MAX_K || p->max_miss < 0 || p->lmax < 4 || p->lmax > KF_MAX_LMAX) return KF_ERR_ARG;
  if (!(p->chi2_cut > 0.f)) return KF_ERR_ARG;
  const bool learned = p->mlp != nullptr && p->top_n > 0;
  if (p->top_n < 0 || p->top_n > KF_MAX_K) return KF_ERR_ARG;
  if (!(p->score_margin >= 0.f) || !(p->score_margin < 3.4e38f)) return KF_ERR_ARG;
  if (p->window_ranking != 0 && p->window_ranking != 1) return KF_ERR_ARG;
  if (p->block_threads != 0 && (p->block_threads < 32 || p->block_threads > 256 || p->block_threads % 32))
    return KF_ERR_ARG;
  if (p->blocks_per_sm < 0) return KF_ERR_ARG;
  if (learned && p->block_threads > kFindMaxBlockLearned) return KF_ERR_CAPACITY;
  if (p->k_capacity < 0 || p->k_capacity > KF_MAX_K) return KF_ERR_ARG;
  int kc = pick_kc(std::max(learned ? std::max(p->k_max, p->top_n) : p->k_max, p->k_capacity));
  if (kc < 0) return KF_ERR_ARG;
  // Adaptive capacity: a first pass at the smallest compiled capacity >= the requested one, when
  // that is below the full capacity (and, with the learned proposal, holds top_n).
  const int ac = p->adaptive_capacity;
  if (ac < 0 || ac > KF_MAX_K) return KF_ERR_ARG;
  int kc1 = ac > 0 ? pick_kc(ac) : 0;
  if (kc1 >= kc || (learned && p->top_n > kc1)) kc1 = 0;
  // Slots for every candidate that is kept are all that a pass needs: such a first pass is the only one
  // (and a detecting pass always has k_max above its slots).
  if (kc1 >= p->k_max) {
    kc = kc1;
    kc1 = 0;
  }
  // Resident blocks per SM for a block size (shared memory and registers), cached per (device,
  // capacity, mode, block size, lmax) so later calls, e.g. inside a stream capture, only launch.
  const int feat = compiled_features(learned, features);
  const int fi = feat == 0 ? 0 : feat == kFeatSteer ? 1 : feat == kFeatMaterial ? 2 : feat == kFeatField ? 3 : 4;
  static int occ_cache[16][6][2][5][8][32] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 16) return KF_ERR_ARG;
  auto occupancy = [&](int kcx, int blk, size_t* smem_out, int* occ_out) {
    const int ki = kcx == 1 ? 0 : kcx == 2 ? 1 : kcx == 4 ? 2 : kcx == 6 ? 3 : kcx == 8 ? 4 : 5;
    size_t sm = 0;
    dispatch_find(kcx, learned, feat, [&](auto k) {
      sm = block_smem_base<decltype(k)::kc, decltype(k)::learned>() +
           warp_smem_bytes<decltype(k)::kc, decltype(k)::learned>(p->lmax) * (blk / 32);
      return KF_OK;
    });
    *smem_out = sm;
    *occ_out = 0;
    if (sm > 227 * 1024) return KF_OK;
    int& cached = occ_cache[dev][ki][learned][fi][blk / 32 - 1][p->lmax];
    if (cached == 0) {
      int o = 0;
      const int rc = dispatch_find(kcx, learned, feat, [&](auto k) {
        return find_occupancy<decltype(k)::kc, decltype(k)::learned, decltype(k)::feat>(blk, sm, &o);
      });
      if (rc != KF_OK) return rc;
      cached = o > 0 ? o : -1;
    }
    *occ_out = cached > 0 ? cached : 0;
    return KF_OK;
  };
  // Block size (the caller's, or the one that keeps the most warps resident per SM), persistent
  // grid and shared memory of the instance with capacity kcx.
  auto choose = [&](int kcx, int* block_out, int* grid_out, size_t* smem_out) {
    int block = p->block_threads;
    size_t smem = 0;
    int occ = 0;
    if (block != 0) {
      const int rc = occupancy(kcx, block, &smem, &occ);
      if (rc != KF_OK) return rc;
    } else {
      int best_warps = 0;
      for (int blk = learned ? kFindMaxBlockLearned : 256; blk >= 64; blk -= 32) {
        size_t sm = 0;
        int o = 0;
        const int rc = occupancy(kcx, blk, &sm, &o);
        if (rc != KF_OK) return rc;
        if (o * blk / 32 > best_warps) {
          best_warps = o * blk / 32;
          block = blk;
          smem = sm;
          occ = o;
        }
      }
    }
    if (occ < 1) return KF_ERR_CAPACITY;
    int bps = p->blocks_per_sm;
    if (bps == 0 || bps > occ) bps = occ;
    const long long groups_per_block = static_cast<long long>(block / 32) * (32 / kcx);
    const long long want = (static_cast<long long>(n_seeds) + groups_per_block - 1) / groups_per_block;
    *block_out = block;
    *grid_out = static_cast<int>(std::max(1LL, std::min<long long>(static_cast<long long>(sms) * bps, want)));
    *smem_out = smem;
    return KF_OK;
  };
  int rc = choose(kc, &plan->block, &plan->grid, &plan->smem);
  if (rc != KF_OK) return rc;
  plan->kc1 = kc1;
  plan->block1 = plan->grid1 = 0;
  plan->smem1 = 0;
  if (kc1 > 0) {
    rc = choose(kc1, &plan->block1, &plan->grid1, &plan->smem1);
    if (rc != KF_OK) return rc;
  }
  plan->kc = kc;
  plan->learned = learned;
  plan->feat = feat;
  auto up = [](size_t v) { return (v + 255) / 256 * 256; };
  plan->off_state = 256;  // after the work counters
  plan->off_surf = up(plan->off_state + static_cast<size_t>(kSeedWords) * n_seeds * sizeof(float));
  plan->off_mlp = up(plan->off_surf + static_cast<size_t>(n_seeds) * sizeof(int));
  plan->ws_bytes = learned ? up(plan->off_mlp + static_cast<size_t>(kFragWords) * sizeof(uint4)) : plan->off_mlp;
  plan->off_ovf = 0;
  if (kc1 > 0) {
    plan->off_ovf = plan->ws_bytes;
    plan->ws_bytes = up(plan->off_ovf + static_cast<size_t>(n_seeds) * sizeof(int));
  }
  // The seed order's list comes last: a workspace without it (the fixed scratch) leaves the seeds
  // in index order.
  plan->need_bytes = plan->off_order = plan->ws_bytes;
  plan->ws_bytes = up(plan->off_order + static_cast<size_t>(n_seeds) * sizeof(int));
  return KF_OK;
}

int launch_seed_states(const DevGeom& G, const DevMat& M, const FindArgs& A, cudaStream_t stream) {
  launch_pdl(k_seed_states<false>, (A.n_seeds + 127) / 128, 128, 0, stream, G, M, A);
  return cudaGetLastError() == cudaSuccess ? KF_OK : KF_ERR_CUDA;
}

// ------------------------------------------------------------------------------------------------
// Scratch of the allocation-free entry point (kf_find_tracks_static): the work counter, the seed
// states for at most KF_STATIC_MAX_SEEDS seeds and the learned proposal's weight fragments,
// laid out as plan_find lays out a caller's workspace. A fixed array in the library: every GPU that loads the library holds it until the
// process exits. In host code g_find_scratch only names the array; its device address comes from
// cudaGetSymbolAddress, looked up once per device.
constexpr size_t static_scratch_bytes() {
  return (((256 + static_cast<size_t>(kSeedWords) * KF_STATIC_MAX_SEEDS * sizeof(float) + 255) / 256 * 256 +
           static_cast<size_t>(KF_STATIC_MAX_SEEDS) * sizeof(int) + 255) /
              256 * 256 +
          static_cast<size_t>(kFragWords) * sizeof(uint4) + 255) /
         256 * 256;
}
static_assert(static_scratch_bytes() == KF_STATIC_SCRATCH_BYTES, "header and library disagree on the scratch size");
static __device__ __align__(256) unsigned char g_find_scratch[static_scratch_bytes()];

int static_scratch(void** ptr) {
  static void* addr[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return KF_ERR_CUDA;
  if (addr[dev] == nullptr) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_find_scratch) != cudaSuccess || p == nullptr) return KF_ERR_CUDA;
    addr[dev] = p;
  }
  *ptr = addr[dev];
  return KF_OK;
}

int launch_find(const DevGeom& G, const DevMat& M, FindArgs& A, const FindPlan& plan, void* ws, size_t ws_bytes,
                cudaStream_t stream) {
  char* base = static_cast<char*>(ws);
  A.counter = reinterpret_cast<int*>(base);
  A.seed_state = reinterpret_cast<float*>(base + plan.off_state);
  A.seed_surf = reinterpret_cast<int*>(base + plan.off_surf);
  A.mlp_frag = nullptr;
  if (plan.learned) {
    uint4* frag = reinterpret_cast<uint4*>(base + plan.off_mlp);
    if (launch_mlp_fragments(A.mlp, frag, stream) != 0) return KF_ERR_CUDA;
    A.mlp_frag = frag;
  }
  // Work counters: [0] the (first) pass's seed queue, [1] the second pass's, [2] the overflow count,
  // [3] the number of seeds in the ordered list, [4] in the front list, [8 ...] the classes' counts, [32 ...]
  // their cursors. (A kernel clears them because a memset would not start under the kernel before.)
  constexpr int kCounters = 56;
  static_assert(kMaxSurf <= 255, "surface numbers share a word with a mark");
  static_assert(8 + kClasses <= 32 && 32 + kClasses <= kCounters && kCounters * sizeof(int) <= 256, "counter area");
  const bool disks = G.n_dpos + G.n_dneg > 0, room = ws_bytes >= plan.ws_bytes, ordered = disks && room;
  int* list = reinterpret_cast<int*>(base + plan.off_order);
  A.front_list = !disks && room ? list : nullptr;
  A.front_count = A.counter + 4;
  launch_pdl(k_clear_counters, 1, 64, 0, stream, A.counter, kCounters);
  A.detect = 0;
  A.ovf_list = A.ovf_count = nullptr;
  A.seed_list = A.seed_list_count = nullptr;
  A.class_count = ordered ? A.counter + 8 : nullptr;
  launch_pdl(k_seed_states<true>, (A.n_seeds + 127) / 128, 128, 0, stream, G, M, A);
  if (ordered) {
    k_order_seeds<<<static_cast<int>((static_cast<long long>(A.n_seeds) + kOrderSeeds - 1) / kOrderSeeds), kOrderThreads,
                    0, stream>>>(A, A.counter + 32, list, A.counter + 3);
    A.seed_list = list;
    A.seed_list_count = A.counter + 3;
  }
  if (plan.kc1 > 0) {
    // First pass at the smaller capacity; its overflowing seeds go to the second pass.
    FindArgs A1 = A;
    A1.detect = 1;
    A1.ovf_list = reinterpret_cast<int*>(base + plan.off_ovf);
    A1.ovf_count = A.counter + 2;
    dispatch_find(plan.kc1, plan.learned, plan.feat, [&](auto k) {
      find_launch_kernel<decltype(k)::kc, decltype(k)::learned, decltype(k)::feat>(G, M, A1, plan.grid1, plan.block1,
                                                                                  plan.smem1, stream);
      return KF_OK;
    });
    A.counter = A.counter + 1;
    A.seed_list = A1.ovf_list;
    A.seed_list_count = A1.ovf_count;
  }
  dispatch_find(plan.kc, plan.learned, plan.feat, [&](auto k) {
    find_launch_kernel<decltype(k)::kc, decltype(k)::learned, decltype(k)::feat>(G, M, A, plan.grid, plan.block,
                                                                                plan.smem, stream);
    return KF_OK;
  });
  return cudaGetLastError() == cudaSuccess ? KF_OK : KF_ERR_CUDA;
}

}  // namespace kfgb
