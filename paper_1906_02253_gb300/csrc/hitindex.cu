// Hit index build: per (event, surface) slab, a counting sort of the hits by bin
// (phi-bin * n_2nd + second-bin), ordered within a bin by (phi sub-bin, hit id). This is the binned
// hit structure behind the per-layer search windows (paper Sec. 3.1) and the reuse of hit data by
// nearby seeds (Sec. 3.2).
//
// One CTA per slab, everything staged in shared memory: the bin (u16) and phi sub-bin (u8) of each
// hit, the bin histogram and its exclusive scan, then an unstable scatter of local hit numbers by
// shared atomics. Each bin's sub-bin counts give its sub-bin offsets; the output pass puts the hit
// at unstable position p of bin [s, e) at s + its rank by (sub-bin, id) among the bin's hits (bins
// hold a handful of hits) and writes the sorted hits, ids and, when asked for, each hit's 16-byte
// search record (cos phi, sin phi, second coordinate, id), so that the search reads one aligned
// record per hit and computes residual angles without trig. The ranks replace a per-bin insertion
// sort, which took 43% of the kernel (one lane per bin, dependent shared loads, lanes diverging
// with the bin sizes).
// Global traffic per hit: one 8-byte read (plus an L2 re-read in the output pass) and a 12-byte
// write (28 bytes with search records).
#include "kf_math.cuh"
#include "pdl.cuh"

namespace kfgb {

static_assert(kPhiSub == 8, "sub-bin offsets are written as eight 16-bit counts");

__global__ void __launch_bounds__(1024, 2) k_build_hit_index(DevGeom G, const float2* __restrict__ hits,
                                                         const int* __restrict__ slab_off, int n_slabs,
                                                         int cap, int* __restrict__ bin_off,
                                                         float2* __restrict__ sorted_hits,
                                                         int* __restrict__ sorted_ids, float4* __restrict__ sorted_rec,
                                                         uint4* __restrict__ sub_off, int* __restrict__ d_status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_begin();
  const int nb = G.n_bins;
  int* hist = reinterpret_cast<int*>(smem_raw);                       // [nb + 1]
  unsigned short* bin = reinterpret_cast<unsigned short*>(hist + nb + 1);  // [cap]
  unsigned short* order = bin + cap;                                  // [cap]
  unsigned char* sub = reinterpret_cast<unsigned char*>(order + cap);  // [cap]
  __shared__ int warp_sums[32];

  for (int sl = blockIdx.x; sl < n_slabs; sl += gridDim.x) {
    const int si = sl % G.n_surf;
    const int h0 = slab_off[sl];
    const int n = slab_off[sl + 1] - h0;
    int* out = bin_off + static_cast<size_t>(sl) * (nb + 1);
    uint4* sout = sub_off ? sub_off + static_cast<size_t>(sl) * nb : nullptr;
    if (n > cap || n < 0) {
      for (int b = threadIdx.x; b <= nb; b += blockDim.x) out[b] = h0;
      if (sout)
        for (int b = threadIdx.x; b < nb; b += blockDim.x) sout[b] = make_uint4(0u, 0u, 0u, 0u);
      if (threadIdx.x == 0 && d_status) atomicOr(d_status, 1);
      __syncthreads();
      continue;
    }
    const int nbs = G.n_phi[si] * G.n_2nd[si];
    const int n2 = G.n_2nd[si];
    for (int b = threadIdx.x; b <= nb; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    // Four hits per thread per iteration, their loads issued together.
    for (int i0 = threadIdx.x; i0 < n; i0 += 4 * blockDim.x) {
      float2 hv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * blockDim.x;
        hv[u] = i < n ? __ldg(hits + h0 + i) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * blockDim.x;
        if (i < n) {
          const int pb = phi_bin(G, si, hv[u].x);
          const int b = pb * n2 + second_bin(G, si, hv[u].y);
          bin[i] = static_cast<unsigned short>(b);
          sub[i] = static_cast<unsigned char>(sub_of(phi_fine(G, si, hv[u].x), pb));
          atomicAdd(&hist[b], 1);
        }
      }
    }
    __syncthreads();
    // Exclusive scan of hist[0, nbs) in place: each thread scans a contiguous chunk.
    const int per = (nbs + blockDim.x - 1) / blockDim.x;
    const int b0 = min(nbs, static_cast<int>(threadIdx.x) * per), b1 = min(nbs, b0 + per);
    int local = 0;
    for (int b = b0; b < b1; ++b) local += hist[b];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) warp_sums[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      const int nw = blockDim.x >> 5;
      int v = lane < nw ? warp_sums[lane] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
      }
      if (lane < nw) warp_sums[lane] = v;  // inclusive over warps
    }
    __syncthreads();
    int run = incl - local + (wid > 0 ? warp_sums[wid - 1] : 0);
    for (int b = b0; b < b1; ++b) {
      const int c = hist[b];
      hist[b] = run;
      run += c;
    }
    __syncthreads();
    for (int b = threadIdx.x; b <= nb; b += blockDim.x) out[b] = h0 + (b < nbs ? hist[b] : n);
    __syncthreads();
    // Unstable scatter: hist[b] becomes the end of bin b.
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const int pos = atomicAdd(&hist[bin[i]], 1);
      order[pos] = static_cast<unsigned short>(i);
    }
    __syncthreads();
    // Sub-bin offsets of each bin (hit counts of its sub-bins, cumulated).
    if (sout) {
      for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        unsigned long long c03 = 0, c47 = 0;  // 16-bit hit counts of sub-bins 0-3 and 4-7
        if (b < nbs) {
          const int e = hist[b];
          const int s = b > 0 ? hist[b - 1] : 0;
          for (int i = s; i < e; ++i) {
            const unsigned sv = sub[order[i]];
            const unsigned long long inc = 1ull << (16 * (sv & 3));
            if (sv < 4) c03 += inc;
            else c47 += inc;
          }
        }
        unsigned cum[kPhiSub];
        unsigned run = 0;
#pragma unroll
        for (int j = 0; j < kPhiSub; ++j) {
          run += static_cast<unsigned>(((j < 4 ? c03 : c47) >> (16 * (j & 3))) & 0xffffull);
          cum[j] = run;
        }
        sout[b] = make_uint4(cum[0] | (cum[1] << 16), cum[2] | (cum[3] << 16), cum[4] | (cum[5] << 16),
                             cum[6] | (cum[7] << 16));
      }
    }
    // Gather: the hit at (unstable) position p of bin [s, e) goes to s + its rank by (sub-bin, id)
    // among the bin's hits; four per thread per iteration with their loads issued together.
    for (int p0 = threadIdx.x; p0 < n; p0 += 4 * blockDim.x) {
      int iv[4], dv[4];
      float2 hv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int p = p0 + u * blockDim.x;
        iv[u] = 0;
        dv[u] = 0;
        if (p < n) {
          const int v = order[p];
          const int b = bin[v];
          const int s = b > 0 ? hist[b - 1] : 0, e = hist[b];
          const unsigned kv = (static_cast<unsigned>(sub[v]) << 16) | static_cast<unsigned>(v);
          int rank = 0;
          for (int q = s; q < e; ++q) {
            const unsigned w = order[q];
            rank += ((static_cast<unsigned>(sub[w]) << 16) | w) < kv;
          }
          iv[u] = v;
          dv[u] = s + rank;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) hv[u] = p0 + u * static_cast<int>(blockDim.x) < n ? __ldg(hits + h0 + iv[u]) : make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int p = p0 + u * blockDim.x;
        if (p < n) {
          const int d = h0 + dv[u];
          sorted_hits[d] = hv[u];
          sorted_ids[d] = h0 + iv[u];
          if (sorted_rec) {
            float s, c;
            sincosf(hv[u].x, &s, &c);
            sorted_rec[d] = make_float4(c, s, hv[u].y, __int_as_float(h0 + iv[u]));
          }
        }
      }
    }
    __syncthreads();
  }
}

// The same index by fine bins (bin * kPhiSub + sub-bin), for surfaces of up to kFineMaxBins bins: the
// histogram counts fine bins (two 16-bit counters a word), so its scan yields the sub-bin offsets
// and the bin offsets at once, a hit's rank is searched only among the hits of its own fine bin
// (0.2 to 1.2 on average here, 2 to 10 in its bin), and a hit keeps one 16-bit word instead of a
// bin and a sub-bin. 200 barrel + disk events (28.6 M hits, 7,000 slabs) take 434 us against 466 us
// with bins and sub-bins apart, the search records 55 us of it; issue and latency bound (a slab is a
// chain of eight block barriers). 512 or 768 threads a block are 2-3% slower, as the largest slab's
// shared memory keeps it at two blocks per SM.
// 16-bit fields of x added up within the word pair by pair: (lo, lo + hi), plus c in both fields.
__device__ __forceinline__ unsigned cumulate(unsigned x, unsigned c) { return x + (x << 16) + c * 0x10001u; }

__global__ void __launch_bounds__(1024, 2)
    k_build_hit_index_fine(const __grid_constant__ DevGeom G, const float2* __restrict__ hits,
                           const int* __restrict__ slab_off, int n_slabs, int cap, int* __restrict__ bin_off,
                           float2* __restrict__ sorted_hits, int* __restrict__ sorted_ids, float4* __restrict__ sorted_rec,
                           uint4* __restrict__ sub_off, int* __restrict__ d_status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_begin();
  const int nb = G.n_bins;
  uint4* hist4 = reinterpret_cast<uint4*>(smem_raw);  // [nb]: the eight counters of each bin
  unsigned* hist = reinterpret_cast<unsigned*>(smem_raw);
  const unsigned short* hist16 = reinterpret_cast<const unsigned short*>(smem_raw);
  unsigned short* fine = reinterpret_cast<unsigned short*>(hist4 + nb);  // [cap]: fine bin of each hit
  unsigned short* order = fine + cap;                                    // [cap]: hits by fine bin
  __shared__ int warp_sums[32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;

  for (int sl = blockIdx.x; sl < n_slabs; sl += gridDim.x) {
    const int si = sl % G.n_surf;
    const int h0 = slab_off[sl];
    const int n = slab_off[sl + 1] - h0;
    int* out = bin_off + static_cast<size_t>(sl) * (nb + 1);
    uint4* sout = sub_off ? sub_off + static_cast<size_t>(sl) * nb : nullptr;
    if (n > cap || n < 0) {
      for (int b = tid; b <= nb; b += blockDim.x) out[b] = h0;
      if (sout)
        for (int b = tid; b < nb; b += blockDim.x) sout[b] = make_uint4(0u, 0u, 0u, 0u);
      if (tid == 0 && d_status) atomicOr(d_status, 1);
      continue;
    }
    const int n2 = G.n_2nd[si];
    for (int b = tid; b < nb; b += blockDim.x) hist4[b] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    // Four hits per thread per iteration, their loads issued together.
    for (int i0 = tid; i0 < n; i0 += 4 * blockDim.x) {
      float2 hv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * blockDim.x;
        hv[u] = i < n ? __ldg(hits + h0 + i) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * blockDim.x;
        if (i < n) {
          const int pb = phi_bin(G, si, hv[u].x);
          const int f = (pb * n2 + second_bin(G, si, hv[u].y)) * kPhiSub + sub_of(phi_fine(G, si, hv[u].x), pb);
          fine[i] = static_cast<unsigned short>(f);
          atomicAdd(&hist[f >> 1], 1u << (16 * (f & 1)));
        }
      }
    }
    __syncthreads();
    // Scan: warp w takes the bins [w per, (w + 1) per), 32 at a time.
    const int per = (nb + 32 * nw - 1) / (32 * nw) * 32, b0 = min(nb, wid * per), b1 = min(nb, b0 + per);
    int sum = 0;
    for (int b = b0 + lane; b < b1; b += 32) {
      const uint4 c = hist4[b];
      const unsigned t = (c.x + c.y) + (c.z + c.w);  // (a bin holds at most 32768 hits: no field carries over)
      sum += static_cast<int>((t & 0xffffu) + (t >> 16));
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) warp_sums[wid] = sum;
    __syncthreads();
    int base = 0;  // hits before this warp's bins
    {
      int v = lane < nw && lane < wid ? warp_sums[lane] : 0;
      base = __reduce_add_sync(0xffffffffu, v);
    }
    for (int bb = b0; bb < b1; bb += 32) {
      const int b = bb + lane;
      const uint4 c = b < b1 ? hist4[b] : make_uint4(0u, 0u, 0u, 0u);
      uint4 in;  // inclusive counts of the bin's sub-bins
      in.x = cumulate(c.x, 0u);
      in.y = cumulate(c.y, in.x >> 16);
      in.z = cumulate(c.z, in.y >> 16);
      in.w = cumulate(c.w, in.z >> 16);
      const int count = static_cast<int>(in.w >> 16);
      int incl = count;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      if (b < b1) {
        const int start = base + incl - count;
        const unsigned s2 = static_cast<unsigned>(start) * 0x10001u;
        hist4[b] = make_uint4(in.x - c.x + s2, in.y - c.y + s2, in.z - c.z + s2, in.w - c.w + s2);
        out[b] = h0 + start;
        if (sout) sout[b] = in;
      }
      base += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (tid == 0) out[nb] = h0 + n;
    __syncthreads();
    // Unstable scatter: a fine bin's counter becomes its end.
    for (int i = tid; i < n; i += blockDim.x) {
      const int f = fine[i], sh = 16 * (f & 1);
      order[(atomicAdd(&hist[f >> 1], 1u << sh) >> sh) & 0xffffu] = static_cast<unsigned short>(i);
    }
    __syncthreads();
    // Gather: the hit at (unstable) position p of its fine bin [s, e) goes to s + its rank by id; four
    // per thread per iteration with their loads issued together.
    for (int p0 = tid; p0 < n; p0 += 4 * blockDim.x) {
      int iv[4], dv[4];
      float2 hv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int p = p0 + u * blockDim.x;
        iv[u] = 0;
        dv[u] = 0;
        if (p < n) {
          const int v = order[p], f = fine[v];
          const int s = f > 0 ? hist16[f - 1] : 0, e = hist16[f];
          int d = p;
          if (e - s > 1) {
            d = s;
            for (int q = s; q < e; ++q) d += order[q] < v;
          }
          iv[u] = v;
          dv[u] = d;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        hv[u] = p0 + u * static_cast<int>(blockDim.x) < n ? __ldg(hits + h0 + iv[u]) : make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int p = p0 + u * blockDim.x;
        if (p < n) {
          const int d = h0 + dv[u];
          sorted_hits[d] = hv[u];
          sorted_ids[d] = h0 + iv[u];
          if (sorted_rec) {
            float sn, cs;
            sincosf(hv[u].x, &sn, &cs);
            sorted_rec[d] = make_float4(cs, sn, hv[u].y, __int_as_float(h0 + iv[u]));
          }
        }
      }
    }
    __syncthreads();
  }
}

}  // namespace kfgb
