// IP pair scanning (Algorithm 2, Sec. 4.1) for one or many routers in one launch.
//
// Each thread takes 16-byte vectors of the pair stream (two packets per
// vector), hashes both addresses with the simple-tabulation tables held in
// shared memory, and sets the r recorders RSEA[i, RHFG[i](cip)][H1(oip)] to 0,
// which for the library's stamp recorders is a store of the sketch's clock.
// Setting a recorder to 0 is idempotent and order-free (Sec. 4.1), so the
// stores need no atomics and no ordering between threads.
#include "ssd_internal.cuh"

namespace ssd {
namespace {

// Algorithm 2 for one pair: DRidx = H1(oip); RHFG[0](cip) from the second table
// set; RHFG[i](cip) = ((cip >> (i-1)*delta) ^ RHFG[0](cip)) mod 2^q for i >= 1.
// The recorders take distance 0: the stamp `now` (the sketch's clock).
__device__ __forceinline__ void scan_pair(uint16_t* __restrict__ dr, uint16_t now, uint32_t cip, uint32_t oip,
                                          const uint32_t* sT, const Dims& d) {
  const uint32_t j = tab_hash(sT, oip) & (d.eta - 1u);
  const uint32_t c0 = tab_hash(sT + 1024, cip) & d.col_mask;
  if (in_bounds(d, j < d.eta && c0 < (1u << d.q))) dr[((uint64_t)c0 << d.log2_eta) | j] = now;
#pragma unroll
  for (uint32_t i = 1; i < SSD_MAX_R; ++i) {
    if (i < d.r) {
      const uint32_t sh = (i - 1u) * d.delta + d.sh0;
      const uint32_t w = sh < 32u ? (cip >> sh) : 0u;
      const uint32_t col = (w ^ c0) & d.col_mask;
      if (in_bounds(d, col < (1u << d.q))) dr[((((uint64_t)i << d.q) | col) << d.log2_eta) | j] = now;
    }
  }
}

// scan_pair on the stored pair (x, y) through a job's view (side and group).
__device__ __forceinline__ void scan_view(uint16_t* __restrict__ dr, uint16_t now, uint32_t view, uint32_t x,
                                          uint32_t y, const uint32_t* sT, const Dims& d) {
  uint32_t cip, oip;
  if (view_pair(view, x, y, cip, oip)) scan_pair(dr, now, cip, oip, sT, d);
}

// touch_pair on the stored pair (x, y) through a job's view; every lane makes the
// call (a pair outside the view's group takes part as a no-op).
template <int CM>
__device__ __forceinline__ void touch_view(uint32_t* bits, uint64_t jbase, uint32_t view, uint32_t x, uint32_t y,
                                           bool live, const uint32_t* sT, const Dims& d, uint32_t r0, uint32_t r1,
                                           uint64_t se0, uint64_t count) {
  uint32_t cip, oip;
  const bool in = view_pair(view, x, y, cip, oip);
  touch_pair<CM>(bits, jbase, cip, oip, live && in, sT, d, r0, r1, se0, count);
}

__device__ __forceinline__ int find_router(const ScanBatch& b, uint64_t v) {
  int lo = 0, hi = b.n - 1;
  while (lo < hi) {  // last j with prefix[j] <= v
    const int mid = (lo + hi + 1) >> 1;
    if (b.prefix[mid] <= v) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// U: 16-byte pair vectors each thread loads before it hashes any of them.
template <int U>
__global__ void __launch_bounds__(kBlock) k_scan(const Dims d, const uint32_t* __restrict__ tables,
                                                 const __grid_constant__ ScanBatch b) {
  __shared__ uint32_t sT[2048];
  __shared__ uint16_t sNow[kMaxBatch];   // each job's stamp: its sketch's clock
  for (int i = threadIdx.x; i < 2048; i += blockDim.x) sT[i] = tables[i];
  if (threadIdx.x < b.n) sNow[threadIdx.x] = (uint16_t)read_tm(b.tm[threadIdx.x]);
  __syncthreads();

  // packets outside the 16-byte aligned bodies: a head when a buffer starts at
  // 8 mod 16, a tail when the body leaves one packet over
  if (blockIdx.x == 0 && threadIdx.x < 2 * b.n) {
    const uint32_t* e = b.edge[threadIdx.x];
    const int j = threadIdx.x >> 1;
    if (e) scan_view(b.dr[j], sNow[j], b.view[j], e[0], e[1], sT, d);
  }

  const uint64_t total = b.prefix[b.n];
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b.n == 1) {
    const uint4* __restrict__ vec = b.vec[0];
    uint16_t* __restrict__ dr = b.dr[0];
    const uint32_t view = b.view[0];
    const uint16_t now = sNow[0];
    for (; v + (U - 1) * stride < total; v += U * stride) {
      uint4 w[U];
#pragma unroll
      for (int u = 0; u < U; ++u) w[u] = __ldcs(vec + v + u * stride);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        scan_view(dr, now, view, w[u].x, w[u].y, sT, d);
        scan_view(dr, now, view, w[u].z, w[u].w, sT, d);
      }
    }
    for (; v < total; v += stride) {
      const uint4 w = __ldcs(vec + v);
      scan_view(dr, now, view, w.x, w.y, sT, d);
      scan_view(dr, now, view, w.z, w.w, sT, d);
    }
  } else {
    for (; v + (U - 1) * stride < total; v += U * stride) {
      uint4 w[U];
      int jj[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t vv = v + u * stride;
        const int j = find_router(b, vv);
        w[u] = __ldcs(b.vec[j] + (vv - b.prefix[j]));
        jj[u] = j;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = jj[u];
        scan_view(b.dr[j], sNow[j], b.view[j], w[u].x, w[u].y, sT, d);
        scan_view(b.dr[j], sNow[j], b.view[j], w[u].z, w[u].w, sT, d);
      }
    }
    for (; v < total; v += stride) {
      const int j = find_router(b, v);
      const uint4 w = __ldcs(b.vec[j] + (v - b.prefix[j]));
      scan_view(b.dr[j], sNow[j], b.view[j], w.x, w.y, sT, d);
      scan_view(b.dr[j], sNow[j], b.view[j], w.z, w.w, sT, d);
    }
  }
}

// Clears the counters of the slot whose first launch this is (only later launches use them): one operation
// less in the chain of a small slot. Called by block 0 of the launch.
__device__ __forceinline__ void clear_counters(DevCounters* c) {
  if (c && threadIdx.x < sizeof(DevCounters) / 4) reinterpret_cast<uint32_t*>(c)[threadIdx.x] = 0;
}
static_assert(sizeof(DevCounters) / 4 <= kBlock, "clear_counters");

// The touch kernels walk the vectors warp by warp (vb = the warp's first
// vector, a multiple of 32 because the grid stride is): every lane of a warp
// runs the same iterations, as set_touch<1> needs; a lane past the end only
// takes part.
template <int U, int CM>
__global__ void __launch_bounds__(kBlock) k_touch(const Dims d, const uint32_t* __restrict__ tables,
                                                  const __grid_constant__ ScanBatch b, uint32_t* __restrict__ bits,
                                                  uint64_t se0, uint64_t count, DevCounters* clear) {
  __shared__ uint32_t sT[2048];
  if (blockIdx.x == 0) clear_counters(clear);
  for (int i = threadIdx.x; i < 2048; i += blockDim.x) sT[i] = tables[i];
  __syncthreads();
  const uint32_t r0 = (uint32_t)(se0 >> d.q), r1 = (uint32_t)((se0 + count - 1) >> d.q);
  const uint32_t lane = threadIdx.x & 31u;
  if (blockIdx.x == 0 && threadIdx.x < 2 * b.n) {
    const uint32_t* e = b.edge[threadIdx.x];
    if (e)
      touch_view<0>(bits, (uint64_t)(threadIdx.x >> 1) * count, b.view[threadIdx.x >> 1], e[0], e[1], true, sT, d, r0,
                    r1, se0, count);
  }
  const uint64_t total = b.prefix[b.n];
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  uint64_t vb = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
  for (; vb + 31 + (U - 1) * stride < total; vb += U * stride) {
    uint4 w[U];
    uint64_t jb[U];
    uint32_t vw[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint64_t vv = vb + lane + u * stride;
      const int j = b.n == 1 ? 0 : find_router(b, vv);
      w[u] = __ldcs(b.vec[j] + (vv - b.prefix[j]));
      jb[u] = (uint64_t)j * count;
      vw[u] = b.view[j];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      touch_view<CM>(bits, jb[u], vw[u], w[u].x, w[u].y, true, sT, d, r0, r1, se0, count);
      touch_view<CM>(bits, jb[u], vw[u], w[u].z, w[u].w, true, sT, d, r0, r1, se0, count);
    }
  }
  for (; vb < total; vb += stride) {
    const uint64_t v = vb + lane;
    const bool live = v < total;
    uint4 w = make_uint4(0, 0, 0, 0);
    uint64_t jb = 0;
    uint32_t vw = 0;
    if (live) {
      const int j = b.n == 1 ? 0 : find_router(b, v);
      w = __ldcs(b.vec[j] + (v - b.prefix[j]));
      jb = (uint64_t)j * count;
      vw = b.view[j];
    }
    touch_view<CM>(bits, jb, vw, w.x, w.y, live, sT, d, r0, r1, se0, count);
    touch_view<CM>(bits, jb, vw, w.z, w.w, live, sT, d, r0, r1, se0, count);
  }
}

// Both hashes of every pair once per slot: packed = RHFG[0](cip) | H1(oip) << q.
__global__ void __launch_bounds__(kBlock) k_prehash(const Dims d, const uint32_t* __restrict__ tables,
                                                    const __grid_constant__ ScanBatch b, uint2* __restrict__ out) {
  __shared__ uint32_t sT[2048];
  for (int i = threadIdx.x; i < 2048; i += blockDim.x) sT[i] = tables[i];
  __syncthreads();
  const uint64_t nvec = b.prefix[1];
  const uint32_t view = b.view[0];
  auto pack = [&](uint32_t x, uint32_t y) {
    uint32_t cip, oip;
    view_pair(view, x, y, cip, oip);   // the side only: grouped views are not pre-hashed
    return make_uint2(cip, (tab_hash(sT + 1024, cip) & d.col_mask) | ((tab_hash(sT, oip) & (d.eta - 1u)) << d.q));
  };
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < nvec; v += stride) {
    const uint4 w = __ldcs(b.vec[0] + v);
    const uint2 p0 = pack(w.x, w.y), p1 = pack(w.z, w.w);
    reinterpret_cast<uint4*>(out)[v] = make_uint4(p0.x, p0.y, p1.x, p1.y);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    uint64_t at = 2 * nvec;
    for (int k = 0; k < 2; ++k) {
      const uint32_t* e = b.edge[k];
      if (e) out[at++] = pack(e[0], e[1]);
    }
  }
}

template <int U, int CM>
__global__ void __launch_bounds__(kBlock) k_touch_packed(const Dims d, const uint4* __restrict__ vec, uint64_t nvec,
                                                         const uint2* __restrict__ tail, uint32_t* __restrict__ bits,
                                                         uint64_t se0, uint64_t count) {
  const uint32_t r0 = (uint32_t)(se0 >> d.q), r1 = (uint32_t)((se0 + count - 1) >> d.q);
  const uint32_t lane = threadIdx.x & 31u;
  if (blockIdx.x == 0 && threadIdx.x == 0 && tail) touch_packed<0>(bits, tail->x, tail->y, true, d, r0, r1, se0, count);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  uint64_t vb = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u);  // as in k_touch
  for (; vb + 31 + (U - 1) * stride < nvec; vb += U * stride) {
    uint4 w[U];
#pragma unroll
    for (int u = 0; u < U; ++u) w[u] = __ldcs(vec + vb + lane + u * stride);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      touch_packed<CM>(bits, w[u].x, w[u].y, true, d, r0, r1, se0, count);
      touch_packed<CM>(bits, w[u].z, w[u].w, true, d, r0, r1, se0, count);
    }
  }
  for (; vb < nvec; vb += stride) {
    const bool live = vb + lane < nvec;
    const uint4 w = live ? __ldcs(vec + vb + lane) : make_uint4(0, 0, 0, 0);
    touch_packed<CM>(bits, w.x, w.y, live, d, r0, r1, se0, count);
    touch_packed<CM>(bits, w.z, w.w, live, d, r0, r1, se0, count);
  }
}

// Per-chunk touch lists of one router (see ListArgs). Each block owns a contiguous range of the pair vectors,
// each of its warps a fixed share. The first walk counts the warp's touches per chunk, one atomic per
// chunk then reserves the block's run in each list, and the second walk hashes the pairs, sets
// chunk 0's bits and writes the other bit indices into the reserved runs. Lane c of a warp keeps chunk c's count,
// then its place in the list: a touch's rank within the warp comes from a ballot, one per chunk of a row
// (two at the core-link size), so nothing is counted in shared memory (grouping the lanes by chunk
// with __match_any_sync and shared atomics took 167 us for 6.25 M pairs, this 111 us). Where a chunk holds
// whole rows every counted pair has one touch in each and the first walk reads nothing (or, for an IP
// group's view, the pairs alone); with a single chunk there is no list and no first walk. Every lane of a warp
// runs the same iterations.
// SUB: the chunks of a row are 2^SUB (0: whole rows per chunk), or any number for -1.
template <int CM, int SUB>
__global__ void __launch_bounds__(kBlock, 4) k_lists(const Dims d, const uint32_t* __restrict__ tables,
                                                  const __grid_constant__ ScanBatch b, const ListArgs a) {
  constexpr int kWarps = kBlock / 32;
  __shared__ uint32_t sT[2048];
  __shared__ uint32_t s_cnt[kWarps][kMaxChunks];
  for (int i = threadIdx.x; i < 2048; i += blockDim.x) sT[i] = tables[i];
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  // chunk of (row, col): whole rows (row >> row_shift) or 2^sub of them per row (col >> log2_count)
  constexpr bool rows = SUB == 0;
  const uint32_t row_shift = rows ? a.log2_count - d.q : 0u, sub = SUB >= 0 ? (uint32_t)SUB : d.q - a.log2_count;
  const uint32_t in_chunk = (1u << a.log2_count) - 1u;   // estimator within its chunk
  const uint64_t total = b.prefix[1];
  uint64_t per = (total + gridDim.x - 1) / gridDim.x;
  per = (per + 31) & ~31ull;
  const uint64_t v0 = (uint64_t)blockIdx.x * per;
  const uint64_t v1 = v0 + per < total ? v0 + per : total;
  const uint32_t view = b.view[0];
  const bool group = ((view >> 1) & 31u) != 0u;
  const uint4* const vec = b.vec[0];

  auto column = [&](uint32_t i, uint32_t cip, uint32_t c0) {
    const uint32_t sh = i ? (i - 1u) * d.delta + d.sh0 : 32u;
    return ((sh < 32u ? (cip >> sh) : 0u) ^ c0) & d.col_mask;
  };
  // f(x, y, live) for every pair of the warp's share, in the same order each time
  auto walk = [&](auto f) {
    constexpr int U = 2;   // vectors in flight
    for (uint64_t vb = v0 + wid * 32; vb < v1; vb += U * kBlock) {
      uint4 w[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        w[u] = vb + u * kBlock + lane < v1 ? __ldcg(vec + vb + u * kBlock + lane) : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (vb + u * kBlock >= v1) break;   // warp-uniform
        const bool live = vb + u * kBlock + lane < v1;
        f(w[u].x, w[u].y, live);
        f(w[u].z, w[u].w, live);
      }
    }
    if (blockIdx.x == 0 && wid == 0) {   // the packets outside the 16-byte body
      const uint32_t* e = lane < 2u ? b.edge[lane] : nullptr;
      f(e ? e[0] : 0u, e ? e[1] : 0u, e != nullptr);
    }
  };

  uint32_t mine = 0;   // lane c: this warp's touches of chunk c, then its next place in the list
  if (a.n_chunks > 1) {
    if (rows) {
      uint32_t pairs = 0;
      if (group) {
        walk([&](uint32_t x, uint32_t y, bool live) {
          uint32_t cip, oip;
          const bool in = view_pair(view, x, y, cip, oip) && live;
          pairs += __popc(__ballot_sync(0xFFFFFFFFu, in));
        });
      } else {
        for (uint64_t vb = v0 + wid * 32; vb < v1; vb += kBlock)
          pairs += 2u * (uint32_t)(v1 - vb < 32u ? v1 - vb : 32u);
        if (blockIdx.x == 0 && wid == 0) pairs += (b.edge[0] != nullptr) + (b.edge[1] != nullptr);
      }
      for (uint32_t i = 0; i < d.r; ++i) mine += (i >> row_shift) == lane ? pairs : 0u;
    } else {
      walk([&](uint32_t x, uint32_t y, bool live) {
        uint32_t cip, oip;
        const bool in = view_pair(view, x, y, cip, oip) && live;
        const uint32_t c0 = tab_hash(sT + 1024, cip) & d.col_mask;
        const uint32_t n_in = __popc(__ballot_sync(0xFFFFFFFFu, in));
#pragma unroll
        for (uint32_t i = 0; i < SSD_MAX_R; ++i) {
          if (i < d.r) {
            const uint32_t c = column(i, cip, c0) >> a.log2_count;
            if (SUB == 1) {
              const uint32_t n1 = __popc(__ballot_sync(0xFFFFFFFFu, in && c));
              mine += lane == 2u * i ? n_in - n1 : lane == 2u * i + 1u ? n1 : 0u;
            } else {
              for (uint32_t k = 0; k < (1u << sub); ++k) {
                const uint32_t n = __popc(__ballot_sync(0xFFFFFFFFu, in && c == k));
                mine += lane == (i << sub) + k ? n : 0u;
              }
            }
          }
        }
      });
    }
    s_cnt[wid][lane] = mine;
    __syncthreads();
    if (threadIdx.x < kMaxChunks) {   // chunk lane: the block's run, and each warp's part of it
      uint32_t sum = 0, n[kWarps];
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        n[w] = s_cnt[w][lane];
        sum += n[w];
      }
      uint32_t at = lane >= 1 && lane < a.n_chunks && sum ? atomicAdd(&a.fill[lane], sum) : 0u;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        s_cnt[w][lane] = at;
        at += n[w];
      }
    }
    __syncthreads();
    mine = s_cnt[wid][lane];
  }
  walk([&](uint32_t x, uint32_t y, bool live) {
    uint32_t cip, oip;
    const bool in = view_pair(view, x, y, cip, oip) && live;
    const uint32_t c0 = tab_hash(sT + 1024, cip) & d.col_mask;
    const uint32_t pos = touch_pos(d, tab_hash(sT, oip) & (d.eta - 1u));
    const uint32_t m_in = __ballot_sync(0xFFFFFFFFu, in), n_in = __popc(m_in), r_in = __popc(m_in & lt);
#pragma unroll
    for (uint32_t i = 0; i < SSD_MAX_R; ++i) {
      if (i < d.r) {
        const uint32_t col = column(i, cip, c0);
        const uint32_t c = rows ? i >> row_shift : (i << sub) + (col >> a.log2_count);
        const uint32_t se = ((i << d.q) | col) & in_chunk;
        const uint32_t bit = (se << d.log2_eta) | pos;   // (a chunk's bits number at most 2^32)
        if (rows ? (i >> row_shift) == 0 : i == 0)   // warp-uniform: some lane may be in chunk 0
          set_touch<CM>(a.touch0, bit, in && c == 0 && in_bounds(d, bit < d.touch_bits));
        if (a.n_chunks == 1) continue;
        uint32_t place = __shfl_sync(0xFFFFFFFFu, mine, c & 31u);
        if (SUB == 0) {
          place += r_in;
          mine += lane == c ? n_in : 0u;
        } else if (SUB == 1) {
          const uint32_t m1 = __ballot_sync(0xFFFFFFFFu, in && (c & 1u));
          const uint32_t r1 = __popc(m1 & lt), n1 = __popc(m1);
          place += (c & 1u) ? r1 : r_in - r1;
          mine += lane == 2u * i ? n_in - n1 : lane == 2u * i + 1u ? n1 : 0u;
        } else {
          for (uint32_t k = 0; k < (1u << sub); ++k) {
            const uint32_t m = __ballot_sync(0xFFFFFFFFu, in && c == (i << sub) + k);
            if (c == (i << sub) + k) place += __popc(m & lt);
            mine += lane == (i << sub) + k ? __popc(m) : 0u;
          }
        }
        if (in && c != 0) {
          if (place < a.cap) a.ent[(uint64_t)(c - 1u) * a.cap + place] = bit;
          else atomicOr(&a.counters->status, SSD_STATUS_INTERNAL);
        }
      }
    }
  });
}

}  // namespace

cudaError_t launch_lists(const Dims& d, const uint32_t* tables, const ScanBatch& b, const ListArgs& a, int grid,
                         const Tuning& tn, cudaStream_t st) {
  static_assert(kMaxChunks == 32, "a lane per chunk");
  if (a.n_chunks > kMaxChunks || b.n != 1) return cudaErrorInvalidValue;
  const int sub = a.log2_count >= d.q ? 0 : d.q - a.log2_count == 1 ? 1 : -1;
#define SSD_LISTS(CM)                                                          \
  do {                                                                         \
    if (sub == 0) k_lists<CM, 0><<<grid, kBlock, 0, st>>>(d, tables, b, a);    \
    else if (sub == 1) k_lists<CM, 1><<<grid, kBlock, 0, st>>>(d, tables, b, a); \
    else k_lists<CM, -1><<<grid, kBlock, 0, st>>>(d, tables, b, a);            \
  } while (0)
  if (tn.combine == 1) SSD_LISTS(1);
  else if (tn.combine == 2) SSD_LISTS(2);
  else SSD_LISTS(0);
#undef SSD_LISTS
  return cudaGetLastError();
}

cudaError_t launch_prehash(const Dims& d, const uint32_t* tables, const ScanBatch& b, uint2* out, int grid,
                           cudaStream_t st) {
  k_prehash<<<grid, kBlock, 0, st>>>(d, tables, b, out);
  return cudaGetLastError();
}

// Launches KERNEL<U, CM> for the tuning's unroll (U) and combine mode (CM).
#define SSD_TUNED_CM(KERNEL, U, GRID, ST, ...)                                             \
  do {                                                                                    \
    if (tn.combine == 1) KERNEL<U, 1><<<GRID, kBlock, 0, ST>>>(__VA_ARGS__);             \
    else if (tn.combine == 2) KERNEL<U, 2><<<GRID, kBlock, 0, ST>>>(__VA_ARGS__);        \
    else KERNEL<U, 0><<<GRID, kBlock, 0, ST>>>(__VA_ARGS__);                             \
  } while (0)
#define SSD_TUNED_LAUNCH(KERNEL, GRID, ST, ...)                                           \
  do {                                                                                    \
    switch (tn.unroll) {                                                                  \
      case 1: SSD_TUNED_CM(KERNEL, 1, GRID, ST, __VA_ARGS__); break;                      \
      case 2: SSD_TUNED_CM(KERNEL, 2, GRID, ST, __VA_ARGS__); break;                      \
      case 8: SSD_TUNED_CM(KERNEL, 8, GRID, ST, __VA_ARGS__); break;                      \
      default: SSD_TUNED_CM(KERNEL, 4, GRID, ST, __VA_ARGS__); break;                     \
    }                                                                                     \
  } while (0)

cudaError_t launch_touch_packed(const Dims& d, const uint4* vec, uint64_t nvec, const uint2* tail, uint32_t* bits,
                                uint64_t se0, uint64_t se_count, int grid, const Tuning& tn, cudaStream_t st) {
  SSD_TUNED_LAUNCH(k_touch_packed, grid, st, d, vec, nvec, tail, bits, se0, se_count);
  return cudaGetLastError();
}

cudaError_t launch_touch(const Dims& d, const uint32_t* tables, const ScanBatch& b, uint32_t* bits, uint64_t se0,
                         uint64_t se_count, int grid, const Tuning& tn, cudaStream_t st, DevCounters* clear) {
  SSD_TUNED_LAUNCH(k_touch, grid, st, d, tables, b, bits, se0, se_count, clear);
  return cudaGetLastError();
}
#undef SSD_TUNED_LAUNCH
#undef SSD_TUNED_CM

cudaError_t launch_scan(const Dims& d, const uint32_t* tables, const ScanBatch& b, int grid, const Tuning& tn,
                        cudaStream_t st) {
  static_assert(sizeof(ScanBatch) < 32000, "kernel parameter block too large");
  switch (tn.unroll) {
    case 1: k_scan<1><<<grid, kBlock, 0, st>>>(d, tables, b); break;
    case 2: k_scan<2><<<grid, kBlock, 0, st>>>(d, tables, b); break;
    case 8: k_scan<8><<<grid, kBlock, 0, st>>>(d, tables, b); break;
    default: k_scan<4><<<grid, kBlock, 0, st>>>(d, tables, b); break;
  }
  return cudaGetLastError();
}

}  // namespace ssd
