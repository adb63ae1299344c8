// Sort of the particles by cell and the work lists of an evaluation, in four
// launches (Sec. 2.1: "for each cell, the set of particles inside is known ... in
// an O(N) procedure"):
//   bin    the cell of every particle (binning.cuh), its record in input order and
//          its arrival number in its cell (one atomic per distinct cell of a warp);
//   scan   exclusive sums of the per-cell counts within blocks of 1024 cells, the
//          block that finishes last summing the block totals;
//   place  the particle indices into their cells in arrival order, and the complete
//          per-cell offsets (particles, near-field work items, source pairs);
//   rank   the stable order (a particle's place in its cell is the number of particles
//          of the cell with a smaller index, so the arrival order, which the scheduling
//          decides, leaves no trace) and the sorted records in both layouts.
// The rank launch compares each particle with all of its cell: as many comparisons as
// the cell has pairs with itself, at 2 instructions each against 15 of the near field,
// which takes those pairs and the ones with 26 or 124 more cells; cells of 1024 particles
// or more are ranked by whole blocks instead (crowded_rank).
// Latency-bound for small systems (4 dependent launches), bound by scattered 4- to
// 16-byte accesses to the records for large ones.  Sort stage by CUDA events against
// the radix sort it replaces (histogram, two scans and a scatter per 8-bit digit, cell
// bounds, two list scans, gather: 12 or 13 launches): 20011 particles / 16^3 cells
// 71 -> 26 us; 2^20 / 32^3 104 -> 65 us; 10^6 / 64^3 135 -> 64 us; 5.6 million in 64
// systems of 32^3 cells 490 -> 350 us; 2^24 / 64^3 1103 -> 990 us; 4096 / 8^3 in FP64
// 66 -> 27 us.
#include "binning.cuh"
#include "internal.cuh"

namespace pmmm {

namespace {

constexpr int CS_THREADS = 256;  // threads of a scan block
constexpr int CS_PER = 4;        // cells per thread
constexpr int CS_BLK = CS_THREADS * CS_PER;
constexpr int CS_NQ = 3;         // quantities scanned: particles, work items, source pairs

// system of particle i: offsets[s] <= i < offsets[s+1]
__device__ __forceinline__ int system_of(const int64_t* __restrict__ off, int nsys, int64_t i) {
  int lo = 0, hi = nsys;  // invariant: off[lo] <= i < off[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (off[mid] <= i) lo = mid;
    else hi = mid;
  }
  return lo;
}

template <typename T>
__global__ void __launch_bounds__(256) bin_count_kernel(const T* __restrict__ pos, const T* __restrict__ q, int64_t n,
                                                        const int64_t* __restrict__ offsets, int nsys, Geo g,
                                                        int64_t Ksys, uint32_t* __restrict__ keys,
                                                        uint32_t* __restrict__ arrival, uint32_t* __restrict__ count,
                                                        T* __restrict__ rec, int* __restrict__ err) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool live = i < n;
  uint32_t key = 0xffffffffu;  // no cell: at most 2^30 cells
  if (live) {
    const uint32_t key0 = offsets ? (uint32_t)((int64_t)system_of(offsets, nsys, i) * Ksys) : 0u;
    key = bin_record<T>(pos, q, i, g, key0, keys, rec, err);
  }
  // one atomic per distinct cell of the warp (inputs that are already sorted by cell
  // would otherwise serialise 32 additions on one address)
  const uint32_t peers = __match_any_sync(0xffffffffu, key);
  const int leader = __ffs(peers) - 1;
  uint32_t base = 0;
  if (live && lane == leader) base = atomicAdd(count + key, (uint32_t)__popc(peers));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (live) arrival[i] = base + __popc(peers & ((1u << lane) - 1u));
}

struct Quant {
  uint32_t v[CS_NQ];
};
__device__ __forceinline__ Quant quantities(uint32_t cnt) {
  Quant q;
  q.v[0] = cnt;
  q.v[1] = (cnt + PP_CHUNK - 1) / PP_CHUNK;
  q.v[2] = (cnt + 1) / 2;
  return q;
}

// Exclusive scan of one Quant per thread over the block; total of the block in *tot
// (every thread).
__device__ __forceinline__ Quant block_scan(Quant q, uint32_t (*sh)[CS_THREADS / 32], Quant* tot) {
  constexpr int NW = CS_THREADS / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Quant inc = q;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
#pragma unroll
    for (int k = 0; k < CS_NQ; ++k) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, inc.v[k], o);
      if (lane >= o) inc.v[k] += x;
    }
  if (lane == 31)
#pragma unroll
    for (int k = 0; k < CS_NQ; ++k) sh[k][warp] = inc.v[k];
  __syncthreads();
  Quant out;
#pragma unroll
  for (int k = 0; k < CS_NQ; ++k) {
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const uint32_t v = sh[k][w];
      if (w < warp) before += v;
      all += v;
    }
    tot->v[k] = all;
    out.v[k] = before + inc.v[k] - q.v[k];
  }
  __syncthreads();
  return out;
}

// Block-local exclusive sums of the cells' quantities (CS_PER consecutive cells per
// thread); the counts are left zeroed for the next evaluation.  The last block to
// finish turns the block totals into their exclusive prefix sums (tot[block][CS_NQ])
// and re-arms the ticket.
__global__ void __launch_bounds__(CS_THREADS) cell_scan_kernel(uint32_t* __restrict__ count, int64_t K, CellLists l) {
  __shared__ uint32_t sh[CS_NQ][CS_THREADS / 32];
  __shared__ bool last;
  const int tid = threadIdx.x;
  const int64_t c0 = (int64_t)blockIdx.x * CS_BLK + (int64_t)tid * CS_PER;
  Quant q[CS_PER], sum;
#pragma unroll
  for (int k = 0; k < CS_NQ; ++k) sum.v[k] = 0u;
#pragma unroll
  for (int j = 0; j < CS_PER; ++j) {
    uint32_t cnt = 0;
    if (c0 + j < K) {
      cnt = count[c0 + j];
      count[c0 + j] = 0u;
    }
    q[j] = quantities(cnt);
#pragma unroll
    for (int k = 0; k < CS_NQ; ++k) sum.v[k] += q[j].v[k];
  }
  Quant tot;
  Quant ex = block_scan(sum, sh, &tot);
#pragma unroll
  for (int j = 0; j < CS_PER; ++j) {
    const int64_t c = c0 + j;
    if (c <= K) {
      l.cs_local[c] = ex.v[0];
      l.item_start[c] = ex.v[1];
      if (l.pair_start) l.pair_start[c] = ex.v[2];
    }
#pragma unroll
    for (int k = 0; k < CS_NQ; ++k) ex.v[k] += q[j].v[k];
  }
  if (tid == 0) {
#pragma unroll
    for (int k = 0; k < CS_NQ; ++k) l.tot[(int64_t)blockIdx.x * CS_NQ + k] = tot.v[k];
    if (blockIdx.x == 0) *l.counter = 0u;
    __threadfence();
    last = atomicAdd(l.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  Quant run;
#pragma unroll
  for (int k = 0; k < CS_NQ; ++k) run.v[k] = 0u;
  for (int64_t b0 = 0; b0 < gridDim.x; b0 += CS_THREADS) {
    const int64_t b = b0 + tid;
    Quant v;
#pragma unroll
    for (int k = 0; k < CS_NQ; ++k) v.v[k] = b < gridDim.x ? __ldcg(l.tot + b * CS_NQ + k) : 0u;
    const Quant e = block_scan(v, sh, &tot);
#pragma unroll
    for (int k = 0; k < CS_NQ; ++k) {
      if (b < gridDim.x) l.tot[b * CS_NQ + k] = run.v[k] + e.v[k];
      run.v[k] += tot.v[k];
    }
  }
  if (tid == 0) *l.ticket = 0u;
}

// Particle indices into their cells in arrival order (order[]), and the complete
// per-cell offsets: block-local sums plus the prefix of the block.
__global__ void __launch_bounds__(256) place_kernel(const uint32_t* __restrict__ keys,
                                                    const uint32_t* __restrict__ arrival, int64_t n, int64_t K,
                                                    CellLists l, uint32_t* __restrict__ order) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    const uint32_t c = keys[i];
    order[l.cs_local[c] + l.tot[(int64_t)(c / CS_BLK) * CS_NQ] + arrival[i]] = (uint32_t)i;
  }
  if (i <= K) {
    const uint32_t* pre = l.tot + (i / CS_BLK) * CS_NQ;
    l.cs[i] = (int)(l.cs_local[i] + pre[0]);
    l.item_start[i] += pre[1];
    if (l.pair_start) l.pair_start[i] += pre[2];
  }
}

// Ranks of the indices that the threads t0 .. of the block hold (the others pass NONE)
// among the indices order[b .. e): the block sorts its own (bitonic, in shared memory),
// every index of the range finds its place between them by bisection and is counted
// there, and a running sum of the counts gives the ranks.  Returns the sorted index that
// thread t0 + i takes on (the i-th), its rank in *rank.  About 30 instructions per index
// and block, against 2 RANK_THREADS for the plain comparison (2^20-particle Plummer
// sphere on 64^3 cells, up to 6300 particles in a cell: sort stage 350 us with the plain
// comparison alone).
constexpr int RANK_THREADS = 256;
constexpr uint32_t RANK_CROWD = 1024;  // cells of at least this many particles
constexpr uint32_t RANK_NONE = 0xffffffffu;

__device__ __forceinline__ uint32_t crowded_rank(const uint32_t* __restrict__ order, uint32_t me, uint32_t b,
                                                 uint32_t e, int t0, uint32_t* rank) {
  __shared__ uint32_t srt[RANK_THREADS], cnt[RANK_THREADS + 1], wsum[RANK_THREADS / 32];
  const int t = threadIdx.x;
  __syncthreads();  // the arrays may still be read from an earlier call
  srt[t] = me;
  cnt[t] = 0u;
  if (t == 0) cnt[RANK_THREADS] = 0u;
  __syncthreads();
  // rolled loops: 32 registers, 56 otherwise, and the kernel is bound by loads in flight
#pragma unroll 1
  for (int k = 2; k <= RANK_THREADS; k <<= 1)
#pragma unroll 1
    for (int o = k >> 1; o > 0; o >>= 1) {
      const int p = t ^ o;
      if (p > t) {
        const uint32_t x = srt[t], y = srt[p];
        if ((x > y) == ((t & k) == 0)) {
          srt[t] = y;
          srt[p] = x;
        }
      }
      __syncthreads();
    }
#pragma unroll 2
  for (uint32_t i = b + t; i < e; i += RANK_THREADS) {
    const uint32_t v = order[i];
    int lo = 0;  // number of own indices <= v
#pragma unroll
    for (int o = RANK_THREADS / 2; o > 0; o >>= 1)
      if (srt[lo + o - 1] <= v) lo += o;
    if (srt[lo] <= v) ++lo;  // only from lo = RANK_THREADS - 1
    atomicAdd(&cnt[lo], 1u);
  }
  __syncthreads();
  uint32_t x = cnt[t];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if ((t & 31) >= o) x += y;
  }
  if ((t & 31) == 31) wsum[t >> 5] = x;
  __syncthreads();
  for (int w = 0; w < (t >> 5); ++w) x += wsum[w];
  cnt[t] = x;  // only this thread's entry has been read so far
  __syncthreads();
  const int i = t >= t0 ? t - t0 : 0;
  *rank = cnt[i];
  return srt[i];
}

// The stable order, and with it everything an evaluation reads of a sorted particle:
// thread s takes the particle at arrival slot s, whose sorted slot is the first slot of
// its cell plus the number of smaller indices in the cell, and writes there its
// original index, cell and record; its half of its source pair (PACK: FP32 pair
// layout, pp.cu), with the dummy partner that completes an odd cell; and the cell of
// the work item that starts with it.  Also (epart not null) zeroes the energy partials of the unused
// item slots (of all of them when the near-field kernel accumulates into them).
// order is 16-byte aligned and readable up to the next multiple of four entries.
template <typename V, bool PACK>
__global__ void __launch_bounds__(RANK_THREADS) rank_gather_kernel(const uint32_t* __restrict__ order,
                                                          const uint32_t* __restrict__ keys, CellLists l, int64_t n,
                                                          int64_t K, const V* __restrict__ rec,
                                                          uint32_t* __restrict__ vals,
                                                          uint32_t* __restrict__ keys_sorted, V* __restrict__ part,
                                                          float* __restrict__ src2, uint32_t* __restrict__ item_cell,
                                                          double4* __restrict__ epart, int64_t max_items,
                                                          int zero_all) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (epart)
    for (int64_t i = (zero_all ? 0 : (int64_t)l.item_start[K]) + s; i < max_items;
         i += (int64_t)gridDim.x * blockDim.x)
      epart[i] = make_double4(0.0, 0.0, 0.0, 0.0);
  if ((int64_t)blockIdx.x * RANK_THREADS >= n) return;  // the whole block
  const bool live = s < n;
  uint32_t me = order[live ? s : n - 1], c = keys[me], j = 0;
  const uint32_t b = (uint32_t)__ldg(l.cs + c), e = (uint32_t)__ldg(l.cs + c + 1);
  // The indices of a crowded cell are ranked by the block as a whole; such a cell is
  // longer than a block, so it holds the block's first slot or its last.  Every other
  // index is compared with all of its cell by its thread.  (Blocks that held parts of two
  // cells compared all their indices so: sort stage of 786432 particles in a Plummer sphere
  // on 32^3 cells 418 us, now 188; 163840 on 16^3 210 us, now 79.)
  const bool crowd = live && e - b >= RANK_CROWD;
  __shared__ uint32_t ends[2][3];  // cell, b, e
  const int nlive = (int)min((int64_t)RANK_THREADS, n - (int64_t)blockIdx.x * RANK_THREADS);
  if (threadIdx.x == 0 || (int)threadIdx.x == nlive - 1) {
    uint32_t* q = ends[threadIdx.x == 0 ? 0 : 1];
    q[0] = crowd ? c : RANK_NONE;
    q[1] = b;
    q[2] = e;
    if (nlive == 1) ends[1][0] = RANK_NONE;  // one thread is both
  }
  __syncthreads();
#pragma unroll 1
  for (int k = 0; k < 2; ++k) {
    const uint32_t ck = ends[k][0];
    if (ck == RANK_NONE || (k == 1 && ck == ends[0][0])) continue;
    const int64_t s0 = (int64_t)ends[k][1] - (int64_t)blockIdx.x * RANK_THREADS;
    uint32_t r;
    const bool mine = live && c == ck;
    const uint32_t v = crowded_rank(order, mine ? me : RANK_NONE, ends[k][1], ends[k][2], s0 > 0 ? (int)s0 : 0, &r);
    if (mine) {
      me = v;
      j = r;
    }
  }
  if (live && !crowd) {
    // whole 16-byte words; the entries outside [b, e) of the first and last are left out
    const uint4* o4 = reinterpret_cast<const uint4*>(order);
    uint32_t w = b / 4;
    const uint32_t w1 = (e + 3) / 4;
    auto edge = [&](uint32_t i) {
      const uint4 v = o4[i];
      const uint32_t t = 4 * i;
      j += (t >= b && t < e && v.x < me) + (t + 1 >= b && t + 1 < e && v.y < me) +
           (t + 2 >= b && t + 2 < e && v.z < me) + (t + 3 >= b && t + 3 < e && v.w < me);
    };
    edge(w++);
#pragma unroll 4
    for (; w + 1 < w1; ++w) {
      const uint4 v = o4[w];
      j += (v.x < me) + (v.y < me) + (v.z < me) + (v.w < me);
    }
    if (w < w1) edge(w);
  }
  if (!live) return;
  const V r = rec[me];
  vals[b + j] = me;
  keys_sorted[b + j] = c;
  part[b + j] = r;
  if (j % PP_CHUNK == 0) item_cell[l.item_start[c] + j / PP_CHUNK] = c;
  if constexpr (PACK) {
    float* o = src2 + 8 * ((int64_t)l.pair_start[c] + j / 2);
    if (b + j + 1 == e && (j & 1) == 0) {
      reinterpret_cast<float4*>(o)[0] = make_float4((float)r.x, 1.0e4f, (float)r.y, 1.0e4f);
      reinterpret_cast<float4*>(o)[1] = make_float4((float)r.z, 1.0e4f, (float)r.w, 0.0f);
    } else {
      o += j & 1;
      o[0] = (float)r.x;
      o[2] = (float)r.y;
      o[4] = (float)r.z;
      o[6] = (float)r.w;
    }
  }
}

inline unsigned grid1(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

int64_t cell_list_totals(int64_t K) { return CS_NQ * ((K + 1 + CS_BLK - 1) / CS_BLK); }

cudaError_t launch_bin_count(const void* pos, const void* q, bool fp64, int64_t n, const int64_t* offsets, int nsys,
                             const Geo& g, int64_t Ksys, uint32_t* keys, uint32_t* arrival, uint32_t* count, void* rec,
                             int* err, cudaStream_t s, int* nl) {
  if (n <= 0) return cudaSuccess;
  if (fp64)
    bin_count_kernel<double><<<grid1(n, 256), 256, 0, s>>>((const double*)pos, (const double*)q, n, offsets, nsys, g,
                                                           Ksys, keys, arrival, count, (double*)rec, err);
  else
    bin_count_kernel<float><<<grid1(n, 256), 256, 0, s>>>((const float*)pos, (const float*)q, n, offsets, nsys, g,
                                                          Ksys, keys, arrival, count, (float*)rec, err);
  ++*nl;
  return cudaGetLastError();
}

cudaError_t launch_cell_sort(const uint32_t* keys, const uint32_t* arrival, uint32_t* count, const void* rec, bool fp64,
                             int64_t n, int64_t K, const CellLists& l, uint32_t* order, uint32_t* vals,
                             uint32_t* keys_sorted, void* part, void* src2, uint32_t* item_cell, double* epart,
                             int64_t max_items, bool zero_all, cudaStream_t s, int* nl) {
  cell_scan_kernel<<<grid1(K + 1, CS_BLK), CS_THREADS, 0, s>>>(count, K, l);
  place_kernel<<<grid1(n > K ? n : K + 1, 256), 256, 0, s>>>(keys, arrival, n, K, l, order);
  const int64_t work = epart && max_items > n ? max_items : n;
  if (work <= 0) {
    *nl += 2;
    return cudaGetLastError();
  }
  const unsigned blocks = grid1(work, RANK_THREADS);
  const int za = zero_all ? 1 : 0;
  if (fp64)
    rank_gather_kernel<double4, false><<<blocks, RANK_THREADS, 0, s>>>(order, keys, l, n, K, (const double4*)rec, vals,
                                                              keys_sorted, (double4*)part, nullptr, item_cell,
                                                              (double4*)epart, max_items, za);
  else
    rank_gather_kernel<float4, true><<<blocks, RANK_THREADS, 0, s>>>(order, keys, l, n, K, (const float4*)rec, vals,
                                                            keys_sorted, (float4*)part, (float*)src2, item_cell,
                                                            (double4*)epart, max_items, za);
  *nl += 3;
  return cudaGetLastError();
}

}  // namespace pmmm
