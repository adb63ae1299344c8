// Batched M2L on the 5th-generation tensor cores (tcgen05), split-BF16 operands
// with FP32 accumulation in tensor memory.
//
// Per wavevector k, the M2L of all systems (Sec. 2.1, real-matrix form of
// App. A.8) is the complex product L~ = A~ M~ with A~ (C x C) assembled from the
// kernel spectra and M~ (C x B).  A spectrum of kernel order j is real for even j and
// imaginary for odd j, so with the channels rotated by a_l = i for odd orders l (1 for
// even) on both sides, A~ becomes a REAL matrix W: L~ = a_l W (a_lam M~), where W holds
// the signed sums of at most two parity-reduced kernel values (negated where l and lam
// are both odd: i i = -1, while the order l + lam is even).  Real and imaginary parts of
// the systems are then columns of one real product,
//   D[(system, part) 128 x channel 64] = X[128 x 64] W^T[64 x 64],
// for 64 systems and C padded to 64 channels (p <= 7): half the multiplications of the
// complex form in a quarter of the operand bytes, and one real entry to assemble per
// matrix element.  Each FP32 operand x is split into x_hi = bf16(x) and
// x_lo = bf16(x - x_hi); D accumulates X_hi W_hi + X_lo W_hi + X_hi W_lo (the
// lo-lo term, below 2^-18 relative, is dropped), so every product carries a
// relative error of at most about 3 * 2^-18.
//
// Spectra are wavevector-major ([k][c][system]), so each wavevector's M~ and L~
// are one contiguous block.  One CTA of 256 threads (two per SM) owns a contiguous range
// of wavevectors; it assembles W once per wavevector and streams the system tiles through
// it: all threads convert the tile's X (loaded one tile ahead) into shared memory (two
// buffers), one thread issues the 12 MMAs (M = 128, N = 64, K = 16) into one of two TMEM
// accumulators and commits them to an mbarrier, and while they run the threads drain the
// previous accumulator (tcgen05.ld) to global memory; TMEM lanes 2n, 2n + 1 hold the
// real and imaginary parts of system n, so a warp stores 128 contiguous bytes of a
// channel, the rotation back being a swap of the two slots.
// Bound by memory for many systems (a wavevector's tile is read and written once, 64 KB
// at C = 64) and by the assembly of W for few.
// A two-level evaluation of 2^20 particles (2304 wavevectors x 512 systems) 2.20 -> 1.99 ms,
// 64 systems of 32^3 cells 4.08 -> 3.93 ms against the complex form of one 512-thread CTA
// per SM that assembled a 128 x 128 W for every tile.  The rest was instruction issue (1694
// warp instructions a tile, 56 % of the issue slots at 37 % of the memory's): addresses as
// 32-bit offsets within a wavevector's block and the odd orders as one constant bit mask,
// 1.98 -> 1.91 ms and 3.87 -> 3.84 ms.
// Shared-memory operands use the no-swizzle K-major layout of core matrices
// (8 rows x 16 bytes): element (r, k) at (r/8)*SBO + (k/8)*LBO + (r%8)*16 + (k%8)*2
// with LBO = 128 B and SBO = 1024 B.  Every mbarrier wait is bounded; on a
// timeout the kernel sets the plan's error flag, releases its tensor memory and
// returns.
#include <cuda_bf16.h>

#include <algorithm>
#include <vector>

#include "internal.cuh"
#include "m2l_table.cuh"
#include "tcgen05.cuh"

namespace pmmm {

namespace {

constexpr int TC_THREADS = 256;
constexpr int TC_CTAS_PER_SM = 2;
constexpr int TC_CH = 64;                         // channels after padding (p <= 7): GEMM N and K
constexpr int TC_NT = 64;                         // most systems per tile: GEMM M = 2 TC_NT
constexpr uint32_t TC_LBO = 128;                  // next core matrix along K
constexpr uint32_t TC_SBO = (TC_CH / 8) * 128;    // next 8-row group
constexpr uint32_t TC_X_BYTES = 2 * TC_NT * TC_CH * 2;  // one split of X: 16 KB
constexpr uint32_t TC_W_BYTES = TC_CH * TC_CH * 2;      // one split of W: 8 KB
constexpr int TC_GK = 256;                        // kernel values of a wavevector ((2p+1)^2 <= 225), the last zero
constexpr uint32_t TC_OFF_W = 2 * 2 * TC_X_BYTES;
constexpr uint32_t TC_OFF_GK = TC_OFF_W + 2 * 2 * TC_W_BYTES;
constexpr uint32_t TC_OFF_BAR = TC_OFF_GK + 2 * TC_GK * 4;
constexpr uint32_t TC_SMEM = TC_OFF_BAR + 32;
constexpr long long TC_WAIT_LIMIT = 1ll << 26;    // mbarrier polls before giving up

using tc::smem_u32;

// hi / lo BF16 split of 8 values, packed in K order (element j at the lower address).
__device__ __forceinline__ void split8(const float* x, uint4& hi, uint4& lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __nv_bfloat162 bh = __floats2bfloat162_rn(x[2 * j], x[2 * j + 1]);
    const float r0 = x[2 * j] - __low2float(bh), r1 = x[2 * j + 1] - __high2float(bh);
    const __nv_bfloat162 bl = __floats2bfloat162_rn(r0, r1);
    h[j] = *reinterpret_cast<const uint32_t*>(&bh);
    l[j] = *reinterpret_cast<const uint32_t*>(&bl);
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// byte offset of the 16-byte chunk (row r, K-group g) in one operand
__device__ __forceinline__ uint32_t chunk_off(int r, int g) {
  return (uint32_t)(r >> 3) * TC_SBO + (uint32_t)g * TC_LBO + (uint32_t)(r & 7) * 16;
}

__device__ __forceinline__ void cp4(uint32_t saddr, const void* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(saddr), "l"(g) : "memory");
}

// bit c set: channel c = l(l+1)+m has an odd order l (c in [l^2, (l+1)^2), c < 64)
constexpr uint64_t TC_ODD = (((1ull << 4) - 1) ^ ((1ull << 1) - 1)) | (((1ull << 16) - 1) ^ ((1ull << 9) - 1)) |
                            (((1ull << 36) - 1) ^ ((1ull << 25) - 1)) | (~0ull ^ ((1ull << 49) - 1));

// Entry table (build_m2l_table_tc): index 1 | index 2 << 10 | sign 2 << 30 | sign 1 << 31.
// nt: systems per tile (at most TC_NT).
__global__ void __launch_bounds__(TC_THREADS, TC_CTAS_PER_SM)
    m2l_tc_kernel(const float2* __restrict__ Mt, const float* __restrict__ Gr, float* __restrict__ Lt,
                  const uint32_t* __restrict__ tab_g, int C, int CG, int B, int nt, int64_t Kh, int64_t kchunk,
                  int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem[];
  float* gkb = reinterpret_cast<float*>(smem + TC_OFF_GK);  // [2][TC_GK]: kernel values of k and k + 1
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + TC_OFF_BAR);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + TC_OFF_BAR + 16);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t kbeg = (int64_t)blockIdx.x * kchunk, kend = min(Kh, kbeg + kchunk);
  const int ntiles = (B + nt - 1) / nt;

  // this thread's two units of W (output channel co, K-group of 8 input channels): table rows
  uint32_t tv[2][8];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int u = tid + q * TC_THREADS, co = u & 63, kg = u >> 6;
#pragma unroll
    for (int j = 0; j < 8; ++j) tv[q][j] = tab_g[co * TC_CH + kg * 8 + j];
  }
  auto fetch_gk = [&](int64_t kk, int slot) {
    if (kk < kend)
      for (int s = tid; s < CG; s += TC_THREADS) cp4(smem_u32(gkb + TC_GK * slot + s), Gr + (int64_t)s * Kh + kk);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (tid < 2) gkb[TC_GK * tid + TC_GK - 1] = 0.f;
  fetch_gk(kbeg, 0);
  if (tid == 0) {
    tc::bar_init(smem_u32(&bars[0]), 1);
    tc::bar_init(smem_u32(&bars[1]), 1);
    tc::fence_proxy_async();
  }
  if (warp == 0) tc::tmem_alloc(tmem_slot, 2 * TC_CH);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t idesc = tc::idesc_bf16_m128(TC_CH);
  const uint32_t sbase = smem_u32(smem);

  // Per element the loops below run a handful of instructions (offsets within a wavevector's
  // block in 32 bits, the odd orders as bit masks of this thread's channels); index
  // arithmetic in 64 bits and range tests per channel had been two thirds of the kernel's
  // 1700 instructions per thread and tile.
  const uint32_t oddx[2] = {(uint32_t)(TC_ODD >> (8 * (tid >> 6))) & 255u,
                            (uint32_t)(TC_ODD >> (8 * ((tid + TC_THREADS) >> 6))) & 255u};
  // X of one tile: unit (system n, K-group cg of 8 channels)
  float2 xm[2][8];
  auto load_x = [&](int64_t k, int t) {
    const float2* Mk = Mt + k * C * B;
    const int n = tid & 63, nch = n < min(nt, B - t * nt) ? C : 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int c0 = 8 * ((tid + q * TC_THREADS) >> 6);
      uint32_t off = (uint32_t)(c0 * B + t * nt + n);
#pragma unroll
      for (int j = 0; j < 8; ++j, off += (uint32_t)B)
        xm[q][j] = c0 + j < nch ? __ldg(Mk + off) : make_float2(0.f, 0.f);
    }
  };
  // drains accumulator `buf` (wavevector k, tile t): warp w reads TMEM lanes 32 (w % 4) ... and
  // channels 32 (w / 4) ...
  auto drain = [&](int buf, int64_t k, int t, uint32_t parity) -> bool {
    // warp-uniform outcome: the TMEM loads below are .sync.aligned
    const bool done = tc::bar_wait(smem_u32(&bars[buf]), parity, TC_WAIT_LIMIT);
    if (!__all_sync(0xffffffffu, done)) return false;
    tc::fence_after();
    const int row = 32 * (warp & 3) + lane, n = row >> 1;
    const uint32_t part = row & 1;
    const int nch = n < min(nt, B - t * nt) ? C : 0;
    float* Lk = Lt + 2 * k * C * B;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c0 = 32 * (warp >> 2) + 16 * h;
      const uint32_t odd = (uint32_t)(TC_ODD >> c0);
      uint32_t off = 2u * (uint32_t)(c0 * B + t * nt + n);
      float v[16];
      tc::ld16(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(buf * TC_CH + c0), v);
      tc::wait_ld();
#pragma unroll
      for (int j = 0; j < 16; ++j, off += 2u * (uint32_t)B) {
        // odd orders: L = i D, so the real part of D is the imaginary part of L and the
        // imaginary part of D minus the real part of L
        const uint32_t o = (odd >> j) & 1u;
        if (c0 + j < nch) Lk[off + (part ^ o)] = __uint_as_float(__float_as_uint(v[j]) ^ ((part & o) << 31));
      }
    }
    tc::fence_before();
    return true;
  };

  int it = 0, tprev = -1;
  int64_t kprev = -1;
  bool ok = true, stop = false;
  if (kbeg < kend && (int)blockIdx.y < ntiles) load_x(kbeg, blockIdx.y);
  for (int64_t k = kbeg; k < kend && !stop; ++k) {
    const int wb = (int)(k - kbeg) & 1;
    unsigned char* Wh = smem + TC_OFF_W + wb * 2 * TC_W_BYTES;
    // this wavevector's kernel values were fetched one wavevector ahead; start the next fetch
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const float* gk = gkb + TC_GK * wb;
    fetch_gk(k + 1, wb ^ 1);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int u = tid + q * TC_THREADS, co = u & 63, kg = u >> 6;
      float w[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t e = tv[q][j];
        const uint32_t g1 = __float_as_uint(gk[e & 255u]) ^ (e & 0x80000000u);
        const uint32_t g2 = __float_as_uint(gk[(e >> 10) & 255u]) ^ ((e << 1) & 0x80000000u);
        w[j] = __uint_as_float(g1) + __uint_as_float(g2);
      }
      uint4 hi, lo;
      split8(w, hi, lo);
      *reinterpret_cast<uint4*>(Wh + chunk_off(co, kg)) = hi;
      *reinterpret_cast<uint4*>(Wh + TC_W_BYTES + chunk_off(co, kg)) = lo;
    }
    for (int t = blockIdx.y; t < ntiles; t += gridDim.y, ++it) {
      const int buf = it & 1;
      unsigned char* Xh = smem + buf * 2 * TC_X_BYTES;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int u = tid + q * TC_THREADS, n = u & 63, cg = u >> 6;
        float xr[8], xi[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const bool odd = (oddx[q] >> j) & 1u;  // times i
          xr[j] = odd ? -xm[q][j].y : xm[q][j].x;
          xi[j] = odd ? xm[q][j].x : xm[q][j].y;
        }
        uint4 rh, rl, ih, il;
        split8(xr, rh, rl);
        split8(xi, ih, il);
        *reinterpret_cast<uint4*>(Xh + chunk_off(2 * n, cg)) = rh;
        *reinterpret_cast<uint4*>(Xh + chunk_off(2 * n + 1, cg)) = ih;
        *reinterpret_cast<uint4*>(Xh + TC_X_BYTES + chunk_off(2 * n, cg)) = rl;
        *reinterpret_cast<uint4*>(Xh + TC_X_BYTES + chunk_off(2 * n + 1, cg)) = il;
      }
      // the next tile's X, in flight during the MMAs and the drain
      if (t + (int)gridDim.y < ntiles)
        load_x(k, t + gridDim.y);
      else if (k + 1 < kend)
        load_x(k + 1, blockIdx.y);
      tc::fence_proxy_async();
      if (__syncthreads_or(!ok)) {  // a wait gave up: every thread leaves
        stop = true;
        break;
      }
      if (tid == 0) {
        tc::fence_after();
        const uint32_t x_h = sbase + buf * 2 * TC_X_BYTES, x_l = x_h + TC_X_BYTES;
        const uint32_t w_h = sbase + TC_OFF_W + wb * 2 * TC_W_BYTES, w_l = w_h + TC_W_BYTES;
        const uint32_t d = tmem + (uint32_t)(buf * TC_CH);
        const uint32_t Xs[3] = {x_h, x_l, x_h}, Ws[3] = {w_h, w_h, w_l};
#pragma unroll
        for (int sp = 0; sp < 3; ++sp)
#pragma unroll
          for (int j = 0; j < TC_CH / 16; ++j)
            tc::mma_bf16(d, tc::desc(Xs[sp] + 256 * j, TC_LBO, TC_SBO), tc::desc(Ws[sp] + 256 * j, TC_LBO, TC_SBO),
                         idesc, (sp | j) != 0);
        tc::commit(smem_u32(&bars[buf]));
      }
      // the previous tile's accumulator, while these MMAs run
      if (it > 0 && !drain(buf ^ 1, kprev, tprev, (uint32_t)(((it - 1) >> 1) & 1))) ok = false;
      kprev = k;
      tprev = t;
    }
  }
  if (!stop && it > 0 && ok && !drain((it - 1) & 1, kprev, tprev, (uint32_t)(((it - 1) >> 1) & 1))) ok = false;
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (__syncthreads_or(!ok)) {
    if (tid == 0) set_err(err, ERRBIT_TIMEOUT);
    // give MMAs still in flight a bounded time to finish before the memory is released
    if (it >= 1) tc::bar_wait(smem_u32(&bars[(it - 1) & 1]), (uint32_t)(((it - 1) >> 1) & 1), TC_WAIT_LIMIT);
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_free(tmem, 2 * TC_CH);
}

}  // namespace

bool m2l_tc_supported(int p) { return p >= 0 && p <= 7; }

// Packed entry table of the rotated real matrix, padded to 64 x 64 channels: the two
// kernel values of every entry (index TC_GK - 1, a zero, where a term is absent) and
// their signs, negated where both orders are odd.
std::vector<uint32_t> build_m2l_table_tc(int p) {
  const int C = (p + 1) * (p + 1);
  std::vector<M2LEntry> t = build_m2l_table(p);
  const uint32_t none = TC_GK - 1;
  std::vector<uint32_t> out((size_t)TC_CH * TC_CH, none | (none << 10));
  auto order = [](int c) {
    int l = 0;
    while ((l + 1) * (l + 1) <= c) ++l;
    return l;
  };
  for (int co = 0; co < C; ++co)
    for (int ci = 0; ci < C; ++ci) {
      const M2LEntry& e = t[(size_t)co * C + ci];
      const int f = (order(co) & order(ci) & 1) ? -1 : 1;
      const uint32_t i1 = e.s1 ? (uint32_t)e.i1 : none, i2 = e.s2 ? (uint32_t)e.i2 : none;
      out[(size_t)co * TC_CH + ci] =
          i1 | (i2 << 10) | (e.s2 * f < 0 ? 1u << 30 : 0u) | (e.s1 * f < 0 ? 1u << 31 : 0u);
    }
  return out;
}

cudaError_t launch_m2l_tc(const void* Mt, const void* Gr, void* Lt, const uint32_t* tab, int p, int B, int64_t Kh,
                          int num_sms, int tile, int* err, cudaStream_t s, int* nl) {
  if (!m2l_tc_supported(p) || B < 1) return cudaErrorInvalidValue;
  const int C = (p + 1) * (p + 1), CG = (2 * p + 1) * (2 * p + 1);
  const int nt = tile == 32 ? 32 : TC_NT;
  // one resident wave: wavevector ranges, and tiles split over blockIdx.y only where there
  // are fewer wavevectors than resident blocks
  const int64_t blocks = (int64_t)TC_CTAS_PER_SM * (num_sms > 0 ? num_sms : 1);
  const int64_t kchunk = (Kh + blocks - 1) / blocks, gx = (Kh + kchunk - 1) / kchunk;
  const int64_t ntiles = (B + nt - 1) / nt, gy = std::max<int64_t>(1, std::min<int64_t>(ntiles, blocks / gx));
  cudaError_t e = cudaFuncSetAttribute(m2l_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM);
  if (e != cudaSuccess) return e;
  m2l_tc_kernel<<<dim3((unsigned)gx, (unsigned)gy), TC_THREADS, TC_SMEM, s>>>(
      (const float2*)Mt, (const float*)Gr, (float*)Lt, tab, C, CG, B, nt, Kh, kchunk, err);
  ++*nl;
  return cudaGetLastError();
}

}  // namespace pmmm

namespace pmmm {
namespace {
// One thread waits on an mbarrier that expects an arrival nobody makes, with the
// bounded wait of the tensor-core kernels; the timeout raises the error flag.
__global__ void wait_timeout_kernel(long long polls, int* err) {
  __shared__ uint64_t bar;
  if (threadIdx.x != 0) return;
  tc::bar_init(tc::smem_u32(&bar), 1);
  if (!tc::bar_wait(tc::smem_u32(&bar), 0, polls)) set_err(err, ERRBIT_TIMEOUT);
}
}  // namespace
}  // namespace pmmm

extern "C" int pmmm_selftest_wait_timeout(void* cuda_stream, int64_t polls) {
  using namespace pmmm;
  if (polls < 1 || polls > (int64_t)1 << 24) return PMMM_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  int* err = nullptr;
  cudaError_t e = cudaMalloc(&err, sizeof(int));
  if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, sizeof(int), s);
  if (e == cudaSuccess) {
    wait_timeout_kernel<<<1, 32, 0, s>>>(polls, err);
    e = cudaGetLastError();
  }
  int h = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (err) cudaFree(err);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? PMMM_ERR_OOM : PMMM_ERR_CUDA;
  return (h & ERRBIT_TIMEOUT) ? PMMM_ERR_TIMEOUT : PMMM_OK;
}
