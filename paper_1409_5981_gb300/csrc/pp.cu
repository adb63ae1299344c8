// Near field (Sec. 2.1, Sec. 2.2): the pure Newtonian 1/r interaction with every
// particle of the (2c+1)^3 masked cells, plus the combination with the far field
// and the scatter back to the caller's order:
//   phi_i   = sign * (phi_far + sum_j q_j / r_ij)
//   force_i = -q_i * sign * (grad_far + sum_j grad(q_j / r_ij))
//
// Work is split into items of (cell, chunk of up to 32 targets), numbered by an
// exclusive scan over the cells so that crowded cells spread over many warps.
// FP32 items (pp_kernel_tma): one warp per item, its R targets in registers, lane l
// owning target l mod TL and source phase l / TL (TL = R rounded up to a power of two,
// so a chunk of 8 targets still keeps 32 lanes busy on 4 source phases); sparse FP32
// systems: one thread per target (pp_target_kernel); FP64: one block per item
// (pp64_kernel).  Pairs at r = 0 (the self pair, and particles that coincide after the
// rounding of their coordinates) add zero.
#include "internal.cuh"
#include "tcgen05.cuh"

namespace pmmm {

namespace {

constexpr int PP_WARPS = 4;
constexpr int CHUNK = PP_CHUNK;

// FP32 reciprocal square root: the hardware approximation (PTX rsqrt.approx,
// relative error below 2^-22.9) with subnormal inputs flushed to zero.  A pair
// distance is never subnormal (the self pair gives exactly zero and is masked),
// so the flush changes no result and spares the subnormal handling of rsqrtf.
__device__ __forceinline__ float rsqrt_ftz(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Pair-interleaved source records for the FP32 near field: the particles of
// cell c occupy pairs pair_start[c] ... (a cell with an odd count ends with a
// dummy of zero charge far outside the box).  Pair j is two 16-byte words
// {x_a, x_b, y_a, y_b}, {z_a, z_b, q_a, q_b}, so that one 128-bit load yields
// the packed operands of two sources.

// FP64 reciprocal square root: the hardware approximation (PTX rsqrt.approx.ftz.f64,
// from the upper word of x, about 20 bits) and one third-order Householder step,
//   y = y0 + y0 e (1/2 + 3/8 e),  e = 1 - x y0^2,
// whose remainder 5/16 e^3 is below 2^-58: five FP64 operations, at 64 cycles of an SM
// quarter each.  Zero x gives 0, subnormal x the library's rsqrt(x); infinite x gives NaN.
__device__ __forceinline__ double rsqrt64(double x) {
  double y0;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(x));
  const double e = fma(-x, y0 * y0, 1.0);
  double y = fma(y0 * e, fma(e, 0.375, 0.5), y0);
  if (__double2hiint(x) < 0x00100000) y = __double_as_longlong(x) == 0 ? 0.0 : rsqrt(x);
  return y;
}

// FP64 near field (c = 1 or 2).  GB300 issues an FP64 instruction of a warp every 64
// cycles per SM quarter, so the pair's 18 FP64 operations bound the kernel and
// everything else is arranged to keep their lanes full and the quarters evenly loaded:
// one block of 4 warps per item, thread t taking target t mod R (R the item's targets)
// and every P-th source from number t / R on of all (2c+1)^3 cells' sources as one list
// (P = 128 / R source phases; 128 - R P lanes idle), the partial sums added by a tree in
// shared memory.  The target's coordinates in the frames of the neighbour cells are held
// per axis and selected by integer operations.  Items come from a global counter; an
// item's results depend only on the item.
// Against one warp per item with power-of-two lane splits, per-cell loops and rsqrt():
// 4096 particles / 8^3 open 303 -> 53 us (512 items over 608 SM quarters: a quarter of
// them idle, others with three), 131072 / 16^3 periodic 4.83 -> 4.02 ms (81 % of the
// FP64 issue rate in the pairs' 18 operations).
constexpr int P64_THREADS = 128;
constexpr int P64_BLOCKS_PER_SM = 2;
// Three blocks where there are many items of next to no pairs (the items are then a chain of
// memory latencies): at least 2^14 particles, at most one to three cells.  60000 in 200
// systems of 16^3 cells 3.65 -> 3.30 ms, 31457 / 64^3 uniform 2.77 -> 2.58 ms, in a Plummer
// sphere 3.59 -> 3.82 ms: consecutive crowded items share an SM, which is why fuller cells
// keep two (Plummer 8192 / 16^3 2.0 ms with two, 2.9 with three, 3.8 with four).
inline int p64_blocks_per_sm(int64_t n, int64_t K) {
  return n >= (1 << 14) && 3 * n <= K ? P64_BLOCKS_PER_SM + 1 : P64_BLOCKS_PER_SM;
}

template <int CUT>
__global__ void __launch_bounds__(P64_THREADS, P64_BLOCKS_PER_SM) pp64_kernel(
    const double* __restrict__ part, const uint32_t* __restrict__ vals, const int* __restrict__ cs, int64_t K,
    const uint32_t* __restrict__ item_start, const uint32_t* __restrict__ item_cell,
    unsigned int* __restrict__ counter, const double* __restrict__ far, PPParams pp, double* __restrict__ phi,
    double* __restrict__ force, double* __restrict__ epart) {
  constexpr int W = 2 * CUT + 1, NN = W * W * W;
  __shared__ int first[NN + 1], off[NN];  // list position e of cell k: first[k] <= e < first[k+1], record e + off[k]
  __shared__ double sum[4][P64_THREADS];
  __shared__ uint32_t next_item;
  const double4* P = reinterpret_cast<const double4*>(part);
  const int tid = threadIdx.x, lane = tid & 31;
  const uint32_t nitems = item_start[K];
  const int nx = pp.n[0], ny = pp.n[1], nz = pp.n[2];
  for (;;) {
    if (tid == 0) next_item = atomicAdd(counter, 1u);
    __syncthreads();
    const uint32_t item = next_item;
    if (item >= nitems) break;
    const int cell = (int)item_cell[item];
    const int tbeg = cs[cell] + (int)(item - item_start[cell]) * CHUNK;
    const int R = min(CHUNK, cs[cell + 1] - tbeg), NP = P64_THREADS / R;
    const int tl = tid % R, ph = tid / R;
    const bool active = ph < NP;
    if (tid < 32) {
      // counts of the cells in (z, y, x) order and their running sum
      const int sbase = cell - cell % pp.ksys, lc = cell - sbase;
      const int ix = lc % nx, iy = (lc / nx) % ny, iz = lc / (nx * ny);
      int run = 0;
      for (int k0 = 0; k0 < NN; k0 += 32) {
        const int k = k0 + lane;
        int b = 0, m = 0;
        if (k < NN) {
          int jx = ix + k % W - CUT, jy = iy + (k / W) % W - CUT, jz = iz + k / (W * W) - CUT;
          bool ok = true;
          if (jx < 0 || jx >= nx) { ok = ok && pp.periodic; jx += (jx < 0) ? nx : -nx; }
          if (jy < 0 || jy >= ny) { ok = ok && pp.periodic; jy += (jy < 0) ? ny : -ny; }
          if (jz < 0 || jz >= nz) { ok = ok && pp.periodic; jz += (jz < 0) ? nz : -nz; }
          if (ok) {
            const int cj = sbase + jx + nx * (jy + ny * jz);
            b = __ldg(cs + cj);
            m = __ldg(cs + cj + 1) - b;
          }
        }
        int v = m;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int u = __shfl_up_sync(0xffffffffu, v, o);
          if (lane >= o) v += u;
        }
        if (k < NN) {
          first[k] = run + v - m;
          off[k] = b - (run + v - m);
        }
        run += __shfl_sync(0xffffffffu, v, 31);
      }
      if (lane == 0) first[NN] = run;
    }
    const double4 xi = P[tbeg + tl];
    double tx[W], ty[W], tz[W];  // the target in the frames of the cells at each axis offset
#pragma unroll
    for (int d = 0; d < W; ++d) {
      tx[d] = xi.x - (double)(d - CUT) * pp.csf[0];
      ty[d] = xi.y - (double)(d - CUT) * pp.csf[1];
      tz[d] = xi.z - (double)(d - CUT) * pp.csf[2];
    }
    __syncthreads();
    double pot = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
    if (active) {
      const int total = first[NN];
      int k = 0;
      auto pair = [&](int e, auto root) {
        while (e >= first[k + 1]) ++k;
        const double4 r = P[e + off[k]];
        const int ex = k % W, ey = (k / W) % W, ez = k / (W * W);
        double ux = tx[0], uy = ty[0], uz = tz[0];
#pragma unroll
        for (int d = 1; d < W; ++d) {
          if (ex == d) ux = tx[d];
          if (ey == d) uy = ty[d];
          if (ez == d) uz = tz[d];
        }
        const double dx = ux - r.x, dy = uy - r.y, dz = uz - r.z;
        const double ri = root(fma(dx, dx, fma(dy, dy, dz * dz)));  // 0 for the self pair
        const double qr = r.w * ri;
        pot += qr;
        const double qr3 = qr * (ri * ri);
        gx = fma(-qr3, dx, gx);
        gy = fma(-qr3, dy, gy);
        gz = fma(-qr3, dz, gz);
      };
      int e = ph;
      for (; e + NP < total; e += 2 * NP) {  // two at a time: 4.02 ms against 5.41 one by one
        pair(e, rsqrt64);
        pair(e + NP, rsqrt64);
      }
      if (e < total) pair(e, rsqrt64);
      // an infinite square (a particle flagged as far outside an open box), whose root is 0:
      // the sums once more with the library's, one test per target instead of one per pair (on
      // the exponent, an integer operation)
      if ((__double2hiint(pot) & 0x7ff00000) == 0x7ff00000) {
        pot = gx = gy = gz = 0.0;
        k = 0;
        for (e = ph; e < total; e += NP) pair(e, [](double x) { return x > 0.0 ? rsqrt(x) : 0.0; });
      }
    }
    sum[0][tid] = pot;
    sum[1][tid] = gx;
    sum[2][tid] = gy;
    sum[3][tid] = gz;
    for (int m = NP; m > 1;) {  // tree over the phases
      const int h = (m + 1) / 2;
      __syncthreads();
      if (ph < m - h)
#pragma unroll
        for (int q = 0; q < 4; ++q) sum[q][tid] += sum[q][tid + h * R];
      m = h;
    }
    __syncthreads();
    if (tid < 32) {
      double e_t = 0.0, f_t[3] = {0.0, 0.0, 0.0};
      if (tid < R) {
        const int s = tbeg + tid;
        const double4 fr = reinterpret_cast<const double4*>(far)[s];
        const double sg = pp.signf, q = P[s].w;
        const double pt = sg * (fr.x + sum[0][tid] * pp.ihf);
        const double g[3] = {sg * (fr.y + sum[1][tid] * pp.ih2f), sg * (fr.z + sum[2][tid] * pp.ih2f),
                             sg * (fr.w + sum[3][tid] * pp.ih2f)};
        const uint32_t o = vals[s];
        if (phi) phi[o] = pt;
        e_t = 0.5 * q * pt;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          f_t[a] = -q * g[a];
          if (force) force[3 * (int64_t)o + a] = f_t[a];
        }
      }
      // deterministic sums of this item's energy and net-force partials
#pragma unroll
      for (int o = 16; epart && o > 0; o >>= 1) {
        e_t += __shfl_xor_sync(0xffffffffu, e_t, o);
#pragma unroll
        for (int a = 0; a < 3; ++a) f_t[a] += __shfl_xor_sync(0xffffffffu, f_t[a], o);
      }
      if (epart && lane == 0) {
        epart[(int64_t)item * 4 + 0] = e_t;
#pragma unroll
        for (int a = 0; a < 3; ++a) epart[(int64_t)item * 4 + 1 + a] = f_t[a];
      }
    }
  }
}

typedef unsigned long long f2;  // two packed floats (low word = first)
__device__ __forceinline__ f2 pk2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void up2(f2 r, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r)); }
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// A two-source step with the subtractions and r^2 packed (f32x2) and the
// arithmetic after the rsqrt in scalar FP32 (faster in the per-target kernel,
// whose lanes follow different neighbour lists).
template <bool SELF>
__device__ __forceinline__ void pp_pair2_mixed(const ulonglong2& A, const ulonglong2& B, f2 tx, f2 ty, f2 tz, f2& pot,
                                               f2& gx, f2& gy, f2& gz) {
  const f2 dx = sub2(tx, A.x), dy = sub2(ty, A.y), dz = sub2(tz, B.x);
  const f2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
  float a, b;
  up2(r2, a, b);
  float ra = rsqrt_ftz(a), rb = rsqrt_ftz(b);
  if (SELF) {
    ra = a > 0.f ? ra : 0.f;
    rb = b > 0.f ? rb : 0.f;
  }
  float qa, qb, dxa, dxb, dya, dyb, dza, dzb;
  up2(B.y, qa, qb);
  up2(dx, dxa, dxb);
  up2(dy, dya, dyb);
  up2(dz, dza, dzb);
  const float qra = qa * ra, qrb = qb * rb;
  float p0, p1, x0, x1, y0, y1, z0, z1;
  up2(pot, p0, p1);
  up2(gx, x0, x1);
  up2(gy, y0, y1);
  up2(gz, z0, z1);
  p0 += qra;
  p1 += qrb;
  const float ca = qra * (ra * ra), cb = qrb * (rb * rb);
  x0 = fmaf(ca, dxa, x0);
  y0 = fmaf(ca, dya, y0);
  z0 = fmaf(ca, dza, z0);
  x1 = fmaf(cb, dxb, x1);
  y1 = fmaf(cb, dyb, y1);
  z1 = fmaf(cb, dzb, z1);
  pot = pk2(p0, p1);
  gx = pk2(x0, x1);
  gy = pk2(y0, y1);
  gz = pk2(z0, z1);
}

// FP32 near field (c = 1 or 2) with the neighbour cells staged by the Tensor Memory
// Accelerator's bulk copies (cp.async.bulk, global -> shared, completion counted in
// bytes on an mbarrier).  Per item the warp lists its (2c+1)^3 neighbour
// cells -- the target's own cell first, then the others in (z, y, x) order --
// numbers their source pairs consecutively and streams them through two
// shared-memory buffers of NT_CAP pairs: a buffer is filled by one bulk copy per
// cell piece (issued by the lane that owns the cell) and completes on its
// mbarrier; the warp waits for it (bounded), moves the staged sources of the
// neighbour cells into the target cell's frame (one packed add per coordinate),
// sweeps the whole chunk with the target fixed (the own cell's pairs, which hold
// the self pair, separately), and refills the buffer with the chunk after next
// while the other buffer's copies are in flight.  A wait that runs out
// raises the device error flag (PMMM_ERR_TIMEOUT), waits once more (bounded) for
// the copies it issued and leaves the kernel.
// Source pairs per buffer (a multiple of 4) and resident blocks per SM, within 227 KB of
// shared memory.  The per-chunk work (wait, copies, shifts of the cells that begin or end
// in it) favours long chunks, the sweeps' latency more blocks.  Near field of 2^20 /
// 32^3 and 2^24 / 64^3 (c = 1), 2^20 / 32^3 (c = 2): 64 pairs, 6 blocks 557 us, 14.6 ms,
// 2.81 ms; 96, 6: 541, 14.3, 2.70; 128, 5: 528, 13.9, 2.62; 160, 5: 518, 13.8, 2.58;
// 192, 4: 549, 14.4, 2.50; 256, 3: 563, 14.3, 2.54.
template <int CUT> constexpr int nt_cap() { return CUT <= 1 ? 160 : 192; }
template <int CUT> constexpr int nt_blocks_per_sm() { return CUT <= 1 ? 5 : 4; }
constexpr long long NT_WAIT_POLLS = 1 << 20;  // polls of at most 1 us each

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void bar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// One step of two sources (pair record A = {x_a, x_b, y_a, y_b}, B = {z_a, z_b,
// q_a, q_b}) for one target, on float2 values with the packed FP32 operations
// (each half an IEEE fp32 operation: t - s is formed as fma(s, -1, t), exactly
// the rounded difference).  The same 13 packed operations and 2 rsqrt for every
// two sources as the per-target kernel's step.
template <bool SELF>
__device__ __forceinline__ void pp_pair_v(const float4& A, const float4& B, float2 tx, float2 ty, float2 tz,
                                          float2& pot, float2& gx, float2& gy, float2& gz) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const float2 dx = __ffma2_rn(make_float2(A.x, A.y), m1, tx);
  const float2 dy = __ffma2_rn(make_float2(A.z, A.w), m1, ty);
  const float2 dz = __ffma2_rn(make_float2(B.x, B.y), m1, tz);
  const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
  float ra = rsqrt_ftz(r2.x), rb = rsqrt_ftz(r2.y);
  if (SELF) {
    ra = r2.x > 0.f ? ra : 0.f;
    rb = r2.y > 0.f ? rb : 0.f;
  }
  const float2 ri = make_float2(ra, rb);
  const float2 qr = __fmul2_rn(make_float2(B.z, B.w), ri);
  pot = __fadd2_rn(pot, qr);
  const float2 qr3 = __fmul2_rn(qr, __fmul2_rn(ri, ri));
  gx = __ffma2_rn(qr3, dx, gx);
  gy = __ffma2_rn(qr3, dy, gy);
  gz = __ffma2_rn(qr3, dz, gz);
}

// Sweep of npair (a multiple of 4) staged source pairs: all of them for SP = 1, the
// pairs ph, ph + SP, ... of this lane's source phase otherwise.
template <bool SELF>
__device__ __forceinline__ void pp_sweep(const float4* __restrict__ src, int npair, int ph, int SP, float2 tx,
                                         float2 ty, float2 tz, float2& pot, float2& gx, float2& gy, float2& gz) {
  if (SP == 1) {
    int j = 0;
    for (; j + 8 <= npair; j += 8) {
      float4 A[8], B[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        A[u] = src[2 * (j + u)];
        B[u] = src[2 * (j + u) + 1];
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) pp_pair_v<SELF>(A[u], B[u], tx, ty, tz, pot, gx, gy, gz);
    }
    for (; j < npair; j += 4) {
      const float4 A0 = src[2 * j], B0 = src[2 * j + 1], A1 = src[2 * j + 2], B1 = src[2 * j + 3];
      const float4 A2 = src[2 * j + 4], B2 = src[2 * j + 5], A3 = src[2 * j + 6], B3 = src[2 * j + 7];
      pp_pair_v<SELF>(A0, B0, tx, ty, tz, pot, gx, gy, gz);
      pp_pair_v<SELF>(A1, B1, tx, ty, tz, pot, gx, gy, gz);
      pp_pair_v<SELF>(A2, B2, tx, ty, tz, pot, gx, gy, gz);
      pp_pair_v<SELF>(A3, B3, tx, ty, tz, pot, gx, gy, gz);
    }
  } else {
    int j = ph;
    for (; j + 3 * SP < npair; j += 4 * SP) {
      float4 A[4], B[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        A[u] = src[2 * (j + u * SP)];
        B[u] = src[2 * (j + u * SP) + 1];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) pp_pair_v<SELF>(A[u], B[u], tx, ty, tz, pot, gx, gy, gz);
    }
    for (; j + SP < npair; j += 2 * SP) {
      const float4 A0 = src[2 * j], B0 = src[2 * j + 1], A1 = src[2 * (j + SP)], B1 = src[2 * (j + SP) + 1];
      pp_pair_v<SELF>(A0, B0, tx, ty, tz, pot, gx, gy, gz);
      pp_pair_v<SELF>(A1, B1, tx, ty, tz, pot, gx, gy, gz);
    }
    if (j < npair) pp_pair_v<SELF>(src[2 * j], src[2 * j + 1], tx, ty, tz, pot, gx, gy, gz);
  }
}

template <int CUT>
__global__ void __launch_bounds__(PP_WARPS * 32, nt_blocks_per_sm<CUT>()) pp_kernel_tma(
    const float* __restrict__ part, const float* __restrict__ src2f, const uint32_t* __restrict__ pair_start,
    const uint32_t* __restrict__ vals, const int* __restrict__ cs, int64_t K, const uint32_t* __restrict__ item_start,
    const uint32_t* __restrict__ item_cell, unsigned int* __restrict__ counter, const float* __restrict__ far,
    PPParams pp, float* __restrict__ phi, float* __restrict__ force, double* __restrict__ epart,
    int* __restrict__ err, float4* __restrict__ near_out) {
  constexpr int W = 2 * CUT + 1, NS = W * W * W, SL = (NS + 31) / 32, SELFK = (NS - 1) / 2;
  constexpr int NT_CAP = nt_cap<CUT>();
  __shared__ __align__(128) float4 sbuf[PP_WARPS][2][2 * NT_CAP];
  __shared__ __align__(8) unsigned long long sbar[PP_WARPS][2];
  __shared__ uint32_t soff[PP_WARPS][NS];  // cell offset of the r-th non-empty segment, a signed byte per axis
  const float4* P = reinterpret_cast<const float4*>(part);
  const char* S2 = reinterpret_cast<const char*>(src2f);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t bar0 = tc::smem_u32(&sbar[warp][0]), bar1 = tc::smem_u32(&sbar[warp][1]);
  const uint32_t buf0 = tc::smem_u32(&sbuf[warp][0][0]), buf1 = tc::smem_u32(&sbuf[warp][1][0]);
  if (lane == 0) {
    tc::bar_init(bar0, 1);
    tc::bar_init(bar1, 1);
    tc::fence_proxy_async();
  }
  __syncwarp();
  uint32_t parity = 0;  // bit b: parity of the next phase of buffer b
  const uint32_t nitems = item_start[K];
  const int nx = pp.n[0], ny = pp.n[1], nz = pp.n[2];
  const float csx = pp.cs32[0], csy = pp.cs32[1], csz = pp.cs32[2];
  uint32_t item = 0;
  bool again = false;  // the same item once more, r = 0 masked in every cell (below)
  for (;;) {
    if (!again) {
      if (lane == 0) item = atomicAdd(counter, 1u);  // one item per atomic: the shortest tail
      item = __shfl_sync(0xffffffffu, item, 0);
    }
    if (item >= nitems) break;  // warp-uniform
    const int cell = (int)item_cell[item];
    const int chunk = (int)(item - item_start[cell]);
    const int tbeg = cs[cell] + chunk * CHUNK;
    const int R = min(CHUNK, cs[cell + 1] - tbeg);
    int TL = 1;
    while (TL < R) TL <<= 1;
    const int SP = 32 / TL;
    const int tl = lane & (TL - 1), ph = lane / TL;
    const bool active = tl < R;
    float4 xi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (active) xi = P[tbeg + tl];
    const int sbase = cell - cell % pp.ksys, lc = cell - sbase;
    const int ix = lc % nx, iy = (lc / nx) % ny, iz = lc / (nx * ny);
    // segment s (lane s % 32, slot s / 32): the own cell for s = 0, then the other
    // cells k = s - 1 (k >= SELFK: s) of the (2c+1)^3 block, x fastest: first pair
    // (global), pair count, first pair in the item's numbering, and the shift that
    // moves the cell's sources into the target cell's frame.  The numbering pads the
    // own cell and the whole list to multiples of 4 pairs with zero-charge dummies.
    int gb[SL], gn[SL], gf[SL], nfull = 0;
#pragma unroll
    for (int j = 0; j < SL; ++j) {
      const int sg = lane + 32 * j;
      gb[j] = gn[j] = 0;
      uint32_t ofs = 0;
      if (sg < NS) {
        const int kk = sg == 0 ? SELFK : (sg - 1 >= SELFK ? sg : sg - 1);
        const int dx = kk % W - CUT, dy = (kk / W) % W - CUT, dz = kk / (W * W) - CUT;
        int jx = ix + dx, jy = iy + dy, jz = iz + dz;
        bool ok = true;
        if (jx < 0 || jx >= nx) { ok = ok && pp.periodic; jx += (jx < 0) ? nx : -nx; }
        if (jy < 0 || jy >= ny) { ok = ok && pp.periodic; jy += (jy < 0) ? ny : -ny; }
        if (jz < 0 || jz >= nz) { ok = ok && pp.periodic; jz += (jz < 0) ? nz : -nz; }
        if (ok) {
          const int cj = sbase + jx + nx * (jy + ny * jz);
          gb[j] = (int)__ldg(pair_start + cj);
          gn[j] = (int)__ldg(pair_start + cj + 1) - gb[j];
        }
        ofs = (uint32_t)(dx & 255) | ((uint32_t)(dy & 255) << 8) | ((uint32_t)(dz & 255) << 16);
      }
      const uint32_t full = __ballot_sync(0xffffffffu, gn[j] > 0);
      if (gn[j] > 0) soff[warp][nfull + __popc(full & ((1u << lane) - 1u))] = ofs;
      nfull += __popc(full);
    }
    const int nself = __shfl_sync(0xffffffffu, gn[0], 0);
    const int nselfp = (nself + 3) & ~3;  // own cell, padded: [0, nselfp)
    int total = 0;
#pragma unroll
    for (int j = 0; j < SL; ++j) {
      const int w = (j == 0 && lane == 0) ? nselfp : gn[j];
      int v = w;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
      }
      gf[j] = total + v - w;
      total += __shfl_sync(0xffffffffu, v, 31);
    }
    const int real_end = total;        // dummies of the tail: [real_end, total)
    total = (total + 3) & ~3;
    const int nch = (total + NT_CAP - 1) / NT_CAP;
    const int nmask = again ? total : nselfp;  // pairs swept with r = 0 masked
    // queues the copies of chunk ch into buffer b (real pairs only)
    auto issue = [&](int ch, int b) {
      const int base = ch * NT_CAP, end = min(base + NT_CAP, total);
      const int dummies = max(0, min(end, nselfp) - max(base, nself)) + max(0, end - max(base, real_end));
      const uint32_t bar = b ? bar1 : bar0, dst = b ? buf1 : buf0;
      if (lane == 0) bar_expect_tx(bar, (uint32_t)(end - base - dummies) * 32u);
      __syncwarp();
      tc::fence_proxy_async();
#pragma unroll
      for (int j = 0; j < SL; ++j) {
        const int lo = max(gf[j], base), hi = min(gf[j] + gn[j], end);
        if (hi > lo)
          bulk_g2s(dst + 32u * (uint32_t)(lo - base), S2 + 32 * ((int64_t)gb[j] + (lo - gf[j])),
                   32u * (uint32_t)(hi - lo), bar);
      }
    };
    for (int c0 = 0; c0 < 2 && c0 < nch; ++c0) issue(c0, c0);
    float2 pot = make_float2(0.f, 0.f), gx = pot, gy = pot, gz = pot;
    const float2 tx = make_float2(xi.x, xi.x), ty = make_float2(xi.y, xi.y), tz = make_float2(xi.z, xi.z);
    int nbeg = 0;  // non-empty segments that begin before the current group of 32 pairs
    bool ok = true;
    for (int ch = 0; ch < nch; ++ch) {
      const int b = ch & 1;
      const uint32_t bar = b ? bar1 : bar0;
      const bool done = tc::bar_wait(bar, (parity >> b) & 1u, NT_WAIT_POLLS);
      if (!__all_sync(0xffffffffu, done)) {
        if (lane == 0) set_err(err, ERRBIT_TIMEOUT);
        tc::bar_wait(bar, (parity >> b) & 1u, NT_WAIT_POLLS);
        if (ch + 1 < nch) tc::bar_wait(b ? bar0 : bar1, (parity >> (b ^ 1)) & 1u, NT_WAIT_POLLS);
        ok = false;
        break;
      }
      parity ^= 1u << b;
      float4* buf = &sbuf[warp][b][0];
      const int base = ch * NT_CAP, end = min(base + NT_CAP, total);
      // dummies: zero charge far outside every cell (they add exact zeros)
      const float4 far4 = make_float4(1.0e4f, 1.0e4f, 1.0e4f, 1.0e4f), farq = make_float4(1.0e4f, 1.0e4f, 0.f, 0.f);
      for (int e = max(base, nself) + lane; e < min(end, nselfp); e += 32) {
        buf[2 * (e - base)] = far4;
        buf[2 * (e - base) + 1] = farq;
      }
      for (int e = max(base, real_end) + lane; e < end; e += 32) {
        buf[2 * (e - base)] = far4;
        buf[2 * (e - base) + 1] = farq;
      }
      // the neighbour cells' sources of this chunk moved into the target cell's frame, 32
      // pairs at a time whatever their cells: the segment of a pair is the number of
      // segments that begin at or before it (one pass per segment, half of its lanes idle
      // at 16 pairs per cell: 2^20 / 32^3 518 us, c = 2 2.50 ms against 494 us, 2.30 ms)
      for (int e0 = base; e0 < end; e0 += 32) {
        uint32_t begins = 0;
#pragma unroll
        for (int j = 0; j < SL; ++j)
          if (gn[j] > 0 && (uint32_t)(gf[j] - e0) < 32u) begins |= 1u << (gf[j] - e0);
        begins = __reduce_or_sync(0xffffffffu, begins);
        const int e = e0 + lane, r = nbeg + __popc(begins & (0xffffffffu >> (31 - lane))) - 1;
        nbeg += __popc(begins);
        if (e >= nselfp && e < min(end, real_end)) {
          const uint32_t ofs = soff[warp][r];
          const float sx = (float)(signed char)(ofs & 255u) * csx, sy = (float)(signed char)((ofs >> 8) & 255u) * csy,
                      sz = (float)(signed char)((ofs >> 16) & 255u) * csz;
          float4 A = buf[2 * (e - base)], B = buf[2 * (e - base) + 1];
          A.x += sx;
          A.y += sx;
          A.z += sy;
          A.w += sy;
          B.x += sz;
          B.y += sz;
          buf[2 * (e - base)] = A;
          buf[2 * (e - base) + 1] = B;
        }
      }
      __syncwarp();
      // own-cell pairs (self pair masked), then the rest of the chunk in one sweep
      const int s1 = min(max(nmask - base, 0), end - base);
      if (s1 > 0) pp_sweep<true>(buf, s1, ph, SP, tx, ty, tz, pot, gx, gy, gz);
      if (end - base > s1) pp_sweep<false>(buf + 2 * s1, end - base - s1, ph, SP, tx, ty, tz, pot, gx, gy, gz);
      __syncwarp();  // every lane is done with buffer b
      if (ch + 2 < nch) issue(ch + 2, b);
    }
    if (!__all_sync(0xffffffffu, ok)) return;
    // r = 0 is masked in the own cell, which holds the self pair.  A pair across a cell face
    // that coincides after the rounding of its coordinates leaves the potential's sum infinite
    // or NaN; the item then runs a second time with every cell masked
    again = !again && !__all_sync(0xffffffffu, !active || isfinite(pot.x + pot.y));
    if (again) continue;
    float ps = pot.x + pot.y, gxs = -(gx.x + gx.y), gys = -(gy.x + gy.y), gzs = -(gz.x + gz.y);
    for (int o = TL; o < 32; o <<= 1) {
      ps += __shfl_xor_sync(0xffffffffu, ps, o);
      gxs += __shfl_xor_sync(0xffffffffu, gxs, o);
      gys += __shfl_xor_sync(0xffffffffu, gys, o);
      gzs += __shfl_xor_sync(0xffffffffu, gzs, o);
    }
    // near sums in units of 1 / hs and 1 / hs^2, each product rounded on its own
    // (no contraction with the far-field addition), so that the split evaluation,
    // which stores them and adds the far field later, gives the same results
    const float np0 = __fmul_rn(ps, pp.ih32), np1 = __fmul_rn(gxs, pp.ih2_32), np2 = __fmul_rn(gys, pp.ih2_32),
                np3 = __fmul_rn(gzs, pp.ih2_32);
    if (near_out) {  // split evaluation: the near sums only, combined later by pp_combine_kernel
      if (active && ph == 0) near_out[tbeg + tl] = make_float4(np0, np1, np2, np3);
      continue;
    }
    float e_t = 0.f, f_t[3] = {0.f, 0.f, 0.f};
    if (active && ph == 0) {
      const int s = tbeg + tl;
      const float4 fr = reinterpret_cast<const float4*>(far)[s];
      const float sg = pp.sign32;
      const float pt = sg * (fr.x + np0);
      const float g0 = sg * (fr.y + np1), g1 = sg * (fr.z + np2), g2 = sg * (fr.w + np3);
      const uint32_t o = vals[s];
      const float q = xi.w;
      if (phi) phi[o] = pt;
      if (force) {
        force[3 * (int64_t)o + 0] = -q * g0;
        force[3 * (int64_t)o + 1] = -q * g1;
        force[3 * (int64_t)o + 2] = -q * g2;
      }
      e_t = 0.5f * q * pt;
      f_t[0] = -q * g0;
      f_t[1] = -q * g1;
      f_t[2] = -q * g2;
    }
    if (!epart) continue;  // no energy asked for
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e_t += __shfl_xor_sync(0xffffffffu, e_t, o);
      f_t[0] += __shfl_xor_sync(0xffffffffu, f_t[0], o);
      f_t[1] += __shfl_xor_sync(0xffffffffu, f_t[1], o);
      f_t[2] += __shfl_xor_sync(0xffffffffu, f_t[2], o);
    }
    if (lane == 0) {
      epart[(int64_t)item * 4 + 0] = (double)e_t;
      epart[(int64_t)item * 4 + 1] = (double)f_t[0];
      epart[(int64_t)item * 4 + 2] = (double)f_t[1];
      epart[(int64_t)item * 4 + 3] = (double)f_t[2];
    }
  }
}

// Combination of a split FP32 evaluation, where the near field ran beside the far
// field and left its sums (potential, gradient, in units of 1 / hs and 1 / hs^2)
// in near_out: one warp per work item, lane = target, the same combination,
// caller-order stores and per-item energy and net-force partials as the
// epilogue of pp_kernel_tma.
__global__ void __launch_bounds__(256) pp_combine_kernel(const float4* __restrict__ part,
                                                         const uint32_t* __restrict__ vals, const int* __restrict__ cs,
                                                         int64_t K, const uint32_t* __restrict__ item_start,
                                                         const uint32_t* __restrict__ item_cell,
                                                         const float4* __restrict__ far,
                                                         const float4* __restrict__ nearv, PPParams pp,
                                                         float* __restrict__ phi, float* __restrict__ force,
                                                         double* __restrict__ epart) {
  const int lane = threadIdx.x & 31;
  const uint32_t nitems = item_start[K];
  const uint32_t wstride = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t item = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; item < nitems; item += wstride) {
    const int cell = (int)item_cell[item];
    const int tbeg = cs[cell] + (int)(item - item_start[cell]) * CHUNK;
    const int R = min(CHUNK, cs[cell + 1] - tbeg);
    float e_t = 0.f, f_t[3] = {0.f, 0.f, 0.f};
    if (lane < R) {
      const int s = tbeg + lane;
      const float4 fr = far[s], nr = nearv[s];
      const float sg = pp.sign32;
      const float pt = sg * (fr.x + nr.x);
      const float g0 = sg * (fr.y + nr.y), g1 = sg * (fr.z + nr.z), g2 = sg * (fr.w + nr.w);
      const uint32_t o = vals[s];
      const float q = part[s].w;
      if (phi) phi[o] = pt;
      if (force) {
        force[3 * (int64_t)o + 0] = -q * g0;
        force[3 * (int64_t)o + 1] = -q * g1;
        force[3 * (int64_t)o + 2] = -q * g2;
      }
      e_t = 0.5f * q * pt;
      f_t[0] = -q * g0;
      f_t[1] = -q * g1;
      f_t[2] = -q * g2;
    }
    if (!epart) continue;  // no energy asked for
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e_t += __shfl_xor_sync(0xffffffffu, e_t, o);
      f_t[0] += __shfl_xor_sync(0xffffffffu, f_t[0], o);
      f_t[1] += __shfl_xor_sync(0xffffffffu, f_t[1], o);
      f_t[2] += __shfl_xor_sync(0xffffffffu, f_t[2], o);
    }
    if (lane == 0) {
      epart[(int64_t)item * 4 + 0] = (double)e_t;
      epart[(int64_t)item * 4 + 1] = (double)f_t[0];
      epart[(int64_t)item * 4 + 2] = (double)f_t[1];
      epart[(int64_t)item * 4 + 3] = (double)f_t[2];
    }
  }
}

constexpr int PPS_THREADS = 256;

// The end of a per-target evaluation for sorted target i (cell, near sums nr in device
// units): adds the far field, each sum in one rounding, stores the results in the caller's order and reduces the energy and
// net-force terms per work item -- a segmented warp scan over lanes of equal item, one
// store per item that lies inside the warp, and two double atomics (commutative, so
// deterministic) on a zeroed slot for an item split between two warps.  Called by whole
// warps (i >= n: no target).
__device__ __forceinline__ void target_epilogue(int64_t i, int64_t n, int cell, float4 nr,
                                                const float4* __restrict__ P, const uint32_t* __restrict__ vals,
                                                const int* __restrict__ cs, const uint32_t* __restrict__ item_start,
                                                const float4* __restrict__ far, const PPParams& pp,
                                                float* __restrict__ phi, float* __restrict__ force,
                                                double* __restrict__ epart) {
  const int lane = threadIdx.x & 31;
  const int64_t wbase = i - lane;
  float e_t = 0.f, f_t0 = 0.f, f_t1 = 0.f, f_t2 = 0.f;
  uint32_t item = 0xffffffffu;
  int64_t tb = 0, te = 0;
  if (i < n) {
    const int c0 = cs[cell], c1 = cs[cell + 1];
    const int chunk = (int)((i - c0) / CHUNK);
    item = item_start[cell] + (uint32_t)chunk;
    tb = c0 + (int64_t)chunk * CHUNK;
    te = min(tb + CHUNK, (int64_t)c1);
    const float4 fr = far[i];
    const float sg = pp.sign32, q = P[i].w;
    const float pt = sg * fmaf(nr.x, pp.ih32, fr.x);
    const float g0 = sg * fmaf(nr.y, pp.ih2_32, fr.y), g1 = sg * fmaf(nr.z, pp.ih2_32, fr.z),
                g2 = sg * fmaf(nr.w, pp.ih2_32, fr.w);
    const uint32_t o = vals[i];
    if (phi) phi[o] = pt;
    if (force) {
      force[3 * (int64_t)o + 0] = -q * g0;
      force[3 * (int64_t)o + 1] = -q * g1;
      force[3 * (int64_t)o + 2] = -q * g2;
    }
    e_t = 0.5f * q * pt;
    f_t0 = -q * g0;
    f_t1 = -q * g1;
    f_t2 = -q * g2;
  }
  if (!epart) return;  // no energy asked for
  // segmented inclusive scan over runs of lanes with the same item
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float ue = __shfl_up_sync(0xffffffffu, e_t, o), u0 = __shfl_up_sync(0xffffffffu, f_t0, o);
    const float u1 = __shfl_up_sync(0xffffffffu, f_t1, o), u2 = __shfl_up_sync(0xffffffffu, f_t2, o);
    const uint32_t uit = __shfl_up_sync(0xffffffffu, item, o);
    if (lane >= o && uit == item) {
      e_t += ue;
      f_t0 += u0;
      f_t1 += u1;
      f_t2 += u2;
    }
  }
  const uint32_t next = __shfl_down_sync(0xffffffffu, item, 1);
  if (i < n && (lane == 31 || next != item)) {
    double* ep = epart + 4 * (int64_t)item;
    if (tb >= wbase && te <= wbase + 32) {
      ep[0] = (double)e_t;
      ep[1] = (double)f_t0;
      ep[2] = (double)f_t1;
      ep[3] = (double)f_t2;
    } else {
      atomicAdd(ep + 0, (double)e_t);
      atomicAdd(ep + 1, (double)f_t0);
      atomicAdd(ep + 2, (double)f_t1);
      atomicAdd(ep + 3, (double)f_t2);
    }
  }
}

// FP32 near field (c = 1 or 2) with one thread per target: for sparsely filled cells,
// where the per-item set-up of the cell-item kernels costs more than the
// interactions.  Thread i takes sorted target i; it walks the (2c+1)^2 neighbour rows
// (dy, dz) and in each row the source pairs of its 2c+1 cells x-c .. x+c as one list,
// two pairs per step (sources of neighbouring targets coincide, so loads are served by
// L1).  One loop per row instead of one per cell: the lanes of a warp wait for each
// other 9 (25) times instead of 27 (125), and row totals of neighbouring targets, which
// share most of their cells, are more alike than cell counts.  A warp whose 32 targets
// lie in one cell (a crowded one) takes its sources through shared memory instead, 32
// pairs of a neighbour cell at a time: the broadcast loads then come from there, at
// twice the rate of L1, and need no per-lane addresses.  Same pairs in the same order
// with the same rounding.  Bound by latency and divergence where cells are sparse, by
// the pair step's operand reads (33 cycles per 64 pairs and SM quarter) where they are
// full.  Against one loop per cell and L1 loads throughout: 20011 particles / 16^3 29 ->
// 20 us; 10^6 / 64^3 195 -> 160 us; 5.6 million in 64 systems 1336 -> 1124 us; 2^20 in a
// Plummer sphere / 64^3 (3.5e10 pairs, up to 6300 particles per cell) 27.9 -> 18.4 ms.
// near_out (split evaluation): the near sums go there, pp_combine_target_kernel ends.

// Sums of one target over npair pairs whose words lie in sa and sb (shared memory).
template <bool SELF>
__device__ __forceinline__ void pp_staged(const float4* __restrict__ sa, const float4* __restrict__ sb, int npair,
                                          float2 tx, float2 ty, float2 tz, float2& pot, float2& gx, float2& gy,
                                          float2& gz) {
  int j = 0;
  for (; j + 4 <= npair; j += 4) {
    float4 A[4], B[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      A[u] = sa[j + u];
      B[u] = sb[j + u];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) pp_pair_v<SELF>(A[u], B[u], tx, ty, tz, pot, gx, gy, gz);
  }
  for (; j < npair; ++j) pp_pair_v<SELF>(sa[j], sb[j], tx, ty, tz, pot, gx, gy, gz);
}

// Adds the near sums of 32 targets of one cell (lane = target): pot, g of pp_target_kernel.
// mask_all (the same for all lanes): r = 0 adds zero in every cell, not in the own one alone.
template <int CUT>
__device__ __forceinline__ void pp_crowd_warp(const float4 xi, int sbase, int ix, int iy, int iz,
                                              const float4* __restrict__ S2, const uint32_t* __restrict__ pair_start,
                                              const PPParams& pp, bool mask_all, float4* sa, float4* sb, float2& pot,
                                              float2& gx, float2& gy, float2& gz) {
  const int lane = threadIdx.x & 31;
  for (int dz = -CUT; dz <= CUT; ++dz)
    for (int dy = -CUT; dy <= CUT; ++dy)
      for (int dx = -CUT; dx <= CUT; ++dx) {
        int jx = ix + dx, jy = iy + dy, jz = iz + dz;
        bool ok = true;
        if (jx < 0 || jx >= pp.n[0]) { ok = ok && pp.periodic; jx += (jx < 0) ? pp.n[0] : -pp.n[0]; }
        if (jy < 0 || jy >= pp.n[1]) { ok = ok && pp.periodic; jy += (jy < 0) ? pp.n[1] : -pp.n[1]; }
        if (jz < 0 || jz >= pp.n[2]) { ok = ok && pp.periodic; jz += (jz < 0) ? pp.n[2] : -pp.n[2]; }
        if (!ok) continue;
        const uint32_t* row = pair_start + sbase + jx + pp.n[0] * (jy + pp.n[1] * jz);
        const int pb = (int)__ldg(row), pe = (int)__ldg(row + 1);
        const float ux = xi.x - (float)dx * pp.cs32[0], uy = xi.y - (float)dy * pp.cs32[1],
                    uz = xi.z - (float)dz * pp.cs32[2];
        const float2 tx = make_float2(ux, ux), ty = make_float2(uy, uy), tz = make_float2(uz, uz);
        const bool mask = mask_all || (dx == 0 && dy == 0 && dz == 0);
        for (int p = pb; p < pe; p += 32) {
          const int m = min(32, pe - p);
          __syncwarp();
          if (lane < m) {
            sa[lane] = __ldg(S2 + 2 * (int64_t)(p + lane));
            sb[lane] = __ldg(S2 + 2 * (int64_t)(p + lane) + 1);
          }
          __syncwarp();
          if (mask)
            pp_staged<true>(sa, sb, m, tx, ty, tz, pot, gx, gy, gz);
          else
            pp_staged<false>(sa, sb, m, tx, ty, tz, pot, gx, gy, gz);
        }
      }
}

template <int CUT>
__global__ void __launch_bounds__(PPS_THREADS, 4) pp_target_kernel(
    const float4* __restrict__ P, const ulonglong2* __restrict__ S2, const uint32_t* __restrict__ pair_start,
    const uint32_t* __restrict__ keys, const uint32_t* __restrict__ vals, const int* __restrict__ cs,
    const uint32_t* __restrict__ item_start, int64_t n, const float4* __restrict__ far, PPParams pp,
    float* __restrict__ phi, float* __restrict__ force, double* __restrict__ epart, float4* __restrict__ near_out) {
  constexpr int W = 2 * CUT + 1;
  const int64_t i = (int64_t)blockIdx.x * PPS_THREADS + threadIdx.x;
  float4 nr = make_float4(0.f, 0.f, 0.f, 0.f);
  __shared__ float4 stage[PPS_THREADS / 32][2][32];
  const int mycell = i < n ? (int)keys[i] : -1;
  const int cell0 = __shfl_sync(0xffffffffu, mycell, 0);  // every lane takes part
  const bool crowd = __all_sync(0xffffffffu, mycell >= 0 && mycell == cell0);
  if (i < n) {
    const float4 xi = P[i];
    const int cell = mycell;
    const int nx = pp.n[0], ny = pp.n[1], nz = pp.n[2];
    const int sbase = cell - cell % pp.ksys, lc = cell - sbase;
    const int ix = lc % nx, iy = (lc / nx) % ny, iz = lc / (nx * ny);
    const float csx = pp.cs32[0], csy = pp.cs32[1], csz = pp.cs32[2];
    float pa = 0.f, pbv = 0.f, xa = 0.f, xb = 0.f, ya = 0.f, yb = 0.f, za = 0.f, zb = 0.f;
    if (crowd) {
      float2 pot = make_float2(0.f, 0.f), gx = pot, gy = pot, gz = pot;
      float4(*st)[32] = stage[threadIdx.x >> 5];
      // r = 0 is looked for in the own cell only (a compare and a select per source).  A pair
      // across a cell face can coincide too, after the rounding of its cell-relative
      // coordinates; its infinite term leaves the sum of the potential infinite or NaN, and
      // the warp then starts again with the test in every cell.
      for (bool mask_all = false;; mask_all = true) {
        pp_crowd_warp<CUT>(xi, sbase, ix, iy, iz, reinterpret_cast<const float4*>(S2), pair_start, pp, mask_all, st[0],
                           st[1], pot, gx, gy, gz);
        if (mask_all || __all_sync(0xffffffffu, isfinite(pot.x + pot.y))) break;
        pot = gx = gy = gz = make_float2(0.f, 0.f);
      }
      pa = pot.x; pbv = pot.y; xa = gx.x; xb = gx.y; ya = gy.x; yb = gy.y; za = gz.x; zb = gz.y;
    } else {
      f2 pot = pk2(0.f, 0.f), gx = pot, gy = pot, gz = pot;
      // the row's cells: x index (wrapped; -1 outside an open box) and the target's x there
      int jx[W];
      float txs[W];
#pragma unroll
      for (int d = 0; d < W; ++d) {
        jx[d] = ix + d - CUT;
        if (jx[d] < 0 || jx[d] >= nx) jx[d] = pp.periodic ? jx[d] + (jx[d] < 0 ? nx : -nx) : -1;
        txs[d] = xi.x - (float)(d - CUT) * csx;
      }
      for (int dz = -CUT; dz <= CUT; ++dz) {
        int jz = iz + dz;
        if (jz < 0 || jz >= nz) {
          if (!pp.periodic) continue;
          jz += (jz < 0) ? nz : -nz;
        }
        const float tzs = xi.z - (float)dz * csz;
        const f2 tz = pk2(tzs, tzs);
        for (int dy = -CUT; dy <= CUT; ++dy) {
          int jy = iy + dy;
          if (jy < 0 || jy >= ny) {
            if (!pp.periodic) continue;
            jy += (jy < 0) ? ny : -ny;
          }
          const float tys = xi.y - (float)dy * csy;
          const f2 ty = pk2(tys, tys);
          const uint32_t* row = pair_start + sbase + nx * (jy + ny * jz);
          // list position e of cell d's pairs: first[d] <= e < first[d + 1], pair e + off[d]
          int first[W], off[W], tot = 0;
#pragma unroll
          for (int d = 0; d < W; ++d) {
            const int b = jx[d] >= 0 ? (int)__ldg(row + jx[d]) : 0;
            const int m = jx[d] >= 0 ? (int)__ldg(row + jx[d] + 1) - b : 0;
            first[d] = tot;
            off[d] = b - tot;
            tot += m;
          }
          auto at = [&](int e, const ulonglong2*& src, f2& tx) {
            int o = off[0];
            float t = txs[0];
#pragma unroll
            for (int d = 1; d < W; ++d)
              if (e >= first[d]) {
                o = off[d];
                t = txs[d];
              }
            src = S2 + 2 * (int64_t)(e + o);
            tx = pk2(t, t);
          };
          const ulonglong2 *s0, *s1;
          f2 tx0, tx1;
          int e = 0;
          for (; e + 2 <= tot; e += 2) {
            at(e, s0, tx0);
            at(e + 1, s1, tx1);
            const ulonglong2 A0 = s0[0], B0 = s0[1], A1 = s1[0], B1 = s1[1];
            pp_pair2_mixed<true>(A0, B0, tx0, ty, tz, pot, gx, gy, gz);
            pp_pair2_mixed<true>(A1, B1, tx1, ty, tz, pot, gx, gy, gz);
          }
          if (e < tot) {
            at(e, s0, tx0);
            pp_pair2_mixed<true>(s0[0], s0[1], tx0, ty, tz, pot, gx, gy, gz);
          }
        }
      }
      up2(pot, pa, pbv);
      up2(gx, xa, xb);
      up2(gy, ya, yb);
      up2(gz, za, zb);
    }
    nr = make_float4(pa + pbv, -(xa + xb), -(ya + yb), -(za + zb));
  }
  if (near_out) {  // split evaluation: the near sums only, combined later by pp_combine_target_kernel
    if (i < n) near_out[i] = nr;
    return;
  }
  target_epilogue(i, n, mycell, nr, P, vals, cs, item_start, far, pp, phi, force, epart);
}

// Combination of a split evaluation with the per-target near field, one thread per
// sorted target.
__global__ void __launch_bounds__(PPS_THREADS) pp_combine_target_kernel(
    const float4* __restrict__ P, const uint32_t* __restrict__ keys, const uint32_t* __restrict__ vals,
    const int* __restrict__ cs, const uint32_t* __restrict__ item_start, int64_t n, const float4* __restrict__ far,
    const float4* __restrict__ nearv, PPParams pp, float* __restrict__ phi, float* __restrict__ force,
    double* __restrict__ epart) {
  const int64_t i = (int64_t)blockIdx.x * PPS_THREADS + threadIdx.x;
  const float4 nr = i < n ? nearv[i] : make_float4(0.f, 0.f, 0.f, 0.f);
  target_epilogue(i, n, i < n ? (int)keys[i] : -1, nr, P, vals, cs, item_start, far, pp, phi, force, epart);
}

}  // namespace

int64_t pp_items_max(int64_t K, int64_t n) { return K + (n + CHUNK - 1) / CHUNK + 1; }

int64_t pp_pairs_max(int64_t K, int64_t n) { return (n + K) / 2 + 1; }

bool pp_per_target_applies(bool fp64, int c) { return !fp64 && c <= 2; }

cudaError_t launch_pp_combine(bool per_target, const void* part, const uint32_t* keys, const uint32_t* vals, int64_t n,
                              const int* cell_start, int64_t K, const uint32_t* item_start, const uint32_t* item_cell,
                              int64_t max_items, const void* far, const void* nearv, PPParams pp, void* phi, void* force,
                              double* epart, cudaStream_t s, int* nl) {
  if (per_target) {
    if (n <= 0) return cudaSuccess;
    pp_combine_target_kernel<<<(unsigned)((n + PPS_THREADS - 1) / PPS_THREADS), PPS_THREADS, 0, s>>>(
        (const float4*)part, keys, vals, cell_start, item_start, n, (const float4*)far, (const float4*)nearv, pp,
        (float*)phi, (float*)force, epart);
    ++*nl;
    return cudaGetLastError();
  }
  if (max_items <= 0) return cudaSuccess;
  const int64_t blocks = (max_items + 7) / 8;  // 8 warps (items) per block, one item per warp
  pp_combine_kernel<<<(unsigned)blocks, 256, 0, s>>>((const float4*)part, vals, cell_start, K, item_start, item_cell,
                                                     (const float4*)far, (const float4*)nearv, pp, (float*)phi,
                                                     (float*)force, epart);
  ++*nl;
  return cudaGetLastError();
}

cudaError_t launch_pp(bool fp64, const void* part, const void* src2, const uint32_t* pair_start, const uint32_t* vals,
                      const uint32_t* keys, int64_t n, bool per_target, const int* cell_start, int64_t K,
                      const uint32_t* item_start, const uint32_t* item_cell, unsigned int* counter, int num_sms,
                      const void* far, PPParams pp, void* phi, void* force, double* epart, int* err, void* near_out,
                      cudaStream_t s, int* nl) {
  const int sms = num_sms > 0 ? num_sms : 1;
  if (fp64) {
    if (near_out) return cudaErrorInvalidValue;  // only the FP32 kernels split
#define PP64(C)                                                                                                    \
  pp64_kernel<C><<<(unsigned)(p64_blocks_per_sm(n, K) * sms), P64_THREADS, 0, s>>>((const double*)part, vals, cell_start, K, \
                                                                             item_start, item_cell, counter,       \
                                                                             (const double*)far, pp, (double*)phi, \
                                                                             (double*)force, epart)
    if (pp.c <= 1) PP64(1); else PP64(2);
#undef PP64
  } else if (per_target) {
    if (n <= 0) return cudaSuccess;
    const unsigned g = (unsigned)((n + PPS_THREADS - 1) / PPS_THREADS);
#define PP_TARGETS(C)                                                                                              \
  pp_target_kernel<C><<<g, PPS_THREADS, 0, s>>>((const float4*)part, (const ulonglong2*)src2, pair_start, keys, vals, \
                                                cell_start, item_start, n, (const float4*)far, pp, (float*)phi,    \
                                                (float*)force, epart, (float4*)near_out)
    if (pp.c <= 1) PP_TARGETS(1); else PP_TARGETS(2);
#undef PP_TARGETS
  } else {
    // persistent launch: nt_blocks_per_sm resident blocks of PP_WARPS warps per SM
#define PP_ITEMS(C)                                                                                                  \
  pp_kernel_tma<C><<<(unsigned)(nt_blocks_per_sm<C>() * sms), PP_WARPS * 32, 0, s>>>(                                \
      (const float*)part, (const float*)src2, pair_start, vals, cell_start, K, item_start, item_cell, counter,       \
      (const float*)far, pp, (float*)phi, (float*)force, epart, err, (float4*)near_out)
    if (pp.c <= 1) PP_ITEMS(1); else PP_ITEMS(2);
#undef PP_ITEMS
  }
  ++*nl;
  return cudaGetLastError();
}

}  // namespace pmmm
