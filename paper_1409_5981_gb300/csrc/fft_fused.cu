// Whole 3-D real FFT of one channel per CTA, for FP32 meshes whose half
// spectrum of the physical z planes fits in shared memory and whose transform
// lengths are at most 32 (32^3 periodic, 16^3 open and smaller).  Same
// transforms, layout and conventions as fft.cu (Sec. 2.1, App. C): spectra
// [channel][Lz][Ly][hx], forward exp(-2 pi i jk/L), inverse unnormalised.
//
//   forward: x pass (two real rows per complex transform) from global memory
//            into shared memory, rows y >= ny and planes z >= nz never stored;
//            y pass in place; z pass from shared memory straight to the spectrum.
//   inverse: z pass from the spectrum into shared memory (planes z < nz), y pass
//            in place (rows y < ny kept), x pass to the real rows x < nx.
// Every 1-D transform is held by one thread in registers; each channel is read and
// written once.  Two families: runtime sizes (fft3_fwd_kernel, fft3_inv_kernel: radix-2
// decimation-in-frequency FFTs, twiddles broadcast from shared memory, output in
// bit-reversed order, reindexed at the store), for non-cubic meshes whose channels fill
// the GPU; and cubes of 8, 16 or 32 cells with every size and twiddle a compile-time
// constant (fft3_cube_fwd_kernel, fft3_cube_inv_kernel, below), for any number of
// channels.  Only cubes, because the axis lengths of 4 to 32, padded or not, combine to
// more than a hundred instances of each kernel.
#include "fft.cuh"
#include "internal.cuh"

namespace pmmm {

namespace {

constexpr int FF_MAX_L = 32;

template <int L>
__host__ __device__ constexpr int bitrev(int k) {
  int r = 0;
  for (int b = 1, m = L >> 1; b < L; b <<= 1, m >>= 1)
    if (k & b) r |= m;
  return r;
}

__device__ __forceinline__ float2 cmul(float2 a, float2 w) {
  return make_float2(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x);
}

// In-register DIF FFT; on return v[bitrev(k)] holds X_k.  tw[t] = exp(-2 pi i t / L);
// the inverse uses the conjugates.
template <int L, bool INV>
__device__ __forceinline__ void fft_reg(float2 (&v)[L], const float2* __restrict__ tw) {
#pragma unroll
  for (int half = L / 2; half >= 1; half >>= 1) {
    const int ts = L / (2 * half);
#pragma unroll
    for (int b = 0; b < L; b += 2 * half) {
#pragma unroll
      for (int j = 0; j < half; ++j) {
        const float2 a = v[b + j], c = v[b + j + half];
        v[b + j] = make_float2(a.x + c.x, a.y + c.y);
        const float2 d = make_float2(a.x - c.x, a.y - c.y);
        if (j == 0) {
          v[b + j + half] = d;
        } else {
          float2 w = tw[j * ts];
          if (INV) w.y = -w.y;
          v[b + j + half] = cmul(d, w);
        }
      }
    }
  }
}

struct FFArgs {
  int nx, ny, nz, Lx, Ly, Lz, hx;
  int64_t Kh;
};

// ---------------------------------------------------------------- forward passes
template <int LX>
__device__ __forceinline__ void fwd_x(const float* __restrict__ src, float2* S, const FFArgs& a, int pr,
                                      const float2* tw) {
  const int nrows = a.nz * a.ny;
  const int r0 = 2 * pr, r1 = r0 + 1;
  const bool has1 = r1 < nrows;
  float2 v[LX];
#pragma unroll
  for (int t = 0; t < LX; ++t) v[t] = make_float2(0.f, 0.f);
  const float* p0 = src + (int64_t)r0 * a.nx;
  const float* p1 = src + (int64_t)r1 * a.nx;
  if ((a.nx & 3) == 0) {
#pragma unroll
    for (int t = 0; t < LX; t += 4) {
      if (t < a.nx) {
        const float4 x0 = *reinterpret_cast<const float4*>(p0 + t);
        const float4 x1 = has1 ? *reinterpret_cast<const float4*>(p1 + t) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[t] = make_float2(x0.x, x1.x);
        if (t + 1 < LX) v[t + 1] = make_float2(x0.y, x1.y);
        if (t + 2 < LX) v[t + 2] = make_float2(x0.z, x1.z);
        if (t + 3 < LX) v[t + 3] = make_float2(x0.w, x1.w);
      }
    }
  } else {
#pragma unroll
    for (int t = 0; t < LX; ++t)
      if (t < a.nx) v[t] = make_float2(p0[t], has1 ? p1[t] : 0.f);
  }
  fft_reg<LX, false>(v, tw);
  const int z0 = r0 / a.ny, y0 = r0 - z0 * a.ny, z1 = r1 / a.ny, y1 = r1 - z1 * a.ny;
  float2* o0 = S + ((int64_t)z0 * a.Ly + y0) * a.hx;
  float2* o1 = S + ((int64_t)z1 * a.Ly + y1) * a.hx;
#pragma unroll
  for (int k = 0; k <= LX / 2; ++k) {
    const float2 Z = v[bitrev<LX>(k)], Zm = v[bitrev<LX>((LX - k) & (LX - 1))];
    // X = (Z + conj Z_-k) / 2 ;  Y = (Z - conj Z_-k) / (2i)
    o0[k] = make_float2(0.5f * (Z.x + Zm.x), 0.5f * (Z.y - Zm.y));
    if (has1) o1[k] = make_float2(0.5f * (Z.y + Zm.y), -0.5f * (Z.x - Zm.x));
  }
}

template <int LY>
__device__ __forceinline__ void fwd_y(float2* S, const FFArgs& a, int col, const float2* tw) {
  const int z = col / a.hx, x = col - z * a.hx;
  float2* base = S + (int64_t)z * a.Ly * a.hx + x;
  float2 v[LY];
#pragma unroll
  for (int t = 0; t < LY; ++t) v[t] = t < a.ny ? base[t * a.hx] : make_float2(0.f, 0.f);
  fft_reg<LY, false>(v, tw);
#pragma unroll
  for (int t = 0; t < LY; ++t) base[t * a.hx] = v[bitrev<LY>(t)];
}

template <int LZ>
__device__ __forceinline__ void fwd_z(const float2* S, float2* __restrict__ dst, const FFArgs& a, int col,
                                      const float2* tw) {
  const int64_t plane = (int64_t)a.Ly * a.hx;
  float2 v[LZ];
#pragma unroll
  for (int t = 0; t < LZ; ++t) v[t] = t < a.nz ? S[t * plane + col] : make_float2(0.f, 0.f);
  fft_reg<LZ, false>(v, tw);
#pragma unroll
  for (int t = 0; t < LZ; ++t) dst[t * plane + col] = v[bitrev<LZ>(t)];
}

// ---------------------------------------------------------------- inverse passes
template <int LZ>
__device__ __forceinline__ void inv_z(const float2* __restrict__ src, float2* S, const FFArgs& a, int col,
                                      const float2* tw) {
  const int64_t plane = (int64_t)a.Ly * a.hx;
  float2 v[LZ];
#pragma unroll
  for (int t = 0; t < LZ; ++t) v[t] = src[t * plane + col];
  fft_reg<LZ, true>(v, tw);
#pragma unroll
  for (int t = 0; t < LZ; ++t)
    if (t < a.nz) S[t * plane + col] = v[bitrev<LZ>(t)];
}

template <int LY>
__device__ __forceinline__ void inv_y(float2* S, const FFArgs& a, int col, const float2* tw) {
  const int z = col / a.hx, x = col - z * a.hx;
  float2* base = S + (int64_t)z * a.Ly * a.hx + x;
  float2 v[LY];
#pragma unroll
  for (int t = 0; t < LY; ++t) v[t] = base[t * a.hx];
  fft_reg<LY, true>(v, tw);
#pragma unroll
  for (int t = 0; t < LY; ++t)
    if (t < a.ny) base[t * a.hx] = v[bitrev<LY>(t)];
}

// Writes the real rows into `rows` (shared memory, nz*ny*nx floats) after the
// caller's barrier; the rows reuse the spectrum's storage.
template <int LX>
__device__ __forceinline__ void inv_x(const float2* S, float* rows, const FFArgs& a, int pr, const float2* tw) {
  const int nrows = a.nz * a.ny;
  const bool mine = 2 * pr < nrows;  // threads past the last pair only join the barrier
  if (!mine) pr = 0;
  const int r0 = 2 * pr, r1 = r0 + 1;
  const bool has1 = mine && r1 < nrows;
  const int z0 = r0 / a.ny, y0 = r0 - z0 * a.ny, z1 = r1 / a.ny, y1 = r1 - z1 * a.ny;
  const float2* i0 = S + ((int64_t)z0 * a.Ly + y0) * a.hx;
  const float2* i1 = S + ((int64_t)z1 * a.Ly + y1) * a.hx;
  float2 v[LX];
#pragma unroll
  for (int k = 0; k <= LX / 2; ++k) {
    const float2 A = i0[k], B = has1 ? i1[k] : make_float2(0.f, 0.f);
    // Z_k = A_k + i B_k, and Z_{L-k} = conj(A_k) + i conj(B_k) (Hermitian rows)
    v[k] = make_float2(A.x - B.y, A.y + B.x);
    if (k > 0 && k < LX / 2) v[LX - k] = make_float2(A.x + B.y, -A.y + B.x);
  }
  fft_reg<LX, true>(v, tw);
  __syncthreads();  // every thread has read its half spectra before the rows overwrite them
  // element x of row r is staged at r*nx + ((x + r/2) mod nx): the row pairs of
  // neighbouring threads start on different banks
  float* p0 = rows + (int64_t)r0 * a.nx;
  float* p1 = rows + (int64_t)r1 * a.nx;
  const int rot = pr & (a.nx - 1);
#pragma unroll
  for (int t = 0; t < LX; ++t)
    if (mine && t < a.nx) {
      const float2 z = v[bitrev<LX>(t)];
      const int xs = (t + rot) & (a.nx - 1);
      p0[xs] = z.x;
      if (has1) p1[xs] = z.y;
    }
}

#define FF_DISPATCH(L, CALL)             \
  switch (L) {                           \
    case 2: { constexpr int LL = 2; CALL; } break;   \
    case 4: { constexpr int LL = 4; CALL; } break;   \
    case 8: { constexpr int LL = 8; CALL; } break;   \
    case 16: { constexpr int LL = 16; CALL; } break; \
    case 32: { constexpr int LL = 32; CALL; } break; \
    default: break;                      \
  }

constexpr int FF_THREADS = 512;  // 128 registers per thread: the 32-point transforms stay in registers

__global__ void __launch_bounds__(FF_THREADS, 1) fft3_fwd_kernel(const float* __restrict__ in, float2* __restrict__ spec,
                                                                FFArgs a, const float2* __restrict__ twx,
                                                                const float2* __restrict__ twy,
                                                                const float2* __restrict__ twz) {
  extern __shared__ __align__(16) unsigned char ff_smem[];
  float2* tx = reinterpret_cast<float2*>(ff_smem);
  float2* ty = tx + FF_MAX_L;
  float2* tz = ty + FF_MAX_L;
  float2* S = tz + FF_MAX_L;
  const int tid = threadIdx.x;
  for (int t = tid; t < FF_MAX_L; t += blockDim.x) {
    if (t < a.Lx) tx[t] = twx[t];
    if (t < a.Ly) ty[t] = twy[t];
    if (t < a.Lz) tz[t] = twz[t];
  }
  __syncthreads();
  const int64_t c = blockIdx.x;
  const float* src = in + c * a.nz * a.ny * a.nx;
  const int npairs = (a.nz * a.ny + 1) / 2;
  for (int pr = tid; pr < npairs; pr += blockDim.x) FF_DISPATCH(a.Lx, fwd_x<LL>(src, S, a, pr, tx));
  __syncthreads();
  for (int col = tid; col < a.nz * a.hx; col += blockDim.x) FF_DISPATCH(a.Ly, fwd_y<LL>(S, a, col, ty));
  __syncthreads();
  float2* dst = spec + c * a.Kh;
  for (int col = tid; col < a.Ly * a.hx; col += blockDim.x) FF_DISPATCH(a.Lz, fwd_z<LL>(S, dst, a, col, tz));
}

__global__ void __launch_bounds__(FF_THREADS, 1) fft3_inv_kernel(const float2* __restrict__ spec, float* __restrict__ out,
                                                                FFArgs a, const float2* __restrict__ twx,
                                                                const float2* __restrict__ twy,
                                                                const float2* __restrict__ twz) {
  extern __shared__ __align__(16) unsigned char ff_smem[];
  float2* tx = reinterpret_cast<float2*>(ff_smem);
  float2* ty = tx + FF_MAX_L;
  float2* tz = ty + FF_MAX_L;
  float2* S = tz + FF_MAX_L;
  const int tid = threadIdx.x;
  for (int t = tid; t < FF_MAX_L; t += blockDim.x) {
    if (t < a.Lx) tx[t] = twx[t];
    if (t < a.Ly) ty[t] = twy[t];
    if (t < a.Lz) tz[t] = twz[t];
  }
  __syncthreads();
  const int64_t c = blockIdx.x;
  const float2* src = spec + c * a.Kh;
  for (int col = tid; col < a.Ly * a.hx; col += blockDim.x) FF_DISPATCH(a.Lz, inv_z<LL>(src, S, a, col, tz));
  __syncthreads();
  for (int col = tid; col < a.nz * a.hx; col += blockDim.x) FF_DISPATCH(a.Ly, inv_y<LL>(S, a, col, ty));
  __syncthreads();
  // x pass: one row pair per thread (npairs <= blockDim, see fft_fused_applies);
  // the real rows go to shared memory, then out with coalesced 16-byte stores
  float* rows = reinterpret_cast<float*>(S);
  FF_DISPATCH(a.Lx, inv_x<LL>(S, rows, a, tid, tx));
  __syncthreads();
  const int64_t nreal = (int64_t)a.nz * a.ny * a.nx;
  float* dst = out + c * nreal;
  const int nxm = a.nx - 1;
  auto staged = [&](int64_t i) {
    const int64_t r = i / a.nx;
    const int x = (int)(i - r * a.nx);
    return rows[r * a.nx + ((x + (int)(r >> 1)) & nxm)];
  };
  if ((nreal & 3) == 0 && (a.nx & 3) == 0) {
    for (int64_t i = tid; i < nreal / 4; i += blockDim.x)
      reinterpret_cast<float4*>(dst)[i] = make_float4(staged(4 * i), staged(4 * i + 1), staged(4 * i + 2),
                                                       staged(4 * i + 3));
  } else {
    for (int64_t i = tid; i < nreal; i += blockDim.x) dst[i] = staged(i);
  }
}

// ---------------------------------------------------------------- cubic meshes
// The same passes for N^3 cells in transforms of L = N or 2 N points per axis, sizes known
// at compile time: constant twiddles and strides, as many threads as the y pass has columns
// (one column per thread), the real rows staged in shared memory by 16-byte copies in both
// directions (a row per thread read from global memory touches 32 lines a load).  Row pairs
// are (r, r + N^2 / 2): lanes then store half spectra hx complex values apart, hx odd.
// Bound by the chain load, three shared-memory passes, store of each CTA (one per SM at
// 32^3); 4096 channels of 32^3: forward 433 -> 260 us, inverse 566 -> 293 us (1.1 GB each,
// 4.2 and 3.8 TB/s) against the runtime-size kernels above, whose y and z passes needed a
// second round for 32 of their 544 columns.
template <int L_, int N_>
struct Cube {
  static constexpr int L = L_, N = N_, HX = L / 2 + 1, PLANE = L * HX, PAIRS = N * N / 2, Q = N / 4;
  static constexpr int T = ((N * HX > PAIRS ? N * HX : PAIRS) + 31) / 32 * 32;
  static constexpr size_t SMEM = sizeof(float2) * N * PLANE;
  // 16-byte chunk q of real row r: rotated so that eight consecutive rows hit all banks
  __device__ static int slot(int r, int q) { return r * N + 4 * ((q + r / (32 / N)) & (Q - 1)); }
};

using cf = cpx<float>;

template <int L, int N>
__global__ void __launch_bounds__(Cube<L, N>::T) fft3_cube_fwd_kernel(const float* __restrict__ in,
                                                                      float2* __restrict__ spec) {
  using K = Cube<L, N>;
  constexpr int HX = K::HX, PLANE = K::PLANE;
  extern __shared__ __align__(16) unsigned char ff_smem[];
  cf* S = reinterpret_cast<cf*>(ff_smem);
  float* rows = reinterpret_cast<float*>(ff_smem);
  const int tid = threadIdx.x;
  const float* src = in + (int64_t)blockIdx.x * (N * N * N);
  for (int i = tid; i < N * N * K::Q; i += K::T) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(rows + K::slot(i / K::Q, i % K::Q));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src + 4 * i) : "memory");
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const bool mine = tid < K::PAIRS;
  const int r0 = mine ? tid : 0, r1 = r0 + K::PAIRS;
  {
    cf v[N], w[L];
#pragma unroll
    for (int q = 0; q < K::Q; ++q) {
      const float4 a = *reinterpret_cast<const float4*>(rows + K::slot(r0, q));
      const float4 b = *reinterpret_cast<const float4*>(rows + K::slot(r1, q));
      v[4 * q] = mk(a.x, b.x);
      v[4 * q + 1] = mk(a.y, b.y);
      v[4 * q + 2] = mk(a.z, b.z);
      v[4 * q + 3] = mk(a.w, b.w);
    }
    dft_pad<float, L, N, -1>(v, w);
    __syncthreads();  // every row has been read before the half spectra overwrite them
    if (mine) {
      cf* o0 = S + (r0 / N) * PLANE + (r0 % N) * HX;
      cf* o1 = S + (r1 / N) * PLANE + (r1 % N) * HX;
#pragma unroll
      for (int k = 0; k < HX; ++k) {
        const cf Z = w[k], Zm = w[(L - k) & (L - 1)];
        o0[k] = mk(0.5f * (Z.x + Zm.x), 0.5f * (Z.y - Zm.y));   // (Z + conj Z_-k) / 2
        o1[k] = mk(0.5f * (Z.y + Zm.y), -0.5f * (Z.x - Zm.x));  // (Z - conj Z_-k) / (2i)
      }
    }
  }
  __syncthreads();
  if (tid < N * HX) {
    cf* base = S + (tid / HX) * PLANE + tid % HX;
    cf v[N], w[L];
#pragma unroll
    for (int t = 0; t < N; ++t) v[t] = base[t * HX];
    dft_pad<float, L, N, -1>(v, w);
#pragma unroll
    for (int t = 0; t < L; ++t) base[t * HX] = w[t];
  }
  __syncthreads();
  cf* dst = reinterpret_cast<cf*>(spec) + (int64_t)blockIdx.x * (L * PLANE);
  for (int col = tid; col < PLANE; col += K::T) {
    cf v[N], w[L];
#pragma unroll
    for (int t = 0; t < N; ++t) v[t] = S[t * PLANE + col];
    dft_pad<float, L, N, -1>(v, w);
#pragma unroll
    for (int t = 0; t < L; ++t) dst[t * PLANE + col] = w[t];
  }
}

template <int L, int N>
__global__ void __launch_bounds__(Cube<L, N>::T) fft3_cube_inv_kernel(const float2* __restrict__ spec,
                                                                      float* __restrict__ out) {
  using K = Cube<L, N>;
  constexpr int HX = K::HX, PLANE = K::PLANE;
  extern __shared__ __align__(16) unsigned char ff_smem[];
  cf* S = reinterpret_cast<cf*>(ff_smem);
  float* rows = reinterpret_cast<float*>(ff_smem);
  const int tid = threadIdx.x;
  const cf* src = reinterpret_cast<const cf*>(spec) + (int64_t)blockIdx.x * (L * PLANE);
  for (int col = tid; col < PLANE; col += K::T) {
    cf v[L];
#pragma unroll
    for (int t = 0; t < L; ++t) v[t] = src[t * PLANE + col];
    dft_reg<float, L, 1>(v);
#pragma unroll
    for (int t = 0; t < N; ++t) S[t * PLANE + col] = v[t];
  }
  __syncthreads();
  if (tid < N * HX) {
    cf* base = S + (tid / HX) * PLANE + tid % HX;
    cf v[L];
#pragma unroll
    for (int t = 0; t < L; ++t) v[t] = base[t * HX];
    dft_reg<float, L, 1>(v);
#pragma unroll
    for (int t = 0; t < N; ++t) base[t * HX] = v[t];
  }
  __syncthreads();
  const bool mine = tid < K::PAIRS;
  const int r0 = mine ? tid : 0, r1 = r0 + K::PAIRS;
  {
    const cf* i0 = S + (r0 / N) * PLANE + (r0 % N) * HX;
    const cf* i1 = S + (r1 / N) * PLANE + (r1 % N) * HX;
    cf v[L];
#pragma unroll
    for (int k = 0; k < HX; ++k) {
      const cf A = i0[k], B = i1[k];
      // Z_k = A_k + i B_k, and Z_{L-k} = conj(A_k) + i conj(B_k) (Hermitian rows)
      v[k] = mk(A.x - B.y, A.y + B.x);
      if (k > 0 && k < L / 2) v[L - k] = mk(A.x + B.y, -A.y + B.x);
    }
    dft_reg<float, L, 1>(v);
    __syncthreads();  // every half spectrum has been read before the rows overwrite them
    if (mine) {
#pragma unroll
      for (int q = 0; q < K::Q; ++q) {
        *reinterpret_cast<float4*>(rows + K::slot(r0, q)) =
            make_float4(v[4 * q].x, v[4 * q + 1].x, v[4 * q + 2].x, v[4 * q + 3].x);
        *reinterpret_cast<float4*>(rows + K::slot(r1, q)) =
            make_float4(v[4 * q].y, v[4 * q + 1].y, v[4 * q + 2].y, v[4 * q + 3].y);
      }
    }
  }
  __syncthreads();
  float4* dst = reinterpret_cast<float4*>(out + (int64_t)blockIdx.x * (N * N * N));
  for (int i = tid; i < N * N * K::Q; i += K::T)
    dst[i] = *reinterpret_cast<const float4*>(rows + K::slot(i / K::Q, i % K::Q));
}

template <int L, int N>
cudaError_t cube_run(bool inverse, const void* in, void* out, int C, cudaStream_t s) {
  using K = Cube<L, N>;
  cudaError_t e = inverse ? cudaFuncSetAttribute(fft3_cube_inv_kernel<L, N>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::SMEM)
                          : cudaFuncSetAttribute(fft3_cube_fwd_kernel<L, N>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::SMEM);
  if (e != cudaSuccess) return e;
  if (inverse)
    fft3_cube_inv_kernel<L, N><<<(unsigned)C, K::T, K::SMEM, s>>>((const float2*)in, (float*)out);
  else
    fft3_cube_fwd_kernel<L, N><<<(unsigned)C, K::T, K::SMEM, s>>>((const float*)in, (float2*)out);
  return cudaGetLastError();
}

// cudaErrorNotSupported: not one of the compiled cubes
cudaError_t cube_launch(bool inverse, const void* in, void* out, const Dims& d, int C, cudaStream_t s) {
  if (fft_cube_applies(false, d)) {
    if (d.Lx == 32 && d.nx == 32) return cube_run<32, 32>(inverse, in, out, C, s);
    if (d.Lx == 16 && d.nx == 16) return cube_run<16, 16>(inverse, in, out, C, s);
    if (d.Lx == 8 && d.nx == 8) return cube_run<8, 8>(inverse, in, out, C, s);
    if (d.Lx == 32 && d.nx == 16) return cube_run<32, 16>(inverse, in, out, C, s);
    if (d.Lx == 16 && d.nx == 8) return cube_run<16, 8>(inverse, in, out, C, s);
  }
  return cudaErrorNotSupported;
}

size_t fused_smem(const Dims& d) { return sizeof(float2) * (3 * FF_MAX_L + (size_t)d.nz * d.Ly * d.hx); }

FFArgs ff_args(const Dims& d) {
  FFArgs a;
  a.nx = d.nx;
  a.ny = d.ny;
  a.nz = d.nz;
  a.Lx = d.Lx;
  a.Ly = d.Ly;
  a.Lz = d.Lz;
  a.hx = d.hx;
  a.Kh = d.Kh;
  return a;
}

}  // namespace

bool fft_cube_applies(bool fp64, const Dims& d) {
  return !fp64 && d.nx == d.ny && d.nx == d.nz && d.Lx == d.Ly && d.Lx == d.Lz && d.Lx >= 8 && d.Lx <= FF_MAX_L &&
         d.nx >= 8 && (d.nx == d.Lx || 2 * d.nx == d.Lx);
}

bool fft_fused_applies(bool fp64, const Dims& d) {
  return !fp64 && d.Lx <= FF_MAX_L && d.Ly <= FF_MAX_L && d.Lz <= FF_MAX_L && d.Lx >= 2 && d.Ly >= 2 &&
         d.Lz >= 2 && fused_smem(d) <= 200 * 1024 && (d.nz * d.ny + 1) / 2 <= FF_THREADS &&
         (int64_t)d.nz * d.Ly * d.hx * 2 >= (int64_t)d.nz * d.ny * d.nx;
}

cudaError_t launch_fft_fused_forward(const void* in, void* spec, const Dims& d, int C, const FftTw& tw, cudaStream_t s,
                                     int* nl) {
  if (C <= 0) return cudaSuccess;
  cudaError_t e = cube_launch(false, in, spec, d, C, s);
  if (e != cudaErrorNotSupported) {
    ++*nl;
    return e;
  }
  const size_t smem = fused_smem(d);
  e = cudaFuncSetAttribute(fft3_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  fft3_fwd_kernel<<<(unsigned)C, FF_THREADS, smem, s>>>((const float*)in, (float2*)spec, ff_args(d),
                                                         (const float2*)tw.x, (const float2*)tw.y, (const float2*)tw.z);
  ++*nl;
  return cudaGetLastError();
}

cudaError_t launch_fft_fused_inverse(const void* spec, void* out, const Dims& d, int C, const FftTw& tw, cudaStream_t s,
                                     int* nl) {
  if (C <= 0) return cudaSuccess;
  cudaError_t e = cube_launch(true, spec, out, d, C, s);
  if (e != cudaErrorNotSupported) {
    ++*nl;
    return e;
  }
  const size_t smem = fused_smem(d);
  e = cudaFuncSetAttribute(fft3_inv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  fft3_inv_kernel<<<(unsigned)C, FF_THREADS, smem, s>>>((const float2*)spec, (float*)out, ff_args(d),
                                                         (const float2*)tw.x, (const float2*)tw.y, (const float2*)tw.z);
  ++*nl;
  return cudaGetLastError();
}

}  // namespace pmmm
