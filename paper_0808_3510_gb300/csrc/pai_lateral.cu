// pai_lateral.cu -- FFTs along a strided axis for power-of-two lengths:
// the lateral transforms of Algorithm 2 (Eq. fft-1a forward, the lateral part
// of Eq. fft-1 inverse) and their transposes.
//
// Data are viewed as A[outer][L][C]: the transform runs along the middle axis
// (length L, element stride C) for every contiguous column c < C and every
// outer index.  The axis is the slow one, so each CTA takes a tile of columns:
//   * the tile is read and written in full 32-byte sectors;
//   * FP column FFTs of length L run in shared memory with the same Stockham
//     passes as the row kernels (16 values per thread per pass);
//   * real-to-complex: columns c, c+1 are paired as z = a + i b (two real
//     FFTs for one complex FFT) and separated after the transform,
//     A[k] = (Z[k] + conj Z[-k]) / 2, B[k] = (Z[k] - conj Z[-k]) / (2i);
//   * complex-to-real: the two half spectra are merged as Z = A + i B over the
//     full range (Hermitian extension, imaginary parts of the self-conjugate
//     bins k = 0, L/2 ignored as in any C2R), inverse transformed, and the
//     real / imaginary parts are the two real columns.
// All transforms are unnormalised.
#include "pai_row_kernels.cuh"

namespace pai {

// Complex values per FFT slot of FP column slots side by side: the padded
// layout, with the slots 16 / FP (mod 16) values apart: the 16 lanes of a
// half-warp in the load and store phases, FP columns times 16 / FP consecutive
// elements, then fall on 16 different banks, in the first pass's writes too
// (17 x0 + r).  (One pad per 32 and a shift of 4 made those accesses two- to
// four-way conflicts: the eight lateral passes of a 256^3 gradient took 356 us
// against 316 now, of 240 their bytes need at the measured copy rate.)
__host__ __device__ constexpr int lateral_slot(int L, int FP) {
  const int s = L + (L >> 4);
  return s + (16 / FP - s % 16 + 16) % 16;
}
// The same for lines handled one after another (rows_fft_kernel, rows_fold_kernel).
__host__ __device__ constexpr int rows_slot(int L) { return L + (L >> 4); }

enum : int { kLatR2C = 0, kLatC2R = 1, kLatC2C = 2, kLatC2CInv = 3 };

// Two adjacent floats, one load when they start on an 8-byte boundary (pairs).
template <bool CHECK>
__device__ __forceinline__ float2 load_pair(const float2* p, int pairs) {
  if (!CHECK || pairs) return *p;
  const float* q = reinterpret_cast<const float*>(p);
  return make_float2(q[0], q[1]);
}

// PRUNED: only the first n of the L points exist on the real side (R2C, C2R)
// or on the input of the C2C / the output of the inverse C2C; the others are
// zeros, or are not stored.  The forward model's box is two to four times the
// image per axis, so most of its traffic is such points: the lateral passes of a
// 128^3 volume in its 512^3 box took 852 us on the whole box, 203 us pruned (and
// with them went 345 us of padding and 18 us of cropping).  (Compiled apart: the
// full kernel keeps its loads without the extra predicate.)  pairs = 0: the
// real buffer is only 4-byte aligned (the forward model takes such buffers;
// the plans' other calls ask for 8 bytes), its floats move one at a time.
template <int KIND, int FP, bool PRUNED>
__global__ void __launch_bounds__(1024) lateral_kernel(const void* vin, void* vout, int L,
                                                       int mshift, int C, long long in_outer, long long out_outer,
                                                       const float2* __restrict__ tw, int twstride, int n,
                                                       int pairs) {
  extern __shared__ __align__(16) float2 smem[];
  constexpr bool kInv = (KIND == kLatC2R || KIND == kLatC2CInv);
  const int tpr = L / kElemsPerThread;
  const int S = lateral_slot(L, FP);
  const int T = blockDim.x;
  const int f = threadIdx.x % FP;  // column group of this thread in the load / store phases
  const int x0 = threadIdx.x / FP;
  const int xs = T / FP;           // = L / 16
  const int half = L >> 1;
  // columns handled by this CTA: real kinds take 2 FP real columns, complex kinds FP
  constexpr int CPT = (KIND == kLatC2C || KIND == kLatC2CInv) ? FP : 2 * FP;
  const int c0 = blockIdx.x * CPT;
  const long long ob = blockIdx.y;
  float2* Z = smem + f * S;
  pdl_wait();

  // ---- load -------------------------------------------------------------
  if (KIND == kLatR2C) {
    const float* in = static_cast<const float*>(vin) + ob * in_outer;
    const bool live = c0 + 2 * f < C;  // C even: pairs are whole
    const float2* src = reinterpret_cast<const float2*>(in + (size_t)x0 * C + c0) + f;
    float2 z[kElemsPerThread];
#pragma unroll
    for (int i = 0; i < kElemsPerThread; ++i)
      z[i] = live && (!PRUNED || x0 + i * xs < n) ? load_pair<PRUNED>(src + (size_t)i * xs * (C / 2), pairs)
                                                  : make_float2(0.f, 0.f);
    first_pass_regs<false>(Z, z, x0);
  } else if (KIND == kLatC2C || KIND == kLatC2CInv) {
    const float2* in = static_cast<const float2*>(vin) + ob * in_outer;
    const bool live = c0 + f < C;
    const float2* src = in + (size_t)x0 * C + c0 + f;
    float2 z[kElemsPerThread];
#pragma unroll
    for (int i = 0; i < kElemsPerThread; ++i)  // plain loads: the C2C may run in place
      z[i] = live && (!PRUNED || kInv || x0 + i * xs < n) ? src[(size_t)i * xs * C] : make_float2(0.f, 0.f);
    first_pass_regs<kInv>(Z, z, x0);
  } else {  // C2R: rows k = 0 .. L/2 of two complex columns per slot
    const float2* in = static_cast<const float2*>(vin) + ob * in_outer;
    const bool live = c0 + 2 * f < C;
    // rows k = x0 + i xs, i = 0 .. 8 (the last only for x0 = 0): loads first
    constexpr int NK = kElemsPerThread / 2 + 1;
    float4 abv[NK];
#pragma unroll
    for (int i = 0; i < NK; ++i) {
      const int k = x0 + i * xs;
      abv[i] = (live && k <= half) ? *reinterpret_cast<const float4*>(in + (size_t)k * C + c0 + 2 * f)
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < NK; ++i) {
      const int k = x0 + i * xs;
      if (k > half) break;
      const float4 ab = abv[i];
      if (k == 0 || k == half) {
        // self-conjugate bins: only the real parts enter a C2R
        Z[padi(k)] = make_float2(ab.x, ab.z);
      } else {
        // Z[k] = A[k] + i B[k];  Z[L-k] = conj A[k] + i conj B[k]
        Z[padi(k)] = make_float2(ab.x - ab.w, ab.y + ab.z);
        Z[padi(L - k)] = make_float2(ab.x + ab.w, ab.z - ab.y);
      }
    }
  }
  __syncthreads();
  {
    const int slot = threadIdx.x / tpr;
    const int lane = threadIdx.x - slot * tpr;
    if (KIND == kLatC2R) fft_smem<kInv, kLayoutFlat>(smem + slot * S, L, mshift, lane, tpr, tw, twstride);
    else fft_rest<kInv, kLayoutFlat>(smem + slot * S, L, mshift, lane, tpr, tw, twstride);
  }

  // ---- store ------------------------------------------------------------
  if (KIND == kLatR2C) {
    float2* out = static_cast<float2*>(vout) + ob * out_outer;
    if (c0 + 2 * f < C) {
      for (int k = x0; k <= half; k += xs) {
        const float2 a = Z[k];
        const float2 b = Z[(L - k) & (L - 1)];
        const float4 o = make_float4(0.5f * (a.x + b.x), 0.5f * (a.y - b.y), 0.5f * (a.y + b.y), 0.5f * (b.x - a.x));
        *reinterpret_cast<float4*>(out + (size_t)k * C + c0 + 2 * f) = o;
      }
    }
  } else if (KIND == kLatC2C || KIND == kLatC2CInv) {
    float2* out = static_cast<float2*>(vout) + ob * out_outer;
    if (c0 + f < C) {
#pragma unroll
      for (int i = 0; i < kElemsPerThread; ++i) {
        const int x = x0 + i * xs;
        if (!PRUNED || !kInv || x < n) out[(size_t)x * C + c0 + f] = Z[x];
      }
    }
  } else {
    float* out = static_cast<float*>(vout) + ob * out_outer;
    if (c0 + 2 * f < C) {
#pragma unroll
      for (int i = 0; i < kElemsPerThread; ++i) {
        const int x = x0 + i * xs;
        if (!PRUNED) {
          *reinterpret_cast<float2*>(out + (size_t)x * C + c0 + 2 * f) = Z[x];
        } else if (x < n) {
          float* o = out + (size_t)x * C + c0 + 2 * f;
          if (pairs) {
            *reinterpret_cast<float2*>(o) = Z[x];
          } else {
            o[0] = Z[x].x;
            o[1] = Z[x].y;
          }
        }
      }
    }
  }
}

int lateral_slots_per_cta(int L) {
  // 8 slots for 256- and 512-point columns (a 256^3 gradient step's four
  // lateral stages gained 22 us over 4; 128-point columns lost with 8)
  int fp = (L >= 256 && L <= 512) ? 8 : 4;
  while (fp > 1 && fp * (L / kElemsPerThread) > 1024) fp >>= 1;
  return fp;
}

size_t lateral_smem_bytes(int L) { return (size_t)lateral_slots_per_cta(L) * lateral_slot(L, lateral_slots_per_cta(L)) * sizeof(float2); }

bool lateral_supported(int L, int C) {
  if (L < 32 || (L & (L - 1)) != 0) return false;
  if ((L / kElemsPerThread) > 1024) return false;
  if (C % 2 != 0) return false;
  return lateral_smem_bytes(L) <= 200 * 1024;
}

template <int KIND, int FP, bool PRUNED>
static cudaError_t lat_launch(const void* in, void* out, int L, int C, int outer, long long in_outer,
                              long long out_outer, const float2* tw, int twstride, cudaStream_t s, bool pdl, int n) {
  const size_t smem = lateral_smem_bytes(L);
  cudaError_t e =
      allow_smem(lateral_kernel<KIND, FP, PRUNED>, smem);
  if (e != cudaSuccess) return e;
  int mshift = 0;
  while ((1 << mshift) < L) ++mshift;
  const int threads = FP * (L / kElemsPerThread);
  constexpr int CPT = (KIND == kLatC2C || KIND == kLatC2CInv) ? FP : 2 * FP;
  dim3 grid((C + CPT - 1) / CPT, outer);
  const void* real = KIND == kLatR2C ? in : out;
  const int pairs = (reinterpret_cast<uintptr_t>(real) & 7) == 0;
  return launch_kernel(lateral_kernel<KIND, FP, PRUNED>, grid, dim3(threads), smem, s, pdl, in, out, L, mshift, C,
                       in_outer, out_outer, tw, twstride, n, pairs);
}

// in_full / out_full: outer strides for L (complex kinds) or L/2 + 1 points; the pruned side has n.
template <int KIND, bool PRUNED>
static cudaError_t lat_dispatch(const void* in, void* out, int L, int C, int outer, const float2* tw, int twstride,
                                cudaStream_t s, bool pdl, int n) {
  const long long full = (long long)L * C, half = (long long)(L / 2 + 1) * C, part = (long long)n * C;
  const long long io = KIND == kLatC2R ? half : KIND == kLatC2CInv ? full : part;
  const long long oo = KIND == kLatR2C ? half : KIND == kLatC2C ? full : part;
  switch (lateral_slots_per_cta(L)) {
    case 8: return lat_launch<KIND, 8, PRUNED>(in, out, L, C, outer, io, oo, tw, twstride, s, pdl, n);
    case 4: return lat_launch<KIND, 4, PRUNED>(in, out, L, C, outer, io, oo, tw, twstride, s, pdl, n);
    case 2: return lat_launch<KIND, 2, PRUNED>(in, out, L, C, outer, io, oo, tw, twstride, s, pdl, n);
    default: return lat_launch<KIND, 1, PRUNED>(in, out, L, C, outer, io, oo, tw, twstride, s, pdl, n);
  }
}

template <int KIND>
static cudaError_t lat_any(const void* in, void* out, int L, int C, int outer, const float2* tw, int twstride,
                           cudaStream_t s, bool pdl, int n) {
  if (n > 0 && n < L) return lat_dispatch<KIND, true>(in, out, L, C, outer, tw, twstride, s, pdl, n);
  return lat_dispatch<KIND, false>(in, out, L, C, outer, tw, twstride, s, pdl, L);
}

// out[o][k][c] = sum_x e^{-2 pi i k x / L} in[o][x][c], k = 0..L/2.
cudaError_t launch_lateral_r2c(const float* in, float2* out, int L, int C, int outer, const float2* tw, int twstride,
                               cudaStream_t s, bool pdl, int n) {
  return lat_any<kLatR2C>(in, out, L, C, outer, tw, twstride, s, pdl, n);
}

// out[o][x][c] = sum over the Hermitian extension of in[o][k][c] of e^{+2 pi i k x / L} (unnormalised C2R).
cudaError_t launch_lateral_c2r(const float2* in, float* out, int L, int C, int outer, const float2* tw, int twstride,
                               cudaStream_t s, bool pdl, int n) {
  return lat_any<kLatC2R>(in, out, L, C, outer, tw, twstride, s, pdl, n);
}

// out[o][k][c] = sum_x e^{-+2 pi i k x / L} in[o][x][c]; in place where a point lies at the same place on both sides
// (each CTA owns its columns): not pruned, or outer = 1.
cudaError_t launch_lateral_c2c(const float2* in, float2* out, int L, int C, int outer, bool inverse, const float2* tw,
                               int twstride, cudaStream_t s, bool pdl, int n) {
  if (in == out && n > 0 && n < L && outer != 1) return cudaErrorInvalidValue;
  if (inverse) return lat_any<kLatC2CInv>(in, out, L, C, outer, tw, twstride, s, pdl, n);
  return lat_any<kLatC2C>(in, out, L, C, outer, tw, twstride, s, pdl, n);
}

// In-place FFT of contiguous lines (the depth transform of Eq. fft-1 and its
// transpose): line r occupies data[r L .. r L + L).  One row slot of L/16
// threads per line; the first pass reads straight from global memory.
template <bool INV>
__global__ void __launch_bounds__(1024) rows_fft_kernel(float2* data, int L, int mshift, int rows,
                                                        const float2* __restrict__ tw, int twstride) {
  extern __shared__ __align__(16) float2 smem[];
  const int tpr = L / kElemsPerThread;
  const int slot = threadIdx.x / tpr;
  const int lane = threadIdx.x - slot * tpr;
  const int rpc = blockDim.x / tpr;
  const int row = blockIdx.x * rpc + slot;
  const bool valid = row < rows;
  float2* X = smem + slot * rows_slot(L);
  float2* line = data + (size_t)(valid ? row : 0) * L;
  pdl_wait();
  {
    constexpr int R = 16;
    const int LR = L / R;
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = line[lane + r * LR];  // plain loads: the transform is in place
    dft_reg<R, INV>(v);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int idx = lane * R + r;
      X[padi(idx)] = v[r];
    }
  }
  __syncthreads();
  fft_rest<INV, kLayoutFlat>(X, L, mshift, lane, tpr, tw, twstride);
  if (valid)
    for (int z = lane; z < L; z += tpr) line[z] = X[z];
}

cudaError_t launch_rows_c2c(float2* data, int L, int rows, bool inverse, const float2* tw, int twstride,
                            cudaStream_t s, bool pdl) {
  if (L < 32 || (L & (L - 1)) != 0 || L / kElemsPerThread > 1024) return cudaErrorInvalidValue;
  int mshift = 0;
  while ((1 << mshift) < L) ++mshift;
  const int tpr = L / kElemsPerThread;
  const int threads = tpr > 128 ? tpr : 128;  // (128 measured 1.5 us faster than 256 per 256^3 depth stage)
  const int rpc = threads / tpr;
  const size_t smem = (size_t)rpc * rows_slot(L) * sizeof(float2);
  const int ctas = (rows + rpc - 1) / rpc;
  void (*k)(float2*, int, int, int, const float2*, int) = inverse ? rows_fft_kernel<true> : rows_fft_kernel<false>;
  const cudaError_t e = allow_smem(k, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(k, dim3(ctas), dim3(threads), smem, s, pdl, data, L, mshift, rows, tw, twstride);
}

// The depth stage of the forward model: lines of n image layers, zero-padded to
// the box depth L and transformed; only c_j = F[j] + F[L - j] is wanted (each
// node pair carries the sum), so a line costs n values read and L/2 + 1
// written instead of L read and L written, and the padded box itself is never
// in memory.
__global__ void __launch_bounds__(1024) rows_fold_kernel(const float2* in, int n, float2* out, int L, int mshift,
                                                         int rows, const float2* __restrict__ tw, int twstride) {
  extern __shared__ __align__(16) float2 smem[];
  const int tpr = L / kElemsPerThread;
  const int slot = threadIdx.x / tpr;
  const int lane = threadIdx.x - slot * tpr;
  const int row = blockIdx.x * (blockDim.x / tpr) + slot;
  const bool valid = row < rows;
  float2* X = smem + slot * rows_slot(L);
  const float2* line = in + (size_t)(valid ? row : 0) * n;
  pdl_wait();
  float2 v[kElemsPerThread];
  if (2 * n <= L && mshift >= 9 && ((mshift - 5) & 3) == 0) {
    // L = 32 16^k: a radix-32 first pass leaves radix-16 passes only (no radix-2
    // pass at the end, 1/4 of the shared-memory traffic).  Butterfly j has inputs
    // x_r at j + r L/32, zero for r >= 16; one thread computes its even outputs (the
    // 16-point DFT of x_r), one its odd ones (of x_r w32^r).
    const int half = tpr >> 1, h = lane >= half ? 1 : 0, j = lane - h * half, L32 = L >> 5;
#pragma unroll
    for (int r = 0; r < kElemsPerThread; ++r) {
      const int z = j + r * L32;
      v[r] = z < n ? line[z] : make_float2(0.f, 0.f);
    }
    if (h) tw32_all(v);
    dft_reg<16, false>(v);
    float2* dst = X + 33 * j + h;
#pragma unroll
    for (int m = 0; m < 16; ++m) dst[2 * m] = v[m];
    __syncthreads();
    fft_rest<false, kLayoutFlat, 2, 5>(X, L, mshift, lane, tpr, tw, twstride, true, 5);
  } else {
#pragma unroll
    for (int r = 0; r < kElemsPerThread; ++r) {
      const int z = lane + r * tpr;
      v[r] = z < n ? line[z] : make_float2(0.f, 0.f);
    }
    first_pass_regs<false>(X, v, lane);
    __syncthreads();
    fft_rest<false, kLayoutFlat>(X, L, mshift, lane, tpr, tw, twstride);
  }
  if (!valid) return;
  float2* o = out + (size_t)row * (L / 2 + 2);
  for (int j = lane; j <= L / 2; j += tpr) {
    float2 y = X[j];
    if (j > 0 && j < L / 2) y = cadd(y, X[L - j]);
    o[j] = y;
  }
}

cudaError_t launch_rows_fold(const float2* in, int n, float2* out, int L, int rows, const float2* tw, int twstride,
                             cudaStream_t s, bool pdl) {
  if (L < 32 || (L & (L - 1)) != 0 || L / kElemsPerThread > 1024) return cudaErrorInvalidValue;
  int mshift = 0;
  while ((1 << mshift) < L) ++mshift;
  const int tpr = L / kElemsPerThread;
  const int threads = tpr > 128 ? tpr : 128;
  const int rpc = threads / tpr;
  const size_t smem = (size_t)rpc * rows_slot(L) * sizeof(float2);
  const cudaError_t e = allow_smem(rows_fold_kernel, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(rows_fold_kernel, dim3((rows + rpc - 1) / rpc), dim3(threads), smem, s, pdl, in, n, out, L,
                       mshift, rows, tw, twstride);
}

}  // namespace pai
