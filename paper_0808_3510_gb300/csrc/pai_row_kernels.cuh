// pai_row_kernels.cuh -- sm_103a row kernels of the NUFFT Fourier reconstruction.
//
// One "row" is one lateral frequency K_lat of the detector data after the
// lateral FFT (Eq. fft-1a).  For every row the forward kernel performs the
// whole one-dimensional nonuniform FFT of Algorithm 1 plus the weight of
// Eq. (fft-0) without leaving the SM:
//
//   1. prescale (Algorithm 1, division by the window) and zero padding to the
//      oversampled length M = c nt, written straight into shared memory;
//   2. the length-M FFT of Eq. (nufft-c), in shared memory (Stockham
//      autosort, radix 16/8/4/2, each thread holding 16 values in registers
//      per pass; at oversampling 2 the first pass skips the zero padding, as
//      two length-8 DFTs or, for M = 32 16^k, as a radix-32 pass shared by
//      two threads);
//   3. the truncated window gather of Eq. (nufft-a) at the nodes
//      omega = c_s sign(Kz) |K| (Eq. dft-2d), multiplied by the weight of
//      Eq. (fft-0), written to the half image spectrum.
//
// The oversampled spectrum of a row therefore never reaches HBM: a row costs
// one read of its nt complex samples and one write of its nz/2+1 (or twice
// that) spectrum values.  The adjoint kernel runs the exact transpose of the
// same steps in reverse order (spread, inverse FFT, prescale).
//
// Conventions fixed by the design (each traced to the paper):
//  * the constant of Fourmont's identity is 1/(2 pi c) (it is the Fourier
//    coefficient of a 2 pi c periodic function); it lives in the prescale;
//  * the phase of the Proposition (Eq. nufft-a) is e^{-i pi (omega - j/c)}:
//    the e^{+i pi j/c} part is applied by storing sample n at position
//    n - nt/2 (mod M) before the FFT, the e^{-i pi omega} part once per node;
//  * taps are wrapped modulo M (the oversampled spectrum is M-periodic by
//    Eq. nufft-c), so nodes beyond the Nyquist band are handled exactly;
//  * node positions are computed in float-float arithmetic (about 44
//    significant bits) because an FP32 node alone would cost 1e-5 relative
//    error at |omega| ~ 3000.
#include <cuda_runtime.h>
#include <stdint.h>

#pragma once
#include "pai_internal.h"

namespace pai {

// Index of element i in the padded layout of a transform in shared memory: one
// padding element every 2^PS.  With PS = 4 a radix-16 first pass (thread j
// writes 16 j .. 16 j + 15) puts the 16 lanes of a half-warp on 16 different
// banks (stride 17), with PS = 5 only on 8; after a radix-32 first pass
// (33 j + q) PS = 5 is the one without conflicts.
template <int PS = 4>
__host__ __device__ __forceinline__ constexpr int padi(int i) {
  return i + (i >> PS);
}

// Complex arithmetic on the packed two-lane FP32 instructions of sm_100+
// (add/sub/mul/fma .rn.f32x2): one instruction per complex add, two per
// complex product.  Each lane rounds exactly like its scalar counterpart.
__device__ __forceinline__ unsigned long long pack2(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long r) {
  float2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)), "l"(pack2(c)));
  return unpack2(r);
}
// (a.x + i a.y)(b.x + i b.y) = a.x (b.x, b.y) + a.y (-b.y, b.x)
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return fma2(make_float2(a.x, a.x), b, mul2(make_float2(a.y, a.y), make_float2(-b.y, b.x)));
}

// cos and sin of 2 pi q / 16, q = 0..7
__host__ __device__ constexpr float cos16(int q) {
  return q == 0 ? 1.0f : q == 1 ? 0.92387953251128674f : q == 2 ? 0.70710678118654752f
       : q == 3 ? 0.38268343236508977f : q == 4 ? 0.0f : q == 5 ? -0.38268343236508977f
       : q == 6 ? -0.70710678118654752f : -0.92387953251128674f;
}
__host__ __device__ constexpr float sin16(int q) {
  return q == 0 ? 0.0f : q == 1 ? 0.38268343236508977f : q == 2 ? 0.70710678118654752f
       : q == 3 ? 0.92387953251128674f : q == 4 ? 1.0f : q == 5 ? 0.92387953251128674f
       : q == 6 ? 0.70710678118654752f : 0.38268343236508977f;
}

// cos and sin of 2 pi q / 32, q = 0..8
__host__ __device__ constexpr float cos32(int q) {
  return q == 0 ? 1.0f : q == 1 ? 0.98078528040323044913f : q == 2 ? 0.92387953251128675613f
       : q == 3 ? 0.83146961230254523708f : q == 4 ? 0.70710678118654752440f : q == 5 ? 0.55557023301960222474f
       : q == 6 ? 0.38268343236508977173f : q == 7 ? 0.19509032201612826785f : 0.0f;
}
__host__ __device__ constexpr float sin32(int q) { return cos32(8 - q); }

// x * e^{-+ 2 pi i q / 32}, q = 0..8  (CONJ: plus sign)
template <int Q, bool CONJ>
__device__ __forceinline__ float2 tw32(float2 x) {
  if (Q == 0) return x;
  if (Q == 8) return CONJ ? make_float2(-x.y, x.x) : make_float2(x.y, -x.x);
  constexpr float c = cos32(Q);
  constexpr float s = CONJ ? sin32(Q) : -sin32(Q);
  return fma2(make_float2(x.x, x.x), make_float2(c, s), mul2(make_float2(x.y, x.y), make_float2(-s, c)));
}

// x * e^{-+ 2 pi i q / 16}  (forward: minus sign; INV: plus sign)
template <int Q, bool INV>
__device__ __forceinline__ float2 twq(float2 x) {
  if (Q == 0) return x;
  if (Q == 4) return INV ? make_float2(-x.y, x.x) : make_float2(x.y, -x.x);
  constexpr float c = cos16(Q);
  constexpr float s = INV ? sin16(Q) : -sin16(Q);
  return fma2(make_float2(x.x, x.x), make_float2(c, s), mul2(make_float2(x.y, x.y), make_float2(-s, c)));
}

template <int R>
__host__ __device__ constexpr int bitrev(int i) {
  int r = 0;
  for (int b = 1, k = R >> 1; b < R; b <<= 1, k >>= 1)
    if (i & b) r |= k;
  return r;
}

// Butterfly stage of an in-register radix-2 DIT FFT of size R (data in
// bit-reversed order).  Stage span m, half h = m/2, twiddle q = k * 16/m.
template <int R, int M2, int K, bool INV>
struct Stage {
  __device__ __forceinline__ static void run(float2 (&a)[R]) {
    constexpr int h = M2 / 2;
#pragma unroll
    for (int g = 0; g < R; g += M2) {
      float2 u = a[g + K];
      float2 t = twq<K * (16 / M2), INV>(a[g + K + h]);
      a[g + K] = cadd(u, t);
      a[g + K + h] = csub(u, t);
    }
    Stage<R, M2, K + 1, INV>::run(a);
  }
};
template <int R, int M2, bool INV>
struct Stage<R, M2, M2 / 2, INV> {
  __device__ __forceinline__ static void run(float2 (&)[R]) {}
};

template <int R, int M2, bool INV>
struct Stages {
  __device__ __forceinline__ static void run(float2 (&a)[R]) {
    Stage<R, M2, 0, INV>::run(a);
    Stages<R, M2 * 2, INV>::run(a);
  }
};
template <int R, bool INV>
struct Stages<R, R * 2, INV> {
  __device__ __forceinline__ static void run(float2 (&)[R]) {}
};

// v <- DFT_R(v): v[k] = sum_r v[r] e^{-+ 2 pi i r k / R}
template <int R, bool INV>
__device__ __forceinline__ void dft_reg(float2 (&v)[R]) {
  float2 a[R];
#pragma unroll
  for (int i = 0; i < R; ++i) a[bitrev<R>(i)] = v[i];
  Stages<R, 2, INV>::run(a);
#pragma unroll
  for (int i = 0; i < R; ++i) v[i] = a[i];
}

// Shared-memory accesses by 32-bit address (16 bytes at a time in the band grids: every kernel declares its
// dynamic shared memory 16-byte aligned, which float2 alone does not make it).
__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ float4 lds4(unsigned a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a)
               : "memory");
  return v;
}
__device__ __forceinline__ float2 lds2(unsigned a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts2(unsigned a, float2 v) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void sts4(unsigned a, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// Layouts of a row slot in shared memory.  Passes between the first and the
// last keep one padding element every 16 or 32 (padi) so strided butterfly accesses
// do not collide in the banks.  The last pass of the forward transform writes
// the spectrum unpadded and repeats its first 2*kMaxH values after index M
// ("ghost cells"), so a node's 2H consecutive taps are plain consecutive
// addresses even when the window wraps around the period M.
enum : int { kLayoutPadded = 0, kLayoutFlat = 1, kLayoutFlatGhost = 2 };

// One in-place Stockham pass of radix R.  Butterfly j (0 <= j < M/R) reads
// X[j + r M/R], twiddles by e^{-+2 pi i r (j mod Ns) / (Ns R)}, and writes its
// R outputs to X[(j - j mod Ns) R + (j mod Ns) + r Ns].  All reads of the
// pass complete (barrier) before any write.  OUT selects the write layout.
// Twiddle powers w^1 .. w^(R-1) from the table entries w^1, w^2, w^4, w^8
// (loaded before the pass barrier); the others are products of at most
// three of them, so each power carries at most three extra roundings.
template <int R>
struct TwBase {
  float2 b[R >= 16 ? 4 : R >= 8 ? 3 : R >= 4 ? 2 : 1];
};

// The twiddle table is two-level (twiddle_table): w^k = hi[k >> 6] lo[k & 63]
// with lo = tw[0..63] and hi = tw[64..], w = e^{-2 pi i / TW}.  Both parts
// together hold 64 + TW/64 values (2.5 KB at TW = 16384), so they stay in L1
// while a full-length table (64 KB at TW = 8192) would miss there; the
// product costs one complex multiply and about one extra rounding.
__device__ __forceinline__ float2 tw_at(const float2* __restrict__ tw, int k) {
  return cmul(__ldg(&tw[kTwLo + (k >> kTwLoShift)]), __ldg(&tw[k & (kTwLo - 1)]));
}

template <int R>
__device__ __forceinline__ void tw_load(TwBase<R>& t, const float2* __restrict__ tw, int step) {
  t.b[0] = tw_at(tw, step);
  if (R >= 4) t.b[1] = tw_at(tw, 2 * step);
  if (R >= 8) t.b[2] = tw_at(tw, 4 * step);
  if (R >= 16) t.b[3] = tw_at(tw, 8 * step);
}

// x * e^{-2 pi i q / 16}, q = 0..15 (a constant once the caller's loop is unrolled)
__device__ __forceinline__ float2 rot16(float2 x, int q) {
  const float c = (q & 8) ? -cos16(q & 7) : cos16(q & 7);
  const float s = (q & 8) ? sin16(q & 7) : -sin16(q & 7);
  return fma2(make_float2(x.x, x.x), make_float2(c, s), mul2(make_float2(x.y, x.y), make_float2(-s, c)));
}

// Base twiddles of butterfly j + i M/16 from those of butterfly j, for the last
// pass of a transform (Ns R = M, so the twiddle index is the butterfly index):
// w^{2^e (j + i M/16)} = w^{2^e j} e^{-2 pi i (2^e i mod 16) / 16}.
template <int R>
__device__ __forceinline__ void tw_shift(TwBase<R>& t, const TwBase<R>& t0, int i) {
  t.b[0] = rot16(t0.b[0], i & 15);
  if (R >= 4) t.b[1] = rot16(t0.b[1], (2 * i) & 15);
  if (R >= 8) t.b[2] = rot16(t0.b[2], (4 * i) & 15);
  if (R >= 16) t.b[3] = rot16(t0.b[3], (8 * i) & 15);
}

template <bool INV>
__device__ __forceinline__ float2 twc(float2 w) {
  return INV ? make_float2(w.x, -w.y) : w;
}

// v[r] *= w^r for r = 1..R-1, each power formed right before its use so only
// the base entries stay live.
template <int R, bool INV>
__device__ __forceinline__ void tw_apply(float2 (&v)[R], const TwBase<R>& t) {
  const float2 w1 = t.b[0];
  v[1] = cmul(v[1], twc<INV>(w1));
  if (R >= 4) {
    const float2 w2 = t.b[1];
    const float2 w3 = cmul(w1, w2);
    v[2] = cmul(v[2], twc<INV>(w2));
    v[3] = cmul(v[3], twc<INV>(w3));
    if (R >= 8) {
      const float2 w4 = t.b[2];
      const float2 w5 = cmul(w1, w4), w6 = cmul(w2, w4), w7 = cmul(w3, w4);
      v[4] = cmul(v[4], twc<INV>(w4));
      v[5] = cmul(v[5], twc<INV>(w5));
      v[6] = cmul(v[6], twc<INV>(w6));
      v[7] = cmul(v[7], twc<INV>(w7));
      if (R >= 16) {
        const float2 w8 = t.b[3];
        v[8] = cmul(v[8], twc<INV>(w8));
        v[9] = cmul(v[9], twc<INV>(cmul(w1, w8)));
        v[10] = cmul(v[10], twc<INV>(cmul(w2, w8)));
        v[11] = cmul(v[11], twc<INV>(cmul(w3, w8)));
        v[12] = cmul(v[12], twc<INV>(cmul(w4, w8)));
        v[13] = cmul(v[13], twc<INV>(cmul(w5, w8)));
        v[14] = cmul(v[14], twc<INV>(cmul(w6, w8)));
        v[15] = cmul(v[15], twc<INV>(cmul(w7, w8)));
      }
    }
  }
}

// Padded addresses without per-element shifts: for a multiple S of 2^PS,
// padi(a + r S) = padi(a) + r (S + S / 2^PS); for a with a mod 32 < 16,
// padi<5>(a + 16 r) = padi<5>(a) + 16 r + r/2 (r < 16); and for a radix-16 first
// pass (Ns = 1) padi(16 j + r) = padi(16 j) + r.
// CHAIN_R: the smallest radix whose last pass derives its twiddles by
// rotation (tw_shift); below it they come from the table.
template <int R, bool INV, int OUT, int CHAIN_R = 2, int PS = 4>
__device__ __forceinline__ void fft_pass(float2* X, int M, int Ns, int lane, int tpr, const float2* __restrict__ tw,
                                         int twstride, bool active = true) {
  constexpr int NB = kElemsPerThread / R;
  float2 v[NB][R];
  TwBase<R> t[NB];
  const int MR = M / R;
  const int tws = (M / (Ns * R)) * twstride;
  // A last pass of radix < 16 (several butterflies per thread, at j = lane +
  // i M/16): their twiddles follow from the first butterfly's by constant
  // rotations (tw_shift) instead of table loads.
  const bool chain = R >= CHAIN_R && NB > 1 && Ns > 1 && Ns * R == M && tpr * kElemsPerThread == M;
  // twiddles do not depend on the data: for radix 16 (one butterfly per
  // thread) their loads are issued before the barrier; smaller radices carry
  // several butterflies per thread and load after it to stay within registers
  if (active) {
    if (Ns > 1 && NB == 1) tw_load<R>(t[0], tw, (lane & (Ns - 1)) * tws);
    if ((MR & ((1 << PS) - 1)) == 0) {
      const int rs = MR + (MR >> PS);
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        const float2* src = X + padi<PS>(lane + i * tpr);
#pragma unroll
        for (int r = 0; r < R; ++r) v[i][r] = src[r * rs];
      }
    } else {
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        const int j = lane + i * tpr;
#pragma unroll
        for (int r = 0; r < R; ++r) v[i][r] = X[padi<PS>(j + r * MR)];
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    if (!active) break;
    const int j = lane + i * tpr;
    const int k = j & (Ns - 1);
    if (Ns > 1) {
      if (NB != 1) {
        if (!chain || i == 0) tw_load<R>(t[i], tw, k * tws);
        else tw_shift<R>(t[i], t[0], i);
      }
      tw_apply<R, INV>(v[i], t[i]);
    }
    dft_reg<R, INV>(v[i]);
    const int base = (j - k) * R + k;
    if (OUT == kLayoutPadded) {
      float2* dst = X + padi<PS>(base);
      if (PS == 5 && Ns == 16) {
#pragma unroll
        for (int r = 0; r < R; ++r) dst[16 * r + (r >> 1)] = v[i][r];
      } else if (Ns > 1 && (Ns & ((1 << PS) - 1)) == 0) {
        const int ws = Ns + (Ns >> PS);
#pragma unroll
        for (int r = 0; r < R; ++r) dst[r * ws] = v[i][r];
      } else if (Ns == 1 && R == 16) {
#pragma unroll
        for (int r = 0; r < R; ++r) dst[r] = v[i][r];
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) X[padi<PS>(base + r * Ns)] = v[i][r];
      }
    } else {
      float2* dst = X + base;
#pragma unroll
      for (int r = 0; r < R; ++r) dst[r * Ns] = v[i][r];
      if (OUT == kLayoutFlatGhost && base < 2 * kMaxH) {
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (base + r * Ns < 2 * kMaxH) X[M + base + r * Ns] = v[i][r];
      }
    }
  }
  __syncthreads();
}

// Sample n of a row's lateral spectrum: src[n], or (paired layout, see
// RowProblem::paired) separated from the transforms of the sample pairs,
// z1 = Z[k][m], z2 = Z[nx - k][m] with m = n/2:
// sample 2m = (z1 + conj z2) / 2, sample 2m+1 = (z1 - conj z2) / (2i).
template <bool PAIRED>
__device__ __forceinline__ float2 row_sample(const float2* src, const float2* src2, int n) {
  if (!PAIRED) return src[n];
  const float2 z1 = src[n >> 1], z2 = src2[n >> 1];
  return (n & 1) ? make_float2(0.5f * (z1.y + z2.y), 0.5f * (z2.x - z1.x))
                 : make_float2(0.5f * (z1.x + z2.x), 0.5f * (z1.y - z2.y));
}

// First forward pass (radix 16, Ns = 1) fed straight from global memory:
// position m = j + r M/16 of the oversampled input holds sample
// n = m + nt/2 (mod M) times the prescale when n < nt, else zero (Algorithm 1
// prescale and zero padding, centred so that the e^{+i pi j/c} part of the
// Proposition's phase is absorbed).  Writes padded.
template <bool PAIRED = false>
__device__ __forceinline__ void fft_first_pass_from_global(float2* X, int M, int nt, int lane, int tpr,
                                                           const float2* src,
                                                           const float* __restrict__ prescale,
                                                           const float2* src2 = nullptr) {
  constexpr int R = 16;
  float2 v[R];
  const int MR = M / R, mask = M - 1, h = nt >> 1;
  if (M == 2 * nt) {
    // Oversampling 2: only the inputs r = 0..3 and 12..15 hold samples (the
    // others fall in the zero padding), a block b_s, s = -4..3, of 8 values.
    // With w = e^{-2 pi i/16}: X[2m] = sum_s b_s w^{2sm} and
    // X[2m+1] = sum_s (b_s w^s) w^{2sm}, two length-8 DFTs.
    float2 c8[8], d8[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int r = q < 4 ? q : q + 8;
      const int n = (lane + r * MR + h) & mask;
      const float2 g = row_sample<PAIRED>(src, src2, n);
      const float s = __ldg(&prescale[n]);
      c8[q] = make_float2(s * g.x, s * g.y);
    }
    d8[0] = c8[0];
    d8[1] = twq<1, false>(c8[1]);
    d8[2] = twq<2, false>(c8[2]);
    d8[3] = twq<3, false>(c8[3]);
    d8[4] = twq<4, true>(c8[4]);  // w^-4 = i
    d8[5] = twq<3, true>(c8[5]);
    d8[6] = twq<2, true>(c8[6]);
    d8[7] = twq<1, true>(c8[7]);
    dft_reg<8, false>(c8);
    dft_reg<8, false>(d8);
    float2* dst = X + padi<5>(lane * R);
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      dst[2 * m] = c8[m];
      dst[2 * m + 1] = d8[m];
    }
    __syncthreads();
    return;
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int m = lane + r * MR;
    const int n = (m + h) & mask;
    float2 a = make_float2(0.f, 0.f);
    if (n < nt) {
      const float2 g = row_sample<PAIRED>(src, src2, n);
      const float s = __ldg(&prescale[n]);
      a = make_float2(s * g.x, s * g.y);
    }
    v[r] = a;
  }
  dft_reg<R, false>(v);
  float2* dst = X + padi<5>(lane * R);
#pragma unroll
  for (int r = 0; r < R; ++r) dst[r] = v[r];
  __syncthreads();
}

// v[r] *= e^{-2 pi i r / 32}, r = 0..15
__device__ __forceinline__ void tw32_all(float2 (&v)[16]) {
  v[1] = tw32<1, false>(v[1]);
  v[2] = tw32<2, false>(v[2]);
  v[3] = tw32<3, false>(v[3]);
  v[4] = tw32<4, false>(v[4]);
  v[5] = tw32<5, false>(v[5]);
  v[6] = tw32<6, false>(v[6]);
  v[7] = tw32<7, false>(v[7]);
  v[8] = tw32<8, false>(v[8]);
  // w32^r = -i w32^(r - 8)
  v[9] = tw32<8, false>(tw32<1, false>(v[9]));
  v[10] = tw32<8, false>(tw32<2, false>(v[10]));
  v[11] = tw32<8, false>(tw32<3, false>(v[11]));
  v[12] = tw32<8, false>(tw32<4, false>(v[12]));
  v[13] = tw32<8, false>(tw32<5, false>(v[13]));
  v[14] = tw32<8, false>(tw32<6, false>(v[14]));
  v[15] = tw32<8, false>(tw32<7, false>(v[15]));
}

// First forward pass of radix 32 at oversampling 2 when M = 32 16^k: the
// transform then takes radix-16 passes only (no radix-2 pass at its end).
// Butterfly j (0 <= j < M/32) has inputs x_r at positions j + r M/32, which
// hold samples for r = 0..7 and r = 24..31 only (the rest is padding), and
// outputs X[32 j + q].  Two threads share it: h = 0 computes the even outputs
// X[32 j + 2m] = sum_s z_s w16^{sm} with z_s = x_s + x_{s+16}, h = 1 the odd
// ones with z_s = (x_s - x_{s+16}) w32^s, w_N = e^{-2 pi i/N}; of each pair
// x_s, x_{s+16} one is padding (s < 8: x_{s+16}; s >= 8: x_s).  Both threads
// load the butterfly's 16 samples.  Writes padded: padi<5>(32 j + q) = 33 j + q.
template <bool PAIRED>
__device__ __forceinline__ void fft_first_pass32_from_global(float2* X, int M, int nt, int lane, int tpr,
                                                             const float2* src,
                                                             const float* __restrict__ prescale,
                                                             const float2* src2) {
  const int half = tpr >> 1, q4 = M >> 2, M32 = M >> 5;
  const int h = lane >= half ? 1 : 0;
  const int j = lane - h * half;
  float2 v[16];
#pragma unroll
  for (int s = 0; s < 16; ++s) {
    const int n = s < 8 ? j + s * M32 + q4 : j + (s - 8) * M32;
    const float2 g = row_sample<PAIRED>(src, src2, n);
    const float p = __ldg(&prescale[n]);
    v[s] = make_float2(p * g.x, p * g.y);
  }
  if (h) {
    v[1] = tw32<1, false>(v[1]);
    v[2] = tw32<2, false>(v[2]);
    v[3] = tw32<3, false>(v[3]);
    v[4] = tw32<4, false>(v[4]);
    v[5] = tw32<5, false>(v[5]);
    v[6] = tw32<6, false>(v[6]);
    v[7] = tw32<7, false>(v[7]);
    // s >= 8: -w32^s = conj(w32^{16-s})
    v[8] = tw32<8, true>(v[8]);
    v[9] = tw32<7, true>(v[9]);
    v[10] = tw32<6, true>(v[10]);
    v[11] = tw32<5, true>(v[11]);
    v[12] = tw32<4, true>(v[12]);
    v[13] = tw32<3, true>(v[13]);
    v[14] = tw32<2, true>(v[14]);
    v[15] = tw32<1, true>(v[15]);
  }
  dft_reg<16, false>(v);
  float2* dst = X + 33 * j + h;
#pragma unroll
  for (int m = 0; m < 16; ++m) dst[2 * m] = v[m];
  __syncthreads();
}

// Whether the forward transform of a row starts with the radix-32 pass.
__device__ __forceinline__ bool first_pass32(int M, int mshift, int nt) {
  return M == 2 * nt && mshift >= 9 && ((mshift - 5) & 3) == 0;
}

// The values a thread loads, elements x0 + i M/16 (i = 0..15), are the inputs
// of butterfly x0 of the first radix-16 Stockham pass (Ns = 1): that pass runs
// on them in registers and writes its outputs 16 x0 + r in the padded layout,
// ready for fft_rest.
template <bool INV>
__device__ __forceinline__ void first_pass_regs(float2* Z, float2 (&z)[kElemsPerThread], int x0) {
  dft_reg<kElemsPerThread, INV>(z);
#pragma unroll
  for (int r = 0; r < kElemsPerThread; ++r) Z[padi(x0 * kElemsPerThread + r)] = z[r];
}

// Remaining passes after a first pass of radix 2^ns_shift (16 or 32: Ns on
// entry); the last pass writes layout OUT.
template <bool INV, int OUT, int CHAIN_R = 2, int PS = 4>
__device__ __forceinline__ void fft_rest(float2* X, int M, int mshift, int lane, int tpr, const float2* tw,
                                         int twstride, bool active = true, int ns_shift = 4) {
  int Ns = 1 << ns_shift;
  int rem = mshift - ns_shift;
  while (rem >= 4) {
    if (rem == 4) {
      fft_pass<16, INV, OUT, CHAIN_R, PS>(X, M, Ns, lane, tpr, tw, twstride, active);
      return;
    }
    fft_pass<16, INV, kLayoutPadded, CHAIN_R, PS>(X, M, Ns, lane, tpr, tw, twstride, active);
    Ns <<= 4;
    rem -= 4;
  }
  if (rem == 3) fft_pass<8, INV, OUT, CHAIN_R, PS>(X, M, Ns, lane, tpr, tw, twstride, active);
  else if (rem == 2) fft_pass<4, INV, OUT, CHAIN_R, PS>(X, M, Ns, lane, tpr, tw, twstride, active);
  else if (rem == 1) fft_pass<2, INV, OUT, CHAIN_R, PS>(X, M, Ns, lane, tpr, tw, twstride, active);
}

// The band grid of an adjoint row (written by the pair spread, see
// adjoint_band): cell c, counted from the row's first cell `lo`, holds the
// sums P[c] over the +x nodes (first half of its 16 bytes) and N[c] over the
// -x nodes (second half); the N sums belong to grid cell -c.  The oversampled
// grid is U[m] = sum over c = m (mod M) of P[c] + sum over c = -m (mod M) of
// N[c].  Cells are stored in four phases, cell c at (c mod 4) ps + c / 4.
struct Band {
  unsigned grid;  // shared-memory address of cell 0
  int ps;         // cells per phase
  int lo, n;      // first cell and number of cells in use
};

// First inverse pass (radix 16, Ns = 1) fed from the band grid (at most M cells
// here), which shares the row slot's memory with the pass's output X: every
// thread holds its 16 inputs before any writes.
__device__ __forceinline__ void fft_first_pass_band(float2* X, int M, int lane, int tpr, const Band& b) {
  constexpr int R = 16;
  float2 v[R];
  const int mask = M - 1;
  const int p0 = lane - b.lo, q0 = -lane - b.lo;
  if ((tpr & 3) == 0) {
    // a thread's inputs are tpr (a multiple of 4) apart, so all lie in one phase
    const int pp = p0 & 3, qp = q0 & 3;
    const unsigned pa = b.grid + ((pp * b.ps) << 4) - (pp << 2), qa = b.grid + ((qp * b.ps) << 4) - (qp << 2) + 8;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = (p0 + r * tpr) & mask, k = (q0 - r * tpr) & mask;
      float2 u = make_float2(0.f, 0.f), w = u;
      if (i < b.n) u = lds2(pa + (i << 2));
      if (k < b.n) w = lds2(qa + (k << 2));
      v[r] = cadd(u, w);
    }
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = (p0 + r * tpr) & mask, k = (q0 - r * tpr) & mask;
      float2 u = make_float2(0.f, 0.f), w = u;
      if (i < b.n) u = lds2(b.grid + (((i & 3) * b.ps + (i >> 2)) << 4));
      if (k < b.n) w = lds2(b.grid + (((k & 3) * b.ps + (k >> 2)) << 4) + 8);
      v[r] = cadd(u, w);
    }
  }
  __syncthreads();
  dft_reg<R, true>(v);
  float2* dst = X + padi(lane * R);
#pragma unroll
  for (int r = 0; r < R; ++r) dst[r] = v[r];
  __syncthreads();
}

// Last pass of an adjoint row's inverse transform (radix R < 16, Ns = M/R,
// 16/R butterflies j = lane + i M/16 per thread, outputs at m = j + r M/R)
// with the crop fused: the outputs that hold samples n = (m + nt/2) mod M <
// nt, times s_n = scale * prescale[n], go straight to dst[n].  At
// oversampling 2 only half of each butterfly's outputs are kept (and
// computed): r < R/4 and r >= 3R/4, for R = 2 the first output of j < M/4 and
// the second of the others.
template <int R, int PS>
__device__ __forceinline__ void fft_last_crop(const float2* X, int M, int nt, int lane, int tpr,
                                              const float2* __restrict__ tw, int twstride, float2* dst,
                                              const float* __restrict__ prescale, float scale) {
  constexpr int NB = kElemsPerThread / R;
  const int MR = M / R, q4 = M >> 2, mask = M - 1, h = nt >> 1;
  float2 v[NB][R];
#pragma unroll
  for (int i = 0; i < NB; ++i)
#pragma unroll
    for (int r = 0; r < R; ++r) v[i][r] = X[padi<PS>(lane + i * tpr + r * MR)];
  TwBase<R> t0, t;
  tw_load<R>(t0, tw, lane * twstride);
  const bool two = M == 2 * nt;
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    const int j = lane + i * tpr;
    if (i == 0) t = t0;
    else tw_shift<R>(t, t0, i);
    tw_apply<R, true>(v[i], t);
    dft_reg<R, true>(v[i]);
    if (two) {
      if (R == 2) {
        // j < M/4 for the first half of the butterflies (i < NB/2)
        const int n = i < NB / 2 ? j + q4 : j + MR - 3 * q4;
        const float2 y = i < NB / 2 ? v[i][0] : v[i][R - 1];
        const float s = scale * __ldg(&prescale[n]);
        dst[n] = make_float2(s * y.x, s * y.y);
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (r >= R / 4 && r < 3 * R / 4) continue;
          const int n = j + r * MR + (r < R / 4 ? q4 : -3 * q4);
          const float s = scale * __ldg(&prescale[n]);
          dst[n] = make_float2(s * v[i][r].x, s * v[i][r].y);
        }
      }
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int n = (j + r * MR + h) & mask;
        if (n < nt) {
          const float s = scale * __ldg(&prescale[n]);
          dst[n] = make_float2(s * v[i][r].x, s * v[i][r].y);
        }
      }
    }
  }
}

// Inverse length-M transform of an adjoint row with the crop fused: radix-16
// passes, then the remaining radix (M/16 strided reads and unit-stride global
// writes; as the first pass its scattered shared-memory writes conflicted
// four to eight ways).  The last pass writes the outputs that hold samples
// straight to dst (fft_last_crop).  When M is a power of 16 the last pass is
// radix 16 (butterfly j = lane, outputs at m = j + r M/16); at oversampling 2
// (M = 2 nt) only r = 0..3 (n = m + M/4) and r = 12..15 (n = m - 3M/4) are
// kept, and only those 8 outputs are computed: with w = e^{+2 pi i/16},
// A = inverse DFT8 of the even inputs and B of the odd,
// Y[t] = A[t] + w^t B[t] (t = 0..3) and Y[t+8] = A[t] - w^t B[t] (t = 4..7).
// BAND: the first pass reads the band grid.  Otherwise (list spreads) the
// remaining radix comes first and radix 16 last: their kernel holds three spreads
// and has no registers left for the three other last passes (tap phases with
// linear interpolation at M = 8192: 100.5 us, 105 with them); and one pad per 32,
// so that rows and node lists fit in shared memory up to the sizes they always did.
template <bool BAND>
__device__ __forceinline__ void fft_inverse_crop(float2* X, int M, int mshift, int nt, int lane, int tpr,
                                                 const float2* __restrict__ tw, int twstride, float2* dst,
                                                 const float* __restrict__ prescale, float scale, bool valid,
                                                 const Band& band) {
  constexpr int PS = BAND ? 4 : 5;
  const int r0 = mshift & 3;
  int Ns = 1;
  if (BAND) {
    fft_first_pass_band(X, M, lane, tpr, band);
    Ns = 16;
  } else if (r0 == 3) {
    fft_pass<8, true, kLayoutPadded, 2, PS>(X, M, 1, lane, tpr, tw, twstride);
    Ns = 8;
  } else if (r0 == 2) {
    fft_pass<4, true, kLayoutPadded, 2, PS>(X, M, 1, lane, tpr, tw, twstride);
    Ns = 4;
  } else if (r0 == 1) {
    fft_pass<2, true, kLayoutPadded, 2, PS>(X, M, 1, lane, tpr, tw, twstride);
    Ns = 2;
  }
  while (Ns * 16 < M) {
    fft_pass<16, true, kLayoutPadded, 2, PS>(X, M, Ns, lane, tpr, tw, twstride);
    Ns <<= 4;
  }
  if (!valid) return;
  if (BAND && r0 != 0) {
    if (r0 == 3) fft_last_crop<8, PS>(X, M, nt, lane, tpr, tw, twstride, dst, prescale, scale);
    else if (r0 == 2) fft_last_crop<4, PS>(X, M, nt, lane, tpr, tw, twstride, dst, prescale, scale);
    else fft_last_crop<2, PS>(X, M, nt, lane, tpr, tw, twstride, dst, prescale, scale);
    return;
  }
  const int j = lane;
  float2 v[16];
  if ((Ns & ((1 << PS) - 1)) == 0) {
    const float2* src = X + padi<PS>(j);
    const int rs = Ns + (Ns >> PS);
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = src[r * rs];
  } else {
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = X[padi<PS>(j + r * Ns)];
  }
  if (Ns > 1) {
    TwBase<16> tb;
    tw_load<16>(tb, tw, j * twstride);
    tw_apply<16, true>(v, tb);
  }
  const int q4 = M >> 2;
  if (M == 2 * nt) {
    float2 a[8], b[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      a[q] = v[2 * q];
      b[q] = v[2 * q + 1];
    }
    dft_reg<8, true>(a);
    dft_reg<8, true>(b);
    b[1] = twq<1, true>(b[1]);
    b[2] = twq<2, true>(b[2]);
    b[3] = twq<3, true>(b[3]);
    b[4] = twq<4, true>(b[4]);
    b[5] = twq<5, true>(b[5]);
    b[6] = twq<6, true>(b[6]);
    b[7] = twq<7, true>(b[7]);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float2 y = q < 4 ? cadd(a[q], b[q]) : csub(a[q], b[q]);
      const int n = q < 4 ? j + q * Ns + q4 : j + (q + 8) * Ns - 3 * q4;
      const float s = scale * __ldg(&prescale[n]);
      dst[n] = make_float2(s * y.x, s * y.y);
    }
    return;
  }
  dft_reg<16, true>(v);
  const int mask = M - 1, h = nt >> 1;
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const int n = (j + r * Ns + h) & mask;
    if (n < nt) {
      const float s = scale * __ldg(&prescale[n]);
      dst[n] = make_float2(s * v[r].x, s * v[r].y);
    }
  }
}

// Length-M FFT (M = 2^mshift >= 32) of a padded row slot, in shared memory;
// the last pass writes layout OUT.
// Threads with active == false take part in the barriers only (used when a
// shorter transform runs on a row slot sized for a longer one).
template <bool INV, int OUT>
__device__ __forceinline__ void fft_smem(float2* X, int M, int mshift, int lane, int tpr, const float2* tw,
                                         int twstride, bool active = true) {
  fft_pass<16, INV, kLayoutPadded>(X, M, 1, lane, tpr, tw, twstride, active);
  fft_rest<INV, OUT>(X, M, mshift, lane, tpr, tw, twstride, active);
}

// ---------------------------------------------------------------------------
// Node position x = c omega = B sqrt(S + az) in float-float arithmetic.
// Returns j0 = floor(x), fr = x - j0 in [0,1), and x0 = FP32 value of x.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void node_position(float2 S, float4 zt, float B2hi, float B2lo, int& j0, float& fr,
                                              float& rx) {
  // s = S + az (two-sum of the high parts, low parts added)
  float s_hi = __fadd_rn(S.x, zt.x);
  float bb = __fsub_rn(s_hi, S.x);
  float err = __fadd_rn(__fsub_rn(S.x, __fsub_rn(s_hi, bb)), __fsub_rn(zt.x, bb));
  float s_lo = __fadd_rn(err, __fadd_rn(S.y, zt.y));
  float t = __fadd_rn(s_hi, s_lo);
  s_lo = __fsub_rn(s_lo, __fsub_rn(t, s_hi));
  s_hi = t;
  // y = B^2 s
  float p = __fmul_rn(B2hi, s_hi);
  float e = fmaf(B2hi, s_hi, -p);
  e = fmaf(B2hi, s_lo, e);
  e = fmaf(B2lo, s_hi, e);
  float y_hi = __fadd_rn(p, e);
  float y_lo = __fsub_rn(e, __fsub_rn(y_hi, p));
  // x = sqrt(y): an FP32 root from the reciprocal square root (a few ulp)
  // plus one Newton correction from the exact residual, which leaves about
  // 44 bits; rx = 1/x to FP32 accuracy is the caller's (x = 0 only for the
  // zero-frequency node, where rx = 0)
  rx = y_hi > 0.0f ? rsqrtf(y_hi) : 0.0f;
  const float x0 = y_hi * rx;
  float q = __fmul_rn(x0, x0);
  float qe = fmaf(x0, x0, -q);
  float r = __fadd_rn(__fsub_rn(__fsub_rn(y_hi, q), qe), y_lo);
  float delta = 0.5f * r * rx;
  float fl = floorf(x0);
  j0 = (int)fl;
  fr = __fadd_rn(__fsub_rn(x0, fl), delta);
  if (fr < 0.0f) {
    fr += 1.0f;
    j0 -= 1;
  } else if (fr >= 1.0f) {
    fr -= 1.0f;
    j0 += 1;
  }
}

// The mirrored node -x = (-j0p - 1) + (1 - frp).  For an integer node fr = 1:
// the tap polynomials cover z = fr - 1/2 in [-1/2, 1/2] with both ends, and
// this is the tap set the forward pair evaluation (node_value_pair) uses.
__device__ __forceinline__ void negate_node(int j0p, float frp, int& j0, float& fr) {
  j0 = -j0p - 1;
  fr = 1.0f - frp;
}

// e^{+i pi nu} for nu = (j0 + fr) nt / M, returned as (cos, sin).
// The integer part is reduced exactly: pi j0 nt / M modulo 2 pi is
// pi m2 / M with m2 = j0 nt mod 2M.  When M = 2 nt that angle is a multiple of
// pi/2 and becomes an exact quarter-turn rotation.
__device__ __forceinline__ float2 node_phase(int j0, float fr, int nt, int M, float nt_over_M) {
  float s2, c2;
  sincospif(fr * nt_over_M, &s2, &c2);
  if (M == 2 * nt) {
    // multiply (c2, s2) by i^(j0 mod 4) with selects, no divergent branch
    const int q = j0 & 3;
    float a = (q & 1) ? -s2 : c2;
    float b = (q & 1) ? c2 : s2;
    if (q & 2) {
      a = -a;
      b = -b;
    }
    return make_float2(a, b);
  }
  const int m2 = (int)(((long long)j0 * (long long)nt) & (2LL * M - 1));
  float s1, c1;
  sincospif((float)m2 / (float)M, &s1, &c1);
  return make_float2(c1 * c2 - s1 * s2, s1 * c2 + c1 * s2);
}

// P(nu) = e^{-i pi nu} sum_t w_t G[(j0 + t) mod M], t = -H+1..H   (Eq. nufft-a).
// U is the flat spectrum with ghost cells: the 2H taps are U[b .. b+2H-1],
// b = (j0 - H + 1) mod M.  Weights are formed pair by pair (tap it and its
// mirror 2H-1-it) and consumed at once.
template <int H>
__device__ __forceinline__ float2 node_value(const float2* U, const WindowPoly& W, int j0, float fr, int M, int nt,
                                             float nt_over_M) {
  const float2* g = U + ((j0 - H + 1) & (M - 1));
  const float z = fr - 0.5f, z2 = z * z;
  float ax = 0.0f, ay = 0.0f;
#pragma unroll
  for (int p = 0; p < H; ++p) {
    float E = W.ce[p][kHalfCoef - 1], O = W.co[p][kHalfCoef - 1];
#pragma unroll
    for (int e = kHalfCoef - 2; e >= 0; --e) {
      E = fmaf(E, z2, W.ce[p][e]);
      O = fmaf(O, z2, W.co[p][e]);
    }
    const float wl = fmaf(z, O, E), wh = fmaf(-z, O, E);
    const float2 gl = g[p], gh = g[2 * H - 1 - p];
    ax = fmaf(wl, gl.x, ax);
    ay = fmaf(wl, gl.y, ay);
    ax = fmaf(wh, gh.x, ax);
    ay = fmaf(wh, gh.y, ay);
  }
  const float2 ph = node_phase(j0, fr, nt, M, nt_over_M);
  return make_float2(fmaf(ax, ph.x, ay * ph.y), fmaf(ay, ph.x, -ax * ph.y));
}

// Interpolation methods of Sec. 4 (no window, prescale 1): the oversampled DFT
// D_j = sum_n e^{-2 pi i j n / M} g_n sits on the grid nu_j = j nt / M, and the
// centred spectrum holds U[j] = e^{+i pi nu_j} D_j, so D_j = e^{-i pi nu_j} U[j mod M].
// LINEAR: (1 - fr) D_j0 + fr D_{j0+1};  NEAREST: D_{j0 + (fr >= 1/2)}.
__device__ __forceinline__ float2 grid_value(const float2* U, int j, int M, int nt, float nt_over_M) {
  const float2 u = U[j & (M - 1)];
  const float2 ph = node_phase(j, 0.0f, nt, M, nt_over_M);
  return make_float2(fmaf(u.x, ph.x, u.y * ph.y), fmaf(u.y, ph.x, -u.x * ph.y));
}

__device__ __forceinline__ float2 node_interp(const float2* U, int method, int j0, float fr, int M, int nt,
                                              float nt_over_M) {
  if (method == PAI_METHOD_NEAREST) return grid_value(U, j0 + (fr >= 0.5f ? 1 : 0), M, nt, nt_over_M);
  const float2 a = grid_value(U, j0, M, nt, nt_over_M);
  const float2 b = grid_value(U, j0 + 1, M, nt, nt_over_M);
  return make_float2(fmaf(fr, b.x - a.x, a.x), fmaf(fr, b.y - a.y, a.y));
}

// The value at a node by the problem's method.  Interpolation plans always run
// with H = 2, so the other instantiations carry no method branch.
template <int H>
__device__ __forceinline__ float2 node_eval(const RowProblem& P, const float2* U, const WindowPoly& W, int j0,
                                            float fr) {
  if constexpr (H == 2) {
    if (P.method >= PAI_METHOD_LINEAR) return node_interp(U, P.method, j0, fr, P.M, P.nt, P.nt_over_M);
  }
  return node_value<H>(U, W, j0, fr, P.M, P.nt, P.nt_over_M);
}

struct RowGeom {
  int d1, d2;     // destination rows (full lateral index) of +nu and -nu nodes
  bool mirror;    // row is not self-conjugate: both destinations are written
  float2 S;       // |K_lat/2pi|^2 as float-float
};

__device__ __forceinline__ RowGeom row_geom(const RowProblem& P, int row) {
  RowGeom g;
  const int half = P.n2 >> 1;
  const int i1 = row / (half + 1);
  const int i2 = row - i1 * (half + 1);
  g.mirror = (i2 > 0) && (i2 < half);
  g.d1 = i1 * P.n2 + i2;
  g.d2 = ((P.n1 - i1) % P.n1) * P.n2 + ((P.n2 - i2) % P.n2);
  g.S = P.rowS[row];
  return g;
}

// Node task i of a row: positive l' (1..nz/2-1), negative l' (mirror rows),
// and one Nyquist task evaluating both nodes at |l'| = nz/2.
__device__ __forceinline__ void node_task(int i, int nzh, int nA, int& lp, bool& neg, bool& nyq) {
  neg = false;
  nyq = false;
  if (i < nzh - 1) {
    lp = i + 1;
  } else if (i == nA - 1) {
    lp = nzh;
    nyq = true;
  } else {
    lp = i - (nzh - 1) + 1;
    neg = true;
  }
}

// Values at the node pair +x and -x (x = c nu = j0 + fr, fr in [0, 1)) from one
// evaluation of the tap polynomials.  The mirrored node is taken as
// -x = (-j0 - 1) + (1 - fr): its offset z' = (1 - fr) - 1/2 = -z, so its tap q
// weighs w_q(-z) = w_{2H-1-q}(z) (phi is even), and its phase
// e^{-i pi (-nu)} is the conjugate of the phase of +x.  Both values come out
// exactly as node_eval would give them for the two nodes, without rounding
// 1 - fr.
template <int H>
__device__ __forceinline__ void node_value_pair(const RowProblem& P, const float2* U, const WindowPoly& W, int j0,
                                                float fr, float2& vp, float2& vn) {
  if constexpr (H == 2) {
    if (P.method >= PAI_METHOD_LINEAR) {
      vp = node_interp(U, P.method, j0, fr, P.M, P.nt, P.nt_over_M);
      vn = node_interp(U, P.method, -j0 - 1, 1.0f - fr, P.M, P.nt, P.nt_over_M);
      return;
    }
  }
  const int mask = P.M - 1;
  const float2* gp = U + ((j0 - H + 1) & mask);
  const float2* gn = U + ((-j0 - H) & mask);
  const float z = fr - 0.5f, z2 = z * z;
  float ax = 0.0f, ay = 0.0f, bx = 0.0f, by = 0.0f;
#pragma unroll
  for (int p = 0; p < H; ++p) {
    float E = W.ce[p][kHalfCoef - 1], O = W.co[p][kHalfCoef - 1];
#pragma unroll
    for (int e = kHalfCoef - 2; e >= 0; --e) {
      E = fmaf(E, z2, W.ce[p][e]);
      O = fmaf(O, z2, W.co[p][e]);
    }
    const float wl = fmaf(z, O, E), wh = fmaf(-z, O, E);
    const float2 pl = gp[p], ph = gp[2 * H - 1 - p];
    const float2 nl = gn[p], nh = gn[2 * H - 1 - p];
    ax = fmaf(wl, pl.x, ax);
    ay = fmaf(wl, pl.y, ay);
    ax = fmaf(wh, ph.x, ax);
    ay = fmaf(wh, ph.y, ay);
    bx = fmaf(wh, nl.x, bx);
    by = fmaf(wh, nl.y, by);
    bx = fmaf(wl, nh.x, bx);
    by = fmaf(wl, nh.y, by);
  }
  const float2 ph = node_phase(j0, fr, P.nt, P.M, P.nt_over_M);
  vp = make_float2(fmaf(ax, ph.x, ay * ph.y), fmaf(ay, ph.x, -ax * ph.y));
  vn = make_float2(fmaf(bx, ph.x, -by * ph.y), fmaf(by, ph.x, bx * ph.y));
}

// Half image spectrum of one row (ZF = false layout): for l' = 1 .. nz/2 one
// task evaluates the node pair +-|K|; destination row d1 takes the +nu value,
// the conjugate row d2 (mirror rows only) the conjugate of the -nu value, and
// the Nyquist entry l' = nz/2 the mean of both (reading of the l = -nz/2 row).
// Self-conjugate rows (no mirror) need the -nu value only at the Nyquist entry.
template <int H>
__device__ __forceinline__ void gather_row(const RowProblem& P, const WindowPoly& W, const float2* X, int row,
                                           int lane) {
  const RowGeom rg = row_geom(P, row);
  const int nzh = P.nz >> 1;
  float2* out1 = P.fh + (size_t)rg.d1 * P.lz;
  float2* out2 = P.fh + (size_t)rg.d2 * P.lz;
  if (lane == 0) {
    out1[0] = make_float2(0.f, 0.f);
    if (rg.mirror) out2[0] = make_float2(0.f, 0.f);
  }
  // the depth-table entry of the next task is loaded one iteration ahead
  float4 zt_next = __ldg(&P.zt[min(lane, nzh - 1) + 1]);
  for (int i = lane; i < nzh; i += P.tpr) {
    const int lp = i + 1;
    const float4 zt = zt_next;
    if (i + P.tpr < nzh) zt_next = __ldg(&P.zt[lp + P.tpr]);
    int j0;
    float fr, rx;
    node_position(rg.S, zt, P.B2hi, P.B2lo, j0, fr, rx);
    const float wt = P.wscale * zt.z * rx;
    if (lp == nzh || rg.mirror) {
      float2 v, u;
      node_value_pair<H>(P, X, W, j0, fr, v, u);
      if (lp == nzh) {
        const float2 a = make_float2(0.5f * wt * (v.x + u.x), 0.5f * wt * (v.y + u.y));
        out1[lp] = a;
        if (rg.mirror) out2[lp] = make_float2(a.x, -a.y);
      } else {
        out1[lp] = make_float2(wt * v.x, wt * v.y);
        out2[lp] = make_float2(wt * u.x, -wt * u.y);
      }
    } else {
      const float2 v = node_eval<H>(P, X, W, j0, fr);
      out1[lp] = make_float2(wt * v.x, wt * v.y);
    }
  }
}

// Depth-row layout: the row's own full depth spectrum F[l], l in
// [-nz/2, nz/2), stored at Zs[l mod nz] (Zs = the row's line of the output),
// from the row's nodes at +nu (l > 0) and -nu (l < 0):  F[l] = W P(sign(l)|K|)
// for 0 < |l| < nz/2, F[0] = 0 (l = 0 rule), F[-nz/2] = W (P(+|K|) + P(-|K|))/2
// (Nyquist rule).  One task per |l| evaluates the node pair.  An inverse depth
// FFT of each line followed by the lateral C2R completes Eq. (fft-1).
template <int H>
__device__ __forceinline__ void gather_row_z(const RowProblem& P, const WindowPoly& W, const float2* X, float2* Zs,
                                             int row, int lane) {
  const float2 S = P.rowS[row];
  const int nzh = P.nz >> 1;
  if (lane == 0) Zs[0] = make_float2(0.f, 0.f);
  float4 zt_next = __ldg(&P.zt[min(lane, nzh - 1) + 1]);
  for (int i = lane; i < nzh; i += P.tpr) {
    const int lp = i + 1;
    const float4 zt = zt_next;
    if (i + P.tpr < nzh) zt_next = __ldg(&P.zt[lp + P.tpr]);
    int j0;
    float fr, rx;
    node_position(S, zt, P.B2hi, P.B2lo, j0, fr, rx);
    const float wt = P.wscale * zt.z * rx;
    float2 v, u;
    node_value_pair<H>(P, X, W, j0, fr, v, u);
    if (lp == nzh) {
      Zs[nzh] = make_float2(0.5f * wt * (v.x + u.x), 0.5f * wt * (v.y + u.y));
    } else {
      Zs[lp] = make_float2(wt * v.x, wt * v.y);
      Zs[P.nz - lp] = make_float2(wt * u.x, wt * u.y);
    }
  }
}

// The next work item for the whole CTA (dynamic scheduling).  A CTA's first
// item is its block index (the grid is never larger than the item list), so
// no CTA waits for a counter before it starts; every further item costs one
// atomic.  The CTAs fetch exactly nitems times in all (nitems - gridDim.x
// items and one empty fetch each), and the atomic counts modulo nitems, so it
// leaves zero for the next launch: no memset runs before the kernel (0.9 us plus
// a launch gap of about 1 us per pass before).  The same holds for launches of
// one shape that overlap (calls on one plan that nobody ordered): every nitems
// tickets hold one empty one per CTA of a launch, so the counter is at zero again
// when the last of them ends, whatever their order.  (Set back by a store of its
// own, it could lose tickets drawn in between, and a later call left out rows.)
__device__ __forceinline__ int next_item(const RowLaunch& L, int* s_item) {
  if (L.nitems <= (int)gridDim.x) return L.nitems;  // one item per CTA: the counter is not used
  __syncthreads();
  if (threadIdx.x == 0) {
    *s_item = (int)(gridDim.x + atomicInc(L.counter, (unsigned)(L.nitems - 1)));
  }
  __syncthreads();
  return *s_item;
}

// ZF = false: writes the half image spectrum fhat[k][l'] (both lateral
// destinations k and -k); ZF = true: writes the row's own full depth spectrum
// F[row][l mod nz] (see gather_row_z).
// PAIRED: the launch holds problems in the paired layout (RowProblem::paired);
// compiled apart so that the kernel of plans without them keeps its registers.
template <int H, bool ZF, bool PAIRED = false>
__global__ void __launch_bounds__(1024) row_forward_kernel(RowLaunch L, WindowPoly W) {
  extern __shared__ __align__(16) float2 smem[];
  __shared__ int s_item;
  pdl_wait();
  for (int item = blockIdx.x; item < L.nitems; item = next_item(L, &s_item)) {
    const WorkItem wi = L.items[item];
    const RowProblem& P = L.problems[wi.problem];
    const int tpr = P.tpr, M = P.M;
    const int slot = threadIdx.x / tpr;
    const int lane = threadIdx.x - slot * tpr;
    const int row = wi.row0 + slot;
    const bool valid = row < P.rows;
    float2* X = smem + slot * P.slot32;
    // first pass straight from the lateral spectrum row (rows past the end read row 0, unused)
    const int srow = valid ? row : 0;
    const bool paired = PAIRED && P.paired != 0;
    const float2* src = P.pt + (size_t)srow * (paired ? P.nt >> 1 : P.nt);
    const float2* src2 = P.pt + (size_t)(srow == 0 ? 0 : P.n2 - srow) * (P.nt >> 1);
    const bool r32 = first_pass32(M, P.mshift, P.nt);
    // (the layout is a template argument so that each path issues its loads
    // back to back)
    if (PAIRED && paired) {
      if (r32) fft_first_pass32_from_global<true>(X, M, P.nt, lane, tpr, src, P.prescale, src2);
      else fft_first_pass_from_global<true>(X, M, P.nt, lane, tpr, src, P.prescale, src2);
    } else {
      if (r32) fft_first_pass32_from_global<false>(X, M, P.nt, lane, tpr, src, P.prescale, src2);
      else fft_first_pass_from_global<false>(X, M, P.nt, lane, tpr, src, P.prescale, src2);
    }
    // (rotated twiddles only in radix-8 last passes: the register pressure of
    // the radix-2/4 ones costs this kernel more than the table loads)
    // (one pad per 32: a second instance of the passes for one pad per 16 cost this kernel more in registers than
    // the first pass's two-way store conflicts: 54.0 against 51.8 us at M = 8192, 137.8 against 135.2 us at 256^3)
    fft_rest<false, kLayoutFlatGhost, 8, 5>(X, M, P.mshift, lane, tpr, L.tw, L.Mmax >> P.mshift, true, r32 ? 5 : 4);
    if (valid) {
      if (!ZF) gather_row<H>(P, W, X, row, lane);
      else gather_row_z<H>(P, W, X, P.fh + (size_t)row * P.nz, row, lane);
    }
  }
}

// ---------------------------------------------------------------------------
// Adjoint
// ---------------------------------------------------------------------------

// Adjoint of the node evaluation.  Windowed methods: the node record carries
// e^{+i pi nu} (the transpose of the node's phase) and the taps weigh
// w_t(fr).  Interpolation methods (H = 2 plans only): the phase belongs to the
// grid cell, e^{+i pi nu_j}, applied to each cell after the spread, and tap
// t = 1, 2 (cells j0, j0+1) weigh 1 - fr, fr (linear) or 1 on the nearer cell.
template <int H>
__device__ __forceinline__ float2 adj_node_phase(const RowProblem& P, int j0, float fr) {
  if constexpr (H == 2) {
    if (P.method >= PAI_METHOD_LINEAR) return make_float2(1.0f, 0.0f);
  }
  return node_phase(j0, fr, P.nt, P.M, P.nt_over_M);
}

__device__ __forceinline__ float interp_tap_weight(int method, int t, float fr) {
  if (method == PAI_METHOD_NEAREST) return (t == 1) ? (fr >= 0.5f ? 0.0f : 1.0f) : (t == 2 ? (fr >= 0.5f ? 1.0f : 0.0f) : 0.0f);
  return (t == 1) ? 1.0f - fr : (t == 2 ? fr : 0.0f);
}

// Where a row's node pairs come from.
struct PairSrc {
  const float2* a;  // ZF: the row's depth spectrum; else the +k line of the half spectrum
  const float2* b;  // else: the -k line
  float2 S;         // |K_lat / 2 pi|^2 as float-float
  bool mirror;      // the row has -nu nodes below the Nyquist entry
};
// The depth index of node pair 0: forward models have a pair at depth frequency 0 too.
template <bool Q>
constexpr int kFirstPair = Q ? 0 : 1;

// Node pair i of a row: the nodes +-x of one depth index l = i + kFirstPair,
// x = j0 + fr, and their values Q+ = qp, Q- = qn: the
// input times the weight and the transpose of the node's phase, e^{+i pi nu}
// for +x and its conjugate for -x.  Q (forward model): both nodes carry c_l / 2
// (wscale holds 1 / (2 n_lat nz)).
template <bool ZF, bool Q>
__device__ __forceinline__ void pair_node(const RowProblem& P, const PairSrc& src, int i, int& j0, float& fr,
                                          float2& qp, float2& qn) {
  const int nzh = P.nz >> 1;
  const int lp = i + kFirstPair<Q>;
  const float4 zt = __ldg(&P.zt[lp]);
  float rx;
  node_position(src.S, zt, P.B2hi, P.B2lo, j0, fr, rx);
  const float2 ph = node_phase(j0, fr, P.nt, P.M, P.nt_over_M);
  float2 yp, yn;  // inputs of the two nodes, real weights applied
  const float wt = P.wscale * zt.z * rx;
  if (Q) {
    const float2 y = src.a[lp];
    yp = yn = make_float2(P.wscale * y.x, P.wscale * y.y);
  } else if (lp == nzh) {
    // Nyquist: both nodes carry half the l = -nz/2 input
    float2 y = src.a[lp];
    if (!ZF && src.mirror) {
      const float2 y2 = src.b[lp];
      y = make_float2(y.x + y2.x, y.y - y2.y);
    }
    yp = yn = make_float2(0.5f * wt * y.x, 0.5f * wt * y.y);
  } else if (ZF) {
    const float2 y = src.a[lp], y2 = src.a[P.nz - lp];
    yp = make_float2(wt * y.x, wt * y.y);
    yn = make_float2(wt * y2.x, wt * y2.y);
  } else {
    const float2 y = src.a[lp];
    yp = make_float2(2.0f * wt * y.x, 2.0f * wt * y.y);
    yn = make_float2(0.f, 0.f);  // self-conjugate row: no -nu node below the Nyquist entry
    if (src.mirror) {
      const float2 y2 = src.b[lp];
      yn = make_float2(2.0f * wt * y2.x, -2.0f * wt * y2.y);
    }
  }
  qp = cmul(yp, ph);
  qn = cmul(yn, make_float2(ph.x, -ph.y));
}

// Cells of a band grid: WIDE 16 bytes (two complex values that take the same
// weights), else 8 bytes (one).
template <bool WIDE>
struct Cell {
  float4 v;
};
template <>
struct Cell<false> {
  float2 v;
};
template <bool WIDE>
constexpr int kCellShift = WIDE ? 4 : 3;

template <bool WIDE>
__device__ __forceinline__ Cell<WIDE> cell_zero() {
  if constexpr (WIDE) return {make_float4(0.f, 0.f, 0.f, 0.f)};
  else return {make_float2(0.f, 0.f)};
}
template <bool WIDE>
__device__ __forceinline__ Cell<WIDE> cell_load(unsigned a) {
  if constexpr (WIDE) return {lds4(a)};
  else return {lds2(a)};
}
template <bool WIDE>
__device__ __forceinline__ void cell_store(unsigned a, const Cell<WIDE>& c) {
  if constexpr (WIDE) sts4(a, c.v);
  else sts2(a, c.v);
}
template <bool WIDE>
__device__ __forceinline__ Cell<WIDE> cell_add(const Cell<WIDE>& a, const Cell<WIDE>& b) {
  if constexpr (WIDE) {
    const float2 p = cadd(make_float2(a.v.x, a.v.y), make_float2(b.v.x, b.v.y));
    const float2 n = cadd(make_float2(a.v.z, a.v.w), make_float2(b.v.z, b.v.w));
    return {make_float4(p.x, p.y, n.x, n.y)};
  } else {
    return {cadd(a.v, b.v)};
  }
}
// w q + g
template <bool WIDE>
__device__ __forceinline__ Cell<WIDE> cell_axpy(float w, const Cell<WIDE>& q, const Cell<WIDE>& g) {
  const float2 ww = make_float2(w, w);
  if constexpr (WIDE) {
    const float2 p = fma2(ww, make_float2(q.v.x, q.v.y), make_float2(g.v.x, g.v.y));
    const float2 n = fma2(ww, make_float2(q.v.z, q.v.w), make_float2(g.v.z, g.v.w));
    return {make_float4(p.x, p.y, n.x, n.y)};
  } else {
    return {fma2(ww, q.v, g.v)};
  }
}
template <bool WIDE>
__device__ __forceinline__ Cell<WIDE> cell_shfl_down(const Cell<WIDE>& c, int d) {
  const unsigned full = 0xffffffffu;
  if constexpr (WIDE)
    return {make_float4(__shfl_down_sync(full, c.v.x, d), __shfl_down_sync(full, c.v.y, d),
                        __shfl_down_sync(full, c.v.z, d), __shfl_down_sync(full, c.v.w, d))};
  else
    return {make_float2(__shfl_down_sync(full, c.v.x, d), __shfl_down_sync(full, c.v.y, d))};
}
// Address of cell i (four phases, see Band).
template <bool WIDE>
__device__ __forceinline__ unsigned cell_at(const Band& b, int i) {
  return b.grid + (((i & 3) * b.ps + (i >> 2)) << kCellShift<WIDE>);
}

// Tap addresses of one lane: tap t of a node whose first cell is cell0 sits at
// a[t & 3] plus t / 4 cells (the four phases make every tap offset but four a
// constant), or, for the first nspill taps, in the warp's spill.
template <bool WIDE>
struct BandTaps {
  unsigned a[4];
  unsigned spill;
  int nspill;
  __device__ __forceinline__ BandTaps(const Band& b, int cell0, unsigned spill_at, int ns)
      : spill(spill_at), nspill(ns) {
#pragma unroll
    for (int j = 0; j < 4; ++j) a[j] = cell_at<WIDE>(b, cell0 + j);
  }
  __device__ __forceinline__ unsigned direct(int t) const { return a[t & 3] + ((t >> 2) << kCellShift<WIDE>); }
  __device__ __forceinline__ unsigned at(int t) const {
    return t < nspill ? spill + (t << kCellShift<WIDE>) : direct(t);
  }
};

// Runs of lanes with equal j0 within a group of gw lanes (nodes are sorted).
struct Runs {
  bool head;    // first lane of its run
  int first;    // that lane
  int last;     // last lane of this lane's run
  int maxrun;   // longest run of the warp
  int mingap;   // least distance of neighbouring runs
  bool sorted;  // rounding did not swap neighbouring nodes
};
__device__ __forceinline__ Runs find_runs(int j0, bool act, int gw) {
  const unsigned full = 0xffffffffu;
  const int l32 = threadIdx.x & 31;
  const bool first = (l32 & (gw - 1)) == 0;
  const int prev = __shfl_up_sync(full, j0, 1);
  Runs r;
  r.head = act && (first || prev != j0);
  const unsigned heads = __ballot_sync(full, r.head), actm = __ballot_sync(full, act);
  const unsigned stop = (heads | ~actm) & (0xfffffffeu << l32);  // the run ends before the next head or idle lane
  r.last = stop ? __ffs(stop) - 2 : 31;
  const unsigned mine = heads & (0xffffffffu >> (31 - l32));
  r.first = mine ? 31 - __clz(mine) : l32;
  r.maxrun = __reduce_max_sync(full, (unsigned)(r.head ? r.last - l32 + 1 : 0));
  r.mingap = __reduce_min_sync(full, (unsigned)(r.head && !first ? max(j0 - prev, 0) : 1 << 20));
  r.sorted = __all_sync(full, !(act && !first && prev > j0));
  return r;
}

template <int H>
__device__ __forceinline__ void tap_pair(const WindowPoly& W, int p, float z, float z2, float& wl, float& wh) {
  float E = W.ce[p][kHalfCoef - 1], O = W.co[p][kHalfCoef - 1];
#pragma unroll
  for (int e = kHalfCoef - 2; e >= 0; --e) {
    E = fmaf(E, z2, W.ce[p][e]);
    O = fmaf(O, z2, W.co[p][e]);
  }
  wl = fmaf(z, O, E);
  wh = fmaf(-z, O, E);
}

// Spreads one node per lane: q times its 2H weights.  Nodes on one cell (a run
// of lanes) take turns; in each turn lanes write distinct cells at one tap,
// neighbouring taps of different lanes may meet, so a __syncwarp separates
// them.  Where all neighbouring nodes are two or more cells apart, two adjacent
// taps of all lanes are still distinct cells and go together.  Long runs (nodes
// crowd where the lateral frequency dominates) sum by shuffles instead: their
// first lane adds.  The order of a cell's terms is fixed in every case.
template <int H, bool WIDE>
__device__ __forceinline__ void band_spread(const WindowPoly& W, const BandTaps<WIDE>& tp, int j0, float fr,
                                            const Cell<WIDE>& q, bool act, int gw) {
  const float z = fr - 0.5f, z2 = z * z;
  const Runs r = find_runs(j0, act, gw);
  float w[2 * H];
#pragma unroll
  for (int p = 0; p < H; ++p) tap_pair<H>(W, p, z, z2, w[p], w[2 * H - 1 - p]);
  const bool ordered = r.sorted && r.maxrun <= 1;
  if (ordered && r.mingap >= 2 && __all_sync(0xffffffffu, tp.nspill <= 0 || !act)) {
#pragma unroll
    for (int t = 0; t < 2 * H; t += 2) {
      if (act) {
        const Cell<WIDE> g0 = cell_load<WIDE>(tp.direct(t)), g1 = cell_load<WIDE>(tp.direct(t + 1));
        cell_store<WIDE>(tp.direct(t), cell_axpy<WIDE>(w[t], q, g0));
        cell_store<WIDE>(tp.direct(t + 1), cell_axpy<WIDE>(w[t + 1], q, g1));
      }
      __syncwarp();
    }
  } else if (r.sorted && r.maxrun > 4) {
    const int l32 = threadIdx.x & 31;
#pragma unroll
    for (int t = 0; t < 2 * H; ++t) {
      Cell<WIDE> v = cell_axpy<WIDE>(w[t], q, cell_zero<WIDE>());
      for (int d = 1; d < r.maxrun; d <<= 1) {
        const Cell<WIDE> u = cell_shfl_down<WIDE>(v, d);
        if (l32 + d <= r.last) v = cell_add<WIDE>(v, u);
      }
      if (r.head) {
        const unsigned a = tp.at(t);
        cell_store<WIDE>(a, cell_add<WIDE>(cell_load<WIDE>(a), v));
      }
      __syncwarp();
    }
  } else {
    // this lane's turn: its place in its run (any lane of its own where rounding swapped two neighbours)
    const int turn = r.sorted ? (threadIdx.x & 31) - r.first : (threadIdx.x & (gw - 1));
    const int turns = r.sorted ? r.maxrun : gw;
    for (int k = 0; k < turns; ++k) {
      const bool on = act && turn == k;
#pragma unroll
      for (int t = 0; t < 2 * H; ++t) {
        if (on) {
          const unsigned a = tp.at(t);
          cell_store<WIDE>(a, cell_axpy<WIDE>(w[t], q, cell_load<WIDE>(a)));
        }
        __syncwarp();
      }
    }
  }
}

// Spreads two neighbouring nodes A and B per lane, d = 0, 1 or 2 cells apart:
// their 2H + 2 cells take both nodes' terms in one read and write each, B's
// weights shifted by d, so a node costs H + 1 accesses instead of 2H, and lanes
// share a cell only where four nodes do.  Runs sum by shuffles.
template <int H, bool WIDE>
__device__ __forceinline__ void band_spread2(const WindowPoly& W, const BandTaps<WIDE>& tp, int j0, float fa,
                                             const Cell<WIDE>& qa, bool act, int gw, int d, float fb,
                                             const Cell<WIDE>& qb) {
  const float za = fa - 0.5f, za2 = za * za, zb = fb - 0.5f, zb2 = zb * zb;
  const Runs r = find_runs(j0, act, gw);
  const int l32 = threadIdx.x & 31;
  // cell u: wa A + (b0, b1 or b2) B, the three candidates for d = 0, 1, 2
  auto cell = [&](int u, float wa, float b0, float b1, float b2) {
    const float wb = d == 0 ? b0 : d == 1 ? b1 : b2;
    const unsigned a = tp.at(u);
    if (r.maxrun <= 1) {
      if (act) cell_store<WIDE>(a, cell_axpy<WIDE>(wb, qb, cell_axpy<WIDE>(wa, qa, cell_load<WIDE>(a))));
    } else {
      Cell<WIDE> v = cell_axpy<WIDE>(wb, qb, cell_axpy<WIDE>(wa, qa, cell_zero<WIDE>()));
      for (int k = 1; k < r.maxrun; k <<= 1) {
        const Cell<WIDE> t = cell_shfl_down<WIDE>(v, k);
        if (l32 + k <= r.last) v = cell_add<WIDE>(v, t);
      }
      if (r.head) cell_store<WIDE>(a, cell_add<WIDE>(cell_load<WIDE>(a), v));
    }
    __syncwarp();
  };
  // from both ends inwards: lower and upper weights of this and the last two pairs
  float l1 = 0.f, l2 = 0.f, u1 = 0.f, u2 = 0.f, ua1 = 0.f, ua2 = 0.f;
#pragma unroll
  for (int p = 0; p < H; ++p) {
    float la, ha, lb, hb;
    tap_pair<H>(W, p, za, za2, la, ha);
    tap_pair<H>(W, p, zb, zb2, lb, hb);
    cell(p, la, lb, l1, l2);
    cell(2 * H + 1 - p, ua2, u2, u1, hb);
    l2 = l1;
    l1 = lb;
    u2 = u1;
    u1 = hb;
    ua2 = ua1;
    ua1 = ha;
  }
  cell(H, ua1, u1, l1, l2);
  cell(H + 1, ua2, u2, u1, l1);
}

// A row's (or unit's) sorted nodes divided over its warps, and the part of the
// band each warp adds to.  Cells at or below the predecessor's last cell go to
// the warp's own spill of kSpill cells and are merged after a barrier; all
// others the warp owns alone, so it zeroes them and begins without a barrier.
template <int H>
struct BandPart {
  // a pass over two nodes adds (zeros) up to kReach cells beyond the second one's last
  static constexpr int kReach = 2;
  static constexpr int kSpill = 2 * H + 4 + kReach;  // at most 32
  int nw, wa, w;       // warps, warps with nodes (as few as hold 32 each, at most nw; np is shared evenly), this warp
  int gw, l;           // lanes per row in a warp, this lane's place
  int n0, n1;          // this warp's nodes
  int lo_w, hi_prev;   // first cell of this warp's nodes, last cell of its predecessor's
  unsigned spills, spill_w;
  int2* bnd;           // first cell and last cell per warp (shared memory)
};

// Sets up the parts and zeroes the cells this warp owns and its spill.
// position(i): cell index j0 of node i.  One cell to spare on either side,
// should rounding swap two neighbouring nodes.
template <int H, bool WIDE, typename Pos>
__device__ __forceinline__ void band_begin(BandPart<H>& b, Band& band, char* slot, int ps, int np, int lane, int threads,
                                           Pos position) {
  constexpr int kSpill = BandPart<H>::kSpill, kShift = kCellShift<WIDE>;
  b.nw = threads > 32 ? threads >> 5 : 1;
  b.gw = threads < 32 ? threads : 32;
  b.w = threads > 32 ? lane >> 5 : 0;
  b.l = lane & (b.gw - 1);
  b.wa = min(b.nw, (np + 31) >> 5);
  const bool on = b.w < b.wa;
  b.n0 = on ? np * b.w / b.wa : np;
  b.n1 = on ? np * (b.w + 1) / b.wa : np;
  band.grid = smem_addr(slot);
  band.ps = ps;
  band.lo = 0;
  band.n = 0;
  b.spills = band.grid + ((4 * ps) << kShift);
  b.spill_w = b.spills + ((b.w * kSpill) << kShift);
  b.bnd = reinterpret_cast<int2*>(slot + ((4 * ps + (b.nw > 1 ? b.nw * kSpill : 0)) << kShift));
  // lanes 0 .. 3: first node of the row, last of this warp, first of this warp, last of the predecessor
  int j = 0;
  if (on && b.l < 4) j = position(b.l == 0 ? 0 : b.l == 1 ? b.n1 - 1 : b.l == 2 ? b.n0 : max(b.n0 - 1, 0));
  const unsigned full = 0xffffffffu;
  const int j_row = __shfl_sync(full, j, 0, b.gw), j_last = __shfl_sync(full, j, 1, b.gw);
  const int j_first = b.nw > 1 ? __shfl_sync(full, j, 2) : j_row, j_prev = b.nw > 1 ? __shfl_sync(full, j, 3) : j_row;
  band.lo = j_row - H;
  b.lo_w = j_first - H;
  b.hi_prev = b.w > 0 ? j_prev + H + 1 + BandPart<H>::kReach : -(1 << 30);
  if (on) {
    const int hi = j_last + H + 1 + BandPart<H>::kReach;
    if (b.l == 0) b.bnd[b.w] = make_int2(b.lo_w, hi);
    const Cell<WIDE> zero = cell_zero<WIDE>();
    for (int c = (b.w > 0 ? b.hi_prev + 1 - band.lo : 0) + b.l; c <= hi - band.lo; c += b.gw)
      cell_store<WIDE>(cell_at<WIDE>(band, c), zero);
    if (b.nw > 1 && b.l < kSpill) cell_store<WIDE>(b.spill_w + (b.l << kShift), zero);
  }
  __syncwarp();
}

// After the spread's barrier: merges the spills (a cell spilled by several
// warps is summed by the first of them, in warp order) and sets band.n.
// fold: cells `fold` apart are one grid value (bands longer than that, for
// coarse time steps or tiny grids, are folded).  uniform over the CTA: nw, ps.
template <int H, bool WIDE>
__device__ __forceinline__ void band_end(const BandPart<H>& b, Band& band, int lane, int threads, int fold) {
  constexpr int kSpill = BandPart<H>::kSpill, kShift = kCellShift<WIDE>;
  if (b.wa > 0) {
    band.lo = b.bnd[0].x;  // (warps without nodes do not have it)
    band.n = b.bnd[b.wa - 1].y + 1 - band.lo;
  }
  if (b.nw > 1) {
    const int c = b.lo_w + b.l;
    if (b.w > 0 && b.w < b.wa && b.l < kSpill && c <= b.hi_prev && (b.w == 1 || c > b.bnd[b.w - 2].y)) {
      const unsigned a = cell_at<WIDE>(band, c - band.lo);
      Cell<WIDE> s = cell_load<WIDE>(a);
      for (int v = b.w; v < b.wa && c >= b.bnd[v].x; ++v)
        s = cell_add<WIDE>(s, cell_load<WIDE>(b.spills + ((v * kSpill + c - b.bnd[v].x) << kShift)));
      cell_store<WIDE>(a, s);
    }
    __syncthreads();
  }
  if (4 * band.ps > fold) {
    for (int i = lane; i < fold && i < band.n - fold; i += threads) {
      const unsigned a = cell_at<WIDE>(band, i);
      Cell<WIDE> g = cell_load<WIDE>(a);
      for (int k = i + fold; k < band.n; k += fold) g = cell_add<WIDE>(g, cell_load<WIDE>(cell_at<WIDE>(band, k)));
      cell_store<WIDE>(a, g);
    }
    __syncthreads();
    band.n = min(band.n, fold);
  }
}

// Adjoint of one row by node pairs (spread mode 3, windowed methods): the
// transpose of the gather, deterministic and without atomics.
//
// The -x node of a pair is taken as (-j0 - 1) + (1 - fr), as the forward
// gather takes it, so its tap at cell -c weighs what the +x node's tap at cell
// c weighs.  Both therefore add with one weight to one 16-byte (WIDE) cell of the
// band grid (struct Band), which covers only the cells the row's nodes reach:
// one read and one write of 16 bytes per tap and pair, half the accesses of
// two separate complex cells.  The first inverse FFT pass reads the grid
// values from the band.
//
// The row's warps take contiguous blocks of the sorted pairs (BandPart).  A
// pair's values are formed right before they are spread (no list in shared
// memory).
//
// What bounds it: shared-memory accesses (32 bytes per tap and pair; 256^3: 81 %
// of their peak, 38 % of the wavefronts bank conflicts, issue slots 55 %), in
// long rows with fewer CTAs also the latency of the tap chain and the barriers
// (2048x4096: 61 % and 42 %); 64 registers at 32 warps per SM measured
// best (56: +6 %, 90 and half the warps: +16 %).  The lists, run sums and float
// atomics it replaced held one CTA per SM for long rows and serialised on equal
// cells: 2048x4096 (M = 8192, H = 8) 126 -> 91 us, 256^3 (M = 1024, H = 6) 224 ->
// 221 us, 666x1500 (M = 4096) 21.6 -> 18.3 us.  Spreading two pairs per lane as
// the forward model does paid at 256^3 (216 us) but not for longer rows or wider
// windows (105 and 19.6 us), whose weights leave the registers.
template <int H, bool ZF, bool Q>
__device__ __forceinline__ bool adjoint_band(const RowProblem& P, const WindowPoly& W, int row, bool valid, int lane,
                                             float2* X, Band& band) {
  PairSrc src{nullptr, nullptr, make_float2(0.f, 0.f), true};
  int np = 0;
  if (valid) {
    np = (P.nz >> 1) + 1 - kFirstPair<Q>;
    if (ZF) {
      src.a = P.fh + (size_t)row * P.zstride;
      src.S = P.rowS[row];
    } else {
      const RowGeom rg = row_geom(P, row);
      src.a = P.fh + (size_t)rg.d1 * P.lz;
      src.b = P.fh + (size_t)rg.d2 * P.lz;
      src.S = rg.S;
      src.mirror = rg.mirror;
    }
  }
  BandPart<H> part;
  band_begin<H, true>(part, band, reinterpret_cast<char*>(X), P.band_ps, np, lane, P.tpr, [&](int i) {
    int j0;
    float fr, rx;
    node_position(src.S, __ldg(&P.zt[i + kFirstPair<Q>]), P.B2hi, P.B2lo, j0, fr, rx);
    return j0;
  });
  // chunks: uniform over the warp (rows sharing a warp have equal counts, or none)
  const int cn = __reduce_max_sync(0xffffffffu, (unsigned)(part.n1 - part.n0));
  for (int c0 = 0; c0 < cn; c0 += part.gw) {
    const int i = part.n0 + c0 + part.l;
    const bool act = i < part.n1;
    int j0 = 0;
    float fr = 0.5f;
    float2 qp = make_float2(0.f, 0.f), qn = qp;
    if (act) pair_node<ZF, Q>(P, src, i, j0, fr, qp, qn);
    const int c = j0 - H + 1;  // first cell
    const BandTaps<true> tp(band, c - band.lo, part.spill_w + ((c - part.lo_w) << 4), part.hi_prev + 1 - c);
    band_spread<H, true>(W, tp, j0, fr, Cell<true>{make_float4(qp.x, qp.y, qn.x, qn.y)}, act, part.gw);
  }
  __syncthreads();  // every warp's cells and spills are complete
  band_end<H, true>(part, band, lane, P.tpr, P.M);
  return src.mirror;
}

// The adjoint row kernel with the pair spread (spread mode 3), a kernel of its
// own so that its register allocation does not carry the other schemes.  Q: the
// discrete forward model by node pairs, for windows that row_model_kernel is not
// used for (see there) and rows that do not fit it.
template <int H, bool ZF, bool Q = false>
__global__ void __launch_bounds__(1024) row_adjoint_pairs_kernel(RowLaunch L, WindowPoly W) {
  extern __shared__ __align__(16) float2 smem[];
  __shared__ int s_item;
  pdl_wait();
  for (int item = blockIdx.x; item < L.nitems; item = next_item(L, &s_item)) {
    const WorkItem wi = L.items[item];
    const RowProblem& P = L.problems[wi.problem];
    const int tpr = P.tpr, M = P.M, nt = P.nt;
    const int slot = threadIdx.x / tpr;
    const int lane = threadIdx.x - slot * tpr;
    const int row = wi.row0 + slot;
    const bool valid = row < P.rows;
    float2* X = smem + slot * P.band_slot;
    Band band;
    const bool mirror = adjoint_band<H, ZF, Q>(P, W, row, valid, lane, X, band);
    const float scale = (valid && !ZF && mirror) ? 0.5f : 1.0f;
    float2* dst = const_cast<float2*>(P.pt) + (size_t)(valid ? row : 0) * nt;
    fft_inverse_crop<true>(X, M, P.mshift, nt, lane, tpr, L.tw, L.Mmax >> P.mshift, dst, P.prescale, scale, valid,
                           band);
  }
}

// t a + conj(t) b
__device__ __forceinline__ float2 model_sample(float2 t, float2 a, float2 b) {
  return fma2(make_float2(t.x, t.x), cadd(a, b), mul2(make_float2(t.y, t.y), make_float2(b.y - a.y, a.x - b.x)));
}

// Last pass of the forward model's transform (radix R < 16, Ns = M/R) with its
// samples g_n = t_n V[n] + conj(t_n) V[M - n], n < nt, formed in registers: M - n
// of butterfly j's outputs j + r Ns are those of butterfly Ns - j, so a thread
// takes the butterflies q and Ns - q together (q = 0: 0 and Ns/2, each its own
// mirror).  Saves a write and two reads of the row in shared memory.
template <int R>
__device__ __forceinline__ void model_last(const float2* X, int M, int nt, int lane, int tpr,
                                           const float2* __restrict__ tw, int twstride,
                                           const float2* __restrict__ tab, float2* dst) {
  const int Ns = M / R;
#pragma unroll
  for (int i = 0; i < 8 / R; ++i) {
    const int q = lane + i * tpr;
    const int ja = q, jb = q == 0 ? Ns >> 1 : Ns - q;
    float2 a[R], b[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      a[r] = X[padi(ja + r * Ns)];
      b[r] = X[padi(jb + r * Ns)];
    }
    TwBase<R> t;
    tw_load<R>(t, tw, ja * twstride);
    tw_apply<R, false>(a, t);
    tw_load<R>(t, tw, jb * twstride);
    tw_apply<R, false>(b, t);
    dft_reg<R, false>(a);
    dft_reg<R, false>(b);
    if (!dst) continue;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int na = ja + r * Ns, nb = jb + r * Ns;
      if (na < nt) dst[na] = model_sample(__ldg(&tab[na]), a[r], q == 0 ? a[(R - r) % R] : b[R - 1 - r]);
      if (nb < nt) dst[nb] = model_sample(__ldg(&tab[nb]), b[r], q == 0 ? b[R - 1 - r] : a[R - 1 - r]);
    }
  }
}

// Forward-model row kernel (the operator Q of Sec. 2 on a padded periodic
// box).  A row's samples are g_n = sum_j c_j cos(2 pi nu_j n / nt), j =
// 0..nz/2, nu_j >= 0 the frequency of |K| (j = 0 included: its frequency is
// the lateral |K|); Zs[j] holds c_j.
//
// The sum is even in n, so it is taken as a NUFFT over the interval (-nt, nt),
// centred at n = 0: a grid of 2M cells at the half-integers m + 1/2, nodes at
// x' = 2 x - 1/2, real window weights and no node phases; the mirrored nodes
// are the reflection m -> -1 - m.  What is left is a cosine transform of M
// cells (type II), taken as one complex transform of length M: with V1 the sum
// over the nodes (no mirror), v[e] = V1[2e] + V1[-1-2e] (indices modulo 2M) and
// its transform V,
//   g_n = t_n V[n] + conj(t_n) V[M - n],   t_n = s_n e^{-i pi n / (2M)},
// s_n the window's prescale over the doubled interval.  Against the node pairs
// of the adjoint (two nodes with phases per index) this halves the values
// spread and drops a sine and cosine per node.  The window's error falls on other
// samples than with the node pairs, so only windows whose error is below rounding
// take this kernel; the others keep the pairs in band grids
// (row_adjoint_pairs_kernel; truncated sinc, 12 taps, 128^3: 1369 us a call, 2683
// with the pair warps and the stored box before both).
//
// PAIR (3-D): rows k1 and -k1 have the same |K| and so the same nodes; a unit
// of 2 tpr threads spreads both rows' values with one set of weights into
// 16-byte cells, then transforms one row with each half of its threads.
//
// What bounds it: shared-memory accesses and instruction issue (128^3: 81 % of
// their peak and 65 % of the slots; 2048x4096: 63 and 60 %, and barriers), about a
// third of the issue node positions and weights.
// 128^3 in its 512^3 box (131 584 rows, M = 512): 1264 us with the node pairs of
// the adjoint and their lists, 957 us with them in band grids, 675 us as this
// kernel, 604 us with two nodes per lane (band_spread2); 2048x4096 in 8192^2
// (4097 rows, M = 8192): 1455, 584, 602 and 477 us; with the last pass forming
// the samples (model_last) another 27 us less each.
template <int H, bool PAIR>
__global__ void __launch_bounds__(1024) row_model_kernel(RowLaunch L, WindowPoly W) {
  extern __shared__ __align__(16) float2 smem[];
  __shared__ int s_item;
  pdl_wait();
  constexpr int kShift = kCellShift<PAIR>;
  for (int item = blockIdx.x; item < L.nitems; item = next_item(L, &s_item)) {
    const WorkItem wi = L.items[item];
    const RowProblem& P = L.problems[wi.problem];
    const int tpr = P.tpr, M = P.M, nzh = P.nz >> 1;
    const int tpu = PAIR ? 2 * tpr : tpr;
    const int slot = threadIdx.x / tpu;
    const int lane_u = threadIdx.x - slot * tpu;
    const int sub = PAIR ? lane_u / tpr : 0, lane = lane_u - sub * tpr;
    const int unit = wi.row0 + slot;
    const bool valid = unit < (PAIR ? (P.n1 / 2 + 1) * (P.n2 / 2 + 1) : P.rows);
    int row_b = -1;  // the partner row (k1, k2) -> (-k1, k2)
    if (PAIR && valid) {
      const int half1 = P.n2 / 2 + 1, i1 = unit / half1;
      if (i1 > 0 && i1 < P.n1 / 2) row_b = (P.n1 - i1) * half1 + (unit - i1 * half1);
    }
    float2* U = smem + (size_t)slot * P.model_slot;
    const float2* za = P.fh + (size_t)(valid ? unit : 0) * P.zstride;
    const float2* zb = P.fh + (size_t)(row_b >= 0 ? row_b : 0) * P.zstride;
    const float2 S = valid ? P.rowS[unit] : make_float2(0.f, 0.f);
    // cell index and fraction of node i on the half-integer grid
    auto node = [&](int i, int& j0, float& fr) {
      float rx;
      node_position(S, __ldg(&P.zt[i]), 4.0f * P.B2hi, 4.0f * P.B2lo, j0, fr, rx);
      fr -= 0.5f;
      if (fr < 0.0f) {
        fr += 1.0f;
        j0 -= 1;
      }
    };
    Band band;
    BandPart<H> part;
    band_begin<H, PAIR>(part, band, reinterpret_cast<char*>(U), P.model_ps, valid ? nzh + 1 : 0, lane_u, tpu, [&](int i) {
      int j0;
      float fr;
      node(i, j0, fr);
      return j0;
    });
    auto value = [&](int i) {
      const float2 ya = za[i];
      if constexpr (PAIR) {
        const float2 yb = row_b >= 0 ? zb[i] : make_float2(0.f, 0.f);
        return Cell<true>{make_float4(P.wscale * ya.x, P.wscale * ya.y, P.wscale * yb.x, P.wscale * yb.y)};
      } else {
        return Cell<false>{make_float2(P.wscale * ya.x, P.wscale * ya.y)};
      }
    };
    const int cn = __reduce_max_sync(0xffffffffu, (unsigned)(part.n1 - part.n0));
    for (int c0 = 0; c0 < cn;) {
      // two nodes per lane while there are enough and they are at most two cells apart
      const bool two = P.model_dense && cn - c0 > part.gw;
      const int step = two ? 2 : 1;
      const int i = part.n0 + c0 + step * part.l;
      c0 += step * part.gw;
      const bool act = i < part.n1;
      int j0 = 0, jb = 0;
      float fr = 0.5f, fb = 0.5f;
      Cell<PAIR> q = cell_zero<PAIR>(), qb = q;
      if (act) {
        q = value(i);
        node(i, j0, fr);
        jb = j0;
      }
      if (two) {
        const bool actb = i + 1 < part.n1;
        if (actb) {
          qb = value(i + 1);
          node(i + 1, jb, fb);
        }
        const int prev = __shfl_up_sync(0xffffffffu, jb, 1);
        // (rounding may move a node by a cell: then one at a time)
        if (__all_sync(0xffffffffu, !act || (jb >= j0 && jb <= j0 + 2 && (part.l == 0 || prev <= j0)))) {
          const int c = j0 - H + 1;
          const BandTaps<PAIR> tp(band, c - band.lo, part.spill_w + ((c - part.lo_w) << kShift), part.hi_prev + 1 - c);
          band_spread2<H, PAIR>(W, tp, j0, fr, q, act, part.gw, jb - j0, fb, qb);
          continue;
        }
      }
      for (int k = 0; k < step; ++k) {
        const bool on = k == 0 ? act : i + 1 < part.n1;
        const int j = k == 0 ? j0 : jb, c = j - H + 1;
        const BandTaps<PAIR> tp(band, c - band.lo, part.spill_w + ((c - part.lo_w) << kShift), part.hi_prev + 1 - c);
        band_spread<H, PAIR>(W, tp, j, k == 0 ? fr : fb, k == 0 ? q : qb, on, part.gw);
      }
    }
    __syncthreads();
    band_end<H, PAIR>(part, band, lane_u, tpu, 2 * M);
    // first pass (radix 16): element e = lane + r M/16; a thread's cells lie 2 M/16 (a multiple of 4) apart, in one phase
    float2* X = U + (PAIR ? sub * P.slot : 0);
    {
      constexpr int R = 16;
      float2 v[R];
      const int mask = 2 * M - 1;
      const int p0 = 2 * lane - band.lo, q0 = -1 - 2 * lane - band.lo;
      const int pp = p0 & 3, qp = q0 & 3;
      const unsigned half = sub << 3;
      const unsigned pa = band.grid + ((pp * band.ps) << kShift) + half;
      const unsigned qa = band.grid + ((qp * band.ps) << kShift) + half;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = (p0 + 2 * r * tpr) & mask, k = (q0 - 2 * r * tpr) & mask;
        float2 a = make_float2(0.f, 0.f), b = a;
        if (i < band.n) a = lds2(pa + ((i >> 2) << kShift));
        if (k < band.n) b = lds2(qa + ((k >> 2) << kShift));
        v[r] = cadd(a, b);
      }
      __syncthreads();  // the band is read before its memory takes the transform
      first_pass_regs<false>(X, v, lane);
    }
    __syncthreads();
    const int row = sub ? row_b : (valid ? unit : -1);
    float2* dst = row >= 0 ? const_cast<float2*>(P.pt) + (size_t)row * P.nt : nullptr;
    const int last = P.mshift & 3, tws = L.Mmax >> P.mshift;
    if (last == 0) {
      fft_rest<false, kLayoutFlat>(X, M, P.mshift, lane, tpr, L.tw, tws);
      if (dst)
        for (int n = lane; n < P.nt; n += tpr) dst[n] = model_sample(__ldg(&P.model_tab[n]), X[n], X[(M - n) & (M - 1)]);
    } else {
      for (int Ns = 16; Ns * 16 <= M; Ns <<= 4)
        fft_pass<16, false, kLayoutPadded>(X, M, Ns, lane, tpr, L.tw, tws);
      if (last == 1) model_last<2>(X, M, P.nt, lane, tpr, L.tw, tws, P.model_tab, dst);
      else if (last == 2) model_last<4>(X, M, P.nt, lane, tpr, L.tw, tws, P.model_tab, dst);
      else model_last<8>(X, M, P.nt, lane, tpr, L.tw, tws, P.model_tab, dst);
    }
  }
}

// ZF = false: input is the half image spectrum (image R2C over all axes) with
// both lateral destinations of a row; ZF = true: input is the row's own full
// depth spectrum Fbar[row][l mod nz].
template <int H, bool ZF>
__global__ void __launch_bounds__(1024) row_adjoint_kernel(RowLaunch L, WindowPoly W) {
  extern __shared__ __align__(16) float2 smem[];
  __shared__ int s_item;
  pdl_wait();
  float4* nodes_all = reinterpret_cast<float4*>(smem + L.fft_region);
  for (int item = blockIdx.x; item < L.nitems; item = next_item(L, &s_item)) {
    const WorkItem wi = L.items[item];
    const RowProblem& P = L.problems[wi.problem];
    const int tpr = P.tpr, M = P.M, nt = P.nt, mask = M - 1;
    const int slot = threadIdx.x / tpr;
    const int lane = threadIdx.x - slot * tpr;
    const int row = wi.row0 + slot;
    const bool valid = row < P.rows;
    float2* X = smem + slot * P.slot32;
    float4* N = nodes_all + slot * (P.nz + 2);
    const int nzh = P.nz >> 1;
    RowGeom rg;
    int nneg = 1, nn = 0;
    // ZF: the row's depth spectrum Fbar[l mod nz] (depth FFT of the lateral R2C of the image)
    const float2* Zs = P.fh + (size_t)(valid ? row : 0) * P.zstride;
    if (valid && ZF && P.qmode) {
      // Discrete forward model (the operator Q of Sec. 2 on a padded periodic
      // box): the row's temporal samples are sum_j c_j cos(2 pi nu_j n / nt)
      // over the depth frequencies j = 0..nz/2, nu_j >= 0 the frequency of
      // |K| (j = 0 included: its frequency is the lateral |K|), with
      // c_j = F[j] + F[-j] (F[0], F[nz/2] alone; Zs[j]).  Each cosine is the node pair
      // +-nu_j with value c_j / 2 (wscale holds 1 / (2 n_lat nz)); the spread
      // below and the inverse FFT then sum the pairs like any adjoint row.
      rg.S = P.rowS[row];
      rg.mirror = true;
      nneg = nzh + 1;
      nn = 2 * nneg;
      for (int j = lane; j <= nzh; j += tpr) {
        const float4 zt = __ldg(&P.zt[j]);
        int j0p, j0;
        float frp, fr, rx;
        node_position(rg.S, zt, P.B2hi, P.B2lo, j0p, frp, rx);
        negate_node(j0p, frp, j0, fr);
        const float2 y = Zs[j];
        const float2 pb = make_float2(P.wscale * y.x, P.wscale * y.y);
        const float2 qp = cmul(pb, node_phase(j0p, frp, nt, M, P.nt_over_M));
        const float2 qn = cmul(pb, node_phase(j0, fr, nt, M, P.nt_over_M));
        N[nneg + j] = make_float4(__int_as_float(j0p), frp, qp.x, qp.y);
        N[nneg - 1 - j] = make_float4(__int_as_float(j0), fr, qn.x, qn.y);
      }
    } else if (valid && ZF) {
      rg.S = P.rowS[row];
      rg.mirror = true;
      nneg = nzh;
      nn = nneg + nzh;
      const int nA = P.nz - 1;
      for (int i = lane; i < nA; i += tpr) {
        int lp;
        bool neg, nyq;
        node_task(i, nzh, nA, lp, neg, nyq);
        const float4 zt = __ldg(&P.zt[lp]);
        int j0p, j0;
        float frp, fr, rx;
        node_position(rg.S, zt, P.B2hi, P.B2lo, j0p, frp, rx);
        const float wt = P.wscale * zt.z * rx;
        negate_node(j0p, frp, j0, fr);
        if (nyq) {
          const float2 y = Zs[nzh];
          const float2 pb = make_float2(0.5f * wt * y.x, 0.5f * wt * y.y);
          const float2 qp = cmul(pb, adj_node_phase<H>(P, j0p, frp));
          const float2 qn = cmul(pb, adj_node_phase<H>(P, j0, fr));
          N[nneg + nzh - 1] = make_float4(__int_as_float(j0p), frp, qp.x, qp.y);
          N[0] = make_float4(__int_as_float(j0), fr, qn.x, qn.y);
        } else if (!neg) {
          const float2 y = Zs[lp];
          const float2 q = cmul(make_float2(wt * y.x, wt * y.y), adj_node_phase<H>(P, j0p, frp));
          N[nneg + lp - 1] = make_float4(__int_as_float(j0p), frp, q.x, q.y);
        } else {
          const float2 y = Zs[P.nz - lp];
          const float2 q = cmul(make_float2(wt * y.x, wt * y.y), adj_node_phase<H>(P, j0, fr));
          N[nzh - lp] = make_float4(__int_as_float(j0), fr, q.x, q.y);
        }
      }
    }
    if (valid && !ZF) {
      rg = row_geom(P, row);
      nneg = rg.mirror ? nzh : 1;
      nn = nneg + nzh;
      // phase 1: node values Q = e^{+i pi nu} * Pbar, stored sorted by position
      const int nA = rg.mirror ? (P.nz - 1) : nzh;
      const float2* in1 = P.fh + (size_t)rg.d1 * P.lz;
      const float2* in2 = P.fh + (size_t)rg.d2 * P.lz;
      for (int i = lane; i < nA; i += tpr) {
        int lp;
        bool neg, nyq;
        node_task(i, nzh, nA, lp, neg, nyq);
        const float4 zt = __ldg(&P.zt[lp]);
        int j0p, j0;
        float frp, fr, rx;
        node_position(rg.S, zt, P.B2hi, P.B2lo, j0p, frp, rx);
        const float wt = P.wscale * zt.z * rx;
        negate_node(j0p, frp, j0, fr);
        if (nyq) {
          float2 y = in1[lp];
          if (rg.mirror) {
            const float2 y2 = in2[lp];
            y.x += y2.x;
            y.y -= y2.y;
          }
          const float2 pb = make_float2(0.5f * wt * y.x, 0.5f * wt * y.y);
          const float2 php = adj_node_phase<H>(P, j0p, frp);
          const float2 phn = adj_node_phase<H>(P, j0, fr);
          const float2 qp = cmul(pb, php), qn = cmul(pb, phn);
          N[nneg + nzh - 1] = make_float4(__int_as_float(j0p), frp, qp.x, qp.y);
          N[0] = make_float4(__int_as_float(j0), fr, qn.x, qn.y);
        } else if (!neg) {
          const float2 y = in1[lp];
          const float2 pb = make_float2(2.0f * wt * y.x, 2.0f * wt * y.y);
          const float2 q = cmul(pb, adj_node_phase<H>(P, j0p, frp));
          N[nneg + lp - 1] = make_float4(__int_as_float(j0p), frp, q.x, q.y);
        } else {
          const float2 y = in2[lp];
          const float2 pb = make_float2(2.0f * wt * y.x, -2.0f * wt * y.y);
          const float2 q = cmul(pb, adj_node_phase<H>(P, j0, fr));
          N[nzh - lp] = make_float4(__int_as_float(j0), fr, q.x, q.y);
        }
      }
    }
    __syncthreads();
    // phase 2: the spread (the transpose of the gather).  Node k adds
    // w_t(fr_k) Q_k to grid cell j0_k + t - H + 1 (mod M), t = 0..2H-1, by one
    // of three schemes (the plan times them and keeps the fastest; the tap
    // phases are also the deterministic choice).  Tap phases: nodes are taken in chunks of at most one node per thread that never mix
    // the two signs (-nu and +nu lists).  Nodes with equal j0 form a run (the
    // list is sorted); for each tap t in turn the head of every run evaluates
    // the tap weight of each of its nodes (tap index uniform over the CTA, so
    // the polynomial coefficients stay constant-bank operands) and adds the
    // run's sum to its cell.  Taps run in the order 0, 2H-1, 1, 2H-2, ... so a
    // tap and its mirror share one evaluation of the pair polynomials.  Within
    // a chunk distinct runs have distinct j0 and the chunk spans fewer than
    // M - 2H cells, so in one tap phase no two heads write the same cell; a
    // barrier separates the tap phases.  Every cell receives its terms in a
    // fixed order (chunk, tap, node): deterministic, no atomics.
    if (L.spread_mode == 1) {
      // shared-memory atomics: every node adds its 2H taps straight into the
      // grid, no tap phases (summation order, hence the last bits, may vary
      // from run to run)
      const bool interp = H == 2 && P.method >= PAI_METHOD_LINEAR;
      for (int g = lane; g < M; g += tpr) X[padi<5>(g)] = make_float2(0.f, 0.f);
      __syncthreads();
      for (int i = lane; i < nn; i += tpr) {
        const float4 nd = N[i];
        const int j0 = __float_as_int(nd.x);
        const float z = nd.y - 0.5f, z2 = z * z;
#pragma unroll
        for (int p = 0; p < H; ++p) {
          float E = W.ce[p][kHalfCoef - 1], O = W.co[p][kHalfCoef - 1];
#pragma unroll
          for (int e = kHalfCoef - 2; e >= 0; --e) {
            E = fmaf(E, z2, W.ce[p][e]);
            O = fmaf(O, z2, W.co[p][e]);
          }
          float wl = fmaf(z, O, E), wh = fmaf(-z, O, E);
          if constexpr (H == 2) {
            if (interp) {
              wl = interp_tap_weight(P.method, p, nd.y);
              wh = interp_tap_weight(P.method, 2 * H - 1 - p, nd.y);
            }
          }
          float2* cl = X + padi<5>((j0 + p - H + 1) & mask);
          float2* ch = X + padi<5>((j0 + H - p) & mask);
          atomicAdd(&cl->x, wl * nd.z);
          atomicAdd(&cl->y, wl * nd.w);
          atomicAdd(&ch->x, wh * nd.z);
          atomicAdd(&ch->y, wh * nd.w);
        }
      }
      __syncthreads();  // every node's taps are in the grid
    } else if (L.spread_mode == 2) {
      // shared-memory atomics per run: the first node of each run of equal j0
      // sums the run's weighted terms for every tap and adds each sum with one
      // atomic, so clusters of nodes on few cells cost few atomics
      const bool interp = H == 2 && P.method >= PAI_METHOD_LINEAR;
      for (int g = lane; g < M; g += tpr) X[padi<5>(g)] = make_float2(0.f, 0.f);
      __syncthreads();
      for (int i = lane; i < nn; i += tpr) {
        const int j0 = __float_as_int(N[i].x);
        if (i > 0 && __float_as_int(N[i - 1].x) == j0) continue;  // not the first node of its run
        int run = 1;
        while (i + run < nn && __float_as_int(N[i + run].x) == j0) ++run;
#pragma unroll
        for (int p = 0; p < H; ++p) {
          float lx = 0.f, ly = 0.f, hx = 0.f, hy = 0.f;  // taps p and 2H-1-p
          for (int r = 0; r < run; ++r) {
            const float4 nd = N[i + r];
            const float z = nd.y - 0.5f, z2 = z * z;
            float E = W.ce[p][kHalfCoef - 1], O = W.co[p][kHalfCoef - 1];
#pragma unroll
            for (int e = kHalfCoef - 2; e >= 0; --e) {
              E = fmaf(E, z2, W.ce[p][e]);
              O = fmaf(O, z2, W.co[p][e]);
            }
            float wl = fmaf(z, O, E), wh = fmaf(-z, O, E);
            if constexpr (H == 2) {
              if (interp) {
                wl = interp_tap_weight(P.method, p, nd.y);
                wh = interp_tap_weight(P.method, 2 * H - 1 - p, nd.y);
              }
            }
            lx = fmaf(wl, nd.z, lx);
            ly = fmaf(wl, nd.w, ly);
            hx = fmaf(wh, nd.z, hx);
            hy = fmaf(wh, nd.w, hy);
          }
          float2* cl = X + padi<5>((j0 + p - H + 1) & mask);
          float2* ch = X + padi<5>((j0 + H - p) & mask);
          atomicAdd(&cl->x, lx);
          atomicAdd(&cl->y, ly);
          atomicAdd(&ch->x, hx);
          atomicAdd(&ch->y, hy);
        }
      }
      __syncthreads();  // every run's taps are in the grid
    } else {
      const int CH = L.chunk;  // <= tpr
      const bool interp = H == 2 && P.method >= PAI_METHOD_LINEAR;
      for (int g = lane; g < M; g += tpr) X[padi<5>(g)] = make_float2(0.f, 0.f);
      const int list_max = (P.nz >> 1) + (P.qmode ? 1 : 0);  // nodes per sign list, at most
      const int half_chunks = (list_max + CH - 1) / CH;         // uniform over the CTA's slots
      for (int c = 0; c < 2 * half_chunks; ++c) {
        const bool pos = c >= half_chunks;
        const int first = pos ? nneg : 0;
        const int count = pos ? nn - nneg : nneg;
        const int c0 = first + (pos ? c - half_chunks : c) * CH;
        const int cn = valid ? max(0, min(CH, first + count - c0)) : 0;
        int j0 = 0, run = 0;  // run length if this thread's node heads a run, else 0
        if (lane < cn) {
          j0 = __float_as_int(N[c0 + lane].x);
          if (lane == 0 || __float_as_int(N[c0 + lane - 1].x) != j0) {
            run = 1;
            while (lane + run < cn && __float_as_int(N[c0 + lane + run].x) == j0) ++run;
          }
        }
        // the head's own node stays in registers for all taps; its polynomial
        // pair (E_p, O_p) serves tap p and its mirror 2H-1-p, which run in
        // consecutive phases
        const float4 nd0 = run > 0 ? N[c0 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float z0 = nd0.y - 0.5f, z0sq = z0 * z0;
        __syncthreads();  // previous chunk's writes (or the zeroing) complete
#pragma unroll
        for (int p = 0; p < H; ++p) {
          float E0 = W.ce[p][kHalfCoef - 1], O0 = W.co[p][kHalfCoef - 1];
#pragma unroll
          for (int e = kHalfCoef - 2; e >= 0; --e) {
            E0 = fmaf(E0, z0sq, W.ce[p][e]);
            O0 = fmaf(O0, z0sq, W.co[p][e]);
          }
#pragma unroll
          for (int side = 0; side < 2; ++side) {
            // tap t = p (side 0) or 2H-1-p (side 1): w(z) = E_p(z^2) +- z O_p(z^2), z = fr - 1/2
            const int t = side == 0 ? p : 2 * H - 1 - p;
            if (run > 0) {
              float w0 = side == 0 ? fmaf(z0, O0, E0) : fmaf(-z0, O0, E0);
              if constexpr (H == 2) {
                if (interp) w0 = interp_tap_weight(P.method, t, nd0.y);
              }
              float sx = w0 * nd0.z, sy = w0 * nd0.w;
              for (int r = 1; r < run; ++r) {
                const float4 nd = N[c0 + lane + r];
                const float z = side == 0 ? nd.y - 0.5f : 0.5f - nd.y;
                const float z2 = z * z;
                float E = W.ce[p][kHalfCoef - 1], O = W.co[p][kHalfCoef - 1];
#pragma unroll
                for (int e = kHalfCoef - 2; e >= 0; --e) {
                  E = fmaf(E, z2, W.ce[p][e]);
                  O = fmaf(O, z2, W.co[p][e]);
                }
                float w = fmaf(z, O, E);
                if constexpr (H == 2) {
                  if (interp) w = interp_tap_weight(P.method, t, nd.y);
                }
                sx = fmaf(w, nd.z, sx);
                sy = fmaf(w, nd.w, sy);
              }
              const int gi = padi<5>((j0 + t - H + 1) & mask);
              float2 x = X[gi];
              x.x += sx;
              x.y += sy;
              X[gi] = x;
            }
            __syncthreads();
          }
        }
      }
    }
    if constexpr (H == 2) {
      // interpolation methods: the grid cells' phases e^{+i pi nu_j}
      if (valid && P.method >= PAI_METHOD_LINEAR)
        for (int g = lane; g < M; g += tpr) X[padi<5>(g)] = cmul(X[padi<5>(g)], node_phase(g, 0.0f, nt, M, P.nt_over_M));
    }
    __syncthreads();
    const float scale = (valid && !ZF && rg.mirror) ? 0.5f : 1.0f;
    float2* dst = const_cast<float2*>(P.pt) + (size_t)(valid ? row : 0) * nt;
    fft_inverse_crop<false>(X, M, P.mshift, nt, lane, tpr, L.tw, L.Mmax >> P.mshift, dst, P.prescale, scale, valid,
                            Band{});
  }
}

}  // namespace pai
