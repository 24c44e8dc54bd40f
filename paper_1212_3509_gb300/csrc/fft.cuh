// Shared-memory Stockham FFT building blocks (power-of-two lengths).
//
// The structured formats apply each 1D Toeplitz factor through a circulant
// embedding and the convolution theorem (Sec. 4.1: DFT / IDFT definitions,
// Eq. dft and Eq. idft with omega = exp(-2 pi i k j / n); Lemmas 4-5: the DFT
// of a CP / Tucker tensor is the 1D DFT of its factor columns).  A real signal
// of length L is transformed as a complex signal of length N = L/2 (even
// samples in the real part, odd samples in the imaginary part) followed by
// the usual split step.
//
// Complex FFT: self-sorting (Stockham) mixed-radix passes.  Pass with radix R
// over sub-transforms of size Ns: item j < N/R loads x[j + r N/R] (r < R),
// multiplies by W^(r (j mod Ns) N/(Ns R)), does an R-point DFT in registers and
// stores to y[(j / Ns) Ns R + (j mod Ns) + r Ns].  Radix 16 passes first,
// then one pass of radix 2, 4 or 8 for the remaining bits.  A pass is done
// in place: all items are read into registers, the group synchronises, then
// writes.
#pragma once

#include <cuda_runtime.h>

namespace demag {

template <typename T> struct cplx_t;
template <> struct cplx_t<float> { using type = float2; };
template <> struct cplx_t<double> { using type = double2; };

template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  C r;
  r.x = a.x * b.x - a.y * b.y;
  r.y = a.x * b.y + a.y * b.x;
  return r;
}
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { C r; r.x = a.x + b.x; r.y = a.y + b.y; return r; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { C r; r.x = a.x - b.x; r.y = a.y - b.y; return r; }
template <typename C> __device__ __forceinline__ C cconj(C a) { a.y = -a.y; return a; }

// FP32 complex add / subtract as one packed instruction on the (re, im) pair
// (add.rn.f32x2 / sub.rn.f32x2): per component the same correctly rounded
// result as a scalar add, half the issue slots of the FFT butterflies.
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  unsigned long long ra, rb, rc;
  asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(rc) : "l"(ra), "l"(rb));
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(rc));
  return r;
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
  unsigned long long ra, rb, rc;
  asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(rc) : "l"(ra), "l"(rb));
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(rc));
  return r;
}

// exp(-2 pi i j / 16) for j = 0..15 (cos, -sin), exact zeros and ones.
__device__ __forceinline__ constexpr double w16_re(int j) {
  return j == 0 ? 1.0 : j == 1 ? 0.92387953251128675613 : j == 2 ? 0.70710678118654752440
       : j == 3 ? 0.38268343236508977173 : j == 4 ? 0.0 : j == 5 ? -0.38268343236508977173
       : j == 6 ? -0.70710678118654752440 : j == 7 ? -0.92387953251128675613 : j == 8 ? -1.0
       : j == 9 ? -0.92387953251128675613 : j == 10 ? -0.70710678118654752440
       : j == 11 ? -0.38268343236508977173 : j == 12 ? 0.0 : j == 13 ? 0.38268343236508977173
       : j == 14 ? 0.70710678118654752440 : 0.92387953251128675613;
}
__device__ __forceinline__ constexpr double w16_im(int j) {
  // -sin(2 pi j / 16) = cos(2 pi (j + 4) / 16)
  return w16_re((j + 4) & 15);
}

// Multiply by exp(s 2 pi i k / R) with compile-time k, R (R <= 16); s = -1
// forward, +1 inverse.  Trivial rotations compile to swaps / negations.
template <int R, int K, bool INV, typename C>
__device__ __forceinline__ C rot(C v) {
  using T = decltype(v.x);
  constexpr int j = (K * (16 / R)) & 15;
  if constexpr (j == 0) {
    return v;
  } else if constexpr (j == 4) {  // forward: -i, inverse: +i
    C r;
    if (INV) { r.x = -v.y; r.y = v.x; } else { r.x = v.y; r.y = -v.x; }
    return r;
  } else if constexpr (j == 8) {
    C r; r.x = -v.x; r.y = -v.y; return r;
  } else if constexpr (j == 12) {
    C r;
    if (INV) { r.x = v.y; r.y = -v.x; } else { r.x = -v.y; r.y = v.x; }
    return r;
  } else {
    C w;
    w.x = (T)w16_re(j);
    w.y = INV ? -(T)w16_im(j) : (T)w16_im(j);
    return cmul(v, w);
  }
}

template <int R, bool INV, int K, typename C>
__device__ __forceinline__ void dft_combine(C (&v)[R], C (&e)[R / 2], C (&o)[R / 2]) {
  if constexpr (K < R / 2) {
    C t = rot<R, K, INV>(o[K]);
    constexpr int j = (K * (16 / R)) & 15;
    if constexpr (j == 4 || j == 12) {
      // +-i: the swap and sign fold into scalar adds (a packed add would need
      // the swapped pair built first)
      v[K].x = e[K].x + t.x;
      v[K].y = e[K].y + t.y;
      v[K + R / 2].x = e[K].x - t.x;
      v[K + R / 2].y = e[K].y - t.y;
    } else {
      v[K] = cadd(e[K], t);
      v[K + R / 2] = csub(e[K], t);
    }
    dft_combine<R, INV, K + 1>(v, e, o);
  }
}

// In-register R-point DFT, radix-2 decimation in time, natural order output.
template <int R, bool INV, typename C>
__device__ __forceinline__ void dft_reg(C (&v)[R]) {
  if constexpr (R == 1) {
    return;
  } else if constexpr (R == 2) {
    C a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  } else {
    C e[R / 2], o[R / 2];
#pragma unroll
    for (int i = 0; i < R / 2; ++i) { e[i] = v[2 * i]; o[i] = v[2 * i + 1]; }
    dft_reg<R / 2, INV>(e);
    dft_reg<R / 2, INV>(o);
    dft_combine<R, INV, 0>(v, e, o);
  }
}

// The first 8 outputs of an inverse 16-point DFT (the kept half of the last
// pass): two 8-point DFTs of the even and odd inputs and the "+" half of the
// final butterflies.
template <int K>
__device__ __forceinline__ void combine_half16(float2 (&v)[16], float2 (&e)[8], float2 (&o)[8]) {
  if constexpr (K < 8) {
    const float2 t = rot<16, K, true>(o[K]);
    if constexpr (K == 4) {  // +i: folded into scalar adds
      v[K].x = e[K].x + t.x;
      v[K].y = e[K].y + t.y;
    } else {
      v[K] = cadd(e[K], t);
    }
    combine_half16<K + 1>(v, e, o);
  }
}

__device__ __forceinline__ void idft16_first_half(float2 (&v)[16]) {
  float2 e[8], o[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    e[i] = v[2 * i];
    o[i] = v[2 * i + 1];
  }
  dft_reg<8, true>(e);
  dft_reg<8, true>(o);
  combine_half16<0>(v, e, o);
}

// v[r] *= exp(-2 pi i r / 16), r < 8
template <int R>
__device__ __forceinline__ void rot16_rows(float2 (&v)[8]) {
  if constexpr (R < 8) {
    v[R] = rot<16, R, false>(v[R]);
    rot16_rows<R + 1>(v);
  }
}

// Forward 16-point DFT of inputs r < 8 (the others are zero): the even outputs
// are the 8-point DFT of the inputs, the odd ones that of x_r W_16^r.
__device__ __forceinline__ void dft16_of_half(const float2 (&x)[8], float2 (&v)[16]) {
  float2 e[8], o[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) e[r] = o[r] = x[r];
  rot16_rows<1>(o);
  dft_reg<8, false>(e);
  dft_reg<8, false>(o);
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    v[2 * m] = e[m];
    v[2 * m + 1] = o[m];
  }
}

// ---- FFT of length N = 16 B, 32 <= N <= 512, in the registers of B lanes ----
//
// Lane l (of the B consecutive lanes of a fibre) holds 16 elements.  In time
// order element r is x[l + B r]; in frequency order element s is X[f(l, s)]
// (rf_freq), a fixed permutation that a product with a spectrum does not mind.
// With f = k1 + 16 k2, X = sum_j W_B^(j k2) [ W_N^(j k1) sum_r W_16^(r k1) x[j + B r] ]:
// a 16-point DFT in registers, one twiddle, one exchange through shared memory
// (16 rows of B, one write and one read of the fibre), and 16 / B DFTs of B
// points in registers; for B = 32 a 32-point one shared by two lanes, its last
// radix-2 step by shuffles.  The inverse takes the same steps backwards.  A
// fibre thus crosses shared memory once per transform where the in-place
// radix-16 passes of fft_inplace cross it once per pass and once to be staged.
// Only the first N / 2 time samples exist (zero padding in, kept half out).
//
// Exchange rows are B + 1 long and a fibre's buffer is N + 17 long (1 mod 16):
// with fibre g in slot rf_slot(g) the fibres that share a half-warp lie B
// apart modulo 16, so rows, columns and (16 fibres of one index) transposed
// reads are all free of bank conflicts.
template <int B> struct RegFft {
  static constexpr int N = 16 * B;
  static constexpr int BS = N + 17;  // buffer elements per fibre
};

template <int B>
__device__ __forceinline__ int rf_slot(int g) {
  if constexpr (B >= 16) return g;
  constexpr int F = B >= 16 ? 1 : 16 / B;  // fibres per half-warp
  return (g & ~15) + (g % F) * B + (g / F) % B;
}

template <int B>
__device__ __forceinline__ int rf_freq(int l, int s) {
  if constexpr (B == 32) return (l & 15) + 16 * (8 * (l >> 4) + (s & 7) + 16 * (s >> 3));
  return l + B * (s / B) + 16 * (s % B);
}

__device__ __forceinline__ float2 shfl_xor2(float2 v, int off) {
  v.x = __shfl_xor_sync(0xffffffffu, v.x, off);
  v.y = __shfl_xor_sync(0xffffffffu, v.y, off);
  return v;
}

// exp(-2 pi i t / 32), t < 8
__device__ __forceinline__ constexpr double w32_re(int t) {
  return t == 0 ? 1.0 : t == 1 ? 0.98078528040323044913 : t == 2 ? 0.92387953251128675613
       : t == 3 ? 0.83146961230254523708 : t == 4 ? 0.70710678118654752440 : t == 5 ? 0.55557023301960222474
       : t == 6 ? 0.38268343236508977173 : 0.19509032201612826785;
}
__device__ __forceinline__ constexpr double w32_im(int t) { return t == 0 ? 0.0 : -w32_re(8 - t); }

template <bool INV, int T>
__device__ __forceinline__ float2 rot32(float2 v) {
  float2 w;
  w.x = (float)w32_re(T);
  w.y = INV ? -(float)w32_im(T) : (float)w32_im(T);
  return T == 0 ? v : cmul(v, w);
}

// The radix-2 step of B = 32 for t = T..7: forward on (B_0, B_1)[k2'], k2' = 8 h + t
template <int T>
__device__ __forceinline__ void rf_join(float2 (&u)[16], const float2 (&other)[8], int h) {
  if constexpr (T < 8) {
    const float2 own = h ? u[8 + T] : u[T];
    const float2 b0 = h ? other[T] : own;
    float2 c = rot32<false, T>(h ? own : other[T]);
    if (h) c = make_float2(c.y, -c.x);  // W_32^(8 + t) = -i W_32^t
    rf_join<T + 1>(u, other, h);        // (reads u[T + 1 ..], u[8 + T + 1 ..] before they are written)
    u[T] = cadd(b0, c);
    u[8 + T] = csub(b0, c);
  }
}
template <int T>
__device__ __forceinline__ void rf_part(float2 (&u)[16], float2 (&send)[8], float2 (&keep)[8], int h) {
  if constexpr (T < 8) {
    const float2 b = cadd(u[T], u[8 + T]);
    float2 c = rot32<true, T>(csub(u[T], u[8 + T]));
    if (h) c = make_float2(-c.y, c.x);  // conj W_32^(8 + t) = i conj W_32^t
    send[T] = h ? b : c;
    keep[T] = h ? c : b;
    rf_part<T + 1>(u, send, keep, h);
  }
}

// Forward: the twiddled 16-point DFTs lie in buf (row k1, column l); u: the spectrum in frequency order.
template <int B>
__device__ __forceinline__ void rf_finish(float2 (&u)[16], float2* buf, int l) {
  if constexpr (B == 32) {
    const int k1 = l & 15, h = l >> 4;
#pragma unroll
    for (int i = 0; i < 16; ++i) u[i] = buf[k1 * (B + 1) + 2 * i + h];
    __syncwarp();
    dft_reg<16, false>(u);
    float2 other[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) other[t] = shfl_xor2(h ? u[t] : u[8 + t], 16);
    rf_join<0>(u, other, h);
  } else {
    constexpr int E = B >= 16 ? 1 : 16 / B;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      float2 w[B];
#pragma unroll
      for (int j = 0; j < B; ++j) w[j] = buf[(l + B * e) * (B + 1) + j];
      dft_reg<B, false>(w);
#pragma unroll
      for (int j = 0; j < B; ++j) u[e * B + j] = w[j];
    }
    __syncwarp();
  }
}

// x: the 8 time samples x[l + B r]; u: the spectrum in frequency order.  pw[r] = W_N^(l r).
template <int B>
__device__ __forceinline__ void rf_forward(const float2 (&x)[8], float2 (&u)[16], float2* buf, int l,
                                           const float2 (&pw)[16]) {
  {
    float2 v[16];
    dft16_of_half(x, v);
#pragma unroll
    for (int k = 0; k < 16; ++k) buf[k * (B + 1) + l] = k ? cmul(v[k], pw[k]) : v[k];
  }
  __syncwarp();
  rf_finish<B>(u, buf, l);
}

// u: a spectrum in frequency order; its inverse B-point DFTs are left in buf (row k1, column l).
template <int B>
__device__ __forceinline__ void rf_begin(float2 (&u)[16], float2* buf, int l) {
  if constexpr (B == 32) {
    const int k1 = l & 15, h = l >> 4;
    float2 send[8], keep[8];
    rf_part<0>(u, send, keep, h);
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const float2 got = shfl_xor2(send[t], 16);
      u[t] = h ? got : keep[t];
      u[8 + t] = h ? keep[t] : got;
    }
    dft_reg<16, true>(u);
#pragma unroll
    for (int i = 0; i < 16; ++i) buf[k1 * (B + 1) + 2 * i + h] = u[i];
  } else {
    constexpr int E = B >= 16 ? 1 : 16 / B;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      float2 w[B];
#pragma unroll
      for (int j = 0; j < B; ++j) w[j] = u[e * B + j];
      dft_reg<B, true>(w);
#pragma unroll
      for (int j = 0; j < B; ++j) buf[(l + B * e) * (B + 1) + j] = w[j];
    }
  }
}

// u: a spectrum in frequency order; v[r], r < 8: x[l + B r] of the unnormalised inverse.
template <int B>
__device__ __forceinline__ void rf_inverse(float2 (&u)[16], float2 (&v)[16], float2* buf, int l,
                                           const float2 (&pw)[16]) {
  rf_begin<B>(u, buf, l);
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float2 y = buf[k * (B + 1) + l];
    v[k] = k ? cmul(y, make_float2(pw[k].x, -pw[k].y)) : y;
  }
  __syncwarp();
  idft16_first_half(v);
}

// Inverse 16-point DFT of w^k v[k] with the powers of w inside its radix-2 steps: eight twiddles
// (16 registers) where separate products keep fifteen.  Outputs r < 8 only with HALF.
struct Twid16 {
  float2 a[4];  // w exp(2 pi i j / 16)
  float2 b[2];  // w^2 exp(2 pi i j / 8)
  float2 c, d;  // w^4, w^8
};

template <int R, int K>
__device__ __forceinline__ float2 tw16_rot(const Twid16& t, float2 v) {
  constexpr int j = K % (R >= 4 ? R / 4 : 1);
  if constexpr (R == 16) return cmul(v, t.a[j]);
  if constexpr (R == 8) return cmul(v, t.b[j]);
  if constexpr (R == 4) return cmul(v, t.c);
  return cmul(v, t.d);
}
template <int R, int K, bool HALF>
__device__ __forceinline__ void tw16_combine(const Twid16& t, const float2 (&e)[R / 2], const float2 (&o)[R / 2],
                                             float2 (&v)[R]) {
  if constexpr (K < R / 2) {
    const float2 p = tw16_rot<R, K>(t, o[K]);
    if constexpr (R >= 4 && K >= R / 4) {  // a further factor i
      v[K].x = e[K].x - p.y;
      v[K].y = e[K].y + p.x;
      if constexpr (!HALF) {
        v[K + R / 2].x = e[K].x + p.y;
        v[K + R / 2].y = e[K].y - p.x;
      }
    } else {
      v[K] = cadd(e[K], p);
      if constexpr (!HALF) v[K + R / 2] = csub(e[K], p);
    }
    tw16_combine<R, K + 1, HALF>(t, e, o, v);
  }
}
template <int R, bool HALF>
__device__ __forceinline__ void tw16_idft(const Twid16& t, float2 (&v)[R]) {
  if constexpr (R > 1) {
    float2 e[R / 2], o[R / 2];
#pragma unroll
    for (int i = 0; i < R / 2; ++i) {
      e[i] = v[2 * i];
      o[i] = v[2 * i + 1];
    }
    tw16_idft<R / 2, false>(t, e);
    tw16_idft<R / 2, false>(t, o);
    tw16_combine<R, 0, HALF>(t, e, o, v);
  }
}

// Radix plan for N = 2^LOGN: number of radix-16 passes and the remainder radix.
template <int LOGN> struct RadixPlan {
  static constexpr int n16 = LOGN / 4;
  static constexpr int rem = 1 << (LOGN % 4);  // 1, 2, 4 or 8
  static constexpr int passes = n16 + (rem > 1 ? 1 : 0);
};

// One Stockham pass of radix R on buf[0..N) by TG threads (local id lt).
// tw(m) returns exp(-2 pi i m / N) (forward twiddle), m < N.
template <int R, int N, int TG, bool INV, typename C, typename TW>
__device__ __forceinline__ void stockham_pass(C* buf, int Ns, int lt, const TW& tw) {
  constexpr int items = N / R;
  constexpr int ipt = (items + TG - 1) / TG;
  C v[ipt][R];
#pragma unroll
  for (int it = 0; it < ipt; ++it) {
    const int j = lt + it * TG;
    if (items % TG == 0 || j < items) {
      const int k = j % Ns;
      const int tstep = k * (N / (Ns * R));
#pragma unroll
      for (int r = 0; r < R; ++r) {
        C x = buf[j + r * items];
        if (r > 0 && Ns > 1) {
          C w = tw(r * tstep);
          if (INV) w.y = -w.y;
          x = cmul(x, w);
        }
        v[it][r] = x;
      }
      dft_reg<R, INV>(v[it]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < ipt; ++it) {
    const int j = lt + it * TG;
    if (items % TG == 0 || j < items) {
      const int k = j % Ns;
      const int base = (j / Ns) * Ns * R + k;
#pragma unroll
      for (int r = 0; r < R; ++r) buf[base + r * Ns] = v[it][r];
    }
  }
  __syncthreads();
}

// Padded shared-memory index: one spare slot per 16, so that strided
// accesses of a Stockham pass fall into distinct banks.
__device__ __forceinline__ int pad16(int i) { return i + (i >> 4); }
// pad16(i + r * S) = pad16(i) + r * (S + S / 16) when S is a multiple of 16
template <int S> struct PadStride { static constexpr int value = S + S / 16; };

// pw[r] = w^r for r < R by a product tree of depth <= 4 (w^2, w^4, w^8 by
// squaring, the rest as one product of those), so each power carries only a
// few roundings of the table value w.
template <int R>
__device__ __forceinline__ void powers(float2 w, float2 (&pw)[R]) {
  pw[0] = make_float2(1.f, 0.f);
  if constexpr (R > 1) pw[1] = w;
  if constexpr (R > 2) pw[2] = cmul(w, w);
  if constexpr (R > 3) pw[3] = cmul(pw[2], w);
  if constexpr (R > 4) {
    pw[4] = cmul(pw[2], pw[2]);
    pw[5] = cmul(pw[4], w);
    pw[6] = cmul(pw[4], pw[2]);
    pw[7] = cmul(pw[4], pw[3]);
  }
  if constexpr (R > 8) {
    pw[8] = cmul(pw[4], pw[4]);
#pragma unroll
    for (int r = 9; r < R; ++r) pw[r] = cmul(pw[8], pw[r - 8]);
  }
}

// Full complex FFT of length N = 2^LOGN in place on buf (unnormalised).
// All threads of the block must call it (it synchronises the block); threads
// of a group share buf.  `lt` is the thread index inside its group of TG.
template <int LOGN, int TG, bool INV, typename C, typename TW>
__device__ __forceinline__ void fft_inplace(C* buf, int lt, const TW& tw) {
  constexpr int N = 1 << LOGN;
  using P = RadixPlan<LOGN>;
  int Ns = 1;
  if constexpr (P::rem > 1) {
    stockham_pass<P::rem, N, TG, INV>(buf, Ns, lt, tw);
    Ns *= P::rem;
  }
  if constexpr (P::n16 > 0) {
#pragma unroll
    for (int p = 0; p < P::n16; ++p) {
      stockham_pass<16, N, TG, INV>(buf, Ns, lt, tw);
      Ns *= 16;
    }
  }
}

}  // namespace demag
