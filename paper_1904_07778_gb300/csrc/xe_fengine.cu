// GPU F-engine (Sec. 2.1): polyphase filter bank, the FFT of two real
// inputs as one complex transform with the Eq. 2 separation, the 18-bit
// output, and the equaliser / requantiser to packed fix_4_3 codes -- one
// fused kernel whose output is the X-engine's input.
//
// A CTA takes one input pair (2k, 2k+1) and a group of consecutive spectra.
// M/8 threads (an "FFT unit"; a CTA holds 2048/M units for M <= 2048, each
// with its own stretch of the group) take two spectra at a time: they filter 8 consecutive samples
// each, store z[n] = y_2k[n] + j y_2k+1[n] of both in padded shared memory,
// and run in-place Stockham FFTs (radix-8 passes, then one radix-2 or radix-4
// pass).  The separated spectra are rounded to 18 bits, equalised, packed, and
// staged per thread until 16 spectra of its channels leave as 16-byte pieces
// of the X-engine's [c][i][t] order: the corner turn happens here.
#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "fengine.h"
#include "xe_internal.h"
#include "xengine.h"

struct fe_ctx {
  int n_inputs = 0, n_chans = 0, taps = 0, shift = 0;
  unsigned flags = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  float* h = nullptr;         // [taps * M] prototype filter
  float2* w = nullptr;        // [M] exp(-2 pi j n / M)
  uint32_t* gain = nullptr;   // [C][N]
};

namespace xe {
namespace {

struct FeArgs {
  const int8_t* adc;
  long long adc_stride;
  const float* h;
  const float2* w;
  const uint32_t* gain;
  uint8_t* out;
  long long out_stride;
  int32_t* v18;
  float* spec;
  unsigned long long* power;
  int n_inputs, n_spectra, taps, layout;
  int pairs_first;  // CTAs in order of input pairs, not of groups of spectra
  int per_unit;  // consecutive spectra of each FFT unit: 2, 4, 8, 16 or 32
  int lo_is_real, vec_in, vec_out;
  int vec_two;  // [c][i][t] pieces of two spectra leave as half words
  int vec_extra;  // both inputs' spectra and 18-bit values as 16 bytes
  float scale;  // 2^-(shift + 1): Eq. 2's halving and the 18-bit scaling
};

__host__ __device__ constexpr int fe_threads(int logm) {
  return (1 << logm) / 8 > 256 ? (1 << logm) / 8 : 256;
}
// One point of padding (16 bytes: both spectra's complex values) per 8 and
// another per 64: aligned runs of 8 points (a quarter-warp's 16-byte accesses)
// stay contiguous, and runs of stride 8 and 64 spread over the banks.
__host__ __device__ constexpr int fe_pad(int n) { return n + (n >> 3) + (n >> 6); }
// Twiddles of the radix-8 passes at Ns = 8 and Ns = 64 in shared memory,
// [k][j-1] for k < Ns, each value twice: they depend only on lt mod Ns, so
// the table is small (threads with equal k read the same entry) and frees the
// registers they would take.  Row k of the Ns = 64 part lies at
// 8 (k mod 8) + k / 8: the threads of a class (below) read neighbouring rows.
constexpr int kTwTable = (8 + 64) * 7;
__host__ __device__ constexpr int tw64_row(int k) { return 8 * (k & 7) + (k >> 3); }
__host__ __device__ constexpr int fe_units(int logm) { return fe_threads(logm) / ((1 << logm) / 8); }
// Codes staged per thread before they leave: its four channels of up to 16
// spectra, two spectra of both inputs to a word.  Only the thread itself reads
// them back.
constexpr int kStageIts = 8;
constexpr long long kL2Bytes = 120 << 20;  // what the L2 (135 MB) holds of a kernel's output
template <int LOGM>
constexpr size_t fe_smem_bytes() {
  constexpr int M = 1 << LOGM;
  return (size_t)fe_units(LOGM) * fe_pad(M) * 16 + kTwTable * 16 +
         (size_t)fe_threads(LOGM) * 4 * (kStageIts * sizeof(uint32_t) + sizeof(float2) + sizeof(uint32_t));
}

// ---- two spectra side by side -------------------------------------------------
// A unit transforms two consecutive spectra at once, and every value of the
// FFT, the separation and the equaliser is a pair of FP32 numbers, one per
// spectrum, in packed instructions (each half rounded as the scalar
// operation would be): half the instructions to issue for the same FP32
// work, and one 16-byte shared-memory access per point of both spectra.
struct C2 {
  uint64_t x, y;  // real and imaginary parts of the two spectra
};
__device__ __forceinline__ uint64_t p_pack(float a, float b) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ void p_unpack(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t p_dup(float a) { return p_pack(a, a); }
__device__ __forceinline__ uint64_t p_add(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t p_sub(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t p_mul(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t p_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t p_neg(uint64_t a) {
  float x, y;
  p_unpack(a, x, y);
  return p_pack(-x, -y);
}

// a b with b's parts given twice each
__device__ __forceinline__ C2 cmul(const C2& a, uint64_t bx, uint64_t by) {
  return {p_fma(a.x, bx, p_neg(p_mul(a.y, by))), p_fma(a.x, by, p_mul(a.y, bx))};
}
__device__ __forceinline__ C2 cadd(const C2& a, const C2& b) { return {p_add(a.x, b.x), p_add(a.y, b.y)}; }
__device__ __forceinline__ C2 csub(const C2& a, const C2& b) { return {p_sub(a.x, b.x), p_sub(a.y, b.y)}; }
// a - j b and a + j b
__device__ __forceinline__ C2 csub_j(const C2& a, const C2& b) { return {p_add(a.x, b.y), p_sub(a.y, b.x)}; }
__device__ __forceinline__ C2 cadd_j(const C2& a, const C2& b) { return {p_sub(a.x, b.y), p_add(a.y, b.x)}; }

// Y[k] = sum_n x[n] (-j)^(nk)
__device__ __forceinline__ void dft4(C2& x0, C2& x1, C2& x2, C2& x3) {
  const C2 t0 = cadd(x0, x2), t1 = csub(x0, x2), t2 = cadd(x1, x3), t3 = csub(x1, x3);
  x0 = cadd(t0, t2);
  x2 = csub(t0, t2);
  x1 = csub_j(t1, t3);
  x3 = cadd_j(t1, t3);
}

// X[k] = sum_n a[n] W8^(nk), W8 = exp(-j pi / 4): two DFT4s of the even and
// odd samples, joined with W8^k.  The factors 1/sqrt2 of W8 and W8^3 go into
// fused multiply-adds with the sums and differences they scale.
__device__ __forceinline__ void dft8(C2 (&a)[8]) {
  C2 e0 = a[0], e1 = a[2], e2 = a[4], e3 = a[6];
  C2 o0 = a[1], o1 = a[3], o2 = a[5], o3 = a[7];
  dft4(e0, e1, e2, e3);
  dft4(o0, o1, o2, o3);
  const uint64_t r = p_dup(0.70710678118654752f), mr = p_dup(-0.70710678118654752f);
  a[0] = cadd(e0, o0);
  a[4] = csub(e0, o0);
  const uint64_t s1 = p_add(o1.x, o1.y), d1 = p_sub(o1.y, o1.x);  // W8 o1 = r (s1 + j d1)
  a[1] = {p_fma(r, s1, e1.x), p_fma(r, d1, e1.y)};
  a[5] = {p_fma(mr, s1, e1.x), p_fma(mr, d1, e1.y)};
  a[2] = csub_j(e2, o2);
  a[6] = cadd_j(e2, o2);
  const uint64_t d3 = p_sub(o3.y, o3.x), s3 = p_add(o3.x, o3.y);  // W8^3 o3 = r (d3 - j s3)
  a[3] = {p_fma(r, d3, e3.x), p_fma(mr, s3, e3.y)};
  a[7] = {p_fma(mr, d3, e3.x), p_fma(r, s3, e3.y)};
}

// Twiddles of one Stockham pass for one thread: butterfly b = lt + r M/8
// multiplies its input j by exp(-2 pi j (b mod Ns) j / (Ns R)), for
// j = 1 .. R-1.  They do not depend on the spectrum, so a thread loads them
// once (from the FP64-rounded table) and keeps them in registers.
template <int M, int R>
__device__ __forceinline__ void load_twiddles(float2 (&tw)[7], const int (&b)[8 / R], int Ns,
                                              const float2* __restrict__ w) {
#pragma unroll
  for (int r = 0; r < 8 / R; ++r) {
    const int step = (b[r] & (Ns - 1)) * (M / (R * Ns));
#pragma unroll
    for (int j = 1; j < R; ++j) tw[r * (R - 1) + j - 1] = __ldg(&w[j * step]);
  }
}

// The butterflies of a thread in a last pass of radix R = 4 or 2 (Ns = M/R,
// outputs b + r Ns): pairs b and Ns - b, whose outputs are each other's
// mirror images M - nu, so that the separation of Eq. 2 happens in registers
// (a pass over shared memory and two barriers less).  b = 0 and b = Ns/2 are
// their own mirrors: thread 0 takes both.
template <int M, int R>
__device__ __forceinline__ void last_butterflies(int lt, int (&b)[8 / R]) {
  constexpr int Ns = M / R;
#pragma unroll
  for (int p = 0; p < 4 / R; ++p) {
    b[2 * p] = lt + p * (M / 8);
    b[2 * p + 1] = p == 0 && lt == 0 ? Ns / 2 : Ns - b[2 * p];
  }
}

__device__ __forceinline__ C2 z_load(const ulonglong2* z, int i) {
  const ulonglong2 v = z[i];
  return {v.x, v.y};
}
__device__ __forceinline__ void z_store(ulonglong2* z, int i, const C2& v) {
  z[i] = make_ulonglong2(v.x, v.y);
}

// The TPU threads of an FFT unit meet (units are whole warps, or parts of one).
template <int TPU, int NT>
__device__ __forceinline__ void unit_sync(int u) {
  if constexpr (TPU == NT)
    __syncthreads();
  else if constexpr (TPU > 32)
    asm volatile("bar.sync %0, %1;" ::"r"(1 + u), "n"(TPU) : "memory");
  else
    __syncwarp();
}

// The points of a unit with equal index mod 8 form a class: every radix-8 pass
// after the first maps a class onto itself.  The TPU / 8 threads lt / (TPU/8)
// = w of the unit take class w's butterflies in those passes and meet among
// themselves: within a warp (M <= 2048), or 64 threads (M = 4096).
template <int TPU>
__device__ __forceinline__ void class_sync(int lt) {
  if constexpr (TPU / 8 > 32)
    asm volatile("bar.sync %0, %1;" ::"r"(1 + lt / (TPU / 8)), "n"(TPU / 8) : "memory");
  else
    __syncwarp();
}
template <int TPU>
__device__ __forceinline__ int class_butterfly(int lt) {
  constexpr int n = TPU >= 8 ? TPU / 8 : 1;
  return 8 * (lt % n) + lt / n;
}

// Butterflies b[] of a Stockham pass of radix R over a unit's M-point
// transforms in z (padded indices): butterfly b reads z[b + j M/R], applies
// its twiddles (registers, or the shared table), and leaves its R outputs in v.
template <int M, int R, bool STW = false>
__device__ __forceinline__ void butterflies(C2 (&v)[8], const ulonglong2* z, const int (&bf)[8 / R], int Ns,
                                            const float2 (&tw)[7], const ulonglong2* stw = nullptr) {
  constexpr int B = 8 / R;       // butterflies per thread
  constexpr int S = M / R;       // input stride
#pragma unroll
  for (int r = 0; r < B; ++r) {
    const int b = bf[r];
    const int pb = fe_pad(b);
#pragma unroll
    for (int j = 0; j < R; ++j)
      v[r * R + j] = z_load(z, S % 64 == 0 ? pb + j * fe_pad(S) : fe_pad(b + j * S));
    if (Ns > 1) {
      const int k = b & (Ns - 1);
      const ulonglong2* row = STW ? stw + (Ns == 64 ? tw64_row(k) : k) * 7 : nullptr;
#pragma unroll
      for (int j = 1; j < R; ++j) {
        if constexpr (STW) {  // radix 8, one butterfly per thread: this thread's row of the table
          const ulonglong2 t = row[j - 1];
          v[r * R + j] = cmul(v[r * R + j], t.x, t.y);
        } else {
          const float2 t = tw[r * (R - 1) + j - 1];
          v[r * R + j] = cmul(v[r * R + j], p_dup(t.x), p_dup(t.y));
        }
      }
    }
  }
  if constexpr (R == 8) {
    dft8(v);
  } else if constexpr (R == 4) {
    dft4(v[0], v[1], v[2], v[3]);
    dft4(v[4], v[5], v[6], v[7]);
  } else {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const C2 a0 = v[2 * r], a1 = v[2 * r + 1];
      v[2 * r] = cadd(a0, a1);
      v[2 * r + 1] = csub(a0, a1);
    }
  }
}

// A radix-8 pass in place: butterfly b writes its outputs to
// (b div Ns) 8 Ns + (b mod Ns) + r Ns.  The first pass (Ns = 1) runs over the
// whole unit, whose barrier separates its loads and stores and ends it; the
// later ones run within the classes, the last one ended by the unit's barrier.
template <int M, int NT, int NS, bool LAST, bool STW = false>
__device__ __forceinline__ void fft_pass8(ulonglong2* z, int u, int lt, const float2 (&tw)[7],
                                          const ulonglong2* stw = nullptr) {
  constexpr int TPU = M / 8;
  const int b = NS == 1 ? lt : class_butterfly<TPU>(lt);
  C2 v[8];
  butterflies<M, 8, STW>(v, z, {b}, NS, tw, stw);
  if constexpr (NS == 1)
    unit_sync<TPU, NT>(u);
  else
    class_sync<TPU>(lt);
  const int k = b & (NS - 1);
  const int to = (b - k) * 8 + k;
  const int base = fe_pad(to);
#pragma unroll
  for (int j = 0; j < 8; ++j)  // (to is a multiple of 8 NS plus less than NS)
    z_store(z, NS == 1 ? base + j : NS == 8 ? base + 9 * j : base + j * fe_pad(NS), v[j]);
  if constexpr (NS == 1 || LAST)
    unit_sync<TPU, NT>(u);
  else
    class_sync<TPU>(lt);
}

// The equaliser in FP32, exactly: while the fix_36_24 product p = v g stays
// below 7.5 2^21 < 2^24 in magnitude, v (g 2^-21) is exact in FP32, and one
// fused multiply-add with 1.5 2^23 rounds it half to even; the sum's low four
// bits are the fix_4_3 code in two's complement.  Larger products saturate at
// +-7, which is the code of every v with p between 6.5 and 7.5 2^21: so the
// spectra are clamped to +-w, an integer w near 7 2^21 / g, and to the 18-bit
// range, before they are rounded to the code.  The interval is 14% of w wide,
// so a thread keeps w as a bfloat16 (an integer: w >= 56), two to a register.
__device__ __forceinline__ uint32_t clamp_bound(float gs) {  // gs = g 2^-21; bfloat16 bits
  const float w = fminf(__fdividef(7.0f, gs), 200000.0f);    // (g = 0: infinity)
  const float i = (w + 12582912.0f) - 12582912.0f;           // an integer
  return (__float_as_uint(i) + 0x8000u) >> 16;
}
// The 18-bit range and w as one clamp: w below 2^17, else 2^17 - 0.75; with
// kClampSkew the lower bound -(w + 0.375) rounds to -w or to -2^17.
constexpr float kClampSkew = 0.375f;
__device__ __forceinline__ float clamp18(uint32_t bits) {
  return fminf(__uint_as_float(bits), 131071.25f);
}

// With a gain of kWideGain or more, everything beyond the 18-bit range
// saturates (2^17 * 120 = 7.5 2^21), and so does all that lies past w: the
// spectra need no clamp before they are rounded, only the code does.  (A
// spectrum stays below 2^21: 128 sum |h| is at most 0.43 2^21, at 4096 samples
// and 16 taps, so v g 2^-21 < 2^18 and both magic roundings keep exact.)
constexpr uint32_t kWideGain = 120;
// A rounded code (the bits of 1.5 2^23 + q) clamped from below, to -7; s4_pack
// then saturates it from above.
__device__ __forceinline__ int code_floor(uint32_t bits) { return __viaddmax_s32((int)bits, -0x4B400000, -7); }
// low << 8 with the byte hi : lo of two codes, saturated to 4 bits, below it
__device__ __forceinline__ uint32_t s4_pack(int hi, int lo, uint32_t low) {
  uint32_t d;
  asm("cvt.pack.sat.s4.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(hi), "r"(lo), "r"(low));
  return d;
}

// n bytes of v (n = 4, 8 or 16) to any address: up to the next word by byte and
// half word, then whole words, then the rest: 8 stores for 16 bytes instead of 16
// (192 inputs x 1024 channels x 2047 spectra 4.1 -> 2.0 ms).  Not inlined: in
// the kernel it costs aligned outputs 0.8%.
__device__ __noinline__ void store_piece(uint8_t* d, uint4 v, int n) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  const int s = (int)(0u - (uint32_t)reinterpret_cast<uintptr_t>(d)) & 3;
  if (s & 1) d[0] = (uint8_t)w[0];
  if (s & 2) *reinterpret_cast<uint16_t*>(d + (s & 1)) = (uint16_t)(w[0] >> (8 * (s & 1)));
  uint32_t last = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (4 * i < n) {
      last = __funnelshift_r(w[i], i < 3 ? w[i + 1] : 0u, 8 * s);
      if (s == 0 || 4 * i + 4 < n) *reinterpret_cast<uint32_t*>(d + s + 4 * i) = last;
    }
  uint8_t* const e = d + n - 4 + s;  // 4 - s bytes remain, in `last`
  if (s && !(s & 2)) *reinterpret_cast<uint16_t*>(e) = (uint16_t)last, last >>= 16;
  if (s & 1) e[s & 2 ? 0 : 2] = (uint8_t)last;
  if (s == 2) *reinterpret_cast<uint16_t*>(e) = (uint16_t)last;
}

// clamp(rne(x), -2^17, 2^17 - 1): clamping first keeps |x| < 2^22, where
// adding 1.5 2^23 rounds x to the nearest integer, ties to even.  Returns
// the sum's bits less those of 1.5 2^23: the integer.
__device__ __forceinline__ int round18(float x) {
  const float c = fminf(fmaxf(x, -131072.0f), 131071.0f);
  return __float_as_int(c + 12582912.0f) - 0x4B400000;
}
// The same from a rounded spectrum's bits (those of 1.5 2^23 + its integer; a
// spectrum stays below 2^21, see kWideGain): two integer instructions.
__device__ __forceinline__ int value18(uint32_t bits) {
  return min(__viaddmax_s32((int)bits, -0x4B400000, -131072), 131071);
}

// Bytes r and r + 1 of w (biased: w holds x ^ 0x80 per byte, x the int8 sample)
// as the floats 1.5 2^23 + 128 + x: the byte becomes the low mantissa bits of
// 1.5 2^23, and subtracting 1.5 2^23 + 128 leaves x (every step exact below 2^24).
__device__ __forceinline__ uint64_t biased_bytes(uint32_t w, int r) {
  return ((uint64_t)__byte_perm(w, 0x4B400000u, 0x7650u + (unsigned)(r + 1)) << 32) |
         __byte_perm(w, 0x4B400000u, 0x7650u + (unsigned)r);
}

constexpr float kByteBias = 12583040.0f;

// Eight samples as pairs of floats, from the 8 bytes of an aligned load or one by one.
__device__ __forceinline__ void samples8(uint64_t (&x)[4], int2 w) {
  const uint32_t b[2] = {(uint32_t)w.x ^ 0x80808080u, (uint32_t)w.y ^ 0x80808080u};
  const uint64_t bias = p_dup(kByteBias);
#pragma unroll
  for (int r = 0; r < 4; ++r) x[r] = p_sub(biased_bytes(b[r >> 1], 2 * (r & 1)), bias);
}
__device__ __forceinline__ int2 load_bytes8(const int8_t* p) {
  uint32_t w[2] = {0u, 0u};
#pragma unroll
  for (int r = 0; r < 8; ++r) w[r >> 2] |= (uint32_t)(uint8_t)p[r] << (8 * (r & 3));
  return make_int2((int)w[0], (int)w[1]);
}

// Two CTAs per SM where 256-thread CTAs fit twice (registers capped at 128).
__host__ __device__ constexpr int fe_min_blocks(int logm) { return logm <= 11 ? 2 : 1; }

// What bounds it: latency.  128 registers a thread (32 hold the two spectra's
// eight points, 52 the taps and the next frames) leave 16 warps an SM, with
// issue slots 47% busy, the shared-memory data pipe 62% and FP32 42%; the time
// is close to proportional to the instructions of an iteration (about 1250 a
// thread), a quarter of them the separation and equaliser.  192 inputs x 1024
// channels x 2048 spectra: 2.02 -> 1.50 ms, in steps (ms): packed pairs and
// 16-byte points 1.94; frames loaded an iteration ahead, 16 staged spectra
// 1.78; the last pass and the separation in registers 1.59; classes within
// warps 1.56; instances for up to four taps 1.55; the code clamped instead of
// the spectra 1.52; no code for the other outputs, and the nibbles swapped
// by word where real parts are low, 1.50.
// POWER: accumulate Eq. 3's power sums, of 18-bit values clamped as integers
// beside the equaliser's own rounding, joined over a CTA's units before they
// are added to the caller's: ADC samples to visibilities and powers of 32 inputs
// x 256 channels x 4096 spectra 201 -> 174 us, 192 x 512 x 2048 1123 -> 929 (with
// the spectra clamped for both in floats, and every unit's sums added globally,
// before).  FRAMED: at most four taps and
// aligned frames, coefficients and frames in registers; otherwise any taps and
// alignment, the next frame's samples and coefficients read ahead (8 taps: fx
// of 64 inputs x 512 channels x 1024 spectra 318 -> 272 us, 192 x 1024 x 2048
// 2.54 -> 2.48 ms).  EXTRA: spectra or 18-bit values go out too (their code, in
// the loop four times over, costs the others 2 to 4%: 192 x 256 x 4096 spectra
// 683 -> 653 us, 192 x 1024 x 2048 1.523 -> 1.497 ms).  (Instances of their own,
// so that each keeps the others' registers free.)
template <int LOGM, bool POWER, bool FRAMED, bool EXTRA>
__global__ void __launch_bounds__(fe_threads(LOGM), fe_min_blocks(LOGM)) fengine_kernel(FeArgs a) {
  constexpr int M = 1 << LOGM, C = M / 2;
  constexpr int TPU = M / 8;                 // threads per FFT unit
  constexpr int NT = fe_threads(LOGM);
  constexpr int U = NT / TPU;                // units per CTA
  constexpr int PM = fe_pad(M);
  constexpr int P8 = LOGM / 3, REM = LOGM % 3;
  extern __shared__ __align__(16) uint8_t fe_smem[];
  const int tid = threadIdx.x, u = tid / TPU, lt = tid % TPU;
  ulonglong2* const z = reinterpret_cast<ulonglong2*>(fe_smem) + u * PM;
  ulonglong2* const ttab = reinterpret_cast<ulonglong2*>(fe_smem) + U * PM;  // [Ns=8 | Ns=64][k][7]
  // [channel of the thread][iteration][thread]: codes of two spectra, both inputs
  uint32_t* const codes = reinterpret_cast<uint32_t*>(ttab + kTwTable) + tid;
  // [channel of the thread][thread]: gains as g 2^-21 (exact) of the two inputs, and
  // their clamp bounds, bfloat16 each (registers are what limits the CTA)
  float2* const gains = reinterpret_cast<float2*>(codes - tid + 4 * kStageIts * NT) + tid;
  uint32_t* const bounds = reinterpret_cast<uint32_t*>(gains - tid + 4 * NT) + tid;
  const int i0 = 2 * (a.pairs_first ? blockIdx.x : blockIdx.y);
  const int grp = a.pairs_first ? blockIdx.y : blockIdx.x;  // the CTA's group of spectra
  const bool has1 = i0 + 1 < a.n_inputs;
  const int N = a.n_inputs;
  // [t][c][i] codes: both inputs' as one half word
  const bool pair16 = has1 && ((N | (int)reinterpret_cast<uintptr_t>(a.out)) & 1) == 0;
  // this unit's spectra tu .. tu + per_unit - 1, two an iteration; the first
  // unit's range, the earliest, says how many iterations the CTA makes
  const int tu = (grp * U + u) * a.per_unit;
  const int n_it = (min(a.per_unit, a.n_spectra - grp * U * a.per_unit) + 1) / 2;

  // per-thread constants: the filter taps of its 8 samples (neighbouring
  // samples in pairs; absent taps are zeros) and the twiddles of every pass
  uint64_t hr[4][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
#pragma unroll
    for (int r = 0; r < 4; r += 2) {
      ulonglong2 v = make_ulonglong2(0, 0);
      if (FRAMED && q < a.taps) v = __ldg(reinterpret_cast<const ulonglong2*>(a.h + q * M + 8 * lt + 2 * r));
      hr[q][r] = v.x, hr[q][r + 1] = v.y;
    }
  }
  // passes at Ns = 8 and 64 read the shared table (filled here, first read
  // after the barrier below); a pass at Ns = 512 (M = 4096) keeps registers
  for (int e = tid; e < kTwTable; e += NT) {
    const int big = e >= 56, q = big ? e - 56 : e, k = q / 7, j = q % 7 + 1;
    const int Ns = big ? 64 : 8;
    if (M >= 8 * Ns) {
      const float2 t = __ldg(&a.w[j * k * (M / (8 * Ns))]);
      ttab[big ? 56 + tw64_row(k) * 7 + j - 1 : e] = make_ulonglong2(p_dup(t.x), p_dup(t.y));
    }
  }
  float2 tw[1][7], twl[7];
  if constexpr (P8 >= 4) load_twiddles<M, 8>(tw[0], {class_butterfly<TPU>(lt)}, 512, a.w);
  constexpr int RL = REM ? 1 << REM : 8;  // radix of the last pass
  int bl[8 / RL] = {};                    // its butterflies, and the channels they give
  if constexpr (REM != 0) {
    last_butterflies<M, RL>(lt, bl);
    load_twiddles<M, RL>(twl, bl, M / RL, a.w);
  }
  // channel k of this thread: the first RL/2 outputs of each butterfly
  // (without a last pass of its own, lt + k TPU)
  auto channel = [&](int k) { return REM ? bl[k / (RL / 2)] + k % (RL / 2) * (M / RL) : lt + k * TPU; };

  unsigned long long pw[4][2];  // only used by the POWER instance
  bool wide = true;             // every gain of this CTA is 0 or kWideGain and more
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const long long g = (long long)channel(k) * N + i0;
    const uint32_t n0 = a.gain[g], n1 = has1 ? a.gain[g + 1] : 0u;
    wide = wide && (n0 == 0 || n0 >= kWideGain) && (n1 == 0 || n1 >= kWideGain);
    const float g0 = (float)n0 * 4.76837158203125e-07f, g1 = (float)n1 * 4.76837158203125e-07f;  // 2^-21
    gains[k * NT] = make_float2(g0, g1);
    bounds[k * NT] = clamp_bound(g0) | (clamp_bound(g1) << 16);
    pw[k][0] = pw[k][1] = 0ull;
  }
  wide = __syncthreads_and(wide);  // (and the table is filled)

  const int8_t* const xt = a.adc + (long long)i0 * a.adc_stride + (long long)tu * M + 8 * lt;
  // the five frames of the unit's next two spectra, both inputs, as loaded:
  // requested an iteration ahead, so that the FFT hides their latency (loads
  // at the filter itself, with the L1 prefetched, cost 18%)
  int2 raw[5][2];
  auto load_frame = [&](int f, int s) {  // frame f of spectra s, s + 1 (if one of them uses it)
    raw[f][0] = raw[f][1] = make_int2(0, 0);
    if (f > min(2, a.n_spectra - tu - s) + a.taps - 2) return;
    const int8_t* x = xt + (long long)(s + f) * M;
    raw[f][0] = __ldg(reinterpret_cast<const int2*>(x));
    if (has1) raw[f][1] = __ldg(reinterpret_cast<const int2*>(x + a.adc_stride));
  };
  if constexpr (FRAMED) {
#pragma unroll
    for (int f = 0; f < 5; ++f) load_frame(f, 0);
  }

  for (int it = 0; it < n_it; ++it) {
    const int s = 2 * it;                              // this unit's spectra: tu + s and the next
    const int n_act = min(2, a.n_spectra - tu - s);    // how many of them exist (<= 0: none)
    // ---- polyphase filter: y[n] = sum_q h[q M + n] x[(t + q) M + n]
    // The two spectra share frames: each is converted once and added into the
    // spectra that use it, in the order of their taps.  Pairs here are
    // neighbouring samples, as the coefficients lie.
    uint64_t y[2][2][4];  // [spectrum][input][sample pair]
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
      for (int r = 0; r < 4; ++r) y[e][0][r] = y[e][1][r] = 0ull;
    if constexpr (FRAMED) {
#pragma unroll
      for (int f = 0; f < 5; ++f) {
        if (f > a.taps) break;
        uint64_t x[2][4];  // (frames past the last spectrum's are zeros)
        samples8(x[0], raw[f][0]);
        samples8(x[1], raw[f][1]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int q = f - e;  // this frame is tap q of spectrum e
          if (q < 0 || q > 3) continue;
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            y[e][0][r] = p_fma(hr[q][r], x[0][r], y[e][0][r]);
            y[e][1][r] = p_fma(hr[q][r], x[1][r], y[e][1][r]);
          }
        }
      }
      // the next iteration's frames: two spectra on, taps - 1 of the five stay
      if (it + 1 < n_it) {
#pragma unroll
        for (int f = 0; f < 5; ++f) {
          if (f < 3 && f <= a.taps - 2)
            raw[f][0] = raw[f + 2][0], raw[f][1] = raw[f + 2][1];
          else
            load_frame(f, s + 2);
        }
      }
    } else {  // any number of taps, any alignment
      uint64_t hp[4] = {0ull, 0ull, 0ull, 0ull};  // the tap before
      ulonglong2 hn[2];                           // the next frame's coefficients and samples
      int2 xn[2];
      auto load = [&](int f) {
        hn[0] = hn[1] = make_ulonglong2(0, 0);
        if (f < a.taps) {
          hn[0] = __ldg(reinterpret_cast<const ulonglong2*>(a.h + f * M + 8 * lt));
          hn[1] = __ldg(reinterpret_cast<const ulonglong2*>(a.h + f * M + 8 * lt + 4));
        }
        const int8_t* xf = xt + (long long)(s + f) * M;
        xn[0] = a.vec_in ? __ldg(reinterpret_cast<const int2*>(xf)) : load_bytes8(xf);
        xf += a.adc_stride;
        xn[1] = !has1 ? make_int2(0, 0) : a.vec_in ? __ldg(reinterpret_cast<const int2*>(xf)) : load_bytes8(xf);
      };
      const int n_f = n_act + a.taps - 1;
      if (n_act > 0) load(0);
#pragma unroll 1
      for (int f = 0; n_act > 0 && f < n_f; ++f) {
        uint64_t x[2][4], hq[4] = {hn[0].x, hn[0].y, hn[1].x, hn[1].y};
        samples8(x[0], xn[0]);
        samples8(x[1], xn[1]);
        if (f + 1 < n_f) load(f + 1);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          if (f < a.taps) {
            y[0][0][r] = p_fma(hq[r], x[0][r], y[0][0][r]);
            y[0][1][r] = p_fma(hq[r], x[1][r], y[0][1][r]);
          }
          if (f > 0 && n_act > 1) {
            y[1][0][r] = p_fma(hp[r], x[0][r], y[1][0][r]);
            y[1][1][r] = p_fma(hp[r], x[1][r], y[1][1][r]);
          }
          hp[r] = hq[r];
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float v[2][2][2];  // [spectrum][input][sample]
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int j = 0; j < 2; ++j) p_unpack(y[e][j][r], v[e][j][0], v[e][j][1]);
#pragma unroll
      for (int i = 0; i < 2; ++i)
        z_store(z, fe_pad(8 * lt) + 2 * r + i, {p_pack(v[0][0][i], v[1][0][i]), p_pack(v[0][1][i], v[1][1][i])});
    }
    unit_sync<TPU, NT>(u);
    // ---- FFTs of y_2k + j y_2k+1 (natural order out)
    fft_pass8<M, NT, 1, P8 == 1>(z, u, lt, twl);  // first pass: no twiddles
    if constexpr (P8 >= 2) fft_pass8<M, NT, 8, P8 == 2, true>(z, u, lt, twl, ttab);
    if constexpr (P8 >= 3) fft_pass8<M, NT, 64, P8 == 3, true>(z, u, lt, twl, ttab + 56);
    if constexpr (P8 >= 4) fft_pass8<M, NT, 512, P8 == 4>(z, u, lt, tw[0]);
    C2 v[8];
    if constexpr (REM != 0) butterflies<M, RL>(v, z, bl, M / RL, twl);
    // ---- Eq. 2 separation, 18-bit rounding, equaliser
    if (n_act > 0) {
      const uint64_t scale = p_dup(a.scale), magic = p_dup(12582912.0f);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int nu = channel(k);
        C2 zp, zm;
        if constexpr (REM != 0) {
          constexpr int H = RL / 2;
          const int q = k / H, r = k % H;  // output r of butterfly q; its mirror is output RL-1-r of butterfly q^1
          zp = v[q * RL + r];
          zm = v[(q ^ 1) * RL + RL - 1 - r];
          if (q < 2 && lt == 0) zm = q == 0 ? v[(RL - r) % RL] : v[RL + RL - 1 - r];  // its own mirror
        } else {
          zp = z_load(z, fe_pad(nu));
          zm = z_load(z, fe_pad((M - nu) & (M - 1)));
        }
        // X[input][re, im] of both spectra
        const uint64_t X[2][2] = {{p_mul(p_add(zp.x, zm.x), scale), p_mul(p_sub(zp.y, zm.y), scale)},
                                  {p_mul(p_add(zp.y, zm.y), scale), p_mul(p_sub(zm.x, zp.x), scale)}};
        if (EXTRA && (a.spec || a.v18)) {
          float x[2][2][2];  // [input][re, im][spectrum]
#pragma unroll
          for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int c = 0; c < 2; ++c) p_unpack(X[j][c], x[j][c][0], x[j][c][1]);
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            if (e >= n_act) break;
            const long long ei = (((long long)(tu + s + e) * C + nu) * N + i0) * 2;
            if (a.spec) {
              float* o = a.spec + ei;
              if (a.vec_extra) {
                *reinterpret_cast<float4*>(o) = make_float4(x[0][0][e], x[0][1][e], x[1][0][e], x[1][1][e]);
              } else {
                *reinterpret_cast<float2*>(o) = make_float2(x[0][0][e], x[0][1][e]);
                if (has1) *reinterpret_cast<float2*>(o + 2) = make_float2(x[1][0][e], x[1][1][e]);
              }
            }
            if (a.v18) {
              int32_t* o = a.v18 + ei;
              const int v[4] = {round18(x[0][0][e]), round18(x[0][1][e]), round18(x[1][0][e]), round18(x[1][1][e])};
              if (a.vec_extra) {
                *reinterpret_cast<int4*>(o) = make_int4(v[0], v[1], v[2], v[3]);
              } else {
                *reinterpret_cast<int2*>(o) = make_int2(v[0], v[1]);
                if (has1) *reinterpret_cast<int2*>(o + 2) = make_int2(v[2], v[3]);
              }
            }
          }
        }
        const float2 gk = gains[k * NT];
        uint32_t q[2][2][2];  // [re, im][input][spectrum]: the bits of 1.5 2^23 + code
        if constexpr (POWER) {  // Eq. 3's sums of the 18-bit values, clamped as integers
#pragma unroll
          for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              const uint64_t r = p_add(X[j][c], magic);
              const int v0 = value18((uint32_t)r), v1 = value18((uint32_t)(r >> 32));
              pw[k][j] += (unsigned long long)((long long)v0 * v0);
              if (n_act > 1) pw[k][j] += (unsigned long long)((long long)v1 * v1);
            }
        }
        if (!wide) {
          const uint32_t bound = bounds[k * NT];
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const uint64_t g = p_dup(j ? gk.y : gk.x);
            const uint32_t wb = j ? bound & 0xFFFF0000u : bound << 16;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              float x0, x1;
              p_unpack(X[j][c], x0, x1);
              // the rounded spectrum, clamped to the bound
              const float hi = clamp18(wb), lo = -(hi + kClampSkew);
              const uint64_t f =
                  p_sub(p_add(p_pack(fminf(fmaxf(x0, lo), hi), fminf(fmaxf(x1, lo), hi)), magic), magic);
              const uint64_t e = p_fma(f, g, magic);
              q[c][j][0] = (uint32_t)e;
              q[c][j][1] = (uint32_t)(e >> 32);
            }
          }
        } else {
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const uint64_t g = p_dup(j ? gk.y : gk.x);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              const uint64_t e = p_fma(p_sub(p_add(X[j][c], magic), magic), g, magic);
              q[c][j][0] = (uint32_t)e;
              q[c][j][1] = (uint32_t)(e >> 32);
            }
          }
        }
        // bytes [spectrum][input], the last one first
        uint32_t word = 0;
#pragma unroll
        for (int b = 3; b >= 0; --b) {
          const int re = code_floor(q[0][b & 1][b >> 1]), im = code_floor(q[1][b & 1][b >> 1]);
          word = s4_pack(re, im, word);
        }
        if (a.lo_is_real) word = ((word >> 4) & 0x0F0F0F0Fu) | ((word & 0x0F0F0F0Fu) << 4);
        if (a.layout == CORR_L_CIT) {
          codes[(k * kStageIts + it % kStageIts) * NT] = word;
        } else if (a.out) {  // [t][c][i]
          uint8_t* o = a.out + ((long long)(tu + s) * C + nu) * N + i0;
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            if (e >= n_act) break;
            if (pair16) {
              *reinterpret_cast<uint16_t*>(o + (long long)e * C * N) = (uint16_t)(word >> (16 * e));
              continue;
            }
            o[(long long)e * C * N] = (uint8_t)(word >> (16 * e));
            if (has1) o[(long long)e * C * N + 1] = (uint8_t)(word >> (16 * e + 8));
          }
        }
      }
    }
    // ---- codes out to [c][i][t], when a stage is full: the thread's own
    // channels, 16 spectra (or all it has, fewer) of each input as one piece
    if (a.out && a.layout == CORR_L_CIT && (it % kStageIts == kStageIts - 1 || it == n_it - 1)) {
      const int first = it / kStageIts * kStageIts;  // iteration of the stage's first spectra
      const int cnt = min(2 * (it + 1 - first), a.n_spectra - tu - 2 * first);
      const int whole = min(a.per_unit, 2 * kStageIts);
#pragma unroll 1
      for (int k = 0; k < 4 && cnt > 0; ++k) {
        int nu = channel(0);  // (a dynamic k)
#pragma unroll
        for (int kk = 1; kk < 4; ++kk)
          if (kk == k) nu = channel(kk);
        const uint32_t* const src = codes + k * kStageIts * NT;
        uint8_t* o = a.out + ((long long)nu * N + i0) * a.out_stride + tu + 2 * first;
        if (cnt == whole && whole >= 4) {
          uint32_t w[2][4];
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const uint32_t w0 = 4 * h < cnt ? src[2 * h * NT] : 0u, w1 = 4 * h < cnt ? src[(2 * h + 1) * NT] : 0u;
            w[0][h] = __byte_perm(w0, w1, 0x6420);
            w[1][h] = __byte_perm(w0, w1, 0x7531);
          }
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            if (j == 1 && !has1) break;
            uint8_t* d = o + j * a.out_stride;
            if (!a.vec_out)
              store_piece(d, make_uint4(w[j][0], w[j][1], w[j][2], w[j][3]), whole);
            else if (whole == 16)
              *reinterpret_cast<uint4*>(d) = make_uint4(w[j][0], w[j][1], w[j][2], w[j][3]);
            else if (whole == 8)
              *reinterpret_cast<uint2*>(d) = make_uint2(w[j][0], w[j][1]);
            else
              *reinterpret_cast<uint32_t*>(d) = w[j][0];
          }
        } else if (a.vec_two && cnt == 2) {
          const uint32_t w = src[0];
          *reinterpret_cast<uint16_t*>(o) = (uint16_t)__byte_perm(w, 0u, 0x4420);
          if (has1) *reinterpret_cast<uint16_t*>(o + a.out_stride) = (uint16_t)__byte_perm(w, 0u, 0x4431);
        } else {
          for (int q = 0; q < cnt; ++q) {
            const uint32_t w = src[(q >> 1) * NT] >> (16 * (q & 1));
            o[q] = (uint8_t)w;
            if (has1) o[a.out_stride + q] = (uint8_t)(w >> 8);
          }
        }
      }
    }
    unit_sync<TPU, NT>(u);  // z is read: the next iteration may fill it
  }

  if constexpr (POWER) {
    // the units of a CTA have the same channels: their sums meet in shared memory
    // (z is free), and one unit's threads add them to the caller's
    unsigned long long* const sums = reinterpret_cast<unsigned long long*>(fe_smem);  // [q][unit][lt]
    if constexpr (U > 1) {
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 8; ++q) sums[q * NT + tid] = pw[q >> 1][q & 1];
      __syncthreads();
    }
    if (U > 1 && u > 0) return;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      unsigned long long v = pw[q >> 1][q & 1];
      for (int e = 1; e < U; ++e) v += sums[q * NT + e * TPU + lt];
      if ((q & 1) == 0 || has1) atomicAdd(a.power + (long long)channel(q >> 1) * N + i0 + (q & 1), v);
    }
  }
}

template <int LOGM, bool POWER, bool FRAMED, bool EXTRA>
cudaError_t fe_launch_one(const FeArgs& a, int n_pairs, cudaStream_t s) {
  constexpr int M = 1 << LOGM;
  constexpr size_t smem = fe_smem_bytes<LOGM>();
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(fengine_kernel<LOGM, POWER, FRAMED, EXTRA>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  // Spectra per unit: as many (few prologues and power additions, the output in
  // whole pieces) as leave five CTAs for six slots of the chip: 8 inputs x 128
  // channels x 4096 spectra 21 us at 8 (256 CTAs) against 25 at 4 and 39 at 32;
  // 64 x 64 x 2048 33 us at 16 (256) against 39 at 4; 16 x 128 x 100 10.8 at 2
  // against 57 at 32.
  // (From 32 to 16, whose pieces are as large, also where 32 leave between one
  // and 16/9 CTAs a slot, for fuller waves: over 16 to 1024 channels and 8 to 192
  // inputs, with powers and without, 16 take 0.83 - 0.90 of the time of 32 at 305
  // to 368 CTAs, 0.97 - 1.03 to 448, 0.91 - 0.96 to 530, and 1.03 - 1.08 from 560 on.)
  // Where the pieces of [c][i][t] codes are whole words at 4, the step to 2 pays
  // only below one CTA for two SMs: 6 inputs x 256 channels x 1024 spectra (192
  // CTAs at 4) 15 us at 4 against 21 at 2 (29 with its pieces in bytes), 3 x 64 x
  // 4096 with spectra (128) 11 against 12.8 (15); 16 x 64 x 200 (32) 10.9 against
  // 9.0.  (Not for 16 and 32 channels, whose units are 4 and 8 threads: 16 x 16 x
  // 4096 8.6 at 4 against 7.0.)
  FeArgs b = a;
  const bool pieces = LOGM >= 7 && a.out && a.layout == CORR_L_CIT &&
                      ((reinterpret_cast<uintptr_t>(a.out) | (uintptr_t)a.out_stride) & 3) == 0;
  const int slots = device_sm_count() * fe_min_blocks(LOGM);
  for (b.per_unit = 32; b.per_unit > 2; b.per_unit /= 2) {
    const int group = b.per_unit * fe_units(LOGM);
    const long long ctas = (long long)((a.n_spectra + group - 1) / group) * n_pairs;
    if (b.per_unit == 32 && ctas > slots && ctas <= slots * 16 / 9) continue;
    if (ctas >= (pieces && b.per_unit == 4 ? device_sm_count() / 2 : slots * 5 / 6)) break;
  }
  // (64 inputs x 64 channels x 128 spectra 10.6 us in bytes, 8.6 in half words)
  b.vec_two = b.per_unit == 2 && ((reinterpret_cast<uintptr_t>(a.out) | (uintptr_t)a.out_stride) & 1) == 0;
  const int group = b.per_unit * fe_units(LOGM);
  // [t][c][i] codes, spectra and 18-bit values: the inputs of a pair are 2 bytes of
  // codes, 8 or 16 of the others, so neighbouring pairs write the same sectors.
  // Together they may be larger than the L2, which then writes out sectors before
  // their other pairs come: CTAs of neighbouring pairs run together (192 inputs x
  // 1024 channels x 2048 spectra 5.1 -> 2.35 ms, 191 x 256 x 8192 5.55 -> 3.05;
  // spectra of 64 x 1024 x 512 276 -> 210 us).  What fits joins there in any order,
  // and neighbouring groups of spectra, which share frames, are better run
  // together (191 x 1024 x 64 codes 167 -> 140 us, 33 x 64 x 2048 33.5 -> 31.2).
  // The line lies between 113 MB, where groups are ahead by up to 17%, and 133 MB,
  // where pairs are by 5 to 50%.  With spectra or 18-bit values groups are ahead
  // below it only from many pairs on (191 x 256 x 128 and codes 121 -> 95 us; 17 and
  // 33 inputs 3 to 14% the other way, 9 and 65 mixed).
  const int groups = (a.n_spectra + group - 1) / group;
  const long long samples = (long long)M * a.n_spectra * n_pairs;  // (of both inputs: M / 2 channels)
  const long long joined = samples * ((a.out && a.layout != CORR_L_CIT ? 1 : 0) + (a.spec ? 8 : 0) + (a.v18 ? 8 : 0));
  b.pairs_first = (joined > kL2Bytes || ((a.spec || a.v18) && n_pairs <= 64)) && groups <= 65535;
  const dim3 grid = b.pairs_first ? dim3(n_pairs, groups) : dim3(groups, n_pairs);
  fengine_kernel<LOGM, POWER, FRAMED, EXTRA><<<grid, fe_threads(LOGM), smem, s>>>(b);
  return cudaGetLastError();
}

template <int LOGM>
cudaError_t fe_launch(const FeArgs& a, int n_pairs, cudaStream_t s) {
  if (a.vec_in && a.taps <= 4) {
    if (a.spec || a.v18)
      return a.power ? fe_launch_one<LOGM, true, true, true>(a, n_pairs, s)
                     : fe_launch_one<LOGM, false, true, true>(a, n_pairs, s);
    return a.power ? fe_launch_one<LOGM, true, true, false>(a, n_pairs, s)
                   : fe_launch_one<LOGM, false, true, false>(a, n_pairs, s);
  }
  return a.power ? fe_launch_one<LOGM, true, false, true>(a, n_pairs, s)
                 : fe_launch_one<LOGM, false, false, true>(a, n_pairs, s);
}

bool fe_is_device(const void* p) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

void fe_free(fe_ctx* f) {
  if (!f) return;
  if (f->stream) cudaStreamSynchronize(f->stream);
  cudaFree(f->h);
  cudaFree(f->w);
  cudaFree(f->gain);
  if (f->own_stream && f->stream) cudaStreamDestroy(f->stream);
  delete f;
}

}  // namespace
}  // namespace xe

using namespace xe;

extern "C" {

int fe_create(int n_inputs, int n_chans, int taps, int shift, unsigned flags, void* stream,
              fe_ctx** out) {
  TraceRange trace_("fe_create");
  if (!out) return CORR_EINVAL;
  *out = nullptr;
  if (n_inputs < 1 || n_inputs > 131070 || n_chans < 16 || n_chans > 2048 ||
      (n_chans & (n_chans - 1)) || taps < 1 || taps > 16 || shift < 0 || shift > 24 ||
      (flags & ~FE_F_LO_IS_REAL))
    return CORR_EINVAL;
  fe_ctx* f = new (std::nothrow) fe_ctx;
  if (!f) return CORR_ENOMEM;
  f->n_inputs = n_inputs;
  f->n_chans = n_chans;
  f->taps = taps;
  f->shift = shift;
  f->flags = flags;
  const int M = 2 * n_chans;
  const long long L = (long long)taps * M;
  // prototype: Hamming window times sinc, in FP64, rounded to FP32
  std::vector<float> h(L);
  const double pi = 3.14159265358979323846;
  for (long long m = 0; m < L; ++m) {
    const double win = 0.54 - 0.46 * std::cos(2.0 * pi * (double)m / (double)(L - 1));
    const double x = ((double)m - (double)(L - 1) / 2.0) / (double)M;
    const double sinc = x == 0.0 ? 1.0 : std::sin(pi * x) / (pi * x);
    h[m] = (float)(win * sinc);
  }
  std::vector<float2> w(M);
  for (int n = 0; n < M; ++n) {
    const double ang = -2.0 * pi * (double)n / (double)M;
    w[n] = make_float2((float)std::cos(ang), (float)std::sin(ang));
  }
  int st = CORR_OK;
  do {
    if (stream) {
      f->stream = (cudaStream_t)stream;
    } else {
      if (cudaStreamCreateWithFlags(&f->stream, cudaStreamNonBlocking) != cudaSuccess) { st = CORR_ECUDA; break; }
      f->own_stream = true;
    }
    if (cudaMalloc(&f->h, L * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&f->w, M * sizeof(float2)) != cudaSuccess ||
        cudaMalloc(&f->gain, (size_t)n_chans * n_inputs * sizeof(uint32_t)) != cudaSuccess) {
      st = CORR_ENOMEM;
      break;
    }
    if (cudaMemcpy(f->h, h.data(), L * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(f->w, w.data(), M * sizeof(float2), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(f->gain, 0, (size_t)n_chans * n_inputs * sizeof(uint32_t)) != cudaSuccess) {
      st = CORR_ECUDA;
      break;
    }
  } while (0);
  if (st != CORR_OK) {
    fe_free(f);
    return st;
  }
  *out = f;
  return CORR_OK;
}

int fe_set_gains(fe_ctx* f, const uint32_t* gain) {
  if (!f || !gain) return CORR_EINVAL;
  const size_t n = (size_t)f->n_chans * f->n_inputs;
  if (fe_is_device(gain)) {
    // checked on the host: a device table is copied back once
    std::vector<uint32_t> hg(n);
    if (cudaMemcpy(hg.data(), gain, n * sizeof(uint32_t), cudaMemcpyDeviceToHost) != cudaSuccess)
      return CORR_ECUDA;
    for (uint32_t v : hg)
      if (v >= (1u << 18)) return CORR_EINVAL;
  } else {
    for (size_t k = 0; k < n; ++k)
      if (gain[k] >= (1u << 18)) return CORR_EINVAL;
  }
  if (cudaMemcpyAsync(f->gain, gain, n * sizeof(uint32_t), cudaMemcpyDefault, f->stream) != cudaSuccess ||
      cudaStreamSynchronize(f->stream) != cudaSuccess)
    return CORR_ECUDA;
  return CORR_OK;
}

int fe_channelise(fe_ctx* f, const int8_t* adc, long long adc_stride, int n_spectra, uint8_t* out,
                  int layout, long long out_stride, int32_t* v18, float* spec, int64_t* power) {
  TraceRange trace_("fe_channelise");
  if (!f || !adc || n_spectra < 1) return CORR_EINVAL;
  const int M = 2 * f->n_chans;
  if (adc_stride < (long long)(n_spectra + f->taps - 1) * M) return CORR_EINVAL;
  if (layout != CORR_L_CIT && layout != CORR_L_TCI) return CORR_EINVAL;
  if (out && layout == CORR_L_CIT && out_stride < n_spectra) return CORR_EINVAL;
  if (!fe_is_device(adc) || (out && !fe_is_device(out)) || (v18 && !fe_is_device(v18)) ||
      (spec && !fe_is_device(spec)) || (power && !fe_is_device(power)))
    return CORR_EINVAL;
  if ((v18 && reinterpret_cast<uintptr_t>(v18) % 8) || (spec && reinterpret_cast<uintptr_t>(spec) % 8) ||
      (power && reinterpret_cast<uintptr_t>(power) % 8))
    return CORR_EINVAL;
  FeArgs a{};
  a.adc = adc;
  a.adc_stride = adc_stride;
  a.h = f->h;
  a.w = f->w;
  a.gain = f->gain;
  a.out = out;
  a.out_stride = out_stride;
  a.v18 = v18;
  a.spec = spec;
  a.power = reinterpret_cast<unsigned long long*>(power);
  a.n_inputs = f->n_inputs;
  a.n_spectra = n_spectra;
  a.taps = f->taps;
  a.layout = layout;
  a.lo_is_real = (f->flags & FE_F_LO_IS_REAL) ? 1 : 0;
  a.vec_in = reinterpret_cast<uintptr_t>(adc) % 8 == 0 && adc_stride % 8 == 0;
  a.vec_extra = f->n_inputs % 2 == 0 && reinterpret_cast<uintptr_t>(a.spec) % 16 == 0 &&
                reinterpret_cast<uintptr_t>(a.v18) % 16 == 0;
  a.vec_out = out && layout == CORR_L_CIT && reinterpret_cast<uintptr_t>(out) % 16 == 0 &&
              out_stride % 16 == 0;
  a.scale = std::ldexp(1.0f, -(f->shift + 1));
  const int pairs = (f->n_inputs + 1) / 2;
  cudaError_t e;
  switch (M) {
    case 32: e = fe_launch<5>(a, pairs, f->stream); break;
    case 64: e = fe_launch<6>(a, pairs, f->stream); break;
    case 128: e = fe_launch<7>(a, pairs, f->stream); break;
    case 256: e = fe_launch<8>(a, pairs, f->stream); break;
    case 512: e = fe_launch<9>(a, pairs, f->stream); break;
    case 1024: e = fe_launch<10>(a, pairs, f->stream); break;
    case 2048: e = fe_launch<11>(a, pairs, f->stream); break;
    case 4096: e = fe_launch<12>(a, pairs, f->stream); break;
    default: return CORR_EINVAL;
  }
  return e == cudaSuccess ? CORR_OK : CORR_ECUDA;
}

int fe_gains_from_power(const int64_t* power, int n_chans, int n_inputs, long long n_spectra,
                        double target_rms, uint32_t* gain) {
  if (!power || !gain || n_chans < 1 || n_inputs < 1 || n_spectra < 1 || !(target_rms > 0.0))
    return CORR_EINVAL;
  const long long n = (long long)n_chans * n_inputs;
  for (long long k = 0; k < n; ++k) {
    if (power[k] < 0) return CORR_EINVAL;
    if (power[k] == 0) {
      gain[k] = 0;
      continue;
    }
    const double rms = std::sqrt((double)power[k] / (2.0 * (double)n_spectra));
    const double g = std::nearbyint(target_rms * 2097152.0 / rms);
    gain[k] = g < 1.0 ? 1u : (g > 262143.0 ? 262143u : (uint32_t)g);
  }
  return CORR_OK;
}

int fe_sync(fe_ctx* f) {
  if (!f) return CORR_EINVAL;
  return cudaStreamSynchronize(f->stream) == cudaSuccess ? CORR_OK : CORR_ECUDA;
}

void fe_destroy(fe_ctx* f) { fe_free(f); }

}  // extern "C"
