// fm_voice.cu -- the 4-operator FM voice: four sine operators in a serial
// phase-modulation stack op3 -> op2 -> op1 -> op0 (Chowning's FM as phase
// modulation), each at f0 x ratio_i with the Voice's ADSR gated by the
// keyboard's note-on duration; out(n) = y_0(n) with y_4 = 0 and
// y_i(n) = level_i E_i(n) sin(2 pi phi_i(n) + y_(i+1)(n)). The paper names a
// 4-operator FM architecture as in development (Sec. 3.2) and specifies no
// more; parameter ranges and the stack are this library's choices.
//
// One CTA renders one voice's chunk of samples (fm_chunk): it draws (or loads)
// the 30 normalized parameters, maps them, turns each operator's frequency
// into a 64-bit fixed-point phase increment (the phase of sample n is the
// exact product n x inc mod 2^64), evaluates the four envelopes at the
// control points the chunk spans, and then renders 4-sample quads. No FP64:
// the increments come from the float-float exp2 of the Voice's control chain.
//
// What bounds it: instruction issue (the 90 MB that a batch of 128 x 4 s
// writes take 13.5 us). So the audio loop runs two samples at a time in packed
// FP32 (f32x2.cuh), a sine is one odd polynomial after a half-turn reduction
// instead of two chosen by quarter turn, levels are folded into the envelopes,
// signals between operators are kept in cycles, and only a quad that meets two
// intervals (never with R a multiple of 4) looks at the second. 128 x 4 s:
// 116 us before, 72 us (error against 64 bits 7.8e-7 -> 3.1e-7: the phases are now
// rounded to 2^-26 cycles where they were cut off at 2^-24).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "control_ff.cuh"
#include "f32x2.cuh"
#include "internal.h"
#include "voice_device.cuh"

namespace synth {
namespace {

constexpr int kFmThreads = 256;
constexpr int kFmCtasPerSm = 4;
constexpr uint32_t kStreamFmParam = 2;

struct FmConst {
  int64_t N, rate_a, rate_b;  // samples; R = rate_a / rate_b samples per control interval
  ff inv_cr;                  // 1 / control rate
  int chunk;                  // samples per CTA (a multiple of 4)
  int max_pts;                // control points a chunk can span
  ff log2_440_over_sr;        // log2(440 / SR)
  alignas(16) FFTables T;     // float-float exp2 tables
};

// Normalized parameter p -> human value, y = lo + (hi - lo) u^c with c = 1
// or 2 (exact products). Layout: midi f0, note-on duration, then per
// operator (0 = carrier) ratio, level, attack, decay, sustain, release, alpha.
__host__ __device__ inline void fm_range(int p, float& lo, float& hi, int& c) {
  if (p < 2) {
    lo = 0.f;
    hi = p == 0 ? 127.f : 4.f;
    c = 1;
    return;
  }
  const int i = (p - 2) / 7, q = (p - 2) % 7;
  const float los[7] = {0.5f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.1f};
  const float his[7] = {8.f, 8.f, 2.f, 2.f, 1.f, 5.f, 6.f};
  const int cs[7] = {2, 2, 2, 2, 1, 2, 2};
  lo = los[q];
  hi = (q == 1 && i == 0) ? 1.f : his[q];  // the carrier's level is an amplitude in [0, 1]
  c = (q == 1 && i == 0) ? 1 : cs[q];
}

// The Voice's ADSR (attack (t/a)^alpha, decay to s, release from the level at
// note-off d); zero-length sections are skipped. The section lengths, the
// note-on duration and the time are float-float, and so are the section
// choice and the time into the section (t - a, t - d): the argument x of
// x^alpha then carries a relative error of a few float roundings wherever
// the section falls in the note. (In FP32 the time alone is off by up to
// t 2^-24 s, which near a section start with alpha < 1 -- where x^alpha is
// steep -- moves the envelope by 1e-5 and more.) x^alpha itself is FP32.
struct FmEnv {
  ff a, dc, r, d;  // attack, decay, release, note-on duration (s)
  float s, alpha;  // sustain level, curve exponent
};
__device__ __forceinline__ float fm_pow(ff x, ff len, float alpha) {
  return powf(ff_to_float(x) / ff_to_float(len), alpha);
}
// Gate-on level at time t.
__device__ __forceinline__ float fm_gate_on(ff t, const FmEnv& E) {
  if (ff_lt(t, E.a)) return fm_pow(t, E.a, E.alpha);
  const ff ta = ff_sub(t, E.a);
  if (ff_lt(ta, E.dc)) return 1.f - (1.f - E.s) * fm_pow(ta, E.dc, E.alpha);
  return E.s;
}
// The envelope at time t; level_d is the gate-on level at note-off. The
// section is chosen first, then one x^alpha.
__device__ __forceinline__ float fm_adsr(ff t, const FmEnv& E, float level_d) {
  float base, scale;
  ff x, len;
  if (ff_lt(t, E.d)) {
    if (ff_lt(t, E.a)) {
      base = 0.f; scale = 1.f; x = t; len = E.a;
    } else {
      x = ff_sub(t, E.a);
      if (!ff_lt(x, E.dc)) return E.s;
      base = 1.f; scale = -(1.f - E.s); len = E.dc;
    }
  } else {
    x = ff_sub(t, E.d);
    if (!ff_lt(x, E.r)) return 0.f;
    base = level_d; scale = -level_d; len = E.r;
  }
  return fmaf(scale, fm_pow(x, len, E.alpha), base);
}

// Operator i's envelope constants from its normalized parameters uo (ratio,
// level, attack, decay, sustain, release, alpha) and the duration parameter
// ud: attack and decay 2 u^2, release 5 u^2 (u^2 exact as a float-float
// product), duration 4 u, sustain u; alpha = 0.1 + 5.9 u^2 as in the
// parameter map.
__device__ __forceinline__ FmEnv fm_env(const float* uo, float ud) {
  FmEnv E;
  E.a = ff_mul_f(two_prod(uo[2], uo[2]), 2.f);
  E.dc = ff_mul_f(two_prod(uo[3], uo[3]), 2.f);
  E.r = ff_mul_f(two_prod(uo[5], uo[5]), 5.f);
  E.d = ff_make(4.f * ud);
  E.s = uo[4];
  E.alpha = fmaf(6.f - 0.1f, uo[6] * uo[6], 0.1f);
  return E;
}

struct __align__(16) FmSmem {
  float u[32];
  unsigned long long inc[4];
  FmEnv env[4];
  float level_d[4];  // gate-on levels at note-off
  float scale[4];    // the carrier's level; a modulator's level in cycles
};

// sin(2 pi t) of two values, |t| < 2^20: with k = rint(2 t) and r = t - k / 2,
// |r| <= 1/4, it is sin(2 pi r) times -1 to the power k. rint by adding and
// taking away 1.5 2^23, which leaves k's parity in the sum's last bit. The odd
// polynomial of r is a minimax fit of sin(2 pi r) / r in r^2 (weighted least
// squares, the weights raised where the error is largest; relative error
// 5.3e-9). In FP32 its error is at most 1.6e-7, 3.6e-8 in the mean square,
// below the rounding of its argument (|t| up to 1.8 cycles: 3.7e-7 rad).
__device__ __forceinline__ f32x2 sin2pi2(f32x2 t) {
  const float magic = 12582912.f;
  const f32x2 m = fma2(t, both2(2.f), both2(magic));
  const f32x2 r = fma2(add2(m, both2(-magic)), both2(-0.5f), t);
  const f32x2 z = mul2(r, r);
  f32x2 p = fma2(z, both2(39.7109784977881f), both2(-76.57500087327254f));
  p = fma2(z, p, both2(81.6022316631156f));
  p = fma2(z, p, both2(-41.34167748601398f));
  p = fma2(z, p, both2(6.283185273828892f));
  float s0, s1, m0, m1;
  unpack2(mul2(r, p), s0, s1);
  unpack2(m, m0, m1);
  return pack2(__uint_as_float(__float_as_uint(s0) ^ (__float_as_uint(m0) << 31)),
               __uint_as_float(__float_as_uint(s1) ^ (__float_as_uint(m1) << 31)));
}

__global__ void __launch_bounds__(kFmThreads, kFmCtasPerSm) fm_render_kernel(const __grid_constant__ FmConst fc,
                                                               uint64_t seed,
                                                               uint64_t batch_index, int batch,
                                                               const float* __restrict__ params_in,
                                                               float* __restrict__ audio,
                                                               float* __restrict__ params_out) {
  __shared__ FmSmem S;
  // per control point the chunk spans: the four envelopes, the first sample
  // of its interval (chunk-relative) and that sample's fraction
  extern __shared__ __align__(16) float fm_dyn[];
  const int max_pts = fc.max_pts;
  float* env = fm_dyn;                                         // [4][max_pts]
  int* sst = reinterpret_cast<int*>(fm_dyn + 4 * max_pts);     // [max_pts]
  float* fr0 = fm_dyn + 5 * max_pts;                           // [max_pts]
  const int tid = threadIdx.x;
  const int v = blockIdx.y;
  const uint64_t g = batch_index * (uint64_t)batch + (uint64_t)v;
  const int64_t s0 = (int64_t)blockIdx.x * fc.chunk;
  const int64_t N = fc.N;
  const int64_t s1 = min(s0 + (int64_t)fc.chunk, N);
  // ---- parameters
  if (params_in == nullptr) {
    if (tid < 8) {
      const uint4 r = philox4x32_10(
          make_uint4((uint32_t)g, (uint32_t)(g >> 32), (uint32_t)tid, kStreamFmParam),
          make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
      S.u[4 * tid + 0] = u01f(r.x);
      S.u[4 * tid + 1] = u01f(r.y);
      S.u[4 * tid + 2] = u01f(r.z);
      S.u[4 * tid + 3] = u01f(r.w);
    }
  } else if (tid < kNumFmParams) {
    S.u[tid] = fminf(fmaxf(params_in[(size_t)v * kNumFmParams + tid], 0.f), 1.f);
  }
  __syncthreads();
  if (tid < kNumFmParams) {
    const float u = S.u[tid];
    if (blockIdx.x == 0 && params_out) params_out[(size_t)v * kNumFmParams + tid] = u;
    float lo, hi;
    int c;
    fm_range(tid, lo, hi, c);
    const int i = (tid - 2) / 7;
    if (tid == 3 + 7 * i)
      S.scale[i] = fmaf(hi - lo, c == 2 ? u * u : u, lo) * (i == 0 ? 1.f : 0.15915494309189535f);
  }
  if (tid < 4) {
    // the operator's increment in cycles per sample, f0 ratio / SR with
    // f0 = 440 2^((m - 69)/12), in float-float (relative error ~1e-14), then
    // its fraction as 64-bit fixed point: phase(n) = n inc mod 2^64 exactly
    const float ur = S.u[2 + 7 * tid];
    const ff m = ff_mul_f(ff_make(127.f), S.u[0]);
    const ff ratio = ff_add_f(ff_mul_f(ff_mul_f(ff_make(ur), ur), 7.5f), 0.5f);
    S.inc[tid] = ff_to_fix64(ff_mul(inc_at_ff(m, fc.log2_440_over_sr, fc.T), ratio));
  } else if (tid >= 32 && tid < 36) {
    const int i = tid - 32;
    const FmEnv E = fm_env(S.u + 2 + 7 * i, S.u[1]);
    S.env[i] = E;
    S.level_d[i] = fm_gate_on(E.d, E);
  }
  __syncthreads();
  // ---- envelopes at the control points the chunk spans
  const int64_t k_lo = s0 * fc.rate_b / fc.rate_a;
  const int64_t k_hi = (s1 - 1) * fc.rate_b / fc.rate_a + 1;
  const int npts = (int)(k_hi - k_lo + 1);
  for (int e = tid; e < 4 * npts; e += kFmThreads) {  // (operator, point) pairs
    const int i = e / npts, j = e - i * npts;
    const ff t = ff_mul_f(fc.inv_cr, (float)(k_lo + j));  // k < 2^24: exact in a float
    env[i * max_pts + j] = S.scale[i] * fm_adsr(t, S.env[i], S.level_d[i]);
  }
  for (int j = tid; j < npts; j += kFmThreads) {
    const int64_t k = k_lo + j;
    const int64_t sk = (k * fc.rate_a + fc.rate_b - 1) / fc.rate_b;
    sst[j] = (int)(sk - s0);
    fr0[j] = (float)(sk * fc.rate_b - k * fc.rate_a) / (float)fc.rate_a;
  }
  __syncthreads();
  // ---- audio
  const float invR = (float)fc.rate_b / (float)fc.rate_a;
  const int n_c = (int)(s1 - s0);
  float* out = audio + (size_t)v * (size_t)N + (size_t)s0;
  const bool vec = (N & 3) == 0 && (reinterpret_cast<uintptr_t>(audio) & 15) == 0;
  for (int q = tid; 4 * q < n_c; q += kFmThreads) {
    const int r0 = 4 * q;
    int j = min((int)((float)r0 * invR), npts - 2);
    while (j + 1 < npts - 1 && sst[j + 1] <= r0) ++j;
    while (j > 0 && sst[j] > r0) --j;
    const uint32_t n0 = (uint32_t)(s0 + r0);  // N < 2^31
    // the four samples' places in interval j, and in j + 1 for those past its start
    const float d0 = (float)(r0 - sst[j]), f0 = fr0[j];
    const f32x2 fu0 = fma2(pack2(d0, d0 + 1.f), both2(invR), both2(f0));
    const f32x2 fu1 = fma2(pack2(d0 + 2.f, d0 + 3.f), both2(invR), both2(f0));
    const int nb = j + 1 < npts - 1 ? sst[j + 1] - r0 : 4;  // samples in interval j
    f32x2 y0 = 0, y1 = 0;  // the operator above, in cycles
#pragma unroll
    for (int op = 3; op >= 0; --op) {
      // the quad's first phase, one 64-bit product; its top 32 bits as a signed
      // fraction of a cycle, exact to 2^-26, and the next samples' by sums of
      // the increment's top bits (an error of 3 2^-32 at most)
      const unsigned long long inc = S.inc[op];
      const uint32_t ph = (uint32_t)((n0 * inc) >> 32), step = (uint32_t)(inc >> 32);
      const f32x2 t0 = fma2(pack2((float)(int)ph, (float)(int)(ph + step)), both2(0x1p-32f), y0);
      const f32x2 t1 = fma2(pack2((float)(int)(ph + 2 * step), (float)(int)(ph + 3 * step)),
                            both2(0x1p-32f), y1);
      const float* en = env + op * max_pts + j;
      const float ea = en[0], eb = en[1];
      const f32x2 da = both2(eb - ea);
      f32x2 e0 = fma2(fu0, da, both2(ea)), e1 = fma2(fu1, da, both2(ea));
      if (nb < 4) {
        const float db = en[2] - eb, fb = fr0[j + 1];
        float e[4];
        unpack2(e0, e[0], e[1]);
        unpack2(e1, e[2], e[3]);
#pragma unroll
        for (int i = 1; i < 4; ++i)
          if (i >= nb) e[i] = fmaf(fmaf((float)(i - nb), invR, fb), db, eb);
        e0 = pack2(e[0], e[1]);
        e1 = pack2(e[2], e[3]);
      }
      y0 = mul2(e0, sin2pi2(t0));
      y1 = mul2(e1, sin2pi2(t1));
    }
    float o4[4];
    unpack2(y0, o4[0], o4[1]);
    unpack2(y1, o4[2], o4[3]);
    if (vec && r0 + 3 < n_c) {
      __stcs(reinterpret_cast<float4*>(out + r0), make_float4(o4[0], o4[1], o4[2], o4[3]));
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (r0 + i < n_c) out[r0 + i] = o4[i];
    }
  }
}

// Samples per CTA of a launch: the cut of a voice that costs least, where a round
// of resident CTAs first spends what kFmSetup samples cost on parameters and
// envelopes (2.2 us), and a last round of fewer CTAs an SM takes the share of a
// full one's time that kFmShare gives (the audio loop is bound by issue; fitted to
// the times below); at equal cost the finer cut. 8192 samples for every launch
// left the last round of CTAs part empty. 128 voices of 4 s: 71.8 -> 65.6 us (12600
// samples; 9288: 69.7, 19600: 67.6, 4096: 79.5), 40: 28.6 -> 24.7, 16: 16.4 -> 13.0
// (4644), one 10.3 -> 9.2; 128 of 1 s 26.3 -> 22.6, 100 of 2.3 s 38.0 -> 32.9. The
// cuts meet the same samples: bit for bit as before.
constexpr int kFmSetup = 1400;
constexpr int kFmShare[kFmCtasPerSm] = {0, 40, 60, 82};  // percent
constexpr int kFmDefaultChunk = 8192, kFmMaxChunk = 20480;
constexpr int kFmMaxPoints = 1900;  // control points whose shared memory lets kFmCtasPerSm CTAs on an SM
int fm_chunk(const VoiceConst& vc, int batch, int sms) {
  const int64_t n = vc.n_samples;
  const int64_t by_points = (int64_t)kFmMaxPoints * vc.rate_a / vc.rate_b;
  if (by_points < kFmDefaultChunk) return kFmDefaultChunk;
  const int64_t cap = std::min<int64_t>(kFmMaxChunk, by_points);
  const int64_t first = (n + cap - 1) / cap;
  int64_t best = 0, chunk = kFmDefaultChunk;
  // CTAs a voice: 32 cuts at most, none below 1024 samples but the first (a launch
  // of short voices takes as long as the call)
  const int64_t last = std::max(first, std::min(first + 31, n / 1024));
  for (int64_t c = first; c <= last; ++c) {
    const int64_t len = (((n + c - 1) / c) + 3) / 4 * 4;
    if (len > cap) continue;
    const int64_t per_sm = ((n + len - 1) / len * batch + sms - 1) / sms;
    const int64_t full = per_sm / kFmCtasPerSm, rest = per_sm % kFmCtasPerSm;
    const int64_t cost = len * full + len * kFmShare[rest] / 100 + (full + (rest > 0)) * kFmSetup;
    if (best == 0 || cost <= best) { best = cost; chunk = len; }
  }
  return (int)chunk;
}

}  // namespace

cudaError_t launch_fm_render(const VoiceConst& vc, uint64_t seed, uint64_t batch_index, int batch,
                             const float* params_in, float* audio, float* params_out,
                             cudaStream_t stream) {
  if (batch <= 0) return cudaSuccess;
  if (batch > 65535) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  FmConst fc;
  fc.N = vc.n_samples;
  fc.rate_a = vc.rate_a;
  fc.rate_b = vc.rate_b;
  fc.inv_cr = ff_from_double(1.0 / vc.control_rate);
  fc.log2_440_over_sr = vc.log2_440_over_sr;
  fc.T = vc.T;
  fc.chunk = fm_chunk(vc, batch, sms);
  fc.max_pts = (int)((int64_t)fc.chunk * vc.rate_b / vc.rate_a) + 3;
  const size_t smem = sizeof(float) * 6 * (size_t)fc.max_pts;
  if (smem > 200 * 1024) return cudaErrorInvalidValue;
  if (smem > 48 * 1024) {
    e = cudaFuncSetAttribute(fm_render_kernel,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
    if (e != cudaSuccess) return e;
  }
  const dim3 grid((unsigned)((vc.n_samples + fc.chunk - 1) / fc.chunk), (unsigned)batch);
  fm_render_kernel<<<grid, kFmThreads, smem, stream>>>(fc, seed, batch_index, batch, params_in,
                                                       audio, params_out);
  return cudaGetLastError();
}

}  // namespace synth
