// render_backward.cu -- adjoint of the Voice render: grad_u = (d audio / d u)^T
// grad_audio for the 78 normalized parameters of every voice.
//
// "Stress-tested differentiable modules" are future work in the paper
// (Sec. 7); this is the reverse-mode derivative of the library's own render.
// Where the forward takes a branch (envelope section, clamp, Nyquist cap,
// square LFO) the derivative is that of the branch taken.
//
// Three kernels (all on the caller's stream, buffers in the caller's workspace):
//  1. bwd_recompute: the forward control rate, one CTA per voice, in the fused
//     render's arithmetic (float-float chain, fixed-point phase sums); its
//     per-interval phase descriptions are the checkpoints from which the
//     audio-rate values are rebuilt;
//  2. bwd_samples: audio-rate reverse pass, eight lanes per control interval:
//     rebuilds every sample, forms d/d(phase) of both VCOs, the amplitude,
//     drive, shape and mixer-gain partials, and the interval's moments for the
//     reverse phase scan;
//  3. bwd_control, one CTA per voice: the reverse scan over intervals (FP64):
//     with C_k = sum of d/d(phase) over all samples from interval k on, the
//     pitch adjoint of control point k is
//     (ln 2 / 12) (M1_k + F1_k C_{k+1} + M2_{k-1} + F2_{k-1} C_k); then the
//     control-rate reverse sweep: modulation mixer, LFOs (with a reverse scan of
//     the LFO phase adjoint), ADSRs, range map -> d/du.
//
// What bounds it: at 64 voices of 1 s the 11 MB of audio gradient take 2 us; the
// per-voice kernels are latency on 64 of 152 SMs, the sample pass is
// instruction issue. So a step goes over the (envelope, point), (LFO, point) or
// (VCO, interval) pairs of a voice and not over points alone, phase sums are
// integers (an FP64 scan waits on the narrow FP64 pipe), and an interval's 21
// sums are added up over 8 lanes, not 32. Kernels of the plain form's modules,
// a warp per interval and a scan kernel that handed FP64 point adjoints on took
// 110.6 us; now 78.0 us.
//
// Precision: every value that goes from one kernel to the next is rounded to float
// once, from float-float (parameters, envelopes, mixer gains and outputs, phases)
// or FP64 (a point's pitch adjoint, whose two ends and running sums cancel).
// Mixer outputs as FP32 sums and pitch adjoints rounded before they were added
// took 76.6 us, and their error against 64 bits was up to 1.7 times that of the
// modules' kernels over a batch (10 times for a voice); now it is theirs, 7.6e-6
// over 1280 voices of 0.1 s and 8.2e-6 over 872 of 0.1 to 2 s.

#include "control_ff.cuh"
#include "internal.h"

namespace synth {

namespace {

constexpr int kStat = 21;  // per-interval partial sums written by bwd_samples
// stat layout: [0..4] sine T, M1, F1, M2, F2; [5..9] square-saw T, M1, F1, M2, F2;
// [10..12] amp grads to the left point (sine, sq, noise); [13..15] to the right
// point; [16] d/d kappa; [17..19] mixer gains g0, g1, g2; [20] d/d shape.

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

struct AdjBuffers {
  float* y;       // [B][80] human-range parameters (78 used)
  float* mix;     // [B][4] mixer gains (3), square-saw shape
  float* env;     // [B][6][P] ADSRs at the control points
  float* phase;   // [B][2][P] LFO phases (cycles, wrapped)
  float* dest;    // [B][5][P] modulation mixer outputs
  SegVco* seg;    // [B][2][K] VCO interval descriptions
  float* kappa;   // [B][2][K] square-saw drive and 1/tanh(drive)
  float* stat;    // [B][K][kStat]
  double2* csum;  // [B][K] both VCOs' sums of d/d(phase) over all later intervals
  float* dtheta;  // [B][2][P]
  float* denv;    // [B][6][P]
  size_t total;
};

AdjBuffers adj_carve(const VoiceConst& vc, int batch, void* ws) {
  const size_t B = (size_t)batch, P = (size_t)vc.K + 1, K = (size_t)vc.K;
  char* base = static_cast<char*>(ws);
  size_t o = 0;
  auto take = [&](size_t bytes) { char* at = base ? base + o : nullptr; o += al256(bytes); return at; };
  AdjBuffers b;
  b.y = reinterpret_cast<float*>(take(sizeof(float) * B * 80));
  b.mix = reinterpret_cast<float*>(take(sizeof(float) * B * 4));
  b.env = reinterpret_cast<float*>(take(sizeof(float) * B * 6 * P));
  b.phase = reinterpret_cast<float*>(take(sizeof(float) * B * 2 * P));
  b.dest = reinterpret_cast<float*>(take(sizeof(float) * B * 5 * P));
  b.seg = reinterpret_cast<SegVco*>(take(sizeof(SegVco) * B * 2 * K));
  b.kappa = reinterpret_cast<float*>(take(sizeof(float) * B * 2 * K));
  b.stat = reinterpret_cast<float*>(take(sizeof(float) * B * K * kStat));
  b.csum = reinterpret_cast<double2*>(take(sizeof(double2) * B * K));
  b.dtheta = reinterpret_cast<float*>(take(sizeof(float) * B * 2 * P));
  b.denv = reinterpret_cast<float*>(take(sizeof(float) * B * 6 * P));
  b.total = o;
  return b;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// 1. forward control rate of a voice, kCP control points (kCP - 1 intervals) at
// a time. Threads 0 .. kCP - 1 take the first LFO and VCO, the others the second.
// ---------------------------------------------------------------------------
constexpr int kCT = 1024;
constexpr int kCP = kCT / 2;
constexpr int kCW = kCP / 32;  // warps of a half

struct RecomputeSmem {
  FFTables T;
  VoiceFF V;
  ff y[kNumParams];
  // the six envelopes; an LFO's output then takes the place of its amplitude
  // envelope (3, 5), a VCO's pitch that of an LFO's rate envelope (2, 4)
  ff env[6][kCP];
  unsigned long long p0[4];  // initial phases: LFOs, VCOs
  unsigned long long warp_tot[2][kCW];
};

// Exclusive sum over each half of the block; tot: the half's whole sum.
__device__ __forceinline__ unsigned long long half_scan(RecomputeSmem& s, unsigned long long x,
                                                        unsigned long long& tot) {
  const int lane = threadIdx.x & 31, half = threadIdx.x / kCP, warp = (threadIdx.x % kCP) >> 5;
  unsigned long long in = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long n = __shfl_up_sync(0xffffffffu, in, o);
    if (lane >= o) in += n;
  }
  __syncthreads();  // the earlier scan's totals are read
  if (lane == 31) s.warp_tot[half][warp] = in;
  __syncthreads();
  unsigned long long before = 0;
  tot = 0;
#pragma unroll
  for (int w = 0; w < kCW; ++w) {
    const unsigned long long t = s.warp_tot[half][w];
    if (w < warp) before += t;
    tot += t;
  }
  return before + in - x;
}

__global__ void __launch_bounds__(kCT) bwd_recompute(const __grid_constant__ VoiceConst vc, int batch,
                                                     const float* __restrict__ params,
                                                     const AdjBuffers b, ScratchHeader* hdr) {
  __shared__ RecomputeSmem s;
  const int v = blockIdx.x, tid = threadIdx.x, half = tid / kCP, p = tid % kCP;
  const int K = vc.K, P = K + 1;
  // every buffer below is addressed at voice v of this batch
  if (!in_bounds(hdr, v, batch)) return;
  const VoiceFF& V = s.V;
  load_tables(s.T, vc.T);
  __syncthreads();
  if (tid < kNumParams) {
    const float u = fminf(fmaxf(params[(size_t)v * kNumParams + tid], 0.f), 1.f);
    s.y[tid] = range_map_ff(u, vc.map_base[tid], vc.map_scale[tid], vc.map_curve[tid],
                            vc.map_code[tid], vc.sym[tid], s.T);
    b.y[(size_t)v * 80 + tid] = ff_to_float(s.y[tid]);
  }
  __syncthreads();
  if (tid < 16) {
    voice_ff_fill(s.V, s.y, tid);
  } else if (tid == 32) {
    const ff sum = ff_add(ff_add(s.y[kMix], s.y[kMix + 1]), s.y[kMix + 2]);
    const ff inv = ff_lt(sum, ff_make(1.f)) ? ff_make(1.f) : ff_rcp(sum);
    float g[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) g[c] = ff_to_float(ff_mul(s.y[kMix + c], inv));
    *reinterpret_cast<float4*>(b.mix + (size_t)v * 4) =
        make_float4(g[0], g[1], g[2], ff_to_float(s.y[kSqr + 3]));
  } else if (tid >= 64 && tid < 68) {
    const int slot[4] = {kLfo + 2, kLfo + 8 + 2, kSine + 2, kSqr + 2};
    s.p0[tid - 64] = ff_to_fix64(ff_mul(s.y[slot[tid - 64]], vc.inv_2pi));
  }
  __syncthreads();
  if (tid < 6) s.V.level_d[tid] = gate_level_ff(tid, V, s.T);
  __syncthreads();
  unsigned long long lfo_carry = s.p0[half], vco_carry = s.p0[2 + half];
  for (int base = 0; base < K; base += kCP - 1) {
    const int nseg = min(kCP - 1, K - base);  // points base .. base + nseg
    for (int i = tid; i < 6 * kCP; i += kCT) {
      const int a = i / kCP, k = i % kCP;
      if (k > nseg || !in_bounds(hdr, base + k, P)) continue;
      const ff e = adsr_ff(ff_mul_f(vc.inv_cr, (float)(base + k)), a, V, s.T);
      s.env[a][k] = e;
      b.env[((size_t)v * 6 + a) * P + base + k] = ff_to_float(e);
    }
    __syncthreads();
    unsigned long long inc = 0, tot;
    if (p < nseg) {
      const ff rate = ff_min(ff_max(ff_add(V.lfo_freq[half], ff_mul(V.lfo_depth[half], s.env[2 + 2 * half][p])),
                                    ff_make(0.f)),
                             ff_make((float)kLfoMaxHz));
      inc = ff_to_fix64(ff_mul(rate, vc.inv_cr));
    }
    const unsigned long long theta = lfo_carry + half_scan(s, inc, tot);
    lfo_carry += tot;
    if (p <= nseg) {
      const ff th = fix64_to_ff(theta);
      b.phase[((size_t)v * 2 + half) * P + base + p] = ff_to_float(th);
      s.env[3 + 2 * half][p] = lfo_ff(th, half, s.env[3 + 2 * half][p], V, s.T);
    }
    __syncthreads();
    if (p <= nseg) {
      const ff src[4] = {s.env[0][p], s.env[1][p], s.env[3][p], s.env[5][p]};
      // the mixer's outputs, two or three a half (the pitch one, then amplitudes): sums
      // in float-float, rounded once
#pragma unroll 1
      for (int j = 2 * half; j < 2 + 3 * half; ++j) {
        ff acc = ff_mul(V.mod_w[0][j], src[0]);
#pragma unroll
        for (int q = 1; q < 4; ++q) acc = ff_add(acc, ff_mul(V.mod_w[q][j], src[q]));
        acc = ff_mul(acc, V.inv_norm[j]);
        b.dest[((size_t)v * 5 + j) * P + base + p] = ff_to_float(acc);
        if (j == 2 * half) s.env[j + 2][p] = ff_add(V.pitch_base[half], ff_mul(V.depth[half], acc));
      }
    }
    __syncthreads();
    ff adv = ff_make(0.f);
    SegVco sv;
    if (p < nseg) {
      const int k = base + p;
      const int64_t rem = vc.n_samples - (int64_t)k * vc.R;
      const int Rk = rem < vc.R ? (int)rem : vc.R;
      float inc_first;
      adv = vco_interval_ff(s.env[2 + 2 * half][p], s.env[2 + 2 * half][p + 1], (float)vc.R, Rk,
                            vc.inv_R, vc.ln2_12R, vc.m_nyq_ff, vc.log2_440_over_sr, s.T, &sv,
                            &inc_first);
      if (half == 1) {  // drive 1 + SR / (8 f) at the (capped) frequency of the interval start
        const float kap = fminf((float)kBrightnessMax, 1.f + 0.125f / inc_first);
        b.kappa[((size_t)v * 2 + 0) * K + k] = kap;
        b.kappa[((size_t)v * 2 + 1) * K + k] = 1.f / tanhf(kap);
      }
    }
    const unsigned long long start =
        vco_carry + half_scan(s, p < nseg ? ff_to_fix64(adv) : 0ull, tot);
    vco_carry += tot;
    if (p < nseg && in_bounds(hdr, base + p, K)) {
      // from 48 bits: a phase cut to 32 bits first rounds the other way in 1% of the intervals,
      // which a steep square-saw shows
      sv.phase0 = ff_to_float(fix64_to_ff(start));
      b.seg[((size_t)v * 2 + half) * K + base + p] = sv;
    }
    __syncthreads();  // the chunk's envelopes are done with
  }
}

// ---------------------------------------------------------------------------
// 2. audio-rate reverse pass. Eight lanes take a control interval (R <= 128), lane
// l its samples 16 l .. 16 l + 15, from the last to the first, so that the sum of
// d/d(phase) over later samples is at hand: over the lane's own it runs along,
// over the later lanes' it enters the moments afterwards (they are linear in it).
// Six blocks an SM (80 registers): issue is at half its rate with five, waiting
// for the sine unit; 79.3 -> 77.3 us. With eight the accumulators spill: 79.7.
// ---------------------------------------------------------------------------
constexpr int kST = 128;
constexpr int kSI = kST / 8;  // intervals per block

// Phases (cycles) and increments of samples j0 .. j0 + 3; the increment of a
// sample whose pitch is capped at Nyquist as 0 (it does not move with the pitch).
__device__ __forceinline__ void vco_quad_and_inc(const SegVco& s, int j0, float ph[4], float inc[4]) {
  vco_quad(s, j0, ph);
  const int jc = s.jc_flags & 0xffff;
  if (j0 + 3 < jc || j0 >= jc) {  // inside one piece: the increments are geometric
    const bool in_b = j0 >= jc;
    const float c = in_b ? s.cB : s.cA;
    const bool lin = (s.jc_flags >> (in_b ? 17 : 16)) & 1;
    const bool cap = (s.jc_flags >> (in_b ? 19 : 18)) & 1;
    const float x = lin ? 0.f : s.x;
    const float e1 = expm1_phase(x);  // q2 - 2 has lost its last bits
    inc[0] = cap ? 0.f : fmaf(c, expm1_phase((float)(j0 - (in_b ? jc : 0)) * x), c);
    inc[1] = fmaf(inc[0], e1, inc[0]);
    inc[2] = fmaf(inc[1], e1, inc[1]);
    inc[3] = fmaf(inc[2], e1, inc[2]);
  } else {
    bool cap[4];
    vco_inc_quad(s, j0, inc, cap);
#pragma unroll
    for (int i = 0; i < 4; ++i) inc[i] = cap[i] ? 0.f : inc[i];
  }
}

__global__ void __launch_bounds__(kST, 6) bwd_samples(const __grid_constant__ VoiceConst vc,
                                                      uint64_t seed, uint64_t batch_index, int batch,
                                                      const float* __restrict__ grad_audio,
                                                      const AdjBuffers b, ScratchHeader* hdr) {
  const int lane = threadIdx.x & 31, l8 = lane & 7;
  const int v = blockIdx.y;
  const int K = vc.K, P = K + 1, R = vc.R;
  const int ki = blockIdx.x * kSI + (threadIdx.x >> 3);
  if (ki - (lane >> 3) >= K) return;  // the warp's first interval is past the end
  const bool valid = ki < K;
  const int k = valid ? ki : K - 1;
  // the interval's control points k and k + 1, its descriptions and its row
  // of statistics belong to voice v of this batch
  if (!in_bounds(hdr, v, batch) || !in_bounds(hdr, k + 1, P)) return;
  const int64_t N = vc.n_samples;
  const float4 mx = *reinterpret_cast<const float4*>(b.mix + (size_t)v * 4);
  const float sigma = mx.w, ip = 1.f / (1.f + sigma);
  const float* d1 = b.dest + ((size_t)v * 5 + 1) * P + k;
  const float a0[3] = {d1[0], d1[2 * P], d1[3 * P]};  // destinations 1, 3, 4
  const float da[3] = {d1[1] - a0[0], d1[2 * P + 1] - a0[1], d1[3 * P + 1] - a0[2]};
  const SegVco& s0 = b.seg[((size_t)v * 2 + 0) * K + k];
  const SegVco& s1 = b.seg[((size_t)v * 2 + 1) * K + k];
  const float kap = b.kappa[((size_t)v * 2 + 0) * K + k];
  const float itk = b.kappa[((size_t)v * 2 + 1) * K + k];
  const int64_t n_first = (int64_t)k * R;
  const int Rk = valid ? (int)min((int64_t)R, N - n_first) : 0;
  const float invR = 1.f / (float)R;
  const uint64_t gv = batch_index * (uint64_t)batch + (uint64_t)v;
  const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
  const float* ga = grad_audio + (size_t)v * N + n_first;
  const bool vec = (N & 3) == 0 && (reinterpret_cast<uintptr_t>(grad_audio) & 15) == 0;

  float acc[24];
#pragma unroll
  for (int i = 0; i < 24; ++i) acc[i] = 0.f;
  float ls[2] = {0.f, 0.f};  // sum of d/d(phase) over the lane's later samples
#pragma unroll 1
  for (int i = 3; i >= 0; --i) {
    const int j0 = 4 * (4 * l8 + i);
    if (j0 >= Rk) continue;
    float ps[4], pq[4], inc[2][4], go4[4];
    vco_quad_and_inc(s0, j0, ps, inc[0]);
    vco_quad_and_inc(s1, j0, pq, inc[1]);
    const uint4 nz = philox4x32_10(make_uint4((uint32_t)gv, (uint32_t)(gv >> 32),
                                              (uint32_t)((n_first + j0) >> 2), kStreamNoise),
                                   key);
    const uint32_t nw[4] = {nz.x, nz.y, nz.z, nz.w};
    if (vec && j0 + 3 < Rk && in_bounds(hdr, (long long)v * N + n_first + j0 + 3, (long long)batch * N)) {
      const float4 t = __ldg(reinterpret_cast<const float4*>(ga + j0));
      go4[0] = t.x; go4[1] = t.y; go4[2] = t.z; go4[3] = t.w;
    } else {
#pragma unroll
      for (int t = 0; t < 4; ++t)
        go4[t] = j0 + t < Rk && in_bounds(hdr, (long long)v * N + n_first + j0 + t, (long long)batch * N)
                     ? ga[j0 + t]
                     : 0.f;
    }
#pragma unroll
    for (int t = 3; t >= 0; --t) {
      const bool on = j0 + t < Rk;
      const float go = go4[t];
      const float fj = (float)(j0 + t) * invR, fl = 1.f - fj;
      float A[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) A[c] = fmaf(fj, da[c], a0[c]);
      // SFU sine, cosine and tanh, as in the forward render
      float xs, xc, sn, cs;
      __sincosf(kTwoPiF * ps[t], &xs, &xc);
      __sincosf(kTwoPiF * pq[t], &sn, &cs);
      const float th = tanh_from_y(kTwoLog2e * kap * sn);
      const float shp = fmaf(sigma, cs, 1.f);
      const float x[3] = {xs, th * itk * shp * ip, fmaf(2.f, u01f(nw[t]), -1.f)};
      const float gg[3] = {go * mx.x, go * mx.y, go * mx.z};
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float dA = gg[c] * x[c];
        acc[10 + c] = fmaf(dA, fl, acc[10 + c]);
        acc[13 + c] = fmaf(dA, fj, acc[13 + c]);
        acc[17 + c] = fmaf(go * A[c], x[c], acc[17 + c]);
      }
      const float sech2 = 1.f - th * th;
      const float gA1 = gg[1] * A[1] * ip;
      const float dphi[2] = {gg[0] * A[0] * kTwoPiF * xc,
                             gA1 * kTwoPiF * itk * (kap * cs * sech2 * shp - th * sigma * sn)};
      // d xq / d kappa with d(1/tanh k)/dk = 1 - (1/tanh k)^2
      acc[16] = fmaf(gA1 * shp, sn * sech2 * itk + th * (1.f - itk * itk), acc[16]);
      acc[20] = fmaf(gA1 * ip * th * itk, cs - 1.f, acc[20]);
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        const float w = on ? inc[o][t] : 0.f, wr = w * fj, wl = w * fl;
        acc[5 * o + 1] = fmaf(wl, ls[o], acc[5 * o + 1]);
        acc[5 * o + 2] += wl;
        acc[5 * o + 3] = fmaf(wr, ls[o], acc[5 * o + 3]);
        acc[5 * o + 4] += wr;
        ls[o] += dphi[o];
      }
    }
  }
  // the later lanes' samples: their sum enters M1 and M2 times F1 and F2
#pragma unroll
  for (int o = 0; o < 2; ++o) {
    float suf = ls[o];  // inclusive over lanes >= l8 of the interval
#pragma unroll
    for (int d = 1; d < 8; d <<= 1) {
      const float t = __shfl_down_sync(0xffffffffu, suf, d, 8);
      if (l8 + d < 8) suf += t;
    }
    float after = __shfl_down_sync(0xffffffffu, suf, 1, 8);
    if (l8 == 7) after = 0.f;
    acc[5 * o + 0] = ls[o];
    acc[5 * o + 1] = fmaf(after, acc[5 * o + 2], acc[5 * o + 1]);
    acc[5 * o + 3] = fmaf(after, acc[5 * o + 4], acc[5 * o + 3]);
  }
  // butterfly reduce-scatter of the 21 (of 24) sums over the 8 lanes: at each step a
  // lane keeps half of its slots and adds its partner's copy of that half; in
  // the end lane l holds the totals of sums 3 l .. 3 l + 2
  static_assert(kStat <= 24, "three sums per lane");
#pragma unroll
  for (int sh = 4, n = 12; sh >= 1; sh >>= 1, n >>= 1) {
    const bool up = (lane & sh) != 0;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float send = up ? acc[i] : acc[i + n];
      const float keep = up ? acc[i + n] : acc[i];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, sh);
    }
  }
  if (valid && l8 < kStat / 3) {
    float* st = b.stat + ((size_t)v * K + k) * kStat + 3 * l8;
#pragma unroll
    for (int i = 0; i < 3; ++i) st[i] = acc[i];
  }
}

// ---------------------------------------------------------------------------
// 3. reverse scan over intervals (FP64) and control-rate reverse sweep, one block
// per voice; the sweep in FP32: a gradient needs a relative accuracy of about
// 1e-3, not the forward's float-float (the forward values it differentiates at
// are recomputed in float-float and rounded to float).
// ---------------------------------------------------------------------------
constexpr int kGY = 80;  // slots of the per-voice human-range gradient d/dy (78 used)
constexpr int kBC = 512;  // threads of the control-rate reverse sweep (one block per voice)

// x^a for x >= 0 and its partials (0 at x <= 0, as the forward's convention).
__device__ __forceinline__ void pow_d(float x, float a, float& p, float& dpx, float& dpa) {
  if (x <= 0.f) { p = 0.f; dpx = 0.f; dpa = 0.f; return; }
  const float lx = logf(x);
  p = expf(a * lx);
  dpx = a * p / x;
  dpa = p * lx;
}

// Gate-on level g(t) and its partials wrt (t, a, dc, s, alpha).
__device__ void gate_on_d(float t, const float* q, float& val, float d[5]) {
  const float a = q[0], dc = q[1], s = q[2], al = q[4];
  for (int i = 0; i < 5; ++i) d[i] = 0.f;
  if (t < a) {
    float p, px, pa;
    pow_d(t / a, al, p, px, pa);
    val = p;
    d[0] = px / a;             // d/dt
    d[1] = -px * t / (a * a);  // d/da
    d[4] = pa;                 // d/dalpha
  } else if (t < a + dc) {
    float p, px, pa;
    const float x = (t - a) / dc;
    pow_d(x, al, p, px, pa);
    val = 1.f - (1.f - s) * p;
    const float dx = -(1.f - s) * px;
    d[0] = dx / dc;
    d[1] = -dx / dc;
    d[2] = -dx * x / dc;
    d[3] = p;
    d[4] = -(1.f - s) * pa;
  } else {
    val = s;
    d[3] = 1.f;
  }
}

// Envelope (Sec. 3.1 reading) partials wrt (a, dc, s, r, alpha, d) at time t.
__device__ void adsr_d(float t, const float* q, float dur, float out[6]) {
  for (int i = 0; i < 6; ++i) out[i] = 0.f;
  float gd[5], val;
  if (t < dur) {
    gate_on_d(t, q, val, gd);
    out[0] = gd[1]; out[1] = gd[2]; out[2] = gd[3]; out[4] = gd[4];
    return;
  }
  const float r = q[3], al = q[4];
  const float tau = t - dur;
  if (!(tau < r)) return;
  gate_on_d(dur, q, val, gd);  // L = g(d)
  const float L = val;
  float p, px, pa;
  const float x = tau / r;
  pow_d(x, al, p, px, pa);
  const float dL = 1.f - p;           // d env / d L
  const float dx = -L * px;           // d env / d x
  out[0] = dL * gd[1];
  out[1] = dL * gd[2];
  out[2] = dL * gd[3];
  out[3] = -dx * x / r;
  out[4] = dL * gd[4] - L * pa;
  out[5] = dL * gd[0] - dx / r;       // via L = g(d) and tau = t - d
}

// Forward LFO shape mix and its derivative wrt the phase.
__device__ __forceinline__ void lfo_shapes(float p, float sh[5], float dsh[5]) {
  float sn, cs;
  sincospif(2.f * p, &sn, &cs);
  sh[0] = sn; dsh[0] = 6.28318530717958647692f * cs;
  sh[1] = 1.f - 4.f * fabsf(p - 0.5f); dsh[1] = (p - 0.5f) < 0.f ? 4.f : -4.f;
  sh[2] = 2.f * p - 1.f; dsh[2] = 2.f;
  sh[3] = 1.f - 2.f * p; dsh[3] = -2.f;
  sh[4] = p < 0.5f ? 1.f : -1.f; dsh[4] = 0.f;
}

// Adds a warp's values into its own row of the per-voice gradient (one row
// per warp, no atomics: the rows are summed in warp order at the end, so the
// gradient is the same on every run).
__device__ __forceinline__ void acc_y(float* gy_warp, int slot, float val) {
  const float w = warp_sum(val);
  if ((threadIdx.x & 31) == 0) gy_warp[slot] += w;
}

// Adds 32 values of each lane up over the warp and lane i's total of value i to
// the warp's row at slot(i): a butterfly reduce-scatter of 31 shuffles.
template <class Slot>
__device__ __forceinline__ void acc_y32(float* gy_warp, float (&r)[32], Slot slot) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int sh = 16; sh >= 1; sh >>= 1) {
    const bool up = (lane & sh) != 0;
#pragma unroll
    for (int i = 0; i < sh; ++i) {
      const float send = up ? r[i] : r[i + sh];
      const float keep = up ? r[i + sh] : r[i];
      r[i] = keep + __shfl_xor_sync(0xffffffffu, send, sh);
    }
  }
  gy_warp[slot(lane)] += r[0];
  __syncwarp();
}

// d y / d u of the range map for parameter p at u (FP32: the FP64 pipe is
// narrow on this GPU, and the gradient needs ~1e-6).
__device__ __forceinline__ float range_map_dydu(const VoiceConst& vc, int p, float u_raw) {
  const float u = fminf(fmaxf(u_raw, 0.f), 1.f);
  const float c = ff_to_float(vc.map_curve[p]);
  const float span = vc.sym[p] ? 2.f * ff_to_float(vc.map_scale[p]) : ff_to_float(vc.map_scale[p]);
  if (!vc.sym[p]) return u <= 0.f ? 0.f : span * c * powf(u, c - 1.f);
  const float s = fabsf(2.f * u - 1.f);
  return s <= 0.f ? 0.f : span * c * powf(s, c - 1.f);
}

__global__ void __launch_bounds__(kBC) bwd_control(const __grid_constant__ VoiceConst vc,
                                                   const AdjBuffers buf,
                                                   const float* __restrict__ u_in,
                                                   float* __restrict__ grad_params,
                                                   int batch, ScratchHeader* hdr) {
  __shared__ float gy[kGY];
  __shared__ float gyw_all[kBC / 32][kGY];  // per-warp partial gradients
  __shared__ float yv[kNumParams];
  __shared__ float warp_tot[2 * (kBC / 32)];
  __shared__ double warp_totd[2 * (kBC / 32)];
  __shared__ double red[4][kBC / 32];
  const int v = blockIdx.x;
  const int K = vc.K, P = K + 1;
  if (!in_bounds(hdr, v, batch)) return;
  const float inv_cr = (float)(1.0 / vc.control_rate);
  const float inv_2pi = 0.15915494309189533577f;
  const double l12 = kLn2 / 12.0;
  float* gyw = gyw_all[threadIdx.x >> 5];
  for (int i = threadIdx.x; i < kGY * (kBC / 32); i += kBC) (&gyw_all[0][0])[i] = 0.f;
  for (int i = threadIdx.x; i < kNumParams; i += kBC) yv[i] = buf.y[(size_t)v * 80 + i];
  const float* stat = buf.stat + (size_t)v * K * kStat;
  double2* csum = buf.csum + (size_t)v * K;
  // C_{idx+1}: sum of d/d(phase) over all later intervals; and the voice's sums
  // of the gain and shape partials
  double total0 = 0.0, total1 = 0.0;
  {
    double part[4] = {0.0, 0.0, 0.0, 0.0};  // dg0, dg1, dg2, dshape
    for (int base = 0; base < K; base += kBC) {
      const int idx = K - 1 - (base + (int)threadIdx.x);  // reversed order
      const bool ok = idx >= 0;
      const float* st = stat + (size_t)(ok ? idx : 0) * kStat;
      double e0 = ok ? (double)st[0] : 0.0, e1 = ok ? (double)st[5] : 0.0, t0, t1;
      if (ok)
        for (int c = 0; c < 4; ++c) part[c] += (double)st[17 + c];
      block_exclusive_scan2<double, kBC>(e0, e1, warp_totd, t0, t1);
      if (ok && in_bounds(hdr, idx, K)) csum[idx] = make_double2(total0 + e0, total1 + e1);
      total0 += t0;
      total1 += t1;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int c = 0; c < 4; ++c) {
      const double w = warp_sum_d(part[c]);
      if (lane == 0) red[c][warp] = w;
    }
  }
  __syncthreads();
  float inv_norm[5], wsum_col[5];
  for (int j = 0; j < 5; ++j) {
    float ws = 0.f;
    for (int i = 0; i < 4; ++i) ws += yv[kMod + 5 * i + j];
    wsum_col[j] = ws;
    inv_norm[j] = 1.f / fmaxf(1.f, ws);
  }
  float lfo_wsum[2];
  for (int l = 0; l < 2; ++l) {
    float ws = 0.f;
    for (int s = 0; s < 5; ++s) ws += yv[kLfo + 8 * l + 3 + s];
    lfo_wsum[l] = ws;
  }
  float* dth = buf.dtheta + (size_t)v * 2 * P;
  float* de = buf.denv + (size_t)v * 6 * P;
  const float* env = buf.env + (size_t)v * 6 * P;

  // pass A: modulation mixer, LFO outputs, pitch
  for (int base = 0; base < P; base += kBC) {
    const int k = base + threadIdx.x;
    const bool ok = k < P;
    const int kk = ok ? k : 0;
    float e[6];
    for (int a = 0; a < 6; ++a) e[a] = env[(size_t)a * P + kk];
    float mix[2], sh[2][5], dsh[2][5], lfo[2];
    for (int l = 0; l < 2; ++l) {
      lfo_shapes(buf.phase[((size_t)v * 2 + l) * P + kk], sh[l], dsh[l]);
      float accm = 0.f;
      for (int s = 0; s < 5; ++s) accm += yv[kLfo + 8 * l + 3 + s] * sh[l][s];
      mix[l] = lfo_wsum[l] < 1e-12f ? 0.f : accm / lfo_wsum[l];
      lfo[l] = e[3 + 2 * l] * mix[l];
    }
    const float src[4] = {e[0], e[1], lfo[0], lfo[1]};
    // the point's pitch and amplitude adjoints: the left end of interval k and the
    // right end of interval k - 1, the pitch ones' sums in FP64 (they cancel)
    float gk[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    double gm0 = 0.0, gm1 = 0.0;
    if (ok && k < K) {
      const float* st = stat + (size_t)k * kStat;
      const double2 c = csum[k];
      gm0 = (double)st[1] + (double)st[2] * c.x;
      gm1 = (double)st[6] + (double)st[7] * c.y;
      // square-saw drive kappa_k = min(50, 1 + SR/(8 f_k)): d kappa / d m =
      // -(kappa - 1) ln2/12 while below the bound and the pitch is uncapped
      const float kap = buf.kappa[((size_t)v * 2 + 0) * K + k];
      if (kap < (float)kBrightnessMax &&
          !((buf.seg[((size_t)v * 2 + 1) * K + k].jc_flags >> 18) & 1))
        gm1 -= (double)st[16] * (double)(kap - 1.f);
      for (int c3 = 0; c3 < 3; ++c3) gk[2 + c3] = st[10 + c3];
    }
    if (ok && k > 0) {
      const float* st = stat + (size_t)(k - 1) * kStat;
      const double2 c = csum[k - 1];
      gm0 += (double)st[3] + (double)st[4] * c.x;
      gm1 += (double)st[8] + (double)st[9] * c.y;
      for (int c3 = 0; c3 < 3; ++c3) gk[2 + c3] += st[13 + c3];
    }
    gk[0] = (float)(l12 * gm0);
    gk[1] = (float)(l12 * gm1);
    const float dd[5] = {yv[kSine + 1] * gk[0], gk[2], yv[kSqr + 1] * gk[1], gk[3], gk[4]};
    float dst[5];
    for (int j = 0; j < 5; ++j) dst[j] = buf.dest[((size_t)v * 5 + j) * P + kk];
    // pitch: m = midi + tune + depth * dest
    const float dm0 = gk[0];
    const float dm1 = gk[1];
    acc_y(gyw, kSqr, dm1);
    acc_y(gyw, kSine + 1, dm0 * dst[0]);
    acc_y(gyw, kSqr + 1, dm1 * dst[2]);
    // the other 32 sums in one go: 20 modulation weights, 10 shape weights, midi, sine tune
    float r[32];
    r[30] = dm0 + dm1;
    r[31] = dm0;
    // dest_j = (sum_i W_ij src_i) / max(1, sum_i W_ij)
    float dsrc[4] = {0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      const float over = wsum_col[j] > 1.f ? 1.f : 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        dsrc[i] += dd[j] * yv[kMod + 5 * i + j] * inv_norm[j];
        r[5 * i + j] = dd[j] * (src[i] * inv_norm[j] - over * dst[j] * inv_norm[j]);
      }
    }
    float dea[6] = {dsrc[0], dsrc[1], 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      const float dl = dsrc[2 + l];
      dea[3 + 2 * l] = dl * mix[l];
      const float dmix = dl * e[3 + 2 * l];
      float dthv = 0.f;
      const bool on = lfo_wsum[l] >= 1e-12f;
#pragma unroll
      for (int s = 0; s < 5; ++s) {
        r[20 + 5 * l + s] = on ? dmix * (sh[l][s] - mix[l]) / lfo_wsum[l] : 0.f;
        dthv += yv[kLfo + 8 * l + 3 + s] * dsh[l][s];
      }
      if (ok) dth[(size_t)l * P + k] = on ? dthv * (dmix / lfo_wsum[l]) : 0.f;
    }
    acc_y32(gyw, r, [](int i) {
      return i < 20 ? kMod + i : i < 25 ? kLfo + 3 + i - 20 : i < 30 ? kLfo + 8 + 3 + i - 25
             : i == 30 ? kMidi : kSine;
    });
    if (ok)
      for (int a = 0; a < 6; ++a) de[(size_t)a * P + k] = dea[a];
  }
  __syncthreads();

  // pass B: reverse scan of the LFO phase adjoint -> d/d(phase increment);
  // increments rate_k / CR with rate = clamp(freq + depth * env_rate, 0, 20)
  float carry0 = 0.f, carry1 = 0.f;
  for (int base = 0; base < P; base += kBC) {
    const int idx = P - 1 - (base + (int)threadIdx.x);
    const bool ok = idx >= 0;
    float a0 = ok ? dth[idx] : 0.f, a1 = ok ? dth[(size_t)P + idx] : 0.f, t0, t1;
    block_exclusive_scan2<float, kBC>(a0, a1, warp_tot, t0, t1);
    for (int l = 0; l < 2; ++l) {
      float dinc = 0.f, er = 0.f, rate_raw = 0.f;
      if (ok) {
        dinc = (l == 0 ? carry0 + a0 : carry1 + a1);  // sum of dtheta over points after idx
        er = env[(size_t)(2 + 2 * l) * P + idx];
        rate_raw = yv[kLfo + 8 * l] + yv[kLfo + 8 * l + 1] * er;
      }
      const bool inside = ok && rate_raw >= 0.f && rate_raw <= (float)kLfoMaxHz;
      const float dr = inside ? dinc * inv_cr : 0.f;
      acc_y(gyw, kLfo + 8 * l, dr);
      acc_y(gyw, kLfo + 8 * l + 1, dr * er);
      if (ok) de[(size_t)(2 + 2 * l) * P + idx] = dr * yv[kLfo + 8 * l + 1];
    }
    carry0 += t0;
    carry1 += t1;
  }
  if (threadIdx.x == 0) {
    gyw[kLfo + 2] += carry0 * inv_2pi;  // theta_0 = frac(phase0 / 2 pi)
    gyw[kLfo + 8 + 2] += carry1 * inv_2pi;
  }
  __syncthreads();

  // pass C: the ADSRs' partials, the (envelope, point) pairs spread over
  // the block; each thread sums its pairs' partials per envelope, then one
  // block-wide sum per partial
  float dur_acc = 0.f;
  float acc[6][5];
#pragma unroll
  for (int a = 0; a < 6; ++a)
#pragma unroll
    for (int q = 0; q < 5; ++q) acc[a][q] = 0.f;
  for (int i = threadIdx.x; i < 6 * P; i += kBC) {
    const int a = i / P, k = i - a * P;
    const float g = de[(size_t)a * P + k];
    if (g != 0.f) {
      float out[6];
      // t_k = k / CR: the float-float product the forward pass uses,
      // rounded to float (no FP64 division per point and envelope)
      adsr_d(ff_to_float(ff_mul_f(vc.inv_cr, (float)k)), yv + kAdsr + 5 * a, yv[kDuration], out);
#pragma unroll
      for (int b = 0; b < 6; ++b)
        if (b == a) {
#pragma unroll
          for (int q = 0; q < 5; ++q) acc[b][q] += g * out[q];
        }
      dur_acc += g * out[5];
    }
  }
  float r[32];
#pragma unroll
  for (int i = 0; i < 30; ++i) r[i] = acc[i / 5][i % 5];
  r[30] = dur_acc;
  r[31] = 0.f;
  acc_y32(gyw, r, [](int i) { return i < 30 ? kAdsr + i : i == 30 ? kDuration : kGY - 1; });
  __syncthreads();
  for (int i = threadIdx.x; i < kGY; i += kBC) {
    float t = 0.f;
    for (int w = 0; w < kBC / 32; ++w) t += gyw_all[w][i];
    gy[i] = t;
  }
  __syncthreads();

  if (threadIdx.x == 0) {
    gy[kSine + 2] += (float)total0 * inv_2pi;  // sums over every sample: d/d(initial phase, cycles)
    gy[kSqr + 2] += (float)total1 * inv_2pi;
    float va[4];
    for (int c = 0; c < 4; ++c) {
      double t = 0.0;
      for (int w = 0; w < kBC / 32; ++w) t += red[c][w];
      va[c] = (float)t;
    }
    gy[kSqr + 3] += va[3];
    // mixer gains g_i = l_i / max(1, sum l)
    const float l0 = yv[kMix], l1 = yv[kMix + 1], l2 = yv[kMix + 2];
    const float sum = l0 + l1 + l2, norm = fmaxf(1.f, sum);
    const float dotg = va[0] * l0 + va[1] * l1 + va[2] * l2;
    for (int c = 0; c < 3; ++c)
      gy[kMix + c] += va[c] / norm - (sum > 1.f ? dotg / (norm * norm) : 0.f);
  }
  __syncthreads();
  // through the range map: d/du = d/dy dy/du
  if (threadIdx.x < kNumParams &&
      in_bounds(hdr, (long long)v * kNumParams + threadIdx.x, (long long)batch * kNumParams)) {
    const size_t i = (size_t)v * kNumParams + threadIdx.x;
    grad_params[i] = gy[threadIdx.x] * range_map_dydu(vc, threadIdx.x, u_in[i]);
  }
}


}  // namespace

size_t backward_workspace_bytes(const VoiceConst& vc, int batch) {
  return adj_carve(vc, batch, nullptr).total;
}

cudaError_t launch_render_backward(const VoiceConst& vc, uint64_t seed, uint64_t batch_index,
                                   int batch, const float* params, const float* grad_audio,
                                   float* grad_params, void* workspace, ScratchHeader* hdr,
                                   cudaStream_t st) {
  if (vc.R > 128) return cudaErrorInvalidValue;
  const AdjBuffers b = adj_carve(vc, batch, workspace);
  bwd_recompute<<<batch, kCT, 0, st>>>(vc, batch, params, b, hdr);
  const dim3 gs((vc.K + kSI - 1) / kSI, batch);
  bwd_samples<<<gs, kST, 0, st>>>(vc, seed, batch_index, batch, grad_audio, b, hdr);
  bwd_control<<<batch, kBC, 0, st>>>(vc, b, params, grad_params, batch, hdr);
  return cudaGetLastError();
}

}  // namespace synth
