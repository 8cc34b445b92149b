// Kramers-Kronig receiver front end (declared in rx_kk.h).
//
// Stage 1 (kk_hilbert_kernel, one 64-thread CTA per two windows of 1024 samples,
// hop 512, packed as real and imaginary parts of one transform): intensity I ->
// a = sqrt(max(I, 1e-30)), ln a (8-bit samples: a table of the 256 codes); FFT;
// multiply by j sign(f) / N and conjugate; the same forward FFT again gives the
// Hilbert image phi (inverse by conjugation); the kept half of the window becomes
// E = a exp(j phi) exp(j 2 pi f_c n / fs), the shift to DC taken from a 64-bit
// fixed-point phase accumulator.
// Stage 2 (kk_filter_kernel, one 64-thread CTA per window): FFT 1024 of the
// field, multiply by the static filter (dispersion inverse x RRC, with the 1/2
// of the decimated DFT and 1/512 of the inverse folded in), keep the 512 bins
// of |f| < fs/4, inverse 512-point FFT, keep the window's centre at 2 samples
// per symbol.
// Both stages hold a transform in the registers of 64 threads, element t + 64 i in
// register i of thread t before and after every FFT: the last pass of the first
// transform, the spectrum's multiplication and the first pass of the second work on the
// same registers, the first and the last pass read and write global memory directly, and
// the pair of FFTs crosses shared memory four times, one barrier each.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <string>
#include <vector>

#include "../../include/rx_kk.h"
#include "fft.cuh"
#include "rx_internal.h"

namespace rx {
namespace {

constexpr int KN = 1024;          // transform length of both stages
constexpr int KH = KN / 2;        // Hilbert overlap and hop (100 % overlap-save)
constexpr int KN2 = KN / 2;       // decimated transform length
constexpr int KDELAY = 1536;      // output delay (samples): the look-ahead of both stages (1280), rounded to 512
constexpr int KHIST = 3072;       // input history kept from earlier buffers (samples)
constexpr int KEDGE = 1024;       // field computed beyond the output range on each side

// Where stream sample s comes from: the current buffer [pos, pos + n), the history
// of earlier buffers [pos - KHIST, pos) (float intensities), or nothing (before the
// stream start or at / after its end: outside, zero log-amplitude and zero field).
struct KkSrc {
  const void *in;
  int dtype;
  int64_t pos, n;
  float scale, offset;
  const float *hist;
  int64_t start, end;
};

__device__ __forceinline__ bool kk_inside(const KkSrc &src, int64_t s) { return s >= src.start && s < src.end; }

__device__ __forceinline__ float kk_intensity(const KkSrc &src, int64_t s) {
  if (s >= src.pos) {
    const int64_t m = s - src.pos;
    const float x = src.dtype == RX_KK_I8 ? (float)reinterpret_cast<const int8_t *>(src.in)[m]
                                          : reinterpret_cast<const float *>(src.in)[m];
    return (x + src.offset) * src.scale;
  }
  return src.hist[s - (src.pos - KHIST)];
}

// A load of what the kernel in front of an overlapped launch writes: coherent, and kept behind
// griddepcontrol.wait (a const __restrict__ pointer or __ldg would let the compiler take it for
// read-only data of the whole kernel, whose life begins while that kernel still writes).
__device__ __forceinline__ float2 kk_load_behind_wait(const float2 *p) {
  float2 v;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
  return v;
}

// ---- transforms of 64 threads: x[i] is element t + 64 i
constexpr int KT = 64;
constexpr int KBUF = KN + KN / 16;       // one float2 of padding per 16: unit- and 16-strided accesses conflict-free
__device__ __forceinline__ int kpad(int i) { return i + (i >> 4); }

// Stockham pass boundary: the R outputs of a pass of stride Ns (butterfly of inputs
// t + 64 r) to buf; the next pass reads elements t + 64 i back.  With two buffers in turn a
// thread is past the barrier of one exchange before any can write that buffer again; with
// ONE buffer a barrier in front keeps the last exchange's reads ahead of the writes.
template <int R, int Ns, int N, bool ONE = false>
__device__ __forceinline__ void kk_exchange(float2 *buf, float2 (&x)[N / KT], int t) {
  static_assert(R == N / KT, "one butterfly per thread");
  const int d = (t / Ns) * Ns * R + (t & (Ns - 1));
  if (ONE) __syncthreads();
#pragma unroll
  for (int r = 0; r < R; ++r) buf[kpad(d + r * Ns)] = x[r];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < R; ++i) x[i] = buf[kpad(t + KT * i)];
}

// x[r] *= W_{Ns R}^{r jm}
template <int R, int Ns, int N>
__device__ __forceinline__ void kk_twiddle(float2 (&x)[R], int jm, const float2 *__restrict__ tw) {
  constexpr int TW = N / (Ns * R);
#pragma unroll
  for (int r = 1; r < R; ++r) x[r] = cmul(x[r], __ldg(&tw[r * jm * TW]));
}

// 1024-point forward FFT, radices 16, 16, 4 (the last as four butterflies j = t + 64 q of
// elements j + 256 r, registers q + 4 r); natural order in and out.
template <bool ONE>
__device__ __forceinline__ void kk_fft1024(float2 (&x)[16], int t, float2 *b0, float2 *b1, const float2 *__restrict__ tw) {
  dft<16>(x);
  kk_exchange<16, 1, KN, ONE>(b0, x, t);
  kk_twiddle<16, 16, KN>(x, t & 15, tw);
  dft<16>(x);
  kk_exchange<16, 16, KN, ONE>(b1, x, t);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float2 v[4] = {x[q], x[q + 4], x[q + 8], x[q + 12]};
    kk_twiddle<4, 256, KN>(v, t + KT * q, tw);
    dft4(v[0], v[1], v[2], v[3]);
#pragma unroll
    for (int r = 0; r < 4; ++r) x[q + 4 * r] = v[r];
  }
}

// Windows 2b and 2b + 1 in one transform pair: window w gives the field of stream
// samples [e0 + 512 w, e0 + 512 w + 512) from the input over [e0 + 512 w - 256,
// e0 + 512 w + 768), written to E[s - e0].  The log-amplitudes of the two windows
// are the real and imaginary parts of one complex sequence: the Hilbert response
// j sign(f) maps real sequences to real ones, so the inverse transform returns the
// first window's phase in its real part and the second's in its imaginary part --
// two windows for the price of one FFT pair.  The second window is the first one 512
// samples on, so a thread's samples t + 64 i (i < 24) serve both.
// CTAs from n_pairs on copy the input history for the next buffer (hist_next): the
// intensities of stream samples [pos + n - KHIST, pos + n).
// Bound by the latency of its loads (samples, twiddles) at 24 warps per SM, 46 % of the issue
// slots busy: 2^22 8-bit samples 46 us (81 with eight shared-memory crossings per pair).
template <bool I8>
__global__ void __launch_bounds__(KT, 12) kk_hilbert_kernel(KkSrc src, int64_t e0, int nwin, int n_pairs,
                                                            const float2 *__restrict__ tw, unsigned long long inc_q,
                                                            float2 *__restrict__ E, float *__restrict__ hist_next) {
  // one transform buffer: 12 CTAs per SM instead of 9
  __shared__ float2 buf[KBUF];
  __shared__ float2 lut[I8 ? 256 : 1];         // (ln a, a) of each code
  __shared__ float amp[2 * KH];                // a of the kept samples, lo + 256 on
  const int t = threadIdx.x;
  if ((int)blockIdx.x >= n_pairs) {
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    const int j = ((int)blockIdx.x - n_pairs) * KT + t;
    if (j < KHIST) hist_next[j] = kk_intensity(src, src.pos + src.n - KHIST + j);   // before the stream start: never read
    return;
  }
  if (I8) {
    for (int c = t; c < 256; c += KT) {
      const float p = fmaxf(((float)(c - 128) + src.offset) * src.scale, 1e-30f);
      lut[c] = make_float2(0.5f * logf(p), sqrtf(p));
    }
    __syncthreads();
  }
  // launched while the kernel in front drains: its results, and the scratch it reads, from here on
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int w0 = 2 * blockIdx.x;
  const bool two = w0 + 1 < nwin;
  const int64_t lo = e0 + (int64_t)w0 * KH - KH / 2;          // first sample of window w0
  // every sample of both windows in the current buffer
  const bool whole = two && lo >= src.pos && lo >= src.start && lo + KN + KH <= src.end;
  const int8_t *in8 = reinterpret_cast<const int8_t *>(src.in) + (lo - src.pos);
  const float *in32 = reinterpret_cast<const float *>(src.in) + (lo - src.pos);
  auto sample = [&](int i) -> float2 {          // (ln a, a) of sample lo + i; (0, 0) outside the stream
    const int64_t s = lo + i;
    if (!whole && !kk_inside(src, s)) return make_float2(0.f, 0.f);
    if (I8 && (whole || s >= src.pos)) return lut[(int)in8[i] + 128];
    const float p = fmaxf(whole ? (in32[i] + src.offset) * src.scale : kk_intensity(src, s), 1e-30f);
    return make_float2(0.5f * logf(p), sqrtf(p));
  };
  // a thread's samples through its own slots of the buffer: one copy of the sample code
  float *const ln = reinterpret_cast<float *>(buf);
#pragma unroll 4
  for (int i = 0; i < 24; ++i) {
    const int m = t + KT * i;
    const float2 v = sample(m);
    ln[m] = v.x;
    if (i >= 4 && i < 20) amp[m - KH / 2] = v.y;
  }
  float2 x[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) x[i] = make_float2(ln[t + KT * i], two ? ln[t + KT * i + KH] : 0.f);
  kk_fft1024<true>(x, t, buf, buf, tw);
  const float inv = 1.f / (float)KN;
#pragma unroll
  for (int i = 0; i < 16; ++i) {                // conj(j sign(f) X / N): bins k = t + 64 i
    const float2 v = x[i];
    x[i] = i < 8 ? make_float2(-v.y * inv, -v.x * inv) : make_float2(v.y * inv, v.x * inv);
    if (i % 8 == 0 && t == 0) x[i] = make_float2(0.f, 0.f);     // k = 0 and N / 2
  }
  // the second transform forms its twiddles' addresses again: held from the first, they
  // would spill
  int t2 = t;
  asm volatile("" : "+r"(t2));
  kk_fft1024<true>(x, t2, buf, buf, tw);
  // inverse = conj of the forward transform of the conjugate: phase of window w0 in
  // the real part, of window w0 + 1 in the (negated) imaginary part
  // (through the thread's own slots of the buffer)
  float *const ph = ln;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    ph[t + KT * i] = x[i + 4].x;
    ph[t + KT * i + KH] = -x[i + 4].y;
  }
  const int n_out = two ? 16 : 8;
#pragma unroll 4
  for (int i = 0; i < n_out; ++i) {
    const int m = t + KT * i;                    // field sample of the pair
    const int64_t s = lo + KH / 2 + m;
    const float a = amp[m];                      // outside the stream: zero field
    // exp(j (phi + 2 pi f_c s / fs)): the turn s inc_q (signed Q0.64) in half turns, rounded from
    // its top 32 bits to the 24 of a float (2^-25 half turns near +-1), phi / pi in two terms,
    // one sine and cosine
    const float turn = (float)(int)(((unsigned long long)s * inc_q) >> 32) * 4.65661287307739258e-10f;   // 2^-31
    // (a 0 there whatever the phase: an infinite intensity leaves none in its whole window)
    const float phi = a > 0.f ? ph[m] : 0.f;
    float sp, cp;
    sincospif(fmaf(phi, 0.31830987334251404f, fmaf(phi, 1.2841276632e-08f, turn)), &sp, &cp);
    E[s - e0] = make_float2(a * cp, a * sp);
  }
}

// Window i0 + b of the static filter: E over [i S - V/2, i S - V/2 + 1024) (E[s - e0]),
// output samples t in [i S, i S + S) inside [o0, o0 + no) at 2 samples/symbol to
// y[(t - o0)/2] (zero before the stream start); optionally the field itself to
// field[t - o0] for every t of the range.
// Bound by load and shared-memory latency: 2^22 samples 43 us (52 with 32 threads, staged loads
// and seven crossings); 14 or 16 CTAs per SM with one buffer measured the same.
__global__ void __launch_bounds__(KT, 12) kk_filter_kernel(const float2 *E, int64_t e0, int64_t i0, int64_t o0,
                                                       int64_t no, int64_t start, int V,
                                                       const float2 *__restrict__ H, const float2 *__restrict__ tw,
                                                       const float2 *__restrict__ tw2, float2 *__restrict__ y,
                                                       float2 *__restrict__ field) {
  __shared__ float2 b0[KBUF], b1[KBUF];
  const int t = threadIdx.x;
  const int S = KN - V;
  const int64_t i = i0 + blockIdx.x;
  const int64_t lo = i * S - V / 2;
  float2 x[16];
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const float2 *src = E + (lo - e0) + t;
#pragma unroll
  for (int q = 0; q < 16; ++q) x[q] = kk_load_behind_wait(src + KT * q);
  if (field) {
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int m = t + KT * q;
      const int64_t tt = lo + m;
      if (m >= V / 2 && m < V / 2 + S && tt >= o0 && tt < o0 + no) field[tt - o0] = x[q];
    }
  }
  kk_fft1024<false>(x, t, b0, b1, tw);
  // keep |f| < fs/4: bins k < 256 -> k, k >= 768 -> k - 512; conjugate for the inverse
  float2 z[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int r = q < 4 ? q : q + 8;
    z[q] = cconj(cmul(x[r], __ldg(&H[t + KT * r])));
  }
  // 512-point forward FFT, radices 8, 8, 8
  dft<8>(z);
  kk_exchange<8, 1, KN2>(b0, z, t);
  kk_twiddle<8, 8, KN2>(z, t & 7, tw2);
  dft<8>(z);
  kk_exchange<8, 8, KN2>(b1, z, t);
  kk_twiddle<8, 64, KN2>(z, t, tw2);
  dft<8>(z);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int m = t + KT * q;
    const int64_t tt = i * S + 2 * (m - V / 4);      // input-rate sample of this output
    if (m < V / 4 || m >= V / 4 + S / 2 || tt < o0 || tt >= o0 + no) continue;
    y[(tt - o0) / 2] = tt >= start ? cconj(z[q]) : make_float2(0.f, 0.f);
  }
}

}  // namespace
}  // namespace rx

using namespace rx;

struct rx_kk {
  double baud = 0, carrier = 0, L_km = 0, D = 0, rolloff = 0;
  int sps = 4, V = KH;
  int64_t max_n = 0;
  unsigned long long inc_q = 0;
  int64_t pos = 0;                  // stream position of the next buffer's first sample
  int64_t start = 0;                // first sample of the current stream
  cudaStream_t stream = nullptr;
  float2 *tw = nullptr, *tw2 = nullptr, *H = nullptr, *Hs = nullptr, *E = nullptr;
  float *hist[2] = {nullptr, nullptr};   // input history ping-pong (KHIST intensities each)
  int cur = 0;
  bool profile = false;
  std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> pending;
  double ms[2] = {0, 0};
  std::string msg;
};

namespace {

rx_status kfail(rx_kk *k, rx_status s, const std::string &m) {
  if (k) k->msg = m;
  return s;
}

void kk_release(rx_kk *k) {
  cudaFree(k->tw);
  cudaFree(k->tw2);
  cudaFree(k->H);
  cudaFree(k->Hs);
  cudaFree(k->E);
  cudaFree(k->hist[0]);
  cudaFree(k->hist[1]);
  k->tw = k->tw2 = k->H = k->Hs = k->E = nullptr;
  k->hist[0] = k->hist[1] = nullptr;
  std::vector<cudaEvent_t> seen;     // consecutive stages share an event
  for (auto &p : k->pending)
    for (cudaEvent_t ev : {p.second.first, p.second.second})
      if (std::find(seen.begin(), seen.end(), ev) == seen.end()) seen.push_back(ev);
  for (cudaEvent_t ev : seen) cudaEventDestroy(ev);
  k->pending.clear();
}

}  // namespace

extern "C" {

rx_status rx_kk_create(rx_kk **out, double baud, int sps, double carrier_hz, double L_km, double D_ps_nm_km,
                       double rolloff, int64_t max_samples) {
  if (!out) return RX_EINVAL;
  *out = nullptr;
  if (!(baud > 0) || !(L_km >= 0) || !(rolloff > 0 && rolloff <= 1) || max_samples <= 0 || max_samples % 2 ||
      carrier_hz != carrier_hz || D_ps_nm_km != D_ps_nm_km)
    return RX_EINVAL;
  if (sps != 4) return RX_EUNSUPPORTED;
  rx_kk *k = new (std::nothrow) rx_kk();
  if (!k) return RX_ENOMEM;
  *out = k;
  k->baud = baud;
  k->sps = sps;
  k->carrier = carrier_hz;
  k->L_km = L_km;
  k->D = D_ps_nm_km;
  k->rolloff = rolloff;
  k->max_n = max_samples;
  const int64_t ncd = n_cd_taps(baud, sps, L_km, D_ps_nm_km, 1550.0);
  k->V = (int)std::max<int64_t>(KH, ((ncd - 1 + 31) / 32) * 32);
  if (k->V >= KN) return kfail(k, RX_EUNSUPPORTED, "dispersion too large for the 1024-point static filter");
  // f_c / fs as a Q0.64 turn increment
  double frac = carrier_hz / (sps * baud);
  frac -= floor(frac);
  k->inc_q = (unsigned long long)(frac * 18446744073709551616.0);
  cudaError_t e = cudaMalloc(&k->tw, KN * sizeof(float2));
  if (e == cudaSuccess) e = cudaMalloc(&k->tw2, KN2 * sizeof(float2));
  if (e == cudaSuccess) e = cudaMalloc(&k->Hs, KN * sizeof(float2));
  if (e == cudaSuccess) e = cudaMalloc(&k->H, KN * sizeof(float2));
  // field scratch: the output range plus KEDGE on each side (a flush covers KDELAY)
  if (e == cudaSuccess)
    e = cudaMalloc(&k->E, (size_t)(std::max<int64_t>(max_samples, KDELAY) + 2 * KEDGE) * sizeof(float2));
  if (e == cudaSuccess) e = cudaMalloc(&k->hist[0], KHIST * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&k->hist[1], KHIST * sizeof(float));
  if (e != cudaSuccess) {
    cudaGetLastError();
    kk_release(k);
    return kfail(k, RX_ENOMEM, "device allocation failed");
  }
  // twiddles of both transform sizes (the scratch filter table is unused)
  e = launch_tables(k->Hs, k->tw, KN, baud, 0.0, 0.0, 1550.0, rolloff, k->stream);
  if (e == cudaSuccess) e = launch_tables(k->Hs, k->tw2, KN2, baud, 0.0, 0.0, 1550.0, rolloff, k->stream);
  // static filter on the input grid: sqrt(sps) RRC x dispersion inverse x the constant that takes back
  // the carrier tone's own dispersion phase (unit symbol gain, no constant phase), with the 1/2 of the
  // decimated DFT and the 1/512 of its inverse
  std::vector<float2> h(KN);
  const double pi = 3.14159265358979323846, fs = sps * baud;
  const double Dsm = D_ps_nm_km * 1e-12 / (1e-9 * 1e3), lam = 1550e-9;
  const double beta2 = -Dsm * lam * lam / (2.0 * pi * 299792458.0);
  const double f1 = (1.0 - rolloff) * baud / 2.0, f2 = (1.0 + rolloff) * baud / 2.0;
  for (int i = 0; i < KN; ++i) {
    const double f = (double)(i < KN / 2 ? i : i - KN) * fs / KN, af = fabs(f);
    double r = 0.0;
    if (af <= f1) r = 1.0;
    else if (af <= f2) r = cos(pi * (af - f1) / (2.0 * rolloff * baud));
    const double w = 2.0 * pi * f, wc = 2.0 * pi * carrier_hz;
    const double ph = -beta2 * (L_km * 1e3) * (w * w - wc * wc) / 2.0;
    const double g = r * sqrt((double)sps) * 0.5 / KN2;
    h[i] = make_float2((float)(g * cos(ph)), (float)(g * sin(ph)));
  }
  if (e == cudaSuccess) e = cudaMemcpy(k->H, h.data(), KN * sizeof(float2), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaStreamSynchronize(k->stream);
  if (e != cudaSuccess) {
    kk_release(k);
    return kfail(k, RX_ECUDA, std::string("create: ") + cudaGetErrorString(e));
  }
  return RX_OK;
}

rx_status rx_kk_set_cuda_stream(rx_kk *k, void *s) {
  if (!k) return RX_EINVAL;
  k->stream = (cudaStream_t)s;
  return RX_OK;
}

rx_status rx_kk_get_overlap(rx_kk *k, int *v) {
  if (!k || !v) return RX_EINVAL;
  *v = k->V;
  return RX_OK;
}

}  // extern "C"

namespace {

int64_t floor_div(int64_t a, int64_t b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// A launch whose CTAs may be placed while the kernel in front of it drains (they wait for
// its end themselves, before they touch memory that it uses).
template <class... KArgs, class... Args>
cudaError_t launch_overlapped(bool overlap, void (*fn)(KArgs...), unsigned grid, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(KT);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, fn, args...);
}

// Output samples [pos - KDELAY, pos - KDELAY + no) of the stream whose input is
// known on [start, end): Hilbert windows over the field range with KEDGE on each
// side, then the static filter's windows over the output range.
rx_status kk_run(rx_kk *k, const KkSrc &src, int64_t no, float *y, float *field) {
  cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
  if (k->profile)
    for (auto &e : ev)
      if (cudaEventCreate(&e) != cudaSuccess) return kfail(k, RX_ECUDA, "event");
  const int64_t o0 = k->pos - KDELAY, e0 = o0 - KEDGE;
  if (ev[0]) cudaEventRecord(ev[0], k->stream);
  const int nwin = (int)((no + 2 * KEDGE) / KH);
  const int n_pairs = (nwin + 1) / 2;
  const unsigned grid = (unsigned)(n_pairs + (src.n > 0 ? KHIST / KT : 0));   // + the history's copy
  const auto hilbert = src.dtype == RX_KK_I8 ? kk_hilbert_kernel<true> : kk_hilbert_kernel<false>;
  // (a buffer's first stage is not: its CTAs, placed early, keep the equaliser's acquisition on
  // another stream from finding an SM, 543 -> 589 us over four buffers; the flush is small)
  cudaError_t e = launch_overlapped(src.n == 0, hilbert, grid, k->stream, src, e0, nwin, n_pairs, (const float2 *)k->tw, k->inc_q, k->E,
                                    k->hist[1 - k->cur]);
  if (ev[1]) cudaEventRecord(ev[1], k->stream);
  const int S = KN - k->V;
  const int64_t i0 = floor_div(o0, S), i1 = floor_div(o0 + no - 1, S);
  if (e == cudaSuccess) {
    e = launch_overlapped(true, kk_filter_kernel, (unsigned)(i1 - i0 + 1), k->stream, (const float2 *)k->E, e0, i0, o0, no, k->start,
                          k->V, (const float2 *)k->H, (const float2 *)k->tw, (const float2 *)k->tw2,
                          reinterpret_cast<float2 *>(y), reinterpret_cast<float2 *>(field));
  }
  if (ev[2]) {
    cudaEventRecord(ev[2], k->stream);
    k->pending.push_back({0, {ev[0], ev[1]}});
    k->pending.push_back({1, {ev[1], ev[2]}});
  }
  if (e != cudaSuccess) return kfail(k, RX_ECUDA, std::string("launch: ") + cudaGetErrorString(e));
  return RX_OK;
}

}  // namespace

extern "C" {

rx_status rx_kk_process(rx_kk *k, const void *in, int dtype, int64_t n, float in_scale, float in_offset, float *y,
                        float *field) {
  if (!k) return RX_EINVAL;
  if (n < 0 || n % KH || n > k->max_n)
    return kfail(k, RX_EINVAL, "sample count must be a multiple of 512 and within max_samples");
  if (dtype != RX_KK_I8 && dtype != RX_KK_F32) return kfail(k, RX_EINVAL, "unknown input dtype");
  if (n == 0) return RX_OK;
  if (!in || !y) return kfail(k, RX_EINVAL, "null input or output");
  if ((uintptr_t)y % 8 || (field && (uintptr_t)field % 8) || (dtype == RX_KK_F32 && (uintptr_t)in % 4))
    return kfail(k, RX_EINVAL, "misaligned buffer");
  KkSrc src{in, dtype, k->pos, n, in_scale, in_offset, k->hist[k->cur], k->start, k->pos + n};
  const rx_status s = kk_run(k, src, n, y, field);
  if (s != RX_OK) return s;
  k->cur = 1 - k->cur;
  k->pos += n;
  return RX_OK;
}

rx_status rx_kk_flush(rx_kk *k, float *y, float *field) {
  if (!k) return RX_EINVAL;
  if (!y) return kfail(k, RX_EINVAL, "null output");
  if ((uintptr_t)y % 8 || (field && (uintptr_t)field % 8)) return kfail(k, RX_EINVAL, "misaligned buffer");
  KkSrc src{nullptr, RX_KK_F32, k->pos, 0, 1.f, 0.f, k->hist[k->cur], k->start, k->pos};
  const rx_status s = kk_run(k, src, KDELAY, y, field);
  if (s != RX_OK) return s;
  k->pos = k->start = 0;     // the stream has ended: the next call starts a new one at 0
  return RX_OK;
}

rx_status rx_kk_get_delay(rx_kk *k, int *delay) {
  if (!k || !delay) return RX_EINVAL;
  *delay = KDELAY;
  return RX_OK;
}

rx_status rx_kk_set_position(rx_kk *k, int64_t pos) {
  if (!k) return RX_EINVAL;
  if (pos < 0) return kfail(k, RX_EINVAL, "stream position must be >= 0");
  k->pos = k->start = pos;
  return RX_OK;
}

rx_status rx_kk_profile(rx_kk *k, int on, double *ms, int reset) {
  if (!k) return RX_EINVAL;
  k->profile = on != 0;
  if (cudaStreamSynchronize(k->stream) != cudaSuccess) return kfail(k, RX_ECUDA, "profile wait");
  // events are shared between consecutive stages: destroy each once
  std::vector<cudaEvent_t> seen;
  for (auto &p : k->pending) {
    float t = 0.f;
    cudaEventElapsedTime(&t, p.second.first, p.second.second);
    k->ms[p.first] += t;
    for (cudaEvent_t ev : {p.second.first, p.second.second})
      if (std::find(seen.begin(), seen.end(), ev) == seen.end()) seen.push_back(ev);
  }
  for (cudaEvent_t ev : seen) cudaEventDestroy(ev);
  k->pending.clear();
  if (ms) {
    ms[0] = k->ms[0];
    ms[1] = k->ms[1];
  }
  if (reset) k->ms[0] = k->ms[1] = 0;
  return RX_OK;
}

void rx_kk_destroy(rx_kk *k) {
  if (!k) return;
  cudaStreamSynchronize(k->stream);
  kk_release(k);
  delete k;
}

const char *rx_kk_last_error(rx_kk *k) { return k ? k->msg.c_str() : "null handle"; }

}  // extern "C"
