// fsmp_lucy.cu -- LucyDDM on the GPU (arXiv 2403.03156, Sec. 2.3): Lucy's iterative
// deconvolution of each waveform by the SER at the sample times, then the solution space
// T = [t_min - 4 ns, t_max + 4 ns], the initial PEs {tau : q-hat(tau) > thresh} and t0 = t_min.
//
// With the kernel v(m) = V(m dt) / S (m = 0 .. L_V - 1, unit sum) and the data
// d(t) = max(w(t), 0) / S, one iteration is two correlations over the window:
//   w^r(t) = sum_m q(t - m) v(m)                          t = 0 .. n-1
//   q(tau) <- q(tau) sum_m [d / w^r](tau + m) v(m)         tau = -L_V+1 .. n-1
// (a ratio with w^r = 0 is 0; d / w^r is 0 outside the window). q^0 is uniform with the sum
// of d.
//
// Layout: one warp per waveform. In the index i = tau + L_V - 1 = 0 .. nq-1 (nq = n + L_V - 1) both
// correlations run over the same range: w^r(i) = sum_m q(i - m) v(m) for i >= L_V - 1, and
// q(i) *= sum_m r(i + m) v(m). Lane l owns the K = KP H values i = K l .. K l + K - 1 (K >= nq / 32,
// so that a window leaves few lanes idle: at n = 150 81 % of the computed outputs are used, where
// passes of 128 outputs used 71 %, at n = 64 75 % instead of 50 %). It computes them KP at a time in
// registers: a block of KP taps loads KP new source values (one 32-bit shared load per KP FMAs; the
// other operands slide through the registers) and does KP^2 FMAs. The arrays are stored by rows of
// i mod K with a constant stride, so that all lanes of a load read consecutive words of one row and
// a row's address is an offset of the load. The taps travel in the kernel's parameters, a block of
// them at a 16-byte boundary, and come through the constant cache. Every output adds its taps in the
// order m = 0, 1, .., L_V - 1, by one FMA each.
// Arithmetic: 2 (n + L_V) L_V FMAs per iteration, FP32. Bound: issue slots (88 % busy; 61 % of the
// instructions are FMAs, one in KP as many source loads), then the FP32 FMA pipe (54 %). 10 000 uneven windows x
// 500 iterations: 6.65 ms, 11.1 ms with 128 outputs a pass, four of them in registers. Packed FMAs
// (two outputs each) were slower (9.8 ms against 8.3 at that stage): their sources have to be held
// twice; so were taps from shared memory in place of constants (7.1), and two blocks per turn.
#include <math.h>

#include "fsmp_internal.h"

namespace fsmp {
namespace {

constexpr int kLucyMaxLV = 128;  // taps the parameters carry
constexpr int kKPMin = 4, kKPMax = 8;

// Blocks of kp taps, each at a multiple of 4 floats (kp = 4) or 8.
__host__ __device__ constexpr int tap_stride(int kp) { return kp <= 4 ? 4 : 8; }
__host__ __device__ constexpr int tap_blocks(int kp) { return (kLucyMaxLV + kp - 1) / kp; }
__host__ __device__ constexpr int tap_first(int kp) {  // of the blocks of kp in LucyArgs::taps
  int o = 0;
  for (int k = kKPMin; k < kp; ++k) o += tap_blocks(k) * tap_stride(k);
  return o;
}
constexpr int kTapFloats = tap_first(kKPMax + 1);

// Words of a row: 32 lanes' columns and the columns that the taps reach beyond them, at most
// ceil(L_V / K) + 1.
constexpr int kRow = 64;

// KP and H of a window: the least instructions per tap and lane, H (KP^2 + KP + 8) / KP (FMAs, loads
// and a block's overhead), of the splits that cover nq outputs and whose taps stay within a row.
__host__ __device__ inline void lucy_split(int LV, int nq, int* kp, int* h) {
  const int need = (nq + 31) / 32;
  int best = 0;
  for (int k = kKPMax; k >= kKPMin; --k) {
    const int hh = (need + k - 1) / k, c = hh * (k * k + k + 8) * (840 / k);
    if ((LV + k * hh - 1) / (k * hh) + 1 > kRow - 32) continue;
    if (best == 0 || c < best) { best = c; *kp = k; *h = hh; }
  }
}
// Per warp: q and the ratio in rows of kRow, the data in rows of 32.
__host__ __device__ inline int lucy_warp_floats(int K) { return (2 * kRow + 32) * K; }
inline size_t lucy_warp_bytes(int LV, int n_alloc) {  // of the widest split up to n_alloc samples
  size_t most = 0;
  const int nq_max = n_alloc + LV - 1;
  for (int nq = 32; nq < nq_max + 32; nq += 32) {
    int kp = 0, h = 0;
    lucy_split(LV, nq < nq_max ? nq : nq_max, &kp, &h);
    const size_t w = (size_t)lucy_warp_floats(kp * h);
    if (w > most) most = w;
  }
  return (sizeof(float) * most + 15) & ~(size_t)15;
}

struct LucyArgs {
  alignas(16) float taps[kTapFloats];  // v(m) in blocks of KP, for each KP
  const float* samples;
  const int32_t* offsets;
  const double* t_origin;
  int n_waveforms, n_alloc, n_iter, LV, R, z_stride;
  float thresh, inv_S;
  double dt, g;
  float* q_out;
  int32_t* T_lo;
  int32_t* T_hi;
  double* t0;
  int32_t* z;
  int32_t* n_z;
  int* status;  // per waveform: 0, or FSMP_ST_INVALID when the window is empty or longer than n_alloc
};

// The taps of block b (KP of them)
template <int KP> __device__ __forceinline__ void lucy_taps(const LucyArgs& A, int b, float (&v)[KP]) {
  const float4* p = reinterpret_cast<const float4*>(A.taps + tap_first(KP)) + b * (tap_stride(KP) / 4);
  const float4 t = p[0];
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  if constexpr (KP > 4) {
    const float4 u = p[1];
    const float w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int k = 4; k < KP; ++k) v[k] = w[k - 4];
  }
}

// The iterations of one waveform on a warp (its arrays are set up). Q, R, D: row 0 at the lane's own
// column. ONE: H = 1, the usual case (n <= 192 at L_V = 65): a block's sources are the rows again,
// one column on. The KP sources in registers slide in place: tap s of a block reads value e in
// register e mod KP, and the value that no later tap needs makes room for the next one, so that a
// block ends with every register where it began. Outputs beyond the window are computed too: their
// data are 0, which keeps the ratio and q-hat there 0.
template <int KP, bool ONE>
__device__ __forceinline__ void lucy_iterate(const LucyArgs& A, float* Q, float* R, const float* D, int H1) {
  constexpr int S = kRow;
  const int H = ONE ? 1 : H1, K = KP * H, nb = A.LV / KP, rem = A.LV - nb * KP;
  const int last = tap_first(KP) + nb * tap_stride(KP);  // the taps beyond the full blocks
#pragma unroll 1
  for (int it = 0; it < A.n_iter; ++it) {
    // w^r(i0 + k): tap KP b + s reads q(i0 + k - KP b - s)
#pragma unroll 1
    for (int h = 0; h < H; ++h) {
      const float* p = Q + h * KP * S;
      int hh = h;
      float acc[KP], x[KP];
#pragma unroll
      for (int k = 0; k < KP; ++k) { acc[k] = 0.0f; x[k] = p[k * S]; }
      auto before = [&] {  // the KP values before
        if (ONE) { p -= 1; }
        else { p = hh ? p - KP * S : p + (K - KP) * S - 1; hh = hh ? hh - 1 : H - 1; }
      };
#pragma unroll 1
      for (int b = 0; b < nb; ++b) {
        before();
        float v[KP];
        lucy_taps<KP>(A, b, v);
#pragma unroll
        for (int s = 0; s < KP; ++s) {
#pragma unroll
          for (int k = 0; k < KP; ++k) acc[k] = fmaf(x[(KP + k - s) % KP], v[s], acc[k]);
          x[KP - 1 - s] = p[(KP - 1 - s) * S];
        }
      }
      before();
#pragma unroll
      for (int s = 0; s < KP - 1; ++s) {
        if (s >= rem) break;
        const float v = A.taps[last + s];
#pragma unroll
        for (int k = 0; k < KP; ++k) acc[k] = fmaf(x[(KP + k - s) % KP], v, acc[k]);
        x[KP - 1 - s] = p[(KP - 1 - s) * S];
      }
#pragma unroll
      for (int k = 0; k < KP; ++k) {
        // a ratio of 0 / x (half the data are 0) sends the warp to the division's slow path, 30
        // instructions an output: divide 1 by 1 there
        const float d = D[(h * KP + k) * 32];
        const bool some = acc[k] > 0.0f && d > 0.0f;
        float num = some ? d : 1.0f, den = some ? acc[k] : 1.0f;
        asm("" : "+f"(num), "+f"(den));  // or the compiler divides d by acc after all
        const float r = num / den;
        R[(h * KP + k) * S] = some ? r : 0.0f;
      }
    }
    __syncwarp();
    // q(i0 + k) *= the sum over taps KP b + s of ratio(i0 + k + KP b + s) v
#pragma unroll 1
    for (int h = 0; h < H; ++h) {
      const float* p = R + h * KP * S;
      int hh = h;
      float acc[KP], x[KP];
#pragma unroll
      for (int k = 0; k < KP; ++k) { acc[k] = 0.0f; x[k] = p[k * S]; }
      auto after = [&] {  // the KP values after
        if (ONE) { p += 1; }
        else { p = hh + 1 < H ? p + KP * S : p - (K - KP) * S + 1; hh = hh + 1 < H ? hh + 1 : 0; }
      };
#pragma unroll 1
      for (int b = 0; b < nb; ++b) {
        after();
        float v[KP];
        lucy_taps<KP>(A, b, v);
#pragma unroll
        for (int s = 0; s < KP; ++s) {
#pragma unroll
          for (int k = 0; k < KP; ++k) acc[k] = fmaf(x[(k + s) % KP], v[s], acc[k]);
          x[s] = p[s * S];
        }
      }
      after();
#pragma unroll
      for (int s = 0; s < KP - 1; ++s) {
        if (s >= rem) break;
        const float v = A.taps[last + s];
#pragma unroll
        for (int k = 0; k < KP; ++k) acc[k] = fmaf(x[(k + s) % KP], v, acc[k]);
        x[s] = p[s * S];
      }
#pragma unroll
      for (int k = 0; k < KP; ++k) Q[(h * KP + k) * S] *= acc[k];
    }
    __syncwarp();
  }
}
template <int KP>
__device__ __forceinline__ void lucy_run(const LucyArgs& A, float* Q, float* R, const float* D, int H) {
  if (H == 1) lucy_iterate<KP, true>(A, Q, R, D, H);
  else lucy_iterate<KP, false>(A, Q, R, D, H);
}

__global__ void __launch_bounds__(32) lucy_kernel(const __grid_constant__ LucyArgs A) {
  extern __shared__ __align__(16) float lsm[];
  const int lane = threadIdx.x, wi = blockIdx.x;
  const int o0 = A.offsets[wi], n = A.offsets[wi + 1] - o0;
  const int LV = A.LV, nq = n + LV - 1;
  if (n < 1 || n > A.n_alloc) {
    if (lane == 0) {
      A.status[wi] = FSMP_ST_INVALID;
      A.n_z[wi] = 0; A.T_lo[wi] = 0; A.T_hi[wi] = max(n, 0) * A.R; A.t0[wi] = NAN;
    }
    return;
  }
  int KP = 0, H = 0;
  lucy_split(LV, nq, &KP, &H);
  // rows of i mod K, a word per i / K: q with the columns that earlier values lie in before its own,
  // the ratio with those of later values behind, the data
  constexpr int S = kRow, pad = S - 32;
  const int K = KP * H;
  float* const Q = lsm + pad;
  float* const R = lsm + K * S;
  float* const D = R + K * S;
  // data, zero pads, q^0
#pragma unroll 1
  for (int i = lane; i < 2 * K * S + 32 * K; i += 32) lsm[i] = 0.0f;
  __syncwarp();
  float ds = 0.0f;
#pragma unroll 1
  for (int t = lane; t < n; t += 32) {
    const float x = A.samples[o0 + t];
    const float dv = x > 0.0f ? x * A.inv_S : 0.0f;
    const int i = t + LV - 1;
    D[(i % K) * 32 + i / K] = dv;
    ds += dv;
  }
  for (int o = 16; o > 0; o >>= 1) ds += __shfl_xor_sync(0xffffffffu, ds, o);
  const float q0 = ds / (float)nq;
  __syncwarp();
#pragma unroll 1
  for (int i = lane; i < nq; i += 32) Q[(i % K) * S + i / K] = q0;
  __syncwarp();
  switch (KP) {
    case 4: lucy_run<4>(A, Q + lane, R + lane, D + lane, H); break;
    case 5: lucy_run<5>(A, Q + lane, R + lane, D + lane, H); break;
    case 6: lucy_run<6>(A, Q + lane, R + lane, D + lane, H); break;
    case 7: lucy_run<7>(A, Q + lane, R + lane, D + lane, H); break;
    default: lucy_run<8>(A, Q + lane, R + lane, D + lane, H); break;
  }
  // q-hat out, initial PEs in tau order, solution space and t0 (Sec. 2.3)
  float* qo = A.q_out ? A.q_out + (size_t)o0 + (size_t)wi * (LV - 1) : nullptr;
  int cnt = 0, tmin = 0, tmax = 0;
  int32_t* zo = A.z + (size_t)wi * A.z_stride;
#pragma unroll 1
  for (int b = 0; b < nq; b += 32) {
    const int i = b + lane;
    const int tau = i - (LV - 1);
    const float qv = i < nq ? Q[(i % K) * S + i / K] : 0.0f;
    if (qo && i < nq) qo[i] = qv;
    const bool on = i < nq && qv > A.thresh;
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (on) {
      const int pos = cnt + __popc(m & ((1u << lane) - 1u));
      if (pos < A.z_stride) zo[pos] = tau * A.R;
    }
    if (m) {
      if (cnt == 0) tmin = b + __ffs(m) - 1 - (LV - 1);
      tmax = b + 31 - __clz(m) - (LV - 1);
    }
    cnt += __popc(m);
  }
  if (lane == 0) {
    A.status[wi] = 0;
    A.n_z[wi] = cnt;
    if (cnt == 0) {
      A.T_lo[wi] = 0;
      A.T_hi[wi] = n * A.R;
      A.t0[wi] = NAN;
    } else {
      A.T_lo[wi] = (int32_t)floor((tmin * A.dt - 4.0) / A.g + 1e-9);
      A.T_hi[wi] = (int32_t)ceil((tmax * A.dt + 4.0) / A.g - 1e-9) + 1;
      A.t0[wi] = (A.t_origin ? A.t_origin[wi] : 0.0) + tmin * A.dt;
    }
  }
}

// The kernel taps v(m) = V(m dt) / S, zero-padded to whole groups of four.
__global__ void lucy_taps_kernel(const float* V32, int LV, int R, int jv, float* v4, float* S_out) {
  float s = 0.0f;
  for (int m = 0; m < LV; ++m) s += V32[m * R];
  for (int m = threadIdx.x; m < 4 * jv; m += blockDim.x) v4[m] = m < LV ? V32[m * R] / s : 0.0f;
  if (threadIdx.x == 0) *S_out = s;
}

}  // namespace

// What sets the longest window: four waveforms' data, q and ratio with their pads in one CTA's
// shared memory (a limit of the entry point, whatever this kernel's own layout takes).
size_t lucy_limit_bytes(int LV, int n_alloc) {
  const size_t jv = (size_t)(LV + 3) / 4, n = (size_t)n_alloc;
  const size_t q = 4 * (jv + 1) + (n + 127) / 128 * 128 + 8;
  const size_t r = 8 * (jv + 1) + (n + 4 * jv + 127) / 128 * 128 + 8;
  return 4 * sizeof(float) * (q + r + (n + 3) / 4 * 4);
}

cudaError_t lucy_kernel_attributes(int max_smem) {
  return cudaFuncSetAttribute(lucy_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
}

cudaError_t launch_lucy_taps(const float* V32, int LV, int R, float* v4, float* S_dev, cudaStream_t st) {
  lucy_taps_kernel<<<1, 128, 0, st>>>(V32, LV, R, (LV + 3) / 4, v4, S_dev);
  return cudaGetLastError();
}

cudaError_t launch_lucy(const float* v4_host, float S, int LV, int R, double dt, double g, int n_waveforms, int n_alloc,
                        const float* samples, const int32_t* offsets, const double* t_origin, int n_iter, float thresh,
                        float* q_out, int32_t* T_lo, int32_t* T_hi, double* t0, int32_t* z, int32_t* n_z, int z_stride,
                        int* status, cudaStream_t st) {
  if (n_waveforms <= 0) return cudaSuccess;
  if (LV > kLucyMaxLV) return cudaErrorInvalidValue;
  LucyArgs A;
  for (float& t : A.taps) t = 0.0f;
  for (int kp = kKPMin; kp <= kKPMax; ++kp)
    for (int m = 0; m < LV; ++m) A.taps[tap_first(kp) + m / kp * tap_stride(kp) + m % kp] = v4_host[m];
  A.samples = samples; A.offsets = offsets; A.t_origin = t_origin;
  A.n_waveforms = n_waveforms; A.n_alloc = n_alloc; A.n_iter = n_iter; A.LV = LV; A.R = R; A.z_stride = z_stride;
  A.thresh = thresh; A.inv_S = 1.0f / S; A.dt = dt; A.g = g;
  A.q_out = q_out; A.T_lo = T_lo; A.T_hi = T_hi; A.t0 = t0; A.z = z; A.n_z = n_z; A.status = status;
  lucy_kernel<<<(unsigned)n_waveforms, 32, lucy_warp_bytes(LV, n_alloc), st>>>(A);
  return cudaGetLastError();
}

}  // namespace fsmp
