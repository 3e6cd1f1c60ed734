// fsmp_pe.cu -- host side of the PE-space chain kernel (arXiv 2403.03156, Sec. 2.4 and Appendix
// A.1) and its dynode-model instances; the kernel itself is in fsmp_pe_kernel.cuh.
#include <type_traits>

#include "fsmp_pe_kernel.cuh"

namespace fsmp {

size_t pe_smem_bytes(const DevModel& M, int n_alloc, int warps, int lanes, int Ns, PeForm form) {
  const int chains = form == kPeTeam ? 1 : warps * (32 / lanes);
  const size_t cmd = form == kPeTeam ? kTeamBytes : 0;
  auto bytes = [&](auto big, auto lane_count, auto mix) {
    constexpr bool BIG = decltype(big)::value, MIX = decltype(mix)::value;
    constexpr int L = decltype(lane_count)::value;
    if (M.precision == FSMP_FP64)
      return pe_block_bytes<double>(M) + chains * pe_chain_bytes<double, BIG, L, MIX>(M.n_cap, n_alloc, M.win_extra, Ns);
    return pe_block_bytes<float>(M) + cmd + chains * pe_chain_bytes<float, BIG, L, MIX>(M.n_cap, n_alloc, M.win_extra, Ns);
  };
  using std::false_type;
  using std::true_type;
  const std::integral_constant<int, 16> l16;
  const std::integral_constant<int, 32> l32;
  if (M.n_comp > 1)
    return lanes == 16 ? bytes(false_type{}, l16, true_type{}) : bytes(false_type{}, l32, true_type{});
  if (pe_big(M.n_cap)) return bytes(true_type{}, l32, false_type{});
  return lanes == 16 ? bytes(false_type{}, l16, false_type{}) : bytes(false_type{}, l32, false_type{});
}

// The state that sets how long a window and how large a capacity a context takes: per chain 216
// bytes of sums, the draws of `lanes` steps, the lists and four vectors of n_cap PEs, the residual,
// log Phi and the C^-1 tile; per CTA the SER, log(i) and 1 / i. It stays what it is when the
// kernel's own layout changes, so that what is refused does not depend on the launch shape.
size_t pe_limit_bytes(const DevModel& M, int n_alloc, int warps, int lanes, int Ns) {
  const bool f64 = M.precision == FSMP_FP64;
  const size_t ts = f64 ? 8 : 4, cs = 2 * ts, n_cap = (size_t)M.n_cap;
  const size_t chain = a16(216) + a16((f64 ? 56 : 28) * (size_t)lanes) + 2 * a16(4 * n_cap) + a16(n_cap) +
                       4 * a16(cs * n_cap) + a16(ts * n_alloc) + a16(ts * M.win_extra) + a16(cs * (size_t)tri(Ns));
  return a16(ts * M.Lt) + a16(ts * (n_cap + 2)) + a16(8 * (n_cap + 2)) + (size_t)(warps * (32 / lanes)) * chain;
}

size_t pe_ws_slot_doubles(int n_cap) { return pe_ws_doubles(n_cap); }

size_t pe_c_entries(int n_cap) { return (size_t)tri(n_cap); }

size_t pe_c_entry_bytes(int precision) {
  return precision == FSMP_FP64 ? sizeof(PeTab<double>::C) : sizeof(PeTab<float>::C);
}

cudaError_t launch_split_ff(const double* a, float* out, size_t n, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  split_ff_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a, out, n);
  return cudaGetLastError();
}

// The pile-up variant (BIG) unrolls the gathers and row passes over C^-1 four ways so that
// their loads overlap; it pays off when chains carry many PEs (C^-1 in global memory) and costs
// registers otherwise.
bool pe_big(int n_cap) { return n_cap > 192; }

// Lanes per chain the kernel is built for: 32, and 16 where chains are small (not BIG).
bool pe_lanes_ok(int lanes, int n_cap) { return lanes == 32 || (lanes == 16 && !pe_big(n_cap)); }

bool pe_team_ok(int precision, int lanes) { return precision != FSMP_FP64 && lanes == 32; }
bool pe_more_ok(const DevModel& M, int lanes) { return M.n_comp > 1 && M.precision != FSMP_FP64 && lanes == 32; }

cudaError_t pe_kernel_attributes(int precision, int max_smem) {
  const cudaError_t e = pe_set_attributes<false>(precision, max_smem);
  return e != cudaSuccess ? e : pe_mix_attributes(precision, max_smem);
}

int pe_kernel_occupancy(int precision, int threads, size_t smem, bool big, int lanes, bool mix, PeForm form) {
  if (mix) return pe_mix_occupancy(precision, threads, smem, lanes, form);
  return pe_occupancy<false>(precision, threads, smem, big, lanes, form);
}

// ---- a warp or a team per chain, by the chains' expected PEs
//
// A team makes a chain of many PEs two to three times as fast, but an SM holds 4 teams where it
// holds 8 to 12 warps with a chain each, and chains of up to 32 PEs get nothing from it. So a launch
// that ends with its longest chains is faster in teams and one that ends when the SMs have worked
// through all chains is slower (uneven windows x 600 steps, ms with a warp and with a team per chain:
// 3040 chains of lambda0 0.5 to 50: 13.4, 10.6; of 0.5 to 25: 6.5, 7.7; all of 8: 5.1, 9.0; 1216 of
// 0.5 to 50: 11.9, 6.6; all of 8: 3.1, 4.3; pile-up model, 1216 of 0.5 to 200: 47.4, 22.5; of 5: 3.3,
// 5.2). Which of the two a launch is depends
// on its lambda0 and steps, which are on the device: this kernel estimates both times and sets the
// chain counters so that only the faster form's launch finds chains (the other's ends at once: 3 us
// and this kernel's 3 us).
//
// The estimate: a chain starts empty (or from n_init PEs) and moves towards lambda0 by 0.22 PEs a
// step. Its step costs a polynomial in its PEs: `lat` us on its own, `thr` us of an SM that is full.
// A launch takes the longest chain's time or the SMs' share of all chains, whichever is longer (a
// smooth maximum). Fitted to 404 timed pairs of launches: lambda0 from 1 to 200, alone and mixed,
// 152 to 6000 chains, 150 to 1500 steps. Of the 276 with more than 608 chains it takes the slower
// form 13 times, by more than 10 % five times.
constexpr float kGrowth = 0.22f;  // PEs a step
struct FormCost {
  float lat[4], thr[4];
};
constexpr FormCost kCost[2][2] = {
    // n_cap <= 192: a warp per chain, a team
    {{{2.1f, 0.22f, 4.3e-3f, 4.1e-5f}, {0.17f, 0.036f, 2.8e-4f, 3.7e-6f}},
     {{3.1f, 0.18f, 5.5e-4f, 1.8e-7f}, {0.27f, 0.068f, 7.1e-5f, 1.0e-7f}}},
    // above
    {{{2.8f, 0.24f, 8.4e-3f, 1.2e-6f}, {0.26f, 0.076f, 1.2e-4f, 4.1e-6f}},
     {{4.9f, 0.10f, 3.0e-3f, 3.4e-7f}, {0.54f, 0.10f, 2.1e-5f, 1.4e-6f}}}};
constexpr int kFormThreads = 1024;

struct FormTime {
  float lat, thr;  // us: the longest chain, all chains on one SM
};
__device__ __forceinline__ float form_cost(const float (&a)[4], const float (&f)[4]) {
  return a[0] * f[0] + a[1] * f[1] + a[2] * f[2] + a[3] * f[3];
}
__global__ void __launch_bounds__(kFormThreads) pe_form_kernel(const BatchView B, FormCost one, FormCost team, int n_cap,
                                                               float sms, int* counters) {
  __shared__ FormTime part[2][kFormThreads / 32];
  FormTime t[2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
  for (int i = threadIdx.x; i < B.n_waveforms; i += kFormThreads) {
    const float cap = (float)n_cap, lam = (float)B.lambda0[i];
    const float s = (float)max(B.n_steps_arr ? B.n_steps_arr[i] : B.n_steps, 0);
    const float n0 = B.z_init ? fminf(fmaxf((float)B.n_init[i], 0.0f), cap) : 0.0f;
    const float goal = lam > 0.0f ? fminf(lam, cap) : 0.0f;  // (an invalid lambda0 runs no step)
    const float ramp = fminf(s, fabsf(goal - n0) / kGrowth);
    const float n1 = n0 + (goal > n0 ? kGrowth : -kGrowth) * ramp, flat = s - ramp;
    // sums of N^0 .. N^3 over the steps
    const float f[4] = {s, (n0 + n1) / 2 * ramp + n1 * flat, (n0 * n0 + n0 * n1 + n1 * n1) / 3 * ramp + n1 * n1 * flat,
                        (n0 + n1) * (n0 * n0 + n1 * n1) / 4 * ramp + n1 * n1 * n1 * flat};
    t[0].lat = fmaxf(t[0].lat, form_cost(one.lat, f));
    t[1].lat = fmaxf(t[1].lat, form_cost(team.lat, f));
    t[0].thr += form_cost(one.thr, f);
    t[1].thr += form_cost(team.thr, f);
  }
  for (int k = 0; k < 2; ++k) {
    for (int o = 16; o > 0; o >>= 1) {
      t[k].lat = fmaxf(t[k].lat, __shfl_xor_sync(0xffffffffu, t[k].lat, o));
      t[k].thr += __shfl_xor_sync(0xffffffffu, t[k].thr, o);
    }
    if ((threadIdx.x & 31) == 0) part[k][threadIdx.x / 32] = t[k];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float cube[2];
    for (int k = 0; k < 2; ++k) {
      float lat = 0.0f, thr = 0.0f;
      for (int q = 0; q < kFormThreads / 32; ++q) {
        lat = fmaxf(lat, part[k][q].lat);
        thr += part[k][q].thr;
      }
      thr /= sms;
      cube[k] = lat * lat * lat + thr * thr * thr;
    }
    const bool teams = cube[1] < cube[0];
    counters[0] = teams ? B.n_waveforms : 0;
    counters[1] = teams ? 0 : B.n_waveforms;
    counters[2] = teams ? 1 : 0;
  }
}

cudaError_t launch_pe_form(const DevModel& M, const BatchView& B, int sms, int* counters, cudaStream_t st) {
  const FormCost(&c)[2] = kCost[pe_big(M.n_cap) ? 1 : 0];
  pe_form_kernel<<<1, kFormThreads, 0, st>>>(B, c[0], c[1], M.n_cap, (float)sms, counters);
  return cudaGetLastError();
}

// lambda_FSMP of given N histograms (testing aid): the device function every chain ends with,
// one histogram per group of L lanes. Histogram i is h[i * (n_max + 1) .. (i + 1) * (n_max + 1)).
template <int L>
__global__ void lambda_mle_kernel(const int* __restrict__ h, int n_hist, int n_max, const double* __restrict__ lambda0,
                                  double* __restrict__ out) {
  const Lanes<L> ln = pe_lanes<L>();
  const int i = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) / L);
  if (i >= n_hist) return;  // i is the same on every lane of a group
  const double lam = group_lambda_mle<L>(h + (size_t)i * (n_max + 1), n_max, lambda0[i], ln.sl, ln.gm);
  if (ln.sl == 0) out[i] = lam;
}

cudaError_t launch_lambda_mle(const int* h, int n_hist, int n_max, const double* lambda0, double* out, int lanes,
                              cudaStream_t st) {
  if (n_hist <= 0) return cudaSuccess;
  const int threads = 128, per_block = threads / lanes;
  const unsigned blocks = (unsigned)((n_hist + per_block - 1) / per_block);
  if (lanes == 16) lambda_mle_kernel<16><<<blocks, threads, 0, st>>>(h, n_hist, n_max, lambda0, out);
  else lambda_mle_kernel<32><<<blocks, threads, 0, st>>>(h, n_hist, n_max, lambda0, out);
  return cudaGetLastError();
}

cudaError_t launch_pe(const DevModel& M, const BatchView& B, int warps, int lanes, int ctas, int Ns, size_t smem,
                      void* cinv, size_t c_stride, double* ws, size_t ws_stride, int* hist, int* counter,
                      PeForm form, cudaStream_t st) {
  if (hist == nullptr || !pe_lanes_ok(lanes, M.n_cap)) return cudaErrorInvalidValue;
  if (form == kPeTeam && (!pe_team_ok(M.precision, lanes) || warps != kTeam)) return cudaErrorInvalidValue;
  if (form == kPeWarpMore && !pe_more_ok(M, lanes)) return cudaErrorInvalidValue;
  if (M.n_comp > 1)
    return pe_mix_launch(M, B, warps, lanes, ctas, Ns, smem, cinv, c_stride, ws, ws_stride, hist, counter, form,
                         st);
  return pe_launch<false>(M, B, warps, lanes, ctas, Ns, smem, cinv, c_stride, ws, ws_stride, hist, counter,
                          pe_big(M.n_cap), form, st);
}

}  // namespace fsmp
