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
