// tkf_states.cu -- the all-states output: the Rauch-Tung-Striebel backward pass (paper Sec. 2:
// the smoother makes every state use every measurement) over the states the forward fit
// stored, so that every entry of every track gets its smoothed parameters and covariance.
//
// The first-surface result of tkf_fit needs no stored states (the smoother is evaluated
// forward there); this pass is what an all-states request adds. Per track, k = N-2 .. 0:
//   A_k    = Cf_k J_{k+1}^T Cp_{k+1}^-1                  (Cp_{k+1} by its L D L^T factor)
//   ps_k   = pf_k + A_k (ps_{k+1} - pp_{k+1})            (phi difference wrapped)
//   Cs_k   = Cf_k + A_k (Cs_{k+1} - Cp_{k+1}) A_k^T
// with the filtered state (pf, Cf) read from the all-states arrays, where the forward pass left
// it, and the predicted state (pp, Cp) and transport Jacobian J from the workspace. Each result
// overwrites the filtered state it came from; the last entry's smoothed state is its filtered
// one. FP64 throughout (the paper attributes its FP32 fit's mismatch to this smoother).
//
// Bound by the FP64 pipe (90 % busy; an entry is 0.9 KB of traffic and about 510 FP64 instructions, 420 with
// FP64 states, against 609 with square roots, divisions and full Jacobian rows): Cp is factored as
// L D L^T with reciprocals by rcp_nr, row 4 of J and, in a field along z, row 3 have one and two terms;
// records move in 16-byte loads. 100,000 mixed tracks of 9.8 entries: 1.08 -> 0.92 ms.

#include "tkf_fp64.cuh"
#include "tkf_internal.cuh"

namespace tkf {
namespace {

constexpr uint32_t kFatal = ~(TKF_TRACK_TOO_FEW_HITS | TKF_TRACK_OUT_OF_FIELD | TKF_TRACK_PROPOSAL_FALLBACK);

__host__ __device__ constexpr int P(int i, int j) { return i <= j ? i * (9 - i) / 2 + j : j * (9 - j) / 2 + i; }

__device__ __forceinline__ double wrap_pi(double x) {
  if (x > kPi) x -= 2.0 * kPi;
  if (x <= -kPi) x += 2.0 * kPi;
  return x;
}

__device__ void nan_entries(const FitArgs& a, uint32_t b0, uint32_t b1) {
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  const size_t nm = size_t(a.n_meas);
  for (uint32_t e = b0; e < b1; ++e) {
    for (int j = 0; j < 5; ++j) a.states_par[size_t(j) * nm + e] = nan;
    for (int j = 0; j < 15; ++j) a.states_cov[size_t(j) * nm + e] = nan;
  }
}

// Thread k takes track perm[k]: the fit's order (most entries first), so that the lanes of a warp
// run backward passes of the same length.
template <bool kAxial, bool kRow4>
__global__ void __launch_bounds__(128) smooth_states_kernel(FitArgs a, const uint32_t* __restrict__ perm) {
  const size_t nm = size_t(a.n_meas);
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < a.n_tracks; k += gridDim.x * blockDim.x) {
    const uint32_t i = perm[k];
    const uint32_t b0 = a.offsets[i], b1 = a.offsets[i + 1];
    if (b1 < b0 || b1 > a.n_meas) continue;  // bad offsets: the track has no entries to write
    const uint32_t N = b1 - b0;
    if (N == 0) continue;
    uint32_t M = 0;
    for (uint32_t e = b0; e < b1; ++e) M += (a.sid[e] & TKF_SID_NO_MEASUREMENT) ? 0u : 1u;
    const uint32_t status = a.status[i];
    if (M == 0 || (status & kFatal)) {  // no fit (the seed was returned), or a failed one
      nan_entries(a, b0, b1);
      continue;
    }
    double ps[5], Cs[15];
    for (int j = 0; j < 5; ++j) ps[j] = a.states_par[size_t(j) * nm + b1 - 1];
    for (int j = 0; j < 15; ++j) Cs[j] = a.states_cov[size_t(j) * nm + b1 - 1];
    bool spd = true;
    for (int k = int(N) - 2; k >= 0 && spd; --k) {
      const uint32_t e = b0 + uint32_t(k);
      const double2* w = reinterpret_cast<const double2*>(a.states_scratch + size_t(e + 1) * kStatesScratch);
      double pf[5], Cf[15], rec[40];
#pragma unroll
      for (int j = 0; j < 20; ++j) {
        const double2 x = w[j];
        rec[2 * j] = x.x;
        rec[2 * j + 1] = x.y;
      }
#pragma unroll
      for (int j = 0; j < 5; ++j) pf[j] = a.states_par[size_t(j) * nm + e];
#pragma unroll
      for (int j = 0; j < 15; ++j) Cf[j] = a.states_cov[size_t(j) * nm + e];
      const double *pp = rec, *Cp = rec + 5, *J = rec + 20;
      // B = J Cf, then X = Cp^-1 B = A^T (Cp, Cf symmetric); row 4 of J is e_4. With kRow4 (FP64
      // states) row 4 of A (column 4 of X) is e_4 too: A J = I - Q (Cf + Q)^-1, and the process noise Q
      // has no q/p element. The mixed path's Cp carries FP32 rounding, which only the full A sees through
      // consistently (1e-8 of the covariance otherwise).
      constexpr int kC = kRow4 ? 4 : 5;  // columns of X to solve for
      double X[5][5];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < kC; ++c) {
          const bool two = kAxial && r == 3;  // the row's first three elements are zeros
          double acc = two ? J[18] * Cf[P(3, c)] : J[5 * r] * Cf[P(0, c)];
#pragma unroll
          for (int q = two ? 4 : 1; q < 5; ++q) acc = fma(J[5 * r + q], Cf[P(q, c)], acc);
          X[r][c] = acc;
        }
#pragma unroll
      for (int c = 0; c < kC; ++c) X[4][c] = Cf[P(4, c)];
      // Cp = L D L^T (unit L below the diagonal), with the reciprocals of D
      double L[5][5], inv[5];
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        double t[5];  // L[c][q] D[q]
        double d = Cp[P(c, c)];
#pragma unroll
        for (int q = 0; q < c; ++q) {
          t[q] = L[q][c];
          L[c][q] = t[q] * inv[q];
          d = fma(-t[q], L[c][q], d);
        }
        spd = spd && d > 0.0;
        inv[c] = d > 1e-290 && d < 1e290 ? rcp_nr(d) : 1.0 / d;
#pragma unroll
        for (int r = c + 1; r < 5; ++r) {  // row c above the diagonal: D[c] L[r][c]
          double acc = Cp[P(c, r)];
#pragma unroll
          for (int q = 0; q < c; ++q) acc = fma(-L[c][q], L[q][r], acc);
          L[c][r] = acc;
        }
      }
      if (!spd) break;
#pragma unroll
      for (int c = 0; c < kC; ++c) {  // solve L D L^T x = column c of B
#pragma unroll
        for (int r = 1; r < 5; ++r)
#pragma unroll
          for (int q = 0; q < r; ++q) X[r][c] = fma(-L[r][q], X[q][c], X[r][c]);
#pragma unroll
        for (int r = 0; r < 5; ++r) X[r][c] *= inv[r];
#pragma unroll
        for (int r = 3; r >= 0; --r)
#pragma unroll
          for (int q = r + 1; q < 5; ++q) X[r][c] = fma(-L[q][r], X[q][c], X[r][c]);
      }
      // A = X^T: A[r][c] = X[c][r]
      double dp[5];
      for (int j = 0; j < 5; ++j) dp[j] = ps[j] - pp[j];
      dp[2] = wrap_pi(dp[2]);
#pragma unroll
      for (int r = 0; r < kC; ++r) {
        double acc = pf[r];
#pragma unroll
        for (int c = 0; c < 5; ++c) acc = fma(X[c][r], dp[c], acc);
        ps[r] = acc;
      }
      if (kRow4) ps[4] = pf[4] + dp[4];
      ps[2] = wrap_pi(ps[2]);
      // Cs = Cf + A (Cs - Cp) A^T: G = A D (5 x 5), then the upper triangle of G A^T
      double D[15];
#pragma unroll
      for (int j = 0; j < 15; ++j) D[j] = Cs[j] - Cp[j];
#pragma unroll
      for (int r = 0; r < kC; ++r) {
        double G[5];
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          double acc = X[0][r] * D[P(0, c)];
#pragma unroll
          for (int q = 1; q < 5; ++q) acc = fma(X[q][r], D[P(q, c)], acc);
          G[c] = acc;
        }
#pragma unroll
        for (int c = r; c < kC; ++c) {
          double acc = Cf[P(r, c)];
#pragma unroll
          for (int q = 0; q < 5; ++q) acc = fma(G[q], X[q][c], acc);
          Cs[P(r, c)] = acc;
        }
        if (kRow4) Cs[P(r, 4)] = Cf[P(r, 4)] + G[4];
      }
      if (kRow4) Cs[P(4, 4)] = Cf[P(4, 4)] + D[P(4, 4)];
      for (int j = 0; j < 5; ++j) a.states_par[size_t(j) * nm + e] = ps[j];
      for (int j = 0; j < 15; ++j) a.states_cov[size_t(j) * nm + e] = Cs[j];
    }
    if (!spd) {  // a predicted covariance that is not positive definite: the track fails
      const double nan = __longlong_as_double(0x7ff8000000000000LL);
      a.status[i] = status | TKF_TRACK_SMOOTHER_NOT_SPD;
      for (int j = 0; j < 5; ++j) a.par[size_t(j) * a.stride + i] = nan;
      for (int j = 0; j < 15; ++j) a.cov[size_t(j) * a.stride + i] = nan;
      a.chi2[i] = nan;
      nan_entries(a, b0, b1);
    }
  }
}

}  // namespace

cudaError_t launch_smooth_states(const FitArgs& a, const uint32_t* perm, bool axial, bool fp64,
                                 cudaStream_t stream) {
  if (a.n_tracks == 0) return cudaSuccess;
  const unsigned blocks = (a.n_tracks + 127) / 128;
  if (axial && fp64)
    smooth_states_kernel<true, true><<<blocks, 128, 0, stream>>>(a, perm);
  else if (axial)
    smooth_states_kernel<true, false><<<blocks, 128, 0, stream>>>(a, perm);
  else if (fp64)
    smooth_states_kernel<false, true><<<blocks, 128, 0, stream>>>(a, perm);
  else
    smooth_states_kernel<false, false><<<blocks, 128, 0, stream>>>(a, perm);
  return cudaGetLastError();
}

}  // namespace tkf
