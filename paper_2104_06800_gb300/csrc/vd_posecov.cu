// Pose covariance from the P3P samples (Sec. III-A "Uncertainty-aware Pose
// Estimation"): an iterative Gaussian fit in se(3) with 3-sigma rejection and
// an eigenvalue floor, one warp per frame, float64.
//
// Lane l owns samples l, l + 32, ... (at most 8 with 256 samples), staged in
// shared memory with their coordinates at the current mean.  Sums over the
// samples are reduce-scatters over the lanes in a fixed order, their results
// broadcast, so all lanes hold bit-identical totals and take the same
// decisions without a barrier.
//
// Bound: the number of float64 instructions of one warp, 64 cycles each on
// this GPU however many lanes are active, on as many SMs as frames.  So the
// small algebra is spread over lanes (a row, column or entry of a 6x6 matrix
// each) in place of all of it in every lane, and coordinates at a mean are
// formed once.  After a 1216 x 368 window of 6 frames, with the visibility
// score: 1504 -> 918 us per call pair (the covariance alone 1.45 -> 0.84 ms).
#include "vd_device.cuh"
#include "vd_geom64.cuh"

#define PC_MAX_ROUNDS 50
#define PC_MEAN_ITERS 50
#define PC_MEAN_TOL 1e-12
#define PC_MIN_INLIERS 7
#define PC_PER_LANE (VD_MAX_SAMPLES / 32)

#define PC_FULL 0xffffffffu

__device__ __forceinline__ double pc_warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(PC_FULL, v, o);
  return v;
}

// acc[0 .. N-1] of every lane (N = 8 or 32) -> the warp's sum of acc[lane /
// (32 / N)], the order of a butterfly over lane bits 4 .. 0.
template <int N>
__device__ __forceinline__ double pc_reduce_scatter(double* acc, int lane) {
#pragma unroll
  for (int s = N / 2, o = 16; s >= 1; s >>= 1, o >>= 1) {
    const bool upper = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const double send = upper ? acc[i] : acc[i + s];
      const double keep = upper ? acc[i + s] : acc[i];
      acc[i] = keep + __shfl_xor_sync(PC_FULL, send, o);
    }
  }
  double v = acc[0];
#pragma unroll
  for (int o = 16 / N; o > 0; o >>= 1) v += __shfl_xor_sync(PC_FULL, v, o);
  return v;
}

// d = log(mu^-1 T) for the 12 doubles of T
__device__ __forceinline__ void pc_coords(const double* mu_inv, const double* T, double* d) {
  double rel[12];
  vd_compose(mu_inv, T, rel);
  vd_se3_log(rel, d);
}

// S <- V diag(max(w, eps)) V^T and Sinv <- S^-1, both 6x6 in shared memory.
// When S - eps I has a Cholesky factor every eigenvalue is already above eps
// and S stays as it is (the inverse from S's own factor); otherwise the
// eigen-decomposition raises the small eigenvalues (every lane computes it).
// sM: 36 doubles of scratch.
//
// Lanes 0-7 factorise S, 8-15 S - eps I, at once: lane 8h + i holds row i (rows
// 6 and 7 repeat row 5).
__device__ void pc_floor(double* S, double* Sinv, double* sM, double eps, int lane) {
  const int i = min(lane & 7, 5), base = lane & 8;
  double a[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) a[j] = S[6 * i + j] - (base && i == j ? eps : 0.0);
  bool ok = true;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
#pragma unroll
    for (int k = 0; k < j; ++k) a[j] -= a[k] * __shfl_sync(PC_FULL, a[k], base + j);
    const double d = __shfl_sync(PC_FULL, a[j], base + j);
    ok = ok && d > 0.0;
    const double ljj = sqrt(d);
    a[j] = i == j ? ljj : a[j] / ljj;          // rows above j are not read again
  }
  if (__all_sync(PC_FULL, ok || lane >= 16)) {
    // column c of M = L^-1 in lane c
    const int c = i;
    double m[6];
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      double v = 0.0;
#pragma unroll
      for (int k = 0; k < r; ++k) v -= __shfl_sync(PC_FULL, a[k], r) * m[k];
      const double num = r == c ? 1.0 : (r > c ? v : 0.0);
      m[r] = num / __shfl_sync(PC_FULL, a[r], r);
    }
    __syncwarp();
    if (lane < 6)
#pragma unroll
      for (int r = 0; r < 6; ++r) sM[6 * r + c] = m[r];
    __syncwarp();
    // entry (p, q), q >= p, of L^-T L^-1 in lane 0 .. 20
    if (lane < 21) {
      int p = 0, q = lane;
      while (q >= 6 - p) q -= 6 - p++;
      q += p;
      double v = 0.0;
      for (int k = q; k < 6; ++k) v += sM[6 * k + p] * sM[6 * k + q];
      Sinv[6 * p + q] = v;
      Sinv[6 * q + p] = v;
    }
    __syncwarp();
    return;
  }
  double A[36], w[6], V[36];
  for (int k = 0; k < 36; ++k) A[k] = S[k];
  __syncwarp();
  vd_jacobi_eig<6>(A, w, V);
  for (int k = 0; k < 6; ++k) w[k] = fmax(w[k], eps);
  for (int r = 0; r < 6; ++r)
    for (int j = 0; j < 6; ++j) {
      double s = 0.0, si = 0.0;
      for (int k = 0; k < 6; ++k) {
        s += V[6 * r + k] * w[k] * V[6 * j + k];
        si += V[6 * r + k] / w[k] * V[6 * j + k];
      }
      if (lane == 0) {
        S[6 * r + j] = s;
        Sinv[6 * r + j] = si;
      }
    }
  __syncwarp();
}

// out[52 t']: mean (12), cov (36), n_samples, n_inliers, rounds, degenerate
__global__ void __launch_bounds__(32)
k_pose_cov(DevParams P, const double* __restrict__ G, const double* __restrict__ sample_pose,
           const double* __restrict__ sample_energy, double eps, double* __restrict__ out) {
  const int t = blockIdx.x + 1;
  const int lane = threadIdx.x;
  const double* Ts = sample_pose + (size_t)(t - 1) * VD_MAX_SAMPLES * 12;
  const double* Es = sample_energy + (size_t)(t - 1) * VD_MAX_SAMPLES;
  __shared__ double T[VD_MAX_SAMPLES][12];   // sample g = lane + 32 k at row g
  unsigned valid = 0;
  int nv = 0;
  for (int k = 0; k < PC_PER_LANE; ++k) {
    const int g = lane + 32 * k;
    const bool ok = g < P.S && Es[g] < INFINITY;
    for (int i = 0; i < 12; ++i) T[g][i] = ok ? Ts[12 * g + i] : 0.0;
    valid |= (unsigned)ok << k;
    nv += ok;
  }
  const int n_samples = (int)pc_warp_sum((double)nv);
  __shared__ double D[VD_MAX_SAMPLES][6];    // the samples' coordinates at the mean
  __shared__ double S[36], Sinv[36], sM[36], sMu[12], sE[12];
  __shared__ unsigned char sV[VD_MAX_SAMPLES];
  double mu[12], mi[12];
  for (int i = 0; i < 12; ++i) mu[i] = G[12 * t + i];
  for (int i = lane; i < 36; i += 32) S[i] = 0.0;
  __syncwarp();
  int rounds = 0, n_in = n_samples, degenerate = n_samples < PC_MIN_INLIERS;
  // each lane reads back only its own rows of D
  auto coords_all = [&]() {
    vd_inverse(mu, mi);
    for (int k = 0; k < PC_PER_LANE; ++k) {
      if (!(valid >> k & 1u)) continue;
      double d[6];
      pc_coords(mi, T[lane + 32 * k], d);
      for (int i = 0; i < 6; ++i) D[lane + 32 * k][i] = d[i];
    }
  };
  if (!degenerate) {
    // robust start: diag((1.4826 median_g |d_gi|)^2) at the mode, the
    // medians selected by rank among the valid samples (exact, no arithmetic)
    coords_all();
    for (int k = 0; k < PC_PER_LANE; ++k)
      sV[lane + 32 * k] = (unsigned char)(valid >> k & 1u);
    __syncwarp();   // every lane's coordinates and flags before the ranks
    const int r1 = (n_samples - 1) / 2, r2 = n_samples / 2;   // middle ranks
    for (int i = 0; i < 6; ++i) {
      double m1 = -1.0, m2 = -1.0;
      for (int k = 0; k < PC_PER_LANE; ++k) {
        if (!(valid >> k & 1u)) continue;
        const int g = lane + 32 * k;
        const double a = fabs(D[g][i]);
        int rank = 0;   // valid samples before g in (value, index) order
        for (int h = 0; h < P.S; ++h) {
          if (!sV[h]) continue;
          const double b = fabs(D[h][i]);
          rank += (b < a) || (b == a && h < g);
        }
        if (rank == r1) m1 = a;
        if (rank == r2) m2 = a;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        m1 = fmax(m1, __shfl_xor_sync(PC_FULL, m1, o));
        m2 = fmax(m2, __shfl_xor_sync(PC_FULL, m2, o));
      }
      const double s = 1.4826 * ((m1 + m2) / 2.0);
      if (lane == 0) S[7 * i] = s * s;
    }
    __syncwarp();
  }
  pc_floor(S, Sinv, sM, eps, lane);
  unsigned prev = 0;
  if (!degenerate) {
    for (int r = 1; r <= PC_MAX_ROUNDS; ++r) {
      rounds = r;
      unsigned inl = 0;
      int ni = 0;
      for (int k = 0; k < PC_PER_LANE; ++k) {
        if (!(valid >> k & 1u)) continue;
        const double* d = D[lane + 32 * k];
        double m = 0.0;
        for (int i = 0; i < 6; ++i) {
          double row = 0.0;
          for (int j = 0; j < 6; ++j) row += Sinv[6 * i + j] * d[j];
          m += d[i] * row;
        }
        if (m <= 9.0) {
          inl |= 1u << k;
          ++ni;
        }
      }
      n_in = __reduce_add_sync(PC_FULL, ni);
      if (r > 1 && !__any_sync(PC_FULL, inl != prev)) break;   // the same inlier set
      if (n_in < PC_MIN_INLIERS) {
        degenerate = 1;
        break;
      }
      // Frechet mean of the inliers (the first step from the coordinates in D)
      for (int it = 0; it < PC_MEAN_ITERS; ++it) {
        if (it > 0) vd_inverse(mu, mi);
        double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int k = 0; k < PC_PER_LANE; ++k) {
          if (!(inl >> k & 1u)) continue;
          double d[6];
          if (it > 0) {
            pc_coords(mi, T[lane + 32 * k], d);
          } else {
            for (int i = 0; i < 6; ++i) d[i] = D[lane + 32 * k][i];
          }
          for (int i = 0; i < 6; ++i) acc[i] += d[i];
        }
        const double mean = pc_reduce_scatter<8>(acc, lane) / n_in;
        double step[6], nrm = 0.0;
        for (int i = 0; i < 6; ++i) {
          step[i] = __shfl_sync(PC_FULL, mean, 4 * i);
          nrm += step[i] * step[i];
        }
        double E[12];
        vd_se3_exp(step, E);
        // mu <- mu o E, an entry per lane
        __syncwarp();
        if (lane == 0)
          for (int i = 0; i < 12; ++i) {
            sMu[i] = mu[i];
            sE[i] = E[i];
          }
        __syncwarp();
        const int row = min(lane >> 2, 2), col = lane & 3;
        const double* m = sMu + 4 * row;
        double v = m[0] * sE[col] + m[1] * sE[4 + col] + m[2] * sE[8 + col];
        if (col == 3) v += m[3];
        for (int i = 0; i < 12; ++i) mu[i] = __shfl_sync(PC_FULL, v, i);
        if (sqrt(nrm) < PC_MEAN_TOL) break;
      }
      // maximum-likelihood covariance at the mean, eigenvalues floored
      coords_all();
      double acc[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) acc[i] = 0.0;
      for (int k = 0; k < PC_PER_LANE; ++k) {
        if (!(inl >> k & 1u)) continue;
        const double* d = D[lane + 32 * k];
#pragma unroll
        for (int i = 0, q = 0; i < 6; ++i)
#pragma unroll
          for (int j = i; j < 6; ++j, ++q) acc[q] += d[i] * d[j];
      }
      const double v = pc_reduce_scatter<32>(acc, lane) / n_in;
      if (lane < 21) {
        int p = 0, q = lane;
        while (q >= 6 - p) q -= 6 - p++;
        q += p;
        S[6 * p + q] = v;
        S[6 * q + p] = v;
      }
      __syncwarp();
      pc_floor(S, Sinv, sM, eps, lane);
      prev = inl;
    }
  }
  if (lane == 0) {
    double* o = out + 52 * (t - 1);
    for (int i = 0; i < 12; ++i) o[i] = mu[i];
    for (int i = 0; i < 36; ++i) o[12 + i] = S[i];
    o[48] = n_samples;
    o[49] = n_in;
    o[50] = rounds;
    o[51] = degenerate;
  }
}

extern "C" vd_status vd_pose_covariance(vd_ctx* c, double eps, vd_pose_cov* out) {
  if (!c || !out || !(eps > 0.0) || !isfinite(eps)) return VD_ERR_ARG;
  if (c->samples_set != (1u << c->N) - 1u) {
    vd_set_error("every frame needs a pose M-step first");
    return VD_ERR_STATE;
  }
  k_pose_cov<<<c->N, 32, 0, c->stream>>>(c->dp, c->G, c->sample_pose, c->sample_energy, eps,
                                         c->pc_out);
  VD_CU(cudaGetLastError());
  double h[52 * VD_MAX_FLOWS];
  VD_CU(cudaMemcpyAsync(h, c->pc_out, sizeof(double) * 52 * c->N, cudaMemcpyDeviceToHost,
                        c->stream));
  VD_CU(cudaStreamSynchronize(c->stream));
  for (int t = 0; t < c->N; ++t) {
    const double* o = h + 52 * t;
    vd_pose_cov& r = out[t];
    for (int i = 0; i < 12; ++i) r.mean[i] = o[i];
    for (int i = 0; i < 36; ++i) r.cov[i] = o[12 + i];
    r.n_samples = (int)o[48];
    r.n_inliers = (int)o[49];
    r.rounds = (int)o[50];
    r.degenerate = (int)o[51];
  }
  return VD_OK;
}

extern "C" vd_status vd_get_frame_samples(vd_ctx* c, int t, double* poses, double* energies) {
  if (!c || t < 1 || t > c->N) return VD_ERR_ARG;
  if (!(c->samples_set >> (t - 1) & 1u)) {
    vd_set_error("frame has no pose M-step yet");
    return VD_ERR_STATE;
  }
  const int S = c->prm.n_pose_samples;
  const size_t f = (size_t)(t - 1) * VD_MAX_SAMPLES;
  if (poses)
    VD_CU(cudaMemcpyAsync(poses, c->sample_pose + 12 * f, sizeof(double) * 12 * S,
                          cudaMemcpyDeviceToHost, c->stream));
  if (energies)
    VD_CU(cudaMemcpyAsync(energies, c->sample_energy + f, sizeof(double) * S,
                          cudaMemcpyDeviceToHost, c->stream));
  VD_CU(cudaStreamSynchronize(c->stream));
  return VD_OK;
}

VD_CHECK_ACCESSOR(posecov)
