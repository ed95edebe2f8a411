// FP64 red-black Gauss-Seidel cycle kernels (A = I).  The FP64 path is bound by the FP64 unit (one
// warp instruction per 64 clocks and SM sub-partition), so these forms leave out work whose
// result is known:
//   * after a red-black sweep the residual of the black nodes is zero but for rounding, so the
//     restriction forms the red nodes' residuals only (2D: three in place of seven per coarse
//     node, 3D: seven in place of fifteen);
//   * before a black-red sweep the prolongation corrects the red nodes only: the sweep's first half
//     replaces every black value from its red neighbours;
//   * products by powers of two are exponent additions.
// On 2D levels of up to kFused64 cells per side, where a half sweep is little more than a launch, a
// level's pre-smoothing with its restriction, and its prolongation with its post-smoothing, are one
// launch each: a block works on a tile plus a halo as deep as its sweeps reach, in shared memory.
#include <cuda_runtime.h>

#include <vector>

#include "fmg_internal.cuh"
#include "fmg_phase.cuh"

namespace fmg {

namespace {

constexpr int kRB = 128;    // threads per block of the per-level kernels
constexpr int kRT = 256;    // threads per block of the tile kernels

inline unsigned cdiv(long long a, long long b) { return (unsigned)((a + b - 1) / b); }

// b - A u at an interior node, 2D: (b + sum of neighbours) - 4 u.
__device__ __forceinline__ double res2(const double* __restrict__ u, const double* __restrict__ b, long long c,
                                       long long np) {
  return fma(-4.0, u[c], b[c] + ((u[c - 1] + u[c + 1]) + (u[c - np] + u[c + np])));
}

// ------------------------------------------------------------------ half sweeps
// One colour in 2D, S rows per thread: the rows' loads (b and the four neighbours, all of the other
// colour) are issued together.  One node per thread took 23.8 us at 2049^2, 5 FP64 operations
// with the product by 1/4; this 20.6, 4 operations (13.3 at the FP64 rate).
template <int S>
__device__ __forceinline__ void k_rbgs2_strip_body(double* __restrict__ u, const double* __restrict__ b, int n,
                                                   int colour) {
  const int j0 = blockIdx.y * S + 1;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const long long np = n + 1;
  double v[S];
  long long c[S];
  bool on[S];
  double q[S][5];
#pragma unroll
  for (int r = 0; r < S; ++r) {
    const int j = j0 + r;
    const int i = ((colour + j) & 1) ? 2 * t + 1 : 2 * t + 2;
    on[r] = i <= n - 1 && j <= n - 1;
    c[r] = on[r] ? (long long)j * np + i : np + 1;
    q[r][0] = u[c[r] - 1];
    q[r][1] = u[c[r] + 1];
    q[r][2] = u[c[r] - np];
    q[r][3] = u[c[r] + np];
    q[r][4] = b[c[r]];
  }
#pragma unroll
  for (int r = 0; r < S; ++r) v[r] = quarter(q[r][4] + ((q[r][0] + q[r][1]) + (q[r][2] + q[r][3])));
#pragma unroll
  for (int r = 0; r < S; ++r)
    if (on[r]) u[c[r]] = v[r];
}
template <int S>
__global__ void __launch_bounds__(kRB) k_rbgs2_strip(double* __restrict__ u, const double* __restrict__ b, int n,
                                                     int colour) {
  pdl_start();
  k_rbgs2_strip_body<S>(u, b, n, colour);
}

// ------------------------------------------------------------------ restriction of red residuals
// 2D: b_c(I, J) = r(2I, 2J) + (r(2I+1, 2J+1) + r(2I-1, 2J-1)) / 2.  The residual at (2I+1, 2J+1) serves
// the coarse nodes (I, J) and (I+1, J+1): a thread walks S coarse rows of a column and takes the
// other one from the lane to its left, one row earlier (a warp's first lane only helps: 31
// columns per warp), so a coarse node costs two residuals, 12 FP64 operations against 49 for the
// seven of the general form.  start: also the coarse level's first red half sweep from zero
// (u_c = b_c / 4 on its red nodes, 0 on the black ones).
template <int S>
__device__ __forceinline__ void k_restrict_rb2_body(const double* __restrict__ u, const double* __restrict__ b,
                                                    int nf, double* __restrict__ bc, double* __restrict__ uc,
                                                    int nc, int start) {
  const int lane = threadIdx.x & 31;
  const int I = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 31 + lane;
  const int J0 = blockIdx.y * S + 1;
  const int J1 = min(J0 + S, nc);
  const long long np = nf + 1;
  const bool din = I < nc;                              // the column of (2I + 1) is interior
  const bool cin = lane > 0 && I >= 1 && I <= nc - 1;   // this thread's coarse column
  auto diag = [&](int J) { return din ? res2(u, b, (long long)(2 * J + 1) * np + 2 * I + 1, np) : 0.0; };
  double dprev = diag(J0 - 1);
#pragma unroll
  for (int k = 0; k < S; ++k) {
    const int J = J0 + k;
    if (J >= J1) break;
    const double d = diag(J);
    const double dm = __shfl_up_sync(0xffffffffu, dprev, 1);
    if (cin) {
      const double r0 = res2(u, b, (long long)(2 * J) * np + 2 * I, np);
      const double v = fma(0.5, d + dm, r0);
      const long long cc = (long long)J * (nc + 1) + I;
      bc[cc] = v;
      if (start) uc[cc] = ((I + J) & 1) ? 0.0 : quarter(v);
    }
    dprev = d;
  }
}
template <int S>
__global__ void k_restrict_rb2(const double* __restrict__ u, const double* __restrict__ b, int nf,
                               double* __restrict__ bc, double* __restrict__ uc, int nc, int start) {
  pdl_start();
  k_restrict_rb2_body<S>(u, b, nf, bc, uc, nc, start);
}

// 3D: the red neighbours of a coarse node are those at +- (1,1,0), (1,0,1), (0,1,1).
__global__ void k_restrict_rb3(const double* __restrict__ u, const double* __restrict__ b, int nf, int lgf,
                               double* __restrict__ bc, double* __restrict__ uc, int nc, int start) {
  pdl_start();
  const int I = blockIdx.x * blockDim.x + threadIdx.x + 1;
  const int J = blockIdx.y + 1;
  const int K = blockIdx.z + 1;
  if (I > nc - 1) return;
  const long long np = nf + 1;
  const long long pl = np * np;
  const long long F = ((long long)(2 * K) * np + 2 * J) * np + 2 * I;
  auto res = [&](long long c) {
    const double s = ((u[c - 1] + u[c + 1]) + (u[c - np] + u[c + np])) + (u[c - pl] + u[c + pl]);
    return b[c] - times_pow2(fma(6.0, u[c], -s), -lgf);
  };
  const double e = ((res(F + 1 + np) + res(F - 1 - np)) + (res(F + 1 + pl) + res(F - 1 - pl))) +
                   (res(F + np + pl) + res(F - np - pl));
  const double v = fma(0.5, e, res(F));
  const long long ncp = nc + 1;
  const long long cc = ((long long)K * ncp + J) * ncp + I;
  bc[cc] = v;
  // the coarse level's red half sweep from zero: u = b n_c / 6
  if (start) uc[cc] = ((I + J + K) & 1) ? 0.0 : times_pow2(v, lgf - 1) * (1.0 / 6.0);
}

// ------------------------------------------------------------------ prolongation onto red nodes
// u += P e_c at the nodes of even i + j [+ l]: where every index is even the coarse value itself,
// else the mean of the two ends of its coarse edge.
__device__ __forceinline__ void k_prolong_rb2_body(const double* __restrict__ e, int nc, double* __restrict__ u) {
  const int nf = 2 * nc;
  const int j = blockIdx.y + 1;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = (j & 1) ? 2 * t + 1 : 2 * t + 2;
  if (i > nf - 1) return;
  const long long cp = nc + 1;
  const long long a = (long long)(j >> 1) * cp + (i >> 1);
  const long long f = (long long)j * (nf + 1) + i;
  if (j & 1)
    u[f] = fma(0.5, e[a] + e[a + cp + 1], u[f]);
  else
    u[f] += e[a];
}
__global__ void k_prolong_rb2(const double* __restrict__ e, int nc, double* __restrict__ u) {
  pdl_start();
  k_prolong_rb2_body(e, nc, u);
}

__global__ void k_prolong_rb3(const double* __restrict__ e, int nc, double* __restrict__ u) {
  pdl_start();
  const int nf = 2 * nc;
  const int j = blockIdx.y + 1, l = blockIdx.z + 1;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = ((j + l) & 1) ? 2 * t + 1 : 2 * t + 2;
  if (i > nf - 1) return;
  const long long cp = nc + 1;
  const long long a = ((long long)(l >> 1) * cp + (j >> 1)) * cp + (i >> 1);
  const long long z = ((long long)((l + 1) >> 1) * cp + ((j + 1) >> 1)) * cp + ((i + 1) >> 1);
  const long long f = ((long long)l * (nf + 1) + j) * (nf + 1) + i;
  if (a == z)
    u[f] += e[a];
  else
    u[f] = fma(0.5, e[a] + e[z], u[f]);
}

// ------------------------------------------------------------------ level start
// u = P u_c (the FMG interpolation) and b = w (g - a f(u)) in one pass; b is zero on the boundary.
// w = 2^wexp when wexp <= 0, else the factor w.
// A thread takes kLS rows (along y in 2D, z in 3D), their loads issued together.
constexpr int kLS = 4;
template <int D>
__device__ __forceinline__ void k_level_start64_body(const double* __restrict__ e, int nc, double* __restrict__ u,
                                                     const double* __restrict__ g, double* __restrict__ b, int kind,
                                                     double a, double w, int wexp) {
  const int n = 2 * nc;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int z0 = (D == 2 ? blockIdx.y : blockIdx.z) * kLS;
  if (i > n) return;
  const long long np = n + 1, cp = nc + 1;
  double ep[kLS], eq[kLS], gv[kLS];
  long long f[kLS];
  int in[kLS];   // 0: past the level, 1: boundary, 2: interior node on a coarse node, 3: between two
#pragma unroll
  for (int r = 0; r < kLS; ++r) {
    const int j = D == 2 ? z0 + r : (int)blockIdx.y, l = D == 3 ? z0 + r : 0;
    f[r] = ((long long)l * np + j) * np + i;
    const bool here = z0 + r <= n;
    const bool inner = here && i > 0 && i < n && j > 0 && j < n && (D == 2 || (l > 0 && l < n));
    const long long p = ((long long)(l >> 1) * cp + (j >> 1)) * cp + (i >> 1);
    const long long q = ((long long)((l + 1) >> 1) * cp + ((j + 1) >> 1)) * cp + ((i + 1) >> 1);
    in[r] = inner ? (p == q ? 2 : 3) : here ? 1 : 0;
    ep[r] = inner ? e[p] : 0.0;
    eq[r] = inner ? e[q] : 0.0;
    gv[r] = inner ? g[f[r]] : 0.0;
  }
#pragma unroll
  for (int r = 0; r < kLS; ++r) {
    if (in[r] < 2) {
      if (in[r] == 1) b[f[r]] = 0.0;
      continue;
    }
    const double v = in[r] == 2 ? ep[r] : times_pow2(ep[r] + eq[r], -1);
    u[f[r]] = v;
    double x;
    if (kind == FMG_F_CUBIC) {
      x = fma(-a, v * v * v, gv[r]);
    } else {
      x = gv[r] - f_only<double>(kind, a, v);
    }
    b[f[r]] = wexp <= 0 ? times_pow2(x, wexp) : w * x;
  }
}
template <int D>
__global__ void k_level_start64(const double* __restrict__ e, int nc, double* __restrict__ u,
                                const double* __restrict__ g, double* __restrict__ b, int kind, double a, double w,
                                int wexp) {
  pdl_start();
  k_level_start64_body<D>(e, nc, u, g, b, kind, a, w, wexp);
}

// ------------------------------------------------------------------ 2D tile kernels
// 8-byte asynchronous global -> shared copy, so that a thread has all its copies in flight at once
// (a loop of loads and stores cost a memory latency per turn: 14 us per launch); zero-fills when off.
__device__ __forceinline__ void cp_async8(double* dst, const double* src, bool on) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(on ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// One colour of a sweep on the local rows and columns lo..hi of a W x W tile whose local (0, 0) is
// global (gx0, gy0); interior nodes only.  The nodes of the region are dealt to the threads in
// one sequence (an FP64 warp instruction costs the same with few lanes as with all).
template <int W>
__device__ __forceinline__ void tile_half64(double* su, const double* sb, int lo, int hi, int colour, int gx0, int gy0,
                                            int n) {
  const int xlo = max(lo, 1 - gx0), xhi = min(hi, n - 1 - gx0);
  const int ylo = max(lo, 1 - gy0), yhi = min(hi, n - 1 - gy0);
  const int cw = (xhi - xlo + 2) >> 1;   // nodes of a colour per row, at most
  if (cw <= 0) return;
  const unsigned magic = ((1u << 20) + cw - 1) / cw;
  const int total = (yhi - ylo + 1) * cw;
  for (int t = threadIdx.x; t < total; t += kRT) {
    const int q = (int)(((unsigned)t * magic) >> 20);
    const int p = t - q * cw;
    const int ly = ylo + q;
    const int lx = xlo + ((colour + gy0 + ly + gx0 + xlo) & 1) + 2 * p;
    if (lx > xhi) continue;
    const int c = ly * W + lx;
    su[c] = quarter(sb[c] + ((su[c - 1] + su[c + 1]) + (su[c - W] + su[c + W])));
  }
}

// NU red-black sweeps on A u = b from u_in (from zero when NULL), then b_c = P^T (b - A u): the red
// residuals of the tile, in shared memory.  u_out and u_in differ (the tiles read each other's
// halo).
template <int NU, int T>
__device__ __forceinline__ void k_pre_rb64_body(const double* __restrict__ u_in, const double* __restrict__ b,
                                                double* __restrict__ u_out, double* __restrict__ bc, int n) {
  constexpr int H = 2 * NU + 2;
  constexpr int W = T + 2 * H;
  constexpr int R = T / 2 + 1;
  extern __shared__ double smd[];
  double* su = smd;
  double* sb = su + W * W;
  double* sd = sb + W * W;   // residuals at (X0 - 1 + 2 i, Y0 - 1 + 2 j)
  const int X0 = blockIdx.x * T, Y0 = blockIdx.y * T;
  const int gx0 = X0 - H, gy0 = Y0 - H;
  const long long np = n + 1;
  for (int t = threadIdx.x; t < W * W; t += kRT) {
    const int ly = t / W, lx = t - ly * W;
    const int gx = gx0 + lx, gy = gy0 + ly;
    const bool on = gx >= 0 && gx <= n && gy >= 0 && gy <= n;
    const long long c = on ? (long long)gy * np + gx : 0;
    cp_async8(&sb[t], b + c, on);
    if (u_in)
      cp_async8(&su[t], u_in + c, on);
    else
      su[t] = 0.0;
  }
  cp_async_wait();
  __syncthreads();
  for (int s = 0; s < 2 * NU; ++s) {
    tile_half64<W>(su, sb, s + 1, W - 2 - s, s & 1, gx0, gy0, n);
    __syncthreads();
  }
  auto res = [&](int c) { return fma(-4.0, su[c], sb[c] + ((su[c - 1] + su[c + 1]) + (su[c - W] + su[c + W]))); };
  for (int t = threadIdx.x; t < R * R; t += kRT) {
    const int j = t / R, i = t - j * R;
    const int gx = X0 - 1 + 2 * i, gy = Y0 - 1 + 2 * j;
    sd[t] = gx > 0 && gx < n && gy > 0 && gy < n ? res((gy - gy0) * W + gx - gx0) : 0.0;
  }
  __syncthreads();
  const int nc = n >> 1;
  for (int t = threadIdx.x; t < (T / 2) * (T / 2); t += kRT) {
    const int j = t / (T / 2), i = t % (T / 2);
    const int I = X0 / 2 + i, J = Y0 / 2 + j;
    if (I < 1 || I > nc - 1 || J < 1 || J > nc - 1) continue;
    bc[(long long)J * (nc + 1) + I] =
        fma(0.5, sd[j * R + i] + sd[(j + 1) * R + i + 1], res((2 * j + H) * W + 2 * i + H));
  }
  for (int t = threadIdx.x; t < T * T; t += kRT) {
    const int ly = t / T, lx = t % T;
    const int gx = X0 + lx, gy = Y0 + ly;
    if (gx > 0 && gx < n && gy > 0 && gy < n) u_out[(long long)gy * np + gx] = su[(ly + H) * W + lx + H];
  }
}
template <int NU, int T>
__global__ void __launch_bounds__(kRT) k_pre_rb64(const double* __restrict__ u_in, const double* __restrict__ b,
                                                  double* __restrict__ u_out, double* __restrict__ bc, int n) {
  pdl_start();
  k_pre_rb64_body<NU, T>(u_in, b, u_out, bc, n);
}

// u_out = NU black-red sweeps on A u = b from u_in + P e_c (the correction on the red nodes).
template <int NU, int T>
__device__ __forceinline__ void k_post_rb64_body(const double* __restrict__ u_in, const double* __restrict__ ec,
                                                 const double* __restrict__ b, double* __restrict__ u_out, int n) {
  constexpr int H = 2 * NU;
  constexpr int W = T + 2 * H;
  extern __shared__ double smd[];
  double* su = smd;
  double* sb = su + W * W;
  const int X0 = blockIdx.x * T, Y0 = blockIdx.y * T;
  const int gx0 = X0 - H, gy0 = Y0 - H;
  const long long np = n + 1, cp = (n >> 1) + 1;
  // the coarse nodes of the tile region, (gx0 / 2 ..) in x and y
  constexpr int CW = W / 2 + 1;
  double* se = sb + W * W;
  const int cx0 = gx0 >> 1, cy0 = gy0 >> 1, nc = n >> 1;
  for (int t = threadIdx.x; t < W * W; t += kRT) {
    const int ly = t / W, lx = t - ly * W;
    const int gx = gx0 + lx, gy = gy0 + ly;
    const bool on = gx >= 0 && gx <= n && gy >= 0 && gy <= n;
    const bool inner = gx > 0 && gx < n && gy > 0 && gy < n;
    const long long c = on ? (long long)gy * np + gx : 0;
    cp_async8(&su[t], (inner ? u_in : u_out) + c, on);   // (the boundary is the result's own)
    cp_async8(&sb[t], b + c, on);
  }
  for (int t = threadIdx.x; t < CW * CW; t += kRT) {
    const int y = t / CW, x = t - y * CW;
    const bool on = cx0 + x >= 0 && cx0 + x <= nc && cy0 + y >= 0 && cy0 + y <= nc;
    cp_async8(&se[t], ec + (on ? (long long)(cy0 + y) * cp + cx0 + x : 0), on);
  }
  cp_async_wait();
  __syncthreads();
  // += P e_c on the red nodes: the coarse value itself, or the mean of a diagonal edge's ends
  for (int t = threadIdx.x; t < W * (W / 2); t += kRT) {
    const int ly = t / (W / 2), lx = 2 * (t - ly * (W / 2)) + ((gx0 + gy0 + ly) & 1);
    const int gx = gx0 + lx, gy = gy0 + ly;
    if (gx > 0 && gx < n && gy > 0 && gy < n) {
      const double* e = se + ((gy >> 1) - cy0) * CW + (gx >> 1) - cx0;
      su[ly * W + lx] = (gx & 1) ? fma(0.5, e[0] + e[CW + 1], su[ly * W + lx]) : su[ly * W + lx] + e[0];
    }
  }
  __syncthreads();
  for (int s = 0; s < 2 * NU; ++s) {
    tile_half64<W>(su, sb, s + 1, W - 2 - s, 1 - (s & 1), gx0, gy0, n);
    __syncthreads();
  }
  for (int t = threadIdx.x; t < T * T; t += kRT) {
    const int ly = t / T, lx = t % T;
    const int gx = X0 + lx, gy = Y0 + ly;
    if (gx > 0 && gx < n && gy > 0 && gy < n) u_out[(long long)gy * np + gx] = su[(ly + H) * W + lx + H];
  }
}
template <int NU, int T>
__global__ void __launch_bounds__(kRT) k_post_rb64(const double* __restrict__ u_in, const double* __restrict__ ec,
                                                   const double* __restrict__ b, double* __restrict__ u_out, int n) {
  pdl_start();
  k_post_rb64_body<NU, T>(u_in, ec, b, u_out, n);
}

template <int NU, int T>
cudaError_t launch_pre(int n, const double* u_in, const double* b, double* u_out, double* bc, cudaStream_t s) {
  constexpr int W = T + 2 * (2 * NU + 2), R = T / 2 + 1;
  const size_t smem = sizeof(double) * (2 * W * W + R * R);
  const unsigned t = cdiv(n + 1, T);
  cudaError_t e = raise_dyn_smem((const void*)k_pre_rb64<NU, T>, smem);
  if (e != cudaSuccess) return e;
  launch_k(k_pre_rb64<NU, T>, dim3(t, t), kRT, smem, s, u_in, b, u_out, bc, n);
  return cudaGetLastError();
}
template <int NU, int T>
cudaError_t launch_post(int n, const double* u_in, const double* ec, const double* b, double* u_out, cudaStream_t s) {
  constexpr int W = T + 4 * NU;
  const size_t smem = sizeof(double) * (2 * W * W + (W / 2 + 1) * (W / 2 + 1));
  const unsigned t = cdiv(n + 1, T);
  cudaError_t e = raise_dyn_smem((const void*)k_post_rb64<NU, T>, smem);
  if (e != cudaSuccess) return e;
  launch_k(k_post_rb64<NU, T>, dim3(t, t), kRT, smem, s, u_in, ec, b, u_out, n);
  return cudaGetLastError();
}

// Cells per side up to which the tile kernels are used, and up to which their tiles are 16^2: a
// level of 128 cells has 64 such tiles, of which each is a third of a 32^2 one's work.
constexpr int kFused64 = 512;
constexpr int kTile16 = 128;

}  // namespace

cudaError_t launch_rbgs2_strip(LevelGeo g, double* u, const double* b, int colour, cudaStream_t s) {
  const dim3 grid(cdiv(g.n / 2, kRB), cdiv(g.n - 1, 4));
  launch_k(k_rbgs2_strip<4>, grid, kRB, 0, s, u, b, g.n, colour);
  return cudaGetLastError();
}

bool fused_rb64_supported(int dim, int n, int nu_pre, int nu_post) {
  return dim == 2 && n <= kFused64 && (n & 1) == 0 && nu_pre >= 1 && nu_pre <= 2 && nu_post >= 1 && nu_post <= 2;
}

cudaError_t launch_pre_rb64(LevelGeo g, int nu, const double* u_in, const double* b, double* u_out, double* bc,
                            cudaStream_t s) {
  if (g.n <= kTile16)
    return nu == 1 ? launch_pre<1, 16>(g.n, u_in, b, u_out, bc, s) : launch_pre<2, 16>(g.n, u_in, b, u_out, bc, s);
  return nu == 1 ? launch_pre<1, 32>(g.n, u_in, b, u_out, bc, s) : launch_pre<2, 32>(g.n, u_in, b, u_out, bc, s);
}

cudaError_t launch_post_rb64(LevelGeo g, int nu, const double* u_in, const double* ec, const double* b, double* u_out,
                             cudaStream_t s) {
  if (g.n <= kTile16)
    return nu == 1 ? launch_post<1, 16>(g.n, u_in, ec, b, u_out, s) : launch_post<2, 16>(g.n, u_in, ec, b, u_out, s);
  return nu == 1 ? launch_post<1, 32>(g.n, u_in, ec, b, u_out, s) : launch_post<2, 32>(g.n, u_in, ec, b, u_out, s);
}

cudaError_t launch_restrict_rb64(int dim, LevelGeo gf, const double* u_f, const double* b_f, LevelGeo gc, double* b_c,
                                 double* u_c, bool start, cudaStream_t s) {
  const int nc = gc.n;
  if (dim == 2) {
    const unsigned warps = cdiv(nc - 1, 31);
    const int S = nc <= 128 ? 1 : (nc <= 512 ? 2 : 4);
    const dim3 grid(cdiv(warps, kRB / 32), cdiv(nc - 1, S));
    if (S == 1)
      launch_k(k_restrict_rb2<1>, grid, kRB, 0, s, u_f, b_f, gf.n, b_c, u_c, nc, start ? 1 : 0);
    else if (S == 2)
      launch_k(k_restrict_rb2<2>, grid, kRB, 0, s, u_f, b_f, gf.n, b_c, u_c, nc, start ? 1 : 0);
    else
      launch_k(k_restrict_rb2<4>, grid, kRB, 0, s, u_f, b_f, gf.n, b_c, u_c, nc, start ? 1 : 0);
  } else {
    int lg = 0;
    while ((1 << lg) < gf.n) ++lg;
    if ((1 << lg) != gf.n) return cudaErrorInvalidValue;
    const unsigned bx = nc <= 32 ? 32 : (nc <= 64 ? 64 : 128);
    launch_k(k_restrict_rb3, dim3(cdiv(nc - 1, bx), nc - 1, nc - 1), bx, 0, s, u_f, b_f, gf.n, lg, b_c, u_c, nc,
             start ? 1 : 0);
  }
  return cudaGetLastError();
}

cudaError_t launch_prolong_rb64(int dim, LevelGeo gc, const double* e_c, LevelGeo gf, double* u_f, cudaStream_t s) {
  const unsigned gx = cdiv(gc.n, kRB);
  if (dim == 2)
    launch_k(k_prolong_rb2, dim3(gx, gf.n - 1), kRB, 0, s, e_c, gc.n, u_f);
  else
    launch_k(k_prolong_rb3, dim3(gx, gf.n - 1, gf.n - 1), kRB, 0, s, e_c, gc.n, u_f);
  return cudaGetLastError();
}

cudaError_t launch_level_start64(int dim, LevelGeo gc, const double* uc, LevelGeo g, double* u, const double* gn,
                                 double* b, int kind, double a, cudaStream_t s) {
  const double h = 1.0 / g.n;
  const double w = dim == 2 ? h * h : h * h * h;
  int lg = 0;
  while ((1 << lg) < g.n) ++lg;
  const int wexp = (1 << lg) == g.n ? -dim * lg : 1;
  const unsigned gx = cdiv(g.n + 1, kRB);
  if (dim == 2)
    launch_k(k_level_start64<2>, dim3(gx, cdiv(g.n + 1, kLS)), kRB, 0, s, uc, gc.n, u, gn, b, kind, a, w, wexp);
  else
    launch_k(k_level_start64<3>, dim3(gx, g.n + 1, cdiv(g.n + 1, kLS)), kRB, 0, s, uc, gc.n, u, gn, b, kind, a, w, wexp);
  return cudaGetLastError();
}

// The 2D kernels, for phase-batched launches.
void phase_kernels_rb64(std::vector<PhaseKernel>& out) {
  out.push_back(phase_kernel<&k_rbgs2_strip_body<4>, kRB, 1>(&k_rbgs2_strip<4>));
  out.push_back(phase_kernel<&k_restrict_rb2_body<1>, kRB, 1>(&k_restrict_rb2<1>));
  out.push_back(phase_kernel<&k_restrict_rb2_body<2>, kRB, 1>(&k_restrict_rb2<2>));
  out.push_back(phase_kernel<&k_restrict_rb2_body<4>, kRB, 1>(&k_restrict_rb2<4>));
  out.push_back(phase_kernel<&k_prolong_rb2_body, kRB, 1>(&k_prolong_rb2));
  out.push_back(phase_kernel<&k_level_start64_body<2>, kRB, 1>(&k_level_start64<2>));
  out.push_back(phase_kernel<&k_pre_rb64_body<1, 16>, kRT, 1>(&k_pre_rb64<1, 16>));
  out.push_back(phase_kernel<&k_pre_rb64_body<2, 16>, kRT, 1>(&k_pre_rb64<2, 16>));
  out.push_back(phase_kernel<&k_pre_rb64_body<1, 32>, kRT, 1>(&k_pre_rb64<1, 32>));
  out.push_back(phase_kernel<&k_pre_rb64_body<2, 32>, kRT, 1>(&k_pre_rb64<2, 32>));
  out.push_back(phase_kernel<&k_post_rb64_body<1, 16>, kRT, 1>(&k_post_rb64<1, 16>));
  out.push_back(phase_kernel<&k_post_rb64_body<2, 16>, kRT, 1>(&k_post_rb64<2, 16>));
  out.push_back(phase_kernel<&k_post_rb64_body<1, 32>, kRT, 1>(&k_post_rb64<1, 32>));
  out.push_back(phase_kernel<&k_post_rb64_body<2, 32>, kRT, 1>(&k_post_rb64<2, 32>));
}

}  // namespace fmg
