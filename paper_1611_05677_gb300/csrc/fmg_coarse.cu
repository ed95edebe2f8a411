// The V(nu_pre, nu_post) cycle on the coarse levels jtop..1 in one launch (Algorithm 3.1 step 1,
// eq. 3.5): the same smoothing steps, restriction P^T, exact level-1 solve and prolongation as the
// per-level kernels, with every level's arrays in shared memory and barriers in place of
// launches.
//
// What bounds it and how it is split.  A coarse level is a few thousand nodes and a cycle about
// ten dependent passes per level, so the cycle is a latency chain; on one SM it is a throughput
// one too, in FP64 above all: an SM issues two FP64 operations per clock, and a 64^2 half sweep
// needs 10^4 of them.  A cluster barrier that orders remote shared-memory stores costs a pass
// about 1400 clocks, a __syncthreads 44.  So only the top level is dealt to the CTAs of a cluster,
// by rows (y in 2D, z planes in 3D), and every CTA then runs the levels below it by itself, all
// CTAs the same arithmetic, from a right-hand side that the restriction stores into every CTA.
// On the top level a CTA holds its own rows and a halo of kHalo rows on either side.  In 2D the
// halo is as deep as two sweeps and the restriction reach (6), so that pre-smoothing runs without
// any exchange on rows that shrink by one per pass, and so does post-smoothing after one exchange;
// in 3D, where a plane is a whole 17^2 slice, it is one plane, exchanged after every pass.
// Measured (one 64^2 cycle, 1/H = 8, inside a solve): FP64 red-black 66 us on one CTA, 28 us here;
// FP32 Chebyshev 18 and 14 us.  With every level dealt to the CTAs and one row of halo (a cluster
// barrier per pass) it was 31 and 20 us.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <vector>

#include "fmg_ff.cuh"
#include "fmg_internal.cuh"
#include "fmg_phase.cuh"

namespace fmg {

namespace {

namespace cg = cooperative_groups;

constexpr int kCT = 512;          // threads per CTA
constexpr int kCS = 8;            // CTAs of a cluster that deals its top level
constexpr int kMaxCL = 8;         // levels at most (2 .. 64 cells per side)
constexpr int kMaxOwn = 64;       // a CTA's own rows of the top level, at most
constexpr int kMaxCoarseN = 64;   // level-1 unknowns (2D: (1/H - 1)^2 <= 49, 3D: <= 27)

template <int D>
constexpr int kHalo = D == 2 ? 6 : 1;

// Cells per side up to which one CTA runs the whole cycle.
__host__ __device__ inline int local_cells(int dim) { return dim == 2 ? 32 : 8; }

// Top-level rows a CTA of a cluster of cs holds at most.
__host__ __device__ inline int held_rows(int dim, int n, int cs) {
  const int h = (n + cs - 1) / cs + 2 * (dim == 2 ? kHalo<2> : kHalo<3>);
  return cs == 1 || h > n + 1 ? n + 1 : h;
}

template <typename T>
struct CoarseArgs {
  T* u;                 // level jtop's nodal arrays
  const T* b;
  const double* Ainv;   // A_1^{-1}
  const float* Ainv32;  // its FP32 copy (FP32 cycles with A = I)
  double* add;          // add_mode 1: add += u (FP64); 2: float-float add += u; 0: u is stored
  int add_mode;
  int n0, jtop, nu_pre, nu_post, zero_start;
  VarCoef vc;
  // Chebyshev coefficients in T: a conversion from FP64 issues at the FP64 rate
  T cd[kMaxCheb], cr[kMaxCheb];
};

// One level as a CTA sees it.  Local index of node (i, j[, l]): (row - lo) rs + (3D: j np) + i.
struct CLevel {
  int n, lg, np, rs;
  int lo;               // first held row (0 below the top level)
  int u, b, d, ua;      // array offsets (elements); the residual goes to d
  unsigned magic;       // 2^20 / (n / 2), rounded up
};

template <typename T, int D, bool CHEB, bool VC>
__device__ __forceinline__ void k_coarse_cluster_body(const CoarseArgs<T>& A) {
  cg::cluster_group cluster = cg::this_cluster();
  const int me = (int)cluster.block_rank();
  const int CS = (int)cluster.num_blocks();
  const int lgcs = 31 - __clz(CS);
  extern __shared__ __align__(16) unsigned char smraw[];
  T* sm = reinterpret_cast<T*>(smraw);
  __shared__ CLevel LV[kMaxCL];
  __shared__ int lo_tab[kCS], hi_tab[kCS];    // top-level rows held by each CTA
  __shared__ unsigned char mask[kMaxOwn];     // per own row: the other CTAs that hold it
  using BT = typename std::conditional<(sizeof(T) == 4 && !VC), float, double>::type;
  __shared__ BT b1[kMaxCoarseN];
  const int tid = threadIdx.x;
  const int jtop = A.jtop;
  const int m1 = A.n0 - 1;
  const int N1 = D == 2 ? m1 * m1 : m1 * m1 * m1;
  const int mrow = D == 2 ? m1 : m1 * m1;     // level-1 unknowns per row
  constexpr int NARR = CHEB ? 4 : 3;
  constexpr int W = kHalo<D>;
  using AT = typename std::conditional<(sizeof(T) == 4 && !VC), float, double>::type;
  const int ntop = A.n0 << (jtop - 1);
  const int rstop = D == 2 ? ntop + 1 : (ntop + 1) * (ntop + 1);
  // own interior rows r of the top level: floor(r CS / n) = rank
  auto own0 = [&](int c) { return max(1, (c * ntop + CS - 1) >> lgcs); };
  auto own1 = [&](int c) { return min(ntop, ((c + 1) * ntop + CS - 1) >> lgcs); };
  const int R0 = own0(me), R1 = own1(me);
  const int lo = CS == 1 ? 0 : max(0, R0 - W), hi = CS == 1 ? ntop : min(ntop, R1 - 1 + W);
  const int held = (hi - lo + 1) * rstop;
  if (tid < jtop) {
    const int j = tid + 1;
    CLevel L;
    L.n = A.n0 << (j - 1);
    L.lg = 31 - __clz(L.n);
    L.np = L.n + 1;
    L.rs = D == 2 ? L.np : L.np * L.np;
    L.lo = j == jtop ? lo : 0;
    const unsigned half = (unsigned)(L.n >> 1);
    L.magic = ((1u << 20) + half - 1) / half;
    int off = 0;
    for (int q = 1; q < j; ++q) {
      const int np = (A.n0 << (q - 1)) + 1;
      off += NARR * (D == 2 ? np * np : np * np * np);
    }
    const int len = (j == jtop ? held_rows(D, L.n, CS) : L.np) * L.rs;
    L.u = off;
    L.b = off + len;
    L.d = off + 2 * len;
    L.ua = off + 3 * len;
    LV[tid] = L;
  }
  if (tid < CS) {
    lo_tab[tid] = CS == 1 ? 0 : max(0, own0(tid) - W);
    hi_tab[tid] = CS == 1 ? ntop : min(ntop, own1(tid) - 1 + W);
  }
  // every array starts at zero (boundary rows and columns stay zero)
  int words = 0;
  for (int q = 1; q < jtop; ++q) {
    const int np = (A.n0 << (q - 1)) + 1;
    words += NARR * (D == 2 ? np * np : np * np * np);
  }
  words += NARR * held_rows(D, ntop, CS) * rstop;
  const int sm_end = (words + 3) & ~3;
  {
    uint4* z = reinterpret_cast<uint4*>(smraw);
    const int nz = sm_end * (int)sizeof(T) / 16;
    for (int i = tid; i < nz; i += kCT) z[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  // all of the above overlaps the predecessor's end; its data is read from here on
  pdl_wait();
  // ---- the global loads are issued together: the held rows of b (and of u), and A_1^{-1}
  constexpr int PL = 4, PA = 6;
  T bv[PL], uv[PL];
  AT av[PA];
  const long long g0 = (long long)lo * rstop;
#pragma unroll
  for (int r = 0; r < PL; ++r) {
    const int i = tid + r * kCT;
    bv[r] = i < held ? A.b[g0 + i] : T(0);
    uv[r] = (i < held && !A.zero_start) ? A.u[g0 + i] : T(0);
  }
  auto ainv_at = [&](int i) -> AT {
    if constexpr (sizeof(AT) == 4)
      return __ldg(A.Ainv32 + i);
    else
      return __ldg(A.Ainv + i);
  };
#pragma unroll
  for (int r = 0; r < PA; ++r) {
    const int i = tid + r * kCT;
    av[r] = i < N1 * N1 ? ainv_at(i) : AT(0);
  }
  __syncthreads();
  const CLevel Lt = LV[jtop - 1];
  AT* ai = reinterpret_cast<AT*>(sm + sm_end);   // A_1^{-1}
#pragma unroll
  for (int r = 0; r < PA; ++r) {
    const int i = tid + r * kCT;
    if (i < N1 * N1) ai[i] = av[r];
  }
  for (int i = tid + PA * kCT; i < N1 * N1; i += kCT) ai[i] = ainv_at(i);
  for (int r = R0 + tid; r < R1; r += kCT) {
    unsigned m = 0;
    for (int c = 0; c < CS; ++c)
      if (c != me && r >= lo_tab[c] && r <= hi_tab[c]) m |= 1u << c;
    mask[r - R0] = (unsigned char)m;
  }
  const bool first_top = CHEB && A.zero_start && A.nu_pre >= 1;
  // buffer a level's smoothing starts in when its first Chebyshev step is taken by the code that
  // writes its right-hand side: u when an even number of steps follows, else ua
  auto cheb_start_off = [&](const CLevel& L) { return ((A.nu_pre - 1) & 1) ? L.ua : L.u; };
  {
    // top level from zero: nothing, or the first Chebyshev step u = d = cr_0 D^{-1} b, pointwise
    // on every held row
    const T e0 = times_pow2(A.cr[0], D == 2 ? 0 : Lt.lg) * (T(1) / T(2 * D));
    const int us = first_top ? cheb_start_off(Lt) : Lt.u;
    auto place = [&](int i, T bval, T uval) {
      sm[Lt.b + i] = bval;
      if (!A.zero_start) sm[Lt.u + i] = uval;
      if (first_top) {   // (b is zero on the boundary)
        const T e = e0 * bval;
        sm[us + i] = e;
        sm[Lt.d + i] = e;
      }
    };
#pragma unroll
    for (int r = 0; r < PL; ++r) {
      const int i = tid + r * kCT;
      if (i < held) place(i, bv[r], uv[r]);
    }
    for (int i = tid + PL * kCT; i < held; i += kCT) place(i, A.b[g0 + i], A.zero_start ? T(0) : A.u[g0 + i]);
  }
  __syncthreads();
  // every CTA has laid out its memory before any remote store
  if (CS > 1) cluster.barrier_arrive();
  bool laid_out = CS == 1;
  auto before_remote = [&]() {
    if (!laid_out) cluster.barrier_wait();
    laid_out = true;
  };

  // f(local index, x, y, row) over the interior nodes of one colour in rows ra .. rb-1
  auto for_colour = [&](const CLevel& L, int ra, int rb, int colour, auto f) {
    ra = max(ra, 1);
    rb = min(rb, L.n);
    const int half = L.n >> 1;
    const int total = D == 2 ? (rb - ra) * half : ((rb - ra) * half) << L.lg;
    for (int t = tid; t < total; t += kCT) {
      int p, y, q;
      if (D == 2) {
        q = (int)(((unsigned)t * L.magic) >> 20);
        p = t - q * half;
        y = ra + q;
      } else {
        p = t & (half - 1);
        y = (t >> (L.lg - 1)) & (L.n - 1);
        q = t >> (2 * L.lg - 1);
        if (y == 0) continue;
      }
      const int row = ra + q;
      const int par = (colour + y + (D == 3 ? row : 0)) & 1;
      const int i = par ? 2 * p + 1 : 2 * p + 2;
      if (i > L.n - 1) continue;
      f((row - L.lo) * L.rs + (D == 3 ? y * L.np : 0) + i, i, y, row);
    }
  };
  // the same over all interior nodes of those rows
  auto for_inner = [&](const CLevel& L, int ra, int rb, auto f) {
    ra = max(ra, 1);
    rb = min(rb, L.n);
    const int total = D == 2 ? (rb - ra) * L.n : ((rb - ra) * L.n) << L.lg;
    for (int t = tid; t < total; t += kCT) {
      int i, y, q;
      if (D == 2) {
        q = (int)(((unsigned)(t >> 1) * L.magic) >> 20);
        i = t - q * L.n;
        y = ra + q;
      } else {
        i = t & (L.n - 1);
        y = (t >> L.lg) & (L.n - 1);
        q = t >> (2 * L.lg);
        if (y == 0) continue;
      }
      if (i == 0) continue;
      const int row = ra + q;
      f((row - L.lo) * L.rs + (D == 3 ? y * L.np : 0) + i, i, y, row);
    }
  };
  // sum of the 2d neighbours
  auto nbsum = [&](const CLevel& L, const T* u, int c) {
    const int np = L.np;
    T s = (u[c - 1] + u[c + 1]) + (u[c - np] + u[c + np]);
    if (D == 3) s += u[c - L.rs] + u[c + L.rs];
    return s;
  };
  auto offsets = [&](const CLevel& L, int* o) {
    o[0] = -1;
    o[1] = 1;
    o[2] = -L.np;
    o[3] = L.np;
    if (D == 3) {
      o[4] = -L.rs;
      o[5] = L.rs;
    }
  };

  // Halo bookkeeping.  `valid`: rows beyond the own ones on which the top level's iterate is
  // current (below the top level every row is local).  A pass that reads neighbours leaves one
  // row less; when none would be left the own rows are stored into the CTAs that hold them.
  int valid = W;
  auto push_rows = [&](int off) {
    const int own = (R1 - R0) * rstop;
    for (int i = tid; i < own; i += kCT) {
      const int q = i / rstop;
      unsigned m = mask[q];
      if (!m) continue;
      const int w = i - q * rstop;
      const T v = sm[off + (R0 + q - lo) * rstop + w];
      while (m) {
        const int t = __ffs(m) - 1;
        m &= m - 1;
        cluster.map_shared_rank(sm, t)[off + (R0 + q - lo_tab[t]) * rstop + w] = v;
      }
    }
  };
  // makes at least `need` halo rows of array `off` current.  A deep halo is overwritten only when
  // no CTA reads it any more (the CTAs' passes are not in step between exchanges); with a halo of
  // one row every pass is followed by an exchange, and what a neighbour may still read of it is
  // the other colour, whose values the store repeats, or the other Chebyshev buffer.  Where that
  // does not hold -- after the prolongation, which adds to the halo rows in place, and after an odd
  // number of Chebyshev steps, whose result is moved to the buffer that the last of them read -- the
  // CTAs have arrived at a barrier behind the pass in question (`behind`), and the store waits for it.
  bool behind = false;
  auto ensure = [&](int off, int need) {
    if (CS == 1 || valid >= need) return;
    before_remote();
    if (W > 1) cluster.sync();
    if (behind) cluster.barrier_wait();
    behind = false;
    push_rows(off);
    cluster.sync();
    valid = W;
  };
  // rows a pass on level j covers when it leaves `v` halo rows current
  auto row_a = [&](int j, int v) { return j == jtop ? (CS == 1 ? 1 : R0 - v) : 1; };
  auto row_b = [&](int j, int v) { return j == jtop ? (CS == 1 ? ntop : R1 + v) : (A.n0 << (j - 1)); };

  auto half_sweep = [&](const CLevel& L, int j, int colour) {
    const T bscale = D == 2 ? T(1) : T(L.n);
    const T* u = sm + L.u;
    if (j == jtop) {
      ensure(L.u, 1);
      --valid;
    }
    for_colour(L, row_a(j, valid), row_b(j, valid), colour, [&](int c, int i, int y, int row) {
      T v;
      if constexpr (VC) {
        int o[2 * D];
        offsets(L, o);
        T w[2 * D];
        edge_weights_t<D, T>(A.vc, j - 1, i, y, row, w);
        T sw = T(0), su = T(0);
#pragma unroll
        for (int e = 0; e < 2 * D; ++e) {
          sw += w[e];
          su += w[e] * u[c + o[e]];
        }
        v = (sm[L.b + c] * bscale + su) / sw;
      } else {
        const T s = nbsum(L, u, c);
        if constexpr (D == 2)
          v = quarter(sm[L.b + c] + s);
        else
          v = (times_pow2(sm[L.b + c], L.lg) + s) * (T(1) / T(6));
      }
      sm[L.u + c] = v;
    });
    __syncthreads();
  };
  // Chebyshev steps k0..steps-1, alternating between u and ua, ending in u.  exchanged: the top level's
  // u goes to the neighbours next.
  auto cheb_steps = [&](const CLevel& L, int j, int steps, int k0, bool exchanged) {
    const T inv2d = T(1) / T(2 * D);
    int us = k0 ? cheb_start_off(L) : L.u;
    int uo = us == L.u ? L.ua : L.u;
    for (int k = k0; k < steps; ++k) {
      const T cd = A.cd[k], cr = A.cr[k];
      const T* u = sm + us;
      if (j == jtop) {
        // a pass over halo rows needs the step direction there too
        if (W > 1 && CS > 1 && valid < 1) {
          before_remote();
          cluster.sync();
          push_rows(L.d);
        }
        ensure(us, 1);
        --valid;
      }
      for_inner(L, row_a(j, valid), row_b(j, valid), [&](int c, int, int, int) {
        const T s = nbsum(L, u, c);
        const T bs = D == 2 ? sm[L.b + c] : times_pow2(sm[L.b + c], L.lg);
        const T z = (bs + s) * inv2d - u[c];
        const T dn = k == 0 ? cr * z : cd * sm[L.d + c] + cr * z;
        sm[L.d + c] = dn;
        sm[uo + c] = u[c] + dn;
      });
      __syncthreads();
      const int t2 = us;
      us = uo;
      uo = t2;
    }
    if (us != L.u) {
      if (W == 1 && CS > 1 && j == jtop && exchanged) {
        before_remote();
        cluster.barrier_arrive();
        behind = true;
      }
      // (current rows only: a neighbour may already store into the others)
      for_inner(L, row_a(j, valid), row_b(j, valid), [&](int c, int, int, int) { sm[L.u + c] = sm[us + c]; });
      __syncthreads();
    }
  };

  // ---- descend
  for (int j = jtop; j >= 2; --j) {
    const CLevel L = LV[j - 1];
    const CLevel C = LV[j - 2];
    if constexpr (CHEB) {
      const bool started = A.nu_pre >= 1 && (j < jtop || A.zero_start);
      cheb_steps(L, j, A.nu_pre, started ? 1 : 0, true);
    } else {
      for (int it = 0; it < A.nu_pre; ++it) {
        half_sweep(L, j, 0);
        half_sweep(L, j, 1);
      }
    }
    // r = b - A u on the own rows and their neighbours (3D: with a halo of one plane only, on the
    // own rows, then exchanged).  After a red-black sweep of the FP64 cycle the residual of the
    // black nodes, just relaxed, is zero but for rounding: it is taken as zero (half the FP64
    // work); the FP32 cycle forms it as its per-level kernels do.
    const T* u = sm + L.u;
    const T inv_n = times_pow2(T(1), -L.lg);   // 3D: h (n is a power of two)
    constexpr int RV = W >= 2 ? 1 : 0;   // halo rows the residual is formed on
    if (j == jtop) ensure(L.u, RV + 1);
    auto res = [&](int c, int i, int y, int row) {
      T r;
      if constexpr (VC) {
        int o[2 * D];
        offsets(L, o);
        T w[2 * D];
        edge_weights_t<D, T>(A.vc, j - 1, i, y, row, w);
        const T uc = u[c];
        T a = T(0);
#pragma unroll
        for (int e = 0; e < 2 * D; ++e) a += w[e] * (uc - u[c + o[e]]);
        r = sm[L.b + c] - (D == 2 ? T(1) : T(1) / T(L.n)) * a;
      } else {
        const T s = nbsum(L, u, c);
        r = sm[L.b + c] - (D == 2 ? T(1) : inv_n) * (T(2 * D) * u[c] - s);
      }
      sm[L.d + c] = r;
    };
    if (!CHEB && sizeof(T) == 8 && A.nu_pre >= 1)
      for_colour(L, row_a(j, RV), row_b(j, RV), 0, res);
    else
      for_inner(L, row_a(j, RV), row_b(j, RV), res);
    __syncthreads();
    if (CS > 1 && j == jtop) before_remote();
    if (CS > 1 && j == jtop && RV == 0) {
      push_rows(L.d);
      cluster.sync();
    }
    // b_c = P^T r, from the top level into every CTA; the coarse level starts from zero
    // (Chebyshev: with its step 0)
    const bool first_c = CHEB && A.nu_pre >= 1 && j - 1 >= 2;
    const T e0c = times_pow2(A.cr[0], D == 2 ? 0 : C.lg) * (T(1) / T(2 * D));
    const int ucs = first_c ? cheb_start_off(C) : C.u;
    const T* r = sm + L.d;
    const bool spread = CS > 1 && j == jtop;
    const bool red_only = !CHEB && sizeof(T) == 8 && A.nu_pre >= 1;
    // coarse rows K with 2K among the own fine rows
    const int ka = spread ? (R0 + 1) >> 1 : 1, kb = spread ? (R1 + 1) >> 1 : C.n;
    for_inner(C, ka, kb, [&](int cc, int I, int J, int K) {
      const int F = (2 * K - L.lo) * L.rs + (D == 3 ? 2 * J * L.np : 0) + 2 * I;
      const int np = L.np;
      T e;
      if constexpr (VC) {
        constexpr int NQ = D == 2 ? 3 : 7;
        const int q[7] = {1, np, 1 + np, L.rs, 1 + L.rs, np + L.rs, 1 + np + L.rs};
        e = T(0);
#pragma unroll
        for (int k = 0; k < NQ; ++k) e += r[F + q[k]] + r[F - q[k]];
      } else if (red_only) {
        // the neighbours of even offset (black residuals are zero)
        e = r[F + np + 1] + r[F - np - 1];
        if (D == 3)
          e += (r[F + L.rs + 1] + r[F - L.rs - 1]) + (r[F + L.rs + np] + r[F - L.rs - np]);
      } else {
        e = (r[F + 1] + r[F - 1]) + (r[F + np] + r[F - np]) + (r[F + np + 1] + r[F - np - 1]);
        if (D == 3) {
          const int pl = L.rs;
          const int o[4] = {pl, 1 + pl, np + pl, 1 + np + pl};
#pragma unroll
          for (int k = 0; k < 4; ++k) e += r[F + o[k]] + r[F - o[k]];
        }
      }
      const T bval = r[F] + T(0.5) * e;
      if (spread) {
        for (int t = 0; t < CS; ++t) cluster.map_shared_rank(sm, t)[C.b + cc] = bval;
        return;
      }
      sm[C.b + cc] = bval;
      if (first_c) {
        sm[ucs + cc] = e0c * bval;
        sm[C.d + cc] = e0c * bval;
      }
    });
    if (spread) {
      cluster.sync();
      if (first_c) {
        const int len = D == 2 ? C.np * C.np : C.np * C.np * C.np;
        for (int i = tid; i < len; i += kCT) {
          const T e1 = e0c * sm[C.b + i];
          sm[ucs + i] = e1;
          sm[C.d + i] = e1;
        }
        __syncthreads();
      }
    } else {
      __syncthreads();
    }
    // the halo that post-smoothing needs travels while the coarser levels run
    if (spread) {
      push_rows(L.u);
      cluster.barrier_arrive();
      valid = W;
    }
  }
  // ---- level 1: u_1 = A_1^{-1} b_1
  {
    const CLevel C = LV[0];
    auto slot = [&](int p) {
      const int row = p / mrow, w = p - row * mrow;
      const int y = D == 3 ? w / m1 : 0;
      return (row + 1) * C.rs + (D == 3 ? (y + 1) * C.np : 0) + (D == 3 ? w - y * m1 : w) + 1;
    };
    if (tid < N1) b1[tid] = (BT)sm[C.b + slot(tid)];
    __syncthreads();
    if constexpr (sizeof(T) == 4 && VC) {
      if (tid < N1) {
        const double* a = reinterpret_cast<const double*>(ai) + (size_t)tid * N1;
        double a0 = 0.0, a1 = 0.0;
        int c = 0;
        for (; c + 1 < N1; c += 2) {
          a0 = fma(a[c], b1[c], a0);
          a1 = fma(a[c + 1], b1[c + 1], a1);
        }
        if (c < N1) a0 = fma(a[c], b1[c], a0);
        sm[C.u + slot(tid)] = (T)(a0 + a1);
      }
    } else if constexpr (sizeof(T) == 4) {
      // a warp per row, four rows at a time
      const int lane = tid & 31, warp = tid >> 5;
      constexpr int NW = kCT / 32;
      const bool h0 = lane < N1, h1 = lane + 32 < N1;   // N_1 <= 64
      const float x0 = h0 ? (float)b1[lane] : 0.f, x1 = h1 ? (float)b1[lane + 32] : 0.f;
      for (int r0 = warp; r0 < N1; r0 += 4 * NW) {
        float acc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int r = r0 + q * NW;
          const float a0 = r < N1 && h0 ? (float)ai[r * N1 + lane] : 0.f;
          const float a1 = r < N1 && h1 ? (float)ai[r * N1 + lane + 32] : 0.f;
          acc[q] = fmaf(a1, x1, a0 * x0);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (lane == 0 && r0 + q * NW < N1) sm[C.u + slot(r0 + q * NW)] = (T)acc[q];
      }
    } else {
      // eight lanes per row: a row costs a chain of N_1 / 8 products and three sums
      const int g = tid & 7;
      for (int r0 = 0; r0 < N1; r0 += kCT / 8) {
        const int r = r0 + (tid >> 3);
        double acc = 0.0;
        if (r < N1)
          for (int c = g; c < N1; c += 8) acc = fma((double)ai[r * N1 + c], b1[c], acc);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (g == 0 && r < N1) sm[C.u + slot(r)] = (T)acc;
      }
    }
    __syncthreads();
  }
  // ---- ascend
  for (int j = 2; j <= jtop; ++j) {
    const CLevel L = LV[j - 1];
    const CLevel C = LV[j - 2];
    if (CS > 1 && j == jtop) cluster.barrier_wait();
    // u += P e_c on every held row; before a red-black sweep on the red nodes only (the sweep's
    // first half replaces every black value from its red neighbours)
    const T* e = sm + C.u;
    auto prol = [&](int c, int i, int y, int row) {
      const int a = (row >> 1) * C.rs + (D == 3 ? (y >> 1) * C.np : 0) + (i >> 1);
      const int z = ((row + 1) >> 1) * C.rs + (D == 3 ? ((y + 1) >> 1) * C.np : 0) + ((i + 1) >> 1);
      sm[L.u + c] += T(0.5) * (e[a] + e[z]);
    };
    const int ra = j == jtop ? lo : 1, rb = j == jtop ? hi + 1 : L.n;
    if (!CHEB && A.nu_post >= 1)
      for_colour(L, ra, rb, 0, prol);
    else
      for_inner(L, ra, rb, prol);
    // (the second half sweep's exchange is the first to store into the rows just corrected)
    if (!CHEB && W == 1 && CS > 1 && j == jtop && A.nu_post >= 1) {
      cluster.barrier_arrive();
      behind = true;
    }
    __syncthreads();
    if constexpr (CHEB) {
      cheb_steps(L, j, A.nu_post, 0, false);
    } else {
      for (int it = 0; it < A.nu_post; ++it) {
        half_sweep(L, j, 1);
        half_sweep(L, j, 0);
      }
    }
  }
  // ---- the own rows of the top level
  for_inner(Lt, R0, R1, [&](int c, int, int, int) {
    const long long g = (long long)lo * rstop + c;
    const T v = sm[Lt.u + c];
    if (A.add_mode == 2)
      ff_store(A.add + g, ff_add_f(ff_load(A.add + g), (float)v));
    else if (A.add_mode == 1)
      A.add[g] += (double)v;
    else
      A.u[g] = v;
  });
}

template <typename T, int D, bool CHEB, bool VC>
__global__ void __launch_bounds__(kCT) k_coarse_cluster(const __grid_constant__ CoarseArgs<T> A) {
  pdl_launch();
  k_coarse_cluster_body<T, D, CHEB, VC>(A);
}

// CTAs of a launch whose top level has n cells per side: one where the whole cycle is local, and
// for contexts that run beside others, where eight CTAs for a cycle take SMs from the other
// streams (32 batched 2D instances: 2.58 ms with clusters, 2.43 ms with one CTA
// each).
int cluster_ctas(int dim, int n) { return n <= local_cells(dim) || !t_pdl ? 1 : kCS; }

}  // namespace

template <typename T>
size_t coarse_cycle_smem(int dim, int n0, int jtop, bool cheb) {
  const int narr = cheb ? 4 : 3;
  size_t tot = 0;
  for (int j = 1; j < jtop; ++j) tot += (size_t)narr * ipow((n0 << (j - 1)) + 1, dim);
  const int n = n0 << (jtop - 1);
  tot += (size_t)narr * held_rows(dim, n, cluster_ctas(dim, n)) * ipow(n + 1, dim - 1);
  tot = (tot + 3) & ~size_t(3);
  const size_t n1 = (size_t)ipow(n0 - 1, dim);
  return tot * sizeof(T) + n1 * n1 * sizeof(double);
}

// Largest mesh (cells per side) the kernel takes.
int coarse_cycle_cells(int dim) { return dim == 2 ? 64 : 16; }

template <typename T, int D, bool CHEB, bool VC>
static cudaError_t launch_cluster(const CoarseArgs<T>& A, int ctas, size_t smem, cudaStream_t s) {
  cudaError_t e = raise_dyn_smem((const void*)k_coarse_cluster<T, D, CHEB, VC>, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(kCT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = t_pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k_coarse_cluster<T, D, CHEB, VC>, A);
}

template <typename T>
cudaError_t launch_coarse_cycle(int dim, int n0, int jtop, T* u, const T* b, int nu_pre, int nu_post,
                                const double* Ainv, const float* Ainv32, const ChebCoef* cheb, bool zero_start,
                                cudaStream_t s, const VarCoef* vc, double* add, int add_mode) {
  const bool v = vc && vc->a64;
  if (sizeof(T) == sizeof(float) && !v && !Ainv32) return cudaErrorInvalidValue;
  if (cheb && (v || nu_pre > kMaxCheb || nu_post > kMaxCheb)) return cudaErrorInvalidValue;
  if (jtop < 2 || jtop > kMaxCL || (n0 << (jtop - 1)) > coarse_cycle_cells(dim)) return cudaErrorInvalidValue;
  const size_t smem = coarse_cycle_smem<T>(dim, n0, jtop, cheb != nullptr);
  const int ctas = cluster_ctas(dim, n0 << (jtop - 1));
  CoarseArgs<T> A = {};
  A.u = u;
  A.b = b;
  A.Ainv = Ainv;
  A.Ainv32 = Ainv32;
  A.add = add;
  A.add_mode = add_mode;
  A.n0 = n0;
  A.jtop = jtop;
  A.nu_pre = nu_pre;
  A.nu_post = nu_post;
  A.zero_start = zero_start ? 1 : 0;
  if (v) A.vc = *vc;
  for (int k = 0; cheb && k < kMaxCheb; ++k) {
    A.cd[k] = (T)cheb->cd[k];
    A.cr[k] = (T)cheb->cr[k];
  }
  if (dim == 2)
    return cheb ? launch_cluster<T, 2, true, false>(A, ctas, smem, s)
           : v  ? launch_cluster<T, 2, false, true>(A, ctas, smem, s)
                : launch_cluster<T, 2, false, false>(A, ctas, smem, s);
  return cheb ? launch_cluster<T, 3, true, false>(A, ctas, smem, s)
         : v  ? launch_cluster<T, 3, false, true>(A, ctas, smem, s)
              : launch_cluster<T, 3, false, false>(A, ctas, smem, s);
}

template size_t coarse_cycle_smem<double>(int, int, int, bool);
template size_t coarse_cycle_smem<float>(int, int, int, bool);
template cudaError_t launch_coarse_cycle<double>(int, int, int, double*, const double*, int, int, const double*,
                                                 const float*, const ChebCoef*, bool, cudaStream_t, const VarCoef*,
                                                 double*, int);
template cudaError_t launch_coarse_cycle<float>(int, int, int, float*, const float*, int, int, const double*,
                                                const float*, const ChebCoef*, bool, cudaStream_t, const VarCoef*,
                                                double*, int);

// The 2D cluster cycles, for phase-batched launches.
void phase_kernels_coarse(std::vector<PhaseKernel>& out) {
  out.push_back(phase_kernel<&k_coarse_cluster_body<float, 2, true, false>, kCT, 1>(&k_coarse_cluster<float, 2, true, false>));
  out.push_back(phase_kernel<&k_coarse_cluster_body<float, 2, false, false>, kCT, 1>(&k_coarse_cluster<float, 2, false, false>));
  out.push_back(phase_kernel<&k_coarse_cluster_body<double, 2, true, false>, kCT, 1>(&k_coarse_cluster<double, 2, true, false>));
  out.push_back(phase_kernel<&k_coarse_cluster_body<double, 2, false, false>, kCT, 1>(&k_coarse_cluster<double, 2, false, false>));
}

}  // namespace fmg
