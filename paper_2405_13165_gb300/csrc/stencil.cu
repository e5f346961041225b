// stencil.cu -- GFDM stencils of Eq. GFDM_Definition (Sec. 2.3), order 2.
//
// One group of G lanes per particle (8 or more for 3D rows of ~180 entries, 4 or
// more for film rows of ~40).  Lanes stride over the row, accumulate the distinct moments of
// A = sum_j w_j p_j p_j^T, reduce them with a reduce-scatter of shuffles, factor
// A (Cholesky) and solve for the four right-hand sides, one per lane.
// FP32 path: one refinement step with the residual b - sum_j c_j p_j of the
// rounded coefficients; particles whose Cholesky pivots are too small or whose
// condition estimate exceeds cond_fp64 are queued and redone in FP64.
#include "internal.cuh"
#include "stencil_common.cuh"

namespace mafp {

// Clouds of at most kStFewRows particles take the wide groups (too few rows for
// the GPU's warps otherwise).
constexpr int64_t kStFewRows = 16384;

// Rounds of rows per warp.  More share a warp's start and its last, partly filled round,
// and leave fewer warps that find no row of the model; but where the rows lie in few warps
// (a column of 3D rows in a wide film) the others are idle.  Whole builds, us, with 1 / 2 /
// 4 rounds --
//   3D (film rounds as below): jet on a film, 70k particles 82 / 93 / 116, 141k 147 / 155 /
//   167, 180k 185 / 185 / 197, 1M 1234 / 1152 / 1146; cube 70k 144 / 146 / 171, 142k 274 /
//   283 / 304, 178k 338 / 344 / 360, 517k 1029 / 1002 / 1016; a film alone, whose 3D pass
//   finds nothing, 160k 111 / 106 / 102;
//   film: 70k 57 / 56 / 61, 131k 96 / 94 / 95, 230k 150 / 145 / 146, 1M 704 / 619 / 583.
// FP64 (its pipe is full with few warps, and uneven warps are its time): jet 66k 1081 /
// 1265 / 1692, cube 134k 5774 / 5919 / 6347, film 131k 1116 / 1146 / 1149.
template <typename C, int M>
static int rounds_of(int64_t n) {
  if (sizeof(C) == 8) return 1;
  if (M == 10) return n > 163840 ? 2 : 1;
  return n > 262144 ? 4 : (n > 65536 ? 2 : 1);
}

// Two warps per block: a block's slot is free again as soon as its two warps'
// rows are done (1M jet cloud, 3D rows: 847 us against 925 with four warps).
constexpr int kBuildThreads = 64;

__global__ void k_reset_queue(DevStatus *st) { pdl_sync(); st->fallback_count = 0; }

// Per-lane cache for the passes after the moments.  FP32: (q, w) of two entries
// together, (q1a, q1b, q2a, q2b) and (q3a, q3b, wa, wb), KC entries per lane (176
// per 3D row, 40 per film row).  FP64: w alone (its exponential is ~25 of the ~55
// FP64 operations that the coefficient pass spends on an entry).  Entries beyond
// it are gathered and recomputed as in the first pass.
template <typename C, int M, int G>
struct StCache {
  static constexpr int KC = pad_to((M == 10 ? 176 : 40) / G, 2);
  static constexpr int BYTES = kBuildThreads * KC * (sizeof(C) == 4 ? (int)sizeof(float4) : 8);
  static constexpr int SMEM = BYTES + (kBuildThreads / G) * StSmem<M, G>::PER_GROUP * (int)sizeof(C);
};

// neighbours a lane gathers ahead of use: 4 for 3D rows (long rows, the loads
// in flight together), 2 for film rows
template <int M> constexpr int kGatherU = M == 10 ? 4 : 2;

// ------------------------------------------------------------------ FP32 rows
// The passes over a row in packed FP32 (two operations per instruction; the FMA
// pipe retires them at the scalar rate, so what falls is the number of
// instructions issued).  The refinement and coefficient passes pack two
// right-hand sides (the coefficients of one entry side by side: lambda_k stays
// in registers once); the moment pass packs the weights and coordinates of two
// entries.
// What bounds it (ncu, jet cloud of 303k particles): 3D, ~6000 instructions per round
// of four rows; the FMA pipe is 51 % busy (a packed FMA with three different operands
// takes 3 cycles of it, measured) and 56 % of the cycles issue, at 13.9 warps per SM of the
// 16 that registers (128) and shared memory (26 KB a block) both allow; an instruction
// waits 1.25 cycles on fixed latencies and 1.14 on its gathers.  Film (4 lanes): issue 58 %,
// FMA pipe 43 %, 16.7 warps of 20 (96 registers).  1M jet cloud, 3D 890 -> 746 us, film
// 300 -> 256 us; with the launch shapes of a new context 2136 -> 889 us for 440k 3D rows.
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  return __ffma2_rn(a, b, c);
}

// Monomials p_1.. of two packed coordinate triples (pairs in 2D); p_0 = 1 is implied.
template <int M>
__device__ __forceinline__ void basis2(float2 a, float2 b, float2 c, float2 (&p)[M]) {
  if constexpr (M == 10) {
    p[1] = a; p[2] = b; p[3] = c;
    p[4] = mul2(a, a); p[5] = mul2(b, b); p[6] = mul2(c, c);
    p[7] = mul2(a, b); p[8] = mul2(a, c); p[9] = mul2(b, c);
  } else {
    p[1] = a; p[2] = b;
    p[3] = mul2(a, a); p[4] = mul2(a, b); p[5] = mul2(b, b);
  }
}

// Process particle i (FP32) with a group of G lanes; results as stencil_particle.
template <int M, int G, bool REFINE>
__device__ __forceinline__ void stencil_row32(int64_t i, const float4 *pos, const uint8_t *model,
                                              const float4 *frame, const long long *row_ptr,
                                              const int32_t *col, float4 *coef,
                                              const StParams<float> &sp, float *sm, int *result,
                                              float *cond_out, float4 *qw) {
  constexpr int NA = Basis<M>::NA, NR = Basis<M>::NR, KL = NR - 1;
  constexpr int VR = pad_to(NR * M, G), VM = pad_to(Moments<M>::N, G);
  constexpr int KP = StCache<float, M, G>::KC / 2, U = kGatherU<M>;
  const int lane = threadIdx.x & (G - 1);
  const unsigned gm = group_mask<G>();
  const float4 xi = ld4(pos + i);
  const uint8_t mi = model[i];
  const float hinv = 1.0f / xi.w, h2inv = hinv * hinv;
  float t1[3] = {0, 0, 0}, t2[3] = {0, 0, 0};
  if constexpr (M == 6) {
    const float4 f1 = ld4(frame + 2 * i), f3 = ld4(frame + 2 * i + 1);
    t1[0] = f1.x; t1[1] = f1.y; t1[2] = f1.z;
    t2[0] = f3.y * t1[2] - f3.z * t1[1];
    t2[1] = f3.z * t1[0] - f3.x * t1[2];
    t2[2] = f3.x * t1[1] - f3.y * t1[0];
  }
  const long long b = row_ptr[i];
  const int len = (int)(row_ptr[i + 1] - b);
  col += b;
  coef += b;

  // U neighbours of the lane (entries e, e + G, ... of the row, their columns
  // given), gathered before any of them is used; slots past the row end load
  // particle i itself and are marked invalid, as are neighbours of the other model
  auto columns = [&](int e, int (&j)[U]) {
#pragma unroll
    for (int u = 0; u < U; ++u) j[u] = e + u * G < len ? col[e + u * G] : -1;
  };
  auto gather = [&](const int *j, int nu, float4 *x, bool *ok) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (u < nu) {
        const int jj = j[u] >= 0 ? j[u] : (int)i;
        x[u] = ld4(pos + jj);
        ok[u] = j[u] >= 0 && model[jj] == mi;
      }
  };
  // (q, w) of two entries, gathered by the caller; w = 0 where an entry is not one
  auto locate = [&](const float4 &xa, const float4 &xb, bool oka, bool okb, float2 &qa, float2 &qb,
                    float2 &qc, float2 &w) {
    const float2 dx = make_float2(xa.x - xi.x, xb.x - xi.x);
    const float2 dy = make_float2(xa.y - xi.y, xb.y - xi.y);
    const float2 dz = make_float2(xa.z - xi.z, xb.z - xi.z);
    const float2 s2 = mul2(fma2(dz, dz, fma2(dx, dx, mul2(dy, dy))), dup2(h2inv));
    const float2 e = make_float2(expf(-sp.alpha * s2.x), expf(-sp.alpha * s2.y));
    w = mul2(add2(e, dup2(-sp.ea)), dup2(sp.inv_den));
    w.x = oka && s2.x <= 1.0f ? w.x : 0.0f;
    w.y = okb && s2.y <= 1.0f ? w.y : 0.0f;
    const float2 hh = dup2(hinv);
    if constexpr (M == 10) {
      qa = mul2(dx, hh); qb = mul2(dy, hh); qc = mul2(dz, hh);
    } else {
      qa = mul2(fma2(dz, dup2(t1[2]), fma2(dx, dup2(t1[0]), mul2(dy, dup2(t1[1])))), hh);
      qb = mul2(fma2(dz, dup2(t2[2]), fma2(dx, dup2(t2[0]), mul2(dy, dup2(t2[1])))), hh);
      qc = qb;
    }
  };

  // ---- moments (the distinct ones), summed one entry after another: two packed
  // entries would take 70 sums and with them the registers of a third of the warps
  float A[VM];
#pragma unroll
  for (int k = 0; k < VM; ++k) A[k] = 0.0f;
  int cnt = 0, kp = 0;
  // the columns are loaded a round ahead of their use (the records too: 828
  // against 805 us in 3D, no difference for film)
  int js[U];
  columns(lane, js);
#pragma unroll 1
  for (int e0 = lane; e0 < len; e0 += U * G, kp += U / 2) {
    float4 xs[U];
    bool oks[U];
    gather(js, U, xs, oks);
    columns(e0 + U * G, js);
#pragma unroll
    for (int u = 0; u < U; u += 2) {
      float2 q[3], w;
      locate(xs[u], xs[u + 1], oks[u], oks[u + 1], q[0], q[1], q[2], w);
      cnt += (oks[u] ? 1 : 0) + (oks[u + 1] ? 1 : 0);
      if (kp + u / 2 < KP) {
        float4 *c = qw + 64 * (kp + u / 2);
        c[0] = make_float4(q[0].x, q[0].y, q[1].x, q[1].y);
        c[32] = make_float4(q[2].x, q[2].y, w.x, w.y);
      }
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          float p[M];
          const float x = v ? q[0].y : q[0].x, y = v ? q[1].y : q[1].x, z = v ? q[2].y : q[2].x;
          p[0] = 1.0f; p[1] = x; p[2] = y;
          if constexpr (M == 10) {
            p[3] = z;
            p[4] = x * x; p[5] = y * y; p[6] = z * z; p[7] = x * y; p[8] = x * z; p[9] = y * z;
          } else {
            p[3] = x * x; p[4] = x * y; p[5] = y * y;
          }
          add_moments<M, float, VM>(A, v ? w.y : w.x, p);
        }
    }
  }
  reduce_scatter<G, VM>(A);
  __syncwarp(gm);
#pragma unroll
  for (int k = 0; k < VM / G; ++k) sm[lane * (VM / G) + k] = A[k];
  float L[NA];
  cnt = group_sum<G>(cnt);
  __syncwarp(gm);
  constexpr MomentTable<M> MT = Moments<M>::T;
#pragma unroll
  for (int k = 0; k < NA; ++k) L[k] = sm[MT.idx[k]];
  __syncwarp(gm);
  float tr = 0;
#pragma unroll
  for (int r = 0; r < M; ++r) tr += L[pk(r, r)];
  float invd[M], pmin, pmax;
  const bool pd = cholesky<M, float, REFINE && M == 10>(L, invd, sp.piv_tol_rel * tr, pmin, pmax);
  const bool ok = pd && cnt >= M;
  const float cond = (pmax / pmin) * (pmax / pmin);
  float *Ls = sm + StSmem<M, G>::SCR;
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NA; ++k) Ls[k] = L[k];
  }
  __syncwarp(gm);
  if (!ok || !(cond <= sp.cond_max)) {
    if (cnt >= M) {
      *result = 2;   // FP64 decides
      return;
    }
    for (int e = lane; e < len; e += G) st4(coef + e, make_float4(0, 0, 0, 0));
    *result = 1;
    *cond_out = INFINITY;
    return;
  }
  // ---- solve: lane k of the group solves right-hand side k, and k + G where there
  // are more than lanes (a warp issues one solve for all of its groups' lanes at
  // once instead of NR in a row; lanes k >= NR repeat one), and the group reads the
  // solutions back from shared memory, as pairs: right-hand sides (0, 1) and (2, 3)
  // in 3D, (0, 1) and 2 for film
  constexpr int NQ = (NR + G - 1) / G;   // solves per lane
  // res[k M + r] (shared): solve for it and put the solution in its place
  auto solve_all = [&](auto &&right) {
    float x[NQ][M];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      float bb[M];
      const int kq = G >= NR ? lane % NR : (lane + q * G < NR ? lane + q * G : NR - 1);
#pragma unroll
      for (int r = 0; r < M; ++r) bb[r] = right(kq, r);
      chol_solve_s<M, float>(Ls, invd, bb, x[q]);
    }
    __syncwarp(gm);   // every lane has its right-hand sides before they are overwritten
#pragma unroll
    for (int q = 0; q < NQ; ++q)
      if (lane + q * G < NR) {
#pragma unroll
        for (int r = 0; r < M; ++r) sm[(lane + q * G) * M + r] = x[q][r];
      }
    __syncwarp(gm);
  };
  float2 l01[M], l2x[M];   // l2x.y: right-hand side 3, or film's correction of the Laplacian
  {
    solve_all([&](int k, int r) { return rhs<M, float>(k, r); });
#pragma unroll
    for (int r = 0; r < M; ++r) {
      l01[r] = make_float2(sm[r], sm[M + r]);
      l2x[r] = make_float2(sm[2 * M + r], M == 10 ? sm[(NR - 1) * M + r] : 0.0f);
    }
    __syncwarp(gm);
  }
  // calls body(e, q and w) for the lane's entries in pairs e and e + G (one loop
  // for cached and uncached entries: the passes' code stays in the instruction
  // cache)
  auto for_pairs = [&](auto &&body) {
#pragma unroll 1
    for (int e = lane, k = 0; e < len; e += 2 * G, ++k) {
      float2 q[3], w;
      if (k < KP) {
        const float4 *c = qw + 64 * k;
        const float4 u = c[0], v = c[32];
        q[0] = make_float2(u.x, u.y);
        q[1] = make_float2(u.z, u.w);
        q[2] = make_float2(v.x, v.y);
        w = make_float2(v.z, v.w);
      } else {   // beyond the cache: gathered again
        float4 xs[2];
        bool oks[2];
        const int j2[2] = {col[e], e + G < len ? col[e + G] : -1};
        gather(j2, 2, xs, oks);
        locate(xs[0], xs[1], oks[0], oks[1], q[0], q[1], q[2], w);
      }
      body(e, q[0], q[1], q[2], w);
    }
  };
  // sums p.lambda of the packed right-hand sides (p_0 = 1)
  auto dots = [&](const float2 (&p)[M], float2 &s01, float2 &s2x) {
    if constexpr (M == 10) {
      // nested: the coefficient pass needs no products then, and three short
      // chains replace one of nine (951 -> 909 us for 440k rows)
      auto poly = [&](const float2 (&l)[M]) {
        const float2 a = fma2(p[1], l[4], fma2(p[2], l[7], fma2(p[3], l[8], l[1])));
        const float2 b = fma2(p[2], l[5], fma2(p[3], l[9], l[2]));
        const float2 c = fma2(p[3], l[6], l[3]);
        return fma2(p[1], a, fma2(p[2], b, fma2(p[3], c, l[0])));
      };
      s01 = poly(l01);
      s2x = poly(l2x);
      return;
    }
    s01 = l01[0];
    s2x = l2x[0];
#pragma unroll
    for (int r = 1; r < M; ++r) {
      s01 = fma2(p[r], l01[r], s01);
      s2x = fma2(p[r], l2x[r], s2x);
    }
  };
  // The Laplacian's refinement correction is kept apart (lo) instead of
  // being added into lambda: its solution has entries ~100x its coefficients on
  // one-sided (free-surface, wall) rows, and rounding lambda + d to FP32 would put
  // back an error A * (rounding of lambda) into the moment conditions, which the
  // applied Laplacian sees divided by h.  Its coefficients are evaluated as
  // w (p.lambda + p.lo).
  float lo[M];
#pragma unroll
  for (int r = 0; r < M; ++r) lo[r] = 0.0f;
  if constexpr (REFINE) {
    // residual b - sum_j c_j p_j of the coefficients as they will be stored
    float2 R01[M], R2x[M];
#pragma unroll
    for (int r = 0; r < M; ++r) R01[r] = R2x[r] = make_float2(0.0f, 0.0f);
    for_pairs([&](int, float2 qa, float2 qb, float2 qc, float2 w) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        float2 p[M], s01, s2x;
        basis2<M>(dup2(u ? qa.y : qa.x), dup2(u ? qb.y : qb.x), dup2(u ? qc.y : qc.x), p);
        dots(p, s01, s2x);
        const float2 ww = dup2(u ? w.y : w.x);
        const float2 c01 = mul2(ww, s01), c2x = mul2(ww, s2x);
        R01[0] = add2(R01[0], c01);
        R2x[0] = add2(R2x[0], c2x);
#pragma unroll
        for (int r = 1; r < M; ++r) {
          R01[r] = fma2(c01, p[r], R01[r]);
          R2x[r] = fma2(c2x, p[r], R2x[r]);
        }
      }
    });
    float R[VR];
#pragma unroll
    for (int k = 0; k < VR; ++k) R[k] = 0.0f;
#pragma unroll
    for (int r = 0; r < M; ++r) {
      R[r] = R01[r].x;
      R[M + r] = R01[r].y;
      R[2 * M + r] = R2x[r].x;
      if (NR == 4) R[(NR - 1) * M + r] = R2x[r].y;
    }
    reduce_scatter<G, VR>(R);
#pragma unroll
    for (int k = 0; k < VR / G; ++k) sm[lane * (VR / G) + k] = R[k];
    __syncwarp(gm);
    {
      // the corrections
      solve_all([&](int k, int r) { return rhs<M, float>(k, r) - sm[k * M + r]; });
#pragma unroll
      for (int r = 0; r < M; ++r) {
        l01[r].x += sm[r];
        l01[r].y += sm[M + r];
        if (NR == 4) l2x[r].x += sm[2 * M + r];
        lo[r] = sm[KL * M + r];
        if (NR == 3) l2x[r].y = lo[r];
      }
    }
    __syncwarp(gm);
  }
  // ---- coefficients: w p.lambda_k (+ w p.lo for the Laplacian) with the
  // operator's scale 1/h or 1/h^2 folded into w (the products are taken onto +0,
  // so an entry of the other model gets +0 whatever the sign of its sum)
  const float2 zero = make_float2(0.0f, 0.0f);
  for_pairs([&](int e, float2 qa, float2 qb, float2 qc, float2 w) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      float2 p[M], s01, s2x;
      basis2<M>(dup2(u ? qa.y : qa.x), dup2(u ? qb.y : qb.x), dup2(u ? qc.y : qc.x), p);
      dots(p, s01, s2x);
      const float wu = u ? w.y : w.x, wg = wu * hinv, wl = wu * h2inv;
      float4 out;
      if constexpr (M == 10) {
        if constexpr (REFINE) {
          const float x = p[1].x, y = p[2].x, z = p[3].x;
          const float a = fmaf(x, lo[4], fmaf(y, lo[7], fmaf(z, lo[8], lo[1])));
          const float b = fmaf(y, lo[5], fmaf(z, lo[9], lo[2]));
          s2x.y += fmaf(x, a, fmaf(y, b, fmaf(z, fmaf(z, lo[6], lo[3]), lo[0])));
        }
        const float2 g = fma2(dup2(wg), s01, zero), gl = fma2(make_float2(wg, wl), s2x, zero);
        out = make_float4(g.x, g.y, gl.x, gl.y);
      } else {
        const float sl = s2x.x + s2x.y;   // (s2x.y = p.lo, zero without refinement)
        const float2 gxy = fma2(make_float2(t1[0], t1[1]), dup2(s01.x),
                                mul2(make_float2(t2[0], t2[1]), dup2(s01.y)));
        const float gz = fmaf(s01.x, t1[2], s01.y * t2[2]);
        const float2 g = fma2(dup2(wg), gxy, zero);
        const float2 gl = fma2(make_float2(wg, wl), make_float2(gz, sl), zero);
        out = make_float4(g.x, g.y, gl.x, gl.y);
      }
      if (u == 0 || e + G < len) st4(coef + e + u * G, out);
    }
  });
  *result = 0;
  *cond_out = cond;
}

// ------------------------------------------------------------ FP64 arithmetic
// Process particle i in FP64 (TS storage) with a group of G lanes.  Returns
// (through *result) 0 = written, 1 = deficient (zeros written).  wc: the lane's
// cache of KC weights (KC = 0: none), 32 apart.
template <typename TS, int M, int G, int KC = 0>
__device__ void stencil_particle(int64_t i, const vec4_t<TS> *pos, const uint8_t *model,
                                 const vec4_t<TS> *frame, const long long *row_ptr,
                                 const int32_t *col, vec4_t<TS> *coef,
                                 const StParams<double> &sp, double *sm, int *result,
                                 float *cond_out, double *wc = nullptr) {
  using C = double;
  constexpr int NA = Basis<M>::NA, NR = Basis<M>::NR;
  using V = vec4_t<TS>;
  const int lane = threadIdx.x & (G - 1);
  const unsigned gm = group_mask<G>();
  const V xi = ld4(pos + i);
  const uint8_t mi = model[i];
  const C hinv = C(1) / C(xi.w);
  C t1[3] = {0, 0, 0}, t2[3] = {0, 0, 0};
  if constexpr (M == 6) {
    const V f1 = ld4(frame + 2 * i), f3 = ld4(frame + 2 * i + 1);
    t1[0] = C(f1.x); t1[1] = C(f1.y); t1[2] = C(f1.z);
    const C n0 = C(f3.x), n1 = C(f3.y), n2 = C(f3.z);
    t2[0] = n1 * t1[2] - n2 * t1[1];
    t2[1] = n2 * t1[0] - n0 * t1[2];
    t2[2] = n0 * t1[1] - n1 * t1[0];
  }
  const long long b = row_ptr[i], e1 = row_ptr[i + 1];
  // ---- moments (the distinct ones)
  constexpr int VM = pad_to(Moments<M>::N, G);
  C A[VM];
#pragma unroll
  for (int k = 0; k < VM; ++k) A[k] = C(0);
  int cnt = 0;
  int kk = 0;   // this lane's running entry index: entry b + lane + kk G
  for (long long e0 = b + lane; e0 < e1; e0 += kGatherU<M> * G, kk += kGatherU<M>) {
    V xs[kGatherU<M>];
    bool oks[kGatherU<M>];
    gather_row<kGatherU<M>, G>(e0, e1, i, mi, col, pos, model, xs, oks);
#pragma unroll
    for (int u = 0; u < kGatherU<M>; ++u) {
      C p[M];
      C w = basis_at<M, C>(xi, xs[u], hinv, t1, t2, sp, p);
      w = oks[u] ? w : C(0);   // other model / past the row end: contributes exact zeros
      cnt += oks[u] ? 1 : 0;
      if constexpr (KC > 0) {
        if (kk + u < KC) wc[(kk + u) * 32] = w;
      }
      add_moments<M, C, VM>(A, w, p);
    }
  }
  cnt = group_sum<G>(cnt);
  reduce_scatter<G, VM>(A);
  __syncwarp(gm);
#pragma unroll
  for (int k = 0; k < VM / G; ++k) sm[lane * (VM / G) + k] = A[k];
  __syncwarp(gm);
  C L[NA];
  constexpr MomentTable<M> MT = Moments<M>::T;
#pragma unroll
  for (int k = 0; k < NA; ++k) L[k] = sm[MT.idx[k]];
  __syncwarp(gm);
  C tr = 0;
#pragma unroll
  for (int r = 0; r < M; ++r) tr += L[pk(r, r)];
  C invd[M], pmin, pmax;
  const bool pd = cholesky<M, C, true>(L, invd, sp.piv_tol_rel * tr, pmin, pmax);
  const bool ok = pd && cnt >= M;
  const C cond = (pmax / pmin) * (pmax / pmin);
  C *Ls = sm + StSmem<M, G>::SCR;
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NA; ++k) Ls[k] = L[k];
  }
  __syncwarp(gm);
  if (!ok) {
    for (long long e = b + lane; e < e1; e += G) st4(coef + e, mk4<TS>(0, 0, 0, 0));
    *result = 1;
    *cond_out = INFINITY;
    return;
  }
  // ---- solve: one right-hand side per lane, as in the FP32 rows
  static_assert(G >= NR, "one lane per right-hand side");
  const int kq = lane % NR;
  C lam[NR][M];
  {
    C bb[M], x[M];
#pragma unroll
    for (int r = 0; r < M; ++r) bb[r] = rhs<M, C>(kq, r);
    chol_solve_s<M, C>(Ls, invd, bb, x);
    if (lane < NR) {
#pragma unroll
      for (int r = 0; r < M; ++r) sm[lane * M + r] = x[r];
    }
    __syncwarp(gm);
#pragma unroll
    for (int k = 0; k < NR; ++k)
#pragma unroll
      for (int r = 0; r < M; ++r) lam[k][r] = sm[k * M + r];
    __syncwarp(gm);
  }
  // ---- coefficients
  const C h2inv = hinv * hinv;
  // the output record of one entry: w p.lambda_k with the operator's scale 1/h or
  // 1/h^2 folded into w
  auto coef_of = [&](const C (&p)[M], C w) -> vec4_t<TS> {
    const C wg = w * hinv, wl = w * h2inv;
    C s[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      C v = lam[k][0];   // p_0 = 1
#pragma unroll
      for (int r = 1; r < M; ++r) v = fma(p[r], lam[k][r], v);
      s[k] = v;
    }
    if constexpr (M == 10) {
      return mk4<TS>(TS(wg * s[0]), TS(wg * s[1]), TS(wg * s[2]), TS(wl * s[3]));
    } else {
      const C gx = wg * fma(s[0], t1[0], s[1] * t2[0]);
      const C gy = wg * fma(s[0], t1[1], s[1] * t2[1]);
      const C gz = wg * fma(s[0], t1[2], s[1] * t2[2]);
      return mk4<TS>(TS(gx), TS(gy), TS(gz), TS(wl * s[2]));
    }
  };
  kk = 0;
  for (long long e0 = b + lane; e0 < e1; e0 += kGatherU<M> * G, kk += kGatherU<M>) {
    V xs[kGatherU<M>];
    bool oks[kGatherU<M>];
    gather_row<kGatherU<M>, G>(e0, e1, i, mi, col, pos, model, xs, oks);
#pragma unroll
    for (int u = 0; u < kGatherU<M>; ++u) {
      const long long e = e0 + (long long)u * G;
      if (e >= e1) break;
      vec4_t<TS> out = mk4<TS>(0, 0, 0, 0);
      if (oks[u]) {
        C p[M], w;
        if (KC > 0 && kk + u < KC) {
          basis_only<M, C>(xi, xs[u], hinv, t1, t2, p);
          w = wc[(kk + u) * 32];
        } else {
          w = basis_at<M, C>(xi, xs[u], hinv, t1, t2, sp, p);
        }
        out = coef_of(p, w);
      }
      st4(coef + e, out);
    }
  }
  *result = 0;
  *cond_out = (float)cond;
}

// Main kernel: every particle of model (M == 10 ? 3D : 2D).  A warp looks at
// `rounds` x 32 / G consecutive particles, and its groups share those of its
// model out, so that a warp of the other model ends at once (a film alone spent
// 57 us in the 3D kernel when every group tested its own particles one by one)
// and mixed warps leave no group idle but in their last round.
template <typename TS, typename C, int M, int G, bool REFINE>
__global__ void __launch_bounds__(kBuildThreads, sizeof(C) == 4 ? (M == 10 ? 7 : 10) : 1) k_stencil(
    int64_t n, const vec4_t<TS> *pos, const uint8_t *model, const vec4_t<TS> *frame,
    const long long *row_ptr, const int32_t *col, vec4_t<TS> *coef, uint8_t *status,
    float *cond, StParams<C> sp, DevStatus *st, int32_t *queue, int rounds) {
  pdl_wait();
  constexpr int SMG = StSmem<M, G>::PER_GROUP, KC = StCache<C, M, G>::KC, ROWS = 32 / G;
  extern __shared__ __align__(16) unsigned char st_smem[];
  C *sm = reinterpret_cast<C *>(st_smem + StCache<C, M, G>::BYTES) + threadIdx.x / G * SMG;
  const int lane = threadIdx.x & (G - 1), wl = threadIdx.x & 31;
  const uint8_t want = M == 10 ? MAFP_MODEL_3D : MAFP_MODEL_2D;
  const int64_t i0 = ((int64_t)blockIdx.x * (kBuildThreads / 32) + threadIdx.x / 32) * rounds * ROWS;
  unsigned todo = __ballot_sync(0xffffffffu, wl < rounds * ROWS && i0 + wl < n &&
                                                 model[i0 + wl] == want);
  while (todo) {
    // group g takes the g-th of the next ROWS particles
    unsigned mine = todo;
    for (int k = 0; k < wl / G; ++k) mine &= mine - 1;
#pragma unroll
    for (int k = 0; k < ROWS; ++k) todo &= todo - 1;
    if (mine) {
      const int64_t i = i0 + __ffs(mine) - 1;
      int res;
      float cd = 0.0f;
      if constexpr (sizeof(C) == 4) {
        float4 *qw = reinterpret_cast<float4 *>(st_smem) + threadIdx.x / 32 * KC * 32 + wl;
        stencil_row32<M, G, REFINE>(i, pos, model, frame, row_ptr, col, coef, sp, sm, &res, &cd,
                                    qw);
      } else {
        double *wc = reinterpret_cast<double *>(st_smem) + threadIdx.x / 32 * KC * 32 + wl;
        stencil_particle<TS, M, G, KC>(i, pos, model, frame, row_ptr, col, coef, sp, sm, &res, &cd,
                                       wc);
      }
      if (lane == 0) {
        if (res == 2) {
          queue[atomicAdd(&st->fallback_count, 1)] = (int32_t)i;
        } else {
          status[i] = res == 0 ? MAFP_STENCIL_OK : MAFP_STENCIL_DEFICIENT;
          cond[i] = res == 0 ? cd : INFINITY;
          if (res == 1) inc_ll(&st->n_deficient);
        }
      }
    }
    __syncwarp();
  }
}

// FP64 redo of the queued particles (FP32 storage), 3D and film by turns.
template <int M, int G>
__device__ __forceinline__ void stencil_redo(const float4 *pos, const uint8_t *model,
                                             const float4 *frame, const long long *row_ptr,
                                             const int32_t *col, float4 *coef, uint8_t *status,
                                             float *cond, const StParams<double> &sp,
                                             DevStatus *st, const int32_t *queue, double *smem) {
  double *sm = smem + threadIdx.x / G * StSmem<M, G>::PER_GROUP;
  const int lane = threadIdx.x & (G - 1);
  const int64_t gid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
  const int64_t ngroups = ((int64_t)gridDim.x * blockDim.x) / G;
  const int nq = st->fallback_count;
  const uint8_t want = M == 10 ? MAFP_MODEL_3D : MAFP_MODEL_2D;
  for (int64_t q = gid; q < nq; q += ngroups) {
    const int64_t i = queue[q];
    if (model[i] != want) continue;
    int res;
    float cd = 0.0f;
    stencil_particle<float, M, G>(i, pos, model, frame, row_ptr, col, coef, sp, sm, &res, &cd);
    if (lane == 0) {
      status[i] = res == 0 ? MAFP_STENCIL_FP64 : MAFP_STENCIL_DEFICIENT;
      cond[i] = res == 0 ? cd : INFINITY;
      if (res == 1) inc_ll(&st->n_deficient);
      else inc_ll(&st->n_fp64_stencil);
    }
  }
}

constexpr int kRedoG = 4;   // small groups: the factorisation is repeated in every lane
__global__ void __launch_bounds__(kBuildThreads) k_stencil_redo(
    const float4 *pos, const uint8_t *model, const float4 *frame, const long long *row_ptr,
    const int32_t *col, float4 *coef, uint8_t *status, float *cond, StParams<double> sp,
    DevStatus *st, const int32_t *queue) {
  pdl_wait();
  static_assert(StSmem<6, kRedoG>::PER_GROUP <= StSmem<10, kRedoG>::PER_GROUP, "film fits");
  __shared__ double smem[(kBuildThreads / kRedoG) * StSmem<10, kRedoG>::PER_GROUP];
  stencil_redo<10, kRedoG>(pos, model, frame, row_ptr, col, coef, status, cond, sp, st, queue, smem);
  __syncthreads();   // the scratch is laid out anew
  stencil_redo<6, kRedoG>(pos, model, frame, row_ptr, col, coef, status, cond, sp, st, queue, smem);
}


template <typename TS, typename C, int M, int G, bool REFINE>
static void launch_stencil(mafp_ctx *ctx, cudaStream_t s, int64_t n, const void *pos_h,
                           const uint8_t *model, const void *frame, const long long *rp,
                           const int32_t *col, void *coef, uint8_t *status, float *cond,
                           const StParams<C> &sp) {
  using V = vec4_t<TS>;
  static const KernelName name("k_stencil<%s,M=%d,G=%d,%s>", sizeof(TS) == 4 ? "f32" : "f64",
                               M, G, REFINE ? "refined" : "plain");
  const int rounds = rounds_of<C, M>(n);
  static_assert(G >= 4, "a warp looks at 32 particles at most");
  const int blocks = (int)((n + (int64_t)rounds * kBuildThreads / G - 1) / (rounds * kBuildThreads / G));
  constexpr int smem = StCache<C, M, G>::SMEM;
  static_assert(smem <= 48 * 1024, "more has to be asked for, per device and function");
  MAFP_TIMED(ctx, s, name.s,
             launch(k_stencil<TS, C, M, G, REFINE>, blocks, kBuildThreads, smem, s, 
                 n, (const V *)pos_h, model, (const V *)frame, rp, col, (V *)coef, status, cond,
                 sp, ctx->d_status, ctx->fallback, rounds));
}

// Lanes per particle.  Clouds of more than kStFewRows: the context's stencil3d_group and
// stencil2d_group, whose default values stand for 8 (3D's 32) and, in FP64, for 4 (film's
// 8).  More lanes repeat the factorisation and leave part of a row's last gather empty --
// 3D, FP32, 8 / 16 / 32 lanes: cube of 20k particles 59 / 60 / 76 us, 80k 164 / 193 / 275;
// FP64, cube 20k 924 / 996 / 1310, jet on a film 40k 677 / 650 / 737; film, FP64, 4 / 8 / 16
// lanes: 20k 216 / 244 / 348, 80k 709 / 869 / 1290.  Smaller clouds, whose rows do not fill
// the GPU: 32 lanes in 3D and, in FP64, 8 on film, whatever is asked for (FP32, cube 4852
// 40 / 32 / 36 us, 10k 45 / 45 / 50; FP64, jet 10k 255 / 208 / 202, cube 5k 292 / 332 / 334);
// their sums are shorter chains too: with 8 and 4 lanes the FP64 outputs lie 0 to 5 %
// further from the exact ones (film 6000 particles 6.7e-15 for 6.4e-15).  Film, FP32:
// always as asked for; the lanes set the order of the sums there, and the Laplacians of a
// curved film are small differences, whose gradients show every change of rounding.
template <typename TS, typename C, bool REFINE>
static int dispatch_stencils(mafp_ctx *ctx, cudaStream_t s, int64_t n, const void *pos_h,
                             const uint8_t *model, const void *frame, const long long *rp,
                             const int32_t *col, void *coef, uint8_t *status, float *cond,
                             const StParams<C> &sp) {
  const bool few = n <= kStFewRows;
  int g3 = ctx->tune.stencil3d_group, g2 = ctx->tune.stencil2d_group;
  if (few) g3 = 32;
  else if (g3 == 32) g3 = 8;
  if (sizeof(C) == 8) g2 = few ? 8 : (g2 == 8 ? 4 : g2);
  switch (g3) {
    case 8: launch_stencil<TS, C, 10, 8, REFINE>(ctx, s, n, pos_h, model, frame, rp, col, coef, status, cond, sp); break;
    case 16: launch_stencil<TS, C, 10, 16, REFINE>(ctx, s, n, pos_h, model, frame, rp, col, coef, status, cond, sp); break;
    default: launch_stencil<TS, C, 10, 32, REFINE>(ctx, s, n, pos_h, model, frame, rp, col, coef, status, cond, sp); break;
  }
  switch (g2) {
    case 4: launch_stencil<TS, C, 6, 4, REFINE>(ctx, s, n, pos_h, model, frame, rp, col, coef, status, cond, sp); break;
    case 16: launch_stencil<TS, C, 6, 16, REFINE>(ctx, s, n, pos_h, model, frame, rp, col, coef, status, cond, sp); break;
    default: launch_stencil<TS, C, 6, 8, REFINE>(ctx, s, n, pos_h, model, frame, rp, col, coef, status, cond, sp); break;
  }
  MAFP_LAUNCH_CHECK(ctx);
  return MAFP_OK;
}

int build_stencils(mafp_ctx *ctx, int64_t n, int32_t dtype, const void *pos_h,
                   const uint8_t *model, const void *frame, const int64_t *row_ptr,
                   const int32_t *col, void *coef, uint8_t *status, float *cond, cudaStream_t s) {
  const long long *rp = reinterpret_cast<const long long *>(row_ptr);
  const int sms = sm_count();
  if (dtype == MAFP_F64) {
    const StParams<double> sp = make_params<double>(ctx->prm, 1e-12);
    return dispatch_stencils<double, double, false>(ctx, s, n, pos_h, model, frame, rp,
                                                          col, coef, status, cond, sp);
  }
  const StParams<float> sp = make_params<float>(ctx->prm, 1e-6);
  const StParams<double> sp64 = make_params<double>(ctx->prm, 1e-12);
  MAFP_TIMED(ctx, s, "k_reset_queue", launch(k_reset_queue, 1, 1, 0, s, ctx->d_status));
  int rc = dtype == MAFP_F32_PLAIN
               ? dispatch_stencils<float, float, false>(ctx, s, n, pos_h, model, frame, rp,
                                                             col, coef, status, cond, sp)
               : dispatch_stencils<float, float, true>(ctx, s, n, pos_h, model, frame, rp,
                                                            col, coef, status, cond, sp);
  if (rc) return rc;
  MAFP_TIMED(ctx, s, "k_stencil_redo",
             launch(k_stencil_redo, sms * 8, kBuildThreads, 0, s, (const float4 *)pos_h, model,
                    (const float4 *)frame, rp, col, (float4 *)coef, status, cond, sp64,
                    ctx->d_status, ctx->fallback));
  MAFP_LAUNCH_CHECK(ctx);
  return MAFP_OK;
}

}  // namespace mafp
