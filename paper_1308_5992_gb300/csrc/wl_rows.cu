// wl_rows.cu -- row-block form of the tile-coloured Kaczmarz sweep (Sec. 3.1)
// for the FP32 and BF16-stored cycles.
//
// A sweep relaxes one unknown after the other: s_i = omega <r, A e_i> / den_i,
// x_i += s_i, r -= s_i A e_i.  For a block of unknowns taken in order this is
// the same as forming every <r, A e_i> from the r the block starts with and
// then solving a small triangular system, since
//   <r - sum_{j<i} s_j A e_j, A e_i> = <r, A e_i> - sum_{j<i} K_ij s_j,
//   K_ij = <A e_j, A e_i>,
// so s = T (<r, A e_i>)_i with T = (den / omega on the diagonal, K below)^-1,
// a constant of the level.  Here a block is one row of a tile (8 sites, 16
// unknowns): the 16 dependent colour steps of a tile become 4 row steps (rows
// i and i + 4 at once, which share no cell of r), at the cost of the product
// with T, 12 of 48 complex multiply-adds per unknown.  T is formed in FP64
// from the stored stencil and rounded once.
//
// Within a row the order is that of wl_tile_order.h: even rows 0 1 2 3, odd
// rows 3 2 1 0 in each 4-site cell, both cells at once.  Two sites couple when
// at most two columns apart, so a cell needs its own 8 inner products and, for
// the left cell of an even row (the right cell of an odd one), 4 of the other
// cell: T has 12 columns.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>

#include "wl_common.cuh"
#include "wl_tile_order.h"

namespace cg = cooperative_groups;

#define RB_KT 8
#define RB_W 10    // window side: tile and halo
#define RB_RS 209  // complex floats between the r windows of two right-hand sides in shared memory:
                   // 200 used; 2 * 209 = 2 (mod 32) puts consecutive right-hand sides in
                   // consecutive bank pairs for the transposing copies

// bytes of one row step of a packed tile: per lane the stencil entries of its
// site for its spin (9 offsets x 2 rows) and its row of T (12 entries)
template <typename S>
__host__ __device__ constexpr int rb_step_bytes() {
  return 32 * (9 * 2 * (int)sizeof(S) + 12 * (int)sizeof(zf));
}

__device__ __forceinline__ int rb_site(const Geo &g, int A0, int B0, int i, int j) {
  int a = A0 + i, b = B0 + j;
  return g.idx(a + b, a - b);
}

// tile `t` of tile colour tc: its origin
__device__ __forceinline__ void rb_origin(const Geo &g, int tc, int t, int &A0, int &B0) {
  int nb4 = g.N / (4 * RB_KT);
  A0 = ((tc & 1) + 2 * (t / nb4)) * RB_KT;
  B0 = ((tc >> 1) + 2 * (t % nb4)) * RB_KT;
}

// stored coefficient as complex double (floats widened on the integer pipes)
__device__ __forceinline__ zd rb_ld64(const zd *p) { return *p; }
__device__ __forceinline__ zd rb_ld64(const zf *p) { return widen<double>(*p); }
__device__ __forceinline__ zd rb_ld64(const zb *p) { return widen<double>(ld<float>(p)); }

// K = <A e_(h2,t2), A e_(h,t)> for sites h, h2 of one row, h2 = h + delta
// columns (|delta| <= 2): column (h, t) has the entries g_s g_t conj(A[h][d][t][s])
template <typename S>
__device__ zd rb_gram(const S *__restrict__ A, int h, int t, int h2, int t2, int delta) {
  zd k = mk(0.0, 0.0);
  for (int da = 0; da < 3; ++da)
    for (int db = 0; db < 3; ++db) {
      int eb = db - delta;  // the same cell seen from h2
      if (eb < 0 || eb > 2) continue;
      const S *p = A + ((long)h * 9 + da * 3 + db) * 4 + t * 2;
      const S *q = A + ((long)h2 * 9 + da * 3 + eb) * 4 + t2 * 2;
      for (int s = 0; s < 2; ++s) k = k + rb_ld64(p + s) * cconj(rb_ld64(q + s));
    }
  double f = (t ^ t2) ? -1.0 : 1.0;
  return mk(f * k.re, f * k.im);
}

// 16 threads per cell of 4 sites: its stencil entries and rows of T, packed in
// the lane order of k_kacz_rows ([tile colour][tile][step][9 + 6][32 lanes]).
// Thread i < 12 forms row i of the block's matrix (in the order of
// relaxation), then column i of its inverse by forward substitution.
#define RBP_CELLS 8
template <typename S>
__global__ void __launch_bounds__(16 * RBP_CELLS) k_rows_pack(Geo g, const S *__restrict__ A, double omega,
                                                              unsigned char *__restrict__ out) {
  __shared__ zd Ms[RBP_CELLS][12][13];
  const int ntile = (g.N / (2 * RB_KT)) * (g.N / (4 * RB_KT));
  const int lc = threadIdx.x >> 4, i = threadIdx.x & 15;
  const int id = blockIdx.x * RBP_CELLS + lc;  // 16 cells a tile: the grid is exact
  const int cell = id & 1, grp = (id >> 1) & 1, step = (id >> 2) & 3, tile = id >> 4;  // tile counts through the colours
  int A0, B0;
  rb_origin(g, tile / ntile, tile % ntile, A0, B0);
  const int row = step + 4 * grp;
  const bool rev = step & 1;
  const bool dep = cell == (rev ? 1 : 0);  // needs the other cell's first two sites
  // site v = 0..5 of the order of relaxation: own sites, and the other cell's
  // first two after the own ones of the same colour (in a cell that needs no
  // other site v = 4, 5 are unused: unit rows)
  auto column = [&](int v) -> int {
    if (!dep) return v < 4 ? cell * 4 + (rev ? 3 - v : v) : -1;
    const int u = v < 4 ? v >> 1 : v - 2, j = rev ? 3 - u : u;  // own, other, own, other, own, own
    return ((v < 4 && (v & 1)) ? 1 - cell : cell) * 4 + j;
  };
  if (i < 12) {
    const int p = i >> 1, t = i & 1, cp = column(p);
    for (int q = 0; q < 6; ++q) {
      const int cq = column(q), dl = cq - cp;
      for (int t2 = 0; t2 < 2; ++t2) {
        zd k = mk(0.0, 0.0);
        if (2 * q + t2 <= i) {
          if (cp < 0 || cq < 0) {
            if (2 * q + t2 == i) k = mk(1.0, 0.0);
          } else if (dl >= -2 && dl <= 2) {
            k = rb_gram(A, rb_site(g, A0, B0, row, cp), t, rb_site(g, A0, B0, row, cq), t2, dl);
            if (2 * q + t2 == i) k = mk(k.re / omega, 0.0);
          }
        }
        Ms[lc][i][2 * q + t2] = k;
      }
    }
  }
  __syncthreads();
  unsigned char *so = out + ((long)tile * 4 + step) * rb_step_bytes<S>();
  S *oa = (S *)so;
  zf *ot = (zf *)(so + 32 * 18 * sizeof(S));
  if (i < 12) {
    const int cq = column(i >> 1), kq = cq < 0 ? 0 : cq / 4 == cell ? 2 * (cq & 3) + (i & 1)
                                       : 8 + 2 * (rev ? (cq & 3) - 2 : (cq & 3)) + (i & 1);  // this column of T
    zd X[12];
#pragma unroll
    for (int r = 0; r < 12; ++r) {
      zd v = mk(r == i ? 1.0 : 0.0, 0.0);
#pragma unroll
      for (int q = 0; q < r; ++q) v = v - Ms[lc][r][q] * X[q];
      double d = Ms[lc][r][r].re;
      X[r] = mk(v.re / d, v.im / d);
      const int cr = column(r >> 1);
      if (cq >= 0 && cr >= 0 && cr / 4 == cell)
        ot[((kq >> 1) * 32 + grp * 16 + cr * 2 + (r & 1)) * 2 + (kq & 1)] = ccast<float>(X[r]);
    }
  }
  if (!dep)  // the columns of the other cell's sites
    for (int e = i; e < 32; e += 16) {
      int u = e >> 2, k = 8 + (e & 3);
      ot[((k >> 1) * 32 + grp * 16 + cell * 8 + u) * 2 + (k & 1)] = mk(0.f, 0.f);
    }
  for (int e = i; e < 4 * 36; e += 16) {
    int b = cell * 4 + e / 36, c = e % 36, d = c >> 2, t = (c >> 1) & 1, p = c & 1;
    oa[(d * 32 + grp * 16 + b * 2 + p) * 2 + t] = A[(long)rb_site(g, A0, B0, row, b) * 36 + c];
  }
}

// stencil entries (rows t = 0 and 1) of one offset, or two entries of T
__device__ __forceinline__ void rb_ld(const zf *p, float2 &a0, float2 &a1) {
  float4 v = *(const float4 *)p;
  a0 = make_float2(v.x, v.y);
  a1 = make_float2(v.z, v.w);
}
__device__ __forceinline__ void rb_ld(const zb *p, float2 &a0, float2 &a1) {
  uint2 u = *(const uint2 *)p;
  a0 = __bfloat1622float2(*(const __nv_bfloat162 *)&u.x);
  a1 = __bfloat1622float2(*(const __nv_bfloat162 *)&u.y);
}
__device__ __forceinline__ float2 rb_swap(float2 v) { return make_float2(v.y, v.x); }
__device__ __forceinline__ float2 rb_shfl_xor1(float2 v) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, 1), __shfl_xor_sync(0xffffffffu, v.y, 1));
}

// One tile colour (a quarter of a sweep): a block per tile and chunk of R
// right-hand sides, a warp per RPT of them.  Lane (row group, column b, spin
// p) = (lane / 16, (lane / 2) % 8, lane % 2) forms the partial products of its
// site's two unknowns over the nine cells of spin p, the pair of lanes of a
// site swaps halves, the 12 inner products a row of T needs go through shared
// memory, and the update of r is summed per column with the neighbours' parts
// taken by shuffles.  A warp never waits for another one between the first
// and the last barrier; its RPT right-hand sides go through each phase
// together, so that their latencies overlap.  Complex products are paired
// FMAs on (re, im) pairs as they lie in memory: sum (a.re x.re, a.im x.im) and
// sum (a.re x.im, a.im x.re), combined once per sum.  The tile's packed rows
// arrive as one bulk copy per row step, all four issued at the start (bounded
// waits; on a timeout *timeout gets 1, r is not written and x may be partly). x and r are not
// declared restrict: their loads have to stay after griddepcontrol.wait.
template <typename S, int R, int RPT>
__global__ void __launch_bounds__(32 * R / RPT, RPT == 1 ? 16 / R : 0) k_kacz_rows(Geo g, int tc, const unsigned char *__restrict__ pk,
                                                            zf *x, zf *r, int nrhs, int *timeout) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  constexpr int NT = 32 * R / RPT, NW = R / RPT, SB = rb_step_bytes<S>();
  unsigned char *cs = sm_raw;                           // [4][SB] packed rows
  float2 *rs = (float2 *)(sm_raw + 4 * SB);             // [R][RB_RS] r of tile + halo, [site][spin]
  float2 *nums = rs + ((R * RB_RS + 1) & ~1);           // [NW][RPT][2][20] inner products
  int *hs = (int *)(nums + R * 40);                     // [100] site index of tile + halo
  uint64_t *mbar = (uint64_t *)(hs + RB_W * RB_W);      // [4], 8-byte aligned: every part above is a multiple of 8
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int ntile = (g.N / (2 * RB_KT)) * (g.N / (4 * RB_KT));
  const int r0 = blockIdx.y * R, Rc = min(R, nrhs - r0);
  int A0, B0;
  rb_origin(g, tc, blockIdx.x, A0, B0);
  if (tid == 0) {
    for (int i = 0; i < 4; ++i) mbar_init(smem_u32(&mbar[i]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    const unsigned char *src = pk + ((long)tc * ntile + blockIdx.x) * 4 * SB;
    for (int i = 0; i < 4; ++i) {
      mbar_arrive_expect_tx(smem_u32(&mbar[i]), SB);
      bulk_g2s(smem_u32(cs + i * SB), src + i * SB, SB, smem_u32(&mbar[i]));
    }
  }
  for (int ls = tid; ls < RB_W * RB_W; ls += NT) hs[ls] = rb_site(g, A0, B0, ls / RB_W - 1, ls % RB_W - 1);
  __syncthreads();
  // this thread's elements of the window, in global and in shared memory
  constexpr int NE = (RB_W * RB_W * 2 * R + NT - 1) / NT;
  float2 *ga[NE];
#pragma unroll
  for (int i = 0; i < NE; ++i) {
    int e = tid + i * NT, q = e % R, row = e / R;
    bool in = e < RB_W * RB_W * 2 * R && q < Rc;
    ga[i] = in ? (float2 *)r + ((long)hs[row >> 1] * 2 + (row & 1)) * nrhs + r0 + q : nullptr;
  }
  const int grp = lane >> 4, b = (lane >> 1) & 7, p = lane & 1;
  const int q0 = w * RPT;
  bool act[RPT];
#pragma unroll
  for (int m = 0; m < RPT; ++m) act[m] = q0 + m < Rc;
  float2 *xa[4];  // x of this lane's unknown in the four row steps
#pragma unroll
  for (int st = 0; st < 4; ++st)
    xa[st] = (float2 *)x + ((long)hs[(st + 4 * grp + 1) * RB_W + b + 1] * 2 + p) * nrhs + r0 + q0;
  // r and x are the previous launch's
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
#pragma unroll
  for (int i = 0; i < NE; ++i) {
    int e = tid + i * NT;
    if (ga[i])
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_u32(rs + (e % R) * RB_RS + e / R)),
                   "l"(ga[i]));
  }
  float2 xp[4][RPT];
#pragma unroll
  for (int st = 0; st < 4; ++st)
#pragma unroll
    for (int m = 0; m < RPT; ++m)
      if (act[m]) xp[st][m] = xa[st][m];
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  const bool edge = b == 0 || b == 7;
  const int eo = b == 0 ? 0 : 4;  // the halo column an edge lane also updates, from its own column - 1
  const float ml = b == 0 ? 0.f : 1.f, mr = b == 7 ? 0.f : 1.f;
  float2 *nw = nums + w * RPT * 40 + grp * 20;
  const int own = (b >> 2) * 8;
  bool ok = true;
#pragma unroll
  for (int st = 0; st < 4; ++st) {
    ok = ok && mbar_wait(smem_u32(&mbar[st]), 0, 1000000000ull);
    if (!__all_sync(0xffffffffu, ok)) {
      ok = false;
      break;
    }
    float2 a0[9], a1[9], T[12];
    const S *ca = (const S *)(cs + st * SB);
    const zf *ct = (const zf *)(cs + st * SB + 32 * 18 * sizeof(S));
#pragma unroll
    for (int d = 0; d < 9; ++d) rb_ld(ca + (d * 32 + lane) * 2, a0[d], a1[d]);
    float2 *rq = rs + q0 * RB_RS + ((st + 4 * grp) * RB_W + b) * 2 + p;
    float2 rc[RPT][3], re[RPT][3];  // own column and, on edge lanes, the halo column beside it
#pragma unroll
    for (int m = 0; m < RPT; ++m) {
      float2 d0 = make_float2(0.f, 0.f), d1 = d0, e0 = d0, e1 = d0;
#pragma unroll
      for (int d = 0; d < 9; ++d) {
        float2 v = rq[m * RB_RS + ((d / 3) * RB_W + d % 3) * 2], vs = rb_swap(v);
        d0 = __ffma2_rn(a0[d], v, d0);
        e0 = __ffma2_rn(a0[d], vs, e0);
        d1 = __ffma2_rn(a1[d], v, d1);
        e1 = __ffma2_rn(a1[d], vs, e1);
        if (d % 3 == 1) rc[m][d / 3] = v;
        if (d % 3 == 0) re[m][d / 3] = v;
        if (d % 3 == 2 && b == 7) re[m][d / 3] = v;
      }
      float2 P0 = make_float2(d0.x - d0.y, e0.x + e0.y), P1 = make_float2(d1.x - d1.y, e1.x + e1.y);
      float2 mine = p ? P1 : P0, recv = rb_shfl_xor1(p ? P0 : P1);
      nw[m * 40 + b * 2 + p] = make_float2(mine.x - recv.x, mine.y - recv.y);
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) rb_ld(ct + (k * 32 + lane) * 2, T[2 * k], T[2 * k + 1]);
    __syncwarp();
    const int oth = (st & 1) ? 4 : 8;  // the 4 inner products beside the own cell's 8
    float2 m0[RPT], m1[RPT];
#pragma unroll
    for (int m = 0; m < RPT; ++m) {
      float2 d0 = make_float2(0.f, 0.f), e0 = d0, d1 = d0, e1 = d0;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        float4 v = *(const float4 *)(nw + m * 40 + (k < 4 ? own + 2 * k : oth + 2 * (k - 4)));
        d0 = __ffma2_rn(T[2 * k], make_float2(v.x, v.y), d0);
        e0 = __ffma2_rn(T[2 * k], make_float2(v.y, v.x), e0);
        d1 = __ffma2_rn(T[2 * k + 1], make_float2(v.z, v.w), d1);
        e1 = __ffma2_rn(T[2 * k + 1], make_float2(v.w, v.z), e1);
      }
      float2 s = make_float2((d0.x - d0.y) + (d1.x - d1.y), (e0.x + e0.y) + (e1.x + e1.y));
      if (act[m]) xa[st][m] = make_float2(xp[st][m].x + s.x, xp[st][m].y + s.y);
      float2 so = rb_shfl_xor1(s);
      // r_(d,p) -= g_p sum_t g_t s_t conj(a[d][t][p])
      m0[m] = p ? make_float2(-so.x, -so.y) : s;
      m1[m] = p ? s : make_float2(-so.x, -so.y);
    }
#pragma unroll
    for (int m = 0; m < RPT; ++m) {
      float2 dl[9], n0 = rb_swap(m0[m]), n1 = rb_swap(m1[m]);
#pragma unroll
      for (int d = 0; d < 9; ++d) {  // m0 conj(a0) + m1 conj(a1)
        float2 u = __ffma2_rn(a1[d], m1[m], __fmul2_rn(a0[d], m0[m]));
        float2 v = __ffma2_rn(a1[d], n1, __fmul2_rn(a0[d], n0));
        dl[d] = make_float2(u.x + u.y, v.x - v.y);
      }
      float2 up[3], dn[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        up[i] = make_float2(__shfl_up_sync(0xffffffffu, dl[i * 3 + 2].x, 2, 16),
                            __shfl_up_sync(0xffffffffu, dl[i * 3 + 2].y, 2, 16));
        dn[i] = make_float2(__shfl_down_sync(0xffffffffu, dl[i * 3].x, 2, 16),
                            __shfl_down_sync(0xffffffffu, dl[i * 3].y, 2, 16));
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        float2 v = dl[i * 3 + 1];
        v = __ffma2_rn(up[i], make_float2(ml, ml), v);
        v = __ffma2_rn(dn[i], make_float2(mr, mr), v);
        rq[m * RB_RS + (i * RB_W + 1) * 2] = make_float2(rc[m][i].x - v.x, rc[m][i].y - v.y);
      }
      if (edge) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          float2 v = b == 0 ? dl[i * 3] : dl[i * 3 + 2];
          rq[m * RB_RS + i * RB_W * 2 + eo] = make_float2(re[m][i].x - v.x, re[m][i].y - v.y);
        }
      }
    }
    __syncwarp();
  }
  if (!__syncthreads_and(ok)) {
    if (tid == 0) {
      mbar_drain(mbar, 4, 0);
      atomicExch(timeout, 1);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < NE; ++i) {
    int e = tid + i * NT;
    if (ga[i]) *ga[i] = rs[(e % R) * RB_RS + e / R];
  }
}

// ------------------------------------------------------------- small levels
// The 16-colour sweep of a 32 x 32 or 16 x 16 level with the same blocks: the
// sites of a row a = const form a ring of N sites (position u; crossing u = N/2
// continues in row a + N/2), and the colours 4 (a mod 4) + (b mod 4) take the
// rings a mod 4 = 0, 1, 2, 3 in turn, in each ring the sites u mod 4 = 0, 1, 2,
// 3.  So a sweep is 4 passes over N / 8 rings each, and in a pass a cell of 4
// sites needs its own 8 inner products and the next cell's first 4.  One block
// per right-hand side, a lane per site of a pass, r and the packed rings in
// shared memory for all sweeps of a level visit, x in registers.
//
// Row of T of unknown (u, t) packed by what its colour j = u mod 4 can need: the
// columns of the cell's colours 0, 1 (all sites), 2, 3 and the next cell's 0
// (j >= 2), the next cell's 1 (j = 3): 15 complex floats a site on average.
template <typename S, int N>
__host__ __device__ constexpr int ring_bytes() {
  return N * (36 * (int)sizeof(S) + 15 * (int)sizeof(zf));
}
// first float4 of the row (t) of T, part q = 0..3, for position u
template <int N>
__host__ __device__ constexpr int ring_t_at(int q, int t, int h, int u) {
  // part 0: 2 float4 a row for all sites; 1: 2 for j >= 2; 2: 1 for j >= 2; 3: 1 for j = 3
  return q == 0   ? (t * 2 + h) * N + u
         : q == 1 ? 4 * N + (t * 2 + h) * (N / 2) + (u >> 2) * 2 + (u & 1)
         : q == 2 ? 6 * N + t * (N / 2) + (u >> 2) * 2 + (u & 1)
                  : 7 * N + t * (N / 4) + (u >> 2);
}

template <typename S, int N>
__global__ void __launch_bounds__(16 * RBP_CELLS) k_rings_pack(Geo g, const S *__restrict__ A, double omega,
                                                               unsigned char *__restrict__ out) {
  __shared__ zd Ms[RBP_CELLS][12][13];
  const int lc = threadIdx.x >> 4, i = threadIdx.x & 15;
  const int id = blockIdx.x * RBP_CELLS + lc;  // N / 4 cells a ring, N / 2 rings: the grid is exact
  const int cell = id % (N / 4), rg = id / (N / 4), pass = rg / (N / 8), row = pass + 4 * (rg % (N / 8));
  auto site = [&](int u) { return g.idx(row + u, row - u); };
  // position of site v = 0..5 of the order of relaxation: own 0, next 0, own 1, next 1, own 2, own 3
  auto column = [&](int v) { return cell * 4 + (v < 4 ? (v >> 1) + 4 * (v & 1) : v - 2); };
  if (i < 12)
    for (int q = 0; q < 6; ++q)
      for (int t2 = 0; t2 < 2; ++t2) {
        const int cp = column(i >> 1), cq = column(q), dl = cq - cp;
        zd k = mk(0.0, 0.0);
        if (2 * q + t2 <= i && dl >= -2 && dl <= 2) k = rb_gram(A, site(cp), i & 1, site(cq), t2, dl);
        if (2 * q + t2 == i) k = mk(k.re / omega, 0.0);
        Ms[lc][i][2 * q + t2] = k;
      }
  __syncthreads();
  unsigned char *so = out + (long)rg * ring_bytes<S, N>();
  S *oa = (S *)so;
  zf *ot = (zf *)(so + N * 36 * sizeof(S));
  if (i < 12) {
    const int v = i >> 1, t2 = i & 1;
    const int k = (v < 4 ? ((v & 1) ? 8 : 0) + 2 * (v >> 1) : 2 * (v - 2)) + t2;  // column of T: own 0..7, next 8..11
    const int q = k < 4 ? 0 : k < 8 ? 1 : k < 10 ? 2 : 3, h = q < 2 ? (k >> 1) & 1 : 0;
    zd X[12];
#pragma unroll
    for (int r = 0; r < 12; ++r) {
      zd w = mk(r == i ? 1.0 : 0.0, 0.0);
#pragma unroll
      for (int c = 0; c < r; ++c) w = w - Ms[lc][r][c] * X[c];
      double d = Ms[lc][r][r].re;
      X[r] = mk(w.re / d, w.im / d);
      const int u = column(r >> 1), j = u & 3;
      if (u < cell * 4 + 4 && (q == 0 || j == 3 || (j == 2 && q < 3)))
        ot[2 * ring_t_at<N>(q, r & 1, h, u) + (k & 1)] = ccast<float>(X[r]);
    }
  }
  for (int e = i; e < 4 * 36; e += 16) {
    int u = cell * 4 + e / 36, c = e % 36;
    oa[((c >> 1) * N + u) * 2 + (c & 1)] = A[(long)site(u) * 36 + c];
  }
}

__device__ __forceinline__ float4 rb_cat(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }

// `sweeps` sweeps for one right-hand side per block; rin (r or the level's
// right-hand side) and xin (x, or NULL for a zero start) are read, x and r
// written.  Bounded waits as in k_kacz_rows.
//
// Bound by shared-memory bandwidth (a pass reads 61 KB) and the chain of a pass.
// Four sweeps of the 32 x 32 level, back to back: 5 right-hand sides with BF16-stored
// stencil 20.6 us (k_kacz_block 61.7), one FP32 right-hand side 16.5 us (k_kacz_coop 160).
template <typename S, int N>
__global__ void __launch_bounds__(N *N / 8) k_kacz_rings(Geo g, int sweeps, const unsigned char *__restrict__ pk,
                                                         const zf *rin, const zf *xin, zf *x, zf *r, int nrhs,
                                                         int *timeout) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  constexpr int NT = N * N / 8, RB = ring_bytes<S, N>(), PB = RB * (N / 8);
  unsigned char *cs = sm_raw;                                // [4][N / 8][RB]
  float4 *rs = (float4 *)(sm_raw + 4 * PB);                  // [N / 2][N] both spins
  float4 *nums = rs + N * N / 2;                             // [N / 8][N] both rows
  uint64_t *mbar = (uint64_t *)(nums + NT);                  // [4]
  const int tid = threadIdx.x, u = tid % N, ig = tid / N, rh = blockIdx.x;
  if (tid == 0) {
    for (int i = 0; i < 4; ++i) mbar_init(smem_u32(&mbar[i]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int i = 0; i < 4; ++i) {
      mbar_arrive_expect_tx(smem_u32(&mbar[i]), PB);
      bulk_g2s(smem_u32(cs + i * PB), pk + (long)i * PB, PB, smem_u32(&mbar[i]));
    }
  }
  const float2 *ri = (const float2 *)rin, *xi = (const float2 *)xin;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    int row = k + 4 * ig;
    long o = (long)g.idx(row + u, row - u) * 2 * nrhs + rh;
    rs[row * N + u] = rb_cat(ri[o], ri[o + nrhs]);
  }
  float2 xr[4][2];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    int row = k + 4 * ig;
    long o = (long)g.idx(row + u, row - u) * 2 * nrhs + rh;
    xr[k][0] = xi ? xi[o] : make_float2(0.f, 0.f);
    xr[k][1] = xi ? xi[o + nrhs] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  bool ok = true;
  for (int sw = 0; sw < sweeps && ok; ++sw) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (sw == 0) {
        ok = ok && mbar_wait(smem_u32(&mbar[k]), 0, 1000000000ull);
        ok = __syncthreads_and(ok);
        if (!ok) break;
      }
      const int row = k + 4 * ig;
      const S *ca = (const S *)(cs + k * PB + ig * RB);
      const zf *ct = (const zf *)(cs + k * PB + ig * RB + N * 36 * sizeof(S));
      // the window: rows row - 1, row, row + 1 (past the last ring the ring 0
      // half a turn on, before the first one the last ring likewise)
      float4 *wr[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        int ro = row + i - 1, sh = 0;
        if (ro < 0) ro += N / 2, sh = N / 2;
        if (ro >= N / 2) ro -= N / 2, sh = N / 2;
        wr[i] = rs + ro * N + ((u + sh) & (N - 1));
      }
      const int ul[3] = {-1, 0, 1};
      float2 a[9][2][2];  // [d][row t][spin]
#pragma unroll
      for (int d = 0; d < 9; ++d)
#pragma unroll
        for (int t = 0; t < 2; ++t) rb_ld(ca + ((d * 2 + t) * N + u) * 2, a[d][t][0], a[d][t][1]);
      float2 d0[2][2], e0[2][2];  // [t][spin]
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int sp = 0; sp < 2; ++sp) d0[t][sp] = e0[t][sp] = make_float2(0.f, 0.f);
      float4 rc[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        float4 *row0 = rs + ((wr[i] - rs) & ~(N - 1));
        const int uu = (int)((wr[i] - rs) & (N - 1));
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          float4 v = row0[(uu + ul[q]) & (N - 1)];
          if (q == 1) rc[i] = v;
          float2 v0 = make_float2(v.x, v.y), v1 = make_float2(v.z, v.w);
          float2 w0 = rb_swap(v0), w1 = rb_swap(v1);
          const int d = i * 3 + q;
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            d0[t][0] = __ffma2_rn(a[d][t][0], v0, d0[t][0]);
            e0[t][0] = __ffma2_rn(a[d][t][0], w0, e0[t][0]);
            d0[t][1] = __ffma2_rn(a[d][t][1], v1, d0[t][1]);
            e0[t][1] = __ffma2_rn(a[d][t][1], w1, e0[t][1]);
          }
        }
      }
      float2 nm[2];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        float re = (d0[t][0].x - d0[t][0].y) - (d0[t][1].x - d0[t][1].y);
        float im = (e0[t][0].x + e0[t][0].y) - (e0[t][1].x + e0[t][1].y);
        nm[t] = t ? make_float2(-re, -im) : make_float2(re, im);
      }
      float4 *nr = nums + ig * N;
      nr[u] = rb_cat(nm[0], nm[1]);
      const int j = u & 3;
      float2 T[2][12];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
#pragma unroll
        for (int c = 4; c < 12; ++c) T[t][c] = make_float2(0.f, 0.f);
        rb_ld(ct + 2 * ring_t_at<N>(0, t, 0, u), T[t][0], T[t][1]);
        rb_ld(ct + 2 * ring_t_at<N>(0, t, 1, u), T[t][2], T[t][3]);
        if (j >= 2) {
          rb_ld(ct + 2 * ring_t_at<N>(1, t, 0, u), T[t][4], T[t][5]);
          rb_ld(ct + 2 * ring_t_at<N>(1, t, 1, u), T[t][6], T[t][7]);
          rb_ld(ct + 2 * ring_t_at<N>(2, t, 0, u), T[t][8], T[t][9]);
        }
        if (j == 3) rb_ld(ct + 2 * ring_t_at<N>(3, t, 0, u), T[t][10], T[t][11]);
      }
      __syncwarp();
      float2 sd[2][2], se[2][2];
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int c = 0; c < 2; ++c) sd[t][c] = se[t][c] = make_float2(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        float4 v = nr[((u & ~3) + c) & (N - 1)];  // the cell's four sites, then the next cell's first two
        float2 v0 = make_float2(v.x, v.y), v1 = make_float2(v.z, v.w), w0 = rb_swap(v0), w1 = rb_swap(v1);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          sd[t][0] = __ffma2_rn(T[t][2 * c], v0, sd[t][0]);
          se[t][0] = __ffma2_rn(T[t][2 * c], w0, se[t][0]);
          sd[t][1] = __ffma2_rn(T[t][2 * c + 1], v1, sd[t][1]);
          se[t][1] = __ffma2_rn(T[t][2 * c + 1], w1, se[t][1]);
        }
      }
      float2 s0 = make_float2((sd[0][0].x - sd[0][0].y) + (sd[0][1].x - sd[0][1].y),
                              (se[0][0].x + se[0][0].y) + (se[0][1].x + se[0][1].y));
      float2 s1 = make_float2((sd[1][0].x - sd[1][0].y) + (sd[1][1].x - sd[1][1].y),
                              (se[1][0].x + se[1][0].y) + (se[1][1].x + se[1][1].y));
      xr[k][0] = make_float2(xr[k][0].x + s0.x, xr[k][0].y + s0.y);
      xr[k][1] = make_float2(xr[k][1].x + s1.x, xr[k][1].y + s1.y);
      // r_(d,sp) -= g_sp (s_0 conj(a[d][0][sp]) - s_1 conj(a[d][1][sp]))
      float2 m1 = make_float2(-s1.x, -s1.y), n0 = rb_swap(s0), n1 = rb_swap(m1);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        float2 dl[3][2];
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
          for (int sp = 0; sp < 2; ++sp) {
            float2 v = __ffma2_rn(a[i * 3 + q][1][sp], m1, __fmul2_rn(a[i * 3 + q][0][sp], s0));
            float2 w = __ffma2_rn(a[i * 3 + q][1][sp], n1, __fmul2_rn(a[i * 3 + q][0][sp], n0));
            dl[q][sp] = make_float2(v.x + v.y, w.x - w.y);
          }
        float2 tot[2];
#pragma unroll
        for (int sp = 0; sp < 2; ++sp) {
          float2 up = make_float2(__shfl_sync(0xffffffffu, dl[2][sp].x, (u - 1) & (N - 1), N),
                                  __shfl_sync(0xffffffffu, dl[2][sp].y, (u - 1) & (N - 1), N));
          float2 dn = make_float2(__shfl_sync(0xffffffffu, dl[0][sp].x, (u + 1) & (N - 1), N),
                                  __shfl_sync(0xffffffffu, dl[0][sp].y, (u + 1) & (N - 1), N));
          tot[sp] = make_float2(dl[1][sp].x + up.x + dn.x, dl[1][sp].y + up.y + dn.y);
        }
        *wr[i] = make_float4(rc[i].x - tot[0].x, rc[i].y - tot[0].y, rc[i].z + tot[1].x, rc[i].w + tot[1].y);
      }
      __syncthreads();
    }
  }
  if (!__syncthreads_and(ok)) {
    if (tid == 0) {
      mbar_drain(mbar, 4, 0);
      atomicExch(timeout, 1);
    }
    return;
  }
  float2 *ro = (float2 *)r, *xo = (float2 *)x;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    int row = k + 4 * ig;
    long o = (long)g.idx(row + u, row - u) * 2 * nrhs + rh;
    float4 v = rs[row * N + u];
    ro[o] = make_float2(v.x, v.y);
    ro[o + nrhs] = make_float2(v.z, v.w);
    xo[o] = xr[k][0];
    xo[o + nrhs] = xr[k][1];
  }
}

// --------------------------------------------------- 16-colour sweeps in FP64
// The ring passes on a level of any size, two launches a pass: k_ring_dots forms
// the inner products of every site of the rings a mod 4 = pass, k_ring_update
// solves the cells' triangular systems and updates x and r.  In FP64 a warp
// instruction takes the SM's FP64 unit 16 cycles and its warp 64, whatever the
// number of active lanes, so a chain of FP64 instructions is what a small level
// waits for: the products of a site are spread over 4 H lanes (row, real or
// imaginary part, and with H = 2, 4 the spin and half of the offsets), the T rows
// over 8 and the update over 12 a site, and nothing is divided.
//
// T [4][n / 4][2][12] (pass, ring and position, row): columns 0..7 the cell's own
// unknowns, 8..11 the next cell's first four.
__global__ void __launch_bounds__(16 * RBP_CELLS) k_ring64_pack(Geo g, const zd *__restrict__ A, double omega,
                                                                zd *__restrict__ T) {
  __shared__ zd Ms[RBP_CELLS][12][13];
  const int N = g.N, lc = threadIdx.x >> 4, i = threadIdx.x & 15;
  const int id = blockIdx.x * RBP_CELLS + lc;  // N / 4 cells a ring, N / 2 rings: the grid is exact
  const int cell = id % (N / 4), rg = id / (N / 4), pass = rg / (N / 8), row = pass + 4 * (rg % (N / 8));
  auto site = [&](int u) { return g.idx(row + u, row - u); };
  auto column = [&](int v) { return cell * 4 + (v < 4 ? (v >> 1) + 4 * (v & 1) : v - 2); };  // as in k_rings_pack
  if (i < 12)
    for (int q = 0; q < 6; ++q)
      for (int t2 = 0; t2 < 2; ++t2) {
        const int cp = column(i >> 1), cq = column(q), dl = cq - cp;
        zd k = mk(0.0, 0.0);
        if (2 * q + t2 <= i && dl >= -2 && dl <= 2) k = rb_gram(A, site(cp), i & 1, site(cq), t2, dl);
        if (2 * q + t2 == i) k = mk(k.re / omega, 0.0);
        Ms[lc][i][2 * q + t2] = k;
      }
  __syncthreads();
  if (i >= 12) return;
  const int v = i >> 1;
  const int k = (v < 4 ? ((v & 1) ? 8 : 0) + 2 * (v >> 1) : 2 * (v - 2)) + (i & 1);
  zd X[12];
#pragma unroll
  for (int r = 0; r < 12; ++r) {
    zd w = mk(r == i ? 1.0 : 0.0, 0.0);
#pragma unroll
    for (int c = 0; c < r; ++c) w = w - Ms[lc][r][c] * X[c];
    double d = Ms[lc][r][r].re;
    X[r] = mk(w.re / d, w.im / d);
    const int u = column(r >> 1);
    if (u < cell * 4 + 4) T[(((long)rg * N + u) * 2 + (r & 1)) * 12 + k] = X[r];
  }
}

// v with its sign flipped where `neg` (on the integer pipe: a negation that is
// not known at compile time costs an instruction of the FP64 unit, and the
// update of a pass took 2860 instead of 1306 cycles with them)
__device__ __forceinline__ double rb_flip(double v, bool neg) {
  return __hiloint2double(__double2hiint(v) ^ (neg ? (int)0x80000000 : 0), __double2loint(v));
}
// component c of a v: c = 0: a.re v.re - a.im v.im, c = 1: a.re v.im + a.im v.re
__device__ __forceinline__ void rb_cfma(double &acc, zd a, zd v, int c) {
  acc = fma(a.re, c ? v.im : v.re, acc);
  acc = fma(rb_flip(a.im, c == 0), c ? v.re : v.im, acc);
}

template <int H>
__global__ void __launch_bounds__(128) k_ring_dots(Geo g, int pass, const zd *__restrict__ A, const zd *r,
                                                   double *num, int nrhs) {
  constexpr int ND = H == 4 ? 5 : 9, NS = H == 1 ? 2 : 1;
  const int N = g.N, n4 = g.nsites() >> 2;
  const long tid = (long)blockIdx.x * 128 + threadIdx.x;
  const int l = (int)(tid % (4 * H)), c = l & 1, t = (l >> 1) & 1;
  const long q = tid / (4 * H);
  const int rh = (int)(q % nrhs);
  const long sp = q / nrhs;
  const bool act = sp < n4;
  const int row = pass + 4 * (int)((act ? sp : 0) / N), u = (int)((act ? sp : 0) % N);
  const int px = (row + u) & (N - 1), py = (row - u) & (N - 1);
  const zd *Ah = A + (long)g.idx(px, py) * 36 + t * 2;
  const int s0 = H == 1 ? 0 : (l >> 2) & 1, dh = H == 4 ? (l >> 3) * 5 : 0;  // offsets 0..4 or 5..8
  zd a[ND][NS];
#pragma unroll
  for (int i = 0; i < ND; ++i)
#pragma unroll
    for (int s = 0; s < NS; ++s) a[i][s] = dh + i < 9 ? Ah[(dh + i) * 4 + s0 + s] : mk(0.0, 0.0);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  double acc[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) acc[s] = 0;
  zd rv[ND][NS];
#pragma unroll
  for (int i = 0; i < ND; ++i)
#pragma unroll
    for (int s = 0; s < NS; ++s)
      rv[i][s] = r[((long)g.nb(px, py, min(dh + i, 8)) * 2 + s0 + s) * nrhs + rh];
#pragma unroll
  for (int i = 0; i < ND; ++i)
#pragma unroll
    for (int s = 0; s < NS; ++s) rb_cfma(acc[s], a[i][s], rv[i][s], c);
  double v;
  if (H == 1) {
    v = acc[0] - acc[NS - 1];
  } else {
    v = rb_flip(acc[0], s0 != 0);
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    if (H == 4) v += __shfl_xor_sync(0xffffffffu, v, 8);
  }
  if (act && l < 4) num[((sp * 2 + t) * nrhs + rh) * 2 + c] = rb_flip(v, t != 0);
}

// W positions of a ring and C right-hand sides per block, W C 12 threads / NI:
// the solutions s of the W sites and the two beside them go to shared memory,
// then every thread sums the update of NI real numbers of r.
template <int W, int C, int NI>
__global__ void __launch_bounds__(W *C * 12 / NI) k_ring_update(Geo g, int pass, const zd *__restrict__ A,
                                                                const zd *__restrict__ T, const double *num,
                                                                double *x, double *r, int nrhs) {
  constexpr int NT = W * C * 12 / NI;
  __shared__ double sm[W + 2][2][C][2];
  const int N = g.N, seg = N / W, tid = threadIdx.x;
  const int ring = blockIdx.x / seg, u0 = (blockIdx.x % seg) * W, row = pass + 4 * ring;
  const int r0 = blockIdx.y * C, Rc = min(C, nrhs - r0);
  // this thread's numbers of r: component, right-hand side, spin, row of the window, position
  zd a[NI][6];
  long ro[NI];
  bool in[NI];
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    int e = tid + i * NT, cc = (e >> 1) % C, q = (e >> 1) / C, s = q & 1, da = (q >> 1) % 3, uw = (q >> 1) / 3;
    in[i] = cc < Rc;
    int ra = row + da - 1, u = u0 + uw;
    ro[i] = (((long)g.idx(ra + u, ra - u) * 2 + s) * nrhs + r0 + cc) * 2 + (e & 1);
#pragma unroll
    for (int k = 0; k < 3; ++k) {  // the sites at u - 1, u, u + 1: this cell is their offset (da, 1 - k + 1)
      const zd *p = A + (long)g.idx(row + u + k - 1, row - u - k + 1) * 36 + (da * 3 + 2 - k) * 4 + s;
      a[i][2 * k] = p[0];
      a[i][2 * k + 1] = p[2];
    }
  }
  // solution items: lane (component, row, hh) takes the columns of unknown hh of the
  // six sites 0..5 from the cell's first; a site of colour j needs its own colours
  // up to j, the next cell's first for j >= 2 and its second for j = 3.  With C >= 4 a
  // warp is one position, so the others cost it nothing (3.25 of 6 on average).
  constexpr int NV = ((W + 2) * C * 8 + NT - 1) / NT;  // items a thread
  auto needed = [](int j, int k) { return k <= j || (k == 4 && j >= 2) || (k == 5 && j == 3); };
  zd tv[NV][6];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    int e = tid + i * NT, uu = min((e >> 3) / C, W + 1), u = (u0 + uu - 1) & (N - 1);
    const zd *Tp = T + ((((long)pass * (N / 8) + ring) * N + u) * 2 + ((e >> 1) & 1)) * 12 + ((e >> 2) & 1);
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if (needed(u & 3, k)) tv[i][k] = Tp[2 * k];
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  double rv[NI];
#pragma unroll
  for (int i = 0; i < NI; ++i) rv[i] = in[i] ? r[ro[i]] : 0.0;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int e = tid + i * NT;
    if (e >= ((W + 2) * C * 8 + 31) / 32 * 32) break;  // whole warps: the halves meet by a shuffle
    const int l = e & 7, c = l & 1, t = (l >> 1) & 1, hh = l >> 2, cc = (e >> 3) % C, uu = (e >> 3) / C;
    const bool on = uu < W + 2 && cc < Rc;
    const int u = (u0 + uu - 1) & (N - 1);
    double v = 0, xv = 0;
    double *xa = x + (((long)g.idx(row + u, row - u) * 2 + t) * nrhs + r0 + cc) * 2 + c;
    const bool mine = on && hh == 0 && uu >= 1 && uu <= W;
    if (on) {
      if (mine) xv = *xa;
      zd nv[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        int us = ((u & ~3) + k) & (N - 1);
        if (needed(u & 3, k)) nv[k] = *(const zd *)(num + ((((long)ring * N + us) * 2 + hh) * nrhs + r0 + cc) * 2);
      }
#pragma unroll
      for (int k = 0; k < 6; ++k)
        if (needed(u & 3, k)) rb_cfma(v, tv[i][k], nv[k], c);
    }
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    if (on && hh == 0) sm[uu][t][cc][c] = v;
    if (mine) *xa = xv + v;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    if (!in[i]) continue;
    int e = tid + i * NT, c = e & 1, cc = (e >> 1) % C, q = (e >> 1) / C, s = q & 1, uw = (q >> 1) / 3;
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int t = 0; t < 2; ++t) {  // r -= g_s g_t s_t conj(a)
        const double *sv = sm[uw + k][t][cc];
        zd av = a[i][2 * k + t];
        const bool neg = s == t;  // g_s g_t = 1: subtract
        rv[i] = fma(rb_flip(av.re, neg), sv[c], rv[i]);
        rv[i] = fma(rb_flip(av.im, neg == (c == 0)), sv[1 - c], rv[i]);
      }
    r[ro[i]] = rv[i];
  }
}

// All sweeps of a 32 x 32 or 64 x 64 level in one launch: a cluster of 16 blocks
// per right-hand side, block (ring group i, segment) holding rows 4 i .. 4 i + 3 of
// W positions with their stencil rows and T in shared memory, and r with a halo
// of one row and one position. Inner products and updated values of r that a
// neighbour's halo holds are stored there as well (distributed shared memory), so
// that every load is the block's own; a cluster barrier (390 cycles) follows the
// inner products and another one the update.  16 passes (four sweeps) of the
// 32 x 32 level with 12 right-hand sides: 56 us, two launches a pass 104 us.
template <int N>
struct RingCluster {
  static constexpr int NG = N / 8, SEG = 16 / NG, W = N / SEG, H = N == 32 ? 4 : 2;
  static constexpr int NT = N == 32 ? 128 : 384;
  zd A[4][W + 2][36];
  zd T[4][W + 2][24];
  zd r[6][W + 2][2];   // rows -1 .. 4, positions -1 .. W
  zd num[W + 10][2];   // positions -4 .. W + 5 of the ring of the pass
  zd s[W + 2][2];
  zd x[4][W][2];
};

template <int N>
__global__ void __launch_bounds__(RingCluster<N>::NT) k_ring64_cluster(Geo g, int sweeps, const zd *__restrict__ A,
                                                                       const zd *__restrict__ T, const zd *rin,
                                                                       const zd *xin, zd *x, zd *r, int nrhs) {
  typedef RingCluster<N> C;
  constexpr int W = C::W, SEG = C::SEG, NG = C::NG, NT = C::NT, H = C::H;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  C *sm = (C *)sm_raw;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), ig = rank / SEG, u0 = (rank % SEG) * W, tid = threadIdx.x, rh = blockIdx.y;
  auto site = [&](int row, int u) { return g.idx(row + u, row - u); };
  for (int e = tid; e < 4 * (W + 2) * 36; e += NT) {
    int k = e / ((W + 2) * 36), q = e / 36 % (W + 2), c = e % 36;
    sm->A[k][q][c] = A[(long)site(4 * ig + k, u0 + q - 1) * 36 + c];
  }
  for (int e = tid; e < 4 * (W + 2) * 24; e += NT) {
    int k = e / ((W + 2) * 24), q = e / 24 % (W + 2), c = e % 24, u = (u0 + q - 1) & (N - 1);
    sm->T[k][q][c] = T[(((long)k * NG + ig) * N + u) * 24 + c];
  }
  for (int e = tid; e < 6 * (W + 2) * 2; e += NT) {
    int k = e / (2 * (W + 2)), q = e / 2 % (W + 2), sp = e & 1;
    sm->r[k][q][sp] = rin[((long)site(4 * ig + k - 1, u0 + q - 1) * 2 + sp) * nrhs + rh];
  }
  for (int e = tid; e < 4 * W * 2; e += NT) {
    int k = e / (2 * W), w = e / 2 % W, sp = e & 1;
    sm->x[k][w][sp] = xin ? xin[((long)site(4 * ig + k, u0 + w) * 2 + sp) * nrhs + rh] : mk(0.0, 0.0);
  }
  // the blocks beside this one along the rings
  C *left = cl.map_shared_rank(sm, ig * SEG + (rank + SEG - 1) % SEG);
  C *right = cl.map_shared_rank(sm, ig * SEG + (rank + 1) % SEG);
  cl.sync();
  for (int sw = 0; sw < sweeps; ++sw)
    for (int k = 0; k < 4; ++k) {
      if (tid < W * 4 * H) {  // whole warps
        const int l = tid % (4 * H), w = tid / (4 * H), c = l & 1, t = (l >> 1) & 1, sp = (l >> 2) & 1;
        const int d0 = H == 4 ? (l >> 3) * 5 : 0, d1 = H == 4 ? min(d0 + 5, 9) : 9;
        double v = 0;
#pragma unroll
        for (int i = 0; i < (H == 4 ? 5 : 9); ++i) {
          int d = d0 + i;
          if (d < d1) rb_cfma(v, sm->A[k][w + 1][d * 4 + t * 2 + sp], sm->r[k + d / 3][w + d % 3][sp], c);
        }
        v = rb_flip(v, sp != 0);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        if (H == 4) v += __shfl_xor_sync(0xffffffffu, v, 8);
        if (l < 4) {
          v = rb_flip(v, t != 0);
          ((double *)&sm->num[w + 4][t])[c] = v;
          if (w >= W - 4) ((double *)&right->num[w - W + 4][t])[c] = v;
          if (w < 6) ((double *)&left->num[w + W + 4][t])[c] = v;
        }
      }
      cl.sync();
      if (tid < ((W + 2) * 8 + 31) / 32 * 32) {
        const int l = tid & 7, c = l & 1, t = (l >> 1) & 1, hh = l >> 2, q = min(tid >> 3, W + 1);
        const int cell = ((q + 3) & ~3) + hh * 3;  // in num: the cell of position q - 1, and the half's first site
        double v = 0;
#pragma unroll
        for (int i = 0; i < 6; ++i) rb_cfma(v, sm->T[k][q][t * 12 + hh * 6 + i], sm->num[cell + (i >> 1)][i & 1], c);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        if (hh == 0) {
          ((double *)&sm->s[q][t])[c] = v;
          if ((tid >> 3) == q && q >= 1 && q <= W) ((double *)&sm->x[k][q - 1][t])[c] += v;
        }
      }
      __syncthreads();
      for (int e = tid; e < W * 12; e += NT) {
        const int c = e & 1, sp = (e >> 1) & 1, i = (e >> 2) % 3, w = (e >> 2) / 3;
        double v = ((const double *)&sm->r[k + i][w + 1][sp])[c];
#pragma unroll
        for (int q = 0; q < 3; ++q)  // the sites at positions w - 1, w, w + 1
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            const double *sv = (const double *)&sm->s[w + q][t];
            zd a = sm->A[k][w + q][(i * 3 + 2 - q) * 4 + t * 2 + sp];
            const bool neg = sp == t;
            v = fma(rb_flip(a.re, neg), sv[c], v);
            v = fma(rb_flip(a.im, neg == (c == 0)), sv[1 - c], v);
          }
        // to every block whose rows (with halo) hold this cell: its own group and,
        // for a first or last row, the group before or after (half a turn on past
        // the last ring); there to the segment and, at its ends, the next one's halo
        int ro = 4 * ig + k + i - 1, u = u0 + w;
        if (ro < 0) ro += N / 2, u += N / 2;
        if (ro >= N / 2) ro -= N / 2, u += N / 2;
#pragma unroll
        for (int n = 0; n < 2; ++n) {
          int gr = ro >> 2, idx = (ro & 3) + 1, un = u;
          if (n == 1) {
            if (idx == 1) gr -= 1, idx = 5;
            else if (idx == 4) gr += 1, idx = 0;
            else break;
            if (gr < 0) gr += NG, un += N / 2;
            if (gr >= NG) gr -= NG, un += N / 2;
          }
          un &= N - 1;
          const int sg = un / W, p = un % W;
          ((double *)&cl.map_shared_rank(sm, gr * SEG + sg)->r[idx][p + 1][sp])[c] = v;
          if (p == 0) ((double *)&cl.map_shared_rank(sm, gr * SEG + (sg + SEG - 1) % SEG)->r[idx][W + 1][sp])[c] = v;
          if (p == W - 1) ((double *)&cl.map_shared_rank(sm, gr * SEG + (sg + 1) % SEG)->r[idx][0][sp])[c] = v;
        }
      }
      cl.sync();
    }
  for (int e = tid; e < 4 * W * 2; e += NT) {
    int k = e / (2 * W), w = e / 2 % W, sp = e & 1;
    long o = ((long)site(4 * ig + k, u0 + w) * 2 + sp) * nrhs + rh;
    r[o] = sm->r[k + 1][w + 1][sp];
    x[o] = sm->x[k][w][sp];
  }
}

// A pass in one launch for few right-hand sides on levels of any size: a cluster of
// N / W blocks holds a ring, each block W positions.  The inner products a
// neighbour's cells need are stored in its shared memory as well; one cluster
// barrier separates them from the update, where the two-launch form has the end of
// one kernel and the start of another.  Blocks write r only after that barrier, so
// no block still reads what another one updates.  The paper's W(4,4) cycles on
// 128 x 128 (2016 passes on 128, 64 and 32): 9.92 -> 9.50 ms a solve.
template <int W>
struct RingPass {
  static constexpr int H = W == 8 ? 4 : 2, NT = W == 8 ? 128 : 192;
};
template <int W>
__global__ void __launch_bounds__(RingPass<W>::NT) k_ring_pass(Geo g, int pass, const zd *__restrict__ A,
                                                               const zd *__restrict__ T, double *x, double *r, int nrhs) {
  constexpr int H = RingPass<W>::H, ND = H == 4 ? 5 : 9;
  __shared__ zd num[W + 10][2];  // positions -4 .. W + 5
  __shared__ zd ss[W + 2][2];
  const int N = g.N, seg = N / W, tid = threadIdx.x, rh = blockIdx.y;
  cg::cluster_group cl = cg::this_cluster();  // the blocks of one ring
  const int me = (int)cl.block_rank(), ring = blockIdx.x / seg, u0 = me * W, row = pass + 4 * ring;
  zd(*left)[2] = cl.map_shared_rank(num, (me + seg - 1) % seg), (*right)[2] = cl.map_shared_rank(num, (me + 1) % seg);
  // constants first: this thread's stencil entries, row of T and update entries
  const int dl = tid % (4 * H), dw = tid / (4 * H), dc = dl & 1, dt = (dl >> 1) & 1, dsp = (dl >> 2) & 1;
  const int dh = H == 4 ? (dl >> 3) * 5 : 0;
  const bool dots = tid < W * 4 * H;
  const int px = (row + u0 + dw) & (N - 1), py = (row - u0 - dw) & (N - 1);
  zd a[ND];
  if (dots) {
    const zd *Ah = A + (long)g.idx(px, py) * 36 + dt * 2 + dsp;
#pragma unroll
    for (int i = 0; i < ND; ++i) a[i] = dh + i < 9 ? Ah[(dh + i) * 4] : mk(0.0, 0.0);
  }
  const int sl = tid & 7, sc = sl & 1, st = (sl >> 1) & 1, sh = sl >> 2, sq = min(tid >> 3, W + 1);
  const int su = (u0 + sq - 1) & (N - 1);
  const bool solve = tid < ((W + 2) * 8 + 31) / 32 * 32, mine = (tid >> 3) == sq && sh == 0 && sq >= 1 && sq <= W;
  zd tv[6];
  if (solve) {
    const zd *Tp = T + ((((long)pass * (N / 8) + ring) * N + su) * 2 + st) * 12 + sh;
#pragma unroll
    for (int k = 0; k < 6; ++k) tv[k] = Tp[2 * k];
  }
  const int uc = tid & 1, us = (tid >> 1) & 1, ui = (tid >> 2) % 3, uw = (tid >> 2) / 3;
  const bool upd = tid < W * 12;
  zd b[6];
  if (upd)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const zd *p = A + (long)g.idx(row + u0 + uw + k - 1, row - u0 - uw - k + 1) * 36 + (ui * 3 + 2 - k) * 4 + us;
      b[2 * k] = p[0];
      b[2 * k + 1] = p[2];
    }
  const long ro = (((long)g.idx(row + ui - 1 + u0 + uw, row + ui - 1 - u0 - uw) * 2 + us) * nrhs + rh) * 2 + uc;
  double *xa = x + (((long)g.idx(row + su, row - su) * 2 + st) * nrhs + rh) * 2 + sc;
  cl.sync();  // every block of the ring runs
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  double v = 0, rv = 0, xv = 0;
  if (dots) {
    zd w[ND];
#pragma unroll
    for (int i = 0; i < ND; ++i)
      w[i] = *(const zd *)(r + (((long)g.nb(px, py, min(dh + i, 8)) * 2 + dsp) * nrhs + rh) * 2);
    if (upd) rv = r[ro];
    if (mine) xv = *xa;
#pragma unroll
    for (int i = 0; i < ND; ++i) rb_cfma(v, a[i], w[i], dc);
    v = rb_flip(v, dsp != 0);
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    if (H == 4) v += __shfl_xor_sync(0xffffffffu, v, 8);
    if (dl < 4) {
      v = rb_flip(v, dt != 0);
      ((double *)&num[dw + 4][dt])[dc] = v;
      if (dw >= W - 4) ((double *)&right[dw - W + 4][dt])[dc] = v;
      if (dw < 6) ((double *)&left[dw + W + 4][dt])[dc] = v;
    }
  } else {
    if (upd) rv = r[ro];
    if (mine) xv = *xa;
  }
  cl.sync();
  if (solve) {
    const int cell = (sq + 3) & ~3;  // in num: the first site of the cell of position sq - 1
    double z = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k) rb_cfma(z, tv[k], num[cell + k][sh], sc);
    z += __shfl_xor_sync(0xffffffffu, z, 4);
    if (sh == 0) ((double *)&ss[sq][st])[sc] = z;
    if (mine) *xa = xv + z;
  }
  __syncthreads();
  if (upd) {
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int t = 0; t < 2; ++t) {  // r -= g_s g_t s_t conj(a)
        const double *sv = (const double *)&ss[uw + k][t];
        const bool neg = us == t;
        rv = fma(rb_flip(b[2 * k + t].re, neg), sv[uc], rv);
        rv = fma(rb_flip(b[2 * k + t].im, neg == (uc == 0)), sv[1 - uc], rv);
      }
    r[ro] = rv;
  }
}

namespace wl {

// raise a kernel's dynamic shared-memory limit once per device
static int rb_smem_limit(const void *fn, size_t bytes, std::atomic<unsigned long long> &done) {
  int dev = 0;
  WL_CUDA(cudaGetDevice(&dev));
  unsigned long long bit = 1ull << (dev & 63);
  if (!(done.load(std::memory_order_acquire) & bit)) {
    WL_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    done.fetch_or(bit, std::memory_order_acq_rel);
  }
  return WL_OK;
}

template <typename S, int R, int RPT>
static int launch_rows(const Level &L, const LevelOps &o, int tc, void *x, void *r, int nrhs, int pdl, cudaStream_t s) {
  constexpr int NW = R / RPT;
  size_t smem = (size_t)4 * rb_step_bytes<S>() + sizeof(zf) * ((R * RB_RS + 1) & ~1) + sizeof(zf) * R * 40 +
                sizeof(int) * RB_W * RB_W + 4 * sizeof(uint64_t);
  static std::atomic<unsigned long long> done{0};
  WL_TRY(rb_smem_limit((const void *)k_kacz_rows<S, R, RPT>, smem, done));
  int *flag = tile_timeout_flag();
  if (!flag) return WL_ECUDA;
  dim3 grid((L.N / (2 * RB_KT)) * (L.N / (4 * RB_KT)), (nrhs + R - 1) / R);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(32 * NW);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = pdl;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  WL_CUDA(cudaLaunchKernelEx(&cfg, k_kacz_rows<S, R, RPT>, L.geo, tc, (const unsigned char *)o.rows.p, (zf *)x, (zf *)r,
                             nrhs, flag));
  return WL_OK;
}

template <typename S>
static int rows_tile(const Level &L, const LevelOps &o, int tc, void *x, void *r, int nrhs, int param, int pdl,
                     cudaStream_t s) {
  switch (param) {
#define RB_CASE(R, RPT) \
  case R | RPT << 8: return launch_rows<S, R, RPT>(L, o, tc, x, r, nrhs, pdl, s);
    RB_CASE(1, 1) RB_CASE(2, 1) RB_CASE(4, 1) RB_CASE(8, 1) RB_CASE(8, 2)
#undef RB_CASE
    default: wl_set_error("internal: no row-block form %d", param); return WL_EINVAL;
  }
}

// the launch parameters (R | RPT << 8) worth timing for nrhs right-hand sides
int rows_candidates(int nrhs, int *out) {
  int n = 0;
  if (nrhs <= 2) out[n++] = 1 | 1 << 8;
  if (nrhs >= 2) out[n++] = 2 | 1 << 8;
  if (nrhs >= 3) out[n++] = 4 | 1 << 8;
  if (nrhs >= 5) {
    out[n++] = 8 | 1 << 8;
    out[n++] = 8 | 2 << 8;
  }
  return n;
}

// Which sweeps take the row-block form.  Two concurrent lanes fill the GPU
// between them, so there the work of a sweep counts and not its latency: with
// the row form (about twice the instructions of k_kacz_tile, a third of its
// dependent steps) on level 1 the 512x512 step of 64 right-hand sides took
// 145.0 ms instead of 143.7, although that level's sweep alone takes 21
// instead of 41.7 us.  (A batch of 16 to 31 with overlap = 1 is one lane, but of the
// width that a lane of a split batch has.  FP64 lanes were not measured.)
bool rows_ok(const wl_amg *a, int l, int prec, int nrhs) {
  // A launch relaxes a quarter of the level's tiles for every right-hand side.  The
  // lines lie where a sweep takes as long as the best tile kernel's.  Tiles x
  // right-hand sides, us a sweep, row form against tile kernel, FP32 (BF16): up to 4
  // right-hand sides, 1024x1024 x 1 = 2048: 71 / 139.5 (59 / 148), 512x512 x 4 = 2048:
  // 35.0 / 46.9 (32.9 / 43.1).  More of them, whose tile kernel has fewer idle lanes:
  // 128x128 x 32 = 1024: 25.1 / 32.9 (24.7 / 37.0), 256x256 x 9 = 1152: 32.4 / 37.0
  // (31.3 / 37.0), x 12 = 1536: 32.9 / 32.9 (32.9 / 37.2), 128x128 x 48 = 1536: 37.0 / 32.9
  // (35.8 / 37.1), 256x256 x 16 = 2048: 37.0 / 32.9 (36.6 / 37.1).
  const Level &L = a->lev[l];
  if ((long)L.n / 256 * nrhs > (nrhs <= 4 ? 2048 : prec == WL_FP32_BF16 ? 1536 : 1280)) return false;
  return !a->is_twin && !(a->prm.overlap && nrhs >= 16) && prec != WL_FP64 && a->prm.kacz_order == 1 && l < a->L - 1 && L.N >= 64 && L.N % (4 * RB_KT) == 0 &&
         a->prm.omega > 0.0;
}

bool rows_form_exists(const wl_amg *a, int l, int prec, int param) {
  bool known = false;
  for (int nrhs : {1, 8}) {  // the parameters rows_candidates hands out
    int c[8], n = rows_candidates(nrhs, c);
    for (int i = 0; i < n; ++i) known |= c[i] == param;
  }
  return known && rows_ok(a, l, prec, 1);
}

// the level's packed rows in precision prec, made on first use (stream s)
int rows_prepare(wl_amg *a, int l, int prec, cudaStream_t s) {
  Level &L = a->lev[l];
  LevelOps &o = prec == WL_FP32 ? L.op32 : L.opbf;
  if (o.rows.p) return WL_OK;
  int nt = L.n / 64;
  int sb = prec == WL_FP32 ? rb_step_bytes<zf>() : rb_step_bytes<zb>();
  WL_TRY(o.rows.alloc((size_t)nt * 4 * sb));
  unsigned grid = nt * 16 / RBP_CELLS;
  if (prec == WL_FP32) k_rows_pack<zf><<<grid, 16 * RBP_CELLS, 0, s>>>(L.geo, o.A.as<zf>(), a->prm.omega, o.rows.as<unsigned char>());
  else k_rows_pack<zb><<<grid, 16 * RBP_CELLS, 0, s>>>(L.geo, o.A.as<zb>(), a->prm.omega, o.rows.as<unsigned char>());
  wl_count_launches(1);
  WL_CUDA(cudaGetLastError());
  return WL_OK;
}

int rows_sweeps(wl_amg *a, int l, int prec, void *x, void *r, int nrhs, int sweeps, int param, cudaStream_t s) {
  const Level &L = a->lev[l];
  for (int sw = 0; sw < sweeps; ++sw)
    for (int tc = 0; tc < 4; ++tc) {
      wl_count_launches(1);
      if (prec == WL_FP32) WL_TRY(rows_tile<zf>(L, L.op32, tc, x, r, nrhs, param, sw + tc > 0, s));
      else WL_TRY(rows_tile<zb>(L, L.opbf, tc, x, r, nrhs, param, sw + tc > 0, s));
    }
  WL_CUDA(cudaGetLastError());
  return WL_OK;
}

// ---- small levels
bool rings_ok(const wl_amg *a, int l, int prec) {
  const Level &L = a->lev[l];
  return prec != WL_FP64 && l < a->L - 1 && (L.N == 32 || L.N == 16) && a->prm.omega > 0.0;
}

template <typename S, int N>
static int rings_pack(const Level &L, LevelOps &o, double omega, cudaStream_t s) {
  WL_TRY(o.rows.alloc((size_t)(N / 2) * ring_bytes<S, N>()));
  k_rings_pack<S, N><<<N * N / 8 / RBP_CELLS, 16 * RBP_CELLS, 0, s>>>(L.geo, o.A.as<S>(), omega,
                                                                     o.rows.as<unsigned char>());
  wl_count_launches(1);
  WL_CUDA(cudaGetLastError());
  return WL_OK;
}

int rings_prepare(wl_amg *a, int l, int prec, cudaStream_t s) {
  Level &L = a->lev[l];
  LevelOps &o = prec == WL_FP32 ? L.op32 : L.opbf;
  if (!tile_timeout_flag()) return WL_ECUDA;  // looked up before a stream capture needs it
  if (o.rows.p) return WL_OK;
  if (prec == WL_FP32) return L.N == 32 ? rings_pack<zf, 32>(L, o, a->prm.omega, s) : rings_pack<zf, 16>(L, o, a->prm.omega, s);
  return L.N == 32 ? rings_pack<zb, 32>(L, o, a->prm.omega, s) : rings_pack<zb, 16>(L, o, a->prm.omega, s);
}

template <typename S, int N>
static int launch_rings(const Level &L, const LevelOps &o, const void *rin, const void *xin, void *x, void *r, int nrhs,
                        int sweeps, cudaStream_t s) {
  const size_t smem = (size_t)(N / 2) * ring_bytes<S, N>() + sizeof(float4) * (N * N / 2 + N * N / 8) + 4 * sizeof(uint64_t);
  static_assert((N / 2) * ring_bytes<S, N>() + 16 * (N * N / 2 + N * N / 8) + 32 <= 227 * 1024, "shared memory");
  static std::atomic<unsigned long long> done{0};
  WL_TRY(rb_smem_limit((const void *)k_kacz_rings<S, N>, smem, done));
  int *flag = tile_timeout_flag();
  if (!flag) return WL_ECUDA;
  k_kacz_rings<S, N><<<nrhs, N * N / 8, smem, s>>>(L.geo, sweeps, o.rows.as<unsigned char>(), (const zf *)rin,
                                                   (const zf *)xin, (zf *)x, (zf *)r, nrhs, flag);
  wl_count_launches(1);
  WL_CUDA(cudaGetLastError());
  return WL_OK;
}

int rings_sweeps(wl_amg *a, int l, int prec, const void *rin, const void *xin, void *x, void *r, int nrhs, int sweeps,
                 cudaStream_t s) {
  const Level &L = a->lev[l];
  const LevelOps &o = prec == WL_FP32 ? L.op32 : L.opbf;
  if (prec == WL_FP32)
    return L.N == 32 ? launch_rings<zf, 32>(L, o, rin, xin, x, r, nrhs, sweeps, s)
                     : launch_rings<zf, 16>(L, o, rin, xin, x, r, nrhs, sweeps, s);
  return L.N == 32 ? launch_rings<zb, 32>(L, o, rin, xin, x, r, nrhs, sweeps, s)
                   : launch_rings<zb, 16>(L, o, rin, xin, x, r, nrhs, sweeps, s);
}

// ---- 16-colour sweeps in FP64
bool rings64_ok(const wl_amg *a, int l, int prec, int nrhs) {
  const Level &L = a->lev[l];
  const bool tile = a->prm.kacz_order == 1 && L.N >= 64;
  return prec == WL_FP64 && !tile && l < a->L - 1 && L.N >= 16 && a->prm.omega > 0.0 && !a->is_twin &&
         !(a->prm.overlap && nrhs >= 16);
}

int rings64_prepare(wl_amg *a, int l, bool stale, cudaStream_t s) {
  Level &L = a->lev[l];
  if (L.op64.rows.p && !stale) return WL_OK;
  WL_TRY(L.op64.rows.alloc(sizeof(zd) * (size_t)L.n * 24));
  k_ring64_pack<<<L.n / 4 / RBP_CELLS, 16 * RBP_CELLS, 0, s>>>(L.geo, L.op64.A.as<zd>(), a->prm.omega,
                                                              L.op64.rows.as<zd>());
  wl_count_launches(1);
  WL_CUDA(cudaGetLastError());
  return WL_OK;
}

template <typename... P, typename... Q>
static int rb_launch(void (*fn)(P...), dim3 grid, int nt, int pdl, cudaStream_t s, Q... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(nt);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = pdl;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  wl_count_launches(1);
  WL_CUDA(cudaLaunchKernelEx(&cfg, fn, args...));
  return WL_OK;
}

template <int N>
static int launch_cluster(const Level &L, const void *rin, const void *xin, void *x, void *r, int nrhs, int sweeps,
                          cudaStream_t s) {
  const size_t smem = sizeof(RingCluster<N>);
  static std::atomic<unsigned long long> done{0}, wide{0};
  WL_TRY(rb_smem_limit((const void *)k_ring64_cluster<N>, smem, done));
  int dev = 0;
  WL_CUDA(cudaGetDevice(&dev));
  unsigned long long bit = 1ull << (dev & 63);
  if (!(wide.load(std::memory_order_acquire) & bit)) {  // clusters of 16 blocks
    WL_CUDA(cudaFuncSetAttribute((const void *)k_ring64_cluster<N>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    wide.fetch_or(bit, std::memory_order_acq_rel);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(16, nrhs);
  cfg.blockDim = dim3(RingCluster<N>::NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 16;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  wl_count_launches(1);
  WL_CUDA(cudaLaunchKernelEx(&cfg, k_ring64_cluster<N>, L.geo, sweeps, (const zd *)L.op64.A.p, (const zd *)L.op64.rows.p,
                             (const zd *)rin, (const zd *)xin, (zd *)x, (zd *)r, nrhs));
  return WL_OK;
}

template <int W>
static int launch_ring_pass(const Level &L, int pass, void *x, void *r, int nrhs, int pdl, cudaStream_t s) {
  static std::atomic<unsigned long long> wide{0};
  int dev = 0;
  WL_CUDA(cudaGetDevice(&dev));
  unsigned long long bit = 1ull << (dev & 63);
  if (!(wide.load(std::memory_order_acquire) & bit)) {
    WL_CUDA(cudaFuncSetAttribute((const void *)k_ring_pass<W>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    wide.fetch_or(bit, std::memory_order_acq_rel);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(L.N / 8 * (L.N / W), nrhs);
  cfg.blockDim = dim3(RingPass<W>::NT);
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = L.N / W;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = pdl;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  wl_count_launches(1);
  WL_CUDA(cudaLaunchKernelEx(&cfg, k_ring_pass<W>, L.geo, pass, (const zd *)L.op64.A.p, (const zd *)L.op64.rows.p,
                             (double *)x, (double *)r, nrhs));
  return WL_OK;
}

// Does the current device (a partition of one, perhaps) hold a cluster of this kernel?
// Asked once per device; raises the kernel's limits on the way.
static bool cluster_fits(const void *fn, int blocks, int nt, size_t smem, std::atomic<unsigned long long> *known) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(known[0].load(std::memory_order_acquire) & bit)) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(nt);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = blocks;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if ((!smem || cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess) &&
        (blocks <= 8 || cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
        cudaOccupancyMaxActiveClusters(&n, fn, &cfg) == cudaSuccess && n > 0)
      known[1].fetch_or(bit, std::memory_order_acq_rel);
    else
      cudaGetLastError();
    known[0].fetch_or(bit, std::memory_order_acq_rel);
  }
  return (known[1].load(std::memory_order_acquire) & bit) != 0;
}
template <int N>
static bool ring_cluster_fits() {
  static std::atomic<unsigned long long> known[2];
  return cluster_fits((const void *)k_ring64_cluster<N>, 16, RingCluster<N>::NT, sizeof(RingCluster<N>), known);
}
template <int W, int BLOCKS>
static bool ring_pass_fits() {
  static std::atomic<unsigned long long> known[2];
  return cluster_fits((const void *)k_ring_pass<W>, BLOCKS, RingPass<W>::NT, 0, known);
}

bool rings64_form(const wl_amg *a, int l, int param, int nrhs) {
  const int N = a->lev[l].N;
  if (param == 1) return N == 32 ? ring_cluster_fits<32>() : N == 64 && ring_cluster_fits<64>();
  if (param == 2 && nrhs <= 4)
    return N == 32 ? ring_pass_fits<8, 4>() : N == 64 ? ring_pass_fits<8, 8>()
         : N == 128 ? ring_pass_fits<8, 16>() : N == 256 && ring_pass_fits<16, 16>();
  return param == 0;
}

// The form of a cycle's sweeps, by level and width alone, since the forms round
// differently.  us a sweep (params 0 / 1 / 2 / the best of the other forms):
//   32x32:   1: 21.7 / 18.7 / 16.5 / 78, 4: 25.7 / 18.5 / 16.5 / 191, 5: 27.6 / 18.7 / - / 193,
//            32: 36.0 / 28.9 / - / 193, 48: 48.3 / 59.6 / - / 193
//   64x64:   1: 21.7 / 26.8 / 16.5 / 78, 4: 27.5 / 27.0 / 18.7 / 211, 6: 34.0 / 27.0 / - / 211,
//            8: 35.9 / 51.6 / - / 213, 64: 125 / 249 / - / 211
//   128x128: 1: 25.7 / - / 22.7 / 78, 2: 29.9 / - / 35.1 / 228, 24: 174 / - / - / 211
//   256x256: 1: 57 / - / 71 / 192, 4: 126 / - / 244 / 216, 5: 189 / - / - / 220
// (over four sweeps, 32x32, one right-hand side: 79 / 47 / 58) and one right-hand side of
// 512x512 146 / 623, of 1024x1024 492 / 2195.  Param 0 works on
// chunks of 4; it meets the cooperative launch at 2^18 site-vectors (128x128 x 32: 212 / 212,
// 256x256 x 8: 213 / 213), and where that launch needs a second block on an SM (152 blocks of
// 2048 site-vectors) again at 3 * 2^17 (128x128 x 48: 308 / 371, 256x256 x 12: 308 / 374,
// x 9: 284 / 219, x 16: 401 / 373).
int rings64_rule(const wl_amg *a, int l, int nrhs) {
  const int N = a->lev[l].N;
  const long n = a->lev[l].n, padded = n * ((nrhs + 3) / 4 * 4);
  if (rings64_form(a, l, 2, nrhs) && (N <= 64 || (N == 128 && nrhs == 1))) return 2;
  if (rings64_form(a, l, 1, nrhs) && nrhs <= (N == 32 ? 32 : 6)) return 1;
  if (nrhs == 1 || padded <= 1L << 18 || (n * nrhs > 152L * 2048 && padded <= 3L << 17)) return 0;
  return -1;
}

// param 0: two launches a pass; 1: one launch of clusters (32 x 32 and 64 x 64); 2:
// one launch of clusters a pass.
// rin, xin as in rings_sweeps (param 0 takes r and x themselves)
int rings64_sweeps(wl_amg *a, int l, const void *rin, const void *xin, void *x, void *r, void *nums, int nrhs, int sweeps,
                   int param, cudaStream_t s) {
  Level &L = a->lev[l];
  if (param == 1)
    return L.N == 32 ? launch_cluster<32>(L, rin, xin, x, r, nrhs, sweeps, s)
                     : launch_cluster<64>(L, rin, xin, x, r, nrhs, sweeps, s);
  if (param == 2) {
    for (int sw = 0; sw < sweeps; ++sw)
      for (int k = 0; k < 4; ++k) {
        if (L.N <= 128) WL_TRY(launch_ring_pass<8>(L, k, x, r, nrhs, sw + k > 0, s));
        else WL_TRY(launch_ring_pass<16>(L, k, x, r, nrhs, sw + k > 0, s));
      }
    return WL_OK;
  }
  const zd *A = L.op64.A.as<zd>(), *T = L.op64.rows.as<zd>();
  double *num = (double *)nums;
  const long items = (long)(L.n / 4) * nrhs;
  // lanes a site: as many as leave at most a warp or so per SM partition (a launch
  // of the dots, one right-hand side: 1.6 us on 64 x 64 with H = 4, 2.0 us on 128 x 128
  // with H = 2; the update 2.6 and 2.7 us)
  const int H = items <= 512 ? 4 : items <= 4096 ? 2 : 1;
  const dim3 gd((unsigned)((items * 4 * H + 127) / 128));
  const int rings = L.N / 8;
  for (int sw = 0; sw < sweeps; ++sw)
    for (int k = 0; k < 4; ++k) {
      const int pdl = sw + k > 0;
      if (H == 4) WL_TRY(rb_launch(k_ring_dots<4>, gd, 128, pdl, s, L.geo, k, A, (const zd *)r, num, nrhs));
      else if (H == 2) WL_TRY(rb_launch(k_ring_dots<2>, gd, 128, pdl, s, L.geo, k, A, (const zd *)r, num, nrhs));
      else WL_TRY(rb_launch(k_ring_dots<1>, gd, 128, pdl, s, L.geo, k, A, (const zd *)r, num, nrhs));
      const double *nm = num;
      if (nrhs == 1)
        WL_TRY(rb_launch(k_ring_update<16, 1, 1>, dim3(rings * (L.N / 16)), 192, 1, s, L.geo, k, A, T, nm, (double *)x,
                         (double *)r, nrhs));
      else if (nrhs == 2)
        WL_TRY(rb_launch(k_ring_update<8, 2, 1>, dim3(rings * (L.N / 8)), 192, 1, s, L.geo, k, A, T, nm, (double *)x,
                         (double *)r, nrhs));
      else
        WL_TRY(rb_launch(k_ring_update<8, 4, 2>, dim3(rings * (L.N / 8), (nrhs + 3) / 4), 192, 1, s, L.geo, k, A, T, nm,
                         (double *)x, (double *)r, nrhs));
    }
  return WL_OK;
}

}  // namespace wl
