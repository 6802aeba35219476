// Inner solve of the mixed path by grid groups: CG on A^T A d = g with every
// alias product formed one grid at a time in shared memory.  Included only by
// fct_solver.cuh.
//
// A^T A = sum_l A_l^T A_l, and a grid's block A_l has one entry per column, so
// q_l = A_l s and t_l = A_l^T q_l need nothing from the other grids: a block
// that holds s (or a slice of it) and q_l in shared memory does both, and only
// the sum over grids t = sum_l t_l and the vector updates cross blocks.
//
// Per iteration (s = residual of the normal equations, as in cg_normal):
//   phase 1, per task (a group of tk_gg grids, one block): p = s + beta p_old
//     into shared memory, q_l = A_l p and |q|^2, then t = sum_{l in group}
//     A_l^T q_l, streamed out (tpart);
//   phase 2, per owner chunk: t = sum over groups of tpart, then x += alpha p,
//     s -= alpha t.
// What bounds it now: latency in the two streams at 16 warps per SM, then the
// phases' fixed costs.  Counters of the sparse D = 100 plans (N = 20000 on 1000
// grids, N = 100000 on 240): DRAM at 36 and 35 % of the copy rate, issue slots 17 and
// 18 % used, per issued instruction 10 and 9 warps at a barrier and 7 and 8 waiting for a load;
// 81 and 98 instructions and 25 and 27 shared-memory wavefronts of the whole launch
// per four steps of a warp.  Time per CG iteration, two-matrix form -> this: sparse
// D = 100, N = 50000, 240 grids 226 -> 70 us; N = 20000, 1000 grids 172 -> 107;
// D = 18 degree 5, 171 grids 56 -> 49 (171 tasks on 152 SMs).
// Two team barriers, as in cg_normal, but every scattered access is to shared
// memory and global traffic is coalesced: 6 bytes of table per entry (read by
// the gather and again by the scatter; the plans above hold 120 and 144 MB of tables,
// and both readings come from DRAM) and 8 + 4 bytes of vectors per coefficient and
// task.
//
// Cell tables.  A cell is one (grid, slice of tk_sl coefficients).  Its rows are
// cut into runs of at most kCellRun entries, sorted by length, 32 to a group:
// lane i of a warp sums run i of the group, one entry a step, so a step is 32
// independent entries and pads are few (sorted lengths).  A warp's groups are
// contiguous, so it streams its steps, four to a block, without looking at group
// boundaries ahead: bit 15 of a step's indices marks the last step of a group,
// where the lanes store their sums and go on to the next 32 runs.  Rows of
// several runs are completed by cell_join.  The order of additions depends only
// on the plan and the block size, so a transform's result is the same bit for
// bit alone, in a batch and for any team size.
#pragma once

#include "fct_common.cuh"

__device__ __forceinline__ uint32_t shared_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ float lds_f32(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t a) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts_f32(uint32_t a, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(shared_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// A grid's part of the shared memory: its row sums (rows, extra slots, one slot
// for idle lanes), then the run destinations of the cell at hand.
__device__ __forceinline__ int cell_q_floats(int rows, int ext) { return (rows + ext + 1 + 3) & ~3; }

// Run destinations of a cell into shared memory (asynchronous copies; kCellIdle
// groups of idle destinations follow the last: they are read ahead).
template <int NW>
__device__ __forceinline__ void cell_load_dest(const DevPlan& P, int cell, uint16_t* dest) {
  const int n16 = (__ldg(P.tk_wtab + static_cast<int64_t>(cell) * (NW + 1) + NW).y + kCellIdle) * 4;
  const uint16_t* src = P.tk_dest + static_cast<int64_t>(cell) * P.tk_gmax * 32;
  for (int i = threadIdx.x; i < n16; i += NW * 32) cp_async16(dest + 8 * i, src + 8 * i);
}

// A step's index is the coefficient in the slice (15 bits) and the mark; the
// byte offset in shared memory is 4 x the coefficient.
__device__ __forceinline__ uint32_t cell_at0(uint32_t v) { return (v & 0x7fffu) << 2; }
__device__ __forceinline__ uint32_t cell_at1(uint32_t v) { return (v >> 14) & 0x1fffcu; }

constexpr int kCellAhead = 4;  // blocks of four steps a warp keeps in flight

// Calls block(indices, values) for the n blocks of four steps of a warp's share of
// a cell, kCellAhead loaded ahead.
template <typename Block>
__device__ __forceinline__ void cell_stream(const uint2* __restrict__ idx, const float4* __restrict__ w, int n,
                                            Block block) {
  uint2 in[kCellAhead];
  float4 wn[kCellAhead];
#pragma unroll
  for (int j = 0; j < kCellAhead; ++j) {
    const int b = min(j, n - 1);
    in[j] = __ldg(idx + b * 32);
    wn[j] = __ldg(w + b * 32);
  }
  int b = 0;
#pragma unroll 1
  for (; b + kCellAhead <= n; b += kCellAhead) {
    uint2 ic[kCellAhead];
    float4 wc[kCellAhead];
#pragma unroll
    for (int j = 0; j < kCellAhead; ++j) {
      ic[j] = in[j];
      wc[j] = wn[j];
    }
#pragma unroll
    for (int j = 0; j < kCellAhead; ++j) {
      const int nb = min(b + kCellAhead + j, n - 1);
      in[j] = __ldg(idx + nb * 32);
      wn[j] = __ldg(w + nb * 32);
    }
#pragma unroll
    for (int j = 0; j < kCellAhead; ++j) block(ic[j], wc[j]);
  }
#pragma unroll
  for (int j = 0; j < kCellAhead - 1; ++j)
    if (b + j < n) block(in[j], wn[j]);
}

// q[dest] (+)= the sums of w p over n blocks of a cell.  ADD: the plan has
// several slices, whose sums add up in q.  sp, sq, sd: shared addresses of the
// slice of p, the grid's row sums and this lane's first destination.  A run's
// place (and, with ADD, its sum so far) is loaded while the runs before it are
// summed: the chain of loads per ending run would bound cells of short rows.
// Its own function (not inlined): the loop needs its registers for the loads in
// flight.
template <bool ADD>
__device__ __noinline__ void cell_gather(const uint2* __restrict__ idx, const float4* __restrict__ w, int n,
                                         uint32_t sp, uint32_t sq, uint32_t sd) {
  float acc = 0.0f;
  uint32_t a = sq + 4 * lds_u16(sd), an = sq + 4 * lds_u16(sd + 64);
  float old = ADD ? lds_f32(a) : 0.0f;
  sd += 128;
  auto end = [&](uint32_t mark) {
    if (mark) {  // the same for all lanes
      sts_f32(a, ADD ? old + acc : acc);
      acc = 0.0f;
      a = an;
      if (ADD) old = lds_f32(a);
      an = sq + 4 * lds_u16(sd);
      sd += 64;
    }
  };
  cell_stream(idx, w, n, [&](uint2 ic, float4 wc) {
    const float p0 = lds_f32(sp + cell_at0(ic.x)), p1 = lds_f32(sp + cell_at1(ic.x));
    const float p2 = lds_f32(sp + cell_at0(ic.y)), p3 = lds_f32(sp + cell_at1(ic.y));
    acc = fmaf(wc.x, p0, acc);
    if (((ic.x | ic.y) & 0x80008000u) == 0) {  // no run ends here
      acc = fmaf(wc.y, p1, acc);
      acc = fmaf(wc.z, p2, acc);
      acc = fmaf(wc.w, p3, acc);
    } else {
      end(ic.x & 0x8000u);
      acc = fmaf(wc.y, p1, acc);
      end(ic.x & 0x80000000u);
      acc = fmaf(wc.z, p2, acc);
      end(ic.y & 0x8000u);
      acc = fmaf(wc.w, p3, acc);
      end(ic.y & 0x80000000u);
    }
  });
}

// t[m] (+)= w q[row] over n blocks of a cell.  Every column has one entry per
// grid, so no two entries of a cell touch the same t; the first grid of a group
// stores, the others add.
template <bool ADD>
__device__ __noinline__ void cell_scatter(const uint2* __restrict__ idx, const float4* __restrict__ w, int n,
                                          uint32_t sv, uint32_t sq, uint32_t sd) {
  float qv = lds_f32(sq + 4 * lds_u16(sd)), qn = lds_f32(sq + 4 * lds_u16(sd + 64));
  uint32_t an = sq + 4 * lds_u16(sd + 128);
  sd += 192;
  auto next = [&](uint32_t mark) {
    if (mark) {
      qv = qn;
      qn = lds_f32(an);
      an = sq + 4 * lds_u16(sd);
      sd += 64;
    }
  };
  cell_stream(idx, w, n, [&](uint2 ic, float4 wc) {
    const uint32_t a0 = sv + cell_at0(ic.x), a1 = sv + cell_at1(ic.x), a2 = sv + cell_at0(ic.y), a3 = sv + cell_at1(ic.y);
    float t0 = 0.0f, t1 = 0.0f, t2 = 0.0f, t3 = 0.0f;
    if (ADD) {  // the four entries of a lane are different columns
      t0 = lds_f32(a0);
      t1 = lds_f32(a1);
      t2 = lds_f32(a2);
      t3 = lds_f32(a3);
    }
    auto term = [&](float wv, float before) { return ADD ? fmaf(wv, qv, before) : __fmul_rn(wv, qv); };
    t0 = term(wc.x, t0);
    if (((ic.x | ic.y) & 0x80008000u) == 0) {
      t1 = term(wc.y, t1);
      t2 = term(wc.z, t2);
      t3 = term(wc.w, t3);
    } else {
      next(ic.x & 0x8000u);
      t1 = term(wc.y, t1);
      next(ic.x & 0x80000000u);
      t2 = term(wc.z, t2);
      next(ic.y & 0x8000u);
      t3 = term(wc.w, t3);
      next(ic.y & 0x80000000u);
    }
    sts_f32(a0, t0);
    sts_f32(a1, t1);
    sts_f32(a2, t2);
    sts_f32(a3, t3);
  });
}

// Rows of several runs: their runs' sums sit in q at extra slots; a thread adds
// up to kCellFew of them, a warp more, in a fixed order.  One slice (ADD =
// false): the total is the row's sum, written back to the extra slots for the
// scatter.  Several: it is added to the row, the extra slots are cleared for the
// next slice, and cell_spread writes the finished row back before the scatter.
// Few-run rows fill tk_comb from its end, the others from its start.
template <int NW, bool ADD>
__device__ __forceinline__ void cell_join(const DevPlan& P, int cell, float* q) {
  const int warp = static_cast<int>(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int2 n = __ldg(P.tk_ncomb + cell);
  const int2* cb = P.tk_comb + static_cast<int64_t>(cell) * P.tk_cmax;
  for (int i = threadIdx.x; i < n.y; i += NW * 32) {
    const int2 c = __ldg(cb + P.tk_cmax - 1 - i);
    const int row = c.x & 0xffff, cnt = (c.x >> 16) & 0xffff;
    float v = 0.0f;
    for (int e = 0; e < cnt; ++e) v += q[c.y + e];
    for (int e = 0; e < cnt; ++e) q[c.y + e] = ADD ? 0.0f : v;
    if (ADD) q[row] += v;
    else q[row] = v;
  }
  for (int i = warp; i < n.x; i += NW) {
    const int2 c = __ldg(cb + i);
    const int row = c.x & 0xffff, cnt = (c.x >> 16) & 0xffff;
    float v = 0.0f;
    for (int e = lane; e < cnt; e += 32) v += q[c.y + e];
    v = warp_sum(v);
    for (int e = lane; e < cnt; e += 32) q[c.y + e] = ADD ? 0.0f : v;
    if (lane == 0) {
      if (ADD) q[row] += v;
      else q[row] = v;
    }
  }
}
template <int NW>
__device__ __forceinline__ void cell_spread(const DevPlan& P, int cell, float* q) {
  const int warp = static_cast<int>(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int2 n = __ldg(P.tk_ncomb + cell);
  const int2* cb = P.tk_comb + static_cast<int64_t>(cell) * P.tk_cmax;
  for (int i = threadIdx.x; i < n.y; i += NW * 32) {
    const int2 c = __ldg(cb + P.tk_cmax - 1 - i);
    const float v = q[c.x & 0xffff];
    for (int e = 0; e < ((c.x >> 16) & 0xffff); ++e) q[c.y + e] = v;
  }
  for (int i = warp; i < n.x; i += NW) {
    const int2 c = __ldg(cb + i);
    const float v = q[c.x & 0xffff];
    for (int e = lane; e < ((c.x >> 16) & 0xffff); e += 32) q[c.y + e] = v;
  }
}

// Phase 1 of one task: the grids l0 .. l0 + ng - 1.  p = s + beta p_old (s at the
// first iteration) slice by slice, the grids' row sums, |q|^2 (scaled by rsf;
// this thread's compensated share is returned), and t of every coefficient to
// tp.  Its own function (not inlined) for its registers; all threads call it, and
// it ends with a block barrier.
template <int BT>
__device__ __noinline__ float2 cells_task(const DevPlan& P, unsigned char* dsm, int l0, int ng, float beta, bool first,
                                          float rsf, float* tp) {
  constexpr int NW = BT / 32;
  const int tid = static_cast<int>(threadIdx.x), warp = tid >> 5, lane = tid & 31;
  const int N = P.N, S = P.tk_slices, SL = P.tk_sl, l1 = l0 + ng;
  float* const qs = reinterpret_cast<float*>(dsm);  // [tk_q] row sums and destinations of the grids
  float* const vs = qs + P.tk_q;                    // [SL + 32] the slice of p, then of t
  const float* const sv = reinterpret_cast<const float*>(P.sp32);
  const float* const pv = sv + ((N + 3) & ~3);
  auto q_of = [&](int l) { return qs + __ldg(P.tk_qoff + l); };
  auto dest_of = [&](int l) {
    return reinterpret_cast<uint16_t*>(q_of(l) + cell_q_floats(__ldg(P.tk_rows + l), P.tk_ext));
  };
  // a cell's row sums, this lane's first destination and this warp's blocks;
  // loaded one cell ahead
  struct Geom {
    const uint2* idx;
    const float4* w;
    int n;
    uint32_t sq, sd;
  };
  auto geom = [&](int l, int s) {
    const int2* wt = P.tk_wtab + static_cast<int64_t>(l * S + s) * (NW + 1) + warp;
    const int2 a = __ldg(wt);
    const int off = __ldg(P.tk_qoff + l), rows = __ldg(P.tk_rows + l);
    Geom g;
    const int64_t at = (static_cast<int64_t>(l * S + s) * P.tk_blocks + a.x) * 32 + lane;
    g.idx = reinterpret_cast<const uint2*>(P.tk_idx) + at;
    g.w = reinterpret_cast<const float4*>(P.tk_w) + at;
    g.n = __ldg(&wt[1].x) - a.x;
    g.sq = shared_addr(qs + off);
    g.sd = g.sq + 4 * cell_q_floats(rows, P.tk_ext) + (a.y * 32 + lane) * 2;
    return g;
  };
  const uint32_t sp = shared_addr(vs);
  if (S > 1) {
    for (int i = tid; i < P.tk_q; i += BT) qs[i] = 0.0f;
    __syncthreads();  // the copies below write the destinations in between
  }
  for (int l = l0; l < l1; ++l) cell_load_dest<NW>(P, l * S, dest_of(l));
  for (int s = 0; s < S; ++s) {
    const int m0 = s * SL, n = min(SL, N - m0);
    if (s > 0) {
      for (int l = l0; l < l1; ++l) cell_load_dest<NW>(P, l * S + s, dest_of(l));
    }
    Geom cur = geom(l0, s);
    if (first) {
#pragma unroll 4
      for (int i = 4 * tid; i < n; i += 4 * BT)
        *reinterpret_cast<float4*>(vs + i) = ldcg(reinterpret_cast<const float4*>(sv + m0 + i));
    } else {
#pragma unroll 4
      for (int i = 4 * tid; i < n; i += 4 * BT) {
        const float4 a = ldcg(reinterpret_cast<const float4*>(sv + m0 + i));
        const float4 b = ldcg(reinterpret_cast<const float4*>(pv + m0 + i));
        *reinterpret_cast<float4*>(vs + i) =
            make_float4(fmaf(beta, b.x, a.x), fmaf(beta, b.y, a.y), fmaf(beta, b.z, a.z), fmaf(beta, b.w, a.w));
      }
    }
    if (tid < 32) vs[SL + tid] = 0.0f;  // what padding entries read
    cp_async_wait();
    __syncthreads();
    for (int l = l0; l < l1; ++l) {
      const Geom g = cur;
      if (l + 1 < l1) cur = geom(l + 1, s);
      if (g.n == 0) continue;
      if (S > 1) cell_gather<true>(g.idx, g.w, g.n, sp, g.sq, g.sd);
      else cell_gather<false>(g.idx, g.w, g.n, sp, g.sq, g.sd);
    }
    __syncthreads();
    for (int l = l0; l < l1; ++l) {
      if (S > 1) cell_join<NW, true>(P, l * S + s, q_of(l));
      else cell_join<NW, false>(P, l * S + s, q_of(l));
    }
    __syncthreads();
  }
  // |q|^2: compensated sums of exact squares
  float hi = 0.0f, lo = 0.0f;
  for (int l = l0; l < l1; ++l) {
    const float* q = q_of(l);
    const int nr = __ldg(P.tk_rows + l);
    for (int i = tid; i < nr; i += BT) {
      const float2 sq = df_square(q[i] * rsf);
      const float2 t = df_two_sum(hi, sq.x);
      hi = t.x;
      lo += t.y + sq.y;
    }
  }
  // t = sum over the grids of A_l^T q_l
  for (int s = 0; s < S; ++s) {
    const int m0 = s * SL, n = min(SL, N - m0);
    Geom cur = geom(l0, s);
    if (S > 1) {
      for (int l = l0; l < l1; ++l) cell_load_dest<NW>(P, l * S + s, dest_of(l));
      for (int l = l0; l < l1; ++l) cell_spread<NW>(P, l * S + s, q_of(l));
      cp_async_wait();
      __syncthreads();
    }
    for (int l = l0; l < l1; ++l) {
      const Geom g = cur;
      if (l + 1 < l1) cur = geom(l + 1, s);
      if (g.n > 0) {
        if (l == l0) cell_scatter<false>(g.idx, g.w, g.n, sp, g.sq, g.sd);
        else cell_scatter<true>(g.idx, g.w, g.n, sp, g.sq, g.sd);
      }
      __syncthreads();
    }
    for (int i = 4 * tid; i < n; i += 4 * BT)
      stcg(reinterpret_cast<float4*>(tp + m0 + i), *reinterpret_cast<const float4*>(vs + i));
    __syncthreads();
  }
  return df_two_sum(hi, lo);
}

// CG on A^T A d = g by grid groups (see the head of this file).  On entry
// s = right-hand side, x = 0, gamma0 = |s|^2; returns as cg_normal does.  s and p
// are the halves of sp32, tpart lives in y0 and the per-task and per-chunk
// partials in y1 (the DCT's buffers, free by now).
template <int BT>
__device__ bool cg_cells(const DevPlan& P, Team& tm, unsigned char* dsm, double gamma0, double tol, int max_iter,
                         int stall, int* iters_out, double* gamma_out, int* status_out) {
  constexpr int NW = BT / 32;
  __shared__ float2 wpart[kUnitGroup][NW];
  __shared__ float sh_ab[2];  // alpha, beta
  __shared__ double sh_gam;
  __shared__ int sh_ctl[3];   // stop flag, status, iterations
  *status_out = FCT_OK;
  *iters_out = 0;
  *gamma_out = gamma0;
  if (!(gamma0 > 0.0) || !isfinite(gamma0)) {
    if (!isfinite(gamma0)) *status_out = FCT_ERR_NONFINITE;
    return true;
  }
  const int N = P.N, K = P.K, NG = P.tk_groups, GG = P.tk_gg;
  const int64_t NP = P.tk_np;
  const int CW = P.tk_cw, LG = P.tk_lg, nown = P.tk_nown;
  const int tid = static_cast<int>(threadIdx.x), warp = tid >> 5, lane = tid & 31;
  float* const tpart = reinterpret_cast<float*>(P.y0);
  float2* const part_r = reinterpret_cast<float2*>(P.y1);
  float2* const part_c = part_r + NG;
  float* const sv = reinterpret_cast<float*>(P.sp32);
  float* const pv = sv + ((N + 3) & ~3);
  float* const xv = P.dx32;
  int e0 = 0;
  frexp(gamma0, &e0);
  const double rs = ldexp(1.0, -(e0 / 2));  // exact scaling near 1/sqrt(gamma0)
  const float rsf = static_cast<float>(rs);
  const double c0 = gamma0 * rs * rs;
  const float2 tol2 = df_of(tol * tol * c0);
  // thread 0's state, in scaled units
  float2 gam = df_of(c0);
  float2 best = gam;
  int best_it = 0, it = 0;
  bool first = true;
  auto flush = [&](float2* part, int u0, int nk) {
    __syncthreads();
    if (tid < nk) {
      stcg(part + u0 + tid * tm.G, warps_sum<NW>(wpart[tid]));
    }
    __syncthreads();
  };
  int ctl = 0;
  for (;;) {
    // ================= phase 1
    {
      if (warp == 0) {
        float2 gnew = gam;
        if (!first) gnew = warp0_sum(part_c, nown);
        if (tid == 0) {
          int c = 0;
          float bt = 0.0f;
          if (!first) {
            ++it;
            if (!isfinite(gnew.x)) {
              c = FCT_ERR_NONFINITE + 16;
            } else {
              bt = df_div(gnew, gam).x;
              gam = gnew;
              if (!df_less(tol2, gam)) c = 1;
              else if (it >= max_iter) c = FCT_ERR_NOCONV + 16;
              else if (stall > 0) {
                if (df_less(gam, best)) {
                  best = gam;
                  best_it = it;
                } else if (it - best_it >= stall) {
                  c = 1;
                }
              }
            }
          }
          sh_ab[1] = bt;
          sh_ctl[0] = c;
        }
      }
      __syncthreads();
      ctl = sh_ctl[0];
      if (ctl != 0) break;
      const float beta = sh_ab[1];
      int kg = 0, u0 = tm.rank;
      for (int g = tm.rank; g < NG; g += tm.G) {
        const int l0 = g * GG;
        const float2 part = warp_sum(cells_task<BT>(P, dsm, l0, min(K, l0 + GG) - l0, beta, first, rsf, tpart + g * NP));
        if (lane == 0) wpart[kg][warp] = part;
        if (++kg == kUnitGroup && g + tm.G < NG) {
          flush(part_r, u0, kg);
          kg = 0;
          u0 = g + tm.G;
        }
      }
      if (!phase_end<NW>(tm, wpart, part_r, u0, kg)) return false;
    }
    // ================= phase 2: t = sum over groups; s, p, x of the owned chunk
    {
      const int mi = tid % CW, gl = tid / CW;
      auto sum_t = [&](int m) -> float {
        float a = 0.0f;
        const float* tp = tpart + m;
        for (int g = gl; g < NG; g += 16 * LG) {
          float v[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = ldcg(tp + min(g + i * LG, NG - 1) * NP);
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (g + i * LG < NG) a += v[i];
        }
        return a;
      };
      float* const comb = reinterpret_cast<float*>(dsm);  // [LG][CW] when LG > 1
      int c = tm.rank;
      float t = 0.0f, so = 0.0f, po = 0.0f, xo = 0.0f;
      auto load = [&](int ch) {
        const int m = ch * CW + mi;
        t = 0.0f;
        if (gl < LG && m < N) {
          if (gl == 0) {
            so = ldcg(sv + m);
            xo = ldcg(xv + m);
            if (!first) po = ldcg(pv + m);
          }
          t = sum_t(m);
        }
      };
      if (warp == 0) {
        const float2 dl = warp0_sum(part_r, NG);
        if (tid == 0) {
          int cc = 0;
          float al = 0.0f;
          if (!isfinite(dl.x)) cc = FCT_ERR_NONFINITE + 16;
          else if (!(dl.x > 0.0f)) cc = 1;  // q = 0: s is already zero to working precision
          else al = df_div(gam, dl).x;
          sh_ab[0] = al;
          sh_ctl[0] = cc;
        }
      }
      if (c < nown) load(c);
      __syncthreads();
      ctl = sh_ctl[0];
      if (ctl != 0) break;
      const float alpha = sh_ab[0], beta = sh_ab[1];
      int k = 0, kg = 0, u0 = c;
      for (; c < nown; c += tm.G, ++k) {
        if (k > 0) load(c);
        if (LG > 1) {
          if (k > 0) __syncthreads();  // the previous chunk's sums are read
          if (gl < LG) comb[gl * CW + mi] = t;
          __syncthreads();
          if (gl == 0)
            for (int w = 1; w < LG; ++w) t += comb[w * CW + mi];
        }
        const int m = c * CW + mi;
        float2 part = make_float2(0.0f, 0.0f);
        if (gl == 0 && m < N) {
          const float pn = first ? so : fmaf(beta, po, so);
          const float sn = fmaf(-alpha, t, so);
          stcg(sv + m, sn);
          stcg(pv + m, pn);
          stcg(xv + m, fmaf(alpha, pn, xo));
          part = df_square(sn * rsf);
        }
        part = warp_sum(part);
        if (lane == 0) wpart[kg][warp] = part;
        if (++kg == kUnitGroup && c + tm.G < nown) {
          flush(part_c, u0, kg);
          kg = 0;
          u0 = c + tm.G;
        }
      }
      if (!phase_end<NW>(tm, wpart, part_c, u0, kg)) return false;
    }
    first = false;
  }
  if (tid == 0) {
    sh_ctl[1] = ctl >= 16 ? ctl - 16 : FCT_OK;
    sh_ctl[2] = it;
    sh_gam = static_cast<double>(gam.x) + static_cast<double>(gam.y);
  }
  __syncthreads();
  *status_out = sh_ctl[1];
  *iters_out = sh_ctl[2];
  *gamma_out = sh_gam / (rs * rs);
  __syncthreads();
  return true;
}
