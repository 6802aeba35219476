// Inner solve of the mixed path by grid groups: CG on A^T A d = g with every
// alias product formed one grid at a time in shared memory.  Included only by
// fct_solver.cuh.
//
// A^T A = sum_l A_l^T A_l, and a grid's block A_l has one entry per column, so
// q_l = A_l s and t_l = A_l^T q_l need nothing from the other grids: a block
// that holds s (or a slice of it) and q_l in shared memory does both, and only
// the sum over grids t = sum_l t_l and the vector updates cross blocks.
//
// The iteration is the form of CG with one point of reduction (Chronopoulos
// and Gear): the operator is applied to the residual s, not to p, so phase 1
// needs no scalar and reads 4 bytes per coefficient:
//   phase 1, per task (a group of tk_gg grids, one block): q_l = A_l s and
//     delta = |q|^2, then t = sum_{l in group} A_l^T q_l, streamed out (tpart);
//   phase 2, per owner chunk: gamma = |s|^2, beta = gamma / gamma_prev,
//     alpha = gamma / (delta - beta gamma / alpha_prev);
//     p = s + beta p, z = t + beta z, x += alpha p, s -= alpha z.
// Two team barriers per iteration, as in cg_normal, but every scattered access
// is to shared memory and global traffic is coalesced: 6 bytes of table per
// entry (read by the gather and again, from L2, by the scatter).
//
// Cell tables.  A cell is one (grid, slice of tk_sl coefficients).  Its rows are
// cut into runs of at most kCellRun entries, sorted by length, 32 to a group:
// lane i of a warp sums run i of the group, one entry a step, so a step is 32
// independent entries and pads are few (sorted lengths).  A warp's groups are
// contiguous, so it streams its steps, four at a time, without looking at group
// boundaries ahead: bit 15 of a step's indices marks the last step of a group,
// where the lanes store their sums and go on to the next 32 runs.  Rows of
// several runs are completed by cell_join.  The order of additions depends only
// on the plan and the block size, so a transform's result is the same bit for
// bit alone, in a batch and for any team size.
#pragma once

#include "fct_common.cuh"

__device__ __forceinline__ float2 df_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  const float e = fmaf(a.x, b.x, -p) + fmaf(a.x, b.y, __fmul_rn(a.y, b.x));
  const float hi = p + e;
  return make_float2(hi, e - (hi - p));
}
__device__ __forceinline__ float2 df_div(float2 a, float2 b) {
  const float q1 = __fdividef(a.x, b.x);
  const float2 qb = df_mul(make_float2(q1, 0.0f), b);
  const float2 r = df_add(a, make_float2(-qb.x, -qb.y));
  const float q2 = __fdividef(r.x, b.x);
  const float hi = q1 + q2;
  return make_float2(hi, q2 - (hi - q1));
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// A grid's part of the shared memory: its row sums (rows, extra slots, one slot
// for idle lanes), then the run destinations of the cell at hand.
__device__ __forceinline__ int cell_q_floats(int rows, int ext) { return (rows + ext + 1 + 3) & ~3; }

struct CellView {  // one cell, as its warp sees it
  const uint2* idx;       // [blocks][32] four steps per lane
  const float4* w;
  const uint16_t* dest;   // shared, [groups][32], this lane's
  int b0, b1;             // this warp's blocks of four steps
};

template <int NW>
__device__ __forceinline__ CellView cell_view(const DevPlan& P, int cell, const uint16_t* dest) {
  const int warp = static_cast<int>(threadIdx.x >> 5), lane = threadIdx.x & 31;
  CellView v;
  const int2* wt = P.tk_wtab + static_cast<int64_t>(cell) * (NW + 1) + warp;
  const int2 a = __ldg(wt), b = __ldg(wt + 1);
  v.b0 = a.x;
  v.b1 = b.x;
  const int64_t base = static_cast<int64_t>(cell) * P.tk_blocks * 32 + lane;
  v.idx = reinterpret_cast<const uint2*>(P.tk_idx) + base;
  v.w = reinterpret_cast<const float4*>(P.tk_w) + base;
  v.dest = dest + a.y * 32 + lane;
  return v;
}

// Run destinations of a cell into shared memory (asynchronous copies; two
// groups of idle destinations follow the last).
template <int NW>
__device__ __forceinline__ void cell_load_dest(const DevPlan& P, int cell, uint16_t* dest) {
  const int n16 = (__ldg(P.tk_wtab + static_cast<int64_t>(cell) * (NW + 1) + NW).y + 2) * 4;
  const uint16_t* src = P.tk_dest + static_cast<int64_t>(cell) * P.tk_gmax * 32;
  for (int i = threadIdx.x; i < n16; i += NW * 32) cp_async16(dest + 8 * i, src + 8 * i);
}

constexpr int kCellAhead = 4;  // blocks of four steps a warp keeps in flight

// q[dest] (+)= the sums of w s over the cell's runs.  ADD: the plan has several
// slices, whose sums add up in q.
template <int NW, bool ADD>
__device__ __forceinline__ void cell_gather(const CellView& v, const float* s, float* q) {
  if (v.b0 >= v.b1) return;
  uint2 in[kCellAhead];
  float4 wn[kCellAhead];
#pragma unroll
  for (int j = 0; j < kCellAhead; ++j) {
    const int b = min(v.b0 + j, v.b1 - 1);
    in[j] = __ldg(v.idx + b * 32);
    wn[j] = __ldg(v.w + b * 32);
  }
  const uint16_t* dp = v.dest;
  float acc = 0.0f;
  for (int b = v.b0; b < v.b1; b += kCellAhead) {
#pragma unroll
    for (int j = 0; j < kCellAhead; ++j) {
      if (b + j >= v.b1) continue;
      const uint2 ic = in[j];
      const float4 wc = wn[j];
      const int nb = min(b + kCellAhead + j, v.b1 - 1);
      in[j] = __ldg(v.idx + nb * 32);
      wn[j] = __ldg(v.w + nb * 32);
      const float s0 = s[ic.x & 0x7fffu], s1 = s[(ic.x >> 16) & 0x7fffu];
      const float s2 = s[ic.y & 0x7fffu], s3 = s[(ic.y >> 16) & 0x7fffu];
      auto end = [&](uint32_t mark) {
        if (mark) {  // the same for all lanes
          const int d = *dp;
          if (ADD) q[d] += acc;
          else q[d] = acc;
          acc = 0.0f;
          dp += 32;
        }
      };
      acc = fmaf(wc.x, s0, acc);
      if (((ic.x | ic.y) & 0x80008000u) == 0) {  // no run ends here
        acc = fmaf(wc.y, s1, acc);
        acc = fmaf(wc.z, s2, acc);
        acc = fmaf(wc.w, s3, acc);
      } else {
        end(ic.x & 0x8000u);
        acc = fmaf(wc.y, s1, acc);
        end(ic.x & 0x80000000u);
        acc = fmaf(wc.z, s2, acc);
        end(ic.y & 0x8000u);
        acc = fmaf(wc.w, s3, acc);
        end(ic.y & 0x80000000u);
      }
    }
  }
}

// t[m] (+)= w q[row] over the cell's entries.  Every column has one entry per
// grid, so no two entries of a cell touch the same t; the first grid of a group
// stores, the others add.
template <int NW, bool ADD>
__device__ __forceinline__ void cell_scatter(const CellView& v, const float* q, float* t) {
  if (v.b0 >= v.b1) return;
  uint2 in[kCellAhead];
  float4 wn[kCellAhead];
#pragma unroll
  for (int j = 0; j < kCellAhead; ++j) {
    const int b = min(v.b0 + j, v.b1 - 1);
    in[j] = __ldg(v.idx + b * 32);
    wn[j] = __ldg(v.w + b * 32);
  }
  const uint16_t* dp = v.dest;
  float qv = q[*dp];
  for (int b = v.b0; b < v.b1; b += kCellAhead) {
#pragma unroll
    for (int j = 0; j < kCellAhead; ++j) {
      if (b + j >= v.b1) continue;
      const uint2 ic = in[j];
      const float4 wc = wn[j];
      const int nb = min(b + kCellAhead + j, v.b1 - 1);
      in[j] = __ldg(v.idx + nb * 32);
      wn[j] = __ldg(v.w + nb * 32);
      const uint32_t a0 = ic.x & 0x7fffu, a1 = (ic.x >> 16) & 0x7fffu, a2 = ic.y & 0x7fffu, a3 = (ic.y >> 16) & 0x7fffu;
      float t0 = 0.0f, t1 = 0.0f, t2 = 0.0f, t3 = 0.0f;
      if (ADD) {  // the four entries of a lane are different columns
        t0 = t[a0];
        t1 = t[a1];
        t2 = t[a2];
        t3 = t[a3];
      }
      auto next = [&](uint32_t mark) {
        if (mark) {
          dp += 32;
          qv = q[*dp];
        }
      };
      auto term = [&](float w, float old) { return ADD ? fmaf(w, qv, old) : w * qv; };
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
      t[a0] = t0;
      t[a1] = t1;
      t[a2] = t2;
      t[a3] = t3;
    }
  }
}

// Rows of several runs: their runs' sums sit in q at extra slots; a warp adds
// them in a fixed order.  One slice (ADD = false): the total is the row's sum,
// written back to the extra slots for the scatter.  Several: it is added to the
// row, and cell_spread writes the finished row back before the scatter.
template <int NW, bool ADD>
__device__ __forceinline__ void cell_join(const DevPlan& P, int cell, float* q) {
  const int warp = static_cast<int>(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int n = __ldg(P.tk_ncomb + cell);
  const int2* cb = P.tk_comb + static_cast<int64_t>(cell) * P.tk_cmax;
  for (int i = warp; i < n; i += NW) {
    const int2 c = __ldg(cb + i);
    const int row = c.x & 0xffff, cnt = (c.x >> 16) & 0xffff;
    float v = 0.0f;
    for (int e = lane; e < cnt; e += 32) v += q[c.y + e];
    v = warp_sum(v);
    if (ADD) {
      if (lane == 0) q[row] += v;
    } else {
      for (int e = lane; e < cnt; e += 32) q[c.y + e] = v;
      if (lane == 0) q[row] = v;
    }
  }
}
template <int NW>
__device__ __forceinline__ void cell_spread(const DevPlan& P, int cell, float* q) {
  const int warp = static_cast<int>(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int n = __ldg(P.tk_ncomb + cell);
  const int2* cb = P.tk_comb + static_cast<int64_t>(cell) * P.tk_cmax;
  for (int i = warp; i < n; i += NW) {
    const int2 c = __ldg(cb + i);
    const float v = q[c.x & 0xffff];
    for (int e = lane; e < ((c.x >> 16) & 0xffff); e += 32) q[c.y + e] = v;
  }
}

// Warp 0: the double-float sums of two lists of partials (every lane).
__device__ __forceinline__ void warp0_sum2(const float2* a, int na, const float2* b, int nb, float2* sa, float2* sb) {
  float2 va = make_float2(0.0f, 0.0f), vb = va;
  for (int i0 = threadIdx.x; i0 < max(na, nb); i0 += 32 * 8) {
    float2 ta[8], tb[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int i = i0 + 32 * j;
      ta[j] = i < na ? ldcg(a + i) : make_float2(0.0f, 0.0f);
      tb[j] = i < nb ? ldcg(b + i) : make_float2(0.0f, 0.0f);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
      for (int j = 0; j < o; ++j) {
        ta[j] = df_add(ta[j], ta[j + o]);
        tb[j] = df_add(tb[j], tb[j + o]);
      }
    va = df_add(va, ta[0]);
    vb = df_add(vb, tb[0]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    va = df_add(va, make_float2(__shfl_xor_sync(0xffffffffu, va.x, o), __shfl_xor_sync(0xffffffffu, va.y, o)));
    vb = df_add(vb, make_float2(__shfl_xor_sync(0xffffffffu, vb.x, o), __shfl_xor_sync(0xffffffffu, vb.y, o)));
  }
  *sa = va;
  *sb = vb;
}

// CG on A^T A d = g by grid groups (see the head of this file).  On entry
// s = right-hand side, x = 0, gamma0 = |s|^2; returns as cg_normal does.  s and p
// are the halves of sp32, z is q32, tpart lives in y0 and the per-task and
// per-chunk partials in y1 (the DCT's buffers, free by now).
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
  const int N = P.N, K = P.K, NG = P.tk_groups, GG = P.tk_gg, S = P.tk_slices, SL = P.tk_sl;
  const int64_t NP = P.tk_np;
  const int CW = P.tk_cw, LG = P.tk_lg, nown = P.tk_nown;
  const int tid = static_cast<int>(threadIdx.x), warp = tid >> 5;
  float* const qs = reinterpret_cast<float*>(dsm);  // [tk_q] row sums of the group's grids
  float* const vs = qs + P.tk_q;                    // [SL + 32] the slice of s, then of t
  float* const tpart = reinterpret_cast<float*>(P.y0);
  float2* const part_r = reinterpret_cast<float2*>(P.y1);
  float2* const part_c = part_r + NG;
  float* const sv = reinterpret_cast<float*>(P.sp32);
  float* const pv = sv + N;
  float* const zv = P.q32;
  float* const xv = P.dx32;
  int e0 = 0;
  frexp(gamma0, &e0);
  const double rs = ldexp(1.0, -(e0 / 2));  // exact scaling near 1/sqrt(gamma0)
  const float rsf = static_cast<float>(rs);
  const double c0 = gamma0 * rs * rs;
  const float tol2 = static_cast<float>(tol * tol * c0);
  // thread 0's state, in scaled units
  const float2 g0 = make_float2(static_cast<float>(c0), static_cast<float>(c0 - static_cast<float>(c0)));
  float2 gam_prev = g0, al_prev = make_float2(1.0f, 0.0f), gam = g0;
  float best = 3.0e38f;
  int best_it = 0;
  auto dest_of = [&](int l) {
    return reinterpret_cast<uint16_t*>(qs + __ldg(P.tk_qoff + l) + cell_q_floats(__ldg(P.tk_rows + l), P.tk_ext));
  };
  auto flush = [&](float2* part, int u0, int nk) {
    __syncthreads();
    if (tid < nk) {
      float2 v = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int w = 0; w < NW; ++w) v = padd(v, wpart[tid][w]);
      stcg(part + u0 + tid * tm.G, v);
    }
    __syncthreads();
  };
  int ctl = 0, it = 0;
  for (;; ++it) {
    // ================= phase 1
    {
      int kg = 0, u0 = tm.rank;
      for (int g = tm.rank; g < NG; g += tm.G) {
        const int l0 = g * GG, l1 = min(K, l0 + GG);
        if (S > 1) {
          for (int i = tid; i < P.tk_q; i += BT) qs[i] = 0.0f;
          __syncthreads();  // the copies below write the destinations in between
        }
        for (int s = 0; s < S; ++s) {
          const int m0 = s * SL, n = min(SL, N - m0);
          for (int i = 4 * tid; i < n; i += 4 * BT) cp_async16(vs + i, sv + m0 + i);
          for (int l = l0; l < l1; ++l) cell_load_dest<NW>(P, l * S + s, dest_of(l));
          if (tid < 32) vs[SL + tid] = 0.0f;  // what padding entries read
          cp_async_wait();
          __syncthreads();
          for (int l = l0; l < l1; ++l) {
            const CellView v = cell_view<NW>(P, l * S + s, dest_of(l));
            float* q = qs + __ldg(P.tk_qoff + l);
            if (S > 1) cell_gather<NW, true>(v, vs, q);
            else cell_gather<NW, false>(v, vs, q);
          }
          __syncthreads();
          for (int l = l0; l < l1; ++l) {
            float* q = qs + __ldg(P.tk_qoff + l);
            if (S > 1) cell_join<NW, true>(P, l * S + s, q);
            else cell_join<NW, false>(P, l * S + s, q);
          }
          if (S > 1) {  // the next slice uses the extra slots again
            __syncthreads();
            for (int l = l0; l < l1; ++l) {
              float* q = qs + __ldg(P.tk_qoff + l) + __ldg(P.tk_rows + l);
              for (int i = tid; i < P.tk_ext; i += BT) q[i] = 0.0f;
            }
          }
        }
        __syncthreads();
        // delta: compensated sums of exact squares
        float hi = 0.0f, lo = 0.0f;
        for (int l = l0; l < l1; ++l) {
          const float* q = qs + __ldg(P.tk_qoff + l);
          const int nr = __ldg(P.tk_rows + l);
          for (int i = tid; i < nr; i += BT) {
            const float2 sq = df_square(q[i] * rsf);
            const float2 t = df_two_sum(hi, sq.x);
            hi = t.x;
            lo += t.y + sq.y;
          }
        }
        const float2 part = warp_sum(df_two_sum(hi, lo));
        if ((tid & 31) == 0) wpart[kg][warp] = part;
        // t = sum over the group's grids of A_l^T q_l
        float* tp = tpart + g * NP;
        for (int s = 0; s < S; ++s) {
          const int m0 = s * SL, n = min(SL, N - m0);
          if (S > 1) {
            for (int l = l0; l < l1; ++l) cell_load_dest<NW>(P, l * S + s, dest_of(l));
            for (int l = l0; l < l1; ++l) cell_spread<NW>(P, l * S + s, qs + __ldg(P.tk_qoff + l));
            if (tid < 32) vs[SL + tid] = 0.0f;
            cp_async_wait();
            __syncthreads();
          }
          for (int l = l0; l < l1; ++l) {
            const CellView v = cell_view<NW>(P, l * S + s, dest_of(l));
            const float* q = qs + __ldg(P.tk_qoff + l);
            if (l == l0) cell_scatter<NW, false>(v, q, vs);
            else cell_scatter<NW, true>(v, q, vs);
            __syncthreads();
          }
          for (int i = 4 * tid; i < n; i += 4 * BT)
            stcg(reinterpret_cast<float4*>(tp + m0 + i), *reinterpret_cast<const float4*>(vs + i));
          __syncthreads();
        }
        if (++kg == kUnitGroup && g + tm.G < NG) {
          flush(part_r, u0, kg);
          kg = 0;
          u0 = g + tm.G;
        }
      }
      if (!phase_end<NW>(tm, wpart, part_r, u0, kg)) return false;
    }
    // ================= phase 2: t = sum over groups; p, z, x, s of the owned chunk
    {
      // gamma's partials alternate: a block may finish this phase while another
      // still reads the previous ones
      const float2* const pc_in = part_c + ((it & 1) ? nown : 0);
      float2* const pc_out = part_c + ((it & 1) ? 0 : nown);
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
      float t = 0.0f, so = 0.0f, po = 0.0f, zo = 0.0f, xo = 0.0f;
      auto load = [&](int ch) {
        const int m = ch * CW + mi;
        t = 0.0f;
        if (gl < LG && m < N) {
          if (gl == 0) {
            so = ldcg(sv + m);
            xo = ldcg(xv + m);
            if (it > 0) {
              po = ldcg(pv + m);
              zo = ldcg(zv + m);
            }
          }
          t = sum_t(m);
        }
      };
      if (warp == 0) {
        float2 gs, dl;
        warp0_sum2(pc_in, it > 0 ? nown : 0, part_r, NG, &gs, &dl);
        if (tid == 0) {
          if (it > 0) gam = gs;
          int cc = 0;
          float2 al = make_float2(0.0f, 0.0f), bt = al;
          if (!isfinite(gam.x) || !isfinite(dl.x)) {
            cc = FCT_ERR_NONFINITE + 16;
          } else if (it > 0 && gam.x <= tol2) {
            cc = 1;
          } else if (it >= max_iter) {
            cc = FCT_ERR_NOCONV + 16;
          } else if (it > 0 && stall > 0) {
            if (gam.x < best) {
              best = gam.x;
              best_it = it;
            } else if (it - best_it >= stall) {
              cc = 1;
            }
          }
          if (cc == 0) {
            float2 den = dl;
            if (it > 0) {
              bt = df_div(gam, gam_prev);
              const float2 u = df_div(df_mul(bt, gam), al_prev);
              den = df_add(dl, make_float2(-u.x, -u.y));
            }
            if (!(den.x > 0.0f)) {
              cc = 1;  // no further progress in this precision
            } else {
              al = df_div(gam, den);
              gam_prev = gam;
              al_prev = al;
            }
          }
          sh_ab[0] = al.x;
          sh_ab[1] = bt.x;
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
          const float pn = it > 0 ? fmaf(beta, po, so) : so;
          const float zn = it > 0 ? fmaf(beta, zo, t) : t;
          const float sn = fmaf(-alpha, zn, so);
          stcg(sv + m, sn);
          stcg(pv + m, pn);
          stcg(zv + m, zn);
          stcg(xv + m, fmaf(alpha, pn, xo));
          part = df_square(sn * rsf);
        }
        part = warp_sum(part);
        if ((tid & 31) == 0) wpart[kg][warp] = part;
        if (++kg == kUnitGroup && c + tm.G < nown) {
          flush(pc_out, u0, kg);
          kg = 0;
          u0 = c + tm.G;
        }
      }
      if (!phase_end<NW>(tm, wpart, pc_out, u0, kg)) return false;
    }
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
