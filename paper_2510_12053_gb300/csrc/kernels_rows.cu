// Stable Neo-Hookean gradient and upper Hessian block rows formed per free
// row from the positions: no per-tet Hessian store.
//
// For a free vertex j and an incident tet, number the other three corners
// 1, 2, 3 so that (j, 1, 2, 3) is positively oriented, and let e_k = x_k - x_j,
//   n_1 = e_2 x e_3, n_2 = e_3 x e_1, n_3 = e_1 x e_2, n_0 = -(n_1 + n_2 + n_3),
//   det = e_1 . n_1,  D = 6 V (rest),  J = det / D.
// With C = cof F, C G_k = n_k / D, and because the rest shape vectors are dual
// to the rest edges, F (G_0 x G_1) = (e_3 - e_2) / D and cyclically.  So the
// energy's derivatives (see kernels_energy.cu for the same terms through F)
//   dE/dx_j          = w V (mu F G_0 + s C G_0)
//   d2E/dx_j dx_l(k) = w V (mu (G_0 . G_k) I + lam_hat C G_0 (C G_k)^T + s [F (G_0 x G_k)]_skew)
// become, with sigma = w s / 6 = c1 det + c0, c1 = w lam_hat / (6 D),
// c0 = -w (lam_hat + mu) / 6 and m_jl = sum_t w V mu G_j . G_l (constant),
//   g_j  = sum_l m_jl e_l + sum_t sigma n_0
//   H_jl = m_jl I + sum_t ( c1 n_0 n_k^T + sigma [e_a - e_b]_skew ),  (a, b) = (3, 2), (1, 3), (2, 1)
//   H_jj = -sum_l m_jl I + sum_t c1 n_0 n_0^T     (+ mass)
// Nothing here divides or needs F or D_m^{-1}: about 60 float operations per
// (row, tet) for the blocks, so each of a tet's four rows forming its own
// share costs less than one thread forming all ten blocks and sending them
// through memory (320 bytes written per tet and gathered again; that pair of
// kernels was bound by this traffic).  32^3 cube (196 608 tets, 33 759 rows),
// one colour: store + gather 36.7 + 35.0 us, here 8.0 us (sigma) + 24.0 us
// (rows); a whole mixed sweep 579 -> 390 us, 64^3 cube 3.47 -> 2.14 ms.
// Float64, 24 x 23 x 25 box: a sweep 1.77 -> 1.35 ms.
//
// The mixed path keeps the gradient in float-float: sigma comes from a small
// per-tet kernel (formed once instead of by four rows), n_0 as one float-float
// cross product of (e_2 - e_1) and (e_3 - e_1).  Lengths are scaled by a power
// of two near the mean edge (exact), so that c1, det and the error terms of
// the products stay well inside float32's range for any unit of length.
#include <algorithm>
#include <cmath>
#include <vector>

#include "cc_internal.cuh"
#include "dmath.cuh"

namespace ccg {

namespace {

// a b - c d in float-float
__device__ __forceinline__ df df_det2(df a, df b, df c, df d) {
  const float p = __fmul_rn(a.hi, b.hi), q = __fmul_rn(c.hi, d.hi);
  const float ep = __fmaf_rn(a.hi, b.hi, -p), eq = __fmaf_rn(c.hi, d.hi, -q);
  const df s = two_sum(p, -q);
  float lo = __fsub_rn(ep, eq);
  lo = __fmaf_rn(a.hi, b.lo, lo);
  lo = __fmaf_rn(a.lo, b.hi, lo);
  lo = __fmaf_rn(-c.hi, d.lo, lo);
  lo = __fmaf_rn(-c.lo, d.hi, lo);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, lo));
}

__device__ __forceinline__ void cross_df(const df (&a)[3], const df (&b)[3], df (&o)[3]) {
  o[0] = df_det2(a[1], b[2], a[2], b[1]);
  o[1] = df_det2(a[2], b[0], a[0], b[2]);
  o[2] = df_det2(a[0], b[1], a[1], b[0]);
}

template <typename T>
__device__ __forceinline__ void cross3(const T* a, const T* b, T* o) {
  o[0] = a[1] * b[2] - a[2] * b[1];
  o[1] = a[2] * b[0] - a[0] * b[2];
  o[2] = a[0] * b[1] - a[1] * b[0];
}

__device__ __forceinline__ df df_scaled_diff(float ah, float al, float bh, float bl, float s) {
  const df d = df_sub(df{ah, al}, df{bh, bl});
  return df{d.hi * s, d.lo * s};  // s is a power of two
}

// ---- per-tet sigma (mixed path) --------------------------------------------
// rec[t] = (sigma hi, sigma lo, c1, 0) of the listed tets, one thread per tet.
// Bound by float-float arithmetic (~230 operations) and the position gather;
// it writes 16 bytes per tet where the Hessian store took 320.
__global__ void __launch_bounds__(128) k_tet_sigma(const int4* __restrict__ tets, const float4* __restrict__ tc,
                                                   const float4* __restrict__ x_hi, const float4* __restrict__ x_lo,
                                                   const int32_t* __restrict__ list, int64_t count, float scale,
                                                   float4* __restrict__ rec) {
  pdl_entry();
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= count) return;
  const int t = list[k];
  const int4 tv = tets[t];
  const float4 c = tc[t];
  const float4 h0 = x_hi[tv.x], l0 = x_lo[tv.x];
  const float4 h[3] = {x_hi[tv.y], x_hi[tv.z], x_hi[tv.w]}, l[3] = {x_lo[tv.y], x_lo[tv.z], x_lo[tv.w]};
  df e[3][3], n1[3];
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    e[v][0] = df_scaled_diff(h[v].x, l[v].x, h0.x, l0.x, scale);
    e[v][1] = df_scaled_diff(h[v].y, l[v].y, h0.y, l0.y, scale);
    e[v][2] = df_scaled_diff(h[v].z, l[v].z, h0.z, l0.z, scale);
  }
  cross_df(e[1], e[2], n1);
  const df det = df_fma(e[0][2], n1[2], df_fma(e[0][1], n1[1], df_mul(e[0][0], n1[0])));
  const df sg = df_fma(det, df{c.x, c.y}, df{c.z, c.w});
  rec[t] = make_float4(sg.hi, sg.lo, c.x, 0.0f);
}

// ---- rows -------------------------------------------------------------------
// Both row kernels give a row eight lanes, four rows to a warp; a warp shares
// nothing with others.  A Kuhn grid's interior row has 24 tets, 14 neighbours
// and 8 upper blocks: three full rounds over the tets and one over the blocks.
// hdr[2 row], hdr[2 row + 1]: (j, first upper block, upper blocks, first ring
// entry), (ring entries, first vertex-tet entry, entries, first block row).
//
// Codes of an off-diagonal upper block (j, l)'s tets, ascending: 4 (the tet's
// position in the row) + c, where l is the local corner k with k mod 3 = c.
// The first eight are in codes8 (0xffff ends them), all of them in rs_code.

// Calls f(code) for every tet of block p in order; cd = codes8[p].
template <typename F>
__device__ __forceinline__ void for_sources(uint4 cd, int p, const int32_t* __restrict__ rs_ptr,
                                            const uint16_t* __restrict__ rs_code, F&& f) {
  const uint32_t w[4] = {cd.x, cd.y, cd.z, cd.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if ((w[i] & 0xffff) == 0xffff) break;
    f(w[i] & 0xffff);
    if ((w[i] >> 16) != 0xffff) f(w[i] >> 16);
  }
  if ((w[3] >> 16) != 0xffff) {  // an edge of more than eight tets: the rest of its list
    const int s1 = rs_ptr[p + 1];
    for (int s = rs_ptr[p] + 8; s < s1; ++s) f((uint32_t)rs_code[s]);
  }
}

// Shared memory of one warp's four rows.  Mixed: per row the ring's edges
// (high parts, then low parts, 16 bytes each) and a 16-byte record per tet
// (sigma, c1, its three ring slots).
__host__ __device__ inline size_t rows_mixed_smem(int max_val, int max_ring) {
  return 4 * (size_t)(2 * max_ring + max_val) * sizeof(float4);
}

// Mixed path:
//   1. the row's 1-ring: edges e_l (float-float) to shared memory, m_jl e_l
//      into the lane's gradient partial;
//   2. its tets, lane t taking tets t, t + 8, ...: n_0 in float-float,
//      gradient and diagonal-block partials in registers;
//   3. a fixed butterfly over the eight lanes for gradient and diagonal block;
//   4. one lane per upper block walks that block's tets in ascending order and
//      forms n_0 and n_k again in float32 from the ring: re-forming them (18
//      operations) costs no more than staging seven vectors per (row, tet) in
//      step 2, and keeps a row at 0.8 KB of shared memory instead of 2.7 KB
//      (staged: 30.9 us against 24.0 on the 32^3 cube, 16 warps an SM
//      against 24).  Instruction issue bounds it (13.3 M warp instructions);
//      80 registers, 8 bytes a thread spilled.
__global__ void __launch_bounds__(256, 3) k_rows_mixed(
    const int4* __restrict__ hdr, int64_t nrows, const int32_t* __restrict__ nbr_idx,
    const float2* __restrict__ ring_m, const float* __restrict__ row_diag, const int32_t* __restrict__ vt_tet,
    const uint32_t* __restrict__ loc, const float4* __restrict__ rec, const uint4* __restrict__ codes8,
    const int32_t* __restrict__ rs_ptr, const uint16_t* __restrict__ rs_code, const float4* __restrict__ x_hi,
    const float4* __restrict__ x_lo, float scale, float inv_scale, const float2* __restrict__ mass_df,
    const float4* __restrict__ xt_hi, const float4* __restrict__ xt_lo, bool dynamic, int max_val, int max_ring,
    float* __restrict__ bsr, float* __restrict__ g_hi, float* __restrict__ g_lo, float4* __restrict__ diag_g) {
  pdl_entry();
  extern __shared__ __align__(16) float4 rows_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane >> 3, t = lane & 7;
  const int64_t row0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * 4;
  if (row0 >= nrows) return;  // whole warps leave together
  const int64_t row = row0 + sub;
  const bool live = row < nrows;
  const int per_row = 2 * max_ring + max_val;
  float4* eh = rows_smem + (4 * warp + sub) * per_row;
  float4* el = eh + max_ring;
  float4* tr = el + max_ring;
  int4 h0 = make_int4(0, 0, 0, 0), h1 = make_int4(0, 0, 0, 0);
  if (live) {
    h0 = __ldg(hdr + 2 * row);
    h1 = __ldg(hdr + 2 * row + 1);
  }
  const int j = h0.x, p0 = h0.y, nup = h0.z, r0 = h0.w, nring = h1.x, e0 = h1.y, val = h1.z, q0 = h1.w;

  // what depends on the row's record alone is loaded first
  constexpr int kPre = 3;
  int tt[kPre];
  uint32_t lc[kPre];
#pragma unroll
  for (int u = 0; u < kPre; ++u)
    if (t + 8 * u < val) {
      tt[u] = vt_tet[e0 + t + 8 * u];
      lc[u] = loc[e0 + t + 8 * u];
    }
  df gd[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
  {
    const float4 jh = x_hi[j], jl = x_lo[j];
    for (int s = t; s < nring; s += 8) {
      const int l = nbr_idx[r0 + s];
      const float2 m = ring_m[r0 + s];
      const float4 lh = x_hi[l], ll = x_lo[l];
      const df e[3] = {df_scaled_diff(lh.x, ll.x, jh.x, jl.x, scale), df_scaled_diff(lh.y, ll.y, jh.y, jl.y, scale),
                       df_scaled_diff(lh.z, ll.z, jh.z, jl.z, scale)};
      eh[s] = make_float4(e[0].hi, e[1].hi, e[2].hi, 0.f);
      el[s] = make_float4(e[0].lo, e[1].lo, e[2].lo, 0.f);
#pragma unroll
      for (int a = 0; a < 3; ++a) gd[a] = df_fma(df{m.x, m.y}, e[a], gd[a]);
    }
  }
  float4 rc[kPre];
#pragma unroll
  for (int u = 0; u < kPre; ++u)
    if (t + 8 * u < val) rc[u] = rec[tt[u]];
  uint4 cd = make_uint4(0, 0, 0, 0);
  float mq = 0.f;
  if (t < nup) {
    if (t > 0) {
      cd = codes8[p0 + t];
      mq = ring_m[r0 + (nring - nup) + t].x;
    } else {
      mq = row_diag[row];
    }
  }
  __syncwarp();

  float dg[6] = {0, 0, 0, 0, 0, 0};  // sum of c1 n_0 n_0^T, upper triangle
  auto tet = [&](int k, uint32_t l3, float4 r) {
    const int s1 = l3 & 255, s2 = (l3 >> 8) & 255, s3 = (l3 >> 16) & 255;
    const float4 a1 = eh[s1], b1 = el[s1], a2 = eh[s2], b2 = el[s2], a3 = eh[s3], b3 = el[s3];
    const df p[3] = {df_sub(df{a2.x, b2.x}, df{a1.x, b1.x}), df_sub(df{a2.y, b2.y}, df{a1.y, b1.y}),
                     df_sub(df{a2.z, b2.z}, df{a1.z, b1.z})};
    const df q[3] = {df_sub(df{a1.x, b1.x}, df{a3.x, b3.x}), df_sub(df{a1.y, b1.y}, df{a3.y, b3.y}),
                     df_sub(df{a1.z, b1.z}, df{a3.z, b3.z})};
    df n0[3];
    cross_df(p, q, n0);  // (e2 - e1) x (e1 - e3) = -(n1 + n2 + n3)
#pragma unroll
    for (int c = 0; c < 3; ++c) gd[c] = df_fma(df{r.x, r.y}, n0[c], gd[c]);
    const float w0 = r.z * n0[0].hi, w1 = r.z * n0[1].hi, w2 = r.z * n0[2].hi;
    dg[0] = fmaf(w0, n0[0].hi, dg[0]);
    dg[1] = fmaf(w0, n0[1].hi, dg[1]);
    dg[2] = fmaf(w0, n0[2].hi, dg[2]);
    dg[3] = fmaf(w1, n0[1].hi, dg[3]);
    dg[4] = fmaf(w1, n0[2].hi, dg[4]);
    dg[5] = fmaf(w2, n0[2].hi, dg[5]);
    // ring slots as bytes (1, 2, 3, 1): corner k's successors are bytes k mod 3 and k mod 3 + 1
    tr[k] = make_float4(r.x, r.z, __uint_as_float((l3 & 0xffffff) | (l3 << 24)), 0.f);
  };
#pragma unroll
  for (int u = 0; u < kPre; ++u)
    if (t + 8 * u < val) tet(t + 8 * u, lc[u], rc[u]);
  for (int k = t + 8 * kPre; k < val; k += 8) tet(k, loc[e0 + k], rec[vt_tet[e0 + k]]);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
#pragma unroll
    for (int c = 0; c < 6; ++c) dg[c] += __shfl_xor_sync(0xffffffffu, dg[c], o);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const df other{__shfl_xor_sync(0xffffffffu, gd[c].hi, o), __shfl_xor_sync(0xffffffffu, gd[c].lo, o)};
      gd[c] = df_add(gd[c], other);
    }
  }
  __syncwarp();
  if (!live) return;
  if (t < 3) {  // component t of the gradient
    df g = t == 0 ? gd[0] : t == 1 ? gd[1] : gd[2];
    g = df{g.hi * inv_scale, g.lo * inv_scale};
    if (dynamic) {
      const float xh = reinterpret_cast<const float*>(x_hi + j)[t], xl = reinterpret_cast<const float*>(x_lo + j)[t];
      const float th = reinterpret_cast<const float*>(xt_hi + j)[t];
      const float tl = reinterpret_cast<const float*>(xt_lo + j)[t];
      g = df_fma(df{mass_df[j].x, mass_df[j].y}, df_sub(df{xh, xl}, df{th, tl}), g);
    }
    g_hi[3 * (int64_t)j + t] = g.hi;
    g_lo[3 * (int64_t)j + t] = g.lo;
  }
  for (int q = t; q < nup; q += 8) {
    float4* dst = reinterpret_cast<float4*>(bsr) + block_row_at<float>(q0, nup, q, 0) / 4;
    if (q == 0) {
      dst[0] = make_float4(dg[0] + mq, dg[1], dg[2], 0.f);
      dst[nup] = make_float4(dg[1], dg[3] + mq, dg[4], 0.f);
      dst[2 * nup] = make_float4(dg[2], dg[4], dg[5] + mq, 0.f);
      if (!dynamic) {
        float4* own = diag_g + 3 * (int64_t)j;
        own[0] = make_float4(dg[0] + mq, dg[1], dg[2], dg[3] + mq);
        own[1] = make_float4(dg[4], dg[5] + mq, gd[0].hi * inv_scale, gd[1].hi * inv_scale);
        own[2] = make_float4(gd[2].hi * inv_scale, 0.f, 0.f, 0.f);
      }
      continue;
    }
    if (q >= 8) {
      cd = codes8[p0 + q];
      mq = ring_m[r0 + (nring - nup) + q].x;
    }
    const float4 e = eh[(nring - nup) + q];
    float H[9] = {mq, 0.f, 0.f, 0.f, mq, 0.f, 0.f, 0.f, mq}, y0 = 0.f, y1 = 0.f, y2 = 0.f;
    for_sources(cd, p0 + q, rs_ptr, rs_code, [&](uint32_t code) {
      const float4 r = tr[code >> 2];
      const uint32_t sl = __float_as_uint(r.z) >> (8 * (code & 3));
      const float4 a = eh[sl & 255], b = eh[(sl >> 8) & 255];
      // n_k = a x b, n_0 = (a - e) x (e - b), y = sigma (b - a)
      const float nk[3] = {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
      const float u0 = a.x - e.x, u1 = a.y - e.y, u2 = a.z - e.z, v0 = e.x - b.x, v1 = e.y - b.y, v2 = e.z - b.z;
      const float n0[3] = {r.y * (u1 * v2 - u2 * v1), r.y * (u2 * v0 - u0 * v2), r.y * (u0 * v1 - u1 * v0)};
      y0 = fmaf(r.x, b.x - a.x, y0);
      y1 = fmaf(r.x, b.y - a.y, y1);
      y2 = fmaf(r.x, b.z - a.z, y2);
#pragma unroll
      for (int rr = 0; rr < 3; ++rr)
#pragma unroll
        for (int c = 0; c < 3; ++c) H[3 * rr + c] = fmaf(n0[rr], nk[c], H[3 * rr + c]);
    });
    dst[0] = make_float4(H[0], H[1] + y2, H[2] - y1, 0.f);
    dst[nup] = make_float4(H[3] - y2, H[4], H[5] + y0, 0.f);
    dst[2 * nup] = make_float4(H[6] + y1, H[7] - y0, H[8], 0.f);
  }
}

// Float64 path: the float64 pipe bounds it, so every vector is formed once.
// Per (row, tet) c1 n_0, n_1, n_2, n_3 and y_k = sigma (e_a - e_b) are staged
// (21 values: an odd pitch) for the lanes that sum the blocks; sigma is formed
// here (its cross product n_1 is needed anyway), without a per-tet pass.
constexpr int kStage64 = 21;
__host__ __device__ inline size_t rows_f64_smem(int max_val, int max_ring) {
  return 4 * (size_t)(kStage64 * max_val + 3 * max_ring) * sizeof(double);
}

__global__ void __launch_bounds__(256, 2) k_rows_f64(
    const int4* __restrict__ hdr, int64_t nrows, const int32_t* __restrict__ nbr_idx,
    const double* __restrict__ ring_m, const double* __restrict__ row_diag, const int32_t* __restrict__ vt_tet,
    const uint32_t* __restrict__ loc, const double2* __restrict__ tc, const uint4* __restrict__ codes8,
    const int32_t* __restrict__ rs_ptr, const uint16_t* __restrict__ rs_code, const double* __restrict__ x, int64_t n,
    const double* __restrict__ mass, const double* __restrict__ xt, bool dynamic, int max_val, int max_ring,
    double* __restrict__ bsr, double* __restrict__ g) {
  pdl_entry();
  extern __shared__ __align__(16) double rows_smem64[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane >> 3, t = lane & 7;
  const int64_t row0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * 4;
  if (row0 >= nrows) return;  // whole warps leave together
  const int64_t row = row0 + sub;
  const bool live = row < nrows;
  double* ring = rows_smem64 + (size_t)(4 * warp + sub) * (kStage64 * max_val + 3 * max_ring);
  double* stage = ring + 3 * max_ring;
  int4 h0 = make_int4(0, 0, 0, 0), h1 = make_int4(0, 0, 0, 0);
  if (live) {
    h0 = __ldg(hdr + 2 * row);
    h1 = __ldg(hdr + 2 * row + 1);
  }
  const int j = h0.x, p0 = h0.y, nup = h0.z, r0 = h0.w, nring = h1.x, e0 = h1.y, val = h1.z, q0 = h1.w;
  double gs[3] = {0.0, 0.0, 0.0};
  const double xj[3] = {x[j], x[n + j], x[2 * n + j]};
  for (int s = t; s < nring; s += 8) {
    const int l = nbr_idx[r0 + s];
    const double m = ring_m[r0 + s];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double e = x[a * n + l] - xj[a];
      ring[3 * s + a] = e;
      gs[a] = fma(m, e, gs[a]);
    }
  }
  __syncwarp();
  double dg[6] = {0, 0, 0, 0, 0, 0};  // sum of c1 n_0 n_0^T, upper triangle
  for (int k = t; k < val; k += 8) {
    const double2 c = tc[vt_tet[e0 + k]];
    const uint32_t l3 = loc[e0 + k];
    const double* e1 = ring + 3 * (l3 & 255);
    const double* e2 = ring + 3 * ((l3 >> 8) & 255);
    const double* e3 = ring + 3 * ((l3 >> 16) & 255);
    double n1[3], n2[3], n3[3], n0[3];
    cross3(e2, e3, n1);
    cross3(e3, e1, n2);
    cross3(e1, e2, n3);
    const double sg = fma(e1[0] * n1[0] + e1[1] * n1[1] + e1[2] * n1[2], c.x, c.y);
    double* st = stage + kStage64 * k;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      n0[a] = -((n1[a] + n2[a]) + n3[a]);
      gs[a] = fma(sg, n0[a], gs[a]);
      st[a] = c.x * n0[a];
      st[3 + a] = n3[a];  // by k mod 3: 0 -> corner 3
      st[6 + a] = n1[a];
      st[9 + a] = n2[a];
      st[12 + a] = sg * (e2[a] - e1[a]);
      st[15 + a] = sg * (e3[a] - e2[a]);
      st[18 + a] = sg * (e1[a] - e3[a]);
    }
    dg[0] = fma(st[0], n0[0], dg[0]);
    dg[1] = fma(st[0], n0[1], dg[1]);
    dg[2] = fma(st[0], n0[2], dg[2]);
    dg[3] = fma(st[1], n0[1], dg[3]);
    dg[4] = fma(st[1], n0[2], dg[4]);
    dg[5] = fma(st[2], n0[2], dg[5]);
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
#pragma unroll
    for (int c = 0; c < 6; ++c) dg[c] += __shfl_xor_sync(0xffffffffu, dg[c], o);
#pragma unroll
    for (int c = 0; c < 3; ++c) gs[c] += __shfl_xor_sync(0xffffffffu, gs[c], o);
  }
  __syncwarp();
  if (!live) return;
  if (t < 3) {  // component t of the gradient
    double v = t == 0 ? gs[0] : t == 1 ? gs[1] : gs[2];
    if (dynamic) v += mass[j] * (x[t * n + j] - xt[t * n + j]);
    g[3 * (int64_t)j + t] = v;
  }
  for (int q = t; q < nup; q += 8) {
    double2* dst = reinterpret_cast<double2*>(bsr + (int64_t)(q0 + q) * 12);
    if (q == 0) {
      const double d = row_diag[row];
      dst[0] = make_double2(dg[0] + d, dg[1]);
      dst[1] = make_double2(dg[2], 0.0);
      dst[2] = make_double2(dg[1], dg[3] + d);
      dst[3] = make_double2(dg[4], 0.0);
      dst[4] = make_double2(dg[2], dg[4]);
      dst[5] = make_double2(dg[5] + d, 0.0);
      continue;
    }
    const double m = ring_m[r0 + (nring - nup) + q];
    double H[9] = {m, 0, 0, 0, m, 0, 0, 0, m}, y[3] = {0, 0, 0};
    for_sources(codes8[p0 + q], p0 + q, rs_ptr, rs_code, [&](uint32_t code) {
      const double* st = stage + kStage64 * (code >> 2);
      const double* nk = st + 3 + 3 * (code & 3);
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        y[r] += nk[9 + r];
#pragma unroll
        for (int c = 0; c < 3; ++c) H[3 * r + c] = fma(st[r], nk[c], H[3 * r + c]);
      }
    });
    dst[0] = make_double2(H[0], H[1] + y[2]);
    dst[1] = make_double2(H[2] - y[1], 0.0);
    dst[2] = make_double2(H[3] - y[2], H[4]);
    dst[3] = make_double2(H[5] + y[0], 0.0);
    dst[4] = make_double2(H[6] + y[1], H[7] - y[0]);
    dst[5] = make_double2(H[8], 0.0);
  }
}

// ---- set-up ------------------------------------------------------------------
// The other corners of a tet, in the order that keeps its orientation with
// corner c first: (c; 1 2 3), (1; 0 3 2), (2; 3 0 1), (3; 2 1 0).
__device__ __forceinline__ int3 other_corners(int c) {
  return c == 0 ? make_int3(1, 2, 3) : c == 1 ? make_int3(0, 3, 2) : c == 2 ? make_int3(3, 0, 1) : make_int3(2, 1, 0);
}

__device__ __forceinline__ int ring_slot(const int32_t* __restrict__ a, int m, int key) {
  int lo = 0, hi = m - 1;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] < key) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ int corner_id(const int4& v, int c) { return c == 0 ? v.x : c == 1 ? v.y : c == 2 ? v.z : v.w; }

// Ring slots of the other corners of every (vertex, tet) entry; one warp per vertex.
__global__ void k_row_locs(int64_t n, const int32_t* __restrict__ vt_ptr, const int32_t* __restrict__ vt_tet,
                           const uint8_t* __restrict__ vt_corner, const int4* __restrict__ tets,
                           const int32_t* __restrict__ nbr_ptr, const int32_t* __restrict__ nbr_idx,
                           uint32_t* __restrict__ loc) {
  const int64_t j = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (j >= n) return;
  const int32_t* nb = nbr_idx + nbr_ptr[j];
  const int m = nbr_ptr[j + 1] - nbr_ptr[j];
  for (int e = vt_ptr[j] + (threadIdx.x & 31); e < vt_ptr[j + 1]; e += 32) {
    const int4 v = tets[vt_tet[e]];
    const int3 o = other_corners(vt_corner[e]);
    loc[e] = (uint32_t)ring_slot(nb, m, corner_id(v, o.x)) | ((uint32_t)ring_slot(nb, m, corner_id(v, o.y)) << 8) |
             ((uint32_t)ring_slot(nb, m, corner_id(v, o.z)) << 16);
  }
}

// m_jl of every ring entry (ascending tets, float64); one warp per vertex.
__global__ void k_ring_weights(int64_t n, const int32_t* __restrict__ vt_ptr, const int32_t* __restrict__ vt_tet,
                               const uint8_t* __restrict__ vt_corner, const int4* __restrict__ tets,
                               const int32_t* __restrict__ nbr_ptr, const int32_t* __restrict__ nbr_idx,
                               const double* __restrict__ Bm, const double* __restrict__ volw,
                               const double2* __restrict__ mat, double* __restrict__ m64,
                               float2* __restrict__ mdf) {
  const int64_t j = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (j >= n) return;
  for (int p = nbr_ptr[j] + (threadIdx.x & 31); p < nbr_ptr[j + 1]; p += 32) {
    const int l = nbr_idx[p];
    double acc = 0.0;
    for (int e = vt_ptr[j]; e < vt_ptr[j + 1]; ++e) {
      const int t = vt_tet[e], cj = vt_corner[e];
      const int4 v = tets[t];
      const int cl = v.x == l ? 0 : v.y == l ? 1 : v.z == l ? 2 : v.w == l ? 3 : -1;
      if (cl < 0) continue;
      const double* B = Bm + 9 * (int64_t)t;
      double gj[3], gl[3];
      for (int a = 0; a < 3; ++a) {
        const double s = -(B[a] + B[3 + a] + B[6 + a]);
        gj[a] = cj == 0 ? s : B[3 * (cj - 1) + a];
        gl[a] = cl == 0 ? s : B[3 * (cl - 1) + a];
      }
      acc += volw[t] * mat[t].x * (gj[0] * gl[0] + gj[1] * gl[1] + gj[2] * gl[2]);
    }
    m64[p] = acc;
    const df d = df_from_double(acc);
    mdf[p] = make_float2(d.hi, d.lo);
  }
}

// Diagonal constants of the free rows: -sum_l m_jl (+ mass when dynamic).
__global__ void k_row_diag(const int32_t* __restrict__ rows, int64_t nrows, const int32_t* __restrict__ nbr_ptr,
                           const double* __restrict__ m64, const double* __restrict__ mass, bool dynamic,
                           double* __restrict__ d64, float* __restrict__ d32) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= nrows) return;
  const int j = rows[k];
  double s = 0.0;
  for (int p = nbr_ptr[j]; p < nbr_ptr[j + 1]; ++p) s += m64[p];
  const double d = (dynamic ? mass[j] : 0.0) - s;
  d64[k] = d;
  d32[k] = (float)d;
}

// Source codes of every off-diagonal upper block of the free rows (ascending
// tets, as for_sources reads them).  The first eight go to codes8 (padded with 0xffff), all of them to rs_code.
__global__ void k_row_codes(const int32_t* __restrict__ rows, int64_t nrows, const int32_t* __restrict__ up_ptr,
                            const int32_t* __restrict__ up_col, const int32_t* __restrict__ vt_ptr,
                            const int32_t* __restrict__ vt_tet, const uint8_t* __restrict__ vt_corner,
                            const int4* __restrict__ tets, const int32_t* __restrict__ rs_ptr,
                            uint16_t* __restrict__ codes8, uint16_t* __restrict__ rs_code) {
  const int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (k >= nrows) return;
  const int j = rows[k];
  for (int p = up_ptr[j] + 1 + (threadIdx.x & 31); p < up_ptr[j + 1]; p += 32) {
    const int l = up_col[p];
    int s = 0;
    for (int e = vt_ptr[j]; e < vt_ptr[j + 1]; ++e) {
      const int4 v = tets[vt_tet[e]];
      const int3 o = other_corners(vt_corner[e]);
      const int w = corner_id(v, o.x) == l ? 1 : corner_id(v, o.y) == l ? 2 : corner_id(v, o.z) == l ? 0 : -1;
      if (w < 0) continue;
      const uint16_t code = (uint16_t)(((e - vt_ptr[j]) << 2) | w);
      if (s < 8) codes8[8 * (int64_t)p + s] = code;
      rs_code[rs_ptr[p] + s] = code;
      ++s;
    }
  }
}

// Warps per CTA: the tuned number, fewer where their rows' shared memory is large.
int rows_wpb(const Mesh& m, size_t per_warp) {
  int wpb = m.tune_gather_wpb > 0 ? m.tune_gather_wpb : 4;
  while (wpb > 1 && wpb * per_warp > kRowsSmemMax) wpb >>= 1;
  return wpb;
}

}  // namespace

void launch_tet_sigma(Mesh& m, const int32_t* list, int64_t count, cudaStream_t s) {
  if (count <= 0) return;
  pdl_launch(k_tet_sigma, (unsigned)((count + 127) / 128), 128, 0, s, (const int4*)m.d_tets.p, (const float4*)m.d_tcdf.p,
             (const float4*)m.mx.x_hi.p, (const float4*)m.mx.x_lo.p, list, count, m.len_scale, m.mx.rec.p);
}

void launch_rows_from_positions(Mesh& m, bool mixed, const double* x, const double* xt, cudaStream_t s) {
  if (m.n_free <= 0) return;
  const bool dyn = m.h > 0.0;
  const size_t per = mixed ? rows_mixed_smem(m.max_valence, m.max_ring) : rows_f64_smem(m.max_valence, m.max_ring);
  const int wpb = rows_wpb(m, per);
  const unsigned grid = (unsigned)((m.n_free + 4 * wpb - 1) / (4 * wpb));
  if (mixed) {
    set_smem_limit(reinterpret_cast<const void*>(k_rows_mixed), wpb * per);
    pdl_launch(k_rows_mixed, grid, 32 * wpb, wpb * per, s, (const int4*)m.d_row_hdr2.p, m.n_free,
               (const int32_t*)m.d_nbr_idx.p, (const float2*)m.d_ring_mdf.p, (const float*)m.d_row_diag32.p,
               (const int32_t*)m.d_vt_tet.p, (const uint32_t*)m.d_loc.p, (const float4*)m.mx.rec.p,
               (const uint4*)m.d_codes8.p, (const int32_t*)m.d_rs_ptr.p, (const uint16_t*)m.d_rs_code.p,
               (const float4*)m.mx.x_hi.p, (const float4*)m.mx.x_lo.p, m.len_scale, 1.0f / m.len_scale,
               (const float2*)m.d_mass_df.p, (const float4*)m.mx.xt_hi.p, (const float4*)m.mx.xt_lo.p, dyn,
               (int)m.max_valence, (int)m.max_ring, m.mx.bsr.p, m.mx.g_hi.p, m.mx.g_lo.p, m.mx.diag_g.p);
  } else {
    set_smem_limit(reinterpret_cast<const void*>(k_rows_f64), wpb * per);
    pdl_launch(k_rows_f64, grid, 32 * wpb, wpb * per, s, (const int4*)m.d_row_hdr2.p, m.n_free,
               (const int32_t*)m.d_nbr_idx.p, (const double*)m.d_ring_m64.p, (const double*)m.d_row_diag64.p,
               (const int32_t*)m.d_vt_tet.p, (const uint32_t*)m.d_loc.p, (const double2*)m.d_tc64.p,
               (const uint4*)m.d_codes8.p, (const int32_t*)m.d_rs_ptr.p, (const uint16_t*)m.d_rs_code.p, x, m.n,
               (const double*)m.d_mass.p, dyn ? xt : nullptr, dyn, (int)m.max_valence, (int)m.max_ring, m.f64.bsr.p,
               m.f64.g.p);
  }
}

// Rest data of the rows formed from the positions (stable Neo-Hookean), built
// on the device from the uploaded topology.  Sets rows_ok: the ring slots fit
// a byte and one warp's four rows fit the shared memory in both precisions.
void build_row_data(Mesh& m, const std::vector<double>& volw) {
  m.rows_ok = m.rows64_fast = false;
  if (m.model != CC_MODEL_SNH) return;
  m.max_ring = 0;
  for (int64_t v = 0; v < m.n; ++v)
    m.max_ring = std::max<int32_t>(m.max_ring, (int32_t)(m.nbr_ptr[v + 1] - m.nbr_ptr[v]));
  if (m.max_ring > 255 || rows_f64_smem(m.max_valence, m.max_ring) > kRowsSmemMax ||
      rows_mixed_smem(m.max_valence, m.max_ring) > kRowsSmemMax)
    return;
  cudaStream_t s = m.stream;
  const int64_t n = m.n, T = m.T, nr = m.n_free;
  const double w = m.h > 0.0 ? m.h * m.h : 1.0;
  double vsum = 0.0;
  for (int64_t t = 0; t < T; ++t) vsum += volw[t];
  // lengths in units of about one mean edge: 6 V' = (2^k)^3 6 V near 1
  const int k = -(int)std::lround(std::log2(6.0 * vsum / w / (double)T) / 3.0);
  m.len_scale = (float)std::ldexp(1.0, std::max(-100, std::min(100, k)));
  const double sc = m.len_scale;
  std::vector<double2> tc(T);
  std::vector<float4> tcdf(T);
  for (int64_t t = 0; t < T; ++t) {
    const double D = 6.0 * (volw[t] / w), lh = m.tet_lh[t], mu = m.tet_mu[t];
    const double c1 = w * lh / (6.0 * D), c0 = -w * (lh + mu) / 6.0;
    tc[t] = make_double2(c1, c0);
    // scaled lengths: sigma' = sigma / sc and c1' = c1 / sc^4 (n' = sc^2 n, e' = sc e)
    const double a = c1 / (sc * sc * sc * sc), b = c0 / sc;
    const float ah = (float)a, bh = (float)b;
    tcdf[t] = make_float4(ah, (float)(a - (double)ah), bh, (float)(b - (double)bh));
  }
  m.d_tc64.upload(tc, s);
  m.d_tcdf.upload(tcdf, s);
  std::vector<int32_t> hdr;
  hdr.reserve(8 * nr);
  for (int64_t v = 0; v < n; ++v) {
    if (m.pinned[v]) continue;
    const int32_t p0 = (int32_t)m.up_ptr[v], r0 = (int32_t)m.nbr_ptr[v], e0 = (int32_t)m.vt_ptr[v];
    const int32_t h[8] = {(int32_t)v, p0, (int32_t)m.up_ptr[v + 1] - p0, r0, (int32_t)m.nbr_ptr[v + 1] - r0, e0,
                          (int32_t)m.vt_ptr[v + 1] - e0, p0};
    hdr.insert(hdr.end(), h, h + 8);
  }
  m.d_row_hdr2.upload(reinterpret_cast<const int4*>(hdr.data()), 2 * nr, s);
  m.d_loc.alloc(4 * T);
  m.d_ring_m64.alloc(m.nbr_idx.size());
  m.d_ring_mdf.alloc(m.nbr_idx.size());
  m.d_row_diag64.alloc(nr);
  m.d_row_diag32.alloc(nr);
  m.d_codes8.alloc(m.nnz_up);
  m.d_rs_code.alloc(m.d_rs_src.count);
  CCG_CUDA(cudaMemsetAsync(m.d_codes8.p, 0xff, m.nnz_up * sizeof(uint4), s));
  const unsigned gn = (unsigned)((n * 32 + 255) / 256), gr = (unsigned)((nr * 32 + 255) / 256);
  k_row_locs<<<gn, 256, 0, s>>>(n, m.d_vt_ptr.p, m.d_vt_tet.p, m.d_vt_corner.p, m.d_tets.p, m.d_nbr_ptr.p,
                                m.d_nbr_idx.p, m.d_loc.p);
  k_ring_weights<<<gn, 256, 0, s>>>(n, m.d_vt_ptr.p, m.d_vt_tet.p, m.d_vt_corner.p, m.d_tets.p, m.d_nbr_ptr.p,
                                    m.d_nbr_idx.p, m.d_Bm.p, m.d_volw.p, m.d_mat64.p, m.d_ring_m64.p, m.d_ring_mdf.p);
  if (nr > 0) {
    k_row_diag<<<(unsigned)((nr + 255) / 256), 256, 0, s>>>(m.d_free_rows.p, nr, m.d_nbr_ptr.p, m.d_ring_m64.p,
                                                            m.d_mass.p, m.h > 0.0, m.d_row_diag64.p, m.d_row_diag32.p);
    k_row_codes<<<gr, 256, 0, s>>>(m.d_free_rows.p, nr, m.d_up_ptr.p, m.d_up_col.p, m.d_vt_ptr.p, m.d_vt_tet.p,
                                   m.d_vt_corner.p, m.d_tets.p, m.d_rs_ptr.p,
                                   reinterpret_cast<uint16_t*>(m.d_codes8.p), m.d_rs_code.p);
  }
  CCG_CUDA(cudaGetLastError());
  CCG_CUDA(cudaStreamSynchronize(s));  // host vectors above go out of scope
  m.rows_ok = true;
  m.rows64_fast = rows_f64_smem(m.max_valence, m.max_ring) <= kRows64FastSmem;
}

}  // namespace ccg
