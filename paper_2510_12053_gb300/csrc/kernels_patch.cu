// Patch solves (Eq. 5 on P = S_i) in float32 with float64 iterative refinement,
// one CTA per free vertex, for patches of at most kPmMaxN = 192 unknowns (every
// 2-ring of a Kuhn grid).
//
// H_PP is assembled in float32 into shared memory and factored by Cholesky
// there; U = -H_PP^{-1} H_Pi is then reached by iterative refinement,
// z += L^{-T} L^{-1} (B - H_PP z), B = -H_Pi, with the residual in float64 from
// the float64 block rows, until the correction is below 1e-12 of z or stops
// shrinking (it then sits at the rounding level of the float64 residual).  A
// patch whose float32 factorization meets a non-positive pivot, or whose last
// correction is above 1e-11 of z, is queued for the float64 kernel (which also
// decides positive definiteness).
//
// The factor lives in 16 x 16 tiles (lower block triangle, 78 KB at 192, two
// CTAs per SM).  Per block column: one warp factors the diagonal tile in
// registers and replaces it by its inverse, a thread per row multiplies the
// panel by that inverse, and the warps update the trailing tiles with 4 x 4
// outputs per lane; warp 0 updates and factors the next diagonal tile first, so
// its serial chain runs beside the other warps' tiles.  The triangular solves
// use the inverted diagonal tiles: two barriers per 16 unknowns.  The residual
// takes a thread per (row block, right-hand side) over a list of the row's
// blocks inside the patch, found once.
// What bounds it: the float64 residual (an interior 2-ring of a Kuhn grid lists
// 644 blocks: 1 932 products with one right-hand side, 17 400 fused operations
// an iteration) and the shared-memory reads of the tile updates together.
// A column-by-column factorisation in packed storage (two barriers and one
// rank-one update per unknown), one thread per row in the residual with its
// neighbours searched again in every iteration, made a solve of the 16^3 cube
// with four sweeps and one rebuild of its 4 335 bases take 13.3 ms; now 2.5 ms.
#include "cc_internal.cuh"

namespace ccg {

namespace {

constexpr int kPmMaxIt = 4;
constexpr int kPmThreads = 256;
constexpr int kPmWarps = kPmThreads / 32;
constexpr int kPmTiles = kPmMaxN / 16;
constexpr int kPmTileFloats = 256 * kPmTiles * (kPmTiles + 1) / 2;
constexpr int kPmMaxBlocks = 1280;  // listed blocks of a patch (an interior 2-ring of a Kuhn grid: 644)
static_assert(kPmMaxN % 16 == 0 && kPmMaxN <= kPmThreads && kPmMaxN / 3 <= 255, "patch kernel sizes");

struct PatchSmem {
  float L[kPmTileFloats];
  double B[3 * kPmMaxN], Z[3 * kPmMaxN];
  float D[3 * kPmMaxN], X[3 * kPmMaxN];
  int32_t blk[kPmMaxBlocks];   // block number of a listed block, bit 31: transposed
  int32_t S[kPmMaxN / 3], first[kPmMaxN / 3 + 1];
  double dmax, zmax;
  int bad;
  uint8_t col[kPmMaxBlocks];   // its column's slot in the support
};

__device__ __forceinline__ int find_in(const int32_t* a, int m, int key) {
  int lo = 0, hi = m - 1;
  while (lo <= hi) {
    const int mid = (lo + hi) >> 1, x = a[mid];
    if (x == key) return mid;
    if (x < key) lo = mid + 1;
    else hi = mid - 1;
  }
  return -1;
}

// Tiles are row-major; a row's four 16-byte chunks are permuted by its number,
// so that eight rows' equal chunks lie in distinct banks.
__device__ __forceinline__ int tile_at(int I, int J) { return (((I * (I + 1)) >> 1) + J) << 8; }
__device__ __forceinline__ int chunk_at(int r, int ch) { return r * 16 + ((ch ^ ((r >> 1) & 3)) << 2); }
__device__ __forceinline__ int elem_at(int r, int c) {
  return tile_at(r >> 4, c >> 4) + chunk_at(r & 15, (c >> 2) & 3) + (c & 3);
}

// Cholesky factor of the diagonal tile t and its inverse, by one warp (lanes
// 16..31 repeat lanes 0..15); the inverse (zero above the diagonal) replaces it.
__device__ void factor_diag(float* t, int* bad) {
  const int lane = threadIdx.x & 31, r = lane & 15;
  float a[16];
#pragma unroll
  for (int ch = 0; ch < 4; ++ch) {
    const float4 v = *reinterpret_cast<const float4*>(t + chunk_at(r, ch));
    a[4 * ch] = v.x; a[4 * ch + 1] = v.y; a[4 * ch + 2] = v.z; a[4 * ch + 3] = v.w;
  }
  float inv[16];  // reciprocal pivots
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    const float d = __shfl_sync(0xffffffffu, a[c], c);
    if (lane == 0 && !(d > 0.0f)) *bad = 1;
    const float piv = sqrtf(fmaxf(d, 1e-30f));
    inv[c] = 1.0f / piv;
    a[c] = r == c ? piv : a[c] * inv[c];
#pragma unroll
    for (int s = c + 1; s < 16; ++s) a[s] = fmaf(-a[c], __shfl_sync(0xffffffffu, a[c], s), a[s]);
  }
  // lane j: column j of the inverse by forward substitution
  float x[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    float acc = q == r ? 1.0f : 0.0f;
#pragma unroll
    for (int k = 0; k < q; ++k) acc = fmaf(-__shfl_sync(0xffffffffu, a[k], q), x[k], acc);
    x[q] = acc * inv[q];
  }
  __syncwarp();
  if (lane < 16) {
#pragma unroll
    for (int q = 0; q < 16; ++q) t[chunk_at(q, r >> 2) + (r & 3)] = x[q];
  }
}

// Tiles (I, J) and (I + 1, J) of the trailing matrix minus P_I P_J^T and
// P_{I+1} P_J^T (panel tiles of block column kb), by one warp; a tile above the
// diagonal or past the last row is left out.
__device__ __forceinline__ void update_pair(float* L, int kb, int I, int J, int nt) {
  const int lane = threadIdx.x & 31, ri = lane >> 2, cj = lane & 3;
  const bool lo = J <= I, hi = I + 1 < nt;
  const float* PI = L + tile_at(I, kb);
  const float* PK = L + tile_at(hi ? I + 1 : I, kb);
  const float* PJ = L + tile_at(J, kb);
  float acc[4][4];
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = 0.0f;
#pragma unroll
  for (int ch = 0; ch < 4; ++ch) {
    float4 a[4], b[4];
    a[0] = *reinterpret_cast<const float4*>(PI + chunk_at(ri, ch));
    a[1] = *reinterpret_cast<const float4*>(PI + chunk_at(ri + 8, ch));
    a[2] = *reinterpret_cast<const float4*>(PK + chunk_at(ri, ch));
    a[3] = *reinterpret_cast<const float4*>(PK + chunk_at(ri + 8, ch));
#pragma unroll
    for (int y = 0; y < 4; ++y) b[y] = *reinterpret_cast<const float4*>(PJ + chunk_at(cj + 4 * y, ch));
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        acc[x][y] = fmaf(a[x].x, b[y].x, acc[x][y]);
        acc[x][y] = fmaf(a[x].y, b[y].y, acc[x][y]);
        acc[x][y] = fmaf(a[x].z, b[y].z, acc[x][y]);
        acc[x][y] = fmaf(a[x].w, b[y].w, acc[x][y]);
      }
  }
  if (lo) {
    float* C = L + tile_at(I, J);
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) C[chunk_at(ri + 8 * x, y) + cj] -= acc[x][y];
  }
  if (hi) {
    float* C = L + tile_at(I + 1, J);
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) C[chunk_at(ri + 8 * x, y) + cj] -= acc[2 + x][y];
  }
}

// The half-warp walks the blocks (S[a], l), l in S or l = i, of row a in
// ascending l: f(t, p, transposed, before) with t the slot of l (m for l = i),
// p the stored block and `before` the row's blocks inside S listed earlier.
// Returns the number of blocks inside S.
template <typename F>
__device__ __forceinline__ int for_row_blocks(int j, int i, int a, const int32_t* S, int m,
                                              const int32_t* __restrict__ up_ptr, const int32_t* __restrict__ nbr_ptr,
                                              const int32_t* __restrict__ nbr_idx, F&& f) {
  const int lane = threadIdx.x & 31, sub = lane & 15, shift = lane & 16;
  const unsigned half = 0xffffu << shift;
  const int r0 = nbr_ptr[j], nring = nbr_ptr[j + 1] - r0, u0 = up_ptr[j], nup = up_ptr[j + 1] - u0;
  const int nlow = nring - (nup - 1);  // ring vertices below j; the others are the row's upper blocks in order
  int count = 0;
  // position 0..nlow-1: lower neighbours, nlow: j itself, then the upper ones
  for (int e0 = 0; e0 <= nring; e0 += 16) {
    const int e = e0 + sub;
    int t = -1, l = 0;
    if (e <= nring) {
      l = e < nlow ? nbr_idx[r0 + e] : e == nlow ? j : nbr_idx[r0 + e - 1];
      t = l == j ? a : l == i ? m : find_in(S, m, l);
    }
    const unsigned in = (__ballot_sync(half, t >= 0 && t < m) >> shift) & 0xffffu;
    if (t >= 0) f(t, l, e < nlow ? -1 : u0 + (e - nlow), count + __popc(in & ((1u << sub) - 1u)));
    count += __popc(in);
  }
  return count;
}

__global__ void __launch_bounds__(kPmThreads, 2) k_patch_basis_mixed(
    const int32_t* __restrict__ verts, const int32_t* __restrict__ sup_ptr, const int32_t* __restrict__ sup_idx,
    const int32_t* __restrict__ up_ptr, const int32_t* __restrict__ up_col, const int32_t* __restrict__ nbr_ptr,
    const int32_t* __restrict__ nbr_idx, const double* __restrict__ bsr, double* __restrict__ Uout,
    int32_t* __restrict__ redo, int32_t* __restrict__ n_redo) {
  extern __shared__ __align__(16) unsigned char pm_smem[];
  PatchSmem& sm = *reinterpret_cast<PatchSmem*>(pm_smem);
  float* L = sm.L;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i = verts[blockIdx.x];
  const int s0 = sup_ptr[i], m = sup_ptr[i + 1] - s0;
  if (m == 0) return;  // the whole CTA leaves
  const int N = 3 * m, nt = (N + 15) >> 4;
  {
    float4* z = reinterpret_cast<float4*>(L);
    for (int k = tid; k < 64 * ((nt * (nt + 1)) >> 1); k += kPmThreads) z[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k = tid; k < 3 * kPmMaxN; k += kPmThreads) {
      sm.B[k] = 0.0;
      sm.Z[k] = 0.0;
      sm.D[k] = 0.0f;
    }
    for (int a = tid; a < m; a += kPmThreads) sm.S[a] = sup_idx[s0 + a];
    if (tid == 0) sm.bad = 0;
  }
  __syncthreads();
  // blocks per row, their places, then the list, the float32 lower triangle and B
  for (int a = tid >> 4; a < m; a += kPmThreads / 16) {
    const int c = for_row_blocks(sm.S[a], i, a, sm.S, m, up_ptr, nbr_ptr, nbr_idx, [](int, int, int, int) {});
    if ((tid & 15) == 0) sm.first[a + 1] = c;
  }
  for (int r = N + tid; r < 16 * nt; r += kPmThreads) L[elem_at(r, r)] = 1.0f;  // padding: the identity
  __syncthreads();
  if (warp == 0) {
    int carry = 0;
    for (int a0 = 0; a0 < m; a0 += 32) {
      const int a = a0 + lane;
      int v = a < m ? sm.first[a + 1] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
      }
      __syncwarp();
      if (a < m) sm.first[a + 1] = carry + v;
      carry += __shfl_sync(0xffffffffu, v, 31);
    }
    if (lane == 0) sm.first[0] = 0;
  }
  __syncthreads();
  const bool listed = sm.first[m] <= kPmMaxBlocks;
  // the rows' blocks inside S and with i; lower ones are found in the neighbour's row
  for (int a = tid >> 4; a < m; a += kPmThreads / 16) {
    const int j = sm.S[a], at = sm.first[a];
    for_row_blocks(j, i, a, sm.S, m, up_ptr, nbr_ptr, nbr_idx, [&](int t, int l, int p, int before) {
      const bool lower = p < 0;
      if (lower) {
        const int q0 = up_ptr[l] + 1;
        p = q0 + find_in(up_col + q0, up_ptr[l + 1] - q0, j);
      }
      const double* Hb = bsr + (int64_t)p * 12;  // H_jl (or H_lj when lower), row r at Hb[4 r]
      if (t == m) {                              // B_a = -H_ji
        for (int r = 0; r < 3; ++r)
          for (int d = 0; d < 3; ++d) sm.B[d * kPmMaxN + 3 * a + r] = lower ? -Hb[4 * d + r] : -Hb[4 * r + d];
        return;
      }
      if (listed) {
        sm.blk[at + before] = lower ? (int)((unsigned)p | 0x80000000u) : p;
        sm.col[at + before] = (uint8_t)t;
      }
      if (lower) return;  // the float32 triangle takes every stored block once, below the diagonal
      for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c)
          if (t > a || c <= r) L[t > a ? elem_at(3 * t + c, 3 * a + r) : elem_at(3 * a + r, 3 * a + c)] = (float)Hb[4 * r + c];
    });
  }
  __syncthreads();
  if (warp == 0) factor_diag(L, &sm.bad);
  __syncthreads();
  for (int kb = 0; kb + 1 < nt; ++kb) {
    const int r = 16 * (kb + 1) + tid;
    if (r < 16 * nt) {  // panel: A L_kk^{-T}, a row per thread
      float* P = L + tile_at(r >> 4, kb);
      const float* T = L + tile_at(kb, kb);
      const int rr = r & 15;
      float a[16];
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        const float4 v = *reinterpret_cast<const float4*>(P + chunk_at(rr, ch));
        a[4 * ch] = v.x; a[4 * ch + 1] = v.y; a[4 * ch + 2] = v.z; a[4 * ch + 3] = v.w;
      }
#pragma unroll
      for (int c4 = 3; c4 >= 0; --c4) {
        float o[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float acc = 0.0f;
#pragma unroll
          for (int ch = 0; ch <= c4; ++ch) {
            const float4 v = *reinterpret_cast<const float4*>(T + chunk_at(4 * c4 + c, ch));
            acc = fmaf(a[4 * ch], v.x, acc);
            acc = fmaf(a[4 * ch + 1], v.y, acc);
            acc = fmaf(a[4 * ch + 2], v.z, acc);
            acc = fmaf(a[4 * ch + 3], v.w, acc);
          }
          o[c] = acc;
        }
        *reinterpret_cast<float4*>(P + chunk_at(rr, c4)) = make_float4(o[0], o[1], o[2], o[3]);
      }
    }
    __syncthreads();
    // row pairs (I, I + 1) from kb + 1, columns kb + 1 .. I + 1: pair g has 2 g + 2 units, g (g + 1) before it
    const int n1 = nt - 1 - kb, pairs = (n1 + 1) >> 1, units = pairs * (pairs + 1) - (n1 & 1);
    int g = 0;
    auto unit = [&](int u) {
      while ((g + 1) * (g + 2) <= u) ++g;
      update_pair(L, kb, kb + 1 + 2 * g, kb + 1 + u - g * (g + 1), nt);
    };
    if (warp == 0) {
      unit(0);
      __syncwarp();
      factor_diag(L + tile_at(kb + 1, kb + 1), &sm.bad);
    } else {
      for (int u = warp; u < units; u += kPmWarps - 1) unit(u);
    }
    __syncthreads();
  }
  bool ok = sm.bad == 0;
  // iterative refinement: D = B - H_PP Z (float64, rounded), X = (L L^T)^{-1} D (float32), Z += X
  bool settled = false;
  double prev = 1e300, ratio = 1e300;
  for (int it = 0; ok && it < kPmMaxIt && !settled; ++it) {
    for (int w = tid; w < 3 * m; w += kPmThreads) {  // right-hand side d of row block a
      const int a = w / 3, d = w - 3 * a;
      const double* Zd = sm.Z + d * kPmMaxN;
      double y0 = 0.0, y1 = 0.0, y2 = 0.0;
      auto add = [&](int p, bool tr, int t) {
        const double2* b = reinterpret_cast<const double2*>(bsr + (int64_t)p * 12);
        const double2 h0 = __ldg(b), h0z = __ldg(b + 1), h1 = __ldg(b + 2), h1z = __ldg(b + 3), h2 = __ldg(b + 4),
                      h2z = __ldg(b + 5);
        const double z0 = Zd[3 * t], z1 = Zd[3 * t + 1], z2 = Zd[3 * t + 2];
        y0 = fma(h0.x, z0, y0);
        y1 = fma(h1.y, z1, y1);
        y2 = fma(h2z.x, z2, y2);
        y0 = fma(tr ? h1.x : h0.y, z1, y0);
        y1 = fma(tr ? h0.y : h1.x, z0, y1);
        y2 = fma(tr ? h0z.x : h2.x, z0, y2);
        y0 = fma(tr ? h2.x : h0z.x, z2, y0);
        y1 = fma(tr ? h2.y : h1z.x, z2, y1);
        y2 = fma(tr ? h1z.x : h2.y, z1, y2);
      };
      if (listed) {
        for (int e = sm.first[a]; e < sm.first[a + 1]; ++e)
          add(sm.blk[e] & 0x7fffffff, sm.blk[e] < 0, sm.col[e]);
      } else {  // more blocks than the list holds: find them again
        const int j = sm.S[a];
        for (int e = nbr_ptr[j]; e < nbr_ptr[j + 1]; ++e) {
          const int l = nbr_idx[e];
          if (l >= j) break;
          const int t = l == i ? -1 : find_in(sm.S, m, l);
          if (t < 0) continue;
          const int q0 = up_ptr[l] + 1;
          add(q0 + find_in(up_col + q0, up_ptr[l + 1] - q0, j), true, t);
        }
        for (int p = up_ptr[j]; p < up_ptr[j + 1]; ++p) {
          const int l = up_col[p], t = l == j ? a : l == i ? -1 : find_in(sm.S, m, l);
          if (t >= 0) add(p, false, t);
        }
      }
      sm.D[d * kPmMaxN + 3 * a] = (float)(sm.B[d * kPmMaxN + 3 * a] - y0);
      sm.D[d * kPmMaxN + 3 * a + 1] = (float)(sm.B[d * kPmMaxN + 3 * a + 1] - y1);
      sm.D[d * kPmMaxN + 3 * a + 2] = (float)(sm.B[d * kPmMaxN + 3 * a + 2] - y2);
    }
    if (tid == 0) {
      sm.dmax = 0.0;
      sm.zmax = 0.0;
    }
    __syncthreads();
    // forward: X_b = L_bb^{-1} D_b, then D below minus L(., b) X_b
    for (int b = 0; b < nt; ++b) {
      if (tid < 48) {
        const int d = tid >> 4, r = tid & 15;
        const float* T = L + tile_at(b, b);
        const float* y = sm.D + d * kPmMaxN + 16 * b;
        float acc = 0.0f;
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          const float4 v = *reinterpret_cast<const float4*>(T + chunk_at(r, ch));
          const float4 u = *reinterpret_cast<const float4*>(y + 4 * ch);
          acc = fmaf(v.x, u.x, acc);
          acc = fmaf(v.y, u.y, acc);
          acc = fmaf(v.z, u.z, acc);
          acc = fmaf(v.w, u.w, acc);
        }
        sm.X[d * kPmMaxN + 16 * b + r] = acc;
      }
      __syncthreads();
      const int r = 16 * (b + 1) + tid;
      if (r < 16 * nt) {
        const float* T = L + tile_at(r >> 4, b);
        float acc[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          const float4 v = *reinterpret_cast<const float4*>(T + chunk_at(r & 15, ch));
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const float4 u = *reinterpret_cast<const float4*>(sm.X + d * kPmMaxN + 16 * b + 4 * ch);
            acc[d] = fmaf(v.x, u.x, acc[d]);
            acc[d] = fmaf(v.y, u.y, acc[d]);
            acc[d] = fmaf(v.z, u.z, acc[d]);
            acc[d] = fmaf(v.w, u.w, acc[d]);
          }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) sm.D[d * kPmMaxN + r] -= acc[d];
      }
      __syncthreads();
    }
    // backward, in place of D: D_b = L_bb^{-T} X_b, then X above minus L(b, .)^T D_b
    for (int b = nt - 1; b >= 0; --b) {
      if (tid < 48) {
        const int d = tid >> 4, r = tid & 15;
        const float* T = L + tile_at(b, b);
        const float* x = sm.X + d * kPmMaxN + 16 * b;
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < 16; ++k) acc = fmaf(T[chunk_at(k, r >> 2) + (r & 3)], x[k], acc);
        sm.D[d * kPmMaxN + 16 * b + r] = acc;
      }
      __syncthreads();
      if (tid < 16 * b) {
        const float* T = L + tile_at(b, tid >> 4);
        const int c = tid & 15;
        float acc[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const float v = T[chunk_at(k, c >> 2) + (c & 3)];
#pragma unroll
          for (int d = 0; d < 3; ++d) acc[d] = fmaf(v, sm.D[d * kPmMaxN + 16 * b + k], acc[d]);
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) sm.X[d * kPmMaxN + tid] -= acc[d];
      }
      __syncthreads();
    }
    double dl = 0.0, zl = 0.0;
    bool nonfinite = false;
    for (int k = tid; k < 3 * N; k += kPmThreads) {
      const int q = (k / N) * kPmMaxN + k % N;
      const double d = (double)sm.D[q], z = sm.Z[q] + d;
      sm.Z[q] = z;
      nonfinite |= !isfinite(d) || !isfinite(z);  // fmax below would drop a NaN
      dl = fmax(dl, fabs(d));
      zl = fmax(zl, fabs(z));
    }
    if (nonfinite) sm.bad = 1;  // float32 overflow in the triangular solves: the float64 kernel redoes the patch
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      dl = fmax(dl, __shfl_xor_sync(0xffffffffu, dl, o));
      zl = fmax(zl, __shfl_xor_sync(0xffffffffu, zl, o));
    }
    if (lane == 0) {  // non-negative doubles order as their bits
      atomicMax(reinterpret_cast<unsigned long long*>(&sm.dmax), (unsigned long long)__double_as_longlong(dl));
      atomicMax(reinterpret_cast<unsigned long long*>(&sm.zmax), (unsigned long long)__double_as_longlong(zl));
    }
    __syncthreads();
    const double dm = sm.dmax, zm = sm.zmax;
    ok = sm.bad == 0;
    __syncthreads();
    if (!ok) break;
    settled = dm <= 1e-12 * zm;
    ratio = zm > 0.0 ? dm / zm : 0.0;
    if (dm > 0.5 * prev) break;  // corrections at the float64 rounding level of the residual
    prev = dm;
  }
  // accepted when the last correction is at most 1e-11 of z (the float64
  // solve's own rounding is about cond(H_PP) * 1e-16)
  if (!(ok && (settled || ratio <= 1e-11))) {
    if (tid == 0) redo[atomicAdd(n_redo, 1)] = i;
    return;
  }
  for (int k = tid; k < 9 * m; k += kPmThreads) {
    const int a = k / 9, q = k % 9, r = q / 3, d = q % 3;
    Uout[(int64_t)(s0 + a) * 9 + q] = sm.Z[d * kPmMaxN + 3 * a + r];
  }
}

}  // namespace

void launch_patch_basis_mixed(Mesh& m, const int32_t* d_verts, int64_t count, int32_t* redo, int32_t* n_redo,
                              cudaStream_t s) {
  set_smem_limit(reinterpret_cast<const void*>(k_patch_basis_mixed), sizeof(PatchSmem));
  k_patch_basis_mixed<<<(unsigned)count, kPmThreads, sizeof(PatchSmem), s>>>(
      d_verts, m.d_sup_ptr.p, m.d_sup_idx.p, m.d_up_ptr.p, m.d_up_col.p, m.d_nbr_ptr.p, m.d_nbr_idx.p, m.f64.bsr.p,
      m.f64.U.p, redo, n_redo);
  CCG_CUDA(cudaGetLastError());
}

}  // namespace ccg
