// Explicit camera Schur complement.  The matrix-free product walks every edge in every
// PCG iteration; here the off-diagonal blocks of S = H_cc + lambda D_c - H_cp H_pp^-1 H_pc
// are formed once per damped system and a PCG iteration only reads them:
//  * k_ex_prepare: per point the factor G of H_pp^-1 = G G^T (G = L^-T, H_pp = L L^T), per
//    edge Y = Jc^T Jp G (DC x 3) and u = G^T b_p, written camera-major;
//  * k_ex_diag: per camera sum Y Y^T (the Schur term of the diagonal block) and sum Y u
//    (of the right-hand side), by segments of the camera's rows;
//  * k_ex_form / k_ex_merge: per block (i, j) of cameras that share points,
//    S_ij = -sum_p Y_ip Y_jp^T over the block's list of row pairs, stored for both rows;
//  * k_ex_pcg: the whole PCG solve in one launch.
// Bounds: k_ex_form the FP64 pipe (300 cameras, 5 million pairs: 2.0 ms) or in FP32 issue
// and the loads of the row pairs (18.5 million pairs: 437 us; 785 without the next pair's
// loads ahead); k_ex_pcg the latency of its exchanges (FP64, 10 cameras: 7.8 us an
// iteration, 300 cameras 14.7; the separate launches took 27 to 40).
// Camera rows Y lie in tiles of 32 rows cut into 16-byte pieces (as the Jacobian rows), so
// a warp that reads consecutive rows of a camera reads contiguous 512-byte blocks.  Every
// sum has a fixed order (lists are in point order, segments are added in order).
#pragma once

#include "schur_common.cuh"

namespace gpo {

template <class Mo, class AT>
struct ExRow {
  static constexpr int DC = Mo::DC, NY = 3 * DC, NV = NY + 3;
  static constexpr int VP = 16 / (int)sizeof(AT);        // values per 16-byte piece
  static constexpr int Q = (NV + VP - 1) / VP;           // pieces of a row
  static constexpr int QY = (NY + VP - 1) / VP;          // pieces that hold Y
  static constexpr int W = Q * VP;
  __host__ __device__ static __forceinline__ size_t piece(size_t row, int q) {
    return ((row >> 5) * Q + q) * 32 + (row & 31);
  }
};

template <class AT, int N>
__device__ __forceinline__ void ex_load(const uint4* Y, size_t row, AT (&v)[N * (16 / sizeof(AT))], int Q) {
  const size_t base = (row >> 5) * (size_t)Q * 32 + (row & 31);
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const uint4 w = __ldg(Y + base + (size_t)q * 32);
    const AT* a = reinterpret_cast<const AT*>(&w);
#pragma unroll
    for (int k = 0; k < (int)(16 / sizeof(AT)); ++k) v[q * (16 / sizeof(AT)) + k] = a[k];
  }
}

// ---------------------------------------------------------------- plan (once per graph)

// Camera-major row of every edge, and the edge of every row.  Scratch: the Y array.
static __global__ void __launch_bounds__(kThreads) k_ex_rows(LaunchSet ls, int* row_edge, int* e_row) {
  GPO_BIND(ch, kl)
  const ChunkRange cr = chunk_range(d, kl);
  for (int q = threadIdx.x; q < cr.nE; q += kThreads) {
    const int e = cr.e0 + d.ch_sorted[cr.e0 + q], s = cr.s0 + d.e_slot[e];
    const int row = d.ex_slot_y0[s] + q - (d.slot_e0[s] - cr.e0);
    row_edge[row] = e;
    e_row[e] = row;
  }
}

// One CTA per camera i walks the camera's rows in order (each warp a contiguous eighth)
// and visits every edge f of the row's point on a camera j > i.  kFill false: counts the
// pairs of each block (i, j).  kFill true: writes them, row order inside a block.
template <bool kFill>
static __global__ void __launch_bounds__(kThreads) k_ex_pairs(LaunchSet ls, const int* row_edge, const int* e_row,
                                                              int nb_max) {
  extern __shared__ int sm[];
  const DevBA& d = ls.probs[0];
  const int i = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int u0 = d.ex_uoff[i], nb = d.ex_uoff[i + 1] - u0;
  if (nb == 0) return;
  int* col = sm;
  int* cnt = sm + nb_max;   // [8][nb]
  const int* src = d.ex_col + d.ex_row[i + 1] - nb;   // the row's columns above i, ascending
  for (int k = threadIdx.x; k < nb; k += kThreads) col[k] = src[k];
  for (int k = threadIdx.x; k < 8 * nb; k += kThreads) cnt[k] = 0;
  __syncthreads();
  const int a0 = d.ex_crow[i], n = d.ex_crow[i + 1] - a0;
  const int ra = a0 + (int)((long long)n * warp / 8), rb = a0 + (int)((long long)n * (warp + 1) / 8);
  int* mine = cnt + warp * nb;
  auto walk = [&](auto&& visit) {
    for (int r0 = ra; r0 < rb; r0 += 32) {
      int o0 = 0, o1 = 0;
      if (r0 + lane < rb) {
        const int p = d.e_pt[row_edge[r0 + lane]];
        o0 = d.pt_off[p];
        o1 = d.pt_off[p + 1];
      }
      const int m = min(32, rb - r0);
      for (int t = 0; t < m; ++t) {
        const int f0 = __shfl_sync(0xffffffffu, o0, t), f1 = __shfl_sync(0xffffffffu, o1, t);
        for (int f = f0 + lane; f < f1; f += 32) {
          const int j = d.e_cam[f];
          if (j <= i) continue;
          int lo = 0, hi = nb - 1;
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (col[mid] < j) lo = mid + 1;
            else hi = mid;
          }
          visit(lo, r0 + t, f);
        }
        __syncwarp();
      }
    }
  };
  walk([&](int k, int, int) { mine[k] += 1; });   // a point's cameras are distinct: no two lanes share k
  __syncthreads();
  for (int k = threadIdx.x; k < nb; k += kThreads) {
    int at = kFill ? d.ex_poff[u0 + k] : 0;
    for (int w = 0; w < 8; ++w) {
      const int c = cnt[w * nb + k];
      cnt[w * nb + k] = at;
      at += c;
    }
    if (!kFill) d.ex_poff[u0 + k] = at;
  }
  if (!kFill) return;
  __syncthreads();
  walk([&](int k, int r, int f) { d.ex_pair[mine[k]++] = make_int2(r, e_row[f]); });
}

// Counts (in ex_poff) to offsets, and the work items of k_ex_form: a block's pairs in
// segments of ex_seg; a block of several segments sums through ex_part and is listed in
// ex_multi.  One CTA.
static __global__ void __launch_bounds__(1024) k_ex_items(LaunchSet ls) {
  __shared__ int ws[32][4];
  __shared__ int carry[4];
  const DevBA& d = ls.probs[0];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x < 4) carry[threadIdx.x] = 0;
  __syncthreads();
  for (int b0 = 0; b0 < d.ex_nbu; b0 += 1024) {
    const int b = b0 + (int)threadIdx.x;
    const int n = b < d.ex_nbu ? d.ex_poff[b] : 0, ns = (n + d.ex_seg - 1) / d.ex_seg;
    int v[4] = {n, ns, ns > 1 ? ns : 0, ns > 1 ? 1 : 0}, x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      x[k] = v[k];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x[k], o);
        if (lane >= o) x[k] += y;
      }
      if (lane == 31) ws[warp][k] = x[k];
    }
    __syncthreads();
    int tot[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      int before = carry[k];
      tot[k] = carry[k];
      for (int w = 0; w < 32; ++w) {
        if (w < warp) before += ws[w][k];
        tot[k] += ws[w][k];
      }
      x[k] = before + x[k] - v[k];   // exclusive
    }
    if (b < d.ex_nbu) {
      d.ex_poff[b] = x[0];
      for (int s = 0; s < ns; ++s)
        d.ex_item[x[1] + s] = make_int4(x[0] + s * d.ex_seg, min(x[0] + n, x[0] + (s + 1) * d.ex_seg), b, ns > 1 ? x[2] + s : -1);
      if (ns > 1) d.ex_multi[x[3]] = make_int4(b, x[2], ns, 0);
    }
    __syncthreads();
    if (threadIdx.x < 4) carry[threadIdx.x] = tot[threadIdx.x];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    d.ex_poff[d.ex_nbu] = carry[0];
    d.ex_count[0] = carry[1];
    d.ex_count[1] = carry[3];
  }
}

// ---------------------------------------------------------------- camera rows

// Damped point block h (6, packed) -> its inverse o and the factor G = L^-T as the packed
// lower triangle of L^-1 (m00 m10 m11 m20 m21 m22).  Not positive definite in this
// precision: Jacobi, in both.
template <class AT>
__device__ __forceinline__ void point_factor(const AT (&h)[6], AT (&o)[6], AT (&m)[6]) {
  inv3(h, o);
  const AT p0 = h[0], i0 = p0 > (AT)0 ? (AT)1 / sqrt(p0) : (AT)0;
  const AT l10 = h[1] * i0, l20 = h[2] * i0;
  const AT p1 = h[3] - l10 * l10, i1 = p1 > (AT)0 ? (AT)1 / sqrt(p1) : (AT)0;
  const AT l21 = (h[4] - l20 * l10) * i1;
  const AT p2 = h[5] - l20 * l20 - l21 * l21, i2 = p2 > (AT)0 ? (AT)1 / sqrt(p2) : (AT)0;
  const AT det = p0 * p1 * p2;
  if (i0 > (AT)0 && i1 > (AT)0 && i2 > (AT)0 && isfinite(det) && isfinite(i0 * i1 * i2)) {
    m[0] = i0;
    m[1] = -l10 * i0 * i1;
    m[2] = i1;
    m[3] = -(l20 * i0 + l21 * m[1]) * i2;
    m[4] = -l21 * i1 * i2;
    m[5] = i2;
  } else {
    o[0] = h[0] > (AT)0 ? (AT)1 / h[0] : (AT)0;
    o[3] = h[3] > (AT)0 ? (AT)1 / h[3] : (AT)0;
    o[5] = h[5] > (AT)0 ? (AT)1 / h[5] : (AT)0;
    o[1] = o[2] = o[4] = (AT)0;
    m[0] = sqrt(o[0]);
    m[2] = sqrt(o[3]);
    m[5] = sqrt(o[5]);
    m[1] = m[3] = m[4] = (AT)0;
  }
}

// One CTA per chunk: H_pp^-1 and G per point, then the camera rows of the chunk's edges in
// slot order (a slot's edges are consecutive rows of its camera).
template <class Mo, class JT>
__global__ void __launch_bounds__(kThreads) k_ex_prepare(LaunchSet ls) {
  using AT = typename AccOf<JT>::T;
  using R = ExRow<Mo, AT>;
  constexpr int M = Mo::M, DC = Mo::DC, NJ = Mo::NJ, JP0 = Dims<Mo>::JP0;
  GPO_BIND(ch, kl)
  if (!d.ex || !d.sc->active) return;
  extern __shared__ __align__(16) unsigned char smem[];
  AT* pv = reinterpret_cast<AT*>(smem);                                  // [np_max][9]: L^-1 (6), u (3)
  int* sb = reinterpret_cast<int*>(pv + 9 * (size_t)ls.np_max);          // [ns_max] row of slot position 0
  const ChunkRange cr = chunk_range(d, kl);
  const Scalars* sc = d.sc;
  const AT lam = (AT)sc->lambda;
  const AT* Hpp = reinterpret_cast<const AT*>(d.Hpp);
  const AT* bp = reinterpret_cast<const AT*>(d.bp);
  AT* Hinv = reinterpret_cast<AT*>(d.Hinv);
  for (int s = threadIdx.x; s < cr.nS; s += kThreads)
    sb[s] = d.ex_slot_y0[cr.s0 + s] - (d.slot_e0[cr.s0 + s] - cr.e0);
  for (int j = threadIdx.x; j < cr.nP; j += kThreads) {
    const size_t pj = cr.p0 + j;
    AT h[6], o[6], m[6], b[3];
#pragma unroll
    for (int k = 0; k < 6; ++k) h[k] = Hpp[6 * pj + k];
#pragma unroll
    for (int k = 0; k < 3; ++k) b[k] = bp[3 * pj + k];
    h[0] += lam * damp_diag(h[0], sc);
    h[3] += lam * damp_diag(h[3], sc);
    h[5] += lam * damp_diag(h[5], sc);
    point_factor(h, o, m);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      Hinv[6 * pj + k] = o[k];
      pv[9 * j + k] = m[k];
    }
    pv[9 * j + 6] = m[0] * b[0];
    pv[9 * j + 7] = m[1] * b[0] + m[2] * b[1];
    pv[9 * j + 8] = m[3] * b[0] + m[4] * b[1] + m[5] * b[2];
  }
  __syncthreads();
  uint4* Y = reinterpret_cast<uint4*>(d.ex_Y);
  for (int q = threadIdx.x; q < cr.nE; q += kThreads) {
    const int i = d.ch_sorted[cr.e0 + q], e = cr.e0 + i;
    const size_t row = (size_t)(sb[d.e_slot[e]] + q);
    const AT* m = pv + 9 * (d.e_pt[e] - cr.p0);
    AT J[NJ];
    load_row_t<NJ>(reinterpret_cast<const JT*>(d.J), (size_t)e, J);
    AT K[M][3];
#pragma unroll
    for (int a = 0; a < M; ++a) {
      const AT* Ja = J + JP0 + 3 * a;
      K[a][0] = Ja[0] * m[0];
      K[a][1] = Ja[0] * m[1] + Ja[1] * m[2];
      K[a][2] = Ja[0] * m[3] + Ja[1] * m[4] + Ja[2] * m[5];
    }
    __align__(16) AT v[R::W];
#pragma unroll
    for (int k = R::NV; k < R::W; ++k) v[k] = (AT)0;
#pragma unroll
    for (int r = 0; r < DC; ++r)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        AT s = J[r] * K[0][k];
#pragma unroll
        for (int a = 1; a < M; ++a) s += J[a * DC + r] * K[a][k];
        v[3 * r + k] = s;
      }
#pragma unroll
    for (int k = 0; k < 3; ++k) v[R::NY + k] = m[6 + k];
    const uint4* s4 = reinterpret_cast<const uint4*>(v);
#pragma unroll
    for (int p = 0; p < R::Q; ++p) Y[R::piece(row, p)] = s4[p];
  }
}

// ---------------------------------------------------------------- diagonal and off-diagonal blocks

template <class AT> constexpr int kExDiagWarps = sizeof(AT) == 8 ? 2 : 4;   // shared memory: 54 sums per lane

// acc + x . y over three values: in FP32 the row's products first, so that the sum over rows
// rounds once per row.
template <class AT>
__device__ __forceinline__ AT ex_dot3(const AT* x, const AT* y, AT acc) {
  if constexpr (sizeof(AT) == 4) return acc + fmaf(x[2], y[2], fmaf(x[1], y[1], x[0] * y[0]));
  else return fma(x[2], y[2], fma(x[1], y[1], fma(x[0], y[0], acc)));
}

// One warp per segment of a camera's rows: sum Y Y^T (packed upper triangle) and sum Y u,
// a row per lane, the lanes added in a fixed order.  S_cc = H_cc + lambda D_c - sum Y Y^T
// cancels and the squares on its diagonal all have one sign, so that in FP32 a long chain of
// additions shows in the solve: the lanes, and the segments in k_cam_finalize, are added by
// ex_chains (64 segments and more in FP64, whose conversions took 4 us of a damped system of
// 100 cameras).  RMS error of S_cc relative to its diagonal, in 2^-23, with one chain throughout
// and so, the matrix-free kernels' on the same graph in brackets: 6 cameras of 33,000 rows
// 0.46, 0.36 (0.37); 4 of 45,000 0.86, 0.52 (0.57).
template <class Mo, class AT>
__global__ void __launch_bounds__(kExDiagWarps<AT> * 32) k_ex_diag(LaunchSet ls) {
  using R = ExRow<Mo, AT>;
  constexpr int DC = Mo::DC, TC = Dims<Mo>::TC, NA = TC + DC, NPA = Dims<Mo>::NPA, WPC = kExDiagWarps<AT>;
  __shared__ AT buf[WPC][NA][33];
  GPO_BIND(xd, xl)
  if (!d.ex || !d.sc->active) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int item = xl * WPC + warp;
  if (item >= d.ex_nd) return;
  const int c = d.ex_dcam[item], r0 = d.ex_crow[c] + (item - d.ex_doff[c]) * d.ex_dseg;
  const int r1 = min(r0 + d.ex_dseg, d.ex_crow[c + 1]);
  AT acc[NA];
#pragma unroll
  for (int k = 0; k < NA; ++k) acc[k] = (AT)0;
  for (int r = r0 + lane; r < r1; r += 32) {
    AT v[R::W];
    ex_load<AT, R::Q>(reinterpret_cast<const uint4*>(d.ex_Y), (size_t)r, v, R::Q);
    int t = 0;
#pragma unroll
    for (int a = 0; a < DC; ++a) {
#pragma unroll
      for (int b = a; b < DC; ++b, ++t) acc[t] = ex_dot3(v + 3 * a, v + 3 * b, acc[t]);
    }
#pragma unroll
    for (int a = 0; a < DC; ++a) acc[TC + a] = ex_dot3(v + 3 * a, v + R::NY, acc[TC + a]);
  }
#pragma unroll
  for (int k = 0; k < NA; ++k) buf[warp][k][lane] = acc[k];
  __syncwarp();
  AT* out = reinterpret_cast<AT*>(d.ex_dpart) + (size_t)item * NPA;
  for (int t = lane; t < NPA; t += 32) out[t] = t < NA ? ex_chains<AT>(buf[warp][t], 1, 32) : (AT)0;
}

template <class Mo, class AT>
__device__ __forceinline__ void ex_store(const DevBA& d, int u, int t, AT v) {
  constexpr int DC = Mo::DC, EL = DC * DC;
  AT* S = reinterpret_cast<AT*>(d.ex_S);
  const int2 at = d.ex_ublk[u];
  S[(size_t)at.x * EL + t] = v;                            // S_ij, column-major
  S[(size_t)at.y * EL + (t % DC) * DC + t / DC] = v;       // S_ji
}

// One warp per work item: -sum Y_i Y_j^T over the item's pairs.  FP32: a pair per lane, all
// of the block's products in the lane's registers; FP64: three lanes per pair, three rows
// each.  The lanes' sums are added in lane order.
template <class Mo, class AT>
__global__ void __launch_bounds__(128) k_ex_form(LaunchSet ls) {
  using R = ExRow<Mo, AT>;
  constexpr int DC = Mo::DC, EL = DC * DC, RS = sizeof(AT) == 8 ? 3 : 1, NG = 32 / RS, RR = DC / RS;
  constexpr int HB = (EL + 1) / 2;   // outputs reduced at a time
  __shared__ AT buf[4][HB][NG + 1];
  GPO_BIND(xf, xl)
  if (!d.ex || !d.sc->active) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane / RS, h = lane % RS;
  const int n_item = d.ex_count[0], stride = d.ex_nxf * 4;
  const uint4* Y = reinterpret_cast<const uint4*>(d.ex_Y);
  AT* part = reinterpret_cast<AT*>(d.ex_part);
  // a warp's items are a grid apart (its CTA's warps work on neighbouring blocks, which
  // share camera rows); the next item and the next pair's rows are known a step ahead
  int item = xl * 4 + warp;
  int4 nit = item < n_item ? d.ex_item[item] : make_int4(0, 0, 0, 0);
  for (; item < n_item; item += stride) {
    const int4 it = nit;
    int2 nx = g < NG && it.x + g < it.y ? __ldg(d.ex_pair + it.x + g) : make_int2(0, 0);
    if (item + stride < n_item) nit = d.ex_item[item + stride];
    AT acc[RR * DC];
#pragma unroll
    for (int k = 0; k < RR * DC; ++k) acc[k] = (AT)0;
    if (g < NG) {
      for (int p = it.x + g; p < it.y; p += NG) {
        const int2 ef = nx;
        if (p + NG < it.y) nx = __ldg(d.ex_pair + p + NG);
        AT yf[R::QY * R::VP], ye[RR * 3 + R::VP];
        ex_load<AT, R::QY>(Y, (size_t)ef.y, yf, R::Q);
        if constexpr (RS == 1) {
          AT w[R::QY * R::VP];
          ex_load<AT, R::QY>(Y, (size_t)ef.x, w, R::Q);
#pragma unroll
          for (int k = 0; k < RR * 3; ++k) ye[k] = w[k];
        } else {
          const AT* src = reinterpret_cast<const AT*>(d.ex_Y);
#pragma unroll
          for (int k = 0; k < RR * 3; ++k) {
            const int o = h * RR * 3 + k;
            ye[k] = __ldg(src + R::piece((size_t)ef.x, 0) * R::VP + (size_t)(o / R::VP) * 32 * R::VP + o % R::VP);
          }
        }
#pragma unroll
        for (int a = 0; a < RR; ++a)
#pragma unroll
          for (int b = 0; b < DC; ++b)
#pragma unroll
            for (int k = 0; k < 3; ++k) acc[a * DC + b] = fma(ye[3 * a + k], yf[3 * b + k], acc[a * DC + b]);
      }
    }
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int t0 = half * HB, t1 = half ? EL : HB;
      if (g < NG) {
#pragma unroll
        for (int a = 0; a < RR; ++a)
#pragma unroll
          for (int b = 0; b < DC; ++b) {
            const int t = b * DC + h * RR + a;
            if (t >= t0 && t < t1) buf[warp][t - t0][g] = acc[a * DC + b];
          }
      }
      __syncwarp();
      for (int t = t0 + lane; t < t1; t += 32) {
        AT s = (AT)0;
        for (int q = 0; q < NG; ++q) s += buf[warp][t - t0][q];
        if (it.w < 0) ex_store<Mo, AT>(d, it.z, t, -s);
        else part[(size_t)it.w * EL + t] = -s;
      }
      __syncwarp();
    }
  }
}

template <class Mo, class AT>
__global__ void __launch_bounds__(128) k_ex_merge(LaunchSet ls) {
  constexpr int EL = Mo::DC * Mo::DC;
  GPO_BIND(xf, xl)
  if (!d.ex || !d.sc->active) return;
  const int lane = threadIdx.x & 31, n = d.ex_count[1];
  for (int m = xl * 4 + (threadIdx.x >> 5); m < n; m += d.ex_nxf * 4) {
    const int4 e = d.ex_multi[m];
    const AT* part = reinterpret_cast<const AT*>(d.ex_part) + (size_t)e.y * EL;
    for (int t = lane; t < EL; t += 32) {
      AT s = part[t];
      for (int q = 1; q < e.z; ++q) s += part[(size_t)q * EL + t];
      ex_store<Mo, AT>(d, e.x, t, s);
    }
  }
}

// ---------------------------------------------------------------- the PCG solve

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of `p` (own shared memory) in the shared memory of CTA `rank` of the cluster.
__device__ __forceinline__ unsigned cluster_addr(const void* p, int rank) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}

// Values travel between the CTAs of a solve as 8-byte words, half of each the epoch (the
// count of the solve's reductions) the value belongs to: a reader that sees the epoch has
// the value, in one round trip and without fences or acquire loads (which would also empty
// the L1 cache that holds the blocks).  A float takes one word, a double two.
template <class T>
__device__ __forceinline__ void ex_pack(T v, unsigned epoch, unsigned long long (&w)[sizeof(T) / 4]) {
  const unsigned long long e = (unsigned long long)epoch << 32;
  if constexpr (sizeof(T) == 4) {
    w[0] = e | __float_as_uint(v);
  } else {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    w[0] = e | (u & 0xffffffffull);
    w[1] = e | (u >> 32);
  }
}
template <class T>
__device__ __forceinline__ bool ex_unpack(const unsigned long long (&w)[sizeof(T) / 4], unsigned epoch, T& v) {
  if constexpr (sizeof(T) == 4) {
    v = __uint_as_float((unsigned)w[0]);
    return (unsigned)(w[0] >> 32) == epoch;
  } else {
    v = __longlong_as_double((long long)((w[0] & 0xffffffffull) | (w[1] << 32)));
    return (unsigned)(w[0] >> 32) == epoch && (unsigned)(w[1] >> 32) == epoch;
  }
}
// Words in global memory.
template <class T>
__device__ __forceinline__ void ex_post(unsigned long long* at, T v, unsigned epoch) {
  unsigned long long w[sizeof(T) / 4];
  ex_pack(v, epoch, w);
  if constexpr (sizeof(T) == 4) asm volatile("st.relaxed.gpu.u64 [%0], %1;" ::"l"(at), "l"(w[0]) : "memory");
  else asm volatile("st.relaxed.gpu.v2.u64 [%0], {%1, %2};" ::"l"(at), "l"(w[0]), "l"(w[1]) : "memory");
}
template <class T>
__device__ __forceinline__ bool ex_poll(const unsigned long long* at, T& v, unsigned epoch) {
  unsigned long long w[sizeof(T) / 4];
  if constexpr (sizeof(T) == 4) asm volatile("ld.relaxed.gpu.u64 %0, [%1];" : "=l"(w[0]) : "l"(at) : "memory");
  else asm volatile("ld.relaxed.gpu.v2.u64 {%0, %1}, [%2];" : "=l"(w[0]), "=l"(w[1]) : "l"(at) : "memory");
  return ex_unpack(w, epoch, v);
}
// Words in shared memory: written into another CTA of the cluster (address of
// cluster_addr), read in the own one.
template <class T>
__device__ __forceinline__ void ex_post_cluster(unsigned at, T v, unsigned epoch) {
  unsigned long long w[sizeof(T) / 4];
  ex_pack(v, epoch, w);
#pragma unroll
  for (int k = 0; k < (int)(sizeof(T) / 4); ++k)
    asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(at + 8 * k), "l"(w[k]) : "memory");
}
template <class T>
__device__ __forceinline__ bool ex_poll_shared(const unsigned long long* at, T& v, unsigned epoch) {
  unsigned long long w[sizeof(T) / 4];
  const unsigned a = (unsigned)__cvta_generic_to_shared(at);
#pragma unroll
  for (int k = 0; k < (int)(sizeof(T) / 4); ++k)
    asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(w[k]) : "r"(a + 8 * k) : "memory");
  return ex_unpack(w, epoch, v);
}
// Bounded waiting by the SM's clock: false once kWaitClocks have passed since the start.
struct ExWait {
  long long t0;
  __device__ __forceinline__ ExWait() : t0(sm_clock()) {}
  __device__ __forceinline__ bool again() const { return sm_clock() - t0 < kWaitClocks; }
};

// Sum over a warp of the lanes' v, n values in all (the lanes past n hold zero), the same in
// every lane.  FP64 additions take a sub-partition's pipe some 70 clocks each on this part, so
// the values are added as 64-bit integers on the scale of the largest: a value's 53-bit
// significand is shifted to leave room for n terms (bits below 2^-52 of the largest term and
// less are cut, as roundings of a floating sum cut them), and the order does not matter.
// Infinities, NaN and values near the smallest exponents are added as they are.
static __device__ __noinline__ double ex_warp_sum(double v, int n) {
  constexpr unsigned full = 0xffffffffu;
  const long long b = __double_as_longlong(v);
  const int x = (int)(b >> 52) & 0x7ff, e = __reduce_max_sync(full, x);
  if (e == 0x7ff || e < 128) {
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(full, v, o);
    return v;
  }
  const int room = 5 - (n > 1 ? 32 - __clz(n - 1) : 0) + 4;   // 2^53 terms n of them fit 62 bits when shifted by this
  const int sh = e - x - room;                                // right shift
  const long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;
  long long q = x == 0 || sh > 62 ? 0ll : (sh >= 0 ? m >> sh : m << -sh);
  if (b < 0) q = -q;
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(full, q, o);
  // q 2^(e - 1023 - 52 - room)
  return __ll2double_rn(q) * __hiloint2double((e - 52 - room) << 20, 0);
}

// Rows of a CTA: ceil(C / G) consecutive cameras; `wpr` warps share a row.
__host__ __device__ inline int ex_rows_per_cta(int C, int G) { return (C + G - 1) / G; }
__host__ __device__ inline int ex_warps_per_row(int rpc) {
  int w = kExThreads / 32;
  while (w > 1 && w * rpc > kExThreads / 32) w >>= 1;
  return w;
}
// A camera's vector in shared memory: coordinate k of the first DC at (k mod 3) GS + k / 3, so
// that a lane's coordinates of a block (columns k mod 3 = its column group) are one vector
// load; the remaining coordinates after them.
template <class Mo, class AT>
struct ExVec {
  static constexpr int DC = Mo::DC, DB = Mo::DB, ST = DC / 3, GS = ST == 3 ? 4 : 2;
  static constexpr int VP = 16 / (int)sizeof(AT);
  static constexpr int W = (3 * GS + DB - DC + VP - 1) / VP * VP;   // values of a camera
  __device__ static __forceinline__ int at(int k) { return k < DC ? (k % 3) * GS + k / 3 : 3 * GS + k - DC; }
  // the ST coordinates of column group cg
  __device__ static __forceinline__ void group(const AT* v, int cg, AT (&o)[ST]) {
    const AT* p = v + cg * GS;
    if constexpr (sizeof(AT) == 4 && ST == 3) {
      const float4 q = *reinterpret_cast<const float4*>(p);
      o[0] = q.x; o[1] = q.y; o[2] = q.z;
    } else if constexpr (sizeof(AT) == 4) {
      const float2 q = *reinterpret_cast<const float2*>(p);
      o[0] = q.x; o[1] = q.y;
    } else {
      const double2 q = *reinterpret_cast<const double2*>(p);
      o[0] = q.x; o[1] = q.y;
      if constexpr (ST == 3) o[2] = p[2];
    }
  }
};
// Shared memory of a solve: nloc cameras in a CTA's column set; nres: most blocks of a CTA's
// rows if they are kept in shared memory, else 0.
template <class Mo, class AT>
__host__ __device__ inline size_t ex_pcg_smem(int C, int G, int nloc, int nres) {
  const int rpc = ex_rows_per_cta(C, G), PW = Mo::kExtra ? Mo::DB : Mo::DC;
  return sizeof(AT) * (2 * (size_t)nloc * ExVec<Mo, AT>::W + Mo::DC * Mo::DC * (size_t)nres +
                       (size_t)rpc * Mo::DB * (7 + 2 * Mo::DB) + (size_t)rpc * ex_warps_per_row(rpc) * PW) +
         sizeof(int) * (size_t)nres;
}

// The sum over a group of CTAs of each one's v[0 .. n-1], by one warp: value w (0 or 1) of the
// reduction `epoch`; value 1 takes part in every second one.  slot_s: [2][kExCluster][4] words
// in the CTA's shared memory (a cluster's slots); red: [2][kExMaxCtas][4] words and the two
// counts of posts (a grid's).  n_slot: CTAs of the group (the test hook adds one that posts
// nothing: a grid waits for its slot, a cluster for an epoch that does not come).  Sets *lost
// on a wait that gave up.
template <class AT, bool kCluster>
__device__ __noinline__ double ex_group_sum(const AT* v, int n, int w, unsigned epoch, int rank, int n_slot,
                                            unsigned long long* slot_s, unsigned long long* red, int* lost) {
  constexpr unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, par = epoch & 1;
  double mine = 0.0;
#pragma unroll 1
  for (int i = lane; i < n; i += 32) mine += (double)v[i];
  mine = ex_warp_sum(mine, 32);
  ExWait wait;
  bool ok = true;
  if constexpr (kCluster) {
    if (lane < kExCluster) ex_post_cluster(cluster_addr(slot_s + (par * kExCluster + rank) * 4 + 2 * w, lane), mine, epoch);
    double u = 0.0;
    const unsigned want = epoch + (unsigned)(n_slot - kExCluster);
    if (lane < kExCluster)
      while (!ex_poll_shared(slot_s + (par * kExCluster + lane) * 4 + 2 * w, u, want) && (ok = wait.again())) {}
    if (!__all_sync(full, ok)) *lost = 1;
    return ex_warp_sum(u, kExCluster);
  } else {
    constexpr int PS = (kExGrid + 32) / 32;   // slots per lane, one more than the grid's
    unsigned long long* slots = red + (size_t)par * 4 * kExMaxCtas + 2 * w;
    // one lane polls a count of the posts first: every CTA polling every slot while the last
    // CTAs arrive keeps the few L2 lines of the slots so busy that the posts wait
    if (lane == 0) {
      unsigned* count = reinterpret_cast<unsigned*>(red + 8 * kExMaxCtas + w);
      ex_post(slots + 4 * rank, mine, epoch);
      asm volatile("red.relaxed.gpu.add.u32 [%0], %1;" ::"l"(count), "r"(1u) : "memory");
      const unsigned want = (unsigned)n_slot * (w ? epoch / 2 : epoch);
      unsigned c;
      do asm volatile("ld.relaxed.gpu.u32 %0, [%1];" : "=r"(c) : "l"(count) : "memory");
      while (c < want && (ok = wait.again()));
    }
    ok = __shfl_sync(full, (int)ok, 0);
    double u[PS];
    bool all;
    do {
      all = true;
#pragma unroll
      for (int k = 0; k < PS; ++k) {
        u[k] = 0.0;
        if (lane + 32 * k < n_slot) all = ex_poll(slots + 4 * (lane + 32 * k), u[k], epoch) && all;
      }
    } while (!__all_sync(full, all) && (ok = __all_sync(full, ok && wait.again())));
    if (!ok) *lost = 1;
#pragma unroll
    for (int k = 1; k < PS; ++k) u[0] += u[k];
    return ex_warp_sum(u[0], 32);
  }
}

// The whole solve of one problem by a group of CTAs: a cluster of kExCluster (small
// problems; several in one launch) or a grid of up to kExGrid (cooperative launch).  A CTA
// owns consecutive block rows and keeps the search direction p of every camera its rows
// touch (its column set) in shared memory, updated there as p = (z + beta p) / n, and its
// rows' blocks as well where they fit.  Two group reductions per iteration, p^T S p and then
// r^T M r with |r|^2 (a warp each), and one exchange of z, which the other warps receive
// while the reduction runs.  Both travel as words that carry their epoch, the partial sums
// of a cluster into every CTA's shared memory, all else through global memory; a value is
// overwritten only after a later reduction has shown that every CTA has read it.  Every CTA
// sums the partials in the same way and so forms the same scalars; rank 0 writes them back.
// The recurrences, guards and stopping rules are those of k_cam_apply and k_pcg_update; the
// inner products are sums of AT products, added exactly to FP64's precision.
template <class Mo, class AT, bool kCluster, bool kRes>
__global__ void __launch_bounds__(kExThreads, 1) k_ex_pcg(LaunchSet ls, int prob0) {
  using V = ExVec<Mo, AT>;
  constexpr int DC = Mo::DC, DB = Mo::DB, TB = Dims<Mo>::TB, EL = DC * DC, NW = kExThreads / 32;
  constexpr int CG = 3, LN = CG * DC, ST = DC / CG;   // columns per step, lanes in use, steps per block
  constexpr int PW = Mo::kExtra ? DB : DC;
  constexpr int ZW = sizeof(AT) / 4;                  // words of a value
  constexpr int ZT = kExThreads - 64, ZK = 4;         // threads that receive z, values each keeps in registers
  constexpr unsigned full = 0xffffffffu;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ DevBA d;
  __shared__ unsigned long long slot_s[2][kExCluster][4];
  __shared__ double is_s;
  __shared__ AT co[4];       // alpha, sigma alpha, 1 / n, beta
  __shared__ int fl[5];      // stop, restart, save best, a wait gave up, r^T M r not positive
  const int G = kCluster ? kExCluster : (int)gridDim.x, rank = (int)blockIdx.x % G;
  const int q = kCluster ? ls.cl_prob[blockIdx.x / kExCluster] : prob0;
  bind_problem(d, ls.probs + q);
  pdl_wait();
  Scalars* sc = d.sc;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (!sc->active || sc->pcg_done) return;   // the same for every CTA of the group
  if (!kCluster && *reinterpret_cast<volatile int*>(ls.err)) {   // an earlier solve's wait gave up
    if (threadIdx.x == 0) sc->active = 0;                        // no step without a solve
    return;
  }
  const int rpc = ex_rows_per_cta(d.C, G), wpr = ex_warps_per_row(rpc), rpp = NW / wpr;
  const int c0 = min(rank * rpc, d.C), nr = min(c0 + rpc, d.C) - c0;
  const int* lcol = d.ex_lcol + d.ex_loff[rank];
  const int nloc = d.ex_loff[rank + 1] - d.ex_loff[rank];
  const int b0 = d.ex_row[c0], nb = d.ex_row[c0 + nr] - b0;
  AT* pl = reinterpret_cast<AT*>(smem);                          // [nloc][V::W] direction
  AT* xl = pl + (size_t)nloc * V::W;                             // [nloc][V::W] x, with restarts
  AT* xs = xl + (size_t)nloc * V::W;                             // [rpc][DB]: x, r, y, g, best x, terms of the sums
  AT* rs = xs + (size_t)rpc * DB;
  AT* ys = rs + (size_t)rpc * DB;
  AT* gs = ys + (size_t)rpc * DB;
  AT* bs = gs + (size_t)rpc * DB;
  AT* da = bs + (size_t)rpc * DB;
  AT* db = da + (size_t)rpc * DB;
  AT* Ss = db + (size_t)rpc * DB;                                // [rpc][DB][DB] diagonal blocks, preconditioner
  AT* Ms = Ss + (size_t)rpc * DB * DB;
  AT* part = Ms + (size_t)rpc * DB * DB;                         // [rpc][wpr][PW]
  AT* Sr = part + (size_t)rpc * wpr * PW;                        // the rows' blocks (kRes) ...
  int* li_s = reinterpret_cast<int*>(Sr + (size_t)nb * EL);      // ... and their columns in the set
  unsigned long long* zw = d.ex_z;
  AT* gx = reinterpret_cast<AT*>(d.x);
  const AT* gz = reinterpret_cast<const AT*>(d.z);
  const AT* Sx = reinterpret_cast<const AT*>(d.ex_S);
  const AT* xH = reinterpret_cast<const AT*>(d.xe_H);
  // The loops of the solve are kept rolled where they are not the work itself: unrolled, the
  // kernel is 95 KB of instructions (32 rolled), which an iteration fetches anew, and each
  // CTA in turn is late by the misses.  An iteration, unrolled -> rolled: 20 cameras (a
  // cluster) 6.6 -> 5.3 us; grids: 777 cameras 10.5 -> 8.8, 1,000 keyframes 11.9 -> 9.3
#pragma unroll 1
  for (int i = tid; i < nr * DB; i += kExThreads) {
    xs[i] = bs[i] = (AT)0;
    rs[i] = gs[i] = reinterpret_cast<const AT*>(d.g)[(size_t)c0 * DB + i];
  }
#pragma unroll 1
  for (int i = tid; i < nr * DB * DB; i += kExThreads) {
    const int c = c0 + i / (DB * DB), a = i % (DB * DB) / DB, b = i % DB;
    const size_t o = (size_t)c * TB + sym_idx(DB, a, b);
    Ss[i] = reinterpret_cast<const AT*>(d.S)[o];
    Ms[i] = reinterpret_cast<const AT*>(d.Minv)[o];
  }
#pragma unroll 1
  for (int i = tid; i < nloc * V::W; i += kExThreads) pl[i] = xl[i] = (AT)0;
  if (kCluster && tid < 2 * kExCluster * 4) (&slot_s[0][0][0])[tid] = 0ull;
  if constexpr (kRes) {
    const AT* src = Sx + (size_t)b0 * EL;
    const int n = nb * EL;
#pragma unroll 1
    for (int i = tid; i < nb; i += kExThreads) li_s[i] = __ldg(d.ex_lidx + b0 + i);
#pragma unroll 4
    for (int i = tid; i < n; i += kExThreads) Sr[i] = __ldg(src + i);
  }
  // the z values this thread receives: entries zi of the column set, their place in z
  const int nz = nloc * DB, z0 = tid - 64;
  AT zr[ZK];
  int zo[ZK];
#pragma unroll
  for (int k = 0; k < ZK; ++k) {
    const int i = z0 + k * ZT;
    zo[k] = z0 >= 0 && i < nz ? lcol[i / DB] * DB + i % DB : -1;
    zr[k] = zo[k] >= 0 ? gz[zo[k]] : (AT)0;
  }
  // scalars of the solve: warp 0 keeps those of r^T M r, warp 1 those of |r|
  const double tol_abs = sc->tol_abs, ratio = sc->ratio;
  const int max_it = sc->max_it, normalize = sc->normalize, restart_every = sc->restart_every;
  double s_rz = sc->rz, s_sigma = 1.0, s_rnorm = sc->rnorm, s_rmin = sc->rmin;
  int pcg_it = 0, products = 0;
  if (tid == 0) {
    co[2] = (AT)1;
    co[3] = (AT)0;
    fl[0] = fl[1] = fl[2] = fl[3] = fl[4] = 0;
    is_s = 1.0;
  }
  __shared__ double sigma_s;
  if (tid == 0) sigma_s = 1.0;
  int fail = 0, breakdown = 0, use_best = 0, have_best = 0, saved = 0;
  unsigned epoch = 0;   // of the group reductions
  if constexpr (kCluster) cluster_sync();   // every CTA has started before its shared memory is written
  else __syncthreads();

  auto group_sum = [&](const AT* v, int w) -> double {
    return ex_group_sum<AT, kCluster>(v, nr * DB, w, epoch, rank, G + ls.debug_wait,
                                      &slot_s[0][0][0], d.ex_red, &fl[3]);
  };
  auto gave_up = [&] {   // leaves the kernel (a cluster's CTAs together: their shared memory is shared)
    if (tid == 0) {
      atomicExch(ls.err, 1);
      sc->active = 0;   // the rest of the iteration, and the iterations after it, leave the problem alone
    }
    if constexpr (kCluster) cluster_sync();
  };
  auto receive_z = [&](int o, AT& z) {
    ExWait wait;
    bool ok = true;
    while (!ex_poll(zw + (size_t)o * ZW, z, epoch) && (ok = wait.again())) {}
    if (!ok) fl[3] = 1;
  };

  for (;;) {
    const int restart = fl[1];
    if (!restart && z0 >= 0) {   // the direction of every camera of the column set
      const AT beta = co[3], inv_n = co[2];
#pragma unroll
      for (int k = 0; k < ZK; ++k) {
        const int i = z0 + k * ZT;
        if (i < nz) {
          AT* p = pl + i / DB * V::W + V::at(i % DB);
          *p = (zr[k] + beta * *p) * inv_n;
        }
      }
#pragma unroll 1
      for (int i = z0 + ZK * ZT; i < nz; i += ZT) {
        const int o = __ldg(lcol + i / DB) * DB + i % DB;
        AT* p = pl + i / DB * V::W + V::at(i % DB);
        AT z = (AT)0;
        if (epoch == 0) z = gz[o];
        else receive_z(o, z);
        *p = (z + beta * *p) * inv_n;
      }
    }
    const AT* vec = restart ? xl : pl;   // a restart's product is of the current solution
    __syncthreads();
#pragma unroll 1
    for (int r = warp / wpr; r < nr; r += rpp) {
      const int sub = warp % wpr, c = c0 + r, cg = lane < LN ? lane / DC : 0;
      AT acc = (AT)0;
      const int b1 = __ldg(d.ex_row + c + 1);
      int b = __ldg(d.ex_row + c) + sub;
      if constexpr (kRes) {
#pragma unroll 4
        for (; b < b1; b += wpr) {
          AT v[ST];
          V::group(vec + li_s[b - b0] * V::W, cg, v);
          const AT* Sb = Sr + (size_t)(b - b0) * EL + (lane < LN ? lane : 0);
#pragma unroll
          for (int s = 0; s < ST; ++s) acc = fma(Sb[s * LN], v[s], acc);
        }
      } else {
        // blocks from the L2 cache: UB blocks of a warp are in flight
        constexpr int UB = 8;
#pragma unroll 1
        for (; b < b1; b += UB * wpr) {
          AT w[UB][ST];
          int li[UB];
#pragma unroll
          for (int k = 0; k < UB; ++k) {
            const int bk = b + k * wpr;
            li[k] = bk < b1 ? __ldg(d.ex_lidx + bk) : 0;
#pragma unroll
            for (int s = 0; s < ST; ++s)
              w[k][s] = bk < b1 && lane < LN ? __ldg(Sx + (size_t)bk * EL + s * LN + lane) : (AT)0;
          }
#pragma unroll
          for (int k = 0; k < UB; ++k) {
            AT v[ST];
            V::group(vec + li[k] * V::W, cg, v);
#pragma unroll
            for (int s = 0; s < ST; ++s) acc = fma(w[k][s], v[s], acc);
          }
        }
      }
      const AT a1 = __shfl_down_sync(full, acc, DC), a2 = __shfl_down_sync(full, acc, 2 * DC);
      AT y = lane < DC ? (acc + a1) + a2 : (AT)0;
      if constexpr (Mo::kExtra) {
        // products with the camera-side edges' off-diagonal blocks, dealt over the row's
        // warps; two lanes per row of the block, half of its columns each
        constexpr int H0 = (DB + 1) / 2;
        const int half = lane / DB, a = lane % DB;
        AT t = (AT)0;
#pragma unroll 1
        for (int u = __ldg(d.xk_off + c) + sub; u < __ldg(d.xk_off + c + 1); u += wpr) {
          const int o = __ldg(d.ex_xl + u);
          if (o < 0) continue;   // unary edge: diagonal only
          const int code = __ldg(d.xk_list + u), side = code & 1;
          const AT* H = xH + (size_t)(code >> 1) * DB * DB;
          const int step = side ? DB : 1, base = side ? a : a * DB;
          if (half < 2) {
#pragma unroll
            for (int j = 0; j < H0; ++j) {
              const int k = half * H0 + j;
              if (k < DB) t += __ldg(H + base + k * step) * vec[o * V::W + V::at(k)];
            }
          }
        }
        t += __shfl_down_sync(full, t, DB);
        y += t;
      }
      if (lane < PW) part[((size_t)r * wpr + sub) * PW + lane] = y;
    }
    __syncthreads();
#pragma unroll 1
    for (int r = warp; r < nr; r += NW) {
      const int c = c0 + r;
      const AT* v = vec + __ldg(d.ex_lown + c) * V::W;
      if (lane < DB) {
        AT yi = (AT)0;
#pragma unroll
        for (int j = 0; j < DB; ++j) yi += Ss[(r * DB + lane) * DB + j] * v[V::at(j)];
        if (lane < PW)
#pragma unroll 1
          for (int s = 0; s < wpr; ++s) yi += part[((size_t)r * wpr + s) * PW + lane];
        ys[r * DB + lane] = yi;
        da[r * DB + lane] = v[V::at(lane)] * yi;
      }
    }
    __syncthreads();
    ++epoch;
    if (warp == 0) {
      const double pAp = group_sum(da, 0);
      int bad = 0;
      double al = 0.0;
      if (!restart) {
        bad = !(pAp > 0.0) || !isfinite(pAp);
        al = bad ? 0.0 : s_rz / pAp;
        if (bad) {   // p^T S p not positive: S is not positive definite at this damping
          if (pcg_it == 0) fail = 1;
          else breakdown = 1;
        }
      }
      if (lane == 0) {
        co[0] = (AT)al;
        co[1] = (AT)(sigma_s * al);
        fl[0] = bad;
      }
    }
    __syncthreads();
    if (fl[3]) return gave_up();
    if (fl[0]) break;
    const AT alpha = co[0], sa = co[1], sn = co[2];
    if (restart_every > 0 && !restart)
#pragma unroll 1
      for (int i = tid; i < nloc * V::W; i += kExThreads) xl[i] += sa * pl[i];
#pragma unroll 1
    for (int r = warp; r < nr; r += NW) {
      const int c = c0 + r, k = r * DB + lane;
      AT ri = (AT)0;
      if (lane < DB) {
        if (restart) {
          ri = gs[k] - ys[k];
        } else {
          xs[k] += sa * pl[__ldg(d.ex_lown + c) * V::W + V::at(lane)];
          ri = rs[k] * sn - alpha * ys[k];
        }
        rs[k] = ri;
      }
      __syncwarp();
      if (lane < DB) {
        AT zi = (AT)0;
#pragma unroll
        for (int j = 0; j < DB; ++j) zi += Ms[(r * DB + lane) * DB + j] * rs[r * DB + j];
        ex_post(zw + ((size_t)c * DB + lane) * ZW, zi, epoch + 1);
        da[k] = ri * zi;
        db[k] = ri * ri;
      }
    }
    __syncthreads();
    ++epoch;
    pcg_it += restart ? 0 : 1;
    products += 1;
    // stopping rules, beta and the normalisation (as pcg_update_finish): warp 0 from
    // r^T M r, warp 1 from |r|^2, while the others receive z
    if (warp == 0) {
      const double rz = group_sum(da, 0);
      const double be = restart ? 0.0 : rz / s_rz;
      s_rz = rz;
      if (lane == 0) {
        co[3] = (AT)be;
        fl[4] = !(rz > 0.0);
      }
    } else if (warp == 1) {
      const double rr = group_sum(db, 1);
      const double is = rr > 0.0 ? rsqrt(rr) : 0.0, n = rr > 0.0 ? rr * is : rr;
      if (restart) s_sigma = 1.0;
      const double rtrue = s_sigma * n;
      int done = 0, save = 0;
      if (ratio > 0.0) {
        if (rtrue < s_rmin) {
          s_rmin = rtrue;
          save = 1;
          have_best = 1;
        } else if (rtrue > ratio * s_rmin) {
          done = 1;
          use_best = 1;
        }
      }
      const bool tol = rtrue <= tol_abs, fin = isfinite(rtrue);
      if (tol || pcg_it >= max_it || !fin) done = 1;
      if (!fin) use_best = 1;
      s_rnorm = rtrue;
      double in = 1.0;
      if (normalize && n > 0.0) {
        in = is;
        s_sigma *= n;
      }
      if (lane == 0) {
        co[2] = (AT)in;
        is_s = in;
        sigma_s = s_sigma;
        fl[0] = done | (tol ? 2 : 0);
        fl[1] = (!restart && restart_every > 0 && pcg_it % restart_every == 0) ? 1 : 0;
        fl[2] = save;
      }
    } else {
#pragma unroll
      for (int k = 0; k < ZK; ++k)
        if (zo[k] >= 0) receive_z(zo[k], zr[k]);
    }
    __syncthreads();
    if (fl[3]) return gave_up();
    if (warp == 0) s_rz = s_rz * is_s * is_s;
    // r^T M r not positive before the tolerance is met: the preconditioned system is not
    // positive definite at this damping (after at least one step)
    if (fl[4] && !(fl[0] & 2)) breakdown = 1;
    if (fl[2]) {
      saved = 1;
#pragma unroll 1
      for (int i = tid; i < nr * DB; i += kExThreads) bs[i] = xs[i];
    }
    if (fl[0] || fl[4]) break;
  }
  if constexpr (kCluster) cluster_sync();   // no CTA's shared memory is written any more
#pragma unroll 1
  for (int i = tid; i < nr * DB; i += kExThreads) {
    gx[(size_t)c0 * DB + i] = xs[i];
    if (saved) reinterpret_cast<AT*>(d.xbest)[(size_t)c0 * DB + i] = bs[i];
  }
  if (rank != 0) return;
  if (tid == 0) {
    sc->rz = s_rz;
    sc->pcg_it = pcg_it;
    sc->pcg_products = products;
    sc->pcg_total += products;
    if (fail) sc->pcg_fail = 1;
    if (breakdown) sc->pcg_breakdown = 1;
    sc->pcg_done = 1;
  }
  if (tid == 32) {
    sc->sigma = s_sigma;
    sc->rnorm = s_rnorm;
    sc->rmin = s_rmin;
    if (use_best) sc->use_best = 1;
    if (have_best) sc->have_best = 1;
  }
}

}  // namespace gpo
