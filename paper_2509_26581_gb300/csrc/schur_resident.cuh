// The PCG of small mixed-precision systems in one launch, on the matrix-free product.
//
// A solve of a few dozen chunks is bound by its launches: a product and a camera kernel of
// a few microseconds each per iteration, started one after the other, and up to a group of
// iterations launched after the last one needed.  Here a problem's chunks are dealt to
// resident CTAs (kResChunks at most each) that keep the chunks' indices and point records
// in shared memory for the whole solve.  A camera's rows and vectors stay in the registers of
// one warp of the CTA that has the camera's unit of the camera half, and every CTA applies
// the stopping rules to its own copy of the solve's scalars, so an iteration passes three
// waits (products, p^T y, residual norms) and no ticket.  The problems of a batch do not
// wait for one another.  The sums and their order are those of k_spmv_pp, k_cam_apply and
// k_pcg_update (bit-identical results).
//
// Bound by latency: of some 26,000 clocks per iteration (20 cameras, 18 chunks) the product's
// four passes take 8,600, the three waits with their arrivals 7,400, the camera half and the
// update 5,500, the FP64 scalars 5,200.  Loops are kept rolled and the division in one copy:
// unrolled (75 KB of text against 52) an iteration took 30,600 clocks.  BF16 solves of two
// LM iterations: 20 cameras, 2,000 points 1,262 -> 850 us; 24 windows of 5 to 40 cameras at
// once 4,246 -> 3,423 us.
//
// Taken when the CTAs fit the device at once with at most kResChunks chunks each (the waits
// need every CTA resident).  Four chunks per CTA at three CTAs per SM measured 3,693 us on
// the 24 windows against 3,557 with two chunks at four.
#pragma once

namespace gpo {

// Shared memory: the passes' scratch, point solutions and slot directions of
// pipe_layout, then per chunk of the CTA the packed edge words, slot records and point
// records.
template <class Mo>
__host__ __device__ inline PipeLayout resident_layout(size_t sA, int ch_max, int np_max, int ns_max, int m) {
  PipeLayout L = pipe_layout<Mo>(sA, ch_max, np_max, ns_max);
  L.prec = L.bsize;                                  // inside a chunk's buffer
  L.bsize += (uint32_t)np_max * (uint32_t)((6 * sA + 8 + 15) & ~(size_t)15);
  L.size = L.buf + (uint32_t)m * L.bsize;
  return L;
}

// Arrival and wait of the solve's barriers: counts that k_cam_finalize clears and that only
// grow during the solve.  Bounded (kWaitClocks): false if the wait gave up.
__device__ __forceinline__ void res_arrive(unsigned int* bar) {
  __syncthreads();
  if (threadIdx.x == 0) red_add_release(bar, 1u);
}
__device__ __forceinline__ bool res_wait(const unsigned int* bar, unsigned int target) {
  __shared__ int ok;
  if (threadIdx.x == 0) {
    ok = 1;
    const long long t0 = sm_clock();
    while (ld_acquire(bar) < target) {
      if (sm_clock() - t0 > kWaitClocks) {
        ok = 0;
        break;
      }
    }
  }
  __syncthreads();
  return ok != 0;
}

// sum_partials' tree over n <= 32 values, one per lane of a warp (the same additions).
__device__ __forceinline__ double res_tree(double x, int n) {
#pragma unroll 1
  for (int s2 = tree_width(n) / 2; s2 > 0; s2 >>= 1) {
    const double y = __shfl_down_sync(0xffffffffu, x, s2);
    if ((int)(threadIdx.x & 31) < s2) x += y;
  }
  return x;
}

// One copy of the division and the root in the kernel: its text has to stay in the
// instruction cache from one iteration to the next.
static __device__ __noinline__ double res_div(double a, double b) { return a / b; }
static __device__ __noinline__ double res_sqrt(double a) { return sqrt(a); }

// seg_sum and component-wise point_sum with their loads issued ahead in batches (the same
// additions in the same order): a CTA or two per SM leave a serial chain of one load per
// addition exposed.
template <class AT>
__device__ __forceinline__ AT seg_sum_ahead(const AT* src, int a, int b) {
  AT s0 = (AT)0, s1 = (AT)0, s2 = (AT)0, s3 = (AT)0;
  int q = a;
#pragma unroll 1
  for (; q + 16 <= b; q += 16) {
    AT v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = src[q + i];
#pragma unroll
    for (int i = 0; i < 16; i += 4) { s0 += v[i]; s1 += v[i + 1]; s2 += v[i + 2]; s3 += v[i + 3]; }
  }
#pragma unroll 1
  for (; q + 4 <= b; q += 4) {
    s0 += src[q];
    s1 += src[q + 1];
    s2 += src[q + 2];
    s3 += src[q + 3];
  }
#pragma unroll 1
  for (; q < b; ++q) s0 += src[q];
  return (s0 + s1) + (s2 + s3);
}
template <class JT, class AT>
__device__ __forceinline__ void point_sum_ahead(const AT* v, int LD, int a, int b, AT (&u)[3]) {
  if constexpr (std::is_same<JT, float>::value) {
    point_sum<JT>(v, LD, a, b, u);
  } else {
    u[0] = u[1] = u[2] = (AT)0;
    int i = a;
#pragma unroll 1
    for (; i + 4 <= b; i += 4) {
      AT t[3][4];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
#pragma unroll
        for (int m = 0; m < 4; ++m) t[k][m] = v[k * LD + i + m];
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
#pragma unroll
        for (int k = 0; k < 3; ++k) u[k] += t[k][m];
      }
    }
#pragma unroll 1
    for (; i < b; ++i) {
#pragma unroll
      for (int k = 0; k < 3; ++k) u[k] += v[k * LD + i];
    }
  }
}

template <class Mo, class JT, int EPT>
__global__ void __launch_bounds__(kThreads, sizeof(JT) == 2 ? 4 : 3) k_pcg_resident(LaunchSet ls, int max_launch) {
  using AT = typename AccOf<JT>::T;
  constexpr int DC = Mo::DC, DB = Mo::DB, NJ = Mo::NJ, TB = Dims<Mo>::TB;
  constexpr size_t PRB = (6 * sizeof(AT) + 8 + 15) & ~(size_t)15;
  static_assert(kThreads == kCamPerBlock * 32 && !Mo::kExtra, "bundle adjustment, camera warps of the product's CTAs");
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ DevBA d;
  __shared__ Scalars s;                        // the solve's scalars, kept alike by every CTA
  __shared__ AT hm[kCamPerBlock / kApplySplit][2 * TB];
  __shared__ AT quarter[kCamPerBlock][DC];
  __shared__ double dots[kCamPerBlock];
  __shared__ AT coef[3];                       // alpha, sigma alpha, 1 / n
  __shared__ double num[6];                    // r^T z, |r|^2; beta, 1 / n, sigma, scaled r^T z
  __shared__ int bad_s;
  __shared__ unsigned int broke;
  __shared__ ChunkRange crs[kResChunks];
  __shared__ int own[3];                       // problem, rank in it, its CTAs
  if (threadIdx.x == 0) {
    int q = 0, b = blockIdx.x, n = 0;
#pragma unroll 1
    for (; q < ls.nprob; ++q) {
      const bool one = ls.nprob == 1, last = q + 1 == ls.nprob;
      const int nch = one ? ls.n_ch : (last ? ls.n_ch : ls.ch_base[q + 1]) - ls.ch_base[q];
      const int ncb = one ? ls.n_cb : (last ? ls.n_cb : ls.cb_base[q + 1]) - ls.cb_base[q];
      n = resident_ctas(nch, ncb, ls.res_m);
      if (b < n) break;
      b -= n;
    }
    own[0] = q; own[1] = b; own[2] = n;
  }
  __syncthreads();
  if (own[0] >= ls.nprob) return;
  bind_problem(d, ls.probs + own[0]);
  if (ls.ex && d.ex) return;                   // solved on its explicit Schur complement
  const int rank = own[1];
  const int chunk_ctas = (d.NCH + ls.res_m - 1) / ls.res_m, units = d.ncblk * kApplySplit;
#pragma unroll 1
  for (int i = threadIdx.x; i < (int)(sizeof(Scalars) / 4); i += kThreads)
    reinterpret_cast<int*>(&s)[i] = reinterpret_cast<const int*>(d.sc)[i];
  const int CH = ls.ch_max, LD = CH + 1, LP = ls.np_max + 1;
  const PipeLayout PL = resident_layout<Mo>(sizeof(AT), CH, ls.np_max, ls.ns_max, ls.res_m);
  AT* vv = reinterpret_cast<AT*>(smem);
  AT* tp = reinterpret_cast<AT*>(smem + PL.tp);
  AT* xs = reinterpret_cast<AT*>(smem + PL.xs);
  const int k0 = rank * ls.res_m, k1 = min(d.NCH, k0 + ls.res_m);
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    const ChunkRange cr = chunk_range(d, k);
    if (threadIdx.x == 0) crs[k - k0] = cr;
    unsigned char* B = smem + PL.buf + (k - k0) * PL.bsize;
#pragma unroll 1
    for (int i = threadIdx.x; i < cr.nE; i += kThreads) reinterpret_cast<uint32_t*>(B)[i] = d.e_meta[cr.e0 + i];
#pragma unroll 1
    for (int i = threadIdx.x; i < cr.nS; i += kThreads) reinterpret_cast<int4*>(B + PL.srec)[i] = d.slot_rec[cr.s0 + i];
    const uint4* pr = reinterpret_cast<const uint4*>(static_cast<const unsigned char*>(d.pt_rec) + (size_t)cr.p0 * PRB);
#pragma unroll 1
    for (int i = threadIdx.x; i < cr.nP * (int)(PRB / 16); i += kThreads) reinterpret_cast<uint4*>(B + PL.prec)[i] = pr[i];
  }
  // the CTA's unit of the camera half (two cameras, four warps each; as in cam_apply_body),
  // whose first warps also keep their camera's rows and vectors for the whole solve
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp % kApplySplit;
  const bool unit = rank < units;
  const int c = unit ? unit_camera(rank / kApplySplit, rank % kApplySplit) : d.C;
  const int2 sr = c < d.C ? make_int2(d.cam_s_off[c], d.cam_s_off[c + 1]) : make_int2(0, 0);
  const bool lead = c < d.C && q == 0 && lane < DB;
  AT g0 = (AT)0, x = (AT)0, xb = (AT)0, r = (AT)0, z = (AT)0, p = (AT)0;
  const size_t o = lead ? DB * (size_t)c + lane : 0;
  AT* const hb = hm[warp / kApplySplit];               // the camera's damped block, then its inverse
  if (c < d.C && q == 0) {
#pragma unroll 1
    for (int j = lane; j < TB; j += 32) {
      hb[j] = reinterpret_cast<const AT*>(d.Hcl)[(size_t)c * TB + j];
      hb[TB + j] = reinterpret_cast<const AT*>(d.Minv)[(size_t)c * TB + j];
    }
  }
  if (lead) {
    g0 = reinterpret_cast<const AT*>(d.g)[o];
    x = reinterpret_cast<const AT*>(d.x)[o];
    xb = reinterpret_cast<const AT*>(d.xbest)[o];
    r = reinterpret_cast<const AT*>(d.r)[o];
    z = reinterpret_cast<const AT*>(d.z)[o];
    p = reinterpret_cast<const AT*>(s.pidx ? d.p2 : d.p)[o];
  }
  const JT* Jg = reinterpret_cast<const JT*>(d.J);
  AT* partV = reinterpret_cast<AT*>(d.partV);
  double* const upart = d.cblk_part + 2 * (size_t)units;   // [camera][r^T z, |r|^2]
  unsigned int* const bar = d.sc->bar;
  __syncthreads();
  if (threadIdx.x == 0) coef[2] = sc_inv_n<AT>(&s);
  if (!s.active || s.pcg_done) return;
  if (*static_cast<volatile int*>(ls.err)) {   // an earlier wait gave up: no step without a solve
    if (threadIdx.x == 0) d.sc->active = 0;
    return;
  }
  bool ok = true;
#pragma unroll 1
  for (int it = 0; it < max_launch; ++it) {
    const int restart = s.restart;
    const AT beta = restart ? (AT)0 : sc_beta<AT>(&s), inv_n = restart ? (AT)1 : sc_inv_n<AT>(&s);
    const AT* zv = reinterpret_cast<const AT*>(restart ? d.x : d.z);
    const AT* pold = restart ? zv : reinterpret_cast<const AT*>(s.pidx ? d.p2 : d.p);
    // ---- the product over the CTA's chunks (the passes of k_spmv_pp)
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
      const ChunkRange cr = crs[k - k0];
      const unsigned char* B = smem + PL.buf + (k - k0) * PL.bsize;
      const uint32_t* meta = reinterpret_cast<const uint32_t*>(B);
      const int4* srec = reinterpret_cast<const int4*>(B + PL.srec);
      uint4 raw[EPT][JTiles<JT, NJ>::Q];   // the threads' rows, read once for passes 1 and 3
#pragma unroll
      for (int m = 0; m < EPT; ++m) {
        const int i = threadIdx.x + m * kThreads;
        if (i < cr.nE) {
#pragma unroll
          for (int t = 0; t < JTiles<JT, NJ>::Q; ++t)
            raw[m][t] = reinterpret_cast<const uint4*>(Jg)[JTiles<JT, NJ>::piece((size_t)(cr.e0 + i), t)];
        }
      }
#pragma unroll 1
      for (int w = threadIdx.x; w < cr.nS * DC; w += kThreads) {
        const int sl = w / DC, j = w - sl * DC;
        const size_t oc = DB * (size_t)srec[sl].z + j;
        xs[w] = (zv[oc] + beta * pold[oc]) * inv_n;
      }
      __syncthreads();
#pragma unroll
      for (int m = 0; m < EPT; ++m) {
        const int i = threadIdx.x + m * kThreads;
        if (i >= cr.nE) break;
        AT row[NJ], a[3];
        load_row<NJ>(reinterpret_cast<const JT*>(raw[m]), row);
        edge_point_term<Mo>(row, xs + DC * (int)((meta[i] >> 10) & 1023u), a);
#pragma unroll
        for (int j = 0; j < 3; ++j) vv[j * LD + i] = a[j];
      }
      __syncthreads();
#pragma unroll 1
      for (int j = threadIdx.x; j < cr.nP; j += kThreads) {
        const AT* hv = reinterpret_cast<const AT*>(B + PL.prec + (size_t)j * PRB);
        const int* se = reinterpret_cast<const int*>(B + PL.prec + (size_t)j * PRB + 6 * sizeof(AT));
        AT u[3], t[3];
        point_sum_ahead<JT>(vv, LD, se[0], se[1], u);
        mul3(hv, u, t);
#pragma unroll
        for (int l = 0; l < 3; ++l) tp[l * LP + j] = t[l];
      }
      __syncthreads();
#pragma unroll
      for (int m = 0; m < EPT; ++m) {
        const int i = threadIdx.x + m * kThreads;
        if (i >= cr.nE) break;
        const uint32_t w = meta[i];
        const int pl = (int)(w >> 20), pos = (int)(w & 1023u);
        AT row[NJ], v[DC];
        load_row<NJ>(reinterpret_cast<const JT*>(raw[m]), row);
        edge_camera_term<Mo>(row, tp[pl], tp[LP + pl], tp[2 * LP + pl], v);
#pragma unroll
        for (int j = 0; j < DC; ++j) vv[j * LD + pos] = v[j];
      }
      __syncthreads();
#pragma unroll 1
      for (int w = threadIdx.x; w < cr.nS * DC; w += kThreads) {
        const int sl = w / DC, comp = w - sl * DC;
        const int4 r4 = srec[sl];
        partV[(size_t)r4.w * DC + comp] = seg_sum_ahead(vv + comp * LD, r4.x, r4.y);
      }
      __syncthreads();   // vv and xs are free again
    }
    if (k0 < k1) res_arrive(bar);
    if (unit) {
      // ---- the camera half
      AT hrow[DB];   // read ahead of the wait
#pragma unroll
      for (int j = 0; j < DB; ++j) hrow[j] = lead ? hb[sym_idx(DB, lane, j)] : (AT)0;
      if (!(ok = res_wait(bar, (unsigned)(chunk_ctas * (it + 1) + ls.debug_wait)))) break;
      AT acc[DC];
#pragma unroll
      for (int k = 0; k < DC; ++k) acc[k] = (AT)0;
#pragma unroll 2
      for (int t = sr.x + q * 32 + lane; t < sr.y; t += 32 * kApplySplit) {
        const AT* src = partV + (size_t)t * DC;
#pragma unroll
        for (int k = 0; k < DC; ++k) acc[k] += src[k];
      }
#pragma unroll
      for (int h = 16; h > 0; h >>= 1) {
#pragma unroll
        for (int k = 0; k < DC; ++k) acc[k] += __shfl_down_sync(0xffffffffu, acc[k], h);
      }
      if (lane == 0) {
#pragma unroll
        for (int k = 0; k < DC; ++k) quarter[warp][k] = acc[k];
      }
      __syncthreads();
      AT pi = (AT)0, yi = (AT)0;
      if (c < d.C && q == 0) {
        AT sv = (AT)0;
        if (lane < DC) {
          sv = quarter[warp][lane];
          for (int j = 1; j < kApplySplit; ++j) sv += quarter[warp + j][lane];
        }
        const AT zs = restart ? x : z, ps = restart ? x : p;
        pi = lane < DB ? (zs + beta * ps) * inv_n : (AT)0;
        if (s.save_best) xb = x;
#pragma unroll
        for (int j = 0; j < DB; ++j) {
          const AT pj = __shfl_sync(0xffffffffu, pi, j);
          if (lane < DB) yi += hrow[j] * pj;
        }
        if (lane < DB) {
          yi -= sv;
          if (!restart) {
            p = pi;
            reinterpret_cast<AT*>(s.pidx ? d.p : d.p2)[o] = pi;
          }
        }
      }
      // ---- alpha from all units' p^T y (a restart's product needs none, but its arrivals
      // count: they show that every unit has read the last update's norms in upart, which
      // the update below overwrites; units without chunks arrive nowhere else before it)
      if (!restart) {
        AT dot = lead ? pi * yi : (AT)0;
#pragma unroll
        for (int h = 16; h > 0; h >>= 1) dot += __shfl_down_sync(0xffffffffu, dot, h);
        if (lane == 0) dots[warp] = (double)dot;
        __syncthreads();
        if (threadIdx.x == 0) {
          double a = 0.0;
          for (int w = 0; w < kCamPerBlock; w += kApplySplit) a += dots[w];   // the other warps' are zero
          d.cblk_part[2 * rank] = a;
        }
      }
      res_arrive(bar + 1);
      if (!(ok = res_wait(bar + 1, (unsigned)units * (unsigned)(it + 1)))) break;
      if (!restart) {
        double pAp = 0.0;   // by two warps, for the two coefficients
        if (units > 32) pAp = sum_partials_first(d.cblk_part, units);
        else if (warp < 2) pAp = res_tree(lane < units ? d.cblk_part[2 * lane] : 0.0, units);
        if (lane == 0 && warp < 2) {
          const int bad = !(pAp > 0.0) || !isfinite(pAp);
          const double alpha = bad ? 0.0 : res_div(s.rz, pAp);
          if (warp == 0) {
            s.pAp = pAp;
            s.alpha = alpha;
            coef[0] = (AT)alpha;
            if (bad && rank == 0) bar[3] = 1u;   // read by every CTA after the update's arrivals
            bad_s = bad;
          } else {
            coef[1] = (AT)(s.sigma * alpha);
          }
        }
      } else if (threadIdx.x == 0) {
        bad_s = 0;
      }
      __syncthreads();
      // ---- the update of the unit's cameras
      if (q == 0) {
        AT rz_c = (AT)0, rr_c = (AT)0, zi = (AT)0, mrow[DB];
#pragma unroll
        for (int j = 0; j < DB; ++j) mrow[j] = lead ? hb[TB + sym_idx(DB, lane, j)] : (AT)0;
        if (lead && !bad_s) {
          if (restart) {
            r = g0 - yi;
          } else {
            x = x + coef[1] * p;
            r = r * coef[2] - coef[0] * yi;
          }
        }
#pragma unroll
        for (int j = 0; j < DB; ++j) {
          const AT rj = __shfl_sync(0xffffffffu, r, j);
          if (lane < DB) zi += mrow[j] * rj;
        }
        if (lead && !bad_s) {
          z = zi;
          rz_c = r * zi;
          rr_c = r * r;
          reinterpret_cast<AT*>(d.z)[o] = z;
          reinterpret_cast<AT*>(d.x)[o] = x;
        }
#pragma unroll
        for (int h = 16; h > 0; h >>= 1) {
          rz_c += __shfl_down_sync(0xffffffffu, rz_c, h);
          rr_c += __shfl_down_sync(0xffffffffu, rr_c, h);
        }
        if (lane == 0) {
          const int uc = unit_camera(rank / kApplySplit, rank % kApplySplit);
          *reinterpret_cast<double2*>(upart + 2 * (size_t)uc) = make_double2((double)rz_c, (double)rr_c);
        }
      }
      res_arrive(bar + 2);
    }
    if (!(ok = res_wait(bar + 2, (unsigned)units * (unsigned)(it + 1)))) break;
    // ---- the stopping rules, by every CTA on the same sums.  One FP64 warp instruction
    // takes a sub-partition some 70 clocks, so the two sums, the divisions and the rules are
    // spread over four warps (each takes the root it needs).
    double rz = 0.0, rr = 0.0;
    if (threadIdx.x == kThreads - 32) broke = *static_cast<volatile unsigned int*>(bar + 3);
    if (d.ncblk <= 32) {
      if (warp < 2) {
        double a = 0.0;
        if (lane < d.ncblk) {
          double v[kCamPerBlock];
#pragma unroll
          for (int w = 0; w < kCamPerBlock; ++w) v[w] = upart[2 * (lane * kCamPerBlock + w) + warp];
#pragma unroll
          for (int w = 0; w < kCamPerBlock; ++w) a += v[w];
        }
        a = res_tree(a, d.ncblk);
        if (lane == 0) num[warp] = a;
      }
      __syncthreads();
      rz = num[0];
      rr = num[1];
    } else {
      // block sums first (into the passes' scratch, unused here), then their tree
      double* blk = reinterpret_cast<double*>(vv);
#pragma unroll 1
      for (int i = threadIdx.x; i < d.ncblk; i += kThreads) {
        double a = 0.0, b = 0.0;
#pragma unroll 1
        for (int w = 0; w < kCamPerBlock; ++w) {
          const double2 v = reinterpret_cast<const double2*>(upart)[i * kCamPerBlock + w];
          a += v.x; b += v.y;
        }
        blk[2 * i] = a;
        blk[2 * i + 1] = b;
      }
      __syncthreads();
      sum_partials(blk, d.ncblk, rz, rr);
    }
    SolveState st;
    RuleFlags fl;
    if (lane == 0 && warp < 4) {
      st.load(&s);
      const double n = warp == 1 ? 0.0 : res_sqrt(rr);
      const bool norm = st.normalize && n > 0.0;
      if (warp == 0) {
        fl = pcg_flags(st, rz, n, restart);
      } else if (warp == 1) {
        num[2] = restart ? 0.0 : res_div(rz, st.rz_old);   // a restart starts the direction from z
      } else if (warp == 2) {
        const double sg = restart ? 1.0 : st.sigma;
        num[3] = norm ? res_div(1.0, n) : 1.0;
        num[4] = norm ? sg * n : sg;
      } else {
        num[5] = norm ? res_div(rz, n * n) : rz;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      if (broke) {   // p^T S p not positive: S is not positive definite at this damping
        s.pcg_done = 1;
        if (s.pcg_it == 0) s.pcg_fail = 1;
        else s.pcg_breakdown = 1;
      } else {
        pcg_record(&s, st, fl, num[2], num[3], num[4], num[5], restart);
        coef[2] = sc_inv_n<AT>(&s);
      }
    }
    __syncthreads();
    if (s.pcg_done) break;
  }
  if (!ok) {
    if (threadIdx.x == 0) {
      atomicExch(ls.err, 1);
      d.sc->active = 0;   // the rest of the iteration, and the iterations after it, leave the problem alone
    }
    return;
  }
  if (lead) {
    reinterpret_cast<AT*>(d.r)[o] = r;
    reinterpret_cast<AT*>(d.xbest)[o] = xb;
  }
  if (rank == 0 && threadIdx.x == 0) {
    Scalars* sc = d.sc;
    sc->rz = s.rz; sc->pAp = s.pAp; sc->alpha = s.alpha; sc->beta = s.beta; sc->inv_n = s.inv_n;
    sc->sigma = s.sigma; sc->rnorm = s.rnorm; sc->rmin = s.rmin;
    sc->beta_f = s.beta_f; sc->inv_n_f = s.inv_n_f;
    sc->pcg_it = s.pcg_it; sc->pcg_done = s.pcg_done; sc->pcg_total = s.pcg_total; sc->pcg_products = s.pcg_products;
    sc->use_best = s.use_best; sc->save_best = s.save_best; sc->have_best = s.have_best;
    sc->pidx = s.pidx; sc->restart = s.restart;
    sc->pcg_fail = s.pcg_fail; sc->pcg_breakdown = s.pcg_breakdown;
    if (s.pcg_done) atomicSub(ls.running, 1);
  }
}

}  // namespace gpo
