// Batched solves and the serving loop: many independent graphs share every kernel
// launch.  A launch set over the graphs lists their descriptors and which CTA belongs
// to which graph (chunks, camera blocks, point blocks); each graph keeps its own LM
// and PCG state, so a graph's result does not depend on the other graphs it runs with.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <deque>
#include <map>
#include <new>
#include <unordered_map>
#include <vector>

#include "graph.h"

using namespace gpo_host;

namespace {

__global__ void k_put_scalars(const DevBA* probs, const Scalars* src, int n) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) *probs[q].sc = src[q];
}

__global__ void k_get_scalars(const DevBA* probs, Scalars* dst, int n) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) dst[q] = *probs[q].sc;
}

// Device tables of a launch set over several finalized graphs (stream-ordered memory).
struct BatchSet {
  gpo::LaunchSet ls{};
  char* mem = nullptr;
  Scalars* staging = nullptr;    // device [n]
  std::vector<int4> grids;       // problems whose PCG takes a whole grid (ls.xg_host)
  int n = 0;

  void release(cudaStream_t st) {
    if (mem) cudaFreeAsync(mem, st);
    mem = nullptr;
    n = 0;
  }
};

// ex_of[q]: problem q solves on its explicit Schur complement (empty: only costs are computed).
gpo_status build_set(gpo_graph* owner, const std::vector<gpo_graph*>& gs, const std::vector<char>& ex_of, BatchSet& out) {
  const int n = (int)gs.size();
  std::vector<DevBA> probs(n);
  std::vector<int> ch_prob, cb_prob, pb_prob, ch_base(n), cb_base(n), pb_base(n);
  std::vector<int> xf_prob, xd_prob, cl_prob, xf_base(n), xd_base(n);   // explicit Schur complement
  int ch_max = 32, ns_max = 1, np_max = 1, mf = 0, ex = 0, cl_smem = 0;
  out.grids.clear();
  for (int q = 0; q < n; ++q) {
    const gpo_graph* g = gs[q];
    probs[q] = g->dev;
    probs[q].ex = !ex_of.empty() && ex_of[q];
    ch_base[q] = (int)ch_prob.size();
    cb_base[q] = (int)cb_prob.size();
    pb_base[q] = (int)pb_prob.size();
    ch_prob.insert(ch_prob.end(), g->ls.n_ch, q);
    cb_prob.insert(cb_prob.end(), g->ls.n_cb, q);
    pb_prob.insert(pb_prob.end(), g->ls.n_pb, q);
    ch_max = std::max(ch_max, g->ls.ch_max);
    ns_max = std::max(ns_max, g->ls.ns_max);
    np_max = std::max(np_max, g->ls.np_max);
    xf_base[q] = (int)xf_prob.size();
    xd_base[q] = (int)xd_prob.size();
    if (!probs[q].ex) {
      mf = 1;
      continue;
    }
    ex = 1;
    xf_prob.insert(xf_prob.end(), g->ls.n_xf, q);
    xd_prob.insert(xd_prob.end(), g->ls.n_xd, q);
    if (g->ex_cluster) {
      cl_prob.push_back(q);
      cl_smem = std::max(cl_smem, g->ex_grid.z);
    } else {
      out.grids.push_back(make_int4(q, g->ex_grid.y, g->ex_grid.z, g->ex_grid.w));
    }
  }
  auto al = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t b_probs = al(n * sizeof(DevBA)), b_stage = al(n * sizeof(Scalars));
  const size_t b_ch = al(std::max<size_t>(1, ch_prob.size()) * 4), b_cb = al(std::max<size_t>(1, cb_prob.size()) * 4);
  const size_t b_pb = al(std::max<size_t>(1, pb_prob.size()) * 4), b_base = al(n * 4);
  const size_t b_xf = al(std::max<size_t>(1, xf_prob.size()) * 4), b_xd = al(std::max<size_t>(1, xd_prob.size()) * 4);
  const size_t total = b_probs + b_stage + b_ch + b_cb + b_pb + b_xf + b_xd + 6 * b_base + 256;
  cudaStream_t st = owner->stream;
  char* mem = nullptr;
  GPO_CUDA(owner, cudaMallocAsync(reinterpret_cast<void**>(&mem), total, st));
  // one host image, one copy (staged before the call returns: the memory is pageable)
  std::vector<char> img(total, 0);
  size_t at = 0;
  auto take = [&](size_t b) {
    const size_t r = at;
    at += b;
    return r;
  };
  auto put = [&](size_t b, const void* src, size_t n_bytes) {
    const size_t r = take(b);
    if (n_bytes) std::memcpy(img.data() + r, src, n_bytes);
    return mem + r;
  };
  auto put_i = [&](size_t b, const std::vector<int>& v) { return reinterpret_cast<int*>(put(b, v.data(), v.size() * 4)); };
  DevBA* probs_d = reinterpret_cast<DevBA*>(put(b_probs, probs.data(), n * sizeof(DevBA)));
  Scalars* stage_d = reinterpret_cast<Scalars*>(mem + take(b_stage));
  int *ch_d = put_i(b_ch, ch_prob), *cb_d = put_i(b_cb, cb_prob), *pb_d = put_i(b_pb, pb_prob);
  int *chb_d = put_i(b_base, ch_base), *cbb_d = put_i(b_base, cb_base), *pbb_d = put_i(b_base, pb_base);
  int* running_d = reinterpret_cast<int*>(mem + take(256));
  int *xf_d = put_i(b_xf, xf_prob), *xd_d = put_i(b_xd, xd_prob);
  int *xfb_d = put_i(b_base, xf_base), *xdb_d = put_i(b_base, xd_base), *cl_d = put_i(b_base, cl_prob);
  GPO_CUDA(owner, cudaMemcpyAsync(mem, img.data(), total, cudaMemcpyHostToDevice, st));
  gpo::LaunchSet ls{};
  ls.probs = probs_d;
  ls.ch_prob = ch_d; ls.ch_base = chb_d;
  ls.cb_prob = cb_d; ls.cb_base = cbb_d;
  ls.pb_prob = pb_d; ls.pb_base = pbb_d;
  ls.running = running_d;
  ls.err = running_d + 1;
  ls.work = running_d + 2;
  ls.spmv_variant = owner->desc.spmv_variant;
  ls.nprob = n;
  ls.n_ch = (int)ch_prob.size();
  ls.n_cb = (int)cb_prob.size();
  ls.n_pb = (int)pb_prob.size();
  ls.ch_max = ch_max;
  ls.ns_max = ns_max;
  ls.np_max = np_max;
  ls.ex = ex; ls.mf = mf;
  ls.xf_prob = xf_d; ls.xf_base = xfb_d;
  ls.xd_prob = xd_d; ls.xd_base = xdb_d;
  ls.cl_prob = cl_d;
  ls.xg_host = out.grids.data();
  ls.n_xf = (int)xf_prob.size();
  ls.n_xd = (int)xd_prob.size();
  ls.n_cl = (int)cl_prob.size();
  ls.n_xg = (int)out.grids.size();
  ls.cl_smem = cl_smem;
  std::vector<int2> sizes;
  for (const gpo_graph* g : gs) sizes.push_back(make_int2(g->ls.n_ch, g->ls.n_cb));
  if (mf && !ex_of.empty() && !cb_prob.empty()) plan_resident(*gs[0]->ks, owner->prec, sizes, ls);
  out.ls = ls;
  out.mem = mem;
  out.staging = stage_d;
  out.n = n;
  return GPO_OK;
}

gpo_status put_scalars(gpo_graph* owner, BatchSet& bs, const std::vector<Scalars>& sc) {
  GPO_CUDA(owner, cudaMemcpyAsync(bs.staging, sc.data(), sc.size() * sizeof(Scalars),
                                  cudaMemcpyHostToDevice, owner->stream));   // pageable: staged before the call returns
  k_put_scalars<<<(bs.n + 127) / 128, 128, 0, owner->stream>>>(bs.ls.probs, bs.staging, bs.n);
  GPO_CUDA(owner, cudaGetLastError());
  return GPO_OK;
}

gpo_status get_scalars(gpo_graph* owner, BatchSet& bs, std::vector<Scalars>& sc) {
  sc.resize(bs.n);
  k_get_scalars<<<(bs.n + 127) / 128, 128, 0, owner->stream>>>(bs.ls.probs, bs.staging, bs.n);
  GPO_CUDA(owner, cudaGetLastError());
  GPO_CUDA(owner, cudaMemcpyAsync(sc.data(), bs.staging, bs.n * sizeof(Scalars), cudaMemcpyDeviceToHost,
                                  owner->stream));
  GPO_CUDA(owner, cudaStreamSynchronize(owner->stream));
  return GPO_OK;
}

// After a wait gave up: switches the problems whose solve was lost on again (their state is
// the one before the iteration).  ran[q]: problem q has taken its step.
gpo_status rearm(gpo_graph* owner, BatchSet& bs, bool stepped, std::vector<char>& ran) {
  std::vector<Scalars> sc;
  if (gpo_status s = get_scalars(owner, bs, sc); s != GPO_OK) return s;
  for (int q = 0; q < bs.n; ++q) {
    ran[q] = stepped && sc[q].active;
    sc[q].active = 1;
  }
  return put_scalars(owner, bs, sc);
}

void report_from(const Scalars& s, double initial_cost, gpo_report* r) {
  r->initial_cost = initial_cost;
  r->final_cost = s.cost;
  r->final_lambda = s.lambda;
  r->iterations = s.iter;
  r->accepted = s.n_accepted;
  r->pcg_iters_total = s.pcg_total;
  r->reserved0 = 0;
  r->final_nu = s.nu;
}

// Device-memory pool of a server: arenas of retired graphs are kept (keyed by size,
// 1 MiB granularity) and handed to the next admitted graphs, so the serving loop does
// not pay cudaMalloc / cudaFree (which synchronises the device) per request.
struct DevPool {
  std::multimap<size_t, void*> free_blocks;
  std::unordered_map<void*, size_t> block_size;
  size_t held = 0;   // bytes obtained from cudaMalloc and not yet returned

  void trim() {
    for (auto& kv : free_blocks) {
      cudaFree(kv.second);
      held -= kv.first;
      block_size.erase(kv.second);
    }
    free_blocks.clear();
  }
};

void* pool_alloc(size_t bytes, void* ctx) {
  DevPool* pool = static_cast<DevPool*>(ctx);
  const size_t b = (bytes + (size_t(1) << 20) - 1) & ~((size_t(1) << 20) - 1);
  auto it = pool->free_blocks.lower_bound(b);
  if (it != pool->free_blocks.end() && it->first <= 2 * b) {   // reuse a block at most twice as big
    void* p = it->second;
    pool->free_blocks.erase(it);
    return p;
  }
  void* p = nullptr;
  if (cudaMalloc(&p, b) != cudaSuccess) {
    cudaGetLastError();
    pool->trim();
    if (cudaMalloc(&p, b) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
  }
  pool->block_size[p] = b;
  pool->held += b;
  return p;
}

void pool_free(void* p, void* ctx) {
  DevPool* pool = static_cast<DevPool*>(ctx);
  auto it = pool->block_size.find(p);
  if (it != pool->block_size.end()) pool->free_blocks.emplace(it->second, p);
}

}  // namespace

// ============================================================== serving loop state

struct gpo_server {
  gpo_server_desc desc{};
  gpo_graph* owner = nullptr;     // empty graph carrying the stream, flags and profiler
  struct Req {
    gpo_graph* g;
    int max_iters;
    gpo_lm_params prm;
    int64_t ticket;
    int done_iters;
    size_t bytes;
    double initial_cost;
    DampingRange damping;
    Scalars start;          // the parameters
    double limit;           // explicit_up_to
    bool ex;                // solves on its explicit Schur complement
    gpo_graph_desc saved;   // the graph's own stream and allocator, restored at retirement
    bool adopted_stream;
  };
  DevPool pool;
  std::deque<Req> queue;
  std::vector<Req> resident;
  std::unordered_map<int64_t, gpo_report> finished;
  size_t used = 0;
  int64_t next_ticket = 0;
  BatchSet set;
  bool dirty = true;
  int64_t steps = 0;
};

extern "C" {

gpo_status gpo_optimize_batch(gpo_graph* const* graphs, int32_t n, int32_t max_iters,
                              const gpo_lm_params* params, gpo_report* reports) {
  if (!graphs || n <= 0 || max_iters < 0) return GPO_ERR_ARG;
  gpo_graph* owner = graphs[0];
  if (!owner) return GPO_ERR_ARG;
  for (int i = 0; i < n; ++i) {
    if (!graphs[i]) return fail(owner, GPO_ERR_ARG, "graph %d is null", i);
    if (graphs[i]->prec != owner->prec || graphs[i]->desc.device != owner->desc.device)
      return fail(owner, GPO_ERR_ARG, "graphs of a batch must share precision and device");
    if (graphs[i]->desc.spmv_variant == 4)
      return fail(owner, GPO_ERR_UNSUPPORTED, "graphs with dynamic Jacobians are solved alone");
    for (int j = 0; j < i; ++j)
      if (graphs[j] == graphs[i]) return fail(owner, GPO_ERR_ARG, "graph %d appears twice", i);
  }
  GPO_CUDA(owner, cudaSetDevice(owner->desc.device));
  for (int i = 0; i < n; ++i) {
    gpo_status s = finalize(graphs[i]);
    if (s != GPO_OK) {
      if (graphs[i] != owner) owner->err = graphs[i]->err;
      return s;
    }
    if (graphs[i]->ks != owner->ks)
      return fail(owner, GPO_ERR_ARG, "graphs of a batch must share the camera kind");
  }
  const gpo_lm_params prm = params_or_default(params);
  if (!(prm.initial_damping > 0.0)) return fail(owner, GPO_ERR_ARG, "initial damping must be positive");
  std::vector<gpo_graph*> gs(graphs, graphs + n);
  BatchSet bs;
  gpo_status s = join_uploads(owner, gs);
  if (s != GPO_OK) return s;
  std::vector<Scalars> sc(n);
  std::vector<DampingRange> damping(n);
  std::vector<double> limit(n);
  for (int i = 0; i < n; ++i) {
    graphs[i]->cost_valid = graphs[i]->state_same = false;   // until the call has ended well
    fill_scalars(graphs[i], prm, prm.initial_damping, sc[i]);
    sc[i].full = 0;   // shared launches run the Schur form
    graphs[i]->pcg_full = 0;
    damping[i].start(sc[i]);
    limit[i] = explicit_up_to(graphs[i], prm);
  }
  const Scalars first = sc[0];   // the parameters, alike for all
  auto choice = [&] {
    std::vector<char> ex(n);
    for (int i = 0; i < n; ++i) ex[i] = damping[i].within(limit[i]) > 0;
    return ex;
  };
  std::vector<char> ex = choice();
  if ((s = build_set(owner, gs, ex, bs)) != GPO_OK) return s;
  int max_it = 1;
  for (auto& x : sc) max_it = std::max(max_it, x.max_it);
  if ((s = put_scalars(owner, bs, sc)) == GPO_OK && (s = launch_initial_cost(owner, bs.ls)) == GPO_OK &&
      (s = get_scalars(owner, bs, sc)) == GPO_OK) {
    std::vector<double> F0(n);
    for (int i = 0; i < n; ++i) {
      F0[i] = sc[i].cost;
      if (!std::isfinite(F0[i])) {
        s = fail(owner, GPO_ERR_NUMERIC, "graph %d: initial cost is not finite (%g)", i, F0[i]);
        break;
      }
    }
    if (s == GPO_OK && (s = ensure_runtime(owner)) == GPO_OK) s = begin_solves(owner, bs.ls);
    for (int it = 0; s == GPO_OK && it < max_iters; ++it) {
      owner->cur_lm_iter = -1;
      bool read = false;
      for (int i = 0; i < n; ++i) read |= damping[i].within(limit[i]) < 0;
      if (read) {   // a damping may have crossed its limit
        if ((s = get_scalars(owner, bs, sc)) != GPO_OK) break;
        for (int i = 0; i < n; ++i) damping[i].start(sc[i]);
      }
      if (std::vector<char> now = choice(); now != ex) {
        ex = std::move(now);
        bs.release(owner->stream);
        if ((s = build_set(owner, gs, ex, bs)) != GPO_OK || (s = begin_solves(owner, bs.ls)) != GPO_OK) break;
      }
      for (auto& d : damping) d.iteration(first);
      bs.ls.debug_wait = std::any_of(gs.begin(), gs.end(), [&](const gpo_graph* g) { return held(g, it); });
      if ((s = solve_system(owner, bs.ls, max_it, false)) != GPO_OK) break;
      s = finish_iteration(owner, bs.ls);
    }
    if (s == GPO_OK && (s = get_scalars(owner, bs, sc)) == GPO_OK)
      for (int i = 0; s == GPO_OK && i < n; ++i) s = lost_solve(owner, sc[i]);
    if (s == GPO_OK) {
      for (int i = 0; i < n; ++i) {
        graphs[i]->last_cost = sc[i].cost;
        graphs[i]->cost_valid = true;
        graphs[i]->hist.clear();
        if (reports) report_from(sc[i], F0[i], &reports[i]);
      }
    }
  }
  if (owner->prof.on) {
    cudaStreamSynchronize(owner->stream);
    prof_resolve(owner);
  }
  bs.release(owner->stream);
  if (cudaStreamSynchronize(owner->stream) == cudaSuccess)
    for (int i = 0; i < n; ++i) graphs[i]->uploading = false;
  return s;
}

gpo_status gpo_server_desc_default(gpo_server_desc* out) {
  if (!out) return GPO_ERR_ARG;
  std::memset(out, 0, sizeof(*out));
  out->precision = GPO_FP32_BF16;
  out->max_resident = 1024;
  return GPO_OK;
}

gpo_status gpo_server_create(const gpo_server_desc* desc, gpo_server** out) {
  if (!desc || !out) return GPO_ERR_ARG;
  if (desc->max_resident <= 0) return GPO_ERR_ARG;
  gpo_graph_desc gd;
  gpo_graph_desc_default(&gd);
  gd.precision = desc->precision;
  gd.device = desc->device;
  gd.cuda_stream = desc->cuda_stream;
  gpo_graph* owner = nullptr;
  gpo_status s = gpo_graph_create(&gd, &owner);
  if (s != GPO_OK) return s;
  if ((s = ensure_runtime(owner)) != GPO_OK) {
    gpo_graph_destroy(owner);
    return s;
  }
  gpo_server* sv = new (std::nothrow) gpo_server();
  if (!sv) {
    gpo_graph_destroy(owner);
    return GPO_ERR_OOM;
  }
  sv->desc = *desc;
  sv->owner = owner;
  *out = sv;
  return GPO_OK;
}

// Gives a graph back its own stream and allocator after the server is done with it.
static void restore_graph(gpo_server::Req& r) {
  r.g->desc.alloc = r.saved.alloc;
  r.g->desc.free = r.saved.free;
  r.g->desc.alloc_ctx = r.saved.alloc_ctx;
  if (r.adopted_stream) r.g->stream = nullptr;
}

gpo_status gpo_server_destroy(gpo_server* sv) {
  if (!sv) return GPO_OK;
  cudaStreamSynchronize(sv->owner->stream);
  for (auto& r : sv->resident) {
    release_device(r.g);
    restore_graph(r);
  }
  for (auto& r : sv->queue) restore_graph(r);
  sv->set.release(sv->owner->stream);
  cudaStreamSynchronize(sv->owner->stream);
  sv->pool.trim();
  gpo_graph_destroy(sv->owner);
  delete sv;
  return GPO_OK;
}

gpo_status gpo_server_submit(gpo_server* sv, gpo_graph* g, int32_t max_iters, const gpo_lm_params* params,
                             int64_t* ticket) {
  if (!sv || !g || max_iters < 0) return GPO_ERR_ARG;
  if (g->prec != sv->owner->prec || g->desc.device != sv->owner->desc.device)
    return fail(sv->owner, GPO_ERR_ARG, "graph precision or device differs from the server's");
  if (g->desc.spmv_variant == 4)
    return fail(sv->owner, GPO_ERR_UNSUPPORTED, "graphs with dynamic Jacobians are solved alone");
  if (g->finalized) return fail(sv->owner, GPO_ERR_STATE, "graph is already resident on the device");
  const gpo::KernelSet* k = &kernels_of(g);
  if (sv->owner->ks && sv->owner->ks != k)
    return fail(sv->owner, GPO_ERR_ARG, "graph camera kind differs from the server's earlier graphs");
  size_t bytes = 0;
  gpo_status s = plan_within(g, sv->desc.memory_budget ? sv->desc.memory_budget : SIZE_MAX, &bytes);
  if (s != GPO_OK) {
    sv->owner->err = g->err;
    return s;
  }
  if (sv->desc.memory_budget && bytes > sv->desc.memory_budget)
    return fail(sv->owner, GPO_ERR_OOM, "graph needs %zu bytes, more than the server budget %zu", bytes,
                (size_t)sv->desc.memory_budget);
  sv->owner->ks = k;
  gpo_server::Req r{g, max_iters, params_or_default(params), sv->next_ticket++, 0, bytes, 0.0, {}, {}, -1.0, false, g->desc, false};
  // a graph without a stream of its own runs on the server's; a graph without an
  // allocator hook takes its arena from the server's pool
  if (!g->stream) {
    g->stream = sv->owner->stream;
    r.adopted_stream = true;
  }
  if (!g->desc.alloc) {
    g->desc.alloc = pool_alloc;
    g->desc.free = pool_free;
    g->desc.alloc_ctx = &sv->pool;
  }
  sv->queue.push_back(r);
  if (ticket) *ticket = r.ticket;
  return GPO_OK;
}

gpo_status gpo_server_step(gpo_server* sv, int32_t* n_resident, int32_t* n_queued, int32_t* n_finished) {
  if (!sv) return GPO_ERR_ARG;
  gpo_graph* owner = sv->owner;
  GPO_CUDA(owner, cudaSetDevice(owner->desc.device));
  int fin = 0;
  gpo_status late = GPO_OK;   // a wait that gave up, reported at the end
  // 1. admission: first come, first served, while slots and memory allow; the new
  //    graphs' initial costs are computed together in shared launches
  std::vector<gpo_server::Req> adm;
  while (!sv->queue.empty() && (int)(sv->resident.size() + adm.size()) < sv->desc.max_resident) {
    gpo_server::Req r = sv->queue.front();
    if (sv->desc.memory_budget && sv->used + r.bytes > sv->desc.memory_budget) break;
    gpo_status s = finalize(r.g);
    if (s != GPO_OK) {
      owner->err = r.g->err;
      return s;
    }
    sv->used += r.g->arena_bytes;
    sv->queue.pop_front();
    adm.push_back(r);
  }
  std::vector<gpo_server::Req> retire;   // graphs leaving the device this step
  if (!adm.empty()) {
    std::vector<gpo_graph*> gs;
    for (auto& r : adm) gs.push_back(r.g);
    BatchSet bs;
    gpo_status s = join_uploads(owner, gs);
    if (s == GPO_OK) s = build_set(owner, gs, {}, bs);
    if (s != GPO_OK) return s;
    std::vector<Scalars> sc(adm.size());
    for (size_t i = 0; i < adm.size(); ++i) {
      fill_scalars(adm[i].g, adm[i].prm, adm[i].prm.initial_damping, sc[i]);
      sc[i].full = 0;   // shared launches run the Schur form
      adm[i].g->pcg_full = 0;
    }
    if ((s = put_scalars(owner, bs, sc)) == GPO_OK && (s = launch_initial_cost(owner, bs.ls)) == GPO_OK)
      s = get_scalars(owner, bs, sc);
    bs.release(owner->stream);
    if (s != GPO_OK) return s;
    for (size_t i = 0; i < adm.size(); ++i) {
      adm[i].initial_cost = sc[i].cost;
      adm[i].start = sc[i];
      adm[i].damping.start(sc[i]);
      adm[i].limit = explicit_up_to(adm[i].g, adm[i].prm);
      adm[i].ex = adm[i].damping.within(adm[i].limit) > 0;
      if (adm[i].max_iters == 0 || !std::isfinite(adm[i].initial_cost)) {
        gpo_report rep;
        report_from(sc[i], adm[i].initial_cost, &rep);
        sv->finished[adm[i].ticket] = rep;
        retire.push_back(adm[i]);
      } else {
        sv->resident.push_back(adm[i]);
        sv->dirty = true;
      }
    }
  }
  if (!sv->resident.empty()) {
    // 2. one LM iteration for every resident graph, in shared launches
    if (sv->dirty) {
      sv->set.release(owner->stream);
      std::vector<gpo_graph*> gs;
      std::vector<char> ex;
      for (auto& r : sv->resident) {
        gs.push_back(r.g);
        ex.push_back(r.ex);
      }
      gpo_status s = build_set(owner, gs, ex, sv->set);
      if (s != GPO_OK) return s;
      sv->dirty = false;
    }
    int max_it = 1;
    for (auto& r : sv->resident) max_it = std::max(max_it, r.prm.pcg_max_iters);
    owner->cur_lm_iter = -1;
    sv->set.ls.debug_wait = std::any_of(sv->resident.begin(), sv->resident.end(),
                                        [](const gpo_server::Req& r) { return held(r.g, r.done_iters); });
    gpo_status s = begin_solves(owner, sv->set.ls);
    if (s == GPO_OK) s = solve_system(owner, sv->set.ls, max_it, false);
    const bool stepped = s == GPO_OK;
    if (s == GPO_OK) s = post_flags(owner, sv->set.ls);
    if (s == GPO_OK) s = finish_iteration(owner, sv->set.ls);
    if (s == GPO_OK) s = read_flags(owner, sv->set.ls);
    std::vector<char> ran(sv->resident.size(), 1);
    if (s == GPO_ERR_TIMEOUT) {   // the solves that were lost are made again by the next step
      late = s;
      s = rearm(owner, sv->set, stepped, ran);
    }
    if (s != GPO_OK) return s;
    ++sv->steps;
    // 3. retirement of graphs that ran all their iterations
    bool any = false, read = false;
    for (size_t i = 0; i < ran.size(); ++i) {
      gpo_server::Req& r = sv->resident[i];
      any |= (r.done_iters += ran[i]) >= r.max_iters;
      if (ran[i]) r.damping.iteration(r.start);
      read |= r.damping.within(r.limit) < 0;
    }
    if (read) {   // a damping may have crossed its limit
      std::vector<Scalars> sc;
      if ((s = get_scalars(owner, sv->set, sc)) != GPO_OK) return s;
      for (size_t i = 0; i < sc.size(); ++i) sv->resident[i].damping.start(sc[i]);
    }
    for (auto& r : sv->resident) {
      const bool ex = r.damping.within(r.limit) > 0;
      sv->dirty |= ex != r.ex;
      r.ex = ex;
    }
    if (any) {
      std::vector<Scalars> sc;
      if ((s = get_scalars(owner, sv->set, sc)) != GPO_OK) return s;
      std::vector<gpo_server::Req> keep;
      for (size_t i = 0; i < sv->resident.size(); ++i) {
        gpo_server::Req& r = sv->resident[i];
        if (r.done_iters < r.max_iters) {
          keep.push_back(r);
          continue;
        }
        gpo_report rep;
        report_from(sc[i], r.initial_cost, &rep);
        sv->finished[r.ticket] = rep;
        r.g->last_cost = sc[i].cost;
        r.g->cost_valid = true;
        r.g->state_same = false;   // a served run: the next single run starts afresh
        retire.push_back(r);
      }
      sv->resident.swap(keep);
      sv->dirty = true;
    }
  }
  if (!retire.empty()) {
    // final states back to the graphs' host arrays: all copies, then one wait
    std::vector<std::vector<double>> pts(retire.size());
    for (size_t i = 0; i < retire.size(); ++i) {
      gpo_status s = download_begin(retire[i].g, pts[i]);
      if (s != GPO_OK) return s;
    }
    GPO_CUDA(owner, cudaStreamSynchronize(owner->stream));
    for (size_t i = 0; i < retire.size(); ++i) {
      gpo_server::Req& r = retire[i];
      if (r.g->stream != owner->stream) GPO_CUDA(owner, cudaStreamSynchronize(r.g->stream));
      download_end(r.g, pts[i]);
      sv->used -= r.g->arena_bytes;
      release_device(r.g);
      restore_graph(r);
      ++fin;
    }
  }
  if (n_resident) *n_resident = (int32_t)sv->resident.size();
  if (n_queued) *n_queued = (int32_t)sv->queue.size();
  if (n_finished) *n_finished = fin;
  return late;
}

gpo_status gpo_server_poll(gpo_server* sv, int64_t ticket, int32_t* done, gpo_report* report) {
  if (!sv || !done) return GPO_ERR_ARG;
  auto it = sv->finished.find(ticket);
  if (it == sv->finished.end()) {
    *done = 0;
    return GPO_OK;
  }
  *done = 1;
  if (report) *report = it->second;
  sv->finished.erase(it);
  return GPO_OK;
}

gpo_status gpo_server_memory(gpo_server* sv, size_t* used_bytes) {
  if (!sv || !used_bytes) return GPO_ERR_ARG;
  *used_bytes = sv->used;
  return GPO_OK;
}

const char* gpo_server_last_error(const gpo_server* sv) { return sv ? sv->owner->err.c_str() : ""; }

}  // extern "C"
