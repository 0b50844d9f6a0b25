// Batched single-source BFS over many graphs in one CUDA-graph launch (an
// extension beyond the paper).  The batch graph holds, for each handle, an
// independent chain
//     k_init -> k_batch_root (root read from a device array) -> device-side
//     iteration loop (conditional WHILE node) -> k_batch_output
// or, for the fixed policies on small graphs (batch_small), the one node k_small; so one
// cudaGraphLaunch runs every BFS, the chains overlapping on the GPU, and the same
// executable graph is replayed with new roots and output pointers.
#include <algorithm>
#include <set>
#include <vector>

#include "ss_device.cuh"

struct slimsell_batch {
  std::vector<slimsell_handle> hs;
  int sr = 0, policy = 0;
  int* d_roots = nullptr;  // [g]
  int** d_dist = nullptr;  // [g] device output pointers (NULL entries allowed), then
  int** d_par = nullptr;   // [g] (one allocation, one copy per run)
  ss::Ctl** d_src = nullptr;  // [g] the handles' control blocks
  ss::Ctl* d_ctl = nullptr;   // [g] their copies side by side, made by the graph's last node: one
                              // copy to the host per run (64 small ones took 95 us of a 64-graph batch)
  ss::Ctl* h_ctl = nullptr;   // [g] pinned
  cudaGraphExec_t exec = nullptr;
  cudaEvent_t done = nullptr;
  int pending = 0;
};

namespace ss {

__global__ void k_batch_root(Dev d, const int* roots, int i) { init_root_state(d, roots[i]); }

__global__ void k_batch_output(Dev d, int* const* dist, int* const* par, int i) {
  write_outputs(d, dist[i], par[i], d.ctl->root_row, (long long)blockIdx.x * blockDim.x + threadIdx.x,
                (long long)gridDim.x * blockDim.x);
}

__global__ void k_batch_collect(Ctl* const* src, Ctl* dst) {
  const unsigned* a = reinterpret_cast<const unsigned*>(src[blockIdx.x]);
  unsigned* o = reinterpret_cast<unsigned*>(dst + blockIdx.x);
  for (int i = threadIdx.x; i < (int)(sizeof(Ctl) / sizeof(unsigned)); i += blockDim.x) o[i] = a[i];
}

static ss_status add_kernel(cudaGraph_t g, void* func, dim3 grid, dim3 block, void** args,
                            const cudaGraphNode_t* deps, size_t ndeps, cudaGraphNode_t* out) {
  cudaKernelNodeParams kp = {};
  kp.func = func;
  kp.gridDim = grid;
  kp.blockDim = block;
  kp.sharedMemBytes = 0;
  kp.kernelParams = args;
  SS_CUDA(cudaGraphAddKernelNode(out, g, deps, ndeps, &kp));
  return SS_OK;
}

static void free_batch(slimsell_batch* b) {
  if (!b) return;
  if (b->done) {
    cudaEventSynchronize(b->done);
    cudaEventDestroy(b->done);
  }
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->d_roots) cudaFree(b->d_roots);
  if (b->d_dist) cudaFree(b->d_dist);
  if (b->d_src) cudaFree(b->d_src);
  if (b->d_ctl) cudaFree(b->d_ctl);
  if (b->h_ctl) cudaFreeHost(b->h_ctl);
  delete b;
}

}  // namespace ss

extern "C" {

ss_status slimsell_batch_create(const slimsell_handle* hs, int32_t g, int32_t semiring,
                                int32_t policy, slimsell_batch_handle* out) {
  using namespace ss;
  set_error("");
  if (!out || !hs || g < 1) {
    set_error("slimsell_batch_create: bad arguments");
    return SS_ERR_INVALID;
  }
  *out = nullptr;
  if (semiring < SS_TROPICAL || semiring > SS_SELMAX || policy < SS_V_FULL || policy > SS_V_LEARNED) {
    set_error("slimsell_batch_create: bad semiring or policy");
    return SS_ERR_INVALID;
  }
  std::set<slimsell_handle> seen;
  for (int i = 0; i < g; ++i) {
    if (!hs[i] || !seen.insert(hs[i]).second) {
      set_error("slimsell_batch_create: handle %d is NULL or repeated", i);
      return SS_ERR_INVALID;
    }
  }
  slimsell_batch* b = new slimsell_batch();
  b->hs.assign(hs, hs + g);
  b->sr = semiring;
  b->policy = policy;
  ss_status s = dmalloc(nullptr, (void**)&b->d_roots, sizeof(int) * (size_t)g);
  if (s == SS_OK) s = dmalloc(nullptr, (void**)&b->d_dist, 2 * sizeof(int*) * (size_t)g);
  if (s == SS_OK) b->d_par = b->d_dist + g;
  if (s == SS_OK) s = dmalloc(nullptr, (void**)&b->d_src, sizeof(Ctl*) * (size_t)g);
  if (s == SS_OK) s = dmalloc(nullptr, (void**)&b->d_ctl, sizeof(Ctl) * (size_t)g);
  if (s == SS_OK) {
    std::vector<Ctl*> src((size_t)g);
    for (int i = 0; i < g; ++i) src[(size_t)i] = hs[i]->ctl;
    if (cudaMemcpy(b->d_src, src.data(), sizeof(Ctl*) * (size_t)g, cudaMemcpyHostToDevice) != cudaSuccess)
      s = cuda_fail(cudaGetLastError(), "cudaMemcpy");
  }
  if (s == SS_OK && cudaHostAlloc((void**)&b->h_ctl, sizeof(Ctl) * (size_t)g, 0) != cudaSuccess)
    s = cuda_fail(cudaGetLastError(), "cudaHostAlloc");
  if (s == SS_OK && cudaEventCreateWithFlags(&b->done, cudaEventDisableTiming) != cudaSuccess)
    s = cuda_fail(cudaGetLastError(), "cudaEventCreate");
  if (s == SS_OK && cudaMemset(b->d_dist, 0, 2 * sizeof(int*) * (size_t)g) != cudaSuccess)
    s = cuda_fail(cudaGetLastError(), "cudaMemset");
  cudaGraph_t graph = nullptr;
  if (s == SS_OK && cudaGraphCreate(&graph, 0) != cudaSuccess)
    s = cuda_fail(cudaGetLastError(), "cudaGraphCreate");
  // largest graphs first: they decide when the batch ends
  std::vector<int> order((size_t)g);
  std::vector<cudaGraphNode_t> ends;  // last node of every chain
  long long batch_slots = 0;
  for (int i = 0; i < g; ++i) {
    order[(size_t)i] = i;
    batch_slots += b->hs[(size_t)i]->slots;
  }
  long long ctas = 0;
  for (auto* h : b->hs) ctas += batch_ctas(h, h->dev(), policy, batch_slots);
  std::stable_sort(order.begin(), order.end(),
                   [&](int x, int y) { return b->hs[(size_t)x]->slots > b->hs[(size_t)y]->slots; });
  for (int o = 0; o < g && s == SS_OK; ++o) {
    const int i = order[(size_t)o];
    slimsell_graph* h = b->hs[(size_t)i];
    Dev d = h->dev();
    int idx = i;
    int* roots = b->d_roots;
    int** dist = b->d_dist;
    int** par = b->d_par;
    if (batch_small(h, d, policy, ctas)) {  // the whole chain in one node
      SmallIo io{};
      io.roots = roots;
      io.dists = dist;
      io.parents = par;
      io.i = idx;
      cudaGraphNode_t n_run;
      s = add_small_node(h, d, semiring, policy, io, batch_slots, graph, &n_run);
      ends.push_back(n_run);
      continue;
    }
    cudaGraphNode_t n_init, n_root, n_loop, n_out;
    void* a_init[] = {&d};
    s = add_kernel(graph, (void*)k_init, dim3(vertex_grid(h, 256)), dim3(256), a_init, nullptr, 0, &n_init);
    void* a_root[] = {&d, &roots, &idx};
    if (s == SS_OK)
      s = add_kernel(graph, (void*)k_batch_root, dim3(1), dim3(1), a_root, &n_init, 1, &n_root);
    if (s == SS_OK) s = add_loop_node(h, d, semiring, policy, graph, &n_root, 1, &n_loop);
    void* a_out[] = {&d, &dist, &par, &idx};
    if (s == SS_OK)
      s = add_kernel(graph, (void*)k_batch_output, dim3(vertex_grid(h, 256)), dim3(256), a_out,
                     &n_loop, 1, &n_out);
    ends.push_back(n_out);
  }
  if (s == SS_OK) {
    Ctl** src = b->d_src;
    Ctl* dst = b->d_ctl;
    void* a_col[] = {&src, &dst};
    cudaGraphNode_t n_col;
    s = add_kernel(graph, (void*)k_batch_collect, dim3(g), dim3(64), a_col, ends.data(), ends.size(), &n_col);
  }
  if (s == SS_OK && cudaGraphInstantiate(&b->exec, graph, 0) != cudaSuccess) {
    b->exec = nullptr;
    s = cuda_fail(cudaGetLastError(), "cudaGraphInstantiate(batch)");
  }
  if (graph) cudaGraphDestroy(graph);
  if (s != SS_OK) {
    free_batch(b);
    return s;
  }
  *out = b;
  return SS_OK;
}

ss_status slimsell_batch_run(slimsell_batch_handle b, const int32_t* d_roots,
                             int32_t* const* h_dist, int32_t* const* h_parent, void* stream) {
  using namespace ss;
  set_error("");
  if (!b || !d_roots) {
    set_error("slimsell_batch_run: NULL argument");
    return SS_ERR_INVALID;
  }
  const int g = (int)b->hs.size();
  cudaStream_t st = (cudaStream_t)stream;
  for (slimsell_handle hg : b->hs) hg->values_semiring = -1;
  if (b->pending) SS_CUDA(cudaEventSynchronize(b->done));
  std::vector<int> roots((size_t)g);
  SS_CUDA(cudaMemcpyAsync(roots.data(), d_roots, sizeof(int) * (size_t)g, cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaStreamSynchronize(st));
  for (int i = 0; i < g; ++i)
    if (roots[(size_t)i] < 0 || roots[(size_t)i] >= b->hs[(size_t)i]->n) {
      set_error("slimsell_batch_run: root %d of graph %d out of range", roots[(size_t)i], i);
      return SS_ERR_INVALID;
    }
  std::vector<int*> outs(2 * (size_t)g, nullptr);
  for (int i = 0; i < g; ++i) {
    if (h_dist) outs[(size_t)i] = h_dist[i];
    if (h_parent) outs[(size_t)(g + i)] = h_parent[i];
  }
  SS_CUDA(cudaMemcpyAsync(b->d_roots, d_roots, sizeof(int) * (size_t)g, cudaMemcpyDeviceToDevice, st));
  SS_CUDA(cudaMemcpyAsync(b->d_dist, outs.data(), 2 * sizeof(int*) * (size_t)g, cudaMemcpyHostToDevice, st));
  for (auto* h : b->hs) {
    if (h->pending) SS_CUDA(cudaEventSynchronize(h->ev_done));
    h->pending = 0;
  }
  SS_CUDA(cudaGraphLaunch(b->exec, st));
  SS_CUDA(cudaMemcpyAsync(b->h_ctl, b->d_ctl, sizeof(Ctl) * (size_t)g, cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaEventRecord(b->done, st));
  b->pending = 1;
  return SS_OK;
}

ss_status slimsell_batch_get_stats(slimsell_batch_handle b, ss_run_stats* out) {
  using namespace ss;
  if (!b || !out) {
    set_error("slimsell_batch_get_stats: NULL argument");
    return SS_ERR_INVALID;
  }
  if (b->pending) SS_CUDA(cudaEventSynchronize(b->done));
  b->pending = 0;
  int err = 0;
  for (size_t i = 0; i < b->hs.size(); ++i) {
    const Ctl& c = b->h_ctl[i];
    ss_run_stats r = {};
    r.iterations = c.k - 1;
    r.semiring = b->sr;
    r.reached = (long long)c.reached;
    r.reached_degree = (long long)c.reached_deg;
    r.slots = (long long)c.total_slots;
    out[i] = r;
    err |= c.error;
  }
  if (err) {
    set_error("slimsell_batch: iteration limit reached (device error flags %d)", err);
    return SS_ERR_CUDA;
  }
  return SS_OK;
}

void slimsell_batch_destroy(slimsell_batch_handle b) { ss::free_batch(b); }

}  // extern "C"
