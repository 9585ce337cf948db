// The server's batcher on the host: serve.cu with the library's solver replaced by
// fakes, so that a batched solve can end in any status.  argv[1]: "fail" (the batch as a
// whole) or "timeout" (systems of it, each with its own status).
#include <chrono>
#include <cstdio>
#include <cstring>
#include <string>

#include "serve.cpp"

static std::atomic<int> g_setups{0}, g_batches{0};
static int g_requests = 0;
static bool g_fail = false;
static const char* kMessage = "the message of the failed batch, longer than a short string";

extern "C" {
void cptr_params_default(cptr_params* p) {
  *p = cptr_params{};
  p->restart = 30;
  p->precond = CPTR_PREC_CPTR;
}
cptr_status cptr_create(cptr_ctx** out, int32_t n, int32_t, const int32_t*, const int32_t*,
                        const double*, const cptr_params*) {
  *out = new cptr_ctx();
  (*out)->N = n;
  return CPTR_OK;
}
cptr_status cptr_setup(cptr_ctx*) {
  if (g_setups++ == 1)  // the first request's batch has begun
    while (g_batches == 0) std::this_thread::yield();
  return CPTR_OK;
}
cptr_status cptr_solve(cptr_ctx*, const double*, double*, double, int, cptr_info*) {
  return CPTR_ERR_INVALID;
}
cptr_status cptr_solve_batch(cptr_ctx* const* c, int n, const double* const*, double* const* x,
                             double, int, cptr_info* infos) {
  if (g_batches++ == 0) {  // the first request alone: the others gather meanwhile
    while (g_setups < g_requests) std::this_thread::yield();
    std::this_thread::sleep_for(std::chrono::milliseconds(200));
  } else if (g_fail) {
    c[0]->err = kMessage;
    return CPTR_ERR_CUDA;
  }
  cptr_status worst = CPTR_OK;
  for (int k = 0; k < n; ++k) {
    const cptr_status st = c[k]->N == 2   ? CPTR_ERR_TIMEOUT
                           : c[k]->N == 3 ? CPTR_ERR_MAXIT
                           : c[k]->N == 4 ? CPTR_ERR_BREAKDOWN
                                          : CPTR_OK;
    infos[k] = cptr_info{};
    infos[k].iters = 10 + c[k]->N;
    infos[k].status = st;
    x[k][0] = c[k]->N;
    if (st == CPTR_ERR_TIMEOUT) {
      worst = st;
      c[0]->err = kMessage;
    }
  }
  return worst;
}
void cptr_destroy(cptr_ctx* c) { delete c; }
cptr_status cptr_get_info(const cptr_ctx*, cptr_info* i) {
  *i = cptr_info{};
  return CPTR_OK;
}
const char* cptr_last_error(const cptr_ctx* c) { return c->err.c_str(); }
const char* cptr_status_str(cptr_status s) { return s == CPTR_ERR_TIMEOUT ? "timeout" : "status"; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaErrorUnknown; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
  a->type = cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
}

int main(int, char** argv) {
  g_fail = !std::strcmp(argv[1], "fail");
  const int cells[] = {1, 5, 2, 3, 4, 6};  // the first one is a batch of its own
  const cptr_status want[] = {CPTR_OK,        CPTR_OK,            CPTR_ERR_TIMEOUT,
                              CPTR_ERR_MAXIT, CPTR_ERR_BREAKDOWN, CPTR_OK};
  g_requests = 6;
  cptr_params p;
  cptr_params_default(&p);
  cptr_server* s = nullptr;
  if (cptr_server_create(&s, 1ull << 40, 1, &p) || cptr_server_set_limits(s, 16, 100)) return 2;
  std::vector<uint64_t> id(6);
  for (int k = 0; k < 6; ++k) {
    std::vector<int32_t> rp(cells[k] + 1), ci(cells[k]);
    for (int i = 0; i < cells[k]; ++i) rp[i + 1] = i + 1, ci[i] = i;
    std::vector<double> v(16 * cells[k], 1.0), b(4 * cells[k], 1.0);
    if (cptr_submit(s, cells[k], rp.data(), ci.data(), v.data(), b.data(), 1e-6, 50, &id[k]))
      return 2;
  }
  int bad = 0;
  for (int k = 0; k < 6; ++k) {
    std::vector<double> x(4 * cells[k], -1.0);
    cptr_info info{};
    cptr_status st;
    while ((st = cptr_poll(s, id[k], x.data(), &info)) == CPTR_PENDING) std::this_thread::yield();
    const cptr_status w = g_fail && k ? CPTR_ERR_CUDA : want[k];
    const bool solved = !(g_fail && k);  // the solver's results are handed over
    if (st != w || info.status != w || (solved && (x[0] != cells[k] || info.iters != 10 + cells[k]))) {
      std::printf("request of %d cells: status %d, info %d, iterations %d, x %g\n", cells[k], st,
                  info.status, info.iters, x[0]);
      ++bad;
    }
  }
  const std::string e = cptr_server_last_error(s);
  if (g_batches != 2 || e.find(kMessage) == std::string::npos) {
    std::printf("%d batches, last error \"%s\"\n", (int)g_batches, e.c_str());
    ++bad;
  }
  cptr_server_destroy(s);
  return bad != 0;
}
