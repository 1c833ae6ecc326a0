// The server (serve.cu) on the host alone: an engine, a solver and a builder that
// only count, and an engine step that fails when told to.  For
// test_host_cpu.py, which replaces the few CUDA calls of the server too.
#include <atomic>
#include <chrono>
#include <thread>

#include "batch_engine.cuh"

static std::atomic<int> fail_steps{0}, fail_code{0}, added{0}, removed{0};

extern "C" {
BF_API void fake_fail(int steps, int code) { fail_code = code; fail_steps = steps; }
BF_API int fake_added() { return added; }
BF_API int fake_removed() { return removed; }
BF_API void* fake_abstraction(int64_t cells, int32_t inputs) {
    bf_abstraction* a = new bf_abstraction();
    a->g.C = cells;
    a->g.U = inputs;
    return a;
}
BF_API int abs_info(const bf_abstraction* a, int64_t* nc, int32_t* nu, int32_t*, int32_t*, int64_t*, int32_t*) {
    if (nc) *nc = a->g.C;
    if (nu) *nu = a->g.U;
    return BF_OK;
}
BF_API int abs_build(const bf_dynamics*, const bf_grid*, const bf_inputs*, double, int32_t, void*, bf_abstraction**) {
    return BF_ERR_UNSUPPORTED;
}
BF_API int abs_build_hybrid(const bf_dynamics*, const bf_grid*, const bf_inputs*, double, int64_t, void*,
                            bf_abstraction**) {
    return BF_ERR_UNSUPPORTED;
}
BF_API void abs_free(bf_abstraction* a) { delete a; }
// a plain solve: long enough for more requests to queue up
BF_API int bf_solve(const bf_abstraction*, const double*, const uint8_t*, const uint8_t*, const bf_solve_opts*, double* V,
                    uint8_t*, int64_t* iters, int32_t* status, void*) {
    std::this_thread::sleep_for(std::chrono::milliseconds(300));
    V[0] = 1.0;
    *iters = 7;
    *status = BF_CONVERGED;
    return BF_OK;
}
}

namespace bfh {
void set_error(const char*, ...) {}
int cuda_fail(cudaError_t, const char*) { return BF_ERR_CUDA; }
bool is_device_ptr(const void*) { return false; }
}  // namespace bfh
size_t solve_ws_bytes(const bf_abstraction*) { return 0; }

namespace bfk {
WordTurn::~WordTurn() {}
}

namespace bfb {
Engine::Engine(cudaStream_t st) : st_(st) {}
Engine::~Engine() {
    for (InstState* s : insts_) delete s;
}
int Engine::add(const bf_abstraction* a, const double*, const unsigned char*, const unsigned char*, const double*,
                long long, double* V, unsigned char*, InstState** out) {
    *out = new InstState;
    (*out)->a = a;
    (*out)->V_host = V;
    insts_.push_back(*out);
    ++added;
    return BF_OK;
}
int Engine::rebuild() { return BF_OK; }
int Engine::step(int, bool) { return BF_OK; }
int Engine::read_counters(std::vector<Counters>& out) {
    if (fail_steps > 0) {
        --fail_steps;
        return fail_code;
    }
    out.assign(insts_.size(), Counters());
    for (Counters& c : out) c.done = 1;
    return BF_OK;
}
int Engine::finish_instance(InstState* s, int64_t* iters, int32_t* status, int* err) {
    s->V_host[0] = 1.0;
    *iters = 7;
    *status = BF_CONVERGED;
    *err = 0;
    return BF_OK;
}
void Engine::remove(InstState* s) {
    for (size_t i = 0; i < insts_.size(); ++i)
        if (insts_[i] == s) insts_.erase(insts_.begin() + i);
    delete s;
    ++removed;
}
size_t Engine::state_bytes(const bf_abstraction*, bool, bool, bool) const { return 100; }
size_t Engine::state_bytes_for(long long, int, bool, bool, bool) { return 100; }
}  // namespace bfb
