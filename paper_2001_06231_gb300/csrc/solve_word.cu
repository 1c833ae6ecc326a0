// solve_word.cu -- kernels of the word engine (word_engine.cuh): all passes of a
// solve as one cooperative launch, and the same phases as separate launches for the
// host-driven and timed forms.
#include <atomic>

#include "word_engine.cuh"

using namespace bfk;

extern __shared__ __align__(16) unsigned char word_smem[];

// One block per SM: 32 warps at 64 registers fill the register file.  The set-up
// is a launch of its own before it (k_word_init): its registers would cost the
// passes spills, and the launch costs no more than the grid barrier it saves.
template <int K>
__global__ void __launch_bounds__(kWordThreads, 1) k_word_solve(const __grid_constant__ WordInst w) {
    WordSmem& sm = *reinterpret_cast<WordSmem*>(word_smem);
    unsigned target = 0u;
    if (*(volatile int*)&w.ctr->err) return;                  // found by k_word_init
    word_start(sm, &w);
    __syncthreads();
    // the pass counter is an int: a solve of 2^31 passes would take hours
    for (int r = 0;; ++r) {
        word_tables<K>(w, nullptr, 0, (r + 1) & 1, r == 0, sm);
        if (!word_barrier(w.ctr, target, sm)) return;
        const bool last = r >= w.cap;
        word_relax<K>(w, nullptr, 0, r & 1, last, sm);
        const unsigned long long v = word_gate(w.ctr, r, sm);
        if (v == 0ull) return;
        if (blockIdx.x == 0 && threadIdx.x == 0) word_close(w, r, last);
        if (((v >> 16) & 0xFFFFull) == 0ull || last || (v >> 32) == 0ull) break;
    }
    if (threadIdx.x == 0 && sm.pairs) atomicAdd(&w.ctr->total_pairs, sm.pairs);
    word_output(w);
}

// Batched form: up to kWordInsts instances, each at its own pass, at most `passes`
// passes (negative: until every one is done).  An instance that was not set up
// yet is set up first; the instances keep their state between launches.  k: the
// launch's barrier counters (zeroed).
__global__ void __launch_bounds__(kWordThreads, 1) k_word_batch(const WordInst* __restrict__ insts, int n, int passes,
                                                                WordCtr* k) {
    WordSmem& sm = *reinterpret_cast<WordSmem*>(word_smem);
    unsigned target = 0u;
    bool fresh = false;
    for (int i = 0; i < n; ++i)
        if (!insts[i].ctr->ready) {
            fresh = true;
            word_init<kWordMany>(insts[i], reinterpret_cast<double*>(word_smem));
        }
    if (fresh && !word_barrier(k, target, sm)) return;
    __syncthreads();
    word_start(sm, nullptr);
    for (int i = threadIdx.x; i < n; i += kWordThreads) {
        WordCtr* c = insts[i].ctr;
        const bool bad = *(volatile int*)&c->err != 0;
        sm.active[i] = !bad && !*(volatile int*)&c->done;
        sm.round[i] = *(volatile long long*)&c->round;
    }
    if (fresh && !word_barrier(k, target, sm)) return;              // every block has read `ready` and `done`
    if (fresh && blockIdx.x == 0)
        for (int i = threadIdx.x; i < n; i += kWordThreads) {
            WordCtr* c = insts[i].ctr;
            c->ready = 1;
            if (c->err) c->done = 1;
        }
    for (int r = 0; passes < 0 || r < passes; ++r) {
        if (word_split(insts, n, sm) == 0 && !__syncthreads_or((int)threadIdx.x < n && sm.active[threadIdx.x])) break;
        word_tables<kWordMany>(insts[0], insts, n, 0, false, sm);
        if (!word_barrier(k, target, sm)) return;
        word_relax<kWordMany>(insts[0], insts, n, 0, false, sm);
        if (!word_barrier(k, target, sm)) return;
        for (int i = threadIdx.x; i < n; i += kWordThreads) {
            if (!sm.active[i]) continue;
            const long long q = sm.round[i];
            const bool last = q >= insts[i].cap;
            const unsigned long long v = *(volatile unsigned long long*)&insts[i].ctr->sums[q & 3];
            if (blockIdx.x == 0) word_close(insts[i], q, last);
            sm.round[i] = q + 1;
            if ((v >> 32) == 0ull || last || (v & 0xFFFFFFFFull) == 0ull) sm.active[i] = 0;
        }
    }
}

template <int K>
__global__ void __launch_bounds__(kWordThreads, 1) k_word_init(const __grid_constant__ WordInst w) {
    word_init<K>(w, reinterpret_cast<double*>(word_smem));
}

template <int K>
__global__ void __launch_bounds__(kWordThreads, 1) k_word_relax(const __grid_constant__ WordInst w, long long r) {
    WordSmem& sm = *reinterpret_cast<WordSmem*>(word_smem);
    word_start(sm, &w);
    __syncthreads();
    word_relax<K>(w, nullptr, 0, (int)(r & 1), r >= w.cap, sm);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (sm.npairs) atomicAdd(&w.ctr->total_pairs, (unsigned long long)sm.npairs);
        if (sm.nf1) atomicAdd(&w.ctr->sums[r & 3], (unsigned long long)sm.nf1 << 32 | sm.nchg);
    }
}

template <int K>
__global__ void __launch_bounds__(kWordThreads, 1) k_word_tables(const __grid_constant__ WordInst w, long long r) {
    WordSmem& sm = *reinterpret_cast<WordSmem*>(word_smem);
    word_start(sm, &w);
    __syncthreads();
    word_tables<K>(w, nullptr, 0, (int)(r & 1), r < 0, sm);
}

__global__ void k_word_close(const __grid_constant__ WordInst w, long long r) { word_close(w, r, r >= w.cap); }

__global__ void __launch_bounds__(kWordThreads, 1) k_word_output(const __grid_constant__ WordInst w) { word_output(w); }

static_assert(sizeof(WordSmem) >= kWordWarps * kWordSlab * sizeof(double), "the set-up stages costs there");

// kWordBox: the spans of every unit (block per unit): the words its cells' boxes
// meet, as at most kWordSpans runs (runs up to 32 words apart are one), relative
// to its first and last word; *used: the tables its lookups read.
constexpr int kSpanWords = 4096;      // words of S bits of the block's bitmap

__global__ void __launch_bounds__(256) k_word_spans(const __grid_constant__ WordInst w, int4* spans, int* used) {
    __shared__ unsigned bits[kSpanWords];
    __shared__ int tabs;
    const int W = (w.S + 31) >> 5;
    for (int un = blockIdx.x; un < w.units; un += gridDim.x) {
        for (int i = threadIdx.x; i < W; i += blockDim.x) bits[i] = 0u;
        if (threadIdx.x == 0) tabs = 0;
        __syncthreads();
        int p, k, n;
        word_unit(w, un, p, k, n);
        const long long last = min((long long)w.g.C, (long long)(k + n) * 32);
        int mine = 0;
        for (int u = 0; u < w.g.U; ++u)
            for (long long c = (long long)k * 32 + threadIdx.x; c < last; c += blockDim.x) {
                int lo[4], wd[4];
                if (!word_box(w, (int)c, u, lo, wd)) continue;
                word_cover(w.g, lo, wd, [&](int t, int e0, int e1, int e2, int e3) {
                    mine |= 1 << t;
                    const int e[4] = {e0, e1, e2, e3};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (!((bits[e[q] >> 10] >> ((e[q] >> 5) & 31)) & 1u))
                            atomicOr(&bits[e[q] >> 10], 1u << ((e[q] >> 5) & 31));
                });
            }
        if (mine) atomicOr(&tabs, mine);
        __syncthreads();
        // runs, found by one warp 1024 words at a time
        if (threadIdx.x < 32) {
            int4* out = spans + (long long)un * kWordSpans;
            out[threadIdx.x] = make_int4(-1, 0, 0, 0);
            __syncwarp();
            if (threadIdx.x == 0) {
                int first = -1, prev = -1, cnt = 0;
                for (int i = 0; i <= W; ++i) {
                    unsigned b = i < W ? bits[i] : 0u;
                    if (i < W && !b) continue;
                    for (; b || i == W; b &= b - 1u) {
                        const int x = i == W ? 0x7FFFFFFF : i * 32 + __ffs(b) - 1;
                        if (first >= 0 && (i == W || x - prev > 32)) {
                            if (cnt < kWordSpans) out[cnt] = make_int4(0, first - k, prev - (k + n - 1), 0);
                            ++cnt;
                            first = -1;
                        }
                        if (i == W) break;
                        if (first < 0) first = x;
                        prev = x;
                    }
                }
                if (cnt > kWordSpans) out[0] = make_int4(-2, 0, 0, 0);
                atomicOr(used, tabs);
            }
        }
        __syncthreads();
    }
}

// The spans of an instance of the box form; *used on the device.  False: too
// many words.
bool word_spans(const WordInst& w, int4* spans, int* used, cudaStream_t st) {
    if ((w.S + 31) / 32 > kSpanWords) return false;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    k_word_spans<<<w.units < 4 * sms ? w.units : 4 * sms, 256, 0, st>>>(w, spans, used);
    return cudaGetLastError() == cudaSuccess;
}

template <int K>
static int word_attr_k() {
    const int b = (int)sizeof(WordSmem);
    BF_CUDA(cudaFuncSetAttribute(k_word_init<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
    BF_CUDA(cudaFuncSetAttribute(k_word_solve<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
    BF_CUDA(cudaFuncSetAttribute(k_word_relax<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
    BF_CUDA(cudaFuncSetAttribute(k_word_tables<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
    return BF_OK;
}

static int word_attr() {
    BF_CUDA(cudaFuncSetAttribute(k_word_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WordSmem)));
    int rc = word_attr_k<kWordOne>();
    if (rc == BF_OK) rc = word_attr_k<kWordClass>();
    return rc ? rc : word_attr_k<kWordBox>();
}

// Blocks of the engine's launches for a grid of `units` units: one per SM, and
// no more than units.  0: the device cannot hold the kernel.
int word_wave(int units) {
    int dev = 0, sms = 148, per_sm = 0, coop = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop || word_attr() != BF_OK) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_word_solve<kWordClass>, kWordThreads, sizeof(WordSmem)) !=
            cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        return 0;
    }
    return units < sms ? units : sms;
}

// Callers with launches of the engine on a device now.
static std::atomic<int> word_callers[64];

WordTurn::WordTurn() {
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    callers = ++word_callers[dev & 63];
}

WordTurn::~WordTurn() { --word_callers[dev & 63]; }

// An equal share of the SMs, an eighth at least.  Microseconds a solve of 1, 2, 4
// and 8 threads with a handle and a stream each, at full width and by shares (GB300):
//   double integrator 64 x 64      487 452 454 454    487 254 129  68
//   double integrator 301 x 205    463 426 424 423    463 255 145  92
//   unicycle 100 x 100 x 32       1121 1085 1082 1091 1121 651 384 261
//   unicycle 200 x 200 x 64       1955 1914 1920 1922 1955 1498 1149 1104
// Narrower than an eighth no more launches fit than threads were measured, and a
// solve takes twice as long alone.
int WordTurn::width(int blocks) const {
    const int n = callers < 8 ? callers : 8, share = sms / n > 0 ? sms / n : 1;
    return blocks < share ? blocks : share;
}

// The quotients by the launch's blocks.
static void word_blocks(WordInst& w, int blocks) {
    GridDesc q;
    memset(&q, 0, sizeof q);
    q.n[0] = blocks;
    grid_divisors(q);
    w.nb_mul = q.dmul[0];
    w.nb_shr = q.dshr[0];
}

// A whole solve: set-up and passes, two launches (counters zeroed by the caller on the stream).
int word_solve(const WordInst& w0, int blocks, cudaStream_t st) {
    WordInst w = w0;
    word_blocks(w, blocks);
    // (the set-up of the box form is the plain one)
    const int words = (w.S + kWordWarps - 1) / kWordWarps, wide = word_wave(words);
    if (w.cls) k_word_init<kWordClass><<<wide, kWordThreads, sizeof(WordSmem), st>>>(w);
    else k_word_init<kWordOne><<<wide, kWordThreads, sizeof(WordSmem), st>>>(w);
    BF_CUDA(cudaGetLastError());
    void* args[] = {(void*)&w};
    const void* k = w.cls ? (const void*)k_word_solve<kWordClass>
                          : (w.lists ? (const void*)k_word_solve<kWordOne> : (const void*)k_word_solve<kWordBox>);
    BF_CUDA(cudaLaunchCooperativeKernel(k, dim3(blocks), dim3(kWordThreads), args,
                                        sizeof(WordSmem), st));
    return BF_OK;
}

// n instances (device array) together, at most `passes` passes (negative: all) on
// `blocks` SMs; k: scratch counters (`fault` stays set when a block gave up waiting).
int word_solve_batch(const WordInst* insts, int n, int passes, int blocks, WordCtr* k, cudaStream_t st) {
    for (int i = 0; i < n; i += kWordInsts) {
        const WordInst* first = insts + i;
        int m = n - i < kWordInsts ? n - i : kWordInsts;
        BF_CUDA(cudaMemsetAsync(&k->bar, 0, sizeof k->bar, st));
        void* args[] = {(void*)&first, (void*)&m, (void*)&passes, (void*)&k};
        BF_CUDA(cudaLaunchCooperativeKernel((const void*)k_word_batch, dim3(blocks), dim3(kWordThreads), args,
                                            sizeof(WordSmem), st));
    }
    return BF_OK;
}

// The same phases launched one by one, the host reading the counters after
// every pass; with relax_ms / rest_ms (or NULL) CUDA events around them.
template <int K>
static int word_solve_host_k(const WordInst& w, int blocks, cudaStream_t st, double* relax_ms, double* rest_ms,
                    long long* launches) {
    cudaEvent_t e[3] = {nullptr, nullptr, nullptr};
    if (relax_ms)
        for (int i = 0; i < 3; ++i) BF_CUDA(cudaEventCreate(&e[i]));
    const size_t sb = sizeof(WordSmem);
    WordCtr hc;
    k_word_init<K><<<blocks, kWordThreads, sb, st>>>(w);
    k_word_tables<K><<<blocks, kWordThreads, sb, st>>>(w, -1);
    long long n = 2, r = 0;
    cudaError_t er = cudaGetLastError();
    for (; er == cudaSuccess; ++r) {
        if (r == 0) {
            er = cudaMemcpyAsync(&hc, w.ctr, sizeof hc, cudaMemcpyDeviceToHost, st);
            if (er == cudaSuccess) er = cudaStreamSynchronize(st);
            if (er != cudaSuccess || hc.err) break;
        }
        if (relax_ms) cudaEventRecord(e[0], st);
        k_word_relax<K><<<blocks, kWordThreads, sb, st>>>(w, r);
        if (relax_ms) cudaEventRecord(e[1], st);
        k_word_close<<<1, 1, 0, st>>>(w, r);
        n += 2;
        er = cudaMemcpyAsync(&hc, w.ctr, sizeof hc, cudaMemcpyDeviceToHost, st);
        if (er == cudaSuccess) er = cudaStreamSynchronize(st);
        if (er != cudaSuccess) break;
        if (relax_ms && hc.round > r) {
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e[0], e[1]);
            *relax_ms += ms;
        }
        if (hc.done) break;
        if (relax_ms) cudaEventRecord(e[1], st);
        k_word_tables<K><<<blocks, kWordThreads, sb, st>>>(w, r);
        ++n;
        if (relax_ms) {
            cudaEventRecord(e[2], st);
            cudaEventSynchronize(e[2]);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e[1], e[2]);
            *rest_ms += ms;
        }
    }
    if (er == cudaSuccess && !hc.err) {
        k_word_output<<<blocks, kWordThreads, 0, st>>>(w);
        ++n;
        er = cudaGetLastError();
    }
    for (int i = 0; i < 3; ++i)
        if (e[i]) cudaEventDestroy(e[i]);
    *launches = n;
    if (er != cudaSuccess) return bfh::cuda_fail(er, "word engine passes");
    return BF_OK;
}

int word_solve_host(const WordInst& w0, int blocks, cudaStream_t st, double* relax_ms, double* rest_ms,
                    long long* launches) {
    WordInst w = w0;
    word_blocks(w, blocks);
    return w.cls ? word_solve_host_k<kWordClass>(w, blocks, st, relax_ms, rest_ms, launches)
         : w.lists ? word_solve_host_k<kWordOne>(w, blocks, st, relax_ms, rest_ms, launches)
                   : word_solve_host_k<kWordBox>(w, blocks, st, relax_ms, rest_ms, launches);
}
