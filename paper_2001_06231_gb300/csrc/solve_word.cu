// solve_word.cu -- kernels of the word engine (word_engine.cuh): a whole solve
// as one cooperative launch, and the same phases as separate launches for the
// host-driven and timed forms.
#include "word_engine.cuh"

using namespace bfk;

extern __shared__ __align__(16) unsigned char word_smem[];

// One block per SM: 32 warps at 64 registers fill the register file.
__global__ void __launch_bounds__(kWordThreads, 1) k_word_solve(const __grid_constant__ WordInst w) {
    WordSmem& sm = *reinterpret_cast<WordSmem*>(word_smem);
    unsigned target = 0u;
    unsigned long long pairs = 0ull, count;
    word_init(w, reinterpret_cast<double*>(word_smem));
    __syncthreads();
    word_start(sm);
    if (!word_barrier(w.ctr, target, sm)) return;
    if (*(volatile int*)&w.ctr->err) return;
    long long r = 0;
    for (;; ++r) {
        word_tables<false>(w, nullptr, 0, r - 1, sm);
        if (!word_barrier(w.ctr, target, sm)) return;
        const bool last = r >= w.cap;
        word_relax<false>(w, nullptr, 0, r, last, sm, pairs, count);
        const unsigned long long v = word_gate(w.ctr, r, count, sm);
        if (v == 0ull) return;
        if (blockIdx.x == 0 && threadIdx.x == 0) word_close(w, r, last);
        if (((v >> 16) & 0xFFFFull) == 0ull || last || (v >> 32) == 0ull) break;
    }
    if (pairs) atomicAdd(&w.ctr->total_pairs, pairs);
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
    unsigned long long pairs = 0ull, count;
    bool fresh = false;
    for (int i = 0; i < n; ++i)
        if (!insts[i].ctr->ready) {
            fresh = true;
            word_init(insts[i], reinterpret_cast<double*>(word_smem));
        }
    if (fresh && !word_barrier(k, target, sm)) return;
    __syncthreads();
    word_start(sm);
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
        word_tables<true>(insts[0], insts, n, 0, sm);
        if (!word_barrier(k, target, sm)) return;
        word_relax<true>(insts[0], insts, n, 0, false, sm, pairs, count);
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

__global__ void __launch_bounds__(kWordThreads, 1) k_word_init(const __grid_constant__ WordInst w) {
    word_init(w, reinterpret_cast<double*>(word_smem));
}

__global__ void __launch_bounds__(kWordThreads, 1) k_word_relax(const __grid_constant__ WordInst w, long long r) {
    WordSmem& sm = *reinterpret_cast<WordSmem*>(word_smem);
    unsigned long long pairs = 0ull, count;
    word_start(sm);
    word_relax<false>(w, nullptr, 0, r, r >= w.cap, sm, pairs, count);
    if (pairs) atomicAdd(&w.ctr->total_pairs, pairs);
    if ((threadIdx.x & 31) == 0 && count) atomicAdd(&w.ctr->sums[r & 3], count);
}

__global__ void __launch_bounds__(kWordThreads, 1) k_word_tables(const __grid_constant__ WordInst w, long long r) {
    word_tables<false>(w, nullptr, 0, r, *reinterpret_cast<WordSmem*>(word_smem));
}

__global__ void k_word_close(const __grid_constant__ WordInst w, long long r) { word_close(w, r, r >= w.cap); }

__global__ void __launch_bounds__(kWordThreads, 1) k_word_output(const __grid_constant__ WordInst w) { word_output(w); }

static_assert(sizeof(WordSmem) >= kWordWarps * kWordSlab * sizeof(double), "the set-up stages costs there");

static int word_attr() {
    BF_CUDA(cudaFuncSetAttribute(k_word_init, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WordSmem)));
    BF_CUDA(cudaFuncSetAttribute(k_word_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WordSmem)));
    BF_CUDA(cudaFuncSetAttribute(k_word_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WordSmem)));
    BF_CUDA(cudaFuncSetAttribute(k_word_relax, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WordSmem)));
    BF_CUDA(cudaFuncSetAttribute(k_word_tables, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WordSmem)));
    return BF_OK;
}

// Blocks of the engine's launches for a grid of `units` units: one per SM, and
// no more than units.  0: the device cannot hold the kernel.
int word_wave(int units) {
    int dev = 0, sms = 148, per_sm = 0, coop = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop || word_attr() != BF_OK) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_word_solve, kWordThreads, sizeof(WordSmem)) !=
            cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        return 0;
    }
    return units < sms ? units : sms;
}

// A whole solve in one launch (counters zeroed by the caller on the stream).
int word_solve(const WordInst& w, int blocks, cudaStream_t st) {
    WordInst arg = w;
    void* args[] = {(void*)&arg};
    BF_CUDA(cudaLaunchCooperativeKernel((const void*)k_word_solve, dim3(blocks), dim3(kWordThreads), args,
                                        sizeof(WordSmem), st));
    return BF_OK;
}

// n instances (device array) together, at most `passes` passes (negative: all);
// k: scratch counters (`fault` stays set when a block gave up waiting).
int word_solve_batch(const WordInst* insts, int n, int passes, WordCtr* k, cudaStream_t st) {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    for (int i = 0; i < n; i += kWordInsts) {
        const WordInst* first = insts + i;
        int m = n - i < kWordInsts ? n - i : kWordInsts;
        BF_CUDA(cudaMemsetAsync(&k->bar, 0, sizeof k->bar, st));
        void* args[] = {(void*)&first, (void*)&m, (void*)&passes, (void*)&k};
        BF_CUDA(cudaLaunchCooperativeKernel((const void*)k_word_batch, dim3(sms), dim3(kWordThreads), args,
                                            sizeof(WordSmem), st));
    }
    return BF_OK;
}

// The same phases launched one by one, the host reading the counters after
// every pass; with relax_ms / rest_ms (or NULL) CUDA events around them.
int word_solve_host(const WordInst& w, int blocks, cudaStream_t st, double* relax_ms, double* rest_ms,
                    long long* launches) {
    cudaEvent_t e[3] = {nullptr, nullptr, nullptr};
    if (relax_ms)
        for (int i = 0; i < 3; ++i) BF_CUDA(cudaEventCreate(&e[i]));
    const size_t sb = sizeof(WordSmem);
    WordCtr hc;
    k_word_init<<<blocks, kWordThreads, sb, st>>>(w);
    k_word_tables<<<blocks, kWordThreads, sb, st>>>(w, -1);
    long long n = 2, r = 0;
    cudaError_t er = cudaGetLastError();
    for (; er == cudaSuccess; ++r) {
        if (r == 0) {
            er = cudaMemcpyAsync(&hc, w.ctr, sizeof hc, cudaMemcpyDeviceToHost, st);
            if (er == cudaSuccess) er = cudaStreamSynchronize(st);
            if (er != cudaSuccess || hc.err) break;
        }
        if (relax_ms) cudaEventRecord(e[0], st);
        k_word_relax<<<blocks, kWordThreads, sb, st>>>(w, r);
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
        k_word_tables<<<blocks, kWordThreads, sb, st>>>(w, r);
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
