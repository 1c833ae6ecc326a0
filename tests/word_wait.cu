// The word engine's waits, for test_host_cpu.py (their limits) and
// test_gpu_words.py (a wait that runs out).
#include "word_engine.cuh"

using namespace bfk;

// Polls that a wait allows.
extern "C" BF_API double spin_limit() { return (double)kWordSpinMax; }

constexpr unsigned kFew = 1000;

extern __shared__ __align__(16) unsigned char wait_smem[];

// Block 0 waits for block 1, which never arrives: out = {did the barrier pass,
// gate's value}.
__global__ void k_wait(WordCtr* k, int gate, int* out) {
    WordSmem& sm = *reinterpret_cast<WordSmem*>(wait_smem);
    if (blockIdx.x == 1) return;
    if (threadIdx.x == 0) {
        sm.nf1 = sm.nchg = sm.npairs = 0u;
        sm.pairs = 0ull;
    }
    unsigned target = 0u;
    const int v = gate ? (word_gate<kFew>(k, 0, sm) != 0ull) : word_barrier<kFew>(k, target, sm);
    if (threadIdx.x == 0) *out = v;
}

// 0, or a CUDA error; *passed and *fault as the kernel leaves them.
extern "C" BF_API int wait_runs_out(int gate, int* passed, int* fault) {
    struct { WordCtr k; int out; } h, *d = nullptr;
    memset(&h, 0, sizeof h);
    h.out = -1;
    cudaError_t e = cudaMalloc((void**)&d, sizeof h);
    if (e == cudaSuccess) e = cudaMemcpy(d, &h, sizeof h, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_wait, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WordSmem));
    if (e == cudaSuccess) {
        k_wait<<<2, 64, sizeof(WordSmem)>>>(&d->k, gate, &d->out);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(&h, d, sizeof h, cudaMemcpyDeviceToHost);
    cudaFree(d);
    *passed = h.out;
    *fault = h.k.fault;
    return (int)e;
}
