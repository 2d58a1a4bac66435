// The order in which the persistent solve kernels take a batch's nodes.
//
// On collapse profiles and core/tail mixes a node's iterations grow with its optical depth per step, rho dt
// (rank correlation with the inner iterations 0.89-0.97), and differ 20-50 fold within a batch.  With nodes
// taken as they come, a long node that starts late leaves most of the chip idle at the end.  Long nodes first
// is the classical remedy (Graham's LPT rule, SIAM J. Appl. Math. 17, 1969).  This kernel sorts the node
// indices by falling rho dt, to 1/8 octave, with one block's counting sort; the solve's results do not depend
// on the order.  Where rho dt hardly varies, as in a batch of relaxation problems at one step, the iterations
// do not follow it (rank correlation 0.14) and the order is close to arbitrary, neither a gain nor a loss.
//
// Used while it pays: more nodes than resident blocks (else every node starts at once) and at most
// kOrderMax (beyond ~150 nodes per block the idle end is below 1%, and one block's three passes over
// the keys would begin to show).  Without and with it: 512 nodes, mixed, 64 energies, 1.51-1.56 and 1.47 ms; 4099
// nodes, FP64, with their gradient, 24.2 and 23.1; O(v/c), 8192 nodes, 46.0 and 44.2; FP64, 6007 nodes, 64
// energies, 66.9 and 65.0; 20001 nodes, 32 energies, 67.4 and 66.3; mixed, 50000 core/tail nodes, 35.4 and 34.4; 1500
// relaxation problems 59.3-60.1 and 59.0.  The sort itself takes 5 us at 1000 nodes and 180 us at 65536, which calls
// of few iterations do not earn back (emission and absorption alone with matter fixed, 32 energies: 1000 nodes 199
// and 206 us, 10000 nodes 1.32 and 1.36 ms).  It also clears the work queue, in place of the memset of the other calls.
#include <cuda_runtime.h>

#include <string>

#include "nmc_internal.h"

namespace nmc {

namespace {

constexpr int kThreads = 1024;
constexpr int kKeys = 512;   // 1/8 octaves of rho dt, falling from the batch's largest: 64 octaves

// rho dt to its exponent and three mantissa bits; 0 for what is not positive and finite
__device__ __forceinline__ int key_of(double rho, double dt) {
    const double x = rho * dt;
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    return u - 1 < 0x7ff0000000000000ull - 1 ? (int)(u >> 49) : 0;
}

__global__ void __launch_bounds__(kThreads) order_kernel(int n, const double* __restrict__ rho, const double* __restrict__ dt,
                                                         int* __restrict__ order, int* queue) {
    __shared__ int first[kKeys];   // counts, then each key's next position
    __shared__ int top;
    const int t = threadIdx.x;
    if (t == 0) {
        *queue = 0;
        top = 0;
    }
    if (t < kKeys) first[t] = 0;
    __syncthreads();
    int mx = 0;
    for (int i = t; i < n; i += kThreads) mx = max(mx, key_of(rho[i], dt[i]));
    atomicMax(&top, mx);
    __syncthreads();
    const int k0 = top;
    for (int i = t; i < n; i += kThreads) atomicAdd(&first[min(max(k0 - key_of(rho[i], dt[i]), 0), kKeys - 1)], 1);
    __syncthreads();
    for (int off = 1; off < kKeys; off <<= 1) {   // inclusive prefix sums
        const int v = t >= off && t < kKeys ? first[t - off] : 0;
        __syncthreads();
        if (t < kKeys) first[t] += v;
        __syncthreads();
    }
    const int before = t > 0 && t < kKeys ? first[t - 1] : 0;
    __syncthreads();
    if (t < kKeys) first[t] = before;
    __syncthreads();
    // the bounds matter only if a caller overwrites rho or dt meanwhile: the passes then disagree, and some
    // entries keep an earlier batch's nodes or are written twice (node_at bounds what is read)
    for (int i = t; i < n; i += kThreads)
        order[min(atomicAdd(&first[min(max(k0 - key_of(rho[i], dt[i]), 0), kKeys - 1)], 1), n - 1)] = i;
}

}  // namespace

int start_queue(nmc_ctx* ctx, SolveArgs& a, long long resident, cudaStream_t stream) {
    cudaError_t e;
    if (a.order && a.n > resident && a.n <= kOrderMax) {
        order_kernel<<<1, kThreads, 0, stream>>>((int)a.n, a.rho, a.dt, a.order, a.queue);
        e = cudaGetLastError();
    } else {
        a.order = nullptr;
        e = cudaMemsetAsync(a.queue, 0, sizeof(int), stream);
    }
    if (e != cudaSuccess) return set_error(ctx, NMC_ECUDA, std::string("work queue: ") + cudaGetErrorString(e));
    return NMC_OK;
}

cudaError_t preload_order() {
    cudaFuncAttributes fa;
    return cudaFuncGetAttributes(&fa, order_kernel);
}

}  // namespace nmc
