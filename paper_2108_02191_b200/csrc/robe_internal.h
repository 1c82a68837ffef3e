// Host-side declarations shared by the translation units of librobe.so.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "robe_device.cuh"

namespace robe {

// Kernels that follow one another in a stream are launched so that each may be set up while the one before
// still runs (programmatic dependent launch): a kernel launched this way calls follow() (robe_device.cuh)
// before it touches memory.  The gap between two small kernels is most of their time.  Measured (B200, us per
// pass): 128-sample lookup 4.7 -> 3.0, 256-sample training step 8.3 -> 4.9, 26 x 1024 rows of 64 16.4 -> 10.6,
// Adam on 26 x 16384 Zipf rows of 16 156 -> 122.
template <class... P, class... A>
inline void launch_next(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);  // (an error stays for cudaGetLastError)
}

constexpr uint64_t kL2SizedBytes = 192ull << 20;  // arrays up to this size count as "of L2 size"

struct Problem {
    MapParams mp;
    const void* array;       // device, M elements
    int dtype;               // 0 fp32, 1 bf16
    int sign;                // 0 / 1
    IdList indices;          // device [nnz], int64 or int32
    const int64_t* offsets;  // device [nbags+1] or nullptr (one-hot)
    int64_t nbags;           // batch * T
    int64_t nnz;
    int32_t* status;         // device status word or nullptr (validation off)
    int l2_keep = 0;         // 1: array reads (forward) and reductions (atomic backward) carry the L2 "keep" policy
    // deterministic backward: a second stream of higher priority with the two events that fork
    // it from and join it to the caller's stream, or all nullptr (everything in the caller's)
    cudaStream_t side = nullptr;
    cudaEvent_t fork_event = nullptr;
    cudaEvent_t join_event = nullptr;
};

// forward: out [nbags, d].  With keep_keys/keep_vals (device, one word per block each) the staged
// kernel also stores every block's start and payload as the sort-based backward wants them;
// *kept says whether the kernel that ran did so.
cudaError_t launch_forward(const Problem& pb, float* out, int variant, cudaStream_t st,
                           uint32_t* keep_keys = nullptr, uint32_t* keep_vals = nullptr,
                           bool* kept = nullptr);

// one-hot rows of any length as one run of elements (robe_flat.cu)
bool flat_ok(const Problem& pb);
cudaError_t launch_forward_flat(const Problem& pb, float* out, cudaStream_t st);
cudaError_t launch_backward_flat(const Problem& pb, const float* grad_out, float* target, float scale,
                                 cudaStream_t st);

// one-hot rows with the repeats of an id served together (robe_rows.cu)
bool rows_ok(const Problem& pb);
cudaError_t launch_forward_rows(const Problem& pb, float* out, cudaStream_t st);
cudaError_t launch_backward_rows(const Problem& pb, const float* grad_out, float* target, float scale,
                                 cudaStream_t st);

// pooled rows of short bags, a run of bags per warp (robe_pool.cu); the forward keeps block starts when asked
bool pool_ok(const Problem& pb, bool backward);
cudaError_t launch_forward_pool(const Problem& pb, float* out, uint32_t* keep_keys, uint32_t* keep_vals, cudaStream_t st);
cudaError_t launch_backward_pool(const Problem& pb, const float* grad_out, float* target, float scale, cudaStream_t st);

// atomic backward: adds scale * g * grad_out into target (fp32 [M])
cudaError_t launch_backward_atomic(const Problem& pb, const float* grad_out, float* target,
                                   float scale, int variant, cudaStream_t st);

// deterministic backward
size_t det_workspace_bytes(const MapParams& mp, int64_t nbags, int64_t nnz, bool bags);
// Adam moments and constants of the deterministic backward's update mode 2
struct AdamState {
    float* m1;     // device [M], first moment
    float* m2;     // device [M], second moment
    float beta1, beta2, eps;
    float bias1;   // 1 - beta1^t
    float bias2;   // 1 - beta2^t
};

// What the strip apply (robe_strips.cu) takes: the sorted blocks and what their sums are for.
struct StripProblem {
    MapParams mp;
    const float* grad_out;
    uint64_t grad_elems;
    float* target;
    float lr;
    AdamState adam;
    const uint32_t* K;
    const uint32_t* V;
    uint64_t nb;
    const int32_t* status;
    void* workspace;     // strips_workspace_bytes, 256-byte aligned
    uint32_t* hot_list;  // strips_list_bytes
};
bool strips_ok(const MapParams& mp, uint64_t nb, bool sign);
size_t strips_workspace_bytes(const MapParams& mp);
size_t strips_list_bytes(const MapParams& mp, uint64_t nb);
// first sorted position of every strip; in st
void launch_strips_prepare(const StripProblem& sp, cudaStream_t st);
// all slots, mode as launch_backward_det's 0, 1, 2, 4.  Slots [0, Z-1) and strips of often repeated ids are served in
// hot_st (st itself, or a stream that has been made to wait for launch_strips_prepare), the others in st.
void launch_strips(const StripProblem& sp, int mode, cudaStream_t st, cudaStream_t hot_st);

// mode 0: target[j] += delta; 1: target = attached array, target[j] = fma(-lr, delta, target[j]);
// 2: Adam step on the attached array with the moments in *adam; 4: Adagrad step on the attached
// array with the accumulators in adam->m2 and adam->eps; 3: binned atomic adds of
// lr * delta terms into target (one sort pass on the top key bits, then red.global in bin order)
// keys_kept: the workspace already holds the block starts and payloads of these ids (left by
// launch_forward or launch_block_keys), so they are not computed again.
cudaError_t launch_backward_det(const Problem& pb, const float* grad_out, float* target, int mode,
                                float lr, const AdamState* adam, void* workspace,
                                size_t workspace_bytes, cudaStream_t st, bool keys_kept = false);
// where in a workspace of the sort-based backward the block starts and payloads go
void block_key_buffers(const Problem& pb, void* workspace, uint32_t** keys, uint32_t** vals);
// block starts and payloads of pb's ids into the workspace (what the backward does first)
cudaError_t launch_block_keys(const Problem& pb, void* workspace, size_t workspace_bytes,
                              cudaStream_t st);

// dense SGD apply of the data-parallel step: array[j] = fma(-lr, grad[j], array[j]) for j < m,
// grad zeroed afterwards when zero_grad
cudaError_t launch_dense_sgd_apply(float* array, float* grad, uint64_t m, float lr, bool zero_grad,
                                   cudaStream_t st);

// id / offset range check into the status word
cudaError_t launch_validate(const Problem& pb, cudaStream_t st);

}  // namespace robe
