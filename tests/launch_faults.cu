// Test helper (not part of the library), for tests/test_launch_faults.py: the
// library's host code with the CUDA runtime calls that it checks replaced by
// ones that fail when told to.  Runs only where no GPU is visible (the kernels
// that it launches would have no memory to work on).
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdio>

static int g_device_count() {
    int n = 0;
    return cudaGetDeviceCount(&n) == cudaSuccess ? n : 0;
}

namespace fake {
int launches = 0, replays = 0, copies = 0, syncs_after_copy = 0;
int fail_launch = -1, fail_copy = -1;  // index of the call that fails
cudaError_t last = cudaSuccess;

template <typename... A>
cudaError_t launch(A&&...) {
    if (launches++ != fail_launch) return cudaSuccess;
    return last = cudaErrorLaunchOutOfResources;
}
cudaError_t get_last() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
template <typename... A>
cudaError_t copy(A&&...) {
    syncs_after_copy = 0;
    return copies++ == fail_copy ? cudaErrorInvalidValue : cudaSuccess;
}
template <typename... A>
cudaError_t sync(A&&...) {
    ++syncs_after_copy;
    return cudaSuccess;
}
template <typename... A>
cudaError_t replay(A&&...) {
    ++replays;
    return cudaSuccess;
}
template <typename... A>
cudaError_t nothing(A&&...) { return cudaSuccess; }
void reset(int launch_index, int copy_index) {
    launches = replays = copies = syncs_after_copy = 0;
    fail_launch = launch_index;
    fail_copy = copy_index;
    last = cudaSuccess;
}
}  // namespace fake

#define cudaLaunchKernelEx fake::launch
#define cudaGetLastError fake::get_last
#define cudaMemcpyAsync fake::copy
#define cudaMemsetAsync fake::nothing
#define cudaStreamSynchronize fake::sync
#define cudaGraphLaunch fake::replay
#include "../paper_1809_08683_gb300/csrc/lbm_gb300.cu"

static int failures = 0;
#define EXPECT(x)                                          \
    do {                                                   \
        if (!(x)) {                                        \
            std::printf("line %d: %s\n", __LINE__, #x);    \
            ++failures;                                    \
        }                                                  \
    } while (0)

static void context(lbm_ctx& c) {
    c.cfg.nx = 40;
    c.cfg.ny = 30;
    c.cfg.precision = LBM_FP64;
    c.eos_set = true;
    c.stream = (cudaStream_t)1;
}

int main() {
    if (g_device_count() != 0) return 77;
    // the macros pass before the replays of a graph does not start
    {
        lbm_ctx c;
        context(c);
        lbm_batch b;
        b.ctxs = {&c};
        b.models = {c.mc};
        b.stream = c.stream;
        b.graph = (cudaGraphExec_t)1;
        b.graph_steps = 2;
        b.set.p_cnt[0] = 1;
        fake::reset(0, -1);
        EXPECT(lbm_batch_step(&b, 4) == LBM_ECUDA);
        EXPECT(fake::launches == 1 && fake::replays == 0 && b.steps == 0 && c.steps == 0);
        fake::reset(-1, -1);
        EXPECT(lbm_batch_step(&b, 4) == LBM_OK);
        EXPECT(fake::launches == 1 && fake::replays == 2 && b.steps == 4 && c.steps == 4);
    }
    // a launch of a lone lattice's steps fails: in one cluster, in node kernels
    for (int cluster = 0; cluster < 2; ++cluster) {
        lbm_ctx c;
        context(c);
        c.n_node = c.n_prep = 1;
        c.cluster_ctas = cluster;
        fake::reset(cluster ? 0 : 2, -1);
        EXPECT(lbm_step(&c, 3) == LBM_ECUDA);
        EXPECT(c.steps == 0);
        fake::reset(-1, -1);
        EXPECT(lbm_step(&c, 3) == LBM_OK);
        EXPECT(c.steps == 3);
    }
    // without a launch table (lbm_set_tile or lbm_set_eos ran out of memory) nothing is launched
    {
        lbm_ctx c;
        context(c);
        fake::reset(-1, -1);
        EXPECT(lbm_step(&c, 2) == LBM_ENOMEM);
        EXPECT(fake::launches == 0 && c.steps == 0);
    }
    // state transfers: no copy from or to the caller's arrays is left in flight
    for (int set = 0; set < 2; ++set)
        for (int k = 0; k < 4; ++k) {
            lbm_ctx c;
            context(c);
            double f = 0.0, g = 0.0;  // addresses only
            fake::reset(-1, k);
            EXPECT((set ? lbm_set_state(&c, &f, &g) : lbm_get_state(&c, &f, &g)) == LBM_ECUDA);
            EXPECT(fake::copies == k + 1 && fake::syncs_after_copy == 1);
        }
    if (!failures) std::printf("ok\n");
    return failures ? 1 : 0;
}
