// ac_internal.h -- helpers shared by the translation units of the library
// (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>

namespace acgb {

// Record the thread's last error message (read by ac_last_error) and
// return `code`.
int set_last_error(int code, const char *fmt, ...);

// Programmatic dependent launch (AC_PDL=0 turns it off): the kernels of a
// pseudo-iteration are launched so that each may be scheduled while its
// predecessor in the stream is still running; every such kernel starts with
// pdl_wait() and then pdl_trigger() (ac_kernels.cuh), so it touches nothing
// before the predecessor has finished and its writes are visible, and lets its
// successor in only then: a kernel waits beside its predecessor alone, which
// is complete when the wait ends, and not beside kernels further back (the
// other order also filled the SMs' slots unevenly, see pdl_trigger).  What
// overlaps is the launch and CTA dispatch, not the work.
inline bool pdl_enabled() {
    static const bool on = [] {
        const char *e = getenv("AC_PDL");
        return !(e && e[0] == '0');
    }();
    return on;
}

// SMs of the GPU that grids are sized for, and the CTAs of a grid-stride pass over N cells.
constexpr int kSMs = 152;
inline int grid_stride_blocks(size_t N) { return (int)((N + 255) / 256 < kSMs * 8 ? (N + 255) / 256 : kSMs * 8); }

// Pseudo-iterations in a captured loop's body: evaluating the loop's condition
// costs 3 us, a tenth of a small grid's iteration (FP64 20x20, steps of 17 and
// 33: 745 and 1421 us with one iteration to a body, 723 and 1366 with four).
// Iterations past the step's end return at once, which takes 4 us an iteration
// on small grids and 8 on 1024x512: a step that ends after one or two loses by
// the body of four (70 and 108 us with one to a body, 81 and 118 with four),
// from the third on it gains or is even.
constexpr int kLoopIters = 4;

// A step that may well end after one or two pseudo-iterations, as its number
// of them says or because it stops on its tolerance (a tank that has come to
// rest starts every step below it), runs two in line ahead of its loop: 71 and
// 108 us on that grid.  Longer steps that stop on a tolerance then gain or
// lose by where they end in a body (100x1, 3 to 6 iterations: 132, 166, 208,
// 242 -> 143, 172, 204, 231; 33: 1154 -> 1163); fixed numbers keep the loop alone.
constexpr int kAtOnceIters = 2;
inline bool may_end_at_once(double tol, int max_iters) { return tol >= 0.0 || max_iters <= kAtOnceIters; }

// Iterations whose kernels a step of `iters` launches: `lead` in line, then whole bodies of the loop.
inline long long launched_iters(long long iters, int lead) {
    return lead + ((iters > lead ? iters - lead : 0) + kLoopIters - 1) / kLoopIters * kLoopIters;
}

// AC_LOG=1 in the environment: the physical-step calls print one line per
// step on stderr (read at every call, so a process may switch it).
inline bool log_enabled() {
    const char *e = getenv("AC_LOG");
    return e && e[0] == '1';
}

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(bool pdl, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       Args... args) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    memset(&attr, 0, sizeof attr);
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace acgb
