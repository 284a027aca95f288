// launch.h -- host-side launchers shared between the translation units of
// the library (internal; the public interface is include/convhull.h).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include <utility>

#include "common.cuh"

namespace ch {

int sm_count();

// Launches a kernel that may be put on the SMs before the kernel before it in
// the stream has been retired (kernel_entry waits for it).  The first kernel of
// a call is launched the ordinary way.
template <class... P, class... A>
inline void launch_next(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, A &&...args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);   // (errors: cudaGetLastError)
}

// instrumentation around every launch (probe.cu)
void probe_before(int kid, cudaStream_t st);
// counts `count` kernel launches of kernel id kid (every launcher calls it)
void note_kernels(int kid, int count);
void probe_after(int kid, cudaStream_t st);

// learn_params (the MLP's BF16 parameters, ch_hull_learned): one more block
// runs the learned proposal into the workspace's LearnScratch.
// spec (with build_polygon, on large sets): the speculative single sweep --
// a sample octagon first, then the sweep writes the points it cannot prove
// inside it as candidates; when its last block proves the sample octagon
// inside the final one (Octagon::spec), the filter's passes test only them
cudaError_t launch_extremes(const float *pts, int64_t n, void *ws, const Layout &L, uint32_t *ext8,
                            bool build_polygon, unsigned long long *zero_ptr, int64_t zero_words,
                            cudaStream_t st, bool spec = false, const void *learn_params = nullptr,
                            float *learn_dirs = nullptr, int32_t *learn_k = nullptr);

cudaError_t launch_octagon(const float *pts, int64_t n, const uint32_t *ext8, void *ws, const Layout &L,
                           unsigned long long *zero_ptr, int64_t zero_words, cudaStream_t st);

// point test + stable compaction.  variant: 0 two passes (needs keep_bits in
// L), 1 single pass, -1 the process-wide choice of ch_filter_variant.
// data_extremes: the polygon was built from the data's own extremes
// (ch_extremes_filter), which allows the speculative sweep's candidates;
// otherwise the vertices are the caller's (ch_filter).
cudaError_t launch_filter(const float *pts, int64_t n, void *ws, const Layout &L, uint32_t *surv_idx,
                          float *surv_pts, uint32_t *surv_count, cudaStream_t st, int variant = -1,
                          bool data_extremes = false);
// the hull step's survivors (sort keys and payloads in buffer 0) with the
// single-pass schedule
cudaError_t launch_filter_keys_single(const float *pts, int64_t n, void *ws, const Layout &L, cudaStream_t st);
// the count pass alone (the data's own extremes), for its keep bits; kdev: the
// device's choice of K, 8: the pass returns at once
cudaError_t launch_filter_count(const float *pts, int64_t n, const int32_t *kdev, void *ws, const Layout &L,
                                cudaStream_t st);

// A second polygon of ch_hull (two passes only): the K-direction polygon
// over the octagon's survivors (launch_kx_sv).
struct KgonStage {
    const float *dirs;       // device, K directions (cos, sin)
    const int32_t *kdev;     // device choice of K, or NULL: K below
    int K;                   // 16, 32 or 64 (8: no stage) when kdev is NULL
    uint32_t *ext_out;       // device, K vertex indices, or NULL
};

// the process-wide compaction schedule (ch_filter_variant)
int filter_variant();

// the filter's scatter pass alone, on keep bits, tile counts and block
// totals that a count pass of `grid` blocks (same layout as the filter's)
// left in ws
cudaError_t launch_filter_scatter(const float *pts, int64_t n, int64_t grid, void *ws, const Layout &L,
                                  uint32_t *surv_idx, float *surv_pts, uint32_t *surv_count, bool keys_mode,
                                  cudaStream_t st);

// blocks per SM set by ch_tune_set for a batched kernel (0: built-in choice)
int tune_value(int knob);

// K-direction filter polygon (kfilter.cu): extremes sweep + polygon, then
// the count pass; returns the count grid through *grid (for the scatter)
cudaError_t launch_kx_extremes(const float *pts, int64_t n, const float *dirs, int K, uint32_t *ext_out, void *ws,
                               const Layout &L, cudaStream_t st);
cudaError_t launch_kx_count(const float *pts, int64_t n, int K, void *ws, const Layout &L, int64_t *grid,
                            cudaStream_t st);

// a K-direction polygon over the octagon's survivors, refining the count
// pass's keep bits; K is the host's (16, 32, 64; 8: nothing)
// or, with kdev, the device's choice.  ext_out (nullable): its vertices.
cudaError_t launch_kx_sv(const float *pts, int64_t n, const float *dirs, const int32_t *kdev, int K, uint32_t *ext_out,
                        void *ws, const Layout &L, cudaStream_t st);
// hull step: the survivors of the octagon (or of the second polygon kg),
// less the points inside a fan of triangles around the centre where that
// pays, as sort keys and payloads; their number in Ctrl::surv_count
cudaError_t launch_hull_filter(const float *pts, int64_t n, void *ws, const Layout &L, const KgonStage *kg,
                               cudaStream_t st);

// radix sort of the survivors by x (nothing when one block will sort them)
cudaError_t launch_sort(void *ws, const Layout &L, cudaStream_t st);

// sort, monotone chains and assembly of the hull from the survivors
cudaError_t launch_hull_stage(void *ws, const Layout &L, uint32_t *hull_idx, uint32_t *hull_count, cudaStream_t st);

// ---- many sets (ch_hull_batched); every stage works per set
// validates offsets (points beyond n_cap: CH_ERR_CAPACITY) and maps tiles to sets
cudaError_t launch_bx_setup(const int64_t *offsets, void *ws, const Layout &L, const BatchLayout &BL,
                            int64_t n_cap, cudaStream_t st);
cudaError_t launch_bx_extremes(const float *pts, void *ws, const Layout &L, const BatchLayout &BL, cudaStream_t st);
cudaError_t launch_bx_filter(const float *pts, void *ws, const Layout &L, const BatchLayout &BL, cudaStream_t st);
cudaError_t launch_bx_sort(void *ws, const Layout &L, const BatchLayout &BL, cudaStream_t st);
cudaError_t launch_bx_chain(void *ws, const Layout &L, const BatchLayout &BL, cudaStream_t st);
// copies every set's chains to its part of hull_idx (after hull_offsets)
cudaError_t launch_bx_assemble(void *ws, const Layout &L, const BatchLayout &BL, const int64_t *hull_offsets,
                               uint32_t *hull_idx, cudaStream_t st);
cudaError_t launch_bx_finish(void *ws, const Layout &L, const BatchLayout &BL, uint32_t *hull_idx,
                             int64_t *hull_offsets, cudaStream_t st);

}  // namespace ch
