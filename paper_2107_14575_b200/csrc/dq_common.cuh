// Shared declarations of the CUDA library: the host layout object, the layout
// view kernels receive, and small device helpers.  Nothing here is used by the
// CPU checker.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>
#include <vector>

#include "dq.h"

// ---------------------------------------------------------------- host layout

struct dq_layout {
    int32_t n_seg = 0;
    int32_t bucket = 0;
    int64_t padded = 0;                 // D32
    int64_t nb = 0;                     // buckets per worker
    std::vector<int64_t> seg_elems;     // n_i
    std::vector<int64_t> seg_offset;    // P_i (elements)
    // device table image: three int32 arrays of n_seg + 1 entries each
    //   [0]            first 32-element group of tensor i (last entry: D32/32)
    //   [n_seg+1]      first bucket of tensor i           (last entry: nb)
    //   [2(n_seg+1)]   valid elements of tensor i         (last entry: 0)
    // A whole-tensor layout appends a second image of the same shape whose middle array counts
    // 4096-element pieces instead of buckets (the pieces dq_tensor_norms reduces first).
    std::vector<int32_t> table;
    const int32_t* dev_table = nullptr; // caller-owned copy, set by bind
    int32_t norm = DQ_NORM_L2;          // member of the l_p family the norm calls compute
    bool whole_tensor = false;          // one bucket per non-empty tensor
    int64_t n_pieces = 0;               // whole-tensor layouts: 4096-element pieces per worker
};

// What a kernel needs to map 32-element groups and buckets to tensors.
struct LayoutView {
    int32_t n_seg;
    int32_t groups_per_bucket;   // bucket / 32
    int32_t total_groups;        // D32 / 32
    int32_t nb;                  // buckets per worker
    int32_t seg0_elems;          // valid elements when n_seg == 1
    const int32_t* seg_group0;   // [n_seg + 1]   (NULL when n_seg == 1)
    const int32_t* seg_bucket0;  // [n_seg + 1]
    const int32_t* seg_elems;    // [n_seg + 1]
};

inline LayoutView make_view(const dq_layout* L)
{
    LayoutView v;
    v.n_seg = L->n_seg;
    v.groups_per_bucket = L->bucket / 32;
    v.total_groups = (int32_t)(L->padded / 32);
    v.nb = (int32_t)L->nb;
    v.seg0_elems = (int32_t)L->seg_elems[0];
    v.seg_group0 = L->dev_table;
    v.seg_bucket0 = L->dev_table ? L->dev_table + (L->n_seg + 1) : nullptr;
    v.seg_elems = L->dev_table ? L->dev_table + 2 * (L->n_seg + 1) : nullptr;
    return v;
}

// The same tensors cut into 4096-element pieces (whole-tensor layouts only): the view the
// first kernel of dq_tensor_norms works on.
inline LayoutView make_piece_view(const dq_layout* L)
{
    LayoutView v;
    const int32_t n1 = L->n_seg + 1;
    v.n_seg = L->n_seg;
    v.groups_per_bucket = 128;
    v.total_groups = (int32_t)(L->padded / 32);
    v.nb = (int32_t)L->n_pieces;
    v.seg0_elems = (int32_t)L->seg_elems[0];
    v.seg_group0 = L->dev_table ? L->dev_table + 3 * n1 : nullptr;
    v.seg_bucket0 = L->dev_table ? L->dev_table + 4 * n1 : nullptr;
    v.seg_elems = L->dev_table ? L->dev_table + 5 * n1 : nullptr;
    return v;
}

// Host-side argument checks shared by the entry points.
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int dq_check_common(const dq_layout* L, int32_t M);   // DQ_OK / DQ_ERR_*
int dq_sm_count();                                    // SMs of the current device (cached per device)

#ifdef __CUDACC__

// Every kernel of the library is launched with programmatic stream serialization and begins
// with grid_dependency_wait(): the grid may be set up while the previous kernel of the stream
// is still draining (which hides the launch latency between the calls of a step), and the wait
// returns once that kernel has completed and its writes are visible, so nothing is read or
// written early.  No kernel signals its dependents ahead of its own end.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline void dq_launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    (void)cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);   // the caller reads cudaGetLastError()
}

// Every store of a kernel to global memory goes through DQ_STORE(pointer, value, base, extent in
// bytes, status word).  In the normal build that is the plain store and nothing else is evaluated.
// Built with -DDQ_CHECKED (build.py --checked -> libdq_checked.so) every store first checks that it
// lies inside [base, base + extent) and, if it does not, raises DQ_STAT_INTERNAL instead of storing:
// the stand-in for a memory checker where none can be run.
#ifdef DQ_CHECKED
__device__ __forceinline__ bool dq_store_allowed(const void* p, const int bytes, const void* base, const int64_t extent_bytes,
                                                 int32_t* status)
{
    const int64_t off = reinterpret_cast<const char*>(p) - reinterpret_cast<const char*>(base);
    if (off >= 0 && off + bytes <= extent_bytes) return true;
    atomicOr(status, DQ_STAT_INTERNAL);
    return false;
}
template <class T>
__device__ __forceinline__ void dq_checked_store(T* p, const T& v, const void* base, const int64_t extent_bytes, int32_t* status)
{
    if (dq_store_allowed(p, (int)sizeof(T), base, extent_bytes, status)) *p = v;
}
#define DQ_STORE(p, v, base, extent_bytes, status) dq_checked_store((p), (v), (base), (int64_t)(extent_bytes), (status))
#else
#define DQ_STORE(p, v, base, extent_bytes, status) (*(p) = (v))
#endif

// Index of the last of n entries (non-decreasing, entry 0 <= x) that is <= x, found by the warp together: 32
// entries are looked at a step, so that 1023 tensors take two steps and not ten.  start(i) is entry i.
// Tensors of zero size repeat a start; the last repeat is the non-empty one.
template <class Start>
__device__ __forceinline__ int last_not_above_by_warp(const int x, const int n, const Start& start)
{
    const int lane = threadIdx.x & 31;
    int lo = 0, len = n, stride;
    do {
        stride = (len + 31) >> 5;
        const int at = lane * stride;
        const uint32_t below = __ballot_sync(0xffffffffu, at < len && start(lo + at) <= x);
        const int skip = (__popc(below) - 1) * stride;
        lo += skip;
        len = len - skip < stride ? len - skip : stride;
    } while (stride > 1);
    return lo;
}

#endif  // __CUDACC__
