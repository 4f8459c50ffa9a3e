// Device functions of common.cuh compiled for the CPU: what they load, and by which kind of load.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>
#include <utility>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace {
const float *g_lo, *g_hi;                                // the array that may be read
int g_bad, g_read_only;                                  // loads outside of it; loads by the read-only path
void look(const void *p, size_t n)
{
    const float *f = (const float *)p;
    if (f < g_lo || f + n > g_hi) ++g_bad;
}
}  // namespace

template <typename T> T __ldg(const T *p) { ++g_read_only; look(p, sizeof(T) / sizeof(float)); return *p; }
static inline void atomicCAS(int *, int, int) {}
static inline float __int_as_float(int i) { float f; memcpy(&f, &i, 4); return f; }
template <typename T> T __ldcg(const T *p) { return *p; }
template <typename T> T __shfl_xor_sync(unsigned, T v, int) { return v; }

#undef __noinline__
#define __noinline__
#define __CUDACC__
#include "common.cuh"

extern "C" {

// positions j .. j + 3 of a row [0, hi) into out, loaded as a row that may have been written late (or not): how many loads went by the
// read-only path
int load4(const float *x, int j, int hi, int late, float *out)
{
    g_lo = x;
    g_hi = x + hi;
    g_bad = g_read_only = 0;
    const float4 v = late ? fspad_load4(FspadLateRow{x}, j, hi, -1.0f) : fspad_load4(x, j, hi, -1.0f);
    out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
    return g_bad ? -1 : g_read_only;
}
// whether a late row can come to a load of the read-only path
int late_row_is_a_pointer() { return std::is_convertible<FspadLateRow, const float *>::value; }
int whole_units(int rows, int row, int V, int j0, int n) { return fspad_whole_units(rows, row, V, j0, n); }

}  // extern "C"
