// Rows of the particle records: where a slot lies, and loads of whole columns.
#pragma once

#include "hydro_internal.cuh"

namespace hyd {

// A particle's record.  Its eight (FP64: sixteen) 16-byte columns are stored
// turned by the row's number: slot q of row s lies at q ^ turn.  A row is a
// whole number of 128-byte lines, so in rows laid out alike the same column of
// different particles shares its four banks: a warp's gather of one column took
// about 29 passes through the L1 data stage, which was busy 80 % of the cycles
// of the mixed flux and gradient kernels.  Turned rows spread a gather over all
// banks: flux stage 2.10 -> 1.45 ms (2.10 M particles, MFM), 1.23 -> 0.92 ms
// (1.07 M tube), gradients of the tube 0.865 -> 0.716 ms.
template <typename R>
struct Row {
    R *p;
    unsigned turn;
    __device__ __forceinline__ Row(R *rec, int64_t s)
        : p(rec + s * REC), turn((unsigned)(s & 7) * (16u / (unsigned)sizeof(R))) {}
    __device__ __forceinline__ R &operator[](unsigned q) const { return p[q ^ turn]; }
    // n consecutive slots from q (n * sizeof(R) and q * sizeof(R) multiples of
    // 16, or an aligned part of one column)
    template <typename V>
    __device__ __forceinline__ V get(unsigned q) const {
        return *reinterpret_cast<const V *>(p + (q ^ turn));
    }
};

// the first N (even) slots of row s
template <int N>
__device__ __forceinline__ void load_row(const float *rec, int64_t s, float v[N]) {
    const Row<const float> r(rec, s);
#pragma unroll
    for (int k = 0; k + 4 <= N; k += 4) {
        const float4 t = r.get<float4>(k);
        v[k] = t.x; v[k + 1] = t.y; v[k + 2] = t.z; v[k + 3] = t.w;
    }
    if (N % 4 == 2) {
        const float2 t = r.get<float2>(N - 2);
        v[N - 2] = t.x; v[N - 1] = t.y;
    }
}
template <int N>
__device__ __forceinline__ void load_row(const double *rec, int64_t s, double v[N]) {
    const Row<const double> r(rec, s);
#pragma unroll
    for (int k = 0; k < N; k += 2) {
        const double2 t = r.get<double2>(k);
        v[k] = t.x; v[k + 1] = t.y;
    }
}

}  // namespace hyd
