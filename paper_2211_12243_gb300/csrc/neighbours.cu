// Bucketed neighbour search (§2.2.3).  The Morton-sorted particles are cut
// into buckets of 32 (one warp each); buckets are grouped 32 at a time into
// a fixed-arity bounding-box tree per periodic box.  One warp walks the tree
// once for its whole bucket (the paper's single search per bucket).  The
// particles of the candidate buckets near the owners' boxes are collected
// into tiles of 32 in shared memory; every lane tests a full tile against
// its own particle and appends the matches to its fixed-stride row of the
// list (or, for long lists, the overflow region).
//
// Membership r_ij < h_search,i is decided exactly as the definition states
// in double precision: a float test on the fixed-point separation settles
// every candidate outside a band around the boundary that covers the float
// error, and the rest are re-tested with the double-precision minimum image.
#include "hydro_internal.cuh"

namespace hyd {

namespace {

constexpr int LIST_WARPS = 4;
constexpr int LIST_CTAS = 6;   // resident CTAs per SM (80 registers; 5: 4 % slower, 8: -1 to +10 %)
constexpr int STACK = 256;

// Squared lengths below the normal floats (a unit of length so large that h is
// below 1e-19) carry an absolute error of a few of the smallest subnormals: every
// pair of a radius with a square below BAND_MIN2 is decided in double, and
// CULL_MIN2 widens the culls (by nothing where the square is a normal float).
constexpr float BAND_MIN2 = 1e-30f;
constexpr float CULL_MIN2 = 8e-45f;

__device__ __forceinline__ uint32_t wmin(uint32_t v) {
    for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ uint32_t wmax(uint32_t v) {
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float wmaxf(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// level 0: bucket boxes from the particles; lo.w the largest search
// radius hs, hi.w the largest smoothing length h (both rounded up)
__global__ void k_aabb_leaf(int64_t nbucket, const int32_t *__restrict__ first,
                            const int32_t *__restrict__ cnt, const uint32_t *__restrict__ qx,
                            const uint32_t *__restrict__ qy, const uint32_t *__restrict__ qz,
                            const double *__restrict__ hs, const double *__restrict__ hh,
                            uint4 *__restrict__ lo, uint4 *__restrict__ hi) {
    int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (b >= nbucket) return;
    int f = first[b], c = cnt[b];
    uint32_t x0 = 0xffffffffu, y0 = 0xffffffffu, z0 = 0xffffffffu, x1 = 0, y1 = 0, z1 = 0;
    float h = 0.f, hm = 0.f;
    if (lane < c) {
        int s = f + lane;
        x0 = x1 = qx[s];
        y0 = y1 = qy[s];
        z0 = z1 = qz[s];
        h = __double2float_ru(hs[s]);
        hm = __double2float_ru(hh[s]);
    }
    x0 = wmin(x0); y0 = wmin(y0); z0 = wmin(z0);
    x1 = wmax(x1); y1 = wmax(y1); z1 = wmax(z1);
    h = wmaxf(h);
    hm = wmaxf(hm);
    if (lane == 0) {
        lo[b] = make_uint4(x0, y0, z0, __float_as_uint(h));
        hi[b] = make_uint4(x1, y1, z1, __float_as_uint(hm));
    }
}

// level >= 1: union of the children's boxes
__global__ void k_aabb_node(int64_t node0, int64_t nnode, const int32_t *__restrict__ first,
                            const int32_t *__restrict__ cnt, uint4 *__restrict__ lo,
                            uint4 *__restrict__ hi) {
    int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (k >= nnode) return;
    int64_t node = node0 + k;
    int f = first[node], c = cnt[node];
    uint32_t x0 = 0xffffffffu, y0 = 0xffffffffu, z0 = 0xffffffffu, x1 = 0, y1 = 0, z1 = 0;
    float h = 0.f, hm = 0.f;
    if (lane < c) {
        uint4 a = lo[f + lane], b = hi[f + lane];
        x0 = a.x; y0 = a.y; z0 = a.z; h = __uint_as_float(a.w);
        x1 = b.x; y1 = b.y; z1 = b.z; hm = __uint_as_float(b.w);
    }
    x0 = wmin(x0); y0 = wmin(y0); z0 = wmin(z0);
    x1 = wmax(x1); y1 = wmax(y1); z1 = wmax(z1);
    h = wmaxf(h);
    hm = wmaxf(hm);
    if (lane == 0) {
        lo[node] = make_uint4(x0, y0, z0, __float_as_uint(h));
        hi[node] = make_uint4(x1, y1, z1, __float_as_uint(hm));
    }
}

// Raise the bounds of the buckets holding the particles idx[0 .. *nidx):
// lo.w to at least their search radius hs, hi.w to at least their h.  In a
// guard round only those particles' radii move, so the tree built before
// the rounds stays exact in its boxes and an upper bound in .w (a bound
// that stays above a radius that shrank only prunes less); the node levels
// are then recomputed from the buckets.  Positive floats order like their
// bit patterns, so the maximum is an integer atomic.  A particle's bucket is
// the last one whose first particle is at or before it (buckets are
// consecutive and non-empty).
__global__ void k_aabb_raise(const int32_t *__restrict__ idx, const int *__restrict__ nidx,
                             const int32_t *__restrict__ first, int64_t nbucket,
                             const double *__restrict__ hs, const double *__restrict__ hh,
                             uint4 *__restrict__ lo, uint4 *__restrict__ hi) {
    const int ni = *nidx;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < ni; t += gridDim.x * blockDim.x) {
        const int s = idx[t];
        int64_t a = 0, b = nbucket - 1;
        while (a < b) {
            const int64_t m = (a + b + 1) >> 1;
            if (first[m] <= s) a = m; else b = m - 1;
        }
        atomicMax(&lo[a].w, __float_as_uint(__double2float_ru(hs[s])));
        atomicMax(&hi[a].w, __float_as_uint(__double2float_ru(hh[s])));
    }
}

// Lower bound of the periodic distance (fixed-point units) between the
// intervals [a0,a1] and [b0,b1] on the circle of 2^32 units: the circular
// distance of the centres minus both half-widths (rounded up), in 32-bit
// integers only (64-bit conversions would run on the FP64 pipe).
__device__ __forceinline__ uint32_t axis_gap(uint32_t a0, uint32_t a1, uint32_t b0, uint32_t b1) {
    uint32_t wa = (a1 - a0 + 1u) >> 1, wb = (b1 - b0 + 1u) >> 1;
    uint32_t ca = a0 + ((a1 - a0) >> 1), cb = b0 + ((b1 - b0) >> 1);
    int32_t dc = (int32_t)(cb - ca);
    uint32_t d = dc < 0 ? (uint32_t)(-(int64_t)dc) : (uint32_t)dc;
    uint32_t w = wa + wb + 2u;
    return d > w ? d - w : 0u;
}

__device__ __forceinline__ bool boxes_near(uint4 alo, uint4 ahi, uint4 blo, uint4 bhi,
                                           const Box &bx, float rad2) {
    float gx = (float)axis_gap(alo.x, ahi.x, blo.x, bhi.x) * bx.s[0];
    float gy = (float)axis_gap(alo.y, ahi.y, blo.y, bhi.y) * bx.s[1];
    float gz = (float)axis_gap(alo.z, ahi.z, blo.z, bhi.z) * bx.s[2];
    return gx * gx + gy * gy + gz * gz <= rad2;
}

struct ListArgs {
    int64_t nbucket;         // buckets to build (of the queue in modes 1, 2)
    const int32_t *node_first, *node_cnt, *node_box, *box_root;
    int64_t nbucket_total;   // node ids below this are buckets
    const uint4 *lo, *hi;
    const uint32_t *qx, *qy, *qz;
    const double *xs, *ys, *zs, *hs;
    const Box *boxes;
    int32_t *nbr_idx;
    int64_t *nbr_off;
    int32_t *nbr_cnt;
    int64_t capacity;
    DevCounters *cnt;
    int cap;   // fixed slots per particle (row s at s cap)
    const int32_t *rows_of; // LIST_ROWS: only these nbucket buckets (NULL: all)
    int32_t *ovf_list;      // queued bucket ids
    int *ovf_count;
    bool nq_dev;            // modes 1, 2: the queue's length is *ovf_count
};

// What a pass of k_build_lists does
enum : int {
    LIST_ROWS = 0,    // write the fixed-stride rows (a bucket with a row longer
                      // than cap is queued in ovf_list)
    LIST_COUNT = 1,   // count and reserve storage (queued buckets)
    LIST_FILL = 2     // write at nbr_off (queued buckets)
};

__device__ __forceinline__ float u2f(uint32_t v) {
    return fmaf(i2f_small((int32_t)(v >> 11)), 2048.0f, i2f_small((int32_t)(v & 0x7FFu)));
}

// circular gap (fixed-point units) between a point and an interval
__device__ __forceinline__ uint32_t point_gap(uint32_t p, uint32_t b0, uint32_t b1) {
    uint32_t w = (b1 - b0 + 1u) >> 1, c = b0 + ((b1 - b0) >> 1);
    int32_t d = (int32_t)(c - p);
    uint32_t e = d < 0 ? 0u - (uint32_t)d : (uint32_t)d;
    return e > w + 2u ? e - w - 2u : 0u;
}

// two floats side by side: one instruction for both
struct Pair {
    unsigned long long v;
};
__device__ __forceinline__ Pair pair(float a, float b) {
    Pair p;
    asm("mov.b64 %0, {%1, %2};" : "=l"(p.v) : "f"(a), "f"(b));
    return p;
}
__device__ __forceinline__ void halves(Pair p, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p.v));
}
__device__ __forceinline__ Pair add2(Pair a, Pair b) {
    Pair p;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(p.v) : "l"(a.v), "l"(b.v));
    return p;
}
__device__ __forceinline__ Pair mul2(Pair a, Pair b) {
    Pair p;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(p.v) : "l"(a.v), "l"(b.v));
    return p;
}
__device__ __forceinline__ Pair fma2(Pair a, Pair b, Pair c) {
    Pair p;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(p.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return p;
}

// The warp's candidates, a ring of two tiles of 32: positions relative to the
// bucket's corner (or the fixed-point ones) and sorted indices;
// and the boxes its owners are culled by
struct Tiles {
    alignas(16) float x[64];
    alignas(16) float y[64];
    alignas(16) float z[64];
    alignas(16) int32_t j[64];
    int32_t stack[STACK];
    uint4 lo[2], hi[2];      // fixed-point corners; .w: largest radius
    // per axis both relative centres and both half widths, negated; the squared
    // reaches
    alignas(16) float2 ctr[3][2];
    float2 reach2;
};

// r < hs decided as the definition states it
__device__ __forceinline__ bool list_exact(const ListArgs &a, const Box &bx, int s, int j) {
    const double ex = fold64(__dsub_rn(a.xs[j], a.xs[s]), bx.L[0]);
    const double ey = fold64(__dsub_rn(a.ys[j], a.ys[s]), bx.L[1]);
    const double ez = fold64(__dsub_rn(a.zs[j], a.zs[s]), bx.L[2]);
    const double h = a.hs[s];
    return r2_exact(ex, ey, ez) < __dmul_rn(h, h);
}

// Neighbour lists: a warp takes 32 / SPLIT owners of a bucket, each held by
// SPLIT lanes.  One walk of the tree finds the buckets near the owners'
// boxes; their particles near those boxes are collected into tiles of 32 in
// shared memory, and a full tile is tested by all owners: four candidates a
// broadcast read, the distances two at a time, two comparisons and one bit of
// the lane's member mask each, without a branch (lane group g of an owner takes
// the g-th part of the tile).  The masks then give the members in the candidates' order,
// which is the walk's -- internal nodes last pushed first, buckets in
// ascending order -- whatever the split.
//
// Bound by instruction issue (about 8 instructions per candidate and warp, 5 to
// append it, 75 per staged bucket of 32; one distance at a time, appends in a
// loop over the mask's bits and exact position differences: 1.35 -> 1.15 ms for
// the 128^3 lattice, 1.05 -> 0.93 for the tube, 3.94 -> 3.45 for 4 M log-normal).
// Measured against lanes that each decided and appended one candidate at a
// time, the owners culled by one box and the band 1e-4 wide (neighbour stage
// with sort and gathers, 1 GB300): 128^3 lattice at 1.15 h 4.99 -> 1.47 ms (its
// fifth lattice shell lies within 1e-4 of the radius, so the FP64 re-tests
// took 72 % of the time), 1.07 M tube at 1.05 h 1.84 -> 1.14 ms, log-normal
// box of 4 M at 1.05 h 6.5 -> 4.15 ms (two boxes instead of one: 20.8 ms with
// one, whose few straddling buckets collected whole octants).  A warp per
// (owner, bucket) pair with the bucket's particles on the lanes was slower
// (128^3: 7.1 ms).  SPLIT > 1 shortens the serial walk of grids that leave the
// GPU idle: 16^3 box 0.21 -> 0.12 ms.
template <int MODE, int SPLIT>
__global__ void __launch_bounds__(LIST_WARPS * 32, LIST_CTAS) k_build_lists(ListArgs a) {
    constexpr int OW = 32 / SPLIT;            // owners of a warp
    __shared__ Tiles tiles_all[LIST_WARPS];
    __shared__ int over_all[LIST_WARPS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Tiles &W = tiles_all[warp];
    const unsigned lt = (1u << lane) - 1u;
    const int ol = lane & (OW - 1), slot = lane / OW;
    const int64_t nb = MODE != LIST_ROWS && a.nq_dev ? (int64_t)*a.ovf_count : a.nbucket;
    const int64_t nitem = nb * SPLIT;
    for (int64_t item0 = blockIdx.x * (int64_t)LIST_WARPS; item0 < nitem;
         item0 += gridDim.x * (int64_t)LIST_WARPS) {
        const int64_t item = item0 + warp;
        int64_t b = item / SPLIT;
        const int sub = SPLIT > 1 ? (int)(item % SPLIT) * OW : 0;
        const bool valid = item < nitem;
        if (valid && MODE != LIST_ROWS) b = a.ovf_list[b];
        if (valid && MODE == LIST_ROWS && a.rows_of) b = a.rows_of[b];
        const int bcnt = valid ? a.node_cnt[b] : 0;
        bool over = false;
        // (warp-uniform; the warps of a CTA meet at the end of LIST_ROWS)
        if (bcnt > sub) {
            const int f0 = a.node_first[b] + sub, nown = min(OW, bcnt - sub);
            const int bid = a.node_box[b];
            const Box bx = a.boxes[bid];
            const uint4 corner = a.lo[b];
            const uint32_t ox = corner.x, oy = corner.y, oz = corner.z;
            const bool own = ol < nown;
            const int s = f0 + min(ol, nown - 1);   // (the lanes past the owners repeat the last)
            const uint32_t sqx = a.qx[s], sqy = a.qy[s], sqz = a.qz[s];
            const double hs = a.hs[s];
            const float hf = (float)hs;
            const float rx = qdiff(ox, sqx, bx.s[0]), ry = qdiff(oy, sqy, bx.s[1]),
                        rz = qdiff(oz, sqz, bx.s[2]);
            // The owners' two boxes (fixed-point corners, largest radius).  A run
            // of Morton-ordered particles that crosses a high-level cell
            // boundary spans a box that may cover much of the domain; cut where
            // consecutive owners differ in their highest coordinate bit, both
            // parts are compact.
            int cut;
            {
                const uint32_t nx = __shfl_down_sync(0xffffffffu, sqx, 1);
                const uint32_t ny = __shfl_down_sync(0xffffffffu, sqy, 1);
                const uint32_t nz = __shfl_down_sync(0xffffffffu, sqz, 1);
                const uint32_t gap = lane < nown - 1 ? (sqx ^ nx) | (sqy ^ ny) | (sqz ^ nz) : 0u;
                const uint32_t top = __reduce_max_sync(0xffffffffu, gap);
                cut = __ffs(__ballot_sync(0xffffffffu, gap == top));   // owners [0, cut) and the rest
            }
            // (the culls take the largest radius by its bits: -0, a negative one and NaN,
            // whose bits are above every radius's, reach nothing)
            const float hru = __double2float_ru(hs);
            const uint32_t hbits = hru > 0.f ? __float_as_uint(hru) : 0u;
            uint4 qlo, qhi;
            __syncwarp();
#pragma unroll
            for (int t = 0; t < 2; t++) {
                // (the lanes of the other part repeat one of this part's; a
                // second part without owners repeats the last owner.  With
                // SPLIT > 1 the lanes from OW on hold all the item's owners
                // again, so its second box spans both parts: no cut there)
                const int src = t == 0 ? min(lane, cut - 1) : max(lane, min(cut, nown - 1));
                const uint32_t x = __shfl_sync(0xffffffffu, sqx, src);
                const uint32_t y = __shfl_sync(0xffffffffu, sqy, src);
                const uint32_t z = __shfl_sync(0xffffffffu, sqz, src);
                const uint32_t r = __shfl_sync(0xffffffffu, hbits, src);
                uint4 lo, hi;
                lo.x = __reduce_min_sync(0xffffffffu, x); hi.x = __reduce_max_sync(0xffffffffu, x);
                lo.y = __reduce_min_sync(0xffffffffu, y); hi.y = __reduce_max_sync(0xffffffffu, y);
                lo.z = __reduce_min_sync(0xffffffffu, z); hi.z = __reduce_max_sync(0xffffffffu, z);
                lo.w = hi.w = __reduce_max_sync(0xffffffffu, r);
                if (lane == 0) { W.lo[t] = lo; W.hi[t] = hi; }
                if (t == 0) { qlo = lo; qhi = hi; }
                else {
                    qlo.x = min(qlo.x, lo.x); qlo.y = min(qlo.y, lo.y); qlo.z = min(qlo.z, lo.z);
                    qhi.x = max(qhi.x, hi.x); qhi.y = max(qhi.y, hi.y); qhi.z = max(qhi.z, hi.z);
                    qlo.w = max(qlo.w, lo.w);
                }
            }
            __syncwarp();
            const float qh = __uint_as_float(qlo.w);
            const float rad2 = (qh * 1.00001f) * (qh * 1.00001f) + CULL_MIN2;
            const float Lmax = (float)fmax(bx.L[0], fmax(bx.L[1], bx.L[2]));
            // Coordinates relative to the bucket's corner: their differences
            // are one periodic image, the nearest one for every pair within
            // the radius while the owners' box (seen from the corner) plus
            // the radius stays below half a period; another image only makes
            // a candidate look farther.
            float big;
            bool rel;
            {
                const float ex = u2f(qhi.x - ox) * bx.s[0], ey = u2f(qhi.y - oy) * bx.s[1],
                            ez = u2f(qhi.z - oz) * bx.s[2];
                big = fmaxf(ex, fmaxf(ey, ez)) + qh;
                rel = ex + qh < 0.49f * (float)bx.L[0] && ey + qh < 0.49f * (float)bx.L[1] &&
                      ez + qh < 0.49f * (float)bx.L[2];
            }
            // The band around hs^2 inside which a float distance does not
            // decide: at r = hs the relative error of r^2 is at most 8.3e-7 X / hs
            // (both coordinates, up to X, rounded twice to 2^-24; three axes) +
            // 8e-10 L / hs (positions cut to L / 2^32) + 5e-7 (the scale's, the
            // difference's, the squares' and the radius's rounding); twice that
            // is taken.  Without relative coordinates X is the
            // separation itself.
            const float ihf = 1.f / hf;
            const float eps = 2e-6f * (rel ? big : hf) * ihf + 2e-9f * Lmax * ihf + 1e-6f;
            float lo2 = hf * hf * (1.0f - eps), hi2 = hf * hf * (1.0f + eps);
            if (!(eps < 0.1f && hf * hf > BAND_MIN2)) { lo2 = -1.0f; hi2 = 3.0e38f; }   // (every pair exactly)
            // the boxes in relative coordinates, their reach widened likewise
            if (lane < 2) {
                const uint4 lo = W.lo[lane], hi = W.hi[lane];
                const float x0 = u2f(lo.x - ox) * bx.s[0], x1 = u2f(hi.x - ox) * bx.s[0];
                const float y0 = u2f(lo.y - oy) * bx.s[1], y1 = u2f(hi.y - oy) * bx.s[1];
                const float z0 = u2f(lo.z - oz) * bx.s[2], z1 = u2f(hi.z - oz) * bx.s[2];
                const float h = __uint_as_float(lo.w);
                const float reach = h + (4e-6f * big + 2e-9f * Lmax + 1e-5f * h);
                auto put = [&](int q, float v0, float v1) {
                    (&W.ctr[q][0].x)[lane] = -0.5f * (v0 + v1);
                    (&W.ctr[q][1].x)[lane] = -0.5f * (v1 - v0);
                };
                put(0, x0, x1);
                put(1, y0, y1);
                put(2, z0, z1);
                (&W.reach2.x)[lane] = reach * reach + CULL_MIN2;
            }
            __syncwarp();
            int32_t *const row =
                MODE == LIST_FILL ? a.nbr_idx + a.nbr_off[s] : a.nbr_idx + (int64_t)s * a.cap;
            // (a reservation that did not fit -- the capacity flag is set and
            // the host rebuilds -- must not write past the buffer)
            const int lim = MODE == LIST_FILL
                ? (int)max((int64_t)0, min(a.capacity - a.nbr_off[s], (int64_t)0x7fffffff))
                : a.cap;
            int count = 0;   // members of the owner's list so far
            int head = 0, fill = 0;   // the ring's first tile (0 or 32) and candidates in it

            // the members among the n <= 32 candidates from `head` (the slots of a
            // short tile past them hold whatever was there before)
            auto test_tile = [&](int n) {
                constexpr int PER = 32 / SPLIT;
                const int t0 = head + slot * PER;
                unsigned in = 0, amb = 0;
                if (rel) {
                    const Pair mx = pair(-rx, -rx), my = pair(-ry, -ry), mz = pair(-rz, -rz);
#pragma unroll
                    for (int k = 0; k < PER; k += 4) {
                        const float4 X = *reinterpret_cast<const float4 *>(W.x + t0 + k);
                        const float4 Y = *reinterpret_cast<const float4 *>(W.y + t0 + k);
                        const float4 Z = *reinterpret_cast<const float4 *>(W.z + t0 + k);
                        float r2[4];
#pragma unroll
                        for (int u = 0; u < 4; u += 2) {
                            const Pair dx = add2(u ? pair(X.z, X.w) : pair(X.x, X.y), mx);
                            const Pair dy = add2(u ? pair(Y.z, Y.w) : pair(Y.x, Y.y), my);
                            const Pair dz = add2(u ? pair(Z.z, Z.w) : pair(Z.x, Z.y), mz);
                            halves(fma2(dz, dz, fma2(dy, dy, mul2(dx, dx))), r2[u], r2[u + 1]);
                        }
#pragma unroll
                        for (int u = 0; u < 4; u++) {
                            if (r2[u] <= hi2) in |= 1u << (k + u);
                            if (r2[u] <= hi2 && r2[u] >= lo2) amb |= 1u << (k + u);
                        }
                    }
                } else {
#pragma unroll 4
                    for (int k = 0; k < PER; k++) {
                        const float dx = qdiff(sqx, __float_as_uint(W.x[t0 + k]), bx.s[0]);
                        const float dy = qdiff(sqy, __float_as_uint(W.y[t0 + k]), bx.s[1]);
                        const float dz = qdiff(sqz, __float_as_uint(W.z[t0 + k]), bx.s[2]);
                        const float r2 = dx * dx + dy * dy + dz * dz;
                        if (r2 <= hi2) in |= 1u << k;
                        if (r2 <= hi2 && r2 >= lo2) amb |= 1u << k;
                    }
                }
                if (n < 32) {
                    const unsigned have = ((1u << n) - 1u) >> (slot * PER);
                    in &= have;
                    amb &= have;
                }
                const int32_t *J = W.j + t0;
                while (amb) {   // within the float band: decide in double
                    const int k = __ffs(amb) - 1;
                    amb &= amb - 1;
                    if (!list_exact(a, bx, s, J[k])) in &= ~(1u << k);
                }
                int pos = count, tot = __popc(in);
                if (SPLIT > 1) {   // after the members the owner's lower lanes found
                    const int mine = tot;
                    tot = 0;
#pragma unroll
                    for (int t = 0; t < SPLIT; t++) {
                        const int c = __shfl_sync(0xffffffffu, mine, t * OW + ol);
                        if (t < slot) pos += c;
                        tot += c;
                    }
                }
                count += tot;
                if (MODE != LIST_COUNT && own) {
                    if (pos + __popc(in) <= lim) {
                        // (a tile near the owners has members of nearly every
                        // candidate: no loop over the bits)
                        int32_t *p = row + pos;
#pragma unroll
                        for (int k = 0; k < PER; k += 4) {
                            const int4 j = *reinterpret_cast<const int4 *>(J + k);
                            if (in & (1u << k)) *p++ = j.x;
                            if (in & (2u << k)) *p++ = j.y;
                            if (in & (4u << k)) *p++ = j.z;
                            if (in & (8u << k)) *p++ = j.w;
                        }
                        in = 0;
                    }
                    while (in) {
                        const int k = __ffs(in) - 1;
                        in &= in - 1;
                        if (pos < lim) row[pos] = J[k];
                        pos++;
                    }
                }
                __syncwarp();
                head ^= 32;
                fill -= 32;
            };

            // one bucket's particles (lane k: particle cf + k): those near the
            // owners' boxes join the ring
            auto stage = [&](int cf, int cc, uint32_t px, uint32_t py, uint32_t pz) {
                bool keep = false;
                float3 c;
                if (rel) {
                    // (two roundings: the band allows for both)
                    c = make_float3((float)(int32_t)(px - ox) * bx.s[0],
                                    (float)(int32_t)(py - oy) * bx.s[1],
                                    (float)(int32_t)(pz - oz) * bx.s[2]);
                    // both boxes at once
                    auto gap = [&](float v, int q) {
                        const float4 m = *reinterpret_cast<const float4 *>(W.ctr[q]);
                        float a0, a1;
                        halves(add2(pair(v, v), pair(m.x, m.y)), a0, a1);
                        halves(add2(pair(fabsf(a0), fabsf(a1)), pair(m.z, m.w)), a0, a1);
                        return pair(fmaxf(a0, 0.f), fmaxf(a1, 0.f));
                    };
                    const Pair gx = gap(c.x, 0), gy = gap(c.y, 1), gz = gap(c.z, 2);
                    const float2 lim2 = W.reach2;
                    float g0, g1;
                    halves(fma2(gz, gz, fma2(gy, gy, mul2(gx, gx))), g0, g1);
                    keep = g0 <= lim2.x || g1 <= lim2.y;
                } else {
                    c = make_float3(__uint_as_float(px), __uint_as_float(py), __uint_as_float(pz));
                    const float gx = u2f(point_gap(px, qlo.x, qhi.x)) * bx.s[0];
                    const float gy = u2f(point_gap(py, qlo.y, qhi.y)) * bx.s[1];
                    const float gz = u2f(point_gap(pz, qlo.z, qhi.z)) * bx.s[2];
                    keep = gx * gx + gy * gy + gz * gz <= rad2;
                }
                keep = keep && lane < cc;
                const unsigned m = __ballot_sync(0xffffffffu, keep);
                if (keep) {
                    const int at = (head + fill + __popc(m & lt)) & 63;
                    W.x[at] = c.x;
                    W.y[at] = c.y;
                    W.z[at] = c.z;
                    W.j[at] = cf + lane;
                }
                fill += __popc(m);
                __syncwarp();
                if (fill >= 32) test_tile(32);
            };

            const int root = a.box_root[bid];
            int sp = 0;
            __syncwarp();
            if (root < a.nbucket_total) {
                // the whole box is one bucket
                const int rf = a.node_first[root], rc = a.node_cnt[root];
                const int j = rf + min(lane, rc - 1);
                stage(rf, rc, a.qx[j], a.qy[j], a.qz[j]);
            } else {
                if (lane == 0) W.stack[0] = root;
                sp = 1;
            }
            __syncwarp();
            while (sp > 0) {
                sp--;
                const int node = W.stack[sp];
                __syncwarp();
                const int nf = a.node_first[node], nc = a.node_cnt[node];
                bool hit = false;
                const int child = nf + lane;
                if (lane < nc) {
                    const uint4 clo = a.lo[child], chi = a.hi[child];
#pragma unroll
                    for (int t = 0; t < 2; t++) {
                        const uint4 lo = W.lo[t];
                        const float h = __uint_as_float(lo.w) * 1.00001f;
                        hit |= boxes_near(lo, W.hi[t], clo, chi, bx, h * h + CULL_MIN2);
                    }
                }
                unsigned m = __ballot_sync(0xffffffffu, hit);
                if (nf < a.nbucket_total) {
                    // children are buckets: the next one's positions are in
                    // flight while one is staged (and a tile tested)
                    if (!m) continue;
                    int cfirst = 0, ccnt = 0;
                    if (hit) { cfirst = a.node_first[child]; ccnt = a.node_cnt[child]; }
                    int k = __ffs(m) - 1;
                    m &= m - 1;
                    int cf = __shfl_sync(0xffffffffu, cfirst, k), cc = __shfl_sync(0xffffffffu, ccnt, k);
                    int j = cf + min(lane, cc - 1);
                    uint32_t px = a.qx[j], py = a.qy[j], pz = a.qz[j];
                    for (;;) {
                        const bool more = m != 0;
                        k = more ? __ffs(m) - 1 : 0;
                        m &= m - 1;
                        const int cf1 = __shfl_sync(0xffffffffu, cfirst, k);
                        const int cc1 = __shfl_sync(0xffffffffu, ccnt, k);
                        uint32_t px1 = 0, py1 = 0, pz1 = 0;
                        if (more) {
                            j = cf1 + min(lane, cc1 - 1);
                            px1 = a.qx[j]; py1 = a.qy[j]; pz1 = a.qz[j];
                        }
                        stage(cf, cc, px, py, pz);
                        if (!more) break;
                        cf = cf1; cc = cc1;
                        px = px1; py = py1; pz = pz1;
                    }
                } else {
                    const int np = __popc(m);
                    if (sp + np > STACK) {
                        if (lane == 0) set_flag(a.cnt, ST_STACK);
                        break;
                    }
                    if (hit) W.stack[sp + __popc(m & lt)] = child;
                    sp += np;
                    __syncwarp();
                }
            }
            if (fill > 0) test_tile(fill);

            if (MODE == LIST_ROWS) {
                // each particle owns cap slots at s * cap; a longer list sends
                // the whole bucket to the count-then-fill passes (which write
                // nbr_off and nbr_cnt of all its particles)
                over = __any_sync(0xffffffffu, own && count > a.cap);
                if (own && slot == 0 && !over) {
                    a.nbr_off[s] = (int64_t)s * a.cap;
                    a.nbr_cnt[s] = count;
                }
            } else if (MODE == LIST_COUNT) {
                // reserve storage in the overflow region for the warp's lists
                const int mine = own && slot == 0 ? count : 0;
                int incl = mine;
                for (int o = 1; o < 32; o <<= 1) {
                    int t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                const int total = __shfl_sync(0xffffffffu, incl, 31);
                unsigned long long gbase = 0;
                if (lane == 0) gbase = atomicAdd(&a.cnt->list_cursor, (unsigned long long)total);
                gbase = __shfl_sync(0xffffffffu, gbase, 0);
                const bool fits = (int64_t)gbase + total <= a.capacity;
                if (!fits && lane == 0) set_flag(a.cnt, ST_LIST_CAPACITY);
                if (own && slot == 0) {
                    a.nbr_off[s] = (int64_t)gbase + (incl - mine);
                    a.nbr_cnt[s] = fits ? mine : 0;   // (nothing stored for lists that do not fit)
                }
            }
        }
        if (MODE == LIST_ROWS) {
            // a bucket is queued once, by the first of its warps
            if (lane == 0) over_all[warp] = over;
            if (SPLIT > 1) __syncthreads(); else __syncwarp();
            if (valid && lane == 0 && warp % SPLIT == 0) {
                int any = 0;
                for (int t = 0; t < SPLIT; t++) any |= over_all[warp + t];
                if (any) a.ovf_list[atomicAdd(a.ovf_count, 1)] = (int32_t)b;
            }
            if (SPLIT > 1) __syncthreads();
        }
    }
}

// One particle's walk of the tree by a warp: visit(first, count) is called for
// every bucket that `near` (a lane's test of a child's box) lets pass, in the
// order of k_build_lists's walk (internal nodes last pushed first, buckets in
// ascending order), with the lane's particle of the bucket prefetched: the walk
// is a chain of dependent loads, so the next bucket's are issued before one is
// visited.  False when the stack overflowed (cannot happen for trees of
// MAX_LEVELS levels).
struct Spot {
    uint32_t qx, qy, qz;
};

template <typename Near, typename Visit>
__device__ __forceinline__ bool walk_particle(int root, int64_t nbucket, const int32_t *node_first,
                                              const int32_t *node_cnt, const uint4 *lo,
                                              const uint4 *hi, const uint32_t *qx,
                                              const uint32_t *qy, const uint32_t *qz,
                                              int32_t *stack, int depth, Near &&near, Visit &&visit) {
    const int lane = threadIdx.x & 31;
    auto spot = [&](int f, int c) {
        const int j = f + min(lane, c - 1);
        return Spot{qx[j], qy[j], qz[j]};
    };
    if (root < nbucket) {
        const int f = node_first[root], c = node_cnt[root];
        visit(f, c, spot(f, c));
        return true;
    }
    __syncwarp();
    if (lane == 0) stack[0] = root;
    int sp = 1;
    __syncwarp();
    while (sp > 0) {
        sp--;
        const int node = stack[sp];
        __syncwarp();
        const int nf = node_first[node], nc = node_cnt[node];
        bool hit = false;
        int cf = 0, cc = 0;
        if (lane < nc) {
            const uint4 l = lo[nf + lane], u = hi[nf + lane];
            if (nf < nbucket) { cf = node_first[nf + lane]; cc = node_cnt[nf + lane]; }
            hit = near(l, u);
        }
        unsigned m = __ballot_sync(0xffffffffu, hit);
        if (nf < nbucket) {
            if (!m) continue;
            int k = __ffs(m) - 1;
            m &= m - 1;
            int f = __shfl_sync(0xffffffffu, cf, k), c = __shfl_sync(0xffffffffu, cc, k);
            Spot p = spot(f, c);
            for (;;) {
                const bool more = m != 0;
                k = more ? __ffs(m) - 1 : 0;
                m &= m - 1;
                const int f1 = __shfl_sync(0xffffffffu, cf, k), c1 = __shfl_sync(0xffffffffu, cc, k);
                Spot p1 = p;
                if (more) p1 = spot(f1, c1);
                visit(f, c, p);
                if (!more) break;
                f = f1; c = c1; p = p1;
            }
            __syncwarp();
        } else {
            const int nh = __popc(m);
            if (sp + nh > depth) return false;
            if (hit) stack[sp + __popc(m & ((1u << lane) - 1u))] = nf + lane;
            sp += nh;
            __syncwarp();
        }
    }
    return true;
}

// the float band around h^2 for separations from the fixed-point positions
// (k_build_lists says where its width comes from)
__device__ __forceinline__ void point_band(double h, const Box &bx, float &lo2, float &hi2) {
    const float hf = (float)h, ih = 1.f / hf;
    const float eps = 3e-6f + 2e-9f * (float)bx.Lmax * ih;
    lo2 = hf * hf * (1.0f - eps);
    hi2 = hf * hf * (1.0f + eps);
    if (!(eps < 0.1f && hf * hf > BAND_MIN2)) { lo2 = -1.0f; hi2 = 3.0e38f; }
}

// Lists of single particles (the N_cond guard's grown particles, whose
// search radii rose): one warp per particle walks the tree with that
// particle's own sphere -- the lanes test a node's children at once, then a
// bucket's particles at once -- instead of rebuilding the lists of the
// particle's whole bucket at its largest radius.  A list holds the same entries
// in the same order as a bucket rebuild would give it.  The members collect in
// shared memory, then the storage is reserved in the overflow region (flagging
// ST_LIST_CAPACITY when it does not fit) and written; a list longer than the
// buffer is written by a second walk.  Warps stride over the *npidx particles
// of pidx (the count is read on the device); with `active` set, only those
// with an ACT_SOLVE flag (a guard round's re-search: the guard particles
// whose root left their radius), and the search-failure flag that the new
// lists answer is cleared.  Two walks, each waiting for every bucket's loads in
// turn, took 80 us a round on a 500k log-normal box; this takes 34 us.
struct PartListArgs {
    const int32_t *pidx;
    const int *npidx;
    const uint8_t *active;
    const int32_t *node_first, *node_cnt, *box_root, *pbox;
    int64_t nbucket_total;
    const uint4 *lo, *hi;
    const uint32_t *qx, *qy, *qz;
    const double *xs, *ys, *zs, *hs;
    const Box *boxes;
    int32_t *nbr_idx;
    int64_t *nbr_off;
    int32_t *nbr_cnt;
    int64_t capacity;
    DevCounters *cnt;
};

constexpr int PL_WARPS = 4;
constexpr int PL_BUF = 1024;   // members a warp collects in shared memory

__global__ void __launch_bounds__(PL_WARPS * 32) k_particle_lists(PartListArgs a) {
    __shared__ int32_t stack_all[PL_WARPS][STACK], buf_all[PL_WARPS][PL_BUF];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int32_t *stack = stack_all[warp], *buf = buf_all[warp];
    const int np = *a.npidx;
    const int nwarps = gridDim.x * PL_WARPS;
    if (a.active && blockIdx.x == 0 && threadIdx.x == 0) atomicAnd(&a.cnt->flags, ~ST_SEARCH);
    for (int g = blockIdx.x * PL_WARPS + warp; g < np; g += nwarps) {
        const int s = a.pidx[g];
        if (a.active && !(a.active[s] & ACT_SOLVE)) continue;   // (warp-uniform: one particle)
        const Box bx = a.boxes[a.pbox[s]];
        const uint32_t px = a.qx[s], py = a.qy[s], pz = a.qz[s];
        const double x = a.xs[s], y = a.ys[s], z = a.zs[s], hs = a.hs[s];
        const double h2 = __dmul_rn(hs, hs);
        float lo2, hi2;
        point_band(hs, bx, lo2, hi2);
        const int root = a.box_root[a.pbox[s]];
        // one walk: the members to shared memory (dst NULL) or to dst
        int count = 0;
        auto walk = [&](int32_t *dst) {
            count = 0;
            return walk_particle(
                root, a.nbucket_total, a.node_first, a.node_cnt, a.lo, a.hi, a.qx, a.qy, a.qz, stack,
                STACK,
                [&](uint4 l, uint4 u) {
                    const float gx = u2f(point_gap(px, l.x, u.x)) * bx.s[0];
                    const float gy = u2f(point_gap(py, l.y, u.y)) * bx.s[1];
                    const float gz = u2f(point_gap(pz, l.z, u.z)) * bx.s[2];
                    return gx * gx + gy * gy + gz * gz <= hi2;
                },
                [&](int f, int c, const Spot &p) {
                    bool in = false;
                    const int j = f + lane;
                    if (lane < c) {
                        const float dx = qdiff(px, p.qx, bx.s[0]);
                        const float dy = qdiff(py, p.qy, bx.s[1]);
                        const float dz = qdiff(pz, p.qz, bx.s[2]);
                        const float r2 = dx * dx + dy * dy + dz * dz;
                        in = r2 < lo2;
                        if (!in && r2 <= hi2) {   // within the float band: decide in double
                            const double ex = fold64(__dsub_rn(a.xs[j], x), bx.L[0]);
                            const double ey = fold64(__dsub_rn(a.ys[j], y), bx.L[1]);
                            const double ez = fold64(__dsub_rn(a.zs[j], z), bx.L[2]);
                            in = r2_exact(ex, ey, ez) < h2;
                        }
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, in);
                    if (in) {
                        const int pos = count + __popc(m & ((1u << lane) - 1u));
                        if (dst) dst[pos] = j;
                        else if (pos < PL_BUF) buf[pos] = j;
                    }
                    count += __popc(m);
                });
        };
        if (!walk(nullptr)) {
            if (lane == 0) set_flag(a.cnt, ST_STACK);
            continue;
        }
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(&a.cnt->list_cursor, (unsigned long long)count);
        base = __shfl_sync(0xffffffffu, base, 0);
        const bool fits = (int64_t)base + count <= a.capacity;
        if (lane == 0) {
            a.nbr_off[s] = (int64_t)base;
            a.nbr_cnt[s] = fits ? count : 0;   // (nothing stored for a list that does not fit)
            if (!fits) set_flag(a.cnt, ST_LIST_CAPACITY);
        }
        __syncwarp();
        if (fits) {
            if (count <= PL_BUF) {
                for (int k = lane; k < count; k += 32) a.nbr_idx[base + k] = buf[k];
            } else {
                walk(a.nbr_idx + base);
            }
        }
        __syncwarp();
    }
}

__global__ void k_export_count(int64_t n, const int32_t *__restrict__ perm,
                               const int32_t *__restrict__ cnt, int64_t *__restrict__ rowlen) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s < n) rowlen[perm[s]] = cnt[s];
    if (s == n) rowlen[n] = 0;
}

// The lists in the caller's indices, ascending: a warp per row maps its entries
// and puts each at its rank among them (the entries are distinct, so the rank
// is the number of smaller ones; compared from shared memory, 32 entries at a
// time).  One thread per row sorting by insertion in global memory took 3.0 ms
// for 79,507 rows of 141 entries; this takes 0.2 ms.
constexpr int EXPORT_ROW = 1024;   // entries of a row held in shared memory
constexpr int EXPORT_WARPS = 4;

__global__ void __launch_bounds__(EXPORT_WARPS * 32)
k_export_fill(int64_t n, const int32_t *__restrict__ perm, const int64_t *__restrict__ off_in,
              const int32_t *__restrict__ cnt, const int32_t *__restrict__ idx_in,
              const int64_t *__restrict__ off_out, int32_t *__restrict__ idx_out) {
    __shared__ __align__(16) int32_t rows[EXPORT_WARPS][EXPORT_ROW];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t s = blockIdx.x * (int64_t)EXPORT_WARPS + warp;
    if (s >= n) return;
    int32_t *row = rows[warp];
    const int c = cnt[s];
    const int32_t *src = idx_in + off_in[s];
    int32_t *dst = idx_out + off_out[perm[s]];
    const int cs = min(c, EXPORT_ROW);
    for (int k = lane; k < cs; k += 32) row[k] = perm[src[k]];
    // (whole groups of four: the slots past the row hold the largest value)
    if (cs < EXPORT_ROW && lane < ((4 - (cs & 3)) & 3)) row[cs + lane] = INT32_MAX;
    __syncwarp();
    for (int k0 = 0; k0 < c; k0 += 32) {
        const int k = k0 + lane;
        const int32_t v = k >= c ? INT32_MAX : k < EXPORT_ROW ? row[k] : perm[src[k]];
        int rank = 0;
        for (int m = 0; m < cs; m += 4) {
            const int4 r = *reinterpret_cast<const int4 *>(row + m);
            rank += (r.x < v) + (r.y < v) + (r.z < v) + (r.w < v);
        }
        for (int m = EXPORT_ROW; m < c; m++) rank += perm[src[m]] < v;   // (very long rows)
        if (k < c) dst[rank] = v;
    }
}

// queue the buckets holding a particle with one of the bits set (bit 0: to
// search again, and then clear the search-failure flag that the rebuild
// answers)
__global__ void k_queue_active(int64_t nbucket, const int32_t *__restrict__ first,
                               const int32_t *__restrict__ cnt, const uint8_t *__restrict__ active,
                               int32_t *__restrict__ queue, int *__restrict__ nqueue,
                               DevCounters *counters, uint8_t bits = 1) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (bits == 1 && w0 == 0 && lane == 0) atomicAnd(&counters->flags, ~ST_SEARCH);
    // (warps stride over the buckets: a small grid covers every bucket)
    for (int64_t b = w0; b < nbucket; b += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        bool act = lane < cnt[b] && (active[first[b] + lane] & bits);
        if (__any_sync(0xffffffffu, act) && lane == 0) queue[atomicAdd(nqueue, 1)] = (int32_t)b;
    }
}

// The particles that hold a guard particle a in their list, i.e. r_ia < h_i
// (the list's own radius: the reverse of a's list), by one walk of the
// bucket tree per guard particle and warp.  The lanes test the children of
// a node at once: a child is entered when the lower bound of its periodic
// distance from a is within the largest search radius of its particles
// (hs >= h), or (use_h) within their largest h when the tree was built --
// the tighter bound for a guard round, where only the guard particles' h
// moved since, and each of those marks itself; the particles of an entered
// bucket are tested exactly, one per lane (the double-precision membership
// of the lists).  Marks ACT_REDO on them and on a itself.  Warps stride
// over the guard particles, whose count is read on the device.
// a guard round marks by scanning every list when it grew more than
// n / MARK_SCAN_RATIO particles (k_mark_by_lists), else by tree walks
constexpr int MARK_SCAN_RATIO = 1024;

__device__ __forceinline__ bool mark_by_scan(int nguard, int64_t n) {
    return (int64_t)nguard * MARK_SCAN_RATIO > n;
}

constexpr int RSTACK = 320;   // 32-ary tree of at most MAX_LEVELS levels
constexpr int RWARPS = 4;

__global__ void __launch_bounds__(RWARPS * 32)
k_mark_reverse(const int32_t *__restrict__ guard_idx, const int *__restrict__ nguard,
               const int32_t *__restrict__ node_first, const int32_t *__restrict__ node_cnt,
               const int32_t *__restrict__ box_root, int64_t nbucket,
               const uint4 *__restrict__ lo, const uint4 *__restrict__ hi,
               const uint32_t *__restrict__ qx, const uint32_t *__restrict__ qy,
               const uint32_t *__restrict__ qz, const double *__restrict__ xs,
               const double *__restrict__ ys, const double *__restrict__ zs,
               const double *__restrict__ h, const int32_t *__restrict__ pbox,
               const Box *__restrict__ boxes, uint8_t *__restrict__ active, DevCounters *cnt,
               bool use_h, int64_t nparticles) {
    __shared__ int32_t stack_all[RWARPS][RSTACK];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ng = *nguard;
    // (a guard round with many grown particles marks by the list scan below)
    if (use_h && mark_by_scan(ng, nparticles)) return;
    const int nwarps = gridDim.x * RWARPS;
    for (int g = blockIdx.x * RWARPS + warp; g < ng; g += nwarps) {
        const int a = guard_idx[g];
        const Box bx = boxes[pbox[a]];
        const uint32_t pax = qx[a], pay = qy[a], paz = qz[a];
        if (lane == 0) active[a] |= ACT_REDO;
        const bool ok = walk_particle(
            box_root[pbox[a]], nbucket, node_first, node_cnt, lo, hi, qx, qy, qz, stack_all[warp],
            RSTACK,
            [&](uint4 l, uint4 u) {
                const float rmax = __uint_as_float(use_h ? u.w : l.w) * 1.0001f;
                const float gx = u2f(point_gap(pax, l.x, u.x)) * bx.s[0];
                const float gy = u2f(point_gap(pay, l.y, u.y)) * bx.s[1];
                const float gz = u2f(point_gap(paz, l.z, u.z)) * bx.s[2];
                return gx * gx + gy * gy + gz * gz <= rmax * rmax + CULL_MIN2;
            },
            [&](int f, int c, const Spot &p) {
                // lane k tests its particle f + k
                const int i = f + lane;
                if (lane >= c || i == a) return;
                const double hi_ = h[i];
                float lo2, hi2;
                point_band(hi_, bx, lo2, hi2);
                const float dx = qdiff(p.qx, pax, bx.s[0]);
                const float dy = qdiff(p.qy, pay, bx.s[1]);
                const float dz = qdiff(p.qz, paz, bx.s[2]);
                const float r2 = dx * dx + dy * dy + dz * dz;
                bool in = r2 < lo2;
                if (!in && r2 <= hi2) {   // within the float band: decide in double
                    const double ex = fold64(__dsub_rn(xs[a], xs[i]), bx.L[0]);
                    const double ey = fold64(__dsub_rn(ys[a], ys[i]), bx.L[1]);
                    const double ez = fold64(__dsub_rn(zs[a], zs[i]), bx.L[2]);
                    in = r2_exact(ex, ey, ez) < __dmul_rn(hi_, hi_);
                }
                if (in) active[i] |= ACT_REDO;
            });
        if (!ok && lane == 0) set_flag(cnt, ST_STACK);
        __syncwarp();
    }
}

// The same marks from the lists: particle i holds a guard particle a in its
// list iff r_ia < h_i falls within the list's radius, and every list is
// complete for r < h_i (after the density stage it holds its members and a
// few entries just beyond), so scanning each particle's own list for a
// guard flag marks every particle the walk would, plus a few whose
// recomputation gives back their unchanged values.  One pass over all lists
// costs about as much as the walks of n / MARK_SCAN_RATIO guard particles:
// each kernel reads the round's guard count on the device and only one of
// them works (the first round grows many particles, the later ones few).
// Eight lanes read a list together, eight consecutive entries (one 32-byte
// sector) at a time, so a warp scans four lists at once with whole-sector
// reads rather than one scattered entry per lane.
constexpr int MARK_GROUP = 8;

__global__ void __launch_bounds__(256)
k_mark_by_lists(int64_t n, const int *__restrict__ nguard, const int64_t *__restrict__ nbr_off,
                const int32_t *__restrict__ nbr_cnt, const int32_t *__restrict__ nbr_idx,
                const uint32_t *__restrict__ gbits, uint8_t *__restrict__ active) {
    if (!mark_by_scan(*nguard, n)) return;
    constexpr int PER_WARP = 32 / MARK_GROUP;
    const int lane = threadIdx.x & 31, sub = lane & (MARK_GROUP - 1);
    const unsigned gmask = ((1u << MARK_GROUP) - 1u) << (lane & ~(MARK_GROUP - 1));
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t s0 = w * PER_WARP; s0 < n; s0 += nw * PER_WARP) {
        const int64_t s = s0 + lane / MARK_GROUP;
        int64_t o = 0;
        int c = 0;
        bool hit = false;
        if (s < n) {
            o = nbr_off[s];
            c = nbr_cnt[s];
            hit = (gbits[s >> 5] >> (s & 31)) & 1u;   // (a guard particle marks itself)
        }
        const int cmax = __reduce_max_sync(0xffffffffu, hit ? 0 : c);
        for (int k0 = 0; k0 < cmax; k0 += MARK_GROUP) {
            bool h = false;
            if (!hit && k0 + sub < c) {
                const int j = nbr_idx[o + k0 + sub];
                h = (gbits[j >> 5] >> (j & 31)) & 1u;
            }
            hit |= (__ballot_sync(0xffffffffu, h) & gmask) != 0u;
            if (__all_sync(0xffffffffu, hit || k0 + MARK_GROUP >= c)) break;
        }
        if (hit && sub == 0) active[s] |= ACT_REDO;
    }
}

// the guard round's particles as a bitmap (one bit per particle, a 32nd of
// the flag bytes: the scan's lookups stay in L1 and L2)
__global__ void k_guard_bits(const int32_t *__restrict__ guard_idx, const int *__restrict__ nguard,
                             uint32_t *__restrict__ gbits) {
    const int ng = *nguard;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < ng; t += gridDim.x * blockDim.x) {
        const int s = guard_idx[t];
        atomicOr(&gbits[s >> 5], 1u << (s & 31));
    }
}

inline unsigned grid_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t mark_guard_reverse(hydro_ctx *c, stream_t st) {
    HYD_CUDA(mark_reverse(c, st, true));
    const int64_t nw = (c->plan.n + 31) / 32;
    HYD_CUDA(c->d_guard_bits.ensure(nw));
    HYD_CUDA(cudaMemsetAsync(c->d_guard_bits.get(), 0, nw * sizeof(uint32_t), st));
    k_guard_bits<<<152 * 4, 256, 0, st>>>(c->d_guard_idx.get(), &c->d_cnt->nguard,
                                          c->d_guard_bits.get());
    HYD_CUDA(launch_check());
    k_mark_by_lists<<<SWEEP_GRID, 256, 0, st>>>(c->plan.n, &c->d_cnt->nguard, c->d_nbr_off.get(),
                                                c->d_nbr_cnt.get(), c->d_nbr_idx.get(),
                                                c->d_guard_bits.get(), c->d_active.get());
    return launch_check();
}

cudaError_t mark_reverse(hydro_ctx *c, stream_t st, bool use_h) {
    const Plan &P = c->plan;
    // (a latency-bound walk per guard particle: as many resident warps as
    // its 40 registers allow, 12 CTAs of 4 warps per SM)
    k_mark_reverse<<<152 * 12, RWARPS * 32, 0, st>>>(
        c->d_guard_idx.get(), &c->d_cnt->nguard, c->d_node_first.get(), c->d_node_cnt.get(),
        c->d_box_root.get(), P.nbucket, c->d_node_aabb.get(), c->d_node_aabb_hi.get(),
        c->d_qx.get(), c->d_qy.get(), c->d_qz.get(), c->d_xs.get(), c->d_ys.get(), c->d_zs.get(),
        c->d_hsorted.get(), c->d_pbox.get(), c->d_boxes.get(), c->d_active.get(), c->d_cnt,
        use_h, P.n);
    return launch_check();
}

cudaError_t build_tree(hydro_ctx *c, stream_t st) {
    const Plan &P = c->plan;
    k_aabb_leaf<<<grid_for(P.nbucket * 32, 256), 256, 0, st>>>(
        P.nbucket, c->d_node_first.get(), c->d_node_cnt.get(), c->d_qx.get(), c->d_qy.get(),
        c->d_qz.get(), c->d_hs.get(), c->d_hsorted.get(), c->d_node_aabb.get(),
        c->d_node_aabb_hi.get());
    HYD_CUDA(launch_check());
    for (int l = 1; l < P.nlevels; l++) {
        int64_t n0 = P.level_off[l], nn = P.level_off[l + 1] - P.level_off[l];
        k_aabb_node<<<grid_for(nn * 32, 256), 256, 0, st>>>(n0, nn, c->d_node_first.get(),
                                                            c->d_node_cnt.get(),
                                                            c->d_node_aabb.get(),
                                                            c->d_node_aabb_hi.get());
        HYD_CUDA(launch_check());
    }
    return cudaSuccess;
}

// the tree's radius bounds raised for the guard round's particles
// (guard_idx, count nguard on the device), the node levels recomputed
cudaError_t raise_tree(hydro_ctx *c, stream_t st) {
    const Plan &P = c->plan;
    k_aabb_raise<<<152 * 4, 256, 0, st>>>(c->d_guard_idx.get(), &c->d_cnt->nguard,
                                          c->d_node_first.get(), P.nbucket, c->d_hs.get(),
                                          c->d_hsorted.get(), c->d_node_aabb.get(),
                                          c->d_node_aabb_hi.get());
    HYD_CUDA(launch_check());
    for (int l = 1; l < P.nlevels; l++) {
        int64_t n0 = P.level_off[l], nn = P.level_off[l + 1] - P.level_off[l];
        k_aabb_node<<<grid_for(nn * 32, 256), 256, 0, st>>>(n0, nn, c->d_node_first.get(),
                                                            c->d_node_cnt.get(),
                                                            c->d_node_aabb.get(),
                                                            c->d_node_aabb_hi.get());
        HYD_CUDA(launch_check());
    }
    return cudaSuccess;
}

static ListArgs list_args(hydro_ctx *c, int cap) {
    // cap: slots per particle in the fixed-stride part of nbr_idx
    const Plan &P = c->plan;
    ListArgs a;
    a.nbucket = P.nbucket;
    a.node_first = c->d_node_first.get();
    a.node_cnt = c->d_node_cnt.get();
    a.node_box = c->d_node_box.get();
    a.box_root = c->d_box_root.get();
    a.nbucket_total = P.nbucket;
    a.lo = c->d_node_aabb.get();
    a.hi = c->d_node_aabb_hi.get();
    a.qx = c->d_qx.get(); a.qy = c->d_qy.get(); a.qz = c->d_qz.get();
    a.xs = c->d_xs.get(); a.ys = c->d_ys.get(); a.zs = c->d_zs.get();
    a.hs = c->d_hs.get();
    a.boxes = c->d_boxes.get();
    a.nbr_idx = c->d_nbr_idx.get();
    a.nbr_off = c->d_nbr_off.get();
    a.nbr_cnt = c->d_nbr_cnt.get();
    a.capacity = (int64_t)c->d_nbr_idx.cap;
    a.cnt = c->d_cnt;
    a.cap = cap;
    a.rows_of = nullptr;
    a.ovf_list = c->d_ovf.get();
    a.ovf_count = &c->d_cnt->ovf_buckets;
    a.nq_dev = false;
    return a;
}

// warps a bucket is divided among: one while that fills the GPU (24 warps
// on each of the 152 SMs), else four
static int list_split(int64_t nbucket) { return nbucket >= 152 * 24 ? 1 : 4; }

template <int MODE>
static cudaError_t launch_lists(const ListArgs &a, int64_t nbucket, stream_t st) {
    // the queue's length on the device: a grid of 8 CTAs per SM strides over it
    const int split = a.nq_dev ? 4 : list_split(nbucket);
    const int64_t ctas = (nbucket * split + LIST_WARPS - 1) / LIST_WARPS;
    const unsigned grid = (unsigned)(a.nq_dev ? std::min<int64_t>(ctas, 152 * 8) : ctas);
    if (split == 1) k_build_lists<MODE, 1><<<grid, LIST_WARPS * 32, 0, st>>>(a);
    else k_build_lists<MODE, 4><<<grid, LIST_WARPS * 32, 0, st>>>(a);
    return launch_check();
}

// one pass over all buckets; buckets with a row longer than cap are queued
// for build_lists_queued().  Layout of nbr_idx: particle s owns the slots [s cap, s cap + cap); lists
// longer than cap live in the overflow region that follows (n cap onwards),
// reserved by build_lists_queued.
cudaError_t build_lists(hydro_ctx *c, int cap, stream_t st) {
    const int64_t n = c->plan.n;
    HYD_CUDA(c->d_nbr_off.ensure(n + 1));
    HYD_CUDA(c->d_nbr_cnt.ensure(n));
    size_t need = (size_t)n * cap + (size_t)c->ovf_reserve;
    if (c->d_nbr_idx.cap < need) HYD_CUDA(c->d_nbr_idx.ensure(need + need / 8));
    HYD_CUDA(c->d_ovf.ensure(c->plan.nbucket));
    c->list_cap = cap;
    HYD_CUDA(set_u64(&c->d_cnt->list_cursor, (unsigned long long)n * cap, st));
    HYD_CUDA(cudaMemsetAsync(&c->d_cnt->ovf_buckets, 0, sizeof(int), st));
    return launch_lists<LIST_ROWS>(list_args(c, cap), c->plan.nbucket, st);
}

// new rows for nq buckets (their lists may lie anywhere; longer ones go to the
// overflow region, where nothing of a whole build is kept)
cudaError_t build_rows_of(hydro_ctx *c, const int32_t *buckets, int nq, stream_t st) {
    HYD_CUDA(set_u64(&c->d_cnt->list_cursor, (unsigned long long)c->plan.n * c->list_cap, st));
    HYD_CUDA(cudaMemsetAsync(&c->d_cnt->ovf_buckets, 0, sizeof(int), st));
    ListArgs a = list_args(c, c->list_cap);
    a.nbucket = nq;
    a.rows_of = buckets;
    HYD_CUDA(launch_lists<LIST_ROWS>(a, nq, st));
    return build_lists_queued_dev(c, st);
}

// the queued buckets: count and reserve in the overflow region, then fill
cudaError_t build_lists_queued(hydro_ctx *c, int nq, stream_t st) {
    ListArgs a = list_args(c, c->list_cap);
    a.nbucket = nq;   // warps index the queue
    HYD_CUDA(launch_lists<LIST_COUNT>(a, nq, st));
    return launch_lists<LIST_FILL>(a, nq, st);
}

// the queued passes over as many warps as there are buckets; the count of
// queued buckets is read by the warps themselves
cudaError_t build_lists_queued_dev(hydro_ctx *c, stream_t st) {
    ListArgs a = list_args(c, c->list_cap);
    a.nq_dev = true;
    HYD_CUDA(launch_lists<LIST_COUNT>(a, c->plan.nbucket, st));
    return launch_lists<LIST_FILL>(a, c->plan.nbucket, st);
}

cudaError_t rebuild_active_lists_dev(hydro_ctx *c, stream_t st, bool guard) {
    // (in a guard round only guard particles can have left their radius)
    if (guard) return guard_particle_lists(c, st, true);
    const Plan &P = c->plan;
    HYD_CUDA(cudaMemsetAsync(&c->d_cnt->ovf_buckets, 0, sizeof(int), st));
    k_queue_active<<<std::min(grid_for(P.nbucket * 32, 256), SWEEP_GRID), 256, 0, st>>>(
        P.nbucket, c->d_node_first.get(), c->d_node_cnt.get(), c->d_active.get(), c->d_ovf.get(),
        &c->d_cnt->ovf_buckets, c->d_cnt);
    HYD_CUDA(launch_check());
    HYD_CUDA(build_tree(c, st));
    return build_lists_queued_dev(c, st);
}

// new lists (in the overflow region) for the buckets that hold a particle
// whose search radius grew; every other list stays as it is.  *nq receives
// the number of buckets rebuilt (the host waits for it).
cudaError_t rebuild_active_lists(hydro_ctx *c, int *nq, stream_t st, bool guard) {
    if (guard) {
        *nq = 0;   // (no bucket rebuilt: the re-searched particles' own lists)
        return guard_particle_lists(c, st, true);
    }
    const Plan &P = c->plan;
    HYD_CUDA(c->d_ovf.ensure(P.nbucket));
    HYD_CUDA(cudaMemsetAsync(&c->d_cnt->ovf_buckets, 0, sizeof(int), st));
    k_queue_active<<<std::min(grid_for(P.nbucket * 32, 256), SWEEP_GRID), 256, 0, st>>>(
        P.nbucket, c->d_node_first.get(), c->d_node_cnt.get(), c->d_active.get(), c->d_ovf.get(),
        &c->d_cnt->ovf_buckets, c->d_cnt);
    HYD_CUDA(launch_check());
    HYD_CUDA(cudaMemcpyAsync(nq, &c->d_cnt->ovf_buckets, sizeof(int), cudaMemcpyDeviceToHost, st));
    HYD_CUDA(cudaStreamSynchronize(st));
    if (*nq == 0) return cudaSuccess;
    // the buckets' search radii changed
    HYD_CUDA(build_tree(c, st));
    return build_lists_queued(c, *nq, st);
}

// new lists, in the overflow region, for the particles of guard_idx (the
// guard round's grown particles, count nguard on the device; only_search:
// only those flagged ACT_SOLVE by the re-search); the tree must hold the
// current positions (its search radii are not used).  Every other list
// stays as it is, compacted or not: a bucket rebuild would give the
// re-searched particles the same lists.
cudaError_t guard_particle_lists(hydro_ctx *c, stream_t st, bool only_search) {
    const Plan &P = c->plan;
    PartListArgs a;
    a.pidx = c->d_guard_idx.get();
    a.npidx = &c->d_cnt->nguard;
    a.active = only_search ? c->d_active.get() : nullptr;
    a.node_first = c->d_node_first.get();
    a.node_cnt = c->d_node_cnt.get();
    a.box_root = c->d_box_root.get();
    a.pbox = c->d_pbox.get();
    a.nbucket_total = P.nbucket;
    a.lo = c->d_node_aabb.get();
    a.hi = c->d_node_aabb_hi.get();
    a.qx = c->d_qx.get(); a.qy = c->d_qy.get(); a.qz = c->d_qz.get();
    a.xs = c->d_xs.get(); a.ys = c->d_ys.get(); a.zs = c->d_zs.get();
    a.hs = c->d_hs.get();
    a.boxes = c->d_boxes.get();
    a.nbr_idx = c->d_nbr_idx.get();
    a.nbr_off = c->d_nbr_off.get();
    a.nbr_cnt = c->d_nbr_cnt.get();
    a.capacity = (int64_t)c->d_nbr_idx.cap;
    a.cnt = c->d_cnt;
    k_particle_lists<<<152 * 8, PL_WARPS * 32, 0, st>>>(a);
    return launch_check();
}

cudaError_t queue_flagged(hydro_ctx *c, uint8_t bits, stream_t st) {
    const Plan &P = c->plan;
    HYD_CUDA(c->d_ovf.ensure(P.nbucket));
    HYD_CUDA(cudaMemsetAsync(&c->d_cnt->ovf_buckets, 0, sizeof(int), st));
    k_queue_active<<<std::min(grid_for(P.nbucket * 32, 256), SWEEP_GRID), 256, 0, st>>>(
        P.nbucket, c->d_node_first.get(), c->d_node_cnt.get(), c->d_active.get(), c->d_ovf.get(),
        &c->d_cnt->ovf_buckets, c->d_cnt, bits);
    return launch_check();
}

cudaError_t export_lists(hydro_ctx *c, hydro_nbrlist *out, stream_t st) {
    const int64_t n = c->plan.n;
    HYD_CUDA(c->d_scan_tmp.ensure((size_t)(n + 1) + (n + 1) / 2048 + 64));
    int64_t *rowlen = c->d_scan_tmp.get();
    int64_t *tmp = rowlen + (n + 1);
    k_export_count<<<grid_for(n + 1, 256), 256, 0, st>>>(n, c->d_perm.get(), c->d_nbr_cnt.get(),
                                                         rowlen);
    HYD_CUDA(launch_check());
    HYD_CUDA(exclusive_scan_i64(rowlen, out->off, n + 1, tmp, st));
    int64_t total = 0;
    HYD_CUDA(cudaMemcpyAsync(&total, out->off + n, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    HYD_CUDA(cudaStreamSynchronize(st));
    out->needed = total;
    if (total > out->capacity || !out->idx) return cudaSuccess;
    k_export_fill<<<grid_for(n, EXPORT_WARPS), EXPORT_WARPS * 32, 0, st>>>(
        n, c->d_perm.get(), c->d_nbr_off.get(), c->d_nbr_cnt.get(), c->d_nbr_idx.get(), out->off,
        out->idx);
    return launch_check();
}

}  // namespace hyd
