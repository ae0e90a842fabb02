// The learned starting pressure of the exact Riemann solver: a 12 -> 64 ->
// 64 -> 1 network on physics-based features of the face problem.
//
//   k_mlp_pack      float parameters -> packed bf16 tiles for the kernels.
//   k_mlp_predict   standalone inference on the 5th-generation tensor cores
//                   (the tile routine of mlp.cuh that the flux kernel also
//                   runs in front of its Riemann solves).
//   k_mlp_grad      training forward + backward of a minibatch (FP32 CUDA
//                   cores, optional BF16 rounding of the operands so that
//                   training sees the inference numerics).
//   k_mlp_adam      Adam update of the FP32 master parameters.
//   k_mlp_feat      features and targets of recorded face problems.
#include <algorithm>

#include "mlp.cuh"

namespace hyd {

namespace {

// training: samples per tile, threads per CTA, entries of a CTA's partial sums
// (the parameters' gradients, then the loss), CTAs at most (two per SM)
constexpr int GRAD_TILE = 16;
constexpr int GRAD_THREADS = 512;
constexpr int GRAD_NS = GRAD_TILE * MLP_NH / GRAD_THREADS;   // samples per thread and output
constexpr int GRAD_NG = GRAD_THREADS / MLP_NH;               // groups of threads with an output each
constexpr int GRAD_ROW = MLP_NTRAIN + 1;
constexpr int GRAD_CTAS = 304;

__device__ __forceinline__ MlpTile &tile_of(unsigned char *raw) {
    return *reinterpret_cast<MlpTile *>((reinterpret_cast<uintptr_t>(raw) + 1023) &
                                        ~(uintptr_t)1023);
}

// float parameters -> the packed blob (bf16 K-major tiles + float vectors)
__global__ void k_mlp_pack(const float *__restrict__ theta, unsigned char *__restrict__ blob) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < MLP_NH * 16) {
        const int o = e >> 4, k = e & 15;
        const float v = k < MLP_NF ? theta[MLP_OFF_W1 + o * MLP_NF + k] : 0.f;
        *reinterpret_cast<__nv_bfloat16 *>(blob + MLP_W1_OFF + kmajor_off(o, k, 2)) =
            __float2bfloat16_rn(v);
        return;
    }
    const int e2 = e - MLP_NH * 16;
    if (e2 < MLP_NH * MLP_NH) {
        const int o = e2 >> 6, k = e2 & 63;
        *reinterpret_cast<__nv_bfloat16 *>(blob + MLP_W2_OFF + kmajor_off(o, k, 8)) =
            __float2bfloat16_rn(theta[MLP_OFF_W2 + e2]);
        return;
    }
    const int e3 = e2 - MLP_NH * MLP_NH;
    if (e3 < (int)(MLP_BLOB - MLP_F_OFF) / 4) {
        float v = 0.f;
        if (e3 < 64) v = theta[MLP_OFF_B1 + e3];
        else if (e3 < 128) v = theta[MLP_OFF_B2 + e3 - 64];
        else if (e3 < 192) v = theta[MLP_OFF_W3 + e3 - 128];
        else if (e3 < 204) v = theta[MLP_OFF_MEAN + e3 - 192];
        else if (e3 < 216) v = theta[MLP_OFF_SCALE + e3 - 204];
        else if (e3 == 216) v = theta[MLP_OFF_B3];
        else if (e3 == 217) v = theta[MLP_OFF_TMEAN];
        else if (e3 == 218) v = theta[MLP_OFF_TSCALE];
        else if (e3 < 231) v = theta[MLP_OFF_XMIN + e3 - 219];
        else if (e3 < 243) v = theta[MLP_OFF_XMAX + e3 - 231];
        reinterpret_cast<float *>(blob + MLP_F_OFF)[e3] = v;
    }
}

// Inference: faces (float rows rho_L, u_L, p_L, rho_R, u_R, p_R, row stride
// n) -> out[i] = p_TS exp(y), or -1 when the face is out of range (see
// mlp_guess); the caller then keeps its plain guess.
__global__ void __launch_bounds__(128) k_mlp_predict(int64_t n, const float *__restrict__ faces,
                                                     const unsigned char *__restrict__ blob,
                                                     GasK<float> K, float *__restrict__ out,
                                                     DevCounters *cnt, int stall) {
    extern __shared__ unsigned char smem_raw[];
    MlpTile &t = tile_of(smem_raw);
    const int tid = threadIdx.x;
    bool ok = mlp_tile_setup(t, blob, stall != 0);
    uint32_t phase = 0;
    const int64_t ntile = (n + 127) / 128;
    for (int64_t tile = blockIdx.x; ok && tile < ntile; tile += gridDim.x) {
        const int64_t i = tile * 128 + tid;
        float x[MLP_NF], pa = 1.f, lts = 0.f;
        bool in = false;
        if (i < n) {
            mlp_features(K, faces[i], faces[n + i], faces[2 * n + i], faces[3 * n + i],
                         faces[4 * n + i], faces[5 * n + i], x, pa);
            lts = x[9];
            in = mlp_standardise(t, x);
        } else {
#pragma unroll
            for (int k = 0; k < MLP_NF; k++) x[k] = 0.f;
        }
        mlp_put_row(t, tid, x);
        const float y = mlp_tile_eval(t, phase, &ok);
        if (ok && i < n) out[i] = mlp_guess(in, pa, lts, y);
    }
    if (!ok && tid == 0) atomicOr(&cnt->flags, ST_MLP);
    mlp_tile_teardown(t);
}

__device__ __forceinline__ float bfr(float v, bool q) {
    return q ? __bfloat162float(__float2bfloat16_rn(v)) : v;
}

// counter-based sample index (splitmix64 of seed, step, slot)
__device__ __forceinline__ int64_t sample_index(uint64_t seed, uint64_t step, uint64_t slot, int64_t n) {
    uint64_t z = seed + 0x9E3779B97F4A7C15ull * (step * 0x100000001B3ull + slot + 1);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (int64_t)(z % (uint64_t)n);
}

// Gradient of 0.5 mean (y - t)^2 over the nb samples of the minibatch: each
// CTA takes tiles of 16 samples and keeps the sums of its tiles in registers.
// In training it writes them (and its share of the loss) to its row of `part`,
// which k_mlp_adam folds -- no atomics, so training is reproducible.  For a
// caller's gradient (grad not NULL) it adds them to the caller's zeroed arrays:
// no scratch of the context, so calls on several streams do not meet.
// A tile's layers are small matrix products with a few outputs per thread: bound by shared-memory reads and latency.  With a batch of 2048 it
// runs on 128 CTAs; one thread per sample on 32 CTAs, the output layer's
// gradient by shared atomics of all threads on one address, took 200 us a step;
// this takes 10 us and the fold with Adam 6 us (64 steps and the inference of
// 262,144 faces: 12.9 -> 1.19 ms; with 256 threads 1.45 ms).
struct GradSmem {
    float W1[MLP_NH * 13], W2[MLP_NH * 65];
    float b1[MLP_NH], b2[MLP_NH], w3[MLP_NH];
    float mean[MLP_NF], scale[MLP_NF];
    float xs[GRAD_TILE][16], target[GRAD_TILE];
    int bad[GRAD_TILE];
    float h1[GRAD_TILE][68], a2[GRAD_TILE][68];   // a2: layer 2 before the ReLU, then da2
    float dy[GRAD_TILE];
    float z[GRAD_TILE][2];
};

__global__ void __launch_bounds__(GRAD_THREADS) k_mlp_grad(const float *__restrict__ theta,
                                                           const float *__restrict__ x,
                                                           const float *__restrict__ t, int64_t n,
                                                           int64_t nb, int random, uint64_t seed,
                                                           uint64_t step, int quant,
                                                           float *__restrict__ part,
                                                           float *__restrict__ grad,
                                                           float *__restrict__ loss) {
    __shared__ __align__(16) GradSmem S;
    const int tid = threadIdx.x;
    const bool q = quant != 0;
    const float b3 = theta[MLP_OFF_B3], tmean = theta[MLP_OFF_TMEAN], tscale = theta[MLP_OFF_TSCALE];
    const float inv = 1.f / (float)nb;
    const int o64 = tid & 63, s0 = (tid >> 6) * GRAD_NS;   // one output, GRAD_NS samples
    const int bo = (tid >> 4) * 2, bk = (tid & 15) * 4;    // a 2 x 4 block of dW2
    float gW2[2][4], gW1[2] = {0.f, 0.f}, gb1 = 0.f, gb2 = 0.f, gw3 = 0.f, gb3 = 0.f, lsum = 0.f;
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) gW2[i][j] = 0.f;
    const int64_t ntile = (nb + GRAD_TILE - 1) / GRAD_TILE;
    bool first = true;
    for (int64_t tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        __syncthreads();
        // the tile's samples, one feature (or the target) per thread; samples
        // with a non-finite feature or target -- an unphysical face -- are skipped
        const int fs = tid / (MLP_NF + 1), fk = tid % (MLP_NF + 1);
        float v = 0.f;
        bool there = false;
        if (fs < GRAD_TILE) {
            const int64_t slot = tile * GRAD_TILE + fs;
            there = slot < nb;
            if (there) {
                const int64_t idx = random ? sample_index(seed, step, slot, n) : slot;
                v = fk < MLP_NF ? x[idx * MLP_NF + fk] : t[idx];
            }
        }
        if (first) {   // (the samples are in flight)
            for (int e = tid; e < MLP_NH * MLP_NF; e += GRAD_THREADS)
                S.W1[(e / MLP_NF) * 13 + e % MLP_NF] = bfr(theta[MLP_OFF_W1 + e], q);
            for (int e = tid; e < MLP_NH * MLP_NH; e += GRAD_THREADS)
                S.W2[(e >> 6) * 65 + (e & 63)] = bfr(theta[MLP_OFF_W2 + e], q);
            if (tid < MLP_NH) {
                S.b1[tid] = theta[MLP_OFF_B1 + tid];
                S.b2[tid] = theta[MLP_OFF_B2 + tid];
                S.w3[tid] = theta[MLP_OFF_W3 + tid];
            } else if (tid < MLP_NH + MLP_NF) {
                S.mean[tid - MLP_NH] = theta[MLP_OFF_MEAN + tid - MLP_NH];
                S.scale[tid - MLP_NH] = theta[MLP_OFF_SCALE + tid - MLP_NH];
            }
            first = false;
        }
        if (tid < GRAD_TILE) S.bad[tid] = 0;
        __syncthreads();
        if (fs < GRAD_TILE) {
            if (!there || !isfinite(v)) atomicOr(&S.bad[fs], 1);
            if (fk < MLP_NF) S.xs[fs][fk] = there ? bfr((v - S.mean[fk]) / S.scale[fk], q) : 0.f;
            else S.target[fs] = v;
        }
        __syncthreads();
        const bool active = tid < GRAD_TILE && !S.bad[tid];
        const float target = active ? S.target[tid] : 0.f;
        if (fs < GRAD_TILE && fk < MLP_NF && S.bad[fs]) S.xs[fs][fk] = 0.f;
        __syncthreads();
        // layer 1
        {
            float a[GRAD_NS];
#pragma unroll
            for (int i = 0; i < GRAD_NS; i++) a[i] = S.b1[o64];
#pragma unroll
            for (int k = 0; k < MLP_NF; k++) {
                const float w = S.W1[o64 * 13 + k];
#pragma unroll
                for (int i = 0; i < GRAD_NS; i++) a[i] += w * S.xs[s0 + i][k];
            }
#pragma unroll
            for (int i = 0; i < GRAD_NS; i++) S.h1[s0 + i][o64] = bfr(fmaxf(a[i], 0.f), q);
        }
        __syncthreads();
        // layer 2 and the output
        {
            float a[GRAD_NS];
#pragma unroll
            for (int i = 0; i < GRAD_NS; i++) a[i] = S.b2[o64];
#pragma unroll 4
            for (int k = 0; k < MLP_NH; k += 4) {
                float4 h[GRAD_NS];
#pragma unroll
                for (int i = 0; i < GRAD_NS; i++) h[i] = *reinterpret_cast<const float4 *>(&S.h1[s0 + i][k]);
                const float *w = &S.W2[o64 * 65 + k];
#pragma unroll
                for (int i = 0; i < GRAD_NS; i++) a[i] += w[0] * h[i].x;
#pragma unroll
                for (int i = 0; i < GRAD_NS; i++) a[i] += w[1] * h[i].y;
#pragma unroll
                for (int i = 0; i < GRAD_NS; i++) a[i] += w[2] * h[i].z;
#pragma unroll
                for (int i = 0; i < GRAD_NS; i++) a[i] += w[3] * h[i].w;
            }
#pragma unroll
            for (int i = 0; i < GRAD_NS; i++) {
                S.a2[s0 + i][o64] = a[i];
                float z = fmaxf(a[i], 0.f) * S.w3[o64];
                for (int m = 16; m > 0; m >>= 1) z += __shfl_xor_sync(0xffffffffu, z, m);
                // (the two warps of four samples: slots 0 and 1)
                if ((tid & 31) == 0) S.z[s0 + i][(tid >> 5) & 1] = z;
            }
        }
        __syncthreads();
        if (tid < GRAD_TILE) {
            const float y = tmean + tscale * (b3 + (S.z[tid][0] + S.z[tid][1]));
            const float d = active ? (y - target) * inv * tscale : 0.f;   // d loss / d z
            S.dy[tid] = d;
            gb3 += d;
            if (active) lsum += 0.5f * (y - target) * (y - target) * inv;
        }
        __syncthreads();
        // da2 in place of a2
#pragma unroll
        for (int i = 0; i < GRAD_NS; i++) {
            const float a = S.a2[s0 + i][o64], d = S.dy[s0 + i];
            const float da = a > 0.f ? d * S.w3[o64] : 0.f;
            gw3 += fmaxf(a, 0.f) * d;
            gb2 += da;
            S.a2[s0 + i][o64] = da;
        }
        __syncthreads();
        // dW2[o][k] = sum_s da2[s][o] h1[s][k]
#pragma unroll 4
        for (int s = 0; s < GRAD_TILE; s++) {
            const float2 d = *reinterpret_cast<const float2 *>(&S.a2[s][bo]);
            const float4 h = *reinterpret_cast<const float4 *>(&S.h1[s][bk]);
            const float dd[2] = {d.x, d.y}, hh[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) gW2[i][j] += dd[i] * hh[j];
        }
        // da1 = (da2 W2) relu'(a1)
        float d1[GRAD_NS] = {};
#pragma unroll 4
        for (int o = 0; o < MLP_NH; o += 4) {
            float4 d[GRAD_NS];
#pragma unroll
            for (int i = 0; i < GRAD_NS; i++) d[i] = *reinterpret_cast<const float4 *>(&S.a2[s0 + i][o]);
            const float w0 = S.W2[o * 65 + o64], w1 = S.W2[(o + 1) * 65 + o64],
                        w2 = S.W2[(o + 2) * 65 + o64], w3 = S.W2[(o + 3) * 65 + o64];
#pragma unroll
            for (int i = 0; i < GRAD_NS; i++) {
                d1[i] += d[i].x * w0;
                d1[i] += d[i].y * w1;
                d1[i] += d[i].z * w2;
                d1[i] += d[i].w * w3;
            }
        }
#pragma unroll
        for (int i = 0; i < GRAD_NS; i++) {
            d1[i] = S.h1[s0 + i][o64] > 0.f ? d1[i] : 0.f;
            gb1 += d1[i];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < GRAD_NS; i++) S.h1[s0 + i][o64] = d1[i];   // (h1 is done with)
        __syncthreads();
        // dW1[o][k] = sum_s da1[s][o] xs[s][k]
#pragma unroll
        for (int i = 0; i < 2; i++) {
            const int e = tid + i * GRAD_THREADS, o = e / MLP_NF, k = e % MLP_NF;
            if (e >= MLP_NH * MLP_NF) break;
            float acc = 0.f;
#pragma unroll
            for (int s = 0; s < GRAD_TILE; s++) acc += S.h1[s][o] * S.xs[s][k];
            gW1[i] += acc;
        }
    }
    // the CTA's sums
    auto put = [&](int e, float v) {
        if (grad) atomicAdd(e < MLP_NTRAIN ? grad + e : loss, v);
        else part[(int64_t)blockIdx.x * GRAD_ROW + e] = v;
    };
#pragma unroll
    for (int i = 0; i < 2; i++)
        if (tid + i * GRAD_THREADS < MLP_NH * MLP_NF) put(MLP_OFF_W1 + tid + i * GRAD_THREADS, gW1[i]);
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) put(MLP_OFF_W2 + (bo + i) * MLP_NH + bk + j, gW2[i][j]);
    // the sums over the sample groups
    __syncthreads();
    float *fold = &S.W2[0];   // (the weights are done with) [3][GRAD_NG][64]
    fold[tid] = gb1;
    fold[GRAD_THREADS + tid] = gb2;
    fold[2 * GRAD_THREADS + tid] = gw3;
    __syncthreads();
    if (tid < 3 * MLP_NH) {
        const float *f = fold + (tid >> 6) * GRAD_THREADS + o64;
        float v = 0.f;
#pragma unroll
        for (int i = 0; i < GRAD_NG; i++) v += f[i * MLP_NH];
        put((tid < 64 ? MLP_OFF_B1 : tid < 128 ? MLP_OFF_B2 : MLP_OFF_W3) + o64, v);
    }
    if (tid < 32) {
        for (int m = 8; m > 0; m >>= 1) {
            gb3 += __shfl_xor_sync(0xffffffffu, gb3, m);
            lsum += __shfl_xor_sync(0xffffffffu, lsum, m);
        }
        if (tid == 0) {
            put(MLP_OFF_B3, gb3);
            put(MLP_NTRAIN, lsum);
        }
    }
}

// Sum of column e of the nrow rows of part, for 32 columns of a CTA: thread
// (column, slice) sums every eighth row, the slices are folded in shared
// memory.  Every thread of the 256 calls it; the sum is returned to the
// threads of slice 0.
__device__ __forceinline__ float fold_column(const float *__restrict__ part, int nrow, int e,
                                             float (*sh)[32]) {
    const int col = threadIdx.x & 31, sl = threadIdx.x >> 5;
    float v = 0.f;
    if (e < GRAD_ROW)
#pragma unroll 8
        for (int r = sl; r < nrow; r += 8) v += part[(int64_t)r * GRAD_ROW + e];
    sh[sl][col] = v;
    __syncthreads();
    return ((sh[0][col] + sh[1][col]) + (sh[2][col] + sh[3][col])) +
           ((sh[4][col] + sh[5][col]) + (sh[6][col] + sh[7][col]));
}

__global__ void __launch_bounds__(256) k_mlp_adam(float *__restrict__ theta,
                                                  const float *__restrict__ part, int nrow,
                                                  float *__restrict__ m, float *__restrict__ v,
                                                  float *__restrict__ loss, float lr, float b1,
                                                  float b2, float eps, int step) {
    __shared__ float sh[8][32];
    const int e = blockIdx.x * 32 + (threadIdx.x & 31);
    const float g = fold_column(part, nrow, e, sh);
    if (threadIdx.x >= 32 || e > MLP_NTRAIN) return;
    if (e == MLP_NTRAIN) {
        *loss = g;
        return;
    }
    float mm = b1 * m[e] + (1.f - b1) * g;
    float vv = b2 * v[e] + (1.f - b2) * g * g;
    m[e] = mm;
    v[e] = vv;
    float mh = mm / (1.f - powf(b1, (float)step));
    float vh = vv / (1.f - powf(b2, (float)step));
    theta[e] -= lr * mh / (sqrtf(vh) + eps);
}

// features x[n][12] and targets ln(p*/p_a) of recorded faces [7][n]
__global__ void k_mlp_feat(int64_t n, const float *__restrict__ faces, GasK<float> K,
                           float *__restrict__ x, float *__restrict__ t) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    float f[MLP_NF], pa;
    mlp_features(K, faces[i], faces[n + i], faces[2 * n + i], faces[3 * n + i], faces[4 * n + i],
                 faces[5 * n + i], f, pa);
    for (int k = 0; k < MLP_NF; k++) x[i * MLP_NF + k] = f[k];
    t[i] = logf(faces[6 * n + i] / pa) - f[9];   // ln(p* / p_TS)
}

// float <-> integer keys with the order of the floats (for atomicMin/Max)
__device__ __forceinline__ int ord_key(float f) {
    const int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float ord_val(int k) {
    return __int_as_float(k >= 0 ? k : k ^ 0x7fffffff);
}

// per-feature and target mean and standard deviation (double accumulators:
// acc[0..11] sums, [12..23] sums of squares, [24], [25] the target's, [26]
// the count) and the feature box (box[0..11] min keys, [12..23] max keys),
// over the samples whose features and target are all finite
__global__ void k_mlp_stats(int64_t n, const float *__restrict__ x, const float *__restrict__ t,
                            double *__restrict__ acc, int *__restrict__ box) {
    double s[MLP_NF + 1], s2[MLP_NF + 1];
    float lo[MLP_NF], hi[MLP_NF];
    for (int k = 0; k <= MLP_NF; k++) s[k] = s2[k] = 0.0;
    for (int k = 0; k < MLP_NF; k++) { lo[k] = 3.0e38f; hi[k] = -3.0e38f; }
    double cnt = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        bool ok = isfinite(t[i]);
        for (int k = 0; k < MLP_NF; k++) ok = ok && isfinite(x[i * MLP_NF + k]);
        if (!ok) continue;
        cnt += 1.0;
        for (int k = 0; k <= MLP_NF; k++) {
            const float f = k < MLP_NF ? x[i * MLP_NF + k] : t[i];
            const double v = f;
            s[k] += v;
            s2[k] += v * v;
            if (k < MLP_NF) { lo[k] = fminf(lo[k], f); hi[k] = fmaxf(hi[k], f); }
        }
    }
    atomicAdd(&acc[2 * MLP_NF + 2], cnt);
    for (int k = 0; k < MLP_NF; k++) {
        atomicAdd(&acc[k], s[k]);
        atomicAdd(&acc[MLP_NF + k], s2[k]);
        atomicMin(&box[k], ord_key(lo[k]));
        atomicMax(&box[MLP_NF + k], ord_key(hi[k]));
    }
    atomicAdd(&acc[2 * MLP_NF], s[MLP_NF]);
    atomicAdd(&acc[2 * MLP_NF + 1], s2[MLP_NF]);
}

__global__ void k_mlp_box_init(int *box) {
    const int k = threadIdx.x;
    if (k < MLP_NF) {
        box[k] = ord_key(3.0e38f);
        box[MLP_NF + k] = ord_key(-3.0e38f);
    }
}

__global__ void k_mlp_set_norm(int64_t n, const double *__restrict__ acc, const int *__restrict__ box,
                               float *__restrict__ theta) {
    int k = threadIdx.x;
    if (k > MLP_NF) return;
    const double cnt = acc[2 * MLP_NF + 2] > 0.0 ? acc[2 * MLP_NF + 2] : 1.0;
    const double sum = k < MLP_NF ? acc[k] : acc[2 * MLP_NF];
    const double sq = k < MLP_NF ? acc[MLP_NF + k] : acc[2 * MLP_NF + 1];
    const double mu = sum / cnt;
    const double var = sq / cnt - mu * mu;
    const double sd = sqrt(var > 0.0 ? var : 0.0);
    if (k < MLP_NF) {
        theta[MLP_OFF_MEAN + k] = (float)mu;
        theta[MLP_OFF_SCALE + k] = (float)(sd + 1e-3);
        theta[MLP_OFF_XMIN + k] = ord_val(box[k]);
        theta[MLP_OFF_XMAX + k] = ord_val(box[MLP_NF + k]);
    } else {
        theta[MLP_OFF_TMEAN] = (float)mu;
        theta[MLP_OFF_TSCALE] = (float)(sd + 1e-6);
    }
}

inline unsigned grid_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t mlp_pack(hydro_ctx *c, stream_t st) {
    HYD_CUDA(c->d_mlp_blob.ensure(MLP_BLOB));
    const int tot = MLP_NH * 16 + MLP_NH * MLP_NH + (int)(MLP_BLOB - MLP_F_OFF) / 4;
    k_mlp_pack<<<grid_for(tot, 256), 256, 0, st>>>(c->d_mlp.get(), c->d_mlp_blob.get());
    return launch_check();
}

cudaError_t mlp_predict(hydro_ctx *c, const float *faces, int64_t n, float *out, stream_t st) {
    const size_t smem = sizeof(MlpTile) + 1024;
    static bool configured = false;
    if (!configured) {
        HYD_CUDA(cudaFuncSetAttribute(k_mlp_predict, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem));
        configured = true;
    }
    const int64_t ntile = (n + 127) / 128;
    const unsigned grid = (unsigned)std::min<int64_t>(ntile > 0 ? ntile : 1, 152 * 4);
    k_mlp_predict<<<grid, 128, smem, st>>>(n, faces, c->d_mlp_blob.get(),
                                           GasK<float>(c->cfg.gamma), out, c->d_cnt,
                                           c->mlp_stall);
    return launch_check();
}

cudaError_t mlp_features(hydro_ctx *c, const float *faces, int64_t n, float *x, float *t,
                         stream_t st) {
    k_mlp_feat<<<grid_for(n, 256), 256, 0, st>>>(n, faces, GasK<float>(c->cfg.gamma), x, t);
    return launch_check();
}

// CTAs (training: rows of partial sums) for nb samples
static int grad_rows(int64_t nb) {
    return (int)std::min<int64_t>((nb + GRAD_TILE - 1) / GRAD_TILE, GRAD_CTAS);
}

cudaError_t mlp_gradient(hydro_ctx *c, const float *x, const float *t, int64_t n, int quant,
                         float *grad, float *loss, stream_t st) {
    k_mlp_grad<<<grad_rows(n), GRAD_THREADS, 0, st>>>(c->d_mlp.get(), x, t, n, n, 0, 0, 0, quant,
                                                      nullptr, grad, loss);
    return launch_check();
}

cudaError_t mlp_train_step(hydro_ctx *c, const float *x, const float *t, int64_t n, int64_t nb,
                           uint64_t seed, uint64_t step, float *m, float *v, float *loss, float lr,
                           int adam_step, stream_t st) {
    const int rows = grad_rows(nb);
    HYD_CUDA(c->d_mlp_grad.ensure((size_t)rows * GRAD_ROW));
    k_mlp_grad<<<rows, GRAD_THREADS, 0, st>>>(c->d_mlp.get(), x, t, n, nb, 1, seed, step, 1,
                                              c->d_mlp_grad.get(), nullptr, nullptr);
    HYD_CUDA(launch_check());
    k_mlp_adam<<<grid_for(GRAD_ROW, 32), 256, 0, st>>>(c->d_mlp.get(), c->d_mlp_grad.get(), rows, m,
                                                       v, loss, lr, 0.9f, 0.999f, 1e-8f, adam_step);
    return launch_check();
}

cudaError_t mlp_normalise(hydro_ctx *c, const float *x, const float *t, int64_t n, double *acc,
                          int *box, stream_t st) {
    HYD_CUDA(cudaMemsetAsync(acc, 0, sizeof(double) * (2 * MLP_NF + 3), st));
    k_mlp_box_init<<<1, 32, 0, st>>>(box);
    HYD_CUDA(launch_check());
    k_mlp_stats<<<256, 256, 0, st>>>(n, x, t, acc, box);
    HYD_CUDA(launch_check());
    k_mlp_set_norm<<<1, 32, 0, st>>>(n, acc, box, c->d_mlp.get());
    return launch_check();
}

}  // namespace hyd
static_assert(hyd::MLP_BLOB == hyd::MLP_BLOB_BYTES, "blob size");
