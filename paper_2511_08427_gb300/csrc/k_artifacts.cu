// Acquisition-artifact simulation on sinograms (Sec. 2.4: detector jitter, Gaussian noise, ring
// artifacts, gantry motion blur). Every random quantity is an input (shifts, noise samples, chosen
// columns), so these are deterministic transforms; sinograms are [batch][V][Nv][Nu], u fastest.
#include <algorithm>

#include "device_common.cuh"

namespace pyronn {

static int ew_blocks(long long n) { return stride_grid(n, 32); }

// out[v][u] = in[v][u - s] (axis 0, one shift per row) or in[v - s][u] (axis 1, one shift per column).
template <typename T>
__global__ void jitter_kernel(const T *__restrict__ in, T *__restrict__ out, const int *__restrict__ shifts, int axis,
                              int nu, int nv, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int u = (int)(i % nu);
        const long long row = i / nu;             // (item, view, v)
        const int v = (int)(row % nv);
        const long long img = row / nv;           // (item, view)
        float val = 0.0f;
        if (axis == 0) {
            const int src = u - shifts[row];
            if (src >= 0 && src < nu) val = to_f32<T>(in[row * nu + src]);
        } else {
            const int src = v - shifts[img * nu + u];
            if (src >= 0 && src < nv) val = to_f32<T>(in[(img * nv + src) * nu + u]);
        }
        out[i] = from_f32<T>(val);
    }
}

template <typename T>
__global__ void noise_kernel(const T *__restrict__ in, T *__restrict__ out, const float *__restrict__ noise, float mean,
                             float sd, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = from_f32<T>(to_f32<T>(in[i]) + fmaf(sd, noise[i], mean));
}

// element (item, view in [v0, v1), v, column index c): out = in * gains[c] at u = columns[c]
template <typename T>
__global__ void ring_kernel(const T *__restrict__ in, T *__restrict__ out, const int *__restrict__ cols,
                            const float *__restrict__ gains, int ncol, int nu, int nv, int n_views, int v0, int v1,
                            long long n) {
    const int nsel = v1 - v0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % ncol);
        long long r = i / ncol;
        const int v = (int)(r % nv);
        r /= nv;
        const int view = v0 + (int)(r % nsel);
        const long long item = r / nsel;
        const int u = cols[c];
        if (u < 0 || u >= nu) continue;
        const long long o = ((item * n_views + view) * nv + v) * nu + u;
        out[o] = from_f32<T>(to_f32<T>(in[o]) * gains[c]);
    }
}

// out(u, v) of view n = (1 / L) sum_j bilinear(in, u + t_j cos a_n, v + t_j sin a_n), t_j = j - (L - 1) / 2
//
// One CTA owns a tile of 32 x 32 pixels of one projection (four rows per thread) and stages it with the
// H = ceil((L - 1) / 2) pixels around it that the line can reach as FP32 in shared memory, zero outside the detector, so
// that no tap needs a test and the x part of a sample serves four rows. Bound by issue slots (about 22 per sample; the
// DRAM traffic of 360 f16 projections of 192 x 384 is 106 MB, 16 us). On GB300, those 360 projections, against one thread
// per pixel reading global memory (blur_far_kernel): 7 samples 596 -> 231 us, 31 samples of FP32 2076 -> 635 us, 77 samples
// 4831 -> 1543 us.
constexpr int BLUR_NT = 256, BLUR_TILE = 32, BLUR_ROWS = 4, BLUR_BOX = 12288;

template <typename T>
__global__ void __launch_bounds__(BLUR_NT) blur_kernel(const T *__restrict__ in, T *__restrict__ out,
                                                       const float *__restrict__ angles, int length, int tiles_u, int tiles_v,
                                                       int nu, int nv, int n_views, long long tiles) {
    extern __shared__ float box[];   // side x side: the tile, H pixels before it, H + 1 after it
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, h = length >> 1, side = BLUR_TILE + 2 * h + 1;
    const float half = 0.5f * (float)(length - 1), M = 12582912.0f;
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long long img = tile / (tiles_u * tiles_v);
        const int in_img = (int)(tile - img * (tiles_u * tiles_v));
        const int u0 = in_img % tiles_u * BLUR_TILE, v0 = in_img / tiles_u * BLUR_TILE;
        const T *src = in + img * (long long)nv * nu;
        __syncthreads();   // the previous tile's readers are done
        for (int x = lane; x < side; x += 32)
#pragma unroll 5
            for (int y = warp; y < side; y += BLUR_NT / 32) {
                const int gx = u0 - h + x, gy = v0 - h + y;
                box[y * side + x] = (unsigned)gx < (unsigned)nu && (unsigned)gy < (unsigned)nv
                                        ? ldg_f32(src + (long long)gy * nu + gx) : 0.0f;
            }
        __syncthreads();
        const int u = u0 + lane, v = v0 + BLUR_ROWS * warp;
        if (v >= nv) continue;
        float ca, sa;
        sincosf(angles[img % n_views], &sa, &ca);
        const bool bad = !(fabsf(ca) <= 1.0f && fabsf(sa) <= 1.0f);   // an angle that is not finite: no position in the box
        if (bad) ca = sa = 0.0f;
        float acc[BLUR_ROWS] = {0.0f, 0.0f, 0.0f, 0.0f};
        // floor(x) = bits(x + 1.5 2^23 rounded down) - 0x4B400000 for |x| < 2^22 (floorf and its conversion to an integer
        // run at a quarter of the rate); the constant and the box's origin are folded into the address (mod 2^32)
        const unsigned row = 4u * (unsigned)side;
        const unsigned base = (unsigned)__cvta_generic_to_shared(box) - (0x4B400000u + (unsigned)(u0 - h)) * 4u -
                              (0x4B400000u + (unsigned)(v0 - h)) * row;
        for (int j = 0; j < length; ++j) {
            const float t = (float)j - half;
            const float x = fmaf(t, ca, (float)u), tx = __fadd_rd(x, M), ax = x - (tx - M);
            const unsigned col = base + 4u * __float_as_uint(tx);
            const f32x2 wx = pack2(1.0f - ax, ax);
#pragma unroll
            for (int r = 0; r < BLUR_ROWS; ++r) {
                const float y = fmaf(t, sa, (float)(v + r)), ty = __fadd_rd(y, M), ay = y - (ty - M);
                const unsigned q = col + row * __float_as_uint(ty);
                const f32x2 w0 = mul2(wx, splat2(1.0f - ay)), w1 = mul2(wx, splat2(ay));
                float s = lo2(w0) * lds_f32<float>(q);
                s = fmaf(hi2(w0), lds_f32<float>(q + 4u), s);
                s = fmaf(lo2(w1), lds_f32<float>(q + row), s);
                acc[r] += fmaf(hi2(w1), lds_f32<float>(q + row + 4u), s);
            }
        }
#pragma unroll
        for (int r = 0; r < BLUR_ROWS; ++r)
            if (u < nu && v + r < nv)
                out[(img * nv + v + r) * nu + u] = from_f32<T>(bad ? __int_as_float(0x7fffffff) : acc[r] / (float)length);
    }
}

template <typename T>
__global__ void blur_far_kernel(const T *__restrict__ in, T *__restrict__ out, const float *__restrict__ angles, int length,
                                int nu, int nv, int n_views, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int u = (int)(i % nu);
        const long long row = i / nu;
        const int v = (int)(row % nv);
        const long long img = row / nv;
        const int view = (int)(img % n_views);
        const T *src = in + img * (long long)nv * nu;
        float ca, sa;
        sincosf(angles[view], &sa, &ca);
        float acc = 0.0f;
        for (int j = 0; j < length; ++j) {
            const float t = (float)j - 0.5f * (float)(length - 1);
            const float x = fmaf(t, ca, (float)u), y = fmaf(t, sa, (float)v);
            const float fx = floorf(x), fy = floorf(y);
            const int x0 = (int)fx, y0 = (int)fy;
            const float ax = x - fx, ay = y - fy;
            float s = 0.0f;
            if (y0 >= 0 && y0 < nv) {
                if (x0 >= 0 && x0 < nu) s += (1.0f - ax) * (1.0f - ay) * to_f32<T>(src[(long long)y0 * nu + x0]);
                if (x0 + 1 >= 0 && x0 + 1 < nu) s += ax * (1.0f - ay) * to_f32<T>(src[(long long)y0 * nu + x0 + 1]);
            }
            if (y0 + 1 >= 0 && y0 + 1 < nv) {
                if (x0 >= 0 && x0 < nu) s += (1.0f - ax) * ay * to_f32<T>(src[(long long)(y0 + 1) * nu + x0]);
                if (x0 + 1 >= 0 && x0 + 1 < nu) s += ax * ay * to_f32<T>(src[(long long)(y0 + 1) * nu + x0 + 1]);
            }
            acc += s;
        }
        out[i] = from_f32<T>(acc / (float)length);
    }
}

#define PYRONN_DISPATCH(dtype, CALL)                                   \
    switch (dtype) {                                                   \
        case PYRONN_F32: { using T = float; CALL; break; }             \
        case PYRONN_BF16: { using T = __nv_bfloat16; CALL; break; }    \
        case PYRONN_F16: { using T = __half; CALL; break; }            \
        default: return (int)cudaErrorInvalidValue;                    \
    }

int launch_sim_jitter(const void *in, void *out, const int *shifts, int axis, int nu, int nv, long long n, int dtype,
                      void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    PYRONN_DISPATCH(dtype, (jitter_kernel<T><<<ew_blocks(n), 256, 0, st>>>((const T *)in, (T *)out, shifts, axis, nu,
                                                                            nv, n)));
    return (int)cudaGetLastError();
}

int launch_sim_noise(const void *in, void *out, const float *noise, float mean, float sd, long long n, int dtype,
                     void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    PYRONN_DISPATCH(dtype, (noise_kernel<T><<<ew_blocks(n), 256, 0, st>>>((const T *)in, (T *)out, noise, mean, sd, n)));
    return (int)cudaGetLastError();
}

int launch_sim_ring(const void *in, void *out, const int *cols, const float *gains, int ncol, int nu, int nv, int n_views,
                    int v0, int v1, int batch, int dtype, void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const long long n = (long long)batch * (v1 - v0) * nv * ncol;
    if (n <= 0) return 0;
    PYRONN_DISPATCH(dtype, (ring_kernel<T><<<ew_blocks(n), 256, 0, st>>>((const T *)in, (T *)out, cols, gains, ncol, nu,
                                                                          nv, n_views, v0, v1, n)));
    return (int)cudaGetLastError();
}

int launch_sim_blur(const void *in, void *out, const float *angles, int length, int nu, int nv, int n_views, long long n,
                    int dtype, void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    // Staged tiles, but for detectors of few rows or columns, whose tiles would be nearly empty (990 views of 42 x 10, 9 samples: 15 us
    // per pixel, 21 staged), few samples in all (3 views of 51 x 64,
    // 3 samples: 4 us per pixel, 6 staged; 9 samples: 6 both ways), lines whose box passes 48 KB, and
    // detectors so long that FP32 positions lose the pixel: these read global memory, one thread per pixel. 2000 views
    // of 16 rows of 384, per pixel and staged: 7 samples 263 and 138 us, 77 samples 1392 and 865; of one row of 513, 3000
    // views, 33 samples: 60 us and (in tiles of 256 x 4) 277.
    const int side = BLUR_TILE + 2 * (length >> 1) + 1;
    if (nv >= 16 && nu >= 16 && side * side <= BLUR_BOX && std::max(nu, nv) < 1 << 21 && n * length >= 1 << 16) {
        const size_t smem = sizeof(float) * (size_t)(side * side);
        const int tiles_u = ceil_div(nu, BLUR_TILE), tiles_v = ceil_div(nv, BLUR_TILE);
        const long long tiles = n / ((long long)nu * nv) * tiles_u * tiles_v;
        const int blocks = (int)std::min(tiles, (long long)1 << 30);
        PYRONN_DISPATCH(dtype, (blur_kernel<T><<<blocks, BLUR_NT, smem, st>>>((const T *)in, (T *)out, angles, length,
                                                                               tiles_u, tiles_v, nu, nv, n_views, tiles)));
        return (int)cudaGetLastError();
    }
    PYRONN_DISPATCH(dtype, (blur_far_kernel<T><<<ew_blocks(n), 256, 0, st>>>((const T *)in, (T *)out, angles, length, nu,
                                                                              nv, n_views, n)));
    return (int)cudaGetLastError();
}

#undef PYRONN_DISPATCH

}  // namespace pyronn
