// Voxel-driven back-projector of 2D images (same operator as bp_direct_kernel, Sec. 2.1): every pixel projected onto
// the row of detector bins, the linear, zero-padded values summed over the views.
//
// One CTA owns a B x B brick of the image for up to NB images of a batch (which share positions and weights)
// and splits the views among G = 256 / B^2 groups of threads, whose sums are added at the end: a 128^2 image has
// 64 bricks of 16^2, too few for the chip, but 256 of 8^2. Positions are relative to the projection of the brick
// centre, as in the 3D bricks: u = u0 + (Qa . d) / w, w = w0 + Pw . d for a pixel at offset d, with u0, w0, Qa and Pw
// formed in FP64, here by all 256 threads, one view each (a few lanes of one warp while the others wait took most
// of the time of the 3D kernel on a 2D image).
//
// Bound by latency: the FP64 set-ups, then the detector reads (L1 / L2), of which four or eight views are in flight at a
// time. On GB300, against the 3D bricks of depth one: 128^2 image, 180 views of 183 bins, 123 -> 17 us (23 with a branch
// around a view's reads, which kept them one after the other; 512^2 image, 720 views of 1024 bins: 388 -> 256 us).
#include <algorithm>

#include "device_common.cuh"

namespace pyronn {

constexpr int B2_NT = 256;

struct B2View {
    float qa0, qa1, fu, pw0;   // two 16-byte words
    float pw1, w0;
    int U0, valid;             // valid = 0: the brick centre is at or behind the source line
};

static __device__ __forceinline__ void bp2d_view_setup(const OpParams &p, int view, double X, double Y, B2View &o) {
    const double *x = p.views64 + (size_t)view * VIEW64_STRIDE;
    double Pa0, Pa1, Pw0 = 0.0, Pw1 = 0.0, a0, w0 = 1.0;
    if (p.perspective) {
        Pa0 = x[0], Pa1 = x[1], Pw0 = x[8], Pw1 = x[9];
        a0 = Pa0 * X + Pa1 * Y + x[3];
        w0 = Pw0 * X + Pw1 * Y + x[11];
    } else {
        Pa0 = x[3] / p.du, Pa1 = x[4] / p.du;
        a0 = ((X - x[0]) * x[3] + (Y - x[1]) * x[4] - p.ou) / p.du + 0.5 * (p.det.nu - 1);
    }
    o.valid = w0 > 0.0;
    if (!o.valid) w0 = 1.0;
    const double u0 = a0 / w0, U = floor(u0);
    o.qa0 = (float)((Pa0 - u0 * Pw0) * p.sx);
    o.qa1 = (float)((Pa1 - u0 * Pw1) * p.sy);
    o.pw0 = (float)(Pw0 * p.sx);
    o.pw1 = (float)(Pw1 * p.sy);
    o.w0 = (float)w0;
    o.fu = (float)(u0 - U);
    o.U0 = (int)fmin(fmax(U, -4.0e6), 4.0e6);   // far off the detector: contributes nothing anyway
}

template <typename T, int B, int NB, bool W2>
__global__ void __launch_bounds__(B2_NT) bp2d_kernel(OpParams p, const T *__restrict__ sino, T *__restrict__ vol) {
    constexpr int PIX = B * B, G = B2_NT / PIX;
    // views whose loads are in flight together (eight for one image: 17 -> 20 us, for eight of 362^2: 303 -> 254 us)
    constexpr int AHEAD = NB == 4 ? 8 : 4;
    __shared__ __align__(16) B2View sv[B2_NT];
    __shared__ float s_sum[G > 1 ? NB * B2_NT : 1];
    const int tid = threadIdx.x, pix = tid % PIX, group = tid / PIX;
    const int bx0 = blockIdx.x * B, by0 = blockIdx.y * B;
    const int b0 = blockIdx.z * NB, nb = min(NB, p.batch - b0);
    const int lx = pix % B, ly = pix / B;
    const float dx = (float)lx - 0.5f * (B - 1), dy = (float)ly - 0.5f * (B - 1);
    const double X = (bx0 + 0.5 * (B - 1) - 0.5 * (p.vol.nx - 1)) * p.sx;
    const double Y = (by0 + 0.5 * (B - 1) - 0.5 * (p.vol.ny - 1)) * p.sy;
    const T *sb = sino + (long long)b0 * p.sino_elems;
    const int nu = p.det.nu;
    float acc[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) acc[i] = 0.0f;
    for (int n0 = 0; n0 < p.n_views; n0 += B2_NT) {
        const int nc = min(B2_NT, p.n_views - n0);
        __syncthreads();
        if (tid < nc) bp2d_view_setup(p, n0 + tid, X, Y, sv[tid]);
        __syncthreads();
#pragma unroll AHEAD
        for (int c = group; c < nc; c += G) {
            const B2View &V = sv[c];
            const float w = fmaf(V.pw0, dx, fmaf(V.pw1, dy, V.w0));
            const bool ahead = V.valid && w > 0.0f;   // no branch: the loads of consecutive views go out together
            const float iw = p.perspective && ahead ? rcp_fast(w) : 1.0f;
            float q = fmaf(fmaf(V.qa0, dx, V.qa1 * dy), iw, V.fu);
            q = fminf(fmaxf(q, -1.0e6f), 1.0e6f);   // the magic addition needs |q| < 2^22
            const float t = __fadd_rd(q, 12582912.0f);
            const float a = q - (t - 12582912.0f);
            const int u = __float_as_int(t) - 0x4B400000 + V.U0;
            const bool in0 = ahead && (unsigned)u < (unsigned)nu, in1 = ahead && (unsigned)(u + 1) < (unsigned)nu;
            const T *r = sb + (long long)(n0 + c) * nu + u;
            const float om = W2 ? iw * iw : 1.0f;
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const float q0 = in0 && i < nb ? ldg_f32(r + i * p.sino_elems) : 0.0f;
                const float q1 = in1 && i < nb ? ldg_f32(r + i * p.sino_elems + 1) : 0.0f;
                acc[i] = fmaf(om, fmaf(a, q1 - q0, q0), acc[i]);
            }
        }
    }
    if (G > 1) {
#pragma unroll
        for (int i = 0; i < NB; ++i) s_sum[i * B2_NT + tid] = acc[i];
        __syncthreads();
        if (group) return;
#pragma unroll
        for (int i = 0; i < NB; ++i)
#pragma unroll
            for (int g = 1; g < G; ++g) acc[i] += s_sum[i * B2_NT + g * PIX + pix];
    }
    const int gx = bx0 + lx, gy = by0 + ly;
    if (gx < p.vol.nx && gy < p.vol.ny) {
        T *o = vol + (long long)b0 * p.vol_elems + (long long)gy * p.vol.nx + gx;
#pragma unroll
        for (int i = 0; i < NB; ++i)
            if (i < nb) o[i * p.vol_elems] = from_f32<T>(acc[i]);
    }
}

template <typename T, int B, int NB>
static int launch_bp2d_t(const OpParams &p, const void *sino, void *vol, cudaStream_t st) {
    const bool w2 = p.perspective && p.weight == PYRONN_BP_INV_W2;
    const int per_launch = 65535 * NB;
    for (int b0 = 0; b0 < p.batch; b0 += per_launch) {
        OpParams q = p;
        q.batch = std::min(p.batch - b0, per_launch);
        const dim3 grid(ceil_div(p.vol.nx, B), ceil_div(p.vol.ny, B), ceil_div(q.batch, NB));
        const T *s = (const T *)sino + b0 * p.sino_elems;
        T *v = (T *)vol + b0 * p.vol_elems;
        if (w2) bp2d_kernel<T, B, NB, true><<<grid, B2_NT, 0, st>>>(q, s, v);
        else bp2d_kernel<T, B, NB, false><<<grid, B2_NT, 0, st>>>(q, s, v);
    }
    return (int)cudaGetLastError();
}

template <typename T, int B>
static int launch_bp2d_nb(const OpParams &p, const void *sino, void *vol, cudaStream_t st) {
    if (p.batch >= 3) return launch_bp2d_t<T, B, 4>(p, sino, vol, st);
    if (p.batch == 2) return launch_bp2d_t<T, B, 2>(p, sino, vol, st);
    return launch_bp2d_t<T, B, 1>(p, sino, vol, st);
}

// 8^2 bricks with four groups of views up to 384^2 pixels, where 16^2 bricks give at most four CTAs per SM; above, 16^2
// bricks (a quarter of the FP64 set-ups). The choice depends on the image alone, not on the batch.
template <typename T>
static int launch_bp2d_b(const OpParams &p, const void *sino, void *vol, cudaStream_t st) {
    return p.vol_elems <= 384 * 384 ? launch_bp2d_nb<T, 8>(p, sino, vol, st) : launch_bp2d_nb<T, 16>(p, sino, vol, st);
}

int launch_bp2d(const OpParams &p, const void *sino, void *vol, int dtype, void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    switch (dtype) {
        case PYRONN_F32: return launch_bp2d_b<float>(p, sino, vol, st);
        case PYRONN_BF16: return launch_bp2d_b<__nv_bfloat16>(p, sino, vol, st);
        case PYRONN_F16: return launch_bp2d_b<__half>(p, sino, vol, st);
        default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace pyronn
