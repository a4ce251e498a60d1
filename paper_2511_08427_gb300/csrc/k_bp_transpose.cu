// Exact transpose of the voxel-driven back-projector for 3D volumes (the gradient of the BP layers): every
// voxel spreads x omega with the bilinear weights of its projection over four detector pixels of every view.
//
// One CTA owns a brick of 16 x 16 x 32 voxels, kept in shared memory over a range of views. The brick's
// shadow on the detector (a box of (2 eu + 1) x (2 ev + 1) pixels around the projection of its centre) is summed in
// shared memory, int32 fixed point, and then added to the sinogram: about one global reduction per ten voxel
// updates instead of four per update. Coordinates are relative to the projection of the brick centre (FP64
// constants per brick and view, bp_common.cuh), as in the brick back-projectors.
//
// Lanes take the 32 voxels of a column along z: for rays that run mostly across z their projections lie on
// different detector rows, whose pitch is odd, hence on different banks (lanes along x would all fall on one
// pixel in the views along x, and a reduction takes one pass per lane that shares a word). Two boxes alternate, so
// one barrier per view separates its sums from their flush and the next view's from the box's last flush.
//
// Fixed point: contributions enter as round(c scale) by one FFMA with 1.5 2^23 (|c| scale <= 2^22), and the scale keeps
// sums below 2^30: |sum| <= max |x| max omega H with H the sum of the weights of the brick's voxels in one pixel. Over a
// row along x or y, the hats along u sum to at most 1 / s_u + 1 (s_u the voxels' distance along u in pixels); over a
// column along z, the hats along v, widened by what v changes over the row's support, to (1 + 2 spread) / s_v + 1;
// and there are 16 rows. Geometries whose bound passes 600 (voxels far smaller than a pixel) would coarsen
// the quantum (2^-22 of the largest contribution up to 256) and keep the direct kernel's FP32 sums. So do, voxel by voxel,
// bricks of a wide range: the quantum is that of the brick's largest value, so pixels that only small values reach would
// lose bits. A brick counts as wide where some 8 x 2 x 4 voxels of it (at least 40 of them nonzero) stay below
// 1 / WIDE_RANGE of its largest value.
//
// Bound by the shared reductions (four per update, two passes where two lanes share a pixel) and issue slots. 256^3
// voxels, 360 views, 400 x 600 detector, FP32: 42.7 -> 8.9 ms; its error against 64 bits falls from 1.7e-6 to 5.4e-7.
#include <algorithm>
#include <cmath>

#include "bp_common.cuh"

namespace pyronn {

constexpr int BPT_Z = 32, BPT_NT = 256, BPT_GROUP = 32;
// fewer updates (voxels x views) than this: the direct kernel, whose threads fill the chip (32^3 voxels, 8 views, 0.26e6
// updates: 20 us against 32; 24 x 32 x 32, 40 views, 0.98e6: 29 and 35; 30 x 33 x 31, 60 views, 1.8e6: 43 and 35)
constexpr long long BPT_MIN_UPDATES = 3LL << 19;
constexpr int BPT_BOX_MAX = 12 * 1024;   // words of one shadow box

struct BptView {
    BpView v;
    float scale, unscale;   // fixed-point steps per unit, and its reciprocal
    int mode;               // 0 nothing reaches the detector, 1 shadow box, 2 voxel by voxel into global memory
};

// Bound on the summed weights of a brick's voxels in one pixel: s, sz the steps along u (row) and v (z), spread the
// change of v over a row's support, which widens the hat along v
static __host__ __device__ inline float bpt_weight_bound(float s, float sz, float spread) {
    return 16.0f * fminf(16.0f, 1.1f / s + 1.0f) * fminf(32.0f, 1.1f * (1.0f + 2.0f * spread) / sz + 1.0f);
}

// Constants of one (brick, view). xmax: bits of max |x| over the brick.
template <bool W2>
static __device__ void bpt_view_setup(const OpParams &p, int view, const double Xb[3], unsigned xmax, int box_cap, BptView &o) {
    bp_view_setup(p, view, Xb, 0.5 * (BPT_Z - 1), o.v);
    const BpView &V = o.v;
    o.mode = 2;
    o.scale = o.unscale = 0.0f;
    if (!V.valid || V.eu < 0) return;
    // depth ratios over the brick and its margin; near the source plane FP32 positions are too coarse to rely on
    // the box
    const float h[3] = {0.5f * (BPB_X - 1) + 1.0f, 0.5f * (BPB_Y - 1) + 1.0f, 0.5f * (BPT_Z - 1) + 1.0f};
    const float sw = fabsf(V.Pw[0]) * h[0] + fabsf(V.Pw[1]) * h[1] + fabsf(V.Pw[2]) * h[2];
    const float wmin = V.w0 - sw, wmax = V.w0 + sw;
    if (!(wmin > 0.25f * V.w0)) return;
    if ((long long)(2 * V.eu + 1) * (2 * V.ev + 1) > box_cap) return;
    if (V.U0 + V.eu < 0 || V.U0 - V.eu >= p.det.nu || V.V0 + V.ev < 0 || V.V0 - V.ev >= p.det.nv) {
        o.mode = 0;
        return;
    }
    // detector steps per voxel: the row axis k (x or y, the wider along u) and z; the steps along u (row) and v (z)
    // from below, the two cross terms from above, with what the depth ratio changes over the shadow
    const float iw = 1.0f / wmax, jw = 1.0f / wmin;
    const int k = fabsf(V.Qa[0]) >= fabsf(V.Qa[1]) ? 0 : 1;
    const float eu = (float)V.eu, ev = (float)V.ev;
    const float s = fmaxf(fabsf(V.Qa[k]) * iw - fabsf(V.Pw[k]) * jw * eu, 1.0e-3f);
    const float cross_v = (fabsf(V.Qb[k]) + fabsf(V.Pw[k]) * ev) * jw / s;   // v over the row's support (|u| < 1)
    const float cross_u = (fabsf(V.Qa[2]) + fabsf(V.Pw[2]) * eu) * jw;
    const float sz = fmaxf(fabsf(V.Qb[2]) * iw - fabsf(V.Pw[2]) * jw * ev - cross_v * cross_u, 1.0e-3f);
    const float H = fmaxf(bpt_weight_bound(s, sz, cross_v), 256.0f);
    // omega at most jw^2 (a little above every rounded 1 / w^2); the scale need not be a power of two, so that the largest
    // possible sum or contribution uses the whole range
    const double bound = (double)__uint_as_float(xmax) * (W2 ? 1.0001 * jw * jw : 1.0001) * H;
    const double scale = 1073741824.0 / bound;
    if (xmax >= 0x7f800000u || !(scale > 1.0e-30) || !(scale < 1.0e30)) return;
    o.scale = (float)scale;
    o.unscale = (float)(1.0 / (double)o.scale);
    o.mode = 1;
}

template <typename T, bool W2>
__global__ void __launch_bounds__(BPT_NT, 4) bpt_brick_kernel(OpParams p, int views_per_cta, int box_cap,
                                                              const T *__restrict__ vol, float *__restrict__ acc) {
    extern __shared__ __align__(16) float bpt_smem[];
    float *const xs = bpt_smem;                                        // [16 y][16 x][32 z]
    unsigned *const boxes = (unsigned *)(bpt_smem + BPB_NT * BPT_Z);   // two shadow boxes, zero between views
    __shared__ BptView sv[BPT_GROUP];
    __shared__ unsigned s_max, s_low;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nbx = (p.vol.nx + BPB_X - 1) / BPB_X, nby = (p.vol.ny + BPB_Y - 1) / BPB_Y;
    const int bx0 = (blockIdx.x % nbx) * BPB_X, by0 = (blockIdx.x / nbx % nby) * BPB_Y, bz0 = (blockIdx.x / (nbx * nby)) * BPT_Z;
    const int v_begin = blockIdx.y * views_per_cta, v_end = min(v_begin + views_per_cta, p.n_views);
    const int b = blockIdx.z;
    const T *vb = vol + (long long)b * p.vol_elems;
    float *ab = acc + (long long)b * p.sino_elems;
    const int nu = p.det.nu, nv = p.det.nv;

    if (tid == 0) s_max = 0u, s_low = 0xffffffffu;
    __syncthreads();
    unsigned big = 0u, low = 0xffffffffu;   // low: the least maximum of 8 x 2 x 4 voxels
    {
        // x fastest in memory: 16 lanes read one row of the brick; stored with z fastest
        static_assert(BPT_NT == BPB_NT, "one thread per column");
        const int x = tid % BPB_X, y = tid / BPB_X, gx = bx0 + x, gy = by0 + y;
        for (int z0 = 0; z0 < BPT_Z; z0 += 4) {
            unsigned most = 0u, nonzero = 0u;
#pragma unroll
            for (int z = z0; z < z0 + 4; ++z) {
                const int gz = bz0 + z;
                const float v = gx < p.vol.nx && gy < p.vol.ny && gz < p.vol.nz
                                    ? ldg_f32(vb + ((long long)gz * p.vol.ny + gy) * p.vol.nx + gx) : 0.0f;
                xs[tid * BPT_Z + z] = v;
                most = max(most, __float_as_uint(fabsf(v)));
                nonzero += v != 0.0f;
            }
            big = max(big, most);
            for (int o = 1; o < 32; o = o == 4 ? 16 : 2 * o) {
                most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
                nonzero += __shfl_xor_sync(0xffffffffu, nonzero, o);
            }
            if (nonzero >= 40u) low = min(low, most);
        }
    }
    big = __reduce_max_sync(0xffffffffu, big);
    low = __reduce_min_sync(0xffffffffu, low);
    if (lane == 0) {
        atomicMax(&s_max, big);
        atomicMin(&s_low, low);
    }
    for (int e = tid; e < 2 * box_cap; e += BPT_NT) boxes[e] = 0u;
    __syncthreads();
    const unsigned xmax = s_max;
    if (xmax == 0u) return;   // an empty brick (the same for every thread)
    // One view voxel by voxel: absolute coordinates, each tap tested, straight to global memory. Lanes along x, whose taps
    // share sectors in most views, values from L1 (a noisy phantom of 256^3, 90 views, most of whose bricks go this
    // way: 5.7 ms with the lanes of a warp along z, 3.0 this way, 14.1 in the direct kernel).
    auto add_direct = [&](int view) {
        float *q = ab + (long long)view * nv * nu;
        const float *P = p.bp[view].P;
        const int gx = bx0 + tid % BPB_X, gy = by0 + tid / BPB_X;
        const float x = (float)gx - p.vol.hx, y = (float)gy - p.vol.hy;
        const long long plane = (long long)p.vol.ny * p.vol.nx;
        const T *col = vb + bz0 * plane + (long long)gy * p.vol.nx + gx;   // the staged values' z order would meet on one bank
        const int planes = gx < p.vol.nx && gy < p.vol.ny ? min(BPT_Z, p.vol.nz - bz0) : 0;
#pragma unroll 4
        for (int k = 0; k < planes; ++k) {
            const float xv = ldg_f32(col + k * plane);
            if (xv == 0.0f) continue;
            const float z = (float)(bz0 + k) - p.vol.hz;
            const float a = fmaf(P[0], x, fmaf(P[1], y, fmaf(P[2], z, P[3])));
            const float bb = fmaf(P[4], x, fmaf(P[5], y, fmaf(P[6], z, P[7])));
            const float w = p.perspective ? fmaf(P[8], x, fmaf(P[9], y, fmaf(P[10], z, P[11]))) : 1.0f;
            if (!(w > 0.0f)) continue;
            const float iw = __frcp_rn(w);
            const float u = fmaf(a, iw, p.det.hu), v = fmaf(bb, iw, p.det.hv);
            if (!(u > -1.0f && u < (float)nu && v > -1.0f && v < (float)nv)) continue;
            const float fu = floorf(u), fv = floorf(v), au = u - fu, av = v - fv;
            const int iu = (int)fu, iv = (int)fv;
            const float val = W2 ? xv * iw * iw : xv, w0 = val * (1.0f - av), w1 = val * av;
            float *r = q + (iv * nu + iu);
            if (iv >= 0 && iu >= 0) atomicAdd(r, w0 * (1.0f - au));
            if (iv >= 0 && iu + 1 < nu) atomicAdd(r + 1, w0 * au);
            if (iv + 1 < nv && iu >= 0) atomicAdd(r + nu, w1 * (1.0f - au));
            if (iv + 1 < nv && iu + 1 < nu) atomicAdd(r + nu + 1, w1 * au);
        }
    };
    if (range_wide(xmax, s_low)) {
        for (int n = v_begin; n < v_end; ++n) add_direct(n);
        return;
    }

    double Xb[3];
    Xb[0] = (bx0 + 0.5 * (BPB_X - 1) - 0.5 * (p.vol.nx - 1)) * p.sx;
    Xb[1] = (by0 + 0.5 * (BPB_Y - 1) - 0.5 * (p.vol.ny - 1)) * p.sy;
    Xb[2] = (bz0 + 0.5 * (BPT_Z - 1) - 0.5 * (p.vol.nz - 1)) * p.sz;
    const float dz = (float)lane - 0.5f * (BPT_Z - 1);
    const f32x2 M2 = splat2(12582912.0f);
    int flip = 0;
    for (int n0 = v_begin; n0 < v_end; n0 += BPT_GROUP) {
        const int nc = min(BPT_GROUP, v_end - n0);
        __syncthreads();   // the previous group's records are done with
        if (tid < nc) bpt_view_setup<W2>(p, n0 + tid, Xb, xmax, box_cap, sv[tid]);
        __syncthreads();
        for (int c = 0; c < nc; ++c) {
            const BpView &V = sv[c].v;
            const int mode = sv[c].mode;
            float *q = ab + (long long)(n0 + c) * nv * nu;
            if (mode == 0) continue;
            if (mode == 2) {
                add_direct(n0 + c);
                continue;
            }
            unsigned *const box = boxes + flip * box_cap;
            flip ^= 1;
            const int eu = V.eu, ev = V.ev, bu = 2 * eu + 1, bv = 2 * ev + 1;
            // tap (floor(qu), floor(qv)) relative to (U0, V0); the box's origin and the magic numbers' bits are folded
            // into the address (unsigned arithmetic mod 2^32)
            const unsigned pitch = 4u * (unsigned)bu;
            const unsigned base = (unsigned)__cvta_generic_to_shared(box) + 4u * (unsigned)eu + pitch * (unsigned)ev -
                                  0x4B400000u * (pitch + 4u);
            const float scale = sv[c].scale;
            const f32x2 qx = pack2(V.Qa[0], V.Qb[0]), qy = pack2(V.Qa[1], V.Qb[1]), qz = pack2(V.Qa[2], V.Qb[2]);
            const f32x2 fuv = pack2(V.fu, V.fv);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int y = 2 * warp + h;
                const float dy = (float)y - 0.5f * (BPB_Y - 1);
                const f32x2 n0y = fma2(splat2(dy), qy, mul2(splat2(dz), qz));
                const float w0y = fmaf(V.Pw[1], dy, fmaf(V.Pw[2], dz, V.w0));
                const float *xr = xs + (y * BPB_X) * BPT_Z + lane;
#pragma unroll 4
                for (int x = 0; x < BPB_X; ++x) {
                    const float xv = xr[x * BPT_Z];
                    if (xv == 0.0f) continue;
                    const float dx = (float)x - 0.5f * (BPB_X - 1);
                    const float iw = rcp_fast(fmaf(V.Pw[0], dx, w0y));
                    const f32x2 qq = fma2(fma2(splat2(dx), qx, n0y), splat2(iw), fuv);
                    const f32x2 t = add2_rd(qq, M2);
                    const f32x2 a = sub2(qq, sub2(t, M2));   // (au, av)
                    const unsigned at = base + 4u * __float_as_uint(lo2(t)) + pitch * __float_as_uint(hi2(t));
                    const float val = (W2 ? xv * iw * iw : xv) * scale;
                    const float v1 = val * hi2(a), v0 = val - v1;
                    const f32x2 vv = pack2(v0, v1);
                    const f32x2 c0 = fma2(vv, splat2(1.0f - lo2(a)), M2), c1 = fma2(vv, splat2(lo2(a)), M2);
                    auto red = [](unsigned addr, float f) {   // no "memory" clobber: the box is read after a barrier
                        asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(addr), "r"((int)(__float_as_uint(f) - 0x4B400000u)));
                    };
                    red(at, lo2(c0));
                    red(at + 4u, lo2(c1));
                    red(at + pitch, hi2(c0));
                    red(at + pitch + 4u, hi2(c1));
                }
            }
            __syncthreads();
            // add the box to the view and clear it; the other box takes the next view meanwhile
            const float unscale = sv[c].unscale, inv_bu = 1.0f / (float)bu;
            for (int e = tid; e < bu * bv; e += BPT_NT) {
                const unsigned s = box[e];
                if (s == 0u) continue;
                box[e] = 0u;
                const int row = (int)(((float)e + 0.5f) * inv_bu), u = V.U0 - eu + (e - row * bu), v = V.V0 - ev + row;
                if ((unsigned)u < (unsigned)nu && (unsigned)v < (unsigned)nv)
                    atomicAdd(q + (v * nu + u), __int2float_rn((int)s) * unscale);
            }
        }
    }
}

// Words of the largest shadow box over every brick and view (0: the kernel does not apply). Rays that run
// mostly along z (direction cosine above 0.7 at the detector's centre) would put the lanes of a warp on one pixel.
int choose_bpt_box(const pyronn_geom *g) {
    if (g->ndim != 3 || g->nz < 8 || g->views_ext.empty()) return 0;
    long long box = 0;
    for (int n = 0; n < g->n_views; ++n) {
        const double *x = g->views_ext.data() + (size_t)n * VIEW64_STRIDE;
        double d[3];
        for (int i = 0; i < 3; ++i)
            d[i] = g->kind == 1 ? x[21 + i] + 0.5 * (g->nu - 1) * x[15 + i] + 0.5 * (g->nv - 1) * x[18 + i] : x[9 + i];
        if (!(std::fabs(d[2]) <= 0.7 * std::sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]))) return 0;
        // the shadow is largest for the bricks nearest the source, at a corner of the volume
        for (int c = 0; c < 8; ++c) {
            const int nb[3] = {(g->nx + BPB_X - 1) / BPB_X, (g->ny + BPB_Y - 1) / BPB_Y, (g->nz + BPT_Z - 1) / BPT_Z};
            const int side[3] = {BPB_X, BPB_Y, BPT_Z}, dim[3] = {g->nx, g->ny, g->nz};
            const double sp[3] = {g->sx, g->sy, g->sz};
            double Xb[3], Pa[3], Pb[3], Pw[3];
            double a0 = 0.0, b0 = 0.0, w0 = 1.0;
            for (int i = 0; i < 3; ++i)
                Xb[i] = (((c >> i) & 1 ? nb[i] - 1 : 0) * side[i] + 0.5 * (side[i] - 1) - 0.5 * (dim[i] - 1)) * sp[i];
            if (g->kind == 1) {
                a0 = x[3], b0 = x[7], w0 = x[11];
                for (int i = 0; i < 3; ++i) {
                    Pa[i] = x[i], Pb[i] = x[4 + i], Pw[i] = x[8 + i];
                    a0 += Pa[i] * Xb[i], b0 += Pb[i] * Xb[i], w0 += Pw[i] * Xb[i];
                }
            } else {
                for (int i = 0; i < 3; ++i) Pa[i] = x[3 + i] / g->du, Pb[i] = x[6 + i] / g->dv, Pw[i] = 0.0;
            }
            double sa = 0.0, sb = 0.0, sw = 0.0;
            for (int i = 0; i < 3; ++i) {
                const double h = 0.5 * (side[i] - 1) + 1.0;
                sa += std::fabs((Pa[i] - a0 / w0 * Pw[i]) * sp[i]) * h;
                sb += std::fabs((Pb[i] - b0 / w0 * Pw[i]) * sp[i]) * h;
                sw += std::fabs(Pw[i] * sp[i]) * h;
            }
            if (!(w0 - sw > 0.25 * w0) || !(sa / (w0 - sw) < 256.0) || !(sb / (w0 - sw) < 256.0)) continue;   // global path
            const int k = std::fabs(Pa[0] - a0 / w0 * Pw[0]) * sp[0] >= std::fabs(Pa[1] - a0 / w0 * Pw[1]) * sp[1] ? 0 : 1;
            const double s = std::fabs(Pa[k] - a0 / w0 * Pw[k]) * sp[k] / w0, sz = std::fabs(Pb[2] - b0 / w0 * Pw[2]) * sp[2] / w0;
            const double spread = std::fabs(Pb[k] - b0 / w0 * Pw[k]) * sp[k] / w0 / std::max(s, 1e-3);
            if (!(bpt_weight_bound((float)std::max(s, 1e-3), (float)std::max(sz, 1e-3), (float)spread) <= 600.0f)) return 0;
            const long long eu = (long long)std::ceil(sa / (w0 - sw)) + 2, ev = (long long)std::ceil(sb / (w0 - sw)) + 2;
            box = std::max(box, (2 * eu + 1) * (2 * ev + 1));
        }
    }
    return box <= BPT_BOX_MAX ? (int)box : 0;
}

bool bpt_bricks_pay(const OpParams &p) { return p.vol_elems * p.batch * p.n_views >= BPT_MIN_UPDATES; }

template <typename T, bool W2>
static int launch_bpt_brick(const OpParams &p, int box_cap, const void *vol, float *acc, cudaStream_t st) {
    const size_t smem = sizeof(float) * (size_t)(BPB_NT * BPT_Z + 2 * box_cap);
    cudaError_t e = cudaFuncSetAttribute(bpt_brick_kernel<T, W2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    const int bricks = ceil_div(p.vol.nx, BPB_X) * ceil_div(p.vol.ny, BPB_Y) * ceil_div(p.vol.nz, BPT_Z);
    // small volumes: the views are split over CTAs (their sums meet in the sinogram's reductions anyway, each
    // view in one CTA) until there are about eight CTAs per SM, at least four views each
    const long long ctas = (long long)bricks * p.batch;
    const int split = (int)std::max<long long>(1, std::min<long long>(ceil_div(p.n_views, 4), stride_grid(1LL << 40, 8) / ctas));
    const int vpc = std::max(ceil_div(p.n_views, split), ceil_div(p.n_views, 65535));
    for (int b0 = 0; b0 < p.batch; b0 += 65535) {
        dim3 grid(bricks, ceil_div(p.n_views, vpc), std::min(p.batch - b0, 65535));
        bpt_brick_kernel<T, W2><<<grid, BPT_NT, smem, st>>>(p, vpc, box_cap, (const T *)vol + b0 * p.vol_elems,
                                                           acc + b0 * p.sino_elems);
    }
    return (int)cudaGetLastError();
}

template <typename T>
static int launch_bpt_t(const OpParams &p, int box_cap, const void *vol, float *acc, cudaStream_t st) {
    return p.perspective && p.weight == PYRONN_BP_INV_W2 ? launch_bpt_brick<T, true>(p, box_cap, vol, acc, st)
                                                         : launch_bpt_brick<T, false>(p, box_cap, vol, acc, st);
}

// acc: zeroed FP32 sinogram
int launch_bpt_bricks(const OpParams &p, int box_cap, const void *vol, float *acc, int dtype, void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    switch (dtype) {
        case PYRONN_F32: return launch_bpt_t<float>(p, box_cap, vol, acc, st);
        case PYRONN_BF16: return launch_bpt_t<__nv_bfloat16>(p, box_cap, vol, acc, st);
        case PYRONN_F16: return launch_bpt_t<__half>(p, box_cap, vol, acc, st);
        default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace pyronn
