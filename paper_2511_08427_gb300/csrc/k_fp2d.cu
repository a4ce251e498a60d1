// Ray-driven forward projector of 2D images (same operator as fp_direct_kernel, Sec. 2.1).
//
// One CTA owns 32 detector bins of up to sixteen consecutive views (one ray per thread, a warp per view; the 16 x 16
// detector tiles of the 3D projectors leave 15 of 16 threads idle on a detector of one row) and marches along the
// rays' dominant axis in slabs: the slab's box, bounded by the end rays of its views, is staged in shared
// memory by row-wise asynchronous copies (zero outside the image) and every ray samples its part of it there, with the
// sample partition and the box-relative positions of the 3D slab projectors. Consecutive views see nearly
// the same box, so they share the cost of staging it. Rows have an odd pitch, so the lanes of a warp read
// different banks whether they spread along x (y march) or along y (x march), and no y-fastest copy of
// the image is needed.
//
// Images of a batch share their geometry: a CTA takes NB of them, interleaved in the box, so that one
// set of positions, floors and weights serves NB images and every tap is one NB-word load.
//
// Bounds: 4 NB shared words per sample (128 B per clock and SM), issue slots, and for one small image the
// slabs' load latency (the grid is only a few CTAs per SM). On GB300, 256^2 image, 512 bins, 360 views, against
// the tiled 3D projector: 567 -> 91 us; eight 362^2 images, 513 bins, 300 views, against the thread-staged one: 20.6 ->
// 0.64 ms. Tiles of 128 bins and four views with loads through registers took 123 us and 0.81 ms (idle SMs at the end,
// few loads in flight), with asynchronous copies 118 us and 0.82 ms, of 64 bins 97 us and 0.68 ms; a second box, loading
// while the first is sampled, changed nothing.
#include <algorithm>
#include <cmath>

#include "device_common.cuh"
#include "host_rays.h"

namespace pyronn {

constexpr int F2_NT = 32;     // bins per CTA
constexpr int F2_VIEWS = 16;  // most views per CTA

template <int NB>
struct F2Word;
template <>
struct F2Word<1> { typedef float type; };
template <>
struct F2Word<2> { typedef float2 type; };
template <>
struct F2Word<4> { typedef float4 type; };

// HELP: warps beyond the CTA's views, which only load boxes
template <typename T, int NB, bool HELP>
__global__ void __launch_bounds__(F2_NT *F2_VIEWS) fp2d_kernel(OpParams p, Fp2dCfg cfg, const T *__restrict__ vol,
                                                     T *__restrict__ sino) {
    typedef typename F2Word<NB>::type Word;
    extern __shared__ __align__(16) unsigned char f2_smem[];
    Word *const box = reinterpret_cast<Word *>(f2_smem);
    // first and last ray of each view, central ray: cx, cy, dx, dy, 1 / dx, 1 / dy
    __shared__ float s_end[2 * F2_VIEWS + 1][6];
    __shared__ int s_srange[2];
    const int tid = threadIdx.x;
    const int nvw = cfg.views, v0 = blockIdx.y * nvw, view = min(v0 + tid / F2_NT, p.n_views - 1);
    const int b0 = blockIdx.z * NB, nb = min(NB, p.batch - b0);
    const int tu0 = blockIdx.x * F2_NT, tu1 = min(tu0 + F2_NT, p.det.nu) - 1;
    const int u = tu0 + tid % F2_NT;
    const bool active = u <= tu1 && v0 + tid / F2_NT < (HELP ? min(v0 + nvw, p.n_views) : p.n_views);
    const T *vb = vol + (long long)b0 * p.vol_elems;
    const FpRec &rec = p.fp[view];
    const int nx = p.vol.nx, ny = p.vol.ny;
    if (tid <= 2 * nvw) {
        const RayIdx c = ray_setup(p.fp[min(v0 + (tid < 2 * nvw ? tid / 2 : 0), p.n_views - 1)], p.vol,
                                   tid == 2 * nvw ? 0.5f * (float)(tu0 + tu1) : (float)(tid & 1 ? tu1 : tu0), 0.0f);
        s_end[tid][0] = c.cx; s_end[tid][1] = c.cy; s_end[tid][2] = c.dx; s_end[tid][3] = c.dy;
        s_end[tid][4] = 1.0f / c.dx; s_end[tid][5] = 1.0f / c.dy;
    }
    if (tid == 0) {
        s_srange[0] = 1 << 30;
        s_srange[1] = -(1 << 30);
    }
    const RayIdx r = ray_setup(rec, p.vol, (float)min(u, tu1), 0.0f);
    int k0 = 0, k1 = -1;
    bool hit = active && ray_k_range(r, p.vol, p.dt, k0, k1);
    __syncthreads();
    const int m = fabsf(s_end[2 * nvw][2]) >= fabsf(s_end[2 * nvw][3]) ? 0 : 1, a1 = 1 - m;   // march and cross axis
    const int Nm = m == 0 ? nx : ny, N1 = m == 0 ? ny : nx;
    const float cm = m == 0 ? r.cx : r.cy, dm = m == 0 ? r.dx : r.dy;
    const bool marchable = fabsf(dm) > 1e-3f * (fabsf(r.dx) + fabsf(r.dy));
    const bool direct_ray = hit && !marchable;
    if (direct_ray) hit = false;
    const float inv_step = marchable ? 1.0f / (p.dt * dm) : 0.0f;
    const int D = cfg.depth, G = cfg.guard;
    const int nslab = (Nm + 1 + D - 1) / D;   // slab s covers floor(q_m) in [-1 + s D, -1 + (s + 1) D)
    const float hdt = 0.5f * p.dt;
    if (hit) {
        const float qa = fmaf(fmaf((float)k0, p.dt, hdt), dm, cm), qb = fmaf(fmaf((float)k1, p.dt, hdt), dm, cm);
        const float qlo = fmaxf(fminf(qa, qb), -1.0f), qhi = fminf(fmaxf(qa, qb), (float)Nm);
        int slo = ((int)floorf(qlo) + 1) / D, shi = ((int)floorf(qhi) + 1) / D;
        slo = max(min(slo, nslab - 1), 0);
        shi = max(min(shi, nslab - 1), 0);
        atomicMin(&s_srange[0], slo);
        atomicMax(&s_srange[1], shi);
    }
    __syncthreads();
    const int s_first = s_srange[0], s_last = s_srange[1];
    float acc[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) acc[i] = 0.0f;
    const float M = 12582912.0f;

    // image i at global index coordinates (off-box samples and rays outside the slab march)
    auto global_sample = [&](float qx, float qy) {
#pragma unroll
        for (int i = 0; i < NB; ++i)
            if (i < nb) acc[i] += trilerp_zero(vb + i * p.vol_elems, p.vol, qx, qy, 0.0f);
    };

    struct Slab {
        int lox, loy, Ex, Ey;   // box origin and extents
        bool staged;
    };
    auto bounds = [&](int s) {
        const int b_lo = -1 + s * D, b_hi = min(b_lo + D, Nm);
        float mn = 3e38f, mx = -3e38f;
        for (int c = 0; c < 2 * nvw; ++c) {
            const float idm = s_end[c][4 + m];
#pragma unroll
            for (int pl = 0; pl < 2; ++pl) {
                const float t = ((float)(pl ? b_hi + G : b_lo - G) - s_end[c][m]) * idm;
                const float q = fmaf(t, s_end[c][2 + a1], s_end[c][a1]);
                mn = fminf(mn, q);
                mx = fmaxf(mx, q);
            }
        }
        const float gf = (float)(G + 2);
        mn = fmaxf(mn, -gf);
        mx = fminf(mx, (float)N1 + gf);
        const int lo1 = max((int)floorf(mn) - 1, -1 - G), hi1 = min((int)floorf(mx) + 2, N1 + G);
        const int lom = b_lo - G, him = b_hi + G;
        Slab S;
        S.lox = m == 0 ? lom : lo1;
        S.loy = m == 0 ? lo1 : lom;
        S.Ex = (m == 0 ? him : hi1) - S.lox + 1;
        S.Ey = (m == 0 ? hi1 : him) - S.loy + 1;
        S.staged = S.Ex > 0 && S.Ey > 0 && (long long)(S.Ex | 1) * S.Ey <= cfg.box_elems;
        return S;
    };
    // A warp loads one row of the box, or two of at most 16 columns (x march). FP32 words go by asynchronous copies, which
    // are all in flight at once; the other types are converted on the way.
    auto stage = [&](const Slab &S) {
        if (!S.staged) return;
        const int lanes = S.Ex <= 16 ? 16 : 32, rows = (int)blockDim.x / lanes, pitch = S.Ex | 1;
#pragma unroll 4
        for (int row = tid / lanes; row < S.Ey; row += rows) {
            const int gy = S.loy + row;
            const bool iny = (unsigned)gy < (unsigned)ny;
            const T *g = vb + (long long)gy * nx;
            for (int x = tid % lanes; x < S.Ex; x += lanes) {
                const int gx = S.lox + x;
                const bool in = iny && (unsigned)gx < (unsigned)nx;
                Word *dst = box + (row * pitch + x);
                if constexpr (sizeof(T) == 4) {
                    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
#pragma unroll
                    for (int i = 0; i < NB; ++i) {
                        const bool ok = in && i < nb;
                        const T *src = ok ? g + i * p.vol_elems + gx : vb;
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d + 4u * i), "l"(src), "r"(ok ? 4 : 0)
                                     : "memory");
                    }
                } else {
                    float w[NB];
#pragma unroll
                    for (int i = 0; i < NB; ++i) w[i] = in && i < nb ? ldg_f32(g + i * p.vol_elems + gx) : 0.0f;
                    if constexpr (NB == 1) *dst = w[0];
                    else if constexpr (NB == 2) *dst = make_float2(w[0], w[1]);
                    else *dst = make_float4(w[0], w[1], w[2], w[3]);
                }
            }
        }
    };
    // the samples of this thread's ray in slab s
    auto march = [&](int s, const Slab &S) {
        const int b_lo = -1 + s * D, b_hi = min(b_lo + D, Nm), lox = S.lox, loy = S.loy, Ex = S.Ex, Ey = S.Ey, pitch = Ex | 1;
        int ka = 0, kb = -1;
        if (hit) {
            if (dm > 0.0f) {
                ka = (int)ceilf(fmaf((float)b_lo - cm, inv_step, -0.5f));
                kb = (int)ceilf(fmaf((float)b_hi - cm, inv_step, -0.5f)) - 1;
            } else {
                ka = (int)floorf(fmaf((float)b_hi - cm, inv_step, -0.5f)) + 1;
                kb = (int)floorf(fmaf((float)b_lo - cm, inv_step, -0.5f));
            }
            ka = max(ka, k0);
            kb = min(kb, k1);
        }
        if (!S.staged) {   // never expected (the host bound covers every tile)
            if (tid == 0) atomicAdd(p.flags + FLAG_SLAB_OVERFLOW, 1);
            for (int k = ka; k <= kb; ++k) {
                const float t = fmaf((float)k, p.dt, hdt);
                global_sample(fmaf(t, r.dx, r.cx), fmaf(t, r.dy, r.cy));
            }
            return;
        }
        if (ka > kb) return;
        const float c0x = fmaf(hdt, r.dx, r.cx - (float)lox), c0y = fmaf(hdt, r.dy, r.cy - (float)loy);
        const float stx = p.dt * r.dx, sty = p.dt * r.dy;
        auto taps = [&](int base, float ax, float ay) {
            const Word *s0 = box + base, *s1 = s0 + pitch;
            if constexpr (NB == 1) {
                const f32x2 c = lerp2(splat2(ax), pack2(s0[0], s1[0]), pack2(s0[1], s1[1]));
                acc[0] += fmaf(ay, hi2(c) - lo2(c), lo2(c));
            } else {
                const Word v00 = s0[0], v01 = s0[1], v10 = s1[0], v11 = s1[1];
                const f32x2 a2 = splat2(ax), b2 = splat2(ay);
                {
                    const f32x2 c = lerp2(b2, lerp2(a2, pack2(v00.x, v00.y), pack2(v01.x, v01.y)),
                                          lerp2(a2, pack2(v10.x, v10.y), pack2(v11.x, v11.y)));
                    acc[0] += lo2(c);
                    acc[1] += hi2(c);
                }
                if constexpr (NB == 4) {
                    const f32x2 c = lerp2(b2, lerp2(a2, pack2(v00.z, v00.w), pack2(v01.z, v01.w)),
                                          lerp2(a2, pack2(v10.z, v10.w), pack2(v11.z, v11.w)));
                    acc[2] += lo2(c);
                    acc[3] += hi2(c);
                }
            }
        };
        // Positions are one correctly rounded FMA of the sample index, hence monotone in it: when the first
        // and the last sample's cells lie in the box, all of them do. The comparisons fail for NaN.
        const float qax = fmaf((float)ka, stx, c0x), qbx = fmaf((float)kb, stx, c0x);
        const float qay = fmaf((float)ka, sty, c0y), qby = fmaf((float)kb, sty, c0y);
        const float ex = (float)(Ex - 1), ey = (float)(Ey - 1);
        if (qax >= 0.f && qbx >= 0.f && qax < ex && qbx < ex && qay >= 0.f && qby >= 0.f && qay < ey && qby < ey) {
            const f32x2 st2 = pack2(stx, sty), c02 = pack2(c0x, c0y), M2 = splat2(M), one2 = splat2(1.0f);
            f32x2 kf2 = splat2((float)ka);
            const unsigned boff = 0x4B400000u * (unsigned)(pitch + 1);   // the magic numbers' bits, folded into the offset
#pragma unroll 4
            for (int k = ka; k <= kb; ++k) {
                const f32x2 q = fma2(kf2, st2, c02);
                const f32x2 t = add2_rd(q, M2);
                const f32x2 a = sub2(q, sub2(t, M2));
                taps((int)((unsigned)__float_as_int(hi2(t)) * (unsigned)pitch + (unsigned)__float_as_int(lo2(t)) - boff),
                     lo2(a), hi2(a));
                kf2 = add2(kf2, one2);
            }
        } else {
            for (int k = ka; k <= kb; ++k) {
                const float qx = fmaf((float)k, stx, c0x), qy = fmaf((float)k, sty, c0y);
                const float tx = __fadd_rd(qx, M), ty = __fadd_rd(qy, M);
                const unsigned ix = (unsigned)(__float_as_int(tx) - 0x4B400000), iy = (unsigned)(__float_as_int(ty) - 0x4B400000);
                if (ix < (unsigned)(Ex - 1) && iy < (unsigned)(Ey - 1)) {
                    taps((int)(iy * (unsigned)pitch + ix), qx - (tx - M), qy - (ty - M));
                } else {
                    atomicAdd(p.flags + FLAG_SLAB_OUT_OF_BOX, 1);
                    global_sample(qx + (float)lox, qy + (float)loy);
                }
            }
        }
    };

    for (int s = s_first; s <= s_last; ++s) {
        const Slab S = bounds(s);
        __syncthreads();   // the previous slab's readers are done
        stage(S);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        march(s, S);
    }
    if (direct_ray) {
        atomicAdd(p.flags + FLAG_SLAB_DIRECT_RAY, 1);
        for (int k = k0; k <= k1; ++k) {
            const float t = fmaf((float)k, p.dt, hdt);
            global_sample(fmaf(t, r.dx, r.cx), fmaf(t, r.dy, r.cy));
        }
    }
    if (active) {
        T *out = sino + (long long)b0 * p.sino_elems + (long long)view * p.det.nu + u;
#pragma unroll
        for (int i = 0; i < NB; ++i)
            if (i < nb) out[i * p.sino_elems] = from_f32<T>(acc[i] * p.dt);
    }
}

// ---------------------------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------------------------

// Largest box (elements per image) of any tile of nvw consecutive views over its slabs. The range of a tile's
// end rays is convex in the plane position, so the first and the last slab of full depth bound the ones between; the one
// behind them may be cut.
static long long fp2d_bound(const pyronn_geom *g, const Fp2dCfg &c, int nvw) {
    const int dims[2] = {g->nx, g->ny};
    long long best = 0;
    for (int v0 = 0; v0 < g->n_views; v0 += nvw)
        for (int tu0 = 0; tu0 < g->nu; tu0 += F2_NT) {
            const int tu1 = std::min(tu0 + F2_NT, g->nu) - 1;
            const RayD ctr = ray_setup_d(g->fp_rec[v0], g, 0.5 * (tu0 + tu1), 0);
            RayD e[2 * F2_VIEWS];
            for (int k = 0; k < 2 * nvw; ++k)
                e[k] = ray_setup_d(g->fp_rec[std::min(v0 + k / 2, g->n_views - 1)], g, k & 1 ? tu1 : tu0, 0);
            const double amax = std::max(std::fabs(ctr.d[0]), std::fabs(ctr.d[1]));
            for (int m = 0; m < 2; ++m) {
                if (std::fabs(ctr.d[m]) < 0.999 * amax) continue;   // the kernel may pick either axis near a tie
                const int a1 = 1 - m, Nm = dims[m], nslab = (Nm + 1 + c.depth - 1) / c.depth;
                for (int s : {0, std::max(nslab - 2, 0), nslab - 1}) {
                    const int b_lo = -1 + s * c.depth, b_hi = std::min(b_lo + c.depth, Nm);
                    double mn = 1e300, mx = -1e300;
                    for (int k = 0; k < 2 * nvw; ++k)
                        for (int pl = 0; pl < 2; ++pl) {
                            const double t = ((pl ? b_hi + c.guard : b_lo - c.guard) - e[k].c[m]) / e[k].d[m];
                            const double q = e[k].c[a1] + t * e[k].d[a1];
                            mn = std::min(mn, q);
                            mx = std::max(mx, q);
                        }
                    const long long e1 = box_extent(mx - mn, 6, dims[a1] + 2 * c.guard + 2);
                    if (e1 < 0) continue;
                    const long long em = c.depth + 2 * c.guard + 1;
                    best = std::max(best, m == 0 ? (em | 1) * e1 : em * (e1 | 1));
                }
            }
        }
    return best;
}

// valid = 0 for 3D geometries, steps of 2^16 voxels or more and boxes above 64 KB (one view, one image).
// Depth: 29 planes and the guard planes of the default step make x-march rows of 32 words, one pass of a
// warp (61 planes: 82 against 91 us and 125 against 165 us for one image, but 482 against 241 us for 32 images of 128^2,
// whose CTAs then have an SM each). Views per CTA: sixteen, eight, four, then two, where that many have a box at most 1.4
// times one view's (closely spaced views; 1.25: 130 us instead of 91, 2: 111) and leave at least 300 CTAs (1000: 128^2
// image, 192 bins, 120 views, 47 us instead of 33). Neither depends on the batch, so a batch gives bit for bit what its
// images give one by one.
Fp2dCfg choose_fp2d_cfg(const pyronn_geom *g) {
    Fp2dCfg c{};
    if (g->ndim != 2) return c;
    const double smin = std::min(g->sx, g->sy);
    if (!(g->dt / smin < 65535.0)) return c;
    c.guard = 1 + (int)std::floor(g->dt / smin);
    c.depth = 29;
    c.views = 1;
    long long best = fp2d_bound(g, c, 1);
    const long long cap = 64 * 1024 / 4, one = best;
    for (int nvw = F2_VIEWS; nvw > 1; nvw >>= 1) {
        if ((long long)ceil_div(g->n_views, nvw) * ceil_div(g->nu, F2_NT) < 300) continue;
        const long long many = fp2d_bound(g, c, nvw);
        if (many > one + one * 2 / 5 || many > cap) continue;
        c.views = nvw;
        best = many;
        break;
    }
    c.box_elems = (int)std::min(best, cap);
    c.valid = best > 0 && best <= cap;
    return c;
}

template <typename T, int NB>
static int launch_fp2d_t(const OpParams &p, const Fp2dCfg &cfg, const void *vol, void *sino, cudaStream_t st) {
    const size_t smem = sizeof(float) * (size_t)NB * (size_t)cfg.box_elems;
    // boxes that would keep a CTA's own warps loading for long (bins much wider than pixels, other types than FP32): more warps
    // load them, one per 64 words and thread, or 128 where the words of several images go by asynchronous copies (128^2 image, 40
    // bins of 5 pixels, 180 views: 59 -> 35 us; three such images of 128 bins of 1.6 pixels, 120 views, BF16: 123 -> 60;
    // eight 362^2 images, 103 words per thread: 642 us, and 650 with eight warps)
    int warps = cfg.views;
    while (warps < F2_VIEWS && (long long)NB * cfg.box_elems > (sizeof(T) == 2 || NB == 1 ? 64LL : 128LL) * F2_NT * warps) warps <<= 1;
    auto kern = warps > cfg.views ? fp2d_kernel<T, NB, true> : fp2d_kernel<T, NB, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    const int per_launch = 65535 * NB;
    for (int b0 = 0; b0 < p.batch; b0 += per_launch)
        for (int v0 = 0; v0 < p.n_views; v0 += 65535 / F2_VIEWS * F2_VIEWS) {
            OpParams q = p;
            q.batch = std::min(p.batch - b0, per_launch);
            q.n_views = std::min(p.n_views - v0, 65535 / F2_VIEWS * F2_VIEWS);
            q.fp = p.fp + v0;
            dim3 grid(ceil_div(p.det.nu, F2_NT), ceil_div(q.n_views, cfg.views), ceil_div(q.batch, NB));
            kern<<<grid, F2_NT * warps, smem, st>>>(q, cfg, (const T *)vol + b0 * p.vol_elems,
                                                         (T *)sino + b0 * p.sino_elems + (long long)v0 * p.det.nu);
        }
    return (int)cudaGetLastError();
}

template <typename T>
static int launch_fp2d_nb(const OpParams &p, const Fp2dCfg &cfg, int nb, const void *vol, void *sino, cudaStream_t st) {
    if (nb == 4) return launch_fp2d_t<T, 4>(p, cfg, vol, sino, st);
    if (nb == 2) return launch_fp2d_t<T, 2>(p, cfg, vol, sino, st);
    return launch_fp2d_t<T, 1>(p, cfg, vol, sino, st);
}

int launch_fp2d(const OpParams &p, const Fp2dCfg &cfg, int nb, const void *vol, void *sino, int dtype, void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    switch (dtype) {
        case PYRONN_F32: return launch_fp2d_nb<float>(p, cfg, nb, vol, sino, st);
        case PYRONN_BF16: return launch_fp2d_nb<__nv_bfloat16>(p, cfg, nb, vol, sino, st);
        case PYRONN_F16: return launch_fp2d_nb<__half>(p, cfg, nb, vol, sino, st);
        default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace pyronn
