// Matched adjoint of 2D images (same operator as adjoint_scatter_kernel, Sec. 2.2 A^T): every sample of
// every ray adds y dt times its four bilinear weights to its cell's corners.
//
// One CTA owns a B x B brick of the image (with a margin of one pixel on every side, so that the corners of
// a sample need no tests) and a range of views, for up to NB images of a batch, which share all positions and
// weights. For each group of views it walks the rays that cross the brick, a warp on 32 adjacent rays of one
// view, and adds the contributions to int32 fixed-point sums in shared memory, one integer reduction per corner
// (FP32 reductions in shared memory are compare-and-swap loops on this GPU, about 3.6 times slower); the
// sums then go to the image by FP32 reductions. The brick, not the slab of the 3D adjoint, is what stays in shared memory:
// a 2D image is small, and the slabs of all views would reduce into the same few lines of L2.
// Splitting the views over CTAs fills the chip: a 256^2 image alone has 16 bricks of 64^2.
//
// Positions are relative to the brick centre with FP64 per-(brick, view) constants, as in the 3D bricks
// (brick_view.cuh), but rays are counted from the middle of the brick's footprint, whose ray passes the centre closely, and
// the step from ray to ray is kept in two parts: counted from the footprint's end, the rounding of the first ray's offset
// and of the step, times up to 130 rays, moved all rays of a view by several 1e-6 pixel. The adjoint of white noise on
// 256^2 pixels, 512 bins, 360 views then has an error of 1.3e-6, against 3.4e-6 (32^2 bricks counted from the end:
// 1.8e-6). Fixed point: contributions enter as round(c 2^e); 2^e is chosen per view group and image so that no
// contribution exceeds 2^22 (then one FFMA with 1.5 2^23 rounds it) and no sum can exceed 2^30, from
// |sum| <= max |y| dt sum_views R_view (1 / delta + 1): R the rays that can cross one pixel's support
// (-1, 1)^2, whose shadow is at most 2 sqrt(2) pixels wide, and delta the distance of consecutive samples in pixels (see
// k_adjoint_slab.cu). A group ends where the bound would pass 256, which keeps the quantum between 2^-22 and 2^-21 of
// the largest contribution. Views whose bound alone passes it (very dense rays), values that are not finite and groups of a
// wide range use FP32 sums: the quantum is that of the largest |y| anywhere in the group, so pixels that only small values
// reach would lose bits that FP32 sums keep. A group counts as wide where some eight adjacent rays of a view (all
// nonzero; five in footprints of less than 16) stay below 1 / WIDE_RANGE of its largest value.
//
// Bound by the shared reductions (4 NB per sample, two passes where two lanes share a word) and issue slots. On GB300,
// 256^2 image, 512 bins, 360 views, against FP32 shared sums in one CTA per 32^2 brick: 4218 -> 110 us (FP32
// sums throughout: 268 us); eight 362^2 images, 513 bins, 300 views: 13.6 -> 0.89 ms.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "brick_view.cuh"

namespace pyronn {

constexpr int A2_NT = 256, A2_CHUNK = 32;
constexpr float A2_GROUP_BOUND = 256.0f;

struct A2View : BrickView {   // A, Eu, D and Cu for the ray u_lo + k_mid
    int k_mid;
    float Aq[2], Eq[2], El[2];   // point on the brick plane in pixels, plus 1/2, and its step per ray in two parts
    float H;   // bound on the sum of the weights of one view's samples in one pixel; huge: unbounded
};

// FP64 constants and the weight bound of one (brick, view), isp the pixels per mm, by four lanes: each projects one corner of the extended
// brick, the first goes on. With all corners in one lane, while the CTA waits for it: 120 us instead of 105 (256^2 image,
// 360 views), 40 instead of 30 (128^2, 120 views).
static __device__ void adj2d_view_setup(const OpParams &p, int view, const double Xb[3], const double elo[3],
                                        const double ehi[3], double2 isp, A2View &V) {
    const int c = threadIdx.x & 3;
    const double X[3] = {(c & 1) ? ehi[0] : elo[0], (c & 2) ? ehi[1] : elo[1], 0.0};
    double u = 0.0, v;
    const bool behind = !brick_corner(p, p.views64 + (size_t)view * VIEW64_STRIDE, X, u, v);
    // the footprint with a bin on either side, clamped to the detector and two bins around it before the conversion
    u = fmin(fmax(u, -2.0), (double)p.det.nu + 1.0);
    int u_lo = behind ? 0 : max((int)ceil(u) - 1, 0), u_hi = behind ? p.det.nu - 1 : min((int)floor(u) + 1, p.det.nu - 1);
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        u_lo = min(u_lo, __shfl_xor_sync(0xffffffffu, u_lo, o));
        u_hi = max(u_hi, __shfl_xor_sync(0xffffffffu, u_hi, o));
    }
    if (c) return;
    V.u_lo = u_lo;
    V.v_lo = 0;
    V.nu_r = u_hi >= u_lo ? u_hi - u_lo + 1 : 0;
    V.nv_r = V.nu_r ? 1 : 0;
    V.H = 3.0e38f;
    if (V.nu_r == 0) return;
    V.k_mid = (u_hi - u_lo) >> 1;
    double at[4];
    brick_view_rays(p, view, Xb, u_lo + V.k_mid, 0, V, at);
    for (int a = 0; a < 2; ++a) {
        const double is = a ? isp.y : isp.x, step = at[2 + a] * is;
        V.Aq[a] = (float)(at[a] * is + 0.5);
        V.Eq[a] = (float)step;
        V.El[a] = (float)(step - (double)V.Eq[a]);
    }
    // perpendicular distance of adjacent rays in pixels at the brick centre, the smaller at the footprint's two
    // ends (it falls towards a flat detector's edges), times the least magnification over the brick
    const float is0 = p.vol.isx, is1 = p.vol.isy;
    float least = 3.0e38f;
    for (int c = 0; c < 2; ++c) {
        const float f = (float)((c ? V.nu_r - 1 : 0) - V.k_mid);
        const float d0 = fmaf(f, V.Cu[0], V.D[0]) * is0, d1 = fmaf(f, V.Cu[1], V.D[1]) * is1;
        least = fminf(least, fabsf(V.Eu[0] * is0 * d1 - V.Eu[1] * is1 * d0) * rsqrtf(fmaf(d0, d0, d1 * d1)));
    }
    if (p.perspective) {
        const double *x = p.views64 + (size_t)view * VIEW64_STRIDE;
        const double *S = x + 12, *nrm = x + 24;
        const double at = (Xb[0] - S[0]) * nrm[0] + (Xb[1] - S[1]) * nrm[1];
        const double half = 0.5 * ((ehi[0] - elo[0]) * fabs(nrm[0]) + (ehi[1] - elo[1]) * fabs(nrm[1]));
        least *= (float)((fabs(at) - half) / fabs(at));   // not above zero where the brick reaches the source plane
    }
    if (!(least > 1.0e-3f)) return;
    const float smax = (float)fmax(p.sx, p.sy);
    V.H = (floorf(1.1f * 2.8284272f / least) + 2.0f) * (smax / p.dt + 1.0f);
}

// int32 reduction / FP32 reduction at a shared-memory address (no "memory" clobber: see k_adjoint_slab.cu)
static __device__ __forceinline__ void a2_red_s32(unsigned addr, int v) {
    asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(addr), "r"(v));
}
static __device__ __forceinline__ void a2_red_f32(unsigned addr, float v) {
    asm volatile("red.shared.add.f32 [%0], %1;" ::"r"(addr), "f"(v));
}

// FP32 sum into global memory. Reductions there flush subnormal sums to zero, so tiny addends, whose sum may
// be one, are added in a register.
static __device__ __forceinline__ void a2_add(float *dst, float v) {
    if (!(fabsf(v) < 1.0e-30f)) {
        atomicAdd(dst, v);
        return;
    }
    unsigned *w = reinterpret_cast<unsigned *>(dst), seen = *reinterpret_cast<volatile unsigned *>(dst), was;
    do {
        was = seen;
        seen = atomicCAS(w, was, __float_as_uint(__uint_as_float(was) + v));
    } while (seen != was);
}

template <int B, int NB>
struct A2Shared {
    static constexpr int PITCH = B + 3;   // B + 2 columns, odd: 32 rows of one column lie on 32 banks
    static constexpr int CELLS = (B + 2) * PITCH;
    unsigned sum[NB][CELLS];              // fixed-point or FP32 sums of the current group, zero between groups
    A2View sv[A2_CHUNK];
    int s_off[A2_CHUNK + 1];              // first ray slot of each view (whole warps per view)
    unsigned ymax[NB], ylow[NB];          // largest |y| dt, and the least maximum of eight adjacent rays
};

// FP32 running sums of the brick where the output is not FP32 (written once at the end)
template <int B, int NB, bool KEEP>
struct A2Kept {
    float acc[NB][KEEP ? B * B : 1];
};

// DENSE: a warp's lanes on rays spread over the footprint instead of adjacent ones, of which all would meet on a word
template <typename T, int B, int NB, bool DENSE>
__global__ void __launch_bounds__(A2_NT, B == 32 ? 4 : 3) adjoint2d_kernel(OpParams p, double2 isp, int views_per_cta, int allow_fixed,
                                                                           const T *__restrict__ sino, T *__restrict__ vol) {
    constexpr bool KEEP = sizeof(T) != 4;
    typedef A2Shared<B, NB> Sh;
    extern __shared__ __align__(16) unsigned char a2_smem[];
    Sh &S = *reinterpret_cast<Sh *>(a2_smem);
    A2Kept<B, NB, KEEP> &K = *reinterpret_cast<A2Kept<B, NB, KEEP> *>(a2_smem + (sizeof(Sh) + 15) / 16 * 16);
    const int tid = threadIdx.x, lane = tid & 31;
    const int nbx = (p.vol.nx + B - 1) / B;
    const int bx0 = (blockIdx.x % nbx) * B, by0 = (blockIdx.x / nbx) * B;
    const int v_begin = blockIdx.y * views_per_cta, v_end = min(v_begin + views_per_cta, p.n_views);
    const int b0 = blockIdx.z * NB, nb = min(NB, p.batch - b0);
    const T *sb = sino + (long long)b0 * p.sino_elems;
    T *vb = vol + (long long)b0 * p.vol_elems;
    const float dt = p.dt, isx = p.vol.isx, isy = p.vol.isy, sx = (float)p.sx, sy = (float)p.sy;
    const int nu = p.det.nu;

    for (int e = tid; e < NB * Sh::CELLS; e += A2_NT) (&S.sum[0][0])[e] = 0u;
    if (KEEP)
        for (int e = tid; e < NB * B * B; e += A2_NT) (&K.acc[0][0])[e] = 0.0f;

    // brick centre and the brick with its margin, relative to the volume centre (mm)
    const double sp[3] = {p.sx, p.sy, p.sz};
    const double hv3[3] = {0.5 * (p.vol.nx - 1), 0.5 * (p.vol.ny - 1), 0.0};
    const int org[3] = {bx0, by0, 0}, ext[3] = {B, B, 1};
    double Xb[3], elo[3], ehi[3];
    for (int a = 0; a < 3; ++a) {
        Xb[a] = (org[a] + 0.5 * (ext[a] - 1) - hv3[a]) * sp[a];
        elo[a] = (org[a] - 1 - hv3[a]) * sp[a];
        ehi[a] = (org[a] + ext[a] - hv3[a]) * sp[a];
    }
    const float Xb0 = (float)Xb[0], Xb1 = (float)Xb[1];
    // index positions relative to column and row B / 2 of the brick with its margin: floor(q) is -B / 2 .. B / 2 for samples
    // that count
    constexpr int HB = B / 2;
    const float M = 12582912.0f;

    for (int n0 = v_begin; n0 < v_end; n0 += A2_CHUNK) {
        const int nc = min(A2_CHUNK, v_end - n0);
        __syncthreads();
        if (tid >> 5 < (4 * nc + 31) >> 5)   // whole warps; the lanes past the last view repeat it
            adj2d_view_setup(p, n0 + min(tid >> 2, nc - 1), Xb, elo, ehi, isp, S.sv[tid >> 2]);
        __syncthreads();
        if (tid == 0) {
            int o = 0;
            for (int c = 0; c < nc; ++c) {
                S.s_off[c] = o;
                o += (S.sv[c].nu_r + 31) & ~31;
            }
            S.s_off[nc] = o;
        }
        for (int c0 = 0, c1; c0 < nc; c0 = c1) {
            // group of views c0 .. c1 - 1: as many as the bound on the fixed-point sums allows
            float H = S.sv[c0].nu_r ? S.sv[c0].H : 0.0f;
            for (c1 = c0 + 1; c1 < nc; ++c1) {
                const float h = S.sv[c1].nu_r ? S.sv[c1].H : 0.0f;
                if (!(H + h <= A2_GROUP_BOUND)) break;
                H += h;
            }
            if (tid < NB) S.ymax[tid] = 0u, S.ylow[tid] = 0xffffffffu;
            __syncthreads();   // also: the ray slots, and the previous group's sums have been flushed
            const int r0 = S.s_off[c0], r1 = S.s_off[c1];
            {
                unsigned big[NB], low[NB];
#pragma unroll
                for (int i = 0; i < NB; ++i) big[i] = 0u, low[i] = 0xffffffffu;
                int c = c0;
                for (int r = r0 + tid; r < r1; r += A2_NT) {   // whole warps: r1 - r0 is a multiple of 32
                    while (r >= S.s_off[c + 1]) ++c;
                    const int k = r - S.s_off[c];
                    const T *q = sb + (long long)(n0 + c) * nu + S.sv[c].u_lo + k;
#pragma unroll
                    for (int i = 0; i < NB; ++i) {
                        const unsigned v = k < S.sv[c].nu_r && i < nb
                                               ? __float_as_uint(fabsf(ldg_f32(q + i * p.sino_elems) * dt)) : 0u;
                        big[i] = max(big[i], v);
                        low[i] = min(low[i], range_run8(v, S.sv[c].nu_r < 16 ? 5 : 8));
                    }
                }
#pragma unroll
                for (int i = 0; i < NB; ++i) {
                    const unsigned w = __reduce_max_sync(0xffffffffu, big[i]), l = __reduce_min_sync(0xffffffffu, low[i]);
                    if (lane == 0 && w) atomicMax(&S.ymax[i], w);
                    if (lane == 0) atomicMin(&S.ylow[i], l);
                }
            }
            __syncthreads();
            // exponent e of the scale per image: max |y| dt 2^e < 2^22, for any finite value (2^e itself may leave the
            // FP32 range, so it is applied as two factors). FP32 sums for the whole group where an image
            // holds a value that is not finite or has a wide range.
            int e2[NB];
            bool fixed = allow_fixed && H <= A2_GROUP_BOUND, any = false;
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const unsigned yb = S.ymax[i];
                e2[i] = 22 + 126 - (int)(yb >> 23);   // |y| dt < 2^(exponent field - 126)
                any = any || yb != 0u;
                if (yb >= 0x7f800000u || range_wide(yb, S.ylow[i])) fixed = false;
            }
            auto pow2 = [](int x) { return __int_as_float((x + 127) << 23); };
            if (!any) continue;   // every ray is zero (the same for every thread)
            int c = c0;
            for (int r = r0 + tid; r < r1; r += A2_NT) {   // whole warps: r1 - r0 is a multiple of 32
                while (r >= S.s_off[c + 1]) ++c;
                const A2View &V = S.sv[c];
                int k = r - S.s_off[c];
                if (DENSE) k = (k & 31) * ((S.s_off[c + 1] - S.s_off[c]) >> 5) + (k >> 5);
                if (k >= V.nu_r) continue;
                const T *yq = sb + (long long)(n0 + c) * nu + V.u_lo + k;
                float y[NB];
                bool some = false;
#pragma unroll
                for (int i = 0; i < NB; ++i) {
                    y[i] = i < nb ? ldg_f32(yq + i * p.sino_elems) * dt : 0.0f;
                    some = some || y[i] != 0.0f;
                    if (fixed) y[i] = y[i] * pow2(e2[i] >> 1) * pow2(e2[i] - (e2[i] >> 1));
                }
                if (!some) continue;
                // the ray's point on the brick plane, direction, and phase (see brick_view.cuh and k_adjoint_brick.cu)
                const float fu = (float)(k - V.k_mid);
                const float qP0 = fmaf(fu, V.Eq[0], fmaf(fu, V.El[0], V.Aq[0])), qP1 = fmaf(fu, V.Eq[1], fmaf(fu, V.El[1], V.Aq[1]));
                const float P0 = (qP0 - 0.5f) * sx, P1 = (qP1 - 0.5f) * sy;
                const float L0 = fu * V.Cu[0], L1 = fu * V.Cu[1];
                const float DL = fmaf(V.D[0], L0, V.D[1] * L1), LL = fmaf(L0, L0, L1 * L1);
                const float eps = (2.0f * DL + LL) / V.nD2;
                const float sq = sqrtf(1.0f + eps), inv = V.inv_nD / sq, g = -eps / (sq * (1.0f + sq));
                const float d0 = (V.D[0] + L0) * inv, d1 = (V.D[1] + L1) * inv;
                const float e = fmaf(Xb0, fmaf(V.dref[0], g, L0 * inv), Xb1 * fmaf(V.dref[1], g, L1 * inv)) +
                                fmaf(P0, d0, P1 * d1);
                const float c_r = (0.5f - V.f) * dt - e;   // sample j lies at j dt + c_r along d from P
                const float qd0 = d0 * isx, qd1 = d1 * isy;
                // samples whose cell lies in the margin-extended brick: -B / 2 <= q < B / 2 + 1 on both axes
                float slo = -3.0e38f, shi = 3.0e38f;
                bool empty = false;
                clip_axis(qP0 + (float)(HB - 1), qd0, B, slo, shi, empty);
                clip_axis(qP1 + (float)(HB - 1), qd1, B, slo, shi, empty);
                if (empty || !(shi > slo)) continue;
                const float idt = 1.0f / dt;
                int j = (int)floorf((slo - c_r) * idt), j1 = (int)ceilf((shi - c_r) * idt);
                const float low = (float)-HB, top = (float)(HB + 1);
                // position of sample j; monotone in j on both axes, so trimming the ends to samples in the brick
                // leaves only samples in the brick
                auto inside = [&](int at) {
                    const float s = fmaf((float)at, dt, c_r);
                    const float q0 = fmaf(s, qd0, qP0), q1 = fmaf(s, qd1, qP1);
                    return q0 >= low && q0 < top && q1 >= low && q1 < top;
                };
                while (j <= j1 && !inside(j)) ++j;
                while (j1 >= j && !inside(j1)) --j1;
                if (j > j1) continue;
                const f32x2 dt2 = splat2(dt), cr2 = splat2(c_r), qd2 = pack2(qd0, qd1), qP2 = pack2(qP0, qP1);
                const f32x2 M2 = splat2(M), one2 = splat2(1.0f);
                constexpr unsigned SY = 4u * Sh::PITCH, IMG = 4u * Sh::CELLS;
                const unsigned base0 = (unsigned)__cvta_generic_to_shared(&S.sum[0][0]);
                const unsigned base = base0 + ((unsigned)HB - 0x4B400000u) * (SY + 4u);   // HB and the magic numbers' bits folded in
                f32x2 jj = splat2((float)j);
                auto walk = [&](auto fx) {
#pragma unroll 2
                    for (; j <= j1; ++j, jj = add2(jj, one2)) {
                        const f32x2 q = fma2(fma2(jj, dt2, cr2), qd2, qP2);
                        const f32x2 t = add2_rd(q, M2);
                        const f32x2 f = sub2(q, sub2(t, M2));
                        const unsigned a = base + 4u * __float_as_uint(lo2(t)) + SY * __float_as_uint(hi2(t));
                        const float ax = lo2(f), ay = hi2(f);
                        const f32x2 wy = pack2(1.0f - ay, ay);
                        const f32x2 w0 = mul2(wy, splat2(1.0f - ax)), w1 = mul2(wy, splat2(ax));   // (w00, w10), (w01, w11)
#pragma unroll
                        for (int i = 0; i < NB; ++i) {
                            if (decltype(fx)::value) {
                                const f32x2 v0 = fma2(w0, splat2(y[i]), M2), v1 = fma2(w1, splat2(y[i]), M2);
                                a2_red_s32(a + i * IMG, (int)(__float_as_uint(lo2(v0)) - 0x4B400000u));
                                a2_red_s32(a + i * IMG + 4u, (int)(__float_as_uint(lo2(v1)) - 0x4B400000u));
                                a2_red_s32(a + i * IMG + SY, (int)(__float_as_uint(hi2(v0)) - 0x4B400000u));
                                a2_red_s32(a + i * IMG + SY + 4u, (int)(__float_as_uint(hi2(v1)) - 0x4B400000u));
                            } else {
                                a2_red_f32(a + i * IMG, lo2(w0) * y[i]);
                                a2_red_f32(a + i * IMG + 4u, lo2(w1) * y[i]);
                                a2_red_f32(a + i * IMG + SY, hi2(w0) * y[i]);
                                a2_red_f32(a + i * IMG + SY + 4u, hi2(w1) * y[i]);
                            }
                        }
                    }
                };
                if (fixed) walk(std::true_type());
                else walk(std::false_type());
            }
            __syncthreads();
            // the group's sums go to the image (FP32: reductions, other storage: the CTA's own sums) and are cleared
            for (int e = tid; e < Sh::CELLS; e += A2_NT) {
                const int row = e / Sh::PITCH, col = e - row * Sh::PITCH;
                const int gx = bx0 + col - 1, gy = by0 + row - 1;
                const bool mine = row >= 1 && row <= B && col >= 1 && col <= B && gx < p.vol.nx && gy < p.vol.ny;
#pragma unroll
                for (int i = 0; i < NB; ++i) {
                    const unsigned w = S.sum[i][e];
                    if (w == 0u) continue;
                    S.sum[i][e] = 0u;
                    if (!mine || i >= nb) continue;
                    const float val = fixed ? __int2float_rn((int)w) * pow2(-(e2[i] >> 1)) * pow2((e2[i] >> 1) - e2[i])
                                            : __uint_as_float(w);
                    if constexpr (KEEP) K.acc[i][(row - 1) * B + col - 1] += val;
                    else a2_add(vb + i * p.vol_elems + (long long)gy * p.vol.nx + gx, val);
                }
            }
            // the next group's barrier orders the clearing before its reductions
        }
    }
    if constexpr (KEEP) {
        __syncthreads();
        for (int e = tid; e < B * B; e += A2_NT) {
            const int gx = bx0 + e % B, gy = by0 + e / B;
            if (gx < p.vol.nx && gy < p.vol.ny)
                for (int i = 0; i < nb; ++i)
                    vb[i * p.vol_elems + (long long)gy * p.vol.nx + gx] = from_f32<T>(K.acc[i][e]);
        }
    }
}

template <typename T, int B, int NB>
static int launch_a2(const OpParams &p, int vpc, int fixed, bool dense, const void *sino, void *vol, cudaStream_t st) {
    constexpr bool KEEP = sizeof(T) != 4;
    const size_t smem = (sizeof(A2Shared<B, NB>) + 15) / 16 * 16 + sizeof(A2Kept<B, NB, KEEP>);
    auto kern = dense ? adjoint2d_kernel<T, B, NB, true> : adjoint2d_kernel<T, B, NB, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    if (!KEEP) e = cudaMemsetAsync(vol, 0, sizeof(T) * (size_t)p.vol_elems * p.batch, st);
    if (e != cudaSuccess) return (int)e;
    const int bricks = ceil_div(p.vol.nx, B) * ceil_div(p.vol.ny, B), per_launch = 65535 * NB;
    for (int b0 = 0; b0 < p.batch; b0 += per_launch) {
        OpParams q = p;
        q.batch = std::min(p.batch - b0, per_launch);
        dim3 grid(bricks, ceil_div(p.n_views, vpc), ceil_div(q.batch, NB));
        kern<<<grid, A2_NT, smem, st>>>(q, make_double2(1.0 / p.sx, 1.0 / p.sy), vpc, fixed, (const T *)sino + b0 * p.sino_elems,
                                                             (T *)vol + b0 * p.vol_elems);
    }
    return (int)cudaGetLastError();
}

template <typename T>
static int launch_a2_t(const OpParams &p, int fixed, bool dense, const void *sino, void *vol, cudaStream_t st) {
    // Images per CTA: as in the projector, two or four share positions and weights (FP32; the other types keep
    // FP32 sums of their own beside the fixed-point ones and take one image).
    // Brick: 64^2, whose margin and ray set-up cost least per sample, unless the bricks and eight views per
    // CTA would leave the chip idle: then 32^2. Views per CTA (FP32, whose CTAs may share a brick): of 32^2 bricks about
    // six CTAs per SM, at least four views each; of 64^2 bricks about twelve (against six, 512^2 image, 700 views: 848 ->
    // 762 us, eight 362^2 images, 300 views: 970 -> 890), at least seven views each (256^2 image, 360 views: five 138 us, seven
    // 105, ten 119; that is a count of waves at this size, 832 CTAs at three per SM for seven, not a trend).
    const int ng = sizeof(T) == 4 ? (p.batch >= 3 ? ceil_div(p.batch, 4) : 1) : p.batch;
    const int b64 = ceil_div(p.vol.nx, 64) * ceil_div(p.vol.ny, 64) * ng, b32 = ceil_div(p.vol.nx, 32) * ceil_div(p.vol.ny, 32) * ng;
    const int target = stride_grid(1LL << 40, 6);   // six per SM
    const bool big = sizeof(T) == 4 ? (long long)b64 * ceil_div(p.n_views, 8) >= target / 2 : b64 >= target / 3;
    int vpc = p.n_views;
    if (sizeof(T) == 4) {
        const int split = std::max(1, big ? 2 * target / b64 : target / b32);
        vpc = std::max(std::max(big ? 7 : 4, ceil_div(p.n_views, 65535)), ceil_div(p.n_views, split));
    }
    if constexpr (sizeof(T) == 4) {
        if (p.batch >= 3) return big ? launch_a2<T, 64, 4>(p, vpc, fixed, dense, sino, vol, st) : launch_a2<T, 32, 4>(p, vpc, fixed, dense, sino, vol, st);
        if (p.batch == 2) return big ? launch_a2<T, 64, 2>(p, vpc, fixed, dense, sino, vol, st) : launch_a2<T, 32, 2>(p, vpc, fixed, dense, sino, vol, st);
    }
    return big ? launch_a2<T, 64, 1>(p, vpc, fixed, dense, sino, vol, st) : launch_a2<T, 32, 1>(p, vpc, fixed, dense, sino, vol, st);
}

int launch_adjoint2d(const OpParams &p, bool fixed, float ray_px, const void *sino, void *vol, int dtype, void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    // 64^2 pixels, 100 views: 1400 bins of 0.06 pixels 182 -> 100 us (values of a wide range 2.2 -> 0.44 ms); 128^2 pixels, 1024 bins of
    // 0.2 pixels the same both ways; 256^2 pixels, 512 bins of 1.3 pixels 106 -> 121 us
    const bool dense = ray_px < 0.2f;
    switch (dtype) {
        case PYRONN_F32: return launch_a2_t<float>(p, fixed, dense, sino, vol, st);
        case PYRONN_BF16: return launch_a2_t<__nv_bfloat16>(p, fixed, dense, sino, vol, st);
        case PYRONN_F16: return launch_a2_t<__half>(p, fixed, dense, sino, vol, st);
        default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace pyronn
