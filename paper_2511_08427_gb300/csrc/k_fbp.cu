// Filtered back-projection filter (Sec. 2.2: x = A^T F^T K F p; Listing 1's ramp filter and FDK
// weights): divergent-beam cosine pre-weighting, a ramp filter along detector rows and the scale that
// makes the 1/w^2-weighted (divergent) or plain (parallel) voxel-driven BP of the output the
// reconstruction. Same operator as the oracle's or_fbp_filter.
//
// The ramp is applied as a direct convolution with its taps (Ram-Lak or Shepp-Logan, unit spacing), which
// keeps each output's rounding relative to its neighbourhood: an FP32 FFT of the row measured four to six times
// the error, because a smooth row's transform is a hundred times its filtered values. It is organised like a matrix product
// with the Toeplitz tap matrix: a CTA filters 8 rows, staged in shared memory column-major, so that the rows of a
// column are 16-byte loads, and a thread accumulates 32 sums of several rows and outputs.
//
// fbp_odd_kernel (Ram-Lak): the taps of even offset are zero but for the central one, so the even outputs need the
// odd columns only and the odd outputs the even ones, half the products. A thread takes 4 rows x 8 outputs of one
// parity; per column it loads one tap (the other seven slide along) and one 16-byte word for 32 FMAs. Taps are stored by
// offset modulo 8, so the lanes, eight outputs apart, read consecutive words. FMAs are scalar: packed ones want
// every tap twice in a register pair, and the moves cost more than they save (271 against 214 us for 60 views of
// 512^2; one row and 16 outputs per thread, rows along the lanes: 253 us; 8 rows and 4 outputs: 246 us). The taps
// nearest the centre are left out of the loop over columns and added afterwards in column order with the central one
// between them: the partial sums stay at the size of the far taps' sums instead of the central product's, and so
// does their rounding (with the central product added last it measured five times the error). Rows of
// any views share a CTA, so detectors of one row fill it.
// Bound by the register file's operand bandwidth beside the FP32 pipe (FMA pipe 55 %, dispatch stalls), 360 views of
// 400 x 600, FP32: 2.44 -> 1.41 ms; 720 views of 1024^2: 30.8 -> 16.6 ms.
//
// fbp_full_kernel (Shepp-Logan, whose taps are all nonzero): 8 rows x 4 consecutive outputs per thread; the kernel
// above with all columns measured the same to 6 % slower.
#include "device_common.cuh"

namespace pyronn {

constexpr int FBP_ROWS = 8, FBP_OUT = 8;   // rows of a CTA; outputs of a thread
constexpr int FBP_FULL_OUT = 4;
constexpr int FBP_NEAR = 8;                // offsets below this are added after the loop over columns

__device__ __forceinline__ float ramp_tap_f(int k, int filter) {
    const float ipi2 = 0.10132118364233778f;   // 1 / pi^2
    if (filter == 1) return -2.0f * ipi2 / (4.0f * (float)k * (float)k - 1.0f);
    if (k == 0) return 0.25f;
    if ((k & 1) == 0) return 0.0f;
    return -ipi2 / ((float)k * (float)k);
}

// Shared-memory layout, in floats, and threads of a row length
struct FbpLayout {
    int half;      // columns of one parity, rounded up to 8
    int rows;      // staged rows: FBP_NEAR zero columns, 2 half columns (zero beyond Nu), FBP_NEAR zero columns
    int stride;    // taps of one residue (offset modulo 8)
    int blocks;    // threads of one parity and row group
};

static __host__ __device__ inline FbpLayout fbp_layout(int nu) {
    FbpLayout l;
    l.half = ((nu + 1) / 2 + 7) & ~7;
    l.rows = (2 * l.half + 2 * FBP_NEAR) * FBP_ROWS;
    l.stride = 2 * (l.half / 8) + 1;
    l.blocks = l.half / FBP_OUT;
    return l;
}

struct FbpAcc {
    float a[FBP_OUT][4];   // four rows
    // a[k] += w c for the rows of one column
    __device__ __forceinline__ void add(int k, float w, const float4 &c) {
        a[k][0] = fmaf(w, c.x, a[k][0]);
        a[k][1] = fmaf(w, c.y, a[k][1]);
        a[k][2] = fmaf(w, c.z, a[k][2]);
        a[k][3] = fmaf(w, c.w, a[k][3]);
    }
};

__device__ __forceinline__ float4 fbp_col(const float *c) { return *reinterpret_cast<const float4 *>(c); }

// acc[k] += sum over columns j of one parity of tap(i0 + k - j) x[2 j + parity]; t: the table's word for
// offset i0, residue 0
__device__ __forceinline__ void fbp_accumulate(const float *t, int stride, const float *cols, int half, FbpAcc &acc) {
    float w[FBP_OUT];
#pragma unroll
    for (int k = 0; k < FBP_OUT; ++k) w[k] = t[k * stride];
    for (int j = 0; j < half; j += 8, cols += 16 * FBP_ROWS) {
        --t;   // offsets i0 - j - 8 .. i0 - j - 1
        float n[FBP_OUT];
#pragma unroll
        for (int k = 0; k < FBP_OUT; ++k) n[k] = t[k * stride];
#pragma unroll
        for (int s = 0; s < 8; ++s) {   // column j + s: taps of offsets i0 - j - s + k
            const float4 c = fbp_col(cols + 2 * s * FBP_ROWS);
#pragma unroll
            for (int k = 0; k < FBP_OUT; ++k) acc.add(k, k >= s ? w[k - s] : n[8 + k - s], c);
        }
#pragma unroll
        for (int k = 0; k < FBP_OUT; ++k) w[k] = n[k];
    }
}

// grid: ceil(rows / per_cta) over all rows of the batch (per_cta at most 8). Dynamic shared memory: the staged rows, then the tap tables of
// offsets 2 n - 1 (even outputs) and 2 n + 1 (odd outputs). NT: most threads of a CTA.
template <typename T, int NT>
__global__ void __launch_bounds__(NT) fbp_odd_kernel(OpParams p, const FbpRec *__restrict__ rec, long long n_rows,
                                                     int per_cta, const T *__restrict__ in, T *__restrict__ out) {
    constexpr int filter = PYRONN_FILTER_RAM_LAK;
    extern __shared__ __align__(16) float fsm[];
    __shared__ float4 s_cos[FBP_ROWS];   // |source - pixel|^2 = x + y (m - z)^2 along the row, w = sdd (0: no weight)
    __shared__ float s_scale[FBP_ROWS];
    __shared__ int s_odd_values;
    const int Nu = p.det.nu;
    const FbpLayout L = fbp_layout(Nu);
    float *rows = fsm + FBP_NEAR * FBP_ROWS;   // rows[m * 8 + r], m from -FBP_NEAR
    float *taps = fsm + L.rows;                // table q, tap n: taps[q * 8 stride + (k & 7) * stride + (k >> 3)], k = n + half
    const int tid = threadIdx.x;
    const long long row0 = (long long)blockIdx.x * per_cta;
    const int nr = (int)min((long long)per_cta, n_rows - row0);
    if (tid == 0) s_odd_values = 0;
    if (tid < nr) {
        const long long id = row0 + tid;
        const FbpRec &R = rec[id / p.det.nv % p.n_views];
        const float v = (float)(id % p.det.nv);
        // from the row's point nearest the source, both terms positive: from its end they cancel on wide fans (1500 pixels
        // of 3.1 mm at 410 mm: weights off by 7e-7 rms, 1e-7 this way)
        float d[3], b = 0.0f, c = 0.0f, near2 = 0.0f;
        for (int i = 0; i < 3; ++i) {
            d[i] = fmaf(v, R.bv[i], R.b0[i]);
            b = fmaf(d[i], R.bu[i], b);
            c = fmaf(R.bu[i], R.bu[i], c);
        }
        const float m0 = c > 0.0f ? -b / c : 0.0f;
        for (int i = 0; i < 3; ++i) {
            const float e = fmaf(m0, R.bu[i], d[i]);
            near2 = fmaf(e, e, near2);
        }
        s_cos[tid] = make_float4(near2, c, m0, R.sdd);
        s_scale[tid] = R.scale;
    }
    for (int e = tid; e < 2 * 8 * L.stride; e += blockDim.x) {
        const int q = e / (8 * L.stride), k = e - q * 8 * L.stride, n = 8 * (k % L.stride) + k / L.stride - L.half;
        const int d = 2 * n + 2 * q - 1;
        taps[e] = d > -FBP_NEAR && d < FBP_NEAR ? 0.0f : ramp_tap_f(d, filter);
    }
    __syncthreads();
    // a value that is not finite, times the zero taps, makes NaN of the whole row: such rows take every tap
    int odd_values = 0;
    const T *src = in + row0 * Nu;
    for (int m = tid - FBP_NEAR; m < 2 * L.half + FBP_NEAR; m += blockDim.x) {
        const bool inside = m >= 0 && m < Nu;
        const float fm = (float)m;
        float val[FBP_ROWS];
#pragma unroll
        for (int r = 0; r < FBP_ROWS; ++r) val[r] = inside && r < nr ? to_f32<T>(src[(long long)r * Nu + m]) : 0.0f;
#pragma unroll
        for (int r = 0; r < FBP_ROWS; ++r)
            if (inside && r < nr) {
                const float4 c = s_cos[r];
                const float t = fm - c.z;
                if (c.w > 0.0f) val[r] *= c.w * rsqrtf(fmaf(c.y * t, t, c.x));   // cosine of the pixel's ray
                if (!(fabsf(val[r]) < __int_as_float(0x7f800000))) odd_values = 1;
            }
        float4 *to = reinterpret_cast<float4 *>(rows + m * FBP_ROWS);
        to[0] = make_float4(val[0], val[1], val[2], val[3]);
        to[1] = make_float4(val[4], val[5], val[6], val[7]);
    }
    if (odd_values) s_odd_values = 1;
    __syncthreads();
    // threads: parity of the outputs, group of four rows, eight outputs u = 2 (i0 + k) + q
    const int part = tid / L.blocks, q = part >> 1, group = part & 1, i0 = (tid - part * L.blocks) * FBP_OUT;
    const bool work = part < 4;
    FbpAcc acc;
    if (work) {
        const float *mine = rows + 4 * group;
#pragma unroll
        for (int k = 0; k < FBP_OUT; ++k) acc.a[k][0] = acc.a[k][1] = acc.a[k][2] = acc.a[k][3] = 0.0f;
        const int at = (i0 + L.half) >> 3;
        fbp_accumulate(taps + q * 8 * L.stride + at, L.stride, mine + (1 - q) * FBP_ROWS, L.half, acc);
        // the near taps, column by column: c = u - offset
        const float *u0 = mine + (2 * i0 + q) * FBP_ROWS;
#pragma unroll
        for (int c = 1 - FBP_NEAR; c < 2 * FBP_OUT - 2 + FBP_NEAR; ++c) {
            const bool own = (c & 1) == 0;   // the outputs' parity
            if (own && (c < 0 || c > 2 * FBP_OUT - 2)) continue;
            const float4 x = fbp_col(u0 + c * FBP_ROWS);
#pragma unroll
            for (int k = 0; k < FBP_OUT; ++k) {
                const int d = 2 * k - c;
                if (d <= -FBP_NEAR || d >= FBP_NEAR || (own && d != 0)) continue;
                acc.add(k, ramp_tap_f(d, filter), x);
            }
        }
        if (s_odd_values)
            for (int j = q; j < 2 * L.half; j += 2) {
                const float4 x = fbp_col(mine + j * FBP_ROWS);
#pragma unroll
                for (int k = 0; k < FBP_OUT; ++k)
                    if (j != 2 * (i0 + k) + q) acc.add(k, 0.0f, x);
            }
    }
    __syncthreads();   // every thread is done with the staged rows: they take the results, for row-wise stores
    if (work)
#pragma unroll
        for (int k = 0; k < FBP_OUT; ++k)
            *reinterpret_cast<float4 *>(rows + (2 * (i0 + k) + q) * FBP_ROWS + 4 * group) =
                make_float4(acc.a[k][0], acc.a[k][1], acc.a[k][2], acc.a[k][3]);
    __syncthreads();
    T *dst = out + row0 * Nu;
    for (int m = tid; m < Nu; m += blockDim.x) {
        const float4 lo = fbp_col(rows + m * FBP_ROWS), hi = fbp_col(rows + m * FBP_ROWS + 4);
        const float val[FBP_ROWS] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
        for (int r = 0; r < FBP_ROWS; ++r)
            if (r < nr) dst[(long long)r * Nu + m] = from_f32<T>(s_scale[r] * val[r]);
    }
}

template <typename T>
static int launch_odd_t(const OpParams &p, const FbpRec *rec, const void *in, void *out, cudaStream_t st) {
    const FbpLayout L = fbp_layout(p.det.nu);
    const int threads = (4 * L.blocks + 31) & ~31;
    const size_t smem = sizeof(float) * ((size_t)L.rows + 2 * 8 * (size_t)L.stride);
    auto kern = threads <= 512 ? fbp_odd_kernel<T, 512> : fbp_odd_kernel<T, 1024>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    const long long n_rows = (long long)p.batch * p.n_views * p.det.nv;
    int per = FBP_ROWS;   // fewer rows per CTA where eight would leave SMs idle (180 rows of 183: 9.3 -> 8.9 us)
    while (per > 1 && (n_rows + per - 1) / per < stride_grid(1LL << 40, 1)) per >>= 1;
    const long long ctas = (n_rows + per - 1) / per;
    if (ctas > 0x7fffffffLL) return (int)cudaErrorInvalidValue;   // more rows than any device's memory holds
    kern<<<(unsigned)ctas, threads, smem, st>>>(p, rec, n_rows, per, (const T *)in, (T *)out);
    return (int)cudaGetLastError();
}

// grid: (ceil(Nv / 8), V * batch); block: ceil(Nu / 4) threads rounded up to a warp; dynamic shared
// memory: 8 Nu (rows, column-major) + 2 Nu + 4 (taps h(-Nu .. Nu + 3)) floats.
template <typename T>
__global__ void fbp_full_kernel(OpParams p, const FbpRec *__restrict__ rec, int filter, const T *__restrict__ in,
                                  T *__restrict__ out) {
    extern __shared__ __align__(16) float fsm[];
    const int Nu = p.det.nu, Nv = p.det.nv;
    float *rows = fsm;                       // rows[m * 8 + r]
    float *taps = fsm + FBP_ROWS * Nu;       // taps[k + Nu] = h(k), k in [-Nu, Nu + 4)
    const int view = blockIdx.y % p.n_views, b = blockIdx.y / p.n_views;
    const int v0 = blockIdx.x * FBP_ROWS;
    const FbpRec R = rec[view];
    const long long base = (long long)b * p.sino_elems + (long long)view * Nv * Nu;
    for (int k = threadIdx.x; k < 2 * Nu + 4; k += blockDim.x) taps[k] = ramp_tap_f(k - Nu, filter);
    for (int e = threadIdx.x; e < FBP_ROWS * Nu; e += blockDim.x) {
        const int r = e / Nu, m = e - r * Nu, v = v0 + r;
        float val = 0.0f;
        if (v < Nv) {
            val = to_f32<T>(in[base + (long long)v * Nu + m]);
            if (R.sdd > 0.0f) {   // divergent beam: cosine of the pixel's ray
                const float dx = fmaf((float)v, R.bv[0], fmaf((float)m, R.bu[0], R.b0[0]));
                const float dy = fmaf((float)v, R.bv[1], fmaf((float)m, R.bu[1], R.b0[1]));
                const float dz = fmaf((float)v, R.bv[2], fmaf((float)m, R.bu[2], R.b0[2]));
                val *= R.sdd * rsqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
            }
        }
        rows[m * FBP_ROWS + r] = val;
    }
    __syncthreads();
    const int u0 = threadIdx.x * FBP_FULL_OUT;
    float acc[FBP_ROWS][FBP_FULL_OUT];
#pragma unroll
    for (int r = 0; r < FBP_ROWS; ++r)
#pragma unroll
        for (int j = 0; j < FBP_FULL_OUT; ++j) acc[r][j] = 0.0f;
    // outputs u0 + j need h(u0 + j - m): at column m the window is h(u0 - m .. u0 + 3 - m); moving to
    // m + 1 shifts it by one tap. For u0 < Nu every index lies in [-Nu, Nu + 3).
    if (u0 < Nu) {
        float t0 = taps[u0 + Nu], t1 = taps[u0 + 1 + Nu], t2 = taps[u0 + 2 + Nu], t3 = taps[u0 + 3 + Nu];
        for (int m = 0; m < Nu; ++m) {
            const float4 a = *reinterpret_cast<const float4 *>(rows + m * FBP_ROWS);
            const float4 c = *reinterpret_cast<const float4 *>(rows + m * FBP_ROWS + 4);
            const float rv[FBP_ROWS] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w};
#pragma unroll
            for (int r = 0; r < FBP_ROWS; ++r) {
                acc[r][0] = fmaf(t0, rv[r], acc[r][0]);
                acc[r][1] = fmaf(t1, rv[r], acc[r][1]);
                acc[r][2] = fmaf(t2, rv[r], acc[r][2]);
                acc[r][3] = fmaf(t3, rv[r], acc[r][3]);
            }
            t3 = t2;
            t2 = t1;
            t1 = t0;
            t0 = taps[u0 - (m + 1) + Nu];
        }
#pragma unroll
        for (int r = 0; r < FBP_ROWS; ++r) {
            const int v = v0 + r;
            if (v >= Nv) continue;
#pragma unroll
            for (int j = 0; j < FBP_FULL_OUT; ++j)
                if (u0 + j < Nu) out[base + (long long)v * Nu + u0 + j] = from_f32<T>(R.scale * acc[r][j]);
        }
    }
}

template <typename T>
static int launch_full_t(const OpParams &p, const FbpRec *rec, int filter, const void *in, void *out, cudaStream_t st) {
    const int nu = p.det.nu;
    int threads = (nu + FBP_FULL_OUT - 1) / FBP_FULL_OUT;
    threads = ((threads + 31) / 32) * 32;
    const size_t smem = sizeof(float) * (size_t)(FBP_ROWS * nu + 2 * nu + 4);
    cudaError_t e = cudaFuncSetAttribute(fbp_full_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    const int per_launch = 65535 / p.n_views > 0 ? 65535 / p.n_views : 1;
    for (int b0 = 0; b0 < p.batch; b0 += per_launch) {
        const int nb = p.batch - b0 < per_launch ? p.batch - b0 : per_launch;
        dim3 grid(ceil_div(p.det.nv, FBP_ROWS), p.n_views * nb);
        fbp_full_kernel<T><<<grid, threads, smem, st>>>(p, rec, filter, (const T *)in + b0 * p.sino_elems,
                                                          (T *)out + b0 * p.sino_elems);
    }
    return (int)cudaGetLastError();
}

template <typename T>
static int launch_fbp_t(const OpParams &p, const FbpRec *rec, int filter, const void *in, void *out, cudaStream_t st) {
    // rows of less than 32 pixels: half the products are not worth the parts (20 pixels: 6 us against 4)
    return filter == PYRONN_FILTER_RAM_LAK && p.det.nu >= 32 ? launch_odd_t<T>(p, rec, in, out, st) : launch_full_t<T>(p, rec, filter, in, out, st);
}

int launch_fbp_filter(const OpParams &p, const FbpRec *rec, int filter, const void *in, void *out, int dtype,
                      void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    switch (dtype) {
        case PYRONN_F32: return launch_fbp_t<float>(p, rec, filter, in, out, st);
        case PYRONN_BF16: return launch_fbp_t<__nv_bfloat16>(p, rec, filter, in, out, st);
        case PYRONN_F16: return launch_fbp_t<__half>(p, rec, filter, in, out, st);
        default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace pyronn
