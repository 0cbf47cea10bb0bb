// k_pyramid.cu -- coarse-to-fine machinery (Sec. 4: "standard coarse-to-fine framework ...
// multiscale pyramid" with warping; the paper gives no details, the readings are stated at
// each kernel): Gaussian pre-smoothing + resampling, level transfer of the fields, derivative
// images, warping + linearisation with the per-warp max of M_s, and precision conversion.
#include <math.h>

#include <algorithm>

#include "tvl1_device.cuh"

namespace tvl1 {

namespace {

constexpr int B2X = 32, B2Y = 8;

__device__ __forceinline__ int reflect_index(int k, int n) {
    // half-sample symmetric extension for any integer k: period 2n, mirrored halves
    const int period = 2 * n;
    int m = k % period;
    if (m < 0) m += period;
    return m < n ? m : period - 1 - m;
}

__device__ __forceinline__ float clampf(float x, float lo, float hi) { return fminf(fmaxf(x, lo), hi); }

// Bilinear value of plane f (H x W, pitch P) at (x, y) inside [0, W-1] x [0, H-1].
template <typename T>
__device__ __forceinline__ float bilinear(const T *f, int H, int W, int P, float x, float y) {
    const float xf = floorf(x), yf = floorf(y);
    const int x0 = (int)xf, y0 = (int)yf;
    const float fx = x - xf, fy = y - yf;
    const int x1 = min(x0 + 1, W - 1), y1 = min(y0 + 1, H - 1);
    const float a = Store<T>::ld(f + (size_t)y0 * P + x0), b = Store<T>::ld(f + (size_t)y0 * P + x1);
    const float c = Store<T>::ld(f + (size_t)y1 * P + x0), d = Store<T>::ld(f + (size_t)y1 * P + x1);
    const float top = (1.f - fx) * a + fx * b;
    const float bot = (1.f - fx) * c + fx * d;
    return (1.f - fy) * top + fy * bot;
}

// Sample position j + d clamped to [0, n-1], as integer part and fraction, in FP64: j + d and
// its fraction are exact there for any FP32 displacement d.
__device__ __forceinline__ void split_pos_f64(int j, float d, int n, int &x0, double &fx) {
    const double xs = (double)j + (double)d;
    if (!(xs > 0.0)) {              // also catches NaN
        x0 = 0;
        fx = 0.0;
    } else if (xs >= (double)(n - 1)) {
        x0 = n - 1;
        fx = 0.0;
    } else {
        const double fl = floor(xs);
        x0 = (int)fl;
        fx = xs - fl;
    }
}

// Bilinear value of an FP32 plane (H x W, pitch P) at (x0 + fx, y0 + fy) in FP64 arithmetic (the
// four samples are exact in FP64).
__device__ __forceinline__ double bilinear_split_f64(const float *f, int H, int W, int P, int x0, double fx, int y0,
                                                     double fy) {
    const int x1 = min(x0 + 1, W - 1), y1 = min(y0 + 1, H - 1);
    const double a = __ldg(f + (size_t)y0 * P + x0), b = __ldg(f + (size_t)y0 * P + x1);
    const double c = __ldg(f + (size_t)y1 * P + x0), d = __ldg(f + (size_t)y1 * P + x1);
    const double top = (1.0 - fx) * a + fx * b;
    const double bot = (1.0 - fx) * c + fx * d;
    return (1.0 - fy) * top + fy * bot;
}

// Separable Gaussian, first along rows (x), then along columns (y); half-sample symmetric border.
__global__ void k_blur_rows(const float *__restrict__ in, float *__restrict__ out, Geom g, GaussTaps t) {
    const int j = blockIdx.x * B2X + threadIdx.x, i = blockIdx.y * B2Y + threadIdx.y;
    if (i >= g.H || j >= g.W) return;
    const float *row = in + (size_t)i * g.pitch;
    float acc = 0.f;
    for (int k = -t.R; k <= t.R; ++k) acc += t.w[k + t.R] * __ldg(row + reflect_index(j + k, g.W));
    out[(size_t)i * g.pitch + j] = acc;
}

__global__ void k_blur_cols(const float *__restrict__ in, float *__restrict__ out, Geom g, GaussTaps t) {
    const int j = blockIdx.x * B2X + threadIdx.x, i = blockIdx.y * B2Y + threadIdx.y;
    if (i >= g.H || j >= g.W) return;
    float acc = 0.f;
    for (int k = -t.R; k <= t.R; ++k) acc += t.w[k + t.R] * __ldg(in + (size_t)reflect_index(i + k, g.H) * g.pitch + j);
    out[(size_t)i * g.pitch + j] = acc;
}

// Coarse pixel centre (j + 0.5) maps to fine x = (j + 0.5) * Wf / Wc - 0.5, clamped.
__global__ void k_resample(const float *__restrict__ fine, Geom gf, float *__restrict__ coarse, Geom gc) {
    const int j = blockIdx.x * B2X + threadIdx.x, i = blockIdx.y * B2Y + threadIdx.y;
    if (i >= gc.H || j >= gc.W) return;
    const float sx = (float)gf.W / (float)gc.W, sy = (float)gf.H / (float)gc.H;
    const float x = clampf((j + 0.5f) * sx - 0.5f, 0.f, (float)(gf.W - 1));
    const float y = clampf((i + 0.5f) * sy - 0.5f, 0.f, (float)(gf.H - 1));
    coarse[(size_t)i * gc.pitch + j] = bilinear<float>(fine, gf.H, gf.W, gf.pitch, x, y);
}

// Level transfer: fine pixel centre maps to coarse x = (j + 0.5) * Wc / Wf - 0.5, clamped.
template <typename T>
__global__ void k_upsample(const T *__restrict__ coarse, Geom gc, T *__restrict__ fine, Geom gf, float scale) {
    const int j = blockIdx.x * B2X + threadIdx.x, i = blockIdx.y * B2Y + threadIdx.y;
    if (i >= gf.H || j >= gf.W) return;
    const float sx = (float)gc.W / (float)gf.W, sy = (float)gc.H / (float)gf.H;
    const float x = clampf((j + 0.5f) * sx - 0.5f, 0.f, (float)(gc.W - 1));
    const float y = clampf((i + 0.5f) * sy - 0.5f, 0.f, (float)(gc.H - 1));
    Store<T>::st(fine + (size_t)i * gf.pitch + j, scale * bilinear<T>(coarse, gc.H, gc.W, gc.pitch, x, y));
}

// Central differences with clamped neighbour indices.
__global__ void k_derivatives(const float *__restrict__ I, Geom g, float *__restrict__ Ix, float *__restrict__ Iy) {
    const int j = blockIdx.x * B2X + threadIdx.x, i = blockIdx.y * B2Y + threadIdx.y;
    if (i >= g.H || j >= g.W) return;
    const int jl = max(j - 1, 0), jr = min(j + 1, g.W - 1), iu = max(i - 1, 0), id = min(i + 1, g.H - 1);
    const size_t o = (size_t)i * g.pitch + j;
    Ix[o] = 0.5f * (__ldg(I + (size_t)i * g.pitch + jr) - __ldg(I + (size_t)i * g.pitch + jl));
    Iy[o] = 0.5f * (__ldg(I + (size_t)id * g.pitch + j) - __ldg(I + (size_t)iu * g.pitch + j));
}

// ---- twofold FP32: a value as an unevaluated sum h + l of two FP32 numbers (about 48 bits), from the
// error-free transformations of sums (Knuth's TwoSum) and products (by FMA).  The warping needs more
// than FP32 (see k_warp) and FP64 runs at 1/64 of the FP32 rate here.
struct F2 {
    float h, l;
};
// a - b exactly
__device__ __forceinline__ F2 two_diff(float a, float b) {
    const float s = __fsub_rn(a, b), t = __fsub_rn(s, a);
    return {s, __fsub_rn(__fsub_rn(a, __fsub_rn(s, t)), __fadd_rn(b, t))};
}
// a + b exactly
__device__ __forceinline__ F2 two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
// h + l with l at most half an ulp of h
__device__ __forceinline__ F2 renorm(float h, float l) {
    const float s = __fadd_rn(h, l);
    return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
// p + w (q - p)
__device__ __forceinline__ F2 lerp2(F2 p, F2 q, float w) {
    const F2 d = two_diff(q.h, p.h);
    const float e = __fadd_rn(d.l, __fsub_rn(q.l, p.l)), m = __fmul_rn(w, d.h);
    const float ml = __fmaf_rn(w, e, __fmaf_rn(w, d.h, -m));
    const F2 s = two_sum(p.h, m);
    return {s.h, __fadd_rn(s.l, __fadd_rn(p.l, ml))};
}
// acc - g u, acc and g twofold
__device__ __forceinline__ F2 sub_mul(F2 acc, F2 g, float u) {
    const float m = __fmul_rn(g.h, u), ml = __fmaf_rn(g.l, u, __fmaf_rn(g.h, u, -m));
    const F2 d = two_diff(acc.h, m);
    return {d.h, __fadd_rn(d.l, __fsub_rn(acc.l, ml))};
}
// Rounds v, known to within `err`, to FP32; false when the interval straddles two FP32 numbers (Ziv's
// rounding test), or when v is not finite.
__device__ __forceinline__ bool round_safe(F2 v, float err, float &out) {
    const F2 r = renorm(v.h, v.l);
    out = __fadd_rn(r.h, __fadd_rn(r.l, err));
    return out == __fadd_rn(r.h, __fsub_rn(r.l, err));
}

// The sample position j + d clamped to [0, n - 1] as a base index p, its neighbour q and the weight
// w of q, an exact FP32 number: for d >= 0 the base is the pixel below the position and w its
// fraction; for d < 0 the base is the pixel above and w the fraction of |d| (1 - fraction would
// need more than 24 bits).
__device__ __forceinline__ void split_pos(int j, float d, int n, int &p, int &q, float &w) {
    w = 0.f;
    if (!(d > (float)-j)) {  // at or below 0; also catches NaN
        p = 0;
    } else if (d >= (float)(n - 1 - j)) {
        p = n - 1;
    } else {
        const float t = truncf(d);  // towards zero
        w = fabsf(d - t);
        p = j + (int)t;
    }
    // inside the image, 0 < j + d < n - 1, the neighbour is too; weight 0: the one FP64 would read
    q = w != 0.f && d < 0.f ? p - 1 : min(p + 1, n - 1);
}

// Warp I1 and its derivatives to (x + u0, y + v0) (clamped), linearise around d0:
// It = I1w - I0 - Ix u0 - Iy v0, so that rho(w, d) = Ix u + Iy v + beta w + It.
// The block max of M_s = beta^2 + Ix^2 + Iy^2 (of the stored, rounded values) raises *ms_max.
// The results are those of the interpolation and It in FP64, rounded once when stored: It is a small
// difference of terms up to |grad I| |d0|, and the L1 data term puts the flow of weakly textured
// pixels on the line Ix u + Iy v + It = 0, so an FP32 It moved those pixels by up to a few 1e-3 px
// over a whole schedule (measured against the FP64 oracle).  FP64 bounded the kernel (33 operations
// of 64 cycles each per 32 pixels and SM quarter).  So the values are formed in twofold FP32, with an
// error of some 2^-45 of the terms' magnitude, and rounded when an error of 2^-41 cannot change the
// rounding; where it could (about one pixel in ten thousand, exact ties, non-finite values) the pixel
// takes the FP64 path, so that every result is the FP64 path's, bit for bit.  Measured at 1920x1080:
// 36 us against 233 all in FP64 (640x480 10 against 37).
template <typename T, typename TF> __global__ void k_warp(const __grid_constant__ PairSet A, int cur, float beta) {
    __shared__ float red[B2X * B2Y / 32];
    const PairIter &P = A.pairs ? A.pairs[blockIdx.z] : A.one;
    const Geom g = P.g;
    if (blockIdx.x * B2X >= g.W || blockIdx.y * B2Y >= g.H) return;  // beyond a smaller pair of the batch
    const float *__restrict__ I0 = P.I0, *__restrict__ I1 = P.I1, *__restrict__ I1x = P.I1x, *__restrict__ I1y = P.I1y;
    const TF *__restrict__ u0 = reinterpret_cast<const TF *>(P.buf[cur].f[F_U]);
    const TF *__restrict__ v0 = reinterpret_cast<const TF *>(P.buf[cur].f[F_V]);
    T *__restrict__ Ix = (T *)P.Ix, *__restrict__ Iy = (T *)P.Iy, *__restrict__ It = (T *)P.It;
    float *ms_max = const_cast<float *>(P.ms_max);
    const int j = blockIdx.x * B2X + threadIdx.x, i = blockIdx.y * B2Y + threadIdx.y;
    float ms = 0.f;
    if (i < g.H && j < g.W) {
        const size_t o = (size_t)i * g.pitch + j;
        const float uu = Store<TF>::ld(u0 + o), vv = Store<TF>::ld(v0 + o), i0 = __ldg(I0 + o);
        int xp, xq, yp, yq;
        float wx, wy;
        split_pos(j, uu, g.W, xp, xq, wx);
        split_pos(i, vv, g.H, yp, yq, wy);
        const size_t rp = (size_t)yp * g.pitch, rq = (size_t)yq * g.pitch;
        float mag;  // sum of the magnitudes of the last interpolation's samples
        auto sample = [&](const float *f) -> F2 {
            const float a = __ldg(f + rp + xp), b = __ldg(f + rp + xq), c = __ldg(f + rq + xp), d = __ldg(f + rq + xq);
            mag = fabsf(a) + fabsf(b) + (fabsf(c) + fabsf(d));
            return lerp2(lerp2(F2{a, 0.f}, F2{b, 0.f}, wx), lerp2(F2{c, 0.f}, F2{d, 0.f}, wx), wy);
        };
        constexpr float EPS = 0x1p-41f, TINY = 1e-36f;  // TINY: products that underflow
        auto bound = [&](float m) { return m > 0.f ? fmaf(m, EPS, TINY) : 0.f; };
        const F2 w1 = sample(I1);
        const float m1 = mag;
        const F2 gx = sample(I1x);
        const float mx = mag;
        const F2 gy = sample(I1y);
        const float my = mag;
        float ix, iy, it;
        F2 t = two_diff(w1.h, i0);
        t.l = __fadd_rn(t.l, w1.l);
        t = sub_mul(sub_mul(t, gx, uu), gy, vv);
        const float mt = m1 + fabsf(i0) + mx * fabsf(uu) + my * fabsf(vv);
        const bool okx = round_safe(gx, bound(mx), ix), oky = round_safe(gy, bound(my), iy);
        if (!(round_safe(t, bound(mt), it) && okx && oky)) {
            int x0, y0;
            double fx, fy;
            split_pos_f64(j, uu, g.W, x0, fx);
            split_pos_f64(i, vv, g.H, y0, fy);
            const double w1d = bilinear_split_f64(I1, g.H, g.W, g.pitch, x0, fx, y0, fy);
            const double gxd = bilinear_split_f64(I1x, g.H, g.W, g.pitch, x0, fx, y0, fy);
            const double gyd = bilinear_split_f64(I1y, g.H, g.W, g.pitch, x0, fx, y0, fy);
            ix = (float)gxd;
            iy = (float)gyd;
            it = (float)(w1d - (double)i0 - gxd * (double)uu - gyd * (double)vv);
        }
        Store<T>::st(Ix + o, ix);
        Store<T>::st(Iy + o, iy);
        Store<T>::st(It + o, it);
        const float gxr = storage_round<T>(ix), gyr = storage_round<T>(iy);
        ms = beta * beta + gxr * gxr + gyr * gyr;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ms = fmaxf(ms, __shfl_down_sync(0xffffffffu, ms, o));
    const int tid = threadIdx.y * B2X + threadIdx.x;
    if ((tid & 31) == 0) red[tid >> 5] = ms;
    __syncthreads();
    if (tid == 0) {
        float m = red[0];
        for (int k = 1; k < B2X * B2Y / 32; ++k) m = fmaxf(m, red[k]);
        // non-negative floats order like their bit patterns
        atomicMax(reinterpret_cast<unsigned int *>(ms_max), __float_as_uint(m));
    }
}

__global__ void k_warp_reset(const __grid_constant__ PairSet A) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= A.n) return;
    float *m = const_cast<float *>(A.pairs[k].ms_max);
    m[0] = 0.f;
    reinterpret_cast<int *>(m)[1] = 0;  // the stop flag
}

// Everything a level starts with, one pixel per thread: the planes were filled, upsampled and
// differentiated by up to 17 launches of a microsecond or two each, most of it launch and drain.
template <typename TD, typename TF> __global__ void k_level_begin(const __grid_constant__ LevelArgs A) {
    const PairIter &P = A.fine.pairs ? A.fine.pairs[blockIdx.z] : A.fine.one;
    const Geom g = P.g;
    const int j = blockIdx.x * B2X + threadIdx.x, i = blockIdx.y * B2Y + threadIdx.y;
    if (i >= g.H || j >= g.W) return;
    const size_t o = (size_t)i * g.pitch + j;
    const Fields &to = P.buf[A.to];
    float x[3] = {0.f, 0.f, 0.f};
    if (!A.first) {
        // fine pixel centre -> coarse x = (j + 0.5) * Wc / Wf - 0.5, clamped, as k_upsample
        const PairIter &C = A.coarse.pairs ? A.coarse.pairs[blockIdx.z] : A.coarse.one;
        const Geom gc = C.g;
        const float sx = (float)gc.W / (float)g.W, sy = (float)gc.H / (float)g.H;
        const float xc = clampf((j + 0.5f) * sx - 0.5f, 0.f, (float)(gc.W - 1));
        const float yc = clampf((i + 0.5f) * sy - 0.5f, 0.f, (float)(gc.H - 1));
        const float scale[3] = {1.f, (float)g.W / (float)gc.W, (float)g.H / (float)gc.H};
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (c > 0 || A.has_w)
                x[c] = scale[c] * bilinear<TF>(reinterpret_cast<const TF *>(C.buf[A.from].f[F_W + c]), gc.H, gc.W, gc.pitch, xc, yc);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        stT<TF>(to.f[F_W + c], o, x[c]);
        if (A.xbar) stT<TF>(to.f[F_WB + c], o, x[c]);
    }
    // the iterations leave w alone without beta: zero in whichever buffer they end
    if (!A.has_w) stT<TF>(P.buf[A.to ^ 1].f[F_W], o, 0.f);
#pragma unroll
    for (int k = F_P1; k <= F_S; ++k) stT<TD>(to.f[k], o, 0.f);
    const int jl = max(j - 1, 0), jr = min(j + 1, g.W - 1), iu = max(i - 1, 0), id = min(i + 1, g.H - 1);
    const float *__restrict__ I = P.I1;
    P.I1x[o] = 0.5f * (__ldg(I + (size_t)i * g.pitch + jr) - __ldg(I + (size_t)i * g.pitch + jl));
    P.I1y[o] = 0.5f * (__ldg(I + (size_t)id * g.pitch + j) - __ldg(I + (size_t)iu * g.pitch + j));
}

template <typename TD, typename TF>
__global__ void k_state_to_f32(const __grid_constant__ PairSet A, const __grid_constant__ PairSet B, int cur, int xbar, int has_w) {
    const PairIter &P = A.pairs ? A.pairs[blockIdx.z] : A.one, &Q = B.pairs ? B.pairs[blockIdx.z] : B.one;
    const Geom g = P.g;
    const int j = blockIdx.x * B2X + threadIdx.x, i = blockIdx.y * B2Y + threadIdx.y;
    if (i >= g.H || j >= g.W) return;
    const size_t o = (size_t)i * g.pitch + j;
    const Fields &f = P.buf[cur], &t = Q.buf[0];
#pragma unroll
    for (int k = 0; k < NFIELDS; ++k)
        if (xbar || k < F_WB) stT<float>(t.f[k], o, is_flow_field(k) ? ldT<TF>(f.f[k], o) : ldT<TD>(f.f[k], o));
    if (!has_w) stT<float>(Q.buf[1].f[F_W], o, 0.f);
}

template <typename TF> __global__ void k_output(Fields f, Geom g, float *u, float *v, float *w) {
    const int j = blockIdx.x * B2X + threadIdx.x, i = blockIdx.y * B2Y + threadIdx.y;
    if (i >= g.H || j >= g.W) return;
    const size_t o = (size_t)i * g.pitch + j;
    u[o] = ldT<TF>(f.f[F_U], o);
    v[o] = ldT<TF>(f.f[F_V], o);
    w[o] = ldT<TF>(f.f[F_W], o);
}

// One pyramid step in one launch: a block stages the fine pixels its coarse tile needs (with the
// blur's margin, mirrored at the border), blurs their rows in shared memory, and forms each coarse
// pixel from the column blurs at its four fine neighbours.  The sums run in the order of k_blur_rows,
// k_blur_cols and k_resample, so the results are theirs bit for bit; those pass two fine planes
// through memory and took 45 us at 1920x1080.
constexpr int PDX = 32, PDY = 16;
struct PyrArgs {
    const float *fine[2];
    float *coarse[2];
    Geom gf, gc;
    GaussTaps t;
    int nx, ny;  // fine columns and rows of a tile, at most
};
__global__ void __launch_bounds__(256) k_pyr_down(const __grid_constant__ PyrArgs A) {
    extern __shared__ float sm[];
    const int R = A.t.R, Hf = A.gf.H, Wf = A.gf.W, Hc = A.gc.H, Wc = A.gc.W;
    const float *__restrict__ in = A.fine[blockIdx.z];
    const float sx = (float)Wf / (float)Wc, sy = (float)Hf / (float)Hc;
    auto px = [&](int j) { return clampf((j + 0.5f) * sx - 0.5f, 0.f, (float)(Wf - 1)); };
    auto py = [&](int i) { return clampf((i + 0.5f) * sy - 0.5f, 0.f, (float)(Hf - 1)); };
    const int j0 = blockIdx.x * PDX, i0 = blockIdx.y * PDY;
    const int x0 = (int)floorf(px(j0)), y0 = (int)floorf(py(i0));
    const int x1 = min((int)floorf(px(min(j0 + PDX, Wc) - 1)) + 1, Wf - 1), y1 = min((int)floorf(py(min(i0 + PDY, Hc) - 1)) + 1, Hf - 1);
    const int nx = x1 - x0 + 1, ny = y1 - y0 + 1, aw = A.nx + 2 * R;
    float *a = sm, *b = sm + (A.ny + 2 * R) * aw;  // the fine pixels; their rows blurred (pitch A.nx)
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int r = ty; r < ny + 2 * R; r += 8) {
        const float *row = in + (size_t)reflect_index(y0 - R + r, Hf) * A.gf.pitch;
        for (int c = tx; c < nx + 2 * R; c += 32) a[r * aw + c] = __ldg(row + reflect_index(x0 - R + c, Wf));
    }
    __syncthreads();
    for (int r = ty; r < ny + 2 * R; r += 8)
        for (int c = tx; c < nx; c += 32) {
            float acc = 0.f;
            for (int k = 0; k <= 2 * R; ++k) acc += A.t.w[k] * a[r * aw + c + k];
            b[r * A.nx + c] = acc;
        }
    __syncthreads();
    const int j = j0 + tx;
    if (j >= Wc) return;
    const float x = px(j), xf = floorf(x), fx = x - xf;
    const int xa = (int)xf - x0, xb = min((int)xf + 1, Wf - 1) - x0;
    for (int i = i0 + ty; i < min(i0 + PDY, Hc); i += 8) {
        const float y = py(i), yf = floorf(y), fy = y - yf;
        const int ya = (int)yf - y0, yb = min((int)yf + 1, Hf - 1) - y0;
        auto blur = [&](int yy, int xx) {
            float acc = 0.f;
            for (int k = 0; k <= 2 * R; ++k) acc += A.t.w[k] * b[(yy + k) * A.nx + xx];
            return acc;
        };
        const float va = blur(ya, xa), vb = blur(ya, xb), vc = blur(yb, xa), vd = blur(yb, xb);
        const float top = (1.f - fx) * va + fx * vb;
        const float bot = (1.f - fx) * vc + fx * vd;
        A.coarse[blockIdx.z][(size_t)i * A.gc.pitch + j] = (1.f - fy) * top + fy * bot;
    }
}

dim3 grid2(int H, int W) { return dim3((W + B2X - 1) / B2X, (H + B2Y - 1) / B2Y); }

}  // namespace

GaussTaps gauss_taps(float eta) {
    GaussTaps t{};
    const double sg = 0.6 * sqrt(1.0 / ((double)eta * (double)eta) - 1.0);
    t.R = (int)ceil(3.0 * sg);
    if (t.R > MAX_GAUSS_R) {
        t.R = -1;
        return t;
    }
    double w[2 * MAX_GAUSS_R + 1], sum = 0.0;
    for (int k = -t.R; k <= t.R; ++k) {
        w[k + t.R] = sg > 0.0 ? exp(-(double)(k * k) / (2.0 * sg * sg)) : 1.0;
        sum += w[k + t.R];
    }
    for (int k = 0; k <= 2 * t.R; ++k) t.w[k] = (float)(w[k] / sum);
    return t;
}

void launch_pyr_down(const float *const *fine, Geom gf, float *const *coarse, Geom gc, int n, const GaussTaps &taps,
                     float *scratch, cudaStream_t s) {
    PyrArgs a{};
    a.gf = gf;
    a.gc = gc;
    a.t = taps;
    // fine pixels between the first and the last coarse centre of a tile, and the neighbours
    a.nx = std::min(gf.W, (int)ceilf((PDX - 1) * ((float)gf.W / (float)gc.W)) + 3);
    a.ny = std::min(gf.H, (int)ceilf((PDY - 1) * ((float)gf.H / (float)gc.H)) + 3);
    const size_t rows = (size_t)a.ny + 2 * taps.R, smem = rows * (2 * (size_t)a.nx + 2 * taps.R) * sizeof(float);
    // A step that keeps nearly all of the pixels blurs four columns for each: from some 2.5 million pixels, where the
    // launches no longer count, the three kernels are faster (3840x2160: 117 us against 126 at eta = 0.95, 113
    // against 115 at 0.9, 128 against 128 at 0.85; 1920x1080: 35.5 against 35.4 at 0.95).
    const double px = (double)gf.H * gf.W;
    const bool three = px > 2.5e6 && px < 1.29 * (double)gc.H * gc.W;
    if (smem <= 48 * 1024 && !three) {
        for (int q = 0; q < n; ++q) {
            a.fine[q] = fine[q];
            a.coarse[q] = coarse[q];
        }
        const dim3 grid((gc.W + PDX - 1) / PDX, (gc.H + PDY - 1) / PDY, n);
        k_pyr_down<<<grid, 256, smem, s>>>(a);
        return;
    }
    for (int q = 0; q < n; ++q) {
        // scratch holds two Hf x pitch planes: rows-blurred and fully blurred
        float *t1 = scratch, *t2 = scratch + (size_t)gf.H * gf.pitch;
        k_blur_rows<<<grid2(gf.H, gf.W), dim3(B2X, B2Y), 0, s>>>(fine[q], t1, gf, taps);
        k_blur_cols<<<grid2(gf.H, gf.W), dim3(B2X, B2Y), 0, s>>>(t1, t2, gf, taps);
        k_resample<<<grid2(gc.H, gc.W), dim3(B2X, B2Y), 0, s>>>(t2, gf, coarse[q], gc);
    }
}

void launch_upsample_f32(const float *coarse, Geom gc, float *fine, Geom gf, float scale, cudaStream_t s) {
    k_upsample<float><<<grid2(gf.H, gf.W), dim3(B2X, B2Y), 0, s>>>(coarse, gc, fine, gf, scale);
}

void launch_derivatives(const float *I, Geom g, float *Ix, float *Iy, cudaStream_t s) {
    k_derivatives<<<grid2(g.H, g.W), dim3(B2X, B2Y), 0, s>>>(I, g, Ix, Iy);
}

namespace {

// f(first pair, grid) for every launch over the pairs of a set: a grid holds 65,535 in its third dimension.
template <typename F> void over_pairs(const PairSet &a, F f) {
    dim3 d = grid2(a.pairs ? a.grid.H : a.one.g.H, a.pairs ? a.grid.W : a.one.g.W);
    const int n = a.pairs ? a.n : 1;
    for (int k = 0; k < n; k += 65535) {
        d.z = std::min(n - k, 65535);
        f(k, d);
    }
}
PairSet from_pair(PairSet a, int k) {
    if (a.pairs) a.pairs += k;
    return a;
}

}  // namespace

void launch_level_begin(const LevelArgs &a, int prec_dual, int prec_flow, cudaStream_t s) {
    over_pairs(a.fine, [&](int k, dim3 grid) {
        LevelArgs b = a;
        b.fine = from_pair(a.fine, k);
        b.coarse = from_pair(a.coarse, k);
        TVL1_DISPATCH_PREC(prec_dual, TD, TVL1_DISPATCH_PREC(prec_flow, TF,
                           k_level_begin<TD, TF><<<grid, dim3(B2X, B2Y), 0, s>>>(b)));
    });
}

void launch_warp(const PairSet &a, int cur, float beta, int prec, int prec_flow, cudaStream_t s) {
    over_pairs(a, [&](int k, dim3 grid) {
        const PairSet b = from_pair(a, k);
        TVL1_DISPATCH_PREC(prec, T, TVL1_DISPATCH_PREC(prec_flow, TF,
                           k_warp<T, TF><<<grid, dim3(B2X, B2Y), 0, s>>>(b, cur, beta)));
    });
}

void launch_warp_reset(const PairSet &a, cudaStream_t s) {
    // one pair: ms_max and the stop flag are adjacent
    if (!a.pairs) cudaMemsetAsync(const_cast<float *>(a.one.ms_max), 0, sizeof(float) + sizeof(int), s);
    else k_warp_reset<<<(a.n + 127) / 128, 128, 0, s>>>(a);
}

void launch_state_to_f32(const PairSet &from, const PairSet &to, int cur, int xbar, int has_w, int prec_dual,
                         int prec_flow, cudaStream_t s) {
    over_pairs(from, [&](int k, dim3 grid) {
        const PairSet f = from_pair(from, k), t = from_pair(to, k);
        TVL1_DISPATCH_PREC(prec_dual, TD, TVL1_DISPATCH_PREC(prec_flow, TF,
                           k_state_to_f32<TD, TF><<<grid, dim3(B2X, B2Y), 0, s>>>(f, t, cur, xbar, has_w)));
    });
}

void launch_output(const Fields &f, Geom g, float *u, float *v, float *w, int prec_flow, cudaStream_t s) {
    TVL1_DISPATCH_PREC(prec_flow, TF, k_output<TF><<<grid2(g.H, g.W), dim3(B2X, B2Y), 0, s>>>(f, g, u, v, w));
}

}  // namespace tvl1
