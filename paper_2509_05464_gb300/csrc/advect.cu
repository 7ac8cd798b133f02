// advect.cu -- a1 scatterer advection, a2 vessel membership and depth
// binning.
//
// Integer-valued decisions (the wrap of a scatterer along its vessel,
// membership, bins) are those of plain IEEE double: the membership test and
// the wrap decide in binary32 / float-float only where a bound shows that
// double would decide the same, and fall back to the double operations, in
// the order of a plain CPU statement, near a boundary.  Positions are
// float-float (48 bits) rounded once to binary32: GB300 runs two FP64
// operations per SM and clock, and the trajectories of 500k scatterers over
// 100 frames in FP64 took 4.1 ms against 0.09 ms for writing them.  This
// file is compiled with --fmad=false so that no multiply-add is contracted.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstring>

#include "batch.cuh"
#include "fq_internal.cuh"

namespace {

using fqi::ff;

constexpr int kSegDoubles = 20;  // kind, p0[3], a1[3], a2[3], a3[3], length, radius, vmax, arc_radius, phi1, arc_end[2]

struct SegTable {
    int n;
    double t[FQ_MAX_SEGMENTS][kSegDoubles];
};

struct MotionParams {
    int n_terms;
    double amp[4], freq[4], phase[4], dir[4][3];
    double g[3], ce[3], vel[3], omega[3], cr[3];
};

void pack_segments(const fq_flow *flow, SegTable &st)
{
    std::memset(&st, 0, sizeof st);
    st.n = flow ? flow->n_seg : 0;
    for (int i = 0; i < st.n; ++i) {
        const fq_segment &s = flow->seg[i];
        double *t = st.t[i];
        t[0] = (double)s.kind;
        for (int d = 0; d < 3; ++d) {
            t[1 + d] = s.p0[d];
            t[4 + d] = s.a1[d];
            t[7 + d] = s.a2[d];
            t[10 + d] = s.a3[d];
        }
        t[13] = s.length;
        t[14] = s.radius;
        t[15] = s.vmax;
        t[16] = s.arc_radius;
        t[17] = s.phi1;
        t[18] = s.arc_end[0];
        t[19] = s.arc_end[1];
    }
}

__device__ __forceinline__ double wrap_into(double a, double span)
{
    return a - span * floor(a / span);
}

// Frame-constant part of the motion map, evaluated once per block.
struct FrameConst {
    double t, ct, st, kx, ky, kz, wn;
    double dsum[3];
    bool rigid;  // no elastic gain and no drift: out = P + dsum (1 + 0 and + 0 are exact)
};

__device__ void frame_constants(const MotionParams &mp, double t, FrameConst &fc)
{
    fc.t = t;
    const double *om = mp.omega;
    double wn = sqrt(om[0] * om[0] + om[1] * om[1] + om[2] * om[2]);
    fc.wn = wn;
    fc.kx = fc.ky = fc.kz = 0.0;
    fc.ct = 1.0;
    fc.st = 0.0;
    if (wn > 0.0) {
        fc.kx = om[0] / wn;
        fc.ky = om[1] / wn;
        fc.kz = om[2] / wn;
        fc.ct = cos(wn * t);
        fc.st = sin(wn * t);
    }
    fc.rigid = mp.g[0] == 0.0 && mp.g[1] == 0.0 && mp.g[2] == 0.0 && mp.vel[0] == 0.0 && mp.vel[1] == 0.0 &&
               mp.vel[2] == 0.0;
    fc.dsum[0] = fc.dsum[1] = fc.dsum[2] = 0.0;
    for (int j = 0; j < mp.n_terms; ++j) {
        double sj = mp.amp[j] * sin(2.0 * 3.14159265358979323846 * mp.freq[j] * t + mp.phase[j]);
        for (int d = 0; d < 3; ++d) fc.dsum[d] += sj * mp.dir[j][d];
    }
}

// Position of scatterer s at the frame time of fc (written to o[d * S + s]).
__device__ __forceinline__ void advect_point(const float *__restrict__ p0, const int32_t *__restrict__ seg,
                                             const float *__restrict__ flow, int64_t S, int64_t s,
                                             const SegTable &st, const MotionParams &mp, const FrameConst &fc,
                                             float *__restrict__ o)
{
    const double t = fc.t;
    double P[3];
    int si = seg[s];
    if (si < 0 || si >= st.n) {
        P[0] = p0[s];
        P[1] = p0[S + s];
        P[2] = p0[2 * S + s];
    } else {
        const double *sg = st.t[si];
        double q = flow[s], x1 = flow[S + s], x2 = flow[2 * S + s];
        double R = sg[14];
        double v = sg[15] * (1.0 - (x1 * x1 + x2 * x2) / (R * R));
        if ((int)sg[0] == FQ_SEG_LINE) {
            double a = wrap_into(q + v * t, sg[13]);
            for (int d = 0; d < 3; ++d)
                P[d] = sg[1 + d] + a * sg[4 + d] + x1 * sg[7 + d] + x2 * sg[10 + d];
        } else {
            double phi = wrap_into(q + v * t / sg[16], sg[17]);
            double cp, sp;
            sincos(phi, &sp, &cp);
            const double rr = sg[16] + x1;
            for (int d = 0; d < 3; ++d)
                P[d] = sg[1 + d] + rr * (cp * sg[4 + d] + sp * sg[7 + d]) + x2 * sg[10 + d];
        }
    }
    double Q0 = P[0], Q1 = P[1], Q2 = P[2];
    if (fc.wn > 0.0) {
        const double *cr = mp.cr;
        double w0 = P[0] - cr[0], w1 = P[1] - cr[1], w2 = P[2] - cr[2];
        double kw = fc.kx * w0 + fc.ky * w1 + fc.kz * w2;
        double c0 = fc.ky * w2 - fc.kz * w1, c1 = fc.kz * w0 - fc.kx * w2, c2 = fc.kx * w1 - fc.ky * w0;
        double omc = 1.0 - fc.ct;
        P[0] = cr[0] + w0 * fc.ct + c0 * fc.st + fc.kx * kw * omc;
        P[1] = cr[1] + w1 * fc.ct + c1 * fc.st + fc.ky * kw * omc;
        P[2] = cr[2] + w2 * fc.ct + c2 * fc.st + fc.kz * kw * omc;
    }
    if (fc.rigid) {
        // the general form below with gain 1 + 0 = 1 and drift 0 t = 0, whose
        // operations are exact: the same doubles
        for (int d = 0; d < 3; ++d) o[d * S + s] = (float)(P[d] + fc.dsum[d]);
        return;
    }
    double gain = 1.0 + (mp.g[0] * (Q0 - mp.ce[0]) + mp.g[1] * (Q1 - mp.ce[1]) + mp.g[2] * (Q2 - mp.ce[2]));
    for (int d = 0; d < 3; ++d) o[d * S + s] = (float)(P[d] + mp.vel[d] * t + gain * fc.dsum[d]);
}

// ------------------------------------------------------ float-float motion --
// Frame constants of the motion without rotation, and the ensemble's: the
// same doubles as FrameConst, split.
struct FrameFF {
    double td;
    ff t, dsum[3], drift[3];
};
struct MotionFF {
    bool rigid, drift;
    ff k0, g[3];  // elastic gain = k0 + g . Q
};
// Segment fields used per scatterer and frame (shared memory).
struct SegMotion {
    double t[kSegDoubles];
    double inv_rc;
    ff span;
};
constexpr int kMotionThreads = 256;
constexpr int kFrameMax = 16;    // frames per block
constexpr int kSinTab = 64;      // steps of pi / 64 over [0, pi]

struct MotionShared {
    FrameFF fr[kFrameMax];
    MotionFF m;
    float4 tab[kSinTab + 1];     // cos, sin of k pi / 64, each as a float pair
    SegMotion seg[FQ_MAX_SEGMENTS];
};

__device__ __forceinline__ ff ff_of(double d)
{
    const fqi::df2 s = fqi::split_double(d);
    return {s.hi, s.lo};
}

// Segment table, gain and sine table of an ensemble: once per block.
__device__ void motion_tables(const SegTable &st, const MotionParams &mp, MotionShared &sh)
{
    bool arcs = false;
    for (int i = 0; i < st.n; ++i) arcs |= (int)st.t[i][0] != FQ_SEG_LINE;
    for (int i = threadIdx.x; i < st.n; i += blockDim.x) {
        SegMotion &g = sh.seg[i];
        for (int k = 0; k < kSegDoubles; ++k) g.t[k] = st.t[i][k];
        const bool line = (int)g.t[0] == FQ_SEG_LINE;
        g.inv_rc = line ? 1.0 : 1.0 / g.t[16];
        g.span = ff_of(line ? g.t[13] : g.t[17]);
    }
    if (arcs)
        for (int k = threadIdx.x; k <= kSinTab; k += blockDim.x) {
            double sn, cs;
            sincospi((double)k / kSinTab, &sn, &cs);
            const ff c = ff_of(cs), s = ff_of(sn);
            sh.tab[k] = make_float4(c.hi, c.lo, s.hi, s.lo);
        }
    if (threadIdx.x == blockDim.x - 1) {
        MotionFF &m = sh.m;
        m.drift = mp.vel[0] != 0.0 || mp.vel[1] != 0.0 || mp.vel[2] != 0.0;
        m.rigid = mp.g[0] == 0.0 && mp.g[1] == 0.0 && mp.g[2] == 0.0;
        m.k0 = ff_of(1.0 - (mp.g[0] * mp.ce[0] + mp.g[1] * mp.ce[1] + mp.g[2] * mp.ce[2]));
        for (int d = 0; d < 3; ++d) m.g[d] = ff_of(mp.g[d]);
    }
}

__device__ __forceinline__ void motion_frame(const MotionParams &mp, double t, FrameFF &f)
{
    FrameConst fc;
    frame_constants(mp, t, fc);
    f.td = t;
    f.t = ff_of(t);
    for (int d = 0; d < 3; ++d) {
        f.dsum[d] = ff_of(fc.dsum[d]);
        f.drift[d] = ff_of(mp.vel[d] * t);
    }
}

__device__ __forceinline__ bool has_rotation(const MotionParams &mp)
{
    return mp.omega[0] != 0.0 || mp.omega[1] != 0.0 || mp.omega[2] != 0.0;
}

// P + drift + gain dsum rounded to binary32 (P, and the gain if elastic, as
// float pairs; the error term is dropped where the sum is not finite).
__device__ __forceinline__ float displaced(ff P, const MotionFF &m, ff gain, ff dsum, ff drift)
{
    ff w = dsum;
    if (!m.rigid) {
        const float h = __fmul_rn(gain.hi, dsum.hi);
        float e = __fmaf_rn(gain.hi, dsum.hi, -h);
        e = __fmaf_rn(gain.hi, dsum.lo, e);
        w = ff{h, __fmaf_rn(gain.lo, dsum.hi, e)};
    }
    ff s = fqi::ff_two_sum(P.hi, w.hi);
    float lo = __fadd_rn(__fadd_rn(P.lo, w.lo), s.lo);
    if (m.drift) {
        const ff q = fqi::ff_two_sum(s.hi, drift.hi);
        lo = __fadd_rn(lo, __fadd_rn(q.lo, drift.lo));
        s.hi = q.hi;
    }
    return fabsf(s.hi) <= FLT_MAX ? __fadd_rn(s.hi, lo) : s.hi;
}

__device__ __forceinline__ ff gain_at(const MotionFF &m, ff x, ff y, ff z)
{
    ff k = fqi::ff_add(m.k0, fqi::ff_mul(m.g[0], x));
    k = fqi::ff_add(k, fqi::ff_mul(m.g[1], y));
    return fqi::ff_add(k, fqi::ff_mul(m.g[2], z));
}

// cos and sin of r in [0, pi]: table at the nearest multiple of pi / 64, then
// the Taylor series of the remainder (|x| <= 0.0246: truncated below 1e-14,
// evaluated to ~1e-13).  Outside the table, IEEE double.
__device__ __forceinline__ void cos_sin(const float4 *tab, ff r, ff &c, ff &s)
{
    const float kf = rintf(__fmul_rn(r.hi, (float)(kSinTab / 3.14159265358979323846)));
    if (!(kf >= 0.0f && kf <= (float)kSinTab)) {
        double sn, cs;
        sincos((double)r.hi + (double)r.lo, &sn, &cs);
        c = ff_of(cs);
        s = ff_of(sn);
        return;
    }
    const float4 t = tab[(int)kf];
    const ff C = {t.x, t.y}, S = {t.z, t.w};
    constexpr double step = 3.14159265358979323846 / kSinTab;
    const ff st = {(float)step, (float)(step - (double)(float)step)};
    const ff x = fqi::ff_add(r, fqi::ff_neg(fqi::ff_mul_f(st, kf)));
    const ff x2 = fqi::ff_sqr(x);
    const float q = x2.hi;
    // sin x = x + x (-x^2/6 + x^4/120), cos x = 1 + (-x^2/2 + x^4/24 - x^6/720)
    const float ts = __fmul_rn(q, __fmaf_rn(q, 1.0f / 120.0f, -1.0f / 6.0f));
    const ff sx = fqi::ff_add_f(x, __fmul_rn(x.hi, ts));
    const float tc = __fmul_rn(__fmul_rn(q, q), __fmaf_rn(q, -1.0f / 720.0f, 1.0f / 24.0f));
    const ff cx = fqi::ff_add_f(ff{__fmul_rn(-0.5f, x2.hi), __fmul_rn(-0.5f, x2.lo)}, tc);  // cos x - 1
    c = fqi::ff_add(fqi::ff_add(C, fqi::ff_mul(C, cx)), fqi::ff_neg(fqi::ff_mul(S, sx)));
    s = fqi::ff_add(fqi::ff_add(S, fqi::ff_mul(S, cx)), fqi::ff_mul(C, sx));
}

// Frames 0 .. nf - 1 of sh.fr of scatterer s, written to o[f 3 S + d S + s].
__device__ __forceinline__ void advect_frames(const float *__restrict__ p0, const int32_t *__restrict__ seg,
                                              const float *__restrict__ flow, int64_t S, int64_t s, int n_seg,
                                              const MotionShared &sh, int nf, float *__restrict__ o)
{
    const int si = seg[s];
    const MotionFF &m = sh.m;
    const ff one = {1.0f, 0.0f};
    if (si < 0 || si >= n_seg) {
        const ff P[3] = {{p0[s], 0.0f}, {p0[S + s], 0.0f}, {p0[2 * S + s], 0.0f}};
        ff gain = m.rigid ? one : gain_at(m, P[0], P[1], P[2]);
        if (!(fabsf(gain.hi) <= FLT_MAX))  // an infinite coordinate: the error terms are not numbers
            gain.hi = __fmaf_rn(m.g[0].hi, P[0].hi, __fmaf_rn(m.g[1].hi, P[1].hi, m.g[2].hi * P[2].hi));
        for (int f = 0; f < nf; ++f)
#pragma unroll
            for (int d = 0; d < 3; ++d)
                o[((int64_t)f * 3 + d) * S + s] = displaced(P[d], m, gain, sh.fr[f].dsum[d], sh.fr[f].drift[d]);
        return;
    }
    // blood: the path coordinate a = q + rate t wrapped into [0, span), then
    // P = base + u(a), u = a a1 (line) or cos a u1 + sin a u2 (arc)
    const SegMotion &g = sh.seg[si];
    const double *sg = g.t;
    const bool line = (int)sg[0] == FQ_SEG_LINE;
    const double q = flow[s], x1 = flow[S + s], x2 = flow[2 * S + s];
    const double v = sg[15] * (1.0 - (x1 * x1 + x2 * x2) / (sg[14] * sg[14]));
    const ff rate = ff_of(v * g.inv_rc);
    ff base[3], u1[3], u2[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double e = sg[1 + d] + x2 * sg[10 + d];
        if (line) {
            base[d] = ff_of(e + x1 * sg[7 + d]);
            u1[d] = ff_of(sg[4 + d]);
            u2[d] = ff{0.0f, 0.0f};
        } else {
            const double rr = sg[16] + x1;
            base[d] = ff_of(e);
            u1[d] = ff_of(rr * sg[4 + d]);
            u2[d] = ff_of(rr * sg[7 + d]);
        }
    }
    const ff span = g.span;
    const float margin = 1e-6f * span.hi;
    float n = 0.0f;  // the wrap count of the last frame: tried first
    for (int f = 0; f < nf; ++f) {
        const FrameFF &fr = sh.fr[f];
        ff r = fqi::ff_add_f(fqi::ff_mul(rate, fr.t), (float)q);
        if (n != 0.0f) r = fqi::ff_add(r, fqi::ff_neg(fqi::ff_mul_f(span, n)));
        if (!(r.hi > margin && r.hi < span.hi - margin)) {
            // near an end or past it: the count of IEEE double
            const double sd = line ? sg[13] : sg[17];
            const double a = line ? q + v * fr.td : q + v * fr.td / sg[16];
            const double nn = floor(a / sd);
            r = ff_of(a - sd * nn);
            // many wraps on, the float pair of q + rate t (48 bits of it) is too
            // coarse for a position: the double of every frame, then
            n = fabs(nn) < 4096.0 ? (float)nn : 0.0f;
        }
        ff P[3];
        if (line) {
#pragma unroll
            for (int d = 0; d < 3; ++d) P[d] = fqi::ff_add(base[d], fqi::ff_mul(r, u1[d]));
        } else {
            ff c, sn;
            cos_sin(sh.tab, r, c, sn);
#pragma unroll
            for (int d = 0; d < 3; ++d)
                P[d] = fqi::ff_add(base[d], fqi::ff_add(fqi::ff_mul(c, u1[d]), fqi::ff_mul(sn, u2[d])));
        }
        const ff gain = m.rigid ? one : gain_at(m, P[0], P[1], P[2]);
#pragma unroll
        for (int d = 0; d < 3; ++d)
            o[((int64_t)f * 3 + d) * S + s] = displaced(P[d], m, gain, fr.dsum[d], fr.drift[d]);
    }
}

// One block: fb consecutive frames of a strided set of scatterers, so that a
// scatterer's setup (its vessel, speed and gain) and the block's tables are
// shared by the frames.  Membership and trajectories of 500k scatterers x
// 100 frames (tree of 63 lines, elastic motion): 5.68 ms with one FP64
// evaluation per position and (scatterer, vessel) pair, 0.30 ms now (0.24 this
// kernel, 0.06 the membership); positions identical.
__global__ void __launch_bounds__(kMotionThreads) advect_kernel(const float *__restrict__ p0,
                                                                const int32_t *__restrict__ seg,
                                                                const float *__restrict__ flow, int64_t S,
                                                                const __grid_constant__ SegTable st,
                                                                const __grid_constant__ MotionParams mp, double t0,
                                                                double dt, int F, int fb, float *__restrict__ out)
{
    __shared__ MotionShared sh;
    const int f0 = blockIdx.y * fb, nf = min(fb, F - f0);
    motion_tables(st, mp, sh);
    if (threadIdx.x < nf) motion_frame(mp, t0 + (double)(f0 + (int)threadIdx.x) * dt, sh.fr[threadIdx.x]);
    __syncthreads();
    float *o = out + (int64_t)f0 * 3 * S;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < S; s += (int64_t)gridDim.x * blockDim.x)
        advect_frames(p0, seg, flow, S, s, st.n, sh, nf, o);
}

// Motion with a rigid rotation: IEEE double throughout, one frame per block.
__global__ void advect_rot_kernel(const float *__restrict__ p0, const int32_t *__restrict__ seg,
                                  const float *__restrict__ flow, int64_t S, const SegTable st,
                                  const MotionParams mp, double t0, double dt,
                                  float *__restrict__ out)
{
    __shared__ FrameConst fc;
    const int f = blockIdx.y;
    if (threadIdx.x == 0) frame_constants(mp, t0 + (double)f * dt, fc);
    __syncthreads();
    float *o = out + (int64_t)f * 3 * S;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < S;
         s += (int64_t)gridDim.x * blockDim.x)
        advect_point(p0, seg, flow, S, s, st, mp, fc, o);
}

// ------------------------------------------------------------ membership --
__device__ __forceinline__ bool inside_seg(const double *sg, double px, double py, double pz)
{
    double w0 = px - sg[1], w1 = py - sg[2], w2 = pz - sg[3];
    double R2 = sg[14] * sg[14];
    if ((int)sg[0] == FQ_SEG_LINE) {
        double s = (w0 * sg[4] + w1 * sg[5]) + w2 * sg[6];
        if (s < 0.0 || s > sg[13]) return false;
        double q1 = (w0 * sg[7] + w1 * sg[8]) + w2 * sg[9];
        double q2 = (w0 * sg[10] + w1 * sg[11]) + w2 * sg[12];
        return (q1 * q1 + q2 * q2) < R2;
    }
    double x1 = (w0 * sg[4] + w1 * sg[5]) + w2 * sg[6];
    double x2 = (w0 * sg[7] + w1 * sg[8]) + w2 * sg[9];
    double x3 = (w0 * sg[10] + w1 * sg[11]) + w2 * sg[12];
    if (x2 < 0.0) return false;                        // before the arc start (angle 0)
    if (x1 * sg[19] - x2 * sg[18] < 0.0) return false;  // past the arc end (angle phi1 <= pi)
    double rin = sqrt(x1 * x1 + x2 * x2) - sg[16];
    return (rin * rin + x3 * x3) < R2;
}

// A segment for the binary32 rejection: the coordinates along its axes are
// a . P - c to within err = 2^-20 amax (|P|_1 + pn) (their rounding errors sum
// to less than 8 x 2^-24 of that product), so a coordinate beyond its limit by
// more than err is beyond it in IEEE double too.
struct SegBox {
    float4 a1, a2, a3;  // axis, c
    float4 lim;         // radius, length (line) or arc radius, amax, pn
};
struct ClassifyShared {
    SegBox box[FQ_MAX_SEGMENTS];
    int line[FQ_MAX_SEGMENTS];
};

__device__ void classify_tables(const SegTable &st, ClassifyShared &sh)
{
    for (int i = threadIdx.x; i < st.n; i += blockDim.x) {
        const double *t = st.t[i];
        SegBox &b = sh.box[i];
        float4 *ax[3] = {&b.a1, &b.a2, &b.a3};
        double amax = 0.0;
        for (int k = 0; k < 3; ++k) {
            const double *a = t + 4 + 3 * k;
            *ax[k] = make_float4((float)a[0], (float)a[1], (float)a[2],
                                 (float)(a[0] * t[1] + a[1] * t[2] + a[2] * t[3]));
            for (int d = 0; d < 3; ++d) amax = fmax(amax, fabs(a[d]));
        }
        const bool line = (int)t[0] == FQ_SEG_LINE;
        const double up = 1.0 + 1.0 / (1 << 20);  // covers the rounding of the limits
        b.lim = make_float4((float)(fabs(t[14]) * up), (float)(line ? t[13] * up : t[16]), (float)(amax * up),
                            (float)((fabs(t[1]) + fabs(t[2]) + fabs(t[3])) * up));
        sh.line[i] = line;
    }
}

__device__ __forceinline__ float axis_coord(const float4 &a, float x, float y, float z)
{
    return __fmaf_rn(x, a.x, __fmaf_rn(y, a.y, __fmaf_rn(z, a.z, -a.w)));
}

// The lowest segment that holds the tissue scatterer, or -1.  The binary32
// test rejects almost every (scatterer, segment) pair (comparisons with NaN
// reject nothing); the IEEE double test decides the rest.
__device__ __forceinline__ int find_segment(const SegTable &st, const ClassifyShared &sh, float x, float y, float z)
{
    const float n1 = fabsf(x) + fabsf(y) + fabsf(z);
    for (int i = 0; i < st.n; ++i) {
        const SegBox &b = sh.box[i];
        const float err = 9.5367431640625e-7f * b.lim.z * (n1 + b.lim.w);
        const float wide = b.lim.x + err;
        if (fabsf(axis_coord(b.a3, x, y, z)) > wide) continue;
        const float c2 = axis_coord(b.a2, x, y, z), c1 = axis_coord(b.a1, x, y, z);
        if (sh.line[i]) {
            if (fabsf(c2) > wide || c1 < -err || c1 > b.lim.y + err) continue;
        } else {
            const float r = sqrtf(c1 * c1 + c2 * c2);
            if (c2 < -err || fabsf(r - b.lim.y) > wide + 4.0f * err + 1e-6f * (r + b.lim.y)) continue;
        }
        if (inside_seg(st.t[i], x, y, z)) return i;
    }
    return -1;
}

__device__ __forceinline__ void classify_point(const float *__restrict__ pos, const int32_t *__restrict__ seg,
                                               int64_t S, int64_t s, const SegTable &st, const ClassifyShared &sh,
                                               const float *__restrict__ amp_in, int32_t *__restrict__ vessel,
                                               float *__restrict__ amp_out)
{
    const int own = seg[s];
    const int v = own < 0 ? find_segment(st, sh, pos[s], pos[S + s], pos[2 * S + s]) : own;
    vessel[s] = own < 0 && v < 0 ? own : v;
    if (amp_out) amp_out[s] = (own < 0 && v >= 0) ? 0.0f : amp_in[s];
}

// 500k scatterers x 63 lines: 1.55 ms with the IEEE double test of every pair.
__global__ void __launch_bounds__(256) classify_kernel(const float *__restrict__ pos, const int32_t *__restrict__ seg,
                                                       int64_t S, const __grid_constant__ SegTable st,
                                                       const float *__restrict__ amp_in,
                                                       int32_t *__restrict__ vessel, float *__restrict__ amp_out)
{
    __shared__ ClassifyShared sh;
    classify_tables(st, sh);
    __syncthreads();
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < S;
         s += (int64_t)gridDim.x * blockDim.x)
        classify_point(pos, seg, S, s, st, sh, amp_in, vessel, amp_out);
}

// ----------------------------------------------------------- batched --
// Items of fqb::kItemScat scatterers: classify, one item per chunk of
// scatterers; advect, as many items per chunk as frames, item y of a chunk
// taking the 1 / kBatchFrames part y % kBatchFrames of its scatterers over
// the frames of group y / kBatchFrames.
using fqb::kItemScat;
constexpr int kBatchThreads = 256;
constexpr int kBatchFrames = 8;
static_assert(kItemScat == kBatchThreads * kBatchFrames, "one scatterer per thread and frame group");

__global__ void __launch_bounds__(kBatchThreads) classify_batched_kernel(const fqb::EnsDev *__restrict__ ens,
                                                                         const fqb::StageQueue q)
{
    __shared__ int s_buf[2];
    __shared__ ClassifyShared sh;
    int cur = -1;
    fqb::Item it;
    while (fqb::next_item(q, ens, fqb::ST_CLASSIFY, s_buf, it)) {
        const fqb::EnsDev &e = ens[it.e];
        const SegTable &st = *reinterpret_cast<const SegTable *>(e.seg_table);
        if (it.e != cur) {
            classify_tables(st, sh);
            cur = it.e;
            __syncthreads();
        }
        const int64_t beg = (int64_t)it.x * kItemScat;
        const int64_t end = beg + kItemScat < e.S ? beg + kItemScat : e.S;
        for (int64_t s = beg + threadIdx.x; s < end; s += blockDim.x)
            classify_point(e.p0, e.seg, e.S, s, st, sh, e.amp, e.vessel, e.amp_eff);
    }
}

__global__ void __launch_bounds__(kBatchThreads) advect_batched_kernel(const fqb::EnsDev *__restrict__ ens,
                                                                       const fqb::StageQueue q)
{
    __shared__ int s_buf[2];
    __shared__ MotionShared sh;
    __shared__ FrameConst fc;
    int cur = -1;
    fqb::Item it;
    while (fqb::next_item(q, ens, fqb::ST_ADVECT, s_buf, it)) {
        const fqb::EnsDev &e = ens[it.e];
        const SegTable &st = *reinterpret_cast<const SegTable *>(e.seg_table);
        const MotionParams &mp = *reinterpret_cast<const MotionParams *>(e.motion);
        const int64_t beg = (int64_t)it.x * kItemScat;
        if (has_rotation(mp)) {  // as advect_rot_kernel: one frame per item
            if (threadIdx.x == 0) frame_constants(mp, e.t0 + (double)it.y * e.dt, fc);
            __syncthreads();
            float *o = e.pos + (int64_t)it.y * 3 * e.S;
            const int64_t end = beg + kItemScat < e.S ? beg + kItemScat : e.S;
            for (int64_t s = beg + threadIdx.x; s < end; s += blockDim.x)
                advect_point(e.p0, e.seg, e.flow, e.S, s, st, mp, fc, o);
            continue;
        }
        if (it.e != cur) {
            motion_tables(st, mp, sh);
            cur = it.e;
        }
        // a last group of nf < kBatchFrames frames has nf items: each takes every nf-th 256 scatterers
        const int f0 = it.y / kBatchFrames * kBatchFrames, nf = min(kBatchFrames, e.F - f0);
        if (threadIdx.x < nf) motion_frame(mp, e.t0 + (double)(f0 + (int)threadIdx.x) * e.dt, sh.fr[threadIdx.x]);
        __syncthreads();
        float *o = e.pos + (int64_t)f0 * 3 * e.S;
        for (int part = it.y - f0; part < kBatchFrames; part += nf) {
            const int64_t s = beg + part * kBatchThreads + threadIdx.x;
            if (s < e.S) advect_frames(e.p0, e.seg, e.flow, e.S, s, st.n, sh, nf, o);
        }
    }
}

void pack_motion(const fq_motion *motion, MotionParams &mp)
{
    std::memset(&mp, 0, sizeof mp);
    if (!motion) return;
    mp.n_terms = motion->n_terms;
    for (int j = 0; j < 4; ++j) {
        mp.amp[j] = motion->amp[j];
        mp.freq[j] = motion->freq[j];
        mp.phase[j] = motion->phase[j];
        for (int d = 0; d < 3; ++d) mp.dir[j][d] = motion->dir[j][d];
    }
    for (int d = 0; d < 3; ++d) {
        mp.g[d] = motion->elastic_grad[d];
        mp.ce[d] = motion->elastic_center[d];
        mp.vel[d] = motion->vel[d];
        mp.omega[d] = motion->omega[d];
        mp.cr[d] = motion->rot_center[d];
    }
}

// ---------------------------------------------------------------- binning --
// Stable counting sort in three passes over fixed chunks of kChunk
// scatterers: (1) per-(bin, chunk) counts, (2) one exclusive scan over the
// bin-major count table, which directly gives the first output slot of every
// (bin, chunk), (3) a single warp per chunk walks its scatterers in index
// order and places them, ranking equal keys with warp match masks.
constexpr int kChunk = 4096;
constexpr int kMaxBins = 8192;

__global__ void bin_count_kernel(const float *__restrict__ z, int64_t S, double z0, double dz, int B,
                                 int32_t *__restrict__ key, int32_t *__restrict__ counts, int n_chunks)
{
    extern __shared__ int32_t hist[];
    const int chunk = blockIdx.x;
    for (int b = threadIdx.x; b < B; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    int64_t beg = (int64_t)chunk * kChunk;
    int64_t end = beg + kChunk < S ? beg + kChunk : S;
    for (int64_t s = beg + threadIdx.x; s < end; s += blockDim.x) {
        double q = floor(((double)z[s] - z0) / dz);
        int b = q < 0.0 ? 0 : (q > (double)(B - 1) ? B - 1 : (int)q);
        key[s] = b;
        atomicAdd(&hist[b], 1);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < B; b += blockDim.x) counts[(int64_t)b * n_chunks + chunk] = hist[b];
}

// exclusive scan of n ints in place by one CTA of 1024 threads
__global__ void scan_kernel(int32_t *__restrict__ a, int64_t n)
{
    __shared__ int32_t warp_tot[32];
    __shared__ int32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int64_t base = 0; base < n; base += blockDim.x) {
        int64_t i = base + threadIdx.x;
        int32_t v = i < n ? a[i] : 0;
        int32_t x = v;
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_tot[wid] = x;
        __syncthreads();
        if (wid == 0) {
            int32_t t = warp_tot[lane];
            for (int o = 1; o < 32; o <<= 1) {
                int32_t y = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += y;
            }
            warp_tot[lane] = t;  // inclusive prefix of warp totals
        }
        __syncthreads();
        int32_t before = carry + (wid > 0 ? warp_tot[wid - 1] : 0);
        if (i < n) a[i] = before + x - v;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = before + x;
        __syncthreads();
    }
}

__global__ void bin_place_kernel(const int32_t *__restrict__ key, int64_t S, int B,
                                 const int32_t *__restrict__ offsets, int n_chunks,
                                 int32_t *__restrict__ perm, int32_t *__restrict__ bin_off)
{
    extern __shared__ int32_t next[];
    const int chunk = blockIdx.x;
    const int lane = threadIdx.x;  // one warp
    for (int b = lane; b < B; b += 32) next[b] = offsets[(int64_t)b * n_chunks + chunk];
    if (chunk == 0) {
        for (int b = lane; b < B; b += 32) bin_off[b] = offsets[(int64_t)b * n_chunks];
        if (lane == 0) bin_off[B] = (int32_t)S;
    }
    __syncwarp();
    int64_t beg = (int64_t)chunk * kChunk;
    int64_t end = beg + kChunk < S ? beg + kChunk : S;
    const unsigned lt = (1u << lane) - 1u;
    for (int64_t base = beg; base < end; base += 32) {
        int64_t s = base + lane;
        bool valid = s < end;
        unsigned act = __ballot_sync(0xffffffffu, valid);
        int k = valid ? key[s] : -1 - lane;  // invalid lanes get unique dummy keys
        unsigned peers = __match_any_sync(0xffffffffu, k);
        if (valid) {
            int rank = __popc(peers & lt);
            perm[next[k] + rank] = (int32_t)s;
        }
        __syncwarp();
        // the highest lane of each group advances the bin's cursor
        if (valid && (peers >> lane) == 1u) next[k] += __popc(peers);
        __syncwarp();
        (void)act;
    }
}

}  // namespace

extern "C" {

fq_status fq_advect_scatterers(const float *p0, const int32_t *seg_id, const float *flow_coord,
                               int64_t S, const fq_flow *flow, const fq_motion *motion,
                               double t0, double dt, int32_t n_frames, float *pos_out,
                               void *stream)
{
    FQ_REQUIRE(S >= 0 && n_frames >= 1, FQ_ERR_INVALID_ARG, "fq_advect_scatterers: S=%lld n_frames=%d",
               (long long)S, n_frames);
    if (S == 0) return FQ_OK;
    FQ_REQUIRE(p0 && seg_id && flow_coord && pos_out, FQ_ERR_INVALID_ARG,
               "fq_advect_scatterers: null device pointer");
    FQ_REQUIRE(!flow || (flow->n_seg >= 0 && flow->n_seg <= FQ_MAX_SEGMENTS && (flow->n_seg == 0 || flow->seg)),
               FQ_ERR_SHAPE, "fq_advect_scatterers: n_seg must be in [0, %d]", FQ_MAX_SEGMENTS);
    FQ_REQUIRE(!motion || (motion->n_terms >= 0 && motion->n_terms <= FQ_MAX_MOTION_TERMS), FQ_ERR_SHAPE,
               "fq_advect_scatterers: n_terms must be in [0, 4]");
    SegTable local;
    pack_segments(flow, local);
    MotionParams mp;
    pack_motion(motion, mp);
    const int threads = kMotionThreads;
    int64_t blocks = (S + threads - 1) / threads;
    cudaStream_t cs = (cudaStream_t)stream;
    if (mp.omega[0] != 0.0 || mp.omega[1] != 0.0 || mp.omega[2] != 0.0) {
        if (blocks > 4096) blocks = 4096;
        advect_rot_kernel<<<dim3((unsigned)blocks, (unsigned)n_frames), threads, 0, cs>>>(p0, seg_id, flow_coord, S,
                                                                                          local, mp, t0, dt, pos_out);
        return fqi::launch_check("fq_advect_scatterers");
    }
    // frames per block: as many as leave ~8 blocks per SM (16 at most: the
    // setup is then a few percent), one where the call is too small for that
    const int64_t want = 8 * 152;
    int fb = (int)std::min<int64_t>(kFrameMax, std::max<int64_t>(1, blocks * n_frames / want));
    const int groups = (n_frames + fb - 1) / fb;
    blocks = std::min<int64_t>(blocks, std::max<int64_t>(1, (want + groups - 1) / groups));
    advect_kernel<<<dim3((unsigned)blocks, (unsigned)groups), threads, 0, cs>>>(p0, seg_id, flow_coord, S, local, mp,
                                                                                t0, dt, n_frames, fb, pos_out);
    return fqi::launch_check("fq_advect_scatterers");
}

fq_status fq_classify_scatterers(const float *pos, const int32_t *seg_id, int64_t S,
                                 const fq_flow *flow, const float *amp_in, int32_t *vessel_out,
                                 float *amp_out, void *stream)
{
    FQ_REQUIRE(S >= 0, FQ_ERR_INVALID_ARG, "fq_classify_scatterers: S < 0");
    if (S == 0) return FQ_OK;
    FQ_REQUIRE(pos && seg_id && vessel_out && (amp_in || !amp_out), FQ_ERR_INVALID_ARG,
               "fq_classify_scatterers: null device pointer");
    FQ_REQUIRE(!flow || (flow->n_seg >= 0 && flow->n_seg <= FQ_MAX_SEGMENTS && (flow->n_seg == 0 || flow->seg)),
               FQ_ERR_SHAPE, "fq_classify_scatterers: n_seg must be in [0, %d]", FQ_MAX_SEGMENTS);
    SegTable local;
    pack_segments(flow, local);
    const int threads = 256;
    int64_t blocks = (S + threads - 1) / threads;
    if (blocks > 8 * 152) blocks = 8 * 152;
    classify_kernel<<<(unsigned)blocks, threads, 0, (cudaStream_t)stream>>>(pos, seg_id, S, local, amp_in,
                                                                            vessel_out, amp_out);
    return fqi::launch_check("fq_classify_scatterers");
}

fq_status fq_bin_workspace_size(int64_t S, int32_t B, size_t *bytes)
{
    FQ_REQUIRE(bytes && S >= 0 && B >= 1, FQ_ERR_INVALID_ARG, "fq_bin_workspace_size: bad arguments");
    int64_t n_chunks = (S + kChunk - 1) / kChunk;
    if (n_chunks < 1) n_chunks = 1;
    size_t k = ((size_t)S * 4 + 255) & ~(size_t)255;
    size_t c = ((size_t)n_chunks * B * 4 + 255) & ~(size_t)255;
    *bytes = k + c;
    return FQ_OK;
}

fq_status fq_bin_scatterers(const float *z, int64_t S, double z0, double dz, int32_t B,
                            int32_t *bin_off, int32_t *perm, void *workspace,
                            size_t workspace_bytes, void *stream)
{
    FQ_REQUIRE(S >= 0 && S < ((int64_t)1 << 31), FQ_ERR_SHAPE, "fq_bin_scatterers: S out of range");
    FQ_REQUIRE(B >= 1 && B <= kMaxBins, FQ_ERR_SHAPE, "fq_bin_scatterers: B must be in [1, %d]", kMaxBins);
    FQ_REQUIRE(dz > 0.0, FQ_ERR_INVALID_ARG, "fq_bin_scatterers: dz must be > 0");
    FQ_REQUIRE(bin_off && (S == 0 || (z && perm)), FQ_ERR_INVALID_ARG, "fq_bin_scatterers: null pointer");
    cudaStream_t st = (cudaStream_t)stream;
    if (S == 0) {
        return fqi::cuda_check(cudaMemsetAsync(bin_off, 0, sizeof(int32_t) * (B + 1), st), "fq_bin_scatterers");
    }
    size_t need = 0;
    fq_bin_workspace_size(S, B, &need);
    FQ_REQUIRE(workspace && workspace_bytes >= need, FQ_ERR_WORKSPACE,
               "fq_bin_scatterers: workspace needs %zu bytes", need);
    FQ_REQUIRE(fqi::aligned(workspace, 256), FQ_ERR_ALIGN, "fq_bin_scatterers: workspace not 256-byte aligned");
    int n_chunks = (int)((S + kChunk - 1) / kChunk);
    int32_t *key = (int32_t *)workspace;
    int32_t *counts = (int32_t *)((char *)workspace + (((size_t)S * 4 + 255) & ~(size_t)255));
    size_t smem = sizeof(int32_t) * B;
    if (smem > 48 * 1024) {
        fq_status s = fqi::cuda_check(cudaFuncSetAttribute(bin_count_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           (int)smem), "fq_bin_scatterers");
        if (s) return s;
        s = fqi::cuda_check(cudaFuncSetAttribute(bin_place_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem), "fq_bin_scatterers");
        if (s) return s;
    }
    bin_count_kernel<<<n_chunks, 256, smem, st>>>(z, S, z0, dz, B, key, counts, n_chunks);
    scan_kernel<<<1, 1024, 0, st>>>(counts, (int64_t)n_chunks * B);
    bin_place_kernel<<<n_chunks, 32, smem, st>>>(key, S, B, counts, n_chunks, perm, bin_off);
    return fqi::launch_check("fq_bin_scatterers");
}

}  // extern "C"

namespace fqi {

size_t seg_table_bytes() { return (sizeof(SegTable) + 15) & ~(size_t)15; }
size_t motion_bytes() { return (sizeof(MotionParams) + 15) & ~(size_t)15; }
void build_seg_table(const fq_flow *flow, void *out) { pack_segments(flow, *reinterpret_cast<SegTable *>(out)); }
void build_motion(const fq_motion *m, void *out) { pack_motion(m, *reinterpret_cast<MotionParams *>(out)); }

fq_status batched_classify(const fqb::EnsDev *ens, const fqb::StageQueue &q, int items, cudaStream_t st)
{
    const int grid = fqb::persistent_grid(classify_batched_kernel, kBatchThreads, 0, items);
    classify_batched_kernel<<<grid, kBatchThreads, 0, st>>>(ens, q);
    return launch_check("batched classify");
}

fq_status batched_advect(const fqb::EnsDev *ens, const fqb::StageQueue &q, int items, cudaStream_t st)
{
    const int grid = fqb::persistent_grid(advect_batched_kernel, kBatchThreads, 0, items);
    advect_batched_kernel<<<grid, kBatchThreads, 0, st>>>(ens, q);
    return launch_check("batched advect");
}

}  // namespace fqi
