// Guide field from splines (Guidefill, arxiv 1611.05319, Section 3.3) for sm_103a.
//
// g(x) = w_Gamma t_Gamma * exp(-d(x, Gamma)^2 / (2 eta^2)) for the nearest
// polyline segment Gamma when d <= 3 eta, else 0, at every hole pixel; w_Gamma =
// |g_Gamma| is the spline's weight (1 unless given, e.g. the coherence factor of
// detected splines).
//
// Two kernels per request:
//   bin_kernel    one thread per polyline point: the segment starting there is
//                 appended to every 32x32-pixel bin its bounding box, grown by
//                 3 eta + 1 px, overlaps (so no segment within 3 eta of a pixel
//                 is missed, FP32 rounding included);
//   guide_kernel  one CTA per eight bins, a warp at a time per strip of 8 rows
//                 of a bin that holds hole pixels: the bin's segments are
//                 staged in shared memory 32 at a time and each hole pixel
//                 takes the nearest one.  A bin whose list overflowed scans
//                 all segments of its frame.
// The nearest-segment choice and the 3-eta cut use a fixed FP32 expression
// with no contraction (ties: lowest segment index), so the decision does not
// depend on the machine; the returned value is the FP64 evaluation's for the
// chosen segment, rounded once to FP32 (formed in pairs of FP32 numbers where
// those settle the rounding, gf_guide_math.cuh).
//
// guide_kernel was bound by FP64 on the SMs with the most hole pixels, with one CTA
// per bin: 329 us on 32 frames of 1920 x 1080 (2.7 M hole pixels).  In pairs, with the
// same CTAs' work dealt to warps, 241 us; with the value evaluated in one place instead
// of unrolled per pixel, which kept the instruction cache missing, and the strips taken
// by whichever warp is free, 129 us.  Overflowed bins test every point of the frame
// against the strip's box, 32 at a time; scanned one by one by every warp they had no more
// warps than strips, and a 512 x 512 frame of 6,000 segments (eta 11) took 8.9 ms (5.8 with
// a CTA per bin), now 0.93.

#include "gf_internal.cuh"

namespace gf {

__global__ void upload_splines_kernel(const __grid_constant__ SplineChunk c)
{
    for (int i = threadIdx.x; i < c.count; i += blockDim.x) {
        c.dst_frames[c.first + i] = c.frames[i];
        c.dst_po[c.first + i] = c.po[i];
        c.dst_bo[c.first + i] = c.bo[i];
    }
    if (c.first == 0)
        for (int j = threadIdx.x; j < GUIDE_EXP; j += blockDim.x) {
            const Pair e = pair_of(exp(-(double)j / 32.0));
            c.dst_exps->h[j] = e.h;
            c.dst_exps->l[j] = e.l;
        }
    if (threadIdx.x == 0 && c.last_chunk) {
        c.dst_po[c.first + c.count] = c.po[c.count];
        c.dst_bo[c.first + c.count] = c.bo[c.count];
    }
}

__device__ __forceinline__ int find_frame(const int32_t *off, int n, int v)
{
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (__ldg(&off[mid]) <= v) lo = mid; else hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(256) bin_kernel(const __grid_constant__ GuideArgs a, int total_points)
{
    int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= total_points) return;
    int f = find_frame(a.point_offset, a.n_frames, gi);
    const SplineFrameDev &F = a.frames[f];
    int i = gi - __ldg(&a.point_offset[f]);
    // spline s with offsets[s] <= i < offsets[s+1]; the segment needs i+1 < offsets[s+1]
    int lo = 0, hi = F.n_splines;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (__ldg(&F.offsets[mid]) <= i) lo = mid; else hi = mid;
    }
    const bool starts = F.n_splines > 0 && i + 1 < F.n_points && i >= __ldg(&F.offsets[0]) &&
                        i + 1 < __ldg(&F.offsets[lo + 1]);
    const float2 A = __ldg(&F.pts[i]), B = starts ? __ldg(&F.pts[i + 1]) : A;
    float vx = __fsub_rn(B.x, A.x), vy = __fsub_rn(B.y, A.y);
    float l2 = __fadd_rn(__fmul_rn(vx, vx), __fmul_rn(vy, vy));
    if (!(l2 > 0.0f)) {
        F.segp[i].il32 = -1.0f;  // no segment starts here (bins that scan every point)
        return;
    }
    {
        // FP64 terms of this segment used by every pixel that picks it (same
        // expressions as a per-pixel evaluation, computed once)
        const double ax = A.x, ay = A.y;
        const double dvx = __dsub_rn((double)B.x, ax), dvy = __dsub_rn((double)B.y, ay);
        const double len = __dsqrt_rn(__dadd_rn(__dmul_rn(dvx, dvx), __dmul_rn(dvy, dvy)));
        double *s = F.seg64 + 8 * (size_t)i;
        const double il = __ddiv_rn(1.0, __dmul_rn(len, len));
        const double tx = __ddiv_rn(dvx, len), ty = __ddiv_rn(dvy, len);
        const float sw = F.weight ? __ldg(&F.weight[lo]) : 1.0f;
        s[0] = ax;
        s[1] = ay;
        s[2] = dvx;
        s[3] = dvy;
        s[4] = il;
        s[5] = tx;
        s[6] = ty;
        s[7] = (double)sw;
        const Pair px = pair_of(dvx), py = pair_of(dvy), pi = pair_of(il), tpx = pair_of(tx), tpy = pair_of(ty);
        float4 *d = reinterpret_cast<float4 *>(F.segp + i);
        d[0] = make_float4(A.x, A.y, px.h, py.h);  // px.h and py.h are vx and vy
        d[1] = make_float4(__fdiv_rn(1.0f, l2), px.l, py.l, pi.h);
        d[2] = make_float4(pi.l, tpx.h, tpx.l, tpy.h);
        d[3] = make_float4(tpy.l, sw, 0.f, 0.f);
    }
    float grow = 3.0f * a.eta + 1.0f;
    float xmin = fminf(A.x, B.x) - grow, xmax = fmaxf(A.x, B.x) + grow;
    float ymin = fminf(A.y, B.y) - grow, ymax = fmaxf(A.y, B.y) + grow;
    int bx0 = max(0, (int)floorf(xmin / BIN)), bx1 = min(F.NBX - 1, (int)floorf(xmax / BIN));
    int by0 = max(0, (int)floorf(ymin / BIN)), by1 = min(F.NBY - 1, (int)floorf(ymax / BIN));
    for (int by = by0; by <= by1; by++)
        for (int bx = bx0; bx <= bx1; bx++) {
            int b = by * F.NBX + bx;
            int pos = atomicAdd(&F.bin_count[b], 1);
            if (pos < BIN_CAP) F.bin_list[(size_t)b * BIN_CAP + pos] = i;
        }
}

// Squared distance from p to the segment a + [0, 1] v with 1/|v|^2 given, in FP32
// with the oracle's expression (no contraction): t = ((p - a).v) * (1/|v|^2)
// clamped to [0, 1], |p - a - t v|^2.
__device__ __forceinline__ float seg_d2(float px, float py, float ax, float ay, float vx, float vy, float inv_l2)
{
    const float wx = __fsub_rn(px, ax), wy = __fsub_rn(py, ay);
    const float dot = __fadd_rn(__fmul_rn(wx, vx), __fmul_rn(wy, vy));
    float t = __fmul_rn(dot, inv_l2);
    if (t < 0.0f) t = 0.0f;
    if (t > 1.0f) t = 1.0f;
    const float qx = __fsub_rn(wx, __fmul_rn(t, vx));
    const float qy = __fsub_rn(wy, __fmul_rn(t, vy));
    return __fadd_rn(__fmul_rn(qx, qx), __fmul_rn(qy, qy));
}

// Hole bits of four labels: bit c is set iff byte c of w is 1 (a hole label).
__device__ __forceinline__ uint32_t hole4(uint32_t w)
{
    const uint32_t r = __vcmpeq4(w, 0x01010101u);  // 0xff in every byte equal to 1
    return ((r >> 7) & 1u) | ((r >> 14) & 2u) | ((r >> 21) & 4u) | ((r >> 28) & 8u);
}

constexpr int GUIDE_WARPS = 8;
constexpr int STRIP = 8;  // rows of a bin per warp

struct GuideWarp {
    float4 av[32];          // segments staged: a.x, a.y, v.x, v.y
    float2 ilid[32];        // 1/|v|^2, segment index (as bits)
    short holes[BIN * STRIP];
    int seg[BIN * STRIP];   // the nearest segment of each hole pixel, -1: none within 3 eta
};

// The FP64 evaluation: t = ((x - a).v) / |v|^2 clamped, d^2 = |x - a - t v|^2, g = (v/|v|)
// e^(-d^2/(2 eta^2)), with the reciprocals 1/|v|^2 and 1/(2 eta^2) precomputed in FP64.
__device__ __noinline__ float2 guide_value64(const double *s, int x, int y, double k2)
{
    const double ax = __ldcg(&s[0]), ay = __ldcg(&s[1]), vx = __ldcg(&s[2]), vy = __ldcg(&s[3]);
    const double inv_l2 = __ldcg(&s[4]), tx = __ldcg(&s[5]), ty = __ldcg(&s[6]), sw = __ldcg(&s[7]);
    const double wx = __dsub_rn((double)x, ax), wy = __dsub_rn((double)y, ay);
    double t = __dmul_rn(__dadd_rn(__dmul_rn(wx, vx), __dmul_rn(wy, vy)), inv_l2);
    if (t < 0.0) t = 0.0;
    if (t > 1.0) t = 1.0;
    const double qx = __dsub_rn(wx, __dmul_rn(t, vx)), qy = __dsub_rn(wy, __dmul_rn(t, vy));
    const double d2 = __dadd_rn(__dmul_rn(qx, qx), __dmul_rn(qy, qy));
    const double ev = exp(-__dmul_rn(d2, k2));
    return make_float2((float)__dmul_rn(__dmul_rn(tx, ev), sw), (float)__dmul_rn(__dmul_rn(ty, ev), sw));
}

// The nearest segments of the strip's hole pixels, P per lane (pixels q = lane + 32 j),
// the segments in the outer loop so that each is read from shared memory once per lane.
template <int P>
__device__ __forceinline__ void nearest_segments(const GuideArgs &a, const SplineFrameDev &F, GuideWarp *gw, int b, int cnt,
                                             int x0, int y0, int nh, float4 box)
{
    const int lane = threadIdx.x & 31;
    float px[P], py[P], best[P];
    int bi[P];
#pragma unroll
    for (int j = 0; j < P; j++) {
        const int q = lane + 32 * j;
        const int e = q < nh ? gw->holes[q] : 0;
        px[j] = (float)(x0 + (e & (BIN - 1)));
        py[j] = (float)(y0 + (e >> 5));
        best[j] = INFINITY;
        bi[j] = 0x7fffffff;
    }
    // the bin's list, or every segment of the frame where that overflowed
    const bool listed = cnt <= BIN_CAP;
    const int total = listed ? cnt : F.n_points;
    for (int s0 = 0; s0 < total; s0 += 32) {
        __syncwarp();  // the previous segments have been read
        // only segments that come within 3 eta of the hole pixels' box matter (one more
        // px for FP32's rounding, as for the bins): about half of the bin's.  Beyond 2^20
        // px that is not enough: the end a + v and the distance that decides are each off
        // by a few 2^-24 of |v| and of the pixel's coordinates.
        bool keep = false;
        int i = 0;
        float4 S0 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s0 + lane < total) {
            i = listed ? __ldg(&F.bin_list[(size_t)b * BIN_CAP + s0 + lane]) : s0 + lane;
            S0 = __ldg(reinterpret_cast<const float4 *>(F.segp + i));
            const float ex = S0.x + S0.z, ey = S0.y + S0.w;
            const bool exact = fabsf(S0.z) + fabsf(S0.w) < 1048576.0f && fmaxf(box.y, box.w) < 1048576.0f;
            keep = !exact ||
                   !(fmaxf(S0.x, ex) < box.x || fminf(S0.x, ex) > box.y || fmaxf(S0.y, ey) < box.z ||
                     fminf(S0.y, ey) > box.w);
            if (!listed) keep = keep && __ldg(&F.segp[i].il32) >= 0.0f;  // points that start no segment
        }
        const unsigned km = __ballot_sync(0xffffffffu, keep);
        if (keep) {
            const int pos = __popc(km & ((1u << lane) - 1u));
            gw->av[pos] = S0;
            gw->ilid[pos] = make_float2(__ldg(&F.segp[i].il32), __int_as_float(i));
        }
        __syncwarp();
        const int m = __popc(km);
        for (int s = 0; s < m; s++) {
            const float4 S = gw->av[s];
            const float2 t = gw->ilid[s];
            const int id = __float_as_int(t.y);
#pragma unroll
            for (int j = 0; j < P; j++) {
                const float d2 = seg_d2(px[j], py[j], S.x, S.y, S.z, S.w, t.x);
                if (d2 < best[j] || (d2 == best[j] && id < bi[j])) {
                    best[j] = d2;
                    bi[j] = id;
                }
            }
        }
    }
    const float t3 = 3.0f * a.eta;
    const float thr = __fmul_rn(t3, t3);
#pragma unroll
    for (int j = 0; j < P; j++)
        if (lane + 32 * j < nh)
            gw->seg[lane + 32 * j] = bi[j] != 0x7fffffff && best[j] <= thr ? bi[j] : -1;
}

// One CTA per eight bins, in 32 strips of STRIP rows.  Lane 8 c + r of a warp reads row r
// of a strip (two 16-byte loads where the row is aligned and inside the frame) into a
// 32-bit hole mask; a CTA without hole pixels, most of them, ends there.  The strips with
// hole pixels are then taken by the warps one at a time (dense strips cost several times
// sparse ones).  The value is evaluated in one place: unrolled per pixel, it made the
// kernel wait for instructions 40 % of the time.
__global__ void __launch_bounds__(32 * GUIDE_WARPS, 4) guide_kernel(const __grid_constant__ GuideArgs a)
{
    constexpr int PER = BIN / STRIP;                 // strips of a bin
    constexpr int ITEMS = 4 * GUIDE_WARPS;           // strips of a CTA
    constexpr int BINS = ITEMS / PER;
    __shared__ GuideWarp s_warp[GUIDE_WARPS];
    __shared__ uint32_t s_mask[ITEMS][STRIP];
    __shared__ int s_frame[ITEMS];
    __shared__ short s_list[ITEMS];
    __shared__ int s_n, s_next;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) s_n = s_next = 0;
    __syncthreads();
    {
        const int item = warp * 4 + (lane >> 3);     // strip item / BINS of bin item % BINS
        const int gb = blockIdx.x * BINS + item % BINS;
        uint32_t hm = 0u;
        int f = 0;
        if (gb < a.total_bins) {
            f = find_frame(a.bin_offset, a.n_frames, gb);
            const SplineFrameDev &F = a.frames[f];
            const int b = gb - __ldg(&a.bin_offset[f]);
            const int W = F.W, bx = b % F.NBX, by = b / F.NBX;
            const int x0 = bx * BIN, y = by * BIN + item / BINS * STRIP + (lane & 7);
            if (y < F.H) {
                const uint8_t *row = F.labels + (size_t)y * W + x0;
                if (x0 + BIN <= W && (reinterpret_cast<uintptr_t>(row) & 15u) == 0) {
                    const uint4 q0 = __ldg(reinterpret_cast<const uint4 *>(row));
                    const uint4 q1 = __ldg(reinterpret_cast<const uint4 *>(row) + 1);
                    hm = hole4(q0.x) | (hole4(q0.y) << 4) | (hole4(q0.z) << 8) | (hole4(q0.w) << 12) |
                         (hole4(q1.x) << 16) | (hole4(q1.y) << 20) | (hole4(q1.z) << 24) | (hole4(q1.w) << 28);
                } else {
                    for (int c = 0; c < BIN && x0 + c < W; c++)
                        if (__ldg(&row[c]) == 1) hm |= 1u << c;
                }
            }
        }
        const unsigned some = __ballot_sync(0xffffffffu, hm != 0u) & (0xffu << (lane & 24));
        if (some) {
            s_mask[item][lane & 7] = hm;
            if ((lane & 7) == 0) {
                s_frame[item] = f;
                s_list[atomicAdd(&s_n, 1)] = (short)item;
            }
        }
    }
    __syncthreads();
    const int n = s_n;
    GuideWarp *gw = &s_warp[warp];
    for (;;) {
        int it = 0;
        if (lane == 0) it = n > 0 ? atomicAdd(&s_next, 1) : n;
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= n) break;
        const int item = s_list[it];
        const int f = s_frame[item];
        const SplineFrameDev &F = a.frames[f];
        const int b = blockIdx.x * BINS + item % BINS - __ldg(&a.bin_offset[f]);
        const int x0 = b % F.NBX * BIN, y0 = b / F.NBX * BIN + item / BINS * STRIP;
        const int cnt = __ldg(&F.bin_count[b]);
        // the hole pixels, row-major: lane l tests column l of each row
        int nh = 0;
        uint32_t cols = 0, rows = 0;
#pragma unroll
        for (int r = 0; r < STRIP; r++) {
            const uint32_t m = s_mask[item][r];
            cols |= m;
            rows |= m ? 1u << r : 0u;
            if ((m >> lane) & 1u) gw->holes[nh + __popc(m & ((1u << lane) - 1u))] = (short)((r << 5) | lane);
            nh += __popc(m);
        }
        __syncwarp();
        const float grow = 3.0f * a.eta + 1.0f;
        const float4 box = make_float4((float)(x0 + __ffs(cols) - 1) - grow, (float)(x0 + 31 - __clz(cols)) + grow,
                                       (float)(y0 + __ffs(rows) - 1) - grow, (float)(y0 + 31 - __clz(rows)) + grow);
        if (nh <= 32) nearest_segments<1>(a, F, gw, b, cnt, x0, y0, nh, box);
        else if (nh <= 64) nearest_segments<2>(a, F, gw, b, cnt, x0, y0, nh, box);
        else if (nh <= 128) nearest_segments<4>(a, F, gw, b, cnt, x0, y0, nh, box);
        else nearest_segments<8>(a, F, gw, b, cnt, x0, y0, nh, box);
#pragma unroll 1
        for (int q = lane; q < nh; q += 32) {
            const int e = gw->holes[q], sgi = gw->seg[q];
            const int x = x0 + (e & (BIN - 1)), y = y0 + (e >> 5);
            float2 out = make_float2(0.0f, 0.0f);
            if (sgi >= 0) {
                SegPair sp;
                const float4 *d = reinterpret_cast<const float4 *>(F.segp + sgi);
                float4 *o = reinterpret_cast<float4 *>(&sp);
#pragma unroll
                for (int i = 0; i < 4; i++) o[i] = __ldg(&d[i]);
                // coordinates that FP32 does not hold go the FP64 way
                const bool sure = max(x, y) < (1 << 24) &&
                                  guide_value((float)x, (float)y, sp, a.k2p, a.ieta, *a.exps, out.x, out.y);
                if (!sure) out = guide_value64(F.seg64 + 8 * (size_t)sgi, x, y, a.k2);
            }
            F.guide[(size_t)y * F.W + x] = out;
        }
        __syncwarp();  // the strip's pixels have been read
    }
}

// g = |g| (cos phi, sin phi) at hole pixels, evaluated in FP64 and rounded once
// (so a CPU evaluation in FP64 gives the same FP32 field).
__global__ void __launch_bounds__(256) angle_kernel(int64_t npx, const uint8_t *labels, const float *mag,
                                                    const float *phi, float2 *guide)
{
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < npx; p += (int64_t)gridDim.x * blockDim.x) {
        if (__ldg(&labels[p]) != 1) continue;
        double m = (double)__ldg(&mag[p]), a = (double)__ldg(&phi[p]);
        guide[p] = make_float2((float)__dmul_rn(m, cos(a)), (float)__dmul_rn(m, sin(a)));
    }
}

}  // namespace gf
