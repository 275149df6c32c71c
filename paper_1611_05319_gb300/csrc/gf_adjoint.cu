// Adjoint of the Guidefill fill (reverse sweep over the steps) for sm_103a.
//
// Differentiates the fill as a map of the known colours, the guidance angle
// field (|g| fixed) and mu, with the step of every pixel, the stall steps and
// every ghost sample's tap set held fixed (they are piecewise constant).  The
// forward's shell map reconstructs every D^(k) (readable at step k iff
// (uint)(s+1) < (uint)(k+1)), so no other forward state is stored.
//
// For a pixel x filled at step k with normalised weights wh_s over its
// readable samples and bilinear values v_s (Algorithm 1, eq. bilinearDef):
//   grad_in[t]  += wh_s * L_t * ubar(x)           for every tap t of sample s
//   grad_phi(x)  = ubar(x) . sum_s wh_s dv_s/dphi  (dp_s/dphi = n gh_perp - m gh)
//   grad_mu     += ubar(x) . sum_s wh_s (lam_s - lam_bar) v_s,
//                  lam_s = d ln w_s / d mu = -mu |g|^2 m^2 / eps^2  (eq. weight)
// Steps run K-1 .. 0; a pixel's ubar is final once every later step (the only
// readers of its value) has scattered into it.
//
// Kernels: adj_prep_kernel (per pixel: copy grad_out -> grad_in, clear
// grad_phi, histogram of shell indices, K), adj_scan_kernel (per frame: step
// offsets), adj_scatter_kernel (per pixel: pixel lists per step),
// adj_kernel (persistent: one cluster per frame, one cluster barrier per step).
//
// adj_kernel is bound by the dependent chain of each step, not by bandwidth.  All
// of a step but ubar is known beforehand (the shell map, the guide field and the
// output image do not change), so between arriving at a step's barrier and waiting
// on it each warp reads the next step's first pixels, packs the readable bits
// around each into row words in shared memory (one load per cell instead of up to
// eight per sample in two passes) and forms the weights' sum; after the barrier
// ubar is the only load ahead of the scatter.  Samples go in mirror pairs as in the
// fill.  16 frames of 512 x 512 (54 steps): 1,626 us -> 492 us.

#include <cooperative_groups.h>

#include "gf_internal.cuh"

namespace cg = cooperative_groups;

namespace gf {

constexpr unsigned AFULL = 0xffffffffu;

__device__ __forceinline__ int adj_find(const int32_t *off, int n, long long v)
{
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if ((long long)__ldg(&off[mid]) <= v) lo = mid; else hi = mid;
    }
    return lo;
}

__global__ void adj_upload_kernel(const __grid_constant__ AdjChunk c)
{
    for (int i = threadIdx.x; i < c.count; i += blockDim.x) {
        c.dst_frames[c.first + i] = c.frames[i];
        c.dst_blk[c.first + i] = c.blk[i];
    }
    for (int i = threadIdx.x; i < c.count; i += blockDim.x) *c.frames[i].grad_mu = 0.0f;
    if (threadIdx.x == 0 && c.last_chunk) c.dst_blk[c.first + c.count] = c.blk[c.count];
}

// One CTA per block of 1024 pixels of a frame; each thread takes four of them, 256
// apart.  The histogram's atomics are made once per warp and value (a frame's first
// shells hold thousands of pixels, and their counters are single addresses): 126 ->
// 27 us on 16 frames of 512 x 512.
__global__ void __launch_bounds__(256) adj_prep_kernel(const __grid_constant__ AdjArgs a)
{
    const int f = adj_find(a.blk_offset, a.n_frames, blockIdx.x);
    const AdjFrameDev &F = a.frames[f];
    const long long base = (long long)((int)blockIdx.x - __ldg(&a.blk_offset[f])) * 1024 + threadIdx.x;
    const long long np = (long long)F.H * F.W;
    const bool copy = F.grad_in != F.grad_out;
    const int lane = threadIdx.x & 31;
    int s[4];
    float4 g[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const long long p = base + 256 * i;
        s[i] = p < np ? __ldg(&F.shell[p]) : -1;
        if (copy && p < np) g[i] = __ldg(&F.grad_out[p]);
    }
    int top = -1;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const long long p = base + 256 * i;
        if (p < np) {
            if (copy) F.grad_in[p] = g[i];
            F.grad_phi[p] = 0.0f;
        }
        top = max(top, s[i]);
        if (__any_sync(AFULL, s[i] >= 0)) {
            const unsigned same = __match_any_sync(AFULL, s[i]);
            if (s[i] >= 0 && (__ffs(same) - 1) == lane) atomicAdd(&F.cnt[s[i]], __popc(same));
        }
    }
    top = __reduce_max_sync(AFULL, top);
    if (lane == 0 && top >= 0) atomicMax(F.K, top + 1);
}

// one CTA per frame: exclusive scan of cnt[0..K) into start[0..K], cursor = start
__global__ void __launch_bounds__(1024) adj_scan_kernel(const __grid_constant__ AdjArgs a)
{
    const AdjFrameDev &F = a.frames[blockIdx.x];
    const int K = __ldcg(F.K);
    __shared__ int carry;
    __shared__ int wsum[32];
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int base = 0; base < K; base += 1024) {
        int i = base + threadIdx.x;
        int v = i < K ? __ldcg(&F.cnt[i]) : 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(AFULL, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[w] = x;
        __syncthreads();
        if (w == 0) {
            int s = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int y = __shfl_up_sync(AFULL, s, o);
                if (lane >= o) s += y;
            }
            wsum[lane] = s;
        }
        __syncthreads();
        int excl = carry + (w > 0 ? wsum[w - 1] : 0) + x - v;
        if (i < K) {
            F.start[i] = excl;
            F.cnt[i] = excl;  // becomes the scatter cursor
        }
        __syncthreads();
        if (threadIdx.x == 1023) carry = excl + v;
        __syncthreads();
    }
    if (threadIdx.x == 0) F.start[K] = carry;
}

__global__ void __launch_bounds__(256) adj_scatter_kernel(const __grid_constant__ AdjArgs a)
{
    const int f = adj_find(a.blk_offset, a.n_frames, blockIdx.x);
    const AdjFrameDev &F = a.frames[f];
    const long long base = (long long)((int)blockIdx.x - __ldg(&a.blk_offset[f])) * 1024 + threadIdx.x;
    const long long np = (long long)F.H * F.W;
    const int lane = threadIdx.x & 31;
    int s[4];
#pragma unroll
    for (int i = 0; i < 4; i++) s[i] = base + 256 * i < np ? __ldg(&F.shell[base + 256 * i]) : -1;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        if (!__any_sync(AFULL, s[i] >= 0)) continue;
        const unsigned same = __match_any_sync(AFULL, s[i]);
        const int first = __ffs(same) - 1;
        int pos = 0;
        if (s[i] >= 0 && first == lane) pos = atomicAdd(&F.cnt[s[i]], __popc(same));
        pos = __shfl_sync(AFULL, pos, first);
        if (s[i] >= 0) F.order[pos + __popc(same & ((1u << lane) - 1u))] = (int32_t)(base + 256 * i);
    }
}

__device__ __forceinline__ bool tap_readable(const AdjFrameDev &F, int x, int y, int k)
{
    if (x < 0 || y < 0 || x >= F.W || y >= F.H) return false;
    return readable_at(__ldg(&F.shell[(size_t)y * F.W + x]), k);
}

struct SampleGeo {
    int ix, iy;        // cell corner (absolute)
    float frx, fry;    // fractional offsets (0 along a single-tap axis)
    bool ok;
};

__device__ __forceinline__ SampleGeo sample_geo(const AdjArgs &a, const AdjFrameDev &F, int x, int y, float nf,
                                                float mf, float ch, float sh, bool rot, int k)
{
    float ox, oy;
    if (rot) {
        ox = __fsub_rn(__fmul_rn(nf, ch), __fmul_rn(mf, sh));
        oy = __fadd_rn(__fmul_rn(nf, sh), __fmul_rn(mf, ch));
        float r0 = rintf(ox);
        if (fabsf(__fsub_rn(ox, r0)) <= a.tau) ox = r0;
        r0 = rintf(oy);
        if (fabsf(__fsub_rn(oy, r0)) <= a.tau) oy = r0;
    } else {
        ox = nf;
        oy = mf;
    }
    const float flx = floorf(ox), fly = floorf(oy);
    SampleGeo g;
    g.frx = __fsub_rn(ox, flx);
    g.fry = __fsub_rn(oy, fly);
    g.ix = x + (int)flx;
    g.iy = y + (int)fly;
    bool ok = tap_readable(F, g.ix, g.iy, k);
    if (g.frx > 0.f) ok = ok && tap_readable(F, g.ix + 1, g.iy, k);
    if (g.fry > 0.f) {
        ok = ok && tap_readable(F, g.ix, g.iy + 1, k);
        if (g.frx > 0.f) ok = ok && tap_readable(F, g.ix + 1, g.iy + 1, k);
    }
    g.ok = ok;
    return g;
}

__device__ __forceinline__ float4 operator-(float4 a, float4 b)
{
    return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
__device__ __forceinline__ float dot4(float4 a, float4 b) { return a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w; }

__device__ __forceinline__ void red_add4(float4 *p, float4 v)
{
    atomicAdd(p, v);
}

// G lanes process pixel x of step k, every tap's readability read from the shell map:
// the pixels whose rotation is not one (|g| of a few denormals, or not finite).  Must
// be called by all 32 lanes.
__device__ __noinline__ void adj_pixel_general(const AdjArgs &a, const AdjFrameDev &F, int p, int k, bool stall, bool act, int G,
                          int j, double &mu_acc)
{
    const int x = p % F.W, y = p / F.W;
    float4 ub = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 g = make_float2(0.f, 0.f);
    if (act) {
        ub = __ldcg(&F.grad_in[p]);
        if (!stall) g = __ldg(&F.guide[p]);
    }
    float ch = 1.f, sh = 0.f, beta = 0.f, a2 = 0.f;
    const bool rot = !stall;
    if (!stall) {
        a2 = __fadd_rn(__fmul_rn(g.x, g.x), __fmul_rn(g.y, g.y));
        float aa = __fsqrt_rn(a2);
        if (aa > 0.f) {
            ch = __fdiv_rn(g.x, aa);
            sh = __fdiv_rn(g.y, aa);
        }
        beta = a.coef32 * a2;
    }
    const bool has_dir = rot && __fsqrt_rn(a2) > 0.f;  // g = 0: unrotated ball, no angle dependence
    // pass 1: readable inverse distances per |m| group
    const int R = a.tab.R;
    float accg[MAX_R + 1];
#pragma unroll
    for (int gi = 0; gi <= MAX_R; gi++) accg[gi] = 0.f;
    if (act) {
#pragma unroll
        for (int gi = 0; gi <= MAX_R; gi++) {
            if (gi > R) break;
            for (int s = a.tab.m_start[gi] + j; s < a.tab.m_start[gi + 1]; s += G) {
                SampleGeo sg = sample_geo(a, F, x, y, a.tab.n_f[s], a.tab.m_f[s], ch, sh, rot, k);
                if (sg.ok) accg[gi] += a.tab.invd[s];
            }
        }
    }
#pragma unroll
    for (int gi = 0; gi <= MAX_R; gi++)
        for (int o = 1; o < G; o <<= 1) accg[gi] += __shfl_xor_sync(AFULL, accg[gi], o);
    int m0 = MAX_R + 1;
#pragma unroll
    for (int gi = MAX_R; gi >= 0; gi--)
        if (accg[gi] > 0.f) m0 = gi;
    float Wn = 0.f;
#pragma unroll
    for (int gi = 0; gi <= MAX_R; gi++)
        if (accg[gi] > 0.f) Wn += expf(-beta * (float)(gi * gi - m0 * m0)) * accg[gi];
    const float invW = Wn > 0.f ? 1.f / Wn : 0.f;
    // pass 2: scatter, angle and mu terms
    const float lam_scale = a.mu > 0.f ? -2.f * a.coef32 / a.mu * a2 : 0.f;  // lam_s = lam_scale * m^2
    float S1 = 0.f, S2 = 0.f, S3 = 0.f, S4 = 0.f;
    if (act && Wn > 0.f) {
        for (int gi = 0; gi <= R; gi++) {
            const float wg = expf(-beta * (float)(gi * gi - m0 * m0)) * invW;
            const float lam = lam_scale * (float)(gi * gi);
            for (int s = a.tab.m_start[gi] + j; s < a.tab.m_start[gi + 1]; s += G) {
                const float nf = a.tab.n_f[s], mf = a.tab.m_f[s];
                SampleGeo sg = sample_geo(a, F, x, y, nf, mf, ch, sh, rot, k);
                if (!sg.ok) continue;
                const float wh = wg * a.tab.invd[s];
                const size_t b = (size_t)sg.iy * F.W + sg.ix;
                const float fx = sg.frx, fy = sg.fry;
                const bool ax = fx > 0.f, ay = fy > 0.f;
                const float4 c00 = __ldg(&F.out[b]);
                const float4 c10 = ax ? __ldg(&F.out[b + 1]) : c00;
                const float4 c01 = ay ? __ldg(&F.out[b + F.W]) : c00;
                const float4 c11 = (ax && ay) ? __ldg(&F.out[b + F.W + 1]) : c00;
                const float wx0 = 1.f - fx, wx1 = fx, wy0 = 1.f - fy, wy1 = fy;
                // value v_s . ubar and its derivative along x and y
                const float d00 = dot4(c00, ub), d10 = dot4(c10, ub), d01 = dot4(c01, ub), d11 = dot4(c11, ub);
                float vu = wx0 * wy0 * d00;
                if (ax) vu += wx1 * wy0 * d10;
                if (ay) vu += wx0 * wy1 * d01;
                if (ax && ay) vu += wx1 * wy1 * d11;
                float gx_ = 0.f, gy_ = 0.f;
                if (ax) gx_ = wy0 * (d10 - d00) + (ay ? wy1 * (d11 - d01) : 0.f);
                if (ay) gy_ = wx0 * (d01 - d00) + (ax ? wx1 * (d11 - d10) : 0.f);
                if (has_dir) {
                    const float dpx = -nf * sh - mf * ch, dpy = nf * ch - mf * sh;
                    S4 += wh * (gx_ * dpx + gy_ * dpy);
                }
                S1 += wh * lam * vu;
                S2 += wh * lam;
                S3 += wh * vu;
                // scatter wh * L_t * ubar into the taps
                float l = wh * wx0 * wy0;
                red_add4(&F.grad_in[b], make_float4(l * ub.x, l * ub.y, l * ub.z, l * ub.w));
                if (ax) {
                    l = wh * wx1 * wy0;
                    red_add4(&F.grad_in[b + 1], make_float4(l * ub.x, l * ub.y, l * ub.z, l * ub.w));
                }
                if (ay) {
                    l = wh * wx0 * wy1;
                    red_add4(&F.grad_in[b + F.W], make_float4(l * ub.x, l * ub.y, l * ub.z, l * ub.w));
                    if (ax) {
                        l = wh * wx1 * wy1;
                        red_add4(&F.grad_in[b + F.W + 1], make_float4(l * ub.x, l * ub.y, l * ub.z, l * ub.w));
                    }
                }
            }
        }
    }
    for (int o = 1; o < G; o <<= 1) {
        S1 += __shfl_xor_sync(AFULL, S1, o);
        S2 += __shfl_xor_sync(AFULL, S2, o);
        S3 += __shfl_xor_sync(AFULL, S3, o);
        S4 += __shfl_xor_sync(AFULL, S4, o);
    }
    if (act && j == 0) {
        F.grad_phi[p] = has_dir ? S4 : 0.f;
        F.grad_in[p] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!stall) mu_acc += (double)(S1 - S2 * S3);
    }
}

// Per-warp shared memory: for each pixel of a batch (32 / G of them) the readable bits
// of rows -RR .. RR around it (bit dx + RR) and its group weights.
constexpr int ADJ_SLOTS = 16;  // pixels per warp and batch: two lanes each at least
template <int RR>
struct AdjWarp {
    uint32_t row[ADJ_SLOTS][2 * RR + 1];
    float eg[ADJ_SLOTS][MAX_R + 1];
};

// What is known of a pixel before its step: everything but ubar.
struct AdjPix {
    int p;          // pixel, -1: none
    float ch, sh;   // rotation
    float a2;       // |g|^2
    float inv;      // 1 / sum of the readable weights, 0 when there is none
    float4 u;       // the pixel's own output (0 when it is not finite)
    int least;      // smallest readable |m|
    bool rot;       // not a stall step
    bool odd;       // to be done by adj_pixel_general
};

// A mirror pair's cell: offset o = (n, m) rotated, snapped; its floor and fraction,
// and the readability of the sample and of its mirror image.
template <int RR>
struct AdjCell {
    int fx, fy;
    float frx, fry;
    bool hx, hy, ok1, ok2;
    __device__ __forceinline__ AdjCell(const uint32_t *row, float n, float m, float ch, float sh, float tau)
    {
        const float ox = __fsub_rn(__fmul_rn(n, ch), __fmul_rn(m, sh));
        const float oy = __fadd_rn(__fmul_rn(n, sh), __fmul_rn(m, ch));
        // to the lattice by adding 1.5 * 2^23; the difference to the nearest integer is exact
        const float tx = ox + 12582912.0f, ty = oy + 12582912.0f;
        const float dx = ox - (tx - 12582912.0f), dy = oy - (ty - 12582912.0f);
        hx = fabsf(dx) > tau;
        hy = fabsf(dy) > tau;
        const bool lx = dx < -tau, ly = dy < -tau;
        frx = lx ? dx + 1.0f : (hx ? dx : 0.0f);
        fry = ly ? dy + 1.0f : (hy ? dy : 0.0f);
        fx = __float_as_int(tx) - 0x4b400000 - (lx ? 1 : 0);
        fy = __float_as_int(ty) - 0x4b400000 - (ly ? 1 : 0);
        const uint32_t need = hx ? 3u : 1u;
        const int e = hy ? 1 : 0, iy = RR + fy, jy = RR - fy;
        const uint32_t m1 = row[iy] & row[iy + e], m2 = row[jy] & row[jy - e];
        ok1 = ((m1 >> (RR + fx)) & need) == need;
        ok2 = ((m2 >> (RR - fx - (hx ? 1 : 0))) & need) == need;
    }
};

// The part of a batch that does not depend on ubar: lane group grp takes entry
// base + grp of the step's list.  Called by all 32 lanes.
template <int RR>
__device__ __forceinline__ AdjPix adj_prepare(const AdjArgs &a, const AdjFrameDev &F, AdjWarp<RR> *aw, const float4 *pairs,
                                              int first, int last, int k, bool stall, int G, int grp, int j)
{
    constexpr int N = 2 * RR + 1;
    AdjPix px;
    const int q = first + grp;
    const bool act = q < last;
    px.p = act ? __ldg(&F.order[q]) : -1;
    px.rot = !stall;
    px.a2 = 0.f;
    px.ch = 1.f;
    px.sh = 0.f;
    px.inv = 0.f;
    px.least = 0;
    px.u = make_float4(0.f, 0.f, 0.f, 0.f);
    px.odd = false;
    const int W = F.W, H = F.H, R = a.tab.R;
    __syncwarp();  // the previous batch's rows and weights have been read
    float beta = 0.f;
    if (act) {
        const int x = px.p % W, y = px.p / W;
        float2 g = make_float2(0.f, 0.f);
        if (!stall) g = __ldg(&F.guide[px.p]);
        px.u = __ldg(&F.out[px.p]);
        if (!(fabsf(px.u.x) + fabsf(px.u.y) + fabsf(px.u.z) + fabsf(px.u.w) < INFINITY))
            px.u = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int r = j; r < N; r += G) {
            const int yy = y + r - RR;
            const bool rin = yy >= 0 && yy < H;
            const int32_t *sp = F.shell + (size_t)(rin ? yy : 0) * W + (x - RR);
            uint32_t m = 0;
#pragma unroll
            for (int c = 0; c < N; c++) {
                const bool in = rin && x - RR + c >= 0 && x - RR + c < W;
                const int32_t v = in ? __ldg(sp + c) : SH_OUTSIDE;
                m |= readable_at(v, k) ? 1u << c : 0u;
            }
            aw->row[grp][r] = m;
        }
        if (!stall) {
            px.a2 = __fadd_rn(__fmul_rn(g.x, g.x), __fmul_rn(g.y, g.y));
            const float aa = __fsqrt_rn(px.a2);
            if (aa > 0.f) {
                px.ch = __fdiv_rn(g.x, aa);
                px.sh = __fdiv_rn(g.y, aa);
            }
            beta = a.coef32 * px.a2;
            px.odd = aa > 0.f && !(__fmaf_rn(px.ch, px.ch, __fmul_rn(px.sh, px.sh)) <= 1.0000005f);
            px.odd = px.odd || !(aa < INFINITY);
        }
        for (int g2 = j; g2 <= R; g2 += G) aw->eg[grp][g2] = expf(-(beta * (float)(g2 * g2)));
    }
    __syncwarp();
    const int npair = a.tab.ns >> 1;
    const bool go = act && !px.odd;
    float S = 0.f;
    int least = MAX_R + 1;  // smallest readable |m|
    auto sum = [&]() {
        S = 0.f;
        if (go)
            for (int i = j; i < npair; i += G) {
                const float4 t = pairs[i];  // n, m, 1/|(n, m)|, |m|
                const AdjCell<RR> c(aw->row[grp], t.x, t.y, px.ch, px.sh, a.tau);
                const int g2 = __float_as_int(t.w);
                const float w = aw->eg[grp][g2] * t.z;
                if (c.ok1) S += w;
                if (c.ok2) S += w;
                if (c.ok1 || c.ok2) least = min(least, g2);
            }
        for (int o = 1; o < G; o <<= 1) {
            S += __shfl_xor_sync(AFULL, S, o);
            least = min(least, __shfl_xor_sync(AFULL, least, o));
        }
    };
    sum();
    // weights that all underflow: relative to the smallest readable exponent
    const bool shift = go && least <= R && !(S >= 1e-18f);
    if (__any_sync(AFULL, shift)) {
        if (shift)
            for (int g2 = j; g2 <= R; g2 += G)
                aw->eg[grp][g2] = expf(-(beta * (float)(g2 * g2 - least * least)));
        __syncwarp();
        sum();
    }
    px.inv = S > 0.f ? 1.f / S : 0.f;
    px.least = least;
    return px;
}

// Scatter, angle and mu terms of a prepared batch.  Called by all 32 lanes.
template <int RR>
__device__ __forceinline__ void adj_apply(const AdjArgs &a, const AdjFrameDev &F, const AdjWarp<RR> *aw, const float4 *pairs,
                                          const AdjPix &px, int k, int G, int grp, int j, double &mu_acc)
{
    if (__any_sync(AFULL, px.odd)) {  // whole batch: rare
        adj_pixel_general(a, F, px.p < 0 ? 0 : px.p, k, !px.rot, px.p >= 0, G, j, mu_acc);
        return;
    }
    const bool act = px.p >= 0;
    float4 ub = make_float4(0.f, 0.f, 0.f, 0.f);
    if (act) ub = __ldcg(&F.grad_in[px.p]);
    const bool has_dir = px.rot && px.a2 > 0.f && __fsqrt_rn(px.a2) > 0.f;  // g = 0: no angle dependence
    const float lam_scale = a.mu > 0.f ? -2.f * a.coef32 / a.mu * px.a2 : 0.f;  // lam_s = lam_scale * m^2
    const int W = F.W, npair = a.tab.ns >> 1;
    float S1 = 0.f, S2 = 0.f, S3 = 0.f, S4 = 0.f;
    if (act && px.inv > 0.f) {
        for (int i = j; i < npair; i += G) {
            const float4 t = pairs[i];
            const AdjCell<RR> c(aw->row[grp], t.x, t.y, px.ch, px.sh, a.tau);
            if (!c.ok1 && !c.ok2) continue;
            const int g2 = __float_as_int(t.w);
            const float wh = aw->eg[grp][g2] * t.z * px.inv;
            // a constant in lam cancels in S1 - S2 S3: taken off here, it costs no digits
            const float lam = lam_scale * (float)(g2 * g2 - px.least * px.least);
            const float gx = 1.f - c.frx, gy = 1.f - c.fry;
            const float dpx = -t.x * px.sh - t.y * px.ch, dpy = t.x * px.ch - t.y * px.sh;
            const ptrdiff_t o = (ptrdiff_t)c.fy * W + c.fx;
            // the sample, then its mirror image: taps at +-(o, o + 1, o + W, o + W + 1)
            float4 v[2][4];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const bool ok = h ? c.ok2 : c.ok1;
                const ptrdiff_t sg = h ? -1 : 1;
                const float4 *b = F.out + px.p + sg * o;
                const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                v[h][0] = ok ? __ldg(b) : z;
                v[h][1] = ok && c.hx ? __ldg(b + sg) : v[h][0];
                v[h][2] = ok && c.hy ? __ldg(b + sg * W) : v[h][0];
                v[h][3] = ok && c.hx && c.hy ? __ldg(b + sg * (W + 1)) : v[h][0];
            }
#pragma unroll
            for (int h = 0; h < 2; h++) {
                if (!(h ? c.ok2 : c.ok1)) continue;
                // relative to the pixel's own value, the average of the samples: constants
                // cancel in the angle and mu terms, and taken off first they cost no digits
                const float d00 = dot4(v[h][0] - px.u, ub), d10 = dot4(v[h][1] - px.u, ub),
                            d01 = dot4(v[h][2] - px.u, ub), d11 = dot4(v[h][3] - px.u, ub);
                float vu = gx * gy * d00;
                if (c.hx) vu += c.frx * gy * d10;
                if (c.hy) vu += gx * c.fry * d01;
                if (c.hx && c.hy) vu += c.frx * c.fry * d11;
                float ex = 0.f, ey = 0.f;
                if (c.hx) ex = gy * (d10 - d00) + (c.hy ? c.fry * (d11 - d01) : 0.f);
                if (c.hy) ey = gx * (d01 - d00) + (c.hx ? c.frx * (d11 - d10) : 0.f);
                if (has_dir) S4 += wh * (ex * dpx + ey * dpy);
                S1 += wh * lam * vu;
                S2 += wh * lam;
                S3 += wh * vu;
                // scatter wh * L_t * ubar into the taps
                const ptrdiff_t sg = h ? -1 : 1;
                float4 *b = F.grad_in + px.p + sg * o;
                float l = wh * gx * gy;
                red_add4(b, make_float4(l * ub.x, l * ub.y, l * ub.z, l * ub.w));
                if (c.hx) {
                    l = wh * c.frx * gy;
                    red_add4(b + sg, make_float4(l * ub.x, l * ub.y, l * ub.z, l * ub.w));
                }
                if (c.hy) {
                    l = wh * gx * c.fry;
                    red_add4(b + sg * W, make_float4(l * ub.x, l * ub.y, l * ub.z, l * ub.w));
                    if (c.hx) {
                        l = wh * c.frx * c.fry;
                        red_add4(b + sg * (W + 1), make_float4(l * ub.x, l * ub.y, l * ub.z, l * ub.w));
                    }
                }
            }
        }
    }
    for (int o = 1; o < G; o <<= 1) {
        S1 += __shfl_xor_sync(AFULL, S1, o);
        S2 += __shfl_xor_sync(AFULL, S2, o);
        S3 += __shfl_xor_sync(AFULL, S3, o);
        S4 += __shfl_xor_sync(AFULL, S4, o);
    }
    if (act && j == 0) {
        F.grad_phi[px.p] = has_dir ? S4 : 0.f;
        F.grad_in[px.p] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (px.rot) mu_acc += (double)(S1 - S2 * S3);
    }
}

template <int RR>
__global__ void __launch_bounds__(CTA_THREADS, 1) adj_kernel(const __grid_constant__ AdjArgs a)
{
    __shared__ AdjFrameDev s_frame;
    __shared__ float4 s_pairs[MAX_SAMPLES / 2];
    extern __shared__ __align__(16) unsigned char adj_smem[];
    AdjWarp<RR> *aw = reinterpret_cast<AdjWarp<RR> *>(adj_smem) + (threadIdx.x >> 5);
    cg::cluster_group cluster = cg::this_cluster();
    const int crank = (int)cluster.block_rank();
    const int csize = (int)cluster.num_blocks();
    const int cid = blockIdx.x / csize;
    const int lane = threadIdx.x & 31;
    const int gw = (threadIdx.x >> 5) * csize + crank;
    const int nw = csize * WARPS_PER_CTA;
    int32_t *slot = a.cluster_frame + 2 * cid;
    for (int i = threadIdx.x; i < a.tab.ns; i += blockDim.x) {
        // the first half of every |m| group holds one sample of each mirror pair
        const int g = (int)fabsf(a.tab.m_f[i]);
        const int g0 = a.tab.m_start[g], half = (a.tab.m_start[g + 1] - g0) >> 1;
        if (i - g0 < half)
            s_pairs[(g0 >> 1) + (i - g0)] = make_float4(a.tab.n_f[i], a.tab.m_f[i], a.tab.invd[i], __int_as_float(g));
    }
    for (int it = 0;; it++) {
        cluster.sync();
        if (crank == 0 && threadIdx.x == 0) slot[it & 1] = atomicAdd(a.frame_cursor, 1);
        cluster.sync();
        const int f = __ldcg(&slot[it & 1]);
        if (f >= a.n_frames) break;
        if (threadIdx.x == 0) s_frame = a.frames[f];
        __syncthreads();
        const AdjFrameDev &F = s_frame;
        const int K = __ldcg(F.K);
        double mu_acc = 0.0;  // signed terms of all of the frame's pixels
        // step k's first batch, prepared while the barrier of step k + 1 is pending
        int b0 = 0, b1 = 0, G = 2, per = 16, grp = 0, j = 0;
        bool stall = false;
        AdjPix px;
        auto prepare = [&](int k) {
            b0 = __ldg(&F.start[k]);
            b1 = __ldg(&F.start[k + 1]);
            stall = F.stall ? ((__ldg(&F.stall[k >> 5]) >> (k & 31)) & 1u) != 0u : false;
            const int cnt = b1 - b0;
            G = 2;
            while (G < 16 && cnt * G * 2 <= 32 * nw) G <<= 1;
            per = 32 / G;
            j = lane & (G - 1);
            grp = lane / G;
            if (b0 + gw * per < b1) px = adj_prepare<RR>(a, F, aw, s_pairs, b0 + gw * per, b1, k, stall, G, grp, j);
        };
        if (K > 0) prepare(K - 1);
        for (int k = K - 1; k >= 0; k--) {
            if (k < K - 1) cluster.barrier_wait();  // the scatters of step k + 1 have arrived
            for (int base = b0 + gw * per; base < b1; base += nw * per) {
                if (base != b0 + gw * per) px = adj_prepare<RR>(a, F, aw, s_pairs, base, b1, k, stall, G, grp, j);
                adj_apply<RR>(a, F, aw, s_pairs, px, k, G, grp, j, mu_acc);
            }
            if (k > 0) {
                cluster.barrier_arrive();
                prepare(k - 1);
            }
        }
        double wsum = mu_acc;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wsum += __shfl_xor_sync(AFULL, wsum, o);
        if (lane == 0 && wsum != 0.0) atomicAdd(F.mu_sum, wsum);
        cluster.sync();
        if (crank == 0 && threadIdx.x == 0) atomicAdd(F.grad_mu, (float)__ldcg(F.mu_sum));
        __syncthreads();
    }
}

// Rows around a pixel that its taps can reach: R where the snap covers the rotation's
// rounding (offsets exceed R by less than 3.5e-6), one more where it does not.
int adj_reach(int R, float tau)
{
    const int r = tau >= 6e-6f ? R : R + 1;
    return r <= 3 ? 3 : (r <= 4 ? 4 : 8);
}

const void *adj_kernel_entry(int rr)
{
    return rr == 3 ? (const void *)adj_kernel<3> : (rr == 4 ? (const void *)adj_kernel<4> : (const void *)adj_kernel<8>);
}

size_t adj_smem_bytes(int rr)
{
    return WARPS_PER_CTA * (rr == 3 ? sizeof(AdjWarp<3>) : (rr == 4 ? sizeof(AdjWarp<4>) : sizeof(AdjWarp<8>)));
}

cudaError_t launch_adj(int rr, const cudaLaunchConfig_t &cfg, const AdjArgs &a)
{
    if (rr == 3) return cudaLaunchKernelEx(&cfg, adj_kernel<3>, a);
    if (rr == 4) return cudaLaunchKernelEx(&cfg, adj_kernel<4>, a);
    return cudaLaunchKernelEx(&cfg, adj_kernel<8>, a);
}

}  // namespace gf
