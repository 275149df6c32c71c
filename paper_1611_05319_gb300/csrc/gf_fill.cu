// Shell-by-shell transport fill (Guidefill, arxiv 1611.05319) for sm_103a.
//
// Kernels:
//   init_kernel   one pass over every frame: the image copied to the output where
//                 that is another, state word per pixel (out_shell),
//                 per 8x8 tile the bitmask of hole pixels (U) and of the initial
//                 active boundary (Qw = d_active D^(0)_h, Notation) from bit
//                 operations on the labels, per-frame hole count.
//   order_kernel  sorts frames by hole size (largest first) into the work queue
//                 (a split schedule gives its first frames to a second launch
//                 with larger clusters, running beside the first).
//   fill_kernel   persistent; one thread-block cluster runs one frame's whole
//                 shell loop (Algorithm 1) at a time, with one hardware cluster
//                 barrier per step, then takes the next frame from the queue;
//                 clusters that find the queue empty join running frames
//                 (Teams, below).
//
// Front tracking.  Per step k the cluster processes a work list of tiles.  A
// tile is on the list of step k+1 iff a pixel was filled at step k within
// reach (ceil(eps)+1 pixels) of it; the tiles are claimed with atomicMax on a
// per-tile step word while list slots are reserved with one warp-aggregated
// atomicAdd (a warp-ballot stream compaction); lost claims leave skip markers.  Inside a tile only pixels within reach of a step-k fill
// are candidates: the only pixels whose ready test can change (new front
// pixels are 8-neighbours of fills, and a waiting pixel's test depends only on
// pixels of its ball).  Candidates get the exact active-boundary test from the
// state words, so the front sets equal a full rescan (Algorithm 1, last line).
// With GF_FLAG_RESCAN every step instead re-tests every unfilled pixel of the
// frame ("Guidefill without tracking", Section 3.6).
//
// State word s per pixel: -1 known, -2 unfilled hole, -3 bystander, k filled at
// step k.  Readable at step k (Omega_h \ (D^(k)_h u B_h), Section 2.1) iff
// (uint)(s+1) < (uint)(k+1).  Step-k fills write k, which no step-k test
// treats as readable, so fills are written in place (Algorithm 1 evaluates
// every front pixel against D^(k)).
//
// Mutable global data is read with plain (weak) loads.  Every value a step reads
// was written before the cluster barrier that began the step (whose wait has
// acquire semantics at cluster scope, so the loads observe those writes), or is
// being written during the step by another warp, in which case the old and the
// new value lead to the same decision: a state word becoming k is unreadable at
// step k like the -2 it replaces, and a neighbour's unfilled mask only filters
// claims.

#include <cooperative_groups.h>

#include "gf_internal.cuh"

namespace cg = cooperative_groups;

namespace gf {

constexpr unsigned FULL = 0xffffffffu;

// A plain load (weak, may be served by L1); see the note on mutable data above.
template <class T>
__device__ __forceinline__ T ld(const T *p)
{
    return *p;
}

// The ball's samples in shared memory as mirror pairs {(n, m), (-n, -m)}, one entry
// per pair, with m < 0, or m = 0 and n < 0: (n, n, m, m), ready for two-wide
// arithmetic, and (1/|(n, m)|, code) with code = |m| | (n + 8) << 8 | (m + 8) << 16.
// (The lanes of a pixel read different entries, which the constant cache would
// serialise.)
__shared__ float4 g_pos[MAX_SAMPLES / 2];
__shared__ float2 g_wt[MAX_SAMPLES / 2];

// ---------------------------------------------------------------------------
// init
// ---------------------------------------------------------------------------
// One warp per strip of 8 pixel rows x 32 tiles (256 columns); lane l owns tile
// column 32 s + l, i.e. 8 pixel columns, and holds the known and hole bits of its
// columns (plus one column each side) for the strip's rows and the row above and
// below.  The active boundary of D^(0)_h (hole pixels with a known 8-neighbour)
// is then a few bit operations per row, the state words are written as two
// 16-byte stores per row and lane, and each lane writes its tile's masks.
// INIT_WARPS strips per CTA.
//
// Also what a fill starts from: the copy of the input where the output is another image
// (CTAs of their own) and the cleared stall bitmap.  With the scratch cleared by the
// descriptor upload and no order kernel for one frame, a single fill is three launches
// instead of six or seven: the 128 x 128 frame 107 -> 96 us a call.

__device__ __forceinline__ uint2 init_label_row(const uint8_t *labels, int W, int H, int y, int x0, bool vec8)
{
    // labels of columns x0 .. x0+7 of row y (0xff outside the image)
    uint2 v = make_uint2(0xffffffffu, 0xffffffffu);
    if (y >= 0 && y < H && x0 < W) {
        const uint8_t *row = labels + (size_t)y * W;
        if (vec8) {
            v = __ldg(reinterpret_cast<const uint2 *>(row + x0));
        } else {
            uint32_t b[8];
#pragma unroll
            for (int c = 0; c < 8; c++) b[c] = (x0 + c < W) ? (uint32_t)__ldg(row + x0 + c) : 0xffu;
            v.x = b[0] | (b[1] << 8) | (b[2] << 16) | (b[3] << 24);
            v.y = b[4] | (b[5] << 8) | (b[6] << 16) | (b[7] << 24);
        }
    }
    return v;
}

__device__ __forceinline__ void init_label_bits(uint2 v, uint32_t &kn, uint32_t &ho)
{
    // known and hole bits, four labels at a time: __vseteq4 sets bit 8i of a word where
    // byte i matches, and the multiply gathers bits 0, 8, 16, 24 into bits 21..24 (the
    // partial products 2^(8i + 7j) are distinct, so nothing carries)
    auto bits4 = [](uint32_t x) { return ((x * 0x00204081u) >> 21) & 0xfu; };
    kn = bits4(__vseteq4(v.x, 0u)) | (bits4(__vseteq4(v.y, 0u)) << 4);
    ho = bits4(__vseteq4(v.x, 0x01010101u)) | (bits4(__vseteq4(v.y, 0x01010101u)) << 4);
}

__global__ void __launch_bounds__(32 * INIT_WARPS, 4) init_kernel(const __grid_constant__ InitArgs a)
{
    const int b = blockIdx.x;
    // frame f with cta_offset[f] <= b < cta_offset[f+1] (a division when every frame
    // takes the same number of CTAs)
    int lo = 0, first = 0;
    if (a.uniform_ctas > 0) {
        lo = b / a.uniform_ctas;
        first = lo * a.uniform_ctas;
    } else {
        int hi = a.n_frames;
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (__ldg(&a.cta_offset[mid]) <= b) lo = mid; else hi = mid;
        }
        first = __ldg(&a.cta_offset[lo]);
    }
    const FrameDev &F = a.frames[lo];
    const int H = F.H, W = F.W, TW = F.TW, TH = F.TH;
    const int strips = (TW + 31) >> 5;
    const int lane = threadIdx.x & 31;
    const int own = init_ctas(TH, W);
    if (b - first >= own) {
        // a CTA that copies colours (src is set)
        const int64_t px = (int64_t)H * W, p0 = (int64_t)(b - first - own) * COPY_PIXELS + threadIdx.x;
        constexpr int N = COPY_PIXELS / (32 * INIT_WARPS);
        float4 v[N];
#pragma unroll
        for (int i = 0; i < N; i++) {
            const int64_t q = p0 + i * (32 * INIT_WARPS);
            if (q < px) v[i] = __ldcs(&F.src[q]);
        }
#pragma unroll
        for (int i = 0; i < N; i++) {
            const int64_t q = p0 + i * (32 * INIT_WARPS);
            if (q < px) F.rgba[q] = v[i];
        }
        return;
    }
    const int unit = (b - first) * INIT_WARPS + (threadIdx.x >> 5);
    if (unit >= TH * strips) return;  // warp-uniform
    if (unit == 0 && lane == 0) {
        // stands unless the frame's fill ends: a frame that no cluster has taken when
        // every one of them has left has no other writer
        gf_stats st = {};
        st.status = GF_ERR_TIMEOUT;
        st.data_switch = -1;
        *F.stats = st;
    }
    if (F.stall_bits) {
        // the stall bitmap starts at zero
        const WordRange r = stall_words((int64_t)H * W, unit, TH * strips);
        for (int w = r.begin + lane; w < r.end; w += 32) F.stall_bits[w] = 0u;
    }
    const int ty = unit / strips, sx = unit - ty * strips;
    const int tx = sx * 32 + lane;
    const bool tile_ok = tx < TW;
    const int x0 = tx * TILE, y0 = ty * TILE;
    const bool vec8 = (W & 7) == 0 && (reinterpret_cast<uintptr_t>(F.labels) & 7u) == 0;
    const bool vec16 = (W & 7) == 0 && (reinterpret_cast<uintptr_t>(F.shell) & 15u) == 0 &&
                       (!F.enter || (reinterpret_cast<uintptr_t>(F.enter) & 15u) == 0);

    // rows y0-1 .. y0+8: bit 0 = column x0-1, bits 1..8 = x0 .. x0+7, bit 9 = x0+8
    uint32_t kn[TILE + 2], ho[TILE + 2];
    uint2 lab[TILE + 2];  // every row's load is issued before the first is used
    int edge[TILE + 2];   // lanes 0 and 31: the label beyond the strip
#pragma unroll
    for (int r = 0; r < TILE + 2; r++) {
        const int y = y0 - 1 + r;
        const int ex = lane == 0 ? x0 - 1 : x0 + 8;
        lab[r] = tile_ok ? init_label_row(F.labels, W, H, y, x0, vec8) : make_uint2(0xffffffffu, 0xffffffffu);
        edge[r] = ((lane == 0 || lane == 31) && y >= 0 && y < H && ex >= 0 && ex < W)
                      ? (int)__ldg(&F.labels[(size_t)y * W + ex]) : 0xff;
    }
#pragma unroll
    for (int r = 0; r < TILE + 2; r++) {
        uint32_t k8, h8;
        init_label_bits(lab[r], k8, h8);
        // the neighbouring columns: from the adjacent lanes, or from memory at the strip's ends
        uint32_t kl = (__shfl_up_sync(FULL, k8, 1) >> 7) & 1u;
        uint32_t kr = __shfl_down_sync(FULL, k8, 1) & 1u;
        if (lane == 0) kl = edge[r] == 0 ? 1u : 0u;
        if (lane == 31) kr = edge[r] == 0 ? 1u : 0u;
        kn[r] = kl | (k8 << 1) | (kr << 9);
        ho[r] = h8 << 1;
    }
    // tile masks and state words of rows y0 .. y0+7
    unsigned long long U = 0ull, Q = 0ull;
#pragma unroll
    for (int r = 1; r <= TILE; r++) {
        uint32_t nb = kn[r - 1] | kn[r + 1];
        nb |= (nb << 1) | (nb >> 1) | (kn[r] << 1) | (kn[r] >> 1);
        const uint32_t f = ho[r] & nb;
        const uint32_t urow = (ho[r] >> 1) & 0xffu, qrow = (f >> 1) & 0xffu;
        U |= (unsigned long long)urow << (8 * (r - 1));
        Q |= (unsigned long long)qrow << (8 * (r - 1));
        const int y = y0 + r - 1;
        if (!tile_ok || y >= H) continue;
        // state word: -1 known, -2 hole, -3 anything else (bystander); outside the
        // image nothing is written
        const uint32_t known = (kn[r] >> 1) & 0xffu;
        int32_t sw[8], en[8];
#pragma unroll
        for (int c = 0; c < 8; c++) {
            // known and hole exclude each other
            static_assert(SH_KNOWN == SH_BYST + 2 && SH_UNFILLED == SH_BYST + 1, "state word values");
            sw[c] = SH_BYST + 2 * (int32_t)((known >> c) & 1u) + (int32_t)((urow >> c) & 1u);
            en[c] = ((qrow >> c) & 1u) ? 0 : -1;
        }
        const size_t o = (size_t)y * W + x0;
        if (vec16) {
            reinterpret_cast<int4 *>(F.shell + o)[0] = make_int4(sw[0], sw[1], sw[2], sw[3]);
            reinterpret_cast<int4 *>(F.shell + o)[1] = make_int4(sw[4], sw[5], sw[6], sw[7]);
            if (F.enter) {
                reinterpret_cast<int4 *>(F.enter + o)[0] = make_int4(en[0], en[1], en[2], en[3]);
                reinterpret_cast<int4 *>(F.enter + o)[1] = make_int4(en[4], en[5], en[6], en[7]);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 8; c++) {
                if (x0 + c < W) {
                    F.shell[o + c] = sw[c];
                    if (F.enter) F.enter[o + c] = en[c];
                }
            }
        }
    }
    int gcount = 0;  // data term: hole pixels of this tile with g != 0
    if ((a.flags & GF_FLAG_DATA) && tile_ok) {
        for (unsigned long long m = U; m; m &= m - 1ull) {
            const int pix = __ffsll((long long)m) - 1;
            const float2 gv = __ldg(&F.guide[(size_t)(y0 + (pix >> 3)) * W + x0 + (pix & 7)]);
            gcount += (gv.x != 0.0f || gv.y != 0.0f) ? 1 : 0;
        }
    }
    const int t = ty * TW + tx;
    if (tile_ok) {
        F.U[t] = U;
        F.Qw[t] = Q;
        F.sched[t] = -1;
        // both fill records whole (mask 0, tag INT32_MIN): 16-byte stores leave no
        // partially written L2 sector to be read back from DRAM
        reinterpret_cast<int4 *>(&F.F[t])[0] = make_int4(0, 0, INT32_MIN, 0);
        reinterpret_cast<int4 *>(&F.F[F.ntiles + t])[0] = make_int4(0, 0, INT32_MIN, 0);
    }
    const int holes = __reduce_add_sync(FULL, __popcll(U));
    const int nq = __reduce_add_sync(FULL, __popcll(Q));
    gcount = __reduce_add_sync(FULL, gcount);
    // step-0 work list: warp-aggregated append of the tiles on the initial front
    const bool has_front = Q != 0ull;
    const unsigned bm = __ballot_sync(FULL, has_front);
    int b0 = 0;
    if (lane == 0) {
        if (holes) atomicAdd(F.holes, holes);
        if (gcount) atomicAdd(F.gleft, gcount);
        if (bm) {
            b0 = atomicAdd(&F.init_count[0], __popc(bm));
            atomicAdd(&F.init_count[1], nq);
        }
    }
    b0 = __shfl_sync(FULL, b0, 0);
    if (has_front) F.init_list[b0 + __popc(bm & ((1u << lane) - 1u))] = t;
}

__global__ void upload_frames_kernel(const __grid_constant__ FrameChunk c)
{
    for (int i = threadIdx.x; i < c.count; i += blockDim.x) {
        c.dst_frames[c.first + i] = c.frames[i];
        c.dst_cta[c.first + i] = c.cta[i];
    }
    if (threadIdx.x == 0 && c.last_chunk) c.dst_cta[c.first + c.count] = c.cta[c.count];
    for (int64_t i = threadIdx.x; i < c.zero16; i += blockDim.x) c.zero[i] = make_uint4(0u, 0u, 0u, 0u);
}

// Frames in decreasing hole size (ties: index), one thread per frame.
__global__ void order_kernel(const FrameDev *frames, int n, int32_t *order, int32_t *cursor)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int hi = ld(frames[i].holes);
        int rank = 0;
        for (int j = 0; j < n; j++) {
            int hj = ld(frames[j].holes);
            if (hj > hi || (hj == hi && j < i)) rank++;
        }
        order[rank] = i;
    }
    if (blockIdx.x == 0 && threadIdx.x < 2) cursor[threadIdx.x] = 0;
}

// ---------------------------------------------------------------------------
// fill
// ---------------------------------------------------------------------------
// NORMAL: a work-list tile, candidates near the last step's fills.  RESCAN:
// every unfilled pixel each step (no tracking).  STALL: the stall rule over the
// waiting front.  REVAL: every unfilled pixel once with eq. ready (the step at
// which the data term of eq. ready2 is switched off), with claims.
enum Mode { NORMAL = 0, RESCAN = 1, STALL = 2, REVAL = 3 };

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// Pixels of the centre tile within Chebyshev distance `reach` of a set bit of
// the 3x3 neighbourhood masks; lane l < 9 holds the mask of neighbour
// (dx, dy) = (l%3 - 1, l/3 - 1).  reach <= 8.
__device__ __forceinline__ unsigned long long dilate_nbr(unsigned long long fm, int reach)
{
    const int lane = threadIdx.x & 31;
    const int gy = lane - 8;  // row in [-8, 16) of the 3-tile column
    const int tr = gy < 0 ? 0 : (gy < 8 ? 1 : 2);
    const int ry = (lane < 24) ? gy - (tr - 1) * 8 : 0;
    unsigned long long mL = __shfl_sync(FULL, fm, tr * 3 + 0);
    unsigned long long mC = __shfl_sync(FULL, fm, tr * 3 + 1);
    unsigned long long mR = __shfl_sync(FULL, fm, tr * 3 + 2);
    uint32_t row = 0;
    if (lane < 24)
        row = (uint32_t)((mL >> (8 * ry)) & 0xffu) | ((uint32_t)((mC >> (8 * ry)) & 0xffu) << 8) |
              ((uint32_t)((mR >> (8 * ry)) & 0xffu) << 16);
    // dilation by doubling: after a pass of step st <= c + 1 a set bit covers the
    // offsets 0 .. c + st (rows: shfl_up/down return the lane's own value at the
    // warp's ends, and lanes 24..31 hold no row)
    uint32_t h = row;
    for (int c = 0; c < reach;) {
        const int st = min(c + 1, reach - c);
        h |= (h << st) | (h >> st);
        c += st;
    }
    uint32_t v = (lane < 24) ? ((h >> 8) & 0xffu) : 0u;
    for (int c = 0; c < reach;) {
        const int st = min(c + 1, reach - c);
        v |= __shfl_up_sync(FULL, v, st) | __shfl_down_sync(FULL, v, st);
        c += st;
    }
    unsigned long long out = 0;
#pragma unroll
    for (int y = 0; y < 8; y++) out |= (unsigned long long)(__shfl_sync(FULL, v, 8 + y) & 0xffu) << (8 * y);
    return out;
}

// FP64 confidence of tile pixel `pix` (eqs. weight, confidence) against c; used only
// inside the FP32 guard band.  The whole warp works on one pixel, every lane on its
// share of the samples.  First the weights are summed over the lanes in a tree, with
// the table's reciprocal distances: that decides unless S_rd is within 1e-12 S_all of
// c S_all, far above the at most 1e-13 by which such sums can differ from any other
// order's.  Otherwise the weights are added in the canonical order with the oracle's
// expressions, exactly as the oracle adds them.  FP64 runs at a 64th of the FP32 rate
// here and a re-check holds up its frame's step: the canonical sums alone, two chains
// of 28 to 148 additions behind a division and a square root per sample, added 11 us
// (eps 3) to 25 us (eps 5) to the step; the tree adds 2 to 4 us.  Must be called by all 32
// lanes.
template <int RW>
__device__ __noinline__ bool warp_ready_fp64(const FillParams &p, const WarpSmem<RW> *ws, int pix, bool ghost)
{
    constexpr int NSLOT = RW == 4 ? 1 : (RW == 5 ? 2 : 5);  // ceil(samples / 32) for ceil(eps) = 3, 4, 7
    const int lane = threadIdx.x & 31;
    const int px = pix & 7, py = pix >> 3;
    const float gx = ws->guide[pix].x, gy = ws->guide[pix].y;
    float ch = 1.0f, sh = 0.0f;
    if (ghost) {
        const float a2f = __fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy));
        const float a = __fsqrt_rn(a2f);
        if (a > 0.0f) {
            ch = __fdiv_rn(gx, a);
            sh = __fdiv_rn(gy, a);
        }
    }
    const double a2 = __dadd_rn(__dmul_rn((double)gx, (double)gx), __dmul_rn((double)gy, (double)gy));
    double e[NSLOT];  // e^-t
    unsigned ok = 0;  // by slot
    double A = 0.0, B = 0.0;
#pragma unroll
    for (int q = 0; q < NSLOT; q++) {
        const int s = q * 32 + lane;
        e[q] = 0.0;
        if (s < p.tab.ns) {
            const int n = p.tab.cn[s], m = p.tab.cm[s];
            float ox, oy;
            if (ghost) {
                const float fn = (float)n, fm = (float)m;
                ox = __fsub_rn(__fmul_rn(fn, ch), __fmul_rn(fm, sh));
                oy = __fadd_rn(__fmul_rn(fn, sh), __fmul_rn(fm, ch));
                float r = rintf(ox);
                if (fabsf(__fsub_rn(ox, r)) <= p.tau) ox = r;
                r = rintf(oy);
                if (fabsf(__fsub_rn(oy, r)) <= p.tau) oy = r;
            } else {
                ox = (float)n;
                oy = (float)m;
            }
            const float flx = floorf(ox), fly = floorf(oy);
            const float frx = __fsub_rn(ox, flx), fry = __fsub_rn(oy, fly);
            const int ix = px + RW + (int)flx, iy = py + RW + (int)fly;
            const uint32_t need = frx > 0.0f ? 3u : 1u;
            bool rd = ix >= 0 && iy >= 0 && ix < WarpSmem<RW>::WS - 1 && iy < WarpSmem<RW>::WS - 1;
            rd = rd && ((ws->rowmask[iy] >> ix) & need) == need;
            if (fry > 0.0f) rd = rd && (((ws->rowmask[iy + 1] >> ix) & need) == need);
            double t;
            if (ghost) {
                t = __dmul_rn(__dmul_rn(p.coef64, a2), (double)(m * m));
            } else {
                const double proj = __dadd_rn(__dmul_rn(-(double)gy, (double)n), __dmul_rn((double)gx, (double)m));
                t = __dmul_rn(__dmul_rn(p.coef64, proj), proj);
            }
            e[q] = exp(-t);
            const double w = e[q] * p.tab.cinv[s];
            A += w;
            if (rd) {
                B += w;
                ok |= 1u << q;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        A += __shfl_xor_sync(FULL, A, o);
        B += __shfl_xor_sync(FULL, B, o);
    }
    const double d = B - p.c64 * A;
    if (fabs(d) > 1e-12 * A) return d > 0.0;  // the same on every lane
    double S_all = 0.0, S_rd = 0.0;
#pragma unroll 1
    for (int q = 0; q < NSLOT; q++) {
        const int s = q * 32 + lane;
        double w = 0.0;
        if (s < p.tab.ns) {
            const int n = p.tab.cn[s], m = p.tab.cm[s];
            double eq = e[0];
#pragma unroll
            for (int i = 1; i < NSLOT; i++) eq = q == i ? e[i] : eq;
            w = __ddiv_rn(eq, __dsqrt_rn((double)(n * n + m * m)));
        }
        for (int src = 0; src < 32; src++) {
            const double wv = __shfl_sync(FULL, w, src);
            const unsigned okv = __shfl_sync(FULL, ok, src);
            if (q * 32 + src < p.tab.ns) {
                S_all = __dadd_rn(S_all, wv);
                if ((okv >> q) & 1u) S_rd = __dadd_rn(S_rd, wv);
            }
        }
    }
    return __ddiv_rn(S_rd, S_all) > p.c64;
}

// Lanes per front pixel of a tile with n front pixels (n capped at 17): as many as
// the warp has for them, and ceil(256 / lanes), with which (lane * y) >> 8 is lane /
// lanes.  Any count of lanes goes: 9 pixels get 3 lanes each and 5 iterations over
// the 14 pairs of eps = 3 where powers of two gave 2 lanes and 7.
__constant__ int2 c_lanes[18] = {{32, 8},  {32, 8},  {16, 16}, {10, 26}, {8, 32},   {6, 43},
                                 {5, 52},  {4, 64},  {4, 64},  {3, 86},  {3, 86},   {2, 128},
                                 {2, 128}, {2, 128}, {2, 128}, {2, 128}, {2, 128},  {1, 256}};

// Two FP32 operations in one instruction (each correctly rounded, as the scalar ones).
__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v)
{
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// Sums over a pixel's readable samples.  The weights' sum is kept with its rounding
// error (lo): the same pattern of readable samples meets a front again and again, and
// an error of the divisor of half an ulp, the same each time, would add up over a
// long chain of shells (a 4K frame with 250 shells was 3.8e-7 off its values in 64
// bits, and is 3e-8 off now).
struct Acc {
    unsigned long long xy, zw;  // colours, two channels a word
    float s, lo;                // weights
};
// s + w, its rounding error added to lo
__device__ __forceinline__ void weight_add(float &s, float &lo, float w)
{
    const float t = __fadd_rn(s, w), b = __fsub_rn(t, s);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(w, b)));
    s = t;
}
__device__ __forceinline__ void acc_add(Acc &a, unsigned long long w, const ulonglong2 &c)
{
    a.xy = fma2(w, c.x, a.xy);
    a.zw = fma2(w, c.y, a.zw);
}

// The set of the pixels `pix` of the lanes with `in` (every lane gets it): two warp
// reductions, where 64-bit atomics on a shared word would be retried lane by lane.
__device__ __forceinline__ unsigned long long pixel_mask(bool in, int pix)
{
    const uint32_t bit = in ? 1u << (pix & 31) : 0u;
    const uint32_t lo = __reduce_or_sync(FULL, pix < 32 ? bit : 0u);
    const uint32_t hi = __reduce_or_sync(FULL, pix < 32 ? 0u : bit);
    return (unsigned long long)hi << 32 | lo;
}

// The readable bits around a pixel as one word (R <= 3): rows -3 .. 3, 8 columns -3
// .. 4 each, bit 8 (dy + 3) + dx + 3.
template <int RW>
__device__ __forceinline__ unsigned long long around(const WarpSmem<RW> *ws, int px, int py)
{
    uint32_t lo = 0, hi = 0;
#pragma unroll
    for (int r = 0; r < 4; r++) lo |= ((ws->rowmask[py + RW - 3 + r] >> (px + RW - 3)) & 0xffu) << (8 * r);
#pragma unroll
    for (int r = 0; r < 3; r++) hi |= ((ws->rowmask[py + RW + 1 + r] >> (px + RW - 3)) & 0xffu) << (8 * r);
    return (unsigned long long)hi << 32 | lo;
}

// The rotated ball of one pixel, over the mirror pairs j, j + G, ...: readable weights
// (from the group weights eg), weighted colours, and the smallest |m| of a readable
// sample, MAX_R + 1 when there is none.
//
// Negation is exact and commutes with every rounding of the rotation and of the
// snap, so the second sample's offset is the exact negative of the first's; the
// pair shares its rotation, snap, floor and weights, and each tap of the second
// sample is the first's tap reflected through the pixel, with the same bilinear
// weight.  Taps of zero weight and the taps of unreadable samples are read from the
// window's zero entry (an unreadable pixel's colour may be anything, and 0 * NaN is
// NaN).
//
// Bound by the dependent instructions of an iteration, so: two-wide arithmetic for
// the rotation and the colours; rounding to the lattice by adding 1.5 * 2^23 (the
// difference d to the nearest integer is exact, and floor and fraction follow from
// its sign) instead of the conversion unit; BITS: the readability of a sample's
// cell as one shift and one mask of a register word, the mirrored sample's with the
// same shift and mask of the reversed word, instead of four shared loads.  BITS
// needs R <= 3 and |offset| <= R after the snap: offsets exceed R by their rounding, at
// most R (2.4e-7 + 2^-22) < 1.5e-6, so a snap of 6e-6 px and more covers it.
// Measured (cycles of a tile's sample passes, one 1080p frame, eps 3): 9 to 16 front
// pixels 8,200 -> 6,100, 17 and more 13,100 -> 8,900, an iteration 620 -> 450.
template <int RW, bool BITS>
__device__ __forceinline__ void rotated_pairs(const FillParams &p, const WarpSmem<RW> *ws, const float *eg, int pix, int j,
                                              int G, float ch, float sh, int &least_, Acc &acc_)
{
    constexpr int WS = WarpSmem<RW>::WS, ZI = WS * WS;
    const int px = pix & 7, py = pix >> 3;
    const ulonglong2 *col = reinterpret_cast<const ulonglong2 *>(ws->col);
    const int cx = px + RW, cy = py + RW, c0 = cy * WS + cx;
    const unsigned long long c1 = pack2(ch, sh), c2 = pack2(-sh, ch);
    const unsigned long long big = pack2(12582912.0f, 12582912.0f), nbig = pack2(-12582912.0f, -12582912.0f);
    const unsigned long long neg1 = pack2(-1.0f, -1.0f);
    const float tau = p.tau;
    const int npair = p.tab.ns >> 1;
    unsigned long long near = 0, rnear = 0;
    if (BITS) {
        near = around<RW>(ws, px, py);
        rnear = __brevll(near);
    }
    int least = MAX_R + 1;
    Acc acc = {0ull, 0ull, 0.f, 0.f};
#pragma unroll 1
    for (int q = j; q < npair; q += G) {
        const ulonglong2 nm = *reinterpret_cast<const ulonglong2 *>(&g_pos[q]);  // (n, n), (m, m)
        const float2 wt = g_wt[q];
        const int gm = __float_as_int(wt.y) & 0xff;  // |m|
        const float w0 = eg[gm] * wt.x;
        const unsigned long long o = add2(mul2(nm.x, c1), mul2(nm.y, c2));  // n ch - m sh, n sh + m ch
        const unsigned long long t = add2(o, big);
        const float2 d = unpack2(fma2(add2(t, nbig), neg1, o));             // o - rint(o), exact
        const float2 tf = unpack2(t);
        const bool hx = fabsf(d.x) > tau, hy = fabsf(d.y) > tau;  // off the lattice line
        const bool lx = d.x < -tau, ly = d.y < -tau;              // floor is the integer below
        const float frx = lx ? d.x + 1.0f : (hx ? d.x : 0.0f);
        const float fry = ly ? d.y + 1.0f : (hy ? d.y : 0.0f);
        const int fx = __float_as_int(tf.x) - 0x4b400000 - (lx ? 1 : 0);
        const int fy = __float_as_int(tf.y) - 0x4b400000 - (ly ? 1 : 0);
        bool ok1, ok2;
        if (BITS) {
            const uint32_t kx = hx ? 3u : 1u;
            const uint32_t need = hy ? kx * 257u : kx;
            const int at = 8 * fy + fx;
            ok1 = ((uint32_t)(near >> (at + 27)) & need) == need;
            ok2 = ((uint32_t)(rnear >> (at + 36)) & need) == need;
        } else {
            const uint32_t need = hx ? 3u : 1u;
            const int dy = hy ? 1 : 0, iy = cy + fy, jy = cy - fy;
            const uint32_t m1 = ws->rowmask[iy] & ws->rowmask[iy + dy];
            const uint32_t m2 = ws->rowmask[jy] & ws->rowmask[jy - dy];
            ok1 = ((m1 >> (cx + fx)) & need) == need;
            ok2 = ((m2 >> (cx - fx - (hx ? 1 : 0))) & need) == need;
        }
        if (ok1 || ok2) least = min(least, gm);
        weight_add(acc.s, acc.lo, (ok1 ? w0 : 0.f) + (ok2 ? w0 : 0.f));  // 0, w0 or 2 w0: exact
        const float gx = 1.f - frx;
        const float2 wy = unpack2(mul2(pack2(w0, w0), pack2(1.f - fry, fry)));
        const float l00 = gx * wy.x, l10 = frx * wy.x, l01 = gx * wy.y, l11 = frx * wy.y;
        const int A0 = c0 + fy * WS + fx, B0 = c0 - fy * WS - fx;
        const bool x1 = ok1 && hx, y1 = ok1 && hy, x2 = ok2 && hx, y2 = ok2 && hy;
        const ulonglong2 a0 = col[ok1 ? A0 : ZI];
        const ulonglong2 a1 = col[x1 ? A0 + 1 : ZI];
        const ulonglong2 a2 = col[y1 ? A0 + WS : ZI];
        const ulonglong2 a3 = col[x1 && hy ? A0 + WS + 1 : ZI];
        const ulonglong2 b0 = col[ok2 ? B0 : ZI];
        const ulonglong2 b1 = col[x2 ? B0 - 1 : ZI];
        const ulonglong2 b2 = col[y2 ? B0 - WS : ZI];
        const ulonglong2 b3 = col[x2 && hy ? B0 - WS - 1 : ZI];
        unsigned long long l = pack2(l00, l00);
        acc_add(acc, l, a0);
        acc_add(acc, l, b0);
        l = pack2(l10, l10);
        acc_add(acc, l, a1);
        acc_add(acc, l, b1);
        l = pack2(l01, l01);
        acc_add(acc, l, a2);
        acc_add(acc, l, b2);
        l = pack2(l11, l11);
        acc_add(acc, l, a3);
        acc_add(acc, l, b3);
    }
    least_ = least;
    acc_ = acc;
}

// The lattice ball of one pixel (offsets (n, m) themselves, one tap per sample),
// over the mirror pairs j, j + G, ...; ISO: the stall rule's weights 1/|(n, m)|.  The
// exponent is even in (n, m), so the pair shares its weight, and the plain sums need
// no exponential per sample to rescale them: a tile with 9 to 16 front pixels at eps
// 5 takes 5,800 cycles instead of 20,400 (a 1500 x 1125 still 2.80 -> 0.96 ms with the
// rest of this kernel).
template <int RW, bool ISO, bool LEAST>
__device__ __forceinline__ void lattice_pairs(const FillParams &p, const WarpSmem<RW> *ws, int pix, int j, int G, float2 g,
                                              float &S_all_, bool &any_, Acc &acc_, float low, float &least_)
{
    constexpr int WS = WarpSmem<RW>::WS, ZI = WS * WS;
    const ulonglong2 *col = reinterpret_cast<const ulonglong2 *>(ws->col);
    const int cx = (pix & 7) + RW, cy = (pix >> 3) + RW, c0 = cy * WS + cx;
    const int npair = p.tab.ns >> 1;
    float S_all = 0.f, least = INFINITY;
    bool any = false;
    Acc acc = {0ull, 0ull, 0.f, 0.f};
#pragma unroll 2
    for (int q = j; q < npair; q += G) {
        const float2 wt = g_wt[q];
        const int code = __float_as_int(wt.y);
        const int n = ((code >> 8) & 0xff) - 8, m = ((code >> 16) & 0xff) - 8;
        float w0 = wt.x, e = 0.f;
        if (!ISO) {
            const float proj = -g.y * (float)n + g.x * (float)m;  // g_perp . (n, m)
            const float t = p.coef32 * proj * proj;
            // relative to `low`: exponents below it are those of samples that are not readable
            w0 *= LEAST ? expf(low - (low > t ? low : t)) : expf(-t);
            e = t;
        }
        const bool ok1 = (ws->rowmask[cy + m] >> (cx + n)) & 1u;
        const bool ok2 = (ws->rowmask[cy - m] >> (cx - n)) & 1u;
        any = any || ok1 || ok2;
        if (LEAST && (ok1 || ok2)) least = fminf(least, e);
        S_all += w0 + w0;
        weight_add(acc.s, acc.lo, (ok1 ? w0 : 0.f) + (ok2 ? w0 : 0.f));
        const int at = m * WS + n;
        const unsigned long long w = pack2(w0, w0);
        acc_add(acc, w, col[ok1 ? c0 + at : ZI]);
        acc_add(acc, w, col[ok2 ? c0 - at : ZI]);
    }
    S_all_ = S_all;
    any_ = any;
    if (LEAST) least_ = least;
    acc_ = acc;
}

struct PixelSums {
    float S_rd, S_all, wsum, lo;
    int cnt;
    float4 acc;
};

// One front pixel by the whole warp, each lane's colour sum relative to the smallest
// weight exponent it has read (the normalisation cancels in the average and keeps
// e^-t from underflowing): rotated balls whose rotation is not one.  Must be called by
// all 32 lanes; every lane gets the result.
template <int RW>
__device__ __noinline__ PixelSums slow_pixel(const FillParams &p, const WarpSmem<RW> *ws, int pix)
{
    constexpr int WS = WarpSmem<RW>::WS;
    const int lane = threadIdx.x & 31;
    const int px = pix & 7, py = pix >> 3;
    const float2 g = ws->guide[pix];
    float ch = 1.0f, sh = 0.0f;
    const float a2 = __fadd_rn(__fmul_rn(g.x, g.x), __fmul_rn(g.y, g.y));
    const float a = __fsqrt_rn(a2);
    if (a > 0.0f) {
        ch = __fdiv_rn(g.x, a);
        sh = __fdiv_rn(g.y, a);
    }
    const float beta = p.coef32 * a2;
    float S_rd = 0.f, S_all = 0.f, tmin = INFINITY, wsum = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    int cnt = 0;
    for (int s = lane; s < p.tab.ns; s += 32) {
        const float nf = p.tab.n_f[s], mf = p.tab.m_f[s], invd = p.tab.invd[s];
        float ox = __fsub_rn(__fmul_rn(nf, ch), __fmul_rn(mf, sh));
        float oy = __fadd_rn(__fmul_rn(nf, sh), __fmul_rn(mf, ch));
        float r0 = rintf(ox);
        if (fabsf(__fsub_rn(ox, r0)) <= p.tau) ox = r0;
        r0 = rintf(oy);
        if (fabsf(__fsub_rn(oy, r0)) <= p.tau) oy = r0;
        const float flx = floorf(ox), fly = floorf(oy);
        const float frx = __fsub_rn(ox, flx), fry = __fsub_rn(oy, fly);
        const int ix = px + RW + (int)flx, iy = py + RW + (int)fly;
        const uint32_t need = frx > 0.0f ? 3u : 1u;
        // a rotation longer than one may leave the window
        bool ok = ix >= 0 && iy >= 0 && ix < WS - 1 && iy < WS - 1;
        ok = ok && ((ws->rowmask[iy] >> ix) & need) == need;
        if (fry > 0.0f) ok = ok && (((ws->rowmask[iy + 1] >> ix) & need) == need);
        const float tt = beta * (mf * mf);
        S_all += expf(-tt) * invd;
        if (ok) {
            S_rd += expf(-tt) * invd;
            cnt++;
            if (tt < tmin) {
                const float sc = expf(tt - tmin);  // 0 for the first readable sample
                acc.x *= sc; acc.y *= sc; acc.z *= sc; acc.w *= sc;
                wsum *= sc;
                tmin = tt;
            }
            const float w = expf(tmin - tt) * invd;
            const float4 *cb = &ws->col[iy * WS + ix];
            const float4 v = cb[0];
            const float l00 = (1.f - frx) * (1.f - fry);
            float4 val = make_float4(l00 * v.x, l00 * v.y, l00 * v.z, l00 * v.w);
            if (frx > 0.f) {
                const float l = frx * (1.f - fry);
                const float4 c1 = cb[1];
                val.x += l * c1.x; val.y += l * c1.y; val.z += l * c1.z; val.w += l * c1.w;
            }
            if (fry > 0.f) {
                const float l = (1.f - frx) * fry;
                const float4 c2 = cb[WS];
                val.x += l * c2.x; val.y += l * c2.y; val.z += l * c2.z; val.w += l * c2.w;
                if (frx > 0.f) {
                    const float l3 = frx * fry;
                    const float4 c3 = cb[WS + 1];
                    val.x += l3 * c3.x; val.y += l3 * c3.y; val.z += l3 * c3.z; val.w += l3 * c3.w;
                }
            }
            acc.x += w * val.x; acc.y += w * val.y; acc.z += w * val.z; acc.w += w * val.w;
            wsum += w;
        }
    }
    float tg = tmin;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) tg = fminf(tg, __shfl_xor_sync(FULL, tg, o));
    const float sc = (tmin == INFINITY) ? 0.f : expf(tg - tmin);
    PixelSums r = {S_rd, S_all, wsum * sc, 0.f, cnt, make_float4(acc.x * sc, acc.y * sc, acc.z * sc, acc.w * sc)};
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        r.S_rd += __shfl_xor_sync(FULL, r.S_rd, o);
        r.S_all += __shfl_xor_sync(FULL, r.S_all, o);
        r.cnt += __shfl_xor_sync(FULL, r.cnt, o);
        r.wsum += __shfl_xor_sync(FULL, r.wsum, o);
        r.acc.x += __shfl_xor_sync(FULL, r.acc.x, o);
        r.acc.y += __shfl_xor_sync(FULL, r.acc.y, o);
        r.acc.z += __shfl_xor_sync(FULL, r.acc.z, o);
        r.acc.w += __shfl_xor_sync(FULL, r.acc.w, o);
    }
    return r;
}

// The colour and weight sums of the pixels of a pass (G lanes each) again, relative to
// the smallest exponent of a readable sample: readable weights that all underflow in
// FP32.  Without the ready test a pixel is filled whatever its weights are; with it a
// rotated ball's ready pixels have S_rd > c S_all >= c times the m = 0 weights, but a
// lattice ball's weights may all be tiny.  Out of line: rare, and inside the passes it
// cost every tile 3 to 10 %; one pixel at a time it made onion-order fills with sharp
// weights up to 1.7 times slower than now.  Must be called by all 32 lanes; `run`
// marks the lanes of the pixels concerned, `least_m` is their smallest readable |m| (of
// the rotated ball), and lane j = 0 of each gets the result.
template <int RW>
__device__ __noinline__ PixelSums redo_pixels(const FillParams &p, WarpSmem<RW> *ws, int pix, int grp, int j, int G,
                                              bool run, bool ghost, int least_m)
{
    const float2 g = ws->guide[pix];
    const int R = p.tab.R;
    float ch = 1.0f, sh = 0.0f, beta = 0.0f;
    if (ghost) {
        const float a2 = __fadd_rn(__fmul_rn(g.x, g.x), __fmul_rn(g.y, g.y));
        const float a = __fsqrt_rn(a2);
        if (a > 0.0f) {
            ch = __fdiv_rn(g.x, a);
            sh = __fdiv_rn(g.y, a);
        }
        beta = p.coef32 * a2;
    }
    Acc acc = {0ull, 0ull, 0.f, 0.f};
    if (ghost) {
        __syncwarp();
        if (run)
            for (int gg = j; gg <= R; gg += G)
                ws->eg[grp][gg] = gg < least_m ? 0.f : expf(-(beta * (float)(gg * gg - least_m * least_m)));
        __syncwarp();
        int unused;
        if (run) rotated_pairs<RW, false>(p, ws, ws->eg[grp], pix, j, G, ch, sh, unused, acc);
    } else {
        float low = 0.f, least = INFINITY, all;  // exponents
        bool any;
        if (run) lattice_pairs<RW, false, true>(p, ws, pix, j, G, g, all, any, acc, low, least);
        for (int o = 1; o < G; o <<= 1) {
            const float l = __shfl_down_sync(FULL, least, o);
            if (j + o < G) least = fminf(least, l);
        }
        low = __shfl_sync(FULL, least, threadIdx.x % 32 - j);
        if (run) lattice_pairs<RW, false, true>(p, ws, pix, j, G, g, all, any, acc, low, least);
    }
    float2 axy = unpack2(acc.xy), azw = unpack2(acc.zw);
    for (int o = 1; o < G; o <<= 1) {
        const float s0 = __shfl_down_sync(FULL, acc.s, o), s1 = __shfl_down_sync(FULL, acc.lo, o);
        const float c0 = __shfl_down_sync(FULL, axy.x, o), c1 = __shfl_down_sync(FULL, axy.y, o);
        const float c2 = __shfl_down_sync(FULL, azw.x, o), c3 = __shfl_down_sync(FULL, azw.y, o);
        if (j + o < G) {
            weight_add(acc.s, acc.lo, s0);
            acc.lo += s1;
            axy.x += c0;
            axy.y += c1;
            azw.x += c2;
            azw.y += c3;
        }
    }
    return PixelSums{0.f, 0.f, acc.s, acc.lo, 0, make_float4(axy.x, axy.y, azw.x, azw.y)};
}

// The three work lists of a cluster (the list of step s in slot s % 3): the
// first DS_LIST entries of each in the shared memory of the cluster's first CTA
// (read and written by every CTA through distributed shared memory, a round trip
// within the GPC), the rest in global memory.
constexpr int DS_LIST = 2048;
struct Lists {
    int32_t *ds;    // [3][DS_LIST] in the first CTA's shared memory
    int32_t *glob;  // [3][list_cap]; entries from nds on
    int cap;        // list_cap
    int nds;        // DS_LIST, or 0 while a team of clusters fills the frame
};
__device__ __forceinline__ void list_put(const Lists &L, int slot, int pos, int32_t v)
{
    if (pos < L.nds) L.ds[slot * DS_LIST + pos] = v;
    else L.glob[(size_t)slot * L.cap + pos] = v;
}
__device__ __forceinline__ int32_t list_get(const Lists &L, int slot, int pos)
{
    return pos < L.nds ? ld(&L.ds[slot * DS_LIST + pos]) : ld(&L.glob[(size_t)slot * L.cap + pos]);
}

struct WarpCounters {
    int filled, delta, evals, err, rechecks;
};

// Neighbour-tile claims of step k (tiles for the work list of step k+1).  A claim
// is an atomicMax of k+1 on the tile's step word; the claim that raises it wins.
// Two ways to turn claims into list entries:
//  * combined: list slots for every claim are reserved together with the claims
//    (one round trip); a lost claim leaves a skip marker (-1) in its slot;
//  * deferred: the warp reserves slots only for the claims it won, once their
//    atomics have returned (at its next tile), and writes the entries one tile
//    later, so the list holds no skip markers.  Used by teams and when a list with
//    markers could be longer than the cluster's warp count, where they would be
//    walked one by one.
// The struct carries the claims of a warp's last tiles between those points.
struct PendingClaims {
    unsigned m1;  // claims made, slots not yet reserved (warp-uniform lane mask)
    unsigned m2;  // slots reserved, entries not yet written (warp-uniform lane mask)
    int nt1, old1;  // per lane: claimed tile, previous step word
    int nt2, old2;  // per lane: entry tile; old2 >= k+1 turns it into a skip marker
    int base2;      // lane 0: first reserved slot
    int k;          // step of the pending claims
};

// Writes the reserved entries (their slot reservation has returned).
__device__ __forceinline__ void claims_write(const FillParams &p, const Lists &lists, PendingClaims &pc, WarpCounters &wc)
{
    if (pc.m2) {  // warp-uniform
        const int lane = threadIdx.x & 31;
        const int base = __shfl_sync(FULL, pc.base2, 0);
        if ((pc.m2 >> lane) & 1u) {
            const int pos = base + __popc(pc.m2 & ((1u << lane) - 1u));
            if (pos < p.list_cap) list_put(lists, (pc.k + 1) % 3, pos, pc.old2 < pc.k + 1 ? pc.nt2 : -1);
            else wc.err = 1;
        }
        pc.m2 = 0u;
    }
}

// Reserves slots for the won claims among the deferred ones (their claims have
// returned).  Stage 2 must be empty.
__device__ __forceinline__ void claims_reserve(GroupCtl *ctl, PendingClaims &pc)
{
    if (pc.m1) {  // warp-uniform
        const int lane = threadIdx.x & 31;
        const bool won = ((pc.m1 >> lane) & 1u) && pc.old1 < pc.k + 1;
        const unsigned wb = __ballot_sync(FULL, won);
        if (wb) {
            if (lane == 0) pc.base2 = atomicAdd(&ctl->step[pc.k % 3].next, __popc(wb));
            pc.nt2 = pc.nt1;
            pc.old2 = INT32_MIN;
            pc.m2 = wb;
        }
        pc.m1 = 0u;
    }
}

// Everything pending is written (before the step's counter flush).
__device__ __forceinline__ void claims_drain(const FillParams &p, GroupCtl *ctl, const Lists &lists, PendingClaims &pc,
                                             WarpCounters &wc)
{
    claims_write(p, lists, pc, wc);
    claims_reserve(ctl, pc);
    claims_write(p, lists, pc, wc);
}

// Processes one tile at step k (one warp): candidates, exact front test, ready
// test and fill in one pass over each front pixel's samples, tile masks, claims
// of the neighbour tiles for step k+1.
template <int RW, int MODE>
__device__ void process_tile(const FillParams &p, const FrameDev &F, WarpSmem<RW> *ws, GroupCtl *ctl,
                             const Lists &lists, int t, int k, unsigned long long cand_in, WarpCounters &wc,
                             PendingClaims &pc, bool defer, bool phase1)
{
    constexpr int WS = WarpSmem<RW>::WS;
    const int lane = threadIdx.x & 31;
    const int W = F.W, H = F.H;
    // the previous tile's shared-memory reads and window copies are complete
    cp_async_wait_all();
    __syncwarp();
    const int tx = t % F.TW, ty = t / F.TW;
    const int x0 = tx * TILE, y0 = ty * TILE;
    const int R = p.tab.R;
    const bool ghost = (p.flags & GF_FLAG_GHOST) != 0;
    const bool smart = (p.flags & GF_FLAG_SMART) != 0;

    // Issue every load that depends only on the tile before using any of them:
    // tile masks, the neighbours' step-(k-1) fills and hole masks, the state
    // window, the guide vectors and (speculatively) the colour window.
    const unsigned long long U = ld(&F.U[t]);
    const unsigned long long Qold = ld(&F.Qw[t]);
    int ftag = INT32_MIN;
    unsigned long long fmsk = 0ull, unb = 0ull;
    const int ndx = lane % 3 - 1, ndy = lane / 3 - 1;
    const int nxt_x = tx + ndx, nxt_y = ty + ndy;
    const bool nvalid = lane < 9 && nxt_x >= 0 && nxt_y >= 0 && nxt_x < F.TW && nxt_y < F.TH;
    const int nt = nxt_y * F.TW + nxt_x;
    if (MODE != RESCAN && nvalid) {
        unb = ld(&F.U[nt]);
        if (MODE == NORMAL && k > 0) {
            const TileF *e = &F.F[(size_t)((k - 1) & 1) * F.ntiles + nt];
            ftag = ld(&e->tag);
            fmsk = ld(&e->mask);
        }
    }
    const int wx0 = x0 - RW, wy0 = y0 - RW;
    // State window: 16-byte loads of 4 columns when the row width is a multiple of 4 and
    // the state array is aligned (4 columns are then wholly inside or wholly outside the
    // frame), else 4 plain loads.  RW = 4: 4 quads of 2 x 8 rows from column x0 - 4; wider
    // windows: 6 quads of 4 rows at a time from column x0 - 8, of which the window is a part
    // (one column per lane and row took 4,400 to 6,800 cycles a tile to issue, with the
    // colour window by divisions, and takes 2,200 to 2,900).
    constexpr int QW = RW == 4 ? 4 : 8;           // lanes per row
    constexpr int QR = 32 / QW;                   // rows per load
    constexpr int QN = (WS + QR - 1) / QR;        // loads
    constexpr int QX = RW == 4 ? 4 : 8;           // columns left of the tile
    int4 sq[QN];
    {
        const bool vec = (W & 3) == 0 && ((uintptr_t)F.shell & 15u) == 0;
        const int gx = x0 - QX + 4 * (lane & (QW - 1));
        const bool qin = RW == 4 || (lane & 7) < 6;
#pragma unroll
        for (int i = 0; i < QN; i++) {
            const int r = lane / QW + QR * i, gy = wy0 + r;
            const bool rin = qin && r < WS && gy >= 0 && gy < H;
            if (vec) {
                sq[i] = (rin && gx >= 0 && gx < W) ? ld(reinterpret_cast<const int4 *>(&F.shell[(size_t)gy * W + gx]))
                                                   : make_int4(SH_OUTSIDE, SH_OUTSIDE, SH_OUTSIDE, SH_OUTSIDE);
            } else {
                int e[4];
#pragma unroll
                for (int b = 0; b < 4; b++)
                    e[b] = (rin && gx + b >= 0 && gx + b < W) ? ld(&F.shell[(size_t)gy * W + gx + b]) : SH_OUTSIDE;
                sq[i] = make_int4(e[0], e[1], e[2], e[3]);
            }
        }
    }
    float2 gv[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    if (MODE != STALL) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int pix = lane + 32 * h;
            const int gx = x0 + (pix & 7), gy = y0 + (pix >> 3);
            if (gx < W && gy < H) gv[h] = __ldg(&F.guide[(size_t)gy * W + gx]);
        }
    }
    if (WS == 16) {
        // lane = 16 (row parity) + column; the column test is the same for every row
        const int c = lane & 15, r0 = lane >> 4;
        const bool cin = (unsigned)(wx0 + c) < (unsigned)W;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int gy = wy0 + r0 + 2 * i;
            if (cin && (unsigned)gy < (unsigned)H)
                cp_async16(&ws->col[(r0 + 2 * i) * 16 + c], &F.rgba[(size_t)gy * W + wx0 + c]);
        }
    } else {
        // blocks of CR rows x CW columns (WS is a multiple of CW), one element per lane
        constexpr int CW = WS % 8 == 0 ? 8 : 6, CR = 32 / CW;
        const int r0 = lane / CW, c0 = lane - r0 * CW;
        const float4 *src = F.rgba + ((ptrdiff_t)(wy0 + r0) * W + wx0 + c0);
        float4 *dst = &ws->col[r0 * WS + c0];
#pragma unroll
        for (int i = 0; i < (WS + CR - 1) / CR; i++) {
            const bool rin = r0 < CR && r0 + CR * i < WS && (unsigned)(wy0 + r0 + CR * i) < (unsigned)H;
#pragma unroll
            for (int c = 0; c < WS / CW; c++)
                if (rin && (unsigned)(wx0 + c0 + CW * c) < (unsigned)W)
                    cp_async16(dst + CR * WS * i + CW * c, src + CW * c);
            src += (ptrdiff_t)CR * W;
        }
    }

    unsigned long long cand;
    unsigned claimable = 0;  // neighbours (by lane) that hold unfilled pixels
    if (MODE != RESCAN) claimable = __ballot_sync(FULL, unb != 0ull);
    if (MODE == NORMAL) {
        if (k > 0) {
            const unsigned long long fm = (ftag == k - 1) ? fmsk : 0ull;
            cand = U & dilate_nbr(fm, R + 1);
        } else {
            cand = U;
        }
    } else {
        cand = cand_in & U;
    }
    if (cand == 0) return;

    // ---- readable bits of the window by ballot; guide vectors of the candidates
    // each lane's 4 readable bits at its quad's columns, OR-ed over the lanes of a row
#pragma unroll
    for (int i = 0; i < QN; i++) {
        const int r = lane / QW + QR * i;
        uint32_t v = (readable_at(sq[i].x, k) ? 1u : 0u) | (readable_at(sq[i].y, k) ? 2u : 0u) |
                     (readable_at(sq[i].z, k) ? 4u : 0u) | (readable_at(sq[i].w, k) ? 8u : 0u);
        v = RW == 4 || (lane & 7) < 6 ? v << (4 * (lane & (QW - 1))) : 0u;
#pragma unroll
        for (int o = 1; o < QW; o <<= 1) v |= __shfl_xor_sync(FULL, v, o);
        if ((lane & (QW - 1)) == 0 && r < WS) ws->rowmask[r] = (v >> (QX - RW)) & ((1u << WS) - 1u);
    }
    if (MODE != STALL) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int pix = lane + 32 * h;
            if ((cand >> pix) & 1ull) ws->guide[pix] = gv[h];
        }
    }
    __syncwarp();

    // ---- exact active-boundary test of the candidates
    unsigned long long P;
    {
        bool f[2];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            int pix = lane + 32 * h;
            int px = pix & 7, py = pix >> 3;
            bool c = (cand >> pix) & 1ull;
            int wc_ = px + RW - 1, wr = py + RW;
            uint32_t nb = ((ws->rowmask[wr - 1] >> wc_) & 7u) | ((ws->rowmask[wr] >> wc_) & 5u) |
                          ((ws->rowmask[wr + 1] >> wc_) & 7u);
            f[h] = c && nb != 0u;
        }
        P = (unsigned long long)__ballot_sync(FULL, f[0]) | ((unsigned long long)__ballot_sync(FULL, f[1]) << 32);
        if (F.enter) {
            unsigned long long nf = P & ~Qold;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                int pix = lane + 32 * h;
                if ((nf >> pix) & 1ull)
                    F.enter[(size_t)(y0 + (pix >> 3)) * W + x0 + (pix & 7)] = k;
            }
        }
    }
    const unsigned long long Qkeep = Qold & ~cand;
    const int nqold = __popcll(Qold);
    const int np = __popcll(P);
    wc.evals += np;
    // the front pixels in increasing order: pixel q of a pass is plist[q]
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int pix = lane + 32 * h;
        if ((P >> pix) & 1ull) ws->plist[__popcll(P & ((1ull << pix) - 1ull))] = (uint8_t)pix;
    }

    // ---- ready test (eqs. weight, confidence, ready) and the fill value in one
    //      pass over the sample pairs, G lanes per front pixel
    unsigned long long Rm = 0ull, Cm = 0ull;  // ready; to be decided in FP64 (warp-uniform)
    if (np) {
        cp_async_wait_all();
        __syncwarp();
        const int2 lanes = c_lanes[p.tab.ns <= 32 ? max(min(np, 17), 2) : min(np, 17)];
        const int G = lanes.x, per = 32 / G;
        const int grp = (lane * lanes.y) >> 8, j = lane - grp * G;  // lane / G, lane % G
        const bool decide = MODE != STALL && smart;
        // weights that cannot all underflow: a pixel has a readable sample iff its sum is
        // positive, or is not ready all the same
        const bool plain = MODE == STALL || (ghost && decide);
        for (int base = 0; base < np; base += per) {
            const int q = base + grp;
            const bool act = grp < per && q < np;
            const int pix = act ? ws->plist[q] : 0;
            float2 g = make_float2(0.f, 0.f);
            if (act && MODE != STALL) g = ws->guide[pix];
            float S_all = 0.f;
            bool any = false, odd = false;
            int least = MAX_R + 1;  // rotated ball: smallest |m| of a readable sample
            Acc acc = {0ull, 0ull, 0.f, 0.f};
            if (MODE != STALL && ghost) {
                float ch = 1.0f, sh = 0.0f;
                const float a2 = __fadd_rn(__fmul_rn(g.x, g.x), __fmul_rn(g.y, g.y));
                const float a = __fsqrt_rn(a2);
                if (a > 0.0f) {
                    ch = __fdiv_rn(g.x, a);
                    sh = __fdiv_rn(g.y, a);
                }
                const float beta = p.coef32 * a2;
                // |g| of a few denormals (or not finite): the rotation is not one, and may
                // carry a sample out of the ball's square.  (Correctly rounded, ch^2 + sh^2
                // is within 3.6e-7 of 1 otherwise.)
                odd = a > 0.0f && !(__fmaf_rn(ch, ch, __fmul_rn(sh, sh)) <= 1.0000005f);
                odd = odd || !(a < INFINITY);
                // group weights e^(-beta g^2), g = |m| = 0..R, shared by the pixel's lanes
                __syncwarp();
                if (act)
                    for (int gg = j; gg <= R; gg += G) ws->eg[grp][gg] = expf(-(beta * (float)(gg * gg)));
                __syncwarp();
                if (act && !odd) {
                    const float *eg = ws->eg[grp];
                    if (RW == 4 && p.tau >= 6e-6f) rotated_pairs<RW, true>(p, ws, eg, pix, j, G, ch, sh, least, acc);
                    else rotated_pairs<RW, false>(p, ws, eg, pix, j, G, ch, sh, least, acc);
                    any = least <= R;
                    if (decide && j == 0)
                        for (int gg = 0; gg <= R; gg++) S_all = __fmaf_rn(eg[gg], p.tab.Dm[gg], S_all);
                }
            } else if (act) {
                float unused;
                lattice_pairs<RW, MODE == STALL, false>(p, ws, pix, j, G, g, S_all, any, acc, 0.f, unused);
            }
            // combine the lanes of a pixel: lane j takes from j + 1, then j + 2, ...
            float2 axy = unpack2(acc.xy), azw = unpack2(acc.zw);
            float S_rd = acc.s, S_lo = acc.lo;
            for (int o = 1; o < G; o <<= 1) {
                const float s0 = __shfl_down_sync(FULL, S_rd, o), s1 = __shfl_down_sync(FULL, S_lo, o);
                const float c0 = __shfl_down_sync(FULL, axy.x, o), c1 = __shfl_down_sync(FULL, axy.y, o);
                const float c2 = __shfl_down_sync(FULL, azw.x, o), c3 = __shfl_down_sync(FULL, azw.y, o);
                const bool in = j + o < G;
                weight_add(S_rd, S_lo, in ? s0 : 0.f);
                S_lo += in ? s1 : 0.f;
                axy.x += in ? c0 : 0.f;
                axy.y += in ? c1 : 0.f;
                azw.x += in ? c2 : 0.f;
                azw.y += in ? c3 : 0.f;
                if (!plain) {
                    const float a1 = __shfl_down_sync(FULL, S_all, o);
                    const bool an = __shfl_down_sync(FULL, (int)any, o) != 0;
                    const int l1 = __shfl_down_sync(FULL, least, o);
                    if (in) {
                        S_all += a1;
                        any = any || an;
                        least = min(least, l1);
                    }
                }
            }
            if (plain) any = S_rd > 0.f;
            float wsum = S_rd;
            if (!plain) {
                const bool redo = act && j == 0 && any && !odd && (decide ? S_all < 1e-18f : S_rd < 1e-18f);
                if (__any_sync(FULL, redo)) {
                    const bool mine = __shfl_sync(FULL, (int)redo, lane - j) != 0;
                    const PixelSums r = redo_pixels<RW>(p, ws, pix, grp, j, G, mine, ghost, __shfl_sync(FULL, least, lane - j));
                    if (redo) {
                        axy = make_float2(r.acc.x, r.acc.y);
                        azw = make_float2(r.acc.z, r.acc.w);
                        wsum = r.wsum;
                        S_lo = r.lo;
                    }
                }
            }
            // rotations that are not one: the general way, one pixel at a time
            if (MODE != STALL && ghost) {
                for (unsigned rb = __ballot_sync(FULL, act && j == 0 && odd); rb; rb &= rb - 1u) {
                    const int src = __ffs(rb) - 1;
                    const PixelSums r = slow_pixel<RW>(p, ws, __shfl_sync(FULL, pix, src));
                    if (lane == src) {
                        S_rd = r.S_rd;
                        S_all = r.S_all;
                        any = r.cnt > 0;
                        axy = make_float2(r.acc.x, r.acc.y);
                        azw = make_float2(r.acc.z, r.acc.w);
                        wsum = r.wsum;
                        S_lo = 0.f;
                    }
                }
            }
            // Smart order: decided in FP32 outside a guard band around c, re-checked in
            // FP64 inside it.  Band: relative 1e-4 for the rotated ball, where the FP32
            // error of both sums is below ~1e-5 relative (the m = 0 terms are exact and
            // the error of each other term is bounded by t e^-t <= 1/e times a few ulp);
            // 1e-3 for the lattice ball, whose projection g_perp.(n, m) can cancel.
            bool ready = any;
            bool recheck = false;
            if (decide) {
                const float d = S_rd - p.c * S_all;
                const float tol = (ghost ? 1e-4f : 1e-3f) * p.c * S_all;
                ready = d > tol;
                recheck = !(d > tol) && !(d < -tol);
            }
            if (phase1 && g.x == 0.0f && g.y == 0.0f) {
                // eq. ready2, first phase: the data term D(x) = |g(x)| must exceed c2 = 0
                ready = false;
                recheck = false;
            }
            const bool take = act && j == 0 && any;
            ready = ready && !recheck;
            if (take && (ready || recheck)) {
                // acc / (wsum + S_lo): the reciprocal's product, corrected once
                const float inv = __frcp_rn(wsum);
                auto quot = [&](float v) {
                    const float x = v * inv;
                    const float y = __fmaf_rn(__fmaf_rn(-x, S_lo, __fmaf_rn(-x, wsum, v)), inv, x);
                    return fabsf(x) < INFINITY ? y : x;
                };
                ws->colr[pix] = make_float4(quot(axy.x), quot(axy.y), quot(azw.x), quot(azw.y));
            }
            Rm |= pixel_mask(take && ready, pix);
            if (__any_sync(FULL, take && recheck)) Cm |= pixel_mask(take && recheck, pix);
        }
    }
    __syncwarp();
    // FP64 re-checks, one pixel at a time with the whole warp
    for (unsigned long long rc = Cm; rc; rc &= rc - 1ull) {
        const int pix = __ffsll((long long)rc) - 1;
        if (warp_ready_fp64<RW>(p, ws, pix, ghost)) Rm |= 1ull << pix;
        wc.rechecks++;
    }
    const int nr = __popcll(Rm);
    if (phase1) {
        // guided pixels filled: the data term stays on while any is left (counted by step;
        // a count kept in one place would change under the warps that read it)
        bool gz[2];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int pix = lane + 32 * h;
            gz[h] = ((Rm >> pix) & 1ull) && (ws->guide[pix].x != 0.0f || ws->guide[pix].y != 0.0f);
        }
        const int ng = __popc(__ballot_sync(FULL, gz[0])) + __popc(__ballot_sync(FULL, gz[1]));
        if (lane == 0 && ng) atomicAdd(&ctl->step[k % 3].guided, ng);
    }

    // ---- the fills (state word k: not readable by any other test of step k)
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int pix = lane + 32 * h;
        if ((Rm >> pix) & 1ull) {
            const size_t o = (size_t)(y0 + (pix >> 3)) * W + x0 + (pix & 7);
            F.rgba[o] = ws->colr[pix];
            F.shell[o] = k;
        }
    }

    // ---- tile bookkeeping
    const unsigned long long Qnew = Qkeep | (P & ~Rm);
    if (lane == 0) {
        if (Rm) {
            F.U[t] = U & ~Rm;
            TileF *e = &F.F[(size_t)(k & 1) * F.ntiles + t];
            e->mask = Rm;
            e->tag = k;
        }
        if (Qnew != 0ull || nqold != 0) F.Qw[t] = Qnew;
    }
    wc.filled += nr;
    wc.delta += __popcll(Qnew) - nqold;

    // the previous tiles' claims and reservations have returned by now
    claims_write(p, lists, pc, wc);
    claims_reserve(ctl, pc);

    // ---- tiles for step k+1: the neighbours within reach of this step's fills
    //      that still hold unfilled pixels.  The list slots are reserved with one
    //      atomicAdd while the claims (atomicMax on the tile's step word) are in
    //      flight; a claim lost to another tile leaves a skip marker (-1).
    if (MODE != RESCAN && Rm) {
        const int reach = R + 1;
        // columns holding a fill: OR of the 8 row bytes; rows holding one: bit 8y of
        // the byte-wise OR, gathered into bit y by the multiply
        unsigned long long cb = Rm | (Rm >> 32);
        cb |= cb >> 16;
        cb |= cb >> 8;
        const uint32_t colocc = (uint32_t)(cb & 0xffu);
        unsigned long long rb = Rm | (Rm >> 4);
        rb |= rb >> 2;
        rb |= rb >> 1;
        const uint32_t rowocc = (uint32_t)(((rb & 0x0101010101010101ull) * 0x0102040810204080ull) >> 56);
        const uint32_t lowm = reach >= 8 ? 0xffu : ((1u << reach) - 1u);
        const bool nL = (colocc & lowm) != 0, nR = (colocc >> (8 - (reach >= 8 ? 8 : reach))) != 0;
        const bool nU = (rowocc & lowm) != 0, nD = (rowocc >> (8 - (reach >= 8 ? 8 : reach))) != 0;
        const bool left = lane == 4 ? (U & ~Rm) != 0ull : ((claimable >> lane) & 1u) != 0u;
        const bool need = nvalid && (ndx == 0 || (ndx < 0 ? nL : nR)) && (ndy == 0 || (ndy < 0 ? nU : nD)) && left;
        const unsigned bm = __ballot_sync(FULL, need);
        if (bm) {
            pc.k = k;
            if (defer) {
                pc.m1 = bm;
                pc.nt1 = nt;
                if (need) pc.old1 = atomicMax(&F.sched[nt], k + 1);
            } else {
                pc.m2 = bm;
                pc.nt2 = nt;
                if (lane == 0) pc.base2 = atomicAdd(&ctl->step[k % 3].next, __popc(bm));
                if (need) pc.old2 = atomicMax(&F.sched[nt], k + 1);
            }
        }
    }
}

// Clears the counters of a step slot.
__device__ __forceinline__ void clear_step(GroupCtl *ctl, int slot)
{
    int4 *c = reinterpret_cast<int4 *>(&ctl->step[slot]), *l = reinterpret_cast<int4 *>(&ctl->later[slot]);
    c[0] = make_int4(0, 0, 0, 0);
    c[1] = make_int4(0, 0, 0, 0);
    l[0] = make_int4(0, 0, 0, 0);
    l[1] = make_int4(0, 0, 0, 0);
}

// The counters of a pass of the step in `slot`.
__device__ __forceinline__ PassCtl *pass_ctl(GroupCtl *ctl, int slot, int pass)
{
    return pass == PASS_EVAL ? &ctl->step[slot].eval : &ctl->later[slot][pass - 1];
}

// Adds a warp's counters of a pass of step k to slot k%3.  With `clear_next`, lane 0 (of
// the first warp of each CTA, in a team of the owner's first CTA) also clears
// the slot of step k+1: its last readers passed the barrier of step k-1 and its
// next writers start after the barrier of step k.  In a team (`acc` set) the
// warps add into the CTA's shared counters, which team_sync sends on with one
// atomic per CTA and counter: hundreds of warps adding to one L2 address would
// take several microseconds a step.
//
// What is kept between steps matters to the tiles' code: the kernel is at the 168
// registers that 12 warps leave a thread, and ptxas orders the sample loops' instructions
// worse with less room.  With the count of guided pixels and the flag of a dead cluster in
// registers and the waits inline the same instructions took up to 5 % longer (a 4K frame
// with a blob 3.16 ms, 960 x 1280 at eps 6 660 us, one 1080p frame 1253 us; as here, with
// both in shared memory and team_sync out of line, 3.06 ms, 637 and 1214 us).
__device__ __forceinline__ void flush_counters(GroupCtl *ctl, int *acc, const WarpCounters &wc, int k, int pass,
                                               bool clear_next)
{
    const int lane = threadIdx.x & 31;
    const int s = k % 3;
    int f = wc.filled, d = wc.delta, e = wc.evals, er = wc.err, rc = wc.rechecks;
    // all lanes hold identical values except err (per lane)
    er = __reduce_or_sync(FULL, er);
    if (lane == 0) {
        if (acc) {
            if (f) atomicAdd(&acc[0], f);
            if (d) atomicAdd(&acc[1], d);
            if (e && pass == PASS_EVAL) atomicAdd(&acc[2], e);
            if (er) atomicOr(&acc[3], er);
            if (rc) atomicAdd(&acc[4], rc);
        } else {
            PassCtl *c = pass_ctl(ctl, s, pass);
            if (f) atomicAdd(&c->filled, f);
            if (d) atomicAdd(&c->front_delta, d);
            if (e && pass == PASS_EVAL) atomicAdd(&c->evals, e);  // Sigma_k |front_k| counts the evaluation pass only
            if (er) atomicOr(&c->err, er);
            if (rc) atomicAdd(&ctl->rechecks, rc);
        }
        if (clear_next) clear_step(ctl, (k + 1) % 3);
    }
}

// ---------------------------------------------------------------------------
// Teams: several clusters on one frame
// ---------------------------------------------------------------------------
// A step of a frame with more tiles than its cluster has warps is bound by
// throughput, and clusters hold 16 CTAs at most.  A cluster that finds the queue
// empty therefore joins the running frame whose step is longest: it takes a
// ticket (want), the frame's first cluster (its owner) answers the tickets taken
// by the start of a step at that step's end (Admission), and the newcomers take
// part from the next step on.  Only clusters that already run ask, so the
// barrier never waits for a CTA that has no SM, and a plain launch does.  When a
// step's list gets short, the members with the highest numbers leave again, and
// with one cluster left the frame goes on under the hardware cluster barrier,
// closed to joins.  Which warp processes a tile changes no result.
//
// Team barrier: every CTA adds one to a counter and polls it.  About 1 us a step
// more than the cluster barrier, which is why a team is only as large as its
// work list.
//
// Every wait for another cluster ends after FillParams::polls polls.  A CTA whose wait
// gave up marks the frame (TeamCtl::dead, which ends the other waits for it) and its
// cluster (s_dead in every CTA of it), goes to the cluster's next barrier, whichever the
// other CTAs come to next, and after that barrier they all leave the kernel: a cluster
// leaves whole, so no barrier counts a CTA that is gone and nobody reads its shared
// memory.  A cluster that gets no answer to its ticket marks the frame too, since its
// owner may count on it from now on.  A frame that a dead cluster was needed for ends
// with GF_ERR_TIMEOUT.
//
// Measured against one cluster of 16 CTAs per frame, whole calls, with the sample loops
// and the 16 warps per CTA of that time: a 4K frame with a 400 x 400 blob (eps 4; first
// steps of 1,400 to 4,100 tiles) 4.47 -> 3.48 ms, a 2000 x 500 onion-order line problem
// (about 700 tiles a step) 2.94 -> 1.69 ms, a 1500 x 1125 lattice-ball still 2.9 -> 1.8 ms,
// 32 uneven 1080p frames (on clusters of 4) 4.83 -> 3.90 ms; thin cracks on one 1080p
// frame, where few steps are that long, 1.32 -> 1.19 ms.  Now, one cluster of 192 warps and
// teams: the 4K frame 4.04 and 3.06 ms, 960 x 1280 at eps 6 807 and 637 us, the line
// problem 2.58 and 1.22 ms, the still 1.08 and 0.58 ms, the 1080p frame 1.27 and 1.21 ms.
constexpr int TEAM_COUNTERS = 5;  // a CTA's counters of a pass: filled, front_delta, evals, err; rechecks

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(uint32_t *p, uint32_t v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_volatile(const int32_t *p) { return *(const volatile int32_t *)p; }

// Clusters that a step of n tiles keeps busy (`unit` warps each, one tile per warp).
__device__ __forceinline__ int team_need(int n, int unit) { return n <= unit ? 1 : (n + unit - 1) / unit; }

// The barrier of a pass of a team's step (slot = step % 3): sends the CTA's counters,
// then waits until `target` arrivals have been counted.  False when this CTA's wait gave
// up (then `dead` is set in every CTA of the cluster; `lost` is the CTA's own).
__device__ __noinline__ bool team_sync(TeamCtl *tc, int *acc, int *lost, int *dead, int slot, int pass,
                                          uint32_t target, uint32_t polls)
{
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        if (lane < TEAM_COUNTERS) {
            const int v = acc[lane];
            acc[lane] = 0;
            // err is 0 or 1 per CTA: a sum serves as well as an OR
            if (v) atomicAdd(lane < 4 ? &pass_ctl(&tc->c, slot, pass)->filled + lane : &tc->c.rechecks, v);
        }
        __syncwarp();
        if (lane == 0) {
            __threadfence();
            atomicAdd(&tc->bar, 1u);
            unsigned n = 0;
            while ((int32_t)(ld_acquire(&tc->bar) - target) < 0) {
                if (++n >= polls || ((n & 63u) == 0u && ld_volatile(&tc->dead))) {
                    *lost = 1;
                    break;
                }
            }
            __threadfence();
            if (*lost) {
                *(volatile int32_t *)&tc->dead = 1;
                cg::cluster_group cluster = cg::this_cluster();
                for (unsigned r = 0; r < cluster.num_blocks(); r++) *cluster.map_shared_rank(dead, r) = 1;
            }
        }
    }
    __syncthreads();
    return *lost == 0;
}

// A frame's statistics, kept by its leader (in shared memory: the other threads need
// no registers for them).
struct Totals {
    long long filled, evals;
    int max_front, stalls, data_switch;
};

// What a cluster does next, in the shared memory of its first CTA: f >= 0 is a
// queue position, -1 nothing is left; with help set the cluster is member
// `member` of the frame's team.
struct Role {
    int32_t f, help, member, owner;
    Admission adm;
};

// Looks for a running frame whose coming step has more tiles than its team has
// warps, takes a ticket and waits for the answer; -1 when no frame wants help.
// Called by the first warp of a cluster's first CTA.
__device__ int team_find(const FillParams &p, int unit, Role *role)
{
    const int lane = threadIdx.x & 31;
    for (unsigned tries = 0; tries < 4096u; tries++) {
        // the frame that lacks most clusters
        int best = 0, bf = -1, pending = 0;
        for (int i = lane; i < p.n_frames; i += 32) {
            const TeamCtl *tc = &p.teams[i];
            const int load = ld_volatile(&tc->load);
            if (load == 0) pending = 1;
            if (load <= 0) continue;
            const int asked = (int)(*(const volatile uint32_t *)&tc->want - *(const volatile uint32_t *)&tc->admitted);
            const int lack = team_need(load, unit) - ld_volatile(&tc->team) - asked;
            if (lack > best) {
                best = lack;
                bf = i;
            }
        }
        const int top = __reduce_max_sync(FULL, best);
        if (top <= 0) {
            // frames taken from the queue but not started yet may want help in a moment
            if (__any_sync(FULL, pending) && tries < 64u) {
                __nanosleep(500);
                continue;
            }
            return -1;
        }
        const int src = __ffs(__ballot_sync(FULL, best == top)) - 1;
        bf = __shfl_sync(FULL, bf, src);
        int got = 0;
        if (lane == 0) {
            TeamCtl *tc = &p.teams[bf];
            const uint32_t ticket = atomicAdd(&tc->want, 1u);
            for (unsigned n = 0;; n++) {
                if ((int32_t)(ld_acquire(&tc->admitted) - ticket) > 0) {
                    role->adm = tc->adm;
                    role->owner = tc->owner;
                    role->member = role->adm.first_member + (int)ticket - role->adm.first_ticket;
                    got = 1;
                    break;
                }
                if (ld_volatile(&tc->load) < 0) break;  // over, or closed
                if (n >= p.polls) {
                    *(volatile int32_t *)&tc->dead = 1;
                    got = -1;
                    break;
                }
            }
        }
        got = __shfl_sync(FULL, got, 0);
        if (got < 0) return -1;
        if (got) return bf;
    }
    return -1;
}

// Every warp of the team visits the frame's tiles (32 at a time); the mode
// selects the tile mask that makes a tile a member (U: rescan, re-evaluation;
// Qw: stall) and is passed on as the tile's candidates.
template <int RW, int MODE>
__device__ __forceinline__ WarpCounters sweep_tiles(const FillParams &p, const FrameDev &F, WarpSmem<RW> *ws, GroupCtl *ctl,
                                                 const Lists lists, int k, int gw, int nw, bool phase1)
{
    const int lane = threadIdx.x & 31;
    WarpCounters wc = {0, 0, 0, 0, 0};
    PendingClaims pc;
    pc.m1 = 0u;
    pc.m2 = 0u;
    for (int base = gw * 32; base < F.ntiles; base += nw * 32) {
        int t = base + lane;
        unsigned long long m = 0;
        if (t < F.ntiles) m = (MODE == RESCAN || MODE == REVAL) ? ld(&F.U[t]) : ld(&F.Qw[t]);
        unsigned bal = __ballot_sync(FULL, m != 0ull);
        while (bal) {
            int i = __ffs(bal) - 1;
            bal &= bal - 1;
            unsigned long long mi = __shfl_sync(FULL, m, i);
            process_tile<RW, MODE>(p, F, ws, ctl, lists, base + i, k, mi, wc, pc, false, phase1);
        }
    }
    claims_drain(p, ctl, lists, pc, wc);
    return wc;
}

template <int RW>
__global__ void __launch_bounds__(FILL_WARPS * 32, 1) fill_kernel(const __grid_constant__ FillParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ FrameDev s_frame;
    WarpSmem<RW> *ws = reinterpret_cast<WarpSmem<RW> *>(smem_raw) + (threadIdx.x >> 5);
    cg::cluster_group cluster = cg::this_cluster();
    const int crank = (int)cluster.block_rank();
    const int csize = (int)cluster.num_blocks();
    const int cid = blockIdx.x / csize;
    // the cluster's control block and the heads of its work lists live in the first
    // CTA's shared memory
    __shared__ GroupCtl s_ctl;
    __shared__ int32_t s_lists[3 * DS_LIST];
    __shared__ Role s_role[2];
    __shared__ int s_acc[TEAM_COUNTERS];  // the CTA's step counters while it is in a team
    __shared__ Totals s_tot;   // the leader's
    __shared__ int s_gleft[FILL_WARPS];  // by warp: hole pixels with g != 0 left, while the data term is on
    __shared__ int s_lost;     // the CTA's wait at a team barrier gave up
    __shared__ int s_gone;     // the cluster leaves (found at a barrier within a frame)
    __shared__ int s_dead;     // that of a CTA of the cluster did: read after cluster barriers only
    GroupCtl *const ds_ctl = cluster.map_shared_rank(&s_ctl, 0);
    const Role *const ds_role = cluster.map_shared_rank(s_role, 0);
    Lists lists;
    lists.ds = cluster.map_shared_rank(s_lists, 0);
    lists.cap = p.list_cap;
    const int unit = csize * FILL_WARPS;  // warps of a cluster
    const bool rescan = (p.flags & GF_FLAG_RESCAN) != 0;
    for (int i = threadIdx.x; i < p.tab.ns; i += blockDim.x) {
        // group |m| = g lists m = -g before m = +g (n ascending within each), and
        // n < 0 before n > 0 for g = 0: the first half of every group holds one
        // sample of each mirror pair, and every group before it has an even count
        const float n = p.tab.n_f[i], m = p.tab.m_f[i];
        const int g = (int)fabsf(m);
        const int g0 = p.tab.m_start[g], half = (p.tab.m_start[g + 1] - g0) >> 1;
        if (i - g0 < half) {
            const int e = (g0 >> 1) + (i - g0);
            g_pos[e] = make_float4(n, n, m, m);
            g_wt[e] = make_float2(p.tab.invd[i], __int_as_float(g | ((int)n + 8) << 8 | ((int)m + 8) << 16));
        }
    }
    if ((threadIdx.x & 31) == 0) ws->col[WarpSmem<RW>::WS * WarpSmem<RW>::WS] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (threadIdx.x < TEAM_COUNTERS) s_acc[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_lost = s_dead = s_gone = 0;
    __syncthreads();

    for (int it = 0;; it++) {
        cluster.sync();  // everyone is done with the previous frame's counters
        if (__syncthreads_or(s_dead)) break;
        if (crank == 0 && threadIdx.x < 32) {
            Role *role = &s_role[it & 1];
            int f = 0, help = 0;
            if (threadIdx.x == 0) {
                f = atomicAdd(p.frame_cursor, 1);
                for (int i = 0; i < 3; i++) clear_step(&s_ctl, i);
                s_ctl.rechecks = 0;
            }
            f = __shfl_sync(FULL, f, 0);
            if (f >= p.n_frames) {
                f = p.teams ? team_find(p, unit, role) : -1;
                help = 1;
            }
            if (threadIdx.x == 0) {
                role->f = f;
                role->help = help;
            }
        }
        cluster.sync();
        const Role *role = ds_role + (it & 1);
        const int f = role->f;
        if (f < 0) break;
        const bool own = role->help == 0;
        const bool leader = own && crank == 0 && threadIdx.x == 0;
        if (threadIdx.x == 0) {
            s_frame = p.frames[p.frame_order[p.order_first + f]];
            __threadfence();  // a joining CTA's L1 holds nothing of the frame's earlier steps
        }
        __syncthreads();
        const FrameDev &F = s_frame;
        TeamCtl *const tc = p.teams ? &p.teams[f] : nullptr;
        lists.glob = p.lists + (size_t)(p.lists_by_frame ? f : (own ? cid : role->owner)) * 3 * p.list_cap;

        // uniform over the clusters that fill the frame: its team of `team` clusters,
        // of which this one is number `member`; bar: arrivals the team's barrier has
        // counted when the running step ends; admitted: tickets answered
        int team = 1, member = 0, admitted = 0;
        uint32_t bar = 0;
        bool open = p.teams != nullptr;
        GroupCtl *ctl = ds_ctl;
        int gw, nw;
        auto shape = [&]() {
            gw = ((threadIdx.x >> 5) * team + member) * csize + crank;  // interleave CTAs
            nw = team * unit;
            ctl = team > 1 ? &tc->c : ds_ctl;
            lists.nds = team > 1 ? 0 : DS_LIST;
        };
        // adds a pass's counters and waits for everyone; `leave`: arrivals owed by
        // CTAs that left the team at the end of the last step
        int leave = 0;
        auto finish = [&](const WarpCounters &w, int k, int pass, bool clear) -> bool {
            flush_counters(ctl, team > 1 ? s_acc : nullptr, w, k, pass, clear);
            if (team == 1) {
                cluster.sync();
                return true;
            }
            bar += (uint32_t)(team * csize + leave);
            leave = 0;
            return team_sync(tc, s_acc, &s_lost, &s_dead, k % 3, pass, bar, p.polls);
        };

        int n_front = 0;
        int status = GF_OK;
        int k = 0;
        if (leader) s_tot = Totals{0, 0, 0, 0, -1};
        const int max_shells = F.max_shells;
        int n_cur = 0;
        // eq. ready2 (GF_FLAG_DATA): phase 1 while hole pixels with g != 0 remain and
        // some front pixel is ready under the data term; `reval`: this step tests every
        // front pixel with eq. ready (the tracked front was built under phase 1)
        bool phase1 = (p.flags & GF_FLAG_DATA) != 0;
        bool reval = false;
        if (own) {
            n_front = ld(&F.init_count[1]);
            n_cur = ld(&F.init_count[0]);
            if (phase1) s_gleft[threadIdx.x >> 5] = ld(F.gleft);
            if (phase1 && ld(F.gleft) == 0) {
                phase1 = false;
                if (leader) s_tot.data_switch = 0;
            }
        } else {
            const Admission &adm = role->adm;
            member = role->member;
            team = adm.team;
            k = adm.k;
            n_cur = adm.n_cur;
            n_front = adm.n_front;
            phase1 = adm.phase1 != 0;
            reval = adm.reval != 0;
            s_gleft[threadIdx.x >> 5] = adm.gleft;
            bar = adm.bar;
            admitted = adm.first_ticket + (adm.team - adm.first_member);
        }
        // tells the clusters whose tickets up to `upto` were answered that they are in
        // the team from step k on
        auto admit = [&](int upto, int team_old) {
            tc->adm.first_ticket = admitted;
            tc->adm.first_member = team_old;
            tc->adm.team = team;
            tc->adm.k = k;
            tc->adm.n_cur = n_cur;
            tc->adm.phase1 = phase1 ? 1 : 0;
            tc->adm.reval = reval ? 1 : 0;
            tc->adm.bar = bar;
            tc->adm.n_front = n_front;
            tc->adm.gleft = s_gleft[threadIdx.x >> 5];
            tc->team = team;
            __threadfence();
            st_release(&tc->admitted, (uint32_t)upto);
        };
        const int sweep_load = max(1, F.ntiles / 8);  // rescan: tiles swept 32 at a time by a warp
        if (own && open) {
            const int load = rescan ? sweep_load : max(n_cur, 1);
            const int need = team_need(load, unit);
            if (leader) {
                tc->owner = cid;
                tc->team = 1;
                __threadfence();
                *(volatile int32_t *)&tc->load = load;
            }
            // clusters without a frame of their own are already looking for one: a
            // moment's wait lets them take part in the first step, the longest of most fills
            const int spare = min(need - 1, (int)(gridDim.x / csize) - p.n_frames);
            if (spare > 0) {
                if (leader) {
                    const long long t0 = clock64();
                    uint32_t w;
                    do {
                        w = *(volatile uint32_t *)&tc->want;
                    } while ((int)w < spare && clock64() - t0 < 8000);
                    s_ctl.step[2].join = (int)w;
                }
                cluster.sync();
                const int w = ld(&ds_ctl->step[2].join);
                if (w > 0) {
                    team = 1 + w;
                    if (leader) admit(w, 1);
                    admitted = w;
                }
            }
        }
        shape();
        // the first item of the current step's work list is loaded ahead, together with
        // the previous step's counters
        int t0_cur = -1;
        if (gw < n_cur) t0_cur = k == 0 ? ld(&F.init_list[gw]) : list_get(lists, k % 3, gw);
        for (;;) {
            const int slot = k % 3;
            WarpCounters wc = {0, 0, 0, 0, 0};
            int asked = 0;
            if (leader && open) asked = (int)*(volatile uint32_t *)&tc->want;
            // The leader's own blocks leave its warp in two parts, and without a __syncwarp
            // after each the parts went through the rest of the step one after the other:
            // 6.7 us a step of one pixel against 5.2 (a 4096-step corridor).
            __syncwarp();
            const bool more = n_cur > nw;
            // lost claims leave markers, up to 1.5 per tile: where they could make the next
            // list longer than the warps, and a second round of it, they are avoided
            // (a 1080p step of about 180 tiles on 256 warps, with CTAs of 16, took 13 us with a
            // list of 400 entries against 9.5 us with a compact one)
            const bool defer = team > 1 || 5 * n_cur > 2 * nw;
            if (rescan) {
                wc = sweep_tiles<RW, RESCAN>(p, F, ws, ctl, lists, k, gw, nw, phase1);
            } else if (reval) {
                wc = sweep_tiles<RW, REVAL>(p, F, ws, ctl, lists, k, gw, nw, false);
            } else {
                // step 0 takes the init kernel's list, later steps the lists built by the claims
                const int n = n_cur;
                PendingClaims pc;
                pc.m1 = 0u;
                pc.m2 = 0u;

                // Item gw goes to warp gw; items beyond the warp count are handed out
                // by a per-step cursor (the next grab is in flight while a tile is
                // processed), so uneven tiles do not leave warps idle at the barrier.
                // Negative items are claims lost to another tile.
                const bool lane0 = (threadIdx.x & 31) == 0;
                int pre = 0;
                if (lane0 && more) pre = atomicAdd(&ctl->step[slot].cursor, 1);
                int t = gw < n ? t0_cur : -1;
                for (;;) {
                    if (t >= 0) process_tile<RW, NORMAL>(p, F, ws, ctl, lists, t, k, 0ull, wc, pc, defer, phase1);
                    if (!more) break;
                    const int nxt = nw + __shfl_sync(FULL, pre, 0);
                    if (nxt >= n) break;
                    t = k == 0 ? ld(&F.init_list[nxt]) : list_get(lists, slot, nxt);
                    if (lane0) pre = atomicAdd(&ctl->step[slot].cursor, 1);
                }
                claims_drain(p, ctl, lists, pc, wc);
            }
            if (leader && open) ctl->step[slot].join = asked;
            if (!finish(wc, k, PASS_EVAL, threadIdx.x < 32 && (team == 1 || (own && crank == 0)))) {
                status = GF_ERR_TIMEOUT;
                break;
            }
            // one round trip: this step's counters and the next step's list
            const int s3n = (k + 1) % 3;
            const int4 c0 = ld(reinterpret_cast<const int4 *>(&ctl->step[slot].eval));
            const int2 c1 = ld(reinterpret_cast<const int2 *>(&ctl->step[slot].next));
            int filled = c0.x, dlt = c0.y, n_next = c1.x;
            const int ev = c0.z, er = c0.w;
            const int join = open ? c1.y : 0;
            int t0_next = gw < p.list_cap ? list_get(lists, s3n, gw) : -1;  // used only if gw < n_next
            int gleft = 1;  // hole pixels with g != 0 left
            if (phase1) {
                gleft = s_gleft[threadIdx.x >> 5] - ld(&ctl->step[slot].guided);
                __syncwarp();
                s_gleft[threadIdx.x >> 5] = gleft;
                __syncwarp();
            }
            if (er) {
                status = GF_ERR_INTERNAL;
                break;
            }
            if (leader) {
                s_tot.evals += ev;
                s_tot.max_front = max(s_tot.max_front, n_front + dlt + filled);
            }
            __syncwarp();
            reval = false;
            if (phase1 && filled == 0) {
                // eq. ready2 fills nothing at this step: eq. ready from this step on,
                // and this step is evaluated again with it (every front pixel)
                phase1 = false;
                if (leader) s_tot.data_switch = k;
                const WarpCounters wr = sweep_tiles<RW, REVAL>(p, F, ws, ctl, lists, k, gw, nw, false);
                if (!finish(wr, k, PASS_AGAIN, false)) {
                    status = GF_ERR_TIMEOUT;
                    break;
                }
                filled = ld(&ctl->later[slot][PASS_AGAIN - 1].filled);
                dlt += ld(&ctl->later[slot][PASS_AGAIN - 1].front_delta);
                const int er1 = ld(&ctl->later[slot][PASS_AGAIN - 1].err);
                n_next = ld(&ctl->step[slot].next);
                t0_next = gw < p.list_cap ? list_get(lists, s3n, gw) : -1;
                if (er1) {
                    status = GF_ERR_INTERNAL;
                    break;
                }
                if (leader) s_tot.max_front = max(s_tot.max_front, n_front + dlt + filled);
            } else if (phase1 && gleft == 0) {
                // every pixel with g != 0 is filled: eq. ready from the next step on
                phase1 = false;
                if (leader) s_tot.data_switch = k + 1;
                reval = true;
            }
            int fk = filled;
            if (filled == 0) {
                if (n_front + dlt == 0) break;  // Algorithm 1: D^(k) exhausted (or the rest unreachable)
                // stall rule: no front pixel is ready; fill the front isotropically
                const WarpCounters ws2 = sweep_tiles<RW, STALL>(p, F, ws, ctl, lists, k, gw, nw, false);
                if (!finish(ws2, k, PASS_STALL, false)) {
                    status = GF_ERR_TIMEOUT;
                    break;
                }
                const int sf = ld(&ctl->later[slot][PASS_STALL - 1].filled);
                const int dlt2 = dlt + ld(&ctl->later[slot][PASS_STALL - 1].front_delta);
                const int er2 = ld(&ctl->later[slot][PASS_STALL - 1].err);
                // the stall fills appended claims to the next step's list
                n_next = ld(&ctl->step[slot].next);
                t0_next = gw < p.list_cap ? list_get(lists, s3n, gw) : -1;
                if (er2) {
                    status = GF_ERR_INTERNAL;
                    break;
                }
                if (sf == 0) break;  // front pixels with no readable sample at all
                n_front += dlt2;
                fk = sf;
                if (leader) s_tot.stalls++;
                if (leader && F.stall_bits) atomicOr(&F.stall_bits[k >> 5], 1u << (k & 31));
            } else {
                n_front += dlt;
            }
            if (leader) s_tot.filled += fk;
            __syncwarp();
            // without deferred claims the list holds markers of lost ones; its tiles are
            // then about as many as this step's, at most one per warp
            const int load = rescan ? sweep_load : (defer ? n_next : min(n_next, nw));
            n_cur = n_next;
            t0_cur = t0_next;
            k++;
            if (k >= max_shells) {
                status = GF_ERR_NO_PROGRESS;
                break;
            }
            if (!open) continue;
            // the team of the next step: with the clusters that asked to join, or
            // without those that its list does not keep busy
            const int need = team_need(load, unit);
            const int team_old = team;
            if (join > admitted) team += join - admitted;
            else if (need < team) team = need;
            if (team == team_old) {
                if (leader) *(volatile int32_t *)&tc->load = max(load, 1);
                __syncwarp();
                continue;
            }
            const int nh = min(n_cur, DS_LIST);  // the list's head moves between shared and global memory
            int32_t *hg = lists.glob + (size_t)s3n * p.list_cap, *hs = lists.ds + s3n * DS_LIST;
            if (team > team_old) {
                if (team_old == 1) {
                    for (int i = crank * blockDim.x + threadIdx.x; i < nh; i += csize * blockDim.x) hg[i] = hs[i];
                    cluster.sync();
                }
                if (leader) {
                    admit(join, team_old);
                    *(volatile int32_t *)&tc->load = max(load, 1);
                }
                admitted = join;
            } else if (team > 1) {
                // a CTA that leaves still counts at the next barrier, so that nobody clears
                // the counters it has read until it has
                leave = (team_old - team) * csize;
                if (leader) {
                    tc->team = team;
                    *(volatile int32_t *)&tc->load = max(load, 1);
                }
                if (member >= team) {
                    __syncthreads();
                    if (threadIdx.x == 0) {
                        __threadfence();
                        atomicAdd(&tc->bar, 1u);
                    }
                    break;
                }
            } else {
                // one cluster goes on alone, under the cluster barrier
                open = false;
                if (leader) *(volatile int32_t *)&tc->load = -1;
                if (member > 0) break;
                if (leader)
                    for (int i = 0; i < 3; i++) clear_step(&s_ctl, i);
                for (int i = crank * blockDim.x + threadIdx.x; i < nh; i += csize * blockDim.x) hs[i] = hg[i];
                cluster.sync();
                if (__syncthreads_or(s_dead)) {
                    status = GF_ERR_TIMEOUT;
                    if (threadIdx.x == 0) s_gone = 1;
                    break;
                }
            }
            shape();
            t0_cur = gw < n_cur ? list_get(lists, s3n, gw) : -1;
        }
        if (leader) {
            if (tc) *(volatile int32_t *)&tc->load = -1;
            const int holes = ld(F.holes);
            gf_stats st;
            st.shells = k;
            st.stalls = s_tot.stalls;
            st.filled = s_tot.filled;
            st.evaluations = s_tot.evals;
            st.max_front = s_tot.max_front;
            st.holes = holes;
            st.rechecks = s_ctl.rechecks + (tc ? ld(&tc->c.rechecks) : 0);
            st.data_switch = s_tot.data_switch;
            st.reserved = 0;
            if (status == GF_OK && s_tot.filled < holes) status = GF_INCOMPLETE;
            st.status = status;
            *F.stats = st;
        }
        __syncthreads();
        if (s_gone) break;
    }
    cp_async_wait_all();  // window copies of a last tile that had no candidates
    // no CTA leaves while another may still read its shared memory (the control
    // block and list heads of the first CTA)
    cluster.sync();
}

const void *fill_kernel_entry(int rw)
{
    if (rw == 4) return (const void *)fill_kernel<4>;
    if (rw == 5) return (const void *)fill_kernel<5>;
    return (const void *)fill_kernel<8>;
}

cudaError_t launch_fill(int rw, const cudaLaunchConfig_t &cfg, const FillParams &p)
{
    if (rw == 4) return cudaLaunchKernelEx(&cfg, fill_kernel<4>, p);
    if (rw == 5) return cudaLaunchKernelEx(&cfg, fill_kernel<5>, p);
    return cudaLaunchKernelEx(&cfg, fill_kernel<8>, p);
}

}  // namespace gf
