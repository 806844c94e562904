// RAM step on FP32 rows with their own non-uniform mesh (Sec. 3 on an arbitrary
// periodic mesh), warp-segment form.
//
// The plan cuts every row into work items, one segment of output cells each; a CTA
// takes an equal share of all rows' items.  Its prologue has one thread per item
// form the row's shift (S0: shift_params, FP64) and locate the source cell of the
// segment's left edge (extended by the residual halo) through the row's index
// function or the plan's bucket table and a short walk (Eq. 16).  After that every
// warp takes items from the CTA's counter, alone:
//   - the source window, kWin cells from two before the segment's first source
//     cell, and the segment's own nodes come into the warp's shared memory with
//     asynchronous copies (4 bytes a lane, coalesced; the next segment's copies are
//     in flight while this one is computed);
//   - lane l takes the window cells 5l..5l+4: their widths, their reconstructions
//     (PLM, Sec. 3.1; PPM, App. A; order 4, the mean of the two quartic
//     interpolants of the cumulative mass; the limiters of App. A.2), kept as the
//     coefficients of each cell's in-cell cumulative G_p(d) (Eq. 18's partial
//     integrals), one 16-byte store per cell;
//   - lane l then takes the segment's edges 5l..5l+4: the first is located among the
//     window's nodes by eight halvings, the others by walking on (Eq. 16), G is
//     evaluated once per edge, and each output mass is Eq. 18 -- the rest of the left
//     source cell, the whole cells in between summed in order, the start of the
//     right source cell -- divided by the output width (Eq. 26); an output cell
//     whose edges both fall on the nodes of one source cell takes that cell's value
//     unchanged;
//   - where the mesh under the segment is finer than at the segment, its edges
//     run past the window: the window moves on to the last edge reached, and the
//     lanes take the edges that are left;
//   - with a residual step (Eq. 6) the sub-steps run in the lanes' registers, the
//     neighbours by shuffles (widths, slopes and fluxes formed once per cell).
//
// Positions are 32-bit fixed point, in units of 2^qshift of the plan's 64-bit
// fraction of the period.  A power-of-two number of units makes the period 2^32
// (or a multiple of it), so that differences modulo 2^32 need no case for the
// wrap; the plan (nseg_fit in ram_segments.h) picks qshift, and how many of a window's
// cells are used, so that a window spans less than 2^32 units and
// every cell at least 2^20 (a mean cell about 2^24).  Source and output widths,
// positions and offsets all come from the same rounded nodes, so that what the
// rounding does is to move the mesh by 2^-24 of a mean cell: the masses stay
// consistent, and the results are no further from the exact ones than those of the
// per-order kernels' 64-bit positions (figures below).  The shift is not rounded: it is
// the same at every step of a steady rotation, so that its rounding would add up.  It is
// a whole number of units, rounded up, and a rest below a unit that is added where the
// cumulative is evaluated (to the offset itself, its rounding would show: 9.3e-8 against
// 8.8e-8 on the 512-row batch).
//
// Why this form: at 16 bytes a cell the step is bound by the instructions it
// issues and by the shared-memory passes of its gathers, not by DRAM (60% of the
// issue slots, 72% of the shared-memory data path, 25% of the measured bandwidth on
// the 512-row batch).  Five cells per lane, an odd number, keep every strided access
// of the shared arrays free of bank conflicts (16-byte ones too), pay for the search
// once per five edges, and form the stencil's differences and reciprocals once per
// neighbour instead of once per use.  One body serves the three orders: three copies
// missed the instruction cache (68.2 us with them, 51.8 without, about 1 of the
// difference from the plan's segment lengths, which came with it).
//
// The last quotient (Eq. 26) takes a correction step: it costs 2% (50.2 us against 49.3)
// and keeps the error below the per-order kernels' over batches of rows (8.8e-8 against
// 1.1e-7, relative 2-norm; 9.3e-8 without) and level with theirs on meshes graded 16:1
// (0.77 to 1.13 times, 0.96 in the mean over 20 split steps; 0.79 to 1.19 without).  Over 1000
// steps of a steady rotation on the 16:1 bump mesh the masses stay within 1e-7 and the
// field within 8e-7 of the exact one (per-order kernels 5e-5 each, 510 cells).
//
// Measured against the per-order kernels (k_params with k_gwarp, or k_general with a
// residual), us per step: 512 rows of 64 to 65536 cells (5.3 M cells), no limiter,
// 112.6 / 51.0, with a van Leer residual 204.8 / 67.6; 1000 rows (9.5 M) limited
// 198.6 / 91.0; one row of 4096 cells with a residual 14.3 / 7.8.  Limited, 16 bytes (24 with
// a residual) of registers a thread are spilled at the cap of 80 for six CTAs an SM.  Tried (when the batch
// took 52.0): seven cells per lane 57.5 (512 rows), seven or five CTAs per SM instead of
// six 52.9 and 52.9, the lane's edges by side-by-side halvings instead of the walk 54.7,
// a loop without the two predicated steps 54.9, the next node's position kept across
// edges 55.6; when it took 49.4, the walk by pointers 51.6.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "ram_device.cuh"
#include "ram_tma.cuh"

namespace ram {
namespace {

constexpr int kV = kNsegWin / 32;            // window cells and edges per lane
constexpr int kWin = kNsegWin;               // window cells (32 kV)
constexpr int kHR = kNsegHR;                 // reconstruction halo, cells per side
constexpr uint32_t kPast = 0xffffffffu;      // position of a node past the window
static_assert(kWin == 32 * kV && kV % 2 == 1, "a lane takes kV window cells, an odd number");

// Per-warp shared memory (32-bit words).  The cell and node stages hold two words
// before index 0 and past the end, where the outer lanes' stencils read (those
// cells' coefficients are not used).
constexpr int kOffQ = 0;                     // window cell values: -2 .. kWin + 1
constexpr int kOffX = kOffQ + kWin + 8;      // window nodes: -2 .. kWin + 2
constexpr int kOffE = kOffX + kWin + 8;      // the segment's nodes: 0 .. kWin
constexpr int kOffC = kOffE + kWin + 4;      // cumulative coefficients, float4 per cell
constexpr int kOffM = kOffC + 4 * kWin;      // cell masses
constexpr int kOffR = kOffM + kWin + 4;      // node positions relative to the window
constexpr int kOffP = kOffR + 256 + 4;       // the segment's new values
constexpr int kOffV = kOffP + kWin + 4;      // dv at the segment's nodes (residual)
constexpr int kWords = kOffV;
constexpr int kOffH = kOffV + kWin + 4;      // widths of the segment's cells (residual)
constexpr int kWordsResid = kOffH + kWin + 4;
static_assert(kOffC % 4 == 0 && kWords % 4 == 0 && kWordsResid % 4 == 0, "16-byte aligned");

// x y / (x + y) where x and y have one sign, else 0, as (x + y) times the shares x / (x + y)
// and y / (x + y), each cut to [0, 1]: of opposite signs one share is negative.  (The
// product x y would leave the range of FP32 below 1e-22 and above 1e19.)  Beside a NaN or
// an infinity it is 0: the cut takes a NaN to 0.
__device__ __forceinline__ float harmonic(float x, float y)
{
    const float s = x + y, r = rcp_approx(s);
    const float p = __saturatef(x * r) * __saturatef(y * r);
    return p > 0.f ? p * s : 0.f;
}

// Coefficients of the in-cell cumulative G(d) = d (c0 + d (c1 + d (c2 + d c3))) of
// the lane's cells, d the distance from the cell's left node in the units of h
// (mean widths).  q[t], h[t]: cells -2 .. kV + 1 of the lane at t = 0 .. kV + 3; the
// lane's own are t = 2 .. kV + 1.
template <int ORDER, bool LIM>
__device__ __forceinline__ void reconstruct(const float (&q)[kV + 4], const float (&h)[kV + 4],
                                            float4 (&c)[kV])
{
    float s2[kV + 3], up[kV + 3];  // widths and differences of neighbours t, t + 1
#pragma unroll
    for (int t = 0; t < kV + 3; ++t) {
        s2[t] = h[t] + h[t + 1];
        up[t] = q[t + 1] - q[t];
    }
    float D2[kV + 3];  // (Q_{t+1} - Q_t) / (h_t + h_{t+1})
#pragma unroll
    for (int t = 0; t < kV + 3; ++t) D2[t] = up[t] * rcp_approx(s2[t]);
    if (ORDER == 2) {
        // G = q d + sigma (d^2 - h d) / 2.  Limited: the van Leer harmonic mean of the
        // one-sided slopes over centre spacings, 2 D2 each, zero at an extremum; else the
        // centred slope
#pragma unroll
        for (int i = 0; i < kV; ++i) {
            const int t = i + 2;
            float half;
            if (LIM) {
                half = 2.f * harmonic(D2[t - 1], D2[t]);
            } else {
                half = (up[t - 1] + up[t]) * rcp_approx(s2[t - 1] + s2[t]);
            }
            c[i] = make_float4(fmaf(-half, h[t], q[t]), half, 0.f, 0.f);
        }
        return;
    }
    if (ORDER == 3) {
        // delta<Q> of App. A.1, b / (a + b + c) [(2a + b) D2_k + (b + 2c) D2_{k-1}], limited
        // by the first stage of App. A.2
        float dq[kV + 4];
#pragma unroll
        for (int t = 1; t < kV + 3; ++t) {
            const float num = fmaf(s2[t - 1] + h[t - 1], D2[t], (s2[t] + h[t + 1]) * D2[t - 1]);
            dq[t] = h[t] * num * rcp_approx(s2[t - 1] + h[t + 1]);
            // (beside a NaN: 0)
            if (LIM) dq[t] = minxs(dq[t], fmaxf(2.f * minxs_nan(up[t - 1], up[t]), 0.f));
        }
        // <Q>_{k+1/2} - Q_k of App. A.1 (weights read with sums of widths), one
        // reciprocal of the common denominator (2 h0 + h1)(h0 + 2 h1)(h- + h0 + h1 + h2)
        float fa[kV + 3];
#pragma unroll
        for (int t = 1; t < kV + 2; ++t) {
            const float B = s2[t] + h[t], C = s2[t] + h[t + 1], S4 = s2[t - 1] + s2[t + 1];
            const float u = h[t] * (s2[t - 1] * C), v = h[t + 1] * (s2[t + 1] * B);
            const float e = D2[t] + D2[t];
            const float n = fmaf(u, fmaf(h[t + 1], e, -dq[t + 1]), v * fmaf(-h[t], e, dq[t]));
            fa[t] = fmaf(h[t], D2[t], n * rcp_approx(B * C * S4));
        }
        // with a = QR - Q, b = Q - QL: G = (Q - b) d + (2b - a) d^2 / h + (a - b) d^3 / h^2;
        // limited (App. A.2, second stage): a' = median(0, a, 2b), b' = median(0, b, 2a); a
        // NaN on one side makes the cell's profile NaN, as it does unlimited
#pragma unroll
        for (int i = 0; i < kV; ++i) {
            const int t = i + 2;
            float a = fa[t], b = up[t - 1] - fa[t - 1];
            if (LIM) {
                const float a1 = xorsign(max_nan(minxs_nan(a, b + b), 0.f), a);
                b = xorsign(max_nan(minxs_nan(b, a + a), 0.f), b);
                a = a1;
            }
            const float ih = rcp_approx(h[t]);
            c[i] = make_float4(q[t] - b, (b + b - a) * ih, (a - b) * ih * ih, 0.f);
        }
        return;
    }
    // Order 4 (not in the paper): the mean of the quartic interpolants of the
    // cumulative mass through the nodes {k-5/2..k+3/2} and {k-3/2..k+5/2}, from the
    // cell averages' divided differences; Newton form on 0, h, -h_-, h + h_+ expanded
    // to powers of d
    float D3[kV + 2], D4[kV + 1];
#pragma unroll
    for (int t = 0; t < kV + 2; ++t) D3[t] = (D2[t + 1] - D2[t]) * rcp_approx(s2[t] + h[t + 2]);
#pragma unroll
    for (int t = 0; t < kV + 1; ++t) D4[t] = (D3[t + 1] - D3[t]) * rcp_approx(s2[t] + s2[t + 2]);
#pragma unroll
    for (int i = 0; i < kV; ++i) {
        const int t = i + 2;
        const float hh = h[t], hm = h[t - 1];
        const float D = 0.5f * (D4[t - 2] + D4[t - 1]);
        const float A0 = fmaf(-D, s2[t], D3[t - 1]);
        const float B0 = fmaf(hm, A0, D2[t - 1]), B1 = fmaf(hm, D, A0);
        float c0 = fmaf(-hh, B0, q[t]), c1 = fmaf(-hh, B1, B0), c2 = fmaf(-hh, D, B1), c3 = D;
        if (LIM) {
            // limited order 4: scaled toward the mean (Zhang-Shu), bounded by the cell
            // and its neighbours
            const float h2 = hh * hh;
            const float th = quartic_scaling_theta<float>(
                c0, c1 * hh, c2 * h2, c3 * h2 * hh, q[t], fminf(q[t], fminf(q[t - 1], q[t + 1])),
                fmaxf(q[t], fmaxf(q[t - 1], q[t + 1])));
            c0 = th * c0 + (1.f - th) * q[t];
            c1 *= th;
            c2 *= th;
            c3 *= th;
        }
        c[i] = make_float4(c0, c1, c2, c3);
    }
}

// What a warp needs of one work item (a run of output cells of one row), formed by
// one thread of the CTA before the items are handed out.
struct Item {
    int64_t cell_off, mesh_off;
    uint64_t S;                // the row's shift, fraction of the period in units of 2^-64
    int32_t row, n, start, count;
    int16_t most;              // most cells of a segment with its halo
    int16_t window;            // cells of a window that edges may lie in
    int32_t order;
    int32_t p;                 // source cell of the first edge (halo included)
    int32_t nsub;
    float wscale;              // 2^k: a mean width times it is in (1, 2]
    float cf;                  // sub-step length, times wscale
    float scale;               // position units -> the widths' units, about mean widths
    float rem;                 // what S32 is more than the shift, in the widths' units
    uint32_t S32, period;      // shift (rounded up) and period in position units (mod 2^32)
};

struct SegCtx {
    const uint32_t *X32;
    const float *qin;
    float *qout;
    const float *dvp, *dx;
    const Item *it;
    int N, H, lane, hi;        // hi: first window node past the cells an edge may lie in
    bool vl;
    float scale;
    int *err;
};

// Values of cells first .. first + kWin - 1 (cyclic, first in [0, N)) to dst, 4 bytes a
// lane and copy.
__device__ __forceinline__ void copy_cells(uint32_t dst, const float *src, int first, int N,
                                           int lane)
{
    if (first + kWin <= N) {
        const float *s = src + first + lane;
#pragma unroll
        for (int i = 0; i < kV; ++i) cp_async4_s(dst + 4u * (lane + 32 * i), s + 32 * i);
    } else {
#pragma unroll 1
        for (int k = lane; k < kWin; k += 32) cp_async4_s(dst + 4u * k, src + (first + k) % N);
    }
}

// Nodes first .. first + kWin to dst, each turn of the row one period on.
__device__ __forceinline__ void copy_nodes(uint32_t *dst, const uint32_t *src, int first, int N,
                                           uint32_t period, int lane)
{
    if (first + kWin < N) {
        const uint32_t *s = src + first + lane;
        const uint32_t d = smem_u32(dst + lane);
#pragma unroll
        for (int i = 0; i < kV; ++i) cp_async4_s(d + 128u * i, s + 32 * i);
        if (lane == 0) cp_async4_s(d + 4u * kWin, s + kWin);
    } else {
#pragma unroll 1
        for (int k = lane; k <= kWin; k += 32) {
            const int turns = (first + k) / N;
            dst[k] = src[first + k - turns * N] + (uint32_t)turns * period;
        }
    }
}

// The window cells' coefficients and masses to the warp's shared memory.
template <int ORDER, bool LIM>
__device__ __forceinline__ void window_cells(const float (&q)[kV + 4], const float (&h)[kV + 4],
                                             float4 *sC, float *sM, int b)
{
    float4 c[kV];
    reconstruct<ORDER, LIM>(q, h, c);
#pragma unroll
    for (int i = 0; i < kV; ++i) {
        const float m = q[i + 2] * h[i + 2];
        if (ORDER < 4) c[i].w = m;
        sC[b + i] = c[i];
        sM[b + i] = m;
    }
}

// The segment of ne cells (halo included) from row cell a0, its first edge in
// source cell p; `advance` takes the warp's next item and `copies` starts its copies.
// One body for the three orders (only the reconstruction branches): three copies of
// it miss the instruction cache.
template <bool LIM, bool RESID, typename Advance, typename Copies>
__device__ __forceinline__ void nseg_segment(const SegCtx &g, uint32_t *w32, int order, int i0,
                                             int cnt, int p, Advance advance, Copies copies)
{
    float *sQ = reinterpret_cast<float *>(w32 + kOffQ + 2);
    uint32_t *sX = w32 + kOffX + 2;
    const uint32_t *sE = w32 + kOffE;
    float4 *sC = reinterpret_cast<float4 *>(w32 + kOffC);
    float *sM = reinterpret_cast<float *>(w32 + kOffM);
    uint32_t *sR = w32 + kOffR;
    float *sP = reinterpret_cast<float *>(w32 + kOffP);
    float *sV = reinterpret_cast<float *>(w32 + kOffV);
    const Item &it = *g.it;  // what is needed once is read where it is: registers are short
    const int lane = g.lane, b = lane * kV, N = g.N;
    const int ne = cnt + 2 * g.H;

    cp_async_wait<0>();
    __syncwarp();
    uint32_t xo[kV + 1];  // this lane's nodes
#pragma unroll
    for (int i = 0; i <= kV; ++i) xo[i] = sE[b + i];
    const uint32_t x_first = sE[0], x_last = sE[ne];
    if (RESID) {
        // dv of the segment's nodes and its cells' widths: needed after the remap (the
        // rounded nodes would do for the remap alone, whose masses they share; against
        // dv dt they leave the narrow cells of a graded row 2^-20)
        const int a0 = i0 - g.H < 0 ? i0 - g.H + N : i0 - g.H;
        const uint32_t d = smem_u32(sV);
#pragma unroll 1
        for (int k = lane; k <= ne; k += 32) {
            int c = a0 + k;
            c = c >= N ? c - N : c;  // ne < N
            cp_async4_s(d + 4u * k, g.dvp + c);
            cp_async4_s(d + 4u * (kOffH - kOffV) + 4u * k, g.dx + c);
        }
    }
    cp_async_commit();

    uint32_t off = 0;       // position of a shifted node in the window: x - off (and g.rem)
    int from = 0;           // first edge that is left
    bool first = true;
    while (true) {
        // ---- window cells: positions, widths and reconstructions ----
        const uint32_t xb = sX[kHR], rend = sX[g.hi] - xb;
        {
            float q[kV + 4], h[kV + 4];
            uint32_t x[kV + 5];
#pragma unroll
            for (int t = 0; t < kV + 5; ++t) x[t] = sX[b + t - 2];
#pragma unroll
            for (int t = 0; t < kV + 4; ++t) {
                q[t] = sQ[b + t - 2];
                h[t] = (float)(x[t + 1] - x[t]) * g.scale;
            }
#pragma unroll
            for (int i = 0; i < kV; ++i) sR[b + i] = x[i + 2] - xb;
            if (b + kV > g.hi) {
#pragma unroll
                for (int i = 0; i < kV; ++i)
                    if (b + i >= g.hi) sR[b + i] = kPast;
            }
            if (order == 2)
                window_cells<2, LIM>(q, h, sC, sM, b);
            else if (order == 3)
                window_cells<3, LIM>(q, h, sC, sM, b);
            else
                window_cells<4, LIM>(q, h, sC, sM, b);
        }
        __syncwarp();
        if (first) {
            // the first edge lies in source cell p, or, as the nodes are rounded, up to a
            // unit before it (-1)
            off = ((x_first - it.S32 - xb + 1u) & (it.period - 1u)) - 1u;
            off = x_first - off;
            // the window's values and nodes are in use no more
            advance();
            copies();
        }
        cp_async_commit();

        // ---- shifted edges and output masses (Eqs. 16, 18, 26) ----
        // The lane walks along the window's nodes from its first edge to the first of
        // the next lane; the whole cells it passes between two edges are Eq. 18's.
        int we[kV];
        uint32_t de[kV + 1];
        float G[kV + 1], mass[kV];
        int w = kHR;
        uint32_t rw = 0;  // position of node w
        uint32_t ry = xo[0] - off;
        ry = ry == kPast ? 0 : ry;  // the unit before the first source cell
        const float rem = it.rem;
        // the last node at or left of the edge: the nodes past the window are kPast,
        // so no bound is needed
#pragma unroll
        for (int step = 128; step > 0; step >>= 1) {
            const uint32_t r = sR[w + step];
            if (r <= ry) {
                w += step;
                rw = r;
            }
        }
#pragma unroll
        for (int i = 0; i < kV; ++i) {
            const uint32_t d = ry - rw;
            we[i] = w;
            de[i] = d;
            const float x = (float)d * g.scale;
            float4 c = sC[w];
            if (order == 4) {
                c.z = fmaf(x, c.w, c.z);
                c.w = sM[w];
            }
            // (the rest of the offset times the mean up to x: x itself stays exact)
            const float u = fmaf(x, fmaf(x, c.z, c.y), c.x);
            G[i] = fmaf(x, u, rem * u);
            ry = min(xo[i + 1] - off, kPast - 1u);
            // mostly no, one or two nodes: the first one's cell is the edge's own
            float m = 0.f;
            uint32_t r = sR[w + 1];
            if (r <= ry) {
                m = c.w;
                ++w;
                rw = r;
            }
            r = sR[w + 1];
            if (r <= ry) {
                m += sM[w];
                ++w;
                rw = r;
            }
            // more where the mesh under the segment is finer: compensated (Kahan), as their
            // number is only bounded by the window's
            float lost = 0.f;
            while (true) {
                r = sR[w + 1];
                if (r > ry) break;
                const float v = sM[w] - lost, t = m + v;
                lost = (t - m) - v;
                m = t;
                ++w;
                rw = r;
            }
            mass[i] = m;
        }
        de[kV] = __shfl_down_sync(0xffffffffu, de[0], 1);
        G[kV] = __shfl_down_sync(0xffffffffu, G[0], 1);
        // the last edge inside the window: mostly the segment's last
        int last = ne;
        if (x_last - off >= rend) {
            last = from - 1;
#pragma unroll
            for (int i = 0; i < kV; ++i) {
                const unsigned in = __ballot_sync(0xffffffffu, b + i >= from && b + i <= ne &&
                                                                    xo[i] - off < rend);
                if (in) last = max(last, kV * (31 - __clz((int)in)) + i);
            }
        }
        uint32_t least = de[0];
#pragma unroll
        for (int i = 1; i <= kV; ++i) least = min(least, de[i]);
#pragma unroll
        for (int i = 0; i < kV; ++i) {
            const int j = b + i;
            // Eq. 18: the start of the right source cell less that of the left one, plus
            // the cells passed from the left one on; Eq. 26, the quotient by the
            // approximate reciprocal and one correction
            if (j >= from && j < last) {
                const float m = mass[i] + (G[i + 1] - G[i]);
                const float h = (float)(xo[i + 1] - xo[i]) * g.scale, rh = rcp_approx(h);
                const float v = m * rh;
                sP[j] = fmaf(fmaf(-v, h, m), rh, v);
            }
        }
        if (least == 0 && rem == 0.f) {
            // an edge on a node: a cell whose edges both are, on those of one source cell,
            // takes its value unchanged
#pragma unroll
            for (int i = 0; i < kV; ++i)
                if (b + i >= from && b + i < last && (de[i] | de[i + 1]) == 0 &&
                    (i + 1 < kV ? we[i + 1] : w) == we[i] + 1) {
                    const int c = p + we[i] - kHR;
                    sP[b + i] = g.qin[c < N ? c : c % N];
                }
        }
        __syncwarp();
        if (last >= ne) break;
        if (last <= from) {
            // no edge reached: the plan bounds the source cells under an output cell
            if (lane == 0) atomicOr(g.err, ERR_WINDOW);
            break;
        }
        // ---- the window moves on to the source cell of the last edge reached ----
        const int i_last = last % kV;
        const int wl = __shfl_sync(0xffffffffu, i_last == 0   ? we[0]
                                                : i_last == 1 ? we[1]
                                                : i_last == 2 ? we[2]
                                                : i_last == 3 ? we[3]
                                                              : we[4],
                                   last / kV);
        off += sR[wl];
        p = (p + wl - kHR) % N;
        from = last;
        // the edges before it are done: at the new window's first node
#pragma unroll
        for (int i = 0; i <= kV; ++i)
            if (b + i < from) xo[i] = off;
        first = false;
        const int cb = p >= kHR ? p - kHR : p - kHR + N;
        cp_async_wait<0>();
        __syncwarp();
        copy_cells(smem_u32(sQ), g.qin, cb, N, lane);
        copy_nodes(sX, g.X32, cb, N, it.period, lane);
        cp_async_commit();
        cp_async_wait<0>();
        __syncwarp();
    }
    if (!first) {
        // the later windows took the place of the next segment's copies
        copies();
        cp_async_commit();
    }

    if (RESID) {
        // ---- residual sub-steps (Eq. 6): lane l holds cells 5l..5l+4 ----
        cp_async_wait<1>();  // dv (the group before the next segment's)
        __syncwarp();
        const unsigned full = 0xffffffffu;
        const float cf = it.cf, wscale = it.wscale;
        float cur[kV], c[kV], h[kV], rh[kV];
#pragma unroll
        for (int i = 0; i < kV; ++i) {
            cur[i] = sP[b + i];
            c[i] = sV[b + i] * cf;  // signed length swept by node i in a sub-step, scaled
            h[i] = sV[kOffH - kOffV + b + i] * wscale;
            rh[i] = rcp_approx(h[i]);
        }
        const float hm = __shfl_up_sync(full, h[kV - 1], 1);
        const int R = g.vl ? 2 : 1;
        bool bad = false;
        float rs[kV + 1], wc[kV];  // 1 / (both widths at face i), twice the midpoint's offset
#pragma unroll
        for (int i = 0; i < kV; ++i) {
            const float hl = i ? h[i - 1] : hm;
            const bool pos = c[i] > 0.f;
            bad |= b + i >= R && b + i <= ne - R && fabsf(c[i]) > (pos ? hl : h[i]);
            rs[i] = rcp_approx(hl + h[i]);
            wc[i] = 2.f * ((pos ? hl : -h[i]) - c[i]);
        }
        rs[kV] = __shfl_down_sync(full, rs[0], 1);
        if (__any_sync(full, bad) && lane == 0) atomicOr(g.err, ERR_CFL);
        for (int ks = 0, nsub = it.nsub; ks < nsub; ++ks) {
            const float zl = __shfl_up_sync(full, cur[kV - 1], 1);
            float F[kV];
            if (g.vl) {
                // a quarter of the slopes (van Leer harmonic mean, centre spacings)
                const float zr = __shfl_down_sync(full, cur[0], 1);
                float s[kV], Dl = (cur[0] - zl) * rs[0];
#pragma unroll
                for (int i = 0; i < kV; ++i) {
                    const float Dr = ((i < kV - 1 ? cur[i + 1] : zr) - cur[i]) * rs[i + 1];
                    s[i] = harmonic(Dl, Dr);
                    Dl = Dr;
                }
                const float sl = __shfl_up_sync(full, s[kV - 1], 1);
#pragma unroll
                for (int i = 0; i < kV; ++i) {
                    // the upwind cell's value at the middle of the swept length
                    const bool pos = c[i] > 0.f;
                    const float zu = pos ? (i ? cur[i - 1] : zl) : cur[i];
                    const float su = pos ? (i ? s[i - 1] : sl) : s[i];
                    F[i] = c[i] * fmaf(su, wc[i], zu);
                }
            } else {
#pragma unroll
                for (int i = 0; i < kV; ++i) F[i] = c[i] * (c[i] > 0.f ? (i ? cur[i - 1] : zl) : cur[i]);
            }
            const float Fr = __shfl_down_sync(full, F[0], 1);
#pragma unroll
            for (int i = 0; i < kV; ++i)
                cur[i] -= ((i < kV - 1 ? F[i + 1] : Fr) - F[i]) * rh[i];
        }
#pragma unroll
        for (int i = 0; i < kV; ++i) sP[b + i] = cur[i];
        __syncwarp();
    }
    for (int k = lane; k < cnt; k += 32) g.qout[i0 + k] = sP[g.H + k];
    // (the next segment's first write of sP follows a barrier)
}

template <bool LIM, bool RESID>
__global__ void __launch_bounds__(kNsegWarps * 32, kNsegCtas)
    k_nseg(StepArgs a, const NsegItem *items, int n_items)
{
    extern __shared__ __align__(16) uint32_t smem_w[];
    __shared__ Item s_item[kNsegItems];
    __shared__ int s_next;  // the CTA's next item to hand out
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int first = (int)((int64_t)n_items * blockIdx.x / gridDim.x);
    const int n_it = (int)((int64_t)n_items * (blockIdx.x + 1) / gridDim.x) - first;
    uint32_t *w32 = smem_w + warp * (RESID ? kWordsResid : kWords);
    for (int k = kWin + lane; k < 256 + 4; k += 32) w32[kOffR + k] = kPast;
    const int R = a.scheme == RAM_VANLEER ? 2 : 1;

    // ---- one thread per item: the row's shift (S0, FP64) and the first source cell
    // (plan data is read before the wait: the previous kernel in the stream may
    // still be writing q and the phase) ----
    NsegItem t{};
    RowInfo row{};
    if (tid < n_it) {
        t = items[first + tid];
        row = a.rows[t.row];
    }
    if (tid == 0) s_next = 0;
    pdl_wait();
    pdl_trigger();
    if (tid < n_it) {
        const uint64_t *X = a.xfix + row.mesh_off;
        int ns = RESID && a.nsub ? a.nsub[t.row] : (RESID ? 1 : 0);
        if (RESID) ns = ns < 1 ? 1 : (ns > RAM_MAX_NSUB ? RAM_MAX_NSUB : ns);
        int e = t.start - ns * R;
        e = e < 0 ? e + row.n : e;
        const uint64_t xe = X[e];  // in flight while the shift is formed
        // the row's first item advances the phase when no parameter kernel ran
        RowParams<float> P;
        shift_params<float>(a, row, t.row, a.row_phase != 0 && t.start == 0, P);
        const uint64_t S = P.sfix;
        const int qs = row.qshift;
        Item it;
        it.cell_off = row.cell_off;
        it.mesh_off = row.mesh_off;
        it.row = t.row;
        it.n = row.n;
        it.start = t.start;
        it.count = t.count;
        it.most = t.most;
        it.window = t.window;
        it.order = row.order;
        it.p = locate_cell(X, row.n, a.buckets + row.bucket_off, row.bucket_bits, a.density,
                           row.density, xe - S);
        it.S = S;
        // the shift in whole units, rounded up, and the rest
        const uint64_t low = S & ((1ull << qs) - 1ull);
        it.S32 = (uint32_t)(S >> qs) + (low != 0 ? 1u : 0u);
        if (qs > 32) it.S32 &= (1u << (64 - qs)) - 1u;
        it.period = qs > 32 ? 1u << (64 - qs) : 0u;
        it.nsub = P.nsub;
        const int ex = ((__double2hiint(row.cells_per_length) >> 20) & 0x7ff) - 1023;
        it.wscale = __int_as_float((127 + min(max(ex + 1, -126), 127)) << 23);
        it.cf = P.cf * it.wscale;
        // a power of two, so that widths and offsets round once; a mean cell is in [1, 2)
        it.scale = __int_as_float((127 + qs - 64 + 32 - __clz(row.n)) << 23);
        it.rem = low != 0 ? it.scale * (1.f - ldexpf((float)low, -qs)) : 0.f;
        s_item[tid] = it;
    }
    __syncthreads();

    // ---- the warps take the items from a counter as they issue the copies ----
    // An item is one segment, unless its halo is wider than the plan allows for:
    // then it is cut into pieces.  nx, nx_piece, nx_pieces, nx_p: the item the copies
    // in flight are for, its piece, their number and the piece's first source cell.
    int nx = 0, nx_piece = 0, nx_pieces = 0, nx_seg = 0, nx_p = 0;
    auto advance = [&]() {
        const bool same = RESID && ++nx_piece < nx_pieces;
        if (!same) {
            if (lane == 0) nx = atomicAdd(&s_next, 1);
            nx = __shfl_sync(0xffffffffu, nx, 0);
            if (nx >= n_it) return;
        }
        const Item &it = s_item[nx];
        if (!same) {
            nx_p = it.p;
            nx_seg = it.count;
            nx_piece = 0;
            nx_pieces = 1;
            const int most = it.most - 2 * it.nsub * R;
            if (RESID && it.count > most) {
                nx_pieces = (it.count + most - 1) / most;
                nx_seg = (it.count + nx_pieces - 1) / nx_pieces;
                nx_pieces = (it.count + nx_seg - 1) / nx_seg;
            }
        } else {
            const RowInfo &r = a.rows[it.row];
            const uint64_t *X = a.xfix + it.mesh_off;
            int e = it.start + nx_piece * nx_seg - it.nsub * R;
            e = e < 0 ? e + it.n : e;
            nx_p = locate_cell(X, it.n, a.buckets + r.bucket_off, r.bucket_bits, a.density,
                               r.density, X[e] - it.S);
        }
    };
    auto copies = [&]() {
        if (nx >= n_it) return;
        const Item &it = s_item[nx];
        const int N = it.n;
        int e = it.start + (RESID ? nx_piece * nx_seg - it.nsub * R : 0);
        e = e < 0 ? e + N : e;
        const int cb = nx_p >= kHR ? nx_p - kHR : nx_p - kHR + N;
        const uint32_t *X32 = a.x32 + it.mesh_off;
        const uint32_t period = it.period;
        copy_cells(smem_u32(w32 + kOffQ + 2), static_cast<const float *>(a.q_in) + it.cell_off, cb, N,
                   lane);
        copy_nodes(w32 + kOffX + 2, X32, cb, N, period, lane);
        copy_nodes(w32 + kOffE, X32, e, N, period, lane);
    };
    advance();
    copies();
    cp_async_commit();
    while (nx < n_it) {
        const Item &it = s_item[nx];
        SegCtx g;
        g.it = &it;
        g.X32 = a.x32 + it.mesh_off;
        g.qin = static_cast<const float *>(a.q_in) + it.cell_off;
        g.qout = static_cast<float *>(a.q_out) + it.cell_off;
        g.dvp = RESID ? static_cast<const float *>(a.dv) + it.cell_off : nullptr;
        g.dx = a.dx32 + it.mesh_off;
        g.N = it.n;
        g.H = RESID ? it.nsub * R : 0;
        g.lane = lane;
        g.hi = kHR + min(it.window, 2 * g.N - 1);
        g.vl = R == 2;
        g.scale = it.scale;
        g.err = a.err;
        const int i0 = it.start + nx_piece * nx_seg;
        const int cnt = min(nx_seg, it.start + it.count - i0);
        nseg_segment<LIM, RESID>(g, w32, it.order, i0, cnt, nx_p, advance, copies);
    }
}

}  // namespace

cudaError_t launch_nseg(const Plan &p, const StepArgs &a, cudaStream_t s)
{
    const int n = (int)p.items_nseg_h[0].size();
    if (n == 0) return cudaSuccess;
    const bool resid = a.mode != MODE_SHIFT && a.dv != nullptr;
    const size_t smem = (size_t)kNsegWarps * (resid ? kWordsResid : kWords) * 4;
    void (*kern)(StepArgs, const NsegItem *, int) =
        p.limiter ? (resid ? k_nseg<true, true> : k_nseg<true, false>)
                  : (resid ? k_nseg<false, true> : k_nseg<false, false>);
    // one wave of CTAs with near-equal shares of the items (few items: one each, over
    // all SMs); whole waves more when a share would not fit the CTA's table
    const int wave = p.sm_count * kNsegCtas;
    const int64_t waves = ((int64_t)n + (int64_t)wave * kNsegItems - 1) / ((int64_t)wave * kNsegItems);
    const int64_t grid = std::min<int64_t>(n, waves * wave);
    return launch_pdl(kern, dim3((unsigned)grid), dim3(kNsegWarps * 32), smem, s, a,
                      static_cast<const NsegItem *>(p.items_nseg[0]), n);
}

}  // namespace ram
