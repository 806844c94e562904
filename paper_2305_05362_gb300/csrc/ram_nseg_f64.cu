// RAM step on FP64 rows with their own non-uniform mesh (Sec. 3 on an arbitrary
// periodic mesh): the warp-segment form of ram_nseg.cu in double precision.
//
// The same windows, walk and residual as the FP32 kernel, on items of its own (nseg_fit in
// ram_segments.h), the plan's 64-bit positions (modulo 2^64, the period; rows about as
// long as a window or shorter halve the units, so that two turns fit) and FP64 widths.
// What differs is
// what bounds it: the FP64 pipe, which takes a warp instruction every 16 cycles of an
// SM.  So every reconstruction is formed once per cell, its shared terms once per
// face (neighbours by shuffles), the limiters decide on the bits, and quotients are
// Newton steps (ram_bits.cuh): about 46 FP64 instructions per source cell and 12 per
// edge for PPM.  The tiled kernels formed the reconstruction of the source cell at
// every edge, three delta<Q> and two faces each time, with range-checked divides: over
// 500 instructions a cell, the FP64 pipe 87-89% busy.  At the cap of 168 registers for
// three CTAs an SM the residual forms spill 316 (limited) and 188 bytes a thread, the
// limited shift 16.
//
// A window that holds a value of 2^1000 or more in magnitude, an infinity or a NaN, or
// only values below 2^-400, has its limiters decided by floating-point comparisons
// (BITS = false), as the tiled kernels do.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "ram_bits.cuh"
#include "ram_device.cuh"
#include "ram_tma.cuh"

namespace ram {
namespace {

constexpr int kV = kNsegWin / 32;            // window cells and edges per lane
constexpr int kWin = kNsegWin;
constexpr int kHR = kNsegHR;
constexpr uint64_t kPast = ~0ull;            // position of a node past the window
constexpr int kWarps = 4, kCtas = 3, kItems = 32;
constexpr unsigned kFull = 0xffffffffu;

// Per-warp shared memory (64-bit words); the stages hold words before index 0 and past
// the end, where the outer lanes' stencils read.
constexpr int kOffQ = 0;                     // window cell values: -2 .. kWin + 1
constexpr int kOffW = kOffQ + kWin + 8;      // window cell widths: -2 .. kWin + 1
constexpr int kOffX = kOffW + kWin + 8;      // window nodes: 0 .. kWin
constexpr int kOffE = kOffX + kWin + 4;      // the segment's nodes: 0 .. kWin
constexpr int kOffC = kOffE + kWin + 4;      // cumulative coefficients, four arrays
constexpr int kLenC = kWin + 4;
constexpr int kOffM = kOffC + 4 * kLenC;     // cell masses
constexpr int kOffR = kOffM + kWin + 4;      // node positions relative to the window
constexpr int kOffP = kOffR + 256 + 4;       // the segment's new values
constexpr int kOffH = kOffP + kWin + 4;      // widths of the segment's cells
constexpr int kOffV = kOffH + kWin + 4;      // dv at the segment's nodes
constexpr int kWords = kOffV + kWin + 4;

// sign(d) min(|d|, 2|dn|, 2|up|) where dn and up have one sign, else 0 (App. A.2, first
// stage)
template <bool BITS> __device__ __forceinline__ double limit_dq(double d, double dn, double up)
{
    if (BITS) return mag_signed(mag_min(mag(d), mag_up(mag_min(mag(dn), mag(up)), 1)), dn, up);
    if (!(up * dn > 0.0)) return 0.0;
    return copysign(fmin(fabs(d), fmin(2.0 * fabs(dn), 2.0 * fabs(up))), d);
}
// App. A.2, second stage, on a = QR - Q, b = Q - QL: flat at an extremum, else neither
// more than twice the other
template <bool BITS> __device__ __forceinline__ void limit_ab(double &a, double &b)
{
    if (BITS) {
        const unsigned long long ma = mag(a), mb = mag(b);
        const double a1 = mag_signed(mag_min(ma, mag_up(mb, 1)), a, b);
        b = mag_signed(mag_min(mb, mag_up(ma, 1)), b, a);
        a = a1;
    } else if (a * b <= 0.0) {
        a = b = 0.0;
    } else if (fabs(b) > 2.0 * fabs(a)) {
        b = 2.0 * a;
    } else if (fabs(a) > 2.0 * fabs(b)) {
        a = 2.0 * b;
    }
}
// dl dr / (dl + dr) where dl and dr have one sign, else 0
template <bool BITS> __device__ __forceinline__ double harmonic(double dl, double dr)
{
    if (BITS) return half_vl_bits(dl, dr);
    const double p = dl * dr;
    return p > 0.0 ? p / (dl + dr) : 0.0;
}

// Coefficients of the in-cell cumulative G(d) = d (c0 + d (c1 + d (c2 + d c3))) of the
// lane's cells.  q, h: the lane's kV cells with one more on each side (index 1 is the
// first own); terms of the faces and cells beyond come from the neighbouring lanes.
template <int ORDER, bool LIM, bool BITS>
__device__ __forceinline__ void reconstruct(const double (&q)[kV + 2], const double (&h)[kV + 2],
                                            double *sC, int b)
{
    double s2[kV + 2], up[kV + 1], D2[kV + 1];  // face t: between cells t and t + 1
#pragma unroll
    for (int t = 0; t <= kV; ++t) {
        s2[t] = h[t] + h[t + 1];
        up[t] = q[t + 1] - q[t];
    }
#pragma unroll
    for (int t = 1; t <= kV; ++t) D2[t] = up[t] * rcp_newton(s2[t]);
    D2[0] = __shfl_up_sync(kFull, D2[kV], 1);
    double *c0 = sC + b, *c1 = c0 + kLenC, *c2 = c1 + kLenC, *c3 = c2 + kLenC;
    if (ORDER == 2) {
#pragma unroll
        for (int i = 0; i < kV; ++i) {
            // half of the slope per unit length
            const double half = LIM ? 2.0 * harmonic<BITS>(D2[i], D2[i + 1])
                                    : (up[i] + up[i + 1]) * rcp_newton(s2[i] + s2[i + 1]);
            c0[i] = fma(-half, h[i + 1], q[i + 1]);
            c1[i] = half;
            c2[i] = 0.0;
        }
        return;
    }
    s2[kV + 1] = __shfl_down_sync(kFull, s2[1], 1);
    if (ORDER == 3) {
        double dq[kV + 2], fa[kV + 1];
#pragma unroll
        for (int t = 1; t <= kV; ++t) {
            const double num = fma(s2[t - 1] + h[t - 1], D2[t], (s2[t] + h[t + 1]) * D2[t - 1]);
            dq[t] = h[t] * num * rcp_newton(s2[t - 1] + h[t + 1]);
            if (LIM) dq[t] = limit_dq<BITS>(dq[t], up[t - 1], up[t]);
        }
        dq[kV + 1] = __shfl_down_sync(kFull, dq[1], 1);
#pragma unroll
        for (int t = 1; t <= kV; ++t) {
            // <Q>_{t+1/2} - Q_t (App. A.1)
            const double B = s2[t] + h[t], C = s2[t] + h[t + 1], S4 = s2[t - 1] + s2[t + 1];
            const double u = h[t] * (s2[t - 1] * C), v = h[t + 1] * (s2[t + 1] * B);
            const double e = D2[t] + D2[t];
            const double n = fma(u, fma(h[t + 1], e, -dq[t + 1]), v * fma(-h[t], e, dq[t]));
            fa[t] = fma(h[t], D2[t], n * rcp_newton(B * C * S4));
        }
        fa[0] = __shfl_up_sync(kFull, fa[kV], 1);
#pragma unroll
        for (int i = 0; i < kV; ++i) {
            double a = fa[i + 1], bb = up[i] - fa[i];
            if (LIM) limit_ab<BITS>(a, bb);
            const double ih = rcp_newton(h[i + 1]);
            c0[i] = q[i + 1] - bb;
            c1[i] = fma(2.0, bb, -a) * ih;
            c2[i] = (a - bb) * ih * ih;
        }
        return;
    }
    // order 4: divided differences of the cell averages (see ram_nseg.cu)
    double D3[kV + 2], D4[kV + 2];  // D3[t]: cells t .. t + 2, D4[t]: cells t .. t + 3
    const double D2r = __shfl_down_sync(kFull, D2[1], 1);  // face kV + 1
    const double hr = __shfl_down_sync(kFull, h[2], 1);    // cell kV + 2
#pragma unroll
    for (int t = 1; t <= kV; ++t) {
        D3[t] = ((t < kV ? D2[t + 1] : D2r) - D2[t]) *
                rcp_newton(s2[t] + (t < kV ? h[t < kV ? t + 2 : 0] : hr));
    }
    D3[0] = __shfl_up_sync(kFull, D3[kV], 1);
    D3[kV + 1] = __shfl_down_sync(kFull, D3[1], 1);
    const double s2rr = __shfl_down_sync(kFull, s2[2], 1);  // face kV + 2
#pragma unroll
    for (int t = 1; t <= kV; ++t)
        D4[t] = (D3[t + 1] - D3[t]) * rcp_newton(s2[t] + (t < kV ? s2[t + 2] : s2rr));
    const double D4l = __shfl_up_sync(kFull, D4[kV - 1], 1);  // cells -1 .. 2
    D4[0] = __shfl_up_sync(kFull, D4[kV], 1);
#pragma unroll
    for (int i = 0; i < kV; ++i) {
        const int t = i + 1;
        const double hh = h[t], hm = h[t - 1];
        const double D = 0.5 * ((i ? D4[t - 2] : D4l) + D4[t - 1]);
        const double A0 = fma(-D, s2[t], D3[t - 1]);
        const double B0 = fma(hm, A0, D2[t - 1]), B1 = fma(hm, D, A0);
        double k0 = fma(-hh, B0, q[t]), k1 = fma(-hh, B1, B0), k2 = fma(-hh, D, B1), k3 = D;
        if (LIM) {
            const double h2 = hh * hh;
            const double th = quartic_scaling_theta<double>(
                k0, k1 * hh, k2 * h2, k3 * h2 * hh, q[t], fmin(q[t], fmin(q[t - 1], q[t + 1])),
                fmax(q[t], fmax(q[t - 1], q[t + 1])));
            k0 = th * k0 + (1.0 - th) * q[t];
            k1 *= th;
            k2 *= th;
            k3 *= th;
        }
        c0[i] = k0;
        c1[i] = k1;
        c2[i] = k2;
        c3[i] = k3;
    }
}

template <bool LIM, bool BITS>
__device__ __forceinline__ void reconstruct_order(int order, const double (&q)[kV + 2],
                                                  const double (&h)[kV + 2], double *sC, int b)
{
    if (order == 2)
        reconstruct<2, LIM, BITS>(q, h, sC, b);
    else if (order == 3)
        reconstruct<3, LIM, BITS>(q, h, sC, b);
    else
        reconstruct<4, LIM, BITS>(q, h, sC, b);
}

// What a warp needs of one work item, formed by one thread of the CTA.
struct Item {
    int64_t cell_off, mesh_off;
    uint64_t S;            // the row's shift, fraction of the period in units of 2^-64
    double cf;             // sub-step length in the widths' units
    double dscale;         // position units to the widths' units
    int32_t wexp;          // these are widths times 2^wexp: a mean width is in (1/2, 1]
    int32_t row, n, start, count, order;
    int16_t most, window;
    int32_t half;          // 1: positions in units of 2^-63 of the period
    int32_t p;             // source cell of the first edge (halo included)
    int32_t nsub;
};

struct Seg {
    const uint64_t *X;
    const double *qin, *dx, *dvp;
    double *qout;
    int N, H, nsub, lane, hi, half, order, wexp;
    bool vl;
    double dscale, cf;
    uint64_t S, period;
    int *err;
};

__device__ __forceinline__ uint64_t below_past(uint64_t r) { return r == kPast ? kPast - 1 : r; }

__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// Values of cells first .. first + kWin - 1 (cyclic, first in [0, N)) to dst.
__device__ __forceinline__ void copy_cells(double *dst, const double *src, int first, int N, int lane)
{
    const uint32_t d = smem_u32(dst);
    if (first + kWin <= N) {
        const double *s = src + first + lane;
#pragma unroll
        for (int i = 0; i < kV; ++i) cp_async8(d + 8u * (lane + 32 * i), s + 32 * i);
    } else {
#pragma unroll 1
        for (int k = lane; k < kWin; k += 32) cp_async8(d + 8u * k, src + (first + k) % N);
    }
}

// Nodes first .. first + kWin to dst, each turn of the row one period on.
__device__ __forceinline__ void copy_nodes(uint64_t *dst, const uint64_t *src, int first, int N,
                                           int half, int lane)
{
    if (first + kWin < N && !half) {
        const uint64_t *s = src + first + lane;
        const uint32_t d = smem_u32(dst + lane);
#pragma unroll
        for (int i = 0; i < kV; ++i) cp_async8(d + 256u * i, s + 32 * i);
        if (lane == 0) cp_async8(d + 8u * kWin, s + kWin);
    } else {
#pragma unroll 1
        for (int k = lane; k <= kWin; k += 32) {
            const int turns = (first + k) / N;
            dst[k] = (src[first + k - turns * N] >> half) + (half ? (uint64_t)turns << 63 : 0ull);
        }
    }
}

// The residual sub-steps (Eq. 6) on the lane's cells; c: signed swept lengths of the
// nodes left of them, h their widths, rh the reciprocals.
template <bool BITS>
__device__ __forceinline__ void residual(double (&cur)[kV], const double (&c)[kV],
                                         const double (&h)[kV], const double (&rh)[kV], int nsub,
                                         bool vl)
{
    double rs[kV + 1], wc[kV];  // 1 / (sum of the widths at face i), twice the midpoint's offset
    if (vl) {
        const double hm = __shfl_up_sync(kFull, h[kV - 1], 1);
#pragma unroll
        for (int i = 0; i < kV; ++i) {
            const double hl = i ? h[i - 1] : hm;
            rs[i] = rcp_newton(hl + h[i]);
            const double o = (__double_as_longlong(c[i]) > 0 ? hl : -h[i]) - c[i];
            wc[i] = o + o;
        }
        rs[kV] = __shfl_down_sync(kFull, rs[0], 1);
    }
    for (int ks = 0; ks < nsub; ++ks) {
        const double zl = __shfl_up_sync(kFull, cur[kV - 1], 1);
        double F[kV];
        if (vl) {
            const double zr = __shfl_down_sync(kFull, cur[0], 1);
            double s[kV], Dl = (cur[0] - zl) * rs[0];
#pragma unroll
            for (int i = 0; i < kV; ++i) {
                const double Dr = ((i < kV - 1 ? cur[i + 1] : zr) - cur[i]) * rs[i + 1];
                s[i] = harmonic<BITS>(Dl, Dr);  // a quarter of the slope
                Dl = Dr;
            }
            const double sl = __shfl_up_sync(kFull, s[kV - 1], 1);
#pragma unroll
            for (int i = 0; i < kV; ++i) {
                const bool pos = __double_as_longlong(c[i]) > 0;
                const double zu = pos ? (i ? cur[i - 1] : zl) : cur[i];
                const double su = pos ? (i ? s[i - 1] : sl) : s[i];
                F[i] = c[i] * fma(su, wc[i], zu);
            }
        } else {
#pragma unroll
            for (int i = 0; i < kV; ++i)
                F[i] = c[i] * (__double_as_longlong(c[i]) > 0 ? (i ? cur[i - 1] : zl) : cur[i]);
        }
        const double Fr = __shfl_down_sync(kFull, F[0], 1);
#pragma unroll
        for (int i = 0; i < kV; ++i)
            cur[i] = fma((i < kV - 1 ? F[i + 1] : Fr) - F[i], -rh[i], cur[i]);
    }
}

// The segment of cnt output cells from i0 (halo H on both sides), its first edge in
// source cell p; `advance` takes the warp's next item, `copies` starts its copies.
template <bool LIM, bool RESID, typename Advance, typename Copies>
__device__ __forceinline__ void segment(const Seg &g, uint64_t *w64, int i0, int cnt, int p,
                                        Advance advance, Copies copies)
{
    double *sQ = reinterpret_cast<double *>(w64 + kOffQ + 2);
    double *sW = reinterpret_cast<double *>(w64 + kOffW + 2);
    uint64_t *sX = w64 + kOffX;
    const uint64_t *sE = w64 + kOffE;
    double *sC = reinterpret_cast<double *>(w64 + kOffC);
    double *sM = reinterpret_cast<double *>(w64 + kOffM);
    uint64_t *sR = w64 + kOffR;
    double *sP = reinterpret_cast<double *>(w64 + kOffP);
    double *sH = reinterpret_cast<double *>(w64 + kOffH);
    double *sV = reinterpret_cast<double *>(w64 + kOffV);
    const int lane = g.lane, b = lane * kV, N = g.N;
    const int ne = cnt + 2 * g.H;

    cp_async_wait<0>();
    __syncwarp();
    uint64_t xo[kV + 1];
#pragma unroll
    for (int i = 0; i <= kV; ++i) xo[i] = sE[b + i];
    const uint64_t x_first = sE[0], x_last = sE[ne];
    {
        // the segment's widths and dv, needed after the search
        const int a0 = i0 - g.H < 0 ? i0 - g.H + N : i0 - g.H;
        const uint32_t d = smem_u32(sH);
#pragma unroll 1
        for (int k = lane; k <= ne; k += 32) {
            int c = a0 + k;
            c = c >= N ? c - N : c;  // ne < N
            cp_async8(d + 8u * k, g.dx + c);
            if (RESID) cp_async8(d + 8u * (kOffV - kOffH) + 8u * k, g.dvp + c);
        }
    }
    cp_async_commit();

    uint64_t off = 0;       // position of a shifted node in the window: x - off
    int from = 0;           // first edge that is left
    bool first = true, odd = false;
    double rh[kV];          // 1 / the widths of the lane's output cells
    while (true) {
        // ---- window cells ----
        const uint64_t xb = sX[kHR], rend = sX[g.hi] - xb;
        {
            double q[kV + 2], h[kV + 2];
            unsigned top = 0;
#pragma unroll
            for (int t = 0; t < kV + 2; ++t) {
                q[t] = sQ[b + t - 1];
                h[t] = scale_pow2(sW[b + t - 1], g.wexp);
                if (t > 0 && t <= kV) top = max(top, mag_hi(q[t]));
            }
            top = __reduce_max_sync(kFull, top);
            odd = odd || top >= kMagBig || (top < kMagSmall && top > 0);
#pragma unroll
            for (int i = 0; i < kV; ++i) {
                sR[b + i] = b + i < g.hi ? sX[b + i] - xb : kPast;
                sM[b + i] = q[i + 1] * h[i + 1];
            }
            if (odd)
                reconstruct_order<LIM, false>(g.order, q, h, sC, b);
            else
                reconstruct_order<LIM, true>(g.order, q, h, sC, b);
        }
        __syncwarp();
        if (first) {
            // the first edge lies in source cell p, up to the rounding of halved units
            off = (x_first - g.S - xb) & (g.period - 1ull);
            if (g.half && off == g.period - 1ull) off = 0;
            off = x_first - off;
            advance();
            copies();
        }
        cp_async_commit();

        // ---- shifted edges and masses (Eqs. 16, 18) ----
        int we[kV];
        uint64_t de[kV + 1];
        double G[kV + 1], mass[kV];
        int w = kHR;
        uint64_t rw = 0;
        uint64_t ry = b < from ? 0ull : below_past(xo[0] - off);
#pragma unroll
        for (int step = 128; step > 0; step >>= 1) {
            const uint64_t r = sR[w + step];
            if (r <= ry) {
                w += step;
                rw = r;
            }
        }
#pragma unroll
        for (int i = 0; i < kV; ++i) {
            const uint64_t d = ry - rw;
            we[i] = w;
            de[i] = d;
            const double x = u64_to_double(d) * g.dscale;
            const double *c = sC + w;
            double y = c[2 * kLenC];
            if (g.order == 4) y = fma(x, c[3 * kLenC], y);
            G[i] = d == 0 ? 0.0 : x * fma(x, fma(x, y, c[kLenC]), c[0]);
            ry = b + i + 1 < from ? 0ull : below_past(xo[i + 1] - off);
            double m = 0.0;
            while (true) {
                const uint64_t r = sR[w + 1];
                if (r > ry) break;
                m += sM[w];
                ++w;
                rw = r;
            }
            mass[i] = m;
        }
        de[kV] = __shfl_down_sync(kFull, de[0], 1);
        G[kV] = __shfl_down_sync(kFull, G[0], 1);
        int last = ne;
        if (x_last - off >= rend) {
            last = from - 1;
#pragma unroll
            for (int i = 0; i < kV; ++i) {
                const unsigned in =
                    __ballot_sync(kFull, b + i >= from && b + i <= ne && xo[i] - off < rend);
                if (in) last = max(last, kV * (31 - __clz((int)in)) + i);
            }
        }
        if (first) {
            cp_async_wait<1>();  // the segment's widths
            __syncwarp();
#pragma unroll
            for (int i = 0; i < kV; ++i)
                rh[i] = rcp_newton(b + i < ne ? scale_pow2(sH[b + i], g.wexp) : 1.0);
        }
#pragma unroll
        for (int i = 0; i < kV; ++i) {
            const int j = b + i;
            if (j >= from && j < last) {
                double val = (mass[i] + (G[i + 1] - G[i])) * rh[i];
                if ((de[i] | de[i + 1]) == 0 && (i + 1 < kV ? we[i + 1] : w) == we[i] + 1) {
                    const int c = p + we[i] - kHR;
                    val = g.qin[c < N ? c : c % N];
                }
                sP[j] = val;
            }
        }
        __syncwarp();
        if (last >= ne) break;
        if (last <= from) {
            if (lane == 0) atomicOr(g.err, ERR_WINDOW);
            break;
        }
        // ---- the window moves on to the source cell of the last edge reached ----
        int wl = 0;
#pragma unroll
        for (int i = 0; i < kV; ++i)
            if (last % kV == i) wl = we[i];
        wl = __shfl_sync(kFull, wl, last / kV);
        off += sR[wl];
        p = (p + wl - kHR) % N;
        from = last;
        first = false;
        const int cb = p >= kHR ? p - kHR : p - kHR + N;
        cp_async_wait<0>();
        __syncwarp();
        copy_cells(sQ, g.qin, cb, N, lane);
        copy_cells(sW, g.dx, cb, N, lane);
        copy_nodes(sX, g.X, cb, N, g.half, lane);
        cp_async_commit();
        cp_async_wait<0>();
        __syncwarp();
    }
    if (!first) {
        copies();
        cp_async_commit();
    }

    if (RESID) {
        double cur[kV], c[kV], h[kV];
        unsigned top = 0;
#pragma unroll
        for (int i = 0; i < kV; ++i) {
            const bool in = b + i < ne;
            cur[i] = in ? sP[b + i] : 0.0;
            h[i] = in ? scale_pow2(sH[b + i], g.wexp) : 1.0;
            c[i] = in || b + i == ne ? sV[b + i] * g.cf : 0.0;
            top = max(top, mag_hi(c[i]));
        }
        odd = __any_sync(kFull, odd || top >= kMagBig);
        const double hm = __shfl_up_sync(kFull, h[kV - 1], 1);
        const int R = g.vl ? 2 : 1;
        bool bad = false;
#pragma unroll
        for (int i = 0; i < kV; ++i)
            bad |= b + i >= R && b + i <= ne - R &&
                   mag_above(c[i], __double_as_longlong(c[i]) > 0 ? (i ? h[i - 1] : hm) : h[i]);
        if (__any_sync(kFull, bad) && lane == 0) atomicOr(g.err, ERR_CFL);
        if (odd)
            residual<false>(cur, c, h, rh, g.nsub, g.vl);
        else
            residual<true>(cur, c, h, rh, g.nsub, g.vl);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < kV; ++i) sP[b + i] = cur[i];
        __syncwarp();
    }
    for (int k = lane; k < cnt; k += 32) g.qout[i0 + k] = sP[g.H + k];
    __syncwarp();
}

template <bool LIM, bool RESID>
__global__ void __launch_bounds__(kWarps * 32, kCtas)
    k_nseg_f64(StepArgs a, const NsegItem *items, int n_items)
{
    extern __shared__ __align__(16) uint64_t smem_d[];
    __shared__ Item s_item[kItems];
    __shared__ int s_next;  // the CTA's next item to hand out
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int first = (int)((int64_t)n_items * blockIdx.x / gridDim.x);
    const int n_it = (int)((int64_t)n_items * (blockIdx.x + 1) / gridDim.x) - first;
    uint64_t *w64 = smem_d + warp * kWords;
    for (int k = kWin + lane; k < 256 + 4; k += 32) w64[kOffR + k] = kPast;
    const int R = a.scheme == RAM_VANLEER ? 2 : 1;

    // one thread per item: the row's shift (S0) and the first source cell
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
        int ns = RESID ? (a.nsub ? a.nsub[t.row] : 1) : 0;
        if (RESID) ns = ns < 1 ? 1 : (ns > RAM_MAX_NSUB ? RAM_MAX_NSUB : ns);
        int e = t.start - ns * R;
        e = e < 0 ? e + row.n : e;
        const uint64_t xe = X[e];
        // the row's first item advances the phase when no parameter kernel ran
        RowParams<double> P;
        shift_params<double>(a, row, t.row, a.row_phase != 0 && t.start == 0, P);
        Item it;
        it.cell_off = row.cell_off;
        it.mesh_off = row.mesh_off;
        it.S = P.sfix;
        it.wexp = ((__double2hiint(row.cells_per_length) >> 20) & 0x7ff) - 1023;
        it.cf = P.cf * scale_pow2(1.0, it.wexp);
        it.half = row.half;
        it.dscale = scale_pow2(row.period, it.wexp) * (it.half ? 0x1p-63 : 0x1p-64);
        it.row = t.row;
        it.n = row.n;
        it.start = t.start;
        it.count = t.count;
        it.most = t.most;
        it.window = t.window;
        it.order = row.order;
        it.p = locate_cell(X, row.n, a.buckets + row.bucket_off, row.bucket_bits, a.density,
                           row.density, xe - P.sfix);
        it.nsub = P.nsub;
        s_item[tid] = it;
    }
    __syncthreads();

    // the warps take the items from a counter as they issue the copies; a halo wider
    // than the plan allows for cuts an item into pieces (see ram_nseg.cu)
    int nx = 0, nx_piece = 0, nx_pieces = 0, nx_seg = 0, nx_p = 0;
    auto advance = [&]() {
        const bool same = RESID && ++nx_piece < nx_pieces;
        if (!same) {
            if (lane == 0) nx = atomicAdd(&s_next, 1);
            nx = __shfl_sync(kFull, nx, 0);
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
        const uint64_t *X = a.xfix + it.mesh_off;
        copy_cells(reinterpret_cast<double *>(w64 + kOffQ + 2),
                   static_cast<const double *>(a.q_in) + it.cell_off, cb, N, lane);
        copy_cells(reinterpret_cast<double *>(w64 + kOffW + 2), a.dx64 + it.mesh_off, cb, N, lane);
        copy_nodes(w64 + kOffX, X, cb, N, it.half, lane);
        copy_nodes(w64 + kOffE, X, e, N, it.half, lane);
    };
    advance();
    copies();
    cp_async_commit();
    while (nx < n_it) {
        const Item &it = s_item[nx];
        Seg g;
        g.X = a.xfix + it.mesh_off;
        g.qin = static_cast<const double *>(a.q_in) + it.cell_off;
        g.dx = a.dx64 + it.mesh_off;
        g.dvp = RESID ? static_cast<const double *>(a.dv) + it.cell_off : nullptr;
        g.qout = static_cast<double *>(a.q_out) + it.cell_off;
        g.N = it.n;
        g.nsub = it.nsub;
        g.H = RESID ? it.nsub * R : 0;
        g.lane = lane;
        g.hi = kHR + min(it.window, 2 * g.N - 1);
        g.half = it.half;
        g.order = it.order;
        g.vl = R == 2;
        g.wexp = it.wexp;
        g.dscale = it.dscale;
        g.cf = it.cf;
        g.period = it.half ? 1ull << 63 : 0ull;
        g.S = it.half ? ((it.S >> 1) + (it.S & 1ull)) & (g.period - 1ull) : it.S;
        g.err = a.err;
        const int i0 = it.start + nx_piece * nx_seg;
        const int cnt = min(nx_seg, it.start + it.count - i0);
        segment<LIM, RESID>(g, w64, i0, cnt, nx_p, advance, copies);
    }
}

template <bool LIM, bool RESID>
cudaError_t launch_t(const Plan &p, const StepArgs &a, cudaStream_t s)
{
    const size_t smem = (size_t)kWarps * kWords * sizeof(uint64_t);
    static bool configured[64] = {false};
    const int dev = p.device < 64 ? p.device : 63;
    if (!configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(k_nseg_f64<LIM, RESID>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    // one wave of CTAs with near-equal shares of the items, whole waves more when a
    // share would not fit the CTA's table
    const int n = (int)p.items_nseg_h[1].size();
    const int wave = p.sm_count * kCtas;
    const int64_t waves = ((int64_t)n + (int64_t)wave * kItems - 1) / ((int64_t)wave * kItems);
    const int64_t grid = std::min<int64_t>(n, waves * wave);
    return launch_pdl(k_nseg_f64<LIM, RESID>, dim3((unsigned)grid), dim3(kWarps * 32), smem, s, a,
                      static_cast<const NsegItem *>(p.items_nseg[1]), n);
}

}  // namespace

cudaError_t launch_nseg_f64(const Plan &p, const StepArgs &a, cudaStream_t s)
{
    if (p.items_nseg_h[1].empty()) return cudaSuccess;
    const bool resid = a.mode != MODE_SHIFT && a.dv != nullptr;
    if (p.limiter)
        return resid ? launch_t<true, true>(p, a, s) : launch_t<true, false>(p, a, s);
    return resid ? launch_t<false, true>(p, a, s) : launch_t<false, false>(p, a, s);
}

}  // namespace ram
