// Transpose of one linear RAM step (limiter off, donor residual) on uniform rows
// (rows with their own mesh: ram_adjoint_nu.cu).
//
// With the limiters off the shift of a uniform row is a fixed stencil: output
// cell m takes the right part of source cell p = m-K-1 and the left part of p+1
// (Eq. 18), and the left partial A_p of the reconstruction is linear in
// Q_{p-2..p+2}, so Q'_m = sum_u beta_u Q_{m-K-1+u} (u = -2..3) with
// beta_u = [u == 0] - alpha_u + alpha_{u-1}.  Its transpose gathers
// g_in[j] = sum_u beta_u g'[j+K+1-u].  The donor residual sub-step
// Q_i <- Q_i - (F_{i+1} - F_i), F_j = c_j Q_up(j), has the transpose
// g_k <- g_k + [c_{k+1} >= 0] c_{k+1} h_{k+1} + [c_k < 0] c_k h_k with
// h_j = g_j - g_{j-1}, and dL/d dv_j = sum over sub-steps of cf Q_up(j) h_j, where
// the forward sub-step states are recomputed from the step input.  The upwind
// side at c_j = 0 is the left cell.
//
// Two kernels.  k_adj_seg (rows of at least 512 cells on 16-byte boundaries) gives
// each warp a run of output cells, V a lane, in registers: one pass over g, dv and
// the step input forms both gradients, neighbours by shuffles, and FP32 rows form
// their shift themselves (no parameter kernel).  k_adj_uniform takes the other rows:
// blockIdx.y = 0 computes g_in for a tile of source cells, blockIdx.y = 1 adds dL/d
// dv for the tile's interfaces (each interface in exactly one tile, so there are no
// atomics).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <vector>

#include "ram_bits.cuh"
#include "ram_device.cuh"

namespace ram {
namespace {

constexpr int kMaxSub = RAM_MAX_NSUB;

// alpha_{-2..2}: coefficients of Q_{p-2..p+2} in the left partial A_p (limiter off)
template <typename T, int ORDER>
__device__ __forceinline__ void alpha_coeffs(const RowParams<T> &P, T al[5])
{
    for (int s = 0; s < 5; ++s) al[s] = T(0);
    if (ORDER == 2) {
        // A = Q c0 + (Q_{p+1} - Q_{p-1})/2 c1
        al[1] = -T(0.5) * P.c[1];
        al[2] = P.c[0];
        al[3] = T(0.5) * P.c[1];
    } else if (ORDER == 3) {
        // A = QL c0 + QR c1 + Q c2 with QL = 7/12(Q_{p-1}+Q_p) - 1/12(Q_{p-2}+Q_{p+1})
        // and QR = 7/12(Q_p+Q_{p+1}) - 1/12(Q_{p-1}+Q_{p+2})
        const T a = T(7) / T(12), b = T(1) / T(12);
        al[0] = -b * P.c[0];
        al[1] = a * P.c[0] - b * P.c[1];
        al[2] = a * P.c[0] + a * P.c[1] + P.c[2];
        al[3] = -b * P.c[0] + a * P.c[1];
        al[4] = -b * P.c[1];
    } else {
        for (int s = 0; s < 5; ++s) al[s] = P.c[s];
    }
}

// beta_u (u = -2..3) from the left partial's coefficients
template <typename T, int ORDER>
__device__ __forceinline__ void beta_coeffs(const RowParams<T> &P, T beta[6])
{
    T al[5];
    alpha_coeffs<T, ORDER>(P, al);
#pragma unroll
    for (int u = -2; u <= 3; ++u)
        beta[u + 2] = (u == 0 ? T(1) : T(0)) - (u <= 2 ? al[u <= 2 ? u + 2 : 0] : T(0)) +
                      (u >= -1 ? al[u >= -1 ? u + 1 : 0] : T(0));
}

constexpr int kSegWarps = 4;

// Cells per lane of the warp-segment kernel.
template <typename T> constexpr int kSegV = sizeof(T) == 4 ? 8 : 4;

// Halo cells at each end of a warp's 32 V cells, whole 16-byte vectors: the sub-steps
// spoil nsub cells at each end, the gather takes 2 on the left and 3 on the right.
template <typename T> __host__ __device__ constexpr int seg_halo(int nsub)
{
    return (nsub + 3 + 16 / (int)sizeof(T) - 1) / (16 / (int)sizeof(T)) * (16 / (int)sizeof(T));
}

__device__ __forceinline__ int wrap_twice(int c, int N)  // c within (-2N, 2N)
{
    if (c < 0) c += N;
    if (c < 0) c += N;
    if (c >= N) c -= N;
    if (c >= N) c -= N;
    return c;
}

// Whether x is above 0 (or a NaN); whether x, not -0.0, is at least 0 and below 0 (FP64: on
// the integer pipe)
__device__ __forceinline__ bool above_0(float x) { return x > 0.f; }
__device__ __forceinline__ bool above_0(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool upward(float x) { return x >= 0.f; }
__device__ __forceinline__ bool downward(float x) { return x < 0.f; }
__device__ __forceinline__ bool upward(double x)
{
    return (unsigned long long)__double_as_longlong(x) <= 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool downward(double x)
{
    return __double2hiint(x) < 0 && mag(x) <= 0x7ff0000000000000ull;
}

template <typename T> struct Vec16;
template <> struct Vec16<float> {
    using V = float4;
};
template <> struct Vec16<double> {
    using V = double2;
};

// M values (whole vectors) from the lane's cells first, first + 1, ... (cyclic), first =
// wfirst + lane V; wfirst is the warp's, in [0, N), whole vectors like N.
template <typename T, int M, int V>
__device__ __forceinline__ void load_cells(const T *row, int wfirst, int lane, int N, T (&out)[M])
{
    using Vec = typename Vec16<T>::V;
    constexpr int VEC = 16 / sizeof(T);
    Vec v[M / VEC];
    if (wfirst + 31 * V + M <= N) {
        const T *src = row + wfirst + lane * V;
#pragma unroll
        for (int c = 0; c < M / VEC; ++c) v[c] = *reinterpret_cast<const Vec *>(src + c * VEC);
    } else {
#pragma unroll
        for (int c = 0; c < M / VEC; ++c) {
            const int i = wfirst + lane * V + c * VEC;
            v[c] = *reinterpret_cast<const Vec *>(row + (i >= N ? i - N : i));
        }
    }
#pragma unroll
    for (int c = 0; c < M / VEC; ++c) {
        const T *e = reinterpret_cast<const T *>(&v[c]);
#pragma unroll
        for (int k = 0; k < VEC; ++k) out[c * VEC + k] = e[k];
    }
}

// Whether two-float arithmetic holds a row's shift as well as FP64 does for FP32 cells
// (the fraction of a cell to 2^-26): less than 2^20 cells, the factors of v0 dt N / L zero
// or well inside the FP32 range.  By their exponents.
__device__ __forceinline__ bool two_float_holds(const StepArgs &a, const RowInfo &row, int r)
{
    const auto expo = [](double x) {
        return (int)((__double_as_longlong(x) >> 52) & 0x7FF) - 1023;
    };
    const int ev = expo(a.v0[r]), ed = expo(a.dt), ec = expo(row.cells_per_length);
    const auto inside = [](int e) { return e == -1023 || (e >= -60 && e <= 60); };
    return inside(ev) && inside(ed) && inside(ec) && ev + ed + ec < 18;
}

// One segment of k_adj_seg: output cells [out0, out0 + stride) of a row.
template <typename T, int ORDER>
__device__ __forceinline__ void adj_segment(const StepArgs &a, const RowInfo &row,
                                            const RowParams<T> &P, const T (&beta)[6], T *st,
                                            int out0, int stride, int H, int lane, const T *g_out,
                                            T *g_in, T *g_dv)
{
    constexpr int V = kSegV<T>, VEC = 16 / sizeof(T);
    using Vec = typename Vec16<T>::V;
    const int N = row.n, nsub = P.nsub;
    const unsigned full = 0xffffffffu;
    const int m0 = out0 - H + lane * V;  // the lane's first cell (may wrap)
    const int mw = wrap_twice(out0 - H, N);  // the warp's first

    T g[V];
    load_cells<T, V, V>(g_out + row.cell_off, mw, lane, N, g);
    if (nsub > 0) {
        // the faces' Courant numbers (face i: left node), and bit i of `up`, `down`: c[i] is
        // at least 0, below 0 (neither for a NaN).  A cell takes nothing from a face that it
        // is downwind of: there 0 times what is not finite would reach it
        T c[V];
        unsigned up = 0, down = 0;
        load_cells<T, V, V>(static_cast<const T *>(a.dv) + row.cell_off, mw, lane, N, c);
#pragma unroll
        for (int i = 0; i < V; ++i) {
            c[i] = fma(c[i], P.cf, T(0));  // -0.0: 0.0
            up |= upward(c[i]) ? 1u << i : 0u;
            down |= downward(c[i]) ? 1u << i : 0u;
        }
        const T cr = __shfl_down_sync(full, c[0], 1);
        up |= (__shfl_down_sync(full, up, 1) & 1u) << V;
        T acc[V], q0[V];
#pragma unroll
        for (int i = 0; i < V; ++i) acc[i] = T(0);
        if (g_dv != nullptr) {
            // the shifted field: source cells p - 2 .. p + V + 2, p = m0 - K - 1, from a
            // vector boundary
            const int off = ((-P.K - 1) % VEC + VEC) % VEC;
            T w[V + 3 * VEC];
            load_cells<T, V + 3 * VEC, V>(static_cast<const T *>(a.q_in) + row.cell_off,
                                          wrap_twice(mw - P.K - 1 - off - VEC, N), lane, N, w);
#pragma unroll
            for (int o = 0; o < VEC; ++o)
                if (o == off) {
#pragma unroll
                    for (int i = 0; i < V; ++i) {
                        // w[o + VEC + i + u] holds cell p + i + u
                        T v = T(0);
#pragma unroll
                        for (int u = -2; u <= 3; ++u) v += beta[u + 2] * w[o + VEC + i + u];
                        q0[i] = P.whole ? w[o + VEC + i + 1] : v;
                    }
                }
        }
        for (int k = nsub - 1; k >= 0; --k) {
            // transposed flux differences h_i = g_i - g_{i-1}
            T h[V + 1];
            h[0] = g[0] - __shfl_up_sync(full, g[V - 1], 1);
#pragma unroll
            for (int i = 1; i < V; ++i) h[i] = g[i] - g[i - 1];
            h[V] = __shfl_down_sync(full, h[0], 1);
            if (g_dv != nullptr) {
                T q[V];
#pragma unroll
                for (int i = 0; i < V; ++i) q[i] = q0[i];
                for (int s = 0; s < k; ++s) {
                    const T zl = __shfl_up_sync(full, q[V - 1], 1);
                    T F[V + 1];
#pragma unroll
                    for (int i = 0; i < V; ++i)
                        F[i] = c[i] * (above_0(c[i]) ? (i ? q[i - 1] : zl) : q[i]);
                    F[V] = __shfl_down_sync(full, F[0], 1);
#pragma unroll
                    for (int i = 0; i < V; ++i) q[i] -= F[i + 1] - F[i];
                }
                const T zl = __shfl_up_sync(full, q[V - 1], 1);
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    // the upwind cell, the left one at c = 0
                    const T qu = up >> i & 1u ? (i ? q[i - 1] : zl) : q[i];
                    acc[i] = fma(qu, h[i], acc[i]);
                }
            }
#pragma unroll
            for (int i = 0; i < V; ++i) {
                if (down >> i & 1u) g[i] = fma(c[i], h[i], g[i]);
                if (up >> (i + 1) & 1u) g[i] = fma(i + 1 < V ? c[i + 1 < V ? i + 1 : 0] : cr, h[i + 1], g[i]);
            }
        }
        if (g_dv != nullptr) {
            T *gd = g_dv + row.cell_off;
#pragma unroll
            for (int c = 0; c < V / VEC; ++c) {
                const int li = lane * V + c * VEC, m = m0 + c * VEC;
                if (li >= H && li < H + stride && m < N) {
                    Vec v = *reinterpret_cast<const Vec *>(gd + m);
                    T *e = reinterpret_cast<T *>(&v);
#pragma unroll
                    for (int k = 0; k < VEC; ++k) e[k] = fma(P.cf, acc[c * VEC + k], e[k]);
                    *reinterpret_cast<Vec *>(gd + m) = v;
                }
            }
        }
    }

    // ---- the shift's transpose: local cell i gives g_in[m0 + i - K] ----
    T e[V + 5];  // g' at local cells -2 .. V + 2
    e[0] = __shfl_up_sync(full, g[V - 2], 1);
    e[1] = __shfl_up_sync(full, g[V - 1], 1);
#pragma unroll
    for (int i = 0; i < V; ++i) e[i + 2] = g[i];
#pragma unroll
    for (int i = 0; i < 3; ++i) e[V + 2 + i] = __shfl_down_sync(full, g[i], 1);
#pragma unroll
    for (int i = 0; i < V; ++i) {
        T v = T(0);
#pragma unroll
        for (int u = -2; u <= 3; ++u) v += beta[u + 2] * e[i + 3 - u];
        st[lane * V + i] = P.whole ? g[i] : v;
    }
    __syncwarp();
    T *gi = g_in + row.cell_off;
    const int cnt = min(stride, N - out0);
    for (int k = lane; k < cnt; k += 32) {
        const int j = out0 + k - P.K;
        gi[j < 0 ? j + N : j] = st[H + k];
    }
    __syncwarp();  // the stage is free again
}

// One warp per segment of output cells [out0, out0 + stride) of a row, its 32 V cells
// from out0 - H on; lane l holds V consecutive ones.  In one pass: the states of the
// donor sub-steps from the step input (state k from state 0 again for each k: one or
// two sub-steps in earnest), the sub-steps' transpose in reverse with dL/d dv, and
// the shift's transpose, g_in[m - K] = sum_u beta_u g'[m + 1 - u].  The shift by K
// leaves g_in unaligned, so it passes through shared memory to be stored a lane a
// word.
//
// Bound by latency at 512 x 2048 cells, where a step's 24 bytes a cell stay in L2:
// steps back to back, one or two sub-steps, PPM, 28.6 us with the tile passes of
// k_adj_uniform and the parameter kernel before them, 8.7 so (FP32; FP64 103 and 63;
// with the upwind sides selected by masks, which took 9.1 to 9.2 us in FP32 timed by
// itself, 58).
// A segment a warp, so that few rows still fill the SMs; registers capped for six
// CTAs an SM in FP32 (9.25 us uncapped).
template <typename T, int ORDER>
__global__ void __launch_bounds__(kSegWarps * 32, sizeof(T) == 4 ? 6 : 4)
    k_adj_seg(StepArgs a, const int32_t *row_ids, const RowParams<T> *pars, const T *g_out,
              T *g_in, T *g_dv)
{
    constexpr int V = kSegV<T>;
    __shared__ __align__(16) T stage[kSegWarps][32 * V];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int seg0 = blockIdx.y * kSegWarps + warp;
    const int r = row_ids[blockIdx.x];
    const RowInfo row = a.rows[r];
    pdl_wait();
    pdl_trigger();
    RowParams<T> P;
    if constexpr (sizeof(T) == 4) {
        if (two_float_holds(a, row, r))
            shift_params_two_float(a, row, r, seg0 == 0 && lane == 0, P);
        else
            shift_params<float>(a, row, r, false, P);
    } else {
        P = pars[r];
    }
    const int N = row.n, nsub = P.nsub;
    const int H = seg_halo<T>(nsub);
    const int stride = 32 * V - 2 * H;
    T beta[6];
    beta_coeffs<T, ORDER>(P, beta);
    // one segment a warp, unless the row has more than a grid can
    for (int64_t seg = seg0; seg * stride < N; seg += (int64_t)gridDim.y * kSegWarps)
        adj_segment<T, ORDER>(a, row, P, beta, stage[warp], (int)(seg * stride), stride, H, lane,
                              g_out, g_in, g_dv);
}

template <typename T, int ORDER>
__global__ void __launch_bounds__(256)
    k_adj_uniform(StepArgs a, const RowParams<T> *pars, const T *g_out, T *g_in, T *g_dv,
                  int tcap)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int wcap = tcap + 2 * kMaxSub + 16;
    T *s0 = reinterpret_cast<T *>(smem_raw);  // wcap
    T *s1 = s0 + wcap;                        // wcap
    T *sv = s1 + wcap;                        // wcap + 1 (Courant numbers)
    T *st = sv + wcap + 1;                    // forward states: kMaxSub x wcap

    const Tile tile = a.tiles[blockIdx.x];
    const RowInfo row = a.rows[tile.row];
    const int N = row.n;
    const int tid = threadIdx.x, nth = blockDim.x;
    pdl_wait();
    const RowParams<T> P = pars[tile.row];
    const int nsub = P.nsub;
    const int K = P.K;
    const int A0 = tile.start, TN = tile.count;
    const T *g = g_out + row.cell_off;
    const T *dv = nsub > 0 ? static_cast<const T *>(a.dv) + row.cell_off : nullptr;
    T al[5];
    alpha_coeffs<T, ORDER>(P, al);
    T beta[6];  // beta_u for u = -2..3
    for (int u = -2; u <= 3; ++u) {
        const T am = (u - 1 >= -2 && u - 1 <= 2) ? al[u - 1 + 2] : T(0);
        const T a0 = (u >= -2 && u <= 2) ? al[u + 2] : T(0);
        beta[u + 2] = (u == 0 ? T(1) : T(0)) - a0 + am;
    }

    if (blockIdx.y == 0) {
        // ---- g_in on source cells [A0, A0+TN): g' on [A0+K-2, A0+K+TN+3) ----
        const int m0 = A0 + K - 2 - nsub;  // first cell of g_out needed
        const int nm = TN + 5 + 2 * nsub;
        for (int i = tid; i < nm; i += nth) s0[i] = g[wrap_index((int64_t)m0 + i, N)];
        if (nsub > 0)
            for (int i = tid; i <= nm; i += nth) sv[i] = dv[wrap_index((int64_t)m0 + i, N)] * P.cf;
        __syncthreads();
        T *cur = s0, *nxt = s1;
        for (int k = 0; k < nsub; ++k) {
            // valid input [k, nm-k) -> output [k+1, nm-k-1)
            for (int i = k + 1 + tid; i < nm - k - 1; i += nth) {
                const T hL = cur[i] - cur[i - 1];      // h at interface i
                const T hR = cur[i + 1] - cur[i];      // h at interface i+1
                const T cL = sv[i], cR = sv[i + 1];
                T v = cur[i];
                if (cR >= T(0)) v += cR * hR;
                if (cL < T(0)) v += cL * hL;
                nxt[i] = v;
            }
            __syncthreads();
            T *t = cur;
            cur = nxt;
            nxt = t;
        }
        // gather: g_in[j] = sum_u beta_u g'[j+K+1-u]; g'[m] sits at cur[m - m0]
        T *gi = g_in + row.cell_off;
        for (int j = tid; j < TN; j += nth) {
            const int base = (A0 + j) + K + 1 - m0;  // index of g'[j+K+1]
            T acc;
            if (P.whole) {
                acc = cur[base - 1];  // Q'_m = Q_{m-K}: g_in[j] = g'[j+K]
            } else {
                acc = T(0);
#pragma unroll
                for (int u = -2; u <= 3; ++u) acc += beta[u + 2] * cur[base - u];
            }
            gi[A0 + j] = acc;
        }
        return;
    }

    // ---- dL/d dv on interfaces [A0, A0+TN) ----
    if (nsub == 0 || g_dv == nullptr) return;
    // forward states on cells [A0-nsub, A0+TN+nsub): Q' from the step input
    const int c0 = A0 - nsub;
    const int nc = TN + 2 * nsub;
    const T *qin = static_cast<const T *>(a.q_in) + row.cell_off;
    // Q'_m = sum_u beta_u Q_{m-K-1+u}
    for (int i = tid; i < nc; i += nth) {
        const int m = c0 + i;
        T v;
        if (P.whole) {
            v = qin[wrap_index((int64_t)m - K, N)];
        } else {
            v = T(0);
#pragma unroll
            for (int u = -2; u <= 3; ++u) v += beta[u + 2] * qin[wrap_index((int64_t)m - K - 1 + u, N)];
        }
        st[i] = v;
    }
    for (int i = tid; i <= nc; i += nth) sv[i] = dv[wrap_index((int64_t)c0 + i, N)] * P.cf;
    __syncthreads();
    // forward donor sub-steps: state k+1 from state k, valid range shrinking by one
    for (int k = 0; k + 1 < nsub; ++k) {
        const T *q = st + (size_t)k * wcap;
        T *qn = st + (size_t)(k + 1) * wcap;
        for (int i = k + 1 + tid; i < nc - k - 1; i += nth) {
            const T cL = sv[i], cR = sv[i + 1];
            const T FL = cL * (cL > T(0) ? q[i - 1] : q[i]);
            const T FR = cR * (cR > T(0) ? q[i] : q[i + 1]);
            qn[i] = q[i] - (FR - FL);
        }
        __syncthreads();
    }
    // backward sweep: g^(nsub) = g_out on the same cells
    for (int i = tid; i < nc; i += nth) s0[i] = g[wrap_index((int64_t)c0 + i, N)];
    __syncthreads();
    T *cur = s0, *nxt = s1;
    T *gd = g_dv + row.cell_off;
    T acc_local[8];
    const int per = (TN + nth - 1) / nth;  // interfaces per thread (<= 8 by the launcher)
    for (int r = 0; r < 8; ++r) acc_local[r] = T(0);
    for (int k = nsub - 1; k >= 0; --k) {
        const T *q = st + (size_t)k * wcap;
        // interfaces j in [A0, A0+TN): cell index i = j - c0 (interface i, between i-1 and i)
        for (int r = 0; r < per; ++r) {
            const int jj = tid * per + r;
            if (jj < TN) {
                const int i = jj + nsub;
                const T c = sv[i];
                const T qup = (c >= T(0)) ? q[i - 1] : q[i];
                acc_local[r] += P.cf * qup * (cur[i] - cur[i - 1]);
            }
        }
        // g^(k) from g^(k+1) on the shrinking range
        const int lo = (nsub - k), hi = nc - (nsub - k);
        for (int i = lo + tid; i < hi; i += nth) {
            const T hL = cur[i] - cur[i - 1];
            const T hR = cur[i + 1] - cur[i];
            const T cL = sv[i], cR = sv[i + 1];
            T v = cur[i];
            if (cR >= T(0)) v += cR * hR;
            if (cL < T(0)) v += cL * hL;
            nxt[i] = v;
        }
        __syncthreads();
        T *t = cur;
        cur = nxt;
        nxt = t;
    }
    for (int r = 0; r < per; ++r) {
        const int jj = tid * per + r;
        if (jj < TN) gd[A0 + jj] += acc_local[r];
    }
}

template <typename T, int ORDER>
cudaError_t launch_adj_tiles(const Plan &p, const StepArgs &a, const Tile *tiles,
                             const std::vector<Tile> &th, const void *g_out, void *g_in,
                             void *g_dv, cudaStream_t s)
{
    if (th.empty()) return cudaSuccess;
    int cap = 0;
    for (const Tile &t : th) cap = cap > t.count ? cap : t.count;
    const int wcap = cap + 2 * kMaxSub + 16;
    const size_t smem = sizeof(T) * ((size_t)3 * wcap + 1 + (size_t)kMaxSub * wcap);
    if (smem > 227 * 1024) return cudaErrorNotSupported;
    static size_t configured[64] = {0};
    const int dev = p.device < 64 ? p.device : 63;
    if (smem > configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(k_adj_uniform<T, ORDER>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        configured[dev] = smem;
    }
    StepArgs b = a;
    b.tiles = tiles;
    b.n_tiles = (int)th.size();
    return launch_pdl(k_adj_uniform<T, ORDER>, dim3((int)th.size(), 2), 256, smem, s, b,
                      static_cast<const RowParams<T> *>(p.row_par), static_cast<const T *>(g_out),
                      static_cast<T *>(g_in), static_cast<T *>(g_dv), cap);
}

// The warp-segment kernel reads and writes 16-byte vectors of every array but g_in.
bool seg_aligned(const StepArgs &a, const void *g_out, const void *g_dv)
{
    for (const void *ptr : {a.q_in, a.dv, g_out, g_dv})
        if ((uintptr_t)ptr % 16) return false;
    return true;
}

template <typename T, int ORDER>
cudaError_t launch_adj_t(const Plan &p, const StepArgs &a, const void *g_out, void *g_in,
                         void *g_dv, bool vec, cudaStream_t s)
{
    constexpr int d = sizeof(T) == 4 ? 0 : 1;
    for (const Tile &t : p.tiles_uniform_h[ORDER])
        if (t.count > 256 * 8) return cudaErrorNotSupported;  // tiles k_adj_uniform does not take
    if (!vec)
        return launch_adj_tiles<T, ORDER>(p, a, p.tiles_uniform[ORDER], p.tiles_uniform_h[ORDER],
                                          g_out, g_in, g_dv, s);
    const std::vector<int32_t> &rows = p.rows_seg_h[d][ORDER];
    if (!rows.empty()) {
        // segments of the longest row at the widest halo; the warps past a row's end leave
        const int stride = 32 * kSegV<T> - 2 * seg_halo<T>(a.dv ? RAM_MAX_NSUB : 0);
        const int segs = (p.seg_nmax[d][ORDER] + stride - 1) / stride;
        const int y = std::min((segs + kSegWarps - 1) / kSegWarps, 65535);
        cudaError_t e = launch_pdl(k_adj_seg<T, ORDER>, dim3((unsigned)rows.size(), y),
                                   dim3(kSegWarps * 32), 0, s, a,
                                   static_cast<const int32_t *>(p.rows_seg[d][ORDER]),
                                   static_cast<const RowParams<T> *>(p.row_par),
                                   static_cast<const T *>(g_out), static_cast<T *>(g_in),
                                   static_cast<T *>(g_dv));
        if (e != cudaSuccess) return e;
    }
    return launch_adj_tiles<T, ORDER>(p, a, p.tiles_rest_seg[d][ORDER], p.tiles_rest_seg_h[d][ORDER],
                                      g_out, g_in, g_dv, s);
}

}  // namespace

cudaError_t launch_adjoint(const Plan &p, ram_dtype dt, const StepArgs &a, const void *g_out,
                           void *g_in, void *g_dv, cudaStream_t s)
{
    // rows with their own mesh and a residual step need the plan's scratch
    const bool nonuni = p.n_uniform_rows < p.n_rows;
    if (nonuni && a.dv != nullptr && p.adj_scratch == nullptr) return cudaErrorNotSupported;
    // a limited plan: every row on the gather adjoint, linearised at the step input
    if (p.adj_all) return launch_adjoint_nu(p, dt, a, g_out, g_in, g_dv, s);
    const bool vec = seg_aligned(a, g_out, g_dv);
    // FP32 warp-segment rows form their own shift
    bool params = dt != RAM_F32 || nonuni || !vec;
    for (int o = 2; o <= 4; ++o) params |= !p.tiles_rest_seg_h[0][o].empty();
    cudaError_t e = params ? launch_params(p, dt, a, s) : cudaSuccess;
    if (e != cudaSuccess) return e;
    if (dt == RAM_F32) {
        if ((e = launch_adj_t<float, 2>(p, a, g_out, g_in, g_dv, vec, s)) != cudaSuccess) return e;
        if ((e = launch_adj_t<float, 3>(p, a, g_out, g_in, g_dv, vec, s)) != cudaSuccess) return e;
        if ((e = launch_adj_t<float, 4>(p, a, g_out, g_in, g_dv, vec, s)) != cudaSuccess) return e;
    } else {
        if ((e = launch_adj_t<double, 2>(p, a, g_out, g_in, g_dv, vec, s)) != cudaSuccess) return e;
        if ((e = launch_adj_t<double, 3>(p, a, g_out, g_in, g_dv, vec, s)) != cudaSuccess) return e;
        if ((e = launch_adj_t<double, 4>(p, a, g_out, g_in, g_dv, vec, s)) != cudaSuccess) return e;
    }
    return nonuni ? launch_adjoint_nu(p, dt, a, g_out, g_in, g_dv, s) : cudaSuccess;
}

}  // namespace ram
