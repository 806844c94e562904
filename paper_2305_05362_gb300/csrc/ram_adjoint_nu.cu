// Transpose of one RAM step on rows with their own mesh (limiter off: the linear
// step; RAM_ADJOINT plans with the limiter on: every row, the PLM / PPM step
// linearised at its input), donor residual.
//
// The remap with the limiter off is linear: output mass M'_i (Eq. 18) is the sum
// over the source cells p that the shifted output cell overlaps of
// G_p(xi_hi) - G_p(xi_lo), the in-cell cumulative of p's reconstruction between
// the overlap's ends (xi in units of p's width), and G_p is linear in the values
// of p's stencil.  Its transpose is a gather by source cell: source cell p,
// shifted by +s, overlaps a few output cells (found like the forward edges, with
// the bucket table on x + s); with u_i = g'_i / dx_i (the transpose of Eq. 26)
// the cotangent of G_p's coefficients is
//   nu_{p,k} = sum_i u_i (xi_hi^k - xi_lo^k)
//            = u_last + sum over the output nodes inside of (u_left - u_right) xi^k.
// The reconstruction's transpose runs backwards over its own steps: from a cell's
// coefficients to a = QR - Q and b = Q - QL, to the faces' offsets from Q, to the
// delta<Q>, to the differences of neighbours and to the cells (PPM); to the slope
// (PLM) or the divided differences (order 4), then the same.  Each is a sum over a
// few neighbours in shared memory, a pass per step, so that every weight is formed
// once.  Through the limiters (RAM_ADJOINT plans) a branch taken at the step input is
// a choice of weights: zero at an extremum, 2 on the difference that bounds delta<Q>,
// a or b twice the other.  A tile of source cells computes nu on itself plus two
// cells per side.
//
// Bound by the FP64 pipe in double precision: carrying the limited reconstruction's
// value with its derivatives along five stencil cells, every weight with range-checked
// divides, took 685 us on 64 rows (597 K cells, PPM, limited), the passes below 184.
//
// The donor residual sub-steps (Eq. 6) with per-cell widths have the transpose
//   lf_j = g_j / dx_j - g_{j-1} / dx_{j-1},  g_up(j) += c_j lf_j,
//   dL/d dv_j += (dt / nsub) Q_up(j) lf_j
// over the sub-steps in reverse, with the forward states recomputed from the
// shifted field (kept in the plan's adjoint scratch); the upwind side at dv = 0
// is the left cell.
#include <cuda_runtime.h>

#include <cstdint>

#include "ram_bits.cuh"
#include "ram_device.cuh"

namespace ram {
namespace {

constexpr int kAH = 4;       // cells staged beyond a tile on each side
constexpr int kArrays = 12;  // shared arrays of a tile's cells

__device__ __forceinline__ float u64f(uint64_t v, float) { return __ull2float_rn(v); }
__device__ __forceinline__ double u64f(uint64_t v, double) { return u64_to_double(v); }
__device__ __forceinline__ float rcp(float x) { return rcp_approx(x); }
__device__ __forceinline__ double rcp(double x) { return rcp_newton(x); }

// x y rounded, not joined with a sum
__device__ __forceinline__ float mul_rn(float x, float y) { return __fmul_rn(x, y); }
__device__ __forceinline__ double mul_rn(double x, double y) { return __dmul_rn(x, y); }

// 2^e (sign = 1) or 2^-e (sign = -1), e the exponent of the normal x
__device__ __forceinline__ double pow2_below(double x, int sign)
{
    const int e = ((__double2hiint(x) >> 20) & 0x7ff) - 1023;
    return __hiloint2double((1023 + sign * e) << 20, 0);
}

// x y > 0, |x| > 2|y|: on the integer pipe in FP64 (x y > 0 also asks that the product
// does not vanish and neither is NaN); in FP32 by the signs alone, as in the forward
// kernel (the product vanishes below 1e-22)
__device__ __forceinline__ bool positive(float x, float y) { return minxs_nan(x, y) > 0.f; }
__device__ __forceinline__ bool positive(double x, double y)
{
    const int hx = __double2hiint(x), hy = __double2hiint(y);
    const unsigned long long mx = mag(x) - 1ull, my = mag(y) - 1ull;
    const int e = ((hx >> 20) & 0x7ff) + ((hy >> 20) & 0x7ff);
    return (hx ^ hy) >= 0 && mx < 0x7ff0000000000000ull && my < 0x7ff0000000000000ull &&
           e > 1023 - 50;
}
__device__ __forceinline__ bool over_twice(float x, float y) { return fabsf(x) > 2.f * fabsf(y); }
__device__ __forceinline__ bool over_twice(double x, double y)
{
    return mag(x) > mag_up(mag(y), 1);
}

template <typename T> __host__ __device__ inline size_t remap_smem(int tcap)
{
    return sizeof(T) * (size_t)kArrays * (tcap + 2 * kAH);
}

// nu[k], k < K, of source cell p of a row: see the head of this file.  gp: the output
// cotangents, divided by the (scaled) widths already when `divided`.
template <typename T, int K>
__device__ __forceinline__ void overlap_moments(const StepArgs &a, const RowInfo &row,
                                                const uint64_t *X, const T *DX, const T *gp,
                                                uint64_t S, T wscale, bool divided, int p, T nu[K])
{
    const int N = row.n;
    const uint64_t y0 = X[p] + S;                              // shifted left node
    const uint64_t wp = (p + 1 < N ? X[p + 1] : 0ull) - X[p];  // width (fixed point)
    const T iw = rcp(u64f(wp, T(0)));
    int i = locate_cell(X, N, a.buckets + row.bucket_off, row.bucket_bits, a.density, row.density,
                        y0);
#pragma unroll
    for (int k = 0; k < K; ++k) nu[k] = T(0);
    T u = divided ? gp[i] : gp[i] * rcp(DX[i] * wscale);
    // the shifted cell [y0, y0 + wp) overlaps output cells i, i + 1, ..., at the last the
    // first one again (a cell that spans all the others): its right end is behind then
    uint64_t walked = 0;
    for (int guard = 0; guard <= N; ++guard) {
        const uint64_t rr = (i + 1 < N ? X[i + 1] : 0ull) - y0;  // output cell's right end
        if (rr >= wp || rr <= walked) break;
        walked = rr;
        i = i + 1 < N ? i + 1 : 0;
        const T un = divided ? gp[i] : gp[i] * rcp(DX[i] * wscale);
        const T xi = u64f(rr, T(0)) * iw;
        T d = (u - un) * xi;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            nu[k] += d;
            if (k + 1 < K) d *= xi;
        }
        u = un;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) nu[k] += u;
}

// One CTA per tile of source cells; local index j is row cell a0 - kAH + j, face j lies
// between cells j and j + 1.
template <typename T, int ORDER, bool LIM>
__global__ void __launch_bounds__(256)
    k_adj_remap_nu(StepArgs a, const RowParams<T> *pars, const T *gprime, T *g_in, int tcap,
                   int divided)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int m = tcap + 2 * kAH;
    T *sh = reinterpret_cast<T *>(smem_raw);  // widths, scaled by a power of two
    T *sq = sh + m;                           // limited: the step input
    T *r2 = sq + m;                           // 1 / (width of both cells at a face)
    T *hn = r2 + m;                           // cotangent of Q_p itself
    T *U = hn + m;                            // cotangent of Q_{j+1} - Q_j
    T *v0 = U + m, *v1 = v0 + m, *v2 = v1 + m, *v3 = v2 + m, *v4 = v3 + m, *v5 = v4 + m,
      *v6 = v5 + m;

    const Tile tile = a.tiles[blockIdx.x];
    const RowInfo row = a.rows[tile.row];
    const int N = row.n;
    const int tid = threadIdx.x, nth = blockDim.x;
    const uint64_t *X = a.xfix + row.mesh_off;
    const T *DX = (sizeof(T) == 4) ? reinterpret_cast<const T *>(a.dx32 + row.mesh_off)
                                   : reinterpret_cast<const T *>(a.dx64 + row.mesh_off);
    const T *gp = gprime + row.cell_off;
    pdl_wait();
    const uint64_t S = pars[tile.row].sfix;
    const int a0 = tile.start, tn = tile.count;
    const int nm = tn + 2 * kAH;
    const T *q0 = static_cast<const T *>(a.q_in) + row.cell_off;
    // the power of two at or below N / L: products of four widths stay in range
    const T wscale = (T)pow2_below(row.cells_per_length, 1);
    for (int j = tid; j < nm; j += nth) {
        const int c = wrap_index((int64_t)a0 - kAH + j, N);
        sh[j] = DX[c] * wscale;
        if (LIM) sq[j] = q0[c];
    }
    __syncthreads();
    for (int j = tid; j < nm - 1; j += nth) r2[j] = rcp(sh[j] + sh[j + 1]);
    __syncthreads();

    if (ORDER == 3) {
        T *al = v0, *be = v1, *dq = v2, *cq = v3, *w2 = v4, *w3 = v5, *fa = v6;
        // delta<Q>_j = al (Q_{j+1} - Q_j) + be (Q_j - Q_{j-1}) (App. A.1); limited: the
        // weights of the branch taken
        for (int j = 1 + tid; j < nm - 1; j += nth) {
            const T hm = sh[j - 1], h0 = sh[j], hp = sh[j + 1];
            const T f = h0 * rcp(hm + h0 + hp);
            T A = f * (T(2) * hm + h0) * r2[j], B = f * (h0 + T(2) * hp) * r2[j - 1];
            if (LIM) {
                const T up = sq[j + 1] - sq[j], dn = sq[j] - sq[j - 1];
                const T d = A * up + B * dn;
                T v = d;
                if (positive(up, dn)) {
                    // sign(d) min(|d|, 2|dn|, 2|up|)
                    if (over_twice(d, dn)) {
                        A = T(0);
                        B = T(2);
                        v = dn + dn;
                    }
                    if (over_twice(v, up)) {
                        A = T(2);
                        B = T(0);
                        v = up + up;
                    }
                } else {
                    A = B = v = T(0);
                }
                dq[j] = v;
            }
            al[j] = A;
            be[j] = B;
        }
        __syncthreads();
        // <Q>_{j+1/2} - Q_j = cq (Q_{j+1} - Q_j) + w2 delta<Q>_{j+1} + w3 delta<Q>_j
        for (int j = 1 + tid; j < nm - 2; j += nth) {
            const T h0 = sh[j], h1 = sh[j + 1], b0 = sh[j - 1] + h0, b2 = h1 + sh[j + 2];
            const T B = T(2) * h0 + h1, C = h0 + T(2) * h1;
            const T inv = rcp(B * C * (b0 + b2));
            const T x2 = -h0 * b0 * C * inv, x3 = h1 * b2 * B * inv;
            const T xq = r2[j] * (h0 - T(2) * (h1 * x2 + h0 * x3));
            cq[j] = xq;
            w2[j] = x2;
            w3[j] = x3;
            if (LIM) fa[j] = xq * (sq[j + 1] - sq[j]) + x2 * dq[j + 1] + x3 * dq[j];
        }
        __syncthreads();
        // cotangents of a = QR - Q and b = Q - QL (App. A.2's second stage when limited);
        // G / h = xi (Q - b) + xi^2 (2b - a) + xi^3 (a - b).  dq is not read again: b's take
        // its place
        T *cb = dq, *ca = U;
        for (int j = 2 + tid; j < nm - 2; j += nth) {
            T nu[3];
            overlap_moments<T, 3>(a, row, X, DX, gp, S, wscale, divided != 0,
                                  wrap_index((int64_t)a0 - kAH + j, N), nu);
            const T h = sh[j];
            T xa = h * (nu[2] - nu[1]), xb = h * (nu[1] - nu[0]) - xa;
            if (LIM) {
                const T fa_ = fa[j], fb = (sq[j] - sq[j - 1]) - fa[j - 1];
                if (!positive(fa_, fb)) {
                    xa = xb = T(0);
                } else if (over_twice(fb, fa_)) {
                    xa += T(2) * xb;  // b = 2a
                    xb = T(0);
                } else if (over_twice(fa_, fb)) {
                    xb += T(2) * xa;  // a = 2b
                    xa = T(0);
                }
            }
            ca[j] = xa;
            cb[j] = xb;
            hn[j] = h * nu[0];
        }
        __syncthreads();
        // the faces' cotangents are ca_j - cb_{j+1}; those of delta<Q>_j through its weights
        for (int j = 3 + tid; j < nm - 3; j += nth) {
            const T c = (ca[j] - cb[j + 1]) * w3[j] + (ca[j - 1] - cb[j]) * w2[j - 1];
            al[j] *= c;
            be[j] *= c;
        }
        __syncthreads();
        T *UU = fa;
        for (int j = 3 + tid; j < nm - 4; j += nth)
            UU[j] = (ca[j] - cb[j + 1]) * cq[j] + cb[j + 1] + al[j] + be[j + 1];
        U = UU;
    } else if (ORDER == 2) {
        // G = h Q xi + s h^2 (xi^2 - xi), s half the slope: 2 x y / (x + y) of the one-sided
        // ones (half each, x on the left) when limited, else the centred one
        T *tl = v0, *tr = v1;
        for (int j = 2 + tid; j < nm - 2; j += nth) {
            T nu[2];
            overlap_moments<T, 2>(a, row, X, DX, gp, S, wscale, divided != 0,
                                  wrap_index((int64_t)a0 - kAH + j, N), nu);
            const T h = sh[j];
            const T cs = h * h * (nu[1] - nu[0]);
            T l, r;
            if (LIM) {
                const T x = (sq[j] - sq[j - 1]) * r2[j - 1], y = (sq[j + 1] - sq[j]) * r2[j];
                l = r = T(0);
                if (positive(x, y)) {
                    const T i = Num<T>::div(T(1), x + y);
                    l = T(2) * cs * (y * i) * (y * i) * r2[j - 1];
                    r = T(2) * cs * (x * i) * (x * i) * r2[j];
                }
            } else {
                l = r = cs * rcp(sh[j - 1] + T(2) * h + sh[j + 1]);
            }
            tl[j] = l;
            tr[j] = r;
            hn[j] = h * nu[0];
        }
        __syncthreads();
        for (int j = 3 + tid; j < nm - 4; j += nth) U[j] = tr[j] + tl[j + 1];
    } else {
        // order 4, G = z (c0 + z (c1 + z (c2 + z c3))): Newton's form on the divided
        // differences D2, D3, D4 of the cell averages (see ram_nseg.cu), backwards
        T *cE2 = v0, *cE3 = v1, *cD = v2, *r3 = v3, *r4 = v4, *t3 = v5, *t4 = v6;
        for (int j = tid; j < nm - 3; j += nth) {
            r3[j] = rcp(sh[j] + sh[j + 1] + sh[j + 2]);
            r4[j] = rcp(sh[j] + sh[j + 1] + sh[j + 2] + sh[j + 3]);
        }
        for (int j = 2 + tid; j < nm - 2; j += nth) {
            T C[4];
            overlap_moments<T, 4>(a, row, X, DX, gp, S, wscale, divided != 0,
                                  wrap_index((int64_t)a0 - kAH + j, N), C);
            const T h = sh[j], hm = sh[j - 1], hp = sh[j + 1];
            T hk = h;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                C[k] *= hk;
                hk *= h;
            }
            const T B0 = C[1] - h * C[0], B1 = C[2] - h * C[1];
            const T A0 = B1 + hm * B0;
            cD[j] = T(0.5) * (C[3] - h * C[2] + hm * B1 - (h + hp) * A0);
            cE2[j] = B0;
            cE3[j] = A0;
            hn[j] = C[0];
        }
        __syncthreads();
        // D4_j (cells j .. j + 3) enters cells j + 1 and j + 2
        for (int j = 1 + tid; j < nm - 4; j += nth) t4[j] = (cD[j + 1] + cD[j + 2]) * r4[j];
        __syncthreads();
        // D3_j (cells j .. j + 2) enters cell j + 1
        for (int j = 2 + tid; j < nm - 4; j += nth) t3[j] = (cE3[j + 1] + t4[j - 1] - t4[j]) * r3[j];
        __syncthreads();
        // D2_j (face j) enters cell j + 1
        for (int j = 3 + tid; j < nm - 4; j += nth) U[j] = (cE2[j + 1] + t3[j - 1] - t3[j]) * r2[j];
    }
    __syncthreads();
    T *gi = g_in + row.cell_off;
    for (int t = tid; t < tn; t += nth) {
        const int j = t + kAH;
        gi[a0 + t] = hn[j] + U[j - 1] - U[j];
    }
}

// Donor residual transpose on a tile of cells [a0, a0+tn) with a halo of nsub
// cells per side: gprime (over the widths) on the tile, and dL/d dv added on the tile's interfaces.
template <typename T>
__global__ void __launch_bounds__(256)
    k_adj_resid_nu(StepArgs a, const RowParams<T> *pars, const T *qs, const T *g_out, T *gprime,
                   T *g_dv, int tcap)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int wc = tcap + 2 * RAM_MAX_NSUB + 2;
    T *sc = reinterpret_cast<T *>(smem_raw);   // wc + 1: dv h (signed swept length)
    T *g0 = sc + wc + 1;                        // wc
    T *g1 = g0 + wc;                            // wc
    T *lf = g1 + wc;                            // wc + 1
    T *rd = lf + wc + 1;                        // wc: 1 / width
    T *st = rd + wc;                        // (RAM_MAX_NSUB + 1) x wc forward states

    const Tile tile = a.tiles[blockIdx.x];
    const RowInfo row = a.rows[tile.row];
    const int N = row.n;
    const int tid = threadIdx.x, nth = blockDim.x;
    const T *DX = (sizeof(T) == 4) ? reinterpret_cast<const T *>(a.dx32 + row.mesh_off)
                                   : reinterpret_cast<const T *>(a.dx64 + row.mesh_off);
    pdl_wait();
    const RowParams<T> P = pars[tile.row];
    const int ns = P.nsub;
    const T h = row.uniform ? P.cf * (T)row.dx : P.cf;  // sub-step length dt / nsub
    const int a0 = tile.start, tn = tile.count;
    const int c0 = a0 - ns;  // first cell of the halo
    const int nc = tn + 2 * ns;
    const T *dv = static_cast<const T *>(a.dv) + row.cell_off;
    const T *q = qs + row.cell_off;
    const T *g = g_out + row.cell_off;
    for (int i = tid; i < nc; i += nth) {
        const int c = wrap_index((int64_t)c0 + i, N);
        rd[i] = rcp(DX[c]);
        st[i] = q[c];
        g0[i] = g[c];
    }
    for (int i = tid; i <= nc; i += nth) sc[i] = dv[wrap_index((int64_t)c0 + i, N)] * h;
    __syncthreads();
    // forward sub-steps: state k+1 on [k+1, nc-k-1) from state k
    for (int k = 0; k + 1 < ns; ++k) {
        const T *qk = st + (size_t)k * wc;
        T *qn = st + (size_t)(k + 1) * wc;
        for (int i = k + 1 + tid; i < nc - k - 1; i += nth) {
            const T cL = sc[i], cR = sc[i + 1];
            const T FL = cL * (cL > T(0) ? qk[i - 1] : qk[i]);
            const T FR = cR * (cR > T(0) ? qk[i] : qk[i + 1]);
            qn[i] = qk[i] - (FR - FL) * rd[i];
        }
        __syncthreads();
    }
    T *cur = g0, *nxt = g1;
    T *gd = g_dv ? g_dv + row.cell_off : nullptr;
    for (int k = ns - 1; k >= 0; --k) {
        const T *qk = st + (size_t)k * wc;
        const int lo = ns - k, hi = nc - (ns - k);  // g^(k) valid on [lo, hi)
        // lf_j for interfaces j in [lo, hi]: g_j / dx_j - g_{j-1} / dx_{j-1}, each rounded
        // alike on both sides of its cell, so that what the interfaces take cancels
        for (int j = lo + tid; j <= hi; j += nth)
            lf[j] = mul_rn(cur[j], rd[j]) - mul_rn(cur[j - 1], rd[j - 1]);
        __syncthreads();
        if (gd)
            for (int j = ns + tid; j < ns + tn; j += nth) {
                const T c = sc[j];
                const T qup = c >= T(0) ? qk[j - 1] : qk[j];
                gd[wrap_index((int64_t)c0 + j, N)] += lf[j] * h * qup;
            }
        for (int i = lo + tid; i < hi; i += nth) {
            T v = cur[i];
            const T cL = sc[i], cR = sc[i + 1];
            if (cR >= T(0)) v += cR * lf[i + 1];  // F_{i+1} takes Q_i when c >= 0
            if (cL < T(0)) v += cL * lf[i];       // F_i takes Q_i when c < 0
            nxt[i] = v;
        }
        __syncthreads();
        T *t = cur;
        cur = nxt;
        nxt = t;
    }
    // divided by the width (in the remap transpose's units): its kernel then need not for
    // every piece of a shifted cell
    T *gpo = gprime + row.cell_off;
    const T iws = (T)pow2_below(row.cells_per_length, -1);
    for (int i = tid; i < tn; i += nth) gpo[a0 + i] = cur[ns + i] * (rd[ns + i] * iws);
}

template <typename T, int ORDER, bool LIM>
cudaError_t launch_adj_remap_nu(const Plan &p, const StepArgs &a, const void *gp, void *g_in,
                                bool divided, cudaStream_t s)
{
    const int n = (int)p.tiles_adj_nu_h[ORDER].size();
    if (n == 0) return cudaSuccess;
    const int tcap = p.adj_nu_tcap;
    const size_t smem = remap_smem<T>(tcap);
    cudaError_t e = cudaFuncSetAttribute(k_adj_remap_nu<T, ORDER, LIM>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    StepArgs b = a;
    b.tiles = p.tiles_adj_nu[ORDER];
    b.n_tiles = n;
    return launch_pdl(k_adj_remap_nu<T, ORDER, LIM>, n, 256, smem, s, b,
                      static_cast<const RowParams<T> *>(p.row_par), static_cast<const T *>(gp),
                      static_cast<T *>(g_in), tcap, divided ? 1 : 0);
}

template <typename T>
cudaError_t launch_adj_nu_t(const Plan &p, const StepArgs &a, const void *g_out, void *g_in,
                            void *g_dv, cudaStream_t s)
{
    const void *gp = g_out;
    const bool resid = a.dv != nullptr;
    if (resid) {
        // the shifted field (the residual step's input) into the scratch
        T *qs = static_cast<T *>(p.adj_scratch);
        T *gprime = qs + p.n_cells;
        // the step's shift alone (MODE_STEP without dv) of the input, by the
        // general kernels (they read the shift from the parameter kernel's output)
        StepArgs f = a;
        f.q_out = qs;
        f.dv = nullptr;
        const ram_dtype dt = sizeof(T) == 4 ? RAM_F32 : RAM_F64;
        cudaError_t e = cudaSuccess;
        if (p.adj_all) {
            // every row: the shift's own parameters (no residual), the uniform and
            // the general kernels, then the step's parameters back for the transposes
            e = launch_params(p, dt, f, s);
            if (e == cudaSuccess) e = launch_uniform(p, dt, f, s);
            if (e == cudaSuccess) e = launch_general(p, dt, f, s);
            if (e == cudaSuccess) e = launch_params(p, dt, a, s);
        } else {
            e = launch_general(p, dt, f, s);
        }
        if (e != cudaSuccess) return e;
        const int tcap = p.adj_nu_tcap;
        const int wc = tcap + 2 * RAM_MAX_NSUB + 2;
        const size_t smem = sizeof(T) * ((size_t)5 * wc + 2 + (size_t)(RAM_MAX_NSUB + 1) * wc);
        if (smem > 227 * 1024) return cudaErrorNotSupported;
        e = cudaFuncSetAttribute(k_adj_resid_nu<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem);
        if (e != cudaSuccess) return e;
        bool first = true;
        for (int o = 2; o <= 4; ++o) {
            const int nt = (int)p.tiles_adj_nu_h[o].size();
            if (nt == 0) continue;
            StepArgs b = a;
            b.tiles = p.tiles_adj_nu[o];
            b.n_tiles = nt;
            const RowParams<T> *pars = static_cast<const RowParams<T> *>(p.row_par);
            if (first) {
                // the first reader of the scratch takes the stream's full ordering (the
                // launches above wait for each other at their end, so a programmatic
                // launch would do)
                k_adj_resid_nu<T><<<nt, 256, smem, s>>>(b, pars, qs, static_cast<const T *>(g_out),
                                                         gprime, static_cast<T *>(g_dv), tcap);
                e = cudaGetLastError();
                first = false;
            } else {
                e = launch_pdl(k_adj_resid_nu<T>, nt, 256, smem, s, b, pars,
                               static_cast<const T *>(qs), static_cast<const T *>(g_out), gprime,
                               static_cast<T *>(g_dv), tcap);
            }
            if (e != cudaSuccess) return e;
        }
        gp = gprime;
    } else if (p.adj_all) {
        cudaError_t e = launch_params(p, sizeof(T) == 4 ? RAM_F32 : RAM_F64, a, s);
        if (e != cudaSuccess) return e;
    }
    if (p.adj_all) {
        // limited PLM / PPM linearised at the step input
        cudaError_t e = launch_adj_remap_nu<T, 2, true>(p, a, gp, g_in, resid, s);
        if (e == cudaSuccess) e = launch_adj_remap_nu<T, 3, true>(p, a, gp, g_in, resid, s);
        return e;
    }
    cudaError_t e = launch_adj_remap_nu<T, 2, false>(p, a, gp, g_in, resid, s);
    if (e == cudaSuccess) e = launch_adj_remap_nu<T, 3, false>(p, a, gp, g_in, resid, s);
    if (e == cudaSuccess) e = launch_adj_remap_nu<T, 4, false>(p, a, gp, g_in, resid, s);
    return e;
}

}  // namespace

cudaError_t launch_adjoint_nu(const Plan &p, ram_dtype dt, const StepArgs &a, const void *g_out,
                              void *g_in, void *g_dv, cudaStream_t s)
{
    if (dt == RAM_F32) return launch_adj_nu_t<float>(p, a, g_out, g_in, g_dv, s);
    return launch_adj_nu_t<double>(p, a, g_out, g_in, g_dv, s);
}

}  // namespace ram
