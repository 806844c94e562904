// The radial sweep of a polar disk, for dimensional splitting in two dimensions
// (Sec. 3.5): the plan's rows are the rings of one shared azimuthal mesh; every
// azimuthal column takes one flux-form upwind step in r in cylindrical geometry,
//   q'_j = q_j - dt (rf[j+1] F_{j+1} - rf[j] F_j) / A_j,  A_j = (rf[j+1]^2 - rf[j]^2)/2,
// with F = vr q_up (donor) or vr times the upwind ring's van Leer profile (the
// harmonic slope over the ring centres' spacings, Sec. 3.1; zero in the two rings
// next to the walls) at the midpoint of the swept interval, and closed walls
// (F = 0 on faces 0 and n_rows).
//
// A CTA takes kRings rings and 128 azimuthal columns.  Its first threads form the
// rings' geometry once, in FP64 from the face radii, in shared memory: an FP64
// instruction holds its pipe for tens of cycles, and formed by every thread the
// geometry kept that pipe 86% busy (51.1 us on 510 rings of 1533 cells in FP32, cold
// caches; now 8.8 us, bound by the latency of the loads and of the geometry; dt / A as a
// quotient of the cells' type instead, which leaves the range of FP32 at radii of 1e19,
// saved 0.2 us of the split step).  A
// thread walks outward along its column with every load of the column in flight
// first: every slope and flux is formed once, and each value is loaded once but for
// the four rings that neighbouring CTAs share (4, 8 or 16 rings per CTA: 31.5, 31.3,
// 31.3 us for the whole split step).
#include <cuda_runtime.h>

#include "ram_device.cuh"

namespace ram {
namespace {

constexpr int kCols = 128;

// Geometry of ring k, in the cells' type.
template <typename T> struct Ring {
    T w;        // rf[k+1] - rf[k]
    T spacing;  // between the centres of rings k - 1 and k, (rf[k+1] - rf[k-1]) / 2
    T ka;       // dt / A_k
    T rl;       // rf[k]
};

template <typename T, int kRings>
__global__ void __launch_bounds__(kCols) k_radial(int nr, int N, const T *q, T *out,
                                                  const double *rf, const T *vr, double dt,
                                                  int vl, int *err)
{
    // rings j0 - 1 .. j0 + kRings + 1 (those inside the disk)
    __shared__ Ring<T> ring[kRings + 3];
    const int j0 = blockIdx.y * kRings;
    pdl_wait();
    pdl_trigger();
    const int i = blockIdx.x * kCols + threadIdx.x;
    const int j1 = min(j0 + kRings, nr);
    // every load of the column first: they overlap with each other and the geometry
    T qv[kRings + 4], vv[kRings + 1];  // rings j0 - 2 .. j1 + 1, faces j0 .. j1
#pragma unroll
    for (int t = 0; t < kRings + 4; ++t) {
        const int k = j0 - 2 + t;
        qv[t] = i < N && k >= 0 && k < nr && k <= j1 + 1 ? q[(size_t)k * N + i] : T(0);
    }
#pragma unroll
    for (int t = 0; t <= kRings; ++t) {
        const int k = j0 + t;
        vv[t] = i < N && k > 0 && k < nr && k <= j1 ? vr[(size_t)k * N + i] : T(0);
    }
    if (threadIdx.x < kRings + 3) {
        const int k = j0 - 1 + (int)threadIdx.x;
        if (k >= 0 && k <= nr) {
            Ring<T> g{};
            const double r0 = rf[k];
            g.rl = (T)r0;
            if (k < nr) {
                const double r1 = rf[k + 1];
                g.w = (T)(r1 - r0);
                g.ka = (T)(dt / (0.5 * (r1 - r0) * (r1 + r0)));
                if (k > 0) g.spacing = (T)(0.5 * (r1 - rf[k - 1]));
            }
            ring[threadIdx.x] = g;
        }
    }
    __syncthreads();
    if (i >= N) return;
    const T h = (T)dt;
    const Ring<T> *const g0 = ring + 1 - j0;  // g0[k]: ring k
    // van Leer slope of ring k from the divided differences on its two sides (flat
    // in the rings next to the walls)
    auto slope = [&](int k, T dl, T dr) -> T {
        if (!vl || k <= 0 || k >= nr - 1) return T(0);
        const T pr = dl * dr;
        return pr > T(0) ? Num<T>::div(T(2) * pr, dl + dr) : T(0);
    };
    auto diff = [&](int k, T ql, T qr) {  // across face k, between rings k - 1 and k
        return k > 0 && k < nr ? Num<T>::div(qr - ql, g0[k].spacing) : T(0);
    };
    bool bad = false;
    // flux through face k from the values and slopes of rings k - 1 and k
    auto flux = [&](int k, T v, T ql, T sl, T qr, T sr) -> T {
        if (k <= 0 || k >= nr) return T(0);
        const T c = v * h;
        T qh = T(0);
        if (c > T(0)) {
            const T w = g0[k - 1].w;
            qh = ql + T(0.5) * sl * (w - c);
            bad |= c > w;
        } else if (c < T(0)) {
            const T w = g0[k].w;
            qh = qr - T(0.5) * sr * (w + c);
            bad |= -c > w;
        }
        return v * qh;
    };
    // ring j0 - 1's slope, then outward
    T dl = diff(j0 - 1, qv[0], qv[1]), dr = diff(j0, qv[1], qv[2]);
    T s_in = slope(j0 - 1, dl, dr);  // slope of the ring inside the face
    T f_in = T(0);
#pragma unroll
    for (int t = 0; t <= kRings; ++t) {
        const int k = j0 + t;  // face k, between rings k - 1 and k
        if (k <= j1) {
            dl = dr;
            dr = diff(k + 1, qv[t + 2], qv[t + 3]);
            const T s = slope(k, dl, dr);
            const T f = flux(k, vv[t], qv[t + 1], s_in, qv[t + 2], s);
            if (t > 0) {
                const Ring<T> &r = g0[k - 1];
                out[(size_t)(k - 1) * N + i] = qv[t + 1] - r.ka * (g0[k].rl * f - r.rl * f_in);
            }
            f_in = f;
            s_in = s;
        }
    }
    if (bad) atomicOr(err, ERR_CFL);
}

template <typename T, int kRings>
cudaError_t launch_radial_t(const Plan &p, const void *q_in, void *q_out, const double *rf,
                            const void *vr, double step, int scheme, cudaStream_t s)
{
    const int nr = p.n_rows, N = p.rows_h[0].n;
    const dim3 grid((N + kCols - 1) / kCols, (nr + kRings - 1) / kRings);
    return launch_pdl(k_radial<T, kRings>, grid, dim3(kCols), 0, s, nr, N,
                      static_cast<const T *>(q_in), static_cast<T *>(q_out), rf,
                      static_cast<const T *>(vr), step, scheme == RAM_VANLEER ? 1 : 0, p.err);
}

}  // namespace

cudaError_t launch_radial(const Plan &p, ram_dtype dt, const void *q_in, void *q_out,
                          const double *rf, const void *vr, double step, int scheme,
                          cudaStream_t s)
{
    return dt == RAM_F32
               ? launch_radial_t<float, 8>(p, q_in, q_out, rf, vr, step, scheme, s)
               : launch_radial_t<double, 8>(p, q_in, q_out, rf, vr, step, scheme, s);
}

}  // namespace ram
