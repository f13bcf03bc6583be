// diag.cu -- FP64 diagnostics: the phi mass and the contact-angle fit.
// Both are reductions in FP64 with warp shuffles and a fixed block order
// (the mass is bit-reproducible run to run).
#include "storage.cuh"

namespace pfk {
namespace {

constexpr int RB = 256;         // reduction block
constexpr int MASS_BLOCKS = 1216;  // 8 per SM on 152 SMs

__device__ __forceinline__ int wrap1(int x, int nx) { return x < 0 ? x + nx : (x >= nx ? x - nx : x); }

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sum over the block; the result is valid in thread 0.
template <int NT>
__device__ double block_sum(double v, double* sh)
{
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double r = 0.0;
    if (wid == 0) {
        r = (lane < NT / 32) ? sh[lane] : 0.0;
        r = warp_sum(r);
    }
    return r;
}

// Pulled g_I at node (x, y), same rule as the step, as a double.
template <int PREC, int I>
__device__ __forceinline__ double pulled_g(const Planes<PREC>& P, const uint8_t* __restrict__ cls, int x, int y,
                                           int nx, int pitch, size_t plane)
{
    using T = Store<PREC>;
    constexpr int X = cx(I), Y = cy(I), O = opp(I);
    size_t src = (size_t)(y - Y) * pitch + wrap1(x - X, nx);
    if (zeta_of(cls[src])) return (double)T::template ld<I>(P.g[I * plane + src]);
    size_t dst = (size_t)(y + Y) * pitch + wrap1(x + X, nx);
    if (zeta_of(cls[dst])) return (double)T::template ld<O>(P.g[O * plane + dst]);
    return (double)T::template ld<O>(P.g[O * plane + (size_t)y * pitch + x]);
}

template <int PREC>
__global__ void __launch_bounds__(RB) k_mass_partial(const uint8_t* __restrict__ cls, Planes<PREC> P, int nx, int ny,
                                                     int pitch, size_t plane, double* __restrict__ partial)
{
    __shared__ double sh[RB / 32];
    step_wait();
    double acc = 0.0;
    const long long N = (long long)nx * ny;
    for (long long t = (long long)blockIdx.x * RB + threadIdx.x; t < N; t += (long long)gridDim.x * RB) {
        int y = (int)(t / nx), x = (int)(t - (long long)y * nx);
        if (!zeta_of(cls[(size_t)y * pitch + x])) continue;
        double v0 = Store<PREC>::g0_double(P.g0[(size_t)y * pitch + x]);
        double v1 = pulled_g<PREC, 1>(P, cls, x, y, nx, pitch, plane);
        double v2 = pulled_g<PREC, 2>(P, cls, x, y, nx, pitch, plane);
        double v3 = pulled_g<PREC, 3>(P, cls, x, y, nx, pitch, plane);
        double v4 = pulled_g<PREC, 4>(P, cls, x, y, nx, pitch, plane);
        double v5 = pulled_g<PREC, 5>(P, cls, x, y, nx, pitch, plane);
        double v6 = pulled_g<PREC, 6>(P, cls, x, y, nx, pitch, plane);
        double v7 = pulled_g<PREC, 7>(P, cls, x, y, nx, pitch, plane);
        double v8 = pulled_g<PREC, 8>(P, cls, x, y, nx, pitch, plane);
        acc += ((v0 + v1) + (v2 + v3)) + ((v4 + v5) + (v6 + v7)) + v8;
    }
    double r = block_sum<RB>(acc, sh);
    if (threadIdx.x == 0) partial[blockIdx.x] = r;
}

__global__ void __launch_bounds__(RB) k_sum_partials(const double* __restrict__ partial, int n,
                                                     double* __restrict__ out)
{
    __shared__ double sh[RB / 32];
    step_wait();
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += RB) acc += partial[i];
    double r = block_sum<RB>(acc, sh);
    if (threadIdx.x == 0) *out = r;
}

// ---------------------------------------------------------------------------
// Contact angle: phi = 1/2 crossings between fluid neighbours, then a circle
// fit (algebraic fit on mean-centred points, Gauss-Newton on the geometric
// distance), then the angle against the wall, all in FP64.
// ---------------------------------------------------------------------------
struct Wall {
    int type;
    double px, py, nx, ny, r, x_lo, x_hi, exclude;
};

__device__ __forceinline__ double wall_distance(const Wall& w, double x, double y)
{
    if (w.type == 0) return (x - w.px) * w.nx + (y - w.py) * w.ny;
    double dx = x - w.px, dy = y - w.py;
    return sqrt(dx * dx + dy * dy) - w.r;
}

__global__ void k_crossings(const uint8_t* __restrict__ cls, const double* __restrict__ phi, int nx, int ny,
                            int pitch, Wall w, double* __restrict__ pts, int cap, int* __restrict__ count)
{
    step_wait();
    int x = blockIdx.x * blockDim.x + threadIdx.x;
    int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= nx || y >= ny) return;
    if ((cls[(size_t)y * pitch + x] & CLS_MASK) != CLS_FLUID) return;
    double a = phi[(size_t)y * nx + x];
    for (int dir = 0; dir < 2; ++dir) {
        int xx = x + (dir == 0), yy = y + (dir == 1);
        if (xx >= nx || yy >= ny) continue;
        if ((cls[(size_t)yy * pitch + xx] & CLS_MASK) != CLS_FLUID) continue;
        double b = phi[(size_t)yy * nx + xx];
        if ((a >= 0.5) == (b >= 0.5)) continue;
        double t = (0.5 - a) / (b - a);
        double qx = x + (dir == 0 ? t : 0.0), qy = y + (dir == 1 ? t : 0.0);
        if (qx < w.x_lo || qx >= w.x_hi) continue;
        if (wall_distance(w, qx, qy) <= w.exclude) continue;
        int k = atomicAdd(count, 1);
        if (k < cap) {
            pts[2 * k] = qx;
            pts[2 * k + 1] = qy;
        }
    }
}

__device__ bool solve3(double A[3][3], double b[3], double z[3])
{
    for (int c = 0; c < 3; ++c) {
        int piv = c;
        for (int r = c + 1; r < 3; ++r)
            if (fabs(A[r][c]) > fabs(A[piv][c])) piv = r;
        if (A[piv][c] == 0.0) return false;
        if (piv != c) {
            for (int k = 0; k < 3; ++k) { double t = A[c][k]; A[c][k] = A[piv][k]; A[piv][k] = t; }
            double t = b[c]; b[c] = b[piv]; b[piv] = t;
        }
        for (int r = c + 1; r < 3; ++r) {
            double m = A[r][c] / A[c][c];
            for (int k = c; k < 3; ++k) A[r][k] -= m * A[c][k];
            b[r] -= m * b[c];
        }
    }
    for (int r = 2; r >= 0; --r) {
        double acc = b[r];
        for (int k = r + 1; k < 3; ++k) acc -= A[r][k] * z[k];
        z[r] = acc / A[r][r];
    }
    return true;
}

constexpr int FB = 512;

// Sums over the block of K values per thread (the first min(n, FB) threads hold
// some), valid in every thread after the call: the values through shared
// memory, one warp per value. (A shuffle reduction of each value in every
// warp costs FB / 32 x 5 FP64 additions a value, this one at most FB / 32 + 5;
// an FP64 addition takes 19 cycles a warp and SM.)
template <int K>
__device__ void sums(const double (&v)[K], int n, double (*s_v)[FB], double* s_tot)
{
    static_assert(K <= FB / 32, "one warp per value");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, m = n < FB ? n : FB;
    if (threadIdx.x < m) {
#pragma unroll
        for (int j = 0; j < K; ++j) s_v[j][threadIdx.x] = v[j];
    }
    __syncthreads();
    if (wid < K) {
        double a = 0.0;
        for (int i = lane; i < m; i += 32) a += s_v[wid][i];
        a = warp_sum(a);
        if (lane == 0) s_tot[wid] = a;
    }
    __syncthreads();
}

// out = {theta_deg, a, b, R, n}; leaves *count at 0 for the next fit. FP64
// instructions bound it (one block, some hundred points, 5 to 7 Gauss-Newton
// steps): with a block reduction per sum it took 72 us on a 256 x 128 lattice, with
// one warp per sum and one division per point 39 us.
__global__ void __launch_bounds__(FB) k_fit(const double* __restrict__ pts, int* __restrict__ count, int cap, Wall w,
                                            double* __restrict__ out)
{
    __shared__ double s_v[9][FB];
    __shared__ double s_tot[9];
    __shared__ double bc[3];
    __shared__ int flag;
    step_wait();
    int n = *count;
    __syncthreads();
    if (threadIdx.x == 0) *count = 0;
    if (n > cap) n = cap;
    if (n < 3) {
        if (threadIdx.x == 0) { out[0] = nan(""); out[1] = out[2] = out[3] = 0.0; out[4] = n; }
        return;
    }
    // mean
    {
        double s[2] = {0.0, 0.0};
        for (int k = threadIdx.x; k < n; k += FB) { s[0] += pts[2 * k]; s[1] += pts[2 * k + 1]; }
        sums(s, n, s_v, s_tot);
    }
    const double mx = s_tot[0] / n, my = s_tot[1] / n;
    __syncthreads();
    // algebraic fit: normal equations of min sum (u^2 + v^2 + D u + E v + F)^2
    {
        double m[8] = {0};
        for (int k = threadIdx.x; k < n; k += FB) {
            const double u = pts[2 * k] - mx, v = pts[2 * k + 1] - my, uu = u * u, vv = v * v, rhs = -(uu + vv);
            m[0] += uu; m[1] += u * v; m[2] += u; m[3] += vv; m[4] += v;
            m[5] += u * rhs; m[6] += v * rhs; m[7] += rhs;
        }
        sums(m, n, s_v, s_tot);
    }
    if (threadIdx.x == 0) {
        const double* t = s_tot;
        double A[3][3] = {{t[0], t[1], t[2]}, {t[1], t[3], t[4]}, {t[2], t[4], (double)n}};
        double b[3] = {t[5], t[6], t[7]}, z[3];
        flag = 0;
        if (solve3(A, b, z)) {
            double a0 = -z[0] / 2.0, b0 = -z[1] / 2.0, R2 = a0 * a0 + b0 * b0 - z[2];
            if (R2 > 0) { bc[0] = a0; bc[1] = b0; bc[2] = sqrt(R2); flag = 1; }
        }
    }
    __syncthreads();
    if (!flag) {
        if (threadIdx.x == 0) { out[0] = nan(""); out[4] = 0; }
        return;
    }
    for (int it = 0; it < 50; ++it) {
        const double a0 = bc[0], b0 = bc[1], R = bc[2];
        // J = (-u / d, -v / d, -1), r = d - R; a point on the centre counts for nothing
        double q[9] = {0};
        for (int k = threadIdx.x; k < n; k += FB) {
            const double u = pts[2 * k] - mx - a0, v = pts[2 * k + 1] - my - b0;
            const double d = sqrt(u * u + v * v);
            if (d == 0.0) continue;
            const double inv = 1.0 / d, J0 = -u * inv, J1 = -v * inv, r = d - R;
            q[0] += J0 * J0; q[1] += J0 * J1; q[2] -= J0; q[3] += J1 * J1; q[4] -= J1;
            q[5] -= J0 * r; q[6] -= J1 * r; q[7] += r; q[8] += 1.0;
        }
        sums(q, n, s_v, s_tot);
        if (threadIdx.x == 0) {
            const double* t = s_tot;
            double A[3][3] = {{t[0], t[1], t[2]}, {t[1], t[3], t[4]}, {t[2], t[4], t[8]}};
            double b[3] = {t[5], t[6], t[7]}, dz[3];
            flag = 0;
            if (solve3(A, b, dz)) {
                bc[0] = a0 + dz[0]; bc[1] = b0 + dz[1]; bc[2] = R + dz[2];
                flag = (fabs(dz[0]) + fabs(dz[1]) + fabs(dz[2]) < 1e-13 * (1.0 + fabs(R))) ? 0 : 1;
            }
        }
        __syncthreads();
        if (!flag) break;
    }
    if (threadIdx.x == 0) {
        double a0 = bc[0] + mx, b0 = bc[1] + my, R = bc[2], ct;
        if (w.type == 0) {
            ct = -((a0 - w.px) * w.nx + (b0 - w.py) * w.ny) / R;
        } else {
            double dx = a0 - w.px, dy = b0 - w.py;
            ct = (R * R + w.r * w.r - (dx * dx + dy * dy)) / (2.0 * R * w.r);
        }
        ct = fmin(1.0, fmax(-1.0, ct));
        out[0] = acos(ct) * (180.0 / 3.14159265358979323846);
        out[1] = a0; out[2] = b0; out[3] = R; out[4] = n;
    }
}

}  // namespace

template <int PREC>
void mass_prec(pflbm_t* h, size_t plane)
{
    launch_after(k_mass_partial<PREC>, dim3(MASS_BLOCKS), dim3(RB), h->stream, (const uint8_t*)h->cls,
                 Planes<PREC>::make(h->pop[h->cur], plane), h->nx, h->ny, h->pitch, plane, h->red);
}

cudaError_t launch_mass(pflbm_t* h, double* d_out)
{
    size_t plane = (size_t)h->ny * h->pitch;
    switch (h->precision) {
        case PFLBM_FP64: mass_prec<PFLBM_FP64>(h, plane); break;
        case PFLBM_FP32: mass_prec<PFLBM_FP32>(h, plane); break;
        case PFLBM_BF16: mass_prec<PFLBM_BF16>(h, plane); break;
        default: mass_prec<PFLBM_FP16>(h, plane); break;
    }
    launch_after(k_sum_partials, dim3(1), dim3(RB), h->stream, (const double*)h->red, (int)MASS_BLOCKS, d_out);
    return cudaGetLastError();
}

size_t mass_scratch_doubles() { return MASS_BLOCKS + 16; }

cudaError_t launch_contact_angle(pflbm_t* h, const pflbm_wall_t* wall, const double* d_phi, double* d_result)
{
    Wall w{wall->type, wall->px, wall->py, wall->nx, wall->ny, wall->r, wall->x_lo, wall->x_hi, wall->exclude};
    int* d_count = (int*)(h->red + MASS_BLOCKS + 12);   // 0 from creation on; every fit leaves it so
    dim3 b(32, 8), g((h->nx + 31) / 32, (h->ny + 7) / 8);
    cudaError_t e = launch_after(k_crossings, g, b, h->stream, (const uint8_t*)h->cls, d_phi, h->nx, h->ny, h->pitch, w,
                                 h->pts, h->pts_cap, d_count);
    if (e == cudaSuccess)
        e = launch_after(k_fit, dim3(1), dim3(FB), h->stream, (const double*)h->pts, d_count, h->pts_cap, w, d_result);
    return e;
}

}  // namespace pfk
