// Reverse-mode derivative of the P3M force: the transposed Jacobian of the accelerations
// applied to a vector field v, (dA/dx)^T v, and the gradient of a mesh density loss.  These
// are the pieces of the adjoint of the kick-drift-kick step (the reverse sweep itself runs on
// the host side).
//
// Mesh part, with E_b = D_b rho the three mesh accelerations (D_b = IFFT(-i k_b G FFT), real,
// D_b^T = IFFT(+i k_b G FFT)) and rho(n) = sum_j W(x_j - n) the CIC counts:
//   out_k = sum_n grad W(x_k - n) [ sum_b v_k,b E_b(n) + psi(n) ],
//   psi = sum_b D_b^T u_b,  u_b(n) = sum_i W(x_i - n) v_i,b.
// Pair part, J(d) = h(r) I + (h'(r)/r) d d^T with h(r) = Gm g(r/r_s) (r^2 + eps^2)^-3/2:
//   out_k = sum_{j: 0 < r_kj < r_c} J(d_kj) (v_j - v_k).
#include <cuda_runtime.h>
#include <cufft.h>
#include <math.h>

#include <type_traits>
#include <vector>

#include "p3m_device.cuh"
#include "p3m_internal.cuh"
#include "state.cuh"
#include "pair_walk.cuh"

namespace {

inline int grid_for(int64_t n, int threads, int num_sms)
{
    int64_t b = (n + threads - 1) / threads;
    int64_t cap = (int64_t)num_sms * 16;
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}

__device__ __forceinline__ int wrap_index(int i, int M)
{
    i %= M;
    return i < 0 ? i + M : i;
}

// CIC stencil in FP64: base node i0 = floor(x M/L), fraction f.
__device__ __forceinline__ void stencil64(double x, double inv_h, int &i0, double &f)
{
    split_floor(__dmul_rn(x, inv_h), i0, f);
}

// The eight CIC nodes around a wrapped position and the fractions in its mesh cell.  Node indices lie in
// [0, M], so one compare wraps them instead of a division.
struct CicNodes {
    size_t row[2][2];
    int z[2];
    double f[3];
    __device__ __forceinline__ CicNodes(double x, double y, double zz, double inv_h, int M)
    {
        int i[3];
        stencil64(x, inv_h, i[0], f[0]);
        stencil64(y, inv_h, i[1], f[1]);
        stencil64(zz, inv_h, i[2], f[2]);
        int j[3][2];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if ((unsigned)i[d] >= (unsigned)M) i[d] = 0;  // (x / h rounded up to M; a position that is NaN)
            j[d][0] = i[d];
            j[d][1] = i[d] + 1 == M ? 0 : i[d] + 1;
        }
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) row[a][b] = ((size_t)j[0][a] * M + j[1][b]) * M;
        z[0] = j[2][0];
        z[1] = j[2][1];
    }
    __device__ __forceinline__ size_t node(int a, int b, int e) const { return row[a][b] + z[e]; }
};

// v_sorted[k] = v[pid[k]] (caller order -> slot order), also an FP32 copy with w = 0.
__global__ void k_to_slots(const double *__restrict__ v, const uint32_t *__restrict__ pid,
                           int64_t n, double *__restrict__ vs, float *__restrict__ vfx)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t j = pid[k];
        const double a = v[j], b = v[n + j], c = v[2 * n + j];
        vs[k] = a;
        vs[n + k] = b;
        vs[2 * n + k] = c;
        if (vfx) {  // FP32 block-SoA copy (per 32-slot block vx[32] vy[32] vz[32])
            float *dst = vfx + (k >> 5) * 96 + (k & 31);
            dst[0] = (float)a;
            dst[32] = (float)b;
            dst[64] = (float)c;
        }
    }
}

// The vector deposit u_b(node) = sum_k W(x_k - node) v_k,b accumulates in signed 64-bit fixed
// point, like the mass deposit, so that its result does not depend on the order of the atomic
// additions.  The scale 2^S comes from the largest |v|: with |v| < 2^e and N < 2^nb, every
// partial sum stays below 2^61 in magnitude for S = 61 - nb - e.

// *out = max |v| over n values, as the bit pattern of a non-negative double (those order like
// unsigned integers, so the maximum does not depend on the order of the atomics either).
__global__ void k_absmax_bits(const double *__restrict__ v, int64_t n, unsigned long long *__restrict__ out)
{
    unsigned long long m = 0ull;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(v[k]));
        m = b > m ? b : m;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, m, o);
        m = x > m ? x : m;
    }
    if ((threadIdx.x & 31) == 0 && m) atomicMax(out, m);
}

// s_out[0] = S for the largest |v| in *maxbits (0 when v is all zero or not finite).
__global__ void k_fix_exponent(const unsigned long long *__restrict__ maxbits, int nb, int *__restrict__ s_out)
{
    const double m = __longlong_as_double((long long)*maxbits);
    int S = 0;
    if (m > 0.0 && m <= 1.7976931348623157e308) {
        int e = 0;
        frexp(m, &e);  // m < 2^e
        S = 61 - nb - e;
        S = S > 1000 ? 1000 : S;
    }
    s_out[0] = S;
}

// u_b(node) += W(x_k - node) v_k,b as round(W v 2^S) on three fixed-point meshes.
// Bound by the FP64 pipe (17 cycles per warp and instruction on an SM).  |W v 2^S| < 2^(61 - nb), so from
// 2^10 particles on (nb > 10, kSmall false) the integer is in the low bits of fma(W, v 2^S, 1.5 2^52): one
// instruction for a product and a conversion, the same rounding to even.  128^3: 0.316 -> 0.208 ms.
template <bool kSmall>
__global__ void k_deposit_vec(const double *__restrict__ pos, const double *__restrict__ v,
                              P3MGeom g, const int *__restrict__ s_dev,
                              unsigned long long *__restrict__ fix)
{
    constexpr double kBig = 0x1.8p52;
    const int M = g.mesh;
    const int64_t n = g.n;
    const size_t M3 = (size_t)M * M * M;
    const double scale = ldexp(1.0, *s_dev);
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        const CicNodes c(pos[k], pos[n + k], pos[2 * n + k], g.inv_h, M);
        const double wx[2] = {1.0 - c.f[0], c.f[0]}, wy[2] = {1.0 - c.f[1], c.f[1]}, wz[2] = {1.0 - c.f[2], c.f[2]};
        const double vb[3] = {v[k] * scale, v[n + k] * scale, v[2 * n + k] * scale};
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const double wab = wx[a] * wy[b];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const double w = wab * wz[e];
                    const size_t node = c.node(a, b, e);
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const long long q = kSmall ? __double2ll_rn(w * vb[d])
                                                   : __double_as_longlong(fma(w, vb[d], kBig)) - __double_as_longlong(kBig);
                        atomicAdd(fix + d * M3 + node, (unsigned long long)q);
                    }
                }
            }
    }
}

// u = fix 2^-S (signed).
template <typename T>
__global__ void k_fix_to_vec(const unsigned long long *__restrict__ fix, size_t n,
                             const int *__restrict__ s_dev, T *__restrict__ u)
{
    const double inv_scale = ldexp(1.0, -*s_dev);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        u[i] = (T)(__ll2double_rn((long long)fix[i]) * inv_scale);
}

// psi_k = sum_b (+i kg_b G(k)) u_b,k with G as in the forward pass (constants included).
template <typename T, typename C2>
__global__ void k_kspace_adjoint(const C2 *__restrict__ ux, const C2 *__restrict__ uy,
                                 const C2 *__restrict__ uz, const T *__restrict__ tk,
                                 const T *__restrict__ tkg, const T *__restrict__ tg, int M,
                                 T gconst, C2 *__restrict__ psi)
{
    const int nz = M / 2 + 1;
    const size_t total = (size_t)M * M * nz;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int iz = (int)(idx % nz);
        const size_t t = idx / nz;
        const int iy = (int)(t % M), ix = (int)(t / M);
        const T kx = tk[ix], ky = tk[iy], kz = tk[iz];
        const T k2 = kx * kx + ky * ky + kz * kz;
        const T G = idx == 0 ? T(0) : gconst * (tg[ix] * tg[iy] * tg[iz]) / k2;
        const C2 a = ux[idx], b = uy[idx], c = uz[idx];
        // i kg G u = G kg (-u.y, u.x)
        const T gx = G * tkg[ix], gy = G * tkg[iy], gz = G * tkg[iz];
        C2 o;
        o.x = -(gx * a.y + gy * b.y + gz * c.y);
        o.y = gx * a.x + gy * b.x + gz * c.x;
        psi[idx] = o;
    }
}

// A finite FP32 value as FP64 by integer operations: the conversion instruction runs on the FP64 pipe.
__device__ __noinline__ double widen_special(float x) { return (double)x; }
__device__ __forceinline__ double widen(float x)
{
    const uint32_t u = __float_as_uint(x);
    // normal numbers; zero, denormal, infinite and NaN take the instruction
    if (((u << 1) - 0x01000000u) >= 0xFE000000u) return widen_special(x);
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }

// out_k += scale sum_corners grad W(x_k - node) [ sum_b v_k,b E_b(node) + psi(node) ]
// (E or v NULL: no first term; psi NULL: no second term).
// Bound by the FP64 pipe.  The gradient of the trilinear interpolant of the eight values by nested
// differences and interpolations (21 FP64 operations where the sum over weights takes 72), and the FP32
// meshes are widened by integer operations (32 values per particle): 128^3 0.563 -> 0.213 ms.
template <typename T>
__global__ void k_gather_grad(const double *__restrict__ pos, P3MGeom g, const T *__restrict__ E,
                              const double *__restrict__ v, const T *__restrict__ psi,
                              double scale, double *__restrict__ out)
{
    const int M = g.mesh;
    const int64_t n = g.n;
    const size_t M3 = (size_t)M * M * M;
    const double factor = scale * g.inv_h;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        const CicNodes c(pos[k], pos[n + k], pos[2 * n + k], g.inv_h, M);
        double vb[3] = {0.0, 0.0, 0.0};
        if (E && v) {
            vb[0] = v[k];
            vb[1] = v[n + k];
            vb[2] = v[2 * n + k];
        }
        double dz[2][2], m[2][2];  // per edge along z: difference, and value at the particle
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                double s[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const size_t node = c.node(a, b, e);
                    s[e] = psi ? widen(psi[node]) : 0.0;
                    if (E && v)
                        s[e] = fma(vb[2], widen(E[2 * M3 + node]),
                                   fma(vb[1], widen(E[M3 + node]), fma(vb[0], widen(E[node]), s[e])));
                }
                dz[a][b] = s[1] - s[0];
                m[a][b] = fma(c.f[2], dz[a][b], s[0]);
            }
        double q[2], dy[2], dzy[2];  // per edge along y, at the particle's z
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            dy[a] = m[a][1] - m[a][0];
            q[a] = fma(c.f[1], dy[a], m[a][0]);
            dzy[a] = fma(c.f[1], dz[a][1] - dz[a][0], dz[a][0]);
        }
        out[k] = fma(factor, q[1] - q[0], out[k]);
        out[n + k] = fma(factor, fma(c.f[0], dy[1] - dy[0], dy[0]), out[n + k]);
        out[2 * n + k] = fma(factor, fma(c.f[0], dzy[1] - dzy[0], dzy[0]), out[2 * n + k]);
    }
}

// Density loss on the mesh: rho holds counts - mean; delta = rho / n_bar; per node
// r = delta - target; loss partial sums per block; ell = 2 r / n_bar written over rho.
template <typename T>
__global__ void __launch_bounds__(256)
    k_loss_mesh(T *__restrict__ rho, const double *__restrict__ target, size_t M3, double inv_nbar,
                double *__restrict__ part)
{
    __shared__ double s[256];
    double acc = 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < M3;
         i += (size_t)gridDim.x * blockDim.x) {
        const double r = (double)rho[i] * inv_nbar - target[i];
        acc += r * r;
        rho[i] = (T)(2.0 * r * inv_nbar);
    }
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = s[0];
}

__global__ void k_sum_parts(double *part, int nb, double *out)
{
    __shared__ double s[256];
    double acc = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) acc += part[b];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = s[0];
}

// ------------------------------------------------------------------ pair part

// h(r)/Gm and h'(r)/(Gm r) for one pair in FP64, g and g' in closed form.
__device__ __forceinline__ void pair_jac(double r2, double eps2, double inv_rs, double &h,
                                         double &hr)
{
    const double r = sqrt(r2), x = r * inv_rs;
    const double s2 = r2 + eps2, s3 = s2 * sqrt(s2);
    const double gval = erfc(0.5 * x) + x * 0.56418958354775628695 * exp(-0.25 * x * x);
    const double gder = -x * x * exp(-0.25 * x * x) * 0.28209479177387814347;
    h = gval / s3;
    hr = (gder * inv_rs / s3 - 3.0 * r * gval / (s3 * s2)) / r;
}

template <typename T>
struct V4Of;
template <>
struct V4Of<float> {
    using type = float4;
};
template <>
struct V4Of<double> {
    using type = double4_16a;
};

// FP64 mode: one warp per work item (up to 32 particles of one cell, most expensive items first),
// like the force pair kernel: the j particles of the 27 neighbour cells in 32-slot blocks, a
// block skipped when no lane's particle is within r_c of its bounding box, evaluated without
// pair tests when it lies within r_c of every lane's particle; j data read through the cache
// and broadcast by shuffles.  out_k += Gm sum_j J(d_kj) (v_j - v_k).
__global__ void __launch_bounds__(32)
    k_pairs_vjp64(const double4_16a *__restrict__ rel, const double *__restrict__ pos,
                  const float4 *__restrict__ block_box, const double *__restrict__ vs,
                  const uint32_t *__restrict__ cell_start, const uint32_t *__restrict__ work,
                  const uint32_t *__restrict__ n_work_ptr,
                  P3MGeom g, float rcull2, float rin2, uint32_t *__restrict__ cursor,
                  double *__restrict__ out)
{
    const int lane = threadIdx.x;
    const int64_t n = g.n;
    const uint32_t n_work = *n_work_ptr;
    const double rc2 = g.r_c * g.r_c, eps2 = g.eps * g.eps, inv_rs = 1.0 / g.r_s;
    const int nc = g.n_c;
    for (;;) {
        uint32_t slot = 0;
        if (lane == 0) slot = atomicAdd(cursor, 1u);
        slot = __shfl_sync(0xffffffffu, slot, 0);
        if (slot >= n_work) break;
        const uint32_t item = slot;
        const uint32_t cell = work[2 * (size_t)item], first = work[2 * (size_t)item + 1];
        const uint32_t cend = cell_start[cell + 1];
        const int cx = (int)(cell % nc), cy = (int)((cell / nc) % nc), cz = (int)(cell / (nc * nc));
        const uint32_t i = first + lane;
        const bool valid = i < cend;
        const uint32_t ii = valid ? i : first;
        const double4_16a xi = rel[ii];
        const double xa = pos[ii], ya = pos[n + ii], za = pos[2 * n + ii];
        const double vix = vs[ii], viy = vs[n + ii], viz = vs[2 * n + ii];
        double o[3] = {0.0, 0.0, 0.0};
        for (int nb = 0; nb < 27; ++nb) {
            const int ux = cx + nb % 3 - 1, uy = cy + (nb / 3) % 3 - 1, uz = cz + nb / 9 - 1;
            const int wx = (ux + nc) % nc, wy = (uy + nc) % nc, wz = (uz + nc) % nc;
            const uint32_t q = ((uint32_t)wz * nc + wy) * nc + wx;
            const uint32_t js = cell_start[q], je = cell_start[q + 1];
            if (js == je) continue;
            const double L = g.box;
            const double ix = ux < 0 ? -L : (ux >= nc ? L : 0.0);
            const double iy = uy < 0 ? -L : (uy >= nc ? L : 0.0);
            const double iz = uz < 0 ? -L : (uz >= nc ? L : 0.0);
            const float cxs = (float)(xa - ix), cys = (float)(ya - iy), czs = (float)(za - iz);
            double ox = 0, oy = 0, oz = 0;
            for (uint32_t b = js >> 5; b * 32u < je; ++b) {
                const float4 lo = __ldg(block_box + 2 * b), hi = __ldg(block_box + 2 * b + 1);
                const float ex = fmaxf(fmaxf(lo.x - cxs, cxs - hi.x), 0.0f);
                const float ey = fmaxf(fmaxf(lo.y - cys, cys - hi.y), 0.0f);
                const float ez = fmaxf(fmaxf(lo.z - czs, czs - hi.z), 0.0f);
                if (!__any_sync(0xffffffffu, valid && ex * ex + ey * ey + ez * ez < rcull2)) continue;
                const float fx = fmaxf(cxs - lo.x, hi.x - cxs);
                const float fy = fmaxf(cys - lo.y, hi.y - cys);
                const float fz = fmaxf(czs - lo.z, hi.z - czs);
                const bool all_in =
                    __all_sync(0xffffffffu, !valid || fx * fx + fy * fy + fz * fz < rin2);
                const uint32_t j0 = max(b * 32, js), j1 = min(b * 32 + 32, je);
                // the block's particles: one coalesced load, then broadcast lane by lane
                const uint32_t jl = min(b * 32 + lane, (uint32_t)(n - 1));
                const double4_16a ql = rel[jl];
                const double vlx = vs[jl], vly = vs[n + jl], vlz = vs[2 * n + jl];
                for (uint32_t j = j0; j < j1; ++j) {
                    const int src = (int)(j - b * 32);
                    const double dx = (__shfl_sync(0xffffffffu, ql.x, src) - xi.x) + ix;
                    const double dy = (__shfl_sync(0xffffffffu, ql.y, src) - xi.y) + iy;
                    const double dz = (__shfl_sync(0xffffffffu, ql.z, src) - xi.z) + iz;
                    const double r2 = dx * dx + dy * dy + dz * dz;
                    const bool in = valid && (all_in || r2 < rc2) && r2 > 0.0;
                    const double w0 = __shfl_sync(0xffffffffu, vlx, src) - vix;
                    const double w1 = __shfl_sync(0xffffffffu, vly, src) - viy;
                    const double w2 = __shfl_sync(0xffffffffu, vlz, src) - viz;
                    if (!all_in && !__any_sync(0xffffffffu, in)) continue;
                    double h, hr;
                    pair_jac(r2, eps2, inv_rs, h, hr);
                    const double dw = dx * w0 + dy * w1 + dz * w2;
                    const double c = in ? hr * dw : 0.0;
                    const double hh = in ? h : 0.0;
                    ox += hh * w0 + c * dx;
                    oy += hh * w1 + c * dy;
                    oz += hh * w2 + c * dz;
                }
            }
            o[0] += ox;
            o[1] += oy;
            o[2] += oz;
        }
        if (valid) {
            out[i] += g.gm * o[0];
            out[n + i] += g.gm * o[1];
            out[2 * n + i] += g.gm * o[2];
        }
    }
}

// FP32 mode: the force kernel's lists (k_pairs_list in pair.cu: groups of 16 particles (8 or 4 of few), candidates
// tested one per lane against the group's box, the accepted ones compacted into a list, two particles
// and two list entries per lane in packed f32x2 arithmetic), here with v beside the coordinates, for
//   out_k += Gm sum_j [h w + (h'/r) (d.w) d],  w = v_j - v_k,
// where h is the force kernel's fitted factor and h'/r, in the additive form, twice the derivative of
// that fit with respect to w = r^2 + eps^2 (scaled lengths, q = s + ab + na t + e s^2, e = c[4], k = ln 2):
//   h = q s^2 + P(t),  h'/r = t (2 k (-na) s^2 - 2 k P'(t)) - (2 (q + e s^2) + s) s^4,
// as accurate as the closed form (1.9e-7 against 3.8e-7 of the force derivative at the cutoff 4.5) and
// without a second exponential.  The general form takes g' = -x^2 exp(-x^2/4)/(2 sqrt(pi)) closed.
// s^4 is never formed: (2 q + ..) s^2 times s^2 (d.w) stays finite for close pairs without softening.
// r = 0 pairs are selected out (their w need not vanish for coincident particles); only the row of the
// own cell can hold them.  Before, all 32 lanes met every j of a tested block with 40 FP32 operations
// and three 8-cycle MUFU operations per pair (36 and one here).  128^3 near-uniform, one call with the
// mesh part: 9.37 -> 6.71 ms, the pair part 7.6 -> 5.5.  What bounds it: of 143 cycles per 32 accepted
// pairs and scheduler, 117 are the evaluation (55 per 32 slots, 47 % of them accepted).  8 or 32
// particles per group, 18 or 20 CTAs per SM and lists of 192 are within 2 % or slower.
constexpr int kVjpChunk = 128, kVjpTerms = 80;  // FP32 terms per partial sum before it joins the FP64 sum
constexpr float kVjpTiny = 1e-24f, kVjpFar = 1e6f;

struct VjpConst2 {
    f2 c[5], d[3];  // P, and -2 k P' as d[0] + d[1] t + d[2] t^2 (additive form)
    f2 na, ab, e2, na2, two;
};

// h, and (h'/r) dw as *c, for both halves of w (see PairFactor)
template <bool kAdditive>
__device__ __forceinline__ f2 pair_jac2(f2 w, f2 dw, const VjpConst2 &k, f2 *c)
{
    const f2 t = f2_pack(ex2_approx(-w.x), ex2_approx(-w.y));
    const f2 rw = f2_pack(rsqrt_approx(w.x), rsqrt_approx(w.y));
    f2 p = kAdditive ? k.c[3] : f2_fma(k.c[4], t, k.c[3]);
    p = f2_fma(p, t, k.c[2]);
    p = f2_fma(p, t, k.c[1]);
    if (kAdditive) {
        const f2 s2 = f2_mul(rw, rw), q = f2_fma(k.c[4], s2, f2_add(rw, f2_fma(k.na, t, k.ab)));
        const f2 h = f2_fma(p, t, f2_fma(q, s2, k.c[0]));
        const f2 dp = f2_fma(f2_fma(k.d[2], t, k.d[1]), t, k.d[0]);
        const f2 inner = f2_mul(t, f2_fma(k.na2, s2, dp));
        const f2 m = f2_mul(f2_fma(k.two, f2_fma(k.c[4], s2, q), rw), s2);
        *c = f2_fma(inner, dw, f2_neg(f2_mul(m, f2_mul(s2, dw))));
        return h;
    }
    // d[0]: exponent of exp(-r^2/(4 r_s^2)) over t's, d[1]: -1/(2 sqrt(pi)) in scaled lengths, d[2]: -3
    p = f2_fma(p, t, k.c[0]);
    const f2 su = f2_add(w, k.e2), eu = f2_mul(w, k.d[0]);
    const f2 s = f2_pack(rsqrt_approx(su.x), rsqrt_approx(su.y));
    const f2 e = f2_pack(ex2_approx(-eu.x), ex2_approx(-eu.y));
    const f2 r = f2_mul(w, rw), s2 = f2_mul(s, s), s3 = f2_mul(s2, s);
    const f2 gv = f2_fma(r, f2_fma(w, p, f2_fma(k.na, t, k.ab)), f2_pack(1.0f, 1.0f));
    const f2 h = f2_mul(gv, s3);
    *c = f2_fma(f2_mul(f2_mul(r, e), f2_mul(s3, k.d[1])), dw, f2_mul(f2_mul(h, k.d[2]), f2_mul(s2, dw)));
    return h;
}

template <bool kAdditive, int kG>
__global__ void __launch_bounds__(32, 16)
    k_pairs_vjp_list(const uint32_t *__restrict__ relq, CutState cut, const float *__restrict__ vfx,
                     const float4 *__restrict__ block_box, const uint32_t *__restrict__ cell_start,
                     const uint32_t *__restrict__ work,
                     const uint32_t *__restrict__ n_work_ptr, P3MGeom g, PairFactor fac, double scale,
                     float rcull2, uint32_t *__restrict__ cursor, double *__restrict__ out)
{
    constexpr int kPairsI = kG / 2, kStride = 2 * (32 / kPairsI), kSub = P3M_PAIR_TI / kG;
    constexpr int kVjpFlush = kVjpTerms * kStride / kVjpChunk;
    __shared__ __align__(16) float list[6][kVjpChunk + 32];  // x, y, z, vx, vy, vz
    __shared__ uint32_t slot[kVjpChunk + 32];                // the sorted slot of each list entry
    __shared__ double sum[6][32];
    __shared__ PairSeg seg[kPairSegs];
    __shared__ LiveBlocks live;

    const int lane = threadIdx.x, ip = lane % kPairsI, js = lane / kPairsI;
    const uint32_t lt = (1u << lane) - 1u;
    const int64_t n = g.n;
    const uint32_t n_units = *n_work_ptr * kSub;
    const int nc = g.n_c;
    const float lambda = fac.lambda, rlist2 = fac.rlist2;
    VjpConst2 kc;
#pragma unroll
    for (int q = 0; q < 5; ++q) kc.c[q] = f2_pack(fac.c[q], fac.c[q]);
    kc.na = f2_pack(fac.na, fac.na);
    kc.ab = f2_pack(fac.ab, fac.ab);
    kc.e2 = f2_pack(fac.e2, fac.e2);
    const float k2 = 2.0f * 0.69314718055994531f;
    kc.na2 = f2_pack(-k2 * fac.na, -k2 * fac.na);
    kc.two = f2_pack(2.0f, 2.0f);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float d = kAdditive ? -k2 * (float)(q + 1) * fac.c[q + 1] : fac.grad[q];
        kc.d[q] = f2_pack(d, d);
    }
    const f2 w0 = kAdditive ? kc.e2 : f2_pack(kVjpTiny, kVjpTiny);

    for (;;) {
        uint32_t unit = 0;
        if (lane == 0) unit = atomicAdd(cursor, 1u);
        unit = __shfl_sync(0xffffffffu, unit, 0);
        if (unit >= n_units) break;
        const uint32_t item = unit / kSub;
        const uint32_t cell = work[2 * (size_t)item];
        const uint32_t first = work[2 * (size_t)item + 1] + (unit % kSub) * kG;
        const uint32_t cend = cell_start[cell + 1];
        if (first >= cend) continue;
        const int cx = (int)(cell % nc), cy = (int)((cell / nc) % nc), cz = (int)(cell / (nc * nc));
        const GroupFrame fr = group_frame<kG>(relq, first, cend, cx, cy, cz, lambda, fac.cell);
        const uint2 blocks = group_ranges(seg, cell_start, g, cx, cy, cz, fr, fac.cell);
#pragma unroll
        for (int q = 0; q < 6; ++q) sum[q][lane] = 0.0;

        // the lane's two particles, coordinates and v negated
        f2 nx[2][3], nv[2][3], o[2][3];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const uint32_t i = min(first + ip + u * kPairsI, cend - 1);
            const uint32_t *q = fix_coords(relq, i);
            const float *v = vfx + (size_t)(i >> 5) * 96 + (i & 31);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const float x = (float)(int)(__ldg(q + 32 * d) - fr.ctr[d]) * -lambda, y = -__ldg(v + 32 * d);
                nx[u][d] = f2_pack(x, x);
                nv[u][d] = f2_pack(y, y);
                o[u][d] = f2_pack(0.0f, 0.0f);
            }
        }
        auto flush = [&]() {
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    sum[3 * u + d][lane] += (double)(o[u][d].x + o[u][d].y);
                    o[u][d] = f2_pack(0.0f, 0.0f);
                }
        };
        // the pairs of a list in the cutoff's band: their terms are made whole or taken back
        auto settle = [&](int count) {
#pragma unroll 1
            for (int k = 0; k < 2 * count; k += kStride) {
                const int p = (k < count ? k : k - count + 1) + 2 * js;  // the first, then the second halves
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    float dx[3], wv[3];
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        dx[d] = list[d][p] + nx[u][d].x;
                        wv[d] = list[3 + d][p] + nv[u][d].x;
                    }
                    const float w = fmaf(dx[2], dx[2], fmaf(dx[1], dx[1], fmaf(dx[0], dx[0], w0.x)));
                    const float part = cut_part(w, fac.cut_m, fac.cut_b);
                    if (part == rintf(part)) continue;
                    const float dw = fmaf(dx[2], wv[2], fmaf(dx[1], wv[1], dx[0] * wv[0]));
                    const uint32_t i = min(first + ip + u * kPairsI, cend - 1);
                    const float t = (cut_inside<true>(relq, cut, g, i, slot[p], dx[0], dx[1], dx[2], fac) ? 1.0f : 0.0f) - part;
                    f2 c, h = pair_jac2<kAdditive>(f2_pack(w, w), f2_pack(dw, dw), kc, &c);
#pragma unroll
                    for (int d = 0; d < 3; ++d) o[u][d].x = fmaf(t * h.x, wv[d], fmaf(t * c.x, dx[d], o[u][d].x));
                }
            }
        };
        // list entries [0, count), count a multiple of kStride
        auto eval = [&](auto own, int count) {
            f2 hits = f2_pack(0.0f, 0.0f);
#pragma unroll 2
            for (int k = 2 * js; k < count; k += kStride) {
                f2 X[3], V[3];
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    X[d] = *(const f2 *)&list[d][k];
                    V[d] = *(const f2 *)&list[3 + d][k];
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    f2 dx[3], wv[3];
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        dx[d] = f2_add(X[d], nx[u][d]);
                        wv[d] = f2_add(V[d], nv[u][d]);
                    }
                    const f2 w = f2_fma(dx[2], dx[2], f2_fma(dx[1], dx[1], f2_fma(dx[0], dx[0], w0)));
                    const f2 dw = f2_fma(dx[2], wv[2], f2_fma(dx[1], wv[1], f2_mul(dx[0], wv[0])));
                    f2 c, h = pair_jac2<kAdditive>(w, dw, kc, &c);
                    f2 in = f2_pack(cut_part(w.x, fac.cut_m, fac.cut_b), cut_part(w.y, fac.cut_m, fac.cut_b));
                    if (decltype(own)::value) {
                        const bool nl = (__float_as_uint(dx[0].x) | __float_as_uint(dx[1].x) | __float_as_uint(dx[2].x)) != 0u;
                        const bool nh = (__float_as_uint(dx[0].y) | __float_as_uint(dx[1].y) | __float_as_uint(dx[2].y)) != 0u;
                        in = f2_pack(nl ? in.x : 0.0f, nh ? in.y : 0.0f);
                    }
                    hits = f2_add(hits, in);
                    h = f2_mul(h, in);
                    c = f2_mul(c, in);
#pragma unroll
                    for (int d = 0; d < 3; ++d) o[u][d] = f2_fma(h, wv[d], f2_fma(c, dx[d], o[u][d]));
                }
            }
            const float total = hits.x + hits.y;
            if (__any_sync(0xffffffffu, total != rintf(total))) settle(count);
        };

        int fill = 0, chunks = 0;
        auto walk = [&](auto own, uint32_t t0, uint32_t t1) {
            for (uint32_t base = t0; base < t1; base += 32) {
                const int nl = live_blocks(base + lane, t1, seg, block_box, fr, fac.length, rcull2, live);
                // the next block's data are loaded while the current one is tested
                uint32_t qn[3];
                float vn[3];
                auto fetch = [&](int k) {
                    const size_t at = (size_t)(live.at[k].word & kBlockMask) * 96 + lane;
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        qn[d] = __ldg(relq + at + 32 * d);
                        vn[d] = __ldg(vfx + at + 32 * d);
                    }
                };
                if (nl) fetch(0);
#pragma unroll 1
                for (int k = 0; k < nl; ++k) {
                    const LiveBlock S = live.at[k];
                    const float x = (float)(int)(qn[0] - S.cx) * lambda, y = (float)(int)(qn[1] - S.cy) * lambda,
                                z = (float)(int)(qn[2] - S.cz) * lambda;
                    const float vx = vn[0], vy = vn[1], vz = vn[2];
                    const bool mine = live.slots[k] >> lane & 1u;
                    if (k + 1 < nl) fetch(k + 1);
                    const float ex = fmaxf(fabsf(x) - fr.half[0], 0.0f), ey = fmaxf(fabsf(y) - fr.half[1], 0.0f),
                                ez = fmaxf(fabsf(z) - fr.half[2], 0.0f);
                    const bool in = mine && ex * ex + ey * ey + ez * ez < rlist2;
                    const uint32_t mm = __ballot_sync(0xffffffffu, in);
                    if (in) {
                        const int p = fill + __popc(mm & lt);
                        list[0][p] = x;
                        list[1][p] = y;
                        list[2][p] = z;
                        list[3][p] = vx;
                        list[4][p] = vy;
                        list[5][p] = vz;
                        slot[p] = (S.word & kBlockMask) << 5 | lane;
                    }
                    fill += __popc(mm);
                    if (fill >= kVjpChunk) {
                        __syncwarp();
                        eval(own, kVjpChunk);
                        __syncwarp();
                        fill -= kVjpChunk;
                        if (lane < fill) {  // (fill < 32 <= kVjpChunk: no overlap)
                            for (int d = 0; d < 6; ++d) list[d][lane] = list[d][kVjpChunk + lane];
                            slot[lane] = slot[kVjpChunk + lane];
                        }
                        if (++chunks % kVjpFlush == 0) flush();
                    }
                }
            }
            // the rest of the list, padded to whole steps with far entries
            const int count = (fill + kStride - 1) / kStride * kStride;
            if (lane < count - fill)
                for (int d = 0; d < 6; ++d) list[d][fill + lane] = d < 3 ? kVjpFar : 0.0f;
            __syncwarp();
            eval(own, count);
            __syncwarp();
            flush();
            fill = 0;
        };
        walk(std::true_type{}, 0u, blocks.x);
        walk(std::false_type{}, blocks.x, blocks.y);
        __syncwarp();
        for (int t = lane; t < 3 * kG; t += 32) {
            const int d = t / kG, k = t % kG;
            const uint32_t i = first + k;
            if (i >= cend) continue;
            double s = 0.0;
#pragma unroll
            for (int o_ = 0; o_ < 32 / kPairsI; ++o_) s += sum[3 * (k / kPairsI) + d][o_ * kPairsI + k % kPairsI];
            out[d * n + i] += scale * s;
        }
        __syncwarp();  // sum is cleared for the next group
    }
}

// ------------------------------------------------------------------ potential energy

// phi_k = G(k) rho_k (the potential spectrum of the forward pass, no gradient).
template <typename T, typename C2>
__global__ void k_kspace_potential(const C2 *__restrict__ rk, const T *__restrict__ tk,
                                   const T *__restrict__ tg, int M, T gconst, int green_only,
                                   C2 *__restrict__ out)
{
    const int nz = M / 2 + 1;
    const size_t total = (size_t)M * M * nz;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int iz = (int)(idx % nz);
        const size_t t = idx / nz;
        const int iy = (int)(t % M), ix = (int)(t / M);
        const T kx = tk[ix], ky = tk[iy], kz = tk[iz];
        const T k2 = kx * kx + ky * ky + kz * kz;
        const T G = idx == 0 ? T(0) : gconst * (tg[ix] * tg[iy] * tg[iz]) / k2;
        C2 o;
        if (green_only) {  // the kernel K = IFFT(G) itself
            o.x = G;
            o.y = T(0);
        } else {
            const C2 r = rk[idx];
            o.x = G * r.x;
            o.y = G * r.y;
        }
        out[idx] = o;
    }
}

// Per particle: Phi_LR(x_k) - S_k, S_k = sum_{c,c'} w_c w_c' K(n_c - n_c') (kself: K at the
// 27 offsets {-1,0,1}^3, index (dx+1)*9 + (dy+1)*3 + (dz+1)); phi_out[k] = that + cst.
template <typename T>
__global__ void k_gather_potential(const double *__restrict__ pos, P3MGeom g,
                                   const T *__restrict__ phi_mesh, const double *__restrict__ kself,
                                   double cst, double *__restrict__ phi_out)
{
    const int M = g.mesh;
    const int64_t n = g.n;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        int i3[3];
        double f3[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) stencil64(pos[d * n + k], g.inv_h, i3[d], f3[d]);
        double w[8];
        double phi = 0.0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int a = c >> 2, b = (c >> 1) & 1, e = c & 1;
            w[c] = (a ? f3[0] : 1.0 - f3[0]) * (b ? f3[1] : 1.0 - f3[1]) * (e ? f3[2] : 1.0 - f3[2]);
            const size_t node = ((size_t)wrap_index(i3[0] + a, M) * M + wrap_index(i3[1] + b, M)) * M +
                                wrap_index(i3[2] + e, M);
            phi += w[c] * (double)phi_mesh[node];
        }
        double self = 0.0;
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
            for (int d = 0; d < 8; ++d) {
                const int dx = (c >> 2) - (d >> 2), dy = ((c >> 1) & 1) - ((d >> 1) & 1),
                          dz = (c & 1) - (d & 1);
                self += w[c] * w[d] * kself[(dx + 1) * 9 + (dy + 1) * 3 + (dz + 1)];
            }
        phi_out[k] = phi - self + cst;
    }
}

// Short-range pair potential: phi_out[k] += -Gm sum_j erfc(r/(2 r_s)) / sqrt(r^2 + eps^2),
// the pair kernel's traversal (work items, block culling, shuffled j blocks).
template <typename T>
__global__ void __launch_bounds__(32)
    k_pairs_potential(const typename V4Of<T>::type *__restrict__ rel, const double *__restrict__ pos,
                      const float4 *__restrict__ block_box, const uint32_t *__restrict__ cell_start,
                      const uint32_t *__restrict__ work,
                      const uint32_t *__restrict__ n_work_ptr, P3MGeom g, float rcull2,
                      uint32_t *__restrict__ cursor, double *__restrict__ phi_out)
{
    using V4 = typename V4Of<T>::type;
    constexpr bool kAbsolute = sizeof(T) == 8;
    const int lane = threadIdx.x;
    const int64_t n = g.n;
    const uint32_t n_work = *n_work_ptr;
    const T rc2 = (T)(g.r_c * g.r_c), eps2 = (T)(g.eps * g.eps), half_inv_rs = (T)(0.5 / g.r_s);
    const int nc = g.n_c;
    for (;;) {
        uint32_t slot = 0;
        if (lane == 0) slot = atomicAdd(cursor, 1u);
        slot = __shfl_sync(0xffffffffu, slot, 0);
        if (slot >= n_work) break;
        const uint32_t item = slot;
        const uint32_t cell = work[2 * (size_t)item], first = work[2 * (size_t)item + 1];
        const uint32_t cend = cell_start[cell + 1];
        const int cx = (int)(cell % nc), cy = (int)((cell / nc) % nc), cz = (int)(cell / (nc * nc));
        const uint32_t i = first + lane;
        const bool valid = i < cend;
        const uint32_t ii = valid ? i : first;
        const V4 xi = rel[ii];
        const double xa = pos[ii], ya = pos[n + ii], za = pos[2 * n + ii];
        double acc = 0.0;
        for (int nb = 0; nb < 27; ++nb) {
            const int ux = cx + nb % 3 - 1, uy = cy + (nb / 3) % 3 - 1, uz = cz + nb / 9 - 1;
            const int wx = (ux + nc) % nc, wy = (uy + nc) % nc, wz = (uz + nc) % nc;
            const uint32_t q = ((uint32_t)wz * nc + wy) * nc + wx;
            const uint32_t js = cell_start[q], je = cell_start[q + 1];
            if (js == je) continue;
            const double L = g.box, cs = g.cs;
            const double imx = ux < 0 ? -L : (ux >= nc ? L : 0.0);
            const double imy = uy < 0 ? -L : (uy >= nc ? L : 0.0);
            const double imz = uz < 0 ? -L : (uz >= nc ? L : 0.0);
            T xs, ys, zs, ix = 0, iy = 0, iz = 0;
            if (kAbsolute) {
                xs = (T)xi.x;
                ys = (T)xi.y;
                zs = (T)xi.z;
                ix = (T)imx;
                iy = (T)imy;
                iz = (T)imz;
            } else {
                xs = (T)((double)xi.x - (((double)wx * cs + imx) - (double)cx * cs));
                ys = (T)((double)xi.y - (((double)wy * cs + imy) - (double)cy * cs));
                zs = (T)((double)xi.z - (((double)wz * cs + imz) - (double)cz * cs));
            }
            const float cxs = (float)(xa - imx), cys = (float)(ya - imy), czs = (float)(za - imz);
            T s = 0;
            for (uint32_t b = js >> 5; b * 32u < je; ++b) {
                const float4 lo = __ldg(block_box + 2 * b), hi = __ldg(block_box + 2 * b + 1);
                const float ex = fmaxf(fmaxf(lo.x - cxs, cxs - hi.x), 0.0f);
                const float ey = fmaxf(fmaxf(lo.y - cys, cys - hi.y), 0.0f);
                const float ez = fmaxf(fmaxf(lo.z - czs, czs - hi.z), 0.0f);
                if (!__any_sync(0xffffffffu, valid && ex * ex + ey * ey + ez * ez < rcull2)) continue;
                const uint32_t j0 = max(b * 32, js), j1 = min(b * 32 + 32, je);
                const uint32_t jl = min(b * 32 + lane, (uint32_t)(n - 1));
                const V4 ql = rel[jl];
                for (uint32_t j = j0; j < j1; ++j) {
                    const int src = (int)(j - b * 32);
                    T dx = __shfl_sync(0xffffffffu, (T)ql.x, src) - xs;
                    T dy = __shfl_sync(0xffffffffu, (T)ql.y, src) - ys;
                    T dz = __shfl_sync(0xffffffffu, (T)ql.z, src) - zs;
                    if (kAbsolute) {
                        dx += ix;
                        dy += iy;
                        dz += iz;
                    }
                    const T r2 = dx * dx + dy * dy + dz * dz;
                    const bool in = valid && r2 < rc2 && r2 > T(0);
                    if (!__any_sync(0xffffffffu, in)) continue;
                    const T term = erfc(sqrt(r2) * half_inv_rs) / sqrt(r2 + eps2);
                    s += in ? term : T(0);
                }
            }
            acc += (double)s;
        }
        if (valid) phi_out[i] -= g.gm * acc;
    }
}

// Sum of m/2 phi over particles, per-block partials then one block (fixed order).
__global__ void __launch_bounds__(256) k_sum_vec(const double *__restrict__ x, int64_t n, double *part)
{
    __shared__ double s[256];
    double a = 0.0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x)
        a += x[k];
    s[threadIdx.x] = a;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = s[0];
}

template <typename T, typename C2>
cudaError_t potential_impl(p3m_ctx *c, double cst, double *phi_slots, double *sum_dev)
{
    const int M = c->g.mesh;
    const size_t nk = (size_t)M * M * (M / 2 + 1);
    C2 *spec = (C2 *)c->frc_k;  // free after the force evaluation; FFT(rho) stays in rho_k
    T *mesh = (T *)c->adj_u;
    const int gk = grid_for((int64_t)nk, 256, c->num_sms);
    c->launches += 2;
    if (!c->kself_ready) {  // K = IFFT(G) near the origin, once per context
        k_kspace_potential<T, C2><<<gk, 256, 0, c->stream>>>(spec, (const T *)c->tab_k,
                                                             (const T *)c->tab_g, M,
                                                             (T)c->green_const, 1, spec);
        cufftResult r = sizeof(T) == 4 ? cufftExecC2R(c->plan_c2r_one, (cufftComplex *)spec, (cufftReal *)mesh)
                                       : cufftExecZ2D(c->plan_c2r_one, (cufftDoubleComplex *)spec,
                                                      (cufftDoubleReal *)mesh);
        if (r != CUFFT_SUCCESS) return cudaErrorUnknown;
        std::vector<T> host((size_t)M * M * M);
        double k27[27];
        cudaError_t e = cudaMemcpyAsync(host.data(), mesh, sizeof(T) * host.size(), cudaMemcpyDeviceToHost,
                                        c->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
        if (e != cudaSuccess) return e;
        for (int t = 0; t < 27; ++t) {
            const int dx = t / 9 - 1, dy = (t / 3) % 3 - 1, dz = t % 3 - 1;
            const size_t node = ((size_t)((dx + M) % M) * M + (dy + M) % M) * M + (dz + M) % M;
            k27[t] = (double)host[node];
        }
        e = cudaMemcpyAsync(c->kself, k27, sizeof(k27), cudaMemcpyHostToDevice, c->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
        if (e != cudaSuccess) return e;
        c->kself_ready = true;
    }
    // potential mesh from the current deposit (c->rho_k holds FFT(rho) after launch_deposit + R2C)
    k_kspace_potential<T, C2><<<gk, 256, 0, c->stream>>>((const C2 *)c->rho_k, (const T *)c->tab_k,
                                                         (const T *)c->tab_g, M, (T)c->green_const, 0,
                                                         spec);
    cufftResult r = sizeof(T) == 4 ? cufftExecC2R(c->plan_c2r_one, (cufftComplex *)spec, (cufftReal *)mesh)
                                   : cufftExecZ2D(c->plan_c2r_one, (cufftDoubleComplex *)spec,
                                                  (cufftDoubleReal *)mesh);
    if (r != CUFFT_SUCCESS) return cudaErrorUnknown;
    c->launches += 1;
    k_gather_potential<T><<<grid_for(c->g.n, 256, c->num_sms), 256, 0, c->stream>>>(
        c->pos, c->g, mesh, c->kself, cst, phi_slots);
    if (c->short_range) {
        int per_sm = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pairs_potential<T>, 32, 0);
        if (e != cudaSuccess) return e;
        e = cudaMemsetAsync(c->counters + 3, 0, sizeof(uint32_t), c->stream);
        if (e != cudaSuccess) return e;
        const double rcull = c->g.r_c * (1.0 + 1e-4) + c->g.box * 1e-6;
        c->launches += 1;
        k_pairs_potential<T><<<c->num_sms * (per_sm < 1 ? 1 : per_sm), 32, 0, c->stream>>>(
            (const typename V4Of<T>::type *)c->rel, c->pos, c->block_box, c->cell_start, c->work,
            c->n_work, c->g, (float)(rcull * rcull), c->counters + 3,
            phi_slots);
    }
    c->launches += 2;
    k_sum_vec<<<1024, 256, 0, c->stream>>>(phi_slots, c->g.n, c->red);
    k_sum_parts<<<1, 256, 0, c->stream>>>(c->red, 1024, sum_dev);
    return cudaGetLastError();
}

template <typename T, typename C2>
cudaError_t vjp_mesh(p3m_ctx *c, const double *v_slots, double *out_slots)
{
    const int M = c->g.mesh;
    const size_t M3 = (size_t)M * M * M, nk = (size_t)M * M * (M / 2 + 1);
    T *u = (T *)c->adj_u;
    unsigned long long *maxbits = (unsigned long long *)(c->fix_exp + 2);
    cudaError_t e = cudaMemsetAsync(maxbits, 0, sizeof(unsigned long long), c->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(c->rho_fix, 0, 3 * M3 * sizeof(unsigned long long), c->stream);
    if (e != cudaSuccess) return e;
    int nb = 0;
    while (nb < 63 && (c->g.n >> nb)) ++nb;
    const int gn = grid_for(c->g.n, 256, c->num_sms);
    c->launches += 6;
    k_absmax_bits<<<gn, 256, 0, c->stream>>>(v_slots, 3 * c->g.n, maxbits);
    k_fix_exponent<<<1, 1, 0, c->stream>>>(maxbits, nb, c->fix_exp);
    auto deposit = nb <= 10 ? k_deposit_vec<true> : k_deposit_vec<false>;
    deposit<<<gn, 256, 0, c->stream>>>(c->pos, v_slots, c->g, c->fix_exp, c->rho_fix);
    k_fix_to_vec<T><<<grid_for((int64_t)(3 * M3), 256, c->num_sms), 256, 0, c->stream>>>(c->rho_fix, 3 * M3,
                                                                                       c->fix_exp, u);
    C2 *uk = (C2 *)c->frc_k;
    for (int b = 0; b < 3; ++b) {
        cufftResult r = sizeof(T) == 4
                            ? cufftExecR2C(c->plan_r2c, (cufftReal *)(u + b * M3), (cufftComplex *)(uk + b * nk))
                            : cufftExecD2Z(c->plan_r2c, (cufftDoubleReal *)(u + b * M3),
                                           (cufftDoubleComplex *)(uk + b * nk));
        if (r != CUFFT_SUCCESS) return cudaErrorUnknown;
    }
    C2 *psik = (C2 *)c->rho_k;
    k_kspace_adjoint<T, C2><<<grid_for((int64_t)nk, 256, c->num_sms), 256, 0, c->stream>>>(
        uk, uk + nk, uk + 2 * nk, (const T *)c->tab_k, (const T *)c->tab_kg, (const T *)c->tab_g, M,
        (T)c->green_const, psik);
    T *psi = (T *)c->rho;
    cufftResult r = sizeof(T) == 4 ? cufftExecC2R(c->plan_c2r_one, (cufftComplex *)psik, (cufftReal *)psi)
                                   : cufftExecZ2D(c->plan_c2r_one, (cufftDoubleComplex *)psik,
                                                  (cufftDoubleReal *)psi);
    if (r != CUFFT_SUCCESS) return cudaErrorUnknown;
    k_gather_grad<T><<<grid_for(c->g.n, 256, c->num_sms), 256, 0, c->stream>>>(
        c->pos, c->g, (const T *)c->frc, v_slots, psi, 1.0, out_slots);
    return cudaGetLastError();
}

cudaError_t vjp_pairs(p3m_ctx *c, const double *v_slots, double *out_slots)
{
    int per_sm = 0;
    const bool fp32 = c->precision == P3M_PREC_MIXED;
    const int group = pair_group(c);
    const bool add = c->pair_factor.additive != 0;
    auto list = group == 4   ? (add ? k_pairs_vjp_list<true, 4> : k_pairs_vjp_list<false, 4>)
                : group == 8 ? (add ? k_pairs_vjp_list<true, 8> : k_pairs_vjp_list<false, 8>)
                             : (add ? k_pairs_vjp_list<true, 16> : k_pairs_vjp_list<false, 16>);
    cudaError_t e = fp32 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, list, 32, 0)
                         : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pairs_vjp64, 32, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    e = cudaMemsetAsync(c->counters + 3, 0, sizeof(uint32_t), c->stream);
    if (e != cudaSuccess) return e;
    const double rcull = c->g.r_c * (1.0 + 1e-4) + c->g.box * 1e-6;
    const double rin = c->g.r_c * (1.0 - 1e-4) - c->g.box * 1e-6;
    const float rcull2 = (float)(rcull * rcull), rin2 = rin > 0.0 ? (float)(rin * rin) : 0.0f;
    c->launches += 1;
    if (fp32) {
        const double len = ldexp(c->g.cs, -kFixBits) / (double)c->pair_factor.lambda;
        list<<<c->num_sms * per_sm, 32, 0, c->stream>>>(
            c->relq, CutState{(const float4 *)c->rel, c->keys}, c->adj_vfx, c->block_box, c->cell_start, c->work,
            c->n_work, c->g, c->pair_factor, c->g.gm / (len * len * len), rcull2,
            c->counters + 3, out_slots);
    } else {
        k_pairs_vjp64<<<c->num_sms * per_sm, 32, 0, c->stream>>>(
            (const double4_16a *)c->rel, c->pos, c->block_box, v_slots, c->cell_start, c->work,
            c->n_work, c->g, rcull2, rin2, c->counters + 3,
            out_slots);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_to_slots(p3m_ctx *c, const double *v, double *vs)
{
    c->launches += 1;
    k_to_slots<<<grid_for(c->g.n, 256, c->num_sms), 256, 0, c->stream>>>(
        v, c->pid, c->g.n, vs, c->precision == P3M_PREC_MIXED ? c->adj_vfx : nullptr);
    return cudaGetLastError();
}

cudaError_t launch_force_vjp(p3m_ctx *c, const double *v_slots, double *out_slots)
{
    cudaError_t e = cudaMemsetAsync(out_slots, 0, 3 * sizeof(double) * c->g.n, c->stream);
    if (e != cudaSuccess) return e;
    if (c->precision == P3M_PREC_MIXED) {
        e = vjp_mesh<float, cufftComplex>(c, v_slots, out_slots);
        if (e == cudaSuccess && c->short_range) e = vjp_pairs(c, v_slots, out_slots);
    } else {
        e = vjp_mesh<double, cufftDoubleComplex>(c, v_slots, out_slots);
        if (e == cudaSuccess && c->short_range) e = vjp_pairs(c, v_slots, out_slots);
    }
    return e;
}

cudaError_t launch_potential(p3m_ctx *c, double cst, double *phi_slots, double *sum_dev)
{
    return c->precision == P3M_PREC_MIXED ? potential_impl<float, cufftComplex>(c, cst, phi_slots, sum_dev)
                                          : potential_impl<double, cufftDoubleComplex>(c, cst, phi_slots, sum_dev);
}

cudaError_t launch_density_loss(p3m_ctx *c, const double *target, double *loss_dev, double *grad_slots)
{
    const int M = c->g.mesh;
    const size_t M3 = (size_t)M * M * M;
    const double inv_nbar = 1.0 / c->g.mean_count;
    const int nb = 1024;
    c->launches += 2;
    if (c->precision == P3M_PREC_MIXED)
        k_loss_mesh<float><<<nb, 256, 0, c->stream>>>((float *)c->rho, target, M3, inv_nbar, c->red);
    else
        k_loss_mesh<double><<<nb, 256, 0, c->stream>>>((double *)c->rho, target, M3, inv_nbar, c->red);
    k_sum_parts<<<1, 256, 0, c->stream>>>(c->red, nb, loss_dev);
    if (grad_slots) {
        cudaError_t e = cudaMemsetAsync(grad_slots, 0, 3 * sizeof(double) * c->g.n, c->stream);
        if (e != cudaSuccess) return e;
        c->launches += 1;
        if (c->precision == P3M_PREC_MIXED)
            k_gather_grad<float><<<grid_for(c->g.n, 256, c->num_sms), 256, 0, c->stream>>>(
                c->pos, c->g, nullptr, nullptr, (const float *)c->rho, 1.0, grad_slots);
        else
            k_gather_grad<double><<<grid_for(c->g.n, 256, c->num_sms), 256, 0, c->stream>>>(
                c->pos, c->g, nullptr, nullptr, (const double *)c->rho, 1.0, grad_slots);
    }
    return cudaGetLastError();
}
