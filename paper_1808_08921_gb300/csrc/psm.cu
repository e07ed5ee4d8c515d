// psm.cu -- a smooth surrogate of the fluid-solid coupling, for the gradient
// of the probe-plane pressure misfit with respect to the sphere positions of
// a fixed packing.  It lies outside the paper's chosen method: with the
// binary solid map of the momentum-exchange coupling (Section 2.3, Eqs.
// 14-15) the misfit is piecewise constant in the centres, so the gradient is
// taken of a surrogate from the family the paper names as the alternative
// (Section 1: Noble and Torczynski's collision weighted by the solid volume
// fraction of each cell).
//
// Model (dense lattice, every node carries populations, deviations
// g = f - w rho_f, FP32 arithmetic):
//   * solid fraction eps(x) = 1 - prod_p (1 - S(R_p - |x - X_p| + 1/2)), S the
//     cubic smoothstep (0 below 0, 3 s^2 - 2 s^3 on [0, 1], 1 above), the
//     distance to the nearest periodic image; the x ends of a non-periodic
//     lattice stay fluid;
//   * collision  g*_i = g_i - a (g_i - g^eq_i) + B Om_i,  a = (1 - B)/tau,
//     B = eps (tau - 1/2) / ((1 - eps) + (tau - 1/2)),
//     Om_i = g_opp(i) - g_i + w_i drho - g^eq_opp(i)  (the bounce-back of the
//     non-equilibrium part towards a resting solid);
//   * streaming of every population to x + c_i; a population leaving the x
//     range comes back reversed (resting wall); then the pressure inlet
//     (Zou-He, Eq. 25) and the outlet, as in the coupled step;
//   * probe: c_s^2 times the mean density over every node of plane probe_x.
// Reverse mode, for L = sum_k l_k(g_k) and the adjoint lam_k = dL/dg_k:
//   mu = S^T B^T lam_{k+1} (the adjoint of the post-collision state:
//   mu_i(x) = lam_i(x + c_i), or lam_opp(i)(x) where the population left the
//   lattice), then
//   lam_k = (1 - a - B) mu + B mu_opp + B (w . mu) 1 + A(nu) + Bv(nu) . c + dl_k/dg_k,
//   nu_i = a mu_i - B mu_opp(i), A and Bv the contractions of nu with
//   dg^eq/d(drho) and dg^eq/dJ;
//   dL/dtau += mu . dg*/dtau, G(x) += mu . dg*/deps at every node, and at the
//   end dL/dX_p = sum_x G(x) deps(x)/dX_p.
#include "common.cuh"
#include "kernels.cuh"

namespace lbmdem {

__device__ __forceinline__ size_t dense(const PsmArgs& A, int x, int y, int z) {
    return ((size_t)x * A.ny + y) * A.nz + z;
}

// node of this thread in the 3-D launch of psm_grid: z along the block's
// threads, y and x from the block indices (no integer division); false past
// the end of a z line or of a plane's lines
__device__ __forceinline__ bool grid_node(const PsmArgs& A, int& x, int& y, int& z, size_t& k) {
    z = blockIdx.x * blockDim.x + threadIdx.x;
    y = blockIdx.y * blockDim.y + threadIdx.y;
    x = blockIdx.z;
    k = dense(A, x, y, z);
    return z < A.nz && y < A.ny;
}

__device__ __forceinline__ double smooth_step(double v) {
    if (v <= 0.0) return 0.0;
    if (v >= 1.0) return 1.0;
    return v * v * (3.0 - 2.0 * v);
}

// node offset from a centre along one axis, nearest periodic image; iL = 1/L
// (the image count differs from that of d / L at most where both images are
// equally far)
__device__ __forceinline__ double image(double d, double L, double iL, bool periodic) {
    return periodic ? d - L * floor(d * iL + 0.5) : d;
}

// One block per segment of a z line.  The block first collects, in index
// order, the spheres that can reach the segment (their distance in the x, y
// plane and to the z interval, with a margin of 0.01 lu over the exact test
// below, far above the FP32 rounding of offsets within the box); its nodes then
// evaluate only those.  Evaluating every sphere at every node is FP64
// arithmetic at 2 lanes per clock and SM: 7.77 ms for 128 spheres on 64 x 64 x
// 256, against 0.31 ms.  The kept spheres go through the same test and product
// in the same order, so eps is the same bit for bit.  A segment reached by more
// than EPS_LIST spheres walks them all.
constexpr int EPS_LIST = 256;
__global__ void k_psm_eps(PsmArgs A, const double* X, const double* R, int n, float* eps) {
    __shared__ int s_list[EPS_LIST];
    __shared__ int s_count[9];  // per warp, then the list's length
    int x, y, z;
    size_t k;
    const bool inside = grid_node(A, x, y, z, k);
    const bool end = !A.px && (x == 0 || x == A.nx - 1);  // uniform over the block
    if (end) {
        if (inside) eps[k] = 0.f;
        return;
    }
    const int z0 = blockIdx.x * blockDim.x, z1 = min(z0 + (int)blockDim.x, A.nz) - 1;
    const double zc = 0.5 * (z0 + z1), iL[3] = {1.0 / A.nx, 1.0 / A.ny, 1.0 / A.nz};
    const float zh = 0.5f * (float)(z1 - z0);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int total = 0;
    for (int p0 = 0; p0 < n; p0 += blockDim.x) {
        const int p = p0 + threadIdx.x;
        bool near = false;
        if (p < n) {
            const float rx = (float)image(x - X[3 * p], A.nx, iL[0], A.px),
                        ry = (float)image(y - X[3 * p + 1], A.ny, iL[1], true);
            const float dz = fmaxf(fabsf((float)image(zc - X[3 * p + 2], A.nz, iL[2], true)) - zh, 0.f);
            const float reach = (float)R[p] + 0.51f;
            near = rx * rx + ry * ry + dz * dz < reach * reach;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, near);
        if (lane == 0) s_count[wid] = __popc(bal);
        __syncthreads();
        int at = total;
        for (int w = 0; w < nw; ++w) {
            if (w < wid) at += s_count[w];
            total += s_count[w];
        }
        at += __popc(bal & ((1u << lane) - 1u));
        if (near && at < EPS_LIST) s_list[at] = p;
        __syncthreads();
    }
    if (!inside) return;
    const bool all = total > EPS_LIST;
    const int m = all ? n : total;
    double keep = 1.0;
    for (int t = 0; t < m; ++t) {
        const int p = all ? t : s_list[t];
        const double rx = image(x - X[3 * p], A.nx, iL[0], A.px), ry = image(y - X[3 * p + 1], A.ny, iL[1], true),
                     rz = image(z - X[3 * p + 2], A.nz, iL[2], true);
        const double d2 = rx * rx + ry * ry + rz * rz, reach = R[p] + 0.5;
        if (d2 >= reach * reach) continue;
        keep *= 1.0 - smooth_step(R[p] - sqrt(d2) + 0.5);
    }
    eps[k] = (float)(1.0 - keep);
}

// collision weights of a node: B, a = (1 - B)/tau
__device__ __forceinline__ void psm_weights(float e, float tau, float& B, float& a) {
    const float sh = tau - 0.5f;
    B = e * sh / ((1.0f - e) + sh);
    a = (1.0f - B) / tau;
}

// Push step.  156 B per node: 24 us at the copy rate on 64 x 64 x 256.  Each
// population is read once and then dead, and its successor is read by the
// next step, so the reads are evict-first.  Pairs of opposite directions share
// their equilibrium terms: 41.4 -> 39 us with both; the reverse step's
// evict-first reads 63 -> 61 us.
__global__ void __launch_bounds__(256) k_psm_step(PsmArgs A, const float* gin, float* gout, const float* eps) {
    int x, y, z;
    size_t k;
    if (!grid_node(A, x, y, z, k)) return;
    float g[Q];
#pragma unroll
    for (int m = 0; m < Q; ++m) g[m] = __ldcs(gin + (size_t)m * A.N + k);
    const RevMoments M = rev_moments(g, A.rho_f);
    float B, a;
    psm_weights(eps[k], A.tau, B, a);
    const int ym = y == 0 ? A.ny - 1 : y - 1, yp = y == A.ny - 1 ? 0 : y + 1;
    const int zm = z == 0 ? A.nz - 1 : z - 1, zp = z == A.nz - 1 ? 0 : z + 1;
    auto put = [&](int m, float gs) {
        int xs = x + cx(m);
        if (A.px) {
            xs = xs < 0 ? A.nx - 1 : (xs >= A.nx ? 0 : xs);
        } else if (xs < 0 || xs >= A.nx) {
            gout[(size_t)opp(m) * A.N + k] = gs;  // resting wall at the x ends
            return;
        }
        const int ys = cy(m) > 0 ? yp : (cy(m) < 0 ? ym : y), zs = cz(m) > 0 ? zp : (cz(m) < 0 ? zm : z);
        gout[(size_t)m * A.N + dense(A, xs, ys, zs)] = gs;
    };
    // g* = g - a d + B Om with d = g - g^eq and Om_m = d_opp(m) - (g_m - w drho);
    // the rest population takes what the moving ones leave of the density, so
    // that the FP32 weights (their sum is 1 + 1.5e-8) conserve mass
    float moving = 0.f;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const int m = pair_m(q), o = opp(m);
        float cu, em, eo;
        rev_eq(M, m, cu, em, eo);
        moving += em + eo;
        const float dm = g[m] - em, d_o = g[o] - eo, wd = wt(m) * M.drho;
        put(m, g[m] - a * dm + B * (d_o - (g[m] - wd)));
        put(o, g[o] - a * d_o + B * (dm - (g[o] - wd)));
    }
    const float e18 = M.drho - moving;
    put(18, g[18] - a * (g[18] - e18) + B * (wt(18) * M.drho - e18));
}

// the pressure inlet and the outlet on the state t + 1 (one thread per line)
__global__ void k_psm_boundary(PsmArgs A, float* g, Source src, unsigned long long t1) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= A.ny * A.nz) return;
    const int y = k / A.nz, z = k - y * A.nz;
    if (A.inlet == 0) {
        const size_t i = dense(A, 0, y, z);
        float f[Q];
#pragma unroll
        for (int m = 0; m < Q; ++m) f[m] = g[(size_t)m * A.N + i];
        pressure_face(f, (float)source_drho(src, t1), 0);
#pragma unroll
        for (int m = 0; m < Q; ++m)
            if (cx(m) > 0) g[(size_t)m * A.N + i] = f[m];
    }
    const size_t o = dense(A, A.nx - 1, y, z);
    if (A.outlet == 0) {
        const size_t u = dense(A, A.nx - 2, y, z);
#pragma unroll
        for (int m = 0; m < Q; ++m)
            if (cx(m) < 0) g[(size_t)m * A.N + o] = g[(size_t)m * A.N + u];
    } else if (A.outlet == 1) {
        float f[Q];
#pragma unroll
        for (int m = 0; m < Q; ++m) f[m] = g[(size_t)m * A.N + o];
        pressure_face(f, 0.f, 1);
#pragma unroll
        for (int m = 0; m < Q; ++m)
            if (cx(m) < 0) g[(size_t)m * A.N + o] = f[m];
    }
}

// sum of the density deviations over plane probe_x (FP64 atomics per warp)
__global__ void k_psm_probe(PsmArgs A, const float* g, double* out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    double s = 0.0;
    if (k < A.ny * A.nz) {
        const size_t i = dense(A, A.probe_x, k / A.nz, k % A.nz);
        float d = 0.f;
#pragma unroll
        for (int m = 0; m < Q; ++m) d += g[(size_t)m * A.N + i];
        s = d;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0 && s != 0.0) atomicAdd(out, s);
}

// B^T in place on the adjoint of the state t + 1 (the transposed Zou-He face
// and outlet) and the amplitude derivative d rho_in / d rho' = shape(t + 1)
__global__ void k_psm_adj_boundary(PsmArgs A, float* a, double shape, double* d_amp) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    double da = 0.0;
    if (k < A.ny * A.nz) {
        const int y = k / A.nz, z = k - y * A.nz;
        const size_t P = A.N;
        if (A.inlet == 0) {
            const size_t i = dense(A, 0, y, z);
            da = (double)adj_face<0>(a + i, P) * shape;
        }
        const size_t o = dense(A, A.nx - 1, y, z);
        if (A.outlet == 0) {
            const size_t u = dense(A, A.nx - 2, y, z);
            adj_copy(a, P, u, o);
        } else if (A.outlet == 1) {
            adj_face<1>(a + o, P);
        }
    }
#pragma unroll
    for (int s = 16; s; s >>= 1) da += __shfl_xor_sync(0xffffffffu, da, s);
    if ((threadIdx.x & 31) == 0 && da != 0.0) atomicAdd(d_amp, da);
}

// lam_k = J^T mu + dl_k / dg_k at every node, with the tau and eps derivatives.
// 248 B per node (39 us at the copy rate on 64 x 64 x 256), but bound by issue
// and occupancy: 2600 instructions per warp at 140 registers took 147 us.  The
// pairwise contractions, the derivatives as two sums with per-node factors
// (no division per direction) and blocks of 256 threads at 80 registers (24
// warps per SM; 119 registers and 16 warps: 83 us) bring it to 63 us.
__global__ void __launch_bounds__(GRAD_THREADS, 3) k_psm_adj_step(PsmArgs A, const float* lin, const float* gt, float* lout,
                                                      const float* eps, float dl, double* d_tau, double* G) {
    int x, y, z;
    size_t k;
    float dt = 0.f;
    if (grid_node(A, x, y, z, k)) {
        const int ym = y == 0 ? A.ny - 1 : y - 1, yp = y == A.ny - 1 ? 0 : y + 1;
        const int zm = z == 0 ? A.nz - 1 : z - 1, zp = z == A.nz - 1 ? 0 : z + 1;
        float mu[Q];
#pragma unroll
        for (int m = 0; m < Q; ++m) {  // S^T: pull the adjoint back along c_m
            int xs = x + cx(m);
            bool out = false;
            if (A.px) xs = xs < 0 ? A.nx - 1 : (xs >= A.nx ? 0 : xs);
            else out = xs < 0 || xs >= A.nx;
            const int ys = cy(m) > 0 ? yp : (cy(m) < 0 ? ym : y), zs = cz(m) > 0 ? zp : (cz(m) < 0 ? zm : z);
            mu[m] = __ldcs(out ? lin + (size_t)opp(m) * A.N + k : lin + (size_t)m * A.N + dense(A, xs, ys, zs));
        }
        float g[Q];
#pragma unroll
        for (int m = 0; m < Q; ++m) g[m] = __ldcs(gt + (size_t)m * A.N + k);
        const RevMoments M = rev_moments(g, A.rho_f);
        const float e = eps[k], tau = A.tau, sh = tau - 0.5f, den = (1.0f - e) + sh;
        float B, a;
        psm_weights(e, tau, B, a);
        // with d_m = g_m - g^eq_m:  Om_m = d_opp(m) - (g_m - w drho), and the
        // tau and eps derivatives are two sums, mu.d and mu.Om, with per-node
        // factors
        RevSums S;
        float sd, so, wmu;
        {
            const float e18 = wt(18) * (M.drho - M.rho * M.uu15);
            sd = mu[18] * (g[18] - e18);
            so = mu[18] * (wt(18) * M.drho - e18);
            wmu = 12.f * mu[18];
        }
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int m = pair_m(q), o = opp(m);
            float cu, em, eo;
            rev_eq(M, m, cu, em, eo);
            const float dm = g[m] - em, d_o = g[o] - eo, wd = wt(m) * M.drho;
            sd += mu[m] * dm + mu[o] * d_o;
            so += mu[m] * (d_o - (g[m] - wd)) + mu[o] * (dm - (g[o] - wd));
            const float p = mu[m] + mu[o], r = mu[m] - mu[o];
            wmu += RevSums::iw(m) * p;
            S.add(m, cu, (a - B) * p, (a + B) * r);  // nu = a mu - B mu_opp
        }
        S.finish(M, (a - B) * mu[18]);
        const float id = 1.0f / (den * den), it = 1.0f / tau;
        const float dB_dtau = e * (1.0f - e) * id, dB_de = sh * (1.0f + sh) * id;
        const float da_dtau = -dB_dtau * it - (1.0f - B) * it * it;
        const float st = dB_dtau * so - da_dtau * sd, se = dB_de * (sd * it + so);
        const float base = B * RevSums::scaled(wmu) + S.A + (x == A.probe_x ? dl : 0.f), keep = 1.0f - a - B;
#pragma unroll
        for (int m = 0; m < Q; ++m) lout[(size_t)m * A.N + k] = keep * mu[m] + B * mu[opp(m)] + (base + S.dot(m));
        G[k] += (double)se;
        dt = st;
    }
    block_sum_to(dt, d_tau + (blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)) % GRAD_COPIES);
}

// dL/dX_p = sum_x G(x) deps(x)/dX_p over the shell where sphere p's
// smoothstep varies (one block per sphere); deps/deps_p = (1 - eps)/(1 - eps_p)
// is the product over the other spheres, deps_p/dX_p = S'(s) (x - X_p)/d
__global__ void k_psm_grad_x(PsmArgs A, const double* G, const float* eps, const double* X, const double* R,
                             double* dX) {
    const int p = blockIdx.x;
    const double X0 = X[3 * p], X1 = X[3 * p + 1], X2 = X[3 * p + 2], Rp = R[p];
    const double reach = Rp + 0.5;
    const int x0 = (int)floor(X0 - reach), x1 = (int)ceil(X0 + reach);
    const int y0 = (int)floor(X1 - reach), y1 = (int)ceil(X1 + reach);
    const int z0 = (int)floor(X2 - reach), z1 = (int)ceil(X2 + reach);
    const int ey = y1 - y0 + 1, ez = z1 - z0 + 1;
    const long long vol = (long long)(x1 - x0 + 1) * ey * ez;
    double s[3] = {0.0, 0.0, 0.0};
    for (long long t = threadIdx.x; t < vol; t += blockDim.x) {
        const int zi = z0 + (int)(t % ez), yi = y0 + (int)((t / ez) % ey), xi = x0 + (int)(t / ((long long)ey * ez));
        int x = xi;
        if (A.px) x = ((x % A.nx) + A.nx) % A.nx;
        else if (x <= 0 || x >= A.nx - 1) continue;  // fluid x ends
        const int y = ((yi % A.ny) + A.ny) % A.ny, z = ((zi % A.nz) + A.nz) % A.nz;
        const double rx = (double)xi - X0, ry = (double)yi - X1, rz = (double)zi - X2;
        const double d = sqrt(rx * rx + ry * ry + rz * rz);
        const double v = Rp - d + 0.5;
        if (v <= 0.0 || v >= 1.0 || d == 0.0) continue;
        const double ep = smooth_step(v), dS = 6.0 * v * (1.0 - v);
        const size_t k = dense(A, x, y, z);
        const double f = G[k] * (1.0 - (double)eps[k]) / (1.0 - ep) * dS / d;
        s[0] += f * rx;
        s[1] += f * ry;
        s[2] += f * rz;
    }
    __shared__ double red[3][32];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int o = 16; o; o >>= 1) s[a] += __shfl_xor_sync(0xffffffffu, s[a], o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0)
        for (int a = 0; a < 3; ++a) red[a][wid] = s[a];
    __syncthreads();
    if (threadIdx.x < 3) {
        double tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[threadIdx.x][w];
        dX[3 * p + threadIdx.x] = tot;
    }
}

// one thread per node: segments of z lines of up to 256 threads and, where
// the lines are shorter, several lines per block up to 256 threads in all
// (lines: 1 for the kernel whose blocks work on one line)
static void psm_grid(const PsmArgs& A, dim3& grid, dim3& block, int lines = 0) {
    const int tz = A.nz >= 256 ? 256 : ((A.nz + 31) / 32) * 32;
    const int ty = lines ? lines : GRAD_THREADS / tz;
    block = dim3(tz, ty, 1);
    grid = dim3((A.nz + tz - 1) / tz, (A.ny + ty - 1) / ty, A.nx);
}

void launch_psm_eps(const PsmArgs& A, const double* X, const double* R, int n, float* eps, cudaStream_t s) {
    dim3 g, b;
    psm_grid(A, g, b, 1);
    k_psm_eps<<<g, b, 0, s>>>(A, X, R, n, eps);
}
void launch_psm_step(const PsmArgs& A, const float* gin, float* gout, const float* eps, cudaStream_t s) {
    dim3 g, b;
    psm_grid(A, g, b);
    k_psm_step<<<g, b, 0, s>>>(A, gin, gout, eps);
}
void launch_psm_boundary(const PsmArgs& A, float* g, const Source& src, unsigned long long t1, cudaStream_t s) {
    if (A.px) return;
    const int n = A.ny * A.nz;
    k_psm_boundary<<<(n + 127) / 128, 128, 0, s>>>(A, g, src, t1);
}
void launch_psm_probe(const PsmArgs& A, const float* g, double* out, cudaStream_t s) {
    const int n = A.ny * A.nz;
    k_psm_probe<<<(n + 127) / 128, 128, 0, s>>>(A, g, out);
}
void launch_psm_adj_boundary(const PsmArgs& A, float* lam, double shape, double* d_amp, cudaStream_t s) {
    if (A.px) return;
    const int n = A.ny * A.nz;
    k_psm_adj_boundary<<<(n + 127) / 128, 128, 0, s>>>(A, lam, shape, d_amp);
}
void launch_psm_adj_step(const PsmArgs& A, const float* lin, const float* gt, float* lout, const float* eps, float dl,
                         double* d_tau, double* G, cudaStream_t s) {
    dim3 g, b;
    psm_grid(A, g, b);
    k_psm_adj_step<<<g, b, 0, s>>>(A, lin, gt, lout, eps, dl, d_tau, G);
}
void launch_psm_grad_x(const PsmArgs& A, const double* G, const float* eps, const double* X, const double* R, int n,
                       double* dX, cudaStream_t s) {
    if (n > 0) k_psm_grad_x<<<n, 256, 0, s>>>(A, G, eps, X, R, dX);
}

}  // namespace lbmdem
