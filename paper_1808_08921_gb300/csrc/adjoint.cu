// adjoint.cu -- reverse-mode (adjoint) kernels of the lattice step for a
// fixed packing, for the gradient of a probe-plane pressure misfit with
// respect to the relaxation time tau and the source amplitude rho'.
//
// With every sphere fixed the coupled step t -> t+1 acts on the natural
// populations n_t (the state entering step t) as
//     n_{t+1} = B_{t+1}( S( C(n_t) ) )
// C: BGK collision at every fluid node (Eqs. 4, 6, 7); S: streaming with
// half-way bounce-back at resting walls, n(x, i) <- n*(x - c_i, i) when
// x - c_i is fluid, else n*(x, opp(i)) (Eqs. 5, 14 with V_b = 0; populations
// from outside the x range reflect the same way); B: the pressure inlet
// (Zou-He, Section 2.4, density rho_f + rho' shape(t+1)) and the outlet.
// For L = sum_t l_t(n_t) the adjoint a_t = dL/dn_t obeys
//     a_t = dl_t/dn_t + J_C(n_t)^T S^T B_{t+1}^T a_{t+1},   a_T = 0,
// and dL/domega = -sum_t (S^T B^T a_{t+1}) . (n_t - n^eq(n_t)) with
// omega = 1/tau, dL/drho' = sum_t (dB_{t+1}/drho_in)^T a_{t+1} shape(t+1).
//   * S^T: s(y, j) = b(y + c_j, j) when y + c_j is fluid, else b(y, opp(j));
//   * J_C^T: n* = (1 - omega) n + omega n^eq(rho, J) with rho = sum n,
//     J = sum c n, so (J_C^T s)_j = (1 - omega) s_j + omega (A + B . c_j),
//     A = sum_i s_i dn^eq_i/drho, B = sum_i s_i dn^eq_i/dJ;
//   * B^T at an inlet node moves the adjoint of the five unknowns onto the
//     knowns through the transposed Zou-He formulas; at a zero-gradient
//     outlet it adds the unknowns' adjoint to the upstream node.
// Populations are deviations g = n - w rho_f throughout (the derivatives are
// the same).  The forward states come from the product path itself: its
// collide kernels write out the natural populations they read.
#include "common.cuh"
#include "kernels.cuh"

namespace lbmdem {

// B^T in place on the adjoint of n_{t+1}: one thread per boundary node pair
// (inlet node of a (y, z) line, outlet node and its upstream node).
__global__ void k_adj_boundary(AdjArgs A, double shape, double* d_amp) {
    const Lat& L = A.L;
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    double da = 0.0;
    if (k < L.ny * L.nz) {
        int y = k / L.nz, z = k - (k / L.nz) * L.nz;
        float* a = A.adj;
        size_t P = L.nSpad;
        bool fl;
        if (A.inlet == 0) {
            uint32_t i = stored_index(L, 0, y, z, fl);
            if (fl && i != NONE) da = (double)adj_face<0>(a + i, P) * shape;
        }
        if (A.outlet == 0 || A.outlet == 1) {
            uint32_t o = stored_index(L, L.nx - 1, y, z, fl);
            if (fl && o != NONE) {
                if (A.outlet == 0) {  // zero gradient: unknowns copied from upstream
                    bool ufl;
                    uint32_t u = stored_index(L, L.nx - 2, y, z, ufl);
                    if (ufl && u != NONE) {
                        adj_copy(a, P, u, o);
                    }
                } else {  // pressure face at rho_f: the mirrored transpose
                    adj_face<1>(a + o, P);
                }
            }
        }
    }
    // block sum of the amplitude derivative, one FP64 atomic per warp
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int o = 16; o; o >>= 1) da += __shfl_xor_sync(full, da, o);
    if ((threadIdx.x & 31) == 0 && da != 0.0) atomicAdd(d_amp, da);
}

void launch_adj_boundary(const AdjArgs& A, double shape, double* d_amp, cudaStream_t s) {
    int n = A.L.ny * A.L.nz;
    if (A.L.px) return;
    k_adj_boundary<<<(n + 127) / 128, 128, 0, s>>>(A, shape, d_amp);
}

// a_t = J_C(n_t)^T S^T b + dl_t/dn_t, and the omega derivative.  240 B per node,
// 18.4 us at the copy rate on 0.52 M fluid nodes; the neighbours from word
// records and link words, as in the odd collide kernel: 25.2 us against 33.4 us
// with a table of 18 indices per node.
__global__ void __launch_bounds__(256) k_adj_step(AdjArgs A, const float* nat, float* out, float dl,
                                                  double* d_omega) {
    const Lat& L = A.L;
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    float dw = 0.f;
    if (i < L.nS) {
        // fluid: a packing of fixed spheres stores no other node
        const size_t P = L.nSpad;
        float g[Q];
#pragma unroll
        for (int m = 0; m < Q; ++m) g[m] = __ldcs(nat + (size_t)m * P + i);
        float s[Q];
        int x, y, z;
        unpack_coord(__ldg(&L.coord[i]), x, y, z);
        uint32_t wall = __ldg(&A.lw[i].x) & LW_MASK;
        for_neighbours(L, x, y, z, wall, [&](int j, uint32_t n) {
            s[j] = (wall >> j) & 1u ? A.adj[(size_t)opp(j) * P + i] : A.adj[(size_t)j * P + n];
        });
        s[18] = A.adj[(size_t)18 * P + i];
        const RevMoments M = rev_moments(g, L.rho_f);
        RevSums R;
        float sw = s[18] * (g[18] - wt(18) * (M.drho - M.rho * M.uu15));
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int m = pair_m(k), o = opp(m);
            float cu, em, eo;
            rev_eq(M, m, cu, em, eo);
            sw += s[m] * (g[m] - em) + s[o] * (g[o] - eo);
            R.add(m, cu, s[m] + s[o], s[m] - s[o]);
        }
        R.finish(M, s[18]);
        const float om = L.tau_inv;
        const float add = x == A.probe_x ? dl : 0.f;
#pragma unroll
        for (int j = 0; j < Q; ++j)
            out[(size_t)j * P + i] = (1.0f - om) * s[j] + om * (R.A + R.dot(j)) + add;
        dw = -sw;
    }
    block_sum_to(dw, d_omega + blockIdx.x % GRAD_COPIES);
}

void launch_adj_step(const AdjArgs& A, const float* nat, float* out, float dl, double* d_omega, cudaStream_t s) {
    if (A.L.nS) k_adj_step<<<(A.L.nS + 255) / 256, 256, 0, s>>>(A, nat, out, dl, d_omega);
}

}  // namespace lbmdem
