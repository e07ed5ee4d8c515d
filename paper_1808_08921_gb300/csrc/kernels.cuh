// kernels.cuh -- launch interfaces between the host orchestration (api.cu)
// and the kernel translation units.
#pragma once

#include "common.cuh"

namespace lbmdem {

// Fused monitors of the collide kernels.
struct Mon {
    double* acc;                    // [5] sum drho, sum j, fluid count (FP64)
    uint32_t* umax_bits;            // max |u|^2 as float bits
    uint32_t* status;
    double* probe_sum;              // [2 * capacity] (sum drho, count) per step, or null
    const unsigned long long* t_dev;
    uint32_t p0, p1;                // compact index range of the probe plane
};

struct Source {
    int waveform;
    double amp, omega, t0;
    long long t_n;
};

struct BC {
    int inlet, outlet;
    Source src;
    const unsigned long long* t_dev;
};

// Eq. 25 and Table 2 at time t (steps completed), in FP64 (evaluated once
// per block).
__device__ __forceinline__ double source_drho(const Source& S, unsigned long long t) {
    if (S.t_n >= 0 && (long long)t > S.t_n) return 0.0;
    double ph = S.omega * (double)t;
    switch (S.waveform) {
        case 0: return S.amp * sin(ph);
        case 1: return S.amp * (1.0 - cos(ph));
        case 2: return S.amp;
        case 3: {
            double a = 0.5 * S.omega * ((double)t - S.t0);  // pi f (t - t0), f = omega / 2 pi
            return S.amp * (1.0 - 2.0 * a * a) * exp(-a * a);
        }
    }
    return 0.0;
}

// Section 2.4, x-normal D3Q19 pressure face on deviations.  side 0: inlet
// (unknown c_x = +1), side 1: outlet (unknown c_x = -1).  Indices are the
// paper's d (1-based) minus one.
__device__ __forceinline__ void pressure_face(float g[Q], float drho_b, int side) {
    float rest = g[18] + g[2] + g[3] + g[4] + g[5] + g[14] + g[15] + g[16] + g[17];
    float Ny = 0.5f * (g[2] + g[14] + g[15] - g[3] - g[16] - g[17]);
    float Nz = 0.5f * (g[4] + g[14] + g[16] - g[5] - g[15] - g[17]);
    if (side == 0) {
        float rux = drho_b - (rest + 2.f * (g[1] + g[10] + g[11] + g[12] + g[13]));
        g[0] = g[1] + rux * (1.f / 3.f);
        g[6] = g[11] + rux * (1.f / 6.f) - Ny;
        g[7] = g[10] + rux * (1.f / 6.f) + Ny;
        g[8] = g[13] + rux * (1.f / 6.f) - Nz;
        g[9] = g[12] + rux * (1.f / 6.f) + Nz;
    } else {
        float rux = (rest + 2.f * (g[0] + g[6] + g[7] + g[8] + g[9])) - drho_b;
        g[1] = g[0] - rux * (1.f / 3.f);
        g[11] = g[6] - rux * (1.f / 6.f) + Ny;
        g[10] = g[7] - rux * (1.f / 6.f) - Ny;
        g[13] = g[8] - rux * (1.f / 6.f) + Nz;
        g[12] = g[9] - rux * (1.f / 6.f) - Nz;
    }
}

// Link word of a stored node (one 8-byte word per node), for the odd collide
// kernel's fluid neighbours (.x) and the links taken inside the collide
// kernels:
//   .x = link mask (bit m, m < 18: the neighbour x + c_m is solid) | sphere A << 18
//   .y = B mask (bit m: that link's neighbour belongs to sphere B) | sphere B << 18
// Sphere indices take 14 bits; LW_NONE stands for no sphere B, and as sphere
// A for a node whose solid neighbours belong to more than two spheres (its
// links then read the owner map).  With more spheres than LW_MAX_SPHERES the
// indices are cut off and only the mask is used.  Built at the layout from the
// owner map and renewed for every converted node and its 18 neighbours.
constexpr uint32_t LW_MASK = (1u << 18) - 1u;
constexpr uint32_t LW_NONE = 0x3fffu;
constexpr int LW_MAX_SPHERES = (int)LW_NONE;  // sphere indices 0 .. LW_NONE - 1

// Compact indices of the stored nodes at z, z + 1 and z - 1 of one z-line
// from one population count: b = z & 31, low the bits below it; the word's
// prev and next serve the line's neighbours outside the word.
struct LineIndex {
    uint32_t c, p, m;
    __device__ __forceinline__ LineIndex(const uint4& r, uint32_t b, uint32_t low, bool top) {
        c = r.y + __popc(r.x & low);
        p = top ? r.w : c + ((r.x >> b) & 1u);
        m = b == 0u ? r.z : c - ((r.x >> ((b - 1u) & 31u)) & 1u);
    }
};

// take(m, n) for the 18 neighbours x + c_m, n the compact index where the
// neighbour is stored (any value where it is not), from nine word records;
// the directions that leave the x range join `wall` before the first call.
template <class Take>
__device__ __forceinline__ void for_neighbours(const Lat& L, int x, int y, int z, uint32_t& wall, Take take) {
    const uint32_t b = z & 31, low = (1u << b) - 1u;
    const bool top = b == 31u || z == L.nz - 1;
    const int ym = y == 0 ? L.ny - 1 : y - 1, yp = y == L.ny - 1 ? 0 : y + 1;
    int xm = x - 1, xp = x + 1;
    if (x == 0) {
        xm = L.px ? L.nx - 1 : 0;
        if (!L.px) wall |= 1u << 1 | 1u << 10 | 1u << 11 | 1u << 12 | 1u << 13;  // c_x = -1
    }
    if (x == L.nx - 1) {
        xp = L.px ? 0 : x;
        if (!L.px) wall |= 1u << 0 | 1u << 6 | 1u << 7 | 1u << 8 | 1u << 9;  // c_x = +1
    }
    const uint32_t nyw = (uint32_t)L.nw * L.ny, wz = (uint32_t)(z >> 5) * L.ny;
    const uint4 *r0 = L.rec + (size_t)x * nyw + wz, *rm = L.rec + (size_t)xm * nyw + wz,
                *rp = L.rec + (size_t)xp * nyw + wz;
    {
        const LineIndex l(__ldg(r0 + y), b, low, top);
        take(4, l.p);
        take(5, l.m);
    }
    {
        const LineIndex l(__ldg(r0 + yp), b, low, top);
        take(2, l.c);
        take(14, l.p);
        take(15, l.m);
    }
    {
        const LineIndex l(__ldg(r0 + ym), b, low, top);
        take(3, l.c);
        take(16, l.p);
        take(17, l.m);
    }
    {
        const LineIndex l(__ldg(rp + y), b, low, top);
        take(0, l.c);
        take(8, l.p);
        take(9, l.m);
    }
    {
        const LineIndex l(__ldg(rm + y), b, low, top);
        take(1, l.c);
        take(12, l.p);
        take(13, l.m);
    }
    auto one = [&](const uint4* r) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(r));
        return v.y + __popc(v.x & low);
    };
    take(6, one(rp + yp));
    take(7, one(rp + ym));
    take(10, one(rm + yp));
    take(11, one(rm + ym));
}

// The inlet / outlet of the step that ended, one thread per boundary node:
// k < ny nz the inlet plane, then the outlet plane.  Where the populations it
// reads are stored follows from the stored words, fixed since the layout, and
// from the link words, which change only after every block of the band kernel
// has ended: boundary blocks inside that kernel work by the map before its
// conversions, and find the places before they wait for the previous kernel.
template <bool AFTER_EVEN, int ST>
struct BoundaryNode {
    uint32_t i;       // the node, NONE: nothing to do
    int side;         // 0 inlet, 1 outlet
    uint32_t src[Q];  // offsets of the populations read
    uint32_t P;       // stride of a population

    // natural population m of fluid node (x, y, z) = n with solid neighbours s;
    // o: the direction against m, to the node (x, y, z) + d it comes from
    __device__ __forceinline__ uint32_t place(const Lat& L, int x, int y, int z, uint32_t n, uint32_t s, int m, int o,
                                              int dx, int dy, int dz) const {
        const uint32_t own = (uint32_t)m * P + n;
        if (!AFTER_EVEN) return own;
        const int xs = x + dx, ys = wrap1(y + dy, L.ny), zs = wrap1(z + dz, L.nz);
        const bool in = xs >= 0 && xs < L.nx;
        const uint4 r = __ldg(&L.rec[word_of(L, in ? xs : x, ys, zs)]);
        return !in || ((s >> o) & 1u) ? own : (uint32_t)o * P + rec_index(r, 1u << (zs & 31));
    }

    __device__ __forceinline__ BoundaryNode(const Lat& L, const BC& bc, const uint2* lw, int k) : i(NONE), P(L.nSpad) {
        const int plane = L.ny * L.nz;
        side = k >= plane;
        if (k >= 2 * plane || (side == 0 && bc.inlet != 0) || (side == 1 && bc.outlet > 1)) return;
        const int yz = side ? k - plane : k, y = yz / L.nz, z = yz - y * L.nz, x = side ? L.nx - 1 : 0;
        // the boundary planes are never solid
        const uint32_t bit = 1u << (z & 31), n = rec_index(L.rec[word_of(L, x, y, z)], bit);
        const uint32_t s = lw[n].x;
        if (side == 1 && bc.outlet == 0) {  // zero gradient: the neighbour's, if it is fluid
            if (x == 0 || (s >> 1) & 1u) return;
            const uint32_t u = rec_index(L.rec[word_of(L, x - 1, y, z)], bit), su = lw[u].x;
#pragma unroll
            for (int m = 0; m < Q; ++m)
                if (cx(m) < 0) src[m] = place(L, x - 1, y, z, u, su, m, opp(m), -cx(m), -cy(m), -cz(m));
        } else {
#pragma unroll
            for (int m = 0; m < Q - 1; ++m) {  // m at the outlet (cx >= 0), the opposite at the inlet
                const int a = side ? -1 : 1;
                if (cx(m) >= 0)
                    src[m] = place(L, x, y, z, n, s, side ? m : opp(m), side ? opp(m) : m, a * cx(m), a * cy(m), a * cz(m));
            }
            src[18] = 18u * P + n;
        }
        i = n;
    }

    // drho: the source's density deviation at the new time
    __device__ __forceinline__ void apply(const Lat& L, const BC& bc, float drho) const {
        if (i == NONE) return;
        auto* f = pops<ST>(L);
        if (side == 1 && bc.outlet == 0) {
#pragma unroll
            for (int m = 0; m < Q; ++m)
                if (cx(m) < 0) f[(size_t)m * P + i] = f[src[m]];
            return;
        }
        // the two faces apart: with the face as a value the compiler contracts
        // the formulas differently and FP16 populations round differently
        float g[Q];
        if (side == 0) {
#pragma unroll
            for (int m = 0; m < Q - 1; ++m)
                if (cx(m) >= 0) g[opp(m)] = to_f<ST>(f[src[m]], L.fsi);
            g[18] = to_f<ST>(f[src[18]], L.fsi);
            pressure_face(g, drho, 0);
#pragma unroll
            for (int m = 0; m < Q; ++m)
                if (cx(m) > 0) f[(size_t)m * P + i] = from_f<ST>(g[m], L.fs);  // source outside: own slot
        } else {
#pragma unroll
            for (int m = 0; m < Q - 1; ++m)
                if (cx(m) >= 0) g[m] = to_f<ST>(f[src[m]], L.fsi);
            g[18] = to_f<ST>(f[src[18]], L.fsi);
            pressure_face(g, 0.f, 1);
#pragma unroll
            for (int m = 0; m < Q; ++m)
                if (cx(m) < 0) f[(size_t)m * P + i] = from_f<ST>(g[m], L.fs);
        }
    }
};

// Link lists for the link kernel.  Links are grouped by (sphere, direction
// m, maybe), each group padded to whole chunks of 32 records, and each
// sphere's groups together padded to whole LINK_WARP records, so a warp
// walks LINK_WARP / 32 chunks of one sphere, each chunk in one direction
// (one record per lane and chunk) and either without or with only `maybe`
// links:
//   warp_p[w]    = sphere index
//   chunk_dir[c] = direction m of chunk c (the solid neighbour is x + c_m),
//                  | 64 for a chunk of `maybe` links, | 128 when the chunk
//                  holds an `in_band` link; warp w owns chunks
//                  w LINK_CHUNKS ... (w + 1) LINK_CHUNKS - 1
//   link[r]      = {cidx of the fluid node x,
//                   (x - org) + 128 packed 8 bits per axis | maybe << 24 |
//                   shared << 25 | in_band << 26}
// `maybe` marks a neighbour inside a band: whether the sphere owns it now
// is decided by the map update's FP32 test (same operands and rounding),
// or by reading the owner map near the FP32 margin or when the band node
// has several candidate spheres (`shared`).  `in_band` marks a fluid node x
// that may itself be covered before the next re-layout (its fluid bit is
// read); every other link node stays fluid.  cidx == NONE pads.
constexpr int LINK_WARP = 256;
constexpr int LINK_CHUNKS = LINK_WARP / 32;  // chunks per warp
constexpr int LINK_GROUPS = 2 * (Q - 1);     // groups per sphere: (direction m, maybe) -> 2 m + maybe
static_assert(LINK_CHUNKS == 4 || LINK_CHUNKS == 8, "4 or 8 chunk directions per warp");

struct LinkLists {
    const uint2* link;
    const uint32_t* warp_p;
    const uint8_t* chunk_dir;  // LINK_CHUNKS bytes per warp
    uint32_t nwarps;
};

// Nodes whose solid/fluid status can change before the next re-layout.
struct Band {
    const uint32_t* coord;  // packed x, y, z
    const int4* cand;       // up to 4 sphere indices, ascending, -1 padded
    const float* slack;     // distance to the nearest candidate surface at the layout (0: always re-test)
    uint32_t n;
};

struct Flip {
    uint32_t coord;
    int32_t old_owner, new_owner;
    uint32_t pad;
};

struct FlipBuf {
    Flip* rec;        // [2][cap] by step parity
    float* scratch;   // [cap][19][19]
    uint8_t* valid;   // [cap][19]
    uint32_t cap;
};

// CTAs of the largest cluster the one-launch DEM takes.
constexpr int DEM_MAX_CTAS = 16;

// Launch of the one-launch DEM: CTAs of its cluster (0: a launch per substep
// serves instead) and threads per CTA.  Chosen once for a packing: the exchange
// slots are laid out for it.
struct DemShape {
    int ctas = 0, threads = 0;
};

// DEM state (Section 2.2).
struct Dem {
    int n, K;
    DemShape shape;
    float dt;                // 1 / K
    float kn, kt, mu;        // Eqs. 11-12 prefactors
    float3 g;                // body force
    int nbmax;
    // per particle
    const double* Xref;
    float4* dX;              // canonical displacement since re-layout
    float4* dXc;             // Kahan compensation
    // records of the launches per substep, [2][n] by substep parity:
    // {dX, Vh.x}, {Vh.yz, Wh.xy}, {Wh.z}
    float4* dXb;
    float4* V;
    float4* W;
    float4* q;
    float4* Vhb;
    float4* Whb;
    float4* Fc;              // contact force (persistent across steps)
    float4* Tc;
    const double* Fh;        // hydrodynamic force/torque sums of this step (Eqs. 18-19)
    const double* Th;
    double* Fh_prev;         // the sums of the previous step
    double* Th_prev;
    float4* Fa;              // applied: mean of this and the previous step (launches per
    float4* Ta;              // substep only: one launch keeps it in registers)
    const float* R;
    const float* invm;
    const float* invI;
    const uint8_t* fixed;
    // neighbour list
    const int* nb_cnt;
    const int* nb_j;
    const float4* nb_dref;   // xyz: X_ref_j + shift - X_ref_i, w: (R_i+R_j)^2 - |xyz|^2
    float4* nb_ft;           // tangential history (force on i)
    const float* nb_R;       // radius of j
    // one-launch form: slots of the exchange (k_dem_ghosts)
    const int* nb_slot;      // [n * nbmax] slot of the neighbour in the sphere's CTA
    const uint16_t* push;    // [n][DEM_MAX_CTAS] slot of the sphere in each CTA, 0xffff where it has none
    const int* foreign;      // [DEM_MAX_CTAS] spheres of other CTAs a CTA holds
    int slots;               // slots per CTA and record buffer
    // outputs for the lattice kernels
    int4* org;
    int4* orgw;
    float4* xf;
    uint32_t* status;
    uint32_t* max_disp_bits;
    uint32_t* disp_layout_bits;
    uint32_t* layout_fresh;
    uint32_t* max_vel_bits;
    float hard_disp;             // displacement at which the layout is invalid
    int px;
    int dry;                 // the fluid is off: DEM steps follow one another directly
    double Lx, Ly, Lz;
};

// lattice.cu
void launch_collide(const Lat& L, const Mon& mon, bool odd, bool monitor, const uint2* lw, float* snap, int tile,
                    cudaStream_t s);
void launch_collide_links(const Lat& L, const Mon& mon, const PartView& P, bool odd, bool monitor, bool few,
                          const uint2* lw, int tile, cudaStream_t s);
void launch_inlet_outlet(const Lat& L, const BC& bc, const uint2* lw, bool after_even, cudaStream_t s);
void launch_plane_sums(const Lat& L, bool after_even, double* out, cudaStream_t s);
void launch_read_fields(const Lat& L, bool after_even, double* rho, double* u, uint8_t* solid,
                        cudaStream_t s);

// coupling.cu
void launch_links(const Lat& L, const PartView& P, const LinkLists& B, cudaStream_t s);
// inlet: null, or the boundary of the previous step, applied on the way;
// early: the previous step's last kernel is the only predecessor on the stream
void launch_map_update(const Lat& L, const PartView& P, const Band& band, const FlipBuf& F,
                       DevStats* st, int step_parity, uint2* lw, const BC* inlet, bool early, bool shared_gpu,
                       cudaStream_t s);
int map_update_launches(uint32_t nband, int step_parity);
void launch_link_words(const Lat& L, uint2* lw, cudaStream_t s);

// dem.cu
void launch_dem_ghosts(const Dem& D, int* nb_slot, uint16_t* push, int* foreign, int* slots, cudaStream_t s);
void launch_dem_init(const Dem& D, cudaStream_t s);
void launch_dem_step(const Dem& D, cudaStream_t s);
DemShape dem_shape(int n);              // for n spheres on the current device
int dem_launches(DemShape h, int K);  // kernels of one launch_dem_step
// adjoint.cu: reverse-mode kernels of the lattice step for a fixed packing
struct AdjArgs {
    Lat L;
    const uint2* lw;  // link words (a fixed packing's never change)
    float* adj;           // [19][nSpad] adjoint of the natural populations
    int inlet, outlet, probe_x;
};
void launch_adj_boundary(const AdjArgs& A, double shape, double* d_amp, cudaStream_t s);
void launch_adj_step(const AdjArgs& A, const float* nat, float* out, float dl, double* d_omega, cudaStream_t s);

// Parameter derivatives of the reverse kernels: each block sums its
// threads' FP32 terms in FP64 and adds the sum to one of GRAD_COPIES FP64
// accumulators (blockIdx % GRAD_COPIES: no long queue of atomics on one
// address); the host adds the copies.  FP64 adds run at 2 lanes per clock and
// SM here, so the terms go through shared memory to one warp, which adds
// blockDim / 32 of them per lane before its five shuffle steps (a tree in
// every warp spends five warp-wide adds on 32 terms).
constexpr int GRAD_COPIES = 64;
constexpr int GRAD_THREADS = 256;  // largest block
__device__ __forceinline__ void block_sum_to(float v, double* dst) {
    __shared__ float part[GRAD_THREADS];
    const unsigned tid = threadIdx.x + blockDim.x * threadIdx.y, nt = blockDim.x * blockDim.y;
    part[tid] = v;
    __syncthreads();
    if (tid < 32) {
        double s = 0.0;
        for (unsigned k = tid; k < nt; k += 32) s += (double)part[k];
#pragma unroll
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (tid == 0 && s != 0.0) atomicAdd(dst, s);
    }
}

// The collision's transpose, pair by pair.  Opposite directions share |c.u|,
// so the equilibria of a pair are an even part plus or minus an odd one, and
// the contractions A = sum_i v_i dn^eq_i/drho and B = sum_i v_i dn^eq_i/dJ
// (dn^eq/dJ = w (3 c + 9 (c.u) c - 3 u)) need only the pair's sum p and
// difference q of v: half the arithmetic of direction-by-direction sums.
struct RevMoments {
    float drho, rho, ux, uy, uz, uu15;
};
__device__ __forceinline__ RevMoments rev_moments(const float g[Q], float rho_f) {
    float drho = 0.f, jx = 0.f, jy = 0.f, jz = 0.f;
#pragma unroll
    for (int m = 0; m < Q; ++m) {
        drho += g[m];
        jx += cx(m) * g[m];
        jy += cy(m) * g[m];
        jz += cz(m) * g[m];
    }
    RevMoments M;
    M.drho = drho;
    M.rho = rho_f + drho;
    const float ir = 1.0f / M.rho;
    M.ux = jx * ir;
    M.uy = jy * ir;
    M.uz = jz * ir;
    M.uu15 = 1.5f * (M.ux * M.ux + M.uy * M.uy + M.uz * M.uz);
    return M;
}
// c.u of direction m and the equilibrium deviations of m and opp(m)
__device__ __forceinline__ void rev_eq(const RevMoments& M, int m, float& cu, float& em, float& eo) {
    cu = (float)cx(m) * M.ux + (float)cy(m) * M.uy + (float)cz(m) * M.uz;
    const float even = M.drho + M.rho * (4.5f * cu * cu - M.uu15), odd = 3.0f * M.rho * cu;
    em = wt(m) * (even + odd);
    eo = wt(m) * (even - odd);
}
// Sums with the integer weights 36 w (1, 2, 12), scaled by 1/36 at the end:
// the FP32 weights add up to 1 + 1.5e-8, a bias that a recursion of hundreds
// of steps turns into 1e-6 of the gradient; scaled() is unbiased.
struct RevSums {
    float A = 0.f, Bx = 0.f, By = 0.f, Bz = 0.f;
    float s = 0.f, cc = 0.f;
    static __device__ __forceinline__ float iw(int m) {
        return m == 18 ? 12.f : (cx(m) * cx(m) + cy(m) * cy(m) + cz(m) * cz(m)) == 1 ? 2.f : 1.f;
    }
    // x / 36, the product corrected by its exact residual
    static __device__ __forceinline__ float scaled(float x) {
        const float q = x * (1.f / 36.f);
        return fmaf(fmaf(-36.f, q, x), 1.f / 36.f, q);
    }
    // the pair (m, opp(m)): p = v_m + v_opp, q = v_m - v_opp
    __device__ __forceinline__ void add(int m, float cu, float p, float q) {
        const float wp = iw(m) * p, t = 9.0f * cu * wp + (3.0f * iw(m)) * q;
        s += wp;
        cc += cu * cu * wp;
        Bx += cx(m) * t;
        By += cy(m) * t;
        Bz += cz(m) * t;
    }
    __device__ __forceinline__ void finish(const RevMoments& M, float v18) {
        s += 12.f * v18;
        A = scaled(s * (1.0f + M.uu15) - 4.5f * cc);
        Bx = scaled(Bx - 3.0f * M.ux * s);
        By = scaled(By - 3.0f * M.uy * s);
        Bz = scaled(Bz - 3.0f * M.uz * s);
    }
    __device__ __forceinline__ float dot(int m) const { return Bx * cx(m) + By * cy(m) + Bz * cz(m); }
};

// Transposed pressure face (Section 2.4) on the adjoint of one boundary node,
// element m at a[m P]: the adjoint of the five unknowns moves onto the knowns
// (the forward formulas are linear in the knowns and in the boundary
// density), the unknowns' adjoint becomes zero.  Side 0: inlet, 1: outlet.
// Returns the derivative in the boundary density.  Every load is issued
// before the first store: written as read-modify-writes the compiler has to
// keep their order (the 19 planes may alias), and the kernel waited for 14
// loads one after another (10.6 -> 4.0 us per launch at 64 x 64 lines).
template <int SIDE>
__device__ __forceinline__ float adj_face(float* a, size_t P) {
    float v[Q];
#pragma unroll
    for (int m = 0; m < Q; ++m) v[m] = a[m * P];
    // the unknowns 0, 6, 7, 8, 9 of the inlet are the knowns of the outlet
    // and the other way round: pairs (unknown, known) share their index pair
    constexpr int in[5] = {0, 6, 7, 8, 9}, out[5] = {1, 11, 10, 13, 12};
    float ar, ay, az, two;
    if (SIDE == 0) {
        ar = v[0] * (1.f / 3.f) + (v[6] + v[7] + v[8] + v[9]) * (1.f / 6.f);
        ay = 0.5f * (v[7] - v[6]);
        az = 0.5f * (v[9] - v[8]);
        two = -2.f * ar;
    } else {
        // forward: rux = rest + 2 (g0 + g6 + g7 + g8 + g9) - drho_b;
        // g1 = g0 - rux/3, g11 = g6 - rux/6 + Ny, g10 = g7 - rux/6 - Ny,
        // g13 = g8 - rux/6 + Nz, g12 = g9 - rux/6 - Nz
        ar = -(v[1] * (1.f / 3.f) + (v[11] + v[10] + v[13] + v[12]) * (1.f / 6.f));
        ay = 0.5f * (v[11] - v[10]);
        az = 0.5f * (v[13] - v[12]);
        two = 2.f * ar;
    }
    const float rest = SIDE == 0 ? -ar : ar;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const int u = SIDE == 0 ? in[k] : out[k], w = SIDE == 0 ? out[k] : in[k];
        a[w * P] = v[w] + (v[u] + two);
        a[u * P] = 0.f;
    }
    a[18 * P] = v[18] + rest;
    a[2 * P] = v[2] + (rest + ay);
    a[3 * P] = v[3] + (rest - ay);
    a[4 * P] = v[4] + (rest + az);
    a[5 * P] = v[5] + (rest - az);
    a[14 * P] = v[14] + (rest + ay + az);
    a[15 * P] = v[15] + (rest + ay - az);
    a[16 * P] = v[16] + (rest - ay + az);
    a[17 * P] = v[17] + (rest - ay - az);
    return ar;
}

// Transposed zero-gradient outlet: the unknowns' adjoint of outlet node o
// goes to the upstream node u.
__device__ __forceinline__ void adj_copy(float* a, size_t P, size_t u, size_t o) {
    constexpr int um[5] = {1, 10, 11, 12, 13};
    float s[5], t[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        s[q] = a[um[q] * P + o];
        t[q] = a[um[q] * P + u];
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        a[um[q] * P + u] = t[q] + s[q];
        a[um[q] * P + o] = 0.f;
    }
}

// psm.cu: the smooth surrogate of the coupling (dense lattice) and its reverse
struct PsmArgs {
    int nx, ny, nz, px, inlet, outlet, probe_x;
    float rho_f, tau;
    size_t N;  // nodes
};
void launch_psm_eps(const PsmArgs& A, const double* X, const double* R, int n, float* eps, cudaStream_t s);
void launch_psm_step(const PsmArgs& A, const float* gin, float* gout, const float* eps, cudaStream_t s);
void launch_psm_boundary(const PsmArgs& A, float* g, const Source& src, unsigned long long t1, cudaStream_t s);
void launch_psm_probe(const PsmArgs& A, const float* g, double* out, cudaStream_t s);
void launch_psm_adj_boundary(const PsmArgs& A, float* lam, double shape, double* d_amp, cudaStream_t s);
void launch_psm_adj_step(const PsmArgs& A, const float* lin, const float* gt, float* lout, const float* eps, float dl,
                         double* d_tau, double* G, cudaStream_t s);
void launch_psm_grad_x(const PsmArgs& A, const double* G, const float* eps, const double* X, const double* R, int n,
                       double* dX, cudaStream_t s);
}  // namespace lbmdem
