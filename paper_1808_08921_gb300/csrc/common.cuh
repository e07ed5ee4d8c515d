// common.cuh -- lattice constants and the device-side views of the state.
//
// Compact lattice (the fluid is ~25% of the nodes in the FCC media, so a dense
// lattice that skips solids would still move ~2x the fluid bytes through
// partially used 32-byte sectors):
//   * S  = stored nodes = every node that is fluid now or within `skin` of a
//          sphere surface on the solid side (it may become fluid before the
//          next re-layout; in a packing of fixed spheres none does, and
//          only the fluid nodes are stored).  Order: x, then 32-node words along z, then y, then
//          z inside the word: a warp's 32 consecutive nodes come from a few
//          neighbouring lines of one word (about 4 x 32 lattice nodes at 25%
//          fluid), and the nodes of the neighbouring lines in x and y are as
//          contiguous as its own.
//   * f  = populations as deviations g_i = f_i - w_i rho_f, structure of
//          arrays [19][nSpad], in place with the AA access pattern; stored as
//          FP32, or as BF16 / FP16 scaled by a power of two (FP16: 2^12, so
//          that deviations of 1e-8 .. 16 stay normal numbers), always
//          collided in FP32.
//   * rec[w] = {stored bits, base, prev, next} for every 32-node word of a
//          z-line (fixed until the next re-layout): a stored node's compact
//          index is base + popc(stored bits & lower bits); prev and next are
//          the indices of the nodes before the word's first and after its
//          last one (periodic in z), so that z +- 1 needs no other record.
//          fluid[w] holds the fluid-now bits.  The word tables (20 B per 32
//          nodes) stay resident in L2.
//   * coord[i] = x << 20 | y << 10 | z of compact node i.
//   * fbits[i / 32] = fluid-now bit of compact node i.
//   * owner[lattice index] = index of the sphere a node belongs to, or FLUID.
//
// AA pattern, with fluid-solid links handled in place (Section 2.3):
//   even step: node x reads slot m of itself, writes post-collision value of
//              direction m into slot opp(m) of itself;
//   odd step:  node x reads direction m from slot opp(m) of x - c_m when that
//              node is fluid, else from slot m of x itself; it writes
//              direction m into slot m of x + c_m when fluid, else into slot
//              opp(m) of x itself.
//   After either step, slot opp(d) of a fluid node x whose neighbour x + c_d
//   is solid holds the post-collision value of direction d; the link kernel
//   turns it into the bounced value (Eq. 14) in place.  Populations arriving
//   from outside the x range are treated the same way (resting wall) before
//   the inlet/outlet overwrite them.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace lbmdem {

constexpr int Q = 19;
constexpr int32_t OWNER_FLUID = 0x7fffffff;
constexpr uint32_t NONE = 0xffffffffu;

// D3Q19 velocities in the column order of Eq. 3 (index m = d - 1).
__host__ __device__ constexpr int cx(int m) {
    return (m == 0 || m == 6 || m == 7 || m == 8 || m == 9) ? 1
           : (m == 1 || m == 10 || m == 11 || m == 12 || m == 13) ? -1
                                                                  : 0;
}
__host__ __device__ constexpr int cy(int m) {
    return (m == 2 || m == 6 || m == 10 || m == 14 || m == 15) ? 1
           : (m == 3 || m == 7 || m == 11 || m == 16 || m == 17) ? -1
                                                                 : 0;
}
__host__ __device__ constexpr int cz(int m) {
    return (m == 4 || m == 8 || m == 12 || m == 14 || m == 16) ? 1
           : (m == 5 || m == 9 || m == 13 || m == 15 || m == 17) ? -1
                                                                 : 0;
}
// Eq. 8 weights by speed class.
__host__ __device__ constexpr float wt(int m) {
    return (cx(m) * cx(m) + cy(m) * cy(m) + cz(m) * cz(m)) == 0 ? 1.0f / 3.0f
           : (cx(m) * cx(m) + cy(m) * cy(m) + cz(m) * cz(m)) == 1 ? 1.0f / 18.0f
                                                                  : 1.0f / 36.0f;
}
// Opposite direction: the pairs of Eq. 3 are (0,1) (2,3) (4,5) (6,11) (7,10)
// (8,13) (9,12) (14,17) (15,16) and 18 alone.
__host__ __device__ constexpr int opp(int m) {
    return m == 18 ? 18
           : m < 6 ? (m ^ 1)
           : m == 6 ? 11
           : m == 11 ? 6
           : m == 7 ? 10
           : m == 10 ? 7
           : m == 8 ? 13
           : m == 13 ? 8
           : m == 9 ? 12
           : m == 12 ? 9
           : m == 14 ? 17
           : m == 17 ? 14
           : m == 15 ? 16
                     : 15;
}

// The nine pairs of opposite directions: pair k is (pair_m(k), opp(pair_m(k))).
__host__ __device__ constexpr int pair_m(int k) {
    return k == 0 ? 0 : k == 1 ? 2 : k == 2 ? 4 : k == 3 ? 6 : k == 4 ? 7 : k == 5 ? 8 : k == 6 ? 9 : k == 7 ? 14 : 15;
}

__host__ __device__ inline uint32_t pack_coord(int x, int y, int z) {
    return ((uint32_t)x << 20) | ((uint32_t)y << 10) | (uint32_t)z;
}
__host__ __device__ inline void unpack_coord(uint32_t c, int& x, int& y, int& z) {
    x = (int)(c >> 20);
    y = (int)((c >> 10) & 1023u);
    z = (int)(c & 1023u);
}

// Lattice geometry and the compact-storage views, passed by value.
struct Lat {
    int nx, ny, nz, nw;   // nw = 32-node words per z-line
    int px;               // x periodic
    uint32_t nS, nSpad;
    void* f;              // [19][nSpad] deviations, element type by `st`
    int st;               // storage: 0 FP32, 1 BF16, 2 FP16 (scaled by fs)
    float fs, fsi;        // storage scale and its inverse (powers of two)
    uint4* rec;           // [nx*nw*ny] {stored bits, base, prev, next}
    uint32_t* fluid;      // [nx*nw*ny] fluid-now bits
    uint32_t* flip;       // [2][nx*nw*ny] nodes the map update of a step made fluid or solid, by step parity
    uint32_t* coord;      // [nSpad]
    uint32_t* fbits;      // [nSpad / 32]
    int32_t* owner;       // [nx*ny*nz]
    float tau_inv;
    float rho_f;
};

__device__ __forceinline__ int wrap1(int a, int L) { return a < 0 ? a + L : (a >= L ? a - L : a); }

// minimum image of an offset -L < d < L
__device__ __forceinline__ int imin_small(int d, int L) {
    if (2 * d > L) return d - L;
    if (2 * d < -L) return d + L;
    return d;
}

// Word of node (x, y, z).
__device__ __forceinline__ uint32_t word_of(const Lat& L, int x, int y, int z) {
    return ((uint32_t)x * L.nw + (uint32_t)(z >> 5)) * L.ny + y;
}
__device__ __forceinline__ uint32_t rec_index(const uint4& r, uint32_t bit) { return r.y + __popc(r.x & (bit - 1u)); }

// Compact index of node (x+dx, y+dy, z+dz) if it is fluid now, else NONE.
// dx, dy, dz in {-1, 0, 1}.  Out-of-range x (non-periodic) returns NONE.
__device__ __forceinline__ uint32_t fluid_index(const Lat& L, int x, int y, int z, int dx, int dy,
                                                int dz) {
    int xs = x + dx;
    if (L.px) {
        xs = wrap1(xs, L.nx);
    } else if (xs < 0 || xs >= L.nx) {
        return NONE;
    }
    int ys = wrap1(y + dy, L.ny), zs = wrap1(z + dz, L.nz);
    const uint32_t wi = word_of(L, xs, ys, zs);
    const uint4 r = __ldg(&L.rec[wi]);
    const uint32_t bit = 1u << (zs & 31);
    return __ldg(&L.fluid[wi]) & bit ? rec_index(r, bit) : NONE;
}

// Compact index of a stored node given directly, NONE if it is not stored
// (used outside the hot kernel; reads the fluid bits with a coherent load
// because the map-update kernels modify them).
__device__ __forceinline__ uint32_t stored_index(const Lat& L, int x, int y, int z, bool& fluid) {
    const uint32_t wi = word_of(L, x, y, z);
    const uint4 r = L.rec[wi];
    const uint32_t bit = 1u << (z & 31);
    fluid = (L.fluid[wi] & bit) != 0;
    return r.x & bit ? rec_index(r, bit) : NONE;
}

__device__ __forceinline__ bool fluid_bit(const Lat& L, uint32_t i) {
    return (L.fbits[i >> 5] >> (i & 31)) & 1u;
}

// Population storage types and their FP32 conversions (round to nearest;
// the scale is a power of two, so scaling is exact).
template <int ST> struct PopT;
template <> struct PopT<0> { using T = float; };
template <> struct PopT<1> { using T = __nv_bfloat16; };
template <> struct PopT<2> { using T = __half; };

template <int ST> __device__ __forceinline__ float to_f(typename PopT<ST>::T v, float fsi);
template <> __device__ __forceinline__ float to_f<0>(float v, float) { return v; }
template <> __device__ __forceinline__ float to_f<1>(__nv_bfloat16 v, float fsi) { return __bfloat162float(v) * fsi; }
template <> __device__ __forceinline__ float to_f<2>(__half v, float fsi) { return __half2float(v) * fsi; }

template <int ST> __device__ __forceinline__ typename PopT<ST>::T from_f(float v, float fs);
template <> __device__ __forceinline__ float from_f<0>(float v, float) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<1>(float v, float fs) { return __float2bfloat16_rn(v * fs); }
template <> __device__ __forceinline__ __half from_f<2>(float v, float fs) { return __float2half_rn(v * fs); }

template <int ST> __device__ __forceinline__ typename PopT<ST>::T* pops(const Lat& L) {
    return static_cast<typename PopT<ST>::T*>(L.f);
}

// The map before this step's map update, from the committed map and the
// nodes that update changed (flip: the masks of the step's parity).
__device__ __forceinline__ uint32_t old_fluid_index(const Lat& L, const uint32_t* flip, int x, int y, int z, int dx,
                                                    int dy, int dz) {
    int xs = x + dx;
    if (L.px) {
        xs = wrap1(xs, L.nx);
    } else if (xs < 0 || xs >= L.nx) {
        return NONE;
    }
    int ys = wrap1(y + dy, L.ny), zs = wrap1(z + dz, L.nz);
    const uint32_t wi = word_of(L, xs, ys, zs);
    const uint4 r = L.rec[wi];
    const uint32_t bit = 1u << (zs & 31);
    return (L.fluid[wi] ^ flip[wi]) & bit ? rec_index(r, bit) : NONE;
}

// Location of population m of fluid node (x,y,z) with compact index i, in the
// state between steps.  after_even = true: the state after an even step
// (natural populations sit in the neighbours' reversed slots).
template <int ST>
__device__ __forceinline__ typename PopT<ST>::T* pop_loc(const Lat& L, bool after_even, int x, int y, int z,
                                                         uint32_t i, int m) {
    typename PopT<ST>::T* f = pops<ST>(L);
    if (!after_even || m == 18) return f + (size_t)m * L.nSpad + i;
    uint32_t s = fluid_index(L, x, y, z, -cx(m), -cy(m), -cz(m));
    if (s == NONE) return f + (size_t)m * L.nSpad + i;
    return f + (size_t)opp(m) * L.nSpad + s;
}

// A launch macro M(AFTER_EVEN, ST) for the state of lattice L (variables L and
// after_even in scope).
#define LBMDEM_BY_STATE(M)                    \
    do {                                      \
        if (after_even) {                     \
            if (L.st == 0) M(true, 0);        \
            else if (L.st == 1) M(true, 1);   \
            else M(true, 2);                  \
        } else {                              \
            if (L.st == 0) M(false, 0);       \
            else if (L.st == 1) M(false, 1);  \
            else M(false, 2);                 \
        }                                     \
    } while (0)

// The same by the map before this step's map update.
template <int ST>
__device__ __forceinline__ typename PopT<ST>::T* old_pop_loc(const Lat& L, const uint32_t* flip, bool after_even, int x,
                                                             int y, int z, uint32_t i, int m) {
    typename PopT<ST>::T* f = pops<ST>(L);
    if (!after_even || m == 18) return f + (size_t)m * L.nSpad + i;
    uint32_t s = old_fluid_index(L, flip, x, y, z, -cx(m), -cy(m), -cz(m));
    if (s == NONE) return f + (size_t)m * L.nSpad + i;
    return f + (size_t)opp(m) * L.nSpad + s;
}

// Particles as seen by the lattice kernels (current time level).
struct PartView {
    int n;
    const double* Xref;   // [n][3] reference centres of the current layout
    const float4* dX;     // [n] displacement since re-layout (xyz), w unused
    const float4* dXc;    // [n] Kahan compensation of dX
    const float4* V;      // [n]
    const float4* W;      // [n]
    const float* R;       // [n]
    const double* Rd;     // [n] radii in FP64 for the exact inside test
    const int4* org;      // [n] integer origin floor(Xref)
    const int4* orgw;     // [n] that origin wrapped into the box (periodic axes)
    const float4* xf;     // [n] X(t) - origin, FP32
    float4* ab;           // [n][Q-1] moving-wall terms of the step's links (alpha - xf.beta, beta)
    float4* pk;           // [n][3] sphere packet of the step: {xf, V.x} {V.y, V.z, W.x, W.y}
                          // {W.z, wrapped origin as int bits}
    double* Fh;           // [NREP][n][3] hydrodynamic force accumulators (summed by the DEM)
    double* Th;           // [NREP][n][3] hydrodynamic torque accumulators
};

// The link kernels spread their atomics over NREP copies of each sphere's
// force and torque accumulators (fewer same-address collisions: with one copy
// the even kernel with links takes 279 instead of 183 us on the 128 x 128 x
// 1024 column); the DEM kernel and the read-out sum the copies.
constexpr int NREP = 4;

// Exact "inside" test shared by painting and the map update: |y - X|^2 < R^2
// in FP64 without contraction, X = Xref + dX (+ compensation).
__device__ __forceinline__ double norm2_exact(double ax, double ay, double az) {
    return __dadd_rn(__dadd_rn(__dmul_rn(ax, ax), __dmul_rn(ay, ay)), __dmul_rn(az, az));
}
__device__ __forceinline__ bool inside_exact(double ax, double ay, double az, double R) {
    return norm2_exact(ax, ay, az) < __dmul_rn(R, R);
}

// FP32 |a|^2 with a fixed rounding (no contraction), used identically by the
// map update and the link kernel so that both take the same decisions.
__device__ __forceinline__ float norm2_rn(float ax, float ay, float az) {
    return __fadd_rn(__fadd_rn(__fmul_rn(ax, ax), __fmul_rn(ay, ay)), __fmul_rn(az, az));
}
// the FP32 inside test decides only outside this relative margin of R^2
constexpr float FP32_MARGIN = 1e-5f;

// |y - X|^2 / R^2 with the same operation order and rounding as the test
// above; among the spheres that contain a node, the smallest ratio owns it.
__device__ __forceinline__ double inside_ratio(double ax, double ay, double az, double R) {
    return __ddiv_rn(norm2_exact(ax, ay, az), __dmul_rn(R, R));
}

__device__ __forceinline__ double minimg(double d, double L, int periodic) {
    if (!periodic) return d;
    return d - L * floor(d / L + 0.5);
}

// Device status bits (latched; host maps them to LBMDEM_ERR_*).
enum : uint32_t {
    ST_UNSTABLE = 1u,
    ST_CAPACITY = 2u,
    ST_SKIN = 4u,
    ST_TIMEOUT = 8u,
};

struct DevStats {
    uint32_t status;
    uint32_t nflip[2];    // conversions queued this step (double-buffered by step parity)
    uint32_t max_disp_bits;  // float bits of max |dX| (non-negative)
    uint32_t max_vel_bits;   // float bits of max |V|
    uint32_t disp_layout_bits;  // float bits of max |dX| seen since the layout build
    unsigned long long t;    // steps begun (the map update counts each step first; between
                             // steps it equals the completed steps)
    unsigned long long flips_total;
    double mon[6];           // sum rho, sum rho u, max|u|, step
    uint32_t max_u_bits;
    uint32_t layout_fresh;   // 1 from a layout build until the first step's DEM
    unsigned long long t_end[2];  // by step parity: t at the end of the last such step, the source time of its inlet
};

// Programmatic dependent launch.  The kernels of a step are launched with
// programmatic stream serialization (launch_pdl): such a kernel may be
// scheduled while its predecessor on the stream is still running, and its
// first statement, pdl_wait(), blocks until the predecessor grid has
// completed and its memory operations are visible, so nothing is read or
// written early.  pdl_trigger() in the predecessor lets the successor launch
// once every block of the predecessor has executed it (blocks that exit
// count as triggered), which hides the successor's launch and block
// scheduling behind the predecessor's tail.  Both are no-ops for a kernel
// launched without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// smem: bytes of dynamic shared memory (at most 48 KB)
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_smem(void (*k)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                                   Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*k)(KArgs...), unsigned grid, unsigned block, cudaStream_t s, Args... args) {
    return launch_pdl_smem(k, grid, block, 0, s, args...);
}

}  // namespace lbmdem
