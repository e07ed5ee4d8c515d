// dem.cu -- the solid phase (Section 2.2, Eqs. 9-12).
//
//  * Every LBM step runs the K velocity-Verlet substeps of length 1/K with the
//    hydrodynamic force and torque of the step held fixed: kick + drift of
//    the own sphere, an exchange of positions and half-step velocities, then
//    the contact forces of the own sphere from its neighbour list and the
//    closing kick.  A team of TEAM threads works on each sphere.  The
//    exchanged records are double-buffered by substep parity, so one
//    synchronisation per substep suffices.  Each pair is evaluated by both
//    spheres with mirror-exact arithmetic, so the two forces are exact
//    negatives and no atomics are needed.  The hydrodynamic force and torque
//    that drive a sphere are the mean of the exchange sums of this and the
//    previous LBM step (the half-way bounce-back force alternates from step
//    to step; the two-step mean of Ladd's momentum-exchange method keeps the
//    explicit coupling of light spheres stable).
//  * k_dem_step_dsm: packings of up to 2048 spheres, one launch per LBM step,
//    one thread-block cluster (one CTA for up to 64 spheres), the spheres'
//    state in registers, the exchange in shared memory.
//  * k_dem_begin / k_dem_substep: larger packings, one launch per substep over
//    the whole GPU, the state in global memory.
//  * neighbour lists: uniform cells of size >= 2 R_max + skin over the
//    periodic y, z box; every periodic image is a separate entry (a sphere in
//    a narrow box can touch two images of the same neighbour).  Rebuilt only
//    at re-layouts; the tangential history is carried over by (j, image).
//
// Positions are X = Xref (FP64, fixed between re-layouts) + dX (FP32 with a
// Kahan compensation term), so the substep loop needs no FP64 arithmetic.
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "layout.cuh"
#include "per_device.cuh"

namespace lbmdem {

__device__ __forceinline__ float3 f3(float4 a) { return make_float3(a.x, a.y, a.z); }
__device__ __forceinline__ float3 crossf(float3 a, float3 b) {
    return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}

constexpr int TEAM = 4;  // threads per sphere: they share its neighbour list

// Reduced radius R_i R_j / (R_i + R_j) of a pair.
__device__ __forceinline__ float reduced_radius(float Ri, float Rj) { return __fdividef(Ri * Rj, Ri + Rj); }

// One contact of sphere i with neighbour entry (j, image) (Eqs. 11-12):
// Hertz normal force, incremental Mindlin tangential force from the
// half-step relative velocity at the contact point, previous tangential
// force projected on the current tangent plane, Coulomb cap.  dl = dX_j -
// dX_i; dr = the entry's reference separation (w: (R_i + R_j)^2 - |xyz|^2);
// Rs the pair's reduced radius.  Updates the history h (force on i) and adds
// the force and torque on i; a pair out of contact (and an unused entry,
// dr.w < 0) adds nothing and clears h.  Without branches, so that the
// contacts of a lane interleave: each is a chain of some 400 cycles.
// The arithmetic is mirror-exact: sphere j, evaluating the same pair,
// obtains exactly the negative force.  Square roots and divisions use the
// hardware approximations (reciprocal square root, fast divide; a few ulp):
// deterministic functions of symmetric operands, so exactness of the pair
// is kept.
__device__ __forceinline__ void pair_contact(const Dem& D, float Ri, float Rj, float Rs, float3 dl, float4 dr,
                                             float3 vi, float3 wi, float3 vj, float3 wj, float dt_inc, float3& h,
                                             float3& F, float3& T) {
    float3 d = make_float3(dr.x + dl.x, dr.y + dl.y, dr.z + dl.z);
    float cut = Ri + Rj;
    // cut^2 - |d|^2 without cancellation: e0 - 2 dref.dl - dl.dl
    float qd = dr.w - (2.f * (dr.x * dl.x + dr.y * dl.y + dr.z * dl.z) + (dl.x * dl.x + dl.y * dl.y + dl.z * dl.z));
    const bool touch = qd > 0.f;
    float d2 = d.x * d.x + d.y * d.y + d.z * d.z;
    float idist = rsqrtf(d2);
    float dist = d2 * idist;
    float delta = __fdividef(qd, cut + dist);
    float3 n = make_float3(d.x * idist, d.y * idist, d.z * idist);
    float rd = Rs * delta;
    float sq = rd * rsqrtf(rd);
    float fn = D.kn * sq * delta;
    float ai = Ri - 0.5f * delta, aj = Rj - 0.5f * delta;
    float3 ri = make_float3(ai * n.x, ai * n.y, ai * n.z);
    float3 rj = make_float3(-(aj * n.x), -(aj * n.y), -(aj * n.z));
    float3 cwj = crossf(wj, rj), cwi = crossf(wi, ri);
    float3 vr = make_float3((vj.x + cwj.x) - (vi.x + cwi.x), (vj.y + cwj.y) - (vi.y + cwi.y),
                            (vj.z + cwj.z) - (vi.z + cwi.z));
    float vn = vr.x * n.x + vr.y * n.y + vr.z * n.z;
    float3 vt = make_float3(vr.x - vn * n.x, vr.y - vn * n.y, vr.z - vn * n.z);
    float hn = h.x * n.x + h.y * n.y + h.z * n.z;
    float kdt = D.kt * sq * dt_inc;
    float3 ft = make_float3(h.x - hn * n.x + kdt * vt.x, h.y - hn * n.y + kdt * vt.y, h.z - hn * n.z + kdt * vt.z);
    float ftm2 = ft.x * ft.x + ft.y * ft.y + ft.z * ft.z;
    float cap = D.mu * fn;
    // |F_t| > mu |F_n|, compared in squares
    const float sc = ftm2 > cap * cap ? cap * rsqrtf(ftm2) : 1.0f;
    // rounded products: with them, a force inside the cap and one on it take
    // the same operations in the sums below
    ft = make_float3(__fmul_rn(ft.x, sc), __fmul_rn(ft.y, sc), __fmul_rn(ft.z, sc));
    float3 Fk = make_float3(-fn * n.x + ft.x, -fn * n.y + ft.y, -fn * n.z + ft.z);
    float3 Tk = crossf(ri, Fk);
    const float3 Fs = make_float3(F.x + Fk.x, F.y + Fk.y, F.z + Fk.z), Ts = make_float3(T.x + Tk.x, T.y + Tk.y, T.z + Tk.z);
    h = touch ? ft : make_float3(0.f, 0.f, 0.f);
    F = touch ? Fs : F;
    T = touch ? Ts : T;
}

// First half kick of velocity Verlet and the drift of one substep:
// half-step velocities vh, wh from the contact (fc, tc), hydrodynamic (fa,
// ta) and body forces; the displacement dx advanced with Kahan-compensated
// FP32 accumulation (compensation c).
__device__ __forceinline__ void kick_drift(const Dem& D, float3 fc, float3 tc, float3 fa, float3 ta, float im,
                                           float iI, float3 v, float3 w, float3& vh, float3& wh, float3& dx,
                                           float3& c) {
    const float dt = D.dt;
    vh = make_float3(v.x + 0.5f * dt * (fc.x + fa.x + D.g.x) * im, v.y + 0.5f * dt * (fc.y + fa.y + D.g.y) * im,
                     v.z + 0.5f * dt * (fc.z + fa.z + D.g.z) * im);
    wh = make_float3(w.x + 0.5f * dt * (tc.x + ta.x) * iI, w.y + 0.5f * dt * (tc.y + ta.y) * iI,
                     w.z + 0.5f * dt * (tc.z + ta.z) * iI);
    float yx = dt * vh.x - c.x, yy = dt * vh.y - c.y, yz = dt * vh.z - c.z;
    float tx = dx.x + yx, ty = dx.y + yy, tz = dx.z + yz;
    c = make_float3((tx - dx.x) - yx, (ty - dx.y) - yy, (tz - dx.z) - yz);
    dx = make_float3(tx, ty, tz);
}

// Orientation over one substep: q <- normalize(q + dt/2 (0, wh) q).
__device__ __forceinline__ void spin(const Dem& D, float3 wh, float4& q) {
    const float dt = D.dt;
    float dq0 = -(wh.x * q.y + wh.y * q.z + wh.z * q.w);
    float3 wxv = crossf(wh, make_float3(q.y, q.z, q.w));
    float4 dq = make_float4(dq0, q.x * wh.x + wxv.x, q.x * wh.y + wxv.y, q.x * wh.z + wxv.z);
    q = make_float4(q.x + 0.5f * dt * dq.x, q.y + 0.5f * dt * dq.y, q.z + 0.5f * dt * dq.z, q.w + 0.5f * dt * dq.w);
    float nq = rsqrtf(q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w);
    q = make_float4(q.x * nq, q.y * nq, q.z * nq, q.w * nq);
}

// Second half kick: V = vh + dt/2 (F + fa + g) / m, W likewise.
__device__ __forceinline__ void close_kick(const Dem& D, float3 vh, float3 wh, float3 F, float3 T, float3 fa,
                                           float3 ta, float im, float iI, float3& v, float3& w) {
    const float dt = D.dt;
    v = make_float3(vh.x + 0.5f * dt * (F.x + fa.x + D.g.x) * im, vh.y + 0.5f * dt * (F.y + fa.y + D.g.y) * im,
                    vh.z + 0.5f * dt * (F.z + fa.z + D.g.z) * im);
    w = make_float3(wh.x + 0.5f * dt * (T.x + ta.x) * iI, wh.y + 0.5f * dt * (T.y + ta.y) * iI,
                    wh.z + 0.5f * dt * (T.z + ta.z) * iI);
}

// sum over the TEAM lanes of a sphere (lanes of a team are consecutive)
__device__ __forceinline__ void team_sum(float3& F, float3& T) {
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int o = 1; o < TEAM; o <<= 1) {
        F.x += __shfl_xor_sync(full, F.x, o);
        F.y += __shfl_xor_sync(full, F.y, o);
        F.z += __shfl_xor_sync(full, F.z, o);
        T.x += __shfl_xor_sync(full, T.x, o);
        T.y += __shfl_xor_sync(full, T.y, o);
        T.z += __shfl_xor_sync(full, T.z, o);
    }
}

// Lattice frame of sphere i after the step (integer origin, wrapped origin,
// FP32 offset of the centre) and its displacement / speed for the
// re-layout decision and the NaN / skin checks.
__device__ __forceinline__ void sphere_frame(const Dem& D, int i, float& dmax, float& vmax, uint32_t& bad) {
    float4 dx = D.dX[i], c = D.dXc[i], v = D.V[i];
    double X0 = D.Xref[3 * i] + (double)dx.x - (double)c.x;
    double X1 = D.Xref[3 * i + 1] + (double)dx.y - (double)c.y;
    double X2 = D.Xref[3 * i + 2] + (double)dx.z - (double)c.z;
    int4 o = make_int4((int)floor(D.Xref[3 * i]), (int)floor(D.Xref[3 * i + 1]), (int)floor(D.Xref[3 * i + 2]), 0);
    D.org[i] = o;
    int wx = D.px ? (int)(((long long)o.x % (long long)D.Lx + (long long)D.Lx) % (long long)D.Lx) : o.x;
    int wy = (int)(((long long)o.y % (long long)D.Ly + (long long)D.Ly) % (long long)D.Ly);
    int wz = (int)(((long long)o.z % (long long)D.Lz + (long long)D.Lz) % (long long)D.Lz);
    D.orgw[i] = make_int4(wx, wy, wz, 0);
    D.xf[i] = make_float4((float)(X0 - o.x), (float)(X1 - o.y), (float)(X2 - o.z), 0.f);
    float dd = sqrtf(dx.x * dx.x + dx.y * dx.y + dx.z * dx.z);
    float vv = sqrtf(v.x * v.x + v.y * v.y + v.z * v.z);
    if (!(dd == dd) || !(vv == vv) || isinf(dd) || isinf(vv)) bad |= ST_UNSTABLE;
    else if (dd >= D.hard_disp) bad |= ST_SKIN;
    dmax = fmaxf(dmax, dd);
    vmax = fmaxf(vmax, vv);
}

// The same outputs for the per-step kernels: the integer origins depend only
// on Xref, which changes only at re-layouts (after which k_dem_init runs
// sphere_frame), so only the FP32 offset of the centre is renewed, from the
// state in registers (every lane of the team holds it).  Lane `tl` < 3 of the
// sphere's team computes axis tl from its Xref and origin; lane 0 checks.
__device__ __forceinline__ void sphere_offset(const Dem& D, int i, int tl, double Xref, int org, float3 dx, float3 c,
                                              float3 v, float& dmax, float& vmax, uint32_t& bad) {
    if (tl < 3) {
        const float d = tl == 0 ? dx.x : tl == 1 ? dx.y : dx.z, k = tl == 0 ? c.x : tl == 1 ? c.y : c.z;
        double X = Xref + (double)d - (double)k;
        reinterpret_cast<float*>(&D.xf[i])[tl] = (float)(X - org);
    }
    if (tl == 0) {
        float dd = sqrtf(dx.x * dx.x + dx.y * dx.y + dx.z * dx.z);
        float vv = sqrtf(v.x * v.x + v.y * v.y + v.z * v.z);
        if (!(dd == dd) || !(vv == vv) || isinf(dd) || isinf(vv)) bad |= ST_UNSTABLE;
        else if (dd >= D.hard_disp) bad |= ST_SKIN;
        dmax = fmaxf(dmax, dd);
        vmax = fmaxf(vmax, vv);
    }
}

// Warp reduction of the maxima and the status bits, one atomic each per warp
// (every lane of the warp calls it).
__device__ __forceinline__ void flush_maxima(const Dem& D, float dmax, float vmax, uint32_t bad) {
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        dmax = fmaxf(dmax, __shfl_xor_sync(full, dmax, o));
        vmax = fmaxf(vmax, __shfl_xor_sync(full, vmax, o));
        bad |= __shfl_xor_sync(full, bad, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (dmax > 0.f) {
            atomicMax(D.max_disp_bits, __float_as_uint(dmax));
            atomicMax(D.disp_layout_bits, __float_as_uint(dmax));
        }
        if (vmax > 0.f) atomicMax(D.max_vel_bits, __float_as_uint(vmax));
        if (bad) atomicOr(D.status, bad);
    }
}

// Hydrodynamic drive of sphere i: the mean of this and the previous step's
// exchange sums.  Lane tl < 3 of the team takes component tl of both (FP64 adds
// run at 2 lanes per clock and SM), then the team shares them.  Every lane
// of the warp calls it; `lead` is the lane of the team's first thread.
__device__ __forceinline__ void hydro_drive(const Dem& D, int i, int tl, bool have, int lead, float3& fa, float3& ta) {
    const unsigned full = 0xffffffffu;
    float hf = 0.f, ht = 0.f;
    if (have && tl < 3) {
        double f = D.Fh[3 * (size_t)i + tl], t = D.Th[3 * (size_t)i + tl];
#pragma unroll
        for (int r = 1; r < NREP; ++r) {
            f += D.Fh[3 * ((size_t)r * D.n + i) + tl];
            t += D.Th[3 * ((size_t)r * D.n + i) + tl];
        }
        hf = 0.5f * (float)(f + D.Fh_prev[3 * (size_t)i + tl]);
        ht = 0.5f * (float)(t + D.Th_prev[3 * (size_t)i + tl]);
        D.Fh_prev[3 * (size_t)i + tl] = f;
        D.Th_prev[3 * (size_t)i + tl] = t;
    }
    fa = make_float3(__shfl_sync(full, hf, lead), __shfl_sync(full, hf, lead + 1), __shfl_sync(full, hf, lead + 2));
    ta = make_float3(__shfl_sync(full, ht, lead), __shfl_sync(full, ht, lead + 1), __shfl_sync(full, ht, lead + 2));
}

// ------------------------------------------------------------ one launch

// The K substeps with every sphere's state in registers of its team.  One
// cluster of C CTAs, spc = blockDim / TEAM spheres per CTA, sphere i in CTA
// i / spc.  Each CTA's shared memory holds the exchanged record of its own
// spheres (slots 0 .. spc - 1) and of the spheres of other CTAs that its own
// neighbour lists name (slots from spc on, assigned by k_dem_ghosts); a sphere
// pushes its record into every CTA that holds it, and all reads of a substep
// are local.  Reading the neighbours through the cluster window instead
// carries each record once per contact, and that window moves about 18 B per
// clock and SM.  The pushes complete a transaction barrier of the receiving
// CTA, which waits for the bytes of all its foreign records; nothing else
// crosses CTAs (a cluster barrier that releases costs 380 to 480 cycles, more
// with remote stores in flight).  The own spheres' records are ordered by
// __syncthreads (30 to 45 cycles).  Three record buffers: a CTA pushes substep
// s + 3 after it has received s + 2 from the CTAs it pushes to (neighbourhood
// is mutual), which they sent after their __syncthreads of s + 1, so all their
// threads are through with substep s.
// 2048 spheres, K = 10: 29 us per step with reads through the cluster window
// and cluster barriers, 22.5 us so; one CTA of 32 spheres 18.5 and 12.9 us.
// The first NBT neighbour entries of each team lane live in registers (with
// their tangential history) for the whole launch; further entries go through
// global memory.
constexpr int DSM_THREADS = 512;
constexpr int DSM_SOLO = 256;  // largest launch of one CTA (twice the registers per thread)
constexpr int DSM_BUFS = 3;
constexpr int NBT = 3;
static_assert(DEM_MAX_CTAS % TEAM == 0, "push targets are split over a team's lanes");

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t cluster_addr(uint32_t a, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
// stores into another CTA's shared memory that count on its barrier
__device__ __forceinline__ void push4(uint32_t a, float4 v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(a),
                 "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void push1(uint32_t a, float v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(a), "f"(v), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ bool bar_done(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0u;
}
// tries before a wait gives up (each suspends for up to some microseconds):
// the status latches a timeout and the step ends with what it has
constexpr int DSM_TRIES = 1 << 16;
constexpr uint32_t RECORD_BYTES = 36;

// The lane's register entries 0 .. U - 1 (warp-uniform U).
template <int U, class Contact>
__device__ __forceinline__ void contacts_n(Contact contact) {
#pragma unroll
    for (int u = 0; u < U; ++u) contact(u);
}

template <bool MULTI>
__global__ void __launch_bounds__(MULTI ? DSM_THREADS : DSM_SOLO, 1) k_dem_step_dsm(Dem D) {
    // exchanged records, [DSM_BUFS][slots]: {dX, Vh.x}, {Vh.yz, Wh.xy}, Wh.z
    extern __shared__ float4 smem[];
    __shared__ __align__(8) unsigned long long bars[DSM_BUFS];
    float4* xa = smem;
    float4* xb = smem + DSM_BUFS * D.slots;
    float* xc = reinterpret_cast<float*>(smem + 2 * DSM_BUFS * D.slots);
    // Launched with a programmatic dependency on the previous kernel: the
    // sphere state and neighbour entries (last written by the previous
    // step's DEM, long complete) are read before waiting for it; the
    // exchange sums it writes, and every write of this kernel, come after.
    // All loads of the state are independent of one another.  With the fluid
    // off the previous kernel is the previous step's DEM itself.
    if (D.dry) pdl_wait();
    const unsigned full = 0xffffffffu;
    const int spc = blockDim.x / TEAM;
    const int tl = threadIdx.x % TEAM, ls = threadIdx.x / TEAM;
    const int i = blockIdx.x * spc + ls;
    const bool have = i < D.n;
    const int lead = (threadIdx.x & 31) & ~(TEAM - 1);  // lane of the team's first thread
    const float3 zero = make_float3(0.f, 0.f, 0.f);
    float3 dx = zero, dxc = zero, v = zero, w = zero, fc = zero, tc = zero;
    float4 q = make_float4(1.f, 0.f, 0.f, 0.f);
    double Xr = 0.0;
    int org = 0;
    float im = 0.f, iI = 0.f, Ri = 1.f;
    bool fixed = true;
    int cnt = 0;
    // slots of this sphere in the CTAs tl, tl + TEAM, ... (16 bits each)
    uint32_t push[DEM_MAX_CTAS / TEAM / 2];
#pragma unroll
    for (int d = 0; d < DEM_MAX_CTAS / TEAM / 2; ++d) push[d] = 0xffffffffu;
    // this lane's neighbour entries tl + u TEAM, u < NBT: slot, radius,
    // reference separation (w < 0: unused) and history
    int nj[NBT];
    float nR[NBT], nRs[NBT];
    float4 ndr[NBT];
    float3 nh[NBT];
#pragma unroll
    for (int u = 0; u < NBT; ++u) {
        nj[u] = 0;
        nR[u] = 1.f;
        ndr[u] = make_float4(0.f, 0.f, 0.f, -1.f);
        nh[u] = zero;
    }
    if (have) {
        cnt = D.nb_cnt[i];
#pragma unroll
        for (int u = 0; u < NBT; ++u) {  // every list holds more than NBT TEAM entries, used or not
            const size_t e = (size_t)i * D.nbmax + tl + u * TEAM;
            nj[u] = D.nb_slot[e];
            nR[u] = D.nb_R[e];
            ndr[u] = D.nb_dref[e];
            nh[u] = f3(D.nb_ft[e]);
        }
        dx = f3(D.dX[i]);
        dxc = f3(D.dXc[i]);
        v = f3(D.V[i]);
        w = f3(D.W[i]);
        q = D.q[i];
        fc = f3(D.Fc[i]);
        tc = f3(D.Tc[i]);
        im = D.invm[i];
        iI = D.invI[i];
        Ri = D.R[i];
        fixed = D.fixed[i] != 0;
        if (tl < 3) {
            Xr = D.Xref[3 * i + tl];
            org = reinterpret_cast<const int*>(&D.org[i])[tl];
        }
        if (MULTI) {
#pragma unroll
            for (int d = 0; d < DEM_MAX_CTAS / TEAM; d += 2) {
                const uint32_t lo = D.push[(size_t)i * DEM_MAX_CTAS + tl + d * TEAM],
                               hi = D.push[(size_t)i * DEM_MAX_CTAS + tl + (d + 1) * TEAM];
                push[d / 2] = lo | (hi << 16);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < NBT; ++u) {
        if (tl + u * TEAM >= cnt || fixed) {
            nj[u] = 0;
            nR[u] = 1.f;
            ndr[u] = make_float4(0.f, 0.f, 0.f, -1.f);
            nh[u] = zero;
        }
        nRs[u] = reduced_radius(Ri, nR[u]);
    }
    const int used = fixed ? 0 : min((cnt - tl + TEAM - 1) / TEAM, NBT);
    const int most = __reduce_max_sync(full, used > 0 ? used : 0);
    uint32_t foreign = 0;  // bytes this CTA receives per substep
    if (MULTI) {  // the barriers exist before a record is pushed at them
        if (threadIdx.x == 0) {
            for (int k = 0; k < DSM_BUFS; ++k)
                asm volatile("mbarrier.init.shared.b64 [%0], 1;" ::"r"(smem_addr(&bars[k])) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        foreign = RECORD_BYTES * (uint32_t)D.foreign[blockIdx.x];
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    pdl_wait();
    pdl_trigger();
    if (blockIdx.x == 0 && threadIdx.x == 0) *D.layout_fresh = 0u;  // this step's map update is done
    float3 fa, ta;
    hydro_drive(D, i, tl, have, lead, fa, ta);
    float dmax = 0.f, vmax = 0.f;
    uint32_t bad = 0;
    for (int s = 0; s < D.K; ++s) {
        const int buf = s % DSM_BUFS, b = buf * D.slots;
        float3 vh = zero, wh = zero;
        if (!fixed) kick_drift(D, fc, tc, fa, ta, im, iI, v, w, vh, wh, dx, dxc);
        const float4 ra = make_float4(dx.x, dx.y, dx.z, vh.x), rb = make_float4(vh.y, vh.z, wh.x, wh.y);
        if (MULTI) {
            const uint32_t bar = smem_addr(&bars[buf]);
            if (threadIdx.x == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"(bar), "r"(foreign) : "memory");
#pragma unroll
            for (int d = 0; d < DEM_MAX_CTAS / TEAM; ++d) {
                const uint32_t slot = (push[d / 2] >> (16 * (d & 1))) & 0xffffu;
                if (slot == 0xffffu) continue;
                const uint32_t rank = tl + d * TEAM, rbar = cluster_addr(bar, rank);
                push4(cluster_addr(smem_addr(&xa[b + slot]), rank), ra, rbar);
                push4(cluster_addr(smem_addr(&xb[b + slot]), rank), rb, rbar);
                push1(cluster_addr(smem_addr(&xc[b + slot]), rank), wh.z, rbar);
            }
        }
        if (have) {
            if (tl == 0) xa[b + ls] = ra;
            if (tl == 1) xb[b + ls] = rb;
            if (tl == 2) xc[b + ls] = wh.z;
        }
        if (!fixed) spin(D, wh, q);
        __syncthreads();
        if (MULTI) {
            const uint32_t bar = smem_addr(&bars[buf]), parity = (uint32_t)(s / DSM_BUFS) & 1u;
            int tries = 0;
            while (!bar_done(bar, parity))
                if (++tries > DSM_TRIES) {
                    bad |= ST_TIMEOUT;
                    break;
                }
        }
        float3 F = zero, T = zero;
        auto contact = [&](int slot, float Rj, float Rs, float4 dr, float3& h) {
            const float4 a = xa[b + slot], c = xb[b + slot];
            const float wz = xc[b + slot];
            pair_contact(D, Ri, Rj, Rs, make_float3(a.x - dx.x, a.y - dx.y, a.z - dx.z), dr, vh, wh,
                         make_float3(a.w, c.x, c.y), make_float3(c.z, c.w, wz), D.dt, h, F, T);
        };
        auto entry = [&](int u) { contact(nj[u], nR[u], nRs[u], ndr[u], nh[u]); };
        if (most == 3) contacts_n<3>(entry);
        else if (most == 2) contacts_n<2>(entry);
        else if (most == 1) contacts_n<1>(entry);
        if (!fixed)
            for (int k = tl + NBT * TEAM; k < cnt; k += TEAM) {  // entries beyond the registers
                const size_t e = (size_t)i * D.nbmax + k;
                float3 h = f3(D.nb_ft[e]);
                contact(D.nb_slot[e], D.nb_R[e], reduced_radius(Ri, D.nb_R[e]), D.nb_dref[e], h);
                D.nb_ft[e] = make_float4(h.x, h.y, h.z, 0.f);
            }
        __syncwarp();
        team_sum(F, T);
        if (fixed) {
            v = w = zero;
        } else {
            fc = F;
            tc = T;
            close_kick(D, vh, wh, F, T, fa, ta, im, iI, v, w);
        }
    }
    if (have) {
#pragma unroll
        for (int u = 0; u < NBT; ++u)
            if (u < used) D.nb_ft[(size_t)i * D.nbmax + tl + u * TEAM] = make_float4(nh[u].x, nh[u].y, nh[u].z, 0.f);
        if (tl == 0) {
            D.dX[i] = make_float4(dx.x, dx.y, dx.z, 0.f);
            D.dXc[i] = make_float4(dxc.x, dxc.y, dxc.z, 0.f);
        } else if (tl == 1) {
            D.V[i] = make_float4(v.x, v.y, v.z, 0.f);
            D.W[i] = make_float4(w.x, w.y, w.z, 0.f);
        } else if (tl == 2) {
            D.q[i] = q;
        } else {
            D.Fc[i] = make_float4(fc.x, fc.y, fc.z, 0.f);
            D.Tc[i] = make_float4(tc.x, tc.y, tc.z, 0.f);
        }
        sphere_offset(D, i, tl, Xr, org, dx, dxc, v, dmax, vmax, bad);
    }
    flush_maxima(D, dmax, vmax, bad);
    if (MULTI) {  // no CTA leaves while another may still push into it (after a wait that gave up)
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// Slots of the exchange for k_dem_step_dsm, one block per CTA of that launch
// (shared memory: a flag per sphere): the spheres of other CTAs that are
// neighbours of this CTA's spheres get the slots from spc on in index order,
// each entry its neighbour's slot, each named sphere its slot in this CTA
// (push, 0xffff elsewhere).  foreign[c] receives the number of those spheres,
// *slots the largest slot count.
__global__ void k_dem_ghosts(Dem D, int spc, int* nb_slot, uint16_t* push, int* foreign, int* slots) {
    extern __shared__ uint8_t need[];
    __shared__ uint32_t part[33];
    const int c = blockIdx.x, i0 = c * spc, i1 = min(i0 + spc, D.n);
    for (int j = threadIdx.x; j < D.n; j += blockDim.x) need[j] = 0;
    __syncthreads();
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x)
        for (int k = 0; k < D.nb_cnt[i]; ++k) {
            const int j = D.nb_j[(size_t)i * D.nbmax + k];
            if (j < i0 || j >= i1) need[j] = 1;
        }
    // and those whose lists name this CTA's spheres: at a distance that rounds
    // to the edge of the skin only one of a pair may list the other, and the
    // record buffers count on pushes going both ways between two CTAs
    for (int j = threadIdx.x; j < D.n; j += blockDim.x) {
        if (j >= i0 && j < i1) continue;
        for (int k = 0; k < D.nb_cnt[j]; ++k) {
            const int i = D.nb_j[(size_t)j * D.nbmax + k];
            if (i >= i0 && i < i1) need[j] = 1;
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int base = spc;
    for (int j0 = 0; j0 < D.n; j0 += blockDim.x) {
        const int j = j0 + threadIdx.x;
        const bool g = j < D.n && need[j];
        const unsigned bal = __ballot_sync(0xffffffffu, g);
        if (lane == 0) part[wid] = __popc(bal);
        __syncthreads();
        int at = base + __popc(bal & ((1u << lane) - 1u));
        for (int k = 0; k < nw; ++k) {
            if (k < wid) at += part[k];
            base += part[k];
        }
        if (j < D.n) push[(size_t)j * DEM_MAX_CTAS + c] = g ? (uint16_t)at : (uint16_t)0xffffu;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        foreign[c] = base - spc;
        atomicMax(slots, base);
    }
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x)
        for (int k = 0; k < D.nb_cnt[i]; ++k) {
            const size_t e = (size_t)i * D.nbmax + k;
            const int j = D.nb_j[e];
            nb_slot[e] = j >= i0 && j < i1 ? j - i0 : (int)push[(size_t)j * DEM_MAX_CTAS + c];
        }
}

// ------------------------------------------------------------ one launch per substep

// Larger packings: k_dem_begin takes the hydrodynamic drive, the first half
// kick and the drift; k_dem_substep evaluates the contacts of substep s and
// closes it, then opens substep s + 1 or, after the last, writes the step's
// outputs.  Chained by programmatic dependent launch, one team per sphere over
// the whole GPU; the records are exchanged through the L2.  About 2 us per
// substep whatever the count (launch hand-over and one round of loads),
// against 18 us for one cluster of 8 CTAs taking several spheres per team with
// the state in global memory (4096 spheres, K = 10: 180 -> 31 us per step).
constexpr int SUB_THREADS = 128;

// q: the lane TEAM - 1 carries the orientation
__device__ __forceinline__ void open_substep(const Dem& D, int i, int tl, int b, float3 dx, float3 c, float4 q,
                                             float3 fc, float3 tc, float3 fa, float3 ta, float3 v, float3 w,
                                             bool fixed, float im, float iI) {
    float3 vh = make_float3(0.f, 0.f, 0.f), wh = vh;
    if (!fixed) kick_drift(D, fc, tc, fa, ta, im, iI, v, w, vh, wh, dx, c);
    if (tl == 0) {
        D.dX[i] = make_float4(dx.x, dx.y, dx.z, 0.f);
        D.dXb[b * D.n + i] = make_float4(dx.x, dx.y, dx.z, vh.x);
    } else if (tl == 1) {
        D.dXc[i] = make_float4(c.x, c.y, c.z, 0.f);
        D.Vhb[b * D.n + i] = make_float4(vh.y, vh.z, wh.x, wh.y);
    } else if (tl == 2) {
        D.Whb[b * D.n + i] = make_float4(wh.z, 0.f, 0.f, 0.f);
    } else if (!fixed) {
        spin(D, wh, q);
        D.q[i] = q;
    }
}
static_assert(TEAM == 4, "open_substep splits its stores over four lanes");

__global__ void __launch_bounds__(SUB_THREADS) k_dem_begin(Dem D) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x, tl = t % TEAM, i = t / TEAM;
    const bool have = i < D.n;
    pdl_wait();
    pdl_trigger();
    if (t == 0) *D.layout_fresh = 0u;  // this step's map update is done
    float3 fa, ta;
    hydro_drive(D, i, tl, have, (threadIdx.x & 31) & ~(TEAM - 1), fa, ta);
    // the team's lanes all read what two of them replace
    float3 dx = make_float3(0.f, 0.f, 0.f), c = dx, fc = dx, tc = dx, v = dx, w = dx;
    float4 q = make_float4(1.f, 0.f, 0.f, 0.f);
    bool fixed = true;
    float im = 0.f, iI = 0.f;
    if (have) {
        dx = f3(D.dX[i]);
        c = f3(D.dXc[i]);
        q = D.q[i];
        fc = f3(D.Fc[i]);
        tc = f3(D.Tc[i]);
        v = f3(D.V[i]);
        w = f3(D.W[i]);
        fixed = D.fixed[i] != 0;
        im = D.invm[i];
        iI = D.invI[i];
    }
    __syncwarp();
    if (!have) return;
    if (tl == 0) D.Fa[i] = make_float4(fa.x, fa.y, fa.z, 0.f);
    if (tl == 1) D.Ta[i] = make_float4(ta.x, ta.y, ta.z, 0.f);
    open_substep(D, i, tl, 0, dx, c, q, fc, tc, fa, ta, v, w, fixed, im, iI);
}

__global__ void __launch_bounds__(SUB_THREADS) k_dem_substep(Dem D, int s) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x, tl = t % TEAM, i = t / TEAM;
    const bool have = i < D.n;
    const int b = s & 1;
    // the lists and constants change only at re-layouts: read ahead of the wait
    int cnt = 0;
    bool fixed = true;
    float Ri = 1.f, im = 0.f, iI = 0.f;
    int nj[NBT];
    float nR[NBT];
    float4 ndr[NBT];
    if (have) {
        fixed = D.fixed[i] != 0;
        cnt = fixed ? 0 : D.nb_cnt[i];
        Ri = D.R[i];
        im = D.invm[i];
        iI = D.invI[i];
    }
#pragma unroll
    for (int u = 0; u < NBT; ++u) {
        const int k = tl + u * TEAM;
        nj[u] = -1;
        if (k < cnt) {
            const size_t e = (size_t)i * D.nbmax + k;
            nj[u] = D.nb_j[e];
            nR[u] = D.nb_R[e];
            ndr[u] = D.nb_dref[e];
        }
    }
    const double Xr = have && tl < 3 ? D.Xref[3 * i + tl] : 0.0;
    const int org = have && tl < 3 ? reinterpret_cast<const int*>(&D.org[i])[tl] : 0;
    pdl_wait();
    pdl_trigger();
    const float3 zero = make_float3(0.f, 0.f, 0.f);
    float3 F = zero, T = zero, dx = zero, vh = zero, wh = zero, c = zero, fa = zero, ta = zero;
    float4 q = make_float4(1.f, 0.f, 0.f, 0.f);
    // every load of the substep is issued before any is used
    float4 xa[NBT], xb[NBT], nh[NBT];
    float xc[NBT];
    if (have) {
        const float4 a = D.dXb[b * D.n + i], e = D.Vhb[b * D.n + i];
        const float z = D.Whb[b * D.n + i].x;
#pragma unroll
        for (int u = 0; u < NBT; ++u) {
            if (tl + u * TEAM >= cnt) continue;
            xa[u] = D.dXb[b * D.n + nj[u]];
            xb[u] = D.Vhb[b * D.n + nj[u]];
            xc[u] = D.Whb[b * D.n + nj[u]].x;
            nh[u] = D.nb_ft[(size_t)i * D.nbmax + tl + u * TEAM];
        }
        c = f3(D.dXc[i]);
        fa = f3(D.Fa[i]);
        ta = f3(D.Ta[i]);
        if (tl == TEAM - 1) q = D.q[i];
        dx = f3(a);
        vh = make_float3(a.w, e.x, e.y);
        wh = make_float3(e.z, e.w, z);
    }
    auto contact = [&](int k, float4 a, float4 e, float z, float3 h, float Rj, float4 dr) {
        pair_contact(D, Ri, Rj, reduced_radius(Ri, Rj), make_float3(a.x - dx.x, a.y - dx.y, a.z - dx.z), dr, vh, wh,
                     make_float3(a.w, e.x, e.y), make_float3(e.z, e.w, z), D.dt, h, F, T);
        D.nb_ft[(size_t)i * D.nbmax + k] = make_float4(h.x, h.y, h.z, 0.f);
    };
#pragma unroll
    for (int u = 0; u < NBT; ++u)
        if (tl + u * TEAM < cnt) contact(tl + u * TEAM, xa[u], xb[u], xc[u], f3(nh[u]), nR[u], ndr[u]);
    for (int k = tl + NBT * TEAM; k < cnt; k += TEAM) {
        const size_t e = (size_t)i * D.nbmax + k;
        const size_t j = b * (size_t)D.n + D.nb_j[e];
        contact(k, D.dXb[j], D.Vhb[j], D.Whb[j].x, f3(D.nb_ft[e]), D.nb_R[e], D.nb_dref[e]);
    }
    __syncwarp();
    team_sum(F, T);
    float dmax = 0.f, vmax = 0.f;
    uint32_t bad = 0;
    if (have) {
        float3 v = zero, w = zero;
        if (!fixed) close_kick(D, vh, wh, F, T, fa, ta, im, iI, v, w);
        if (s + 1 < D.K) {
            open_substep(D, i, tl, b ^ 1, dx, c, q, F, T, fa, ta, v, w, fixed, im, iI);
        } else {
            if (tl == 0) D.V[i] = make_float4(v.x, v.y, v.z, 0.f);
            if (tl == 1) D.W[i] = make_float4(w.x, w.y, w.z, 0.f);
            if (tl == 2 && !fixed) D.Fc[i] = make_float4(F.x, F.y, F.z, 0.f);
            if (tl == 3 && !fixed) D.Tc[i] = make_float4(T.x, T.y, T.z, 0.f);
            sphere_offset(D, i, tl, Xr, org, dx, c, v, dmax, vmax, bad);
        }
    }
    if (s + 1 == D.K) flush_maxima(D, dmax, vmax, bad);
}

// Initial contact forces (no tangential increment) and the spheres' lattice
// frame, after set_packing and after every re-layout.
__global__ void __launch_bounds__(SUB_THREADS) k_dem_init(Dem D) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x, tl = t % TEAM, i = t / TEAM;
    const bool have = i < D.n;
    float3 F = make_float3(0.f, 0.f, 0.f), T = F;
    if (have) {
        const float3 xi = f3(D.dX[i]), vi = f3(D.V[i]), wi = f3(D.W[i]);
        const int cnt = D.nb_cnt[i];
        for (int k = tl; k < cnt; k += TEAM) {
            const size_t e = (size_t)i * D.nbmax + k;
            const int j = D.nb_j[e];
            const float3 xj = f3(D.dX[j]);
            float3 h = f3(D.nb_ft[e]);
            pair_contact(D, D.R[i], D.R[j], reduced_radius(D.R[i], D.R[j]),
                         make_float3(xj.x - xi.x, xj.y - xi.y, xj.z - xi.z), D.nb_dref[e], vi, wi, f3(D.V[j]),
                         f3(D.W[j]), 0.f, h, F, T);
            D.nb_ft[e] = make_float4(h.x, h.y, h.z, 0.f);
        }
    }
    team_sum(F, T);
    float dmax = 0.f, vmax = 0.f;
    uint32_t bad = 0;
    if (have && tl == 0) {
        D.Fc[i] = make_float4(F.x, F.y, F.z, 0.f);
        D.Tc[i] = make_float4(T.x, T.y, T.z, 0.f);
        sphere_frame(D, i, dmax, vmax, bad);
    }
    flush_maxima(D, dmax, vmax, bad);
}

// ------------------------------------------------------------ launches

constexpr size_t dsm_smem(int slots) { return (size_t)slots * DSM_BUFS * RECORD_BYTES; }

// Largest cluster (CTAs of DSM_THREADS threads) k_dem_step_dsm can run with on
// the current device, 0 where it cannot run.
static int find_dsm_cluster() {
    const size_t most = dsm_smem(DEM_MAX_CTAS * DSM_THREADS / TEAM);  // every sphere in every CTA
    if (cudaFuncSetAttribute(k_dem_step_dsm<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaFuncSetAttribute(k_dem_step_dsm<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) !=
            cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    for (int C : {DEM_MAX_CTAS, 8}) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(C, 1, 1);
        cfg.blockDim = dim3(DSM_THREADS, 1, 1);
        cfg.dynamicSmemBytes = most;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = C;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int ncl = 0;
        if (cudaOccupancyMaxActiveClusters(&ncl, k_dem_step_dsm<true>, &cfg) == cudaSuccess && ncl > 0) return C;
        cudaGetLastError();
    }
    return 0;
}

// The smallest CTAs that fit: a CTA holds half an SM's registers at 256
// threads, so DEM clusters of concurrent columns (batches) find room next to
// the lattice kernels.
DemShape dem_shape(int n) {
    static PerDevice<int> cluster;
    int dev = 0;
    cudaGetDevice(&dev);
    const int cmax = cluster.get(dev, find_dsm_cluster);
    const long long need = (long long)TEAM * (n > 0 ? n : 1);
    if (cmax <= 0 || need > (long long)cmax * DSM_THREADS) return {};
    const int T = need <= (long long)cmax * (DSM_THREADS / 2) ? DSM_THREADS / 2 : DSM_THREADS;
    const int C = (int)((need + T - 1) / T);
    return {C, C == 1 ? (int)(((need + 31) / 32) * 32) : T};
}

void launch_dem_ghosts(const Dem& D, int* nb_slot, uint16_t* push, int* foreign, int* slots, cudaStream_t s) {
    const DemShape h = D.shape;
    cudaMemsetAsync(slots, 0, sizeof(int), s);
    if (D.n <= 0 || !h.ctas) return;
    if (h.ctas < DEM_MAX_CTAS) cudaMemsetAsync(push, 0xff, sizeof(uint16_t) * (size_t)D.n * DEM_MAX_CTAS, s);
    k_dem_ghosts<<<h.ctas, 256, D.n, s>>>(D, h.threads / TEAM, nb_slot, push, foreign, slots);
}

int dem_launches(DemShape h, int K) { return h.ctas ? 1 : K + 1; }

void launch_dem_init(const Dem& D, cudaStream_t s) {
    const unsigned blocks = (unsigned)(((long long)TEAM * D.n + SUB_THREADS - 1) / SUB_THREADS);
    if (D.n > 0) k_dem_init<<<blocks, SUB_THREADS, 0, s>>>(D);
}

void launch_dem_step(const Dem& D, cudaStream_t s) {
    const int C = D.shape.ctas;
    if (!C) {
        const unsigned blocks = (unsigned)(((long long)TEAM * D.n + SUB_THREADS - 1) / SUB_THREADS);
        launch_pdl(k_dem_begin, blocks, SUB_THREADS, s, D);
        for (int k = 0; k < D.K; ++k) launch_pdl(k_dem_substep, blocks, SUB_THREADS, s, D, k);
        return;
    }
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // pdl_wait before the sums are read
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = C;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = C > 1 ? 2 : 1;
    cfg.gridDim = dim3(C, 1, 1);
    cfg.blockDim = dim3(D.shape.threads, 1, 1);
    cfg.dynamicSmemBytes = dsm_smem(D.slots);
    if (C > 1) cudaLaunchKernelEx(&cfg, k_dem_step_dsm<true>, D);
    else cudaLaunchKernelEx(&cfg, k_dem_step_dsm<false>, D);
}

// ------------------------------------------------------------ neighbour lists

__device__ __forceinline__ int floordiv(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }
__device__ __forceinline__ int floormod(int a, int b) { return a - floordiv(a, b) * b; }

// Cell of a position: periodic axes use the wrapped coordinate and return
// the wrap count k (X = X_wrapped + k L); the x axis clamps when not periodic.
__device__ __forceinline__ int cell_axis(double X, double lo, double h, int nc, double L, int periodic,
                                         int& k) {
    if (periodic) {
        k = (int)floor(X / L);
        double xw = X - k * L;
        int c = (int)floor(xw / h);
        return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
    }
    k = 0;
    int c = (int)floor((X - lo) / h);
    return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
}

__global__ void k_cell_count(const double* X, int n, CellGrid G, int* cell_of, int* count) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int kx, ky, kz;
    int cx_ = cell_axis(X[3 * i], G.lo.x, G.h.x, G.nc.x, G.L.x, G.px, kx);
    int cy_ = cell_axis(X[3 * i + 1], 0.0, G.h.y, G.nc.y, G.L.y, 1, ky);
    int cz_ = cell_axis(X[3 * i + 2], 0.0, G.h.z, G.nc.z, G.L.z, 1, kz);
    int c = (cx_ * G.nc.y + cy_) * G.nc.z + cz_;
    cell_of[i] = c;
    atomicAdd(&count[c], 1);
}

__global__ void k_cell_fill(const int* cell_of, int n, int* fill, int* order) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int slot = atomicAdd(&fill[cell_of[i]], 1);
    order[slot] = i;
}

// Per sphere: all (j, image) within R_i + R_j + skin, sorted by (j, image),
// tangential history copied from the previous list where the key matches.
__global__ void k_nb_build(NbBuild B) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B.n) return;
    const CellGrid& G = B.G;
    double Xi[3] = {B.X[3 * i], B.X[3 * i + 1], B.X[3 * i + 2]};
    int ki[3];
    int ci[3];
    ci[0] = cell_axis(Xi[0], G.lo.x, G.h.x, G.nc.x, G.L.x, G.px, ki[0]);
    ci[1] = cell_axis(Xi[1], 0.0, G.h.y, G.nc.y, G.L.y, 1, ki[1]);
    ci[2] = cell_axis(Xi[2], 0.0, G.h.z, G.nc.z, G.L.z, 1, ki[2]);
    int nc[3] = {G.nc.x, G.nc.y, G.nc.z};
    int per[3] = {G.px, 1, 1};
    double L[3] = {G.L.x, G.L.y, G.L.z};
    size_t base = (size_t)i * B.nbmax;
    int cnt = 0;
    double Ri = B.R[i];
    for (int dx = -1; dx <= 1; ++dx) {
        int ux = ci[0] + dx;
        int wx = ux, sx = 0;
        if (per[0]) {
            wx = floormod(ux, nc[0]);
            sx = floordiv(ux, nc[0]);
        } else if (ux < 0 || ux >= nc[0]) {
            continue;
        }
        for (int dy = -1; dy <= 1; ++dy) {
            int uy = ci[1] + dy, wy = floormod(uy, nc[1]), sy = floordiv(uy, nc[1]);
            for (int dz = -1; dz <= 1; ++dz) {
                int uz = ci[2] + dz, wz = floormod(uz, nc[2]), sz = floordiv(uz, nc[2]);
                int c = (wx * nc[1] + wy) * nc[2] + wz;
                for (int a = B.start[c]; a < B.start[c + 1]; ++a) {
                    int j = B.order[a];
                    if (j == i) continue;
                    int kj[3];
                    cell_axis(B.X[3 * j], G.lo.x, G.h.x, G.nc.x, G.L.x, G.px, kj[0]);
                    cell_axis(B.X[3 * j + 1], 0.0, G.h.y, G.nc.y, G.L.y, 1, kj[1]);
                    cell_axis(B.X[3 * j + 2], 0.0, G.h.z, G.nc.z, G.L.z, 1, kj[2]);
                    int s[3] = {per[0] ? sx - kj[0] + ki[0] : 0, sy - kj[1] + ki[1], sz - kj[2] + ki[2]};
                    double d[3];
                    for (int q = 0; q < 3; ++q) d[q] = (B.X[3 * j + q] + s[q] * L[q]) - Xi[q];
                    double cut = Ri + B.R[j] + B.skin;
                    double dd = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
                    if (dd >= cut * cut) continue;
                    if (cnt >= B.nbmax) {
                        atomicOr(B.status, ST_CAPACITY);
                        continue;
                    }
                    size_t e = base + cnt++;
                    B.nj[e] = j;
                    B.nsh[4 * e] = (int8_t)s[0];
                    B.nsh[4 * e + 1] = (int8_t)s[1];
                    B.nsh[4 * e + 2] = (int8_t)s[2];
                    B.nsh[4 * e + 3] = 0;
                    // the overlap is later formed from e0 = (R_i + R_j)^2 - |dref|^2,
                    // taken here in FP64 from the unrounded offset, so FP32 never
                    // cancels two ~2R numbers (nor carries dref's rounding)
                    double c2 = Ri + B.R[j];
                    double e0 = c2 * c2 - dd;
                    B.dref[e] = make_float4((float)d[0], (float)d[1], (float)d[2], (float)e0);
                }
            }
        }
    }
    // insertion sort by (j, sx, sy, sz)
    auto key = [&](size_t e) -> long long {
        return ((long long)B.nj[e] << 24) | ((long long)(B.nsh[4 * e] + 8) << 16) |
               ((long long)(B.nsh[4 * e + 1] + 8) << 8) | (long long)(B.nsh[4 * e + 2] + 8);
    };
    for (int a = 1; a < cnt; ++a) {
        size_t ea = base + a;
        long long ka = key(ea);
        int j = B.nj[ea];
        int8_t sh[4] = {B.nsh[4 * ea], B.nsh[4 * ea + 1], B.nsh[4 * ea + 2], 0};
        float4 dr = B.dref[ea];
        int b = a - 1;
        while (b >= 0 && key(base + b) > ka) {
            size_t eb = base + b, eb1 = base + b + 1;
            B.nj[eb1] = B.nj[eb];
            for (int q = 0; q < 4; ++q) B.nsh[4 * eb1 + q] = B.nsh[4 * eb + q];
            B.dref[eb1] = B.dref[eb];
            --b;
        }
        size_t e = base + b + 1;
        B.nj[e] = j;
        for (int q = 0; q < 4; ++q) B.nsh[4 * e + q] = sh[q];
        B.dref[e] = dr;
    }
    // carry the tangential history over
    int oc = B.old_cnt ? B.old_cnt[i] : 0;
    for (int a = 0; a < cnt; ++a) {
        size_t e = base + a;
        float4 h = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int b = 0; b < oc; ++b) {
            size_t o = base + b;
            if (B.old_j[o] == B.nj[e] && B.old_sh[4 * o] == B.nsh[4 * e] &&
                B.old_sh[4 * o + 1] == B.nsh[4 * e + 1] && B.old_sh[4 * o + 2] == B.nsh[4 * e + 2]) {
                h = B.old_ft[o];
                break;
            }
        }
        B.ft[e] = h;
        B.nR[e] = (float)B.R[B.nj[e]];
    }
    B.cnt[i] = cnt;
}


void launch_cells(const double* X, int n, const CellGrid& G, int* cell_of, int* count, int* start,
                  int* fill, int* order, uint32_t* scan_tmp, cudaStream_t s) {
    int ncell = G.nc.x * G.nc.y * G.nc.z;
    // count[ncell] stays 0, so the exclusive scan of ncell + 1 counts also
    // leaves the total in start[ncell]; the fill cursors start as a copy
    cudaMemsetAsync(count, 0, sizeof(int) * (ncell + 1), s);
    if (n > 0) k_cell_count<<<(n + 255) / 256, 256, 0, s>>>(X, n, G, cell_of, count);
    exclusive_scan(reinterpret_cast<const uint32_t*>(count), reinterpret_cast<uint32_t*>(start), (size_t)ncell + 1,
                   scan_tmp, s);
    cudaMemcpyAsync(fill, start, sizeof(int) * ncell, cudaMemcpyDeviceToDevice, s);
    if (n > 0) k_cell_fill<<<(n + 255) / 256, 256, 0, s>>>(cell_of, n, fill, order);
}

void launch_nb_build(const NbBuild& B, cudaStream_t s) {
    if (B.n > 0) k_nb_build<<<(B.n + 127) / 128, 128, 0, s>>>(B);
}

// Spheres whose surface may reach a band node before the next re-layout
// (|y - Xref| < R + skin, all images), ascending, at most 4, and the node's
// slack: its distance to the nearest candidate surface.  The owner of the
// node is a function of the candidates' inside tests (and, inside two or
// more spheres, of their distance ratios), so it cannot change while every
// sphere stays closer than the slack to its layout position; a node inside
// two or more candidates, or a boundary-plane node, is flagged 0 (always
// re-tested) or never changes (planes stay fluid) respectively.
__global__ void k_band_cand(BandCand B) {
    uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= B.n) return;
    const CellGrid& G = B.G;
    int x, y, z;
    unpack_coord(B.coord[k], x, y, z);
    double P[3] = {(double)x, (double)y, (double)z};
    int kk[3], ci[3];
    ci[0] = cell_axis(P[0], G.lo.x, G.h.x, G.nc.x, G.L.x, G.px, kk[0]);
    ci[1] = cell_axis(P[1], 0.0, G.h.y, G.nc.y, G.L.y, 1, kk[1]);
    ci[2] = cell_axis(P[2], 0.0, G.h.z, G.nc.z, G.L.z, 1, kk[2]);
    int nc[3] = {G.nc.x, G.nc.y, G.nc.z};
    double L[3] = {G.L.x, G.L.y, G.L.z};
    const double iL[3] = {1.0 / G.L.x, 1.0 / G.L.y, 1.0 / G.L.z};  // once per node, not per candidate
    int per[3] = {G.px, 1, 1};
    int c4[4] = {-1, -1, -1, -1};
    int nfound = 0, ninside = 0;
    double slack = 1e30;
    for (int dx = -1; dx <= 1; ++dx) {
        int ux = ci[0] + dx, wx = ux;
        if (per[0]) wx = floormod(ux, nc[0]);
        else if (ux < 0 || ux >= nc[0]) continue;
        for (int dy = -1; dy <= 1; ++dy) {
            int wy = floormod(ci[1] + dy, nc[1]);
            for (int dz = -1; dz <= 1; ++dz) {
                int wz = floormod(ci[2] + dz, nc[2]);
                int c = (wx * nc[1] + wy) * nc[2] + wz;
                for (int a = B.start[c]; a < B.start[c + 1]; ++a) {
                    int p = B.order[a];
                    bool dup = false;
                    for (int q = 0; q < nfound; ++q) dup |= c4[q] == p;
                    if (dup) continue;
                    double d2 = 0;
                    for (int q = 0; q < 3; ++q) {
                        double d = P[q] - B.X[3 * p + q];
                        if (per[q]) d -= L[q] * floor(d * iL[q] + 0.5);
                        d2 += d * d;
                    }
                    double r = B.R[p] + B.skin;
                    if (d2 >= r * r) continue;
                    slack = fmin(slack, fabs(sqrt(d2) - B.R[p]));
                    ninside += d2 < B.R[p] * B.R[p];
                    if (nfound >= 4) {
                        atomicOr(B.status, ST_CAPACITY);
                        continue;
                    }
                    // insert sorted
                    int q = nfound++;
                    while (q > 0 && c4[q - 1] > p) {
                        c4[q] = c4[q - 1];
                        --q;
                    }
                    c4[q] = p;
                }
            }
        }
    }
    B.cand[k] = make_int4(c4[0], c4[1], c4[2], c4[3]);
    if (ninside >= 2) slack = 0.0;
    if (!G.px && (x == 0 || x == B.nx - 1)) slack = 1e30;  // inlet/outlet planes stay fluid
    B.slack[k] = (float)slack;
    if (B.band_dense) B.band_dense[((size_t)x * B.ny + y) * B.nz + z] = nfound >= 2 ? 2 : 1;
}

void launch_band_cand(const BandCand& B, cudaStream_t s) {
    if (B.n > 0) k_band_cand<<<(B.n + 255) / 256, 256, 0, s>>>(B);
}

// Band list ordered by slack (bucket sort, order inside a bucket arbitrary):
// the nodes a step has to re-test -- slack up to the displacement since the
// layout -- then form a prefix of the list and fill whole warps, and the
// warps past it leave after one coalesced load.
constexpr int SLACK_BUCKETS = 1024;
static_assert(SLACK_HIST == SLACK_BUCKETS + 1, "bucket counts and the total");
__device__ __forceinline__ int slack_bucket(float slack, float top) {
    float b = slack * (float)SLACK_BUCKETS / top;
    return b < (float)(SLACK_BUCKETS - 1) ? (int)b : SLACK_BUCKETS - 1;
}
__global__ void k_slack_hist(const float* slack, uint32_t n, float top, uint32_t* hist) {
    uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) atomicAdd(&hist[slack_bucket(slack[k], top)], 1u);
}
__global__ void k_slack_scatter(const uint32_t* coord, const int4* cand, const float* slack, uint32_t n, float top,
                                uint32_t* next, uint32_t* coord2, int4* cand2, float* slack2) {
    uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    uint32_t pos = atomicAdd(&next[slack_bucket(slack[k], top)], 1u);
    coord2[pos] = coord[k];
    cand2[pos] = cand[k];
    slack2[pos] = slack[k];
}
void launch_band_sort(const uint32_t* coord, const int4* cand, const float* slack, uint32_t n, double skin,
                      uint32_t* hist, uint32_t* scan_tmp, uint32_t* coord2, int4* cand2, float* slack2,
                      cudaStream_t s) {
    if (n == 0) return;
    const float top = (float)(2.0 * skin);  // band nodes lie within skin of a surface
    cudaMemsetAsync(hist, 0, sizeof(uint32_t) * (SLACK_BUCKETS + 1), s);
    k_slack_hist<<<(n + 255) / 256, 256, 0, s>>>(slack, n, top, hist);
    exclusive_scan(hist, hist, SLACK_BUCKETS + 1, scan_tmp, s);
    k_slack_scatter<<<(n + 255) / 256, 256, 0, s>>>(coord, cand, slack, n, top, hist, coord2, cand2, slack2);
}

__global__ void k_rebase(double* Xref, float4* dX, float4* dXc, int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float4 d = dX[i], c = dXc[i];
    Xref[3 * i] += (double)d.x - (double)c.x;
    Xref[3 * i + 1] += (double)d.y - (double)c.y;
    Xref[3 * i + 2] += (double)d.z - (double)c.z;
    dX[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    dXc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

void launch_rebase(double* Xref, float4* dX, float4* dXc, int n, cudaStream_t s) {
    if (n > 0) k_rebase<<<(n + 255) / 256, 256, 0, s>>>(Xref, dX, dXc, n);
}

}  // namespace lbmdem
