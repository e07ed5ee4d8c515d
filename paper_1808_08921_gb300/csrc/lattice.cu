// lattice.cu -- fluid kernels on the compact AA lattice:
//   * collide+stream, even and odd parity (Section 2.1, Eqs. 4-8), with the
//     probe-plane density and the FP64 mass/momentum totals fused in;
//   * pressure inlet with the oscillating density and the outlet
//     (Section 2.4, Eq. 25, Table 2);
//   * read-out of rho and u (Eq. 7) for any parity.
// Populations are stored as deviations g = f - w rho_f; every formula below is
// the paper's written in g (the weights sum to one, and sum_m w_m c_m = 0).
#include "common.cuh"
#include "kernels.cuh"

namespace lbmdem {

static_assert(cx(opp(7)) == -cx(7) && cy(opp(7)) == -cy(7), "opp");

// Four consecutive populations of one plane (the even kernel's vector
// access): 16 B for FP32, 8 B for the 16-bit forms, streamed (evict-first).
template <int ST> __device__ __forceinline__ float4 ld4(const typename PopT<ST>::T* p, float fsi);
template <> __device__ __forceinline__ float4 ld4<0>(const float* p, float) {
    return __ldcs(reinterpret_cast<const float4*>(p));
}
template <> __device__ __forceinline__ float4 ld4<1>(const __nv_bfloat16* p, float fsi) {
    uint2 r = __ldcs(reinterpret_cast<const uint2*>(p));
    float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r.x));
    float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r.y));
    return make_float4(a.x * fsi, a.y * fsi, b.x * fsi, b.y * fsi);
}
template <> __device__ __forceinline__ float4 ld4<2>(const __half* p, float fsi) {
    uint2 r = __ldcs(reinterpret_cast<const uint2*>(p));
    float2 a = __half22float2(*reinterpret_cast<const __half2*>(&r.x));
    float2 b = __half22float2(*reinterpret_cast<const __half2*>(&r.y));
    return make_float4(a.x * fsi, a.y * fsi, b.x * fsi, b.y * fsi);
}
template <int ST> __device__ __forceinline__ void st4(typename PopT<ST>::T* p, float4 v, float fs);
template <> __device__ __forceinline__ void st4<0>(float* p, float4 v, float) {
    __stcs(reinterpret_cast<float4*>(p), v);
}
template <> __device__ __forceinline__ void st4<1>(__nv_bfloat16* p, float4 v, float fs) {
    __nv_bfloat162 a = __floats2bfloat162_rn(v.x * fs, v.y * fs), b = __floats2bfloat162_rn(v.z * fs, v.w * fs);
    uint2 r;
    r.x = *reinterpret_cast<const uint32_t*>(&a);
    r.y = *reinterpret_cast<const uint32_t*>(&b);
    __stcs(reinterpret_cast<uint2*>(p), r);
}
template <> __device__ __forceinline__ void st4<2>(__half* p, float4 v, float fs) {
    __half2 a = __floats2half2_rn(v.x * fs, v.y * fs), b = __floats2half2_rn(v.z * fs, v.w * fs);
    uint2 r;
    r.x = *reinterpret_cast<const uint32_t*>(&a);
    r.y = *reinterpret_cast<const uint32_t*>(&b);
    __stcs(reinterpret_cast<uint2*>(p), r);
}

// Eq. 4 with the equilibrium of Eq. 6 and the moments of Eq. 7, on deviations.
// Returns the moments of the pre-collision state.
__device__ __forceinline__ void bgk(float g[Q], float tau_inv, float rho_f, float& drho, float& jx,
                                    float& jy, float& jz) {
    drho = 0.f;
    jx = jy = jz = 0.f;
#pragma unroll
    for (int m = 0; m < Q; ++m) {
        drho += g[m];
        if (cx(m)) jx += cx(m) > 0 ? g[m] : -g[m];
        if (cy(m)) jy += cy(m) > 0 ? g[m] : -g[m];
        if (cz(m)) jz += cz(m) > 0 ? g[m] : -g[m];
    }
    float rho = rho_f + drho;
    float ir = 1.0f / rho;
    float ux = jx * ir, uy = jy * ir, uz = jz * ir;
    float uu15 = 1.5f * (ux * ux + uy * uy + uz * uz);
    float om = 1.0f - tau_inv;
#pragma unroll
    for (int m = 0; m < Q; ++m) {
        float cu = (float)cx(m) * ux + (float)cy(m) * uy + (float)cz(m) * uz;
        float geq = wt(m) * (drho + rho * (3.0f * cu + 4.5f * cu * cu - uu15));
        g[m] = om * g[m] + tau_inv * geq;
    }
}

struct MonAcc {
    float drho, jx, jy, jz, umax2, cnt;
    float pdrho, pcnt;  // probe plane
    int bad;
};

__device__ __forceinline__ void mon_add(MonAcc& a, float drho, float jx, float jy, float jz,
                                        float rho_f) {
    a.drho += drho;
    a.cnt += 1.f;
    a.jx += jx;
    a.jy += jy;
    a.jz += jz;
    float ir = 1.0f / (rho_f + drho);
    float u2 = (jx * jx + jy * jy + jz * jz) * ir * ir;
    a.umax2 = fmaxf(a.umax2, u2);
    if (!(drho == drho) || !(u2 == u2)) a.bad = 1;
}

// Warp + block reduction of the monitors, one FP64 atomic per block per
// quantity; the probe sums use warp-aggregated atomics.
template <bool MON>
__device__ __forceinline__ void mon_flush(const MonAcc& a, const Mon& mon, bool probe_any) {
    const unsigned full = 0xffffffffu;
    if (mon.probe_sum != nullptr) {
        if (__any_sync(full, a.pcnt > 0.f)) {
            float s = a.pdrho, c = a.pcnt;
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                s += __shfl_xor_sync(full, s, o);
                c += __shfl_xor_sync(full, c, o);
            }
            if ((threadIdx.x & 31) == 0) {
                unsigned long long t = *mon.t_dev - 1ull;  // the map update counted this step
                atomicAdd(&mon.probe_sum[2 * t], (double)s);
                atomicAdd(&mon.probe_sum[2 * t + 1], (double)c);
            }
        }
    }
    if (!MON) return;
    __shared__ double sh[6][32];
    double v[5] = {a.drho, a.jx, a.jy, a.jz, a.cnt};
    float um = a.umax2;
    int bad = a.bad;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
#pragma unroll
        for (int k = 0; k < 5; ++k) v[k] += __shfl_xor_sync(full, v[k], o);
        um = fmaxf(um, __shfl_xor_sync(full, um, o));
        bad |= __shfl_xor_sync(full, bad, o);
    }
    int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        for (int k = 0; k < 5; ++k) sh[k][wid] = v[k];
        sh[5][wid] = (double)um;
        if (bad) atomicOr(mon.status, ST_UNSTABLE);
    }
    __syncthreads();
    if (wid == 0) {
        int nw = blockDim.x >> 5;
        double r[6];
        for (int k = 0; k < 6; ++k) r[k] = lane < nw ? sh[k][lane] : 0.0;
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            for (int k = 0; k < 5; ++k) r[k] += __shfl_xor_sync(full, r[k], o);
            r[5] = fmax(r[5], __shfl_xor_sync(full, r[5], o));
        }
        if (lane == 0) {
            for (int k = 0; k < 5; ++k) atomicAdd(&mon.acc[k], r[k]);
            atomicMax(mon.umax_bits, __float_as_uint((float)r[5]));
        }
    }
}

// Even step: node-local.  Each thread owns 4 consecutive compact nodes and
// moves them with 128-bit loads and stores; solid nodes inside a quad are
// processed harmlessly (their slots are never read while they are solid).
// SNAP: the natural populations the step starts from also go to snap
// ([19][nSpad] FP32) for the reverse sweep, from the registers they are
// collided in.
template <bool MON, int ST, bool SNAP>
__global__ void __launch_bounds__(256) k_collide_even(Lat L, Mon mon, float* snap) {
    pdl_wait();
    pdl_trigger();
    auto* f = pops<ST>(L);
    uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t i0 = t * 4u;
    MonAcc a = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    bool active = i0 < L.nS;
    uint32_t bits = 0;
    if (active) {
        bits = (L.fbits[i0 >> 5] >> (i0 & 31)) & 0xfu;
        active = bits != 0;
    }
    if (active) {
        float4 v[Q];
#pragma unroll
        for (int m = 0; m < Q; ++m)
            v[m] = ld4<ST>(f + (size_t)m * L.nSpad + i0, L.fsi);
        if (SNAP) {
#pragma unroll
            for (int m = 0; m < Q; ++m) __stcs(reinterpret_cast<float4*>(snap + (size_t)m * L.nSpad + i0), v[m]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float g[Q];
#pragma unroll
            for (int m = 0; m < Q; ++m) g[m] = (&v[m].x)[k];
            float drho, jx, jy, jz;
            bgk(g, L.tau_inv, L.rho_f, drho, jx, jy, jz);
#pragma unroll
            for (int m = 0; m < Q; ++m) (&v[opp(m)].x)[k] = g[m];
            if ((bits >> k) & 1u) {
                if (MON) mon_add(a, drho, jx, jy, jz, L.rho_f);
                uint32_t i = i0 + k;
                if (i >= mon.p0 && i < mon.p1) {
                    a.pdrho += drho;
                    a.pcnt += 1.f;
                }
            }
        }
#pragma unroll
        for (int m = 0; m < Q; ++m)
            st4<ST>(f + (size_t)m * L.nSpad + i0, v[m], L.fs);
    }
    mon_flush<MON>(a, mon, true);
}

// ---- collide with the step's links (one node per lane)
//
// Where a node's post-collision values are written its links can be bounced.
// For a link direction m of fluid node x (x + c_m solid, owned by sphere p)
// the value leaving towards the wall, g~_m, goes to slot opp(m) of x, in an
// even step as in an odd one, as g~_m - delta (Eq. 14, moving wall),
//     delta = 6 w_m rho_f c_m . U,   U = V + W x r,   r = x - X,
// the wall velocity at x (the half-link offset c_m / 2 drops out because
// c_m . (W x c_m) = 0), and adds the link force c_m (2 g~_m - delta) of
// Eq. 15 (counted about the rest state, as the link kernel does) and its
// torque r x c_m (2 g~_m - delta) of Eq. 19 to the sphere.  A node's links
// belong to one sphere or two, each leaving its six sums in a column of
// shared memory until the populations are stored; then the warp sums the
// columns sphere by sphere and adds each sum with one FP64 atomic per
// component.  The rare node of more than two spheres adds its own sums.

// The links of node (x, y, z) to sphere p (bit m of msk: direction m): g
// becomes what the slots take, out the sums.  u is 6 rho_f / 36 times the wall
// velocity, so that delta is c.u, twice that on the axes, and a pair of
// opposite directions shares it.
__device__ __forceinline__ void node_links(const Lat& L, const PartView& P, int x, int y, int z, int p, uint32_t msk,
                                           float g[Q], float out[6]) {
    const float4 a = P.pk[3 * (size_t)p], b = P.pk[3 * (size_t)p + 1], c = P.pk[3 * (size_t)p + 2];
    const int ox = __float_as_int(c.y), oy = __float_as_int(c.z), oz = __float_as_int(c.w);
    const int ix = L.px ? imin_small(x - ox, L.nx) : x - ox;
    const int iy = imin_small(y - oy, L.ny), iz = imin_small(z - oz, L.nz);
    const float rx = (float)ix - a.x, ry = (float)iy - a.y, rz = (float)iz - a.z;
    const float s = L.rho_f * (1.0f / 6.0f);
    const float ux = s * (a.w + (b.w * rz - c.x * ry)), uy = s * (b.x + (c.x * rx - b.z * rz)),
                uz = s * (b.y + (b.z * ry - b.w * rx));
    float fx = 0.f, fy = 0.f, fz = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int m = pair_m(k), o = opp(m);
        float t = 0.f;
        if (cx(m)) t += cx(m) > 0 ? ux : -ux;
        if (cy(m)) t += cy(m) > 0 ? uy : -uy;
        if (cz(m)) t += cz(m) > 0 ? uz : -uz;
        const float d = k < 3 ? 2.0f * t : t;
        const bool hm = (msk >> m) & 1u, ho = (msk >> o) & 1u;
        float q = 0.f;
        if (hm) {
            q = 2.0f * g[m] - d;
            g[m] -= d;
        }
        if (ho) {
            q -= 2.0f * g[o] + d;
            g[o] += d;
        }
        if (cx(m)) fx += cx(m) > 0 ? q : -q;
        if (cy(m)) fy += cy(m) > 0 ? q : -q;
        if (cz(m)) fz += cz(m) > 0 ? q : -q;
    }
    out[0] = fx;
    out[1] = fy;
    out[2] = fz;
    out[3] = ry * fz - rz * fy;
    out[4] = rz * fx - rx * fz;
    out[5] = rx * fy - ry * fx;
}

// A lane's sums for two spheres (a and b, -1: none), in a column of shared
// memory: force and torque of a, then of b.
constexpr int LINK_COLS = 12;

struct LinkSums {
    float* col;
    int a, b;
};

__device__ __forceinline__ void sums_put(float* c, const float v[6]) {
#pragma unroll
    for (int k = 0; k < 6; ++k) c[k * 32] = v[k];
}

// All links of a node with link word w.
__device__ __forceinline__ void all_links(const Lat& L, const PartView& P, int x, int y, int z, uint2 w, uint32_t rep,
                                          float g[Q], LinkSums& n) {
    float v[6];
    int pa = (int)(w.x >> 18), pb = (int)(w.y >> 18);
    uint32_t mb = w.y & LW_MASK, ma = w.x & LW_MASK & ~mb;
    if (pa == (int)LW_NONE) {
        // neighbours of more than two spheres: their owners from the map, the
        // third sphere's links (and a further one's) here, by this lane alone
        int own[Q - 1];
#pragma unroll
        for (int m = 0; m < Q - 1; ++m) {
            if (!((w.x >> m) & 1u)) continue;
            int xs = x + cx(m);
            if (L.px) xs = wrap1(xs, L.nx);
            own[m] = __ldg(&L.owner[((size_t)xs * L.ny + wrap1(y + cy(m), L.ny)) * L.nz + wrap1(z + cz(m), L.nz)]);
        }
        uint32_t rem = w.x & LW_MASK;
        auto next = [&](int& p) {  // the links of the first remaining direction's sphere
            p = -1;
            uint32_t sub = 0u;
#pragma unroll
            for (int m = 0; m < Q - 1; ++m) {
                if (!((rem >> m) & 1u)) continue;
                if (p < 0) p = own[m];
                if (own[m] == p) sub |= 1u << m;
            }
            rem &= ~sub;
            return sub;
        };
        ma = next(pa);
        mb = next(pb);
        while (rem) {
            int p;
            const uint32_t sub = next(p);
            node_links(L, P, x, y, z, p, sub, g, v);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                atomicAdd(P.Fh + 3 * ((size_t)rep * P.n + p) + k, (double)v[k]);
                atomicAdd(P.Th + 3 * ((size_t)rep * P.n + p) + k, (double)v[k + 3]);
            }
        }
    }
    n.a = pa;
    node_links(L, P, x, y, z, pa, ma, g, v);
    sums_put(n.col, v);
    if (mb) {
        n.b = pb;
        node_links(L, P, x, y, z, pb, mb, g, v);
        sums_put(n.col + 6 * 32, v);
    }
}

// The warp's columns, sphere by sphere.
__device__ __forceinline__ void columns_add(const PartView& P, uint32_t rep, LinkSums& n) {
    const unsigned full = 0xffffffffu;
    const uint32_t lane = threadIdx.x & 31;
    const int comp = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
    const bool adds = (lane & 3) == 0 && comp < 6;
    double* dst = (comp < 3 ? P.Fh + comp : P.Th + (comp - 3)) + 3 * (size_t)rep * P.n;
    for (;;) {
        const int mine = n.a >= 0 ? n.a : n.b;
        const unsigned act = __ballot_sync(full, mine >= 0);
        if (!act) break;
        const int p = __shfl_sync(full, mine, __ffs(act) - 1);
        float s8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (n.a == p || n.b == p) {  // not both
            const float* v = n.a == p ? n.col : n.col + 6 * 32;
#pragma unroll
            for (int c = 0; c < 6; ++c) s8[c] = v[c * 32];
            if (n.a == p) n.a = -1;
            else n.b = -1;
        }
        // transposing butterfly (lane l ends with component 4 b4 + 2 b3 + b2)
        {
            const bool up = lane & 16;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float keep = up ? s8[c + 4] : s8[c], send = up ? s8[c] : s8[c + 4];
                s8[c] = keep + __shfl_xor_sync(full, send, 16);
            }
        }
        {
            const bool up = lane & 8;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float keep = up ? s8[c + 2] : s8[c], send = up ? s8[c] : s8[c + 2];
                s8[c] = keep + __shfl_xor_sync(full, send, 8);
            }
        }
        {
            const bool up = lane & 4;
            const float keep = up ? s8[1] : s8[0], send = up ? s8[0] : s8[1];
            s8[0] = keep + __shfl_xor_sync(full, send, 4);
        }
        s8[0] += __shfl_xor_sync(full, s8[0], 2);
        s8[0] += __shfl_xor_sync(full, s8[0], 1);
        if (adds) atomicAdd(dst + 3 * (size_t)p, (double)s8[0]);
    }
}

// Collision of a node whose links are taken with it: opposite directions share
// their equilibrium terms, and the rest population takes what the moving
// ones leave of the density, so that the FP32 weights conserve mass.
__device__ __forceinline__ void bgk_pairs(float g[Q], float tau_inv, float rho_f, float& drho, float& jx, float& jy,
                                          float& jz) {
    float s[9], d[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        s[k] = g[pair_m(k)] + g[opp(pair_m(k))];
        d[k] = g[pair_m(k)] - g[opp(pair_m(k))];
    }
    drho = (s[0] + s[1]) + (s[2] + s[3]) + ((s[4] + s[5]) + (s[6] + s[7])) + (s[8] + g[18]);
    jx = jy = jz = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int m = pair_m(k);
        if (cx(m)) jx += cx(m) > 0 ? d[k] : -d[k];
        if (cy(m)) jy += cy(m) > 0 ? d[k] : -d[k];
        if (cz(m)) jz += cz(m) > 0 ? d[k] : -d[k];
    }
    const float rho = rho_f + drho, ir = 1.0f / rho;
    const float ux = jx * ir, uy = jy * ir, uz = jz * ir;
    const float om = 1.0f - tau_inv;
    // weight 1/36 terms times 1 / tau: odd part lo c.j, even part e + q (c.u)^2.
    // What 12 lo misses of 1 / tau would be a bias of the momentum at every
    // step (jx off by 1.7e-6 instead of 0.7e-6 after 64 steps at tau 0.67), so
    // the axes take it
    const float lo = tau_inv * (1.0f / 12.0f), miss = 0.5f * fmaf(-12.0f, lo, tau_inv);
    const float t36 = lo * (1.0f / 3.0f), q = 4.5f * t36 * rho;
    const float e = t36 * (drho - 1.5f * (jx * ux + jy * uy + jz * uz));
    float moving = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int m = pair_m(k), o = opp(m);
        float cu = 0.f, cj = 0.f;
        if (cx(m)) cu += cx(m) > 0 ? ux : -ux, cj += cx(m) > 0 ? jx : -jx;
        if (cy(m)) cu += cy(m) > 0 ? uy : -uy, cj += cy(m) > 0 ? jy : -jy;
        if (cz(m)) cu += cz(m) > 0 ? uz : -uz, cj += cz(m) > 0 ? jz : -jz;
        float ev = e + (q * cu) * cu, od = lo * cj;
        if (k < 3) {
            ev *= 2.0f;
            od = fmaf(miss, cj, 2.0f * od);
        }
        moving += ev;
        g[m] = om * g[m] + (ev + od);
        g[o] = om * g[o] + (ev - od);
    }
    g[18] = om * g[18] + (tau_inv * drho - 2.0f * moving);
}

template <int ST> __device__ __forceinline__ float ld1(const typename PopT<ST>::T* p, float fsi) {
    return to_f<ST>(*p, fsi);
}
template <> __device__ __forceinline__ float ld1<0>(const float* p, float) { return __ldcs(p); }
template <int ST> __device__ __forceinline__ void st1(typename PopT<ST>::T* p, float v, float fs) {
    *p = from_f<ST>(v, fs);
}
template <> __device__ __forceinline__ void st1<0>(float* p, float v, float) { __stcs(p, v); }

// Even step with the step's links.  152 B per node and its 12 B of words (104
// us on the 128 x 128 x 1024 column) against about 880 instructions per warp: the
// issue slots (65%) and the loads' latency bound it together, at 36 warps
// per SM.  184 us with register slots per lane over two runs of nodes, 72
// registers and every direction worked through alone; 181 so (64 and 48
// registers are no faster).
template <bool MON, int ST>
__global__ void __maxnreg__(56)
k_collide_even_links(Lat L, Mon mon, PartView P, const uint2* __restrict__ lwp) {
    pdl_wait();
    pdl_trigger();
    auto* f = pops<ST>(L);
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x, rep = (i >> 5) % NREP;
    MonAcc a = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    extern __shared__ float s_col[];  // [warp][LINK_COLS][lane]
    LinkSums n = {s_col + (threadIdx.x >> 5) * (LINK_COLS * 32) + (threadIdx.x & 31), -1, -1};
    if (i < L.nS && fluid_bit(L, i)) {
        float g[Q];
#pragma unroll
        for (int m = 0; m < Q; ++m) g[m] = ld1<ST>(f + (size_t)m * L.nSpad + i, L.fsi);
        const uint2 w = __ldg(&lwp[i]);
        const uint32_t cw = __ldg(&L.coord[i]);
        float drho, jx, jy, jz;
        bgk_pairs(g, L.tau_inv, L.rho_f, drho, jx, jy, jz);
        if (MON) mon_add(a, drho, jx, jy, jz, L.rho_f);
        if (i >= mon.p0 && i < mon.p1) {
            a.pdrho += drho;
            a.pcnt += 1.f;
        }
        if (w.x & LW_MASK) {
            int x, y, z;
            unpack_coord(cw, x, y, z);
            all_links(L, P, x, y, z, w, rep, g, n);
        }
#pragma unroll
        for (int m = 0; m < Q; ++m) st1<ST>(f + (size_t)opp(m) * L.nSpad + i, g[m], L.fs);
    }
    columns_add(P, rep, n);
    mon_flush<MON>(a, mon, true);
}

// ---- even step with few links
//
// The same for lattices where few nodes have links (a sphere alone in a box):
// two slots per lane in registers carry the sums of two spheres over
// EVEN_ROUNDS runs of nodes, the collision is that of the other steps.  What
// such a flow has across its axis (plane momenta, the torque on the sphere) is
// little more than the rounding of these sums, and callers keep the rounding
// they had: over twelve boxes of 28^3 to 160^3, R 8 to 9, they move by up to
// 2.5e-5 of themselves, with the paired collision and the columns by up to
// 3.5e-4.  Time per even step: 60^3 10.5 us against 9.2 us with columns, 160^3
// 115 and 110 us; with 5.3 links per node (128 x 128 x 1024 column) 184 and
// 180 us.

struct LinkSlot {
    int p;
    float v[6];  // force xyz, torque xyz
};

__device__ __forceinline__ void slot_put(LinkSlot& s, int p, const float v[6]) {
    if (s.p < 0) {
        s.p = p;
#pragma unroll
        for (int c = 0; c < 6; ++c) s.v[c] = v[c];
    } else {
#pragma unroll
        for (int c = 0; c < 6; ++c) s.v[c] += v[c];
    }
}

__device__ __forceinline__ void slot_add(LinkSlot& s0, LinkSlot& s1, const PartView& P, int p, const float v[6],
                                         uint32_t rep) {
    if (s0.p == p || s0.p < 0) {
        slot_put(s0, p, v);
    } else if (s1.p == p || s1.p < 0) {
        slot_put(s1, p, v);
    } else {  // a third sphere: add the second slot to the sums and reuse it
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            atomicAdd(P.Fh + 3 * ((size_t)rep * P.n + s1.p) + c, (double)s1.v[c]);
            atomicAdd(P.Th + 3 * ((size_t)rep * P.n + s1.p) + c, (double)s1.v[c + 3]);
        }
        s1.p = -1;
        slot_put(s1, p, v);
    }
}

// The links of node (x, y, z) to sphere p (bit m of msk: direction m).
__device__ __forceinline__ void slot_links(const Lat& L, const PartView& P, int x, int y, int z, int p, uint32_t msk,
                                           float g[Q], float out[6]) {
    const float4 a = P.pk[3 * (size_t)p], b = P.pk[3 * (size_t)p + 1], c = P.pk[3 * (size_t)p + 2];
    const int ox = __float_as_int(c.y), oy = __float_as_int(c.z), oz = __float_as_int(c.w);
    const int ix = L.px ? imin_small(x - ox, L.nx) : x - ox;
    const int iy = imin_small(y - oy, L.ny), iz = imin_small(z - oz, L.nz);
    const float rx = (float)ix - a.x, ry = (float)iy - a.y, rz = (float)iz - a.z;
    const float Ux = a.w + (b.w * rz - c.x * ry), Uy = b.x + (c.x * rx - b.z * rz), Uz = b.y + (b.z * ry - b.w * rx);
    const float s6 = 6.0f * L.rho_f;
    float fx = 0.f, fy = 0.f, fz = 0.f;
#pragma unroll
    for (int m = 0; m < Q - 1; ++m) {
        if (!((msk >> m) & 1u)) continue;
        const float cu = (float)cx(m) * Ux + (float)cy(m) * Uy + (float)cz(m) * Uz;
        const float d = (s6 * wt(m)) * cu;
        const float v = g[m];
        g[m] = v - d;
        const float q = 2.0f * v - d;
        if (cx(m)) fx += cx(m) > 0 ? q : -q;
        if (cy(m)) fy += cy(m) > 0 ? q : -q;
        if (cz(m)) fz += cz(m) > 0 ? q : -q;
    }
    out[0] = fx;
    out[1] = fy;
    out[2] = fz;
    out[3] = ry * fz - rz * fy;
    out[4] = rz * fx - rx * fz;
    out[5] = rx * fy - ry * fx;
}

// owner of the neighbour x + c_m (a link direction, so in range)
__device__ __forceinline__ int neighbour_owner(const Lat& L, int x, int y, int z, int m) {
    int xs = x + cx(m);
    if (L.px) xs = wrap1(xs, L.nx);
    const int ys = wrap1(y + cy(m), L.ny), zs = wrap1(z + cz(m), L.nz);
    return L.owner[((size_t)xs * L.ny + ys) * L.nz + zs];
}

// Each warp takes EVEN_ROUNDS consecutive runs of 32 nodes, one node per
// lane and run (coalesced); the lanes' sphere slots carry over from run to
// run (neighbouring runs mostly touch the same spheres), so the warp sums
// them once per 32 EVEN_ROUNDS nodes.
constexpr int EVEN_ROUNDS = 2;

// 72 registers (a few spills to L1): 28 resident warps per SM instead of 24
// at the 80 the kernel would otherwise take.  Launched with up to 256 threads
// per block.
template <bool MON, int ST>
__global__ void __maxnreg__(72) k_collide_even_slots(Lat L, Mon mon, PartView P, const uint2* __restrict__ lwp) {
    pdl_wait();
    pdl_trigger();
    auto* f = pops<ST>(L);
    const uint32_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t rep = gw % NREP;
    MonAcc a = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    LinkSlot s0, s1;
    s0.p = s1.p = -1;
#pragma unroll
    for (int c = 0; c < 6; ++c) s0.v[c] = s1.v[c] = 0.f;
    for (int run = 0; run < EVEN_ROUNDS; ++run) {
    const uint32_t i = (gw * EVEN_ROUNDS + run) * 32u + (threadIdx.x & 31);
    if (i < L.nS && fluid_bit(L, i)) {
        float g[Q];
#pragma unroll
        for (int m = 0; m < Q; ++m) g[m] = ld1<ST>(f + (size_t)m * L.nSpad + i, L.fsi);
        const uint2 w = __ldg(&lwp[i]);
        const uint32_t cw = __ldg(&L.coord[i]);
        float drho, jx, jy, jz;
        bgk(g, L.tau_inv, L.rho_f, drho, jx, jy, jz);
        if (MON) mon_add(a, drho, jx, jy, jz, L.rho_f);
        if (i >= mon.p0 && i < mon.p1) {
            a.pdrho += drho;
            a.pcnt += 1.f;
        }
        const uint32_t mask = w.x & LW_MASK;
        if (mask) {
            int x, y, z;
            unpack_coord(cw, x, y, z);
            const uint32_t pa = w.x >> 18, pb = w.y >> 18, sel = w.y & LW_MASK;
            float v[6];
            if (pa != LW_NONE) {
                slot_links(L, P, x, y, z, (int)pa, mask & ~sel, g, v);
                slot_add(s0, s1, P, (int)pa, v, rep);
                if (sel) {
                    slot_links(L, P, x, y, z, (int)pb, sel, g, v);
                    slot_add(s0, s1, P, (int)pb, v, rep);
                }
            } else {
                // neighbours of more than two spheres: one sphere at a time
                uint32_t rem = mask;
                while (rem) {
                    int p = -1;
#pragma unroll
                    for (int m = 0; m < Q - 1; ++m)
                        if (p < 0 && ((rem >> m) & 1u)) p = neighbour_owner(L, x, y, z, m);
                    uint32_t sub = 0u;
#pragma unroll
                    for (int m = 0; m < Q - 1; ++m)
                        if (((rem >> m) & 1u) && neighbour_owner(L, x, y, z, m) == p) sub |= 1u << m;
                    slot_links(L, P, x, y, z, p, sub, g, v);
                    slot_add(s0, s1, P, p, v, rep);
                    rem &= ~sub;
                }
            }
        }
#pragma unroll
        for (int m = 0; m < Q; ++m) st1<ST>(f + (size_t)opp(m) * L.nSpad + i, g[m], L.fs);
    }
    }
    // the warp's slots, sphere by sphere: lanes holding the sphere contribute
    const unsigned full = 0xffffffffu;
    const uint32_t lane = threadIdx.x & 31;
    for (;;) {
        const int mine = s0.p >= 0 ? s0.p : s1.p;
        const unsigned act = __ballot_sync(full, mine >= 0);
        if (!act) break;
        const int p = __shfl_sync(full, mine, __ffs(act) - 1);
        float s8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (s0.p == p) {
#pragma unroll
            for (int c = 0; c < 6; ++c) s8[c] += s0.v[c];
            s0.p = -1;
        }
        if (s1.p == p) {
#pragma unroll
            for (int c = 0; c < 6; ++c) s8[c] += s1.v[c];
            s1.p = -1;
        }
        // transposing butterfly (lane l ends with component 4 b4 + 2 b3 + b2)
        {
            const bool up = lane & 16;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float keep = up ? s8[c + 4] : s8[c], send = up ? s8[c] : s8[c + 4];
                s8[c] = keep + __shfl_xor_sync(full, send, 16);
            }
        }
        {
            const bool up = lane & 8;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float keep = up ? s8[c + 2] : s8[c], send = up ? s8[c] : s8[c + 2];
                s8[c] = keep + __shfl_xor_sync(full, send, 8);
            }
        }
        {
            const bool up = lane & 4;
            const float keep = up ? s8[1] : s8[0], send = up ? s8[0] : s8[1];
            s8[0] = keep + __shfl_xor_sync(full, send, 4);
        }
        s8[0] += __shfl_xor_sync(full, s8[0], 2);
        s8[0] += __shfl_xor_sync(full, s8[0], 1);
        const int comp = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
        if ((lane & 3) == 0 && comp < 6) {
            const size_t r = (size_t)rep * P.n + p;
            double* dst = comp < 3 ? P.Fh + 3 * r + comp : P.Th + 3 * r + (comp - 3);
            atomicAdd(dst, (double)s8[0]);
        }
    }
    mon_flush<MON>(a, mon, true);
}

// Odd step: node x gathers direction m from slot opp(m) of x - c_m (or from
// its own slot m when x - c_m is solid or outside), collides, and scatters
// direction m to slot m of x + c_m (or its own slot opp(m)): the population
// leaving along m and the one arriving against it share one location, so the
// 18 element offsets are formed once and the update is in place.  Which
// neighbours are fluid is read from the node's link word (a solid neighbour is
// a link), where they are stored from nine word records: five lines that give
// three neighbours each and four that give one.  Testing each neighbour's
// fluid bit in its record, with two index regions per record and a second
// record past a word's end, took 174 us on the 128 x 128 x 1024 column and 157
// on 160^3 (all fluid), this form 160 and 138 with the offsets in registers
// (64; 80 leave fewer warps: 164 and 144; 48 spill: 225 and 172).  It waits
// for its chain of three dependent loads, so the warps in flight count: the
// offsets wait in shared memory from the loads to the stores, which leaves
// 40 registers and 48 warps per SM, 139 and 120 us.  152 B per fluid node
// plus its 8 B link word: 98 and 97 us at the copy rate.
//
// With LINKS the step's links are taken here too (see above), at 56 registers:
// 191 us on the same column (64: 196, 48 with spills: 196) against 138 and
// 141 in a link kernel that loads and stores the links' populations again.
template <bool MON, int ST, bool SNAP, bool LINKS>
__global__ void __maxnreg__(LINKS ? 56 : 40)
k_collide_odd(Lat L, Mon mon, const uint2* __restrict__ lw, float* snap, PartView P) {
    pdl_wait();
    pdl_trigger();
    auto* f = pops<ST>(L);
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    MonAcc a = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    extern __shared__ uint32_t s_off[];  // [warp][Q - 1][lane]
    uint32_t* off = s_off + (threadIdx.x >> 5) * ((Q - 1) * 32) + (threadIdx.x & 31);
    // three independent loads: then the word records, then the populations
    const bool in = i < L.nS;
    const uint32_t cw = in ? __ldcs(&L.coord[i]) : 0u, lwx = in ? __ldg(&lw[i].x) : 0u;
    LinkSums n = {reinterpret_cast<float*>(s_off + (blockDim.x >> 5) * ((Q - 1) * 32)) +
                      (threadIdx.x >> 5) * (LINK_COLS * 32) + (threadIdx.x & 31),
                  -1, -1};
    if (in && fluid_bit(L, i)) {
        uint32_t wall = lwx & LW_MASK;  // directions without a fluid neighbour
        int x, y, z;
        unpack_coord(cw, x, y, z);
        float g[Q];
        // the place of the population between x and x + c_m, whose compact
        // index is n: a 32-bit offset (19 nSpad < 2^32, checked at the layout)
        auto take = [&](int m, uint32_t n) {
            const uint32_t o = (wall >> m) & 1u ? (uint32_t)opp(m) * L.nSpad + i : (uint32_t)m * L.nSpad + n;
            off[m * 32] = o;
            g[opp(m)] = to_f<ST>(f[o], L.fsi);
        };
        for_neighbours(L, x, y, z, wall, take);
        g[18] = to_f<ST>(f[18u * L.nSpad + i], L.fsi);
        if (SNAP) {
#pragma unroll
            for (int m = 0; m < Q; ++m) __stcs(snap + (size_t)m * L.nSpad + i, g[m]);
        }
        float drho, jx, jy, jz;
        if (LINKS) bgk_pairs(g, L.tau_inv, L.rho_f, drho, jx, jy, jz);
        else bgk(g, L.tau_inv, L.rho_f, drho, jx, jy, jz);
        if (LINKS && (lwx & LW_MASK)) all_links(L, P, x, y, z, __ldg(&lw[i]), (i >> 5) % NREP, g, n);
#pragma unroll
        for (int m = 0; m < Q - 1; ++m) f[off[m * 32]] = from_f<ST>(g[m], L.fs);
        f[18u * L.nSpad + i] = from_f<ST>(g[18], L.fs);
        if (MON) mon_add(a, drho, jx, jy, jz, L.rho_f);
        if (i >= mon.p0 && i < mon.p1) {
            a.pdrho += drho;
            a.pcnt += 1.f;
        }
    }
    if (LINKS) columns_add(P, (i >> 5) % NREP, n);
    mon_flush<MON>(a, mon, true);
}

template <int ST>
static void launch_collide_links_st(const Lat& L, const Mon& mon, const PartView& P, bool odd, bool monitor,
                                    bool few, const uint2* lw, int tile, cudaStream_t s) {
    if (few && !odd) {
        const uint32_t nodes = tile * EVEN_ROUNDS, blocks = (L.nS + nodes - 1) / nodes;
        if (monitor) launch_pdl(k_collide_even_slots<true, ST>, blocks, tile, s, L, mon, P, lw);
        else launch_pdl(k_collide_even_slots<false, ST>, blocks, tile, s, L, mon, P, lw);
        return;
    }
    const uint32_t blocks = (L.nS + tile - 1) / tile;
    const size_t smem = (size_t)(LINK_COLS + (odd ? Q - 1 : 0)) * tile * sizeof(float);
    float* none = nullptr;
    if (odd) {
        if (monitor) launch_pdl_smem(k_collide_odd<true, ST, false, true>, blocks, tile, smem, s, L, mon, lw, none, P);
        else launch_pdl_smem(k_collide_odd<false, ST, false, true>, blocks, tile, smem, s, L, mon, lw, none, P);
    } else {
        if (monitor) launch_pdl_smem(k_collide_even_links<true, ST>, blocks, tile, smem, s, L, mon, P, lw);
        else launch_pdl_smem(k_collide_even_links<false, ST>, blocks, tile, smem, s, L, mon, P, lw);
    }
}

// few: a lattice of few links per node (even steps only)
void launch_collide_links(const Lat& L, const Mon& mon, const PartView& P, bool odd, bool monitor, bool few,
                          const uint2* lw, int tile, cudaStream_t s) {
    if (L.nS == 0) return;
    switch (L.st) {
        case 0: launch_collide_links_st<0>(L, mon, P, odd, monitor, few, lw, tile, s); break;
        case 1: launch_collide_links_st<1>(L, mon, P, odd, monitor, few, lw, tile, s); break;
        default: launch_collide_links_st<2>(L, mon, P, odd, monitor, few, lw, tile, s); break;
    }
}

template <int ST>
static void launch_collide_st(const Lat& L, const Mon& mon, bool odd, bool monitor, const uint2* lw, float* snap,
                              int tile, cudaStream_t s) {
    const uint32_t threads = odd ? L.nS : (L.nS + 3) / 4, blocks = (threads + tile - 1) / tile;
    const size_t smem = (size_t)(Q - 1) * tile * sizeof(uint32_t);  // 4.6 KB per 64 threads
    if (odd) {
        if (snap) launch_pdl_smem(k_collide_odd<false, ST, true, false>, blocks, tile, smem, s, L, mon, lw, snap, PartView{});
        else if (monitor) launch_pdl_smem(k_collide_odd<true, ST, false, false>, blocks, tile, smem, s, L, mon, lw, snap, PartView{});
        else launch_pdl_smem(k_collide_odd<false, ST, false, false>, blocks, tile, smem, s, L, mon, lw, snap, PartView{});
    } else {
        if (snap) launch_pdl(k_collide_even<false, ST, true>, blocks, tile, s, L, mon, snap);
        else if (monitor) launch_pdl(k_collide_even<true, ST, false>, blocks, tile, s, L, mon, snap);
        else launch_pdl(k_collide_even<false, ST, false>, blocks, tile, s, L, mon, snap);
    }
}

// tile: threads per block (64, 128 or 256; the kernels are bounded for 256);
// snap: null, or where the state before the step goes (not with monitor)
void launch_collide(const Lat& L, const Mon& mon, bool odd, bool monitor, const uint2* lw, float* snap, int tile,
                    cudaStream_t s) {
    if (L.nS == 0) return;
    switch (L.st) {
        case 0: launch_collide_st<0>(L, mon, odd, monitor, lw, snap, tile, s); break;
        case 1: launch_collide_st<1>(L, mon, odd, monitor, lw, snap, tile, s); break;
        default: launch_collide_st<2>(L, mon, odd, monitor, lw, snap, tile, s); break;
    }
}

// ------------------------------------------------------------ inlet / outlet

template <bool AFTER_EVEN, int ST>
__global__ void k_inlet_outlet(Lat L, BC bc, const uint2* lw) {
    __shared__ float s_drho;
    if (threadIdx.x == 0) s_drho = (float)source_drho(bc.src, *bc.t_dev);
    const BoundaryNode<AFTER_EVEN, ST> node(L, bc, lw, blockIdx.x * blockDim.x + threadIdx.x);
    __syncthreads();
    node.apply(L, bc, s_drho);
}

void launch_inlet_outlet(const Lat& L, const BC& bc, const uint2* lw, bool after_even, cudaStream_t s) {
    if (L.px) return;
    if (bc.inlet != 0 && bc.outlet > 1) return;
    int n = 2 * L.ny * L.nz;
    int blocks = (n + 127) / 128;
#define LBMDEM_IO(AE, ST) k_inlet_outlet<AE, ST><<<blocks, 128, 0, s>>>(L, bc, lw)
    LBMDEM_BY_STATE(LBMDEM_IO);
#undef LBMDEM_IO
}

// ------------------------------------------------------------ read-out

template <bool AFTER_EVEN, int ST>
__global__ void k_read_fields(Lat L, double* rho, double* u, uint8_t* solid) {
    size_t N = (size_t)L.nx * L.ny * L.nz;
    size_t n = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    int z = (int)(n % L.nz);
    size_t r = n / L.nz;
    int y = (int)(r % L.ny);
    int x = (int)(r / L.ny);
    bool fl;
    uint32_t i = stored_index(L, x, y, z, fl);
    fl = fl && i != NONE;
    if (solid) solid[n] = fl ? 0 : 1;
    double d = 0, jx = 0, jy = 0, jz = 0;
    if (fl) {
#pragma unroll
        for (int m = 0; m < Q; ++m) {
            double g = (double)to_f<ST>(*pop_loc<ST>(L, AFTER_EVEN, x, y, z, i, m), L.fsi);
            d += g;
            jx += cx(m) * g;
            jy += cy(m) * g;
            jz += cz(m) * g;
        }
    }
    double rr = fl ? (double)L.rho_f + d : 0.0;
    if (rho) rho[n] = rr;
    if (u) {
        u[n] = fl ? jx / rr : 0.0;
        u[N + n] = fl ? jy / rr : 0.0;
        u[2 * N + n] = fl ? jz / rr : 0.0;
    }
}

void launch_read_fields(const Lat& L, bool after_even, double* rho, double* u, uint8_t* solid,
                        cudaStream_t s) {
    size_t N = (size_t)L.nx * L.ny * L.nz;
    unsigned blocks = (unsigned)((N + 255) / 256);
#define LBMDEM_RF(AE, ST) k_read_fields<AE, ST><<<blocks, 256, 0, s>>>(L, rho, u, solid)
    LBMDEM_BY_STATE(LBMDEM_RF);
#undef LBMDEM_RF
}

// ------------------------------------------------------------ plane means

// Sums over the fluid nodes of every x plane of the current state: out[3 x]
// += sum (rho - rho_f), out[3 x + 1] += sum rho u_x, out[3 x + 2] += count.
// A plane's nodes are one range of the compact order (from its first word's
// base); PLANE_SPLIT blocks share a plane, every thread adds
// its nodes' FP32 terms in FP64, and each block adds its sums to the plane's
// with one atomic per quantity.  FP64 adds run at 2 lanes per clock and SM
// here, so the count of them decides: one per node and quantity, against 64
// when every lane summed its whole warp (128 x 128 x 1024 column, 4.15 M
// fluid nodes: 1568 -> 100 us; 160^3, all fluid: 1449 -> 81 us).  The parity is
// a template parameter: as a run-time branch around every population it keeps
// the 19 loads of a node one behind the other (252 us).
constexpr int PLANE_SPLIT = 4, PLANE_THREADS = 256;

template <bool AFTER_EVEN, int ST>
__global__ void __launch_bounds__(PLANE_THREADS) k_plane_sums(Lat L, double* out) {
    const int px = blockIdx.x / PLANE_SPLIT, part = blockIdx.x % PLANE_SPLIT;
    const size_t w0 = (size_t)px * L.ny * L.nw;
    const uint32_t lo = L.rec[w0].y, hi = px + 1 == L.nx ? L.nS : L.rec[w0 + (size_t)L.ny * L.nw].y;
    double sd = 0.0, sj = 0.0;
    uint32_t n = 0;
    for (uint32_t i = lo + part * PLANE_THREADS + threadIdx.x; i < hi; i += PLANE_SPLIT * PLANE_THREADS) {
        if (!fluid_bit(L, i)) continue;
        int x, y, z;
        unpack_coord(L.coord[i], x, y, z);
        float d = 0.f, jx = 0.f;
#pragma unroll
        for (int m = 0; m < Q; ++m) {
            const float g = to_f<ST>(*pop_loc<ST>(L, AFTER_EVEN, x, y, z, i, m), L.fsi);
            d += g;
            jx += cx(m) * g;
        }
        sd += (double)d;
        sj += (double)jx;
        ++n;
    }
    const unsigned full = 0xffffffffu;
    n = __reduce_add_sync(full, n);
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        sd += __shfl_xor_sync(full, sd, o);
        sj += __shfl_xor_sync(full, sj, o);
    }
    __shared__ double sh[2][PLANE_THREADS / 32];
    __shared__ uint32_t shn[PLANE_THREADS / 32];
    if ((threadIdx.x & 31) == 0) {
        sh[0][threadIdx.x >> 5] = sd;
        sh[1][threadIdx.x >> 5] = sj;
        shn[threadIdx.x >> 5] = n;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double v = 0.0;
        for (int w = 0; w < PLANE_THREADS / 32; ++w) v += sh[threadIdx.x][w];
        if (v != 0.0) atomicAdd(&out[3 * px + threadIdx.x], v);
    } else if (threadIdx.x == 2) {
        uint32_t v = 0;
        for (int w = 0; w < PLANE_THREADS / 32; ++w) v += shn[w];
        if (v) atomicAdd(&out[3 * px + 2], (double)v);
    }
}

void launch_plane_sums(const Lat& L, bool after_even, double* out, cudaStream_t s) {
    const unsigned blocks = (unsigned)L.nx * PLANE_SPLIT;
    if (!L.nS) return;
#define LBMDEM_PS(AE, ST) k_plane_sums<AE, ST><<<blocks, PLANE_THREADS, 0, s>>>(L, out)
    LBMDEM_BY_STATE(LBMDEM_PS);
#undef LBMDEM_PS
}

}  // namespace lbmdem
