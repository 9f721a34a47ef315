// Hessian-vector products H(X_t) V_t of the physical potential, one cluster of CL
// CTAs per frame (CL > 1 splits the block rows, bonds and angles between the
// CTAs; each then writes its share of the atoms, summing the partials of all). Used by
// the double backward of the energy (the gradient of sum_t |grad U(X_t)|^2 is
// sum_t 2 H(X_t) grad U(X_t); the Onsager-Machlup action of Eq. (SOM) contains (grad U)^2).
// A warp takes a row of an 8-atom block I against up to 32 later blocks: the blocks whose
// boxes lie within r_c, of these the atoms within r_c of some atom of I, and these 64 at a
// time, two per lane, the two pairs of a lane in packed FP32 operations.
//
// For a pair term phi(r) with d = x_j - x_i and w = v_j - v_i:
//   (Hv)_j = phi'' (d.w) d / r^2 + (phi'/r) (w - (d.w) d / r^2),  (Hv)_i = -(Hv)_j,
// with the shifted-force phi' (the shift is linear in r, so phi'' is unchanged).
// For an angle term k/2 (theta - theta0)^2:
//   H v = k (grad theta . v) grad theta + k (theta - theta0) D_v(grad theta),
// D_v being the directional derivative along v, written out by hand below.
// Each chunk of 64 atoms sums its terms in FP32 in a fixed order (8 for an entry, 16 and a
// tree over the quarters of the warp for an atom of I); those sums go to 2^-20 fixed-point
// partials held as 32-bit words (32-bit shared atomics), so results are bit-reproducible, and
// the same for every cluster size, since units and chunks do not depend on it. (400 frames of
// 1200 atoms 783 -> 518 us against pairs of whole blocks in scalar operations with three
// atomics a component; 50 frames of 560 54 -> 43, 3 of 1199 138 -> 38 us.)
#include <cooperative_groups.h>

#include "scps_internal.h"

namespace cg = cooperative_groups;

namespace scps {

namespace {

constexpr unsigned kFullMask = 0xffffffffu;
constexpr int kHvpSeg = 32;          // candidate blocks J per work unit (one per lane)
constexpr int kHvpMaxBlocks = kMaxChainAtoms / 8;  // 8-atom blocks per frame

struct HvpShared {
    float4* xq;      // (x, y, z, qs)
    float4* vq;      // direction v
    float2* lj;
    unsigned long long* ex;  // exclusion mask per atom slot
    // 2^-20 fixed-point partials v of 3 components per slot: the low 20 bits (unsigned), the
    // rest q = v >> 20 as a sum modulo 2^32 and coarse sums of round(q / 2^22), which only the
    // largest terms (stiff bonds) touch. (A slot takes at most 256 sums as an entry, 40 as a block
    // atom, and its bonds and angles; up to 1023 terms are exact, see coarse_shift.)
    unsigned *L0, *L1;
    int* H;
    float4* blo;     // boxes of the 8-atom blocks
    float4* bhi;
    uint16_t* buf;   // per warp: the atoms of its unit
    int nta;
};

__device__ __forceinline__ void hred(const HvpShared& sm, int k, float x) {
    const long long v = f2fix(x), q = v >> 20;
    atomicAdd(&sm.L0[k], (unsigned)(v & 0xfffffll));
    atomicAdd(&sm.L1[k], (unsigned)q);
    const int h = (int)(((q >> 21) + 1) >> 1);
    if (h) atomicAdd(&sm.H[k], h);
}

__device__ __forceinline__ void hadd(const HvpShared& sm, int i, float x, float y, float z) {
    hred(sm, 3 * i, x);
    hred(sm, 3 * i + 1, y);
    hred(sm, 3 * i + 2, z);
}

// phi'(r)/r of the shifted-force pair potential, the negative of phi'' - phi'(r)/r over r^2, for
// two pairs. 1/r^2 is the square of the reciprocal root corrected by one Newton step, so that
// it is as exact as the division it stands for.
template <int ELEC>
__device__ __forceinline__ void pair_derivs2(float2 r2, float2 sig, float2 eps24, float2 qq,
                                             const PairConst& pc, float2& p1, float2& c2) {
    const float2 ir = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
    float2 ir2 = mul2(ir, ir);
    ir2 = fma2(ir2, fma2(neg2(r2), ir2, dup2(1.0f)), ir2);
    const float2 sig2 = mul2(sig, sig);
    const float2 s2 = mul2(sig2, ir2);
    const float2 s6 = mul2(mul2(s2, s2), s2);
    const float2 s12 = mul2(s6, s6);
    const float2 ei = mul2(eps24, ir2);
    p1 = mul2(ei, fma2(dup2(-2.0f), s12, s6));                   // LJ phi'/r
    float2 pp = mul2(ei, fma2(dup2(26.0f), s12, mul2(dup2(-7.0f), s6)));  // LJ phi''
    const float2 k2 = mul2(sig2, dup2(pc.inv_rc2));
    const float2 c6 = mul2(mul2(k2, k2), k2);
    const float2 a_ljc = mul2(mul2(eps24, c6), fma2(dup2(2.0f), c6, dup2(-1.0f)));
    float2 cc = dup2(0.0f);
    if (ELEC == ELEC_DDIEL) {        // phi = (qq/2) / r^2
        const float2 t = mul2(mul2(qq, ir2), ir2);
        p1 = fma2(dup2(-1.0f), t, p1);
        pp = fma2(dup2(3.0f), t, pp);
        cc = mul2(qq, dup2(pc.inv_rc3));
    } else if (ELEC == ELEC_RF) {    // phi = qq (1/r + krf r^2 - crf)
        const float2 ir3 = mul2(ir2, ir);
        p1 = fma2(qq, fma2(dup2(-1.0f), ir3, dup2(2.0f * pc.krf)), p1);
        pp = fma2(qq, fma2(dup2(2.0f), ir3, dup2(2.0f * pc.krf)), pp);
        cc = mul2(qq, dup2(fmaf(pc.inv_rc2, 1.0f, -2.0f * pc.krf * pc.rc)));
    } else if (ELEC == ELEC_PLAIN) { // phi = qq / r
        const float2 t = mul2(qq, mul2(ir2, ir));
        p1 = fma2(dup2(-1.0f), t, p1);
        pp = fma2(dup2(2.0f), t, pp);
        cc = mul2(qq, dup2(pc.inv_rc2));
    }
    p1 = fma2(fma2(a_ljc, dup2(pc.inv_rc), cc), ir, p1);  // phi_sf' = phi' - phi'(rc)
    c2 = mul2(fma2(dup2(-1.0f), p1, pp), ir2);
}

// The pairs of two atoms per lane (j0, j1; dead: the far slot) with the 8 atoms of block I: at
// iteration t lane l takes block atom (l & 7) ^ t against both. The i sums move by one xor
// exchange per iteration and component within a quarter warp and come home with the last; the
// j sums stay in the lane. xm: exclusion bits by block atom (low byte j0, next j1).
template <int ELEC>
__device__ __forceinline__ void hvp_chunk(const HvpShared& sm, const PairConst& pc, int I, int j0,
                                          int j1, bool live0, bool live1, unsigned xm, int lane) {
    const int l8 = lane & 7;
    const float4 xa = sm.xq[j0], xb = sm.xq[j1], va = sm.vq[j0], vb = sm.vq[j1];
    const float2 la = sm.lj[j0], lb = sm.lj[j1];
    float hix = 0.f, hiy = 0.f, hiz = 0.f;
    float2 hx = dup2(0.f), hy = dup2(0.f), hz = dup2(0.f);
#pragma unroll 2
    for (int t = 0; t < 8; ++t) {
        const int a = l8 ^ t, i = 8 * I + a;
        const float4 xi = sm.xq[i], vi = sm.vq[i];
        const float2 li = sm.lj[i];
        const float2 dx = make_float2(xa.x - xi.x, xb.x - xi.x), dy = make_float2(xa.y - xi.y, xb.y - xi.y),
                     dz = make_float2(xa.z - xi.z, xb.z - xi.z);
        const float2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
        const bool ok0 = live0 && r2.x < pc.rc2 && !((xm >> a) & 1u);
        const bool ok1 = live1 && r2.y < pc.rc2 && !((xm >> (8 + a)) & 1u);
        float2 p1, c2;
        pair_derivs2<ELEC>(r2, make_float2(li.x + la.x, li.x + lb.x), make_float2(li.y * la.y, li.y * lb.y),
                           make_float2(xi.w * xa.w, xi.w * xb.w), pc, p1, c2);
        const float2 wx = make_float2(va.x - vi.x, vb.x - vi.x), wy = make_float2(va.y - vi.y, vb.y - vi.y),
                     wz = make_float2(va.z - vi.z, vb.z - vi.z);
        float2 c1 = mul2(c2, fma2(dx, wx, fma2(dy, wy, mul2(dz, wz))));
        c1 = make_float2(ok0 ? c1.x : 0.f, ok1 ? c1.y : 0.f);
        p1 = make_float2(ok0 ? p1.x : 0.f, ok1 ? p1.y : 0.f);
        const float2 ax = fma2(c1, dx, mul2(p1, wx)), ay = fma2(c1, dy, mul2(p1, wy)),
                     az = fma2(c1, dz, mul2(p1, wz));
        hx = add2(hx, ax);
        hy = add2(hy, ay);
        hz = add2(hz, az);
        hix -= ax.x + ax.y;
        hiy -= ay.x + ay.y;
        hiz -= az.x + az.y;
        const int m = t < 7 ? t ^ (t + 1) : 7;  // to the lane that takes atom i next
        hix = __shfl_xor_sync(kFullMask, hix, m);
        hiy = __shfl_xor_sync(kFullMask, hiy, m);
        hiz = __shfl_xor_sync(kFullMask, hiz, m);
    }
    if (live0) hadd(sm, j0, hx.x, hy.x, hz.x);
    if (live1) hadd(sm, j1, hx.y, hy.y, hz.y);
    // the four quarters' shares of the block's atoms (FP32, a fixed order)
    hix += __shfl_xor_sync(kFullMask, hix, 8);
    hiy += __shfl_xor_sync(kFullMask, hiy, 8);
    hiz += __shfl_xor_sync(kFullMask, hiz, 8);
    hix += __shfl_xor_sync(kFullMask, hix, 16);
    hiy += __shfl_xor_sync(kFullMask, hiy, 16);
    hiz += __shfl_xor_sync(kFullMask, hiz, 16);
    if (lane < 8) hadd(sm, 8 * I + lane, hix, hiy, hiz);
}

__device__ void hvp_bond(const HvpShared& sm, const TopoDev& tp, int b) {
    const int2 ij = tp.bond_ij[b];
    const float2 par = tp.bond_par[b];
    const float4 a = sm.xq[ij.x], c = sm.xq[ij.y];
    const float4 va = sm.vq[ij.x], vc = sm.vq[ij.y];
    const float dx = c.x - a.x, dy = c.y - a.y, dz = c.z - a.z;
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float r = sqrtf(r2);
    const float p1 = par.y * (r - par.x) / r;  // phi'/r
    const float wx = vc.x - va.x, wy = vc.y - va.y, wz = vc.z - va.z;
    const float dw = fmaf(dx, wx, fmaf(dy, wy, dz * wz));
    const float c1 = (par.y - p1) * dw / r2;
    const float ax = fmaf(c1, dx, p1 * wx), ay = fmaf(c1, dy, p1 * wy), az = fmaf(c1, dz, p1 * wz);
    hadd(sm, ij.y, ax, ay, az);
    hadd(sm, ij.x, -ax, -ay, -az);
}

__device__ __forceinline__ float3 f3(float x, float y, float z) { return make_float3(x, y, z); }
__device__ __forceinline__ float dot3(float3 a, float3 b) { return fmaf(a.x, b.x, fmaf(a.y, b.y, a.z * b.z)); }
__device__ __forceinline__ float3 cross3(float3 a, float3 b) {
    return f3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float3 lin(float a, float3 x, float b, float3 y) {
    return f3(fmaf(a, x.x, b * y.x), fmaf(a, x.y, b * y.y), fmaf(a, x.z, b * y.z));
}

__device__ void hvp_angle(const HvpShared& sm, const TopoDev& tp, int q) {
    const int4 ijk = tp.ang_ijk[q];
    const float2 par = tp.ang_par[q];
    const float4 A = sm.xq[ijk.x], B = sm.xq[ijk.y], Cc = sm.xq[ijk.z];
    const float4 VA = sm.vq[ijk.x], VB = sm.vq[ijk.y], VC = sm.vq[ijk.z];
    const float3 u = f3(A.x - B.x, A.y - B.y, A.z - B.z), w = f3(Cc.x - B.x, Cc.y - B.y, Cc.z - B.z);
    const float3 du = f3(VA.x - VB.x, VA.y - VB.y, VA.z - VB.z);
    const float3 dw = f3(VC.x - VB.x, VC.y - VB.y, VC.z - VB.z);
    const float3 c = cross3(u, w);
    const float sn = sqrtf(dot3(c, c));
    const float cs = dot3(u, w);
    const float ru2 = dot3(u, u), rw2 = dot3(w, w);
    const float dth = atan2f(sn, cs) - par.x;
    // grad theta: G_i = (cs u / |u|^2 - w) / sn, G_k = (cs w / |w|^2 - u) / sn, G_j = -(G_i + G_k)
    const float isn = 1.0f / sn;
    const float3 Gi = lin(cs / ru2 * isn, u, -isn, w);
    const float3 Gk = lin(cs / rw2 * isn, w, -isn, u);
    // directional derivatives along v
    const float dcs = dot3(du, w) + dot3(u, dw);
    const float3 dc = f3(cross3(du, w).x + cross3(u, dw).x, cross3(du, w).y + cross3(u, dw).y,
                         cross3(du, w).z + cross3(u, dw).z);
    const float dsn = dot3(c, dc) * isn;
    const float dru2 = 2.0f * dot3(u, du), drw2 = 2.0f * dot3(w, dw);
    const float ai = (dcs / ru2 - cs * dru2 / (ru2 * ru2)) * isn;
    const float ak = (dcs / rw2 - cs * drw2 / (rw2 * rw2)) * isn;
    const float3 dGi = f3(ai * u.x + (cs / ru2) * isn * du.x - isn * dw.x - Gi.x * dsn * isn,
                          ai * u.y + (cs / ru2) * isn * du.y - isn * dw.y - Gi.y * dsn * isn,
                          ai * u.z + (cs / ru2) * isn * du.z - isn * dw.z - Gi.z * dsn * isn);
    const float3 dGk = f3(ak * w.x + (cs / rw2) * isn * dw.x - isn * du.x - Gk.x * dsn * isn,
                          ak * w.y + (cs / rw2) * isn * dw.y - isn * du.y - Gk.y * dsn * isn,
                          ak * w.z + (cs / rw2) * isn * dw.z - isn * du.z - Gk.z * dsn * isn);
    // grad theta . v with G_j = -(G_i + G_k): G_i.(v_i - v_j) + G_k.(v_k - v_j)
    const float gv = dot3(Gi, du) + dot3(Gk, dw);
    const float k = par.y;
    const float3 hi = lin(k * gv, Gi, k * dth, dGi);
    const float3 hk = lin(k * gv, Gk, k * dth, dGk);
    // the centre gets -(H v)_i - (H v)_k since G_j = -(G_i + G_k) and D_v G_j = -(D_v G_i + D_v G_k)
    hadd(sm, ijk.x, hi.x, hi.y, hi.z);
    hadd(sm, ijk.z, hk.x, hk.y, hk.z);
    hadd(sm, ijk.y, -(hi.x + hk.x), -(hi.y + hk.y), -(hi.z + hk.z));
}

}  // namespace

template <int CL>
__device__ __forceinline__ void hvp_cluster_sync() {
    if (CL == 1)
        __syncthreads();
    else
        cg::this_cluster().sync();
}

template <int ELEC, int CL>
__global__ void __launch_bounds__(1024)
k_hvp_frames(const TopoDev* __restrict__ topo_ptr, RunParams P, const float* __restrict__ X,
             const float* V, float* HV, int nta, int split) {  // (HV may be V)
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int next_row, n_units;
    __shared__ int upre[kHvpMaxBlocks];  // first work unit of each row of blocks
    const TopoDev tp = *topo_ptr;
    const int n = tp.n_atoms, nbs = nta / 8;
    HvpShared sm;
    char* p = (char*)smem_raw;
    sm.nta = nta;
    sm.xq = (float4*)p; p += sizeof(float4) * nta;
    sm.vq = (float4*)p; p += sizeof(float4) * nta;
    sm.blo = (float4*)p; p += sizeof(float4) * nbs;
    sm.bhi = (float4*)p; p += sizeof(float4) * nbs;
    sm.ex = (unsigned long long*)p; p += sizeof(unsigned long long) * nta;
    sm.H = (int*)p; p += sizeof(int) * 3 * nta;
    sm.L1 = (unsigned*)p; p += sizeof(unsigned) * 3 * nta;
    sm.L0 = (unsigned*)p; p += sizeof(unsigned) * 3 * nta;
    sm.lj = (float2*)p; p += sizeof(float2) * nta;
    sm.buf = (uint16_t*)p + (threadIdx.x >> 5) * 8 * kHvpSeg;
    const long long f = blockIdx.x / CL;
    const int rank = CL == 1 ? 0 : (int)cg::this_cluster().block_rank();
    const float* xf = X + f * n * 3;
    const float* vf = V + f * n * 3;
    for (int i = threadIdx.x; i < nta; i += blockDim.x) {
        if (i < n) {
            sm.xq[i] = make_float4(xf[3 * i], xf[3 * i + 1], xf[3 * i + 2], tp.qs[i]);
            sm.vq[i] = make_float4(vf[3 * i], vf[3 * i + 1], vf[3 * i + 2], 0.f);
            sm.lj[i] = tp.lj[i];
            sm.ex[i] = tp.excl[i];
        } else {
            sm.xq[i] = make_float4(1.0e5f * (float)(i + 1), 0.f, 0.f, 0.f);
            sm.vq[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            sm.lj[i] = make_float2(0.f, 0.f);
            sm.ex[i] = 0ull;
        }
    }
    for (int i = threadIdx.x; i < 3 * nta; i += blockDim.x) {
        sm.H[i] = 0;
        sm.L1[i] = 0u;
        sm.L0[i] = 0u;
    }
    if (threadIdx.x == 0) next_row = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int l8 = lane & 7, q = lane >> 3;
    for (int b0 = 4 * warp; b0 < nbs; b0 += 4 * nw) {  // block boxes (valid atoms only)
        const int b = b0 + q;
        const int a = 8 * b + l8;
        const bool valid = b < nbs && a < n;
        const float4 x = valid ? sm.xq[a] : make_float4(0.f, 0.f, 0.f, 0.f);
        float lx = valid ? x.x : 3.0e38f, ly = valid ? x.y : 3.0e38f, lz = valid ? x.z : 3.0e38f;
        float hx = valid ? x.x : -3.0e38f, hy = valid ? x.y : -3.0e38f, hz = valid ? x.z : -3.0e38f;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            lx = fminf(lx, __shfl_xor_sync(kFullMask, lx, o));
            ly = fminf(ly, __shfl_xor_sync(kFullMask, ly, o));
            lz = fminf(lz, __shfl_xor_sync(kFullMask, lz, o));
            hx = fmaxf(hx, __shfl_xor_sync(kFullMask, hx, o));
            hy = fmaxf(hy, __shfl_xor_sync(kFullMask, hy, o));
            hz = fmaxf(hz, __shfl_xor_sync(kFullMask, hz, o));
        }
        if (l8 == 0 && b < nbs) {
            sm.blo[b] = make_float4(lx, ly, lz, 0.f);
            sm.bhi[b] = make_float4(hx, hy, hz, 0.f);
        }
    }
    __syncthreads();
    const int t0 = threadIdx.x * CL + rank, tstep = blockDim.x * CL;
    for (int b = t0; b < tp.n_bonds; b += tstep) hvp_bond(sm, tp, b);
    for (int a = t0; a < tp.n_angles; a += tstep) hvp_angle(sm, tp, a);
    // work units: the rows of blocks I with I % CL == rank, each cut into segments of kHvpSeg
    // candidate blocks J >= I (long rows first); a warp pulls a unit, tests its blocks
    // against I's box and their atoms against I's, and takes the hits 64 at a time. In a cluster
    // `split` warps may share a unit: each makes the tests and takes its chunks of 64 (the
    // same chunks, so the same sums)
    const int parts = CL == 1 ? 1 : split;
    if (warp == 0) {
        int run = 0;
        for (int r0 = 0; r0 < nbs; r0 += 32) {
            const int I = r0 + lane;
            const int ns = (I < nbs && I % CL == rank) ? (nbs - I + kHvpSeg - 1) / kHvpSeg : 0;
            int x = ns;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(kFullMask, x, o);
                if (lane >= o) x += y;
            }
            if (I < nbs) upre[I] = run + x - ns;  // first unit of row I
            run += __shfl_sync(kFullMask, x, 31);
        }
        if (lane == 0) n_units = run;
    }
    __syncthreads();
    for (;;) {
        int u = 0;
        if (lane == 0) u = atomicAdd(&next_row, 1);
        u = __shfl_sync(kFullMask, u, 0);
        if (u >= n_units * parts) break;
        const int part = u % parts;
        u /= parts;
        int lo = 0, hi = nbs;  // the last row whose first unit is <= u
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (upre[mid] <= u) lo = mid; else hi = mid;
        }
        int I = lo;
        while (I % CL != rank) --I;  // rows of the other CTA own no units here
        const int j0 = I + kHvpSeg * (u - upre[I]);
        const float4 al = sm.blo[I], ah = sm.bhi[I];
        if (!(al.x <= ah.x)) continue;  // no atoms in block I (warp-uniform)
        const int J = j0 + lane;
        bool hit = false;
        if (J < nbs) {
            const float4 bl = sm.blo[J], bh = sm.bhi[J];
            const float gx = fmaxf(0.f, fmaxf(al.x - bh.x, bl.x - ah.x));
            const float gy = fmaxf(0.f, fmaxf(al.y - bh.y, bl.y - ah.y));
            const float gz = fmaxf(0.f, fmaxf(al.z - bh.z, bl.z - ah.z));
            hit = bl.x <= bh.x && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < P.pc.rc2;
        }
        unsigned m = __ballot_sync(kFullMask, hit);
        const unsigned lt = (1u << lane) - 1u;
        int count = 0;
        while (m) {  // four hit blocks at a time, one atom per lane: those within r_c of an atom of I
            unsigned mm = m;
            for (int k = 0; k < q; ++k) mm &= mm - 1u;
            const int src = __ffs(mm) - 1;
            m &= m - 1u;
            m &= m - 1u;
            m &= m - 1u;
            m &= m - 1u;
            const int j = src >= 0 ? 8 * (j0 + src) + l8 : n;
            bool near = false;
            if (j < n) {
                const float4 xj = sm.xq[j];
                float dmin = 3.0e38f;
#pragma unroll
                for (int a = 0; a < 8; ++a) {  // (empty slots sit far away)
                    const float4 xi = sm.xq[8 * I + a];
                    const float dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
                    dmin = fminf(dmin, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
                }
                near = dmin < P.pc.rc2;
            }
            const unsigned nm = __ballot_sync(kFullMask, near);
            if (near) sm.buf[count + __popc(nm & lt)] = (uint16_t)j;
            count += __popc(nm);
        }
        __syncwarp();
        for (int k0 = 64 * part; k0 < count; k0 += 64 * parts) {
            const int k = k0 + 2 * lane;
            const bool live0 = k < count, live1 = k + 1 < count;
            const int ja = live0 ? sm.buf[k] : 8 * I, jb = live1 ? sm.buf[k + 1] : 8 * I;
            // excluded pairs, and the pairs of block I with itself once (j after i)
            unsigned xm = 0u;
            if (sm.buf[k0] < 8 * I + 8 + kExclWindow) {
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    const int i = 8 * I + a;
                    const unsigned long long ex = sm.ex[i];
                    const int da = ja - i + kExclWindow, db = jb - i + kExclWindow;
                    if (ja <= i || (da < 2 * kExclWindow && ((ex >> da) & 1ull))) xm |= 1u << a;
                    if (jb <= i || (db < 2 * kExclWindow && ((ex >> db) & 1ull))) xm |= 256u << a;
                }
            }
            hvp_chunk<ELEC>(sm, P.pc, I, ja, jb, live0, live1, xm, lane);
        }
        __syncwarp();  // (the next unit overwrites the buffer)
    }
    hvp_cluster_sync<CL>();  // every partial of the cluster is complete
    float* out = HV + f * n * 3;
    for (int k = threadIdx.x + rank * blockDim.x; k < 3 * n; k += CL * blockDim.x) {
        long long h = sm.H[k], l0 = sm.L0[k];
        unsigned l1 = sm.L1[k];
#pragma unroll
        for (int r = 1; r < CL; ++r) {
            const unsigned p = (unsigned)((rank + r) & (CL - 1));
            h += cg::this_cluster().map_shared_rank(sm.H, p)[k];
            l0 += cg::this_cluster().map_shared_rank(sm.L0, p)[k];
            l1 += cg::this_cluster().map_shared_rank(sm.L1, p)[k];
        }
        out[k] = fix2f((join_coarse(h, l1, 22) << 20) + l0);
    }
    hvp_cluster_sync<CL>();  // no CTA leaves while its shared memory may still be read
}

size_t hvp_smem_bytes(int nta, int threads) {
    const int nbs = nta / 8;
    return sizeof(float4) * 2 * nta + sizeof(float4) * 2 * nbs + sizeof(unsigned long long) * nta +
           (sizeof(int) + 2 * sizeof(unsigned)) * 3 * (size_t)nta + sizeof(float2) * nta +
           sizeof(uint16_t) * 8 * kHvpSeg * (threads / 32);
}

template <int ELEC, int CL>
static cudaError_t launch_hvp_t(const TopoDev* topo, const RunParams& P, const float* X,
                                const float* V, float* HV, long long n_frames, int nta, int threads,
                                cudaStream_t s) {
    // A small chain has fewer units than a cluster has warps, and the longest sets the time: 4
    // frames of 160 atoms 16.6 -> 13.1 us, of 304 20.6 -> 16.4; 28 frames (four CTAs) 16.9 -> 13.7 and
    // 21.7 -> 19.2; 76 frames of 304 atoms (two CTAs) 25.4 -> 23.2. With 560 atoms the tests made
    // more than once cost more (27.8 -> 33.8).
    const int split = nta > 320 ? 1 : CL >= 4 ? 4 : 2;
    const size_t smem = hvp_smem_bytes(nta, threads);
    auto kern = k_hvp_frames<ELEC, CL>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_frames * CL));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kern, topo, P, X, V, HV, nta, split);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// Threads of a lone CTA: a chain has as many work units as 8-atom blocks, or a few more, so that
// many threads of a small one only wait at its barriers and keep other frames off the SM. 1000
// frames of 17 atoms 32.3 us with 512 threads, 19.2 with 256, 13.5 with 128; of 44 atoms 36.0,
// 25.0, 21.2 (but 200 frames 11.2, 10.9, 13.5); of 100 atoms 60.9, 49.0; of 160 atoms 83.3, 79.1
// (200 frames 25.9, 30.4).
static int lone_threads(long long n_frames, int nta, int n_sm) {
    if (nta <= 32) return 128;
    if (nta <= 64) return 256;
    if (n_frames <= n_sm) return nta <= 128 ? 512 : 1024;
    return nta <= 128 ? 256 : 512;
}

// Few frames: a cluster of 1024-thread CTAs per frame, so that the frames spread over the
// SMs; many frames, or small ones (28 frames of 44 atoms 9.3 us with one CTA, 10.9 with two or four;
// of 100 atoms 13.0, and 12.1 with four; of 200 atoms 21.8, and 15.1 with four): one CTA each.
template <int ELEC>
static cudaError_t launch_hvp_e(const TopoDev* topo, const RunParams& P, const float* X,
                                const float* V, float* HV, long long n_frames, int nta,
                                cudaStream_t s) {
    int dev = 0, n_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int lone = lone_threads(n_frames, nta, n_sm);
    if (nta <= 64) return launch_hvp_t<ELEC, 1>(topo, P, X, V, HV, n_frames, nta, lone, s);
    if (10 * n_frames <= n_sm) return launch_hvp_t<ELEC, 8>(topo, P, X, V, HV, n_frames, nta, 1024, s);
    if (5 * n_frames <= n_sm) return launch_hvp_t<ELEC, 4>(topo, P, X, V, HV, n_frames, nta, 1024, s);
    if (2 * n_frames <= n_sm) return launch_hvp_t<ELEC, 2>(topo, P, X, V, HV, n_frames, nta, 1024, s);
    return launch_hvp_t<ELEC, 1>(topo, P, X, V, HV, n_frames, nta, lone, s);
}

cudaError_t launch_hvp(int elec, const TopoDev* topo, const RunParams& P, const float* X,
                       const float* V, float* HV, long long n_frames, int nta, cudaStream_t s) {
    switch (elec) {
        case ELEC_DDIEL: return launch_hvp_e<ELEC_DDIEL>(topo, P, X, V, HV, n_frames, nta, s);
        case ELEC_RF: return launch_hvp_e<ELEC_RF>(topo, P, X, V, HV, n_frames, nta, s);
        case ELEC_PLAIN: return launch_hvp_e<ELEC_PLAIN>(topo, P, X, V, HV, n_frames, nta, s);
        default: return launch_hvp_e<ELEC_NONE>(topo, P, X, V, HV, n_frames, nta, s);
    }
}

}  // namespace scps
