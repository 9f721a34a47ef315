// Resident rMD step kernel for chain replicas, and the frame evaluator.
//
// One thread-block cluster of CL CTAs (1, 2, 4 or 8) owns one replica for a
// whole launch of n_steps steps. Positions, velocities and fixed-point force
// partials live in shared memory; the CTAs of a cluster split the force work
// between them (the warps of each CTA pull their items from a counter in their
// own shared memory) and read each other's partials through distributed shared
// memory. Every step evaluates
//   bonded terms + non-bonded pairs from a pair list              -grad U
//   z(X) of Eq. (zrMD) from C_ij of Eq. (Cij) in float-float     collective coordinate
//   ratchet of Eq. (FrMD) in FP64 (z < z_m: z_m = z, no bias)   bias force
//   BAOAB update with Philox4x32-10 noise (Eq. Lang)
// and writes a frame every save_interval steps. Each CTA of a cluster integrates a
// share of the atoms and writes their new positions into every CTA's copy.
//
// Pair list. Atoms are grouped in blocks of 8 consecutive chain atoms. For each
// block I the list holds, in ascending order, every atom j of a later block that
// lies within r_list = r_c + skin of some atom of I, in chunks of 16 (the last one
// padded with a far-away sentinel slot). A work item is one block against one
// chunk (128 pairs) on a quarter warp: lane l keeps entries 2 l and 2 l + 1 of the chunk
// and takes block atom l ^ t against both at its iteration t, two FP32 pairs per packed
// operation, so the i-force accumulators move by one xor exchange per iteration while the
// j-forces stay in place (64 replicas x 560 atoms: 18.9 us per step; these items alone took it
// from 26.7, with chunks of 8, one entry per lane and scalar operations, to 21.8; the same bits). Pairs inside a block form 28-pair
// items of their own. The list is rebuilt when a bound on the largest displacement
// since the last build reaches skin/2, or after rebuild_every steps, so no pair
// inside r_c is ever missing.
//
// Summation. Every pair term s (x_j - x_i) is rounded to an integer multiple of
// 2^-13 kJ mol^-1 nm^-1 and summed in integers, bonded terms likewise, bias-gradient
// terms to 2^-20 units. The shared-memory partials are sums modulo 2^32, added with
// 32-bit atomics, with coarse sums of the large terms beside them that fix the total, so
// every sum is exact and independent of the order of the additions. Results are
// therefore the same bits whichever warp or CTA takes an item, whatever the list
// skin or rebuild cadence, and across a checkpoint and resume.
#pragma once

#include <cooperative_groups.h>

#include <algorithm>
#include <climits>

#include "scps_internal.h"

namespace cg = cooperative_groups;

namespace scps {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr unsigned kNonFinite = 0xffffffffu;  // Scalars::vmax2: beyond the bits of any float
constexpr int kFlagGradCoarse = 256;  // Scalars::flag: coarse words of G were touched
constexpr float kForceLimit13 = 8.192e12f;  // 1e9 kJ mol^-1 nm^-1 in 2^-13 units
constexpr int kChunk = 32;    // contacts / bonds / angles per work item (one per lane)

extern __shared__ __align__(16) unsigned char smem_raw[];

// A pair item held in shared memory: descriptor, exclusion masks and the chunk's entries
// (the same data as the global item table, mask table and j entries, without their latency).
struct __align__(16) CacheItem {
    uint32_t desc, pad[3];
    uint8_t xm[kListChunk];
    uint16_t j[kListChunk];
};

// Partials of one kind and parity: per atom slot three modular words, then, after those of all
// slots, three coarse words per slot (see red3).
struct Part {
    unsigned* L;
    int* H;
};

// Shared-memory arrays of one CTA, laid out from smem_raw by the slot count alone (every
// address is an offset computed from nta, so that no pointers stay in registers). Atom slots:
// nta real or padding slots plus 8 sentinel slots (a block far from everything) that absorb
// the padding of list chunks. For both parities of the evaluated step, F: force partials of
// this CTA in 2^-13 units; G: partials of sum_p (C - C0) C'(u) (x_p - x_i) over the native
// contacts this CTA evaluated, in 2^-20 units (the bias gradient without its ratchet factor,
// known only once z is complete).
struct Shared {
    int nta;       // atom slots
    int lc_cap;    // capacity of lc in items
    int fsh, gsh;  // coarse units of the F and G partials (TopoDev)
    __device__ __forceinline__ int na8() const { return nta + 8; }
    // positions with scaled charges, nta + 8
    __device__ __forceinline__ float4* xq() const { return (float4*)smem_raw; }
    // LJ parameters (sigma/2, sqrt(24 eps)), nta + 8
    __device__ __forceinline__ float2* lj() const { return (float2*)(smem_raw + 16 * na8()); }
    // velocities (w: 1/m), nta
    __device__ __forceinline__ float4* v() const { return (float4*)(smem_raw + 24 * na8()); }
    // noise of the next O half step per atom (sd times Gaussian numbers); w: the atom's
    // |F_bias|^2 / m of the step just closed. During a list rebuild it holds the block boxes
    // and chunk counts instead.
    __device__ __forceinline__ float4* xi() const { return v() + nta; }
    __device__ __forceinline__ Part part(int k) const {
        Part p;
        p.L = (unsigned*)(smem_raw + 24 * na8() + 32 * nta + 24 * na8() * k);
        p.H = (int*)(p.L + 3 * na8());
        return p;
    }
    __device__ __forceinline__ Part F(int b) const { return part(b); }
    __device__ __forceinline__ Part G(int b) const { return part(2 + b); }
    // this CTA's pair items when they fit
    __device__ __forceinline__ CacheItem* lc() const {
        return (CacheItem*)(smem_raw + 120 * na8() + 32 * nta);
    }
};

// List slab of this replica or frame (see scps_internal.h for the layout).
struct ListDev {
    uint16_t* jl;               // j entries of all blocks
    uint32_t* items;            // this CTA's item table
    uint8_t* excl;              // exclusion masks, kListMasks bytes per block
    int nbs;                    // blocks of the slab layout (nta / 8)
};

struct Scalars {
    TopoDev tp;         // the replica's topology and list slab (shared memory: read where
    ListDev list;       // needed instead of held in registers)
    PairConst pc;       // for the slow path of a pair item
    int work_next[2];   // this CTA's work counter, by parity of the evaluated step
    int status;         // replica status (identical in every CTA of a cluster): written by this
                        // CTA's warp 0 alone, before the barrier that ends a decision
    int bias_on;
    int flag[2];        // force-range bits raised during the evaluation of a given parity
    int n_items;        // pair items in this CTA's item table
    int cached;         // 1: the items are held in shared memory (Shared::lc)
    int n_diag;         // blocks whose inner pairs this CTA evaluates
    int build_next;     // block counter of a list build
    unsigned vmax2[2];  // largest |v1|^2 + |v2|^2 of the update, by parity (float bits), or
                        // kNonFinite: some CTA's new state is not finite. Raised by every CTA
                        // before the barrier that closes the update, read only after it
    long long pair_slots;  // pairs one evaluation with the current list takes
    long long n_saved;
    double zm, z, epot, T;
    float kb;           // the bias force on an atom is kb times its bias gradient
    uint16_t cnt[kMaxChainAtoms / 8], cntn[kMaxChainAtoms / 8];  // list chunks per block, near ones
    unsigned zw[2][3];       // this CTA's share of z by parity: sums of its bits 0..19, 20..39 and
                             // 40 up (units of 2^-40), which 32-bit atomics add
    long long red_e[2][32];  // per-warp shares of the potential energy (units of 2^-20)
    // contact-map tube bias
    double sm, wm;                      // running minima of s_lambda and w_lambda
    float gam_sum;                      // sum_k gamma_k
    float gam[kMaxTubeK];               // gamma_k = dF/dD_k weights of the evaluated step
    int work_next2[2];                  // counter of the second work phase, by parity
    long long red_d[2][kMaxTubeK];      // this CTA's share of sum_p (C_p - A_kp)^2 (2^-40), by parity
};

__device__ __forceinline__ long long warp_sum_ll(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    return v;
}

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    return v;
}

// Adds an integer vector to the partials of slot k: the modular words always, the coarse
// words only when a component rounds to a non-zero multiple of 2^sh (rarely: one shared
// atomic per component instead of the two of an integer part and a fraction part; returns
// whether it did).
__device__ __forceinline__ bool red3(const Part& p, int k, int vx, int vy, int vz, int sh) {
    unsigned* L = p.L + 3 * k;
    atomicAdd(L, (unsigned)vx);
    atomicAdd(L + 1, (unsigned)vy);
    atomicAdd(L + 2, (unsigned)vz);
    const unsigned half = 1u << (sh - 1);
    if ((((unsigned)vx + half) | ((unsigned)vy + half) | ((unsigned)vz + half)) >> sh) {
        const int hx = ((vx >> (sh - 1)) + 1) >> 1, hy = ((vy >> (sh - 1)) + 1) >> 1,
                  hz = ((vz >> (sh - 1)) + 1) >> 1;
        int* H = p.H + 3 * k;
        if (hx) atomicAdd(H, hx);
        if (hy) atomicAdd(H + 1, hy);
        if (hz) atomicAdd(H + 2, hz);
        return true;
    }
    return false;
}

// The same for 64-bit components (the slow path of a pair item).
__device__ __forceinline__ void red3_64(const Part& p, int k, long long vx, long long vy,
                                        long long vz, int sh) {
    atomicAdd(p.L + 3 * k, (unsigned)vx);
    atomicAdd(p.L + 3 * k + 1, (unsigned)vy);
    atomicAdd(p.L + 3 * k + 2, (unsigned)vz);
    atomicAdd(p.H + 3 * k, (int)(((vx >> (sh - 1)) + 1) >> 1));
    atomicAdd(p.H + 3 * k + 1, (int)(((vy >> (sh - 1)) + 1) >> 1));
    atomicAdd(p.H + 3 * k + 2, (int)(((vz >> (sh - 1)) + 1) >> 1));
}

// Slow path of a pair term: s13 d (2^-13 units, rounded exactly as on the fast path, so the
// sums are the same integers whichever path a pair takes) to atom i and its negative to atom
// j, in 64-bit; a non-finite term or one above 1e9 kJ/mol/nm raises the force-range flag.
__device__ __forceinline__ void add_pair13(const Part& F, int* flag, int sh, int i, int j, float s13,
                                           float dx, float dy, float dz) {
    const float tx = s13 * dx, ty = s13 * dy, tz = s13 * dz;
    const float lim = kForceLimit13;
    if (!(fabsf(tx) <= lim && fabsf(ty) <= lim && fabsf(tz) <= lim)) atomicOr(flag, SCPS_FLAG_FORCE_RANGE);
    const long long qx = __float2ll_rn(tx), qy = __float2ll_rn(ty), qz = __float2ll_rn(tz);
    red3_64(F, i, qx, qy, qz, sh);
    red3_64(F, j, -qx, -qy, -qz, sh);
}

// Bonded terms: integer multiples of 2^-13 kJ mol^-1 nm^-1 (one conversion each); a term
// that is non-finite or beyond 2.6e5 kJ mol^-1 nm^-1 (a bond stretched by more than 1 nm)
// raises the force-range flag, which freezes the replica.
__device__ __forceinline__ void add_term13(const Shared& sm, const Part& F, int* flag, int i,
                                           float fx, float fy, float fz) {
    if (!(fmaxf(fabsf(fx), fmaxf(fabsf(fy), fabsf(fz))) < 2.6e5f) ||
        !(isfinite(fx) && isfinite(fy) && isfinite(fz)))
        atomicOr(flag, SCPS_FLAG_FORCE_RANGE);
    red3(F, i, __float2int_rn(fx * kPairScale), __float2int_rn(fy * kPairScale),
         __float2int_rn(fz * kPairScale), sm.fsh);
}

// Cluster helpers: CL == 1 degenerates to a plain CTA.
template <int CL>
__device__ __forceinline__ void cluster_barrier() {
    if (CL == 1)
        __syncthreads();
    else
        cg::this_cluster().sync();
}

template <int CL, class T>
__device__ __forceinline__ T* rank_ptr(T* p, int rank) {
    if (CL == 1) return p;
    return cg::this_cluster().map_shared_rank(p, (unsigned)rank);
}

template <int CL>
__device__ __forceinline__ int cta_rank() {
    if (CL == 1) return 0;
    return (int)cg::this_cluster().block_rank();
}

// ---------------------------------------------------------------------------
// Pair items
// ---------------------------------------------------------------------------

template <int CL>
__device__ __forceinline__ ListDev list_of(unsigned char* slab, int nta, int rank) {
    ListDev L;
    L.nbs = nta >> 3;
    L.jl = (uint16_t*)slab;
    const long long part = list_items_part(L.nbs, CL);  // items of one CTA of the cluster
    unsigned char* items = slab + list_jl_bytes(L.nbs);
    L.items = (uint32_t*)items + rank * part;
    L.excl = items + list_items_bytes(L.nbs);
    return L;
}

// The 128 pairs of one item (block I against a chunk of 16 list entries, of which this lane
// holds j0 and j1) on a quarter warp, fast path: at iteration t lane l takes block atom l ^ t
// against both entries, the two pairs in one packed operation. The sums of the block atoms
// move by one xor exchange per iteration and component, those of the entries stay in the
// lane; all are integers in 32-bit registers. Items near their block (NEARX) take the excluded
// pairs from the masks xm (low byte entry j0, high byte j1). Returns false (and adds nothing)
// when the integer sums of the item could overflow; the caller then takes the slow path. They
// cannot while every |s| of the quarter warp is up to pc.s_lim / 2 (16 terms for a block atom, 8
// for an entry), nor, looked at only where one is larger, while every |s| is up to pc.s_lim and
// the lanes' largest |s| add up to no more than 4 pc.s_lim (a block atom takes two terms from
// each lane). Close atoms mostly meet one at a time, and a launch waits for its slowest frame: 28
// frames of 44 atoms 16.5 -> 9.9 us, of 100 atoms 18.3 -> 12.0, against every item with an |s|
// beyond pc.s_lim / 2 on the slow path.
//
// Bound by the FMA pipe: 33 packed operations per two pairs, and next to it the XU pipe (two
// rsqrt, six conversions, 2.1 clocks each). Packing the two entries, which stay in registers,
// rather than two block atoms needs no register copies of (x, x) for the other operand: the
// six operations that meet the block atom are scalar ones.
template <int ELEC, bool ENERGY, bool NEARX>
__device__ __forceinline__ bool pair_item_fast(const Shared& sm, const Part& F,
                                               const PairConst& pc, int I, int j0, int j1,
                                               unsigned xm, int lane, long long& e18) {
    const int l8 = lane & 7, q = lane >> 3;
    const Entries n = pack_entries(sm.xq()[j0], sm.xq()[j1], sm.lj()[j0], sm.lj()[j1]);
    int fix = 0, fiy = 0, fiz = 0;
    int fax = 0, fay = 0, faz = 0, fbx = 0, fby = 0, fbz = 0;
    long long ei = 0;
    float most = 0.0f;  // largest |s| of this lane, times 2^13 (NaN: some pair's is)
    bool bad = false;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const int a = l8 ^ t, i = 8 * I + a;
        const float4 xi = sm.xq()[i];
        const float2 li = sm.lj()[i];
        const float2 dx = make_float2(n.x.x - xi.x, n.x.y - xi.x),
                     dy = make_float2(n.y.x - xi.y, n.y.y - xi.y),
                     dz = make_float2(n.z.x - xi.z, n.z.y - xi.z);
        const float2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
        bool ok0 = r2.x < pc.rc2, ok1 = r2.y < pc.rc2;
        if (NEARX) {
            ok0 = ok0 && !((xm >> a) & 1u);
            ok1 = ok1 && !((xm >> (8 + a)) & 1u);
        }
        const LJPair2 lj = lj_pair2(make_float2(li.x + n.s.x, li.x + n.s.y),
                                    make_float2(li.y * n.e.x, li.y * n.e.y), pc);
        float2 e;
        float2 ms = pair_ms2<ELEC, ENERGY>(r2, lj, make_float2(xi.w * n.q.x, xi.w * n.q.y), pc, &e);
        ms.x = ok0 ? ms.x : 0.0f;
        ms.y = ok1 ? ms.y : 0.0f;
        most = max_nan(most, max_nan(fabsf(ms.x), fabsf(ms.y)));
        const float2 fx = mul2(ms, dx), fy = mul2(ms, dy), fz = mul2(ms, dz);
        // (the terms come out negated: they are the entries' share)
        const int ax = __float2int_rn(fx.x), bx = __float2int_rn(fx.y);
        const int ay = __float2int_rn(fy.x), by = __float2int_rn(fy.y);
        const int az = __float2int_rn(fz.x), bz = __float2int_rn(fz.y);
        if (ENERGY) {  // (e comes scaled by 2^13)
            const float lim_e = kPairScale * kPairEMax, se = kPairEScale / kPairScale;
            bad = bad || (ok0 && !(fabsf(e.x) < lim_e)) || (ok1 && !(fabsf(e.y) < lim_e));
            ei += (ok0 ? __float2int_rn(e.x * se) : 0) + (ok1 ? __float2int_rn(e.y * se) : 0);
        }
        fax += ax;
        fay += ay;
        faz += az;
        fbx += bx;
        fby += by;
        fbz += bz;
        fix -= ax + bx;
        fiy -= ay + by;
        fiz -= az + bz;
        if (t < 7) {  // the sums of block atom l8 ^ t go to the lane that takes it next
            fix = __shfl_xor_sync(kFull, fix, t ^ (t + 1));
            fiy = __shfl_xor_sync(kFull, fiy, t ^ (t + 1));
            fiz = __shfl_xor_sync(kFull, fiz, t ^ (t + 1));
        }
    }
    const float lim = kPairScale * pc.s_lim;
    unsigned over = __ballot_sync(kFull, bad || !(most <= 0.5f * lim));
    if (over) {
        float sum = most;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) sum += __shfl_xor_sync(kFull, sum, o);
        over = __ballot_sync(kFull, bad || !(most <= lim) || !(sum <= 4.0f * lim));
        if ((over >> (8 * q)) & 0xffu) return false;
    }
    red3(F, 8 * I + (l8 ^ 7), fix, fiy, fiz, sm.fsh);  // lane l ends with atom l ^ 7's sums
    red3(F, j0, fax, fay, faz, sm.fsh);
    red3(F, j1, fbx, fby, fbz, sm.fsh);
    if (ENERGY) e18 += ei;
    return true;
}

// Slow path of an item: the same pairs with 64-bit sums (rounded per pair as on the fast path) and
// the range check (a force beyond 1e9 kJ/mol/nm or a non-finite one freezes the replica). As
// there, the block atoms' sums move from lane to lane and the entries' stay, and each goes to the
// partials once. Its first call in a launch costs about 5 us (it is small, and reads the pair
// constants and masks from shared memory, so that little has to come from far: 8 us with them
// read from the launch parameters and tables and with atomics for every pair).
template <int ELEC, bool ENERGY>
__device__ __noinline__ long long pair_item_slow(Shared sm, int b, Scalars* sc, int I, int j0, int j1,
                                                 unsigned xm) {
    const int l8 = threadIdx.x & 7;
    const unsigned quarter = 0xffu << (threadIdx.x & 24);  // (the quarter's lanes all come here)
    const Part F = sm.F(b);
    const PairConst& pc = sc->pc;
    long long e18 = 0;
    bool out = false;
#pragma unroll 1
    for (int u = 0; u < 2; ++u) {
        const int j = u ? j1 : j0;
        const float4 xj = sm.xq()[j];
        const float2 lj = sm.lj()[j];
        long long fi[3] = {}, fj[3] = {};
#pragma unroll 1
        for (int t = 0; t < 8; ++t) {
            const int a = l8 ^ t, i = 8 * I + a;
            const float4 xi = sm.xq()[i];
            const float2 li = sm.lj()[i];
            const float dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            if (r2 < pc.rc2 && !((xm >> (8 * u + a)) & 1u)) {
                float e = 0.f;
                const float s13 = kPairScale * pair_s<ELEC, ENERGY>(r2, li.x + lj.x, li.y * lj.y,
                                                                    xi.w * xj.w, pc, &e);
                const float f[3] = {s13 * dx, s13 * dy, s13 * dz};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const long long q = __float2ll_rn(f[c]);
                    out = out || !(fabsf(f[c]) <= kForceLimit13);
                    fi[c] += q;
                    fj[c] -= q;
                }
                if (ENERGY) e18 += __float2ll_rn(e * kPairEScale);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) fi[c] = __shfl_xor_sync(quarter, fi[c], (t ^ (t + 1)) & 7);
        }
        red3_64(F, 8 * I + l8, fi[0], fi[1], fi[2], sm.fsh);  // (the last exchange brought them home)
        red3_64(F, j, fj[0], fj[1], fj[2], sm.fsh);
    }
    if (out) atomicOr(&sc->flag[b], SCPS_FLAG_FORCE_RANGE);
    return e18;
}

// One batch of four pair items (one per quarter warp) from this CTA's item table.
template <int ELEC, bool ENERGY>
__device__ __forceinline__ void pair_batch(const Shared& sm, Scalars& sc, const RunParams& P, int b,
                                           int batch, int lane, long long& e18) {
    const int it = 4 * batch + (lane >> 3), l8 = lane & 7;
    int I = 0;  // idle quarter: block 0 against the far sentinel slot (zero terms)
    unsigned jj = (unsigned)sm.nta * 0x10001u, xm = 0u;
    bool near = false;
    if (it < sc.n_items) {
        if (sc.cached) {
            const CacheItem& c = sm.lc()[it];
            const uint32_t d = c.desc;
            I = (int)(d >> 17);
            near = (d >> 16) & 1u;
            jj = ((const unsigned*)c.j)[l8];
            if (near) xm = ((const uint16_t*)c.xm)[l8];
        } else {
            const ListDev& L = sc.list;
            const uint32_t d = __ldcg(L.items + it);
            I = (int)(d >> 17);
            near = (d >> 16) & 1u;
            jj = __ldcg((const unsigned*)(L.jl + list_jl_off(L.nbs, I) + kListChunk * (int)(d & 0xffffu)) + l8);
            if (near)
                xm = __ldcg((const uint16_t*)(L.excl + kListMasks * I + kListChunk * (int)(d & 0xffffu)) + l8);
        }
    }
    const int j0 = (int)(jj & 0xffffu), j1 = (int)(jj >> 16);
    const Part F = sm.F(b);
    bool done;
    if (__any_sync(kFull, near))
        done = pair_item_fast<ELEC, ENERGY, true>(sm, F, P.pc, I, j0, j1, xm, lane, e18);
    else
        done = pair_item_fast<ELEC, ENERGY, false>(sm, F, P.pc, I, j0, j1, 0u, lane, e18);
    if (!done) {
        const long long es = pair_item_slow<ELEC, ENERGY>(sm, b, &sc, I, j0, j1, near ? xm : 0u);
        if (ENERGY) e18 += es;
    }
}

// The 28 pairs inside block I on a quarter warp: at round k = 1..4 lane l takes the pair
// (l, (l + k) & 7) (round 4 on lanes 0..3 only), so every pair comes once; the second
// atom's accumulators rotate one lane per round and return home with one exchange.
template <int ELEC, bool ENERGY>
__device__ __forceinline__ void diag_item(const Shared& sm, Scalars& sc, const PairConst& pc, int b0,
                                          int I, int lane, long long& e18) {
    const TopoDev& tp = sc.tp;
    const Part F = sm.F(b0);
    const int l8 = lane & 7, q = lane >> 3;
    const int src = (lane & 24) | ((l8 + 1) & 7);
    const int i = 8 * I + l8;
    const float4 xa = sm.xq()[i];
    const float2 la = sm.lj()[i];
    const unsigned long long em = i < tp.n_atoms ? tp.excl[i] : 0ull;
    int fax = 0, fay = 0, faz = 0, fbx = 0, fby = 0, fbz = 0;
    long long ei = 0;
    bool bad = false;
#pragma unroll
    for (int k = 1; k <= 4; ++k) {
        const int b = 8 * I + ((l8 + k) & 7);
        const float4 xb = sm.xq()[b];
        const float2 lb = sm.lj()[b];
        const float dx = xb.x - xa.x, dy = xb.y - xa.y, dz = xb.z - xa.z;
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        const bool ok = r2 < pc.rc2 && (k < 4 || l8 < 4) && !((em >> (b - i + kExclWindow)) & 1ull);
        float e = 0.f;
        float s = pair_s<ELEC, ENERGY>(r2, la.x + lb.x, la.y * lb.y, xa.w * xb.w, pc, &e);
        s = ok ? s : 0.0f;
        bad = bad || !(fabsf(s) <= pc.s_lim);
        if (ENERGY) bad = bad || (ok && !(fabsf(e) < kPairEMax));
        const float s13 = s * kPairScale;
        const int tx = __float2int_rn(s13 * dx), ty = __float2int_rn(s13 * dy),
                  tz = __float2int_rn(s13 * dz);
        fax += tx;
        fay += ty;
        faz += tz;
        fbx -= tx;
        fby -= ty;
        fbz -= tz;
        if (ENERGY) ei += ok ? __float2int_rn(e * kPairEScale) : 0;
        if (k < 4) {
            fbx = __shfl_sync(kFull, fbx, src);
            fby = __shfl_sync(kFull, fby, src);
            fbz = __shfl_sync(kFull, fbz, src);
        }
    }
    const int home = (lane & 24) | ((l8 + 4) & 7);
    fbx = __shfl_sync(kFull, fbx, home);
    fby = __shfl_sync(kFull, fby, home);
    fbz = __shfl_sync(kFull, fbz, home);
    if (!((__ballot_sync(kFull, bad) >> (8 * q)) & 0xffu)) {
        red3(F, i, fax + fbx, fay + fby, faz + fbz, sm.fsh);
        if (ENERGY) e18 += ei;
        return;
    }
    for (int k = 1; k <= 4; ++k) {  // slow path (quarter-uniform)
        const int b = 8 * I + ((l8 + k) & 7);
        const float4 xb = sm.xq()[b];
        const float2 lb = sm.lj()[b];
        const float dx = xb.x - xa.x, dy = xb.y - xa.y, dz = xb.z - xa.z;
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        if (!(r2 < pc.rc2 && (k < 4 || l8 < 4) && !((em >> (b - i + kExclWindow)) & 1ull))) continue;
        float e = 0.f;
        const float s = pair_s<ELEC, ENERGY>(r2, la.x + lb.x, la.y * lb.y, xa.w * xb.w, pc, &e);
        add_pair13(F, &sc.flag[b0], sm.fsh, i, b, s * kPairScale, dx, dy, dz);
        if (ENERGY) e18 += __float2ll_rn(e * kPairEScale);
    }
}

// ---------------------------------------------------------------------------
// Bonded terms, contacts, noise
// ---------------------------------------------------------------------------

template <bool ENERGY>
__device__ __forceinline__ float bond_term(const Shared& sm, Scalars& sc, int par_, int b) {
    const TopoDev& tp = sc.tp;
    const Part F = sm.F(par_);
    int* flag = &sc.flag[par_];
    const int2 ij = tp.bond_ij[b];
    const float2 par = tp.bond_par[b];
    const float4 a = sm.xq()[ij.x], c = sm.xq()[ij.y];
    const float dx = c.x - a.x, dy = c.y - a.y, dz = c.z - a.z;
    const float r = sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    const float dr = r - par.x;
    const float f = par.y * dr / r;
    add_term13(sm, F, flag, ij.x, f * dx, f * dy, f * dz);
    add_term13(sm, F, flag, ij.y, -f * dx, -f * dy, -f * dz);
    return ENERGY ? 0.5f * par.y * dr * dr : 0.0f;
}

template <bool ENERGY>
__device__ __forceinline__ float angle_term(const Shared& sm, Scalars& sc, int par_, int q) {
    const TopoDev& tp = sc.tp;
    const Part F = sm.F(par_);
    int* flag = &sc.flag[par_];
    const int4 ijk = tp.ang_ijk[q];
    const float2 par = tp.ang_par[q];
    const float4 a = sm.xq()[ijk.x], b = sm.xq()[ijk.y], c = sm.xq()[ijk.z];
    const float ux = a.x - b.x, uy = a.y - b.y, uz = a.z - b.z;
    const float wx = c.x - b.x, wy = c.y - b.y, wz = c.z - b.z;
    const float cx = uy * wz - uz * wy, cy = uz * wx - ux * wz, cz = ux * wy - uy * wx;
    const float sn = sqrtf(fmaf(cx, cx, fmaf(cy, cy, cz * cz)));
    const float cs = fmaf(ux, wx, fmaf(uy, wy, uz * wz));
    const float ru2 = fmaf(ux, ux, fmaf(uy, uy, uz * uz));
    const float rw2 = fmaf(wx, wx, fmaf(wy, wy, wz * wz));
    const float dth = atan2f(sn, cs) - par.x;
    // F_i = g (cs u / |u|^2 - w) / sn, F_k = g (cs w / |w|^2 - u) / sn, g = -k dth
    const float g = -par.y * dth / sn;
    const float au = cs / ru2, aw = cs / rw2;
    const float fix = g * fmaf(au, ux, -wx), fiy = g * fmaf(au, uy, -wy), fiz = g * fmaf(au, uz, -wz);
    const float fkx = g * fmaf(aw, wx, -ux), fky = g * fmaf(aw, wy, -uy), fkz = g * fmaf(aw, wz, -uz);
    add_term13(sm, F, flag, ijk.x, fix, fiy, fiz);
    add_term13(sm, F, flag, ijk.z, fkx, fky, fkz);
    add_term13(sm, F, flag, ijk.y, -(fix + fkx), -(fiy + fky), -(fiz + fkz));
    return ENERGY ? 0.5f * par.y * dth * dth : 0.0f;
}

// Adds h (x_p - x_i) to G_i and its negative to G_p (2^-20 fixed point). |h| <= |C - C0|
// |dC/du| < 1 and h |x_p - x_i| stays far below 2^11, so one conversion to a 32-bit count
// of 2^-20 units rounds exactly as the 64-bit conversion would.
__device__ __forceinline__ void add_grad(const Shared& sm, Scalars& sc, int b, int i, int p, float h,
                                         float dx, float dy, float dz) {
    const float h20 = h * 1048576.0f;  // 2^20
    const int gx = __float2int_rn(h20 * dx), gy = __float2int_rn(h20 * dy),
              gz = __float2int_rn(h20 * dz);
    const Part G = sm.G(b);
    if (red3(G, i, gx, gy, gz, sm.gsh) | red3(G, p, -gx, -gy, -gz, sm.gsh))
        atomicOr(&sc.flag[b], kFlagGradCoarse);
}

// One native contact (i, p): (C - C0)^2 in float-float, returned as a 2^-40
// fixed-point value. h (x_p - x_i) with h = (C - C0) dC/du goes to G_i and its
// negative to G_p, so that grad_i (C - C0)^2 = -4 h (x_p - x_i) / r0^2 is
// -4 G_i / r0^2 summed over the atom's contacts (Eq. zrMD, Eq. Cij).
__device__ __forceinline__ long long contact_term(const Shared& sm, Scalars& sc, const RunParams& P,
                                                  int par_, int c) {
    const TopoDev& tp = sc.tp;
    const int2 ij = tp.con_ij[c];
    const float4 a = sm.xq()[ij.x], b = sm.xq()[ij.y];
    const ff r2 = ff_dist2(a, b);
    const ff u = ff_mul(r2, P.inv_r0sq_ff);
    const ff C = contact_C_ff(u);
    const float2 c0 = tp.con_C0[c];
    const ff d = ff_add(C, ff{-c0.x, -c0.y});
    const float h = (d.hi + d.lo) * contact_dC_du(u.hi);
    add_grad(sm, sc, par_, ij.x, ij.y, h, b.x - a.x, b.y - a.y, b.z - a.z);
    return ff2fix40(ff_sqr(d));
}

// Noise of the O half step of global step `step` for atoms 32 q .. 32 q + 31:
// sqrt((1 - c1^2) kT / m_i) times Gaussian numbers from Philox4x32-10 with
// counter (atom, replica id, step, 0). Drawn during the evaluation that precedes the
// O half step, by warps that then go on to pull work items (the update stays short).
__device__ __forceinline__ void noise_chunk(const Shared& sm, const TopoDev& tp, const RunParams& P,
                                            uint32_t rep_id, long long step, int q, int lane) {
    const int i = q * kTile + lane;
    if (i < tp.n_atoms) {
        const uint4 rb = philox4x32_10(make_uint4((uint32_t)i, rep_id, (uint32_t)step, 0u), P.key0,
                                       P.key1);
        const float4 g = normals4_f32(rb);
        const float sd = tp.noise_sd[i];
        // xyz only: w holds the atom's bias-functional term, which warp 0 may still be
        // summing while the next evaluation starts
        sm.xi()[i].x = sd * g.x;
        sm.xi()[i].y = sd * g.y;
        sm.xi()[i].z = sd * g.z;
    }
}

__device__ __forceinline__ float box_gap2(float4 al, float4 ah, float4 bl, float4 bh) {
    const float gx = fmaxf(0.f, fmaxf(al.x - bh.x, bl.x - ah.x));
    const float gy = fmaxf(0.f, fmaxf(al.y - bh.y, bl.y - ah.y));
    const float gz = fmaxf(0.f, fmaxf(al.z - bh.z, bl.z - ah.z));
    return fmaf(gx, gx, fmaf(gy, gy, gz * gz));
}

// C(u) of Eq. (Cij) in FP32, u = (r / r0)^2 (the tube variables need no more).
__device__ __forceinline__ float contact_C_f32(float u) {
    const float u2 = u * u;
    const float num = 1.0f + u + u2;
    return num / (num + u2 * u + u2 * u2);
}

// Contact-map tube bias, first pass over two items of kTubeItem native contacts, one per
// half warp (c0: the first contact of this half's item; has: the half has an item): the
// items' shares of sum_p (C_p(X) - <C_p(t'_k)>)^2 for every reference slice k, each
// item's share rounded to fixed point (2^-40) and added to the lanes' running sums dacc
// (exact integer sums: independent of which warp takes which item). Half lanes 0..7
// compute C of their item's contacts; then half lane l takes slices l, l + 16, ... The
// reference maps are stored by item, slice-major inside an item (the eight contacts'
// values of one slice side by side, zero past the last contact), so a lane reads the
// eight values of its slice with two 16-byte loads. Lane l keeps the sums of slices l,
// l + 32, ...: of each pair of 16-slice blocks the half keeps one block's values and
// swaps the other with the opposite half.
__device__ __forceinline__ void tube_pass1(const Shared& sm, const TopoDev& tp, const RunParams& P,
                                           int c0, bool has, int lane, long long* dacc) {
    const int hl = lane & 15;
    const bool h1 = lane & 16;
    const int nq = has ? min(kTubeItem, tp.n_contacts - c0) : 0;
    float C = 0.f;
    if (hl < nq) {
        const int2 ij = tp.con_ij[c0 + hl];
        const float4 a = sm.xq()[ij.x], q = sm.xq()[ij.y];
        const float dx = q.x - a.x, dy = q.y - a.y, dz = q.z - a.z;
        C = contact_C_f32(fmaf(dx, dx, fmaf(dy, dy, dz * dz)) * P.inv_r0sq);
    }
    const int K = P.tube_k;
    const float4* slab = reinterpret_cast<const float4*>(tp.tube_A) + (size_t)(c0 / kTubeItem) * K * 2;
    float even = 0.f;  // this lane's sum of the even block of the current pair of blocks
#pragma unroll
    for (int blk = 0; blk < kMaxTubeK / 16; ++blk) {
        if (blk * 16 >= K) break;
        const int k = blk * 16 + hl;
        const bool in = has && k < K;
        const float4 lo = in ? __ldg(slab + 2 * k) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 hi = in ? __ldg(slab + 2 * k + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float a[kTubeItem] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        float acc = 0.f;
#pragma unroll
        for (int q = 0; q < kTubeItem; ++q) {
            const float d = __shfl_sync(kFull, C, (lane & 16) | q) - a[q];
            acc = q < nq ? fmaf(d, d, acc) : acc;
        }
        const bool last = (blk + 1) * 16 >= K;
        if ((blk & 1) == 0 && !last) {
            even = acc;
            continue;
        }
        const float e0 = (blk & 1) ? even : acc, o1 = (blk & 1) ? acc : 0.f;
        const float other = __shfl_xor_sync(kFull, h1 ? e0 : o1, 16);
        dacc[blk >> 1] += __float2ll_rn((h1 ? o1 : e0) * 1099511627776.0f) +  // 2^40
                          __float2ll_rn(other * 1099511627776.0f);
    }
}

// Contact-map tube bias, second pass over two items of kTubeItem contacts, one per
// half warp (c0: the first contact of this half's item; has: the half has an item):
// with gamma_k the weights of the ratchet forces on the slices (dF/dD_k), the force on
// the atoms of contact p is beta_p grad C_p with beta_p = (2/N0) sum_k gamma_k
// (C_p - <C_p(t'_k)>); h = beta_p C'(u) goes to G like the z gradient (F = -2/r0^2 G).
// The dots sum_k gamma_k <C_p(t'_k)> are formed with lane l of a half on slices l,
// l + 16, ... (two 16-byte loads per slice, the eight contacts' values side by side)
// and reduced over the half for the eight contacts at once: three exchange steps
// halve the values each lane holds, one more finishes the sums, so half lane L ends
// with the dot of contact L >> 1. The order of every sum is fixed. Two items per warp
// keep twice the loads in flight per L2 round trip.
__device__ __forceinline__ void tube_pass2(const Shared& sm, Scalars& sc, const TopoDev& tp,
                                           const RunParams& P, int b, int c0, bool has, int lane) {
    const int hl = lane & 15;
    const int nq = has ? min(kTubeItem, tp.n_contacts - c0) : 0;
    // the contact of half lane l (l < nq; clamped elsewhere) is read first, so that its
    // latency overlaps the slice loads
    const int2 ij = has ? tp.con_ij[c0 + min(hl, nq - 1)] : make_int2(0, 0);
    const int K = has ? P.tube_k : 0;
    const float4* slab = reinterpret_cast<const float4*>(tp.tube_A) + (size_t)(c0 / kTubeItem) * K * 2;
    float v[kTubeItem];
#pragma unroll
    for (int q = 0; q < kTubeItem; ++q) v[q] = 0.f;
#pragma unroll
    for (int blk = 0; blk < kMaxTubeK / 16; ++blk) {
        if (blk * 16 >= P.tube_k) break;
        const int k = blk * 16 + hl;
        const bool in = k < K;
        const float g = in ? sc.gam[k] : 0.f;
        const float4 lo = in ? __ldg(slab + 2 * k) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 hi = in ? __ldg(slab + 2 * k + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float a[kTubeItem] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
        for (int q = 0; q < kTubeItem; ++q) v[q] = fmaf(g, a[q], v[q]);
    }
    const bool b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
    float w4[4], w2[2];
#pragma unroll
    for (int q = 0; q < 4; ++q)
        w4[q] = (b3 ? v[q + 4] : v[q]) + __shfl_xor_sync(kFull, b3 ? v[q] : v[q + 4], 8);
#pragma unroll
    for (int q = 0; q < 2; ++q)
        w2[q] = (b2 ? w4[q + 2] : w4[q]) + __shfl_xor_sync(kFull, b2 ? w4[q] : w4[q + 2], 4);
    float w1 = (b1 ? w2[1] : w2[0]) + __shfl_xor_sync(kFull, b1 ? w2[0] : w2[1], 2);
    w1 += __shfl_xor_sync(kFull, w1, 1);
    const float dot = __shfl_sync(kFull, w1, (lane & 16) | ((hl & 7) * 2));
    // every lane stays to the end (all exchanges above are full-warp); lanes >= nq
    // of a half hold a copy of its last contact and add nothing
    const bool live = hl < nq;
    const float4 a = sm.xq()[ij.x], q = sm.xq()[ij.y];
    const float dx = q.x - a.x, dy = q.y - a.y, dz = q.z - a.z;
    const float u = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) * P.inv_r0sq;
    const float C = contact_C_f32(u);
    const float h = live ? 2.0f * tp.tube_inv_n0 * (C * sc.gam_sum - dot) * contact_dC_du(u) : 0.f;
    if (live) add_grad(sm, sc, b, ij.x, ij.y, h, dx, dy, dz);
}

// Tube variables and their ratchets from the summed slice distances (warp 0):
// D_k = sum_p (C_p - <C_p(t'_k)>)^2 / N0, pi_k = exp(-lambda D_k) / sum,
// w = -(1/lambda) log sum_k exp(-lambda D_k), s = 1 - (1/t) sum_k t'_k pi_k
// (Eq. sX, Eq. wX with the average maps); F^s, F^w of Eq. (Fs), Eq. (Fw) through
// gamma_k = c_s ds/dD_k + c_w dw/dD_k, ds/dD_k = (lambda/t) pi_k (t'_k - <t'>),
// dw/dD_k = pi_k. The D_k are exact fixed-point sums; their differences to the
// smallest are taken in integers and the weights in FP32 (the FP64 pipe of this GPU
// is 64 times slower); s and w are compared with their running minima in FP64.
// Sums over k are in a fixed order (lane order, then a fixed tree).
template <int CL>
__device__ void tube_decide(Scalars& sc, const TopoDev& tp, const RunParams& P, int b, int lane) {
    const int K = P.tube_k;
    constexpr int NB = kMaxTubeK / 32;
    float tk[NB];  // slice times, loaded first (their latency overlaps the exchange)
    long long dk[NB];
    long long dmin = LLONG_MAX;
#pragma unroll
    for (int blk = 0; blk < NB; ++blk) {
        const int k = blk * 32 + lane;
        tk[blk] = k < K ? (float)P.tube_time[k] : 0.f;
        dk[blk] = LLONG_MAX;
        if (k < K) {
            long long t = 0;
            for (int q = 0; q < CL; ++q) t += rank_ptr<CL>(&sc.red_d[b][0], q)[k];
            dk[blk] = t;
            dmin = min(dmin, t);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmin = min(dmin, __shfl_xor_sync(kFull, dmin, o));
    const float scale = 9.094947017729282e-13f * tp.tube_inv_n0;  // 2^-40 / N0
    const float lam = (float)P.tube_lambda;
    float e[NB], Z = 0.f, Zt = 0.f;
#pragma unroll
    for (int blk = 0; blk < NB; ++blk) {
        const int k = blk * 32 + lane;
        e[blk] = k < K ? expf(-lam * ((float)(dk[blk] - dmin) * scale)) : 0.f;
        Z += e[blk];
        Zt += e[blk] * tk[blk];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Z += __shfl_down_sync(kFull, Z, o);
        Zt += __shfl_down_sync(kFull, Zt, o);
    }
    Z = __shfl_sync(kFull, Z, 0);
    Zt = __shfl_sync(kFull, Zt, 0);
    const float inv_Z = 1.0f / Z;
    const float tbar = Zt * inv_Z;
    const float inv_t = (float)(1.0 / P.tube_t);
    const double sv = 1.0 - (double)(tbar * inv_t);
    const double wv = (double)dmin * 9.094947017729282e-13 * (double)tp.tube_inv_n0 -
                      (double)(logf(Z) / lam);
    double cs = 0.0, cw = 0.0;  // ratchets, theta(0) = 1
    const double sm0 = sc.sm, wm0 = sc.wm;
    if (!(sv < sm0)) cs = -P.tube_ks * (sv - sm0);
    if (!(wv < wm0)) cw = -P.tube_kw * (wv - wm0);
    const float cs_l = (float)cs * lam * inv_t, cw_f = (float)cw;
    float gsum = 0.f;
#pragma unroll
    for (int blk = 0; blk < NB; ++blk) {
        const int k = blk * 32 + lane;
        if (k < K) {
            const float pi = e[blk] * inv_Z;
            const float g = fmaf(cs_l * pi, tk[blk] - tbar, cw_f * pi);
            sc.gam[k] = g;
            gsum += g;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) gsum += __shfl_down_sync(kFull, gsum, o);
    __syncwarp();
    if (lane == 0) {
        if (sv < sm0) sc.sm = sv;
        if (wv < wm0) sc.wm = wv;
        sc.gam_sum = gsum;
        sc.z = sv;  // frames record s_lambda and its running minimum
        sc.zm = fmin(sm0, sv);
        sc.kb = -2.0f * P.inv_r0sq;
        sc.bias_on = (cs != 0.0 || cw != 0.0) ? 1 : 0;
    }
}

// Force and bias gradient of one atom, summed over the cluster.
struct AtomSums {
    float fx, fy, fz, gx, gy, gz;
};

// Sums the partials of atom i for parity b (those of the other CTAs through distributed shared
// memory; all loads are issued before any sum is formed). grad: the bias gradient as well; its
// coarse words are read only when some CTA of the cluster has touched them.
template <int CL>
__device__ __forceinline__ AtomSums load_sums(const Shared& sm, Scalars& sc, int b, int rank, int i,
                                              bool grad) {
    const Part F = sm.F(b), G = sm.G(b);
    int fh[3], hg[3] = {0, 0, 0};
    unsigned fl[3], gl[3];
    int flags = sc.flag[b];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        fh[c] = F.H[3 * i + c];
        fl[c] = F.L[3 * i + c];
        gl[c] = grad ? G.L[3 * i + c] : 0u;
    }
#pragma unroll
    for (int q = 1; q < CL; ++q) {
        const int p = (rank + q) & (CL - 1);
        const int* pFH = rank_ptr<CL>(F.H, p) + 3 * i;
        const unsigned* pFL = rank_ptr<CL>(F.L, p) + 3 * i;
        const unsigned* pGL = rank_ptr<CL>(G.L, p) + 3 * i;
        int rh[3], rf = *rank_ptr<CL>(&sc.flag[b], p);
        unsigned rl[3], ql[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            rh[c] = pFH[c];
            rl[c] = pFL[c];
            ql[c] = grad ? pGL[c] : 0u;
        }
        flags |= rf;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            fh[c] += rh[c];
            fl[c] += rl[c];
            gl[c] += ql[c];
        }
    }
    if (grad && (flags & kFlagGradCoarse))
        for (int p = 0; p < CL; ++p)
            for (int c = 0; c < 3; ++c) hg[c] += rank_ptr<CL>(G.H, p)[3 * i + c];
    AtomSums a;  // (force: 2^-13 to 2^-20 units)
    a.fx = fix2f(join_coarse(fh[0], fl[0], sm.fsh) * 128);
    a.fy = fix2f(join_coarse(fh[1], fl[1], sm.fsh) * 128);
    a.fz = fix2f(join_coarse(fh[2], fl[2], sm.fsh) * 128);
    a.gx = grad ? fix2f(join_coarse(hg[0], gl[0], sm.gsh)) : 0.f;
    a.gy = grad ? fix2f(join_coarse(hg[1], gl[1], sm.gsh)) : 0.f;
    a.gz = grad ? fix2f(join_coarse(hg[2], gl[2], sm.gsh)) : 0.f;
    return a;
}

// The same for the atom of a group of four lanes, one component per lane (a quarter of the remote
// loads in a row); every lane of the group gets the result. Called by whole warps.
template <int CL>
__device__ __forceinline__ AtomSums load_sums4(const Shared& sm, Scalars& sc, int b, int rank, int i,
                                               bool grad) {
    const Part F = sm.F(b), G = sm.G(b);
    const int lane = threadIdx.x & 31, k = 3 * i + min(lane & 3, 2);
    int fh = F.H[k], hg = 0, flags = sc.flag[b];
    unsigned fl = F.L[k], gl = grad ? G.L[k] : 0u;
#pragma unroll
    for (int q = 1; q < CL; ++q) {
        const int p = (rank + q) & (CL - 1);
        flags |= *rank_ptr<CL>(&sc.flag[b], p);
        fh += rank_ptr<CL>(F.H, p)[k];
        fl += rank_ptr<CL>(F.L, p)[k];
        gl += grad ? rank_ptr<CL>(G.L, p)[k] : 0u;
    }
    if (grad && (flags & kFlagGradCoarse))
        for (int p = 0; p < CL; ++p) hg += rank_ptr<CL>(G.H, p)[k];
    const float f = fix2f(join_coarse(fh, fl, sm.fsh) * 128);
    const float g = grad ? fix2f(join_coarse(hg, gl, sm.gsh)) : 0.f;
    const int l0 = lane & ~3;
    AtomSums a;
    a.fx = __shfl_sync(kFull, f, l0);
    a.fy = __shfl_sync(kFull, f, l0 + 1);
    a.fz = __shfl_sync(kFull, f, l0 + 2);
    a.gx = __shfl_sync(kFull, g, l0);
    a.gy = __shfl_sync(kFull, g, l0 + 1);
    a.gz = __shfl_sync(kFull, g, l0 + 2);
    return a;
}

// ---------------------------------------------------------------------------
// Pair list build
// ---------------------------------------------------------------------------

// Builds the pair list of the positions in shared memory: the block boxes, then for the
// blocks I with I % CL == rank (one warp per block) the ascending list of atoms j of
// later blocks within sqrt(rlist2) of some atom of I, then (after a cluster barrier, so
// that every CTA's entries are complete and their counts, written to all CTAs, are there)
// this CTA's item table. Items are numbered over all blocks, chunks near a block (first j
// within the exclusion window of the block) first; item k goes to CTA k % CL. Called by every
// thread of every CTA of the cluster; on return the CTA is synchronised (the counts are
// written again only after the cluster barrier of an evaluation).
template <int CL>
__device__ __noinline__ void build_list(const Shared& sm, Scalars& sc, float rlist2) {
    const TopoDev& tp = sc.tp;
    const ListDev L = sc.list;
    const int n = tp.n_atoms, nb = (n + 7) >> 3;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = cta_rank<CL>();
    // scratch in the xi array (128 B per block): boxes (2 nb float4), the two prefix arrays
    // (nb ints each, one more for the total) and per warp the candidate blocks of its row
    float4* blo = sm.xi();
    float4* bhi = sm.xi() + nb;
    int* pren = (int*)(sm.xi() + 2 * nb);
    int* pref = pren + nb;
    uint8_t* cand = (uint8_t*)(pref + nb + 1) + warp * nb;
    __syncthreads();  // warp 0 may still be summing the bias terms held in the xi array
    if (tid == 0) sc.build_next = 0;
    for (int I = tid; I < nb; I += blockDim.x) {
        float4 lo = make_float4(3.0e38f, 3.0e38f, 3.0e38f, 0.f);
        float4 hi = make_float4(-3.0e38f, -3.0e38f, -3.0e38f, 0.f);
        for (int a = 8 * I; a < min(8 * I + 8, n); ++a) {
            const float4 x = sm.xq()[a];
            lo.x = fminf(lo.x, x.x);
            lo.y = fminf(lo.y, x.y);
            lo.z = fminf(lo.z, x.z);
            hi.x = fmaxf(hi.x, x.x);
            hi.y = fmaxf(hi.y, x.y);
            hi.z = fmaxf(hi.z, x.z);
        }
        blo[I] = lo;
        bhi[I] = hi;
    }
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    for (;;) {  // this CTA's blocks, one warp each, pulled in order (early blocks have most work)
        int m = 0;
        if (lane == 0) m = atomicAdd(&sc.build_next, 1);
        const int I = __shfl_sync(kFull, m, 0) * CL + rank;
        if (I >= nb) break;
        const float4 bl = blo[I], bh = bhi[I];
        const int i0 = 8 * I;
        uint16_t* out = L.jl + list_jl_off(L.nbs, I);
        int nc = 0;  // candidate blocks, ascending
        for (int J0 = I + 1; J0 < nb; J0 += 32) {
            const int J = J0 + lane;
            const bool c = J < nb && box_gap2(bl, bh, blo[J], bhi[J]) < rlist2;
            const unsigned cm = __ballot_sync(kFull, c);
            if (c) cand[nc + __popc(cm & lt)] = (uint8_t)J;
            nc += __popc(cm);
        }
        __syncwarp();
        int count = 0;
        for (int g = 0; g < nc; g += 8) {  // eight candidates at a time, two atoms per lane:
            // lane (c, s) tests atom s of candidates g + c and g + 4 + c, packed
            const int ca = g + (lane >> 3), cb = ca + 4;
            const int ja = ca < nc ? 8 * cand[ca] + (lane & 7) : n;
            const int jb = cb < nc ? 8 * cand[cb] + (lane & 7) : n;
            const float4 far = make_float4(1.0e18f, 0.f, 0.f, 0.f);
            const float4 xa = ja < n ? sm.xq()[ja] : far, xb = jb < n ? sm.xq()[jb] : far;
            float da = 3.0e38f, db = 3.0e38f;
#pragma unroll
            for (int a = 0; a < 8; ++a) {  // (the padding slots of a last block are far)
                const float4 xi = sm.xq()[i0 + a];
                const float2 dx = make_float2(xa.x - xi.x, xb.x - xi.x),
                             dy = make_float2(xa.y - xi.y, xb.y - xi.y),
                             dz = make_float2(xa.z - xi.z, xb.z - xi.z);
                const float2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
                da = fminf(da, r2.x);
                db = fminf(db, r2.y);
            }
            const bool ha = da < rlist2, hb = db < rlist2;
            const unsigned ma = __ballot_sync(kFull, ha), mb = __ballot_sync(kFull, hb);
            if (ha) out[count + __popc(ma & lt)] = (uint16_t)ja;
            count += __popc(ma);
            if (hb) out[count + __popc(mb & lt)] = (uint16_t)jb;
            count += __popc(mb);
        }
        // the entries near the block come first: lane s tests atom s after the block and writes
        // its exclusion mask (bit a for block atom a; zero past the near entries)
        const int jn = i0 + 8 + lane;
        const bool in = lane < kExclWindow - 1 && jn < n;
        const float4 xn = in ? sm.xq()[jn] : make_float4(1.0e18f, 0.f, 0.f, 0.f);
        const unsigned long long exa = (lane < 8 && i0 + lane < n) ? tp.excl[i0 + lane] : 0ull;
        float dn = 3.0e38f;
        unsigned byte = 0u;
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            const float4 xi = sm.xq()[i0 + a];
            const float dx = xn.x - xi.x, dy = xn.y - xi.y, dz = xn.z - xi.z;
            dn = fminf(dn, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
            const unsigned long long ex = __shfl_sync(kFull, exa, a);
            const int dj = 8 + lane - a + kExclWindow;
            if (dj < 2 * kExclWindow && ((ex >> dj) & 1ull)) byte |= 1u << a;
        }
        const bool hn = dn < rlist2;
        const unsigned mn = __ballot_sync(kFull, hn);
        const int n_near = __popc(mn);
        uint8_t* mask = L.excl + kListMasks * I;
        if (hn) mask[__popc(mn & lt)] = (uint8_t)byte;
        if (lane >= n_near) mask[lane] = 0;
        __syncwarp();  // (the candidate list is overwritten by the warp's next row)
        const int chunks = (count + kListChunk - 1) / kListChunk;
        if (lane < kListChunk * chunks - count) out[count + lane] = (uint16_t)sm.nta;
        if (lane < CL) {  // every CTA of the cluster gets the counts
            *rank_ptr<CL>(&sc.cnt[I], lane) = (uint16_t)chunks;
            // chunks with an entry near the block
            *rank_ptr<CL>(&sc.cntn[I], lane) = (uint16_t)((n_near + kListChunk - 1) / kListChunk);
        }
    }
    __threadfence();  // entries are read back with L2 loads (also by the other CTAs)
    cluster_barrier<CL>();  // every block's entries and counts are complete
    if (warp == 0) {  // prefix sums over blocks: near chunks, then the remaining ones
        const int per = (nb + 31) >> 5, I0 = min(per * lane, nb), I1 = min(I0 + per, nb);
        int runn = 0, runf = 0;
        for (int I = I0; I < I1; ++I) {
            runn += sc.cntn[I];
            runf += sc.cnt[I] - sc.cntn[I];
        }
        int sn = runn, sf = runf;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int yn = __shfl_up_sync(kFull, sn, o), yf = __shfl_up_sync(kFull, sf, o);
            if (lane >= o) {
                sn += yn;
                sf += yf;
            }
        }
        int pn = sn - runn, pf = sf - runf;
        for (int I = I0; I < I1; ++I) {
            pren[I] = pn;
            pref[I] = pf;
            pn += sc.cntn[I];
            pf += sc.cnt[I] - sc.cntn[I];
        }
        runn = __shfl_sync(kFull, sn, 31);
        runf = __shfl_sync(kFull, sf, 31);
        const int total = runn + runf;
        if (lane == 0) {
            sc.n_items = (total - rank + CL - 1) / CL;
            sc.cached = sc.n_items <= sm.lc_cap ? 1 : 0;
            sc.n_diag = (nb - rank + CL - 1) / CL;
            sc.work_next[0] = 0;
            sc.work_next[1] = 0;
            sc.pair_slots = 8ll * kListChunk * total + 28ll * nb;  // pairs evaluated per step with this list
        }
        // the total number of near chunks, for the far items' numbering
        if (lane == 0) pref[nb] = runn;
    }
    __syncthreads();
    const int tot_near = pref[nb];
    const bool cached = sc.cached;
    // one item per thread: its block is the last whose first chunk number is not beyond it
    for (int it = tid; it < sc.n_items; it += blockDim.x) {
        const int k = it * CL + rank;
        const bool near = k < tot_near;
        const int* pre = near ? pren : pref;
        const int key = near ? k : k - tot_near;
        int lo = 0, hi = nb;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (pre[mid] <= key) lo = mid; else hi = mid;
        }
        const int c = key - pre[lo] + (near ? 0 : (int)sc.cntn[lo]);
        const uint32_t d = ((uint32_t)lo << 17) | ((uint32_t)near << 16) | (uint32_t)c;
        if (cached) {  // the chunk's entries: two 16-byte loads (chunks are 32-aligned)
            CacheItem& ci = sm.lc()[it];
            const uint4* e = (const uint4*)(L.jl + list_jl_off(L.nbs, lo) + kListChunk * c);
            const uint4 e0 = __ldcg(e), e1 = __ldcg(e + 1);
            if (near) *(uint4*)ci.xm = __ldcg((const uint4*)(L.excl + kListMasks * lo + kListChunk * c));
            ci.desc = d;
            ((uint4*)ci.j)[0] = e0;
            ((uint4*)ci.j)[1] = e1;
        } else {
            L.items[it] = d;
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Force evaluation
// ---------------------------------------------------------------------------

// First tile (of 32 atoms) of the share of nt tiles that CTA `rank` of cl integrates.
__device__ __forceinline__ int own_lo(int nt, int rank, int cl) { return nt * rank / cl; }

// Force evaluation of the configuration in shared memory (pair list current) for
// the evaluated step of parity b. Work items come from the queue of this CTA; its
// share goes to the parity-b partials. With noise_step >= 0 the CTA also draws the
// Gaussian numbers of that step's O half step for the atoms it integrates. Ends with a cluster barrier: the partials of every CTA are
// complete (the bias gradient of the tube bias is not: see finish_evaluation).
template <int ELEC, bool ENERGY, int CL, bool TUBE>
__device__ void evaluate_work(const Shared& sm, Scalars& sc, const RunParams& P, int b,
                              bool do_ratchet, uint32_t rep_id, long long noise_step) {
    const TopoDev& tp = sc.tp;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const int nt = tp.n_tiles, rank = cta_rank<CL>();
    if (noise_step >= 0)  // of the atoms this CTA integrates
        for (int q = own_lo(nt, rank, CL) + warp; q < own_lo(nt, rank + 1, CL); q += nw)
            noise_chunk(sm, tp, P, rep_id, noise_step, q, lane);
    // Work list of this CTA: pair batches (four items from its item table each), blocks
    // with themselves (four per batch), then its shares of the contact, bond and angle
    // chunks (global chunk g belongs to CTA g % CL). Under the contact-map tube bias the
    // contact items are first-pass units of two items of kTubeItem contacts (loads from
    // the reference maps in L2), interleaved one to one with the pair batches so that
    // their memory latency overlaps arithmetic.
    const int n_pb = (sc.n_items + 3) >> 2;
    const int n_db = (sc.n_diag + 3) >> 2;
    const bool tube = TUBE && do_ratchet;  // contact-map tube bias: two work phases
    const int ncon = (P.bias == 1 || P.bias == 5) ? tp.n_contacts : 0;  // frames: z too
    const int g_con = tube ? ((ncon + kTubeItem - 1) / kTubeItem + 1) / 2  // two items a unit
                           : (ncon + kChunk - 1) / kChunk;
    const int g_bond = (tp.n_bonds + kChunk - 1) / kChunk;
    const int g_ang = (tp.n_angles + kChunk - 1) / kChunk;
    const int n_con = (g_con - rank + CL - 1) / CL;
    const int n_bond = (g_bond - rank + CL - 1) / CL;
    const int n_ang = (g_ang - rank + CL - 1) / CL;
    const int m_mix = tube ? min(n_pb, n_con) : 0;
    const int e_pair = n_pb + n_con;          // pair batches and contact items end here
    const int e_diag = e_pair + n_db;
    const int e_bond = e_diag + n_bond;
    const int e_all = e_bond + n_ang;
    int* counter = &sc.work_next[b];
    long long e18 = 0, e20 = 0, zacc = 0;  // fixed point: sums independent of the work order
    long long dacc[TUBE ? kMaxTubeK / 32 : 1];  // first-pass slice sums of this lane
#pragma unroll
    for (int q = 0; q < (TUBE ? kMaxTubeK / 32 : 1); ++q) dacc[q] = 0;
    int m_next = 0;  // the next work index is pulled while the current item runs
    if (lane == 0) m_next = atomicAdd(counter, 1);
    for (;;) {
        const int k = __shfl_sync(kFull, m_next, 0);
        if (k >= e_all) break;
        if (lane == 0) m_next = atomicAdd(counter, 1);
        if (k < e_pair) {
            int kp = -1, kc = -1;  // pair batch or contact item
            if (k < 2 * m_mix) {
                if (k & 1) kc = k >> 1; else kp = k >> 1;
            } else {
                const int r = k - 2 * m_mix;
                if (r < n_pb - m_mix) kp = m_mix + r; else kc = m_mix + r - (n_pb - m_mix);
            }
            if (kp >= 0) {
                pair_batch<ELEC, ENERGY>(sm, sc, P, b, kp, lane, e18);
            } else {
                const int g = kc * CL + rank;
                if (tube) {
                    if constexpr (TUBE) {
                        const int c0 = (2 * g + (lane >> 4)) * kTubeItem;
                        tube_pass1(sm, tp, P, c0, c0 < ncon, lane, dacc);
                    }
                } else {
                    const int c = g * kChunk + lane;
                    if (c < ncon) zacc += contact_term(sm, sc, P, b, c);
                }
            }
        } else if (k < e_diag) {
            const int d = 4 * (k - e_pair) + (lane >> 3);
            const int I = d < sc.n_diag ? d * CL + rank : (sm.nta >> 3);
            diag_item<ELEC, ENERGY>(sm, sc, P.pc, b, I, lane, e18);
        } else if (k < e_bond) {
            const int q = ((k - e_diag) * CL + rank) * kChunk + lane;
            if (q < tp.n_bonds) {
                const float eb = bond_term<ENERGY>(sm, sc, b, q);
                if (ENERGY) e20 += f2fix(eb);
            }
        } else {
            const int q = ((k - e_bond) * CL + rank) * kChunk + lane;
            if (q < tp.n_angles) {
                const float ea = angle_term<ENERGY>(sm, sc, b, q);
                if (ENERGY) e20 += f2fix(ea);
            }
        }
    }
    if constexpr (TUBE) {
        if (tube) {  // one add per slice and warp into this CTA's share
#pragma unroll
            for (int blk = 0; blk < kMaxTubeK / 32; ++blk) {
                const int kk = blk * 32 + lane;
                if (kk < P.tube_k && dacc[blk] != 0)
                    atomicAdd((unsigned long long*)&sc.red_d[b][kk], (unsigned long long)dacc[blk]);
            }
        }
    }
    if (ncon > 0 && !tube) {
        const unsigned z0 = __reduce_add_sync(kFull, (unsigned)zacc & 0xfffffu),
                       z1 = __reduce_add_sync(kFull, (unsigned)(zacc >> 20) & 0xfffffu),
                       z2 = __reduce_add_sync(kFull, (unsigned)(zacc >> 40));
        if (lane == 0) {
            atomicAdd(&sc.zw[b][0], z0);
            atomicAdd(&sc.zw[b][1], z1);
            if (z2) atomicAdd(&sc.zw[b][2], z2);
        }
    }
    long long e = 0;
    if (ENERGY) e = warp_sum_ll((e18 << 2) + e20);  // 2^-18 pair energy units to 2^-20
    if (ENERGY && lane == 0) sc.red_e[b][warp] = e;
    cluster_barrier<CL>();
}

// The end of an evaluation: z, energy and flags summed over the cluster and the ratchet
// decision (warp 0 of every CTA, from the same fixed-point sums); under the tube bias also its
// variables and the second work phase, which completes the bias gradient. On return the CTA is
// synchronised.
template <bool ENERGY, int CL, bool TUBE>
__device__ void finish_evaluation(const Shared& sm, Scalars& sc, const RunParams& P, int b,
                                  bool do_ratchet) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const bool tube = TUBE && do_ratchet;
    // (the partials of the other parity are cleared atom by atom in the update that follows;
    // the slice sums of the tube bias here)
    if (tube)
        for (int i = tid; i < P.tube_k; i += blockDim.x) sc.red_d[b ^ 1][i] = 0;
    // shares of z, energy and flags from every CTA of the cluster (integer sums); all
    // remote loads are issued before any is used
    if (warp == 0) {
        unsigned zq[CL][3];
        long long eq[CL];
        int fq[CL];
#pragma unroll
        for (int q = 0; q < CL; ++q) {
            const unsigned* z = rank_ptr<CL>(&sc.zw[b][0], q);
#pragma unroll
            for (int c = 0; c < 3; ++c) zq[q][c] = lane == 0 ? z[c] : 0u;
            eq[q] = (ENERGY && lane < nw) ? rank_ptr<CL>(&sc.red_e[b][0], q)[lane] : 0;
            fq[q] = lane == 0 ? *rank_ptr<CL>(&sc.flag[b], q) : 0;
        }
        long long zt = 0, et = 0;
        int fl = 0;
#pragma unroll
        for (int q = 0; q < CL; ++q) {
            zt += ((long long)zq[q][2] << 40) + ((long long)zq[q][1] << 20) + (long long)zq[q][0];
            et += eq[q];
            fl |= fq[q];
        }
        if (ENERGY) et = warp_sum_ll(et);
        if (lane == 0) {
            if (ENERGY) sc.epot = (double)et * 9.5367431640625e-07;  // 2^-20
            if (fl & SCPS_FLAG_FORCE_RANGE) sc.status |= SCPS_FLAG_FORCE_RANGE;
            float kb = 0.f;
            int on = 0;
            if (P.bias == 1 || (P.bias == 5 && !tube)) {  // (frame evaluation: z as well)
                // z = zt 2^-40: the count goes into the mantissa of 4096 (whose last bit is
                // 2^-40), one FP64 subtraction instead of a conversion and a product (an FP64
                // instruction costs about 70 clocks that every warp waits for)
                const double z = zt < (1ll << 52)
                                     ? __longlong_as_double(0x40B0000000000000ll | zt) - 4096.0
                                     : (double)zt * 9.094947017729282e-13;
                sc.z = z;
                if (do_ratchet && P.bias == 1) {  // Eq. (FrMD) with theta(0) = 1
                    const double zm = sc.zm, dz = z - zm;
                    if (below_zero(dz)) {  // z < z_m
                        sc.zm = z;
                    } else {
                        const double factor = -P.k_R * dz;
                        on = (__double_as_longlong(factor) << 1) != 0;  // not zero
                        kb = -(float)factor * 4.0f * P.inv_r0sq;
                    }
                }
            }
            sc.kb = kb;
            sc.bias_on = on;
            sc.work_next[b] = 0;  // every pull of this evaluation is done
        }
        if (tube) tube_decide<CL>(sc, sc.tp, P, b, lane);
    }
    __syncthreads();
    if (tube) {  // second work phase: the bias force per contact, then G is complete
        int* counter2 = &sc.work_next2[b];
        const int rank = cta_rank<CL>(), ncon = sc.tp.n_contacts;
        const int n2 = (ncon + kTubeItem - 1) / kTubeItem;
        int m2 = 0;  // the next item index is pulled while the current item runs
        if (lane == 0) m2 = atomicAdd(counter2, 1);
        for (;;) {  // units of two items of this CTA, one per half warp
            const int u = __shfl_sync(kFull, m2, 0);
            if (2 * u * CL + rank >= n2) break;
            if (lane == 0) m2 = atomicAdd(counter2, 1);
            const int k = (2 * u + (lane >> 4)) * CL + rank;
            tube_pass2(sm, sc, sc.tp, P, b, k * kTubeItem, k < n2, lane);
        }
        cluster_barrier<CL>();  // the other CTAs read this CTA's G next
        if (tid == 0) sc.work_next2[b] = 0;
    }
}

// Atom slots: real atoms, padding slots and the 8 sentinel slots far apart from
// everything (no charge, no LJ).
__device__ __forceinline__ float4 far_slot(int i) {
    return make_float4(1.0e5f * (float)(i + 1), 0.f, 0.f, 0.f);
}

}  // namespace

// WIDE: at most kMaxThreadsPair threads per CTA, which leaves 80 registers per thread (every
// cluster of several CTAs, and a lone CTA that has an SM to itself: 1200 atoms 78.0 us per step
// against 84.0 with 1024 threads of 64 registers, 304 atoms 14.4 against 15.4). Otherwise up to
// 1024 threads of 64 registers: for callers who ask for more threads, and where more CTAs on an SM
// save a wave (wide_form).
template <int ELEC, int CL, bool TUBE, bool WIDE>
__global__ void __launch_bounds__(WIDE ? kMaxThreadsPair : 1024, 1)
k_resident(const TopoDev* __restrict__ topos, const RepDev* __restrict__ reps, StateDev st,
           RunParams P, int nta, int lc_cap) {
    __shared__ Scalars sc;
    const RepDev rep = reps[blockIdx.x / CL];  // this launch's replicas, in any order
    const int r = rep.index;
    const int rank = cta_rank<CL>();
    if (threadIdx.x == 0) {
        sc.tp = topos[rep.topo];
        sc.pc = P.pc;
        sc.list = list_of<CL>(P.list_base + rep.list_off, nta, rank);
    }
    __syncthreads();
    const TopoDev& tp = sc.tp;
    const Shared sm = {nta, lc_cap, tp.f_shift, tp.g_shift};
    const int n = tp.n_atoms;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    for (int i = tid; i < sm.na8(); i += blockDim.x) {
        if (i < n) {
            const float4 x = st.x[rep.atom_off + i];
            sm.xq()[i] = make_float4(x.x, x.y, x.z, tp.qs[i]);
            sm.lj()[i] = tp.lj[i];
            const float4 v = st.v[rep.atom_off + i];
            sm.v()[i] = make_float4(v.x, v.y, v.z, tp.inv_m[i]);
        } else {
            sm.xq()[i] = far_slot(i);
            sm.lj()[i] = make_float2(0.f, 0.f);
            if (i < nta) sm.v()[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    for (int i = tid; i < 24 * sm.na8(); i += blockDim.x) sm.F(0).L[i] = 0u;  // F and G, both parities
    if (tid == 0) {
        sc.zm = st.zm[r];
        sc.z = st.z[r];
        sc.T = st.T[r];
        sc.status = st.status[r];
        sc.n_saved = st.n_saved[r];
        sc.flag[0] = 0;
        sc.flag[1] = 0;
        sc.bias_on = 0;
        sc.work_next[0] = 0;
        sc.work_next[1] = 0;
        sc.work_next2[0] = 0;
        sc.work_next2[1] = 0;
        sc.vmax2[0] = 0u;
        sc.vmax2[1] = 0u;
        for (int q = 0; q < 6; ++q) (&sc.zw[0][0])[q] = 0u;
        sc.sm = st.sm[r];
        sc.wm = st.wm[r];
    }
    for (int i = tid; i < kMaxTubeK; i += blockDim.x) {
        sc.red_d[0][i] = 0;
        sc.red_d[1][i] = 0;
    }
    long long step = st.step[r];
    int builds = 0;  // pair-list builds in this launch
    bool nonfinite = false;  // an update left the FP32 range (the same in all threads of the cluster)
    cluster_barrier<CL>();  // every CTA of the cluster is initialised before any remote access
    const float hdt = P.half_dt;
    if (sc.status == 0 && P.n_steps > 0) {
        build_list<CL>(sm, sc, P.rlist2);
        // displacement bound since the last build and steps since then (identical in every
        // thread of the cluster: same inputs, same arithmetic)
        float disp = 0.f;
        int since = 0;
        builds = 1;
        // the O half step that follows an evaluation uses the noise of the same step index
        evaluate_work<ELEC, false, CL, TUBE>(sm, sc, P, (int)(step & 1), true, rep.rep_id, step);
        // The sums of a thread's first atom are loaded as soon as the partials are complete,
        // beside the ratchet decision that the other warps would wait for (the tube bias
        // completes its gradient after the decision and loads then).
        const bool grad = P.bias != 0;
        // the atoms this CTA integrates; their new positions go to every CTA
        const int a0 = kTile * own_lo(tp.n_tiles, rank, CL),
                  a1 = min(n, kTile * own_lo(tp.n_tiles, rank + 1, CL));
        // One thread per atom, four lanes where the threads suffice (the first of them goes on
        // to integrate it); warp 0, which decides, takes no atoms where the others suffice. The
        // latency of the remote loads is what this part of a step waits for: one replica of 560
        // atoms (eight CTAs) 11.7 -> 10.4 us per step, of 304 (four) 8.65 -> 8.06, 64 of 560
        // (two, warp 0 freed) 19.2 -> 18.9.
        const int own = a1 - a0;
        const bool four = CL > 2 && 4 * own + 32 <= (int)blockDim.x;
        const int it = own * (four ? 4 : 1) + 32 <= (int)blockDim.x ? tid - 32 : tid;
        const int i0 = it < 0 ? a1 : a0 + (four ? it >> 2 : it);  // this thread's first atom
        auto load_first = [&](int b) -> AtomSums {
            AtomSums a = {};
            if (four) {
                if (it >= 0 && a0 + ((it & ~31) >> 2) < a1)
                    a = load_sums4<CL>(sm, sc, b, rank, min(i0, a1 - 1), grad);
            } else if (i0 < a1) {
                a = load_sums<CL>(sm, sc, b, rank, i0, grad);
            }
            return a;
        };
        AtomSums first = {};
        if (!TUBE) first = load_first((int)(step & 1));
        finish_evaluation<false, CL, TUBE>(sm, sc, P, (int)(step & 1), true);
        // position of `step` in the save cycle and ring slot of the next frame, kept as
        // counters so that the loop has no 64-bit divisions
        int save_phase = P.save_interval > 0 ? (int)(step % P.save_interval) : -1;
        int slot = P.max_frames > 0 ? (int)(sc.n_saved % P.max_frames) : 0;
        for (long long s = 0; s <= P.n_steps; ++s) {
            // B of the step just evaluated (s > 0), then A of the next one (s < n_steps)
            const bool do_b = s > 0, do_a = s < P.n_steps;
            const int b = (int)(step & 1), nb = b ^ 1;
            const bool bias = sc.bias_on;
            const bool save = do_b && save_phase == 0;
            const float kb = sc.kb;  // F_bias = kb G
            float vm2 = 0.f;  // largest |v after B|^2 + |v after O|^2 of this thread's atoms
            bool finite = true;
            // the other parity's partials were last read before this evaluation's cluster
            // barrier (here and in the other CTAs): clear them for the next one
            {
                uint4* f = (uint4*)sm.F(nb).L;
                uint4* g = (uint4*)sm.G(nb).L;
                for (int i = tid; i < 3 * sm.na8() / 2; i += blockDim.x)
                    f[i] = g[i] = make_uint4(0u, 0u, 0u, 0u);
            }
            if (TUBE) first = load_first(b);
            if (!four || (tid & 3) == 0) {
                for (int i = i0; i < a1; i += blockDim.x) {
                    const AtomSums a = i == i0 ? first : load_sums<CL>(sm, sc, b, rank, i, grad);
                    float4 v = sm.v()[i];
                    const float im = v.w;
                    float fx = a.fx, fy = a.fy, fz = a.fz;
                    if (bias) {
                        // (rounding spelled out: trajectories amplify the last bit)
                        const float bx = __fmul_rn(kb, a.gx), by = __fmul_rn(kb, a.gy),
                                    bz = __fmul_rn(kb, a.gz);
                        if (do_b)  // (rank 0 sums the bias functional)
                            rank_ptr<CL>(sm.xi(), 0)[i].w = fmaf(bz, bz, fmaf(bx, bx, __fmul_rn(by, by))) * im;
                        fx = __fadd_rn(fx, bx);
                        fy = __fadd_rn(fy, by);
                        fz = __fadd_rn(fz, bz);
                    }
                    float4 x = sm.xq()[i];
                    if (do_b) {  // B: closes the evaluated step
                        v.x = fmaf(hdt * im, fx, v.x);
                        v.y = fmaf(hdt * im, fy, v.y);
                        v.z = fmaf(hdt * im, fz, v.z);
                        if (save) {
                            float* fr = st.frames + 3 * (rep.frame_off + (long long)slot * n + i);
                            fr[0] = x.x;
                            fr[1] = x.y;
                            fr[2] = x.z;
                        }
                    }
                    if (do_a) {  // B A O A of the next step
                        v.x = fmaf(hdt * im, fx, v.x);
                        v.y = fmaf(hdt * im, fy, v.y);
                        v.z = fmaf(hdt * im, fz, v.z);
                        const float v1 = fmaf(v.x, v.x, fmaf(v.y, v.y, v.z * v.z));
                        x.x = fmaf(hdt, v.x, x.x);
                        x.y = fmaf(hdt, v.y, x.y);
                        x.z = fmaf(hdt, v.z, x.z);
                        const float4 xi = sm.xi()[i];  // drawn during the evaluation
                        v.x = fmaf(P.c1, v.x, xi.x);
                        v.y = fmaf(P.c1, v.y, xi.y);
                        v.z = fmaf(P.c1, v.z, xi.z);
                        x.x = fmaf(hdt, v.x, x.x);
                        x.y = fmaf(hdt, v.y, x.y);
                        x.z = fmaf(hdt, v.z, x.z);
                        vm2 = fmaxf(vm2, v1 + fmaf(v.x, v.x, fmaf(v.y, v.y, v.z * v.z)));
                        finite = finite && isfinite(x.x) && isfinite(x.y) && isfinite(x.z) &&
                                 isfinite(v.x) && isfinite(v.y) && isfinite(v.z);
#pragma unroll
                        for (int q = 0; q < CL; ++q) rank_ptr<CL>(sm.xq(), q)[i] = x;
                    }
                    sm.v()[i] = v;
                }
            }
            if (do_a) {  // largest speed of the step (positive floats order as their bits)
                const unsigned wm = __reduce_max_sync(kFull, finite ? __float_as_uint(vm2) : kNonFinite);
                if (lane < CL && wm) atomicMax(rank_ptr<CL>(&sc.vmax2[b], lane), wm);
            }
            if (tid == 0) {
                sc.flag[nb] = 0;
                sc.vmax2[nb] = 0u;
                sc.zw[nb][0] = sc.zw[nb][1] = sc.zw[nb][2] = 0u;
            }
            cluster_barrier<CL>();  // every CTA has the new positions
            if (rank == 0 && warp == 0 && do_b && bias) {  // atoms in a fixed order, whatever the CTA shape
                float tsum = 0.f;
                for (int i = lane; i < n; i += 32) tsum += sm.xi()[i].w;
                tsum = warp_sum_f(tsum);
                if (lane == 0) sc.T += P.dt_over_gamma * (double)tsum;
            }
            if (tid == 0 && do_b) {
                if (save) {
                    if (rank == 0) {
                        const long long fi = (long long)r * P.max_frames + slot;
                        st.fz[fi] = sc.z;
                        st.fzm[fi] = sc.zm;
                        st.fe[fi] = sc.epot;
                        st.fT[fi] = sc.T;
                    }
                    sc.n_saved += 1;
                }
            }
            // leave after the last B, when a force was out of range, or when the new state is
            // non-finite. Every thread of the cluster must leave at the same place, so each word
            // read here is one that no CTA can write before all have read it: the force-range bit
            // belongs to a decision and the speed bound to an update, with a cluster barrier
            // between either and its next writer. (One word for both would let a CTA that is
            // already in the next update stop one that still has to take it.)
            if (save) slot = slot + 1 == P.max_frames ? 0 : slot + 1;
            const unsigned vmax = sc.vmax2[b];
            nonfinite = do_a && vmax == kNonFinite;
            if (!do_a || sc.status != 0 || nonfinite) break;
            ++step;
            if (save_phase >= 0) save_phase = save_phase + 1 == P.save_interval ? 0 : save_phase + 1;
            // |x_new - x_old| <= dt/2 (|v after B| + |v after O|) <= dt/2 sqrt(2 vmax2) per
            // atom; a pair inside r_c now was inside r_c + 2 disp at the build, so the list
            // stays complete while 2 disp < skin (a 1 % margin covers the FP32 rounding)
            disp += hdt * sqrtf(2.0f * __uint_as_float(vmax));
            ++since;
            if (disp >= 0.99f * P.skin_half || (P.rebuild_every > 0 && since >= P.rebuild_every)) {
                build_list<CL>(sm, sc, P.rlist2);
                disp = 0.f;
                since = 0;
                ++builds;
            }
            const bool save_next = save_phase == 0;
            if (save_next)
                evaluate_work<ELEC, true, CL, TUBE>(sm, sc, P, nb, true, rep.rep_id, step);
            else
                evaluate_work<ELEC, false, CL, TUBE>(sm, sc, P, nb, true, rep.rep_id, step);
            if (!TUBE) first = load_first(nb);
            if (save_next)
                finish_evaluation<true, CL, TUBE>(sm, sc, P, nb, true);
            else
                finish_evaluation<false, CL, TUBE>(sm, sc, P, nb, true);
            if (sc.status != 0) break;  // force out of range: frozen before the update
        }
    }
    __syncthreads();
    const int status = sc.status | (nonfinite ? SCPS_FLAG_NONFINITE : 0);
    // write back the state: each CTA the atoms it integrated, rank 0 the scalars
    for (int i = kTile * own_lo(tp.n_tiles, rank, CL) + tid;
         i < min(n, kTile * own_lo(tp.n_tiles, rank + 1, CL)); i += blockDim.x) {
        const float4 x = sm.xq()[i];
        st.x[rep.atom_off + i] = make_float4(x.x, x.y, x.z, 0.f);
        const float4 v = sm.v()[i];
        st.v[rep.atom_off + i] = make_float4(v.x, v.y, v.z, 0.f);
    }
    if (rank == 0) {
        if (tid == 0) {
            st.zm[r] = sc.zm;
            st.z[r] = sc.z;
            st.sm[r] = sc.sm;
            st.wm[r] = sc.wm;
            st.T[r] = sc.T;
            st.status[r] = status;
            st.step[r] = step;
            st.n_saved[r] = sc.n_saved;
            if (st.pair_slots && status == 0 && P.n_steps > 0) st.pair_slots[r] = sc.pair_slots;
            if (st.list_builds) st.list_builds[r] = builds;
        }
    }
    cluster_barrier<CL>();  // no CTA leaves while its shared memory may still be read
}

// Energy, forces and z of n_frames configurations (no bias, no state); one cluster of CL
// CTAs per frame, each cluster with its own list slab. With CL > 1 the work is split
// between the CTAs as in the resident kernel and each CTA writes its share of the atoms'
// forces, summing the fixed-point partials of all (the same integers as with one CTA).
template <int ELEC, int CL>
__global__ void __launch_bounds__(1024, 1)
k_eval_frames(const TopoDev* __restrict__ topo_ptr, RunParams P, const float* __restrict__ X,
              double* __restrict__ U, float* __restrict__ F, double* __restrict__ Z, int nta,
              int lc_cap) {
    __shared__ Scalars sc;
    const long long f = blockIdx.x / CL;
    const int rank = cta_rank<CL>();
    if (threadIdx.x == 0) {
        sc.tp = *topo_ptr;
        sc.pc = P.pc;
        sc.list = list_of<CL>(P.list_base + (blockIdx.x / CL) * P.list_slab, nta, rank);
    }
    __syncthreads();
    const TopoDev& tp = sc.tp;
    const Shared sm = {nta, lc_cap, tp.f_shift, tp.g_shift};
    const int n = tp.n_atoms;
    const float* xf = X + f * n * 3;
    for (int i = threadIdx.x; i < sm.na8(); i += blockDim.x) {
        if (i < n) {
            sm.xq()[i] = make_float4(xf[3 * i], xf[3 * i + 1], xf[3 * i + 2], tp.qs[i]);
            sm.lj()[i] = tp.lj[i];
        } else {
            sm.xq()[i] = far_slot(i);
            sm.lj()[i] = make_float2(0.f, 0.f);
        }
    }
    for (int i = threadIdx.x; i < 24 * sm.na8(); i += blockDim.x) sm.F(0).L[i] = 0u;  // F and G
    if (threadIdx.x == 0) {
        sc.zm = 0.0;
        sc.z = 0.0;
        sc.status = 0;
        sc.flag[0] = 0;
        sc.zw[0][0] = sc.zw[0][1] = sc.zw[0][2] = 0u;
        sc.work_next[0] = 0;
    }
    cluster_barrier<CL>();  // every CTA of the cluster is initialised before any remote access
    build_list<CL>(sm, sc, P.rlist2);
    evaluate_work<ELEC, true, CL, false>(sm, sc, P, 0, false, 0u, -1);
    finish_evaluation<true, CL, false>(sm, sc, P, 0, false);
    if (F) {
        float* ff_out = F + f * n * 3;
        const Part own = sm.F(0);
        // one component per thread: the words of a small share come from many threads at once
        for (int k = threadIdx.x + rank * blockDim.x; k < 3 * n; k += CL * blockDim.x) {
            int h = own.H[k];
            unsigned l = own.L[k];
#pragma unroll
            for (int q = 1; q < CL; ++q) {
                h += rank_ptr<CL>(own.H, (rank + q) & (CL - 1))[k];
                l += rank_ptr<CL>(own.L, (rank + q) & (CL - 1))[k];
            }
            ff_out[k] = fix2f(join_coarse(h, l, sm.fsh) * 128);  // 2^-13 to 2^-20 units
        }
    }
    if (threadIdx.x == 0 && rank == 0) {
        U[f] = sc.epot;
        if (Z) Z[f] = sc.z;
    }
    cluster_barrier<CL>();  // no CTA leaves while its shared memory may still be read
}

// Shared memory of a launch (kern_chain.cu).
size_t launch_smem(int nta, int threads, int cl, int* lc_cap);

// Grid of `count` clusters of CL CTAs.
template <int CL>
struct ClusterLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    ClusterLaunch(long long count, int threads, size_t smem, cudaStream_t stream) {
        cfg.gridDim = dim3((unsigned)(count * CL));
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = CL;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
};

template <int ELEC, int CL, bool TUBE, bool WIDE>
static cudaError_t launch_resident_t(const TopoDev* topos, const RepDev* reps, const StateDev& st,
                                     const RunParams& P, int nta, int threads, cudaStream_t stream) {
    int lc_cap = 0;
    const size_t smem = launch_smem(nta, threads, CL, &lc_cap);
    auto kern = k_resident<ELEC, CL, TUBE, WIDE>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const ClusterLaunch<CL> L(P.n_replicas, threads, smem, stream);
    e = cudaLaunchKernelEx(&L.cfg, kern, topos, reps, st, P, nta, lc_cap);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template <int CL, bool WIDE>
cudaError_t launch_resident_cl(int elec, const TopoDev* topos, const RepDev* reps,
                                      const StateDev& st, const RunParams& P, int nta, int threads,
                                      cudaStream_t stream) {
    if (P.bias == 5) {  // contact-map tube bias: its own instantiation
        switch (elec) {
            case ELEC_DDIEL: return launch_resident_t<ELEC_DDIEL, CL, true, WIDE>(topos, reps, st, P, nta, threads, stream);
            case ELEC_RF: return launch_resident_t<ELEC_RF, CL, true, WIDE>(topos, reps, st, P, nta, threads, stream);
            case ELEC_PLAIN: return launch_resident_t<ELEC_PLAIN, CL, true, WIDE>(topos, reps, st, P, nta, threads, stream);
            default: return launch_resident_t<ELEC_NONE, CL, true, WIDE>(topos, reps, st, P, nta, threads, stream);
        }
    }
    switch (elec) {
        case ELEC_DDIEL: return launch_resident_t<ELEC_DDIEL, CL, false, WIDE>(topos, reps, st, P, nta, threads, stream);
        case ELEC_RF: return launch_resident_t<ELEC_RF, CL, false, WIDE>(topos, reps, st, P, nta, threads, stream);
        case ELEC_PLAIN: return launch_resident_t<ELEC_PLAIN, CL, false, WIDE>(topos, reps, st, P, nta, threads, stream);
        default: return launch_resident_t<ELEC_NONE, CL, false, WIDE>(topos, reps, st, P, nta, threads, stream);
    }
}

template <int ELEC, int CL>
static cudaError_t launch_eval_t(const TopoDev* topo, const RunParams& P, const float* X, double* U,
                                 float* F, double* Z, long long n_frames, int nta, int threads,
                                 cudaStream_t stream) {
    int lc_cap = 0;
    const size_t smem = launch_smem(nta, threads, CL, &lc_cap);
    auto kern = k_eval_frames<ELEC, CL>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const ClusterLaunch<CL> L(n_frames, threads, smem, stream);
    e = cudaLaunchKernelEx(&L.cfg, kern, topo, P, X, U, F, Z, nta, lc_cap);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template <int CL>
cudaError_t launch_eval_cl(int elec, const TopoDev* topo, const RunParams& P, const float* X, double* U,
                           float* F, double* Z, long long n_frames, int nta, int threads,
                           cudaStream_t stream) {
    switch (elec) {
        case ELEC_DDIEL: return launch_eval_t<ELEC_DDIEL, CL>(topo, P, X, U, F, Z, n_frames, nta, threads, stream);
        case ELEC_RF: return launch_eval_t<ELEC_RF, CL>(topo, P, X, U, F, Z, n_frames, nta, threads, stream);
        case ELEC_PLAIN: return launch_eval_t<ELEC_PLAIN, CL>(topo, P, X, U, F, Z, n_frames, nta, threads, stream);
        default: return launch_eval_t<ELEC_NONE, CL>(topo, P, X, U, F, Z, n_frames, nta, threads, stream);
    }
}

// Clusters of CL CTAs that the device can run at once in the given shape (0 on failure).
template <int CL>
int max_clusters_cl(int nta, int threads) {
    int lc_cap = 0, n = 0;
    const size_t smem = launch_smem(nta, threads, CL, &lc_cap);
    auto kern = k_resident<ELEC_DDIEL, CL, true, true>;
    const ClusterLaunch<CL> L(1, threads, smem, 0);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kern, &L.cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return n;
}

#define SCPS_RESIDENT_LAUNCHERS(PREFIX, CL, WIDE)                                                   \
    PREFIX template cudaError_t launch_resident_cl<CL, WIDE>(int, const TopoDev*, const RepDev*,    \
                                                             const StateDev&, const RunParams&,     \
                                                             int, int, cudaStream_t);
#define SCPS_EVAL_LAUNCHERS(PREFIX, CL)                                                             \
    PREFIX template cudaError_t launch_eval_cl<CL>(int, const TopoDev*, const RunParams&,           \
                                                   const float*, double*, float*, double*,          \
                                                   long long, int, int, cudaStream_t);
#define SCPS_MAX_CLUSTERS(PREFIX, CL) PREFIX template int max_clusters_cl<CL>(int, int);

// bytes of the kernels' static shared block
constexpr size_t kChainStaticSmem = sizeof(Scalars);

}  // namespace scps
