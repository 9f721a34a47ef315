// Solvated periodic box: rMD replicas of one chain in LJ + Coulomb solvent
// (reaction field), cubic box, column-sorted slots and atom-level pair lists.
//
// Per step (kernels in stream order):
//   [rebuild, when due]  wrap; sort atoms into ncol x ncol columns in (x, y),
//                        by z inside a column (ties by atom id); cut every
//                        column into tiles of 32 slots (the last one padded);
//                        inside a tile, order by x into two halves of 16 and
//                        each half by y, so that slots 8q..8q+7 form a compact
//                        cluster; cluster boxes; per 8-slot cluster the list
//                        of atoms of later clusters within r_c + skin of one of
//                        its atoms, each with the periodic shift of its cluster
//                        (the cluster takes the minimum image pair by pair where
//                        that shift might not hold until the next rebuild)
//   pairs                one warp per cluster, 64 list entries at a
//                        time on quarter warps, every pair once; all force
//                        terms summed in fixed point (order-free)
//   chain                one CTA per replica: bonds, angles, z(X) of Eq.
//                        (zrMD), the ratchet of Eq. (FrMD), the bias force
//   integrate            BAOAB half steps with Philox noise keyed by atom id
// A rebuild is due every `rebuild_every` steps, or earlier when an atom has
// moved more than skin/2 since the last one, so every pair inside the cutoff
// is always in the list; once one live replica is due, all live replicas of the
// batch rebuild together. Forces are integer sums of per-pair terms (order-free);
// positions are wrapped into the box at each rebuild, so runs that rebuild at
// other steps agree to rounding.
#include <type_traits>

#include "scps_internal.h"

namespace scps {

namespace {

constexpr unsigned kFullB = 0xffffffffu;
constexpr int kNumKeys = 8192;  // ncol^2 * nz <= kNumKeys
constexpr int kMaxCols = 256;   // ncol <= 16
constexpr int kSortThreads = 1024;
// k_box_pairs: warps (clusters) per CTA and warps per SM. One warp per CTA: the lists of a
// tile's clusters differ in length, and warps of one CTA would wait for the longest (16 x
// 24 560 sites: 388 us against 423 with four). 20 warps leave 96 registers each; 24 and 28
// take 398 and 408 us, since the kernel is bound by its instruction mix, not by latency.
constexpr int kPairWarps = 1;
constexpr int kPairRegWarps = 20;

__device__ __forceinline__ float wrapc(float x, float L, float invL) {
    return x - L * floorf(x * invL);
}

__device__ __forceinline__ float min_img(float d, float L, float invL) {
    return d - L * rintf(d * invL);
}

// The same for two differences (rint by the addition that drops the fraction bits, exact for
// quotients below 2^22).
__device__ __forceinline__ float2 min_img2(float2 d, float L, float invL) {
    const float2 q = add2(mul2(d, dup2(invL)), dup2(12582912.0f));
    return fma2(dup2(-L), add2(q, dup2(-12582912.0f)), d);
}

// number of lanes whose (key, lane) is below this lane's
__device__ __forceinline__ int warp_rank(float key, int lane, bool member, unsigned group) {
    int rank = 0;
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
        const float kk = __shfl_sync(kFullB, key, k);
        const bool in = (group >> k) & 1u;
        rank += (member && in && (kk < key || (kk == key && k < lane))) ? 1 : 0;
    }
    return rank;
}

}  // namespace

// Rebuild decision of replicas [r0, r0 + nr) by one CTA: a replica rebuilds when forced
// (need set), or, when `auto_ok`, as soon as one live replica of the batch is due (its
// rebuild_every steps are up or its largest displacement reaches skin/2). Lists of all live
// replicas are then rebuilt together: one rebuild of the whole batch keeps the GPU full,
// where replicas due at different steps would each rebuild alone. Values are read before
// any is written, so the decision is the same whatever the thread order. Returns 1 to all
// threads when some replica rebuilds.
__device__ int box_decide_batch(const BoxDev& B, const StateDev& st, int r0, int nr, int auto_ok) {
    int due = 0;
    if (auto_ok)
        for (int r = r0 + threadIdx.x; r < r0 + nr; r += blockDim.x) {
            const float d2 = __uint_as_float(B.maxd2[r]);
            due |= st.status[r] == 0 && (B.since[r] >= B.rebuild_every || d2 >= B.skin2_quarter);
        }
    due = __syncthreads_or(due);
    int any = 0;
    for (int r = r0 + threadIdx.x; r < r0 + nr; r += blockDim.x) {
        const int decide = st.status[r] == 0 && (B.need[r] || due);
        B.need[r] = decide;  // the later rebuild kernels run iff set
        if (decide) {
            B.since[r] = 0;
            B.maxd2[r] = 0u;
            B.nbuild[r] += 1;
        }
        any |= decide;
    }
    return __syncthreads_or(any);
}

// Rebuild, step 1a: the decision (one CTA for the batch); the key counts of the replicas
// that rebuild are cleared by k_box_clear_hist.
__global__ void k_box_decide(BoxDev B, StateDev st, int r0, int nr, int auto_ok) {
    box_decide_batch(B, st, r0, nr, auto_ok);
}

// Graph form of step 1a (one CTA for all R replicas): the same decision, and the graph's
// conditional value: 1 when some replica rebuilds, so that the rebuild kernels run at all
// only then.
__global__ void k_box_decide_graph(BoxDev B, StateDev st, int R, cudaGraphConditionalHandle h) {
    const int any = box_decide_batch(B, st, 0, R, 1);
    if (threadIdx.x == 0) {
        cudaGraphSetConditional(h, any ? 1u : 0u);
        if (any) B.nevent[0] += 1;
    }
}

__global__ void k_box_clear_hist(BoxDev B, int r0) {
    const int r = blockIdx.y + r0;
    if (!B.need[r]) return;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < kNumKeys) B.hist[(size_t)r * kNumKeys + k] = 0;
}

// Rebuild, step 1b (slots): wrap into the box, key = (column, z bin), count keys.
__global__ void k_box_key(BoxDev B, int r0) {
    const int r = blockIdx.y + r0;
    if (!B.need[r]) return;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= B.np) return;
    const size_t base = (size_t)r * B.np;
    B.id2[base + s] = -1;
    const int a = B.id[base + s];
    if (a < 0) return;
    float4 p = B.pos[base + s];
    p.x = wrapc(p.x, B.L, B.invL);
    p.y = wrapc(p.y, B.L, B.invL);
    p.z = wrapc(p.z, B.L, B.invL);
    B.pos[base + s] = p;
    const float cs = (float)B.ncol * B.invL, zs = (float)B.nz * B.invL;
    const int qx = min((int)(p.x * cs), B.ncol - 1), qy = min((int)(p.y * cs), B.ncol - 1),
              qz = min((int)(p.z * zs), B.nz - 1);
    const int k = (qx * B.ncol + qy) * B.nz + qz;
    B.key[base + s] = k;
    atomicAdd(&B.hist[(size_t)r * kNumKeys + k], 1);
}

// Rebuild, step 1c (one CTA of 1024 threads per replica): exclusive scan of the
// key counts (they become running cursors); first compact position and first
// tile of every column (each column starts a tile); the coarse unit of the force sums.
__global__ void __launch_bounds__(kSortThreads) k_box_scan(BoxDev B, int r0) {
    __shared__ int wtot[32];
    __shared__ int tiles[kMaxCols], most;
    const int r = blockIdx.x + r0;
    if (!B.need[r]) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    int* hist = B.hist + (size_t)r * kNumKeys;
    int* col_first = B.colinfo + (size_t)r * 2 * (kMaxCols + 1);
    int* col_tile = col_first + kMaxCols + 1;
    constexpr int kPer = kNumKeys / kSortThreads;
    int loc[kPer], sum = 0;
    const int k0 = tid * kPer;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        loc[q] = hist[k0 + q];
        sum += loc[q];
    }
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFullB, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wtot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int t = lane < nw ? wtot[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFullB, t, o);
            if (lane >= o) t += y;
        }
        wtot[lane] = t;
    }
    __syncthreads();
    int run = (warp > 0 ? wtot[warp - 1] : 0) + x - sum;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        hist[k0 + q] = run;
        run += loc[q];
    }
    __syncthreads();
    const int ncols = B.ncol * B.ncol;
    for (int c = tid; c <= ncols; c += blockDim.x) col_first[c] = c < ncols ? hist[c * B.nz] : B.n_atoms;
    __syncthreads();
    if (warp == 0) {  // prefix sums of the columns' tiles, kMaxCols / 32 columns per lane
        constexpr int kCols = kMaxCols / 32;
        int nt[kCols], sum = 0;
#pragma unroll
        for (int q = 0; q < kCols; ++q) {
            const int c = kCols * lane + q;
            nt[q] = c < ncols ? (col_first[c + 1] - col_first[c] + 31) >> 5 : 0;
            sum += nt[q];
        }
        int x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFullB, x, o);
            if (lane >= o) x += y;
        }
        int t = x - sum;
#pragma unroll
        for (int q = 0; q < kCols; ++q) {
            const int c = kCols * lane + q;
            if (c <= ncols) col_tile[c] = t;  // (the end: <= nt by the capacity ceil(n/32) + ncol^2)
            t += nt[q];
        }
        if (lane == 31 && ncols == kMaxCols) col_tile[ncols] = t;
        if (lane == 0) most = 0;
    }
    __syncthreads();
    // A slot takes one sum from every list it is in and one for its own cluster's share. Only
    // clusters of the columns in reach can list it (k_box_list), so four times the most tiles in
    // reach of a column bounds the lists; the coarse unit is chosen for that many terms.
    const int reach = (int)ceilf(sqrtf(B.rlist2) / (B.L / (float)B.ncol));
    const int span = min(2 * reach + 1, B.ncol);  // columns in reach, per axis
    for (int c = tid; c < ncols; c += blockDim.x) {
        int sum = 0;
        for (int d = 0; d < span; ++d) {
            const int q = c / B.ncol * B.ncol + (c % B.ncol + d) % B.ncol;
            sum += col_tile[q + 1] - col_tile[q];
        }
        tiles[c] = sum;  // of `span` columns from c on in y
    }
    __syncthreads();
    for (int c = tid; c < ncols; c += blockDim.x) {
        int sum = 0;
        for (int d = 0; d < span; ++d) sum += tiles[(c / B.ncol + d) % B.ncol * B.ncol + c % B.ncol];
        atomicMax(&most, sum);  // (of the span x span columns from c on: every centre comes up once)
    }
    __syncthreads();
    if (tid == 0) B.shift[r] = coarse_shift(4ll * most + 1, kBoxShift);
}

// Rebuild, step 1d (atoms): the atom ids go into the padded column layout, positions and
// velocities into atom order (step 1f gathers them). Within a key the atomics give an
// arbitrary order, which step 1e replaces by atom-id order.
__global__ void k_box_scatter(BoxDev B, int r0) {
    const int r = blockIdx.y + r0;
    if (!B.need[r]) return;
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= B.n_atoms) return;
    const size_t base = (size_t)r * B.np;
    const int* col_first = B.colinfo + (size_t)r * 2 * (kMaxCols + 1);
    const int* col_tile = col_first + kMaxCols + 1;
    const int s = B.slot_of[(size_t)r * B.n_atoms + a];
    const int k = B.key[base + s];
    const int p = atomicAdd(&B.hist[(size_t)r * kNumKeys + k], 1);
    const int c = k / B.nz;
    const int dst = col_tile[c] * 32 + (p - col_first[c]);
    B.pos2[base + a] = B.pos[base + s];
    B.vel2[base + a] = B.vel[base + s];
    B.id2[base + dst] = a;
}

// Rebuild, step 1e (slots): each key's atoms in id order, from id2 to id; a slot's rank is
// the number of smaller ids of its key (a few loads side by side; an insertion sort per key, a
// chain of dependent ones, took 51 us where this takes 8). hist[k] now ends key k, so
// key k spans [hist[k - 1], hist[k]).
__global__ void k_box_keyorder(BoxDev B, int r0) {
    const int r = blockIdx.y + r0;
    if (!B.need[r]) return;
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= B.np) return;
    const size_t base = (size_t)r * B.np;
    const int a = B.id2[base + d];
    if (a < 0) {
        B.id[base + d] = -1;
        return;
    }
    const int* hist = B.hist + (size_t)r * kNumKeys;
    const int* col_first = B.colinfo + (size_t)r * 2 * (kMaxCols + 1);
    const int* col_tile = col_first + kMaxCols + 1;
    const int k = B.key[base + B.slot_of[(size_t)r * B.n_atoms + a]];
    const int c = k / B.nz;
    const int lo = k > 0 ? hist[k - 1] : 0, hi = hist[k];
    const size_t off = base + col_tile[c] * 32 - col_first[c];
    int rank = 0;
    for (int q = lo; q < hi; ++q) rank += B.id2[off + q] < a ? 1 : 0;
    B.id[off + lo + rank] = a;
}

// Rebuild, step 1f (one warp per tile): inside each tile, two halves of 16 by x,
// each ordered by y (padding last), so that slots 8q .. 8q+7 form compact
// clusters; final slot arrays, reference positions, LJ parameters, slot_of.
__global__ void k_box_subsort(BoxDev B, const TopoDev* __restrict__ topo, int r0) {
    const int r = blockIdx.y + r0;
    if (!B.need[r]) return;
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= B.nt) return;
    const int lane = threadIdx.x & 31;
    const size_t base = (size_t)r * B.np;
    const int s0 = t * 32 + lane;
    const int a = B.id[base + s0];  // (the other lanes read theirs before any write below)
    const bool valid = a >= 0;
    const float4 p = B.pos2[base + max(a, 0)];
    const float4 v = B.vel2[base + max(a, 0)];
    const float kx = valid ? p.x : 3.0e38f, ky = valid ? p.y : 3.0e38f;
    const int rx = warp_rank(kx, lane, true, kFullB);
    const unsigned upper = __ballot_sync(kFullB, rx >= 16);
    const bool hi = rx >= 16;
    const int ry = warp_rank(ky, lane, true, hi ? upper : ~upper);
    const int s = t * 32 + (hi ? 16 : 0) + ry;
    if (valid) {
        B.pos[base + s] = p;
        B.vel[base + s] = v;
        B.id[base + s] = a;
        B.pos_ref[base + s] = p;
        B.par[base + s] = topo->lj[a];
        B.slot_of[(size_t)r * B.n_atoms + a] = s;
    } else {
        const float4 far = make_float4(1.0e5f * (float)(s + 1), 0.f, 0.f, 0.f);
        B.pos[base + s] = far;
        B.vel[base + s] = make_float4(0.f, 0.f, 0.f, 0.f);
        B.id[base + s] = -1;
        B.pos_ref[base + s] = far;
        B.par[base + s] = make_float2(0.f, 0.f);
    }
}

// Rebuild step 2 (one warp per tile): boxes of the tile and of each 8-slot cluster, and whether
// the cluster holds chain atoms or only atoms with the LJ parameters of the last atom (a solvent
// site), whose pair constants the pair kernel then computes once.
__global__ void k_box_tiles(BoxDev B, const TopoDev* __restrict__ topo, int r0) {
    const int r = blockIdx.y + r0;
    if (!B.need[r]) return;
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= B.nt) return;
    const int lane = threadIdx.x & 31;
    const int s = t * 32 + lane;
    const float4 p = B.pos[(size_t)r * B.np + s];
    const int a = B.id[(size_t)r * B.np + s];
    const bool valid = a >= 0;
    const float2 ref = topo->lj[B.n_atoms - 1];
    const float2 par = B.par[(size_t)r * B.np + s];
    const unsigned pure = __ballot_sync(kFullB, !valid || (par.x == ref.x && par.y == ref.y));
    const unsigned chain = __ballot_sync(kFullB, valid && a < B.n_chain);
    float lx = valid ? p.x : 3.0e38f, ly = valid ? p.y : 3.0e38f, lz = valid ? p.z : 3.0e38f;
    float hx = valid ? p.x : -3.0e38f, hy = valid ? p.y : -3.0e38f, hz = valid ? p.z : -3.0e38f;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        lx = fminf(lx, __shfl_xor_sync(kFullB, lx, o));
        ly = fminf(ly, __shfl_xor_sync(kFullB, ly, o));
        lz = fminf(lz, __shfl_xor_sync(kFullB, lz, o));
        hx = fmaxf(hx, __shfl_xor_sync(kFullB, hx, o));
        hy = fmaxf(hy, __shfl_xor_sync(kFullB, hy, o));
        hz = fmaxf(hz, __shfl_xor_sync(kFullB, hz, o));
    }
    if ((lane & 7) == 0) {  // the box of the 8-slot cluster of this lane
        const size_t c = (size_t)r * 4 * B.nt + 4 * t + (lane >> 3);
        const unsigned mine = 0xffu << (lane & ~7);
        const bool cpure = (pure & mine) == mine;
        B.clo[c] = make_float4(lx, ly, lz, cpure ? 1.f : 0.f);
        B.chi[c] = make_float4(hx, hy, hz, 0.f);
        B.cflag[c] = ((chain & mine) ? 1 : 0) | (cpure ? 4 : 0);
    }
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) {  // and of the tile
        lx = fminf(lx, __shfl_xor_sync(kFullB, lx, o));
        ly = fminf(ly, __shfl_xor_sync(kFullB, ly, o));
        lz = fminf(lz, __shfl_xor_sync(kFullB, lz, o));
        hx = fmaxf(hx, __shfl_xor_sync(kFullB, hx, o));
        hy = fmaxf(hy, __shfl_xor_sync(kFullB, hy, o));
        hz = fmaxf(hz, __shfl_xor_sync(kFullB, hz, o));
    }
    if (lane == 0) {
        B.tlo[(size_t)r * B.nt + t] = make_float4(lx, ly, lz, 0.f);
        B.thi[(size_t)r * B.nt + t] = make_float4(hx, hy, hz, 0.f);
    }
}

// Rebuild step 3 (one warp per 8-slot i cluster c): the pair list of c. Its own 8 slots
// come first (the pair kernel takes those pairs once, j slot after i slot); then, from the
// clusters after c in slot order whose boxes come within r_list of c's box, the atoms within
// r_list of some atom of c (minimum-image distances), in ascending slot order. Each entry
// carries the periodic shift s (per axis -1, 0 or 1 in units of L) that takes its cluster's
// box centre nearest to c's. Where a coordinate difference of some atom of c and the entry
// under s, plus the skin (the most two atoms can close in before the next rebuild), reaches
// L / 2, s may stop being the minimum image of that pair: c is then flagged for the per-pair
// minimum image.
//
// One CTA per tile, one warp per cluster. Instructions bound it, so the candidates narrow in
// three steps: the CTA's warps share a test of tile boxes against the tile's box (32 tiles at a
// time, over the columns in reach), each warp tests the clusters of the hit tiles (eight tiles
// at a time), and the hit clusters' atoms are tested in batches of 64, two per lane in packed
// operations (16 x 24 560 sites, a rebuild of all lists: 292 us, and 662 with each warp scanning all
// clusters of the columns and taking 32 atoms at a time).
constexpr int kListWords = 16;  // 32-tile words of a segment of the tile test

__global__ void __launch_bounds__(128) k_box_list(BoxDev B, StateDev st, int r0) {
    __shared__ float4 sxi[4][8];
    __shared__ int col_tile[kMaxCols + 1];  // first tile of each column (and the end)
    __shared__ unsigned word[kListWords];   // hit tiles of a segment, 32 per word, from tile wt[]
    __shared__ int wt[kListWords];
    __shared__ int tile_hit[32 * kListWords];  // the same as a list
    __shared__ uint32_t cand[4][40];           // per warp: hit clusters and their shift codes
    const int r = blockIdx.y + r0;
    if (!B.need[r]) return;
    const int ncl = 4 * B.nt;
    const int ncols = B.ncol * B.ncol;
    for (int k = threadIdx.x; k <= ncols; k += blockDim.x)
        col_tile[k] = B.colinfo[(size_t)r * 2 * (kMaxCols + 1) + kMaxCols + 1 + k];
    __syncthreads();
    const int w = threadIdx.x >> 5;
    const int tt = blockIdx.x, c = 4 * tt + w;
    const int lane = threadIdx.x & 31, l8 = lane & 7, q = lane >> 3;
    const unsigned lt = (1u << lane) - 1u;
    const size_t base = (size_t)r * B.np;
    const size_t ci = (size_t)r * ncl + c;
    uint32_t* out = B.ent + ci * B.max_ent;
    constexpr uint32_t kNoShift = (1u << 24) | (1u << 26) | (1u << 28);
    const float4 al = B.clo[ci], ah = B.chi[ci];
    const int si = 8 * c + l8;
    const unsigned ivalid = __ballot_sync(kFullB, B.id[base + si] >= 0) & 0xffu;
    if (lane < 8) {
        sxi[w][lane] = B.pos[base + si];
        out[lane] = (uint32_t)si | kNoShift | (al.w != 0.f ? 1u << 30 : 0u);
    }
    __syncwarp();
    int count = 8;
    bool inexact = false;
    const float room = 0.5f * B.L - 2.0f * sqrtf(B.skin2_quarter);  // L/2 - skin
    const float cx = 0.5f * (al.x + ah.x), cy = 0.5f * (al.y + ah.y), cz = 0.5f * (al.z + ah.z);
    const float hx = 0.5f * (ah.x - al.x), hy = 0.5f * (ah.y - al.y), hz = 0.5f * (ah.z - al.z);
    int nc = 0;  // hit clusters waiting in cand[w]

    // atoms of the hit clusters cand[w][0 .. nh), nh <= 8: lane 8 k + a takes atom a of the
    // k-th and of the (k + 4)-th
    auto take_atoms = [&](int nh) {
        uint32_t h[2];
        float4 x[2];
        bool in[2], keep[2];
        float px[2], py[2], pz[2], dm[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            h[u] = q + 4 * u < nh ? cand[w][q + 4 * u] : 0u;
            const int sj = 8 * (int)(h[u] & 0xffffffu) + l8;  // (the first cluster's where there is none)
            in[u] = B.id[base + sj] >= 0 && q + 4 * u < nh;
            x[u] = B.pos[base + sj];
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {  // under the cluster's shift
            px[u] = x[u].x + (float)((int)((h[u] >> 24) & 3u) - 1) * B.L;
            py[u] = x[u].y + (float)((int)((h[u] >> 26) & 3u) - 1) * B.L;
            pz[u] = x[u].z + (float)((int)((h[u] >> 28) & 3u) - 1) * B.L;
            // dm bounds every per-axis separation from c's atoms
            dm[u] = fmaxf(fabsf(px[u] - cx) + hx, fmaxf(fabsf(py[u] - cy) + hy, fabsf(pz[u] - cz) + hz));
        }
        float2 d2 = dup2(3.0e38f);
#pragma unroll
        for (int t = 0; t < 8; ++t) {  // empty slots of c sit far away (x beyond 1e5 nm)
            const float4 a = sxi[w][t];
            const float2 dx = make_float2(px[0] - a.x, px[1] - a.x),
                         dy = make_float2(py[0] - a.y, py[1] - a.y),
                         dz = make_float2(pz[0] - a.z, pz[1] - a.z);
            const float2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
            d2.x = fminf(d2.x, r2.x);
            d2.y = fminf(d2.y, r2.y);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            float d = u ? d2.y : d2.x;
            if (in[u] && !(dm[u] < 0.5f * B.L)) {  // the shift may not be the minimum image
                // box distance of the atom's own nearest image (in a small box not the
                // cluster's), which bounds that of every image
                const float bx = fmaxf(0.f, fabsf(min_img(x[u].x - cx, B.L, B.invL)) - hx),
                            by = fmaxf(0.f, fabsf(min_img(x[u].y - cy, B.L, B.invL)) - hy),
                            bz = fmaxf(0.f, fabsf(min_img(x[u].z - cz, B.L, B.invL)) - hz);
                d = 3.0e38f;
                if (fmaf(bx, bx, fmaf(by, by, bz * bz)) < B.rlist2)
                    for (int t = 0; t < 8; ++t) {
                        if (!((ivalid >> t) & 1u)) continue;
                        const float4 a = sxi[w][t];
                        const float mx = min_img(x[u].x - a.x, B.L, B.invL),
                                    my = min_img(x[u].y - a.y, B.L, B.invL),
                                    mz = min_img(x[u].z - a.z, B.L, B.invL);
                        d = fminf(d, fmaf(mx, mx, fmaf(my, my, mz * mz)));
                    }
            }
            keep[u] = in[u] && d < B.rlist2;
            inexact = inexact || (keep[u] && !(dm[u] < room));
            const unsigned kb = __ballot_sync(kFullB, keep[u]);
            const int pos = count + __popc(kb & lt);
            if (keep[u] && pos < B.max_ent)
                out[pos] = (uint32_t)(8 * (int)(h[u] & 0xffffffu) + l8) | (h[u] & 0x7f000000u);
            count += __popc(kb);
        }
    };

    // the hit tiles of ns words: their list, then (each warp) their clusters and atoms
    auto take_tiles = [&](int ns) {
        __syncthreads();
        const unsigned mine = lane < ns ? word[lane] : 0u;
        int incl = __popc(mine);
#pragma unroll
        for (int o = 1; o < kListWords; o <<= 1) {
            const int y = __shfl_up_sync(kFullB, incl, o);
            if (lane >= o) incl += y;
        }
        const int total = __shfl_sync(kFullB, incl, kListWords - 1);
        for (int k = w; k < ns; k += 4) {
            const unsigned m = word[k];
            const int off = __shfl_sync(kFullB, incl, k) - __popc(m);
            if ((m >> lane) & 1u) tile_hit[off + __popc(m & lt)] = wt[k] + lane;
        }
        __syncthreads();
        if (ivalid)
            for (int b = 0; b < total; b += 8) {
                const int k = b + (lane >> 2);
                const int jc = k < total ? 4 * tile_hit[k] + (lane & 3) : 0;
                bool hit = false;
                uint32_t code = 0;
                if (jc > c) {
                    const float4 bl = B.clo[(size_t)r * ncl + jc], bh = B.chi[(size_t)r * ncl + jc];
                    if (bl.x <= bh.x) {  // the cluster holds atoms
                        const float dx = 0.5f * (bl.x + bh.x) - cx, dy = 0.5f * (bl.y + bh.y) - cy,
                                    dz = 0.5f * (bl.z + bh.z) - cz;
                        const float sx = -rintf(dx * B.invL), sy = -rintf(dy * B.invL),
                                    sz = -rintf(dz * B.invL);
                        const float ex = fabsf(fmaf(sx, B.L, dx)), ey = fabsf(fmaf(sy, B.L, dy)),
                                    ez = fabsf(fmaf(sz, B.L, dz));
                        const float wx = hx + 0.5f * (bh.x - bl.x), wy = hy + 0.5f * (bh.y - bl.y),
                                    wz = hz + 0.5f * (bh.z - bl.z);
                        // lower bound of any periodic-image distance between the two boxes
                        const float gx = fmaxf(0.f, ex - wx), gy = fmaxf(0.f, ey - wy),
                                    gz = fmaxf(0.f, ez - wz);
                        hit = fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < B.rlist2;
                        code = ((uint32_t)(sx + 1.f) << 24) | ((uint32_t)(sy + 1.f) << 26) |
                               ((uint32_t)(sz + 1.f) << 28) | (bl.w != 0.f ? 1u << 30 : 0u);
                    }
                }
                const unsigned m = __ballot_sync(kFullB, hit);
                if (hit) cand[w][nc + __popc(m & lt)] = (uint32_t)jc | code;
                nc += __popc(m);
                __syncwarp();
                while (nc >= 8) {
                    take_atoms(8);
                    nc -= 8;
                    const uint32_t rest = lane < nc ? cand[w][8 + lane] : 0u;
                    __syncwarp();
                    if (lane < nc) cand[w][lane] = rest;
                    __syncwarp();
                }
            }
        __syncthreads();  // the words may be written again
    };

    const float4 tl = B.tlo[(size_t)r * B.nt + tt], th = B.thi[(size_t)r * B.nt + tt];
    if (tl.x <= th.x) {  // the tile holds atoms
        const float tx = 0.5f * (tl.x + th.x), ty = 0.5f * (tl.y + th.y), tz = 0.5f * (tl.z + th.z);
        const float ux = 0.5f * (th.x - tl.x), uy = 0.5f * (th.y - tl.y), uz = 0.5f * (th.z - tl.z);
        // r_list and room for the rounding of the box centres and widths
        const float rt = sqrtf(B.rlist2) + 4.0e-6f * B.L, rt2 = rt * rt;
        // candidate columns: an atom within r_list of c lies at most `reach` columns away in x
        // and in y (periodically); columns in ascending order keep the entries ascending
        const float colw = B.L / (float)B.ncol;
        const int reach = (int)ceilf(sqrtf(B.rlist2) / colw);
        int lo = 0, hi = ncols;  // the tile's column: the last one whose first tile is <= tt
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (col_tile[mid] <= tt) lo = mid; else hi = mid;
        }
        const int qx = lo / B.ncol, qy = lo % B.ncol;
        // the columns in reach in y: [y0, y1) and, around the face, [y2, ncol)
        int y0 = qy - reach, y1 = qy + reach + 1, y2 = B.ncol;
        if (2 * reach + 1 >= B.ncol) {
            y0 = 0;
            y1 = B.ncol;
        } else if (y0 < 0) {
            y2 = y0 + B.ncol;
            y0 = 0;
        } else if (y1 > B.ncol) {
            y2 = y0;
            y0 = 0;
            y1 -= B.ncol;
        }
        int ns = 0;  // words of the segment (the same in every warp; word k is warp k % 4's)
        for (int ix = 0; ix < B.ncol; ++ix) {
            const int ddx = abs(ix - qx);
            if (min(ddx, B.ncol - ddx) > reach) continue;
            for (int part = 0; part < 2; ++part) {
                const int a = ix * B.ncol + (part ? y2 : y0), e = ix * B.ncol + (part ? B.ncol : y1);
                if (a >= e) continue;
                const int t1 = col_tile[e];
                for (int t0 = max(tt, col_tile[a]); t0 < t1; t0 += 32) {
                    if ((ns & 3) == w) {
                        const int t = t0 + lane;
                        bool hit = false;
                        if (t < t1) {
                            const float4 bl = B.tlo[(size_t)r * B.nt + t], bh = B.thi[(size_t)r * B.nt + t];
                            const float dx = 0.5f * (bl.x + bh.x) - tx, dy = 0.5f * (bl.y + bh.y) - ty,
                                        dz = 0.5f * (bl.z + bh.z) - tz;
                            const float ex = fabsf(min_img(dx, B.L, B.invL)),
                                        ey = fabsf(min_img(dy, B.L, B.invL)),
                                        ez = fabsf(min_img(dz, B.L, B.invL));
                            const float gx = fmaxf(0.f, ex - (ux + 0.5f * (bh.x - bl.x))),
                                        gy = fmaxf(0.f, ey - (uy + 0.5f * (bh.y - bl.y))),
                                        gz = fmaxf(0.f, ez - (uz + 0.5f * (bh.z - bl.z)));
                            hit = bl.x <= bh.x && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < rt2;
                        }
                        const unsigned m = __ballot_sync(kFullB, hit);
                        if (lane == 0) {
                            word[ns] = m;
                            wt[ns] = t0;
                        }
                    }
                    if (++ns == kListWords) {
                        take_tiles(ns);
                        ns = 0;
                    }
                }
            }
        }
        if (ns > 0) take_tiles(ns);
        if (nc > 0) take_atoms(nc);
    }
    const int padded = (count + 7) & ~7;
    const int k = count + lane;
    if (k < padded && k < B.max_ent) out[k] = kBoxNoSlot | (1u << 30);  // padding: far, "pure"
    const bool overflow = padded > B.max_ent;
    const bool any_inexact = __any_sync(kFullB, inexact);
    if (lane == 0) {
        B.nent[ci] = overflow ? (B.max_ent & ~7) : padded;
        if (any_inexact) B.cflag[ci] |= 2;
        if (overflow) atomicOr(&st.status[r], SCPS_FLAG_LIST_OVERFLOW);
    }
}

// The i cluster of a warp in shared memory.
struct BoxCluster {
    float4 x[8];  // (x, y, z, qs)
    float2 lj[8];
    int id[8];
    unsigned long long ex[8];  // exclusion masks of its chain atoms
    unsigned redo[kBoxMaxEnt / 512];  // quarters of chunks to redo pair by pair, 8 chunks per word
};

// Adds an integer vector (2^-13 units) to the force sums of slot s (acc: the replica's three
// modular, three coarse and three upper arrays of np words); the coarse words only when a component
// rounds to a non-zero multiple of 2^sh. (Six words per slot side by side, which need fewer
// address computations, touch more sectors per atomic: 409 against 388 us.)
__device__ __forceinline__ void box_red3(const BoxDev& B, unsigned* acc, int sh, int s, int vx, int vy, int vz) {
    unsigned* L = acc + s;
    const size_t np = (size_t)B.np;
    atomicAdd(L, (unsigned)vx);
    atomicAdd(L + np, (unsigned)vy);
    atomicAdd(L + 2 * np, (unsigned)vz);
    const unsigned half = 1u << (sh - 1);
    if ((((unsigned)vx + half) | ((unsigned)vy + half) | ((unsigned)vz + half)) >> sh) {
        int* H = (int*)L + 3 * np;
        const int hx = ((vx >> (sh - 1)) + 1) >> 1, hy = ((vy >> (sh - 1)) + 1) >> 1,
                  hz = ((vz >> (sh - 1)) + 1) >> 1;
        if (hx) atomicAdd(H, hx);
        if (hy) atomicAdd(H + np, hy);
        if (hz) atomicAdd(H + 2 * np, hz);
    }
}

// The same for one 64-bit component (d = 0, 1, 2). Of its coarse count only the low sh bits (signed)
// go to the coarse word, so that as many terms as the coarse unit is chosen for keep it within 31
// bits; the rest, which takes a term beyond 2.7e8 kJ mol^-1 nm^-1 at the usual unit (colliding
// sites), goes to the upper word. The three together hold what a 64-bit sum would.
__device__ __forceinline__ void box_red64(const BoxDev& B, unsigned* acc, int sh, int s, int d, long long v) {
    const size_t np = (size_t)B.np;
    unsigned* L = acc + s + d * np;
    atomicAdd(L, (unsigned)v);
    const long long h = ((v >> (sh - 1)) + 1) >> 1;
    const int lo = (int)((unsigned)h << (32 - sh)) >> (32 - sh);
    if (lo) atomicAdd((int*)L + 3 * np, lo);
    if (lo != h) {
        atomicAdd(L + 6 * np, (unsigned)((h - lo) >> sh));
        *B.big = 1;
    }
}

// The pairs of two list entries per lane with the 8 atoms of the i cluster: at iteration t
// lane l takes cluster atom (l & 7) ^ t against both entries, the two pairs in one packed
// operation. The i sums move by one xor exchange per iteration and component inside a quarter
// warp and come home with the last (fi, lane l: atom l & 7; with the entries' sign); the j sums
// stay in the lane (fj). Each pair term s (x_j - x_i) is rounded to 2^-13 units and summed in
// 32-bit registers. MASKED: bit a of the low (first entry) or second byte of xm leaves out the
// pair with cluster atom a (the cluster's own slots, whose pairs count once, excluded pairs,
// and with the per-pair minimum image, MINIMG, empty slots). FAST: every atom has the reference
// LJ parameters, whose pair constants U are computed once. Returns the lanes where some |s|
// exceeds pc.s_lim / 2 (the 32-bit sums of 16 terms of their quarters could overflow; the caller
// redoes those pair by pair at the end of the list).
//
// FAST takes 24 packed operations, two rsqrt and six roundings per two pairs; all roundings as
// conversions would make the XU pipe (2.1 clocks an instruction) the bound, so z goes through
// the FMA pipe instead. Unrolled by four: with all eight iterations in a row warps at different
// places wait for instructions (1.3 of 7 clocks between two of a warp; a step of 16 x 24 560
// sites 515 -> 499 us, 504 unrolled by two).
template <int ELEC, bool ENERGY, bool MASKED, bool MINIMG, bool FAST>
__device__ __forceinline__ unsigned box_chunk(const BoxDev& B, const PairConst& pc, const LJPair2& U,
                                              const BoxCluster& ci, const Entries& n, unsigned xm,
                                              int lane, int* fi, int (*fj)[3], long long& e18) {
    const int l8 = lane & 7, q = lane >> 3;
    const float lim = 0.5f * kPairScale * pc.s_lim;
    int fx = 0, fy = 0, ax = 0, ay = 0, bx = 0, by = 0;
    unsigned fz = 0u, az = 0u, bz = 0u;  // (z terms carry kIntMagicBits: sums modulo 2^32)
    long long ech = 0;
    bool bad = false;
#pragma unroll 4
    for (int t = 0; t < 8; ++t) {
        const int a = l8 ^ t;
        const float4 xi = ci.x[a];
        float2 dx = make_float2(n.x.x - xi.x, n.x.y - xi.x), dy = make_float2(n.y.x - xi.y, n.y.y - xi.y),
               dz = make_float2(n.z.x - xi.z, n.z.y - xi.z);
        if (MINIMG) {
            dx = min_img2(dx, B.L, B.invL);
            dy = min_img2(dy, B.L, B.invL);
            dz = min_img2(dz, B.L, B.invL);
        }
        const float2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
        bool ok0 = r2.x < pc.rc2, ok1 = r2.y < pc.rc2;
        if (MASKED) {
            ok0 = ok0 && !((xm >> a) & 1u);
            ok1 = ok1 && !((xm >> (8 + a)) & 1u);
        }
        LJPair2 Q = U;
        if (!FAST) {
            const float2 li = ci.lj[a];
            Q = lj_pair2(make_float2(li.x + n.s.x, li.x + n.s.y), make_float2(li.y * n.e.x, li.y * n.e.y), pc);
        }
        float2 e;
        float2 ms = pair_ms2<ELEC, ENERGY>(r2, Q, make_float2(xi.w * n.q.x, xi.w * n.q.y), pc, &e);
        ms.x = ok0 ? ms.x : 0.0f;
        ms.y = ok1 ? ms.y : 0.0f;
        bad = bad || !(fabsf(ms.x) <= lim) || !(fabsf(ms.y) <= lim);
        if (ENERGY) {  // (e comes scaled by 2^13)
            const float lim_e = kPairScale * kPairEMax, se = kPairEScale / kPairScale;
            bad = bad || (ok0 && !(fabsf(e.x) < lim_e)) || (ok1 && !(fabsf(e.y) < lim_e));
            ech += (ok0 ? __float2int_rn(e.x * se) : 0) + (ok1 ? __float2int_rn(e.y * se) : 0);
        }
        const float2 tx = mul2(ms, dx), ty = mul2(ms, dy), tz = mul2(ms, dz);
        const int cx = __float2int_rn(tx.x), dx_ = __float2int_rn(tx.y);
        const int cy = __float2int_rn(ty.x), dy_ = __float2int_rn(ty.y);
        const int2 iz = round2_biased(tz);
        ax += cx;
        ay += cy;
        az += (unsigned)iz.x;
        bx += dx_;
        by += dy_;
        bz += (unsigned)iz.y;
        fx += cx + dx_;
        fy += cy + dy_;
        fz += (unsigned)iz.x + (unsigned)iz.y;
        const int m = (t ^ (t + 1)) & 7;  // to the lane that takes atom a next
        fx = __shfl_xor_sync(kFullB, fx, m);
        fy = __shfl_xor_sync(kFullB, fy, m);
        fz = __shfl_xor_sync(kFullB, fz, m);
    }
    // the biases of the z sums: 8 terms of an entry, 16 of a cluster atom
    const unsigned bias8 = 8u * (unsigned)kIntMagicBits;
    fi[0] = fx;
    fi[1] = fy;
    fi[2] = (int)(fz - 2u * bias8);
    fj[0][0] = ax;
    fj[0][1] = ay;
    fj[0][2] = (int)(az - bias8);
    fj[1][0] = bx;
    fj[1][1] = by;
    fj[1][2] = (int)(bz - bias8);
    const unsigned over = __ballot_sync(kFullB, bad);
    if (ENERGY && !((over >> (8 * q)) & 0xffu)) e18 += ech;
    return over;
}

// Eight entries per quarter warp (mine: the quarter has some) that failed the fast path, one
// per lane, pair by pair: every pair term, rounded to 2^-13 units as on the fast path, is summed
// in 64 bits, so the forces are the same integers on either path. As there, the entry's slot gets
// one sum and the cluster's atoms' sums move from lane to lane and come home (ai, with the
// entries' sign). For whole warps, once the list has been gone through: inside that loop it costs
// the loop registers (up to 39 us for 2 x 6400 sites, which take 34.4).
template <int ELEC, bool ENERGY, bool MINIMG>
__device__ __forceinline__ void box_chunk_slow(const BoxDev& B, const PairConst& pc, const BoxCluster& ci,
                                               float4 xj, float2 lj, int sj, unsigned xm, bool mine,
                                               unsigned* acc, int sh, long long* ai, long long& e18) {
    const int l8 = threadIdx.x & 7;
    long long fi[3] = {}, fj[3] = {};
#pragma unroll 1
    for (int t = 0; t < 8; ++t) {
        const int a = l8 ^ t;
        const float4 xi = ci.x[a];
        float dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
        if (MINIMG) {
            dx = min_img(dx, B.L, B.invL);
            dy = min_img(dy, B.L, B.invL);
            dz = min_img(dz, B.L, B.invL);
        }
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        if (mine && r2 < pc.rc2 && !((xm >> a) & 1u)) {
            float ep = 0.f;
            const float2 li = ci.lj[a];
            const float s = pair_s<ELEC, ENERGY>(r2, li.x + lj.x, li.y * lj.y, xi.w * xj.w, pc, &ep);
            const float ms13 = -s * kPairScale;
            const float f[3] = {ms13 * dx, ms13 * dy, ms13 * dz};
            // (one pair of a quarter is beyond the fast path's limit, few are beyond 32 bits)
            const bool small = fmaxf(fabsf(f[0]), fmaxf(fabsf(f[1]), fabsf(f[2]))) < 2.1e9f && s == s;
#pragma unroll
            for (int k = 0; k < 3; ++k) {  // (sums modulo 2^64)
                const long long q = small ? (long long)__float2int_rn(f[k]) : __float2ll_rn(f[k]);
                fi[k] = (long long)((unsigned long long)fi[k] + (unsigned long long)q);
                fj[k] = (long long)((unsigned long long)fj[k] + (unsigned long long)q);
            }
            if (ENERGY) e18 += __float2ll_rn(ep * kPairEScale);
        }
        const int m = (t ^ (t + 1)) & 7;
#pragma unroll
        for (int k = 0; k < 3; ++k) fi[k] = __shfl_xor_sync(kFullB, fi[k], m);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        ai[k] = (long long)((unsigned long long)ai[k] + (unsigned long long)fi[k]);
        if (mine && sj != (int)kBoxNoSlot) box_red64(B, acc, sh, sj, k, fj[k]);
    }
}

// Non-bonded forces of one 8-slot i cluster on one warp, each pair once (Newton's third
// law): its list 64 entries at a time, two per lane. After a chunk each lane adds its entries'
// sums to their slots and its share of a cluster atom's sums to 64-bit registers, which go to
// the cluster's slots at the end. Entries carry their periodic shift unless MINIMG; padding
// entries sit far away from everything.
// SHIFT: the coarse unit when the replica has the usual one (a constant in the loop: 33.7 us for
// 2 x 6400 sites, and 34.6 with a variable), else 0.
template <int ELEC, bool ENERGY, bool EXCL, bool MINIMG, int SHIFT>
__device__ __forceinline__ void box_cluster_forces(const BoxDev& B, const TopoDev& tp,
                                                   const RunParams& P, int r, int c, int lane,
                                                   bool ipure, BoxCluster& ci) {
    const size_t base = (size_t)r * B.np;
    const size_t cl = (size_t)r * 4 * B.nt + c;
    const uint32_t* lst = B.ent + cl * B.max_ent;
    const int n = B.nent[cl];
    unsigned* acc = B.facc + 9 * base;
    const int sh = SHIFT ? SHIFT : B.shift[r];
    const float2 ref = tp.lj[B.n_atoms - 1];
    const LJPair u1 = lj_pair(ref.x + ref.x, ref.y * ref.y, P.pc);
    const LJPair2 U = {dup2(u1.sig2), dup2(u1.eps24 * kPairScale), dup2(u1.c6), dup2(u1.a_ljc * kPairScale)};
    const int l8 = lane & 7;
    unsigned empty = 0u;  // empty slots of the cluster
    if (MINIMG) empty = __ballot_sync(kFullB, lane < 8 && ci.id[l8] < 0) & 0xffu;
    long long ai[3] = {};  // minus this lane's share of cluster atom l8
    long long e18 = 0;
    bool redo = false;
    auto entry = [&](int k) -> uint32_t { return k < n ? __ldg(lst + k) : (kBoxNoSlot | (1u << 30)); };
    auto position = [&](uint32_t e) -> float4 {
        const int sj = (int)(e & kBoxNoSlot);
        return sj != (int)kBoxNoSlot ? B.pos[base + sj]
                                     : make_float4(1.0e18f, 0.f, 0.f, 0.f);  // beyond any cutoff
    };
    auto shifted = [&](uint32_t e, float4 x) -> float4 {
        if (!MINIMG) {
            x.x = fmaf((float)((int)((e >> 24) & 3u) - 1), B.L, x.x);
            x.y = fmaf((float)((int)((e >> 26) & 3u) - 1), B.L, x.y);
            x.z = fmaf((float)((int)((e >> 28) & 3u) - 1), B.L, x.z);
        }
        return x;
    };
    auto mask = [&](uint32_t e, int k) -> unsigned {
        const int sj = (int)(e & kBoxNoSlot);
        if (sj == (int)kBoxNoSlot) return MINIMG ? 0xffu : 0u;
        unsigned m = k < 8 ? (0xffu << k) & 0xffu : 0u;  // own slots: j slot after i slot
        if (MINIMG) m |= empty;
        if (EXCL) {
            const int idj = B.id[base + sj];
            if (MINIMG && idj < 0) m = 0xffu;
            if (idj >= 0 && idj < B.n_chain)
                for (int a = 0; a < 8; ++a) {
                    const unsigned dj = (unsigned)(idj - ci.id[a] + kExclWindow);
                    if (dj < 2u * kExclWindow && ((ci.ex[a] >> dj) & 1ull)) m |= 1u << a;
                }
        }
        return m;
    };
    auto entry_lj = [&](uint32_t e) {
        const int sj = (int)(e & kBoxNoSlot);
        return sj != (int)kBoxNoSlot ? B.par[base + sj] : make_float2(0.f, 0.f);
    };
    // the next chunk's positions and the entries after it are loaded before a chunk is computed
    uint32_t en[2] = {entry(lane), entry(32 + lane)};
    float4 xn[2] = {position(en[0]), position(en[1])};
    uint32_t e2[2] = {entry(64 + lane), entry(96 + lane)};
    for (int k0 = 0; k0 < n; k0 += 64) {
        const uint32_t e[2] = {en[0], en[1]};
        const float4 x[2] = {shifted(e[0], xn[0]), shifted(e[1], xn[1])};
        float2 lj[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            en[k] = e2[k];
            xn[k] = position(en[k]);
            e2[k] = entry(k0 + 128 + 32 * k + lane);
        }
        bool fast = false;
        if constexpr (!EXCL && !MINIMG) fast = __all_sync(kFullB, ipure && ((e[0] & e[1]) >> 30 & 1u));
        if (!fast) {
            lj[0] = entry_lj(e[0]);
            lj[1] = entry_lj(e[1]);
        }
        const Entries en = pack_entries(x[0], x[1], lj[0], lj[1]);
        unsigned xm = 0u;
        if (EXCL || MINIMG || k0 == 0) xm = mask(e[0], k0 + lane) | (mask(e[1], k0 + 32 + lane) << 8);
        int fi[3], fj[2][3];
        unsigned over;
        if (EXCL || MINIMG || k0 == 0) {
            if (fast)
                over = box_chunk<ELEC, ENERGY, true, MINIMG, true>(B, P.pc, U, ci, en, xm, lane, fi, fj, e18);
            else
                over = box_chunk<ELEC, ENERGY, true, MINIMG, false>(B, P.pc, U, ci, en, xm, lane, fi, fj, e18);
        } else {
            if (fast)
                over = box_chunk<ELEC, ENERGY, false, MINIMG, true>(B, P.pc, U, ci, en, xm, lane, fi, fj, e18);
            else
                over = box_chunk<ELEC, ENERGY, false, MINIMG, false>(B, P.pc, U, ci, en, xm, lane, fi, fj, e18);
        }
        const bool good = !((over >> (lane & 24)) & 0xffu);
        if (over) {  // (uniform in the warp)
            redo = true;
            const unsigned bad = __ballot_sync(kFullB, !good && l8 == 0);  // bits 0, 8, 16, 24
            if (lane == 0) ci.redo[k0 >> 9] |= ((bad * 0x01020408u) >> 24 & 0xfu) << (k0 >> 4 & 28);
        }
        if (good) {
#pragma unroll
            for (int d = 0; d < 3; ++d) ai[d] += fi[d];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int sj = (int)(e[k] & kBoxNoSlot);
                if (sj != (int)kBoxNoSlot) box_red3(B, acc, sh, sj, fj[k][0], fj[k][1], fj[k][2]);
            }
        }
    }
    __syncwarp();
    for (int w = 0; redo && w < (n + 511) >> 9; ++w) {
        unsigned m = ci.redo[w];
        while (m) {  // two failed quarters of 16 entries at a time, eight entries per quarter warp
            const int q0 = __ffs(m) - 1;
            m &= m - 1u;
            const int q1 = m ? __ffs(m) - 1 : -1;
            m &= m - 1u;
            const int qq = lane < 16 ? q0 : q1;
            const bool mine = qq >= 0;
            const int k = mine ? 512 * w + 64 * (qq >> 2) + 8 * (qq & 3) + 32 * (lane >> 3 & 1) + l8 : n;
            const uint32_t e = entry(k);
            box_chunk_slow<ELEC, ENERGY, MINIMG>(B, P.pc, ci, shifted(e, position(e)), entry_lj(e),
                                                 (int)(e & kBoxNoSlot), mask(e, k), mine, acc, sh, ai, e18);
        }
    }
    // the four quarters' shares of each cluster atom
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        ai[d] += __shfl_xor_sync(kFullB, ai[d], 8);
        ai[d] += __shfl_xor_sync(kFullB, ai[d], 16);
    }
    if (lane < 8 && ci.id[lane] >= 0) {
#pragma unroll
        for (int d = 0; d < 3; ++d) box_red64(B, acc, sh, 8 * c + lane, d, -ai[d]);
    }
    if (ENERGY) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) e18 += __shfl_xor_sync(kFullB, e18, o);
        if (lane == 0 && e18 != 0) atomicAdd((unsigned long long*)&B.epair[r], (unsigned long long)e18);
    }
}

// Non-bonded forces: one warp per 8-slot i cluster, the variant chosen by its flags.
template <int ELEC, bool ENERGY>
__global__ void __launch_bounds__(32 * kPairWarps, kPairRegWarps / kPairWarps) k_box_pairs(BoxDev B, const TopoDev* __restrict__ topo,
                                                                 RunParams P, int r0) {
    __shared__ BoxCluster ci[kPairWarps];
    const int r = blockIdx.y + r0;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c = blockIdx.x * kPairWarps + w;
    if (c >= 4 * B.nt) return;
    const TopoDev& tp = *topo;
    if (lane < 8) {
        const size_t sl = (size_t)r * B.np + 8 * c + lane;
        ci[w].x[lane] = B.pos[sl];
        ci[w].lj[lane] = B.par[sl];
        const int a = B.id[sl];
        ci[w].id[lane] = a;
        ci[w].ex[lane] = (a >= 0 && a < B.n_chain) ? tp.excl[a] : 0ull;
    }
    if (lane < kBoxMaxEnt / 512) ci[w].redo[lane] = 0u;
    __syncwarp();
    const int fl = B.cflag[(size_t)r * 4 * B.nt + c];
    const bool pure = (fl & 4) != 0;
    auto forces = [&](auto shift) {
        constexpr int S = decltype(shift)::value;
        switch (fl & 3) {
            case 0: box_cluster_forces<ELEC, ENERGY, false, false, S>(B, tp, P, r, c, lane, pure, ci[w]); break;
            case 1: box_cluster_forces<ELEC, ENERGY, true, false, S>(B, tp, P, r, c, lane, pure, ci[w]); break;
            default: box_cluster_forces<ELEC, ENERGY, true, true, S>(B, tp, P, r, c, lane, pure, ci[w]); break;
        }
    };
    if (B.shift[r] == kBoxShift)
        forces(std::integral_constant<int, kBoxShift>());
    else
        forces(std::integral_constant<int, 0>());
}

// Total non-bonded force on slot s of replica r (fixed point), which is cleared for the
// next evaluation.
__device__ __forceinline__ float4 take_nb_force(const BoxDev& B, int r, int s) {
    const size_t np = (size_t)B.np;
    unsigned* L = B.facc + 9 * (size_t)r * np + s;
    unsigned w[6];
    const int big = *B.big, sh = B.shift[r];
#pragma unroll
    for (int d = 0; d < 6; ++d) w[d] = L[d * np];
    float f[3];
#pragma unroll
    for (int d = 0; d < 3; ++d)  // 2^-13 to 2^-20 units
        f[d] = fix2f(join_coarse((int)w[3 + d], w[d], sh) * 128);
    if (big)  // some upper word has been added to
        for (int d = 0; d < 3; ++d) {
            const long long up = (long long)L[(6 + d) * np] << sh;
            f[d] = fix2f(join_coarse((int)w[3 + d] + up, w[d], sh) * 128);
            L[(6 + d) * np] = 0u;
        }
#pragma unroll
    for (int d = 0; d < 6; ++d) L[d * np] = 0u;
    return make_float4(f[0], f[1], f[2], 0.f);
}

// Chain terms of one replica: bonds, angles (minimum image), z and the ratchet,
// the bias force; writes fch (bonded + bias) per chain atom. Also closes the
// rebuild bookkeeping of the step.
template <bool ENERGY>
__global__ void __launch_bounds__(512) k_box_chain(BoxDev B, const TopoDev* __restrict__ topo,
                                                   StateDev st, RunParams P, int r0,
                                                   int do_ratchet, int count_step) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ long long zred[16];
    __shared__ double ered[16];
    __shared__ double s_factor;
    __shared__ int s_bias;
    const int r = blockIdx.x + r0;
    const TopoDev tp = *topo;
    const int nch = B.n_chain, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float4* x = (float4*)smem_raw;                       // nch chain positions
    long long* F = (long long*)(x + nch);                // 3 nch fixed point
    float* hc = (float*)(F + 3 * nch);                   // contacts
    const size_t base = (size_t)r * B.np;
    for (int a = tid; a < nch; a += blockDim.x) x[a] = B.pos[base + B.slot_of[(size_t)r * B.n_atoms + a]];
    for (int i = tid; i < 3 * nch; i += blockDim.x) F[i] = 0;
    __syncthreads();
    const float L = B.L, iL = B.invL;
    double eb = 0.0;
    for (int b = tid; b < tp.n_bonds; b += blockDim.x) {
        const int2 ij = tp.bond_ij[b];
        const float2 par = tp.bond_par[b];
        const float dx = min_img(x[ij.y].x - x[ij.x].x, L, iL), dy = min_img(x[ij.y].y - x[ij.x].y, L, iL),
                    dz = min_img(x[ij.y].z - x[ij.x].z, L, iL);
        const float rr = sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        const float dr = rr - par.x;
        const float f = par.y * dr / rr;
        const long long qx = f2fix(f * dx), qy = f2fix(f * dy), qz = f2fix(f * dz);
        atomicAdd((unsigned long long*)&F[3 * ij.x], (unsigned long long)qx);
        atomicAdd((unsigned long long*)&F[3 * ij.x + 1], (unsigned long long)qy);
        atomicAdd((unsigned long long*)&F[3 * ij.x + 2], (unsigned long long)qz);
        atomicAdd((unsigned long long*)&F[3 * ij.y], (unsigned long long)(-qx));
        atomicAdd((unsigned long long*)&F[3 * ij.y + 1], (unsigned long long)(-qy));
        atomicAdd((unsigned long long*)&F[3 * ij.y + 2], (unsigned long long)(-qz));
        if (ENERGY) eb += 0.5 * (double)par.y * (double)dr * (double)dr;
    }
    for (int q = tid; q < tp.n_angles; q += blockDim.x) {
        const int4 ijk = tp.ang_ijk[q];
        const float2 par = tp.ang_par[q];
        const float ux = min_img(x[ijk.x].x - x[ijk.y].x, L, iL), uy = min_img(x[ijk.x].y - x[ijk.y].y, L, iL),
                    uz = min_img(x[ijk.x].z - x[ijk.y].z, L, iL);
        const float wx = min_img(x[ijk.z].x - x[ijk.y].x, L, iL), wy = min_img(x[ijk.z].y - x[ijk.y].y, L, iL),
                    wz = min_img(x[ijk.z].z - x[ijk.y].z, L, iL);
        const float cx = uy * wz - uz * wy, cy = uz * wx - ux * wz, cz = ux * wy - uy * wx;
        const float sn = sqrtf(fmaf(cx, cx, fmaf(cy, cy, cz * cz)));
        const float cs = fmaf(ux, wx, fmaf(uy, wy, uz * wz));
        const float ru2 = fmaf(ux, ux, fmaf(uy, uy, uz * uz));
        const float rw2 = fmaf(wx, wx, fmaf(wy, wy, wz * wz));
        const float dth = atan2f(sn, cs) - par.x;
        const float g = -par.y * dth / sn;
        const float au = cs / ru2, aw = cs / rw2;
        const float f1x = g * fmaf(au, ux, -wx), f1y = g * fmaf(au, uy, -wy), f1z = g * fmaf(au, uz, -wz);
        const float f3x = g * fmaf(aw, wx, -ux), f3y = g * fmaf(aw, wy, -uy), f3z = g * fmaf(aw, wz, -uz);
        const long long a1 = f2fix(f1x), a2 = f2fix(f1y), a3 = f2fix(f1z);
        const long long c1 = f2fix(f3x), c2 = f2fix(f3y), c3 = f2fix(f3z);
        atomicAdd((unsigned long long*)&F[3 * ijk.x], (unsigned long long)a1);
        atomicAdd((unsigned long long*)&F[3 * ijk.x + 1], (unsigned long long)a2);
        atomicAdd((unsigned long long*)&F[3 * ijk.x + 2], (unsigned long long)a3);
        atomicAdd((unsigned long long*)&F[3 * ijk.z], (unsigned long long)c1);
        atomicAdd((unsigned long long*)&F[3 * ijk.z + 1], (unsigned long long)c2);
        atomicAdd((unsigned long long*)&F[3 * ijk.z + 2], (unsigned long long)c3);
        atomicAdd((unsigned long long*)&F[3 * ijk.y], (unsigned long long)(-a1 - c1));
        atomicAdd((unsigned long long*)&F[3 * ijk.y + 1], (unsigned long long)(-a2 - c2));
        atomicAdd((unsigned long long*)&F[3 * ijk.y + 2], (unsigned long long)(-a3 - c3));
        if (ENERGY) eb += 0.5 * (double)par.y * (double)dth * (double)dth;
    }
    // z of Eq. (zrMD): (C - C0)^2 in float-float, summed in 2^-40 fixed point
    long long zacc = 0;
    if (P.bias == 1) {
        for (int c = tid; c < tp.n_contacts; c += blockDim.x) {
            const int2 ij = tp.con_ij[c];
            const float4 a = x[ij.x], b = x[ij.y];
            // exact float-float separation, then the minimum-image shift (a multiple of L)
            ff dx = ff_diff(b.x, a.x), dy = ff_diff(b.y, a.y), dz = ff_diff(b.z, a.z);
            dx = ff_add_f(dx, -L * rintf((b.x - a.x) * iL));
            dy = ff_add_f(dy, -L * rintf((b.y - a.y) * iL));
            dz = ff_add_f(dz, -L * rintf((b.z - a.z) * iL));
            const ff u = ff_mul(ff_r2(dx, dy, dz), P.inv_r0sq_ff);
            const ff C = contact_C_ff(u);
            const float2 c0 = tp.con_C0[c];
            const ff d = ff_add(C, ff{-c0.x, -c0.y});
            hc[c] = (d.hi + d.lo) * contact_dC_du(u.hi);
            zacc += ff2fix40(ff_sqr(d));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        zacc += __shfl_down_sync(kFullB, zacc, o);
        eb += __shfl_down_sync(kFullB, eb, o);
    }
    if (lane == 0) {
        zred[warp] = zacc;
        ered[warp] = eb;
    }
    __syncthreads();
    if (tid == 0) {
        long long zt = 0;
        double et = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            zt += zred[w];
            et += ered[w];
        }
        double factor = 0.0;
        if (P.bias == 1) {
            const double z = (double)zt * 9.094947017729282e-13;  // 2^-40
            st.z[r] = z;
            if (do_ratchet) {  // Eq. (FrMD) with theta(0) = 1
                if (z < st.zm[r])
                    st.zm[r] = z;
                else
                    factor = -P.k_R * (z - st.zm[r]);
            }
        }
        s_factor = factor;
        s_bias = factor != 0.0;
        if (ENERGY) B.eb[r] = et;
        if (B.need[r])
            B.need[r] = 0;  // the rebuild of this step is complete
        else if (count_step)
            B.since[r] += 1;
    }
    __syncthreads();
    const float k = -(float)s_factor * 4.0f * P.inv_r0sq;
    float tb = 0.f;
    for (int a = tid; a < nch; a += blockDim.x) {
        float bx = 0.f, by = 0.f, bz = 0.f;
        if (s_bias) {
            const float4 xa = x[a];
            for (int q = tp.con_off[a]; q < tp.con_off[a + 1]; ++q) {
                const int2 cp = tp.con_nbr[q];
                const float4 xp = x[cp.y];
                const float h = hc[cp.x];
                bx = fmaf(h, min_img(xp.x - xa.x, L, iL), bx);
                by = fmaf(h, min_img(xp.y - xa.y, L, iL), by);
                bz = fmaf(h, min_img(xp.z - xa.z, L, iL), bz);
            }
            bx *= k;
            by *= k;
            bz *= k;
            tb += (bx * bx + by * by + bz * bz) * tp.inv_m[a];
        }
        B.fch[(size_t)r * nch + a] = make_float4(fix2f(F[3 * a]) + bx, fix2f(F[3 * a + 1]) + by,
                                                 fix2f(F[3 * a + 2]) + bz, 0.f);
    }
    // bias functional: fixed order (lane tree, then warps in index order)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tb += __shfl_down_sync(kFullB, tb, o);
    __shared__ float tred[16];
    if (lane == 0) tred[warp] = tb;
    __syncthreads();
    if (tid == 0 && s_bias && count_step) {
        float ts = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) ts += tred[w];
        st.T[r] += (double)P.dt / P.gamma * (double)ts;
    }
}

// BAOAB half steps per slot: B closes the evaluated step, A starts the next one. The largest
// squared displacement since the list build goes to the replica's bound with at most one atomic
// per warp (every lane reaches the warp reduction; the slots of a warp share their replica).
// Latency bounds it: loads ahead of all stores, and an atomic only where it raises the bound
// (one per warp on 16 addresses of a line made it 48 us for 16 x 24 560 sites, now 19).
__global__ void k_box_integrate(BoxDev B, const TopoDev* __restrict__ topo, StateDev st,
                                RunParams P, const uint32_t* __restrict__ rep_ids, long long step,
                                int do_b, int do_a, int step_from_state) {
    const int r = blockIdx.y;
    if (step_from_state) step = st.step[r];  // graph form: the counter the step graph advanced
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const size_t base = (size_t)r * B.np;
    float d2 = 0.f;
    if (s < B.np) {
        // all loads that need nothing but the slot go out together
        const int a = B.id[base + s];
        float4 v = B.vel[base + s];
        float4 x = B.pos[base + s];
        const float4 p0 = B.pos_ref[base + s];
        const bool live = a >= 0 && st.status[r] == 0;
        const TopoDev& tp = *topo;
        const float im = tp.inv_m[max(a, 0)], sd = tp.noise_sd[max(a, 0)];
        float4 f = take_nb_force(B, r, s);  // also clears the sums (frozen replicas too)
        if (live) {
            if (a < B.n_chain) {
                const float4 c = B.fch[(size_t)r * B.n_chain + a];
                f.x += c.x;
                f.y += c.y;
                f.z += c.z;
            }
            const float hdt = P.half_dt;
            if (do_b) {
                v.x = fmaf(hdt * im, f.x, v.x);
                v.y = fmaf(hdt * im, f.y, v.y);
                v.z = fmaf(hdt * im, f.z, v.z);
            }
            if (do_a) {
                v.x = fmaf(hdt * im, f.x, v.x);
                v.y = fmaf(hdt * im, f.y, v.y);
                v.z = fmaf(hdt * im, f.z, v.z);
                x.x = fmaf(hdt, v.x, x.x);
                x.y = fmaf(hdt, v.y, x.y);
                x.z = fmaf(hdt, v.z, x.z);
                const uint4 rb = philox4x32_10(make_uint4((uint32_t)a, rep_ids[r], (uint32_t)step, 0u),
                                               P.key0, P.key1);
                const float4 xi = normals4_f32(rb);
                v.x = fmaf(P.c1, v.x, sd * xi.x);
                v.y = fmaf(P.c1, v.y, sd * xi.y);
                v.z = fmaf(P.c1, v.z, sd * xi.z);
                x.x = fmaf(hdt, v.x, x.x);
                x.y = fmaf(hdt, v.y, x.y);
                x.z = fmaf(hdt, v.z, x.z);
                if (!(isfinite(x.x) && isfinite(x.y) && isfinite(x.z) && isfinite(v.x) &&
                      isfinite(v.y) && isfinite(v.z)))
                    atomicOr(&st.status[r], SCPS_FLAG_NONFINITE);
                B.pos[base + s] = x;
                const float ddx = x.x - p0.x, ddy = x.y - p0.y, ddz = x.z - p0.z;
                d2 = fmaf(ddx, ddx, fmaf(ddy, ddy, ddz * ddz));
            }
            B.vel[base + s] = v;
        }
    }
    if (do_a) {  // non-negative floats order as unsigned
        const unsigned m = __reduce_max_sync(kFullB, __float_as_uint(d2));
        // (the bound only grows: a warp below it, whatever its age, has nothing to add)
        if ((threadIdx.x & 31) == 0 && m > __ldcg(&B.maxd2[r])) atomicMax(&B.maxd2[r], m);
    }
}

// Frame output of the evaluated configuration (positions in atom-id order).
__global__ void k_box_frame(BoxDev B, StateDev st, RunParams P, long long frame_atoms) {
    const int r = blockIdx.y;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= B.np) return;
    const int a = B.id[(size_t)r * B.np + s];
    if (a < 0) return;
    const long long slot = st.n_saved[r] % P.max_frames;
    const float4 x = B.pos[(size_t)r * B.np + s];
    float* fr = st.frames + 3 * ((long long)r * frame_atoms + slot * B.n_atoms + a);
    fr[0] = x.x;
    fr[1] = x.y;
    fr[2] = x.z;
}

// Frame scalars; the potential energy is the fixed-point pair energy (2^-18 units, cleared
// here) plus the bonded energy.
__global__ void k_box_frame_scalars(BoxDev B, StateDev st, RunParams P, int R) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R) return;
    const long long slot = st.n_saved[r] % P.max_frames;
    const long long fi = (long long)r * P.max_frames + slot;
    st.fz[fi] = st.z[r];
    st.fzm[fi] = st.zm[r];
    st.fe[fi] = (double)B.epair[r] * 3.814697265625e-06 + B.eb[r];  // 2^-18
    st.fT[fi] = st.T[r];
    st.n_saved[r] += 1;
    B.epair[r] = 0;
}

__global__ void k_box_step_count(StateDev st, int R, long long k) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < R && st.status[r] == 0) st.step[r] += k;
}

// ------------------------------------------------------------------ host side
size_t box_chain_smem(int n_chain, int n_contacts) {
    return sizeof(float4) * n_chain + sizeof(long long) * 3 * n_chain + sizeof(float) * n_contacts;
}

// The rebuild kernels after the decision (each returns at once for a replica that does not
// rebuild), for replicas [r0, r0 + nr).
static void box_rebuild(const BoxDev& B, const TopoDev* topo, const StateDev& st, int r0, int nr,
                        cudaStream_t s) {
    k_box_key<<<dim3((B.np + 255) / 256, nr), 256, 0, s>>>(B, r0);
    k_box_scan<<<nr, kSortThreads, 0, s>>>(B, r0);
    k_box_scatter<<<dim3((B.n_atoms + 255) / 256, nr), 256, 0, s>>>(B, r0);
    k_box_keyorder<<<dim3((B.np + 255) / 256, nr), 256, 0, s>>>(B, r0);
    const dim3 gt((B.nt + 3) / 4, nr);       // one warp per tile
    k_box_subsort<<<gt, 128, 0, s>>>(B, topo, r0);
    k_box_tiles<<<gt, 128, 0, s>>>(B, topo, r0);
    k_box_list<<<dim3(B.nt, nr), 128, 0, s>>>(B, st, r0);
}

// Pair forces of replicas [r0, r0 + nr).
static void box_pairs_launch(const BoxDev& B, const TopoDev* topo, const RunParams& P, int r0, int nr,
                             int elec, bool energy, cudaStream_t s) {
    const dim3 gg((4 * B.nt + kPairWarps - 1) / kPairWarps, nr);
#define PAIRS(E)                                                                                \
    switch (elec) {                                                                             \
        case ELEC_DDIEL: k_box_pairs<ELEC_DDIEL, E><<<gg, 32 * kPairWarps, 0, s>>>(B, topo, P, r0); break;  \
        case ELEC_RF: k_box_pairs<ELEC_RF, E><<<gg, 32 * kPairWarps, 0, s>>>(B, topo, P, r0); break;        \
        case ELEC_PLAIN: k_box_pairs<ELEC_PLAIN, E><<<gg, 32 * kPairWarps, 0, s>>>(B, topo, P, r0); break;  \
        default: k_box_pairs<ELEC_NONE, E><<<gg, 32 * kPairWarps, 0, s>>>(B, topo, P, r0); break;           \
    }
    if (energy) {
        PAIRS(true)
    } else {
        PAIRS(false)
    }
#undef PAIRS
}

// Chain terms and the ratchet of replicas [r0, r0 + nr) (independent of the pair forces: the
// integrator adds the two).
static void box_chain_launch(const BoxDev& B, const TopoDev* topo, const StateDev& st,
                             const RunParams& P, int r0, int nr, int ncon_max, bool energy,
                             int do_ratchet, int count_step, cudaStream_t s) {
    const size_t smem = box_chain_smem(B.n_chain, ncon_max);
    if (energy)
        k_box_chain<true><<<nr, 512, smem, s>>>(B, topo, st, P, r0, do_ratchet, count_step);
    else
        k_box_chain<false><<<nr, 512, smem, s>>>(B, topo, st, P, r0, do_ratchet, count_step);
}

// Pair forces, then the chain terms and the ratchet, of replicas [r0, r0 + nr).
static void box_forces(const BoxDev& B, const TopoDev* topo, const StateDev& st, const RunParams& P,
                       int r0, int nr, int elec, int ncon_max, bool energy, int do_ratchet,
                       int count_step, cudaStream_t s) {
    box_pairs_launch(B, topo, P, r0, nr, elec, energy, s);
    box_chain_launch(B, topo, st, P, r0, nr, ncon_max, energy, do_ratchet, count_step, s);
}

// One force evaluation of replicas [r0, r0 + nr): rebuild when forced (or, when
// `auto_ok`, when due), pair forces, chain terms and the ratchet.
static cudaError_t box_eval(const BoxDev& B, const TopoDev* topo, const StateDev& st,
                            const RunParams& P, int r0, int nr, int elec, int ncon_max,
                            bool energy, int do_ratchet, int count_step, int auto_ok,
                            cudaStream_t s) {
    k_box_decide<<<1, 256, 0, s>>>(B, st, r0, nr, auto_ok);
    k_box_clear_hist<<<dim3((kNumKeys + 255) / 256, nr), 256, 0, s>>>(B, r0);
    box_rebuild(B, topo, st, r0, nr, s);
    box_forces(B, topo, st, P, r0, nr, elec, ncon_max, energy, do_ratchet, count_step, s);
    return cudaGetLastError();
}

// Dynamic shared memory k_box_chain may request on the current device: the opt-in per-block
// limit less its static shared block; 0 when the device cannot be queried.
size_t box_chain_smem_limit() {
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return 0;
    size_t stat = 0;
    for (const void* k : {(const void*)k_box_chain<true>, (const void*)k_box_chain<false>}) {
        cudaFuncAttributes a;
        if (cudaFuncGetAttributes(&a, k) != cudaSuccess) return 0;
        stat = a.sharedSizeBytes > stat ? a.sharedSizeBytes : stat;
    }
    return (size_t)optin > stat ? (size_t)optin - stat : 0;
}

cudaError_t box_prepare(const BoxDev& B, int n_contacts_max) {
    const size_t smem = box_chain_smem(B.n_chain, n_contacts_max);
    cudaError_t e = cudaFuncSetAttribute(k_box_chain<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_box_chain<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return e;
}

// One MD step of replicas [0, R) as a graph: the step counters, the rebuild decision (which
// sets the graph's conditional value), the rebuild kernels inside a conditional node (run
// only when some replica rebuilds), the forces, [the frame], the B half step and, unless
// `last`, the A half step of the next one (noise counter read from the step counters),
// [the frame scalars].
static cudaError_t box_step_graph(const BoxDev& B, const TopoDev* topo, const StateDev& st,
                                  const RunParams& P, const uint32_t* rep_ids, int R, int elec,
                                  int ncon_max, bool save, bool last, long long frame_atoms,
                                  cudaStream_t cs, cudaStream_t cs2, cudaGraph_t* def,
                                  cudaGraphExec_t* exec) {
    const dim3 ga((B.np + 255) / 256, R);
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaGraphCreate(&g, 0);
    if (e != cudaSuccess) return e;
    cudaGraphConditionalHandle h;
    e = cudaGraphConditionalHandleCreate(&h, g, 0, cudaGraphCondAssignDefault);
    if (e == cudaSuccess) e = cudaStreamBeginCaptureToGraph(cs, g, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) {
        cudaGraphDestroy(g);
        return e;
    }
    k_box_step_count<<<(R + 127) / 128, 128, 0, cs>>>(st, R, 1);
    k_box_decide_graph<<<1, 256, 0, cs>>>(B, st, R, h);
    cudaStreamCaptureStatus cst;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    cudaGraphNode_t cond = nullptr;
    cudaGraphNodeParams cp = {};
    e = cudaStreamGetCaptureInfo(cs, &cst, nullptr, nullptr, &deps, nullptr, &nd);
    if (e == cudaSuccess) {
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = h;
        cp.conditional.type = cudaGraphCondTypeIf;
        cp.conditional.size = 1;
        e = cudaGraphAddNode(&cond, g, deps, nullptr, nd, &cp);
    }
    if (e == cudaSuccess) e = cudaStreamUpdateCaptureDependencies(cs, &cond, nullptr, 1, cudaStreamSetCaptureDependencies);
    if (e == cudaSuccess) {
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        e = cudaStreamBeginCaptureToGraph(cs2, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            k_box_clear_hist<<<dim3((kNumKeys + 255) / 256, R), 256, 0, cs2>>>(B, 0);
            box_rebuild(B, topo, st, 0, R, cs2);
            const cudaError_t le = cudaGetLastError();
            e = cudaStreamEndCapture(cs2, &body);
            if (e == cudaSuccess) e = le;
        }
    }
    cudaEvent_t fork = nullptr, join = nullptr;
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&join, cudaEventDisableTiming);
    if (e == cudaSuccess) {  // the chain terms run beside the pair forces (second branch)
        e = cudaEventRecord(fork, cs);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(cs2, fork, 0);
        if (e == cudaSuccess) {
            box_chain_launch(B, topo, st, P, 0, R, ncon_max, save, 1, 1, cs2);
            e = cudaEventRecord(join, cs2);
        }
        if (e == cudaSuccess) {
            box_pairs_launch(B, topo, P, 0, R, elec, save, cs);
            e = cudaStreamWaitEvent(cs, join, 0);
        }
    }
    if (e == cudaSuccess) {
        if (save) k_box_frame<<<ga, 256, 0, cs>>>(B, st, P, frame_atoms);
        k_box_integrate<<<ga, 256, 0, cs>>>(B, topo, st, P, rep_ids, 0, 1, last ? 0 : 1, 1);
        if (save) k_box_frame_scalars<<<(R + 127) / 128, 128, 0, cs>>>(B, st, P, R);
        e = cudaGetLastError();
    }
    cudaGraph_t out = nullptr;
    const cudaError_t ce = cudaStreamEndCapture(cs, &out);
    if (e == cudaSuccess) e = ce;
    if (fork) cudaEventDestroy(fork);
    if (join) cudaEventDestroy(join);
    if (e == cudaSuccess) e = cudaGraphInstantiate(exec, g, 0);
    if (e != cudaSuccess) {
        cudaGraphDestroy(g);
        return e;
    }
    *def = g;
    return cudaSuccess;
}

void BoxGraphs::reset() {
    for (int v = 0; v < 4; ++v) {
        if (exec[v]) cudaGraphExecDestroy(exec[v]);
        if (def[v]) cudaGraphDestroy(def[v]);
        exec[v] = nullptr;
        def[v] = nullptr;
    }
}

// n_steps steps of replicas [0, R) on stream s: the current configuration is evaluated
// again (no scheduled rebuild here, so the result does not depend on how steps are split into
// calls) and its A half step taken; then every step is one launch of a step graph from G
// (regular, last, save, save and last; captured on first use), or, without G, the same
// kernels launched one by one.
cudaError_t box_run(const BoxDev& B, const TopoDev* topo, const StateDev& st, const RunParams& P,
                    const uint32_t* rep_ids, int R, int elec, int ncon_max, long long step0,
                    long long n_steps, long long frame_atoms, BoxGraphs* G, cudaStream_t s) {
    const dim3 ga((B.np + 255) / 256, R);
    cudaError_t e = box_eval(B, topo, st, P, 0, R, elec, ncon_max, false, 1, 0, 0, s);
    if (e != cudaSuccess) return e;
    k_box_integrate<<<ga, 256, 0, s>>>(B, topo, st, P, rep_ids, step0, 0, 1, 0);
    for (long long k = 1; k <= n_steps; ++k) {
        const long long step = step0 + k;
        const bool save = P.save_interval > 0 && step % P.save_interval == 0;
        const bool last = k == n_steps;
        if (G) {
            const int v = (save ? 2 : 0) + (last ? 1 : 0);
            if (!G->exec[v]) {
                e = box_step_graph(B, topo, st, P, rep_ids, R, elec, ncon_max, save, last,
                                   frame_atoms, G->cap, G->cap2, &G->def[v], &G->exec[v]);
                if (e != cudaSuccess) return e;
            }
            e = cudaGraphLaunch(G->exec[v], s);
            if (e != cudaSuccess) return e;
            continue;
        }
        k_box_step_count<<<(R + 127) / 128, 128, 0, s>>>(st, R, 1);
        e = box_eval(B, topo, st, P, 0, R, elec, ncon_max, save, 1, 1, 1, s);
        if (e != cudaSuccess) return e;
        if (save) k_box_frame<<<ga, 256, 0, s>>>(B, st, P, frame_atoms);
        k_box_integrate<<<ga, 256, 0, s>>>(B, topo, st, P, rep_ids, step, 1, last ? 0 : 1, 0);
        if (save) k_box_frame_scalars<<<(R + 127) / 128, 128, 0, s>>>(B, st, P, R);
    }
    return cudaGetLastError();
}

// Energy and forces of one configuration X (atom order) in the evaluation slot r_eval.
__global__ void k_box_load_frame(BoxDev B, const TopoDev* __restrict__ topo, StateDev st,
                                 const float* __restrict__ X, int r) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= B.np) return;
    const size_t base = (size_t)r * B.np;
    if (s < B.n_atoms) {
        B.pos[base + s] = make_float4(X[3 * s], X[3 * s + 1], X[3 * s + 2], topo->qs[s]);
        B.vel[base + s] = make_float4(0.f, 0.f, 0.f, 0.f);
        B.id[base + s] = s;
        B.slot_of[(size_t)r * B.n_atoms + s] = s;
    } else {
        B.id[base + s] = -1;
    }
    if (s == 0) {
        B.need[r] = 1;
        st.status[r] = 0;
    }
}

cudaError_t box_load(const BoxDev& B, const TopoDev* topo, const StateDev& st, const float* X,
                     int r, cudaStream_t s) {
    k_box_load_frame<<<(B.np + 255) / 256, 256, 0, s>>>(B, topo, st, X, r);
    return cudaGetLastError();
}

// Forces of the evaluation slot r in atom order (F may be NULL: the j parts are
// cleared all the same).
__global__ void k_box_store_forces(BoxDev B, int r, float* __restrict__ F) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= B.np) return;
    const size_t base = (size_t)r * B.np;
    float4 f = take_nb_force(B, r, s);
    const int a = B.id[base + s];
    if (a < 0 || !F) return;
    if (a < B.n_chain) {
        const float4 c = B.fch[(size_t)r * B.n_chain + a];
        f.x += c.x;
        f.y += c.y;
        f.z += c.z;
    }
    F[3 * a] = f.x;
    F[3 * a + 1] = f.y;
    F[3 * a + 2] = f.z;
}

__global__ void k_box_store_energy(BoxDev B, StateDev st, int r, double* U, double* Z) {
    *U = (double)B.epair[r] * 3.814697265625e-06 + B.eb[r];  // 2^-18
    B.epair[r] = 0;
    if (Z) *Z = st.z[r];
}

cudaError_t box_energy_forces(const BoxDev& B, const TopoDev* topo, const StateDev& st,
                              const RunParams& P, int r_eval, int elec, int ncon_max,
                              const float* X, double* U, float* F, double* Z, cudaStream_t s) {
    const int g = (B.np + 255) / 256;
    k_box_load_frame<<<g, 256, 0, s>>>(B, topo, st, X, r_eval);
    cudaError_t e = box_eval(B, topo, st, P, r_eval, 1, elec, ncon_max, true, 0, 0, 0, s);
    if (e != cudaSuccess) return e;
    k_box_store_forces<<<g, 256, 0, s>>>(B, r_eval, F);
    k_box_store_energy<<<1, 1, 0, s>>>(B, st, r_eval, U, Z);
    return cudaGetLastError();
}

}  // namespace scps
