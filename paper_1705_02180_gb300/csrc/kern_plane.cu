// Two-dimensional models, one particle per replica, overdamped Langevin
// (Euler-Maruyama) in FP64, a whole launch of steps in one kernel.
//   model 0: U = (x^2 - 1)^2 + y^2 (double well)
//   model 1: the asymmetric funnel of Eq. (U) with the parameters of Table 1
// Biases (P.bias):
//   2: ratchet of Eq. (FrMD) on z = (x - x_ref)^2
//   3: ratchet on z = sqrt(x^2 + y^2), the distance from the funnel centre
//   4: tube variables s_lambda, w_lambda of a reference path <X(t'_k)> (the
//      configuration-space form used for the funnel): D_k = |X - <X(t'_k)>|^2,
//      pi_k = exp(-lambda D_k) / sum, w = -(1/lambda) log sum_k exp(-lambda D_k),
//      s = 1 - (1/t) sum_k t'_k pi_k, each with its own ratchet (forces F^w, F^s of
//      Eq. Fw and Eq. Fs; z_m of Eq. FrMD replaced by s_m and w_m)
//
// What bounds these kernels is the FP64 pipe: a warp's FP64 instruction takes about 68 clocks
// of its quarter of the SM, whether one lane is active or all, and a second one of the same
// warp waits for it (measured; log 2310, sqrt 730, sincospi 2060, exp 1130, a division 470
// clocks). A step is a serial chain, so its time is the number of FP64 instructions its warp
// issues. Both kernels therefore keep everything that is not part of the chain out of that
// warp (the Gaussian numbers depend only on the step counter), spread what is alike over its
// lanes (divisions, the slices of a path), and test signs in integers.
#include <algorithm>

#include "scps_internal.h"

namespace scps {

namespace {

constexpr unsigned kFullP = 0xffffffffu;
constexpr double kA1 = 30.0, kA2 = 20.0, kA3 = 6.0, kS1 = 1.0, kS2 = 2.0, kS3 = 0.5;
constexpr double kW = 0.03, kYm = 0.0, kXm = 1.5;
constexpr int kPlaneProducers = 3;  // warps drawing noise beside the stepping warp

// The lanes of a stepping warp: 32 >> lg copies of each of 1 << lg replicas; lane l holds
// copy l >> lg of replica l & ((1 << lg) - 1). With four copies or more, like terms are
// computed one per copy and exchanged.
struct Lanes {
    int lane, lg;
    __device__ __forceinline__ int g() const { return lane & ((1 << lg) - 1); }
    __device__ __forceinline__ int copy() const { return lane >> lg; }
    __device__ __forceinline__ bool wide() const { return lg <= 3; }
    __device__ __forceinline__ double from(double v, int c) const {
        return __shfl_sync(kFullP, v, (c << lg) + g());
    }
};

// a b + c d with one rounding in the first product. Trajectories amplify the last bit, so
// every sum of products states which of them is fused: results do not hang on what the
// compiler would choose for another arrangement of the code around it.
__device__ __forceinline__ double dot2(double a, double b, double c, double d) {
    return __fma_rn(a, b, __dmul_rn(c, d));
}

// n0 / d0 and n1 / d1.
__device__ __forceinline__ double2 div_two(const Lanes& L, double n0, double d0, double n1, double d1) {
    if (!L.wide()) return make_double2(n0 / d0, n1 / d1);
    const bool first = L.copy() == 0;
    const double q = (first ? n0 : n1) / (first ? d0 : d1);
    return make_double2(L.from(q, 0), L.from(q, 1));
}

__device__ __forceinline__ double funnel_u(double x, double y) {
    const double r2 = x * x + y * y;
    const double d2 = (x - kXm) * (x - kXm) + (y - kYm) * (y - kYm);
    const double a = r2 + kS1 * kS1, b = r2 + kS2 * kS2, c = d2 + kS3 * kS3;
    return kW * kW * r2 * r2 - kA1 * kS1 * kS1 / (a * a) + kA2 * kS2 * kS2 / (b * b) -
           kA3 * kS3 * kS3 / (c * c);
}

__device__ __forceinline__ double2 funnel_f(const Lanes& L, double x, double y) {
    const double r2 = dot2(x, x, y, y);
    const double X = x - kXm;
    const double d2 = dot2(X, X, y, y);
    const double a = r2 + kS1 * kS1, b = r2 + kS2 * kS2, c = d2 + kS3 * kS3;
    double qa, qb, gd;  // the three terms of the shape n / d^3
    const double na = 2.0 * kA1 * kS1 * kS1, nb = 2.0 * kA2 * kS2 * kS2, nc = -2.0 * kA3 * kS3 * kS3;
    if (L.wide()) {
        const int k = L.copy();
        const double d = k == 0 ? a : k == 1 ? b : c;
        const double q = (k == 0 ? na : k == 1 ? nb : nc) / (d * d * d);
        qa = L.from(q, 0);
        qb = L.from(q, 1);
        gd = L.from(q, 2);
    } else {
        qa = na / (a * a * a);
        qb = nb / (b * b * b);
        gd = nc / (c * c * c);
    }
    // -dU/dr2 for the terms in r2, -dU/dd2 for the gate term
    const double gr = __dadd_rn(__fma_rn(-2.0 * kW * kW, r2, -qa), qb);
    return make_double2(2.0 * dot2(gd, X, gr, x), 2.0 * dot2(gd, y, gr, y));
}

__device__ __forceinline__ double2 model_force(const Lanes& L, int model, double2 p) {
    if (model == 1) return funnel_f(L, p.x, p.y);
    return make_double2(-4.0 * p.x * (p.x * p.x - 1.0), -2.0 * p.y);
}

__device__ __forceinline__ double model_energy(int model, double2 p) {
    if (model == 1) return funnel_u(p.x, p.y);
    return (p.x * p.x - 1.0) * (p.x * p.x - 1.0) + p.y * p.y;
}

// Tube variables at p: s, w and their gradients (one lane, all slices).
__device__ void tube_vars(const RunParams& P, double2 p, double* s, double* w, double2* gs,
                          double2* gw) {
    double dmin = 1e300;
    for (int k = 0; k < P.tube_k; ++k) {
        const double2 q = P.tube_ref[k];
        const double dx = p.x - q.x, dy = p.y - q.y, d = dot2(dx, dx, dy, dy);
        dmin = d < dmin ? d : dmin;
    }
    // sums with the largest weight scaled to 1 (the formulas are unchanged)
    double S = 0.0, St = 0.0;
    double2 g1 = make_double2(0.0, 0.0), g2 = make_double2(0.0, 0.0);
    for (int k = 0; k < P.tube_k; ++k) {
        const double2 q = P.tube_ref[k];
        const double dx = p.x - q.x, dy = p.y - q.y;
        const double e = exp(-P.tube_lambda * (dot2(dx, dx, dy, dy) - dmin));
        const double et = __dmul_rn(e, P.tube_time[k]);
        S = __dadd_rn(S, e);
        St = __dadd_rn(St, et);
        g1.x = __fma_rn(2.0 * e, dx, g1.x);  // sum e_k grad D_k
        g1.y = __fma_rn(2.0 * e, dy, g1.y);
        g2.x = __fma_rn(2.0 * et, dx, g2.x);  // sum e_k t_k grad D_k
        g2.y = __fma_rn(2.0 * et, dy, g2.y);
    }
    const double tm = St / S;  // <t'> under pi
    *w = dmin - log(S) / P.tube_lambda;
    *s = 1.0 - tm / P.tube_t;
    *gw = make_double2(g1.x / S, g1.y / S);  // sum pi_k grad D_k
    const double c = P.tube_lambda / P.tube_t;
    *gs = make_double2(c * (g2.x / S - __dmul_rn(tm, g1.x) / S),
                       c * (g2.y / S - __dmul_rn(tm, g1.y) / S));
}

// Ring buffer position and save phase of a replica as counters (no 64-bit division per step).
struct Saver {
    int phase, slot;
    long long ns;
    __device__ __forceinline__ void init(const RunParams& P, long long step, long long n_saved) {
        ns = n_saved;
        phase = P.save_interval > 0 ? (int)(step % P.save_interval) : -1;
        slot = P.max_frames > 0 ? (int)(n_saved % P.max_frames) : 0;
    }
    // counts a step; true when it is saved
    __device__ __forceinline__ bool step(const RunParams& P) {
        if (phase < 0) return false;
        phase = phase + 1 == P.save_interval ? 0 : phase + 1;
        return phase == 0;
    }
    __device__ __forceinline__ void saved(const RunParams& P) {
        ++ns;
        slot = slot + 1 == P.max_frames ? 0 : slot + 1;
    }
};

__device__ __forceinline__ void save_position(const StateDev& st, const RunParams& P, int r, int slot,
                                              double2 p, double T) {
    const long long fi = (long long)r * P.max_frames + slot;
    st.frames[2 * fi] = (float)p.x;
    st.frames[2 * fi + 1] = (float)p.y;
    st.fe[fi] = model_energy(P.toy_model, p);
    st.fT[fi] = T;
}

__device__ __forceinline__ double2 draw_noise(const RunParams& P, uint32_t id, long long step) {
    const uint4 rb = philox4x32_10(make_uint4(0u, id, (uint32_t)step, 0u), P.key0, P.key1);
    return normals2_f64(rb.x, rb.y);
}

}  // namespace

// Biases without many slices: a CTA steps 1 << lg replicas on its first warp (one lane each,
// the other lanes repeat them) while three more warps draw the noise of the next batch of
// 3 * (32 >> lg) steps, one step of one replica per lane. The double well (256 replicas, two
// per CTA) takes 0.51 us per step against 3.6 us with noise and step in one lane. (Replicas are spread over the SMs first: lg is the smallest for which
// there is at most one CTA per SM, up to a full warp of replicas.)
template <int BIAS>
__global__ void __launch_bounds__(32 * (1 + kPlaneProducers))
k_plane(StateDev st, RunParams P, const uint32_t* __restrict__ rep_ids, int lg) {
    __shared__ double2 noise[2][32 * kPlaneProducers];
    const int warp = threadIdx.x >> 5;
    const Lanes L = {(int)(threadIdx.x & 31), lg};
    const int G = 1 << lg, per = 32 >> lg, batch = kPlaneProducers * per;
    const int slot_r = blockIdx.x * G + L.g();
    const bool mine = slot_r < P.n_replicas && L.copy() == 0;
    const int r = min(slot_r, P.n_replicas - 1);
    const long long step0 = st.step[r];
    const uint32_t id = rep_ids[r];
    auto draw = [&](long long s0, int buf) {
        const long long s = s0 + (warp - 1) * per + L.copy();
        if (s < P.n_steps) noise[buf][(warp - 1) * 32 + L.lane] = draw_noise(P, id, step0 + s);
    };
    double2 p = st.xy[r];
    double zm = st.zm[r], T = st.T[r], sm = st.sm[r], wm = st.wm[r];
    Saver sv;
    sv.init(P, step0, st.n_saved[r]);
    const double a = P.toy_dt_over_gamma, sd = P.toy_sd, xr = P.toy_x_ref;
    if (warp > 0) draw(0, 0);
    __syncthreads();
    int buf = 0;
    for (long long s0 = 0; s0 < P.n_steps; s0 += batch, buf ^= 1) {
        if (warp > 0) {
            draw(s0 + batch, buf ^ 1);
        } else {
            const int m = (int)min((long long)batch, P.n_steps - s0);
            for (int k = 0; k < m; ++k) {
                double2 f = model_force(L, P.toy_model, p);
                double bx = 0.0, by = 0.0;
                if (BIAS == 2) {  // Eq. (FrMD) with theta(0) = 1
                    const double d = p.x - xr, z = d * d, dz = z - zm;
                    const bool low = below_zero(dz);
                    bx = low ? 0.0 : (-2.0 * P.k_R) * dz * d;
                    zm = low ? z : zm;
                    T += a * (bx * bx);
                    f.x += bx;
                } else if (BIAS == 3) {
                    const double z = sqrt(dot2(p.x, p.x, p.y, p.y)), dz = z - zm;
                    const double2 gz = div_two(L, p.x, z, p.y, z);
                    const bool low = below_zero(dz);
                    const double fac = -P.k_R * dz;
                    bx = low || !(z > 0.0) ? 0.0 : fac * gz.x;
                    by = low || !(z > 0.0) ? 0.0 : fac * gz.y;
                    zm = low ? z : zm;
                } else if (BIAS == 4) {
                    double s, w;
                    double2 gs, gw;
                    tube_vars(P, p, &s, &w, &gs, &gw);
                    double fs = 0.0, fw = 0.0;
                    if (s < sm) sm = s; else fs = -P.tube_ks * (s - sm);
                    if (w < wm) wm = w; else fw = -P.tube_kw * (w - wm);
                    bx = dot2(fs, gs.x, fw, gw.x);
                    by = dot2(fs, gs.y, fw, gw.y);
                }
                if (BIAS >= 3) {
                    f.x += bx;
                    f.y += by;
                    T = __fma_rn(a, dot2(bx, bx, by, by), T);  // (dt / gamma) |F_bias|^2, unit mass
                }
                const double2 xi = noise[buf][k * G + L.g()];
                p.x = p.x + a * f.x + sd * xi.x;
                p.y = p.y + a * f.y + sd * xi.y;
                if (sv.step(P)) {
                    if (mine) {
                        double z = 0.0, zmin = 0.0;
                        if (BIAS == 2 || BIAS == 3) {
                            z = BIAS == 2 ? (p.x - xr) * (p.x - xr) : sqrt(p.x * p.x + p.y * p.y);
                            zmin = zm < z ? zm : z;
                        } else if (BIAS == 4) {  // frames record s_lambda and its running minimum
                            double w;
                            double2 gs, gw;
                            tube_vars(P, p, &z, &w, &gs, &gw);
                            zmin = sm < z ? sm : z;
                        }
                        const long long fi = (long long)r * P.max_frames + sv.slot;
                        save_position(st, P, r, sv.slot, p, T);
                        st.fz[fi] = z;
                        st.fzm[fi] = zmin;
                    }
                    sv.saved(P);
                }
            }
        }
        __syncthreads();
    }
    if (warp > 0 || !mine) return;
    double z;  // of the final configuration (s_lambda for the tube bias)
    if (BIAS == 3) {
        z = sqrt(p.x * p.x + p.y * p.y);
    } else if (BIAS == 4) {
        double w;
        double2 gs, gw;
        tube_vars(P, p, &z, &w, &gs, &gw);
    } else {
        z = (p.x - xr) * (p.x - xr);
    }
    st.xy[r] = p;
    st.zm[r] = zm;
    st.sm[r] = sm;
    st.wm[r] = wm;
    st.z[r] = z;
    st.T[r] = T;
    st.step[r] = step0 + P.n_steps;
    st.n_saved[r] = sv.ns;
    if (!(isfinite(p.x) && isfinite(p.y))) st.status[r] = 1;
}

// Factors of the terms of one slice: e_k, e_k t_k, 1, and the components of X - <X(t'_k)>.
struct Term {
    double f[5];
};

// Tube bias, one replica per warp (see tube_by_warps): slice k on lane k & 31 (NB slices per lane,
// kept in registers for up to 128 slices; NB = 0 reads them from memory). 512 replicas x 100
// slices: 12.5 us per step against 145 us with one lane per replica walking all slices. Every sum keeps the order of that plain walk (the lane-tree sums that
// would save a quarter of the time change the last bits, which these trajectories amplify to
// 1e-6 of the bias functional within a round), so results depend neither on the lanes nor on
// how many replicas run beside one another.
template <int NB>
__global__ void __launch_bounds__(128)
k_plane_tube(StateDev st, RunParams P, const uint32_t* __restrict__ rep_ids) {
    __shared__ double2 noise_s[4][32];
    __shared__ Term term[4][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = blockIdx.x * (blockDim.x >> 5) + warp;
    if (r >= P.n_replicas) return;  // (whole warps; no block-wide barrier below)
    const Lanes L = {lane, 0};
    const int K = P.tube_k;
    constexpr int NR = NB > 0 ? NB : 1;
    double2 ref[NR];
    double tk[NR];
    if (NB > 0) {
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int k = lane + 32 * i;
            ref[i] = k < K ? P.tube_ref[k] : make_double2(0.0, 0.0);
            tk[i] = k < K ? P.tube_time[k] : 0.0;
        }
    }
    const uint32_t id = rep_ids[r];
    double2 p = st.xy[r];
    double T = st.T[r], sm = st.sm[r], wm = st.wm[r], z = 0.0;
    const long long step0 = st.step[r];
    Saver sv;
    sv.init(P, step0, st.n_saved[r]);
    const double a = P.toy_dt_over_gamma, sd = P.toy_sd, c = P.tube_lambda / P.tube_t;
    bool pending = false;  // a frame waits for its s_lambda, which the next evaluation gives
    for (long long s = 0;; ++s) {
        // distances, and the smallest (non-negative FP64 values order as their bits)
        double dx[NR], dy[NR];
        unsigned long long best = ~0ull;
        auto dist = [&](double ex, double ey) { return dot2(ex, ex, ey, ey); };
        if (NB > 0) {
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                dx[i] = p.x - ref[i].x;
                dy[i] = p.y - ref[i].y;
                if (lane + 32 * i < K)
                    best = min(best, (unsigned long long)__double_as_longlong(dist(dx[i], dy[i])));
            }
        } else {
            for (int k = lane; k < K; k += 32) {
                const double2 q = P.tube_ref[k];
                best = min(best, (unsigned long long)__double_as_longlong(dist(p.x - q.x, p.y - q.y)));
            }
        }
        const unsigned hi = __reduce_min_sync(kFullP, (unsigned)(best >> 32));
        const unsigned lo = __reduce_min_sync(kFullP, (unsigned)(best >> 32) == hi ? (unsigned)best : ~0u);
        const double dmin = __longlong_as_double((long long)(((unsigned long long)hi << 32) | lo));
        // sums with the largest weight scaled to 1 (the formulas are unchanged). The lanes
        // compute the weights of 32 slices at a time and leave the factors of each slice's
        // terms in shared memory; then lane v adds term v of every slice in turn: one FP64
        // instruction per slice for all six sums, in the order of a plain loop.
        double acc = 0.0;
        // lane v: S, St, and half of g1 and g2 (e_k X, e_k t_k X)
        const int iu = (0x110010 >> (4 * min(lane, 5))) & 7, iw = (0x434322 >> (4 * min(lane, 5))) & 7;
        auto block = [&](int k0, double ex, double ey, double t) {
            const double e = exp(-P.tube_lambda * (dist(ex, ey) - dmin));
            Term& w = term[warp][lane];
            w.f[0] = e;
            w.f[1] = __dmul_rn(e, t);
            w.f[2] = 1.0;
            w.f[3] = ex;
            w.f[4] = ey;
            __syncwarp();
            const int m = min(32, K - k0);
#pragma unroll 8
            for (int k = 0; k < m; ++k) acc = __fma_rn(term[warp][k].f[iu], term[warp][k].f[iw], acc);
            __syncwarp();
        };
        if (NB > 0) {
#pragma unroll
            for (int i = 0; i < NR; ++i) block(32 * i, dx[i], dy[i], tk[i]);
        } else {
            for (int k0 = 0; k0 < K; k0 += 32) {
                const int k = min(k0 + lane, K - 1);
                const double2 q = P.tube_ref[k];
                block(k0, p.x - q.x, p.y - q.y, P.tube_time[k]);
            }
        }
        const double S = __shfl_sync(kFullP, acc, 0), St = __shfl_sync(kFullP, acc, 1);
        const double tm = St / S;  // <t'> under pi
        // lanes 2..5: g1 / S and g2 / S, lanes 6, 7: tm g1 / S (all halved)
        const double g1x = __shfl_sync(kFullP, acc, 2), g1y = __shfl_sync(kFullP, acc, 3);
        double num = acc;
        if (lane == 6) num = tm * g1x;
        if (lane == 7) num = tm * g1y;
        const double q = num / S;
        const double2 gw = make_double2(__shfl_sync(kFullP, q, 2), __shfl_sync(kFullP, q, 3));
        const double2 gs = make_double2(c * (__shfl_sync(kFullP, q, 4) - __shfl_sync(kFullP, q, 6)),
                                        c * (__shfl_sync(kFullP, q, 5) - __shfl_sync(kFullP, q, 7)));
        const double2 wt = div_two(L, log(S), P.tube_lambda, tm, P.tube_t);
        const double w_ = dmin - wt.x, s_ = 1.0 - wt.y;
        z = s_;
        if (pending) {
            if (lane == 0) {
                const long long fi = (long long)r * P.max_frames + sv.slot;
                st.fz[fi] = s_;  // frames record s_lambda and its running minimum
                st.fzm[fi] = sm < s_ ? sm : s_;
            }
            sv.saved(P);
            pending = false;
        }
        if (s == P.n_steps) break;
        if ((s & 31) == 0) {  // the noise of the next 32 steps, one per lane
            __syncwarp();
            if (s + lane < P.n_steps) noise_s[warp][lane] = draw_noise(P, id, step0 + s + lane);
            __syncwarp();
        }
        const double ds = s_ - sm, dw = w_ - wm;
        const bool ls = below_zero(ds), lw = below_zero(dw);
        // (twice the factors: gs and gw are half the gradients)
        const double fs = ls ? 0.0 : -2.0 * P.tube_ks * ds, fw = lw ? 0.0 : -2.0 * P.tube_kw * dw;
        sm = ls ? s_ : sm;
        wm = lw ? w_ : wm;
        const double bx = dot2(fs, gs.x, fw, gw.x), by = dot2(fs, gs.y, fw, gw.y);
        double2 f = model_force(L, P.toy_model, p);
        f.x += bx;
        f.y += by;
        T = __fma_rn(a, dot2(bx, bx, by, by), T);  // (dt / gamma) |F_bias|^2, unit mass
        const double2 xi = noise_s[warp][s & 31];
        p.x = p.x + a * f.x + sd * xi.x;
        p.y = p.y + a * f.y + sd * xi.y;
        if (sv.step(P)) {
            if (lane == 0) save_position(st, P, r, sv.slot, p, T);
            pending = true;
        }
    }
    if (lane) return;
    st.xy[r] = p;
    st.sm[r] = sm;
    st.wm[r] = wm;
    st.z[r] = z;
    st.T[r] = T;
    st.step[r] = step0 + P.n_steps;
    st.n_saved[r] = sv.ns;
    if (!(isfinite(p.x) && isfinite(p.y))) st.status[r] = 1;
}

// Whether a warp per replica takes the tube sums (k_plane_tube), or a lane per replica (k_plane).
// Below eight slices most lanes of a warp would idle in the exp that dominates a slice. Above,
// a step of a warp is shorter by far, but a quarter of an SM takes the lanes of a warp (32
// replicas) in the time of one, and warps one after another, so the lanes win with many replicas:
// the cheaper of waves x measured time per step wins (40 steps, us: a warp 207 with 8 slices,
// 435 with 100; a lane 656 and 5130. 4096 replicas x 8 slices: 1429 us as warps, 660 as lanes;
// 32 768 x 100: 22 667 and 11 694). Both sum in the same order: the bits are the same.
constexpr int kTubeWarpMin = 8;

bool tube_by_warps(int R, int K, int n_sm) {
    if (K < kTubeWarpMin) return false;
    const long long warps = (R + 4ll * n_sm - 1) / (4 * n_sm), lanes = (R + 128ll * n_sm - 1) / (128 * n_sm);
    return warps * (163 + 1.4 * K + 33 * ((K + 31) / 32)) < lanes * (230 + 54.0 * K);
}

cudaError_t launch_toy(const StateDev& st, const RunParams& P, const uint32_t* rep_ids,
                       cudaStream_t stream) {
    int dev = 0, n_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int R = P.n_replicas;
    if (P.bias == 4 && tube_by_warps(R, P.tube_k, n_sm)) {
        // one warp per quarter of an SM, spread over all SMs first
        const int per = std::min(4, (R + n_sm - 1) / n_sm);
        const dim3 grid((R + per - 1) / per);
        const int nb = (P.tube_k + 31) / 32;
        if (nb == 1) k_plane_tube<1><<<grid, 32 * per, 0, stream>>>(st, P, rep_ids);
        else if (nb == 2) k_plane_tube<2><<<grid, 32 * per, 0, stream>>>(st, P, rep_ids);
        else if (nb == 3) k_plane_tube<3><<<grid, 32 * per, 0, stream>>>(st, P, rep_ids);
        else if (nb == 4) k_plane_tube<4><<<grid, 32 * per, 0, stream>>>(st, P, rep_ids);
        else k_plane_tube<0><<<grid, 32 * per, 0, stream>>>(st, P, rep_ids);
        return cudaGetLastError();
    }
    int lg = 0;
    while (lg < 5 && (R + (1 << lg) - 1) >> lg > n_sm) ++lg;
    const dim3 grid((R + (1 << lg) - 1) >> lg);
    const int th = 32 * (1 + kPlaneProducers);
    if (P.bias == 2) k_plane<2><<<grid, th, 0, stream>>>(st, P, rep_ids, lg);
    else if (P.bias == 3) k_plane<3><<<grid, th, 0, stream>>>(st, P, rep_ids, lg);
    else if (P.bias == 4) k_plane<4><<<grid, th, 0, stream>>>(st, P, rep_ids, lg);
    else k_plane<0><<<grid, th, 0, stream>>>(st, P, rep_ids, lg);
    return cudaGetLastError();
}

}  // namespace scps
