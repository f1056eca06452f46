// Body of the persistent single-right-hand-side shifted-COCG kernel.  See
// solver.cuh for the algorithm; this file holds the phases.
#pragma once
#include <type_traits>

#include "solver.cuh"

namespace scocg {

// A warp sum parked in a double-sized scratch slot in its own type, so that
// only the final sum over warps uses the FP64 pipe: an FP64 instruction holds
// the SM's FP64 pipe for 16 cycles whatever its active lanes.
__device__ __forceinline__ void park(double* slot, double v) { *slot = v; }
__device__ __forceinline__ void park(double* slot, float v) { *reinterpret_cast<float*>(slot) = v; }
__device__ __forceinline__ void park(double* slot, dfs v) { *reinterpret_cast<dfs*>(slot) = v; }
template <typename T> __device__ __forceinline__ double unpark(const double* slot);
template <> __device__ __forceinline__ double unpark<double>(const double* slot) { return *slot; }
template <> __device__ __forceinline__ double unpark<float>(const double* slot) {
    return (double)*reinterpret_cast<const float*>(slot);
}
template <> __device__ __forceinline__ double unpark<dfs>(const double* slot) {
    return to_double(*reinterpret_cast<const dfs*>(slot));
}

// Where a CTA's partial sums of one reduction go: value j to part[j * G] (read
// after a grid barrier), or, with pk set, to packet pk[j * G] = {value, tag}
// that the other CTAs wait for directly (grids up to kPktCtas = 32).
struct PartialOut {
    double* part;
    ulonglong2* pk;
    int G;
    unsigned long long tag;
    bool skip;               // fault injection: do not publish
    __device__ __forceinline__ void put(int j, double t) const {
        if (!pk) part[(size_t)j * G] = t;
        else if (!skip) st_packet(pk + (size_t)j * G, t, tag);
    }
};

// CTA sums of the first nv of NV per-thread values, of which only the warps
// with place wi < nw hold any: warp j < nv publishes sum j (the caller
// synchronises the CTA before anyone reuses scratch).  Each sum is a tree, not
// a chain: a serial FP64 chain over 16 warps was ~0.5 us of every seed
// iteration, twice.
template <int NV, typename T, int kScratch>
__device__ __forceinline__ void block_partials(T (&v)[NV], double (&scratch)[kScratch], const PartialOut& out, int wi,
                                               int nv = NV, int nw = kWarps) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    static_assert(kScratch >= NV * (std::is_same<T, double>::value ? kBlock : kWarps), "scratch too small");
    if constexpr (std::is_same<T, double>::value) {
        // FP64 values: every thread parks its values and nv warps sum them,
        // instead of five-step FP64 warp sums in all warps
        if (wi < nw)
#pragma unroll
            for (int j = 0; j < NV; ++j)
                if (j < nv) scratch[j * kBlock + 32 * wi + lane] = v[j];
        __syncthreads();
        if (out.pk && warp < nv && lane == 0) fence_acq_rel();   // the CTA's writes come before its packets
        if (warp < nv) {
            double a[4] = {0.0, 0.0, 0.0, 0.0};
            for (int w = 0; w < nw; w += 4)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (w + q < nw) {
                        const double t = scratch[warp * kBlock + 32 * (w + q) + lane];
                        a[q] = w == 0 ? t : a[q] + t;
                    }
            if (nw > 2) { a[0] += a[2]; if (nw > 3) a[1] += a[3]; }
            if (nw > 1) a[0] += a[1];
            const double t = warp_sum(a[0]);
            if (lane == 0) out.put(warp, t);
        }
    } else {
        // the warp-level part in the values' own type, the sum over warps in FP64
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            if (j >= nv) break;
            const T t = warp_sum(v[j]);
            if (lane == 0) park(scratch + j * kWarps + wi, t);
        }
        __syncthreads();
        if (out.pk && warp < nv && lane == 0) fence_acq_rel();
        if (warp < nv) {
            double t = lane < kWarps ? unpark<T>(scratch + warp * kWarps + lane) : 0.0;
#pragma unroll
            for (int o = kWarps / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) out.put(warp, t);
        }
    }
}

// per-thread accumulation of u^T v (bilinear) in the vector precision
__device__ __forceinline__ void acc_bil(double& re, double& im, double2 u, double2 v) {
    re = fma(u.x, v.x, fma(-u.y, v.y, re)); im = fma(u.x, v.y, fma(u.y, v.x, im));
}
__device__ __forceinline__ void acc_bil(float& re, float& im, float2 u, float2 v) {
    re = fmaf(u.x, v.x, fmaf(-u.y, v.y, re)); im = fmaf(u.x, v.y, fmaf(u.y, v.x, im));
}
__device__ __forceinline__ void acc_nrm(double& s, double2 u) { s = fma(u.x, u.x, fma(u.y, u.y, s)); }
__device__ __forceinline__ void acc_nrm(float& s, float2 u) { s = fmaf(u.x, u.x, fmaf(u.y, u.y, s)); }
// compensated: products exact to DF, sums with TwoSum; the real and
// imaginary parts as one packed pair, (re, im) += (u.re, u.re) (v.re, v.im)
// + (-u.im, u.im) (v.im, v.re)
__device__ __forceinline__ void acc_bil(dfs& re, dfs& im, float4 u, float4 v) {
    float2 h = make_float2(re.hi, im.hi), l = make_float2(re.lo, im.lo);
    pk_acc_prod(h, l, make_float2(u.x, u.x), make_float2(u.z, u.z), hi2(v), lo2(v));
    pk_acc_prod(h, l, make_float2(-u.y, u.y), make_float2(-u.w, u.w), make_float2(v.y, v.x), make_float2(v.w, v.z));
    re = dfs{h.x, l.x};
    im = dfs{h.y, l.y};
}
__device__ __forceinline__ void acc_nrm(dfs& s, float4 u) {
    df_acc_prod(s, cre(u), cre(u));
    df_acc_prod(s, cim(u), cim(u));
}

// Per-thread accumulation of rho = r^T r and ||r||^2, and the thread's totals
// (re rho, im rho, ||r||^2) after its last row.
template <typename AT, typename V>
__device__ __forceinline__ void acc_rr(AT& re, AT& im, AT& nrm, V ri) {
    acc_bil(re, im, ri, ri);
    acc_nrm(nrm, ri);
}
template <typename AT>
__device__ __forceinline__ void end_rr(AT&, AT&, AT&) {}
// complex128: sum of x^2 - y^2, of x y and of y^2 (four FP64 FMAs a row
// instead of six), combined once per thread
template <>
__device__ __forceinline__ void acc_rr<double, double2>(double& re, double& xy, double& yy, double2 ri) {
    re = fma(ri.x, ri.x, fma(-ri.y, ri.y, re));
    xy = fma(ri.x, ri.y, xy);
    yy = fma(ri.y, ri.y, yy);
}
template <>
__device__ __forceinline__ void end_rr<double>(double& re, double& xy, double& yy) {
    xy += xy;
    yy = fma(2.0, yy, re);
}
// Compensated vectors: rho = sum (x^2 - y^2) + 2i sum x y from three
// pair-exact products (the doubling is exact), and ||r||^2 from the high
// parts in FP32: it only feeds the convergence test, where a relative
// accuracy of 1e-7 is ample.
template <>
__device__ __forceinline__ void acc_rr<dfs, float4>(dfs& re, dfs& im, dfs& nrm, float4 ri) {
    // (re, im) += (x, x) (x, 2y) + (-y, 0) (y, 0), packed
    float2 h = make_float2(re.hi, im.hi), l = make_float2(re.lo, im.lo);
    pk_acc_prod(h, l, make_float2(ri.x, ri.x), make_float2(ri.z, ri.z), make_float2(ri.x, 2.f * ri.y),
                make_float2(ri.z, 2.f * ri.w));
    pk_acc_prod(h, l, make_float2(-ri.y, 0.f), make_float2(-ri.w, 0.f), make_float2(ri.y, 0.f),
                make_float2(ri.w, 0.f));
    re = dfs{h.x, l.x};
    im = dfs{h.y, l.y};
    nrm.hi = fmaf(ri.x, ri.x, fmaf(ri.y, ri.y, nrm.hi));
}

// Per-thread accumulation of the r partials: rho = r^T r, ||r||^2, c_0^T r.
template <typename R>
__device__ __forceinline__ void acc_r(typename Acc<R>::T (&acc)[5], typename Vec<R>::T ri,
                                     const typename Vec<R>::T* c0) {
    acc_rr(acc[0], acc[1], acc[2], ri);
    if (c0) acc_bil(acc[3], acc[4], *c0, ri);
}

// r_{n+1} = r_n - alpha_n q_n (one fused multiply-add for compensated vectors)
template <typename V>
__device__ __forceinline__ V r_update(V r, V al, V q) { return vsub(r, vcfma(al, q, vzero<V>())); }
template <>
__device__ __forceinline__ double2 r_update<double2>(double2 r, double2 al, double2 q) {
    return vcfma(make_double2(-al.x, -al.y), q, r);
}
template <>
__device__ __forceinline__ float4 r_update<float4>(float4 r, float4 al, float4 q) {
    return vcfma(make_float4(-al.x, -al.y, -al.z, -al.w), q, r);
}

// A CTA's share of the rows and where its part of q lives.  Its units are
// numbered lu = 0 .. nloc - 1 and its rows t = 0 .. nrow - 1; every phase of an
// iteration gives a row to the same CTA, so q, which only the row's owner
// reads, can stay in shared memory (on): it is then neither written to nor read
// from L2, and the first reduction's release has no vector stores to wait for.
// A strided apply (Hubbard, q in global memory) uses contiguous rows in the
// row-wise phases.
template <class Apply, typename V>
struct RowShare {
    static constexpr bool kStrided = Apply::kMap == kMapStrided;
    static constexpr int kRpu = Apply::kRowsPerUnit;
    int G, cta, nloc, nrow;
    int64_t ubeg, rbeg;
    bool on;
    V* q_s;
    V* q_g;
    __device__ __forceinline__ RowShare(int64_t n, int64_t nunits, int G_, int cta_, bool on_, V* qs, V* qg)
        : G(G_), cta(cta_), on(!kStrided && on_), q_s(qs), q_g(qg) {
        if constexpr (kStrided) {
            ubeg = cta;
            nloc = cta < nunits ? (int)((nunits - cta + G - 1) / G) : 0;
            rbeg = (int64_t)cta * n / G;
            nrow = (int)((int64_t)(cta + 1) * n / G - rbeg);
        } else {
            ubeg = (int64_t)cta * nunits / G;
            nloc = (int)((int64_t)(cta + 1) * nunits / G - ubeg);
            rbeg = ubeg * kRpu;
            nrow = (int)(min(n, rbeg + (int64_t)nloc * kRpu) - rbeg);
        }
    }
    __device__ __forceinline__ int64_t unit(int lu) const { return kStrided ? ubeg + (int64_t)G * lu : ubeg + lu; }
    __device__ __forceinline__ int64_t row(int t) const { return rbeg + t; }
    // place of the row that `lane` owns in unit lu
    __device__ __forceinline__ int place(int lu, int lane) const { return lu * kRpu + lane / (32 / kRpu); }
    __device__ __forceinline__ V get(int t, int64_t r) const { return on ? q_s[t] : q_g[r]; }
    __device__ __forceinline__ void put(int t, int64_t r, V v) const {
        if (on) q_s[t] = v; else q_g[r] = v;
    }
};

// CTA sums of the accumulated partials into values 0..2 (0..4 with dense
// projections) of this CTA's column of the value-major partials (value j at
// part[j * G]); the extra dense projections m >= 1 are summed in separate
// passes over r into values 3 + 2m.
template <typename R, class Share, int kScratch>
__device__ __forceinline__ void finish_r_partials(const SolveArgs<R>& a, typename Acc<R>::T (&acc)[5],
                                                  const Share& sh, double (&scratch)[kScratch],
                                                  const PartialOut& out) {
    using AT = typename Acc<R>::T;
    const int tid = threadIdx.x;
    const int nw = min(kWarps, (sh.nrow + 31) >> 5);   // warps that hold rows
    end_rr(acc[0], acc[1], acc[2]);
    block_partials<5>(acc, scratch, out, tid >> 5, a.cvec ? 5 : 3, max(nw, 1));
    for (int m = 1; m < a.nproj && a.cvec; ++m) {
        AT w2[2] = {};
        for (int t = tid; t < sh.nrow; t += kBlock) {
            const int64_t i = sh.row(t);
            acc_bil(w2[0], w2[1], a.cvec[(size_t)m * a.n + i], a.r[i]);
        }
        __syncthreads();   // the sums above have been read from scratch
        const PartialOut om{out.part + (size_t)(3 + 2 * m) * out.G, nullptr, out.G, 0ull, false};   // more than one: no packets
        block_partials<2>(w2, scratch, om, tid >> 5, 2, max(nw, 1));
    }
}

template <typename R, class Share, int kScratch>
__device__ __forceinline__ void r_partials(const SolveArgs<R>& a, const Share& sh, double (&scratch)[kScratch],
                                           const PartialOut& out) {
    typename Acc<R>::T acc[5] = {};
    for (int t = threadIdx.x; t < sh.nrow; t += kBlock) {
        const int64_t i = sh.row(t);
        acc_r<R>(acc, a.r[i], a.cvec ? a.cvec + i : nullptr);
    }
    finish_r_partials(a, acc, sh, scratch, out);
}

#ifdef SCOCG_CHECKED
#define SCOCG_TRACE(ph)                                                    \
    do {                                                                   \
        if (threadIdx.x == 0 && a.trace) {                                 \
            volatile int* t_ = a.trace + 2 * cta;                          \
            t_[0] = s.n; t_[1] = (ph);                                     \
            __threadfence_system();                                        \
        }                                                                  \
    } while (0)
#else
#define SCOCG_TRACE(ph) do { } while (0)
#endif

// Optional per-phase wall-time accounting (-DSCOCG_PHASE_TIMERS): thread 0 of
// each CTA adds the time spent since the previous mark to slot `k` of its row in
// a.phase_ns ([grid][8] nanoseconds).
#ifdef SCOCG_PHASE_TIMERS
#define SCOCG_MARK(k)                                                      \
    do {                                                                   \
        if (threadIdx.x == 0 && a.phase_ns) {                              \
            const uint64_t t_ = globaltimer_ns();                          \
            a.phase_ns[8 * cta + (k)] += t_ - t_mark;                      \
            t_mark = t_;                                                   \
        }                                                                  \
    } while (0)
#else
#define SCOCG_MARK(k) do { } while (0)
#endif

// The inputs of one phase C (the per-shift update of seed iteration n): the
// seed scalars alpha_n, beta_{n-1}, alpha_n beta_{n-1} / alpha_{n-1},
// (||r_{n+1}|| / ||b||)^2 and c_m^T r_n.  Phase C can run one iteration late,
// inside the next phase A, from this copy.
struct ShiftInputs {
    double2 alpha, beta_prev, t2;
    double rn_b2;
    int n;
    double2 cr[kMaxProj];
};

// The per-shift state of a CTA's own shifts in shared memory, one slot per
// owning thread: each seed iteration reads and writes it once, and a global
// load after a grid barrier is a round trip to L2 (300 to 800 cycles).  Used
// when every owner is in warp 0 and a shift has at most kOwnM projections; the
// state is copied to the global arrays at the end of the solve.
constexpr int kOwn = 32, kOwnM = 2;
struct OwnShifts {
    double2 pi_prev[kOwn], pi_cur[kOwn], sigma[kOwn], alpha_k[kOwn], inv_cur[kOwn];
    double2 P[kOwn * kOwnM], X[kOwn * kOwnM];
    double resid[kOwn];
    int frozen[kOwn], iters[kOwn];
};
__device__ __forceinline__ ShiftState own_view(OwnShifts& o) {
    return ShiftState{o.pi_prev, o.pi_cur, o.sigma, o.alpha_k, o.inv_cur, o.P, o.X, o.frozen, o.iters, o.resid};
}

// pi_{n+1} = (1 + alpha sigma) pi_n + t2 (pi_n - pi_{n-1}), t2 = alpha_n beta_{n-1} /
// alpha_{n-1}.  With the operations spelt out, so that every place that forms it
// from the same inputs has the same bits: the full-vector mode's steps and the
// recurrence would otherwise use different numbers wherever pi_{n+1} comes out of
// a cancellation, and x^k loses what they differ by (t2 rounded in another order
// there: errors of x 20 to 35 % larger at Im z = 0.1, up to 25 times on single systems).
__device__ __forceinline__ double2 pi_next(double2 alpha, double2 t2, double2 sigma, double2 pc, double2 pp) {
    const auto mul = [](double2 a, double2 b) {
        return c2(fma(a.x, b.x, -__dmul_rn(a.y, b.y)), fma(a.x, b.y, __dmul_rn(a.y, b.x)));
    };
    const auto add = [](double2 a, double2 b) { return c2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y)); };
    return add(mul(add(c2(1, 0), mul(alpha, sigma)), pc), mul(t2, add(pc, c2(-pp.x, -pp.y))));
}

// t2 from beta_{n-1} / alpha_{n-1}, which is known before alpha_n
__device__ __forceinline__ double2 shift_t2(double2 alpha, double2 ratio) {
    return c2(fma(alpha.x, ratio.x, -__dmul_rn(alpha.y, ratio.y)), fma(alpha.x, ratio.y, __dmul_rn(alpha.y, ratio.x)));
}

// Phase C for the shift in slot k of S: the pi three-term recurrence, the
// projected p^k and x^k, the residual estimate and freezing.  Sets bad for a
// zero or non-finite pi (its state is then left as it was), active when the
// shift stays unconverged.
__device__ __forceinline__ void shift_update(const ShiftState& S, int k, const ShiftInputs& c, int M, double tol,
                                             double tol2, int& active, int& bad) {
    const double2 pp = S.pi_prev[k], pc = S.pi_cur[k], ic = S.inv_cur[k];
    const double2 pn = pi_next(c.alpha, c.t2, S.sigma[k], pc, pp);
    const double2 in = crecip(pn);
    const double2 ratio = cmul(pp, ic);                        // pi_{n-1} / pi_n
    const double2 beta_k = cmul(cmul(ratio, ratio), c.beta_prev);
    const double2 ak = cmul(cmul(pc, in), c.alpha);            // alpha^k_n
    const double res2 = c.rn_b2 * cabs2(in);
    if (cabs2(pn) == 0.0 || !cfinite(pn) || !cfinite(in)) {
        bad = 1;
        return;
    }
    for (int m = 0; m < M; ++m) {
        const size_t o = (size_t)k * M + m;
        const double2 P = cadd(cmul(c.cr[m], ic), cmul(beta_k, S.P[o]));
        S.P[o] = P;
        S.X[o] = cadd(S.X[o], cmul(ak, P));
    }
    S.alpha_k[k] = ak;
    S.pi_prev[k] = pc;
    S.pi_cur[k] = pn;
    S.inv_cur[k] = in;
    S.resid[k] = res2;
    S.iters[k] = c.n + 1;
    if (tol > 0.0 && res2 <= tol2) S.frozen[k] = 1;
    else active = 1;
}

// Applies whose phase A runs in two passes (they declare kTwoPass and
// provide units1 / pass1 and units2 / pass2, see ApplyHubbard2).
template <class A, class = void>
struct HasTwoPass : std::false_type {};
template <class A>
struct HasTwoPass<A, std::void_t<decltype(A::kTwoPass)>> : std::integral_constant<bool, A::kTwoPass> {};

// Decision word of the per-iteration checks: kGoOn continues, any other value
// ends the solve with that status (SCOCG_OK is 0, so 0 cannot mean "go on").
constexpr int kGoOn = 0x7fffffff;

// Phase A's third partial: the unconverged shifts of a CTA after the last
// phase C and whether a pi^k became zero or non-finite, as two integers (their
// sums need no FP64 arithmetic).
__device__ __forceinline__ double pack_counts(int active, int bad) { return __hiloint2double(bad, active); }
__device__ __forceinline__ void sum_counts(const double* part, int G, int& active, int& bad) {
    const int lane = threadIdx.x & 31;
    int act = 0, any = 0;
    for (int c = lane; c < G; c += 32) {
        const double v = __ldcg(part + c);
        act += __double2loint(v);
        any |= __double2hiint(v);
    }
    active = __reduce_add_sync(0xffffffffu, act);
    bad = __reduce_or_sync(0xffffffffu, any);
}

// A packet's tag: the reduction's number in the low word; phase A's first
// packet carries the CTA's shift counts in the high word.
__device__ __forceinline__ unsigned long long packet_tag(unsigned no, int active, int bad) {
    return ((unsigned long long)((unsigned)active | (bad ? 0x80000000u : 0u)) << 32) | no;
}

// Waits for nv packets of each of the G <= 32 CTAs (warp j < nv for packet j,
// lane c for CTA c) and leaves their sums, the same in every CTA, in out[0..nv)
// and the counts of packet 0 in counts[0..1] (counts[2]: a wait was given up).  One round trip through L2
// instead of the barrier's arrival, its poll and then the loads of the
// partials (32 CTAs: 1.1 us against 1.25 + 0.6; at 64 CTAs the packets' all-to-all
// traffic makes it the slower one).  A packet is rewritten only
// after a later reduction that every CTA takes part in.  The wait is bounded
// like the grid barrier's; false ends the solve.
__device__ __forceinline__ bool packet_sums(const GridSync& g, const ulonglong2* pk, int G, int nv, unsigned no,
                                            double* out, int* counts) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < nv) {
        double v = 0.0;
        unsigned aux = 0u, any = 0u;
        if (lane < G) {
            unsigned long long tag = 0;
            uint64_t t0 = 0;
            for (unsigned turn = 1;; ++turn) {
                v = ld_packet(pk + (size_t)warp * G + lane, tag);
                if ((unsigned)tag == no) break;
                if (turn & 63u) continue;
                const uint64_t t = globaltimer_ns();
                if (t0 == 0) t0 = t;
                if (ld_volatile_i32(g.status) < 0 || t - t0 > g.timeout_ns) {
                    atomicCAS(g.status, 0, (int)SCOCG_ERR_TIMEOUT);
                    atomicCAS(g.status, 1, (int)SCOCG_ERR_TIMEOUT);
                    counts[2] = 1;
                    break;
                }
            }
            aux = (unsigned)(tag >> 32) & 0x7fffffffu;
            any = (unsigned)(tag >> 63);
        }
        __syncwarp();
        fence_acq_rel();   // the CTA's later loads see the writes before the packets
        const double t = warp_sum(v);
        if (lane == 0) out[warp] = t;
        if (warp == 0) {
            aux = __reduce_add_sync(0xffffffffu, aux);
            any = __reduce_or_sync(0xffffffffu, any);
            if (lane == 0) { counts[0] = (int)aux; counts[1] = (int)any; }
        }
    }
    __syncthreads();
    return counts[2] == 0;
}

// Order in which the warps take units when warps 0 and 1 first do scalar work:
// they get the last two places of each round.
__device__ __forceinline__ int rotated_place(int warp) { return (warp + kWarps - 2) % kWarps; }

// a / b by one warp (all lanes return it): the products a conj(b) and |b|^2
// run in different lanes of the same instructions.  A warp issues an FP64
// instruction every 64 cycles however few lanes are active, so the serial time
// of scalar code is its instruction count (cdiv: 17 of them, here 10).
__device__ __forceinline__ double2 warp_cdiv(double2 a, double2 b) {
    const int role = threadIdx.x & 3;
    const int e = max(__double2hiint(b.x) & 0x7ff00000, __double2hiint(b.y) & 0x7ff00000) >> 20;
    if (e < 1023 - 400 || e > 1023 + 400) return cdiv(a, b);   // |b|^2 needs scaling (uniform)
    const double u = role == 0 ? a.x : role == 1 ? a.y : b.x;
    const double v = role == 0 ? a.y : role == 1 ? -a.x : b.y;
    const double p = fma(u, b.x, v * b.y);     // a.x b.x + a.y b.y | a.y b.x - a.x b.y | |b|^2
    const double inv = __drcp_rn(__shfl_sync(0xffffffffu, p, 2));
    const double y = p * inv;
    return c2(__shfl_sync(0xffffffffu, y, 0), __shfl_sync(0xffffffffu, y, 1));
}
// one component (cc = 0: real, 1: imaginary) of a b + c
__device__ __forceinline__ double cfma_part(double2 a, double2 b, int cc, double c) {
    return fma(a.x, cc ? b.y : b.x, fma(a.y, cc ? b.x : -b.y, c));
}
// the lane pair's complex number from each lane's component
__device__ __forceinline__ double2 pair_of(double part, int cc) {
    const double o = __shfl_xor_sync(0xffffffffu, part, 1);
    return cc ? c2(o, part) : c2(part, o);
}
// rho_new / rho from inv = 1 / rho (known before rho_new), with one correction
// step: two lanes of a warp, six FP64 instructions.
__device__ __forceinline__ double2 warp_quot(double2 a, double2 b, double2 inv) {
    const int cc = threadIdx.x & 1;
    const double2 y = pair_of(cfma_part(a, inv, cc, 0.0), cc);
    const double2 r = pair_of(cfma_part(c2(-y.x, -y.y), b, cc, cc ? a.y : a.x), cc);
    return pair_of(cfma_part(r, inv, cc, cc ? y.y : y.x), cc);
}

// Phase C for the CTA's nown shifts in shared memory, by one warp: eight lanes
// per shift, four shifts at a time, the independent products of the update in
// lane pairs of the same instructions (24 FP64 instructions instead of ~80 in
// one lane; see warp_cdiv).  Lane pair g = 0: pi and its reciprocal, 1:
// beta^k, 2 and 3: the projections; lane cc of a pair: real or imaginary part.
__device__ __forceinline__ void shift_update_warp(OwnShifts& o, int nown, const ShiftInputs& c, int M, double tol,
                                                  double tol2, int& active, int& bad) {
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31, g = (lane >> 1) & 3, cc = lane & 1, b8 = lane & 24;
    int act = 0, bd = 0;
    for (int k0 = 0; k0 < nown; k0 += 4) {
        const int kk = k0 + (lane >> 3);
        const bool live = kk < nown && !o.frozen[kk];
        if (!__any_sync(kAll, live)) continue;
        const int k = kk < nown ? kk : 0;
        const double2 pp = o.pi_prev[k], pc = o.pi_cur[k], ic = o.inv_cur[k];
        const int m = g == 2 ? 1 : 0;                      // the projection of pair g = 3 (0) or 2 (1)
        const bool has_p = g == 3 || (g == 2 && M > 1);
        const double2 Po = has_p ? o.P[k * M + m] : c2(0, 0), Xo = has_p ? o.X[k * M + m] : c2(0, 0);
        const double2 cr1 = M > 1 ? c.cr[1] : c2(0, 0);
        // 1 + alpha sigma | pi_{n-1} / pi_n | t2 (pi_n - pi_{n-1}) | c_0^T r / pi_n
        const double2 A1 = g == 0 ? c.alpha : g == 1 ? pp : g == 2 ? c.t2 : c.cr[0];
        const double2 B1 = g == 0 ? o.sigma[k] : g == 2 ? csub(pc, pp) : ic;
        const double s1 = cfma_part(A1, B1, cc, g == 0 && cc == 0 ? 1.0 : 0.0);
        const double2 U = pair_of(s1, cc);
        const double v = __shfl_sync(kAll, s1, b8 | 4 | cc);
        // pi_{n+1} | (pi_{n-1} / pi_n)^2 | c_1^T r / pi_n
        const double2 A2 = g == 2 ? cr1 : U, B2 = g == 0 ? pc : g == 1 ? U : ic;
        const double s2 = cfma_part(A2, B2, cc, g == 0 ? v : 0.0);
        const double2 W = pair_of(s2, cc);
        // |pi_{n+1}|^2 | beta^k
        const double b1 = g == 0 ? W.x : cc ? c.beta_prev.y : c.beta_prev.x;
        const double b2 = g == 0 ? W.y : cc ? c.beta_prev.x : -c.beta_prev.y;
        const double s3 = fma(W.x, b1, W.y * b2);
        const double d = __shfl_sync(kAll, s3, b8);
        const double2 pn = c2(__shfl_sync(kAll, s2, b8), __shfl_sync(kAll, s2, b8 | 1));
        const double2 bk = c2(__shfl_sync(kAll, s3, b8 | 2), __shfl_sync(kAll, s3, b8 | 3));
        const double Pn = cfma_part(bk, Po, cc, g == 3 ? s1 : s2);        // p^k_m (pairs 2, 3)
        const double2 Pc = pair_of(Pn, cc);
        const int e = max(__double2hiint(pn.x) & 0x7ff00000, __double2hiint(pn.y) & 0x7ff00000) >> 20;
        const bool plain = e >= 1023 - 400 && e <= 1023 + 400;            // |pi|^2 and its reciprocal in range
        const double inv = __drcp_rn(d);
        const double2 in = pair_of((cc ? -pn.y : pn.x) * inv, cc);
        const double2 w = pair_of(cfma_part(pc, in, cc, 0.0), cc);
        const double2 ak = pair_of(cfma_part(w, c.alpha, cc, 0.0), cc);   // alpha^k_n
        const double Xn = cfma_part(ak, Pc, cc, cc ? Xo.y : Xo.x);
        const double res2 = c.rn_b2 * inv;
        __syncwarp();                                                     // every lane has read the old state
        if (live && plain) {
            double* P = reinterpret_cast<double*>(o.P + k * M + m);
            double* X = reinterpret_cast<double*>(o.X + k * M + m);
            if (has_p) { P[cc] = Pn; X[cc] = Xn; }
            if (g == 0) reinterpret_cast<double*>(o.alpha_k + k)[cc] = cc ? ak.y : ak.x;
            if (g == 1) reinterpret_cast<double*>(o.inv_cur + k)[cc] = cc ? in.y : in.x;
            if (g == 0) {
                reinterpret_cast<double*>(o.pi_prev + k)[cc] = cc ? pc.y : pc.x;
                reinterpret_cast<double*>(o.pi_cur + k)[cc] = cc ? pn.y : pn.x;
            }
            if ((lane & 7) == 0) {
                o.resid[k] = res2;
                o.iters[k] = c.n + 1;
                if (tol > 0.0 && res2 <= tol2) o.frozen[k] = 1;
                else act = 1;
            }
        } else if (live && (lane & 7) == 0) {
            int a1 = 0, b1_ = 0;
            shift_update(own_view(o), k, c, M, tol, tol2, a1, b1_);
            act = a1;
            bd |= b1_;
        }
        active += __popc(__ballot_sync(kAll, act));
        act = 0;
        __syncwarp();
    }
    bad |= __any_sync(kAll, bd);
}

// The first phase A of a solve continued from a ResumeState: the stopped
// apply's r^T q partial again, from the stored r_n and q_n over the same rows
// in the same order (so the continued solve matches an uninterrupted one bit
// for bit), and the shift count as its deferred phase C left it.
template <typename R, class Apply, class Share, int kScratch>
__device__ __forceinline__ void resume_partials(const SolveArgs<R>& a, const Apply& ap, const Share& sh, int nwA,
                                             bool active, double (&scratch)[kScratch], const PartialOut& out) {
    using AT = typename Acc<R>::T;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wi = a.rstate->rotated != 0 ? rotated_place(warp) : warp;
    AT rq[2] = {};
    if constexpr (HasTwoPass<Apply>::value) {
        using V = typename Vec<R>::T;
        for (int64_t u = sh.cta + (int64_t)sh.G * wi; u < ap.template units2<V>(); u += (int64_t)sh.G * kWarps)
            for (int k = 0; k < Apply::template kRows<V>; ++k) {
                int64_t row;
                if (ap.template row2_of<V>(u, lane, k, row)) acc_bil(rq[0], rq[1], a.r[row], a.q[row]);
            }
    } else {
        for (int lu = wi; lu < sh.nloc; lu += kWarps) {
            int64_t row;
            if (ap.row_of(sh.unit(lu), lane, row)) acc_bil(rq[0], rq[1], a.r[row], sh.get(sh.place(lu, lane), row));
        }
    }
    const int act = __syncthreads_count(active);
    PartialOut o = out;
    o.tag = packet_tag((unsigned)out.tag, act, 0);
    block_partials<2>(rq, scratch, o, wi, 2, nwA);
    if (tid == 64) a.partA[2 * sh.G + sh.cta] = pack_counts(act, 0);
    __syncthreads();
}

// Thread 0 of CTA 0 at the end of a solve: the state a later launch continues
// from when the solve stopped at max_iter (right after the apply of iteration
// n).  Out of line, so that the solve loop's code is the same with or without it.
static __device__ __noinline__ void save_resume_state(ResumeState* rs, const SeedScalars& s, int status, int M,
                                               bool rotated) {
    rs->valid = status == SCOCG_NOT_CONVERGED;
    rs->n = s.n; rs->seed = s.seed; rs->n_switch = s.n_switch; rs->n_replace = s.n_replace;
    rs->replace_on = s.replace_on;
    rs->rotated = rotated;
    rs->alpha_prev = s.alpha_prev; rs->beta_prev = s.beta_prev; rs->rho = s.rho; rs->rho_prev = s.rho_prev;
    rs->zs = s.zs; rs->reserved = 0.0; rs->bnorm = s.bnorm;
    for (int m = 0; m < M; ++m) rs->cr_cur[m] = s.cr_cur[m];
}

// The whole solve of one system, run by its G co-resident CTAs (this one is
// number cta among them).
// kResume: the instantiation that continues a stopped solve (a.resume = 1):
// its init takes the stored state and its first phase A only forms the
// stopped apply's partials again.
template <typename R, class Apply, bool kResume = false>
__device__ __forceinline__ void cocg_body(const SolveArgs<R>& a, const Apply& ap, const int G, const int cta) {
    using V = typename Vec<R>::T;
    using AT = typename Acc<R>::T;
    constexpr bool kMixed = std::is_same<R, float>::value;   // complex64 vectors
    constexpr bool kFull = std::is_same<R, double>::value;   // full-vector mode compiled (FP64 only)
    __shared__ SeedScalars s;
    __shared__ int s_flag[8];            // 0, 1: this CTA's shift counts; 2, 3: decision; 4: seed converged; 5, 6: grid counts; 7: lost
    __shared__ double s_min[kWarps];
    __shared__ int s_arg[kWarps];
    __shared__ ShiftInputs s_c;          // inputs of a deferred phase C
    __shared__ OwnShifts s_own;
    // block_partials: five sums over the rows, in FP64 over threads, else over
    // warps (and one FP64 sum over threads, ||b||^2)
    __shared__ double s_scratch[kFull ? kScratchNV * kBlock : kBlock];
    __shared__ int64_t s_cidx[kMaxProj];
    // z_s, beta_{n-1}, alpha_n in the vector type, converted once by thread 0
    // whenever they change (every thread converting them would queue all
    // warps on the FP64 pipe at each phase start)
    __shared__ V s_vs[3];
    SCOCG_DYN_SHARED(double2, s_full);   // full-vector mode: per-shift scalars of the iteration
    __shared__ int s_nact;               // and the number of unconverged shifts

    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    // phase A visits units in the apply's order (kMap)
    const RowShare<Apply, V> sh(a.n, a.nunits, G, cta, a.q_smem != 0,
                                reinterpret_cast<V*>(reinterpret_cast<char*>(s_full) + full_smem(a.Xf ? a.K : 0)),
                                a.q);
    // warps that visit a unit (all of them when there are enough)
    const int nwA = max(1, min(kWarps, sh.nloc));
    const int M = a.nproj;
    const bool dense_proj = a.cvec != nullptr;
    const int nred = dense_proj ? 3 + 2 * M : 3;
    double* myB = a.partB + cta;              // value-major partials: value j at myB[j * G]
    unsigned long long epoch = 0;
    const double tol2 = a.tol * a.tol;
    const int k_own = cta + tid * G;          // the shift this thread owns (if < K)
    const bool owns = k_own < a.K;
    // Phase C may be deferred into the next phase A when every shift owner of
    // every CTA is in warp 0 (K <= 32 G) and no per-shift vectors are formed:
    // warp 0 then updates the shifts while the other warps apply H.  Seed
    // switching needs the shifts of the same iteration, so an iteration whose
    // seed has converged runs phase C in place.
    bool defer_ok = a.K <= 32 * G;
    if constexpr (kFull) defer_ok = defer_ok && a.Xf == nullptr;
    // the own shifts' state: in shared memory where it fits (OwnShifts)
    const bool own_sm = defer_ok && M <= kOwnM;
    auto state = [&]() { return own_sm ? own_view(s_own) : a.S; };
    const int ko = own_sm ? tid : k_own;      // this thread's slot in it
    auto update_own = [&](int& act, int& bad) {
        if (own_sm) shift_update(own_view(s_own), tid, s_c, M, a.tol, tol2, act, bad);
        else shift_update(a.S, k_own, s_c, M, a.tol, tol2, act, bad);
    };
    const int nown = min(kOwn, (a.K - cta + G - 1) / G);   // the CTA's own shifts (own_sm: all of them)
    // few own shifts: eight lanes each (three passes of ~24 FP64 instructions
    // at most); more: one lane each (~80)
    const bool own_wide = own_sm && nown <= 12;
    if (tid < M && !dense_proj) s_cidx[tid] = a.cidx[tid];
    // small grids exchange their partial sums as packets (packet_sums)
    const bool pkt = a.pk != nullptr;
    unsigned red_no = 0;                      // number of the last packet reduction
    const PartialOut outB{myB, nullptr, G, 0ull, false};
    bool pending = false;                     // a deferred phase C waits for the next phase A

    int status = SCOCG_NOT_CONVERGED;
    bool done = false;
#ifdef SCOCG_PHASE_TIMERS
    uint64_t t_mark = globaltimer_ns();
#endif

    // ------------------------------------------------------------ init: r_0 = b, q_{-1} = 0
    // (or, continuing a solve stopped at max_iter, the stored state)
    if constexpr (kResume) {
        if (tid == 0) {
            const ResumeState& rs = *a.rstate;
            s.rho = rs.rho; s.rho_prev = rs.rho_prev;
            s.alpha_prev = rs.alpha_prev; s.beta_prev = rs.beta_prev;
            s.bnorm = rs.bnorm; s.inv_b2 = 1.0 / (s.bnorm * s.bnorm);
            s.seed = rs.seed; s.zs = rs.zs;
            s_vs[0] = Vec<R>::make(s.zs);
            s_vs[1] = Vec<R>::make(s.beta_prev);
            s.n = rs.n;
            s.active = a.K;
            s.replace_on = rs.replace_on; s.n_switch = rs.n_switch; s.n_replace = rs.n_replace;
            s.shift_iters = 0;
        }
        if (tid < M) s.cr_cur[tid] = a.rstate->cr_cur[tid];
        const ShiftState S = state();
        if (own_sm && owns) {
            S.pi_prev[ko] = a.S.pi_prev[k_own]; S.pi_cur[ko] = a.S.pi_cur[k_own]; S.inv_cur[ko] = a.S.inv_cur[k_own];
            S.sigma[ko] = a.S.sigma[k_own]; S.alpha_k[ko] = a.S.alpha_k[k_own];
            for (int m = 0; m < M; ++m) {
                S.P[ko * M + m] = a.S.P[(size_t)k_own * M + m];
                S.X[ko * M + m] = a.S.X[(size_t)k_own * M + m];
            }
            S.frozen[ko] = a.S.frozen[k_own]; S.iters[ko] = a.S.iters[k_own]; S.resid[ko] = a.S.resid[k_own];
        }
        // s_flag[4] (seed converged) decides whether the next apply takes a
        // deferred shift update and visits its units rotated: restored so
        // that a stop right after this pass records the stopped one's order
        if (tid < 8) s_flag[tid] = tid == 4 ? (a.rstate->rotated ? 0 : 1) : 0;
        __syncthreads();
        if (sh.on) {
            for (int t = tid; t < sh.nrow; t += kBlock) sh.q_s[t] = a.q[sh.row(t)];
            __syncthreads();
        }
        resume_partials(a, ap, sh, nwA, owns && !S.frozen[ko], s_scratch,
                         PartialOut{a.partA + cta, pkt ? a.pk + cta : nullptr, G, (unsigned long long)(++red_no), false});
    } else {
        double nb = 0.0;
        const ShiftState S = state();
        for (int t = tid; t < sh.nrow; t += kBlock) {
            const int64_t i = sh.row(t);
            const double2 bi = a.b[i];
            a.r[i] = Vec<R>::make(bi);
            sh.put(t, i, vzero<V>());
            if constexpr (kMixed) {
                a.p_seed[i] = vzero<V>(); a.x_hi[i] = vzero<V>(); a.x_lo[i] = vzero<V>();
            }
            if constexpr (kFull)
                if (a.Xf)
                    for (int k = 0; k < a.K; ++k) { a.Xf[(size_t)k * a.n + i] = c2(0, 0); a.Pf[(size_t)k * a.n + i] = c2(0, 0); }
            nb = fma(bi.x, bi.x, fma(bi.y, bi.y, nb));
        }
        double v1[1] = {nb};
        block_partials<1>(v1, s_scratch, PartialOut{a.partC + (size_t)cta * kPartC, nullptr, G, 0ull, false}, warp);
        __syncthreads();
        r_partials(a, sh, s_scratch, outB);
        if (owns) {
            S.pi_prev[ko] = c2(1, 0); S.pi_cur[ko] = c2(1, 0); S.inv_cur[ko] = c2(1, 0);
            S.sigma[ko] = csub(a.z[k_own], a.z[a.seed]);
            S.alpha_k[ko] = c2(0, 0);
            for (int m = 0; m < M; ++m) { S.P[(size_t)ko * M + m] = c2(0, 0); S.X[(size_t)ko * M + m] = c2(0, 0); }
            S.frozen[ko] = 0; S.iters[ko] = 0; S.resid[ko] = 1.0;
        }
        if (tid < 8) s_flag[tid] = 0;
        if (!grid_barrier(a.sync, epoch)) return;
        grid_sum_vm1(a.partB, nred, s.red, G);
        grid_sum(a.partC, kPartC, 1, s.red + nred, G);
        if (tid == 0) {
            s.rho = c2(s.red[0], s.red[1]);
            s.bnorm = sqrt(s.red[nred]);
            s.inv_b2 = 1.0 / (s.bnorm * s.bnorm);
            s.alpha_prev = c2(1, 0);
            s.beta_prev = c2(0, 0);
            s.seed = a.seed;
            s.zs = a.z[a.seed];
            s_vs[0] = Vec<R>::make(s.zs);
            s_vs[1] = Vec<R>::make(s.beta_prev);
            s.n = 0;
            s.active = a.K;
            s.replace_on = kMixed && a.replace_every > 0;
            s.n_switch = 0; s.n_replace = 0; s.shift_iters = 0;
        }
        if (tid < M) {
            s.cr_cur[tid] = dense_proj ? c2(s.red[3 + 2 * tid], s.red[4 + 2 * tid])
                                       : (chk(a.dbg, 12, s_cidx[tid], a.n) ? Vec<R>::wide(__ldcg(a.r + s_cidx[tid])) : c2(0, 0));
        }
        __syncthreads();
        if (s.bnorm == 0.0) {                 // b = 0: x = 0 solves every shift
            if (owns) { S.frozen[ko] = 1; S.resid[ko] = 0.0; }
            status = SCOCG_OK;
            done = true;
        }
    }

    // ------------------------------------------------------------ iterations
    int it = s.n;                             // seed iteration, every thread's own copy
    // scalars of the next reductions that depend on the last iteration only,
    // by warp 1 while the other warps apply H
    auto prepare_scalars = [&]() {
        const double2 ir = warp_cdiv(c2(1, 0), s.rho);
        const double2 gr = warp_cdiv(s.beta_prev, s.alpha_prev);
        if (lane == 0) { s.inv_rho = ir; s.t2_ratio = gr; }
    };
    bool skip_a = kResume;                    // the continued solve's first phase A ran before it stopped
    while (!done) {
        SCOCG_TRACE(1);
        SCOCG_MARK(7);
        // ---- phase A: q_n = (z_s - H) r_n + beta_{n-1} q_{n-1}; partial r_n^T q_n
        // (with a deferred phase C of iteration n-1 in warp 0)
        if (!skip_a) {
            AT rq[2] = {};
            // (z_s and beta are read from shared memory where they are used: kept
            // in registers across the apply they would be spilled)

            const bool c_here = pending;           // uniform over the grid
            if (c_here && warp == 0) {
                int act = 0, bad = 0;
                if (own_wide) {
                    shift_update_warp(s_own, nown, s_c, M, a.tol, tol2, act, bad);
                } else {
                    if (owns && !state().frozen[ko]) update_own(act, bad);
                    act = __popc(__ballot_sync(0xffffffffu, act));
                    bad = __any_sync(0xffffffffu, bad);
                }
                if (lane == 0) { s_flag[0] = act; s_flag[1] = bad; }
            }
            if (warp == 1) prepare_scalars();
            // all warps apply H; with a deferred phase C the unit order is
            // rotated so that warps 0 and 1 take the last places in each round
            // and, when the rounds do not come out even, one unit fewer
            const int wi = c_here ? rotated_place(warp) : warp;
            if constexpr (HasTwoPass<Apply>::value) {
                // two passes over the units in two orders, a grid barrier between
                const int64_t n1 = ap.template units1<V>(), n2 = ap.template units2<V>(), step = (int64_t)G * kWarps;
                for (int64_t u = cta + (int64_t)G * wi; u < n1; u += step) ap.pass1(u, lane, s_vs[0], s_vs[1], (const V*)a.r, a.q);
                if (!grid_barrier(a.sync, epoch)) return;
                for (int64_t u = cta + (int64_t)G * wi; u < n2; u += step)
                    ap.pass2(u, lane, (const V*)a.r, a.q,
                             [&](int64_t row, V qn) { acc_bil(rq[0], rq[1], a.r[row], qn); });
            } else {
                for (int lu = wi; lu < sh.nloc; lu += kWarps) {
                    int64_t row;
                    V w;
                    if (ap(sh.unit(lu), lane, s_vs[0], (const V*)a.r, row, w)) {
                        const int t = sh.place(lu, lane);
                        const V qn = vcfma(s_vs[1], sh.get(t, row), w);
                        sh.put(t, row, qn);
                        acc_bil(rq[0], rq[1], a.r[row], qn);
                    }
                }
            }
            ++red_no;
            // (only thread 0's tag is read, and it has set the counts itself)
            const unsigned long long tag = pkt && tid == 0 ? packet_tag(red_no, s_flag[0], s_flag[1]) : red_no;
            block_partials<2>(rq, s_scratch,
                              PartialOut{a.partA + cta, pkt ? a.pk + cta : nullptr, G, tag,
                                         a.debug_inject == 1 && cta == 0 && it == 3}, wi, 2, nwA);
            pending = false;
            if (!pkt && tid == 64) a.partA[2 * G + cta] = pack_counts(s_flag[0], s_flag[1]);
        } else if (warp == 1) {
            prepare_scalars();
        }
        skip_a = false;
        SCOCG_TRACE(2);
        SCOCG_MARK(0);
        if (pkt) {
            if (!packet_sums(a.sync, a.pk, G, 2, red_no, s.red, s_flag + 5)) return;
            SCOCG_TRACE(3);
            SCOCG_MARK(1);
        } else {
            if (!grid_barrier(a.sync, epoch, a.debug_inject == 1 && cta == 0 && it == 3)) return;
            SCOCG_TRACE(3);
            SCOCG_MARK(1);
            if (warp == 2) {
                int act, bad;
                sum_counts(a.partA + 2 * G, G, act, bad);
                if (lane == 0) { s_flag[5] = act; s_flag[6] = bad; }
            }
            grid_sum_vm1(a.partA, 2, s.red, G);
        }
        // warp 0 forms alpha while thread 32 makes the other checks
        if (warp == 0) {
            double2 al = warp_cdiv(s.rho, c2(s.red[0], s.red[1]));
            if (a.debug_inject == 2 && it == 3) al = c2(__longlong_as_double(0x7ff8000000000000ll), 0);
            if (lane == 0) {
                s.alpha = al;
                s_vs[2] = Vec<R>::make(al);
                s_flag[3] = cfinite(al);
            }
        } else if (tid == 32) {
            const double2 rq = c2(s.red[0], s.red[1]);
            const int active = it == 0 ? a.K : s_flag[5];
            int st = kGoOn;
            if (it > 0 && s_flag[6] != 0) st = SCOCG_ERR_BREAKDOWN;
            else if (active == 0) st = SCOCG_OK;
            else if (it >= a.max_iter) st = SCOCG_NOT_CONVERGED;
            else if (cabs2(s.rho) == 0.0 || cabs2(rq) == 0.0 || !cfinite(rq)) st = SCOCG_ERR_BREAKDOWN;
            if (st == kGoOn) s.shift_iters += active;
            s.active = active;
            s_flag[2] = st;
        }
        __syncthreads();
        SCOCG_MARK(6);
        if (s_flag[2] != kGoOn || !s_flag[3]) {
            status = s_flag[2] != kGoOn ? s_flag[2] : (int)SCOCG_ERR_BREAKDOWN;
            break;
        }

        // ---- full-vector mode: this iteration's shift scalars for all shifts
        // (every CTA computes them; t2, pi and its reciprocal bit for bit as phase
        // C does, see pi_next).  The
        // directions are stored as pt^k = p^k / t_k with t_k = 1 / pi^k of the
        // iteration that wrote them, so that pt^k_n = r_n + cp pt^k_{n-1} and
        // x^k += cx pt^k take one complex FMA each:
        // cp = beta^k t_k pi^k_n, cx = alpha^k / pi^k_n.
        if constexpr (kFull) {
            if (a.Xf) {
                double2* s_cp = s_full;
                double2* s_cx = s_full + a.K;
                double2* s_t = s_full + 2 * a.K;
                int* s_list = reinterpret_cast<int*>(s_full + 3 * a.K);   // the unconverged shifts, in any order
                if (tid == 0) s_nact = 0;
                __syncthreads();
                const double2 t2 = shift_t2(s.alpha, s.t2_ratio);   // phase C's, see pi_next
                for (int k = tid; k < a.K; k += kBlock) {
                    if (__ldcg(a.S.frozen + k)) continue;
                    const double2 pp = __ldcg(a.S.pi_prev + k), pc = __ldcg(a.S.pi_cur + k);
                    const double2 ic = __ldcg(a.S.inv_cur + k);
                    const double2 ratio = cmul(pp, ic);
                    const double2 pn = pi_next(s.alpha, t2, __ldcg(a.S.sigma + k), pc, pp);
                    const double2 in = crecip(pn);
                    const double2 t = it == 0 ? c2(1, 0) : s_t[k];
                    s_cp[k] = cmul(cmul(cmul(cmul(ratio, ratio), s.beta_prev), pc), t);
                    s_cx[k] = cmul(cmul(cmul(pc, in), s.alpha), ic);
                    s_t[k] = ic;
                    s_list[atomicAdd(&s_nact, 1)] = k;
                }
                __syncthreads();
                // Warps take 32-row chunks of the CTA's rows; when there are
                // fewer chunks than warps, several warps share a chunk's shifts.
                // Four shifts' vectors are in flight per warp.
                const int nch = (sh.nrow + 31) >> 5, nact = s_nact;
                const int share = nch < kWarps ? kWarps / max(nch, 1) : 1;
                for (int c = warp / share; c < nch; c += kWarps / share) {
                    if (32 * c + lane >= sh.nrow) continue;
                    const int64_t i = sh.row(32 * c + lane);
                    const double2 ri = a.r[i];
                    constexpr int kU = 4;
                    for (int j0 = (warp % share) * kU; j0 < nact; j0 += share * kU) {
                        double2 p[kU], x[kU];
                        int kk[kU];
#pragma unroll
                        for (int u = 0; u < kU; ++u) {
                            kk[u] = j0 + u < nact ? s_list[j0 + u] : -1;
                            if (kk[u] >= 0) { p[u] = a.Pf[(size_t)kk[u] * a.n + i]; x[u] = a.Xf[(size_t)kk[u] * a.n + i]; }
                        }
#pragma unroll
                        for (int u = 0; u < kU; ++u) {
                            if (kk[u] < 0) continue;
                            const double2 pn = vcfma(s_cp[kk[u]], p[u], ri);
                            a.Pf[(size_t)kk[u] * a.n + i] = pn;
                            a.Xf[(size_t)kk[u] * a.n + i] = vcfma(s_cx[kk[u]], pn, x[u]);
                        }
                    }
                }
                __syncthreads();   // the rows' r_n have been read
            }
        }

        // ---- phase B: r_{n+1} = r_n - alpha_n q_n; partials rho, ||r||^2, c^T r
        {
            const V al = s_vs[2];
            const V bp = s_vs[1];
            const bool track_x = kMixed && s.replace_on;
            const bool plain = !track_x;
            AT acc[5] = {};
            if (plain) {
                // one row ahead: the next row's loads are in flight while this
                // row is updated and stored (same rows, same order per thread)
                V ro = vzero<V>(), qo = vzero<V>(), co = vzero<V>();
                if (tid < sh.nrow) {
                    const int64_t i = sh.row(tid);
                    ro = a.r[i]; qo = sh.get(tid, i);
                    if (a.cvec) co = a.cvec[i];
                }
                for (int t = tid; t < sh.nrow; t += kBlock) {
                    V r1 = vzero<V>(), q1 = vzero<V>(), c1 = vzero<V>();
                    if (t + kBlock < sh.nrow) {
                        const int64_t i1 = sh.row(t + kBlock);
                        r1 = a.r[i1]; q1 = sh.get(t + kBlock, i1);
                        if (a.cvec) c1 = a.cvec[i1];
                    }
                    const V rn = r_update(ro, al, qo);
                    a.r[sh.row(t)] = rn;
                    acc_r<R>(acc, rn, a.cvec ? &co : nullptr);
                    ro = r1; qo = q1; co = c1;
                }
            }
            for (int t = tid; !plain && t < sh.nrow; t += kBlock) {
                const int64_t i = sh.row(t);
                const V ro = a.r[i];
                if constexpr (kMixed) {
                    if (track_x) {
                        // p_n = r_n + beta_{n-1} p_{n-1};  x_{n+1} = x_n + alpha_n p_n (compensated sum)
                        const V p = vcfma(bp, a.p_seed[i], ro);
                        a.p_seed[i] = p;
                        const V inc = vcfma(al, p, vzero<V>());
                        const V hi = a.x_hi[i];
                        V lo = a.x_lo[i];
                        const float sx = hi.x + inc.x, bx = sx - hi.x;
                        const float sy = hi.y + inc.y, by = sy - hi.y;
                        lo.x += (hi.x - (sx - bx)) + (inc.x - bx);
                        lo.y += (hi.y - (sy - by)) + (inc.y - by);
                        a.x_hi[i] = make_float2(sx, sy);
                        a.x_lo[i] = lo;
                    }
                }
                const V rn = r_update(ro, al, sh.get(t, i));
                a.r[i] = rn;
                acc_r<R>(acc, rn, a.cvec ? a.cvec + i : nullptr);
            }
            __syncthreads();
            ++red_no;
            finish_r_partials(a, acc, sh, s_scratch,
                              PartialOut{myB, pkt ? a.pk + 2 * G + cta : nullptr, G, red_no, false});
        }
        SCOCG_TRACE(4);
        SCOCG_MARK(2);
        if (pkt) {
            if (!packet_sums(a.sync, a.pk + 2 * G, G, nred, red_no, s.red, s_flag + 5)) return;
        } else {
            if (!grid_barrier(a.sync, epoch)) return;
            SCOCG_TRACE(5);
            SCOCG_MARK(3);
            grid_sum_vm1(a.partB, nred, s.red, G);
        }
        SCOCG_MARK(5);
        // the scalars of this iteration: independent FP64 chains run in three
        // warps at once
        if (tid < M) {
            s.cr_next[tid] = dense_proj ? c2(s.red[3 + 2 * tid], s.red[4 + 2 * tid])
                                        : (chk(a.dbg, 12, s_cidx[tid], a.n) ? Vec<R>::wide(__ldcg(a.r + s_cidx[tid])) : c2(0, 0));
            s_c.cr[tid] = s.cr_cur[tid];
            s.cr_cur[tid] = s.cr_next[tid];
        }
        if (tid == 96) {
            s_c.t2 = shift_t2(s.alpha, s.t2_ratio);
            s_c.alpha = s.alpha; s_c.beta_prev = s.beta_prev; s_c.n = it;
        } else if (tid == 32) {
            s_c.rn_b2 = s.red[2] * s.inv_b2;
            s_flag[4] = a.tol > 0.0 && s_c.rn_b2 <= tol2;    // the seed (pi = 1) has converged
        } else if (warp == 2) {
            const double2 be = warp_quot(c2(s.red[0], s.red[1]), s.rho, s.inv_rho);
            if (lane == 0) {
                s.beta_next = be;
                s_vs[1] = Vec<R>::make(be);
            }
        }
        __syncthreads();

        // ---- phase C: per-shift scalar recurrences for this CTA's shifts
        // (one complex reciprocal per shift; 1/pi^k_n is carried between
        // iterations and residuals are compared squared), here or deferred
        const bool seed_conv = s_flag[4] != 0;
        const bool defer = defer_ok && !seed_conv;
        if (!defer) {
            int my_active = 0, my_bad = 0;
            if (owns && !state().frozen[ko]) update_own(my_active, my_bad);
            const int cnt_active = __syncthreads_count(my_active);
            const int any_bad = __syncthreads_or(my_bad);
            if (tid == 0) { s_flag[0] = cnt_active; s_flag[1] = any_bad; }
        }
        pending = defer;
        ++it;
        // (read next by warp 1, and after further CTA synchronisations by others)
        if (tid == 32) {
            s.beta_prev = s.beta_next;
            s.alpha_prev = s.alpha;
            s.rho_prev = s.rho;
            s.rho = c2(s.red[0], s.red[1]);
            s.n = it;
        }
        if (warp == 1) __syncwarp();
        if (kMixed || seed_conv) __syncthreads();

        // ---- seed switching (Sec. III.C) once the seed has converged
        SCOCG_TRACE(6);
        SCOCG_MARK(4);
        if (seed_conv) {
            SCOCG_TRACE(7);
            // local candidate: the unconverged shift with the smallest |pi| (largest residual)
            double best = INFINITY;
            int arg = 0x7fffffff;
            const ShiftState S = state();
            if (owns && !S.frozen[ko]) { best = -cabs2(S.inv_cur[ko]); arg = k_own; }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
                if (ob < best || (ob == best && oa < arg)) { best = ob; arg = oa; }
            }
            if (lane == 0) { s_min[warp] = best; s_arg[warp] = arg; }
            __syncthreads();
            if (tid == 0) {
                for (int w = 1; w < kWarps; ++w)
                    if (s_min[w] < best || (s_min[w] == best && s_arg[w] < arg)) { best = s_min[w]; arg = s_arg[w]; }
                // the candidate's recurrence values travel with it, so that no CTA
                // reads them after their owner has rebased them below
                double* pc = a.partC + (size_t)cta * kPartC;
                pc[0] = (double)s_flag[0]; pc[1] = best; pc[2] = (double)arg; pc[3] = (double)s_flag[1];
                if (arg < a.K && chk(a.dbg, 10, arg, a.K)) {
                    const int ka = own_sm ? (arg - cta) / G : arg;
                    const double2 pp = S.pi_prev[ka], pq = S.pi_cur[ka], ak = S.alpha_k[ka];
                    pc[4] = pp.x; pc[5] = pp.y; pc[6] = pq.x; pc[7] = pq.y; pc[8] = ak.x; pc[9] = ak.y;
                }
            }
            SCOCG_TRACE(8);
            if (!grid_barrier(a.sync, epoch)) return;
            SCOCG_TRACE(9);
            __shared__ double s_sw[6];
            if (tid == 0) {
                double tot = 0, bad = 0, gbest = INFINITY;
                int garg = 0x7fffffff, gc = -1;
                for (int c = 0; c < G; ++c) {
                    const double* pc = a.partC + (size_t)c * kPartC;
                    tot += __ldcg(pc); bad += __ldcg(pc + 3);
                    const double b2 = __ldcg(pc + 1);
                    const int a2 = (int)__ldcg(pc + 2);
                    if (b2 < gbest || (b2 == gbest && a2 < garg)) { gbest = b2; garg = a2; gc = c; }
                }
                int st = kGoOn;
                if (bad != 0.0) st = SCOCG_ERR_BREAKDOWN;
                else if (tot == 0.0) st = SCOCG_OK;
                else if (!a.allow_switch) st = SCOCG_ERR_BREAKDOWN;
                else if (gc < 0 || !chk(a.dbg, 11, garg, a.K)) st = SCOCG_ERR_BREAKDOWN;
                else
                    for (int j = 0; j < 6; ++j) s_sw[j] = __ldcg(a.partC + (size_t)gc * kPartC + 4 + j);
                s_flag[2] = st;
                s_flag[3] = garg;
            }
            __syncthreads();
            if (s_flag[2] != kGoOn) { status = s_flag[2]; break; }
            const int s2 = s_flag[3];
            SCOCG_TRACE(10 + 100 * s2);
            const double2 pin = c2(s_sw[0], s_sw[1]);        // pi^{s'}_n
            const double2 pin1 = c2(s_sw[2], s_sw[3]);       // pi^{s'}_{n+1}
            const double2 alpha_s2 = c2(s_sw[4], s_sw[5]);   // alpha^{s'}_n
            // r' = r_{n+1} / pi'_{n+1};  q' = (r_n / pi'_n - r_{n+1} / pi'_{n+1}) / alpha'_n,
            // with r_n = r_{n+1} + alpha_n q_n
            const double2 inv1 = cdiv(c2(1, 0), pin1);
            const double2 ca = cdiv(csub(cdiv(c2(1, 0), pin), inv1), alpha_s2);   // times r_{n+1}
            const double2 cb = cdiv(cdiv(s.alpha_prev, pin), alpha_s2);           // times q_n
            const V v_inv1 = Vec<R>::make(inv1), v_ca = Vec<R>::make(ca), v_cb = Vec<R>::make(cb);
            for (int t = tid; t < sh.nrow; t += kBlock) {
                const int64_t i = sh.row(t);
                const V ri = a.r[i], qi = sh.get(t, i);
                sh.put(t, i, vcfma(v_cb, qi, vcfma(v_ca, ri, vzero<V>())));
                a.r[i] = vcfma(v_inv1, ri, vzero<V>());
            }
            SCOCG_TRACE(11);
            if (owns && chk(a.dbg, 13, s2, a.K)) {
                if (k_own == s2) {
                    S.pi_prev[ko] = c2(1, 0); S.pi_cur[ko] = c2(1, 0); S.inv_cur[ko] = c2(1, 0);
                } else {
                    S.pi_prev[ko] = cdiv(S.pi_prev[ko], pin);
                    S.pi_cur[ko] = cdiv(S.pi_cur[ko], pin1);
                    S.inv_cur[ko] = cmul(S.inv_cur[ko], pin1);
                }
                S.sigma[ko] = csub(a.z[k_own], a.z[s2]);
            }
            __syncthreads();
            if (tid == 0) {
                const double2 ratio = cdiv(pin, pin1);
                s.rho = cdiv(s.rho, cmul(pin1, pin1));
                s.beta_prev = cmul(cmul(ratio, ratio), s.beta_prev);
                s.alpha_prev = alpha_s2;
                s.seed = s2;
                s.zs = a.z[s2];
                s_vs[0] = Vec<R>::make(s.zs);
                s_vs[1] = Vec<R>::make(s.beta_prev);
                s.n_switch += 1;
                s.replace_on = 0;        // the new seed's full solution is not tracked
            }
            if (tid < M) s.cr_cur[tid] = cmul(s.cr_cur[tid], inv1);
            SCOCG_TRACE(12);
            if (!grid_barrier(a.sync, epoch)) return;
            SCOCG_TRACE(13);
        }

        // ---- MIXED: FP64 true-residual replacement r_{n+1} = b - (z_s - H) x_{n+1}
        if constexpr (kMixed) {
            if (s.replace_on && it % a.replace_every == 0) {
                for (int t = tid; t < sh.nrow; t += kBlock) {
                    const int64_t i = sh.row(t);
                    const V hi = a.x_hi[i], lo = a.x_lo[i];
                    a.xd[i] = c2((double)hi.x + (double)lo.x, (double)hi.y + (double)lo.y);
                }
                if (!grid_barrier(a.sync, epoch)) return;
                const double2 zs = s.zs;
                for (int lu = warp; lu < sh.nloc; lu += kWarps) {
                    int64_t row;
                    double2 w;
                    if (ap(sh.unit(lu), lane, zs, (const double2*)a.xd, row, w)) {
                        const double2 bi = a.b[row];
                        a.r[row] = Vec<R>::make(c2(bi.x - w.x, bi.y - w.y));
                    }
                }
                if (!grid_barrier(a.sync, epoch)) return;
                r_partials(a, sh, s_scratch, outB);
                if (!grid_barrier(a.sync, epoch)) return;
                grid_sum_vm1(a.partB, nred, s.red, G);
                if (tid == 0) {
                    s.rho = c2(s.red[0], s.red[1]);
                    s.beta_prev = cdiv(s.rho, s.rho_prev);
                    s_vs[1] = Vec<R>::make(s.beta_prev);
                    s.n_replace += 1;
                }
                if (tid < M) {
                    s.cr_cur[tid] = dense_proj ? c2(s.red[3 + 2 * tid], s.red[4 + 2 * tid])
                                               : (chk(a.dbg, 12, s_cidx[tid], a.n) ? Vec<R>::wide(__ldcg(a.r + s_cidx[tid])) : c2(0, 0));
                }
                __syncthreads();
            }
        }
    }

    // ------------------------------------------------------------ outputs
    SCOCG_TRACE(20);
    // what a continuation starts from
    if (sh.on && a.rstate && status == SCOCG_NOT_CONVERGED)
        for (int t = tid; t < sh.nrow; t += kBlock) a.q[sh.row(t)] = sh.q_s[t];
    const ShiftState S = state();
    if (owns) {
        for (int m = 0; m < M; ++m) a.G[(size_t)m * a.K + k_own] = S.X[(size_t)ko * M + m];
        if (own_sm) {
            a.S.pi_prev[k_own] = S.pi_prev[ko]; a.S.pi_cur[k_own] = S.pi_cur[ko]; a.S.inv_cur[k_own] = S.inv_cur[ko];
            a.S.sigma[k_own] = S.sigma[ko]; a.S.alpha_k[k_own] = S.alpha_k[ko];
            for (int m = 0; m < M; ++m) {
                a.S.P[(size_t)k_own * M + m] = S.P[ko * M + m];
                a.S.X[(size_t)k_own * M + m] = S.X[ko * M + m];
            }
            a.S.frozen[k_own] = S.frozen[ko]; a.S.iters[k_own] = S.iters[ko]; a.S.resid[k_own] = S.resid[ko];
        }
    }
    if (cta == 0 && tid == 0) {
        // the stopping apply took the deferred shift update (and rotated its
        // units) when the iteration before had not converged the seed
        if (a.rstate) save_resume_state(a.rstate, s, status, M, defer_ok && s_flag[4] == 0);
        a.stats->iters = s.n;
        a.stats->n_switch = s.n_switch;
        a.stats->seed = s.seed;
        a.stats->n_replace = s.n_replace;
        a.stats->shift_iters = s.shift_iters;
        a.stats->status = status;
        if (status != SCOCG_OK) atomicCAS(a.sync.status, 0, status);
    }
}

// One solve on the whole grid.
// CTAs per SM the persistent kernel is compiled for: two (64 registers a
// thread) hide the latency of the FP32-pipe modes; FP64 solves are bound by
// the FP64 pipe, where one CTA per SM (128 registers, half the CTAs at every
// grid barrier) measured faster.
#ifndef SCOCG_DF_CTAS_PER_SM
#define SCOCG_DF_CTAS_PER_SM 2
#endif
template <typename R> struct MinBlocks { static constexpr int value = 2; };
template <> struct MinBlocks<double> { static constexpr int value = 1; };
template <> struct MinBlocks<DF> { static constexpr int value = SCOCG_DF_CTAS_PER_SM; };

template <typename R, class Apply, bool kResume = false>
__global__ void __launch_bounds__(kBlock, MinBlocks<R>::value) cocg_persistent(SolveArgs<R> a, Apply ap) {
    cocg_body<R, Apply, kResume>(a, ap, (int)gridDim.x, (int)blockIdx.x);
}

// Several independent solves in one launch: CTAs [cta_off[s], cta_off[s+1])
// run system s with its own arguments, barrier counter and partials.
template <typename R, class Apply>
__global__ void __launch_bounds__(kBlock, 2) cocg_multi(const SolveArgs<R>* args, const Apply* aps,
                                                        const int* cta_off, int nsys) {
    int sys = 0;
    while (sys + 1 < nsys && cta_off[sys + 1] <= (int)blockIdx.x) ++sys;
    const SolveArgs<R> a = args[sys];
    const Apply ap = aps[sys];
    cocg_body(a, ap, cta_off[sys + 1] - cta_off[sys], (int)blockIdx.x - cta_off[sys]);
}

}  // namespace scocg
