// Batched ground states of many small impurity-type models, every
// (N_up, N_dn) sector, in one persistent launch (the impurity-solver use case
// that motivates the paper, Sec. I and VI).
//
// Each CTA takes sectors from a device work queue (largest first) and runs a
// whole mixed-precision Lanczos on one sector inside shared memory: FP32
// vectors, dots in two-float sums finished in FP64, FP64 tridiagonal
// eigenpair, a second pass of the recurrence that forms the Ritz vector in
// FP64, and an FP64 H·v for the Rayleigh quotient.  The H·v is the method of
// the paper on the fly: per element unrank (per-spin lists), diagonal, hops
// with the sign from the popcount of the bits between the two sites, and the
// target's rank by combinadics (Fig. algr) -- the per-spin hop lists are
// ranked once per sector and reused by every step.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "gbr_common.h"
#include "tridiag.cuh"

namespace gbr {

constexpr int kBatchThreads = 256;   // default CTA size of the batch solver
constexpr int kBatchMaxL = 10;

struct SectorDesc {
    int model, L, Nup, Ndn;
    int Dup, Ddn;
    int64_t off;       // start-vector offset
};

struct ModelDev {
    int L;
    double h[kBatchMaxL * kBatchMaxL];
    double U[kBatchMaxL];
};

// A team: T consecutive threads of a CTA that solve one sector, with a named
// barrier of their own (a warp needs none).
template <int T> __device__ __forceinline__ void team_sync(int bar) {
    if (T == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(T) : "memory");
}

// Sum over the team in FP64, valid in the first warp.  A dependent FP64 operation
// takes about 150 clocks on this GPU, so each warp sums its own threads (five
// steps) and only the first warp what the others left in red; ends without a
// barrier behind it.
template <int T> __device__ __forceinline__ double team_sum(double v, double *red, int bar) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if (T == 32) return v;
    const int lane = threadIdx.x & 31, w = (threadIdx.x % T) >> 5;
    if (lane == 0) red[w] = v;
    team_sync<T>(bar);
    if (w == 0) {
        v = lane < T / 32 ? red[lane] : 0.0;
#pragma unroll
        for (int o = T / 64; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
        v = __shfl_sync(0xFFFFFFFFu, v, 0);
    }
    return v;
}

__device__ __forceinline__ void ffp(float &hi, float &lo, float a, float b) {
    const float p = a * b;
    const float e = fmaf(a, b, -p);
    const float t = hi + p;
    const float bp = t - hi;
    lo += ((hi - (t - bp)) + (p - bp)) + e;
    hi = t;
}

// k-th (0-based) L-bit pattern with N bits set in increasing order, by
// the greedy combinatorial-number-system unranking (Eq. unrank)
__device__ uint32_t unrank_small(int L, int N, int r, const uint32_t *bin) {
    uint32_t a = 0;
    int c = L - 1;
    for (int k = N; k >= 1; --k) {
        while (c >= 0 && (int)bin[c * (kBatchMaxL + 1) + k] > r) --c;
        a |= 1u << c;
        r -= (int)bin[c * (kBatchMaxL + 1) + k];
        --c;
    }
    return a;
}

// Fig. algr
__device__ __forceinline__ int rank_small(uint32_t a, const uint32_t *bin) {
    int i = 0, k = 1;
    while (a) {
        const int c = __ffs(a) - 1;
        a &= a - 1u;
        i += (int)bin[c * (kBatchMaxL + 1) + k];
        ++k;
    }
    return i;
}

struct SpinLists {
    uint32_t *st;      // states
    uint8_t *cnt;      // hops per state
    uint32_t *ent;     // [state][hm]: offset of the target's element | (2 bond + sign) << 16
    float *d32;        // one-body diagonal (the FP64 one is summed on the fly)
    int hm;            // stride of ent (odd: neighbouring states in different banks)
};

// builds the per-spin state list and hop lists of one spin species; mul: distance
// in the vector between neighbouring ranks of this spin
template <int T>
__device__ void build_spin(int L, int N, int D, int mul, const double *h, const uint8_t *bidx, const uint32_t *bin,
                           const SpinLists &s) {
    for (int r = threadIdx.x % T; r < D; r += T) {
        const uint32_t a = unrank_small(L, N, r, bin);
        s.st[r] = a;
        double d = 0.0;
        int k = 0;
        for (int p = 0; p < L; ++p) {
            if (!((a >> p) & 1u)) continue;
            d += h[p * L + p];
            for (int q = 0; q < L; ++q) {
                if (q == p || ((a >> q) & 1u) || h[p * L + q] == 0.0) continue;
                const uint32_t b = a ^ ((1u << p) | (1u << q));
                const int lo = min(p, q), hi = max(p, q);
                const uint32_t between = ((1u << hi) - 1u) & ~((1u << (lo + 1)) - 1u);
                const uint32_t sg = (uint32_t)(__popc(a & between) & 1);
                if (k < s.hm) s.ent[r * s.hm + k] = (uint32_t)(rank_small(b, bin) * mul) | ((2u * bidx[p * L + q] + sg) << 16);
                ++k;
            }
        }
        s.cnt[r] = (uint8_t)min(k, s.hm);
        s.d32[r] = (float)d;
    }
}

// sum of h_pp over the occupied sites of one spin pattern (ascending p)
__device__ __forceinline__ double diag64(uint32_t a, const double *h, int L) {
    double d = 0.0;
    while (a) {
        const int p = __ffs(a) - 1;
        a &= a - 1u;
        d += h[p * L + p];
    }
    return d;
}

// (H x)_i of element i = (ru, rd), x in shared or global memory (hs: the L x L
// one-body matrix, for the FP64 diagonal; umask: sites with U != 0; cf: the bonds'
// coefficients with both signs).  An entry holds the target's element and the
// signed coefficient's place, so that a hop is three loads and one FMA.
template <typename T>
__device__ __forceinline__ T hv_small(const SectorDesc &sd, const SpinLists &up, const SpinLists &dn, const T *cf,
                                      const T *U, uint32_t umask, const double *hs, const T *x, int ru, int rd) {
    const uint32_t au = up.st[ru], ad = dn.st[rd];
    T dg = (sizeof(T) == 8) ? (T)(diag64(au, hs, sd.L) + diag64(ad, hs, sd.L)) : (T)(up.d32[ru] + dn.d32[rd]);
    uint32_t both = au & ad & umask;
    while (both) {
        dg += U[__ffs(both) - 1];
        both &= both - 1u;
    }
    const T *row = x + ru * sd.Ddn, *col = x + rd;
    T acc = dg * row[rd];
    const uint32_t *e = up.ent + ru * up.hm;
    int n = up.cnt[ru];
    for (int k = 0; k < n; ++k) acc += cf[e[k] >> 16] * col[e[k] & 0xFFFFu];
    e = dn.ent + rd * dn.hm;
    n = dn.cnt[rd];
    for (int k = 0; k < n; ++k) acc += cf[e[k] >> 16] * row[e[k] & 0xFFFFu];
    return acc;
}

struct TeamVars {
    double lam_hint, gap_hint, inv_n0;   // warm start of the convergence test's eigenvalue search; 1 / |start|
    float ak, bk, inv;                   // alpha_k, beta_{k+1} and 1 / beta_{k+1} of the step
    int cur, conv, end, kdone;
    uint32_t umask;                      // sites with U != 0
};

// Longest recurrence whose solver arrays (12 KiB) go to shared memory: the
// solver's chains read one entry a step, which from L2 costs several times the
// arithmetic of the step.
constexpr int kBatchTriSmem = 512;

// A team's shared memory for one sector (host and device lay it out alike).
struct TeamLay {
    int v, vp, w, st_up, st_dn, cnt_up, cnt_dn, ent_up, ent_dn, d_up, d_dn, alpha, beta, svec, scratch, hs, cf64, cf32, U64,
        U32, bidx, bytes;
    int hm_up, hm_dn;
};
__host__ __device__ inline TeamLay team_lay(const SectorDesc &sd, int T, int hmax, int nb, int iters, int tri_smem) {
    TeamLay l;
    int at = (int)((sizeof(TeamVars) + 15) & ~(size_t)15);
    auto take = [&](int bytes) { const int q = at; at += (bytes + 15) & ~15; return q; };
    const int D = sd.Dup * sd.Ddn, K = iters < D ? iters : D, L = sd.L;
    auto hops = [&](int N) { const int m = N * (L - N); return (m < hmax ? m : hmax) | 1; };
    l.hm_up = hops(sd.Nup);
    l.hm_dn = hops(sd.Ndn);
    l.v = take(D * 4);
    l.vp = take(D * 4);
    l.w = take(D * 4);
    l.st_up = take(sd.Dup * 4);
    l.st_dn = take(sd.Ddn * 4);
    l.cnt_up = take(sd.Dup);
    l.cnt_dn = take(sd.Ddn);
    l.ent_up = take(sd.Dup * l.hm_up * 4);
    l.ent_dn = take(sd.Ddn * l.hm_dn * 4);
    l.d_up = take(sd.Dup * 4);
    l.d_dn = take(sd.Ddn * 4);
    l.alpha = take((K + 2) * 8);
    l.beta = take((K + 2) * 8);
    l.svec = take((K + 2) * 8);
    // one double per warp for the sums and, for short recurrences, the solver's
    // 3 (K + 2) doubles in the same place: both are the first warp's between barriers
    const int red = T / 32 * 8, tri = tri_smem ? (K + 2) * 24 : 0;
    l.scratch = take(red > tri ? red : tri);
    l.hs = take(L * L * 8);
    l.cf64 = take(2 * nb * 8);
    l.cf32 = take(2 * nb * 4);
    l.U64 = take(L * 8);
    l.U32 = take(L * 4);
    l.bidx = take(L * L);
    l.bytes = at;
    return l;
}

// Size classes of the sectors: 0 = the whole CTA (as many threads as it has),
// then teams of 128, 64 and 32 threads, several in a CTA.
constexpr int kBatchClasses = 4;
struct BatchLay {
    int hmax, nb, iters, tri_smem, bytes;   // bytes: shared memory of a CTA
    int beg[kBatchClasses + 1];             // sectors of each class in the sorted list
    int64_t slot;                           // doubles of global scratch per CTA
};
// doubles of global scratch of a sector: x, the restart's source (D each), the solver's 3 (K + 2);
// an even number, so that every team's solver work starts on a 16-byte boundary (the second
// run keeps its coefficients there in packs)
__host__ __device__ inline int64_t team_slot(int64_t D, int iters) {
    const int64_t K = iters < D ? iters : D;
    return (2 * D + 3 * (K + 2) + 1) & ~(int64_t)1;
}

template <int T>
__device__ void solve_sector(const SectorDesc sd, const ModelDev &m, const double *__restrict__ start, const BatchLay &bl,
                             unsigned char *smem, double *xg, int bar, const uint32_t *bin, double *outE, int *outK) {
    const TeamLay l = team_lay(sd, T, bl.hmax, bl.nb, bl.iters, bl.tri_smem);
    const int tid = threadIdx.x % T;
    TeamVars &tv = *reinterpret_cast<TeamVars *>(smem);
    float *v = (float *)(smem + l.v), *vp = (float *)(smem + l.vp);
    float *const w = (float *)(smem + l.w);
    const SpinLists up{(uint32_t *)(smem + l.st_up), smem + l.cnt_up, (uint32_t *)(smem + l.ent_up), (float *)(smem + l.d_up), l.hm_up};
    const SpinLists dn{(uint32_t *)(smem + l.st_dn), smem + l.cnt_dn, (uint32_t *)(smem + l.ent_dn), (float *)(smem + l.d_dn), l.hm_dn};
    double *alpha = (double *)(smem + l.alpha), *beta = (double *)(smem + l.beta), *svec = (double *)(smem + l.svec);
    double *red = (double *)(smem + l.scratch);
    double *hs = (double *)(smem + l.hs), *cf64 = (double *)(smem + l.cf64), *U64 = (double *)(smem + l.U64);
    float *cf32 = (float *)(smem + l.cf32), *U32 = (float *)(smem + l.U32);
    uint8_t *bidx = smem + l.bidx;
    const int L = sd.L, D = sd.Dup * sd.Ddn, K = min(bl.iters, D);
    double *x = xg, *hx = xg + D;
    double *work = bl.tri_smem ? red : xg + 2 * (int64_t)D;
    for (int i = tid; i < L * L; i += T) hs[i] = m.h[i];
    for (int i = tid; i < L; i += T) {
        U64[i] = m.U[i];
        U32[i] = (float)m.U[i];
    }
    team_sync<T>(bar);
    if (tid == 0) {
        uint32_t um = 0;
        for (int a = 0; a < L; ++a) um |= U64[a] != 0.0 ? 1u << a : 0u;
        tv.umask = um;
        int nb = 0;
        for (int a = 0; a < L; ++a)
            for (int b = 0; b < L; ++b) {
                const double c = hs[a * L + b];
                if (a == b || c == 0.0) continue;
                bidx[a * L + b] = (uint8_t)nb;
                cf64[2 * nb] = c;
                cf64[2 * nb + 1] = -c;
                cf32[2 * nb] = (float)c;
                cf32[2 * nb + 1] = -(float)c;
                ++nb;
            }
    }
    team_sync<T>(bar);
    build_spin<T>(L, sd.Nup, sd.Dup, sd.Ddn, hs, bidx, bin, up);
    build_spin<T>(L, sd.Ndn, sd.Ddn, 1, hs, bidx, bin, dn);
    // Restarted Lanczos: each cycle stops as soon as the lowest Ritz pair
    // of T has converged to FP32 level (residual estimate
    // beta_{k+1} |s_k| <= 1e-6 max(|alpha|, beta), tested after 4 steps and
    // then at half the distance the decrease so far predicts (4 to 16
    // steps), with a warm-started eigenvalue search and the last
    // eigenvector component alone, and at the last step of the cycle), which keeps the FP32
    // recurrence from running on after convergence and spoiling the Ritz
    // vector; a cycle that ends unconverged restarts from its Ritz vector
    // (at most three cycles).  Each cycle runs the recurrence twice: once
    // for the scalars, once more (bit identical) to accumulate the Ritz
    // vector x in FP64.
    //
    // this thread's elements i = tid + j T as (ru, rd)
    const int dru = T / sd.Ddn, drd = T - dru * sd.Ddn;
    const int ru0 = tid / sd.Ddn, rd0 = tid - ru0 * sd.Ddn;
    auto next = [&](int &ru, int &rd) {
        ru += dru;
        rd += drd;
        if (rd >= sd.Ddn) {
            rd -= sd.Ddn;
            ++ru;
        }
    };
    for (int cyc = 0; cyc < 3; ++cyc) {
        if (cyc > 0)
            for (int i = tid; i < D; i += T) hx[i] = x[i];
        team_sync<T>(bar);
        auto source = [&](int i) { return (float)(cyc == 0 ? start[sd.off + i] : hx[i]); };
        const uint32_t umask = tv.umask;
        float fh = 0.f, fl = 0.f;
        for (int i = tid; i < D; i += T) {
            const float f = source(i);
            ffp(fh, fl, f, f);
        }
        const double n2 = team_sum<T>((double)fh + (double)fl, red, bar);
        if (tid == 0) {
            tv.inv_n0 = 1.0 / sqrt(n2);
            tv.conv = 0;
            tv.end = 0;
            tv.lam_hint = 0.0;
            tv.gap_hint = 0.0;
        }
        team_sync<T>(bar);
        // the first run: scalars
        for (int i = tid; i < D; i += T) v[i] = (float)((double)source(i) * tv.inv_n0);
        team_sync<T>(bar);
        // the first warp's: step of the next test, step and residual of the last one
        int next_check = 4, k_last = 0;
        float r_last = 0.f;
        double scale = 0.0;
        for (int k = 0; k < K; ++k) {
            const float bk = tv.bk;   // beta_k (k > 0)
            float ah = 0.f, al = 0.f;
            for (int i = tid, ru = ru0, rd = rd0; i < D; i += T, next(ru, rd)) {
                float wi = hv_small<float>(sd, up, dn, cf32, U32, umask, hs, v, ru, rd);
                if (k) wi = __fmaf_rn(-bk, vp[i], wi);
                w[i] = wi;
                ffp(ah, al, wi, v[i]);
            }
            const double a = team_sum<T>((double)ah + (double)al, red, bar);
            if (tid == 0) {
                alpha[k] = a;
                tv.ak = (float)a;
            }
            scale = fmax(scale, fabs(a));
            team_sync<T>(bar);
            const float ak = tv.ak;
            float bh = 0.f, blo = 0.f;
            for (int i = tid; i < D; i += T) {
                const float wi = __fmaf_rn(-ak, v[i], w[i]);
                w[i] = wi;
                ffp(bh, blo, wi, wi);
            }
            const double b2 = team_sum<T>((double)bh + (double)blo, red, bar);
            if (tid < 32) {
                const double b = sqrt(fmax(b2, 0.0));
                const int kd = k + 1;
                scale = fmax(scale, b);
                bool conv = b <= 1e-13 * scale;
                if (tid == 0) {
                    beta[kd] = b;
                    tv.bk = (float)b;
                    tv.inv = 1.0f / (float)b;   // FP32: the FP64 divide is slow here
                }
                __syncwarp();
                if (!conv && kd == next_check && kd < K) {
                    // residual estimate from the last eigenvector component alone
                    const Tri t = tri_stage(alpha, beta, kd, scale, work);
                    const double lam = tri_lowest_warm(t, &tv.lam_hint, &tv.gap_hint);
                    // relative to the scale, which the prediction needs in FP32 only
                    const double r = b * tri_last_component(t, lam);
                    const float rr = (float)(r * tri_unit(scale)), thr = (float)(1e-6 * (scale * tri_unit(scale)));
                    if (r <= 1e-6 * scale) {
                        conv = true;
                    } else {
                        // next test at half the distance the geometric decrease since
                        // the last test predicts, 4 to 16 steps ahead
                        int gap = 4;
                        if (r_last > 0.f && rr < r_last) {
                            const float per_step = logf(rr / r_last) / (float)(kd - k_last);
                            const float steps = logf(thr / rr) / per_step;
                            gap = 4 * max(1, min(4, (int)(0.5f * steps / 4.0f)));
                        }
                        next_check = kd + gap;
                        r_last = rr;
                        k_last = kd;
                    }
                }
                if (conv || kd >= K) {
                    // the Ritz pair of the final T for the second run (the vectors'
                    // memory is free: it takes the recurrence from below)
                    const Tri t = tri_stage(alpha, beta, kd, scale, work);
                    const double lam = tri_lowest_warm(t, &tv.lam_hint, &tv.gap_hint);
                    if (!tri_vector_twisted(t, beta, lam, svec, (double *)(smem + l.v)) && tid == 0)
                        tridiag_vector_thread(alpha, beta, kd, lam / t.unit, svec, work);
                    if (tid == 0) {
                        if (conv || b * fabs(svec[kd - 1]) <= 1e-6 * scale) tv.conv = 1;
                        tv.kdone = kd;
                        tv.end = 1;
                    }
                }
            }
            team_sync<T>(bar);
            if (tv.end) break;
            // v_{k+1} takes the place of v_{k-1}
            const float inv = tv.inv;
            for (int i = tid; i < D; i += T) vp[i] = w[i] * inv;
            float *t = vp;
            vp = v;
            v = t;
            team_sync<T>(bar);
        }
        // the second run, one pass a step: the same vectors with the stored
        // scalars, summed into x (the solver's arrays are free: they hold the
        // scalars in FP32, as the first run used them)
        float4 *sf = reinterpret_cast<float4 *>(work);
        const int steps = tv.kdone;
        for (int k = tid; k + 1 < steps; k += T)
            sf[k] = make_float4(k ? (float)beta[k] : 0.f, (float)alpha[k], 1.0f / (float)beta[k + 1], 0.f);
        for (int i = tid; i < D; i += T) {
            const float f = (float)((double)source(i) * tv.inv_n0);
            v[i] = f;
            x[i] = svec[0] * (double)f;
        }
        team_sync<T>(bar);
        for (int k = 0; k + 1 < steps; ++k) {
            const float4 c = sf[k];
            const double sk = svec[k + 1];
            for (int i = tid, ru = ru0, rd = rd0; i < D; i += T, next(ru, rd)) {
                const double xi = x[i];
                float wi = hv_small<float>(sd, up, dn, cf32, U32, umask, hs, v, ru, rd);
                if (k) wi = __fmaf_rn(-c.x, vp[i], wi);
                wi = __fmaf_rn(-c.y, v[i], wi) * c.z;
                vp[i] = wi;   // read by this thread alone
                x[i] = fma(sk, (double)wi, xi);
            }
            float *t = vp;
            vp = v;
            v = t;
            team_sync<T>(bar);
        }
        if (tv.conv) break;
    }
    team_sync<T>(bar);
    // FP64 Rayleigh quotient of the Ritz vector
    double xhx = 0.0, xx = 0.0;
    for (int i = tid, ru = ru0, rd = rd0; i < D; i += T, next(ru, rd)) {
        const double xi = x[i];
        xhx = fma(xi, hv_small<double>(sd, up, dn, cf64, U64, tv.umask, hs, x, ru, rd), xhx);
        xx = fma(xi, xi, xx);
    }
    const double num = team_sum<T>(xhx, red, bar);
    team_sync<T>(bar);
    const double den = team_sum<T>(xx, red, bar);
    if (tid == 0) {
        *outE = num / den;
        *outK = tv.kdone;
    }
    team_sync<T>(bar);
}

template <int NT, int T>
__device__ void batch_class(int cls, const SectorDesc *__restrict__ secs, const ModelDev *__restrict__ models,
                            const double *__restrict__ start, const BatchLay &bl, unsigned char *smem, double *xg,
                            int *counter, const uint32_t *bin, double *outE, int *outK) {
    if (bl.beg[cls] == bl.beg[cls + 1]) return;
    constexpr int teams = NT / T;
    const int team = threadIdx.x / T, bar = 1 + team;
    smem += team * (bl.bytes / teams & ~15);
    xg += team * (bl.slot / teams & ~(int64_t)1);   // at least an (even) team_slot
    TeamVars &tv = *reinterpret_cast<TeamVars *>(smem);
    while (true) {
        if (threadIdx.x % T == 0) tv.cur = bl.beg[cls] + atomicAdd(counter + cls, 1);
        team_sync<T>(bar);
        const int si = tv.cur;
        if (si >= bl.beg[cls + 1]) break;
        const SectorDesc sd = secs[si];
        solve_sector<T>(sd, models[sd.model], start, bl, smem, xg, bar, bin, outE + si, outK + si);
    }
    __syncthreads();   // the next class lays the shared memory out anew
}

// One persistent launch over all sectors, largest class first, each class's
// sectors from a device work queue.
//
// A sector is a long chain of short steps (FP64 sums and tridiagonal searches
// whose dependent operations take about 150 clocks each, barriers, and vector
// loops that a small sector does not fill the CTA with), so small ones go to
// teams: several sectors side by side in a CTA, in the shared memory that a whole
// CTA's sector has.  256 impurity models (16,620 sectors of up to 4,900 states):
// 12.3 ms in the kernel at 256 threads, against 19.3 ms with one sector a CTA; 128
// threads 16.1, 512 threads 22.0 ms.  Three models (192 sectors, no queue): 1.6 ms,
// the largest sector's own time.
//
// xg: per-CTA scratch of bl.slot doubles for the FP64 Ritz vector, the restart's
// source and, for long recurrences, the tridiagonal solver's work (global memory; each CTA
// reuses its own slot, which stays in L2), so that the shared memory holds only the FP32
// recurrence and three CTAs fit on an SM.
//
// NT threads per CTA (128, 256 or 512; the autotuner's choice), at most
// 64 K / (NT x 3 x 256 / NT) registers a thread so that three CTAs fit on an SM
// at 256 and the register budget per SM stays the same at the other sizes.
template <int NT>
__global__ void __launch_bounds__(NT, (NT >= 512 ? 1 : 768 / NT)) k_batch(const SectorDesc *__restrict__ secs,
                                                         const ModelDev *__restrict__ models,
                                                         const double *__restrict__ start, const BatchLay bl,
                                                         int *counter, double *__restrict__ outE, int *__restrict__ outK,
                                                         double *__restrict__ xg) {
    extern __shared__ __align__(16) unsigned char smr[];
    __shared__ uint32_t bin[(kBatchMaxL + 1) * (kBatchMaxL + 1)];
    for (int i = threadIdx.x; i < (kBatchMaxL + 1) * (kBatchMaxL + 1); i += NT) {
        const int n = i / (kBatchMaxL + 1), k = i % (kBatchMaxL + 1);
        // C(n, k) by the multiplicative formula (small n)
        uint32_t c = (k > n) ? 0u : 1u;
        for (int j = 1; j <= k && k <= n; ++j) c = c * (uint32_t)(n - k + j) / (uint32_t)j;
        bin[i] = c;
    }
    __syncthreads();
    xg += (size_t)blockIdx.x * bl.slot;
    batch_class<NT, NT>(0, secs, models, start, bl, smr, xg, counter, bin, outE, outK);
    if (NT > 128) batch_class<NT, NT == 128 ? 64 : 128>(1, secs, models, start, bl, smr, xg, counter, bin, outE, outK);
    batch_class<NT, 64>(2, secs, models, start, bl, smr, xg, counter, bin, outE, outK);
    batch_class<NT, 32>(3, secs, models, start, bl, smr, xg, counter, bin, outE, outK);
}

static int sector_list(int n_models, const gbr_model_desc *models, std::vector<SectorDesc> &secs, int64_t *n_states) {
    secs.clear();
    int64_t off = 0;
    for (int m = 0; m < n_models; ++m) {
        const int L = models[m].L;
        if (L < 1 || L > kBatchMaxL) return set_error(GBR_EINVAL, "model %d: L=%d out of range 1..%d", m, L, kBatchMaxL);
        if (!models[m].h) return set_error(GBR_EINVAL, "model %d: h is NULL", m);
        for (int nu = 0; nu <= L; ++nu)
            for (int nd = 0; nd <= L; ++nd) {
                SectorDesc s;
                s.model = m; s.L = L; s.Nup = nu; s.Ndn = nd;
                s.Dup = (int)binom(L, nu);
                s.Ddn = (int)binom(L, nd);
                s.off = off;
                off += (int64_t)s.Dup * s.Ddn;
                secs.push_back(s);
            }
    }
    if (n_states) *n_states = off;
    return GBR_OK;
}

}  // namespace gbr

using namespace gbr;

extern "C" int gbr_batch_layout(int n_models, const gbr_model_desc *models, int64_t *n_sectors, int64_t *n_states) {
    clear_error();
    if (n_models < 0 || (n_models > 0 && !models)) return set_error(GBR_EINVAL, "bad model list");
    std::vector<SectorDesc> secs;
    int rc = sector_list(n_models, models, secs, n_states);
    if (rc) return rc;
    if (n_sectors) *n_sectors = (int64_t)secs.size();
    return GBR_OK;
}

namespace gbr {
// CTA size and CTAs per SM of the batch solver (process-wide; 0 = as many as
// fit), set by gbr_batch_set_shape or gbr_batch_tune
static int g_batch_threads = kBatchThreads, g_batch_per_sm = 0;

template <int NT>
static int batch_grid(int grid_req_per_sm, int nsec, const BatchLay &bl, int *grid) {
    auto kern = k_batch<NT>;
    GBR_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bl.bytes));
    int per_sm = 0;
    GBR_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, (size_t)bl.bytes));
    per_sm = std::max(1, per_sm);
    if (grid_req_per_sm > 0) per_sm = std::min(per_sm, grid_req_per_sm);
    *grid = std::max(1, std::min<int>(nsec, sm_count() * per_sm));
    return GBR_OK;
}

// Class of every sector and the CTA's shared memory: what the largest sector needs
// for the whole CTA; a smaller one goes to the smallest team whose size suits it
// and whose share of that memory holds it.
// The limits keep a team's vector loops (sixteen elements a thread at most) at its FP64
// chains' length: 256 impurity models 12.9 ms in the call with these, 13.6 with 1,200, 400
// and 64, 12.6 with 2,000, 800 and 128, where 90 models then take 5.6 instead of 5.2 ms.
constexpr int kBatchTeam[kBatchClasses] = {0, 128, 64, 32};
constexpr int kBatchTeamMax[kBatchClasses] = {0, 1600, 500, 100};   // states
static void batch_plan(const std::vector<SectorDesc> &secs, int threads, BatchLay *bl, std::vector<int> *cls) {
    bl->bytes = 0;
    for (const SectorDesc &s : secs) bl->bytes = std::max(bl->bytes, team_lay(s, threads, bl->hmax, bl->nb, bl->iters, bl->tri_smem).bytes);
    cls->assign(secs.size(), 0);
    bl->slot = 0;
    for (size_t i = 0; i < secs.size(); ++i) {
        const SectorDesc &s = secs[i];
        const int D = s.Dup * s.Ddn;
        int teams = 1;
        for (int c = kBatchClasses - 1; c >= 1; --c) {
            const int T = kBatchTeam[c], n = threads / T;
            if (T >= threads || D > kBatchTeamMax[c]) continue;
            if (team_lay(s, T, bl->hmax, bl->nb, bl->iters, bl->tri_smem).bytes > (bl->bytes / n & ~15)) continue;
            (*cls)[i] = c;
            teams = n;
            break;
        }
        bl->slot = std::max(bl->slot, teams * team_slot(D, bl->iters));
    }
}

static int batch_run(int n_models, const gbr_model_desc *models, const double *d_start, int iters, double *h_E0,
                     int *h_arg, double *h_sector_E, cudaStream_t st, int threads, int per_sm_req, float *ms_out) {
    if (n_models < 1 || !models) return set_error(GBR_EINVAL, "bad model list");
    if (!d_start || !h_E0) return set_error(GBR_EINVAL, "NULL argument");
    if (iters < 1 || iters > 4096) return set_error(GBR_EINVAL, "iters=%d out of range 1..4096", iters);
    std::vector<SectorDesc> secs;
    int64_t n_states = 0;
    int rc = sector_list(n_models, models, secs, &n_states);
    if (rc) return rc;
    std::vector<ModelDev> md((size_t)n_models);
    int maxD = 1, hmax = 1, nbmax = 1;
    for (int m = 0; m < n_models; ++m) {
        const int L = models[m].L;
        memset(&md[(size_t)m], 0, sizeof(ModelDev));
        md[(size_t)m].L = L;
        for (int p = 0; p < L; ++p) {
            for (int q = 0; q < L; ++q) {
                const double a = models[m].h[p * L + q];
                if (!std::isfinite(a) || a != models[m].h[q * L + p])
                    return set_error(GBR_EINVAL, "model %d: h not finite and symmetric at (%d,%d)", m, p, q);
                md[(size_t)m].h[p * L + q] = a;
            }
            md[(size_t)m].U[p] = models[m].U ? models[m].U[p] : 0.0;
        }
        int nb = 0;
        for (int p = 0; p < L; ++p)
            for (int q = 0; q < L; ++q)
                if (p != q && models[m].h[p * L + q] != 0.0) ++nb;
        if (nb > 0x7FFF) return set_error(GBR_EINVAL, "too many bonds");
        // largest hop count of any per-spin state: N (L - N) bounds it, and so do the
        // bonds, each of which lets at most one of its ends hop
        for (int N = 0; N <= L; ++N) hmax = std::max(hmax, std::min(N * (L - N), nb / 2));
        nbmax = std::max(nbmax, nb);
    }
    for (const SectorDesc &s : secs) maxD = std::max(maxD, s.Dup * s.Ddn);
    const int K = std::min(iters, maxD);
    BatchLay bl;
    bl.hmax = hmax;
    bl.nb = nbmax;
    bl.iters = K;
    int dev = 0, optin = 0;
    GBR_CUDA_TRY(cudaGetDevice(&dev));
    GBR_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    std::vector<int> cls;
    // the solver's arrays in shared memory if they fit there
    for (bl.tri_smem = K <= kBatchTriSmem ? 1 : 0;; bl.tri_smem = 0) {
        batch_plan(secs, threads, &bl, &cls);
        if (bl.bytes + 1024 <= optin) break;
        if (!bl.tri_smem) return set_error(GBR_EINVAL, "largest sector needs %d bytes of shared memory (limit %d)", bl.bytes, optin);
    }
    // by class, the largest sectors first
    std::vector<SectorDesc> order(secs);
    std::vector<int> idx(secs.size());
    for (size_t i = 0; i < idx.size(); ++i) idx[i] = (int)i;
    std::stable_sort(idx.begin(), idx.end(), [&](int a, int b) {
        if (cls[(size_t)a] != cls[(size_t)b]) return cls[(size_t)a] < cls[(size_t)b];
        return (int64_t)secs[(size_t)a].Dup * secs[(size_t)a].Ddn > (int64_t)secs[(size_t)b].Dup * secs[(size_t)b].Ddn;
    });
    for (int c = 0; c <= kBatchClasses; ++c)
        bl.beg[c] = (int)std::count_if(cls.begin(), cls.end(), [&](int k) { return k < c; });
    for (size_t i = 0; i < idx.size(); ++i) order[i] = secs[(size_t)idx[i]];
    const int nsec = (int)order.size();
    int grid = 1;
    rc = threads == 128 ? batch_grid<128>(per_sm_req, nsec, bl, &grid)
                        : (threads == 512 ? batch_grid<512>(per_sm_req, nsec, bl, &grid) : batch_grid<256>(per_sm_req, nsec, bl, &grid));
    if (rc) return rc;
    // one allocation: queue counters, sectors and models (copied together), results, scratch
    auto r256 = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t at_sec = 256, at_mod = at_sec + r256(order.size() * sizeof(SectorDesc)),
                 at_E = at_mod + r256(md.size() * sizeof(ModelDev)), at_K = at_E + r256(order.size() * 8),
                 at_x = at_K + r256(order.size() * 4);
    DevBuf dev_buf;
    if ((rc = dev_buf.alloc(at_x + (size_t)grid * (size_t)bl.slot * 8))) return rc;
    std::vector<unsigned char> blob(at_E, 0);
    memcpy(blob.data() + at_sec, order.data(), order.size() * sizeof(SectorDesc));
    memcpy(blob.data() + at_mod, md.data(), md.size() * sizeof(ModelDev));
    unsigned char *dp = dev_buf.as<unsigned char>();
    GBR_CUDA_TRY(cudaMemcpyAsync(dp, blob.data(), blob.size(), cudaMemcpyHostToDevice, st));
    int *ctr = reinterpret_cast<int *>(dp), *dK = reinterpret_cast<int *>(dp + at_K);
    const SectorDesc *dsec = reinterpret_cast<const SectorDesc *>(dp + at_sec);
    const ModelDev *dmod = reinterpret_cast<const ModelDev *>(dp + at_mod);
    double *dE = reinterpret_cast<double *>(dp + at_E), *dx = reinterpret_cast<double *>(dp + at_x);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (ms_out) {
        GBR_CUDA_TRY(cudaEventCreate(&e0));
        GBR_CUDA_TRY(cudaEventCreate(&e1));
        cudaEventRecord(e0, st);
    }
    if (threads == 128) k_batch<128><<<grid, 128, (size_t)bl.bytes, st>>>(dsec, dmod, d_start, bl, ctr, dE, dK, dx);
    else if (threads == 512) k_batch<512><<<grid, 512, (size_t)bl.bytes, st>>>(dsec, dmod, d_start, bl, ctr, dE, dK, dx);
    else k_batch<256><<<grid, 256, (size_t)bl.bytes, st>>>(dsec, dmod, d_start, bl, ctr, dE, dK, dx);
    GBR_LAUNCH_CHECK();
    count_launches(1);
    if (ms_out) {
        cudaEventRecord(e1, st);
        GBR_CUDA_TRY(cudaEventSynchronize(e1));
        cudaEventElapsedTime(ms_out, e0, e1);
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
    }
    std::vector<double> E(order.size());
    GBR_CUDA_TRY(cudaMemcpyAsync(E.data(), dE, E.size() * 8, cudaMemcpyDeviceToHost, st));
    GBR_CUDA_TRY(cudaStreamSynchronize(st));
    std::vector<double> Es(secs.size());
    for (size_t i = 0; i < idx.size(); ++i) Es[(size_t)idx[i]] = E[i];
    if (h_sector_E) memcpy(h_sector_E, Es.data(), Es.size() * 8);
    // per model minimum with the tie rule: within 1e-10 |E| prefer lower N, then lower N_up
    size_t s0 = 0;
    for (int m = 0; m < n_models; ++m) {
        const int L = models[m].L;
        const size_t ns = (size_t)(L + 1) * (L + 1);
        double best = Es[s0];
        for (size_t j = 0; j < ns; ++j) best = std::min(best, Es[s0 + j]);
        const double tol = 1e-10 * std::max(1.0, std::fabs(best));
        int bu = -1, bd = -1;
        for (int N = 0; N <= 2 * L && bu < 0; ++N)
            for (int nu = 0; nu <= L; ++nu) {
                const int nd = N - nu;
                if (nd < 0 || nd > L) continue;
                if (Es[s0 + (size_t)(nu * (L + 1) + nd)] <= best + tol) { bu = nu; bd = nd; break; }
            }
        h_E0[m] = best;
        if (h_arg) { h_arg[2 * m] = bu; h_arg[2 * m + 1] = bd; }
        s0 += ns;
    }
    return GBR_OK;
}
}  // namespace gbr

extern "C" int gbr_batch_solve(int n_models, const gbr_model_desc *models, const double *d_start, int iters,
                               double *h_E0, int *h_arg, double *h_sector_E, void *stream) {
    clear_error();
    return batch_run(n_models, models, d_start, iters, h_E0, h_arg, h_sector_E, (cudaStream_t)stream,
                     g_batch_threads, g_batch_per_sm, nullptr);
}

extern "C" int gbr_batch_set_shape(int threads, int ctas_per_sm) {
    clear_error();
    if (threads != 128 && threads != 256 && threads != 512)
        return set_error(GBR_EINVAL, "threads %d must be 128, 256 or 512", threads);
    if (ctas_per_sm < 0 || ctas_per_sm > 32) return set_error(GBR_EINVAL, "ctas_per_sm %d out of range 0..32", ctas_per_sm);
    g_batch_threads = threads;
    g_batch_per_sm = ctas_per_sm;
    return GBR_OK;
}

extern "C" int gbr_batch_get_shape(int *threads, int *ctas_per_sm) {
    clear_error();
    if (!threads || !ctas_per_sm) return set_error(GBR_EINVAL, "NULL argument");
    *threads = g_batch_threads;
    *ctas_per_sm = g_batch_per_sm;
    return GBR_OK;
}

extern "C" int gbr_batch_tune(int n_models, const gbr_model_desc *models, const double *d_start, int iters,
                              int *h_shape, float *h_ms, void *stream) {
    clear_error();
    if (!h_shape) return set_error(GBR_EINVAL, "NULL argument");
    std::vector<double> E((size_t)std::max(n_models, 1));
    float best = 1e30f;
    int bt = kBatchThreads, bp = 0, i = 0;
    for (int t : {128, 256, 512})
        for (int p : {0, 2, 1}) {
            float ms = 0.f;
            const int rc = batch_run(n_models, models, d_start, iters, E.data(), nullptr, nullptr,
                                     (cudaStream_t)stream, t, p, &ms);
            if (rc) return rc;
            if (h_ms) h_ms[i] = ms;
            ++i;
            if (ms < best) { best = ms; bt = t; bp = p; }
        }
    g_batch_threads = bt;
    g_batch_per_sm = bp;
    h_shape[0] = bt;
    h_shape[1] = bp;
    return GBR_OK;
}
