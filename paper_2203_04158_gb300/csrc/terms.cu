// General operator-product terms (Appendix: Eqs. Talpha1, Talpha2, ci and the
// product rule of Fig. mul) and an on-the-fly H·v over a trie-ranked state
// set for any list of such terms -- e.g. the O(M^3) two-body terms of the
// momentum-basis Hubbard ring (Sec. V-C, Eq. Hk) in a total-momentum sector.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "ham.h"

namespace gbr {

// Building blocks, Eqs. ci: c_i has v = 1, m = r = x = 2^i, l = 0,
// s = 2^i - 1; the creator c^dag_i exchanges l and r.
static gbr_term block(int orbital, bool creator) {
    gbr_term t;
    const uint64_t b = 1ull << orbital;
    t.v = 1.0;
    t.m = b;
    t.x = b;
    t.s = b - 1;
    t.l = creator ? b : 0;
    t.r = creator ? 0 : b;
    return t;
}

// Product T = T_a T_b (Fig. mul): Pauli check on the shared orbitals, union
// of the masks, outer demands r (right) and l (left) with the inner factor
// taking precedence on its own mask, the change mask x = l xor r, the sign
// mask outside m, and the sign of the reordering found by applying both
// factors' sign masks along the way to the state |r>.
static gbr_term mul(const gbr_term &a, const gbr_term &b) {
    gbr_term t;
    t.v = (((a.r ^ b.l) & a.m & b.m) != 0) ? 0.0 : a.v * b.v;
    t.m = a.m | b.m;
    t.r = b.r | (a.r & ~b.m);
    t.l = a.l | (b.l & ~a.m);
    t.x = t.l ^ t.r;
    t.s = (a.s ^ b.s) & ~t.m;
    uint64_t z = t.r;
    uint64_t p = z & b.s;
    z ^= b.x;
    p ^= z & a.s;
    if (__builtin_popcountll(p) & 1) t.v = -t.v;
    return t;
}

struct TermK {
    int nterms;
    int H;
    int shift[kMaxChunks];
    int width[kMaxChunks];
    int64_t padded, n;
};

// Two masks of a term in the narrowest word that holds M orbitals: (m, l) decides
// whether the term acts, (x, s) gives its target and sign.
template <typename W> struct alignas(2 * sizeof(W)) MaskPair { W a, b; };

__device__ __forceinline__ int parity(uint32_t a) { return __popc(a) & 1; }
__device__ __forceinline__ int parity(uint64_t a) { return __popcll(a) & 1; }

// Every term applied from the left to a member alpha (Eq. Talpha2):
// <alpha| T = v delta(alpha & m, l) (-1)^h(alpha & s) <alpha ^ x|,
// so y_i gathers v (-1)^... x_j at j = rank(alpha ^ x) -- the row of H, for
// any term list, Hermitian or not.  Ranks by the trie walk of Fig.
// trielookup; check = 1 drops targets outside the set.
//
// A warp takes S consecutive members.  Its lanes first test 32 terms at a time
// against each of them and append the terms that act to the member's queue in
// shared memory (ballot and prefix count); then G = 32 / S lanes per member work
// their queue off, two entries a lane at a time, so that the walks run with full
// warps: of the 1,752 terms of the 12-site momentum ring about a tenth act on a
// given member, and a thread per member ran nearly every term with 3 of its 32
// lanes.  The lanes' sums meet in a fixed butterfly: n terms round at most
// n / G + log2 G times on the way to y_i, where one chain rounds n times (166 random
// terms against extended precision: the largest error a third of the chain's).
//
// Bound: instruction issue (67 % of the slots) and the walks' loads.  12-site
// momentum ring, 71,188 members, FP64: 134 us, against 737 us for a thread per
// member; its 6,350-member 10-site sibling 13 against 343 us; 20 members of the
// 6-site ring 3.5 against 89 us (there a thread went through every term alone).
// The walk reads all levels through L1: with the leading levels staged in shared
// memory and a branch per level it took 142 us.
//
// S: four members share the loads of the terms, but leave a quarter of the warps;
// one member a warp below kTermOneBelow members per multiprocessor, where four
// would leave schedulers without work.
constexpr int kTermOneBelow = 64;
constexpr int kTermThreads = 256, kTermTile = 128, kTermUnroll = 2;

template <typename T, typename E, typename W, int S, bool BISECT>
__global__ void __launch_bounds__(kTermThreads) k_term_hv(const TermK tk, const E *__restrict__ trie,
                                                          const uint64_t *__restrict__ states,
                                                          const MaskPair<W> *__restrict__ ml,
                                                          const MaskPair<W> *__restrict__ xs, const T *__restrict__ vs,
                                                          int check, const T *__restrict__ x, T *__restrict__ y) {
    constexpr int G = 32 / S, UG = kTermUnroll * G, Q = kTermTile + UG;   // room for a tile and what the last one left
    __shared__ int queues[kTermThreads / 32][S][Q];
    const E last = (E)(tk.padded - 1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const int g = lane / G, gl = lane % G;
    int(*queue)[Q] = queues[warp];
    const int64_t nw = (int64_t)gridDim.x * (kTermThreads / 32);
    for (int64_t i0 = ((int64_t)blockIdx.x * (kTermThreads / 32) + warp) * S; i0 < tk.n; i0 += nw * S) {
        W a[S];
        int cnt[S];
#pragma unroll
        for (int s = 0; s < S; ++s) {
            a[s] = (W)states[i0 + s < tk.n ? i0 + s : tk.n - 1];
            cnt[s] = 0;
        }
        const int64_t i = i0 + g;
        W mine = a[0];
#pragma unroll
        for (int s = 1; s < S; ++s)
            if (g == s) mine = a[s];
        T acc = 0;
        for (int t0 = 0; t0 < tk.nterms; t0 += kTermTile) {
            MaskPair<W> c[kTermTile / 32];
#pragma unroll
            for (int u = 0; u < kTermTile / 32; ++u) {
                c[u] = ml[t0 + u * 32 + lane];
            }
#pragma unroll
            for (int u = 0; u < kTermTile / 32; ++u) {
                const int t = t0 + u * 32 + lane;
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    const bool acts = (a[s] & c[u].a) == c[u].b;
                    const unsigned who = __ballot_sync(0xFFFFFFFFu, acts);
                    if (acts) queue[s][cnt[s] + __popc(who & below)] = t;
                    cnt[s] += __popc(who);
                }
            }
            __syncwarp();
            // whole rounds of this member's entries; what is left waits for the next tile
            const bool end = t0 + kTermTile >= tk.nterms;
            int have = cnt[0];
#pragma unroll
            for (int s = 1; s < S; ++s)
                if (g == s) have = cnt[s];
            // (none for lanes past the last member: a diagonal term reads x at the member's place)
            const int todo = i >= tk.n ? 0 : end ? have : have - have % UG;
            for (int e = gl; e < todo; e += UG) {
                MaskPair<W> d[kTermUnroll];
                T v[kTermUnroll];
                bool on[kTermUnroll];
#pragma unroll
                for (int u = 0; u < kTermUnroll; ++u) {
                    on[u] = e + u * G < todo;
                    const int t = queue[g][on[u] ? e + u * G : e];
                    d[u] = xs[t];
                    v[u] = vs[t];
                }
                E k[kTermUnroll];
#pragma unroll
                for (int u = 0; u < kTermUnroll; ++u) k[u] = 0;
                if (BISECT) {
#pragma unroll
                    for (int u = 0; u < kTermUnroll; ++u) {
                        // the established baseline: lower bound in the sorted member list
                        const uint64_t b = (uint64_t)(mine ^ d[u].a);
                        int64_t lo = 0, len = tk.n;
                        while (len > 0) {
                            const int64_t half = len >> 1;
                            if (__ldg(states + lo + half) < b) { lo += half + 1; len -= half + 1; } else { len = half; }
                        }
                        k[u] = (E)lo;
                    }
                } else {
                    for (int lvl = 0; lvl < tk.H; ++lvl) {
                        const uint32_t mask = (1u << tk.width[lvl]) - 1u;
#pragma unroll
                        for (int u = 0; u < kTermUnroll; ++u) {
                            E idx = k[u] + (E)((uint32_t)((mine ^ d[u].a) >> tk.shift[lvl]) & mask);
                            idx = idx > last ? last : idx;
                            k[u] = __ldg(trie + idx);
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < kTermUnroll; ++u) {
                    if (!d[u].a) {
                        k[u] = (E)i;   // diagonal term
                    } else if ((check || BISECT) && !(k[u] < (E)tk.n && __ldg(states + k[u]) == (uint64_t)(mine ^ d[u].a))) {
                        on[u] = false;
                    }
                }
#pragma unroll
                for (int u = 0; u < kTermUnroll; ++u)
                    if (on[u]) acc += (parity(mine & d[u].b) ? -v[u] : v[u]) * x[k[u]];
            }
            if (end) break;
            __syncwarp();
            // a member with a whole round done has at least as many free slots as are left
            if (todo)
                for (int e = gl; e < have - todo; e += G) queue[g][e] = queue[g][todo + e];
            __syncwarp();
#pragma unroll
            for (int s = 0; s < S; ++s) cnt[s] %= UG;
        }
        __syncwarp();
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
        if (gl == 0 && i < tk.n) y[i] = acc;
    }
}

}  // namespace gbr

using namespace gbr;

struct gbr_termham {
    int M = 0;
    int bisect = 0;     // 1: rank by bisection in the member list instead of the trie
    int64_t n = 0;
    int nterms = 0;
    int64_t elements = 0;
    gbr_trie *trie = nullptr;
    // the terms' masks, in 32-bit words if M allows, and coefficients
    gbr::DevBuf ml, xs, v64, v32;
    gbr::LzWork lzw;    // Lanczos work buffers
    ~gbr_termham() { gbr_trie_destroy(trie); }
};

extern "C" int gbr_term_mul(const gbr_term *a, const gbr_term *b, gbr_term *out) {
    clear_error();
    if (!a || !b || !out) return set_error(GBR_EINVAL, "NULL argument");
    *out = mul(*a, *b);
    return GBR_OK;
}

extern "C" int gbr_term_product(const int *ops, int nops, double coef, gbr_term *out) {
    clear_error();
    if (!out || (nops > 0 && !ops) || nops < 0) return set_error(GBR_EINVAL, "bad operator list");
    gbr_term t;
    t.v = coef;
    t.m = t.l = t.r = t.x = t.s = 0;
    for (int o = 0; o < nops; ++o) {
        const int code = ops[o];
        if (code < 0 || (code >> 1) >= 64) return set_error(GBR_EINVAL, "operator code %d out of range", code);
        t = mul(t, block(code >> 1, code & 1));
    }
    *out = t;
    return GBR_OK;
}

namespace gbr {
template <typename W> static int upload_terms(gbr_termham *T, const gbr_term *t, int n) {
    // whole tiles: what follows the terms acts on no state
    std::vector<MaskPair<W>> ml(((size_t)n + kTermTile - 1) / kTermTile * kTermTile, MaskPair<W>{0, 1}), xs((size_t)n);
    std::vector<double> v64((size_t)n);
    for (int i = 0; i < n; ++i) {
        ml[(size_t)i] = {(W)t[i].m, (W)t[i].l};
        xs[(size_t)i] = {(W)t[i].x, (W)t[i].s};
        v64[(size_t)i] = t[i].v;
    }
    std::vector<float> v32(v64.begin(), v64.end());
    int rc = T->ml.upload(ml.data(), ml.size() * sizeof(ml[0]));
    if (!rc) rc = T->xs.upload(xs.data(), xs.size() * sizeof(xs[0]));
    if (!rc) rc = T->v64.upload(v64.data(), v64.size() * 8);
    if (!rc) rc = T->v32.upload(v32.data(), v32.size() * 4);
    return rc;
}
}  // namespace gbr

extern "C" int gbr_termham_create(int M, const gbr_term *h_terms, int nterms, const uint64_t *h_states, int64_t n,
                                  int R, gbr_termham **out) {
    clear_error();
    if (!out) return set_error(GBR_EINVAL, "out is NULL");
    *out = nullptr;
    if (M < 1 || M > 64) return set_error(GBR_EINVAL, "M=%d out of range 1..64", M);
    if (nterms < 1 || !h_terms) return set_error(GBR_EINVAL, "empty term list");
    const uint64_t all = M == 64 ? ~0ull : ((1ull << M) - 1);
    for (int t = 0; t < nterms; ++t) {
        if ((h_terms[t].m | h_terms[t].l | h_terms[t].r | h_terms[t].x | h_terms[t].s) & ~all)
            return set_error(GBR_EINVAL, "term %d touches orbitals at or above M", t);
        if (!std::isfinite(h_terms[t].v)) return set_error(GBR_EINVAL, "term %d has a non-finite coefficient", t);
    }
    gbr_termham *T = new (std::nothrow) gbr_termham();
    if (!T) return set_error(GBR_ENOMEM, "host allocation failed");
    T->M = M;
    T->n = n;
    T->nterms = nterms;
    // most significant chunk first: neighbouring members share their walks
    int rc = trie_create(h_states, n, M, R, 1, false, &T->trie);
    if (!rc) {
        // matrix elements: every (member, term) pair whose left demand holds
        int64_t el = 0;
        for (int64_t i = 0; i < n; ++i)
            for (int t = 0; t < nterms; ++t)
                if ((h_states[i] & h_terms[t].m) == h_terms[t].l && h_terms[t].v != 0.0) ++el;
        T->elements = el;
        rc = M <= 32 ? upload_terms<uint32_t>(T, h_terms, nterms) : upload_terms<uint64_t>(T, h_terms, nterms);
    }
    if (rc) { delete T; return rc; }
    *out = T;
    return GBR_OK;
}

extern "C" void gbr_termham_destroy(gbr_termham *T) { delete T; }

extern "C" int gbr_termham_set_bisect(gbr_termham *T, int bisect) {
    clear_error();
    if (!T) return set_error(GBR_EINVAL, "NULL handle");
    T->bisect = bisect ? 1 : 0;
    return GBR_OK;
}

extern "C" int gbr_termham_info(const gbr_termham *T, int64_t *dim, int64_t *elements, int64_t *trie_elements) {
    clear_error();
    if (!T) return set_error(GBR_EINVAL, "NULL handle");
    if (dim) *dim = T->n;
    if (elements) *elements = T->elements;
    if (trie_elements) *trie_elements = T->trie->size;
    return GBR_OK;
}

namespace gbr {
template <typename T, typename E, typename W>
static int launch_term_kernel(const gbr_termham *Th, const TermK &tk, const T *x, T *y, int check, cudaStream_t st) {
    const gbr_trie *tr = Th->trie;
    // one member a warp while that leaves warps idle, else four
    const int S = Th->n < (int64_t)sm_count() * kTermOneBelow ? 1 : 4;
    auto kern = Th->bisect ? (S == 1 ? k_term_hv<T, E, W, 1, true> : k_term_hv<T, E, W, 4, true>)
                           : (S == 1 ? k_term_hv<T, E, W, 1, false> : k_term_hv<T, E, W, 4, false>);
    const int64_t per = (int64_t)(kTermThreads / 32) * S;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((Th->n + per - 1) / per, (int64_t)sm_count() * 8));
    kern<<<(int)blocks, kTermThreads, 0, st>>>(tk, tr->t.as<E>(), tr->members.as<uint64_t>(), Th->ml.as<MaskPair<W>>(),
                                                  Th->xs.as<MaskPair<W>>(),
                                                  sizeof(T) == 8 ? (const T *)Th->v64.p : (const T *)Th->v32.p, check, x, y);
    GBR_LAUNCH_CHECK();
    count_launches(1);
    return GBR_OK;
}

template <typename T, typename E>
static int launch_term_hv(const gbr_termham *Th, const T *x, T *y, int check, cudaStream_t st) {
    const gbr_trie *tr = Th->trie;
    TermK tk;
    memset(&tk, 0, sizeof(tk));
    tk.nterms = Th->nterms;
    tk.H = tr->H;
    for (int l = 0; l < tr->H; ++l) { tk.shift[l] = tr->shift[l]; tk.width[l] = tr->width[l]; }
    tk.padded = tr->padded;
    tk.n = Th->n;
    if (Th->M <= 32) return launch_term_kernel<T, E, uint32_t>(Th, tk, x, y, check, st);
    return launch_term_kernel<T, E, uint64_t>(Th, tk, x, y, check, st);
}
}  // namespace gbr

namespace gbr {
// y = H x over the set with membership checks (the Lanczos operator)
static int term_apply(const void *obj, const void *x, void *y, int fp, cudaStream_t st) {
    const gbr_termham *T = static_cast<const gbr_termham *>(obj);
    if (T->trie->wide) {
        if (fp == 64) return launch_term_hv<double, uint64_t>(T, (const double *)x, (double *)y, 1, st);
        return launch_term_hv<float, uint64_t>(T, (const float *)x, (float *)y, 1, st);
    }
    if (fp == 64) return launch_term_hv<double, uint32_t>(T, (const double *)x, (double *)y, 1, st);
    return launch_term_hv<float, uint32_t>(T, (const float *)x, (float *)y, 1, st);
}
}  // namespace gbr

extern "C" int gbr_termham_lanczos(const gbr_termham *T, const gbr_lanczos_opts *o, const double *d_v0,
                                   gbr_lanczos_result *res, double *h_alpha, double *h_beta, double *h_ritz,
                                   void *stream) {
    clear_error();
    if (!T) return set_error(GBR_EINVAL, "NULL handle");
    const LzOp op{nullptr, T, &term_apply, T->n, &const_cast<gbr_termham *>(T)->lzw};
    return lanczos_solve(op, o, d_v0, res, h_alpha, h_beta, h_ritz, stream);
}

extern "C" int gbr_termham_hv(const gbr_termham *T, const void *d_x, void *d_y, int fp, int check, void *stream) {
    clear_error();
    if (!T) return set_error(GBR_EINVAL, "NULL handle");
    if (fp != 32 && fp != 64) return set_error(GBR_EINVAL, "fp=%d must be 32 or 64", fp);
    if (!d_x || !d_y) return set_error(GBR_EINVAL, "NULL vector");
    const size_t s = fp == 64 ? 8 : 4;
    const uintptr_t xa = (uintptr_t)d_x, ya = (uintptr_t)d_y;
    if ((xa | ya) % s) return set_error(GBR_EINVAL, "vectors must be aligned to their element size");
    const uintptr_t bytes = (uintptr_t)T->n * s;
    if (xa < ya + bytes && ya < xa + bytes) return set_error(GBR_EINVAL, "x and y overlap");
    cudaStream_t st = (cudaStream_t)stream;
    if (T->trie->wide) {
        if (fp == 64) return launch_term_hv<double, uint64_t>(T, (const double *)d_x, (double *)d_y, check, st);
        return launch_term_hv<float, uint64_t>(T, (const float *)d_x, (float *)d_y, check, st);
    }
    if (fp == 64) return launch_term_hv<double, uint32_t>(T, (const double *)d_x, (double *)d_y, check, st);
    return launch_term_hv<float, uint32_t>(T, (const float *)d_x, (float *)d_y, check, st);
}
