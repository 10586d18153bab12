// On-the-fly H·v over an arbitrary sorted set of states, ranked by the packed
// trie (Sec. IV of Wallerberger & Held): the case the combinadics cannot
// index -- sectors cut by further quantum numbers, or unions of spin
// sectors such as all S_z at fixed particle number.  No spin factorisation:
// every hop of every member is ranked by a walk of Fig. trielookup over the
// full 2L-bit pattern, and (check mode) verified against the member list.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "ham.h"

struct gbr_setham {
    int L = 0, R = 0;
    int bisect = 0;             // 1: rank by bisection in the member list instead of the trie
    int64_t n = 0;
    int64_t elements = 0;
    gbr::HamK k{};
    gbr_trie *trie = nullptr;
    int nent = 0, has_diag = 0;
    gbr::DevBuf hops;           // ends and between-masks of every bond of both spins
    gbr::DevBuf hc64, hc32;     // and their coefficients
    gbr::DevBuf hd64, hd32;     // L diagonal one-body terms h_pp
    gbr::DevBuf uv64, uv32;     // U class values
    gbr::LzWork lzw;            // Lanczos work buffers
    ~gbr_setham() { gbr_trie_destroy(trie); }
};

namespace gbr {

struct SetTrieK {
    int H;
    int shift[kMaxChunks];
    int width[kMaxChunks];
    int64_t padded, n;
    int nent;        // entries of the hop table
    int has_diag;    // any h_pp != 0
};

// One undirected bond of one spin in the narrowest word that holds 2L orbitals:
// its two orbitals and the orbitals strictly between them.
template <typename W> struct alignas(2 * sizeof(W)) SetHop { W ends, between; };

__device__ __forceinline__ int bit_count(uint32_t a) { return __popc(a); }
__device__ __forceinline__ int bit_count(uint64_t a) { return __popcll(a); }

// TPS threads per member.  A thread first tests its share of the bonds of both
// spins against the member (a hop exists where exactly one end is occupied, in
// either direction with the same coefficient, h being symmetric) and keeps the
// answers as a 32-bit mask, then works off the set bits: every round of that
// loop is two whole hops for every thread that has them left, their walks side by
// side.  Nested loops over occupied sites and their empty neighbours left lanes
// idle at both levels: 2,527 warp instructions per 32 members of the 12-site ring's
// every-S_z set at 12.5 hops a member, against 1,580.
//
// Bound: instruction issue and the latency of the walks.  That set (2.7e6 members):
// 142 us FP32 and 202 us FP64, against 266 and 414 us (172 and 199 us with one hop
// a round); 2,002 members of the 7-site ring 4.1 against 12.5 us.
//
// TPS: eight threads a member where that does not fill the chip's 2,048 threads a
// multiprocessor twice over (48,620 members 7.3 us, against 16.6 us with the one
// thread of before), two up to one member per thread, else one.
constexpr int kSetThreads = 256;

template <typename T, typename E, typename W, int TPS, bool BISECT>
__global__ void __launch_bounds__(kSetThreads) k_set_hv(const SetTrieK tk, const E *__restrict__ t,
                                                        const uint64_t *__restrict__ states, const HamK hk,
                                                        const SetHop<W> *__restrict__ hops, const T *__restrict__ hc,
                                                        const T *__restrict__ hd, const T *__restrict__ uv, int check,
                                                        const T *__restrict__ x, T *__restrict__ y) {
    extern __shared__ __align__(16) unsigned char smr[];
    SetHop<W> *sh = reinterpret_cast<SetHop<W> *>(smr);
    T *sc = reinterpret_cast<T *>(sh + tk.nent);
    T *hds = sc + tk.nent;
    for (int i = threadIdx.x; i < tk.nent; i += kSetThreads) {
        sh[i] = hops[i];
        sc[i] = hc[i];
    }
    for (int i = threadIdx.x; i < hk.L; i += kSetThreads) hds[i] = hd[i];
    __syncthreads();
    const E last = (E)(tk.padded - 1);
    const int L = hk.L;
    const W lowmask = (W)((1ull << L) - 1);
    const int g = threadIdx.x % TPS;
    const int64_t stride = (int64_t)gridDim.x * (kSetThreads / TPS);
    // the members of one warp end together: TPS consecutive lanes share one, and
    // every lane takes part in the butterfly
    const int64_t rounds = (tk.n + stride - 1) / stride;
    for (int64_t rd = 0; rd < rounds; ++rd) {
        const int64_t i = rd * stride + (int64_t)blockIdx.x * (kSetThreads / TPS) + threadIdx.x / TPS;
        const bool live = i < tk.n;
        const W a = live ? (W)states[i] : W(0);
        T acc = 0;
        if (live && g == 0) {
            // diagonal: one-body h_pp n_p for both spins, U on doubly occupied sites
            const uint32_t ad = (uint32_t)(a & lowmask), au = (uint32_t)(a >> L);
            T dg = 0;
            if (tk.has_diag) {
                uint32_t occ = ad | au;
                while (occ) {
                    const int p = __ffs(occ) - 1;
                    occ &= occ - 1u;
                    dg += hds[p] * (T)(((ad >> p) & 1u) + ((au >> p) & 1u));
                }
            }
            for (int c = 0; c < hk.nucls; ++c) dg += __ldg(uv + c) * (T)__popc(ad & au & hk.umask[c]);
            acc = dg * x[i];
        }
        for (int e0 = 0; e0 < tk.nent; e0 += 32 * TPS) {
            // bit j: entry e0 + j TPS + g
            uint32_t act = 0;
            const int ne = (tk.nent - e0 - g + TPS - 1) / TPS < 32 ? (tk.nent - e0 - g + TPS - 1) / TPS : 32;
            for (int j = 0; j < ne; ++j) {
                const W ends = sh[e0 + j * TPS + g].ends;
                const W m = a & ends;
                if (m != 0 && m != ends) act |= 1u << j;
            }
            if (!live) act = 0;
            // two hops a round, their walks side by side (the second may be missing)
            while (act) {
                int e[2];
                bool on[2];
                W b[2];
                E k[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    on[u] = act != 0;
                    e[u] = on[u] ? e0 + (__ffs(act) - 1) * TPS + g : e[0];
                    act &= act - 1u;
                    b[u] = a ^ sh[e[u]].ends;
                    k[u] = 0;
                }
                if (BISECT) {
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        // the established baseline: lower bound in the sorted member list
                        int64_t lo = 0, len = tk.n;
                        while (len > 0) {
                            const int64_t half = len >> 1;
                            if (__ldg(states + lo + half) < (uint64_t)b[u]) { lo += half + 1; len -= half + 1; } else { len = half; }
                        }
                        k[u] = (E)lo;
                    }
                } else {
                    // Fig. trielookup on the full pattern, indices clamped into the table
                    for (int lvl = 0; lvl < tk.H; ++lvl) {
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const E idx = k[u] + (E)((uint32_t)(b[u] >> tk.shift[lvl]) & ((1u << tk.width[lvl]) - 1u));
                            k[u] = __ldg(t + (idx > last ? last : idx));
                        }
                    }
                }
                if (check || BISECT) {
#pragma unroll
                    for (int u = 0; u < 2; ++u) on[u] = on[u] && k[u] < (E)tk.n && __ldg(states + k[u]) == (uint64_t)b[u];
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const T c = sc[e[u]];
                    if (on[u]) acc += ((bit_count(a & sh[e[u]].between) & 1) ? -c : c) * x[k[u]];
                }
            }
        }
#pragma unroll
        for (int o = TPS / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
        if (live && g == 0) y[i] = acc;
    }
}

template <typename T, typename E, typename W>
static int launch_set_kernel(const gbr_setham *S, const SetTrieK &tk, const T *x, T *y, int check, cudaStream_t st) {
    const gbr_trie *tr = S->trie;
    const bool d = sizeof(T) == 8;
    const size_t smem = (size_t)tk.nent * (sizeof(SetHop<W>) + sizeof(T)) + (size_t)S->L * sizeof(T);
    const int64_t full = (int64_t)sm_count() * 2048;   // threads the chip holds
    const int tps = S->n * 4 <= full ? 8 : (S->n <= full ? 2 : 1);
    auto kern = S->bisect ? (tps == 8 ? k_set_hv<T, E, W, 8, true> : tps == 2 ? k_set_hv<T, E, W, 2, true> : k_set_hv<T, E, W, 1, true>)
                          : (tps == 8 ? k_set_hv<T, E, W, 8, false> : tps == 2 ? k_set_hv<T, E, W, 2, false> : k_set_hv<T, E, W, 1, false>);
    const int64_t per = kSetThreads / tps;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((S->n + per - 1) / per, (int64_t)sm_count() * 8));
    if (smem > 48 * 1024) GBR_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<(int)blocks, kSetThreads, smem, st>>>(tk, tr->t.as<E>(), tr->members.as<uint64_t>(), S->k, S->hops.as<SetHop<W>>(),
                                                 (const T *)(d ? S->hc64.p : S->hc32.p), (const T *)(d ? S->hd64.p : S->hd32.p),
                                                 (const T *)(d ? S->uv64.p : S->uv32.p), check, x, y);
    GBR_LAUNCH_CHECK();
    count_launches(1);
    return GBR_OK;
}

template <typename T, typename E>
static int launch_set_hv(const gbr_setham *S, const T *x, T *y, int check, cudaStream_t st) {
    const gbr_trie *tr = S->trie;
    SetTrieK tk;
    memset(&tk, 0, sizeof(tk));
    tk.H = tr->H;
    for (int l = 0; l < tr->H; ++l) { tk.shift[l] = tr->shift[l]; tk.width[l] = tr->width[l]; }
    tk.padded = tr->padded;
    tk.n = S->n;
    tk.nent = S->nent;
    tk.has_diag = S->has_diag;
    if (2 * S->L <= 32) return launch_set_kernel<T, E, uint32_t>(S, tk, x, y, check, st);
    return launch_set_kernel<T, E, uint64_t>(S, tk, x, y, check, st);
}

// Hop table of both spins: every bond p < q, spin down first.
template <typename W> static int upload_hops(gbr_setham *S, const double *h) {
    const int L = S->L;
    std::vector<SetHop<W>> hops;
    std::vector<double> c;
    for (int off : {0, L})
        for (int p = 0; p < L; ++p)
            for (int q = p + 1; q < L; ++q) {
                if (h[p * L + q] == 0.0) continue;
                const uint64_t ends = (1ull << p) | (1ull << q), between = ((1ull << q) - 1) & ~((2ull << p) - 1);
                hops.push_back({(W)(ends << off), (W)(between << off)});
                c.push_back(h[p * L + q]);
            }
    S->nent = (int)hops.size();
    if (hops.empty()) {   // nothing to read, but the buffers exist
        hops.push_back({0, 0});
        c.push_back(0.0);
    }
    std::vector<float> c32(c.begin(), c.end());
    int rc = S->hops.upload(hops.data(), hops.size() * sizeof(hops[0]));
    if (!rc) rc = S->hc64.upload(c.data(), c.size() * 8);
    if (!rc) rc = S->hc32.upload(c32.data(), c32.size() * 4);
    return rc;
}

// y = H x on the set with membership checks (the Lanczos operator; a set
// not closed under H gets the projected operator P H P)
static int set_apply(const void *obj, const void *x, void *y, int fp, cudaStream_t st) {
    const gbr_setham *S = static_cast<const gbr_setham *>(obj);
    if (S->trie->wide) {
        if (fp == 64) return launch_set_hv<double, uint64_t>(S, (const double *)x, (double *)y, 1, st);
        return launch_set_hv<float, uint64_t>(S, (const float *)x, (float *)y, 1, st);
    }
    if (fp == 64) return launch_set_hv<double, uint32_t>(S, (const double *)x, (double *)y, 1, st);
    return launch_set_hv<float, uint32_t>(S, (const float *)x, (float *)y, 1, st);
}

}  // namespace gbr

using namespace gbr;

extern "C" int gbr_setham_lanczos(const gbr_setham *S, const gbr_lanczos_opts *o, const double *d_v0,
                                  gbr_lanczos_result *res, double *h_alpha, double *h_beta, double *h_ritz,
                                  void *stream) {
    clear_error();
    if (!S) return set_error(GBR_EINVAL, "NULL handle");
    const LzOp op{nullptr, S, &set_apply, S->n, &const_cast<gbr_setham *>(S)->lzw};
    return lanczos_solve(op, o, d_v0, res, h_alpha, h_beta, h_ritz, stream);
}

extern "C" int gbr_setham_create_ordered(int L, const double *h, const double *U, const uint64_t *h_states,
                                         int64_t n, int R, int msb_first, gbr_setham **out) {
    clear_error();
    if (!out) return set_error(GBR_EINVAL, "out is NULL");
    *out = nullptr;
    if (L < 1 || L > kMaxL) return set_error(GBR_EINVAL, "L=%d out of range 1..%d", L, kMaxL);
    if (!h || !h_states) return set_error(GBR_EINVAL, "NULL argument");
    if (n < 1) return set_error(GBR_EINVAL, "empty state set");
    for (int p = 0; p < L; ++p)
        for (int q = 0; q < L; ++q) {
            const double a = h[p * L + q];
            if (!std::isfinite(a) || a != h[q * L + p]) return set_error(GBR_EINVAL, "h not finite and symmetric at (%d,%d)", p, q);
        }
    gbr_setham *S = new (std::nothrow) gbr_setham();
    if (!S) return set_error(GBR_ENOMEM, "host allocation failed");
    S->L = L;
    S->R = R;
    S->n = n;
    std::vector<uint16_t> pairs, bidx;
    int rc = build_hamk(L, h, U, GBR_RANK_STAGGERED, &S->k, &pairs, &bidx);
    if (!rc) rc = trie_create(h_states, n, 2 * L, R, msb_first, false, &S->trie);   // validates order, duplicates, width
    if (rc) { delete S; return rc; }
    // elements: the diagonal plus every hop of every member (for a set closed
    // under H, exactly the matrix elements one H·v visits)
    int64_t el = n;
    const uint64_t lowmask = (1ull << L) - 1;
    for (int64_t i = 0; i < n; ++i) {
        const uint32_t sp[2] = {(uint32_t)(h_states[i] & lowmask), (uint32_t)(h_states[i] >> L)};
        for (int s = 0; s < 2; ++s)
            for (int p = 0; p < L; ++p)
                if ((sp[s] >> p) & 1u) el += __builtin_popcount(S->k.nbr[p] & ~sp[s]);
    }
    S->elements = el;
    std::vector<double> hd((size_t)L), uv(kMaxUClasses, 0.0);
    for (int p = 0; p < L; ++p) {
        hd[(size_t)p] = h[p * L + p];
        if (hd[(size_t)p] != 0.0) S->has_diag = 1;
    }
    for (int c = 0; c < S->k.nucls; ++c) uv[(size_t)c] = S->k.uval[c];
    std::vector<float> hd32(hd.begin(), hd.end()), uv32(uv.begin(), uv.end());
    rc = 2 * L <= 32 ? upload_hops<uint32_t>(S, h) : upload_hops<uint64_t>(S, h);
    if (!rc) rc = S->hd64.upload(hd.data(), hd.size() * 8);
    if (!rc) rc = S->uv64.upload(uv.data(), uv.size() * 8);
    if (!rc) rc = S->hd32.upload(hd32.data(), hd32.size() * 4);
    if (!rc) rc = S->uv32.upload(uv32.data(), uv32.size() * 4);
    if (rc) { delete S; return rc; }
    *out = S;
    return GBR_OK;
}

extern "C" int gbr_setham_create(int L, const double *h, const double *U, const uint64_t *h_states, int64_t n, int R,
                                 gbr_setham **out) {
    return gbr_setham_create_ordered(L, h, U, h_states, n, R, 1, out);
}

extern "C" void gbr_setham_destroy(gbr_setham *S) { delete S; }

extern "C" int gbr_setham_set_bisect(gbr_setham *S, int bisect) {
    clear_error();
    if (!S) return set_error(GBR_EINVAL, "NULL handle");
    S->bisect = bisect ? 1 : 0;
    return GBR_OK;
}

extern "C" int gbr_setham_info(const gbr_setham *S, int64_t *dim, int64_t *elements, int64_t *trie_elements) {
    clear_error();
    if (!S) return set_error(GBR_EINVAL, "NULL handle");
    if (dim) *dim = S->n;
    if (elements) *elements = S->elements;
    if (trie_elements) *trie_elements = S->trie->size;
    return GBR_OK;
}

extern "C" int gbr_setham_hv(const gbr_setham *S, const void *d_x, void *d_y, int fp, int check, void *stream) {
    clear_error();
    if (!S) return set_error(GBR_EINVAL, "NULL handle");
    if (fp != 32 && fp != 64) return set_error(GBR_EINVAL, "fp=%d must be 32 or 64", fp);
    if (!d_x || !d_y) return set_error(GBR_EINVAL, "NULL vector");
    const size_t s = fp == 64 ? 8 : 4;
    const uintptr_t xa = (uintptr_t)d_x, ya = (uintptr_t)d_y;
    if ((xa | ya) % s) return set_error(GBR_EINVAL, "vectors must be aligned to their element size");
    const uintptr_t bytes = (uintptr_t)S->n * s;
    if (xa < ya + bytes && ya < xa + bytes) return set_error(GBR_EINVAL, "x and y overlap");
    cudaStream_t st = (cudaStream_t)stream;
    if (S->trie->wide) {
        if (fp == 64) return launch_set_hv<double, uint64_t>(S, (const double *)d_x, (double *)d_y, check, st);
        return launch_set_hv<float, uint64_t>(S, (const float *)d_x, (float *)d_y, check, st);
    }
    if (fp == 64) return launch_set_hv<double, uint32_t>(S, (const double *)d_x, (double *)d_y, check, st);
    return launch_set_hv<float, uint32_t>(S, (const float *)d_x, (float *)d_y, check, st);
}
