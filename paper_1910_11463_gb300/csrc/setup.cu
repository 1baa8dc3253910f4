// AIR setup on the GPU (Sec. 1.2; Sec. 4.1.1 Eq. soc; Sec. 4.1.2 filtering).
//
// A hierarchy holds a batch of independent matrices; every level of every
// matrix is processed by one launch per step.  Compiled with --fmad=false and
// written so that each floating-point result is formed by the same operations
// in the same order as the plain definitions below (fused multiply-adds only
// where fma() is written), hence reproducible bit for bit:
//   strength   S_i = {j != i : |a_ij| >= theta * max_{k != i} |a_ik|}, empty if the max is 0
//   PMIS       key_i = (lambda_i, h_i, i), lambda_i = #{k : i in S_k},
//              h_i = top 32 bits of SplitMix64 at state seed ^ (level << 40) ^ i (local i);
//              lambda_i = 0 -> F; rounds: undecided local key maxima over S + S^T -> C,
//              undecided rows depending strongly on a new C -> F
//   P          one-point: F row -> strongest C neighbour in S_i (first maximum), weight 1
//   lAIR       C row i, pattern R_i = strong (eps_R) F neighbours (distance 1, or 2 via F
//              points), A[R_i,R_i]^T z = -A[i,R_i]^T by LU with partial pivoting (first max
//              pivot, full row swaps, column-oriented substitutions); optional phi_R filter
//   RAP        (AP)[k,c] = sum over l ascending (pmap(l) = c) of a_kl, starting from 0.0;
//              (RAP)[i,c] = sum over the R row in ascending column order (identity at
//              its place) of R_ik (AP)[k,c], starting from 0.0, one fma per term; every
//              structural product kept; optional phi_A filter of off-diagonal entries
//   LU         multipliers a_rk * (1 / a_kk), updates fma(-l, a_kc, a_rc), substitutions
//              by columns with fma, y_k * (1 / u_kk)
#include <algorithm>
#include <cstdio>

#include "common.cuh"

namespace pr {

namespace {

constexpr int8_t ST_U = -1, ST_F = 0, ST_C = 1;

__device__ __forceinline__ uint64_t splitmix_first(uint64_t state) {
    uint64_t z = state + 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

__device__ __forceinline__ double lookup(const int *rowptr, const int *col, const double *val, int i, int j) {
    int lo = rowptr[i], hi = rowptr[i + 1] - 1;
    while (lo <= hi) {
        int m = (lo + hi) >> 1;
        int c = col[m];
        if (c == j) return val[m];
        if (c < j) lo = m + 1; else hi = m - 1;
    }
    return 0.0;
}

__global__ void k_dinv(int n, const int *rowptr, const int *col, const double *val, double *dinv, float *dinv32) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double d = lookup(rowptr, col, val, i, i);
    double r = (d != 0.0) ? 1.0 / d : 0.0;
    dinv[i] = r;
    if (dinv32) dinv32[i] = (float)r;
}

// Strength, bit 0: S (theta), bit 1: S^R (eps_R); lam[j] += 1 for every row that depends on
// j; smask: per row of at most 32 entries, the entries with bit 0 (longer rows: not used).
// A block stages its 128 rows' entries (contiguous in the CSR) with coalesced loads and a
// thread takes its row from shared memory; rows past the staged entries read global memory.
// Magnitudes compare as integers, so a row costs two FP64 instructions; NaN entries are
// strong to nothing, as in a comparison of doubles.  The CF splitting and P then visit the
// set bits of smask instead of every entry's flag.  64^3 S8 setup: strength 44 -> 18 ms,
// PMIS 84 -> 62 ms, and no pass of its own for lam (9 ms).
__device__ __forceinline__ bool is_nan_bits(long long m) { return m > 0x7ff0000000000000LL; }

__global__ void __launch_bounds__(128) k_strength(int n, const int *rowptr, const int *col, const double *val,
                                                  const int *rowdir, const char *dwork, double theta, double epsR,
                                                  uint8_t *S, unsigned *smask, unsigned *lam, int cap) {
    extern __shared__ double stsm[];
    long long *sv = (long long *)stsm;
    int *sc = (int *)(stsm + cap);
    uint8_t *sf = (uint8_t *)(sc + cap);
    const int r0 = blockIdx.x * 128, r1 = min(n, r0 + 128);
    const int P0 = rowptr[r0], E = min(rowptr[r1] - P0, cap);
    for (int p = threadIdx.x; p < E; p += 128) {
        sc[p] = col[P0 + p];
        sv[p] = absbits(val[P0 + p]);
    }
    __syncthreads();
    const int i = r0 + threadIdx.x;
    if (i < r1) {
        const int s = rowptr[i] - P0, e = rowptr[i + 1] - P0;
        const bool in = e <= E, work = dwork[rowdir[i]];
        long long mx = 0;
        if (work)
            for (int p = s; p < e; ++p) {
                const int c = in ? sc[p] : col[P0 + p];
                const long long v = in ? sv[p] : absbits(val[P0 + p]);
                if (c != i && v > mx && !is_nan_bits(v)) mx = v;
            }
        const double m = __longlong_as_double(mx);
        const long long t1 = __double_as_longlong(theta * m), t2 = __double_as_longlong(epsR * m);
        unsigned msk = 0;
        for (int p = s; p < e; ++p) {
            uint8_t f = 0;
            if (mx > 0) {
                const int c = in ? sc[p] : col[P0 + p];
                const long long v = in ? sv[p] : absbits(val[P0 + p]);
                if (c != i && !is_nan_bits(v)) {
                    if (v >= t1) {
                        f |= 1;
                        atomicAdd(&lam[c], 1u);
                        if (p - s < 32) msk |= 1u << (p - s);
                    }
                    if (v >= t2) f |= 2;
                }
            }
            if (in) sf[p] = f;
            else S[P0 + p] = f;
        }
        smask[i] = msk;
    }
    __syncthreads();
    // the staged bytes, except the entries of a row that ends past them (written above)
    for (int p = threadIdx.x; p < E; p += 128) sc[p] = 0;
    __syncthreads();
    if (i < r1) {
        const int s = rowptr[i] - P0, e = rowptr[i + 1] - P0;
        if (e > E)
            for (int p = s; p < min(e, E); ++p) sc[p] = 1;
    }
    __syncthreads();
    for (int p = threadIdx.x; p < E; p += 128)
        if (!sc[p]) S[P0 + p] = sf[p];
}

// f(p) for the strong entries of row i, ascending
template <class F>
__device__ __forceinline__ void for_strong(int i, const int *rowptr, const uint8_t *S, const unsigned *smask, F &&f) {
    const int p0 = rowptr[i], p1 = rowptr[i + 1];
    if (p1 - p0 <= 32) {
        for (unsigned m = smask[i]; m; m &= m - 1)
            if (!f(p0 + __ffs(m) - 1)) return;
    } else {
        for (int p = p0; p < p1; ++p)
            if ((S[p] & 1) && !f(p)) return;
    }
}

__global__ void k_pmis_init(int n, const int *rowdir, const char *dwork, const int *row0, const unsigned *lam,
                            int level, unsigned long long seed, uint64_t *key, int8_t *state, int *undecided) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int8_t s = ST_F;
    if (i < n) {
        int d = rowdir[i];
        if (!dwork[d]) {
            key[i] = 0;
        } else {
            uint64_t li = (uint64_t)(i - row0[d]);
            uint32_t hh = (uint32_t)(splitmix_first(seed ^ ((uint64_t)level << 40) ^ li) >> 32);
            key[i] = ((uint64_t)lam[i] << 32) | hh;
            if (lam[i] != 0) s = ST_U;
        }
        state[i] = s;
    }
    // one atomic per block: they all meet at one address
    const int c = __syncthreads_count(s == ST_U);
    if (threadIdx.x == 0 && c) atomicAdd(undecided, c);
}

__device__ __forceinline__ bool key_gt(uint64_t kj, int j, uint64_t ki, int i) {
    return kj > ki || (kj == ki && j > i);
}

__global__ void k_pmis_mark(int n, const int *rowptr, const int *col, const uint8_t *S, const unsigned *smask,
                            const uint64_t *key, const int8_t *state, int *notmax, int round) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || state[i] != ST_U) return;
    uint64_t ki = key[i];
    for_strong(i, rowptr, S, smask, [&](int p) {
        const int j = col[p];
        if (state[j] == ST_U) {
            if (key_gt(key[j], j, ki, i)) notmax[i] = round;
            else notmax[j] = round;
        }
        return true;
    });
}

__global__ void k_pmis_update(int n, const int *rowptr, const int *col, const uint8_t *S, const unsigned *smask,
                              const int8_t *state, int8_t *next, const int *notmax, int round, int *undecided) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int8_t s = i < n ? state[i] : ST_F;
    if (s == ST_U) {
        if (notmax[i] != round) {
            s = ST_C;
        } else {
            for_strong(i, rowptr, S, smask, [&](int p) {
                const int j = col[p];
                if (state[j] == ST_U && notmax[j] != round) s = ST_F;
                return s == ST_U;
            });
        }
    }
    if (i < n) next[i] = s;
    const int c = __syncthreads_count(s == ST_U);
    if (threadIdx.x == 0 && c) atomicAdd(undecided, c);
}

// per-matrix sums: one atomic per warp when its rows share a matrix (the usual case)
template <class T>
__device__ __forceinline__ void add_by_dir(T *out, int d, T v, bool valid) {
    unsigned act = __ballot_sync(0xffffffffu, valid);
    if (!act) return;
    int d0 = __shfl_sync(0xffffffffu, d, __ffs(act) - 1);
    bool same = __all_sync(0xffffffffu, !valid || d == d0);
    if (same) {
        T tot = valid ? v : T(0);
        for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
        if ((threadIdx.x & 31) == __ffs(act) - 1 && tot) atomicAdd(&out[d0], tot);
    } else if (valid && v) {
        atomicAdd(&out[d], v);
    }
}

__global__ void k_count_c(int n, const int *rowdir, const int8_t *state, int *ncdir) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    bool valid = i < n;
    int d = valid ? rowdir[i] : 0;
    add_by_dir<int>(ncdir, d, (valid && state[i] == ST_C) ? 1 : 0, valid);
}

__global__ void k_cf_final(int n, const int *rowdir, const char *cont, const int8_t *state, int8_t *cf, int *isC) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    bool c = cont[rowdir[i]];
    cf[i] = c ? (state[i] == ST_C ? CF_C : CF_F) : CF_COARSEST;
    isC[i] = (c && state[i] == ST_C) ? 1 : 0;
}

__global__ void k_cpts(int n, const int8_t *cf, const int *cidx, int *cpts) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (cf[i] == CF_C) cpts[cidx[i]] = i;
}

__global__ void k_pmap(int n, const int *rowptr, const int *col, const double *val, const uint8_t *S,
                       const unsigned *smask, const int8_t *cf, const int *cidx, int *pmap) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int8_t c = cf[i];
    if (c == CF_COARSEST) { pmap[i] = -1; return; }
    if (c == CF_C) { pmap[i] = cidx[i]; return; }
    int best = -1;
    long long bv = -1;
    for_strong(i, rowptr, S, smask, [&](int p) {
        const int j = col[p];
        if (cf[j] == CF_C) {
            const long long v = absbits(val[p]);
            if (v > bv) { bv = v; best = j; }
        }
        return true;
    });
    pmap[i] = best >= 0 ? cidx[best] : -1;
}

// ---- lAIR ------------------------------------------------------------------
// The pattern of C row i is the set of its strong F neighbours j and, at distance 2,
// of their strong F neighbours, ascending.  Bit 2 of S marks an entry that is eps_R-
// strong with an F column, so the passes below test one byte instead of gathering the
// CF flag of every column (twice), and nf[row] counts a row's marked entries, so the
// candidates of a C row are counted without visiting its neighbours' rows.  Eight lanes
// per row: rows hold 7-16 entries on the fine levels, read as one line.
constexpr uint8_t S_RF = 4;

__global__ void k_mark_rf(int n, const int *rowptr, const int *col, const int8_t *cf, uint8_t *S, int *nf) {
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int i = (int)(tid >> 3), g = (int)(tid & 7);
    int c = 0;
    if (i < n)
        for (int p = rowptr[i] + g; p < rowptr[i + 1]; p += 8) {
            const uint8_t f = S[p];
            if ((f & 2) && cf[col[p]] == CF_F) { S[p] = f | S_RF; ++c; }
        }
    for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (i < n && g == 0) nf[i] = c;
}

// distance 1: the C rows alone are marked and counted (their marked entries are the
// pattern)
__global__ void k_mark_rf1(int nc, const int *cpts, const int *rowptr, const int *col, const int8_t *cf, uint8_t *S,
                           int *ncand) {
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int ic = (int)(tid >> 3), g = (int)(tid & 7);
    int c = 0;
    if (ic < nc) {
        const int i = cpts[ic];
        for (int p = rowptr[i] + g; p < rowptr[i + 1]; p += 8) {
            const uint8_t f = S[p];
            if ((f & 2) && cf[col[p]] == CF_F) { S[p] = f | S_RF; ++c; }
        }
    }
    for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (ic < nc && g == 0) ncand[ic] = c;
}

// distance 2: candidates (with repeats) of every C row.  Rows with more than PAT_BIG of them go to
// the list of the bitmap kernel (any order: a row's pattern has its own place).
constexpr int PAT_SMALL = 64, PAT_MID = 256, PAT_BIG = 1024;

__global__ void k_lair_ncand(int nc, const int *cpts, const int *rowptr, const int *col, const uint8_t *S,
                             const int *nf, int *ncand, int *big, int *nbig) {
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int ic = (int)(tid >> 3), g = (int)(tid & 7);
    int c = 0;
    if (ic < nc) {
        const int i = cpts[ic];
        for (int p = rowptr[i] + g; p < rowptr[i + 1]; p += 8)
            if (S[p] & S_RF) c += 1 + nf[col[p]];
    }
    for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (ic < nc && g == 0) {
        ncand[ic] = c;
        if (c > PAT_BIG) big[atomicAdd(nbig, 1)] = ic;
    }
}

// distance 1: the marked entries of the C row, in order (ncand is then the pattern's
// size); eight lanes per row
__global__ void k_lair_pattern1(int nc, const int *cpts, const int *rowptr, const int *col, const uint8_t *S,
                                const int *candptr, int *cand) {
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int ic = (int)(tid >> 3), g = (int)(tid & 7);
    const int lane = threadIdx.x & 31, sh = lane & ~7;
    int p0 = 0, p1 = 0, out = 0;
    if (ic < nc) {
        const int i = cpts[ic];
        p0 = rowptr[i];
        p1 = rowptr[i + 1];
        out = candptr[ic];
    }
    int len = p1 - p0;
    for (int o = 16; o > 0; o >>= 1) len = max(len, __shfl_xor_sync(0xffffffffu, len, o));
    for (int t = 0; t < len; t += 8) {
        const int p = p0 + t + g;
        const bool in = p < p1 && (S[p] & S_RF);
        const unsigned m = (__ballot_sync(0xffffffffu, in) >> sh) & 0xffu;
        if (in) cand[out + __popc(m & ((1u << g) - 1u))] = col[p];
        out += __popc(m);
    }
}

// distance 2: G lanes per C row with lo < ncand <= hi.  The candidates go into a hash
// table of CAP >= 2 hi slots in shared memory (so it is at most half full), the distinct
// ones are compacted and written at their rank.  A thread per row with an insertion sort
// of its candidates in global memory took O(ncand^2) dependent accesses: 5.3 ms a level on
// an 18^3 x 6 tet matrix (rows of 120 entries, thousands of candidates), where the three
// classes and the bitmap kernel below now take 0.1 ms.  With few candidates (G = 8) a lane
// walks a neighbour's short row; a warp (G = 32) takes the neighbours' rows one after the
// other, lanes across the row.  A warp looks at rb rows' counts together and then takes
// the rows of its class, since most rows of a fine level belong to the smallest class.
template <int G, int CAP, int HI>
__global__ void __launch_bounds__(128) k_lair_pattern2(int nc, const int *cpts, const int *rowptr, const int *col,
                                                       const uint8_t *S, const int *candptr, const int *ncand, int lo,
                                                       int rb, int *cand, int *npat) {
    extern __shared__ int psm[];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, g = lane % G, q = lane / G;
    const int grp = threadIdx.x / G;   // group of the block
    const unsigned gmask = G == 32 ? FULL : (((1u << (G & 31)) - 1u) << (q * G));
    int *keys = psm + grp * (CAP + HI), *list = keys + CAP;
    auto insert = [&](int c) {
        unsigned h = ((unsigned)c * 2654435761u) & (CAP - 1);
        while (true) {   // ends: at most HI <= CAP / 2 distinct columns
            const int prev = atomicCAS(&keys[h], -1, c);
            if (prev == -1 || prev == c) return;
            h = (h + 1) & (CAP - 1);
        }
    };
    // the pattern of row ic (mine: it belongs to the class; whole warps arrive here)
    auto row = [&](int ic, bool mine) {
        for (int t = g; t < CAP; t += G) keys[t] = -1;
        __syncwarp();
        int p0 = 0, p1 = 0;
        if (mine) {
            const int i = cpts[ic];
            p0 = rowptr[i];
            p1 = rowptr[i + 1];
        }
        if (G < 32) {
            for (int p = p0 + g; p < p1; p += G) {
                if (!(S[p] & S_RF)) continue;
                const int j = col[p];
                insert(j);
                const int e = rowptr[j + 1];
                for (int r = rowptr[j]; r < e; r += 4) {   // four entries' loads before their insertions
                    int c[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) c[u] = (r + u < e && (S[r + u] & S_RF)) ? col[r + u] : -1;
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (c[u] >= 0) insert(c[u]);
                }
            }
        } else {
            for (int t = p0; t < p1; t += 32) {
                const int p = t + lane;
                const bool in = p < p1 && (S[p] & S_RF);
                int j = 0, rs = 0, re = 0;
                if (in) {
                    j = col[p];
                    rs = rowptr[j];
                    re = rowptr[j + 1];
                    insert(j);
                }
                for (unsigned b = __ballot_sync(FULL, in); b; b &= b - 1) {
                    const int src = __ffs(b) - 1;
                    const int s0 = __shfl_sync(FULL, rs, src), s1 = __shfl_sync(FULL, re, src);
                    for (int r = s0 + lane; r < s1; r += 32)
                        if (S[r] & S_RF) insert(col[r]);
                }
            }
        }
        __syncwarp();
        int u = 0;
        for (int t0 = 0; t0 < CAP; t0 += G) {
            const int k = keys[t0 + g];
            const unsigned b = __ballot_sync(FULL, k >= 0) & gmask;
            if (k >= 0) list[u + __popc(b & ((1u << lane) - 1u))] = k;
            u += __popc(b);
        }
        __syncwarp();
        if (mine) {
            const int base = candptr[ic];
            for (int e = g; e < u; e += G) {
                const int k = list[e];
                int rank = 0;
                for (int f = 0; f < u; ++f) rank += list[f] < k;
                cand[base + rank] = k;
            }
            if (g == 0) npat[ic] = u;
        }
        __syncwarp();
    };
    if (G < 32) {
        const int ic = blockIdx.x * (128 / G) + grp;
        const int m = ic < nc ? ncand[ic] : HI + 1;
        const bool mine = m <= HI && m >= lo;
        if (__any_sync(FULL, mine)) row(ic, mine);
    } else {
        const long long r0 = (blockIdx.x * 4LL + grp) * rb;
        const int m = (lane < rb && r0 + lane < nc) ? ncand[r0 + lane] : HI + 1;
        for (unsigned b = __ballot_sync(FULL, m <= HI && m >= lo); b; b &= b - 1) row((int)r0 + __ffs(b) - 1, true);
    }
}

// distance 2, rows with more than PAT_BIG candidates: a CTA per row marks the candidates
// in a bitmap of PAT_WIN columns (32 KB of shared memory), whose set bits come out
// ascending and distinct; neighbourhoods spread over more columns take further windows
// over the row's column range.  Grid-stride over the list k_lair_ncand filled.
constexpr int PAT_WIN = 1 << 18;

__global__ void __launch_bounds__(256) k_lair_pattern2_big(const int *big, const int *nbig, const int *cpts,
                                                           const int *rowptr, const int *col, const uint8_t *S,
                                                           const int *candptr, int *cand, int *npat) {
    __shared__ unsigned bits[PAT_WIN / 32];
    __shared__ int red[2][8], wsum[8];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int n = *nbig;
    for (int k = blockIdx.x; k < n; k += gridDim.x) {
        const int ic = big[k], i = cpts[ic], p0 = rowptr[i], p1 = rowptr[i + 1];
        // every candidate to f: a warp per marked neighbour, lanes across its row
        auto visit = [&](auto f) {
            for (int p = p0 + w; p < p1; p += 8) {
                if (!(S[p] & S_RF)) continue;
                const int j = col[p];
                if (lane == 0) f(j);
                for (int r = rowptr[j] + lane; r < rowptr[j + 1]; r += 32)
                    if (S[r] & S_RF) f(col[r]);
            }
        };
        int lo = 0x7fffffff, hi = -1;
        visit([&](int c) { lo = min(lo, c); hi = max(hi, c); });
        for (int o = 16; o > 0; o >>= 1) {
            lo = min(lo, __shfl_xor_sync(FULL, lo, o));
            hi = max(hi, __shfl_xor_sync(FULL, hi, o));
        }
        if (lane == 0) { red[0][w] = lo; red[1][w] = hi; }
        __syncthreads();
        for (int t = 0; t < 8; ++t) { lo = min(lo, red[0][t]); hi = max(hi, red[1][t]); }
        int out = candptr[ic];
        const int out0 = out;
        for (long long c0 = lo; c0 <= hi; c0 += PAT_WIN) {
            const int nw = (int)((min((long long)hi - c0 + 1, (long long)PAT_WIN) + 31) / 32);   // words in use
            const int per = (nw + 255) / 256;                                                    // words per thread
            for (int t = threadIdx.x; t < nw; t += 256) bits[t] = 0u;
            __syncthreads();
            visit([&](int c) {
                const long long d = c - c0;
                if (d >= 0 && d < PAT_WIN) atomicOr(&bits[d >> 5], 1u << (d & 31));
            });
            __syncthreads();
            const int t0 = min((int)threadIdx.x * per, nw), t1 = min(t0 + per, nw);
            int cnt = 0;
            for (int t = t0; t < t1; ++t) cnt += __popc(bits[t]);
            int inc = cnt;
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(FULL, inc, o);
                if (lane >= o) inc += v;
            }
            if (lane == 31) wsum[w] = inc;
            __syncthreads();
            int before = inc - cnt, tot = 0;
            for (int t = 0; t < 8; ++t) {
                if (t < w) before += wsum[t];
                tot += wsum[t];
            }
            int at = out + before;
            for (int t = t0; t < t1; ++t)
                for (unsigned b = bits[t]; b; b &= b - 1) cand[at++] = (int)(c0 + 32LL * t) + __ffs(b) - 1;
            out += tot;
            __syncthreads();   // bits, wsum and red are written again
        }
        if (threadIdx.x == 0) npat[ic] = out - out0;
        __syncthreads();
    }
}

// lAIR systems binned by size, 4, 8, 16 or 32 lanes to a system of up to 8, 16, 32 or 64
// unknowns, with shared workspaces sized to the bin (the smaller they are, the more
// systems are in flight per SM); global workspaces beyond 64, and a dense kernel past 256
constexpr int LAIR_CLASSES = 12;
constexpr int LAIR_BIG = LAIR_CLASSES - 1, LAIR_SLOT = LAIR_BIG - 2;   // dense; first class with global slots
__device__ __forceinline__ int lair_class(int np) {
    return np <= 4 ? 0 : np <= 6 ? 1 : np <= 8 ? 2 : np <= 12 ? 3 : np <= 16 ? 4 : np <= 24 ? 5 : np <= 32 ? 6
         : np <= 48 ? 7 : np <= 64 ? 8 : np <= 128 ? 9 : np <= 256 ? 10 : 11;
}



// Warp per C row.  Shared memory per warp: M (nmax^2 doubles), y (nmax
// doubles), pattern (nmax ints), pivots (nmax ints).
__device__ __forceinline__ int pat_find(const int *pat, int np, int k) {
    int lo = 0, hi = np - 1;
    while (lo <= hi) {
        int m = (lo + hi) >> 1;
        int v = pat[m];
        if (v == k) return m;
        if (v < k) lo = m + 1; else hi = m - 1;
    }
    return -1;
}

// A caller's matrix may repeat a column within a row (its entries ascend, so the repeats
// are neighbours).  Products and strength take every entry; a local system takes the last.
__device__ __forceinline__ bool last_of_run(int p, int p1, const int *col) { return p + 1 >= p1 || col[p + 1] != col[p]; }

// f(p) for the marked entries (S_RF) of the run of one column that holds the marked entry
// p, in order, by the lane of the first of them (lanes of a group hold neighbouring
// entries, and only one may touch the column's unknown)
template <class F>
__device__ __forceinline__ void marked_run(int p, int p0, int p1, const int *col, const uint8_t *S, F &&f) {
    const int c = col[p];
    for (int q = p - 1; q >= p0 && col[q] == c; --q)
        if (S[q] & S_RF) return;
    f(p);
    for (int q = p + 1; q < p1 && col[q] == c; ++q)
        if (S[q] & S_RF) f(q);
}

// ---- nAIR of degree 1 (Neumann series cut after the linear term) -----------
// On the distance-2 pattern (sorted, from k_lair_pattern2):
//   t_k = a_ik for strong F neighbours k of i (else 0); for every strong F
//   neighbour j of i (ascending) and every strong F neighbour k of j
//   (ascending): t_k = fma(a_ij, n_jk, t_k), n_jk = -(a_jk * (1/a_jj));
//   z_k = -(t_k * (1/a_kk)), i.e. Z_i = -A_CF^s[i,:] (I + N) D^{-1} with
//   N = I - D^{-1} A_FF^s.  A zero diagonal on the way empties the row (counted
//   as singular).
// Eight lanes per C row: lanes across a neighbour's row (one lane takes all entries of a
// column, so each t_k takes its terms in the row's order), pattern and t in shared memory up to
// NAIR_SH unknowns, in the row's slots of cand and zval beyond.  (A thread per row that searched and
// accumulated in global memory took 1.6 ms a level on 27^3, 8 directions.)
constexpr int NAIR_SH = 96;

__global__ void __launch_bounds__(128) k_nair(int nc, const int *cpts, const int *rowptr, const int *col,
                                              const double *val, const uint8_t *S, const double *dinv,
                                              const int *candptr, const int *cand, const int *npat,
                                              const int *zrowptr, int *zcol, double *zval, int *keep, int *nsing_dir,
                                              const int *rowdir, double phi_R) {
    __shared__ double tsh[16][NAIR_SH];
    __shared__ int psh[16][NAIR_SH];
    const unsigned FULL = 0xffffffffu;
    const int grp = threadIdx.x >> 3, lane = threadIdx.x & 31, g = lane & 7, q0 = lane & ~7;
    const int ic = blockIdx.x * 16 + grp;
    const bool has = ic < nc;
    const int i = has ? cpts[ic] : 0, np = has ? npat[ic] : 0;
    const int base = has ? zrowptr[ic] : 0;
    const int *cp = has ? cand + candptr[ic] : nullptr;
    const bool sh = np <= NAIR_SH;
    double *t = sh ? tsh[grp] : zval + base;
    const int *pat = sh ? psh[grp] : cp;
    for (int e = g; e < np; e += 8) {
        t[e] = 0.0;
        if (sh) psh[grp][e] = cp[e];
    }
    __syncwarp();
    const int p0 = has ? rowptr[i] : 0, p1 = has ? rowptr[i + 1] : 0;
    for (int p = p0 + g; p < p1; p += 8)
        if (S[p] & S_RF)
            marked_run(p, p0, p1, col, S, [&](int q) { t[pat_find(pat, np, col[q])] = val[q]; });
    __syncwarp();
    bool singular = false;
    int len = p1 - p0;
    for (int o = 16; o > 0; o >>= 1) len = max(len, __shfl_xor_sync(FULL, len, o));
    for (int c0 = 0; c0 < len; c0 += 8) {
        const int p = p0 + c0 + g;
        const bool in = p < p1 && (S[p] & S_RF);
        const int j = in ? col[p] : 0;
        const double aij = in ? val[p] : 0.0, rj = in ? dinv[j] : 0.0;
        const int js = in ? rowptr[j] : 0, je = in ? rowptr[j + 1] : 0;
        if (in && rj == 0.0) singular = true;
        unsigned m = (__ballot_sync(FULL, in) >> q0) & 0xffu;   // the group's neighbours of this pass
        while (__any_sync(FULL, m != 0)) {
            const int src = q0 + (m ? __ffs(m) - 1 : 0);
            const double a = __shfl_sync(FULL, aij, src), r = __shfl_sync(FULL, rj, src);
            const int s0 = __shfl_sync(FULL, js, src), s1 = __shfl_sync(FULL, je, src);
            if (m)
                for (int q = s0 + g; q < s1; q += 8) {
                    if (!(S[q] & S_RF)) continue;
                    const int e = pat_find(pat, np, col[q]);
                    marked_run(q, s0, s1, col, S, [&](int k) { t[e] = fma(a, -(val[k] * r), t[e]); });
                }
            __syncwarp();
            m &= m - 1;
        }
    }
    for (int e = g; e < np; e += 8)
        if (dinv[pat[e]] == 0.0) singular = true;
    singular = ((__ballot_sync(FULL, singular) >> q0) & 0xffu) != 0;
    long long zmb = 0;
    if (!singular)
        for (int e = g; e < np; e += 8) {
            const double z = -(t[e] * dinv[pat[e]]);
            t[e] = z;
            zmb = max(zmb, absbits(z));
        }
    for (int o = 4; o > 0; o >>= 1) zmb = max(zmb, __shfl_xor_sync(FULL, zmb, o, 8));
    const double thr = phi_R * __longlong_as_double(zmb);
    __syncwarp();
    int kept = 0, npm = np;
    for (int o = 16; o > 0; o >>= 1) npm = max(npm, __shfl_xor_sync(FULL, npm, o));
    for (int e0 = 0; e0 < npm; e0 += 8) {
        const int e = e0 + g;
        const double z = e < np ? t[e] : 0.0;
        const bool k_ = e < np && !singular && !(phi_R > 0.0 && fabs(z) < thr);
        const unsigned b = (__ballot_sync(FULL, k_) >> q0) & 0xffu;
        __syncwarp();   // t of this pass is read before zval, which may be its place, is written
        if (k_) {
            const int off = base + kept + __popc(b & ((1u << g) - 1u));
            zcol[off] = pat[e];
            zval[off] = z;
        }
        kept += __popc(b);
    }
    if (has && g == 0) {
        if (singular) atomicAdd(&nsing_dir[rowdir[i]], 1);
        keep[ic] = kept;
    }
}


// 1 / p for a pivot p.  A pivot of magnitude 1 (the unit diagonal of the
// block-scaled level 0, which most eliminations leave untouched) is its own
// reciprocal, exactly, so it takes no division: an FP64 division occupies the FP64
// pipe for a whole warp instruction however few lanes take part, and one per pivot
// was most of the FP64 work left once zero-multiplier rows are skipped.
__device__ __forceinline__ double pivot_recip(double p) {
    const long long mag = __double_as_longlong(p) & 0x7fffffffffffffffLL;   // |p| == 1, integer test
    return mag == 0x3ff0000000000000LL ? p : 1.0 / p;
}

// The FP64 pipe takes a whole warp instruction for any number of active lanes, so
// the O(n^2) passes of the local solves keep their zero tests and signed zeros on
// the integer pipe.
__device__ __forceinline__ bool is_zero_bits(double x) { return (__double_as_longlong(x) & 0x7fffffffffffffffLL) == 0; }
// a * r for a zero a and a finite nonzero r: the zero with the product's sign
__device__ __forceinline__ double zero_times(double a, double r) {
    return __longlong_as_double((__double_as_longlong(a) ^ __double_as_longlong(r)) & (long long)0x8000000000000000ULL);
}
// y * r for a reciprocal r of magnitude 1 (unit pivot): exact sign flip or y itself
__device__ __forceinline__ double times_recip(double y, double r) {
    const long long rb = __double_as_longlong(r);
    if ((rb & 0x7fffffffffffffffLL) == 0x3ff0000000000000LL)
        return __longlong_as_double(__double_as_longlong(y) ^ (rb & (long long)0x8000000000000000ULL));
    return y * r;
}

// Systems past the mask kernels' largest: a warp per system, dense, workspace at
// gbuf + goff[w].
__global__ void k_lair_solve_dense(int nwork, const int *worklist, const int *cpts, const int *rowptr, const int *col,
                             const double *val, const int *candptr, const int *cand, const int *npat,
                             const int *zrowptr, int *zcol, double *zval, int *keep, int *nsing_dir,
                                   const int *rowdir, double phi_R, const long long *goff, double *gbuf) {
    constexpr int G = 32;
    const unsigned FULL = 0xffffffffu;
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int g = lane % G, q = lane / G;
    int wpb = blockDim.x >> 5;
    constexpr int SPW = 32 / G;   // systems per warp
    const unsigned gmask = (G == 32) ? FULL : (((1u << (G & 31)) - 1u) << (q * G));   // this group's lanes
    for (int wb = (blockIdx.x * wpb + warp) * SPW; wb < nwork; wb += gridDim.x * wpb * SPW) {
        int w = wb + q;
        bool has = w < nwork;
        int ic = has ? worklist[w] : 0;
        int i = has ? cpts[ic] : 0;
        int np = has ? npat[ic] : 0;
        double *M = gbuf + (has ? goff[w] : 0);
        double *y = M + (size_t)np * np;
        double *rv = y + np;                  // pivot reciprocals
        int *pat = (int *)(rv + np);
        int *piv = pat + np;
        int *rl = piv + np;                   // rows below the pivot with a nonzero multiplier
        if (has) {
            const int *cp = cand + candptr[ic];
            for (int t = g; t < np; t += G) { pat[t] = cp[t]; y[t] = -0.0; }
            for (int idx = g; idx < np * np; idx += G) M[idx] = 0.0;
        }
        __syncwarp();
        if (has) {
            // M[r][c] = a(pat[c], pat[r]): lane per pattern row, one pass over it, the
            // loads of four entries issued before their lookups
            for (int c = g; c < np; c += G) {
                const int j = pat[c], p1 = rowptr[j + 1];
                for (int p = rowptr[j]; p < p1; p += 4) {
                    int cc[4];
                    double vv[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        cc[u] = p + u < p1 ? col[p + u] : -1;
                        vv[u] = p + u < p1 ? val[p + u] : 0.0;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (cc[u] < 0) continue;
                        const int r = pat_find(pat, np, cc[u]);
                        if (r >= 0) M[r * np + c] = vv[u];
                    }
                }
            }
            for (int p = rowptr[i] + g; p < rowptr[i + 1]; p += G) {
                int r = pat_find(pat, np, col[p]);
                if (r >= 0 && last_of_run(p, rowptr[i + 1], col)) y[r] = -val[p];
            }
        }
        __syncwarp();
        long long mxb = 0;
        for (int idx = g; idx < np * np; idx += G) mxb = max(mxb, absbits(M[idx]));
        for (int o = G / 2; o > 0; o >>= 1) mxb = max(mxb, __shfl_xor_sync(FULL, mxb, o, G));
        long long tinyb = absbits(1e-14 * __longlong_as_double(mxb));
        int kmax = np;
        for (int o = 16; o > 0; o >>= 1) kmax = max(kmax, __shfl_xor_sync(FULL, kmax, o));
        bool singular = false;
        for (int k = 0; k < kmax; ++k) {
            bool act = k < np && !singular;
            long long bv = -1;
            int br = k;
            bool nzb = false;   // a nonzero below the diagonal among this lane's rows
            if (act)
                for (int r = k + g; r < np; r += G) {
                    long long v = absbits(M[r * np + k]);
                    if (r > k && v != 0) nzb = true;
                    if (v > bv) { bv = v; br = r; }
                }
            // Most columns have nothing below the diagonal: when no group of the warp has,
            // every pivot stays on the diagonal (the only candidate that is not zero,
            // held by the group's first lane) and the step has no multipliers to compute
            // and nothing to update.
            const bool any_nz = __ballot_sync(FULL, nzb) != 0u;
            if (any_nz) {
                for (int o = G / 2; o > 0; o >>= 1) {
                    long long ov = __shfl_xor_sync(FULL, bv, o, G);
                    int orr = __shfl_xor_sync(FULL, br, o, G);
                    if (ov > bv || (ov == bv && orr < br)) { bv = ov; br = orr; }
                }
            } else {
                bv = __shfl_sync(FULL, bv, q * G);
                br = k;
            }
            if (act && !(bv > tinyb)) { singular = true; act = false; }
            if (act) {
                if (g == 0) piv[k] = br;
                if (br != k)
                    for (int c = g; c < np; c += G) {
                        double t = M[k * np + c];
                        M[k * np + c] = M[br * np + c];
                        M[br * np + c] = t;
                    }
            }
            __syncwarp();
            // multipliers, and the list of rows whose multiplier is not zero: a zero
            // multiplier's update adds exact zeros, so those rows are skipped, as in the
            // reference LU (in the local systems of these operators most multipliers are
            // zero).  The bound on the rows below the pivot is uniform over the warp, so
            // every lane reaches each ballot.
            // (a zero entry's multiplier is the signed zero a * rd gives, set with
            // integer operations; the others are computed for the listed rows only)
            int m = 0;
            if (!any_nz) {
                // only zeros below: their multipliers are those zeros, with the sign
                // flipped under a negative pivot (the sign of 1 / pivot, so no division
                // here: the reciprocals of such pivots are taken together after the
                // elimination)
                const double pk = act ? M[k * np + k] : 0.0;   // k < np only for an active group
                if (act && __double_as_longlong(pk) < 0)
                    for (int r = k + 1 + g; r < np; r += G) M[r * np + k] = zero_times(M[r * np + k], pk);
                __syncwarp();
                continue;
            }
            // the pivot's reciprocal: one lane of the group divides, the others take it
            double rd = 0.0;
            if (act && g == 0) rd = pivot_recip(M[k * np + k]);
            rd = __shfl_sync(FULL, rd, q * G);
            for (int j0 = 0; j0 < kmax - k - 1; j0 += G) {
                const int r = k + 1 + j0 + g;
                bool nzr = false;
                if (act && r < np) {
                    const double a = M[r * np + k];
                    nzr = !is_zero_bits(a);
                    if (!nzr) M[r * np + k] = zero_times(a, rd);
                }
                const unsigned msk = __ballot_sync(FULL, nzr) & gmask;
                if (nzr) rl[m + __popc(msk & ((1u << lane) - 1u))] = r;
                m += __popc(msk);
            }
            __syncwarp();
            if (act)
                for (int t = g; t < m; t += G) {
                    const double l = M[rl[t] * np + k] * rd;
                    M[rl[t] * np + k] = l;
                    if (is_zero_bits(l)) rl[t] = -1;   // underflowed to zero: skipped too
                }
            __syncwarp();
            if (act) {
                // lane g updates entries g, g + G, ... of the m x wd block (listed rows,
                // trailing columns) in row-major order (the fewest FP64 instructions:
                // every lane busy until the last entries), four entries per pass with all
                // their loads issued before the updates; (list index, column) advance by
                // (G / wd, G % wd) per entry with at most one carry, so no division per
                // entry
                const int wd = np - k - 1;
                if (wd > 0 && m > 0) {
                    const int tot = m * wd;
                    const int dr = G / wd, dc = G - dr * wd;
                    int r = g / wd, c = g - r * wd;
                    for (int e = g; e < tot; e += 4 * G) {
                        int Ro[4], Co[4];
                        bool ok[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int rr = e + u * G < tot ? rl[r] : -1;
                            ok[u] = rr >= 0;
                            Ro[u] = ok[u] ? rr * np : 0;
                            Co[u] = k + 1 + c;
                            r += dr;
                            c += dc;
                            if (c >= wd) { c -= wd; ++r; }
                        }
                        double a[4], b[4], mv[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (ok[u]) { a[u] = M[Ro[u] + k]; b[u] = M[k * np + Co[u]]; mv[u] = M[Ro[u] + Co[u]]; }
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (ok[u]) M[Ro[u] + Co[u]] = fma(-a[u], b[u], mv[u]);
                    }
                }
            }
            __syncwarp();
        }
        bool solve = has && !singular && np > 0;
        // every pivot's reciprocal for the back substitution, G at a time (the same
        // values the elimination took for its multipliers)
        if (solve)
            for (int k = g; k < np; k += G) rv[k] = pivot_recip(M[k * np + k]);
        if (solve && g == 0)
            for (int k = 0; k < np; ++k)
                if (piv[k] != k) { double t = y[k]; y[k] = y[piv[k]]; y[piv[k]] = t; }
        __syncwarp();
        for (int k = 0; k < kmax; ++k) {
            if (solve && k < np) {
                double yk = y[k];
                for (int r = k + 1 + g; r < np; r += G) y[r] = fma(-M[r * np + k], yk, y[r]);
            }
            __syncwarp();
        }
        for (int k = kmax - 1; k >= 0; --k) {
            if (solve && k < np && g == 0) y[k] = times_recip(y[k], rv[k]);
            __syncwarp();
            if (solve && k < np) {
                double yk = y[k];
                for (int r = g; r < k; r += G) y[r] = fma(-M[r * np + k], yk, y[r]);
            }
            __syncwarp();
        }
        long long zmb = 0;
        if (solve)
            for (int t = g; t < np; t += G) zmb = max(zmb, absbits(y[t]));
        for (int o = G / 2; o > 0; o >>= 1) zmb = max(zmb, __shfl_xor_sync(FULL, zmb, o, G));
        double thr = phi_R * __longlong_as_double(zmb);
        int kept = 0;
        int base = has ? zrowptr[ic] : 0;
        int tmax = np;
        for (int o = 16; o > 0; o >>= 1) tmax = max(tmax, __shfl_xor_sync(FULL, tmax, o));
        // keep in ascending order: ballot-compacted write within the group
        for (int t0 = 0; t0 < tmax; t0 += G) {
            int t = t0 + g;
            bool k_ = solve && t < np && !(phi_R > 0.0 && fabs(y[t]) < thr);
            unsigned msk = __ballot_sync(FULL, k_) & gmask;
            if (k_) {
                int off = kept + __popc(msk & ((1u << lane) - 1u));
                zcol[base + off] = pat[t];
                zval[base + off] = y[t];
            }
            kept += __popc(msk);
        }
        if (has && g == 0) {
            if (singular) atomicAdd(&nsing_dir[rowdir[i]], 1);
            keep[ic] = solve ? kept : 0;
        }
        __syncwarp();
    }
}

// Systems of up to 256 unknowns on column masks.  G lanes take a system (32 / G systems a
// warp), lane g the columns g, g + G, ... and the same entries of y; cm holds, per column,
// the rows that may be nonzero.  The local matrices are A_FF restricted to a neighbourhood
// of an upwind operator: a few entries per row, almost nothing below the diagonal, so with
// the masks a pivot step whose column has no row below costs a shuffle of its mask instead
// of a scan of the column, and elimination, fill-in and both substitutions touch stored
// entries only.  Entries outside the masks are never read (the workspace is not cleared)
// and stand for +0.0; forward substitution runs with the elimination, so L is not kept.
//
// The results are those of the dense elimination bit for bit.  What a dense pass does with
// a zero is kept: a zero multiplier takes the sign of the pivot, and y - 0 * y_k changes
// only the sign of a zero y (-0.0 becomes +0.0 when the product is +0.0), unless y_k is
// not finite.  (Partial pivoting keeps multipliers at most 1 in magnitude, and a system
// that holds an infinity or a NaN fails its first pivot test, so the update of an unstored
// entry is always a zero.)
//
// Measured against the dense kernels (a thread a system up to 8 unknowns, 8 to 32 lanes on
// cleared workspaces beyond): 64^3 S8 1311 -> 1232 ms (79 of 210 ms of local solves; the
// three smallest bins alone 41 ms), an 18^3 x 6 tet matrix 29.6 -> 25.6 ms; with the bins
// past 64 unknowns and blocks small enough to fill an SM, 40^3 x 6 tets S4 537 -> 507 ms.
// What bounds it: each FP64 warp instruction holds the SM's FP64 pipe for 16 cycles
// whatever its active lanes, and the dense passes issued one per column, row and step; the
// workspaces (odd row stride: columns are read without bank conflicts) set the resident
// warps.
__device__ __forceinline__ double sub_zero_product(double y, bool neg_zero_factor, double yk) {
    // y - z * yk for a zero z (negative: neg_zero_factor)
    const long long kb = __double_as_longlong(yk);
    if ((kb & 0x7ff0000000000000LL) == 0x7ff0000000000000LL) return fma(neg_zero_factor ? 0.0 : -0.0, yk, y);
    const bool plus = neg_zero_factor != (kb < 0);   // the product -z * yk is +0.0
    return (plus && __double_as_longlong(y) == (long long)0x8000000000000000ULL) ? 0.0 : y;
}

// W words of row bits; bit indices are per lane or uniform, word indices constants
template <int W>
struct RowMask {
    unsigned long long w[W];
    __device__ __forceinline__ bool has(int r) const {
        if (W == 1) return (w[0] >> r) & 1ULL;
        bool b = false;
#pragma unroll
        for (int k = 0; k < W; ++k)
            if ((r >> 6) == k) b = (w[k] >> (r & 63)) & 1ULL;
        return b;
    }
    __device__ __forceinline__ void set(int r) {
#pragma unroll
        for (int k = 0; k < W; ++k)
            if (W == 1 || (r >> 6) == k) w[k] |= 1ULL << (r & 63);
    }
    __device__ __forceinline__ void flip(int r) {
#pragma unroll
        for (int k = 0; k < W; ++k)
            if (W == 1 || (r >> 6) == k) w[k] ^= 1ULL << (r & 63);
    }
    // a row past r
    __device__ __forceinline__ bool any_past(int r) const {
        bool b = false;
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const unsigned long long m = (r >> 6) == k ? w[k] & ~((2ULL << (r & 63)) - 1ULL) : (r >> 6) < k ? w[k] : 0ULL;
            b |= m != 0;
        }
        return b;
    }
};

// column k's mask, to every lane of its group (first lane q0)
template <int G, int R, int W>
__device__ __forceinline__ RowMask<W> mask_column(const RowMask<W> (&cm)[R], int k, int q0) {
    RowMask<W> x;
#pragma unroll
    for (int j = 0; j < W; ++j) {
        unsigned long long v = cm[0].w[j];
#pragma unroll
        for (int t = 1; t < R; ++t) {
            const unsigned long long u = cm[t].w[j];
            v = k / G == t ? u : v;
        }
        x.w[j] = __shfl_sync(0xffffffffu, v, q0 + (k & (G - 1)));
    }
    return x;
}

// G lanes, R columns a lane: systems of up to G R unknowns.  GLOBAL: the workspace is a
// slot of gbuf per warp (systems of more than 64 unknowns; nothing is cleared and little is
// touched, so the slots in use stay in L2), else shared memory.  M is column-major: a
// column's rows are read by consecutive lanes.
template <int G, int R, bool GLOBAL>
__global__ void k_lair_solve_mask(int nwork, const int *worklist, const int *cpts, const int *rowptr, const int *col,
                                  const double *val, const int *candptr, const int *cand, const int *npat,
                                  const int *zrowptr, int *zcol, double *zval, int *keep, int *nsing_dir,
                                  const int *rowdir, double phi_R, int nmax, double *gbuf) {
    typedef unsigned long long u64;
    constexpr int PN = R * G;     // pattern slots: a power of two >= nmax
    constexpr int SPW = 32 / G;   // systems per warp
    constexpr int W = (PN + 63) / 64;
    extern __shared__ double smem[];
    const unsigned FULL = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    const int g = lane % G, q = lane / G, q0 = q * G;
    const unsigned gmask = G == 32 ? FULL : ((1u << (G & 31)) - 1u);   // (shifted down to the group)
    const int ld = nmax | 1;
    const size_t msz = (size_t)nmax * ld;
    double *ws = smem + ((size_t)warp * SPW + q) * ((GLOBAL ? 0 : msz) + nmax + PN / 2);
    double *M = GLOBAL ? gbuf + ((size_t)blockIdx.x * wpb + warp) * msz : ws;
    double *ys = ws + (GLOBAL ? 0 : msz);
    int *pat = (int *)(ys + nmax);
    auto find = [&](int k) {   // position of column k in the pattern, or -1
        int pos = 0;
#pragma unroll
        for (int h = PN / 2; h > 0; h >>= 1)
            if (pat[pos + h - 1] < k) pos += h;
        return pat[pos] == k ? pos : -1;
    };
    auto bcast = [&](const double (&v)[R], int k) {
        double x = v[0];
#pragma unroll
        for (int t = 1; t < R; ++t) {
            const double u = v[t];
            x = k / G == t ? u : x;
        }
        return __shfl_sync(FULL, x, q0 + (k & (G - 1)));
    };
    for (int wb = (blockIdx.x * wpb + warp) * SPW; wb < nwork; wb += gridDim.x * wpb * SPW) {
        const int w = wb + q;
        const bool has = w < nwork;
        const int ic = has ? worklist[w] : 0;
        const int i = has ? cpts[ic] : 0;
        const int np = has ? npat[ic] : 0;
        const int *cp = has ? cand + candptr[ic] : nullptr;
#pragma unroll
        for (int t = 0; t < R; ++t) {
            const int c = g + G * t;
            pat[c] = c < np ? cp[c] : 0x7fffffff;
            if (c < np) ys[c] = -0.0;
        }
        __syncwarp();
        // column c of the system is row pat[c] of A: four entries' loads before their lookups
        RowMask<W> cm[R];
        long long mxb = 0;
#pragma unroll
        for (int t = 0; t < R; ++t) {
            RowMask<W> x;
#pragma unroll
            for (int k = 0; k < W; ++k) x.w[k] = 0;
            const int c = g + G * t, j = c < np ? pat[c] : 0, p1 = c < np ? rowptr[j + 1] : 0;
            int last = -1;
            bool repeats = false;
            long long cmax = 0;
            for (int p = c < np ? rowptr[j] : 0; p < p1; p += 4) {
                int cc[4], r[4];
                double vv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    cc[u] = p + u < p1 ? col[p + u] : -1;
                    vv[u] = p + u < p1 ? val[p + u] : 0.0;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    r[u] = find(cc[u]);
                    repeats |= r[u] >= 0 && r[u] == last;
                    last = r[u];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (r[u] >= 0) {
                        M[(size_t)c * ld + r[u]] = vv[u];
                        x.set(r[u]);
                        cmax = max(cmax, absbits(vv[u]));
                    }
            }
            if (repeats) {   // the last value of a repeated column stands (see last_of_run)
                cmax = 0;
                for (int r = 0; r < np; ++r)
                    if (x.has(r)) cmax = max(cmax, absbits(M[(size_t)c * ld + r]));
            }
            mxb = max(mxb, cmax);
            cm[t] = x;
        }
        if (has)
            for (int p = rowptr[i] + g; p < rowptr[i + 1]; p += G) {
                const int r = find(col[p]);
                if (r >= 0 && last_of_run(p, rowptr[i + 1], col)) ys[r] = -val[p];
            }
        __syncwarp();
        double y[R];
#pragma unroll
        for (int t = 0; t < R; ++t) y[t] = g + G * t < np ? ys[g + G * t] : 0.0;
        int kmax = np;
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) mxb = max(mxb, __shfl_xor_sync(FULL, mxb, o, G));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) kmax = max(kmax, __shfl_xor_sync(FULL, kmax, o));
        const long long tinyb = absbits(1e-14 * __longlong_as_double(mxb));
        // reciprocals of the diagonal as gathered, all at once: a division holds the FP64 pipe
        // for a hundred cycles and more however few lanes take part, and most rows reach
        // their pivot step unchanged, so one per step and one per row again at the end was
        // much of the pipe's work on the levels without a unit diagonal
        double d0[R], rv[R];
#pragma unroll
        for (int t = 0; t < R; ++t) {
            const int c = g + G * t;
            d0[t] = c < np && cm[t].has(c) ? M[(size_t)c * ld + c] : 1.0;
            rv[t] = pivot_recip(d0[t]);
        }
        bool singular = false;
        for (int k = 0; k < kmax; ++k) {
            bool act = k < np && !singular;
            RowMask<W> mk = mask_column<G, R, W>(cm, k, q0);
            double *Mk = M + (size_t)k * ld;
            double pk = act && mk.has(k) ? Mk[k] : 0.0;
            const bool need = act && mk.any_past(k);
            long long bv = absbits(pk);
            int br = k;
            const bool step = __any_sync(FULL, need);
            if (step) {   // pivot: the first largest magnitude of rows k.. (unstored rows are zero)
                if (need) {
                    bv = -1;
#pragma unroll
                    for (int t = 0; t < R; ++t) {
                        const int r = g + G * t;
                        if (r < k || r >= np) continue;
                        const long long v = mk.has(r) ? absbits(Mk[r]) : 0;
                        if (v > bv) { bv = v; br = r; }
                    }
                }
#pragma unroll
                for (int o = G / 2; o > 0; o >>= 1) {
                    const long long ov = __shfl_xor_sync(FULL, bv, o, G);
                    const int orr = __shfl_xor_sync(FULL, br, o, G);
                    if (ov > bv || (ov == bv && orr < br)) { bv = ov; br = orr; }
                }
            }
            if (act && !(bv > tinyb)) { singular = true; act = false; }
            const bool elim = act && need;
            if (step) {
                const bool swp = elim && br != k;
                if (__any_sync(FULL, swp)) {
                    const double yk0 = bcast(y, k);
                    double yb = 0.0;
#pragma unroll
                    for (int t = 0; t < R; ++t) {
                        const double x = __shfl_sync(FULL, y[t], q0 + (br & (G - 1)));
                        if (br / G == t) yb = x;
                    }
                    if (swp) {
#pragma unroll
                        for (int t = 0; t < R; ++t) {
                            const int c = g + G * t;
                            if (c < np) {
                                double *Mc = M + (size_t)c * ld;
                                const double tv = Mc[k];
                                Mc[k] = Mc[br];
                                Mc[br] = tv;
                            }
                            if (c == k) y[t] = yb;
                            else if (c == br) y[t] = yk0;
                            if (cm[t].has(k) != cm[t].has(br)) { cm[t].flip(k); cm[t].flip(br); }
                        }
                        if (mk.has(k) != mk.has(br)) { mk.flip(k); mk.flip(br); }
                    }
                    __syncwarp();
                    if (swp) pk = Mk[k];
                }
            }
            const double yk = bcast(y, k);
            const bool negp = __double_as_longlong(pk) < 0;   // the sign of a zero multiplier
            if (!step) {
                if (act)
#pragma unroll
                    for (int t = 0; t < R; ++t)
                        if (g + G * t > k) y[t] = sub_zero_product(y[t], negp, yk);
                continue;
            }
            // the pivot's reciprocal: one lane of the group divides if the pivot has changed
            double rd = bcast(rv, k);
            const double dk = bcast(d0, k);   // (every lane takes part in the broadcasts)
            const bool redo = elim && __double_as_longlong(pk) != __double_as_longlong(dk);
            if (__any_sync(FULL, redo)) {
                double r1 = rd;
                if (redo && g == 0) r1 = pivot_recip(pk);
                rd = __shfl_sync(FULL, r1, q0);
            }
            RowMask<W> Lm;   // rows whose multiplier is not zero
#pragma unroll
            for (int j = 0; j < W; ++j) Lm.w[j] = 0;
            double l[R];
#pragma unroll
            for (int t = 0; t < R; ++t) {
                const int r = g + G * t;
                const bool inb = elim && r > k && mk.has(r);
                const double a = inb ? Mk[r] : 0.0;
                const bool nz = inb && !is_zero_bits(a);
                l[t] = nz ? a * rd : 0.0;
                const bool upd = nz && !is_zero_bits(l[t]);
                if (act && r > k) {
                    if (upd) y[t] = fma(-l[t], yk, y[t]);
                    else {
                        // zero multiplier: zero entry times the reciprocal, or an underflow
                        const bool neg = nz ? __double_as_longlong(l[t]) < 0 : (__double_as_longlong(a) < 0) != negp;
                        y[t] = sub_zero_product(y[t], neg, yk);
                    }
                }
                const unsigned b = (__ballot_sync(FULL, upd) >> q0) & gmask;
                Lm.w[G * t / 64] |= (u64)b << (G * t % 64);
            }
#pragma unroll
            for (int j = 0; j < W; ++j) {
                u64 rem = Lm.w[j];
                while (__any_sync(FULL, rem != 0)) {
                    const int r = 64 * j + (rem ? __ffsll((long long)rem) - 1 : 0);
                    double lr = 0.0;
#pragma unroll
                    for (int t = 0; t < R; ++t) {
                        if (W > 1 && G * t / 64 != j) continue;
                        const double x = __shfl_sync(FULL, l[t], q0 + (r & (G - 1)));
                        if (r / G == t) lr = x;
                    }
                    if (rem) {
#pragma unroll
                        for (int t = 0; t < R; ++t) {
                            const int c = g + G * t;
                            const bool bk = cm[t].has(k), brr = cm[t].has(r);
                            if (c > k && c < np && (bk || brr)) {
                                double *Mc = M + (size_t)c * ld;
                                const double mv = brr ? Mc[r] : 0.0, bkv = bk ? Mc[k] : 0.0;
                                Mc[r] = fma(-lr, bkv, mv);
                            }
                        }
                    }
                    rem &= rem - 1;
                }
            }
#pragma unroll
            for (int t = 0; t < R; ++t)
                if (g + G * t > k && cm[t].has(k)) {
#pragma unroll
                    for (int j = 0; j < W; ++j) cm[t].w[j] |= Lm.w[j];
                }
            __syncwarp();
        }
        const bool solve = has && !singular && np > 0;
#pragma unroll
        for (int t = 0; t < R; ++t) {
            const int c = g + G * t;
            const double p = solve && c < np ? M[(size_t)c * ld + c] : d0[t];
            if (__double_as_longlong(p) != __double_as_longlong(d0[t])) rv[t] = pivot_recip(p);
        }
        for (int k = kmax - 1; k >= 0; --k) {
            const bool act = solve && k < np;
            const RowMask<W> mk = mask_column<G, R, W>(cm, k, q0);
#pragma unroll
            for (int t = 0; t < R; ++t)
                if (act && g + G * t == k) y[t] = times_recip(y[t], rv[t]);
            const double yk = bcast(y, k);
            if (act)
#pragma unroll
                for (int t = 0; t < R; ++t) {
                    const int r = g + G * t;
                    if (r >= k) continue;
                    if (mk.has(r)) y[t] = fma(-M[(size_t)k * ld + r], yk, y[t]);
                    else y[t] = sub_zero_product(y[t], false, yk);
                }
        }
        long long zmb = 0;
#pragma unroll
        for (int t = 0; t < R; ++t)
            if (solve && g + G * t < np) zmb = max(zmb, absbits(y[t]));
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) zmb = max(zmb, __shfl_xor_sync(FULL, zmb, o, G));
        const double thr = phi_R * __longlong_as_double(zmb);
        const int base = has ? zrowptr[ic] : 0;
        int kept = 0;
#pragma unroll
        for (int t = 0; t < R; ++t) {
            const int c = g + G * t;
            const bool k_ = solve && c < np && !(phi_R > 0.0 && fabs(y[t]) < thr);
            const unsigned b = (__ballot_sync(FULL, k_) >> q0) & gmask;
            if (k_) {
                const int off = kept + __popc(b & ((1u << g) - 1u));
                zcol[base + off] = pat[c];
                zval[base + off] = y[t];
            }
            kept += __popc(b);
        }
        if (has && g == 0) {
            if (singular) atomicAdd(&nsing_dir[rowdir[i]], 1);
            keep[ic] = solve ? kept : 0;
        }
        __syncwarp();
    }
}

__global__ void k_compact_rows(int nrows, const int *oldptr, const int *newptr, const int *col_in,
                               const double *val_in, int *col_out, double *val_out) {
    long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    int r = (int)(tid >> 3), g = (int)(tid & 7);
    if (r >= nrows) return;
    int o = oldptr[r], nn = newptr[r], cnt = newptr[r + 1] - newptr[r];
    for (int t = g; t < cnt; t += 8) { col_out[nn + t] = col_in[o + t]; val_out[nn + t] = val_in[o + t]; }
}

// ---- RAP ---------------------------------------------------------------------
// A P by rows: (AP)[k,c] = the row's entries with pmap = c added in ascending order from
// 0.0, columns ascending, in the row's own slots of apcol/apval.
//
// Rows of up to AP_SHORT entries (7-16 on the fine levels, where the rows are): a block
// stages its 128 rows' entries, contiguous in the CSR, with coalesced loads (coarse column
// and value) in shared memory; a thread merges and sorts its row there in place; the slots
// go back coalesced.  One thread per row keeps every lane of the FP64 adds busy.  A thread
// per row on 64-entry local arrays spent its time on local memory and on 32 rows' strided
// lines: on 64^3 S8 (80 directions) 106 ms of a setup, 48 ms of which this saves; an
// 18^3 x 6 tet matrix (rows of up to 682 entries) is set up and solved in 29.6 ms instead
// of 43.7.  Longer rows go to a list.
constexpr int AP_SHORT = 32;

__global__ void __launch_bounds__(128) k_ap(int n, const int *rowptr, const int *col, const double *val,
                                            const int *pmap, const int8_t *cf, int *aplen, int *apcol,
                                            double *apval, int cap, int *longrow, int *nlong) {
    extern __shared__ double apsm[];
    double *sv = apsm;
    int *sc = (int *)(apsm + cap);
    const int r0 = blockIdx.x * 128, r1 = min(n, r0 + 128);
    const int P0 = rowptr[r0], E = min(rowptr[r1] - P0, cap);
    for (int p = threadIdx.x; p < E; p += 128) {
        sc[p] = pmap[col[P0 + p]];
        sv[p] = val[P0 + p];
    }
    __syncthreads();
    const int k = r0 + threadIdx.x;
    if (k < r1) {
        const int s = rowptr[k] - P0, e = rowptr[k + 1] - P0;
        int len = 0;
        if (cf[k] == CF_COARSEST) {
            aplen[k] = 0;
        } else if (e > s && (e > E || e - s > AP_SHORT)) {   // (an empty row has no product: aplen 0 below)
            longrow[atomicAdd(nlong, 1)] = k;
        } else {
            for (int p = s; p < e; ++p) {   // slot s + len <= p: the merge runs in place
                const int c = sc[p];
                if (c < 0) continue;
                const double v = sv[p];
                int t = s;
                while (t < s + len && sc[t] != c) ++t;
                if (t == s + len) { sc[t] = c; sv[t] = 0.0 + v; ++len; }
                else sv[t] = sv[t] + v;
            }
            for (int a = s + 1; a < s + len; ++a) {
                const int c = sc[a];
                const double v = sv[a];
                int b = a;
                while (b > s && sc[b - 1] > c) { sc[b] = sc[b - 1]; sv[b] = sv[b - 1]; --b; }
                sc[b] = c;
                sv[b] = v;
            }
            aplen[k] = len;
        }
    }
    __syncthreads();
    for (int p = threadIdx.x; p < E; p += 128) {   // (a listed row's slots are written again)
        apcol[P0 + p] = sc[p];
        apval[P0 + p] = sv[p];
    }
}

// Listed rows with lo < entries <= CAP / 2: a warp per row, a hash table of CAP slots in
// shared memory.  32 entries at a time: each lane finds its column's slot, then the first
// lane of every slot adds the values of its lanes in lane order, so a slot's additions keep
// the entry order.  The slots are then ranked by column.
template <int CAP>
__global__ void k_ap_long(const int *longrow, const int *nlong, int lo, const int *rowptr, const int *col,
                          const double *val, const int *pmap, int *aplen, int *apcol, double *apval) {
    extern __shared__ double apsm[];
    const unsigned FULL = 0xffffffffu;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    double *vals = apsm + (size_t)w * CAP;
    int *keys = (int *)(apsm + (size_t)wpb * CAP) + (size_t)w * (CAP + CAP / 2), *list = keys + CAP;
    const int n = *nlong;
    for (int q = blockIdx.x * wpb + w; q < n; q += gridDim.x * wpb) {
        const int k = longrow[q], s = rowptr[k], e = rowptr[k + 1];
        if (e - s <= lo || e - s > CAP / 2) continue;
        for (int t = lane; t < CAP; t += 32) keys[t] = -1;
        __syncwarp();
        for (int p0 = s; p0 < e; p0 += 32) {
            const int p = p0 + lane;
            const int c = p < e ? pmap[col[p]] : -1;
            const double v = p < e ? val[p] : 0.0;
            int slot = -1;
            if (c >= 0) {
                unsigned h = ((unsigned)c * 2654435761u) & (CAP - 1);
                while (true) {   // ends: at most CAP / 2 distinct columns
                    const int prev = atomicCAS(&keys[h], -1, c);
                    if (prev == -1) vals[h] = 0.0;
                    if (prev == -1 || prev == c) break;
                    h = (h + 1) & (CAP - 1);
                }
                slot = (int)h;
            }
            __syncwarp();
            const unsigned same = __match_any_sync(FULL, slot);
            const bool head = slot >= 0 && (int)__ffs(same) - 1 == lane;
            double acc = head ? vals[slot] : 0.0;
            unsigned rem = head ? same : 0u;
            while (__any_sync(FULL, rem)) {
                const double t = __shfl_sync(FULL, v, rem ? __ffs(rem) - 1 : lane);
                if (rem) acc = acc + t;
                rem &= rem - 1;
            }
            if (head) vals[slot] = acc;
            __syncwarp();
        }
        int m = 0;
        for (int t0 = 0; t0 < CAP; t0 += 32) {
            const bool occ = keys[t0 + lane] >= 0;
            const unsigned b = __ballot_sync(FULL, occ);
            if (occ) list[m + __popc(b & ((1u << lane) - 1u))] = t0 + lane;
            m += __popc(b);
        }
        __syncwarp();
        for (int a = lane; a < m; a += 32) {
            const int c = keys[list[a]];
            int rank = 0;
            for (int f = 0; f < m; ++f) rank += keys[list[f]] < c;
            apcol[s + rank] = c;
            apval[s + rank] = vals[list[a]];
        }
        if (lane == 0) aplen[k] = m;
        __syncwarp();
    }
}

// Listed rows with more entries than that: a thread per row in the row's slots.
__global__ void k_ap_serial(const int *longrow, const int *nlong, int lo, const int *rowptr, const int *col,
                            const double *val, const int *pmap, int *aplen, int *apcol, double *apval) {
    const int n = *nlong;
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        const int k = longrow[q], s = rowptr[k], e = rowptr[k + 1];
        if (e - s <= lo) continue;
        int len = 0;
        for (int p = s; p < e; ++p) {
            int c = pmap[col[p]];
            if (c < 0) continue;
            int t = 0;
            while (t < len && apcol[s + t] != c) ++t;
            if (t == len) { apcol[s + t] = c; apval[s + t] = 0.0; ++len; }
            apval[s + t] = apval[s + t] + val[p];
        }
        for (int a = 1; a < len; ++a) {
            int c = apcol[s + a];
            double v = apval[s + a];
            int b = a;
            while (b > 0 && apcol[s + b - 1] > c) {
                apcol[s + b] = apcol[s + b - 1];
                apval[s + b] = apval[s + b - 1];
                --b;
            }
            apcol[s + b] = c;
            apval[s + b] = v;
        }
        aplen[k] = len;
    }
}

__global__ void k_rap_bound(int nc, const int *cpts, const int *zrowptr, const int *zcol, const int *aplen, int *U) {
    int ic = blockIdx.x * blockDim.x + threadIdx.x;
    if (ic >= nc) return;
    int u = aplen[cpts[ic]];
    for (int t = zrowptr[ic]; t < zrowptr[ic + 1]; ++t) u += aplen[zcol[t]];
    U[ic] = u;
}

__device__ __forceinline__ unsigned hslot(int c, unsigned mask) { return ((unsigned)c * 2654435761u) & mask; }

// G lanes per coarse row (32/G rows per warp).  Table: keys (int, -1 empty)
// and values, in shared memory (hcap slots per row, sized to the row's bin) or
// in global scratch (cap per row given by gptr).  Output: sorted, filtered
// entries at ucol/uval[uptr[ic]...], count in cnt[ic].  Magnitude maxima use
// integer keys; the phi_A filter costs nothing when it is off (filt == 0).
// A row's table has the first power of two >= its bound U (at least 64) slots:
// U bounds the row's distinct columns, so linear probing always finds a slot, and
// on the transport operators the distinct columns are on average 20-55% of U, so
// tables stay about half full or less.  Each slot's additions follow the R-row
// order whatever the table size, so the size changes no bit of the result.
template <int G, bool GLOBAL_TABLE>
__global__ void k_rap(int nrows_work, const int *worklist, const int *cpts, const int *zrowptr, const int *zcol,
                      const double *zval, const int *aprow, const int *aplen, const int *apcol, const double *apval,
                      const int *uptr, const int *U, int filt, double phiA, int *cnt, int *ucol, double *uval, int hcap,
                      const long long *gptr, int *gkeys, double *gvals, int *overflow, int *err) {
    extern __shared__ double smem2[];
    const unsigned FULL = 0xffffffffu;
    constexpr int SPW = 32 / G;
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int g = lane % G, q = lane / G;
    int wpb = blockDim.x >> 5;
    unsigned gmask = (G == 32) ? FULL : (((1u << (G & 31)) - 1u) << (q * G));
    for (int wb = (blockIdx.x * wpb + warp) * SPW; wb < nrows_work; wb += gridDim.x * wpb * SPW) {
        int w = wb + q;
        bool has = w < nrows_work;
        int ic = has ? worklist[w] : 0;
        int *keys = nullptr;
        double *vals = nullptr;
        int cap = 0;
        if (has) {
            if (GLOBAL_TABLE) {
                long long off = gptr[w];
                cap = (int)(gptr[w + 1] - off);
                keys = gkeys + off;
                vals = gvals + off;
            } else {
                int slot = warp * SPW + q;
                vals = smem2 + (size_t)slot * hcap;
                keys = (int *)(smem2 + (size_t)wpb * SPW * hcap) + (size_t)slot * hcap;
                if (U[ic] > hcap) {
                    if (g == 0) { cnt[ic] = -1; atomicAdd(overflow, 1); }
                    has = false;
                } else {
                    cap = 64;
                    while (cap < U[ic]) cap <<= 1;
                }
            }
        }
        unsigned mask = (unsigned)cap - 1u;
        for (int t = g; t < cap; t += G) keys[t] = -1;
        __syncwarp();
        int i = has ? cpts[ic] : 0;
        int z0 = has ? zrowptr[ic] : 0, z1 = has ? zrowptr[ic + 1] : 0;
        int nr = has ? z1 - z0 + 1 : 0;   // R row entries, identity included
        int nrmax = nr;
        for (int o = 16; o > 0; o >>= 1) nrmax = max(nrmax, __shfl_xor_sync(FULL, nrmax, o));
        // The R row in ascending column order (the identity at column i); each step's
        // chain of loads (its column, then its AP row, then the AP row's first entry
        // of this lane) is issued one step ahead, while the previous step's entries
        // go into the table.  The additions into each slot keep the R-row order.
        bool placed = false;
        int t = z0;
        int zc = (t < z1) ? zcol[t] : 0x7fffffff;   // the next Z column
        auto advance = [&](int &k, double &r) {
            if (!placed && zc > i) { k = i; r = 1.0; placed = true; }
            else { k = zc; r = zval[t]; ++t; zc = (t < z1) ? zcol[t] : 0x7fffffff; }
        };
        int k_c = 0, a_c = 0, l_c = 0, c_c = 0;
        double r_c = 0.0, v_c = 0.0;
        if (nr > 0) {
            advance(k_c, r_c);
            a_c = aprow[k_c];
            l_c = aplen[k_c];
            if (g < l_c) { c_c = apcol[a_c + g]; v_c = apval[a_c + g]; }
        }
        for (int step = 0; step < nrmax; ++step) {
            int k_n = 0, a_n = 0, l_n = 0, c_n = 0;
            double r_n = 0.0, v_n = 0.0;
            if (step + 1 < nr) {
                advance(k_n, r_n);
                a_n = aprow[k_n];
                l_n = aplen[k_n];
                if (g < l_n) { c_n = apcol[a_n + g]; v_n = apval[a_n + g]; }
            }
            if (step < nr) {
                const double r = r_c;
                const int a0 = a_c, al = l_c;
                for (int qq = g; qq < al; qq += G) {
                    int c;
                    double v;
                    if (qq == g) { c = c_c; v = v_c; }
                    else { c = apcol[a0 + qq]; v = apval[a0 + qq]; }
                    unsigned hs = hslot(c, mask);
                    int probes = 0;
                    bool ok = false;
                    while (probes++ < cap) {
                        int prev = atomicCAS(&keys[hs], -1, c);
                        if (prev == -1) { vals[hs] = 0.0; ok = true; break; }
                        if (prev == c) { ok = true; break; }
                        hs = (hs + 1) & mask;
                    }
                    if (ok) vals[hs] = fma(r, v, vals[hs]);
                    else atomicOr(err, DERR_HASH_OVERFLOW);
                }
            }
            __syncwarp();
            k_c = k_n; r_c = r_n; a_c = a_n; l_c = l_n; c_c = c_n; v_c = v_n;
        }
        const int base = has ? uptr[ic] : 0;
        // The phi_A filter (threshold from the table), then the kept entries are packed in
        // the table itself and each is written at its column's rank among them, once.
        // (Ranking from an unsorted list in the output arrays read every column through L2
        // right after it was written, and the filter took another pass.)
        double thr = 0.0;
        if (filt) {
            long long mxb = 0;
            for (int sl = g; sl < cap; sl += G)
                if (keys[sl] >= 0 && keys[sl] != ic) mxb = max(mxb, absbits(vals[sl]));
            for (int o = G / 2; o > 0; o >>= 1) mxb = max(mxb, __shfl_xor_sync(FULL, mxb, o, G));
            thr = phiA * __longlong_as_double(mxb);
        }
        int m = 0;
        int capmax = cap;
        for (int o = 16; o > 0; o >>= 1) capmax = max(capmax, __shfl_xor_sync(FULL, capmax, o));
        for (int s0 = 0; s0 < capmax; s0 += G) {   // kept entries move to the table's front
            const int sl = s0 + g;
            const int key = sl < cap ? keys[sl] : -1;
            const double v = sl < cap ? vals[sl] : 0.0;
            const bool k_ = key >= 0 && !(filt && key != ic && fabs(v) < thr);
            const unsigned msk = __ballot_sync(FULL, k_) & gmask;
            __syncwarp();   // every slot of the pass is read before one is written (a ballot orders no memory)
            if (k_) {
                const int off = m + __popc(msk & ((1u << lane) - 1u));
                keys[off] = key;
                vals[off] = v;
            }
            m += __popc(msk);
            __syncwarp();
        }
        for (int e = g; e < m; e += G) {
            const int ce = keys[e];
            int rank = 0;
            for (int f = 0; f < m; ++f) rank += keys[f] < ce;
            ucol[base + rank] = ce;
            uval[base + rank] = vals[e];
        }
        if (has && g == 0) cnt[ic] = m;
        __syncwarp();
    }
}

__global__ void k_gather_int(int n, const int *src, const int *idx, int *out) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) out[k] = src[idx[k]];
}

__global__ void k_gather_rowdir(int nc, const int *cpts, const int *rowdir, int *rowdir_c) {
    int ic = blockIdx.x * blockDim.x + threadIdx.x;
    if (ic < nc) rowdir_c[ic] = rowdir[cpts[ic]];
}

__global__ void k_rowlen_dir(int n, const int *rowptr, const int *rowdir, unsigned long long *nnzdir) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    bool valid = i < n;
    int d = valid ? rowdir[i] : 0;
    add_by_dir<unsigned long long>(nnzdir, d, valid ? (unsigned long long)(rowptr[i + 1] - rowptr[i]) : 0ULL, valid);
}

__global__ void k_fill_int8(int n, int8_t *a, int8_t v) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = v;
}

__global__ void k_fill_int(int n, int *a, int v) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = v;
}

__device__ __forceinline__ int rap_bin(int u) { return u <= 128 ? 0 : u <= 512 ? 1 : u <= 2048 ? 2 : 3; }



__global__ void k_overflow_caps(int nover, const int *list, const int *U, long long *capw) {
    int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= nover) return;
    long long c = 64;
    while (c < (long long)U[list[w]]) c <<= 1;
    capw[w] = c;
}

__global__ void k_big_rows(int nbig, const int *list, const int *npat, long long *goff) {
    int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= nbig) return;
    long long np = npat[list[w]];
    goff[w] = np * np + 4 * np;
}


// class of every system, and the largest system of each class with global slots (bmax)
__global__ void k_lair_classes(int nc, const int *npat, int8_t *cls, int *bmax) {
    int ic = blockIdx.x * blockDim.x + threadIdx.x;
    const int np = ic < nc ? npat[ic] : 0, c = lair_class(np);
    if (ic < nc) cls[ic] = (int8_t)c;
    for (int k = LAIR_SLOT; k < LAIR_BIG; ++k) {
        const int mx = __reduce_max_sync(0xffffffffu, c == k ? np : 0);
        if (mx > 0 && (threadIdx.x & 31) == 0) atomicMax(&bmax[k - LAIR_SLOT], mx);
    }
}

__global__ void k_rap_classes(int nc, const int *U, int8_t *cls) {
    int ic = blockIdx.x * blockDim.x + threadIdx.x;
    if (ic < nc) cls[ic] = (int8_t)rap_bin(U[ic]);
}

template <class T>
void d2h(T *h, const T *d, size_t count, cudaStream_t s) {
    PR_CUDA(cudaMemcpyAsync(h, d, count * sizeof(T), cudaMemcpyDeviceToHost, s));
    PR_CUDA(cudaStreamSynchronize(s));
}

// Rows 0..n-1 grouped by class (ascending row order inside each class):
// list[start[c] .. start[c] + count[c]).  A counting sort, deterministic: per
// block of PART_BS rows the rows of each class (counted by warp ballots), an
// exclusive scan over (class, block), and a scatter at each row's rank among the
// rows of its class before it.  One host read (the class counts).
constexpr int PART_BS = 256;
constexpr int PART_MAXC = 16;

__global__ void __launch_bounds__(PART_BS) k_class_hist(int n, const int8_t *cls, int nclass, int nblk, int *hist) {
    __shared__ int wc[PART_BS / 32][PART_MAXC];
    const int i = blockIdx.x * PART_BS + threadIdx.x;
    const int c = (i < n && cls[i] >= 0 && cls[i] < nclass) ? cls[i] : -1;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int k = 0; k < nclass; ++k) {
        const unsigned m = __ballot_sync(0xffffffffu, c == k);
        if (lane == 0) wc[w][k] = __popc(m);
    }
    __syncthreads();
    if ((int)threadIdx.x < nclass) {
        int t = 0;
        for (int ww = 0; ww < PART_BS / 32; ++ww) t += wc[ww][threadIdx.x];
        hist[threadIdx.x * nblk + blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(PART_BS) k_class_scatter(int n, const int8_t *cls, int nclass, int nblk,
                                                           const int *off, int *list) {
    __shared__ int wc[PART_BS / 32][PART_MAXC];
    const int i = blockIdx.x * PART_BS + threadIdx.x;
    const int c = (i < n && cls[i] >= 0 && cls[i] < nclass) ? cls[i] : -1;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int rank_in_warp = 0;
    for (int k = 0; k < nclass; ++k) {
        const unsigned m = __ballot_sync(0xffffffffu, c == k);
        if (lane == 0) wc[w][k] = __popc(m);
        if (c == k) rank_in_warp = __popc(m & ((1u << lane) - 1u));
    }
    __syncthreads();
    if (c < 0) return;
    int before = 0;
    for (int ww = 0; ww < w; ++ww) before += wc[ww][c];
    list[off[c * nblk + blockIdx.x] + before + rank_in_warp] = i;
}

__global__ void k_class_counts(int nclass, int nblk, const int *off, const int *extra, int nextra, int *out) {
    const int c = threadIdx.x;
    if (c <= nclass) out[c] = off[c * nblk];   // class starts, and the total
    else if (c - nclass - 1 < nextra) out[c] = extra[c - nclass - 1];
}

// extra (device, nextra values): read together with the counts into hextra
void partition_by_class(const int8_t *cls, int n, int nclass, int *list, int *start, int *count, cudaStream_t s,
                        const int *extra = nullptr, int nextra = 0, int *hextra = nullptr) {
    PR_REQUIRE(nclass >= 1 && nclass <= PART_MAXC && nclass + 1 + nextra <= 32, PAIR_ERR_DEVICE,
               "partition_by_class: too many classes");
    if (n <= 0) {
        for (int c = 0; c < nclass; ++c) { start[c] = 0; count[c] = 0; }
        for (int k = 0; k < nextra; ++k) hextra[k] = 0;
        return;
    }
    const int nblk = (int)blocks_for(n, PART_BS);
    const int nh = nclass * nblk;
    int *hist = dmalloc<int>(nh, s), *off = dmalloc<int>(nh + 1, s), *cs = dmalloc<int>(nclass + 1 + nextra, s);
    k_class_hist<<<nblk, PART_BS, 0, s>>>(n, cls, nclass, nblk, hist);
    PR_LAUNCH();
    scan_exclusive(hist, off, nh, s, false);
    k_class_scatter<<<nblk, PART_BS, 0, s>>>(n, cls, nclass, nblk, off, list);
    PR_LAUNCH();
    k_class_counts<<<1, 32, 0, s>>>(nclass, nblk, off, extra, nextra, cs);
    PR_LAUNCH();
    int h[32];
    d2h(h, cs, nclass + 1 + nextra, s);
    for (int c = 0; c < nclass; ++c) { start[c] = h[c]; count[c] = h[c + 1] - h[c]; }
    for (int k = 0; k < nextra; ++k) hextra[k] = h[nclass + 1 + k];
    dfree(hist, s);
    dfree(off, s);
    dfree(cs, s);
}

__global__ void k_split_len(int n, const int *srow, const int *rowptr, int *len) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) {
        int i = srow[k];
        len[k] = rowptr[i + 1] - rowptr[i];
    }
}

// entries of split row k (row srow[k]) copied to sptr[k].., eight lanes per row
template <class T>
__global__ void k_split_copy(int n, const int *srow, const int *rowptr, const int *col, const double *val,
                             const int *sptr, int *scol, T *sval) {
    long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    int k = (int)(tid >> 3), g = (int)(tid & 7);
    if (k >= n) return;
    int i = srow[k];
    int a = rowptr[i], len = rowptr[i + 1] - a, d = sptr[k];
    for (int q = g; q < len; q += 8) {
        scol[d + q] = col[a + q];
        sval[d + q] = (T)val[a + q];
    }
}

// ---- sliced ELL (SELL-32) copies for the V-cycle's row dot products -------------
// Rows are taken in windows of 256 and ordered inside each window by decreasing
// length (ties by position); every 32 consecutive positions form a slice whose
// entries are stored column-major with the slice's first (longest) row setting its
// width: entry j of the row at lane t of slice s sits at ptr[s] + 32 j + t.
constexpr int SELL_WIN = 256;

// rows[q] (or q when rows is null), q < nr: CSR row of list position q
__global__ void k_sell_rank(int nr, const int *rows, const int *rowptr, int *out_row, int *out_len) {
    __shared__ int sl[SELL_WIN];
    const int t = threadIdx.x, q = blockIdx.x * SELL_WIN + t;
    const int r = q < nr ? (rows ? rows[q] : q) : -1;
    const int len = r >= 0 ? rowptr[r + 1] - rowptr[r] : -1;
    sl[t] = len;
    __syncthreads();
    int rank = 0;
    for (int u = 0; u < SELL_WIN; ++u) {
        const int lu = sl[u];
        rank += (lu > len || (lu == len && u < t)) ? 1 : 0;
    }
    const int pos = blockIdx.x * SELL_WIN + rank;
    out_row[pos] = r;
    out_len[pos] = len > 0 ? len : 0;
}

__global__ void k_sell_width(int ns, const int *len, int *w32) {
    int sl = blockIdx.x * blockDim.x + threadIdx.x;
    if (sl < ns) w32[sl] = 32 * len[32 * sl];
}

template <class T>
__global__ void k_sell_fill(int npos, const int *prow, const int *plen, const int *sptr, const int *rowptr,
                            const int *col, const double *val, int *scol, T *sval) {
    int pos = blockIdx.x * blockDim.x + threadIdx.x;
    if (pos >= npos) return;
    const int r = prow[pos];
    if (r < 0) return;
    const int a = rowptr[r], len = plen[pos];
    const int base = sptr[pos >> 5] + (pos & 31);
    for (int j = 0; j < len; ++j) {
        scol[base + 32 * j] = col[a + j];
        sval[base + 32 * j] = (T)val[a + j];
    }
}

// 16-bit column offsets: an entry's column minus its row, when every stored entry
// of a store fits (the relaxation stores of the coarse levels: their stencils stay
// within a few mesh planes of the row); the padding slots are never read
// offsets are taken from the row's own index, or (rowbase, the restriction's Z
// rows) from the fine row of its coarse point
__global__ void k_sell_off_check(int npos, const int *prow, const int *plen, const int *sptr, const int *scol,
                                 const int *rowbase, int *bad) {
    const int pos = blockIdx.x * blockDim.x + threadIdx.x;
    if (pos >= npos) return;
    const int q = prow[pos];
    if (q < 0) return;
    const int r = rowbase ? rowbase[q] : q;
    const int len = plen[pos], base = sptr[pos >> 5] + (pos & 31);
    for (int j = 0; j < len; ++j) {
        const int off = scol[base + 32 * j] - r;
        if (off < -32767 || off > 32767) { atomicOr(bad, 1); return; }
    }
}

__global__ void k_sell_to16(int npos, const int *prow, const int *plen, const int *sptr, const int *scol,
                            const int *rowbase, short *col16) {
    const int pos = blockIdx.x * blockDim.x + threadIdx.x;
    if (pos >= npos) return;
    const int q = prow[pos];
    if (q < 0) return;
    const int r = rowbase ? rowbase[q] : q;
    const int len = plen[pos], base = sptr[pos >> 5] + (pos & 31);
    for (int j = 0; j < len; ++j) col16[base + 32 * j] = (short)(scol[base + 32 * j] - r);
}

// P columns of a store's entries and rows (Sell::pcol, pown); *bad: an offset from the
// row's origin (its own P column, else its first entry's) leaves 16 bits
__global__ void k_sell_pcol(int npos, const int *prow, const int *plen, const int *sptr, const int *scol,
                            const int *pmap, int *pcol, int *pown, int *bad) {
    const int pos = blockIdx.x * blockDim.x + threadIdx.x;
    if (pos >= npos) return;
    const int r = prow[pos];
    if (r < 0) { pown[pos] = -2; return; }
    const int len = plen[pos], base = sptr[pos >> 5] + (pos & 31);
    const int own = pmap[r];
    int org = own;
    bool far = false;
    for (int j = 0; j < len; ++j) {
        const int c = pmap[scol[base + 32 * j]];
        pcol[base + 32 * j] = c;
        if (c < 0) continue;
        if (org < 0) org = c;
        far |= c - org < -32767 || c - org > 32767;
    }
    pown[pos] = own >= 0 ? own : -2 - max(org, 0);
    if (far) atomicOr(bad, 1);
}

__global__ void k_sell_pcol16(int npos, const int *prow, const int *plen, const int *sptr, const int *pcol,
                              const int *pown, short *pcol16) {
    const int pos = blockIdx.x * blockDim.x + threadIdx.x;
    if (pos >= npos || prow[pos] < 0) return;
    const int len = plen[pos], base = sptr[pos >> 5] + (pos & 31);
    const int o = pown[pos], org = o >= 0 ? o : -2 - o;
    for (int j = 0; j < len; ++j) {
        const int c = pcol[base + 32 * j];
        pcol16[base + 32 * j] = (short)(c < 0 ? -32768 : c - org);
    }
}

void sell_off_check(Sell &S, const int *rowbase, int *bad, cudaStream_t s) {
    if (S.nrows <= 0) return;
    k_sell_off_check<<<blocks_for(S.npos, 256), 256, 0, s>>>(S.npos, S.row, S.len, S.ptr, S.col, rowbase, bad);
    PR_LAUNCH();
}

void sell_to16(Sell &S, const int *rowbase, cudaStream_t s) {
    if (S.nrows <= 0) return;
    S.col16 = dmalloc<short>(std::max<long long>(S.nnz, 1), s);
    k_sell_to16<<<blocks_for(S.npos, 256), 256, 0, s>>>(S.npos, S.row, S.len, S.ptr, S.col, rowbase, S.col16);
    PR_LAUNCH();
    dfree(S.col, s);
    S.col = nullptr;
}

// 16-bit column offsets of one store, where they fit
void sell_compress_cols(Hier &h, Sell &S, const int *rowbase = nullptr) {
    if (S.nrows <= 0 || !S.col) return;
    cudaStream_t s = h.stream;
    int *bad = dmalloc<int>(1, s);
    PR_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), s));
    sell_off_check(S, rowbase, bad, s);
    int hb = 0;
    d2h(&hb, bad, 1, s);
    dfree(bad, s);
    if (!hb) sell_to16(S, rowbase, s);
}

// the F and C stores of a level: P columns of the F store, and 16-bit offsets where they
// fit (one host read for the three checks)
void sell_finish_fc(Hier &h, Level &L) {
    cudaStream_t s = h.stream;
    Sell &F = L.sF;
    int *bad = dmalloc<int>(3, s);
    PR_CUDA(cudaMemsetAsync(bad, 0, 3 * sizeof(int), s));
    if (F.nrows > 0) {
        F.pcol = dmalloc<int>(std::max<long long>(F.nnz, 1), s);
        F.pown = dmalloc<int>(F.npos, s);
        k_sell_pcol<<<blocks_for(F.npos, 256), 256, 0, s>>>(F.npos, F.row, F.len, F.ptr, F.col, L.pmap, F.pcol, F.pown,
                                                            bad + 2);
        PR_LAUNCH();
    }
    sell_off_check(F, nullptr, bad, s);
    sell_off_check(L.sC, nullptr, bad + 1, s);
    int hb[3] = {0, 0, 0};
    d2h(hb, bad, 3, s);
    dfree(bad, s);
    if (!hb[0]) sell_to16(F, nullptr, s);
    if (!hb[1]) sell_to16(L.sC, nullptr, s);
    if (!hb[2] && F.nrows > 0) {
        F.pcol16 = dmalloc<short>(std::max<long long>(F.nnz, 1), s);
        k_sell_pcol16<<<blocks_for(F.npos, 256), 256, 0, s>>>(F.npos, F.row, F.len, F.ptr, F.pcol, F.pown, F.pcol16);
        PR_LAUNCH();
        dfree(F.pcol, s);
        F.pcol = nullptr;
    }
}

// SELL copy of nr rows of a CSR matrix (list rows, or rows 0..nr-1), values in the
// V-cycle's precision
void build_sell(Hier &h, Sell &S, const int *rows, int nr, const int *rowptr, const int *col, const double *val) {
    cudaStream_t s = h.stream;
    const int BS = 256;
    S.nrows = nr;
    if (nr <= 0) return;
    const int nwin = (nr + SELL_WIN - 1) / SELL_WIN;
    S.npos = nwin * SELL_WIN;
    const int ns = S.npos / 32;
    S.row = dmalloc<int>(S.npos, s);
    S.len = dmalloc<int>(S.npos, s);
    k_sell_rank<<<nwin, SELL_WIN, 0, s>>>(nr, rows, rowptr, S.row, S.len);
    PR_LAUNCH();
    int *w32 = dmalloc<int>(ns, s);
    k_sell_width<<<blocks_for(ns, BS), BS, 0, s>>>(ns, S.len, w32);
    PR_LAUNCH();
    S.ptr = dmalloc<int>(ns + 1, s);
    S.nnz = scan_exclusive(w32, S.ptr, ns, s);
    dfree(w32, s);
    S.col = dmalloc<int>(std::max<long long>(S.nnz, 1), s);
    if (h.prm.precision >= 1) {
        S.val = dmalloc<float>(std::max<long long>(S.nnz, 1), s);
        k_sell_fill<float><<<blocks_for(S.npos, BS), BS, 0, s>>>(S.npos, S.row, S.len, S.ptr, rowptr, col, val,
                                                                 S.col, (float *)S.val);
    } else {
        S.val = dmalloc<double>(std::max<long long>(S.nnz, 1), s);
        k_sell_fill<double><<<blocks_for(S.npos, BS), BS, 0, s>>>(S.npos, S.row, S.len, S.ptr, rowptr, col, val,
                                                                  S.col, (double *)S.val);
    }
    PR_LAUNCH();
}

// CF split of one level (see Level): the row order [F | C | coarsest], SELL copies
// of the F and C rows (with_fc) and a CSR copy of the coarsest rows with the
// coarsest segments' positions in it
void build_split(Hier &h, Level &L, bool with_fc) {
    cudaStream_t s = h.stream;
    const int BS = 256;
    const int n = L.n;
    const size_t es = h.prm.precision >= 1 ? sizeof(float) : sizeof(double);
    int st[3] = {0, 0, 0}, cnt[3] = {0, 0, 0};
    L.srow = dmalloc<int>(std::max(n, 1), s);
    partition_by_class(L.cf, n, 3, L.srow, st, cnt, s);
    PR_REQUIRE(cnt[0] + cnt[1] + cnt[2] == n, PAIR_ERR_DEVICE, "CF split does not cover the level's rows");
    L.nF = cnt[0];
    L.nC = cnt[1];
    const int kX = L.nF + L.nC, nx = n - kX;
    if (with_fc) {
        build_sell(h, L.sF, L.srow, L.nF, L.rowptr, L.col, L.val);
        build_sell(h, L.sC, L.srow + L.nF, L.nC, L.rowptr, L.col, L.val);
        sell_finish_fc(h, L);
    }
    if (nx > 0) {
        int *len = dmalloc<int>(nx, s);
        k_split_len<<<blocks_for(nx, BS), BS, 0, s>>>(nx, L.srow + kX, L.rowptr, len);
        PR_LAUNCH();
        L.sptr = dmalloc<int>(nx + 1, s);
        long long tot = scan_exclusive(len, L.sptr, nx, s);
        dfree(len, s);
        L.scol = dmalloc<int>(std::max<long long>(tot, 1), s);
        L.sval = dmalloc<char>(std::max<long long>(tot, 1) * es, s);
        if (h.prm.precision >= 1)
            k_split_copy<float><<<blocks_for((long long)nx * 8, BS), BS, 0, s>>>(
                nx, L.srow + kX, L.rowptr, L.col, L.val, L.sptr, L.scol, (float *)L.sval);
        else
            k_split_copy<double><<<blocks_for((long long)nx * 8, BS), BS, 0, s>>>(
                nx, L.srow + kX, L.rowptr, L.col, L.val, L.sptr, L.scol, (double *)L.sval);
        PR_LAUNCH();
    }
    // coarsest segments are whole matrices, ascending in row order, so each one is a
    // contiguous run of the coarsest group; positions relative to the group's start
    std::vector<int> s0;
    long long pos = 0, prev = -1;
    for (int d = 0; d < h.ndir; ++d)
        if (L.nrows[d] > 0 && L.coarsest[d]) {
            PR_REQUIRE(L.row0[d] > prev, PAIR_ERR_DEVICE, "coarsest segments out of row order");
            prev = L.row0[d];
            s0.push_back((int)pos);
            pos += L.nrows[d];
        }
    PR_REQUIRE(pos == nx, PAIR_ERR_DEVICE, "coarsest rows differ from the coarsest segments");
    PR_REQUIRE((int)s0.size() == L.n_cseg, PAIR_ERR_DEVICE, "coarsest segment count mismatch");
    // a segment too large for the one-CTA shared-memory sweeps: SELL copy of every
    // coarsest row of the level, swept grid-wide
    bool big = false;
    for (int d = 0; d < h.ndir; ++d)
        if (L.nrows[d] > 0 && L.coarsest[d]) {
            const size_t nr = (size_t)L.nrows[d], nz = (size_t)L.nnzdir[d];
            big |= nz * (es + sizeof(int)) + 4 * nr * es + (nr + 1) * sizeof(int) > (size_t)CS_SMEM;
        }
    if (big) {
        build_sell(h, L.sX, L.srow + kX, nx, L.rowptr, L.col, L.val);
        sell_compress_cols(h, L.sX);
    }
    if (!s0.empty()) {
        L.d_cseg_s0 = dmalloc<int>(s0.size(), s);
        PR_CUDA(cudaMemcpyAsync(L.d_cseg_s0, s0.data(), sizeof(int) * s0.size(), cudaMemcpyHostToDevice, s));
        PR_CUDA(cudaStreamSynchronize(s));
    }
}

}  // namespace

void free_level(Level &L, cudaStream_t s) {
    void *ptrs[] = {L.rowptr, L.col, L.val, L.dinv, L.dinv32, L.cf, L.pmap, L.rowdir, L.cpts,
                    L.zrowptr, L.zcol, L.zval, L.d_row0, L.d_cseg_row0, L.d_cseg_n,
                    L.srow, L.sptr, L.scol, L.sval, L.d_cseg_s0, L.cB, L.d_cB_off,
                    L.sF.ptr, L.sF.row, L.sF.len, L.sF.col, L.sF.col16, L.sF.val, L.sF.pcol, L.sF.pown, L.sF.pcol16, L.sC.ptr, L.sC.row, L.sC.len,
                    L.sC.col, L.sC.col16, L.sC.val, L.sZ.ptr, L.sZ.row, L.sZ.len, L.sZ.col, L.sZ.col16, L.sZ.val,
                    L.sX.ptr, L.sX.row, L.sX.len, L.sX.col, L.sX.col16, L.sX.val, L.vb, L.vx, L.vxn, L.vy};
    for (void *p : ptrs) dfree(p, s);
    L = Level();
}

static void finish_segments(Hier &h, Level &L) {
    cudaStream_t s = h.stream;
    std::vector<int> r0, nn;
    for (int d = 0; d < h.ndir; ++d)
        if (L.nrows[d] > 0 && L.coarsest[d]) { r0.push_back(L.row0[d]); nn.push_back(L.nrows[d]); }
    L.n_cseg = (int)r0.size();
    if (L.n_cseg) {
        L.d_cseg_row0 = dmalloc<int>(L.n_cseg, s);
        L.d_cseg_n = dmalloc<int>(L.n_cseg, s);
        PR_CUDA(cudaMemcpyAsync(L.d_cseg_row0, r0.data(), sizeof(int) * r0.size(), cudaMemcpyHostToDevice, s));
        PR_CUDA(cudaMemcpyAsync(L.d_cseg_n, nn.data(), sizeof(int) * nn.size(), cudaMemcpyHostToDevice, s));
        PR_CUDA(cudaStreamSynchronize(s));
    }
}

void build_hierarchy(Hier &h) {
    cudaStream_t s = h.stream;
    const air_params &prm = h.prm;
    const int ND = h.ndir;
    const int BS = 256;
    int *d_count = dmalloc<int>(1, s);
    char *dwork = dmalloc<char>(ND, s);
    char *dcont = dmalloc<char>(ND, s);
    int *dnc = dmalloc<int>(ND, s);
    long long *dnnz = dmalloc<long long>(ND, s);
    cudaEvent_t ev[4];
    for (auto &e : ev) PR_CUDA(cudaEventCreate(&e));
    struct EvFree {
        cudaEvent_t *e;
        ~EvFree() { for (int k = 0; k < 4; ++k) cudaEventDestroy(e[k]); }
    } evfree{ev};
    auto phase_ms = [&](int a, int b) {
        float ms = 0;
        PR_CUDA(cudaEventSynchronize(ev[b]));
        PR_CUDA(cudaEventElapsedTime(&ms, ev[a], ev[b]));
        return (double)ms;
    };
    for (int l = 0;; ++l) {
        Level &L = h.lev[l];
        int n = L.n;
        L.dinv = dmalloc<double>(n, s);
        if (prm.precision >= 1) L.dinv32 = dmalloc<float>(n, s);
        k_dinv<<<blocks_for(n, BS), BS, 0, s>>>(n, L.rowptr, L.col, L.val, L.dinv, L.dinv32);
        PR_LAUNCH();
        L.cf = dmalloc<int8_t>(n, s);
        L.pmap = dmalloc<int>(n, s);
        // per-matrix stats of this level
        PR_CUDA(cudaMemsetAsync(dnnz, 0, sizeof(long long) * ND, s));
        k_rowlen_dir<<<blocks_for(n, BS), BS, 0, s>>>(n, L.rowptr, L.rowdir, (unsigned long long *)dnnz);
        PR_LAUNCH();
        std::vector<long long> nnzd(ND);
        d2h(nnzd.data(), dnnz, ND, s);
        L.nnzdir.assign(ND, 0);
        for (int d = 0; d < ND; ++d) L.nnzdir[d] = (int)nnzd[d];
        L.ncdir.assign(ND, 0);
        L.nnzZdir.assign(ND, 0);
        L.singular.assign(ND, 0);
        L.coarsest.assign(ND, 0);
        std::vector<char> work(ND, 0);
        bool any = false;
        for (int d = 0; d < ND; ++d) {
            if (L.nrows[d] == 0) continue;
            bool last = L.nrows[d] <= prm.max_coarse || l >= prm.max_levels - 1 || l >= 63;
            L.coarsest[d] = last;
            work[d] = !last;
            any |= !last;
        }
        if (!any) {
            k_fill_int8<<<blocks_for(n, BS), BS, 0, s>>>(n, L.cf, CF_COARSEST);
            PR_LAUNCH();
            k_fill_int<<<blocks_for(n, BS), BS, 0, s>>>(n, L.pmap, -1);
            PR_LAUNCH();
            finish_segments(h, L);
            break;
        }
        PR_CUDA(cudaMemcpyAsync(dwork, work.data(), ND, cudaMemcpyHostToDevice, s));
        PR_CUDA(cudaEventRecord(ev[0], s));
        long long nnz = L.nnz;
        uint8_t *S = dmalloc<uint8_t>(nnz, s);
        unsigned *smask = dmalloc<unsigned>(n, s);
        unsigned *lam = dmalloc<unsigned>(n, s);
        PR_CUDA(cudaMemsetAsync(lam, 0, sizeof(unsigned) * n, s));
        {
            // staged entries per block: a quarter more than its rows hold on average
            const int cap = (int)std::min<long long>(3072, std::max<long long>(512, 160 * nnz / n)) & ~7;
            k_strength<<<blocks_for(n, 128), 128, (size_t)cap * 13, s>>>(n, L.rowptr, L.col, L.val, L.rowdir, dwork,
                                                                        prm.theta, prm.eps_R, S, smask, lam, cap);
            PR_LAUNCH();
        }
        uint64_t *key = dmalloc<uint64_t>(n, s);
        int8_t *st0 = dmalloc<int8_t>(n, s), *st1 = dmalloc<int8_t>(n, s);
        int *notmax = dmalloc<int>(n, s);
        PR_CUDA(cudaMemsetAsync(notmax, 0, sizeof(int) * n, s));
        PR_CUDA(cudaMemsetAsync(d_count, 0, sizeof(int), s));
        k_pmis_init<<<blocks_for(n, BS), BS, 0, s>>>(n, L.rowdir, dwork, L.d_row0, lam, l,
                                                     (unsigned long long)prm.seed, key, st0, d_count);
        PR_LAUNCH();
        int und = 0;
        d2h(&und, d_count, 1, s);
        // rounds in groups of PMIS_GROUP between host reads: a round after the last
        // undecided point is gone changes nothing, and the per-round counts give the
        // exact round count
        constexpr int PMIS_GROUP = 4;
        int *rcount = dmalloc<int>(PMIS_GROUP, s);
        int round = 0;
        while (und > 0) {
            PR_REQUIRE(round < 10000, PAIR_ERR_DEVICE, "PMIS did not terminate");
            PR_CUDA(cudaMemsetAsync(rcount, 0, sizeof(int) * PMIS_GROUP, s));
            for (int g = 0; g < PMIS_GROUP; ++g) {
                const int rd = round + 1 + g;
                k_pmis_mark<<<blocks_for(n, BS), BS, 0, s>>>(n, L.rowptr, L.col, S, smask, key, st0, notmax, rd);
                PR_LAUNCH();
                k_pmis_update<<<blocks_for(n, BS), BS, 0, s>>>(n, L.rowptr, L.col, S, smask, st0, st1, notmax, rd,
                                                               rcount + g);
                PR_LAUNCH();
                std::swap(st0, st1);
            }
            int cnt[PMIS_GROUP];
            d2h(cnt, rcount, PMIS_GROUP, s);
            int g = 0;
            while (g < PMIS_GROUP - 1 && cnt[g] > 0) ++g;
            round += g + 1;
            und = cnt[g];
        }
        dfree(rcount, s);
        L.pmis_rounds = round;
        PR_CUDA(cudaEventRecord(ev[1], s));
        PR_CUDA(cudaMemsetAsync(dnc, 0, sizeof(int) * ND, s));
        k_count_c<<<blocks_for(n, BS), BS, 0, s>>>(n, L.rowdir, st0, dnc);
        PR_LAUNCH();
        std::vector<int> ncd(ND);
        d2h(ncd.data(), dnc, ND, s);
        std::vector<char> cont(ND, 0);
        bool anycont = false;
        for (int d = 0; d < ND; ++d) {
            if (!work[d]) continue;
            int nc_ = ncd[d];
            bool stall = nc_ == 0 || (double)nc_ >= 0.9 * (double)L.nrows[d];
            if (stall) L.coarsest[d] = 1;
            else { cont[d] = 1; anycont = true; L.ncdir[d] = nc_; }
        }
        PR_CUDA(cudaMemcpyAsync(dcont, cont.data(), ND, cudaMemcpyHostToDevice, s));
        int *isC = dmalloc<int>(n, s);
        int *cidx = dmalloc<int>(n + 1, s);
        k_cf_final<<<blocks_for(n, BS), BS, 0, s>>>(n, L.rowdir, dcont, st0, L.cf, isC);
        PR_LAUNCH();
        long long nct = scan_exclusive(isC, cidx, n, s);
        dfree(isC, s); dfree(lam, s); dfree(key, s); dfree(st0, s); dfree(st1, s); dfree(notmax, s);
        if (!anycont || nct == 0) {
            k_fill_int<<<blocks_for(n, BS), BS, 0, s>>>(n, L.pmap, -1);
            PR_LAUNCH();
            dfree(S, s); dfree(smask, s); dfree(cidx, s);
            finish_segments(h, L);
            break;
        }
        int nc = (int)nct;
        L.nc = nc;
        L.cpts = dmalloc<int>(nc, s);
        k_cpts<<<blocks_for(n, BS), BS, 0, s>>>(n, L.cf, cidx, L.cpts);
        PR_LAUNCH();
        k_pmap<<<blocks_for(n, BS), BS, 0, s>>>(n, L.rowptr, L.col, L.val, S, smask, L.cf, cidx, L.pmap);
        PR_LAUNCH();
        dfree(cidx, s);
        dfree(smask, s);

        // ---- lAIR -----------------------------------------------------------
        const int rdist = prm.nair ? 2 : prm.distance;   // nAIR degree 1 uses the distance-2 pattern
        int *ncand = dmalloc<int>(nc, s);
        int *pbig = nullptr;   // distance 2: [count, rows with many candidates]
        if (rdist < 2) {
            k_mark_rf1<<<blocks_for(8LL * nc, BS), BS, 0, s>>>(nc, L.cpts, L.rowptr, L.col, L.cf, S, ncand);
            PR_LAUNCH();
        } else {
            int *nf = dmalloc<int>(n, s);
            k_mark_rf<<<blocks_for(8LL * n, BS), BS, 0, s>>>(n, L.rowptr, L.col, L.cf, S, nf);
            PR_LAUNCH();
            pbig = dmalloc<int>((size_t)nc + 1, s);
            PR_CUDA(cudaMemsetAsync(pbig, 0, sizeof(int), s));
            k_lair_ncand<<<blocks_for(8LL * nc, BS), BS, 0, s>>>(nc, L.cpts, L.rowptr, L.col, S, nf, ncand, pbig + 1,
                                                                 pbig);
            PR_LAUNCH();
            dfree(nf, s);
        }
        int *candptr = dmalloc<int>(nc + 1, s);
        long long ncandt = scan_exclusive(ncand, candptr, nc, s);
        int *cand = dmalloc<int>(ncandt, s);
        int *npat = ncand;   // distance 1: the candidates are the pattern
        int *zr = candptr;     // and their offsets the rows of Z
        long long nz = ncandt;
        if (rdist < 2) {
            k_lair_pattern1<<<blocks_for(8LL * nc, BS), BS, 0, s>>>(nc, L.cpts, L.rowptr, L.col, S, candptr, cand);
            PR_LAUNCH();
        } else {
            // one launch per size class over all rows (a row of another class costs its
            // count), no partition and no host read
            npat = dmalloc<int>(nc, s);
            const int rb = std::max(1, std::min(32, nc / (152 * 48)));   // rows per warp, enough warps to fill the chip
            auto pat2 = [&](auto kern, int G, int cap, int lo, int hi) {
                const size_t sm = (size_t)(128 / G) * (cap + hi) * sizeof(int);
                const int rows = G < 32 ? 128 / G : 4 * rb;
                kern<<<blocks_for(nc, rows), 128, sm, s>>>(nc, L.cpts, L.rowptr, L.col, S, candptr, ncand, lo, rb, cand,
                                                          npat);
                PR_LAUNCH();
            };
            pat2(k_lair_pattern2<8, 2 * PAT_SMALL, PAT_SMALL>, 8, 2 * PAT_SMALL, 0, PAT_SMALL);
            pat2(k_lair_pattern2<32, 2 * PAT_MID, PAT_MID>, 32, 2 * PAT_MID, PAT_SMALL + 1, PAT_MID);
            pat2(k_lair_pattern2<32, 2 * PAT_BIG, PAT_BIG>, 32, 2 * PAT_BIG, PAT_MID + 1, PAT_BIG);
            k_lair_pattern2_big<<<std::min<unsigned>(nc, 152u * 6u), 256, 0, s>>>(pbig + 1, pbig, L.cpts, L.rowptr,
                                                                                 L.col, S, candptr, cand, npat);
            PR_LAUNCH();
            dfree(ncand, s);
            zr = dmalloc<int>(nc + 1, s);
            nz = scan_exclusive(npat, zr, nc, s);
        }
        dfree(pbig, s);
        int *zc = dmalloc<int>(nz, s);
        double *zv = dmalloc<double>(nz, s);
        int *keep = dmalloc<int>(nc, s);
        int *dsing = dmalloc<int>(ND, s);
        PR_CUDA(cudaMemsetAsync(dsing, 0, sizeof(int) * ND, s));
        if (prm.nair) {
            k_nair<<<blocks_for(nc, 16), 128, 0, s>>>(nc, L.cpts, L.rowptr, L.col, L.val, S, L.dinv, candptr, cand, npat,
                                                      zr, zc, zv, keep, dsing, L.rowdir, prm.phi_R);
            PR_LAUNCH();
        } else {
            // rows binned by system size; shared memory per warp sized to the bin
            int8_t *ccls = dmalloc<int8_t>(nc, s);
            int *dbmax = dmalloc<int>(LAIR_BIG - LAIR_SLOT, s);
            PR_CUDA(cudaMemsetAsync(dbmax, 0, sizeof(int) * (LAIR_BIG - LAIR_SLOT), s));
            k_lair_classes<<<blocks_for(nc, BS), BS, 0, s>>>(nc, npat, ccls, dbmax);
            PR_LAUNCH();
            int hc[LAIR_CLASSES], hstart[LAIR_CLASSES];
            int *list = dmalloc<int>(nc, s);
            int cls_n[LAIR_CLASSES] = {4, 6, 8, 12, 16, 24, 32, 48, 64};   // then the largest at hand
            partition_by_class(ccls, nc, LAIR_CLASSES, list, hstart, hc, s, dbmax, LAIR_BIG - LAIR_SLOT,
                               cls_n + LAIR_SLOT);
            dfree(ccls, s);
            dfree(dbmax, s);
            // blocks of one to four warps, so that the shared memory of an SM fills evenly
            auto mask_bin = [&](int c, auto kern, int G, int R) {
                if (!hc[c]) return;
                const int nm = cls_n[c], spw = 32 / G;
                const size_t per = ((size_t)nm * (nm | 1) + nm + G * R / 2) * sizeof(double) * spw;   // per warp
                const int wpb = per > 16 * 1024 ? 1 : per > 8 * 1024 ? 2 : 4;
                const size_t sm = per * wpb;
                const unsigned grid = std::min<unsigned>(blocks_for(hc[c], wpb * spw), 152u * 256u);
                if (sm > 48 * 1024) allow_max_dyn_smem(kern);
                kern<<<grid, 32 * wpb, sm, s>>>(hc[c], list + hstart[c], L.cpts, L.rowptr, L.col, L.val, candptr,
                                                cand, npat, zr, zc, zv, keep, dsing, L.rowdir, prm.phi_R, nm, nullptr);
                PR_LAUNCH();
            };
            // more than 64 unknowns: a warp a system, its workspace a slot of global memory
            // for the largest system of the class
            auto mask_big = [&](int c, auto kern, int R, unsigned warps) {
                if (!hc[c]) return;
                const int nm = cls_n[c];
                const unsigned grid = std::min<unsigned>(hc[c], warps);
                double *gbuf = dmalloc<double>((size_t)grid * nm * (nm | 1), s);
                kern<<<grid, 32, ((size_t)nm + 16 * R) * sizeof(double), s>>>(
                    hc[c], list + hstart[c], L.cpts, L.rowptr, L.col, L.val, candptr, cand, npat, zr, zc, zv, keep,
                    dsing, L.rowdir, prm.phi_R, nm, gbuf);
                PR_LAUNCH();
                dfree(gbuf, s);
            };
            for (int c = 0; c <= 2; ++c) mask_bin(c, k_lair_solve_mask<4, 2, false>, 4, 2);
            for (int c = 3; c <= 4; ++c) mask_bin(c, k_lair_solve_mask<8, 2, false>, 8, 2);
            for (int c = 5; c <= 6; ++c) mask_bin(c, k_lair_solve_mask<16, 2, false>, 16, 2);
            for (int c = 7; c <= 8; ++c) mask_bin(c, k_lair_solve_mask<32, 2, false>, 32, 2);
            mask_big(LAIR_SLOT, k_lair_solve_mask<32, 4, true>, 4, 152u * 20u);
            mask_big(LAIR_SLOT + 1, k_lair_solve_mask<32, 8, true>, 8, 152u * 12u);
            int nbig = hc[LAIR_BIG];
            if (nbig > 0) {
                long long *goff = dmalloc<long long>(nbig + 1, s);
                k_big_rows<<<blocks_for(nbig, BS), BS, 0, s>>>(nbig, list + hstart[LAIR_BIG], npat, goff);
                PR_LAUNCH();
                const long long gtot = scan_exclusive_ll(goff, nbig, s);
                double *gbuf = dmalloc<double>(gtot, s);
                k_lair_solve_dense<<<std::min<unsigned>(nbig, 152u * 16u), 32, 0, s>>>(
                    nbig, list + hstart[LAIR_BIG], L.cpts, L.rowptr, L.col, L.val, candptr, cand, npat, zr, zc, zv, keep,
                    dsing, L.rowdir, prm.phi_R, goff, gbuf);
                PR_LAUNCH();
                dfree(gbuf, s); dfree(goff, s);
            }
            dfree(list, s);
        }
        d2h(L.singular.data(), dsing, ND, s);
        dfree(dsing, s);
        int *zr2 = dmalloc<int>(nc + 1, s);
        long long nz2 = scan_exclusive(keep, zr2, nc, s);
        if (nz2 != nz) {
            int *zc2 = dmalloc<int>(nz2, s);
            double *zv2 = dmalloc<double>(nz2, s);
            k_compact_rows<<<blocks_for(8LL * nc, BS), BS, 0, s>>>(nc, zr, zr2, zc, zv, zc2, zv2);
            PR_LAUNCH();
            dfree(zc, s); dfree(zv, s);
            zc = zc2; zv = zv2;
        }
        if (zr != candptr) dfree(zr, s);
        L.zrowptr = zr2; L.zcol = zc; L.zval = zv; L.nnzZ = nz2;
        dfree(keep, s); dfree(cand, s); dfree(candptr, s); dfree(npat, s);
        dfree(S, s);

        PR_CUDA(cudaEventRecord(ev[2], s));
        // ---- RAP ------------------------------------------------------------
        int *aplen = dmalloc<int>(n, s);
        int *apcol = dmalloc<int>(nnz, s);
        double *apval = dmalloc<double>(nnz, s);
        {
            // staged entries per block: a quarter more than its rows hold on average (rows
            // past it go to the list with the long ones)
            const int cap = (int)std::min<long long>(128 * AP_SHORT, std::max<long long>(512, 160 * nnz / n));
            int *lng = dmalloc<int>((size_t)n + 1, s);   // [count, listed rows]
            PR_CUDA(cudaMemsetAsync(lng, 0, sizeof(int), s));
            k_ap<<<blocks_for(n, 128), 128, (size_t)cap * 12, s>>>(n, L.rowptr, L.col, L.val, L.pmap, L.cf, aplen, apcol,
                                                                  apval, cap, lng + 1, lng);
            PR_LAUNCH();
            auto longer = [&](auto kern, int slots, int wpb, int lo) {
                const size_t sm = (size_t)wpb * slots * (sizeof(double) + sizeof(int) * 3 / 2);
                if (sm > 48 * 1024) allow_max_dyn_smem(kern);
                kern<<<std::min<unsigned>(blocks_for(n, wpb), 152u * 8u), 32 * wpb, sm, s>>>(
                    lng + 1, lng, lo, L.rowptr, L.col, L.val, L.pmap, aplen, apcol, apval);
                PR_LAUNCH();
            };
            longer(k_ap_long<256>, 256, 8, 0);
            longer(k_ap_long<2048>, 2048, 4, 128);
            k_ap_serial<<<std::min<unsigned>(blocks_for(n, 64), 152u), 64, 0, s>>>(lng + 1, lng, 1024, L.rowptr, L.col,
                                                                                 L.val, L.pmap, aplen, apcol, apval);
            PR_LAUNCH();
            dfree(lng, s);
        }
        int *U = dmalloc<int>(nc, s);
        k_rap_bound<<<blocks_for(nc, BS), BS, 0, s>>>(nc, L.cpts, L.zrowptr, L.zcol, aplen, U);
        PR_LAUNCH();
        int *uptr = dmalloc<int>(nc + 1, s);
        long long ut = scan_exclusive(U, uptr, nc, s);
        int *ucol = dmalloc<int>(ut, s);
        double *uval = dmalloc<double>(ut, s);
        int *cnt = dmalloc<int>(nc, s);
        {
            // rows binned by their bound U: tables of 128 / 512 / 2048 slots in
            // shared memory, larger rows in global scratch
            int8_t *rcls = dmalloc<int8_t>(nc, s);
            k_rap_classes<<<blocks_for(nc, BS), BS, 0, s>>>(nc, U, rcls);
            PR_LAUNCH();
            int hb[4], bstart[4];
            int *rlist = dmalloc<int>(nc, s);
            partition_by_class(rcls, nc, 4, rlist, bstart, hb, s);
            dfree(rcls, s);
            const int caps[3] = {128, 512, 2048};
            int filt = prm.phi_A > 0.0 ? 1 : 0;
            PR_CUDA(cudaMemsetAsync(d_count, 0, sizeof(int), s));
            for (int c = 0; c < 3; ++c) {
                if (!hb[c]) continue;
                int hcap = caps[c];
                bool grp = c == 0;   // small rows: 8 lanes per row, 4 rows per warp
                int spw = grp ? 4 : 1;
                int wpb = std::max(1, std::min(16, (200 * 1024) / (hcap * 12 * spw)));
                size_t sm = (size_t)hcap * wpb * spw * (sizeof(double) + sizeof(int));
                unsigned grid = std::min<unsigned>(blocks_for(hb[c], wpb * spw), 152u * 32u);
                if (grp) {
                    allow_max_dyn_smem(k_rap<8, false>);
                    k_rap<8, false><<<grid, 32 * wpb, sm, s>>>(hb[c], rlist + bstart[c], L.cpts, L.zrowptr, L.zcol,
                                                               L.zval, L.rowptr, aplen, apcol, apval, uptr, U, filt,
                                                               prm.phi_A, cnt, ucol, uval, hcap, nullptr, nullptr,
                                                               nullptr, d_count, h.d_err);
                } else {
                    allow_max_dyn_smem(k_rap<32, false>);
                    k_rap<32, false><<<grid, 32 * wpb, sm, s>>>(hb[c], rlist + bstart[c], L.cpts, L.zrowptr, L.zcol,
                                                                L.zval, L.rowptr, aplen, apcol, apval, uptr, U, filt,
                                                                prm.phi_A, cnt, ucol, uval, hcap, nullptr, nullptr,
                                                                nullptr, d_count, h.d_err);
                }
                PR_LAUNCH();
            }
            int nover = hb[3];
            if (nover > 0) {
                int *list = rlist + bstart[3];
                long long *capw = dmalloc<long long>(nover + 1, s);
                k_overflow_caps<<<blocks_for(nover, BS), BS, 0, s>>>(nover, list, U, capw);
                PR_LAUNCH();
                const long long gtot = scan_exclusive_ll(capw, nover, s);
                int *gk = dmalloc<int>(gtot, s);
                double *gv = dmalloc<double>(gtot, s);
                k_rap<32, true><<<std::min<unsigned>(nover, 152u * 16u), 32, 0, s>>>(
                    nover, list, L.cpts, L.zrowptr, L.zcol, L.zval, L.rowptr, aplen, apcol, apval, uptr, U, filt,
                    prm.phi_A, cnt, ucol, uval, 0, capw, gk, gv, d_count, h.d_err);
                PR_LAUNCH();
                dfree(gk, s); dfree(gv, s); dfree(capw, s);
            }
            int nrej = 0;
            d2h(&nrej, d_count, 1, s);
            PR_REQUIRE(nrej == 0, PAIR_ERR_DEVICE, "RAP row exceeded its table bin");
            dfree(rlist, s);
        }
        Level C;
        C.n = nc;
        C.rowptr = dmalloc<int>(nc + 1, s);
        C.nnz = scan_exclusive(cnt, C.rowptr, nc, s);
        C.col = dmalloc<int>(C.nnz, s);
        C.val = dmalloc<double>(C.nnz, s);
        k_compact_rows<<<blocks_for(8LL * nc, BS), BS, 0, s>>>(nc, uptr, C.rowptr, ucol, uval, C.col, C.val);
        PR_LAUNCH();
        dfree(ucol, s); dfree(uval, s); dfree(uptr, s); dfree(U, s); dfree(cnt, s);
        dfree(aplen, s); dfree(apcol, s); dfree(apval, s);
        C.rowdir = dmalloc<int>(nc, s);
        k_gather_rowdir<<<blocks_for(nc, BS), BS, 0, s>>>(nc, L.cpts, L.rowdir, C.rowdir);
        PR_LAUNCH();
        // nnz of Z per matrix (host, from the Z row pointer at the coarse row ranges)
        {
            C.row0.assign(ND, 0);
            C.nrows.assign(ND, 0);
            std::vector<int> bidx(ND + 1);
            int r = 0;
            for (int d = 0; d < ND; ++d) {
                C.row0[d] = r;
                C.nrows[d] = cont[d] ? L.ncdir[d] : 0;
                bidx[d] = r;
                r += C.nrows[d];
            }
            bidx[ND] = r;
            int *didx = dmalloc<int>(ND + 1, s), *dz = dmalloc<int>(ND + 1, s);
            PR_CUDA(cudaMemcpyAsync(didx, bidx.data(), sizeof(int) * (ND + 1), cudaMemcpyHostToDevice, s));
            k_gather_int<<<blocks_for(ND + 1, BS), BS, 0, s>>>(ND + 1, L.zrowptr, didx, dz);
            PR_LAUNCH();
            std::vector<int> zb(ND + 1);
            d2h(zb.data(), dz, ND + 1, s);   // also orders the host copy of bidx before it is freed
            for (int d = 0; d < ND; ++d) L.nnzZdir[d] = zb[d + 1] - zb[d];
            dfree(didx, s);
            dfree(dz, s);
        }
        C.d_row0 = dmalloc<int>(ND, s);
        PR_CUDA(cudaMemcpyAsync(C.d_row0, C.row0.data(), sizeof(int) * ND, cudaMemcpyHostToDevice, s));
        PR_CUDA(cudaEventRecord(ev[3], s));
        h.t_phase[0] += phase_ms(0, 1);
        h.t_phase[1] += phase_ms(1, 2);
        h.t_phase[2] += phase_ms(2, 3);
        finish_segments(h, L);
        h.lev.push_back(C);
    }
    int err = 0;
    d2h(&err, h.d_err, 1, s);
    dfree(d_count, s); dfree(dwork, s); dfree(dcont, s); dfree(dnc, s); dfree(dnnz, s);
    PR_REQUIRE(err == 0, PAIR_ERR_DEVICE, "setup kernel reported device error bits " + std::to_string(err));
    // V-cycle storage in the cycle precision: the CF split with SELL copies of the F
    // and C rows (the block-form level 0 relaxes without them) and of Z
    for (size_t l = 0; l < h.lev.size(); ++l) {
        Level &L = h.lev[l];
        build_split(h, L, !(l == 0 && h.bsr0));
        if (L.n_cseg && L.sX.nrows == 0) coarsest_dense(h, L);
        if (L.nc > 0) {
            build_sell(h, L.sZ, nullptr, L.nc, L.zrowptr, L.zcol, L.zval);
            sell_compress_cols(h, L.sZ, L.cpts);   // offsets from each coarse point's fine row
        }
    }
    PR_CUDA(cudaStreamSynchronize(s));
}

}  // namespace pr
