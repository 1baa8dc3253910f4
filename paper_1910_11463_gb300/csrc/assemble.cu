// Upwind DG assembly on the structured hex Q1 mesh with block-inverse scaling
// (Eq. weak_form_transport; Sec. 1.3).  Compiled with --fmad=false: every
// product and sum below is rounded as written, in the order written (fused
// multiply-adds only where fma() is written), so the scaled operator is
// reproducible bit for bit.
//
// One thread per (element, direction).  Per element K and direction Omega:
//   m1[i][j] = (2 or 1) h / 6,  g1[i][j] = -1/2 (i = 0), +1/2 (i = 1)
//   L_KK[a][b] = sigma_t mass(a,b) - ((mu gx + eta gy) + xi gz)
//                + |Omega_d| face_d(a,b)   on each outflow face (both nodes on it)
//   L_KK'[a][b] = -|Omega_d| face_d(a,b)   a on K's inflow face, b on K''s face
// L_KK is factored by LU with partial pivoting; the stored blocks are
// D_K^{-1} L_KK' (8 x 4, the four columns of the upwind element's face nodes)
// and W_K = D_K^{-1} M_K (8 x 8, for right-hand sides).
#include "common.cuh"

namespace pr {

namespace {

// LU with partial pivoting (first maximum), multipliers a_rk * (1 / a_kk),
// updates fma(-l, a_kc, a_rc); column-oriented substitutions with fma and
// y_k * (1 / u_kk).  The same operation sequence as every LU in the library
// (lu_step, lu_solve below).

struct HexFactors {
    double m1[2][2];
};

__device__ __forceinline__ double face_f(const double (*m1)[2], int d, int a, int b) {
    int ax = a & 1, ay = (a >> 1) & 1, az = (a >> 2) & 1;
    int bx = b & 1, by = (b >> 1) & 1, bz = (b >> 2) & 1;
    return (d == 0) ? m1[ay][by] * m1[az][bz] : (d == 1) ? m1[ax][bx] * m1[az][bz] : m1[ax][bx] * m1[ay][by];
}

// rows of element e in direction m: 8 * (1 + 4 * upwind neighbours)
__global__ void k_hex_rowcounts(int n, int ndir, const double *omega, int *counts) {
    long long E = (long long)n * n * n;
    long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= E * ndir) return;
    int m = (int)(tid / E);
    int e = (int)(tid % E);
    int idx[3] = {e % n, (e / n) % n, e / (n * n)};
    int c = 1;
    for (int d = 0; d < 3; ++d) {
        double o = omega[3 * m + d];
        if (o == 0.0) continue;
        if (o > 0.0 ? idx[d] > 0 : idx[d] < n - 1) c += 4;
    }
    long long r0 = (long long)m * 8 * E + 8LL * e;
    for (int a = 0; a < 8; ++a) counts[r0 + a] = c;
}

// One thread per element, a block within one direction.  What depends on the direction and
// the mesh width alone (mass, advection and outflow-face entries, the right-hand sides of
// the face and mass columns) is formed once per block in shared memory by the expressions
// above, so an element's block is one product, one difference and at most three additions
// an entry.  The factors stay in registers (every index a compile-time one, row exchanges
// as predicated moves), and each group of four solved columns goes through shared memory
// to whole 32-256 byte runs of the outputs.  The FP64 pipe bounds it: about 1700
// operations an element (factorisation 180, twenty solves of 64, 180 for the block) at 2
// lanes a clock and SM.  64^3, 15 directions: 21.3 ms a launch before (2900
// operations, the factors and columns in local memory), 12.4 ms now.
constexpr int HA_BS = 128;

// step K of the factorisation (a template, so that every loop bound and index is a
// constant and D stays in registers)
template <int N, int K = 0>
__device__ __forceinline__ void lu_step(double (&D)[N * N], int (&piv)[N], double (&rinv)[N], int &singular) {
    int p = K;
    long long mx = absbits(D[K * N + K]);
#pragma unroll
    for (int r = K + 1; r < N; ++r) {
        const long long v = absbits(D[r * N + K]);
        if (v > mx) { mx = v; p = r; }
    }
    piv[K] = p;
    if (!(mx > 0)) singular = 1;
    if (p != K) {
#pragma unroll
        for (int r = K + 1; r < N; ++r)
#pragma unroll
            for (int c = 0; c < N; ++c) {
                const double u = D[K * N + c], v = D[r * N + c];
                D[K * N + c] = p == r ? v : u;
                D[r * N + c] = p == r ? u : v;
            }
    }
    const double rd = 1.0 / D[K * N + K];
    rinv[K] = rd;   // row K is final from here on: the back substitution reuses it
#pragma unroll
    for (int r = K + 1; r < N; ++r) {
        const double l = D[r * N + K] * rd;
        D[r * N + K] = l;
#pragma unroll
        for (int c = K + 1; c < N; ++c) D[r * N + c] = fma(-l, D[K * N + c], D[r * N + c]);
    }
    if constexpr (K < N - 1) lu_step<N, K + 1>(D, piv, rinv, singular);
}

template <int N, int K = 0>
__device__ __forceinline__ void lu_swap(const int (&piv)[N], double (&y)[N]) {
#pragma unroll
    for (int r = K + 1; r < N; ++r) {
        const double u = y[K], v = y[r];
        y[K] = piv[K] == r ? v : u;
        y[r] = piv[K] == r ? u : v;
    }
    if constexpr (K < N - 2) lu_swap<N, K + 1>(piv, y);
}
template <int N, int K = 0>
__device__ __forceinline__ void lu_fwd(const double (&D)[N * N], double (&y)[N]) {
#pragma unroll
    for (int r = K + 1; r < N; ++r) y[r] = fma(-D[r * N + K], y[K], y[r]);
    if constexpr (K < N - 2) lu_fwd<N, K + 1>(D, y);
}
template <int N, int K = N - 1>
__device__ __forceinline__ void lu_bwd(const double (&D)[N * N], const double (&rinv)[N], double (&y)[N]) {
    y[K] = y[K] * rinv[K];
#pragma unroll
    for (int r = 0; r < K; ++r) y[r] = fma(-D[r * N + K], y[K], y[r]);
    if constexpr (K > 0) lu_bwd<N, K - 1>(D, rinv, y);
}
template <int N>
__device__ __forceinline__ void lu_solve(const double (&D)[N * N], const int (&piv)[N], const double (&rinv)[N],
                                         double (&y)[N]) {
    lu_swap<N>(piv, y);
    lu_fwd<N>(D, y);
    lu_bwd<N>(D, rinv, y);
}

__global__ void __launch_bounds__(HA_BS) k_hex_assemble(int n, const double *omega, const double *sigma_t,
                                                        const int *rowptr, int *col, double *val, double *bsr64,
                                                        float *bsr32, double *W, double *Gin, int *err) {
    __shared__ double mass[64], adv[64], fo[3][64], fin[3][4][8];
    __shared__ double stage[HA_BS / 32][32][33];   // per lane: [row][column of the group]
    __shared__ int scol[HA_BS / 32][32][4];        // per lane: first entry, row length, offset, first column
    const long long E = (long long)n * n * n;
    const unsigned nbE = (unsigned)((E + HA_BS - 1) / HA_BS);   // blocks of a direction
    const int m = (int)(blockIdx.x / nbE);
    const double om[3] = {omega[3 * m], omega[3 * m + 1], omega[3 * m + 2]};
    const double h = 1.0 / (double)n;
    double m1[2][2];
    for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 2; ++j) m1[i][j] = ((i == j) ? 2.0 : 1.0) * h / 6.0;
    const double g1[2][2] = {{-0.5, -0.5}, {0.5, 0.5}};
    int out[3], in[3];
    for (int d = 0; d < 3; ++d) { out[d] = om[d] > 0.0 ? 1 : 0; in[d] = 1 - out[d]; }
    if (threadIdx.x < 64) {
        const int t = threadIdx.x, a = t >> 3, b = t & 7;
        const int ax = a & 1, ay = (a >> 1) & 1, az = (a >> 2) & 1;
        const int bx = b & 1, by = (b >> 1) & 1, bz = (b >> 2) & 1;
        mass[t] = (m1[ax][bx] * m1[ay][by]) * m1[az][bz];
        const double gx = (g1[ax][bx] * m1[ay][by]) * m1[az][bz];
        const double gy = (m1[ax][bx] * g1[ay][by]) * m1[az][bz];
        const double gz = (m1[ax][bx] * m1[ay][by]) * g1[az][bz];
        adv[t] = (om[0] * gx + om[1] * gy) + om[2] * gz;
        fo[0][t] = fabs(om[0]) * (m1[ay][by] * m1[az][bz]);
        fo[1][t] = fabs(om[1]) * (m1[ax][bx] * m1[az][bz]);
        fo[2][t] = fabs(om[2]) * (m1[ax][bx] * m1[ay][by]);
    } else if (threadIdx.x < 64 + 12) {   // column t of axis d: the upwind element's t-th face node
        const int d = (threadIdx.x - 64) / 4, t = (threadIdx.x - 64) % 4;
        int b = 0, seen = 0;
        for (; b < 8; ++b)
            if (((b >> d) & 1) == out[d] && seen++ == t) break;
        const double w = fabs(om[d]);
        for (int a = 0; a < 8; ++a) fin[d][t][a] = (((a >> d) & 1) != in[d]) ? 0.0 : -(w * face_f(m1, d, a, b));
    }
    __syncthreads();
    const long long e0 = (long long)(blockIdx.x % nbE) * HA_BS + (threadIdx.x & ~31);   // the warp's first element
    const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
    if (e0 >= E) return;   // whole warps
    const bool has = e0 + lane < E;
    const int e = (int)(has ? e0 + lane : E - 1);
    const int nel = (int)min(32LL, E - e0);
    const double st = sigma_t[e];
    double D[64];
    {
        const bool nz[3] = {om[0] != 0.0, om[1] != 0.0, om[2] != 0.0};
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                double v = st * mass[a * 8 + b] - adv[a * 8 + b];
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    if (nz[d] && ((a >> d) & 1) == out[d] && ((b >> d) & 1) == out[d]) v = v + fo[d][a * 8 + b];
                D[a * 8 + b] = v;
            }
    }
    int piv[8];
    double rinv[8];
    int sing = 0;
    lu_step<8>(D, piv, rinv, sing);
    if (sing && has) atomicOr(err, 1);   // (the host stops before anything reads the rows)

    const int idx[3] = {e % n, (e / n) % n, e / (n * n)};
    const int stride[3] = {1, n, n * n};
    // an entry's place in its row: upwind elements and the element itself by index
    bool up[3], low[3];
    int cnt = 1;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        up[d] = om[d] > 0.0 ? idx[d] > 0 : (om[d] < 0.0 && idx[d] < n - 1);
        low[d] = om[d] > 0.0;   // the upwind element has the lower index
        if (up[d]) cnt += 4;
    }
    int off[3], self = 0, run = 0;
#pragma unroll
    for (int d = 2; d >= 0; --d)
        if (up[d] && low[d]) { off[d] = run; run += 4; }
    self = run++;
#pragma unroll
    for (int d = 0; d < 3; ++d)
        if (up[d] && !low[d]) { off[d] = run; run += 4; }
        else if (!up[d]) off[d] = 0;
    const long long N = 8 * E;
    const long long rowbase = (long long)m * N + 8LL * e;
    const int rp = col ? rowptr[rowbase] : 0;   // the element's rows are equally long
    if (col && has)
        for (int a = 0; a < 8; ++a) {
            col[rp + a * cnt + self] = (int)(rowbase + a);
            val[rp + a * cnt + self] = 1.0;
        }
    double(*sg)[33] = stage[wq];
    int(*sc)[4] = scol[wq];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
#pragma unroll 1
        for (int t = 0; t < 4; ++t) {
            double y[8];
#pragma unroll
            for (int a = 0; a < 8; ++a) y[a] = fin[d][t][a];
            lu_solve<8>(D, piv, rinv, y);
#pragma unroll
            for (int a = 0; a < 8; ++a) sg[lane][a * 4 + t] = up[d] ? y[a] : 0.0;
        }
        sc[lane][0] = rp;
        sc[lane][1] = cnt;
        sc[lane][2] = up[d] ? off[d] : -1;
        sc[lane][3] = (int)((long long)m * N) + 8 * (low[d] ? e - stride[d] : e + stride[d]);
        __syncwarp();
        for (int k = lane; k < nel * 32; k += 32) {
            const int el = k >> 5, q = k & 31, a = q >> 2, t = q & 3;
            const double v = sg[el][q];
            const long long at = (((long long)m * E + e0 + el) * 3 + d) * 32 + q;
            if (bsr64) bsr64[at] = v;
            if (bsr32) bsr32[at] = (float)v;
            if (col && sc[el][2] >= 0) {
                // face node t of the upwind element: out on axis d, t's bits on the others
                const int o = out[d];
                const int b = d == 0 ? (o | (t << 1)) : d == 1 ? ((t & 1) | (o << 1) | ((t >> 1) << 2)) : (t | (o << 2));
                const int p = sc[el][0] + a * sc[el][1] + sc[el][2] + t;
                col[p] = sc[el][3] + b;
                val[p] = v;
            }
        }
        __syncwarp();
    }
    if (Gin) {
        // D_K^{-1} sum over boundary inflow faces of |Omega_d| int_F phi_b phi_a (unit inflow)
        double y[8];
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            double acc = 0.0;
            for (int d = 0; d < 3; ++d) {
                if (om[d] == 0.0) continue;
                bool bnd = om[d] > 0.0 ? idx[d] == 0 : idx[d] == n - 1;
                if (!bnd || ((a >> d) & 1) != in[d]) continue;
                double w = fabs(om[d]), s = 0.0;
                for (int b = 0; b < 8; ++b)
                    if (((b >> d) & 1) == in[d]) s = s + w * face_f(m1, d, a, b);
                acc = acc + s;
            }
            y[a] = acc;
        }
        lu_solve<8>(D, piv, rinv, y);
        if (has)
#pragma unroll
            for (int a = 0; a < 8; ++a) Gin[((long long)m * E + e) * 8 + a] = y[a];
    }
    if (W) {
#pragma unroll 1
        for (int g = 0; g < 2; ++g) {
#pragma unroll 1
            for (int t = 0; t < 4; ++t) {
                const int b = 4 * g + t;
                double y[8];
#pragma unroll
                for (int a = 0; a < 8; ++a) y[a] = mass[a * 8 + b];
                lu_solve<8>(D, piv, rinv, y);
#pragma unroll
                for (int a = 0; a < 8; ++a) sg[lane][a * 4 + t] = y[a];
            }
            __syncwarp();
            for (int k = lane; k < nel * 32; k += 32) {
                const int el = k >> 5, q = k & 31;
                W[((long long)m * E + e0 + el) * 64 + (q >> 2) * 8 + 4 * g + (q & 3)] = sg[el][q];
            }
            __syncwarp();
        }
    }
}


// ---- tetrahedra, P1 -----------------------------------------------------------
// Local node a = tet vertex a; face f = the triangle without vertex f.
// e_k = x_k - x_0; c23 = e2 x e3, c31 = e3 x e1, c12 = e1 x e2; det = e1 . c23;
// grad l1 = c23 / det, grad l2 = c31 / det, grad l3 = c12 / det,
// grad l0 = -((grad l1 + grad l2) + grad l3); |K| = |det| / 6; od_a = Omega . grad l_a;
// face flux (Omega.n)|F| = -(od_f (3 |K|)).
// L_KK[a][b] = sigma_t (c_ab |K| / 20) - (od_a |K|) / 4 + sum_{outflow f, a,b != f} (fl_f c_ab) / 12
// L_KK'[a][b'] = (fl_f c) / 12 on the inflow face f (c = 2 on the same vertex, else 1).
// What a tet's geometry alone fixes (the gradients and |K|) is formed once per tet by
// k_tet_geom and read back for every direction: its ten divisions were most of the FP64
// work of an element, again for each of the 24 or 80 directions and again for the row
// counts.
__device__ __forceinline__ void cross3(const double *a, const double *b, double *c) {
    c[0] = a[1] * b[2] - a[2] * b[1];
    c[1] = a[2] * b[0] - a[0] * b[2];
    c[2] = a[0] * b[1] - a[1] * b[0];
}
__device__ __forceinline__ double dot3(const double *a, const double *b) { return (a[0] * b[0] + a[1] * b[1]) + a[2] * b[2]; }

// geometry, one array of T per component: gradients (4 x 3), then |K| (-1: zero volume)
constexpr int TET_GEOM = 13;

__global__ void k_tet_geom(int T, const double *verts, const int *tets, double *geom) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const int *tv = tets + 4LL * t;
    double x[4][3], e[3][3], gr[4][3], c23[3], c31[3], c12[3];
    for (int a = 0; a < 4; ++a)
        for (int k = 0; k < 3; ++k) x[a][k] = verts[3 * tv[a] + k];
    for (int j = 0; j < 3; ++j)
        for (int k = 0; k < 3; ++k) e[j][k] = x[j + 1][k] - x[0][k];
    cross3(e[1], e[2], c23);
    cross3(e[2], e[0], c31);
    cross3(e[0], e[1], c12);
    const double det = dot3(e[0], c23);
    if (det == 0.0) { geom[(TET_GEOM - 1LL) * T + t] = -1.0; return; }
    for (int k = 0; k < 3; ++k) {
        gr[1][k] = c23[k] / det;
        gr[2][k] = c31[k] / det;
        gr[3][k] = c12[k] / det;
        gr[0][k] = -((gr[1][k] + gr[2][k]) + gr[3][k]);
    }
    for (int a = 0; a < 4; ++a)
        for (int k = 0; k < 3; ++k) geom[(3LL * a + k) * T + t] = gr[a][k];
    geom[(TET_GEOM - 1LL) * T + t] = fabs(det) / 6.0;
}

struct TetGeom {
    double od[4], fl[4], vol;
};

__device__ __forceinline__ bool tet_geom(const double *geom, int T, int t, const double *om, TetGeom &g) {
    g.vol = geom[(TET_GEOM - 1LL) * T + t];
    if (g.vol == -1.0) return false;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const double gr[3] = {geom[(3LL * a) * T + t], geom[(3LL * a + 1) * T + t], geom[(3LL * a + 2) * T + t]};
        g.od[a] = dot3(om, gr);
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) g.fl[f] = -(g.od[f] * (3.0 * g.vol));
    return true;
}

__global__ void k_tet_rowcounts(int T, int ndir, const double *omega, const double *geom, const int *nbr, int *counts) {
    long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= (long long)T * ndir) return;
    int m = (int)(tid / T), t = (int)(tid % T);
    const double om[3] = {omega[3 * m], omega[3 * m + 1], omega[3 * m + 2]};
    TetGeom g;
    int c = 1;
    if (tet_geom(geom, T, t, om, g))
        for (int f = 0; f < 4; ++f)
            if (g.fl[f] < 0.0 && nbr[4LL * t + f] >= 0) c += 3;
    *reinterpret_cast<int4 *>(counts + ((long long)m * T + t) * 4) = make_int4(c, c, c, c);
}

// Thread per (tet, direction); the factors in registers, each solved column stored at once.
// FP64-pipe bound.  40^3 x 6 tets, 24 directions, row counts and assembly: 40^3 S4 solve
// 471 -> 454 ms, 20^3 exact sweeps 23.3 -> 20.5 ms against a geometry per (tet, direction)
// and a division per matrix entry.
// (2 x and 1 x |K| / 20, flux / 12 differ by an exact factor of two, so each takes one
// division.)
__global__ void __launch_bounds__(128) k_tet_assemble(int T, int ndir, const double *omega, const double *geom,
                                                      const int *tets, const int *nbr, const double *sigma_t,
                                                      const int *rowptr, int *col, double *val, double *W,
                                                      double *Gin, int *err) {
    long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= (long long)T * ndir) return;
    int m = (int)(tid / T), t = (int)(tid % T);
    const double om[3] = {omega[3 * m], omega[3 * m + 1], omega[3 * m + 2]};
    TetGeom g;
    if (!tet_geom(geom, T, t, om, g)) { atomicOr(err, 1); return; }
    const int4 tv4 = *reinterpret_cast<const int4 *>(tets + 4LL * t);
    const int4 nb4 = *reinterpret_cast<const int4 *>(nbr + 4LL * t);
    const int tv[4] = {tv4.x, tv4.y, tv4.z, tv4.w}, nb[4] = {nb4.x, nb4.y, nb4.z, nb4.w};
    const double st = sigma_t[t];
    const double ms1 = g.vol / 20.0, ms2 = 2.0 * ms1;   // mass entries off and on the diagonal
    double f1[4];                                       // face entries: flux / 12, twice that on the diagonal
#pragma unroll
    for (int f = 0; f < 4; ++f) f1[f] = g.fl[f] / 12.0;
    double D[16];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            double v = st * (a == b ? ms2 : ms1) - g.od[a] * g.vol / 4.0;
#pragma unroll
            for (int f = 0; f < 4; ++f)
                if (g.fl[f] > 0.0 && a != f && b != f) v = v + (a == b ? 2.0 * f1[f] : f1[f]);
            D[a * 4 + b] = v;
        }
    int piv[4], sing = 0;
    double rinv[4];
    lu_step<4>(D, piv, rinv, sing);
    if (sing) { atomicOr(err, 1); return; }
    const long long N = 4LL * T;
    const long long rowbase = (long long)m * N + 4LL * t;
    // an entry's place in its row: upwind tets and the tet itself by index
    bool up[4];
    int len = 1, self = 0;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        up[f] = g.fl[f] < 0.0 && nb[f] >= 0;
        if (up[f]) {
            len += 3;
            if (nb[f] <= t) self += 3;
        }
    }
    const int rp = col ? rowptr[rowbase] : 0;   // the tet's rows are equally long
    if (col)
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            col[rp + a * len + self] = (int)(rowbase + a);
            val[rp + a * len + self] = 1.0;
        }
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        if (!up[f]) continue;
        int off = nb[f] > t ? 1 : 0;
#pragma unroll
        for (int h = 0; h < 4; ++h)
            if (h != f && up[h] && (nb[h] < nb[f] || (nb[h] == nb[f] && h < f))) off += 3;
        const int4 u4 = *reinterpret_cast<const int4 *>(tets + 4LL * nb[f]);
        const int uv[4] = {u4.x, u4.y, u4.z, u4.w};
        int u = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            bool onface = false;
#pragma unroll
            for (int a = 0; a < 4; ++a) onface |= a != f && tv[a] == uv[b];
            if (!onface || u >= 3) continue;
            double y[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) y[a] = a == f ? 0.0 : tv[a] == uv[b] ? 2.0 * f1[f] : f1[f];
            lu_solve<4>(D, piv, rinv, y);
            if (col)
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    col[rp + a * len + off + u] = (int)((long long)m * N + 4LL * nb[f] + b);
                    val[rp + a * len + off + u] = y[a];
                }
            ++u;
        }
        if (u != 3) atomicOr(err, 2);
    }
    if (Gin) {
        // D^{-1} (boundary inflow faces: sum_b |fl_f| c_ab / 12, unit inflow)
        double y[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            double acc = 0.0;
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                if (!(g.fl[f] < 0.0) || nb[f] >= 0 || a == f) continue;
                double s2 = 0.0;
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (b != f) s2 = s2 + -(a == b ? 2.0 * f1[f] : f1[f]);
                acc = acc + s2;
            }
            y[a] = acc;
        }
        lu_solve<4>(D, piv, rinv, y);
#pragma unroll
        for (int a = 0; a < 4; ++a) Gin[((long long)m * T + t) * 4 + a] = y[a];
    }
    if (W) {
        double *We = W + ((long long)m * T + t) * 16;
        double w[16];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            double y[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) y[a] = a == b ? ms2 : ms1;
            lu_solve<4>(D, piv, rinv, y);
#pragma unroll
            for (int a = 0; a < 4; ++a) w[a * 4 + b] = y[a];
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) reinterpret_cast<double2 *>(We)[q] = make_double2(w[2 * q], w[2 * q + 1]);
    }
}

}  // namespace

// Assembles 'ndir' directions (omega: device [ndir][3]).  Any output may be
// null.  CSR: rowptr (ndir * 8 n^3 + 1), col/val (hex_nnz entries), rows and
// columns offset by m * 8 n^3.  Block form: bsr64/bsr32 [dir][elem][axis][a][4].
// W [dir][elem][8][8] = D^{-1} M.  Gin [dir][N] = D^{-1} (unit boundary inflow).
void hex_assemble(int n, int ndir, const double *omega_d, const double *sigma_t, int *rowptr, int *col,
                  double *val, double *bsr64, float *bsr32, double *W, double *Gin, int *d_err, cudaStream_t s) {
    long long E = (long long)n * n * n;
    long long rows = 8 * E * ndir;
    PR_REQUIRE(rows < 0x7fffffffLL, PAIR_ERR_UNSUPPORTED, "hex batch has more than 2^31 rows");
    if (rowptr) {
        int *counts = dmalloc<int>(rows, s);
        k_hex_rowcounts<<<blocks_for(E * ndir, 256), 256, 0, s>>>(n, ndir, omega_d, counts);
        PR_LAUNCH();
        scan_exclusive(counts, rowptr, (int)rows, s, false);
        dfree(counts, s);
    }
    k_hex_assemble<<<blocks_for(E, HA_BS) * ndir, HA_BS, 0, s>>>(n, omega_d, sigma_t, rowptr, col, val, bsr64, bsr32, W,
                                                                 Gin, d_err);
    PR_LAUNCH();
}

// Tetrahedral mesh, 'ndir' directions: CSR (rows/cols offset by m * 4T), W
// [dir][tet][4][4] = D^{-1} M, Gin [dir][4T].  TET_ROWPTR computes the row pointer and
// returns nnz; TET_VALUES assembles on a row pointer it computed (returns 0).
long long tet_assemble(int T, int ndir, const double *omega_d, const double *verts, const int *tets, const int *nbr,
                       const double *sigma_t, int *rowptr, int *col, double *val, double *W, double *Gin, int *d_err,
                       cudaStream_t s, TetPass pass) {
    long long rows = 4LL * T * ndir;
    PR_REQUIRE(rows < 0x7fffffffLL, PAIR_ERR_UNSUPPORTED, "tet batch has more than 2^31 rows");
    // the kernels read tets and nbr as int4: caller arrays that are not 16-byte aligned are
    // copied first
    int *ctets = nullptr, *cnbr = nullptr;
    auto aligned = [&](const int *p, int *&copy) -> const int * {
        if (reinterpret_cast<uintptr_t>(p) % 16 == 0) return p;
        copy = dmalloc<int>(4LL * T, s);
        PR_CUDA(cudaMemcpyAsync(copy, p, sizeof(int) * 4LL * T, cudaMemcpyDeviceToDevice, s));
        return copy;
    };
    const int *at = pass == TET_VALUES ? aligned(tets, ctets) : tets;
    const int *an = pass == TET_VALUES ? aligned(nbr, cnbr) : nbr;
    double *geom = dmalloc<double>((size_t)TET_GEOM * T, s);
    k_tet_geom<<<blocks_for(T, 128), 128, 0, s>>>(T, verts, at, geom);
    PR_LAUNCH();
    long long nnz = 0;
    if (pass == TET_ROWPTR) {
        int *counts = dmalloc<int>(rows, s);
        k_tet_rowcounts<<<blocks_for((long long)T * ndir, 256), 256, 0, s>>>(T, ndir, omega_d, geom, an, counts);
        PR_LAUNCH();
        nnz = scan_exclusive(counts, rowptr, (int)rows, s);
        dfree(counts, s);
    } else {
        k_tet_assemble<<<blocks_for((long long)T * ndir, 128), 128, 0, s>>>(T, ndir, omega_d, geom, at, an, sigma_t,
                                                                            rowptr, col, val, W, Gin, d_err);
        PR_LAUNCH();
    }
    dfree(geom, s);
    dfree(ctets, s);
    dfree(cnbr, s);
    return nnz;
}

// Stored entries of the scaled operator of one direction (closed form).
long long hex_nnz(int n, const double *omega_h) {
    long long E = (long long)n * n * n, nnz = 8 * E;
    for (int d = 0; d < 3; ++d)
        if (omega_h[d] != 0.0) nnz += 32LL * n * n * (n - 1);
    return nnz;
}

}  // namespace pr
