// Grid side of the PIC step: metric tables at the Yee points (Sec. 2.1),
// the stable sort of particles by cell, the deterministic volume-weighted
// deposit (Sec. 2.3) and the FDTD leapfrog (Sec. 2.1, 2.5).
//
// Deposit pipeline (no floating-point atomics, bitwise reproducible):
//   k_dep_particle  one thread per particle (in cell order): the 4x4
//                   trapezoidal subvolumes of sqrt(gamma) on each sub-grid
//                   -> 16 node shares (rho, j^ph, j^r, j^th); on fine grids
//                   from per-cell polynomials (dep_poly.cuh);
//   k_dep_cell      one warp per cell, one lane per record row and
//                   particle parity: fixed-order sums of the cell's
//                   particles' shares into its 20 stencil slots;
//   k_dep_node      one thread per node: fixed-order sum of the slots of the
//                   (up to six) cells touching it, / (2 pi V_dual).
// The FDTD's metric factors come from tables built once.
#include <math.h>
#include <string.h>

#include "dep_poly.cuh"
#include "fpic_internal.h"

namespace fpic {

// ---------------------------------------------------------------------------
// Metric tables
// ---------------------------------------------------------------------------
// Points: 0 (i, j), 1 (i+1/2, j), 2 (i, j+1/2), 3 (i+1/2, j+1/2).  First what
// cleaning and the deposits read: sqrt(gamma), g^rph, g^rr, g^thth, 2 pi x the
// dual-cell volumes; then the field update's coefficients (see the FDTD
// section), each product of metric factors, average weights and reciprocal
// spacings formed once: 11 FP64 operations for E or H at a node instead of
// 35, and no factor read that is not used as it is.  Then sin/cos of the
// integer and half th nodes.
enum {
    T_SG0, T_SG1, T_SG2, T_URP0, T_URR1, T_UTT2, T_DUAL0, T_DUAL1, T_DUAL2,
    // E_r = ER_D D^r + ER_P0 D^ph_i + ER_P1 D^ph_{i+1}; E_th, E_ph alike (0: row i - 1, 1: row i, held at the ends)
    F_ER_D, F_ER_P0, F_ER_P1, F_ET_D, F_ET_B0, F_ET_B1, F_EP_D, F_EP_R0, F_EP_R1, F_EP_T0, F_EP_T1,
    F_HR_B, F_HR_P0, F_HR_P1, F_HT_B, F_HT_D0, F_HT_D1, F_HP_B, F_HP_R0, F_HP_R1, F_HP_T0, F_HP_T1,
    // curls: 1 / (sqrt(gamma) x spacing)
    F_BR, F_BT, F_BPR, F_BPT, F_DR, F_DT, F_DPR, F_DPT,
    // -4 pi J, J = alpha j - rho beta: JR j^r + JR0 rho_i + JR1 rho_{i+1}, JT j^th, JP j^ph
    F_JR, F_JR0, F_JR1, F_JT, F_JP,
    MT_N
};

struct Tabs {
    const double* m;   // MT_N tables of size sz, then 2 (Nth+1) + 2 Nth trig values
    size_t sz;
    int ld;
    __device__ __forceinline__ double at(int t, int i, int j) const
    {
        return m[(size_t)t * sz + (size_t)i * ld + j];
    }
};

__device__ __forceinline__ double sqrtg_sc(const BH& bh, double r, double s, double c)
{
    // sqrt(gamma) = rho^2 sqrt(xi) sin th = sin th sqrt(rho^2 (rho^2 + 2 M r))
    const double rho2 = fma(bh.a2, c * c, r * r);
    return s * sqrt(rho2 * fma(bh.twoM, r, rho2));
}

__device__ double trap16_dev(const BH& bh, double x0, double x1, double y0, double y1)
{
    const double wt[4] = {0.5, 1.0, 1.0, 0.5};
    const double hx = (x1 - x0) / 3.0, hy = (y1 - y0) / 3.0;
    double acc = 0.0;
    for (int l = 0; l < 4; ++l) {
        double s, c;
        sincos(y0 + l * hy, &s, &c);
        double row = 0.0;
        for (int k = 0; k < 4; ++k) row = fma(wt[k], sqrtg_sc(bh, x0 + k * hx, s, c), row);
        acc = fma(wt[l], row, acc);
    }
    return acc * hx * hy;
}

// A thread walks `rows` rows of one th column: the trigonometry of its
// points and of the dual cells' quadrature is taken once, and each row's
// metric serves the averages of its neighbours.
__device__ __forceinline__ double dual_sum(const BH& bh, double x0, double x1, double dy, const double s[4],
                                           const double A[4])
{
    const double hx = (x1 - x0) / 3.0;
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double x = x0 + k * hx, X = x * x;
        double row = 0.0;
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            const double P = X + A[l], q = P * fma(bh.twoM, x, P);
            const double f = s[l] * (q * rsqrt_nr(q));
            row += (l == 0 || l == 3) ? 0.5 * f : f;
        }
        acc += (k == 0 || k == 3) ? 0.5 * row : row;
    }
    return 2.0 * M_PI * acc * hx * (dy / 3.0);
}

__global__ void __launch_bounds__(128) k_metric_tables(BH bh, GridDev G, double* m, size_t sz, int rows)
{
    const int j = blockIdx.x * 128 + threadIdx.x, i0 = blockIdx.y * rows, i1 = min(i0 + rows, G.Nr + 1);
    if (j > G.Nth) return;
    const bool in = j < G.Nth;               // half th points exist
    const double mfpi = -4.0 * M_PI;
    double sn, cn, sh, ch;
    sincos(G.tn[j], &sn, &cn);
    sincos(G.th[j], &sh, &ch);
    if (blockIdx.y == 0) {
        double* trig = m + (size_t)MT_N * sz;
        trig[j] = sn;
        trig[(G.Nth + 1) + j] = cn;
        if (in) {
            trig[2 * (G.Nth + 1) + j] = sh;
            trig[2 * (G.Nth + 1) + G.Nth + j] = ch;
        }
    }
    // th lattices of the dual cells about the integer and the half node
    double sa[4], Aa[4], sb[4], Ab[4];
    const double ya0 = j == 0 ? G.tn[0] : G.th[j - 1], ya1 = in ? G.th[j] : G.tn[G.Nth];
    const double yb0 = G.tn[j], yb1 = in ? G.tn[j + 1] : yb0;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        double s, c;
        sincos(ya0 + l * ((ya1 - ya0) / 3.0), &s, &c);
        sa[l] = s;
        Aa[l] = bh.a2 * c * c;
        sincos(yb0 + l * ((yb1 - yb0) / 3.0), &s, &c);
        sb[l] = s;
        Ab[l] = bh.a2 * c * c;
    }
    const double itn = in ? G.itn[j] : 0.0, ith = G.ith[j > 0 ? j - 1 : G.Nth - 1];
    Geo g0, g1, g2, g3, n0, n2;
    double s1m, s3m;                         // sqrt(gamma) of points 1 and 3 one row below (held at row 0)
    geo_eval(bh, G.rn[i0], sn, cn, g0);
    geo_eval(bh, G.rn[i0], sh, ch, g2);
    {
        const int im = max(i0 - 1, 0);
        geo_eval(bh, G.rh[im], sn, cn, g1);
        s1m = g1.sqrtg;
        geo_eval(bh, G.rh[im], sh, ch, g3);
        s3m = g3.sqrtg;
    }
    for (int i = i0; i < i1; ++i) {
        const bool half = i < G.Nr;          // half r points exist
        double* o = m + (size_t)i * G.ld + j;
        auto put = [&](int t, double v) { o[(size_t)t * sz] = v; };
        const double x0 = i == 0 ? G.rn[0] : G.rh[i - 1], x1 = half ? G.rh[i] : G.rn[G.Nr];
        if (half) {
            geo_eval(bh, G.rh[i], sn, cn, g1);
            geo_eval(bh, G.rh[i], sh, ch, g3);
            geo_eval(bh, G.rn[i + 1], sn, cn, n0);
            geo_eval(bh, G.rn[i + 1], sh, ch, n2);
        }
        const double s1 = half ? g1.sqrtg : s1m, s3 = half ? g3.sqrtg : s3m;    // held at the last row
        const double irn = half ? G.irn[i] : 0.0, irh = (i >= 1 && half) ? G.irh[i - 1] : 0.0;
        {   // (i, j)
            const double is = 1.0 / g0.sqrtg, k = 0.5 * g0.alpha * g0.grp * is;
            put(T_SG0, g0.sqrtg);
            put(T_URP0, g0.gurp);
            put(T_DUAL0, dual_sum(bh, x0, x1, ya1 - ya0, sa, Aa));
            put(F_EP_D, g0.alpha * g0.gpp);
            put(F_EP_R0, k * s1m);
            put(F_EP_R1, k * s1);
            put(F_EP_T0, 0.5 * g0.beta * s1m);
            put(F_EP_T1, 0.5 * g0.beta * s1);
            put(F_DPR, irh * is);
            put(F_DPT, ith * is);
            put(F_JP, mfpi * g0.alpha);
        }
        if (in) {   // (i, j+1/2)
            const double is = 1.0 / g2.sqrtg, k = 0.5 * g2.alpha * g2.grp * is;
            put(T_SG2, g2.sqrtg);
            put(T_UTT2, g2.gutt);
            put(T_DUAL2, dual_sum(bh, x0, x1, yb1 - yb0, sb, Ab));
            put(F_ET_D, g2.alpha * g2.gtt);
            put(F_ET_B0, -0.5 * g2.beta * s3m);
            put(F_ET_B1, -0.5 * g2.beta * s3);
            put(F_HR_B, g2.alpha * g2.grr);
            put(F_HR_P0, k * s3m);
            put(F_HR_P1, k * s3);
            put(F_BR, itn * is);
            put(F_DT, irh * is);
            put(F_JT, mfpi * g2.alpha);
        }
        if (half) {   // (i+1/2, j)
            const double is = 1.0 / g1.sqrtg, k = 0.5 * g1.alpha * g1.grp * is;
            put(T_SG1, g1.sqrtg);
            put(T_URR1, g1.gurr);
            put(T_DUAL1, dual_sum(bh, G.rn[i], G.rn[i + 1], ya1 - ya0, sa, Aa));
            put(F_ER_D, g1.alpha * g1.grr);
            put(F_ER_P0, k * g0.sqrtg);
            put(F_ER_P1, k * n0.sqrtg);
            put(F_HT_B, g1.alpha * g1.gtt);
            put(F_HT_D0, 0.5 * g1.beta * g0.sqrtg);
            put(F_HT_D1, 0.5 * g1.beta * n0.sqrtg);
            put(F_BT, irn * is);
            put(F_DR, ith * is);
            put(F_JR, mfpi * g1.alpha);
            put(F_JR0, -0.5 * mfpi * g1.beta * is * g0.sqrtg);
            put(F_JR1, -0.5 * mfpi * g1.beta * is * n0.sqrtg);
        }
        if (half && in) {   // (i+1/2, j+1/2)
            const double is = 1.0 / g3.sqrtg, k = 0.5 * g3.alpha * g3.grp * is;
            put(F_HP_B, g3.alpha * g3.gpp);
            put(F_HP_R0, k * g2.sqrtg);
            put(F_HP_R1, k * n2.sqrtg);
            put(F_HP_T0, -0.5 * g3.beta * g2.sqrtg);
            put(F_HP_T1, -0.5 * g3.beta * n2.sqrtg);
            put(F_BPR, irn * is);
            put(F_BPT, itn * is);
        }
        s1m = s1;
        s3m = s3;
        g0 = n0;
        g2 = n2;
    }
}

int build_metric_tables(fpic_ctx* c)
{
    const size_t sz = (size_t)(c->Nr + 1) * c->ld;
    const size_t tot = (size_t)MT_N * sz + 2 * (size_t)(c->Nth + 1) + 2 * (size_t)c->Nth;
    retire(c, (void**)&c->d_metric);
    FPIC_CUDA(cudaMalloc(&c->d_metric, tot * sizeof(double)));
    c->metric_stride = sz;
    // the trigonometry of a thread costs about two rows: as few rows as keep
    // two blocks on every SM, 16 at most
    const long long cols = c->Nth / 128 + 1;
    int rows = 16;
    while (rows > 1 && cols * (c->Nr / rows + 1) < 2LL * c->sm_count) rows >>= 1;
    k_metric_tables<<<dim3((unsigned)cols, (unsigned)(c->Nr / rows + 1)), 128>>>(c->bh, c->G, c->d_metric, sz, rows);
    FPIC_CUDA(cudaGetLastError());
    return 0;
}

// ---------------------------------------------------------------------------
// Stable sort by cell
// ---------------------------------------------------------------------------
struct SortBufs {
    uint32_t *key, *perm, *perm2, *count, *cursor, *off, *bsum;
    void* tmp;
};

// count[k] += 1 for each valid lane's key k, one atomic per distinct key of
// the warp (particles arrive nearly sorted by cell: most of a warp shares one
// key, and same-address atomics would serialise).  Every lane of the warp
// calls it; an invalid lane's 64-bit key matches no valid one.
__device__ __forceinline__ void count_key(uint32_t* count, uint32_t k, bool valid)
{
    const unsigned peers = __match_any_sync(0xffffffffu, valid ? (unsigned long long)k : (1ull << 32));
    if (valid && (threadIdx.x & 31) == (unsigned)(__ffs(peers) - 1)) atomicAdd(&count[k], (unsigned)__popc(peers));
}

__global__ void k_keys(GridDev G, const double* r, const double* th, const uint8_t* alive, uint32_t* key,
                       uint32_t* cell, uint32_t* count, long long n, uint32_t C)
{
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const bool valid = p < n;
    uint32_t k = 0;
    if (valid) {
        int i, j;
        double w;
        const double rr = r[p];
        double tt, thv;
        int mh;
        theta_views(G, th[p], tt, thv, mh);
        const float lr = __logf((float)rr);
        locate(G.rn, G.irn, G.Nr + 1, rr, (lr - G.lr0) * G.ilr, i, w);
        locate(G.tn, G.itn, G.Nth + 1, tt, ((float)tt - G.t0) * G.it, j, w);
        const uint32_t c = (uint32_t)i * (uint32_t)G.Nth + (uint32_t)j;
        if (cell) cell[p] = c;
        k = alive[p] ? c : C;
        key[p] = k;
    }
    count_key(count, k, valid);
}

// exclusive scan of count[0..m) into off[0..m], m + 1 outputs; three phases
constexpr int SCAN_B = 1024, SCAN_PER = 4;
__global__ void k_scan_blocks(const uint32_t* in, uint32_t* out, uint32_t* bsum, long long m)
{
    __shared__ uint32_t sh[SCAN_B];
    const long long base = (long long)blockIdx.x * SCAN_B * SCAN_PER;
    uint32_t v[SCAN_PER], tot = 0;
    for (int k = 0; k < SCAN_PER; ++k) {
        const long long idx = base + (long long)threadIdx.x * SCAN_PER + k;
        v[k] = idx < m ? in[idx] : 0u;
        tot += v[k];
    }
    sh[threadIdx.x] = tot;
    __syncthreads();
    for (int o = 1; o < SCAN_B; o <<= 1) {
        uint32_t t = threadIdx.x >= (unsigned)o ? sh[threadIdx.x - o] : 0u;
        __syncthreads();
        sh[threadIdx.x] += t;
        __syncthreads();
    }
    uint32_t run = sh[threadIdx.x] - tot;   // exclusive prefix of this thread
    for (int k = 0; k < SCAN_PER; ++k) {
        const long long idx = base + (long long)threadIdx.x * SCAN_PER + k;
        if (idx < m) out[idx] = run;
        run += v[k];
    }
    if (threadIdx.x == SCAN_B - 1) bsum[blockIdx.x] = sh[SCAN_B - 1];
}

// In-place exclusive scan of bsum[0..nb), bsum[nb] = the total: one block of
// SCAN_B threads, each over a contiguous run of ceil(nb / SCAN_B) entries.
__global__ void __launch_bounds__(SCAN_B) k_scan_bsum(uint32_t* bsum, int nb)
{
    __shared__ uint32_t wsum[SCAN_B / 32];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int per = (nb + SCAN_B - 1) / SCAN_B;
    const int lo = min(nb, t * per), hi = min(nb, lo + per);
    uint32_t tot = 0;
    for (int b = lo; b < hi; ++b) tot += bsum[b];
    uint32_t inc = tot;                 // inclusive scan of the thread totals
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        uint32_t w = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    uint32_t run = inc - tot + (wid > 0 ? wsum[wid - 1] : 0u);
    for (int b = lo; b < hi; ++b) {
        const uint32_t v = bsum[b];
        bsum[b] = run;
        run += v;
    }
    if (t == SCAN_B - 1) bsum[nb] = run;
}

__global__ void k_scan_add(uint32_t* out, const uint32_t* bsum, long long m, int nb)
{
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx < m) out[idx] += bsum[idx / (SCAN_B * SCAN_PER)];
    if (idx == 0) out[m] = bsum[nb];
}

__global__ void k_scatter(const uint32_t* key, const uint32_t* off, uint32_t* cursor, uint32_t* perm, long long n)
{
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const bool valid = p < n;
    const uint32_t k = valid ? key[p] : 0u;
    // one atomic per distinct key of the warp; lanes of a key take
    // consecutive places in lane order (every lane takes part in the match)
    const unsigned peers = __match_any_sync(0xffffffffu, valid ? (unsigned long long)k : (1ull << 32));
    const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (valid && lane == leader) base = atomicAdd(&cursor[k], (unsigned)__popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (valid) perm[off[k] + base + (uint32_t)__popc(peers & ((1u << lane) - 1u))] = (uint32_t)p;
}

// Order a bucket (perm[b0] .. perm[b1 - 1]) by particle index (rank = number of
// smaller indices in the bucket), by a warp.
__device__ __forceinline__ void rank_bucket(uint32_t b0, uint32_t b1, const uint32_t* perm, uint32_t* perm2)
{
    const int lane = threadIdx.x & 31;
    // a bucket already in index order (the usual case: nearly sorted input,
    // whole warps placed in lane order) is copied as it is
    bool sorted = true;
    for (uint32_t a = b0 + lane; a + 1 < b1; a += 32) sorted = sorted && perm[a] < perm[a + 1];
    if (__all_sync(0xffffffffu, sorted)) {
        for (uint32_t a = b0 + lane; a < b1; a += 32) perm2[a] = perm[a];
        return;
    }
    for (uint32_t a = b0 + lane; a < b1; a += 32) {
        const uint32_t x = perm[a];
        uint32_t rank = 0;
        for (uint32_t b = b0; b < b1; ++b) rank += perm[b] < x ? 1u : 0u;
        perm2[b0 + rank] = x;
    }
}

// Every bucket, one warp per cell: its one bucket, or (SETS 2) the two of the
// cell, C apart.  Removed particles (last bucket) are handled by k_dead_rank.
template <int SETS>
__global__ void k_bucket_rank(const uint32_t* off, const uint32_t* perm, uint32_t* perm2, uint32_t C)
{
    const long long cell = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    if (cell >= C) return;
    const uint32_t c0 = SETS > 1 ? off[(size_t)C + cell] : 0u, c1 = SETS > 1 ? off[(size_t)C + cell + 1] : 0u;
    rank_bucket(off[cell], off[cell + 1], perm, perm2);
    if (SETS > 1) rank_bucket(c0, c1, perm, perm2);
}

// Removed particles keep their relative order: position = off[C] + number of
// removed particles with a smaller index.  Blocks of DEAD_T threads cover
// DEAD_PER x DEAD_T consecutive particles (thread t takes particles
// base + k DEAD_T + t); k_dead_count writes each block's count, an exclusive
// scan turns the counts into block offsets, and k_dead_place ranks the
// block's removed particles by ballots in index order.
constexpr int DEAD_T = 256, DEAD_PER = 16, DEAD_W = DEAD_T / 32;

__global__ void __launch_bounds__(DEAD_T) k_dead_count(const uint8_t* alive, uint32_t* bcnt, long long n)
{
    __shared__ uint32_t ws[DEAD_W];
    const long long base = (long long)blockIdx.x * DEAD_PER * DEAD_T;
    uint32_t d = 0;
#pragma unroll
    for (int k = 0; k < DEAD_PER; ++k) {
        const long long q = base + (long long)k * DEAD_T + threadIdx.x;
        d += (q < n && !alive[q]) ? 1u : 0u;
    }
    d = __reduce_add_sync(0xffffffffu, d);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = d;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < DEAD_W; ++w) t += ws[w];
        bcnt[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(DEAD_T) k_dead_place(const uint8_t* alive, const uint32_t* boff,
                                                       const uint32_t* off, uint32_t* perm2, long long n, uint32_t C)
{
    __shared__ uint32_t pre[DEAD_PER * DEAD_W];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long base = (long long)blockIdx.x * DEAD_PER * DEAD_T;
    unsigned m[DEAD_PER];
#pragma unroll
    for (int k = 0; k < DEAD_PER; ++k) {
        const long long q = base + (long long)k * DEAD_T + threadIdx.x;
        m[k] = __ballot_sync(0xffffffffu, q < n && !alive[q]);
        if (lane == 0) pre[k * DEAD_W + wid] = (uint32_t)__popc(m[k]);
    }
    __syncthreads();
    if (threadIdx.x == 0) {             // exclusive prefix in index order (k, then warp)
        uint32_t run = 0;
        for (int e = 0; e < DEAD_PER * DEAD_W; ++e) {
            const uint32_t v = pre[e];
            pre[e] = run;
            run += v;
        }
    }
    __syncthreads();
    const uint32_t at = off[C] + boff[blockIdx.x];
#pragma unroll
    for (int k = 0; k < DEAD_PER; ++k)
        if ((m[k] >> lane) & 1u) {
            const long long q = base + (long long)k * DEAD_T + threadIdx.x;
            perm2[at + pre[k * DEAD_W + wid] + (uint32_t)__popc(m[k] & ((1u << lane) - 1u))] = (uint32_t)q;
        }
}

template <typename T>
__global__ void k_gather_perm(const T* __restrict__ src, T* __restrict__ dst, const uint32_t* __restrict__ perm,
                              long long n)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < n) dst[i] = src[perm[i]];
}

// Every particle array permuted at once (the deposit's sort): one pass
// gathers them all through the permutation into a staging area (11 x n
// doubles, then n u32, then 3 x n bytes), reading the permutation once, and
// one pass copies them back, instead of a gather and a copy per array.
struct PermArrays {
    double* d[11];
    uint8_t* b[3];
    uint32_t* u;
};

__global__ void k_gather_all(PermArrays a, const uint32_t* __restrict__ perm, double* __restrict__ stage, long long n)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t j = perm[i];
    uint32_t* su = (uint32_t*)(stage + 11 * n);
    uint8_t* sb = (uint8_t*)(su + n);
#pragma unroll
    for (int k = 0; k < 11; ++k)
        if (a.d[k]) stage[k * n + i] = a.d[k][j];
    if (a.u) su[i] = a.u[j];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (a.b[k]) sb[k * n + i] = a.b[k][j];
}

__global__ void k_copy_all(PermArrays a, const double* __restrict__ stage, long long n)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t* su = (const uint32_t*)(stage + 11 * n);
    const uint8_t* sb = (const uint8_t*)(su + n);
#pragma unroll
    for (int k = 0; k < 11; ++k)
        if (a.d[k]) a.d[k][i] = stage[k * n + i];
    if (a.u) a.u[i] = su[i];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (a.b[k]) a.b[k][i] = sb[k * n + i];
}

static int scan_u32(const uint32_t* in, uint32_t* out, uint32_t* bsum, long long m, cudaStream_t s)
{
    const int nb = (int)((m + SCAN_B * SCAN_PER - 1) / (SCAN_B * SCAN_PER));
    k_scan_blocks<<<nb, SCAN_B, 0, s>>>(in, out, bsum, m);
    k_scan_bsum<<<1, SCAN_B, 0, s>>>(bsum, nb);
    k_scan_add<<<(unsigned)((m + 255) / 256 + 1), 256, 0, s>>>(out, bsum, m, nb);
    return check_cuda(cudaGetLastError(), "scan");
}

// Scratch2 layout for sort + deposit.
struct Work {
    uint32_t *key, *perm, *perm2, *count, *cursor, *off, *bsum, *flag, *pos;
    double* tmp;        // n doubles (permutation buffer)
    double* rec;        // 16 x n deposit shares
    uint32_t* code;     // n stencil offsets
    double* part;       // 20 x C cell partials
};

static int work_layout(fpic_ctx* c, long long n, bool deposit, Work& w, size_t extra_bytes = 0,
                       void** extra = nullptr, int buckets_per_cell = 1)
{
    const long long C = (long long)c->Nr * c->Nth * buckets_per_cell;
    const long long nbs = (n > C + 2 ? n : C + 2) / (SCAN_B * SCAN_PER) + 2;
    size_t bytes = 0;
    auto take = [&](size_t b) { size_t o = bytes; bytes += (b + 255) & ~(size_t)255; return o; };
    size_t o_key = take(4 * n), o_perm = take(4 * n), o_perm2 = take(4 * n), o_count = take(4 * (C + 2)),
           o_cursor = take(4 * (C + 2)), o_off = take(4 * (C + 2)), o_bsum = take(4 * nbs), o_flag = take(4 * n),
           o_pos = take(4 * (n + 1)), o_tmp = take(8 * n);
    size_t o_rec = 0, o_code = 0, o_part = 0;
    if (deposit) {
        o_rec = take(16 * 8 * (size_t)n);
        o_code = take(4 * n);
        o_part = take(20 * 8 * (size_t)C);
    }
    const size_t o_extra = extra_bytes ? take(extra_bytes) : 0;
    int rc = ensure_scratch2(c, bytes);
    if (rc) return rc;
    char* b = (char*)c->d_scratch2;
    if (extra) *extra = extra_bytes ? (void*)(b + o_extra) : nullptr;
    w.key = (uint32_t*)(b + o_key);
    w.perm = (uint32_t*)(b + o_perm);
    w.perm2 = (uint32_t*)(b + o_perm2);
    w.count = (uint32_t*)(b + o_count);
    w.cursor = (uint32_t*)(b + o_cursor);
    w.off = (uint32_t*)(b + o_off);
    w.bsum = (uint32_t*)(b + o_bsum);
    w.flag = (uint32_t*)(b + o_flag);
    w.pos = (uint32_t*)(b + o_pos);
    w.tmp = (double*)(b + o_tmp);
    w.rec = deposit ? (double*)(b + o_rec) : nullptr;
    w.code = deposit ? (uint32_t*)(b + o_code) : nullptr;
    w.part = deposit ? (double*)(b + o_part) : nullptr;
    return 0;
}

// stage: nullable, room for 12 x n doubles (the deposit's record buffer,
// unused until the sort is done): every array is permuted in two passes.
static int sort_impl(fpic_ctx* c, fpic_particles* p, Work& w, cudaStream_t s, double* stage = nullptr)
{
    const long long n = p->n;
    const uint32_t C = (uint32_t)c->Nr * (uint32_t)c->Nth;
    const unsigned nb = (unsigned)((n + 255) / 256);
    FPIC_CUDA(cudaMemsetAsync(w.count, 0, 4 * ((size_t)C + 2), s));
    FPIC_CUDA(cudaMemsetAsync(w.cursor, 0, 4 * ((size_t)C + 2), s));
    k_keys<<<nb, 256, 0, s>>>(c->G, p->r, p->th, p->alive, w.key, p->cell, w.count, n, C);
    int rc = scan_u32(w.count, w.off, w.bsum, (long long)C + 1, s);
    if (rc) return rc;
    k_scatter<<<nb, 256, 0, s>>>(w.key, w.off, w.cursor, w.perm, n);
    k_bucket_rank<1><<<(unsigned)(((long long)C * 32 + 255) / 256), 256, 0, s>>>(w.off, w.perm, w.perm2, C);
    // removed particles: per-block counts in w.pos (nbd + 1 <= n + 1 entries)
    const unsigned nbd = (unsigned)((n + DEAD_PER * DEAD_T - 1) / (DEAD_PER * DEAD_T));
    k_dead_count<<<nbd, DEAD_T, 0, s>>>(p->alive, w.pos, n);
    k_scan_bsum<<<1, SCAN_B, 0, s>>>(w.pos, (int)nbd);
    k_dead_place<<<nbd, DEAD_T, 0, s>>>(p->alive, w.pos, w.off, w.perm2, n, C);
    FPIC_CUDA(cudaGetLastError());
    double* d8[] = {p->r, p->th, p->ph, p->ur, p->uth, p->uph, p->qm, p->w, p->H0, p->D0, p->Hn};
    if (stage) {
        PermArrays a;
        for (int k = 0; k < 11; ++k) a.d[k] = d8[k];
        a.b[0] = p->alive; a.b[1] = p->scheme; a.b[2] = p->iters;
        a.u = p->cell;
        k_gather_all<<<nb, 256, 0, s>>>(a, w.perm2, stage, n);
        k_copy_all<<<nb, 256, 0, s>>>(a, stage, n);
        FPIC_CUDA(cudaGetLastError());
        return 0;
    }
    for (double* a : d8) {
        if (!a) continue;
        k_gather_perm<double><<<nb, 256, 0, s>>>(a, w.tmp, w.perm2, n);
        FPIC_CUDA(cudaMemcpyAsync(a, w.tmp, 8 * (size_t)n, cudaMemcpyDeviceToDevice, s));
    }
    uint8_t* d1[] = {p->alive, p->scheme, p->iters};
    for (uint8_t* a : d1) {
        if (!a) continue;
        k_gather_perm<uint8_t><<<nb, 256, 0, s>>>(a, (uint8_t*)w.tmp, w.perm2, n);
        FPIC_CUDA(cudaMemcpyAsync(a, w.tmp, (size_t)n, cudaMemcpyDeviceToDevice, s));
    }
    if (p->cell) {
        k_gather_perm<uint32_t><<<nb, 256, 0, s>>>(p->cell, (uint32_t*)w.tmp, w.perm2, n);
        FPIC_CUDA(cudaMemcpyAsync(p->cell, w.tmp, 4 * (size_t)n, cudaMemcpyDeviceToDevice, s));
    }
    FPIC_CUDA(cudaGetLastError());
    return 0;
}

// ---------------------------------------------------------------------------
// Deposit (Sec. 2.3)
// ---------------------------------------------------------------------------

// (s, c) of angle x + h from (s, c) of x and (sin h, cos h - 1).
__device__ __forceinline__ void rotate(double s, double c, double sh, double cm, double& so, double& co)
{
    so = fma(s, cm, fma(c, sh, s));
    co = fma(c, cm, fma(-s, sh, c));
}

// sin/cos at the 7 lattice th values of the th cell [y0, y1] split at t:
// y0 + l hc (l = 0..3, y0 + 3 hc = t), t + l hd (l = 1..3, t + 3 hd = y1).
// The end points come in (node tables, the particle's own sin/cos); the
// interior points are angle-addition rotations by hc, 2 hc, hd, 2 hd.
__device__ __forceinline__ void theta_lattice(double hc, double hd, double s0, double c0, double st, double ct,
                                              double s1, double c1, double sy[7], double cy[7])
{
    double sh, cm;
    sy[0] = s0; cy[0] = c0;
    sy[3] = st; cy[3] = ct;
    sy[6] = s1; cy[6] = c1;
    sincos_step(hc, sh, cm);
    rotate(s0, c0, sh, cm, sy[1], cy[1]);
    // double angle: sin 2h = 2 sin h cos h, cos 2h - 1 = 2 (cos h - 1)(cos h + 1)
    rotate(s0, c0, 2.0 * fma(sh, cm, sh), 2.0 * cm * (cm + 2.0), sy[2], cy[2]);
    sincos_step(hd, sh, cm);
    rotate(st, ct, sh, cm, sy[4], cy[4]);
    rotate(st, ct, 2.0 * fma(sh, cm, sh), 2.0 * cm * (cm + 2.0), sy[5], cy[5]);
}

// 4x4 trapezoid lattice of a sub-grid cell [x0, x1] x [y0, y1] split at
// (r, t): the four subvolumes V00 = [x0,r]x[y0,t], V10 = [r,x1]x[y0,t],
// V01 = [x0,r]x[t,y1], V11 = [r,x1]x[t,y1], each by its own 4 x 4 rule; the
// points of the 7 x 7 lattice are evaluated once.  With X = x^2,
// B = X + 2 M x and A = a^2 cos^2 th, sqrt(gamma) = sin th sqrt((X + A)(B + A))
// and the radicand is X B + A (X + B + A): two operations per point.  The
// sin th factor is applied once per lattice row.
// The three sub-grids of a particle share lattice lines: the split column
// x = r of the (i, j) and (i+1/2, j) lattices (same th rows) and the split
// row th = t of the (i, j) and (i, j+1/2) lattices (same r columns), when
// neither split point was clamped.  col / row carry those 7 values: written
// by every call, read instead of evaluated with COL_IN / ROW_IN.
template <bool COL_IN = false, bool ROW_IN = false>
__device__ __forceinline__ void subvolumes(const BH& bh, double x0, double x1, double r, double hc, double hd,
                                           const double sy[7], const double cy[7], double V[4], double col[7],
                                           double row[7])
{
    const double third = 1.0 / 3.0;
    const double ha = (r - x0) * third, hb = (x1 - r) * third;
    double P[7], Q[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        const double x = k < 3 ? fma((double)k, ha, x0) : (k == 3 ? r : fma((double)(k - 3), hb, r));
        const double X = x * x, B = fma(bh.twoM, x, X);
        P[k] = X * B;
        Q[k] = X + B;
    }
    // the lattice values are 2 sqrt(...) (sqrt2_dep): a common factor of the
    // four subvolumes, which only enter as ratios
    double S00 = 0, S10 = 0, S01 = 0, S11 = 0;
#pragma unroll
    for (int l = 0; l < 7; ++l) {
        const double A = bh.a2 * (cy[l] * cy[l]);
        double f[7];
#pragma unroll
        for (int k = 0; k < 7; ++k) {
            if (ROW_IN && l == 3) f[k] = row[k];
            else if (COL_IN && k == 3) f[k] = col[l];
            else f[k] = sqrt2_dep(fma(A, Q[k] + A, P[k]));
        }
        if (!COL_IN) col[l] = f[3];
        if (!ROW_IN && l == 3) {
#pragma unroll
            for (int k = 0; k < 7; ++k) row[k] = f[k];
        }
        // trapezoid weights 1/2, 1, 1, 1/2 along r on each half; the row's
        // th weight (1/2 at the ends and the split row) times sin th
        const double ra = fma(0.5, f[0] + f[3], f[1] + f[2]);
        const double rb = fma(0.5, f[3] + f[6], f[4] + f[5]);
        const double ws = (l == 0 || l == 3 || l == 6) ? 0.5 * sy[l] : sy[l];
        if (l <= 3) { S00 = fma(ws, ra, S00); S10 = fma(ws, rb, S10); }
        if (l >= 3) { S01 = fma(ws, ra, S01); S11 = fma(ws, rb, S11); }
    }
    V[0] = S00 * (ha * hc);
    V[1] = S10 * (hb * hc);
    V[2] = S01 * (ha * hd);
    V[3] = S11 * (hb * hd);
}

// The same lattices in paired-FP32 arithmetic (ff.cuh): the lattice
// coordinates and step sizes, the sin/cos rotations of the th lattice, the
// radicand, its square root, the trapezoid sums and the subvolumes run on
// the FP32 pipe (about 48 bits; the square root to about 2^-44, against
// 2^-39.6 for the FP64 form above), which issues 64 times the FP64 rate.
// The values are sqrt(...) itself (no factor 2).
struct BHff {
    ff twoM, a2, third;
};

__device__ __forceinline__ void rotate_ff(ff s, ff c, ff sh, ff cm, ff& so, ff& co)
{
    so = ff_add(s, ff_add(ff_mul(c, sh), ff_mul(s, cm)));
    co = ff_add(c, ff_add(ff_neg(ff_mul(s, sh)), ff_mul(c, cm)));
}

// sin and cos of th = x + d from those of a node x (table doubles) and an
// offset d under a cell (a double: the difference of two close doubles,
// formed in FP64).
__device__ __forceinline__ void sincos_from_node(double s0, double c0, double d, ff& s, ff& c)
{
    ff sh, cm;
    sincos_step_ff(d, sh, cm);
    rotate_ff(ff_cut(s0), ff_cut(c0), sh, cm, s, c);
}

// The 7 th values of the lattice of [y0, y1] split at t: y0 + l hc
// (l = 0..3), t + l hd (l = 1..3); the end points' sin/cos come in.
__device__ __forceinline__ void theta_lattice_ff(ff hc, ff hd, ff s0, ff c0, ff st, ff ct, ff s1, ff c1, ff sy[7],
                                                 ff cy[7])
{
    sy[0] = s0; cy[0] = c0;
    sy[3] = st; cy[3] = ct;
    sy[6] = s1; cy[6] = c1;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
        const int b = 3 * half;
        ff sh, cm;
        sincos_step_ff(half ? hd : hc, sh, cm);
        rotate_ff(sy[b], cy[b], sh, cm, sy[b + 1], cy[b + 1]);
        // double angle: sin 2h = 2 sin h (1 + (cos h - 1)), cos 2h - 1 = 2 (cos h - 1)(cos h - 1 + 2)
        const ff sh2 = ff_scale(ff_add(sh, ff_mul(sh, cm)), 2.f);
        const ff cm2 = ff_scale(ff_mul(cm, ff_add(cm, ff_of(2.f))), 2.f);
        rotate_ff(sy[b], cy[b], sh2, cm2, sy[b + 2], cy[b + 2]);
    }
}

// One sub-grid lattice in paired FP32, row by row (the row loop is not
// unrolled: one copy of the code serves every row and, through
// k_dep_particle_ff's loop, every sub-grid): r columns x0 + k ha (k = 0..3,
// x0 + 3 ha = r), r + k hb (k = 1..3).  col_in / row_in: take the split
// column / row from col / row instead of evaluating them; put_shared: store
// this lattice's split column and row there.  V: the four subvolumes.
__device__ __forceinline__ void subvolumes_ff(const BHff& bh, ff x0f, ff rf, ff ha, ff hb, ff hc, ff hd,
                                              const ff* sy, const ff* cy, ff V[4], ff* col, ff row[7],
                                              bool col_in, bool row_in, bool put_shared)
{
    ff P[7], Q[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        ff x;
        if (k == 0) x = x0f;
        else if (k < 3) x = ff_add(x0f, k == 1 ? ha : ff_scale(ha, 2.f));
        else if (k == 3) x = rf;
        else x = ff_add(rf, k == 4 ? hb : (k == 5 ? ff_scale(hb, 2.f) : ff_mulf(hb, 3.f)));
        const ff X = ff_sqr(x), B = ff_add(X, ff_mul(bh.twoM, x));
        P[k] = ff_mul(X, B);
        Q[k] = ff_add_ge(B, X);                        // B = X + 2 M x >= X
    }
    ff S00 = ff_of(0.f), S10 = ff_of(0.f), S01 = ff_of(0.f), S11 = ff_of(0.f);
#pragma unroll 1
    for (int l = 0; l < 7; ++l) {
        ff f[7];
        if (row_in && l == 3) {
#pragma unroll
            for (int k = 0; k < 7; ++k) f[k] = row[k];
        } else {
            const ff A = ff_mul(bh.a2, ff_sqr(cy[l]));
#pragma unroll
            for (int k = 0; k < 7; ++k)
                if (k != 3 || !col_in) f[k] = ff_sqrt(ff_add(P[k], ff_mul(A, ff_add(Q[k], A))));
            if (col_in) f[3] = col[l];
        }
        if (put_shared) {
            col[l] = f[3];
            if (l == 3) {
#pragma unroll
                for (int k = 0; k < 7; ++k) row[k] = f[k];
            }
        }
        // trapezoid weights 1/2, 1, 1, 1/2 along r on each half; the row's
        // th weight (1/2 at the ends and the split row) times sin th.  Along
        // a row sqrt(gamma) grows with r (both factors of the radicand do),
        // so f[k] <= f[k'] for k < k': the pair sums take the fast two-sum
        const ff ra = ff_add(ff_scale(ff_add_ge(f[3], f[0]), 0.5f), ff_add_ge(f[2], f[1]));
        const ff rb = ff_add(ff_scale(ff_add_ge(f[6], f[3]), 0.5f), ff_add_ge(f[5], f[4]));
        const ff ws = ff_scale(sy[l], (l == 0 || l == 3 || l == 6) ? 0.5f : 1.f);
        if (l <= 3) { S00 = ff_add(S00, ff_mul(ws, ra)); S10 = ff_add(S10, ff_mul(ws, rb)); }
        if (l >= 3) { S01 = ff_add(S01, ff_mul(ws, ra)); S11 = ff_add(S11, ff_mul(ws, rb)); }
    }
    V[0] = ff_mul(S00, ff_mul(ha, hc));
    V[1] = ff_mul(S10, ff_mul(hb, hc));
    V[2] = ff_mul(S01, ff_mul(ha, hd));
    V[3] = ff_mul(S11, ff_mul(hb, hd));
}

struct DepK {
    BH bh;
    BHff bhf;        // 2M and a^2 as paired floats
    GridDev G;
    const double* trig;  // sin tn[0..Nth], cos tn[0..Nth], sin th[0..Nth-1], cos th[0..Nth-1]
    const double *r, *th, *ur, *uth, *uph, *qm, *w;
    long long n_alive;
    double* rec;     // 16 x n
    uint32_t* code;  // (i1 - i0 + 1) | (j1 - j0 + 1) << 2
};

__device__ __forceinline__ double clampd(double x, double lo, double hi)
{
    return x < lo ? lo : (x > hi ? hi : x);
}

__global__ void __launch_bounds__(256) k_dep_particle(DepK k)
{
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (p >= k.n_alive) return;
    const GridDev& G = k.G;
    const double r = k.r[p], t = k.th[p];
    // FIDO three-velocity v^i = gamma^ij u_j / Gamma at the particle
    double s, c;
    sincos(t, &s, &c);
    Geo g;
    geo_eval(k.bh, r, s, c, g);
    const double ur = k.ur[p], ut = k.uth[p], up = k.uph[p];
    const double Ur = fma(g.gurr, ur, g.gurp * up), Ut = g.gutt * ut, Up = fma(g.gurp, ur, g.gupp * up);
    const double iG = rsqrt_nr(fma(ur, Ur, fma(ut, Ut, fma(up, Up, 1.0))));
    const double Q = k.w[p] * k.qm[p];
    const double vr = Ur * iG, vt = Ut * iG, vp = Up * iG;
    // clamped positions and cells on the integer and half node lists
    const double rn_c = clampd(r, G.rn[0], G.rn[G.Nr]), rh_c = clampd(r, G.rh[0], G.rh[G.Nr - 1]);
    const double tn_c = clampd(t, G.tn[0], G.tn[G.Nth]), th_c = clampd(t, G.th[0], G.th[G.Nth - 1]);
    int i0, i1, j0, j1;
    double wd;
    const float lr = __logf((float)r);
    locate(G.rn, G.irn, G.Nr + 1, rn_c, (lr - G.lr0) * G.ilr, i0, wd);
    locate(G.rh, G.irh, G.Nr, rh_c, (lr - G.lrh0) * G.ilr, i1, wd);
    locate(G.tn, G.itn, G.Nth + 1, tn_c, ((float)t - G.t0) * G.it, j0, wd);
    locate(G.th, G.ith, G.Nth, th_c, ((float)t - G.th0) * G.it, j1, wd);
    // sin/cos at the clamped th (the particle's own unless clamped at an edge)
    double stn = s, ctn = c, sth = s, cth = c;
    if (tn_c != t) sincos(tn_c, &stn, &ctn);
    if (th_c != t) sincos(th_c, &sth, &cth);
    const double* sn = k.trig;
    const double* cn = k.trig + (G.Nth + 1);
    const double* sh = k.trig + 2 * (G.Nth + 1);
    const double* ch = sh + G.Nth;
    const double third = 1.0 / 3.0;
    double sy[7], cy[7], V[4], col[7], row[7];
    const long long n = k.n_alive;
    // the split column / row are shared between the sub-grids unless clamped
    const bool share = (rn_c == rh_c) && (tn_c == th_c);
    // (i, j): rho and j^ph
    const double y0 = G.tn[j0], y1 = G.tn[j0 + 1];
    double hc = (tn_c - y0) * third, hd = (y1 - tn_c) * third;
    theta_lattice(hc, hd, sn[j0], cn[j0], stn, ctn, sn[j0 + 1], cn[j0 + 1], sy, cy);
    subvolumes(k.bh, G.rn[i0], G.rn[i0 + 1], rn_c, hc, hd, sy, cy, V, col, row);
    double iV = rcp_nr(V[0] + V[1] + V[2] + V[3]);
    // share of node (i+a, j+b) = V(opposite corner) / V
    const double w00 = V[3] * iV, w10 = V[2] * iV, w01 = V[1] * iV, w11 = V[0] * iV;
    k.rec[0 * n + p] = Q * w00; k.rec[1 * n + p] = Q * w10; k.rec[2 * n + p] = Q * w01; k.rec[3 * n + p] = Q * w11;
    const double Qp = Q * vp;
    k.rec[4 * n + p] = Qp * w00; k.rec[5 * n + p] = Qp * w10; k.rec[6 * n + p] = Qp * w01; k.rec[7 * n + p] = Qp * w11;
    // (i+1/2, j): j^r  (same th lattice)
    {
        double row_rh[7];   // this lattice's split row (r columns of the half grid): not shared
        if (share) subvolumes<true, false>(k.bh, G.rh[i1], G.rh[i1 + 1], rh_c, hc, hd, sy, cy, V, col, row_rh);
        else subvolumes(k.bh, G.rh[i1], G.rh[i1 + 1], rh_c, hc, hd, sy, cy, V, col, row_rh);
    }
    iV = rcp_nr(V[0] + V[1] + V[2] + V[3]);
    const double Qr = Q * vr;
    k.rec[8 * n + p] = Qr * (V[3] * iV); k.rec[9 * n + p] = Qr * (V[2] * iV);
    k.rec[10 * n + p] = Qr * (V[1] * iV); k.rec[11 * n + p] = Qr * (V[0] * iV);
    // (i, j+1/2): j^th
    const double z0 = G.th[j1], z1 = G.th[j1 + 1];
    hc = (th_c - z0) * third;
    hd = (z1 - th_c) * third;
    theta_lattice(hc, hd, sh[j1], ch[j1], sth, cth, sh[j1 + 1], ch[j1 + 1], sy, cy);
    if (share) subvolumes<false, true>(k.bh, G.rn[i0], G.rn[i0 + 1], rn_c, hc, hd, sy, cy, V, col, row);
    else subvolumes(k.bh, G.rn[i0], G.rn[i0 + 1], rn_c, hc, hd, sy, cy, V, col, row);
    iV = rcp_nr(V[0] + V[1] + V[2] + V[3]);
    const double Qt = Q * vt;
    k.rec[12 * n + p] = Qt * (V[3] * iV); k.rec[13 * n + p] = Qt * (V[2] * iV);
    k.rec[14 * n + p] = Qt * (V[1] * iV); k.rec[15 * n + p] = Qt * (V[0] * iV);
    k.code[p] = (uint32_t)(i1 - i0 + 1) | ((uint32_t)(j1 - j0 + 1) << 2);
}

// x clamped to [lo, hi] by integer compares of the order-preserving keys:
// the value the FP64 compares give for non-NaN x (a -0 below lo = +0 comes
// back as +0), without FP64-pipe instructions.
__device__ __forceinline__ double clamp_key(double x, double lo, double hi)
{
    const long long kx = okey(x);
    return kx < okey(lo) ? lo : (kx > okey(hi) ? hi : x);
}

__device__ __forceinline__ bool same_bits(double a, double b)
{
    return __double_as_longlong(a) == __double_as_longlong(b);
}

// The charge times the FIDO three-velocity gamma^ij u_j / Gamma, the terms
// shared as in eval_rhs_sc_t (24 FP64 instructions besides the reciprocal's and
// the two roots' six; through the metric's components 5 more, k_dep_particle_poly
// 552 -> 532 us at 4.0e6 particles with the sin/cos series in paired FP32).  FP64:
// the 1/sin^2 th of g^phph and the cancellation between the two terms of U^r and
// U^ph want more than paired FP32's 46 bits.
__device__ __forceinline__ void charge_flux(const BH& bh, double r, double s, double c, double ur, double ut, double up,
                                            double Q, double& Qr, double& Qt, double& Qp)
{
    const double s2 = s * s, rho2 = fma(bh.a2, c * c, r * r);
    const double gpp = rcp_nr(rho2 * s2), irho2 = gpp * s2;
    const double alpha = rsqrt_nr(fma(bh.twoM * irho2, r, 1.0));
    const double gurp = bh.a * irho2, g1 = fma(bh.a * s2, ur, up), iu = (alpha * alpha) * ur, tu = gpp * up;
    const double W = fma(bh.a * ur, g1 + up, ut * ut);
    const double QiG = Q * rsqrt_nr(fma(iu, ur, 1.0 + fma(W, irho2, tu * up)));
    Qr = QiG * fma(gurp, g1, iu);
    Qt = QiG * (irho2 * ut);
    Qp = QiG * fma(gurp, ur, tu);
}

// The deposit's per-particle pass: the sin/cos of the lattices' split
// points (angle addition from the node tables by the in-cell offset), the
// three sub-grid lattices, their subvolumes, weights and the charge products
// in paired FP32; FP64 keeps the particle's sin/cos th and FIDO velocity,
// the node-coordinate differences (the step sizes) and the final sum of
// each share's two floats.
__global__ void __launch_bounds__(256) k_dep_particle_ff(DepK k)
{
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (p >= k.n_alive) return;
    const GridDev& G = k.G;
    const BHff& bh = k.bhf;
    const double r = k.r[p], t = k.th[p];
    // clamped positions and cells on the integer and half node lists
    const double rn_c = clamp_key(r, G.rn[0], G.rn[G.Nr]), rh_c = clamp_key(r, G.rh[0], G.rh[G.Nr - 1]);
    const double tn_c = clamp_key(t, G.tn[0], G.tn[G.Nth]), th_c = clamp_key(t, G.th[0], G.th[G.Nth - 1]);
    int i0, i1, j0, j1;
    double wd;
    const float lr = __logf(f32_est(r)), tf = f32_est(t);
    locate(G.rn, G.irn, G.Nr + 1, rn_c, (lr - G.lr0) * G.ilr, i0, wd);
    locate(G.rh, G.irh, G.Nr, rh_c, (lr - G.lrh0) * G.ilr, i1, wd);
    locate(G.tn, G.itn, G.Nth + 1, tn_c, (tf - G.t0) * G.it, j0, wd);
    locate(G.th, G.ith, G.Nth, th_c, (tf - G.th0) * G.it, j1, wd);
    const double* sn = k.trig;
    const double* cn = k.trig + (G.Nth + 1);
    const double* sh = k.trig + 2 * (G.Nth + 1);
    const double* ch = sh + G.Nth;
    // sin/cos th of the particle in FP64 by angle addition from a node of
    // its cell: the lower node where cos >= 0, the upper one elsewhere, so
    // that sin(x + d) = sin x + (sin x (cos d - 1) + cos x sin d) adds terms
    // of one sign and sin th keeps its relative accuracy up to the poles
    // (g^pp = 1 / (rho^2 sin^2 th) in the velocity needs it); the offset's
    // sin / cos - 1 by the series (libm beyond a cell: a clamped th).
    const int jn = j0 + (__double2hiint(cn[j0]) < 0 ? 1 : 0);
    double s, c;
    sincos_near(G.tn[jn], sn[jn], cn[jn], t, s, c);
    // ... and at the split points of the two th lattices in paired FP32 (the
    // integer lattice's is the particle's own th unless clamped)
    ff stn, ctn, sth, cth;
    if (same_bits(tn_c, t)) {
        stn = ff_cut(s);
        ctn = ff_cut(c);
    } else {
        sincos_from_node(sn[jn], cn[jn], tn_c - G.tn[jn], stn, ctn);
    }
    sincos_from_node(sh[j1], ch[j1], th_c - G.th[j1], sth, cth);
    const double Qd = k.w[p] * k.qm[p];
    double Fr, Ft, Fp;
    charge_flux(k.bh, r, s, c, k.ur[p], k.uth[p], k.uph[p], Qd, Fr, Ft, Fp);
    const ff Q = ff_cut(Qd), Qr = ff_cut(Fr), Qt = ff_cut(Ft), Qp = ff_cut(Fp);
    const long long n = k.n_alive;
    // the split column / row are shared between the sub-grids unless clamped
    const bool share = same_bits(rn_c, rh_c) && same_bits(tn_c, th_c);
    ff sy[7], cy[7], col[7], row[7];
    ff hc = ff_of(0.f), hd = ff_of(0.f);
    // sub-grid 0: (i, j), rho and j^ph; 1: (i+1/2, j), j^r (the th lattice of
    // 0); 2: (i, j+1/2), j^th.  One copy of the lattice code serves all three.
#pragma unroll 1
    for (int sg = 0; sg < 3; ++sg) {
        if (sg != 1) {
            const bool hth = sg == 2;
            const int jj = hth ? j1 : j0;
            const double* Y = hth ? G.th : G.tn;
            const double* sY = hth ? sh : sn;
            const double* cY = hth ? ch : cn;
            const double tc = hth ? th_c : tn_c;
            hc = ff_mul(ff_cut(tc - Y[jj]), bh.third);
            hd = ff_mul(ff_cut(Y[jj + 1] - tc), bh.third);
            theta_lattice_ff(hc, hd, ff_cut(sY[jj]), ff_cut(cY[jj]), hth ? sth : stn, hth ? cth : ctn,
                             ff_cut(sY[jj + 1]), ff_cut(cY[jj + 1]), sy, cy);
        }
        const bool hr = sg == 1;
        const double x0 = hr ? G.rh[i1] : G.rn[i0], x1 = hr ? G.rh[i1 + 1] : G.rn[i0 + 1];
        const double rc = hr ? rh_c : rn_c;
        const ff ha = ff_mul(ff_cut(rc - x0), bh.third), hb = ff_mul(ff_cut(x1 - rc), bh.third);
        ff V[4];
        subvolumes_ff(bh, ff_cut(x0), ff_cut(rc), ha, hb, hc, hd, sy, cy, V, col, row, share && sg == 1,
                      share && sg == 2, sg == 0);
        const ff iV = ff_rcp(ff_add(ff_add(V[0], V[1]), ff_add(V[2], V[3])));
        // share of node (i+a, j+b) = V(opposite corner) / V
        const ff w00 = ff_mul(V[3], iV), w10 = ff_mul(V[2], iV), w01 = ff_mul(V[1], iV), w11 = ff_mul(V[0], iV);
        const int b = sg == 0 ? 0 : 4 + 4 * sg;
        const ff Qs = sg == 0 ? Q : (sg == 1 ? Qr : Qt);
        k.rec[(b + 0) * n + p] = ff_to(ff_mul(Qs, w00)); k.rec[(b + 1) * n + p] = ff_to(ff_mul(Qs, w10));
        k.rec[(b + 2) * n + p] = ff_to(ff_mul(Qs, w01)); k.rec[(b + 3) * n + p] = ff_to(ff_mul(Qs, w11));
        if (sg == 0) {
            k.rec[4 * n + p] = ff_to(ff_mul(Qp, w00)); k.rec[5 * n + p] = ff_to(ff_mul(Qp, w10));
            k.rec[6 * n + p] = ff_to(ff_mul(Qp, w01)); k.rec[7 * n + p] = ff_to(ff_mul(Qp, w11));
        }
    }
    k.code[p] = (uint32_t)(i1 - i0 + 1) | ((uint32_t)(j1 - j0 + 1) << 2);
}

// Builds the cells' polynomials (sub-grid blockIdx.z; a thread walks `rows`
// cells down one th column, whose trigonometry it takes once), the 1-D
// tables and the largest bound over the cells (poly_worst, as the bits of a
// non-negative float).  Once per grid, about 60 FP64 operations a cell.
struct PolyBuild {
    BH bh;
    GridDev G;
    float4* c[3];
    float2* ir[2];
    float4* t[2];
    unsigned* bound;
    int rows;
};

__device__ __forceinline__ float2 pair_of(double d)
{
    const float h = (float)d;
    return make_float2(h, (float)(d - (double)h));
}

template <int DEG>
__global__ void __launch_bounds__(128) k_poly_build(const __grid_constant__ PolyBuild k)
{
    const int sg = blockIdx.z, j = blockIdx.x * 128 + threadIdx.x;
    const GridDev& G = k.G;
    const bool hr = sg == 1, hth = sg == 2;
    const int i0 = blockIdx.y * k.rows, i1 = min(i0 + k.rows, G.Nr - hr);
    float e = 0.f;
    if (j < G.Nth - hth) {
        const double* X = hr ? G.rh : G.rn;
        const double* Y = hth ? G.th : G.tn;
        const double dy = Y[j + 1] - Y[j], y = 0.5 * (Y[j] + Y[j + 1]);
        double s, co;
        sincos(y, &s, &co);
        PolyTheta<DEG> th;
        poly_theta<DEG>(k.bh.a, s, co, dy, th);
        for (int i = i0; i < i1; ++i) {
            const double dx = X[i + 1] - X[i];
            double f[4][4];
            float q[DEG + 2][DEG + 2];
            poly_series<DEG>(k.bh.M, 0.5 * (X[i] + X[i + 1]), dx, th, f, q);
            e = poly_worst(e, poly_bound<DEG>(q));
            float4* c = k.c[sg] + ((size_t)i * G.Nth + j) * (poly_stride(DEG) / 4);
            const float2 f10 = pair_of(f[1][0]), f01 = pair_of(f[0][1]), f20 = pair_of(f[2][0]),
                         f11 = pair_of(f[1][1]), f02 = pair_of(f[0][2]);
            c[0] = make_float4(f10.x, f10.y, f01.x, f01.y);
            c[1] = make_float4(f20.x, f20.y, f11.x, f11.y);
            c[2] = make_float4(f02.x, f02.y, q[3][0], q[2][1]);
            c[3] = make_float4(q[1][2], q[0][3], q[4][0], q[3][1]);
            c[4] = make_float4(q[2][2], q[1][3], q[0][4], q[5][0]);
            c[5] = make_float4(q[4][1], q[3][2], q[2][3], q[1][4]);
            if constexpr (DEG > 5) {
                c[6] = make_float4(q[0][5], q[6][0], q[5][1], q[4][2]);
                c[7] = make_float4(q[3][3], q[2][4], q[1][5], q[0][6]);
            } else {
                c[6] = make_float4(q[0][5], 0.f, 0.f, 0.f);
            }
            if (j == 0 && sg < 2) k.ir[sg][i] = pair_of(1.0 / dx);
        }
        if (i0 == 0 && sg != 1) {
            const double tau = dy * co / s;
            const float2 it = pair_of(1.0 / dy), tp = pair_of(tau), d2 = pair_of(0.5 * dy * dy), d6 = pair_of(dy * dy / 6.0);
            float4* t = k.t[hth] + 2 * j;
            t[0] = make_float4(it.x, it.y, tp.x, tp.y);
            t[1] = make_float4(d2.x, d2.y, d6.x, d6.y);
            if (!(s > 0.0 && dy <= POLY_MAX_DTH && fabs(tau) <= POLY_MAX_TAU)) e = INFINITY;
        }
    }
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(e));
    if ((threadIdx.x & 31) == 0) atomicMax(k.bound, m);
}

// A few cells of the first row, where the bound is largest on a log grid: false
// where the grid is not worth a look.
template <int DEG>
static bool poly_may(const fpic_ctx* c, const double* X, const double* Y)
{
    for (int q = 0; q < 16; ++q) {
        const int j = (int)((long long)q * (c->Nth - 1) / 15);
        const double y = 0.5 * (Y[j] + Y[j + 1]);
        PolyTheta<DEG> th;
        double f[4][4];
        float g[DEG + 2][DEG + 2];
        poly_theta<DEG>(c->a, sin(y), cos(y), Y[j + 1] - Y[j], th);
        poly_series<DEG>(c->M, 0.5 * (X[0] + X[1]), X[1] - X[0], th, f, g);
        if (!(poly_bound<DEG>(g) <= poly_tol(DEG))) return false;
    }
    return true;
}

// The polynomials of the context's grid (built on first use, with a wait for
// the bound); T filled and deg their degree where they may be used, else 0.  Not
// built while the stream is being captured, nor beyond POLY_MAX_BYTES, nor (until
// the next fpic_set_grid) after an allocation that failed: the lattices serve.
constexpr size_t POLY_MAX_BYTES = (size_t)16 << 30;

static int poly_tables(fpic_ctx* c, PolyTab& T, int& deg, cudaStream_t s)
{
    deg = 0;
    const size_t cells = (size_t)c->Nr * c->Nth, row = ((size_t)c->Nr + 31) & ~(size_t)31;
    const bool fresh = c->poly_grid != c->grid_gen;
    int want = c->poly_deg;
    if (fresh) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        FPIC_CUDA(cudaStreamIsCapturing(s, &cap));
        if (cap != cudaStreamCaptureStatusNone) return 0;
        c->poly_deg = 0;
        c->poly_grid = c->grid_gen;
        retire(c, &c->d_poly);
        // spacings far beyond what the bound admits: not worth a look
        const double* X = (const double*)c->h_nodes.data();
        const double* Y = X + (size_t)c->Nr + 1 + c->Nr;
        double dr = 0.0, dt = 0.0;
        for (int i = 0; i < c->Nr; ++i) dr = fmax(dr, (X[i + 1] - X[i]) / X[i]);
        for (int j = 0; j < c->Nth; ++j) dt = fmax(dt, Y[j + 1] - Y[j]);
        const size_t bytes = 3 * cells * poly_stride(6) * 4 + 2 * row * 8 + 4 * (size_t)c->Nth * 16 + 256;
        if (bytes > POLY_MAX_BYTES || dr > 0.05 || dt > POLY_MAX_DTH) return 0;
        want = poly_may<5>(c, X, Y) ? 5 : poly_may<6>(c, X, Y) ? 6 : 0;
        if (!want) return 0;
        if (cudaMalloc(&c->d_poly, bytes) != cudaSuccess) {
            cudaGetLastError();
            c->d_poly = nullptr;
            return 0;
        }
    }
    if (!c->d_poly) return 0;
    PolyBuild k{c->bh, c->G, {}, {}, {}, nullptr, 8};
    for (;; want = 6) {
        char* b = (char*)c->d_poly;
        const size_t per = cells * poly_stride(want) * 4;
        for (int q = 0; q < 3; ++q) k.c[q] = (float4*)(b + q * per);
        b += 3 * per;
        for (int q = 0; q < 2; ++q) k.t[q] = (float4*)b + q * 2 * (size_t)c->Nth;
        b += 4 * (size_t)c->Nth * 16;
        for (int q = 0; q < 2; ++q) k.ir[q] = (float2*)b + q * row;
        k.bound = (unsigned*)(b + 2 * row * 8);
        if (!fresh) break;
        const long long cols = (c->Nth + 127) / 128;
        while (k.rows > 1 && 3 * cols * (c->Nr / k.rows) < 8LL * c->sm_count) k.rows >>= 1;
        const dim3 grid((unsigned)cols, (unsigned)((c->Nr + k.rows - 1) / k.rows), 3);
        FPIC_CUDA(cudaMemsetAsync(k.bound, 0, 4, s));
        if (want == 5) k_poly_build<5><<<grid, 128, 0, s>>>(k);
        else k_poly_build<6><<<grid, 128, 0, s>>>(k);
        float e = 0.f;
        FPIC_CUDA(cudaMemcpyAsync(&e, k.bound, 4, cudaMemcpyDeviceToHost, s));
        FPIC_CUDA(cudaStreamSynchronize(s));
        if (e <= poly_tol(want)) {
            c->poly_deg = want;
            break;
        }
        if (want == 6) {
            FPIC_CUDA(cudaFree(c->d_poly));
            c->d_poly = nullptr;
            break;
        }
    }
    if (!c->poly_deg) return 0;
    const double* X = (const double*)c->h_nodes.data();      // rn, rh, tn, th (th with one node more)
    const size_t m[4] = {(size_t)c->Nr + 1, (size_t)c->Nr, (size_t)c->Nth + 1, (size_t)c->Nth};
    for (int q = 0; q < 4; ++q) {
        T.lo[q] = X[0];
        T.hi[q] = X[m[q] - 1];
        X += m[q];
    }
    for (int q = 0; q < 3; ++q) T.c[q] = k.c[q];
    for (int q = 0; q < 2; ++q) {
        T.ir[q] = k.ir[q];
        T.t[q] = k.t[q];
    }
    deg = c->poly_deg;
    return 0;
}

// The cell of x (held to [lo, hi]) on the m nodes X, est an FP32 estimate of
// it, and the fractions of the cell below (al) and above (ab) x in paired
// FP32, each from its own FP64 difference so that a small share keeps its
// relative accuracy.
__device__ __forceinline__ int cell_split(const double* __restrict__ X, int m, double lo, double hi, double x,
                                          float est, double& d0, double& d1)
{
    const long long klo = okey(lo), khi = okey(hi);
    long long kx = okey(x);
    x = kx < klo ? lo : (kx > khi ? hi : x);
    kx = okey(x);
    int i = max(0, min(__float2int_rd(est), m - 2));
    double X0 = __ldg(X + i), X1 = __ldg(X + i + 1);
    while (i > 0 && kx < okey(X0)) {
        X1 = X0;
        X0 = __ldg(X + --i);
    }
    while (i < m - 2 && kx >= okey(X1)) {
        X0 = X1;
        X1 = __ldg(X + ++i + 1);
    }
    d0 = x - X0;
    d1 = X1 - x;
    return i;
}

// The per-particle pass on grids with polynomials: the same trapezoid rules'
// node shares as k_dep_particle_ff without evaluating their 133 lattice
// points.  FP64 keeps the particle's sin/cos th and FIDO velocity and the
// positions' offsets in their cells.  The shares are stored as pairs of
// floats: turning them into doubles is integer work that k_dep_cell, bound
// by its FP64 additions, has the issue slots for.  FP64-pipe
// bound (61 % busy, some 57 instructions a particle) at 92 instead of 370
// instructions per charge share: 1511 -> 532 us at 4.0e6 particles on
// 512 x 512, 23.7 -> 9 ms at 6.4e7 on 1024 x 1024 (64 or 80 registers alike).
template <int DEG>
__global__ void __launch_bounds__(256, 4) k_dep_particle_poly(const __grid_constant__ DepK k,
                                                              const __grid_constant__ PolyTab T)
{
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (p >= k.n_alive) return;
    const GridDev& G = k.G;
    const double r = k.r[p], t = k.th[p];
    const float lr = __logf(f32_est(r)), tf = f32_est(t);
    double d0, d1;
    const int j0 = cell_split(G.tn, G.Nth + 1, T.lo[2], T.hi[2], t, (tf - G.t0) * G.it, d0, d1);
    Mom X[2], Y[2];
    MomT E[2];
    {
        const float4 t0 = __ldg(T.t[0] + 2 * j0), t1 = __ldg(T.t[0] + 2 * j0 + 1);
        const ff inv = {t0.x, t0.y};
        moments(ff_mul(ff_from(d0), inv), ff_mul(ff_from(d1), inv), Y);
        moments_th<DEG>(Y, {t0.z, t0.w}, {t1.x, t1.y}, {t1.z, t1.w}, E);
    }
    // FIDO three-velocity, as k_dep_particle_ff (sin/cos th by angle addition
    // from the node on the side where the terms share a sign)
    ff Q, Qr, Qt, Qp;
    {
        const double* sn = k.trig;
        const double* cn = k.trig + (G.Nth + 1);
        const int jn = j0 + (__double2hiint(cn[j0]) < 0 ? 1 : 0);
        double s, c;
        sincos_near(G.tn[jn], sn[jn], cn[jn], t, s, c);
        const double Qd = k.w[p] * k.qm[p];
        double Fr, Ft, Fp;
        charge_flux(k.bh, r, s, c, k.ur[p], k.uth[p], k.uph[p], Qd, Fr, Ft, Fp);
        Q = ff_from(Qd);
        Qr = ff_from(Fr);
        Qt = ff_from(Ft);
        Qp = ff_from(Fp);
    }
    const long long n = k.n_alive;
    float2* rec = (float2*)k.rec + p;
    auto put = [&](int row, ff q, const ff w[4]) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const ff v = ff_mul(q, w[b]);
            rec[(row + b) * n] = make_float2(v.hi, v.lo);
        }
    };
    ff w[4];
    const int i1 = cell_split(G.rh, G.Nr, T.lo[1], T.hi[1], r, (lr - G.lrh0) * G.ilr, d0, d1);
    {   // (i+1/2, j): j^r
        const float2 ir = __ldg(T.ir[1] + i1);
        moments(ff_mul(ff_from(d0), {ir.x, ir.y}), ff_mul(ff_from(d1), {ir.x, ir.y}), X);
        poly_shares<DEG>(T.c[1] + ((size_t)i1 * G.Nth + j0) * (poly_stride(DEG) / 4), X, E, w);
        put(8, Qr, w);
    }
    const int i0 = cell_split(G.rn, G.Nr + 1, T.lo[0], T.hi[0], r, (lr - G.lr0) * G.ilr, d0, d1);
    {   // (i, j): rho and j^ph
        const float2 ir = __ldg(T.ir[0] + i0);
        moments(ff_mul(ff_from(d0), {ir.x, ir.y}), ff_mul(ff_from(d1), {ir.x, ir.y}), X);
        poly_shares<DEG>(T.c[0] + ((size_t)i0 * G.Nth + j0) * (poly_stride(DEG) / 4), X, E, w);
        put(0, Q, w);
        put(4, Qp, w);
    }
    const int j1 = cell_split(G.th, G.Nth, T.lo[3], T.hi[3], t, (tf - G.th0) * G.it, d0, d1);
    {   // (i, j+1/2): j^th
        const float4 t0 = __ldg(T.t[1] + 2 * j1), t1 = __ldg(T.t[1] + 2 * j1 + 1);
        const ff inv = {t0.x, t0.y};
        moments(ff_mul(ff_from(d0), inv), ff_mul(ff_from(d1), inv), Y);
        moments_th<DEG>(Y, {t0.z, t0.w}, {t1.x, t1.y}, {t1.z, t1.w}, E);
        poly_shares<DEG>(T.c[2] + ((size_t)i0 * G.Nth + j1) * (poly_stride(DEG) / 4), X, E, w);
        put(12, Qt, w);
    }
    k.code[p] = (uint32_t)(i1 - i0 + 1) | ((uint32_t)(j1 - j0 + 1) << 2);
}

// Slots of a cell (i0, j0): rho[a + 2b] (0..3), j^ph[a + 2b] (4..7),
// j^r[k + 3b] at half-r node i0 - 1 + k (8..13), j^th[a + 2k] at half-th
// node j0 - 1 + k (14..19).  A particle with offsets (ko, kt) (each 0 or 1)
// puts record rows 0..7 in slots 0..7, rows 8 + 2b and 9 + 2b in slots
// 8 + 3b + ko and 9 + 3b + ko, rows 12 + a and 14 + a in slots 14 + a + 2 kt
// and 16 + a + 2 kt.
//
// One warp per cell, its particles 32 at a time: every lane loads one
// particle's 16 shares and code (coalesced, no load depending on another)
// into shared memory; then lane l sums record row l / 2 over the group's
// particles of parity l & 1, into one of two accumulators chosen by the
// particle's offset bit (ko for the j^r rows, kt for the j^th rows, none
// for rows 0..7): 16 FP64 additions per particle, each lane busy.  The
// accumulator is chosen by integer selects, so each addition is one FP64
// instruction.  At the end the two parities are added and lane q < 20
// assembles slot q from at most two (row, accumulator) pairs.  Every
// addition has a fixed order: bitwise reproducible.
constexpr int DEP_CELL_WARPS = 8, DEP_CELL_LD = 33;   // row stride 33: conflict-free shared-memory columns

__device__ __forceinline__ double sel_bits(bool p, double a, double b)
{
    double r;
    asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\tselp.b64 %0, %1, %2, q;\n\t}"
        : "=d"(r) : "d"(a), "d"(b), "r"((unsigned)p));
    return r;
}

// PAIRS: the shares are pairs of floats (k_dep_particle_poly).  The high
// floats are summed in FP64, the low ones (2^-24 of them) in FP32: 2^-48 of the
// sum of |share|, under the shares' own rounding, at one FP64 addition to four
// shares, after a tree of exact FP32 two-sums whose errors join the low floats
// (one addition a share: deposit of 4.0e6 particles on 512^2 1136 -> 1108 us).  The
// low sums join the FP64 ones after every 128 particles: in a crowded cell they
// would lose what is small beside them (16384 equal shares 3e-12 off).  The 16
// conversions a particle are not in the FP64-bound kernel before it.
template <bool PAIRS>
__global__ void __launch_bounds__(32 * DEP_CELL_WARPS) k_dep_cell(const double* __restrict__ rec,
                                                                   const uint32_t* __restrict__ code,
                                                                   const uint32_t* __restrict__ off,
                                                                   double* __restrict__ part, long long n, uint32_t C)
{
    __shared__ double sv[DEP_CELL_WARPS][16 * DEP_CELL_LD];
    __shared__ uint32_t sc[DEP_CELL_WARPS][32];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long cell = blockIdx.x * (long long)DEP_CELL_WARPS + wid;
    if (cell >= C) return;                  // whole warps: one cell per warp
    double* v = sv[wid];
    uint32_t* cw = sc[wid];
    const uint32_t b0 = off[cell], b1 = off[cell + 1];
    if (b0 == b1) {                         // an empty cell
        if (lane < 20) part[(size_t)lane * C + cell] = 0.0;
        return;
    }
    const int row = lane >> 1, par = lane & 1;
    const int bsh = row >= 12 ? 2 : 0;      // the offset bit this row splits on
    const uint32_t bmask = row >= 8 ? 1u : 0u;
    double acc0 = 0.0, acc1 = 0.0;
    float lo0 = 0.f, lo1 = 0.f;
    for (uint32_t base = b0; base < b1; base += 32) {
        const uint32_t cnt = min(32u, b1 - base);
        const bool live = (uint32_t)lane < cnt;
        const size_t a = (size_t)base + lane;
        double x[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) x[q] = live ? __ldg(rec + (size_t)q * n + a) : 0.0;
        const uint32_t cd = live ? __ldg(code + a) : 0u;
        __syncwarp();                       // the previous group's reads are done
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q * DEP_CELL_LD + lane] = x[q];
        cw[lane] = cd;
        __syncwarp();
        const int kend = (int)(cnt + 1) >> 1;
        if (PAIRS) {
            // four particles to an addition: their high floats by a tree of
            // exact two-sums, whose errors join the low floats
            for (int k = 0; k < kend; k += 4) {
                float h[2][4], l[2] = {0.f, 0.f};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int pp = 2 * (k + u) + par;      // particles past the group's end hold zeros
                    const double y = v[row * DEP_CELL_LD + pp];
                    const float2 f = make_float2(__uint_as_float((unsigned)__double2loint(y)),
                                                 __uint_as_float((unsigned)__double2hiint(y)));
                    const bool bit = ((cw[pp] >> bsh) & bmask) != 0u;
                    h[0][u] = bit ? 0.f : f.x;
                    h[1][u] = bit ? f.x : 0.f;
                    l[0] += bit ? 0.f : f.y;
                    l[1] += bit ? f.y : 0.f;
                }
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const ff a = ff_sum2(h[m][0], h[m][1]), c = ff_sum2(h[m][2], h[m][3]), t = ff_sum2(a.hi, c.hi);
                    l[m] += (a.lo + c.lo) + t.lo;
                    h[m][0] = t.hi;
                }
                acc0 += f2d_bits(h[0][0]);
                acc1 += f2d_bits(h[1][0]);
                lo0 += l[0];
                lo1 += l[1];
            }
            if (((base - b0) & 96u) == 96u) {
                acc0 += f2d_bits(lo0);
                acc1 += f2d_bits(lo1);
                lo0 = lo1 = 0.f;
            }
            continue;
        }
        for (int k = 0; k < kend; ++k) {
            const int pp = 2 * k + par;     // a particle past the group's end holds zeros
            const double y = v[row * DEP_CELL_LD + pp];
            const bool bit = ((cw[pp] >> bsh) & bmask) != 0u;
            const double s = sel_bits(bit, acc1, acc0) + y;
            acc1 = sel_bits(bit, s, acc1);
            acc0 = sel_bits(bit, acc0, s);
        }
    }
    acc0 += __shfl_xor_sync(0xffffffffu, acc0, 1);
    acc1 += __shfl_xor_sync(0xffffffffu, acc1, 1);
    // slot q = lane: rows ra (accumulator ua) and rb (accumulator 0, if any)
    int ra = lane, rb = -1;
    bool ua = false;
    if (lane >= 8 && lane < 14) {
        const int b = (lane - 8) / 3, kk = (lane - 8) % 3;
        ra = kk == 2 ? 9 + 2 * b : 8 + 2 * b;
        ua = kk != 0;
        rb = kk == 1 ? 9 + 2 * b : -1;
    } else if (lane >= 14 && lane < 20) {
        const int aa = (lane - 14) & 1, kk = (lane - 14) >> 1;
        ra = kk == 2 ? 14 + aa : 12 + aa;
        ua = kk != 0;
        rb = kk == 1 ? 14 + aa : -1;
    }
    const int la = 2 * (ra & 15), lb = 2 * (rb & 15);
    const double xa0 = __shfl_sync(0xffffffffu, acc0, la), xa1 = __shfl_sync(0xffffffffu, acc1, la);
    const double xb0 = __shfl_sync(0xffffffffu, acc0, lb);
    double tot = (ua ? xa1 : xa0) + (rb >= 0 ? xb0 : 0.0);
    if (PAIRS) {
        lo0 += __shfl_xor_sync(0xffffffffu, lo0, 1);
        lo1 += __shfl_xor_sync(0xffffffffu, lo1, 1);
        const float la0 = __shfl_sync(0xffffffffu, lo0, la), la1 = __shfl_sync(0xffffffffu, lo1, la);
        const float lb0 = __shfl_sync(0xffffffffu, lo0, lb);
        tot += f2d_bits((ua ? la1 : la0) + (rb >= 0 ? lb0 : 0.f));
    }
    if (lane < 20) part[(size_t)lane * C + cell] = tot;
}

struct NodeK {
    int Nr, Nth, ld;
    const double* part;
    uint32_t C;
    Tabs T;
    double *rho, *jr, *jt, *jp;
};

__global__ void k_dep_node(NodeK k)
{
    const int i = blockIdx.y;
    const int Nr = k.Nr, Nth = k.Nth;
    auto P = [&](int q, int ci, int cj) -> double {
        return k.part[(size_t)q * k.C + (size_t)ci * Nth + cj];
    };
    for (int j = threadIdx.x; j <= Nth; j += blockDim.x) {
        const size_t o = (size_t)i * k.ld + j;
        // rho, j^ph at (i, j): cells (i - a, j - b), slot a + 2b
        double sr = 0.0, sp = 0.0;
        for (int b = 0; b < 2; ++b)
            for (int a = 0; a < 2; ++a) {
                const int ci = i - a, cj = j - b;
                if (ci < 0 || ci >= Nr || cj < 0 || cj >= Nth) continue;
                sr += P(a + 2 * b, ci, cj);
                sp += P(4 + a + 2 * b, ci, cj);
            }
        k.rho[o] = sr / k.T.at(T_DUAL0, i, j);
        k.jp[o] = sp / k.T.at(T_DUAL0, i, j);
        // j^r at (i+1/2, j): cells (i + 1 - kk, j - b), slot kk + 3b
        if (i < Nr) {
            double sj = 0.0;
            for (int b = 0; b < 2; ++b)
                for (int kk = 0; kk < 3; ++kk) {
                    const int ci = i + 1 - kk, cj = j - b;
                    if (ci < 0 || ci >= Nr || cj < 0 || cj >= Nth) continue;
                    sj += P(8 + kk + 3 * b, ci, cj);
                }
            k.jr[o] = sj / k.T.at(T_DUAL1, i, j);
        }
        // j^th at (i, j+1/2): cells (i - a, j + 1 - kk), slot a + 2 kk
        if (j < Nth) {
            double sj = 0.0;
            for (int kk = 0; kk < 3; ++kk)
                for (int a = 0; a < 2; ++a) {
                    const int ci = i - a, cj = j + 1 - kk;
                    if (ci < 0 || ci >= Nr || cj < 0 || cj >= Nth) continue;
                    sj += P(14 + a + 2 * kk, ci, cj);
                }
            k.jt[o] = sj / k.T.at(T_DUAL2, i, j);
        }
    }
}

// ---------------------------------------------------------------------------
// FDTD (Sec. 2.1, Eqs. m3, m4, Ei; Sec. 2.5)
// ---------------------------------------------------------------------------
// Four launches a step, k_step_B twice in stage 1 and k_step_D twice in stage
// 2, each an auxiliary field and the update by its curl in one pass:
//   E_r (i+1/2,j) = alpha (g_rr D^r + g_rp <D^ph>),  E_th (i,j+1/2) = alpha g_tt
//   D^th - sqrtg beta <B^ph>,  E_ph (i,j) = alpha (g_rp <D^r> + g_pp D^ph) +
//   sqrtg beta <B^th>  (Eq. Ei; <.> the sqrtg-weighted mean of the two rows);
//   H_r (i,j+1/2) = alpha (g_rr B^r + g_rp <B^ph>),  H_th (i+1/2,j) = alpha g_tt
//   B^th + sqrtg beta <D^ph>,  H_ph (i+1/2,j+1/2) = alpha (g_rp <B^r> + g_pp
//   B^ph) - sqrtg beta <D^th>.
// A warp owns 31 adjacent columns (its 32nd lane holds the neighbour column
// the th differences need, exchanged by shuffles) and walks down `rows` rows
// with the neighbouring rows' values in registers: every array is read once
// and E, H go to memory only where the caller gets them (sub-steps 3 and 9).
// Bound by the FP64 pipe (75-78 % busy on about 160 operations a node and
// step; halvings and the tests for a factor of one are integer operations),
// with 140 doubles a node of traffic behind it.  Before, with E, H and the
// averages as arrays of their own, their metric products per node and the
// absorbing layer's exp and pow in every thread, it was 13 launches: a step
// on 1024 x 1024 809 -> 400 us, 4196 x 1024 full-theta 2645 -> 1433 us.
struct FK {
    int rows;           // rows of a warp, at most 16
    GridDev G;
    Tabs T;
    double dt, chi0, lam, r_abs, r_max;
    int conserving;     // sources are coordinate currents J (fpic_deposit_conserving)
};

struct P3 {
    double* p[3];
};

struct C3 {
    const double* p[3];
};

constexpr int FD_THREADS = 128, FD_COLS = 31;    // columns of a warp

// x^n with the products' rounding errors carried along: within an ulp.
__device__ __forceinline__ double powi_acc(double x, int n)
{
    double h = x, l = 0.0;
    for (int k = 1; k < n; ++k) {
        const double t = h * x, e = fma(h, x, -t);
        l = fma(l, x, e);
        h = t;
    }
    return h + l;
}

// Absorbing-layer factor exp(-chi dt), chi = chi0 ((r - r_abs)/(r_max -
// r_abs))^lambda beyond r_abs (Eqs. abs0-abs2).  A small whole lambda by
// multiplications: pow's latency would be most of a short launch.
__device__ __forceinline__ double damp(const FK& k, double r)
{
    if (k.chi0 <= 0.0 || r <= k.r_abs) return 1.0;
    const double x = (r - k.r_abs) / (k.r_max - k.r_abs);
    const int n = (int)k.lam;
    const double y = (k.lam == (double)n && n >= 1 && n <= 8) ? powi_acc(x, n) : pow(x, k.lam);
    return exp(-k.chi0 * y * k.dt);
}

// The factors of rows i0 .. i0 + 15, integer (lanes 0-15) and half (16-31).
__device__ __forceinline__ double damp_rows(const FK& k, int i0, int lane)
{
    const int i = i0 + (lane & 15);
    if (lane < 16) return i <= k.G.Nr ? damp(k, k.G.rn[i]) : 1.0;
    return i < k.G.Nr ? damp(k, k.G.rh[i]) : 1.0;
}

// Full-theta domain (Sec. 2.5, periodic in th): columns 0..Nth-1 are the
// distinct points; the thread of column 0 also stores its values in column
// Nth, the image the seam's stencils and the push's gather read.
__device__ __forceinline__ void put(double* F, size_t o, int j, const GridDev& G, double v)
{
    F[o] = v;
    if (G.full && j == 0) F[o + G.Nth] = v;
}

// Eq. (m4) + (abs0): Bout = (Bin - dt curl E / sqrtg) exp(-chi dt).  FIRST
// (sub-steps 1, 2): E from D = (D0 + D1) / 2 and B1, Bin = (B0 + B1) / 2; else
// (sub-steps 3, 4) E from D1 and Bh, stored, and Bin = B1.
template <bool FIRST>
__global__ void __launch_bounds__(FD_THREADS) k_step_B(const __grid_constant__ FK k, C3 D0, C3 D1, C3 B0, C3 B1,
                                                       C3 Bh, P3 E, P3 Bout)
{
    const GridDev& G = k.G;
    const int lane = threadIdx.x & 31;
    const int Nr = G.Nr, Nth = G.Nth;
    const int j = (blockIdx.x * (FD_THREADS / 32) + (threadIdx.x >> 5)) * FD_COLS + lane;
    if (j - lane > Nth) return;              // whole warps
    const int i0 = blockIdx.y * k.rows, i1 = min(i0 + k.rows, Nr + 1);
    const int jend = G.full ? Nth - 1 : Nth;
    const bool out = lane < FD_COLS && j <= jend;
    const bool in = j < Nth;                 // half th points
    // column read: the image column is column 0 itself, idle lanes read the last
    const int jj = (G.full && j == Nth) ? 0 : min(j, Nth);
    const double dmp = damp_rows(k, i0, lane);
    const size_t ld = (size_t)G.ld, sz = k.T.sz;
    const C3& Be = FIRST ? B1 : Bh;
    auto mean = [](double x, double y) { return half_of(x + y); };
    auto D = [&](int c, size_t o) { return FIRST ? mean(__ldg(D0.p[c] + o), __ldg(D1.p[c] + o)) : __ldg(D1.p[c] + o); };
    size_t o = (size_t)i0 * ld + jj;
    const double* T = k.T.m + o;
    auto tab = [&](int t) { return __ldg(T + (size_t)t * sz); };
    // row i0's E_th, E_ph
    double Dr, Dp = D(2, o), Bt, Bp, Et, Ep;
    {
        const size_t om = i0 > 0 ? o - ld : o, oc = i0 < Nr ? o : o - ld;
        const double Drm = D(0, om), Btm = __ldg(Be.p[1] + om), Bpm = __ldg(Be.p[2] + om);
        Dr = D(0, oc);
        Bt = __ldg(Be.p[1] + oc);
        Bp = __ldg(Be.p[2] + oc);
        Et = fma(tab(F_ET_D), D(1, o), fma(tab(F_ET_B0), Bpm, tab(F_ET_B1) * Bp));
        Ep = fma(tab(F_EP_D), Dp, fma(tab(F_EP_R0), Drm, tab(F_EP_R1) * Dr));
        Ep = fma(tab(F_EP_T0), Btm, fma(tab(F_EP_T1), Bt, Ep));
    }
    for (int i = i0; i < i1; ++i, o += ld, T += ld) {
        const double dn = __shfl_sync(0xffffffffu, dmp, i - i0), dh = __shfl_sync(0xffffffffu, dmp, 16 + i - i0);
        const double EpR = __shfl_down_sync(0xffffffffu, Ep, 1);
        if (!FIRST && out) {
            if (in) put(E.p[1], o, j, G, Et);
            put(E.p[2], o, j, G, Ep);
        }
        if (out && in) {   // B^r (i, j+1/2)
            const double b = FIRST ? mean(__ldg(B0.p[0] + o), __ldg(B1.p[0] + o)) : __ldg(B1.p[0] + o);
            double v = fma(-k.dt, tab(F_BR) * (EpR - Ep), b);
            if (!is_one(dn)) v *= dn;
            put(Bout.p[0], o, j, G, v);
        }
        if (i == Nr) break;
        // row i+1 (its own half row held at Nr - 1)
        const size_t on = o + ld, oc = i + 1 < Nr ? on : o;
        const double Dpn = D(2, on), Drn = D(0, oc), Btn = __ldg(Be.p[1] + oc), Bpn = __ldg(Be.p[2] + oc);
        const double Er = fma(tab(F_ER_D), Dr, fma(tab(F_ER_P0), Dp, tab(F_ER_P1) * Dpn));
        auto tabn = [&](int t) { return __ldg(T + ld + (size_t)t * sz); };
        const double Etn = fma(tabn(F_ET_D), D(1, on), fma(tabn(F_ET_B0), Bp, tabn(F_ET_B1) * Bpn));
        double Epn = fma(tabn(F_EP_D), Dpn, fma(tabn(F_EP_R0), Dr, tabn(F_EP_R1) * Drn));
        Epn = fma(tabn(F_EP_T0), Bt, fma(tabn(F_EP_T1), Btn, Epn));
        const double ErR = __shfl_down_sync(0xffffffffu, Er, 1);
        if (out) {
            if (!FIRST) put(E.p[0], o, j, G, Er);
            {   // B^th (i+1/2, j)
                const double b = FIRST ? mean(__ldg(B0.p[1] + o), Bt) : __ldg(B1.p[1] + o);
                double v = fma(k.dt, tab(F_BT) * (Epn - Ep), b);
                if (!is_one(dh)) v *= dh;
                put(Bout.p[1], o, j, G, v);
            }
            if (in) {   // B^ph (i+1/2, j+1/2)
                const double b = FIRST ? mean(__ldg(B0.p[2] + o), Bp) : __ldg(B1.p[2] + o);
                double v = fma(-k.dt, fma(tab(F_BPR), Etn - Et, -tab(F_BPT) * (ErR - Er)), b);
                if (!is_one(dh)) v *= dh;
                put(Bout.p[2], o, j, G, v);
            }
        }
        Et = Etn;
        Ep = Epn;
        Dr = Drn;
        Dp = Dpn;
        Bt = Btn;
        Bp = Bpn;
    }
}

struct Src {
    const double *j[3], *rho;
};

// Eq. (m3) + (abs1): Dout = (Din + dt [curl H / sqrtg - 4 pi J]) exp(-chi dt).
// FIRST (sub-steps 7, 8): H from B and D = D1, Din = (D0 + D1) / 2, J the mean
// of both levels; else (9, 10) H from B and D = Dw, stored, Din = D1, J = S1.
// Interior points; the boundaries follow from them (Sec. 2.5, reading: zero
// gradient where a stencil is one-sided, D^ph = 0 on the axis) and are stored
// by the threads of the rows and columns they copy.  Full-theta domain: D^r
// and D^ph at j = 0 too, their backward th difference across the seam (half
// node Nth-1), no th boundary.
template <bool FIRST>
__global__ void __launch_bounds__(FD_THREADS) k_step_D(const __grid_constant__ FK k, C3 D0, C3 D1, C3 D, C3 B, Src S0,
                                                       Src S1, P3 H, P3 Dout)
{
    const GridDev& G = k.G;
    const int lane = threadIdx.x & 31;
    const int Nr = G.Nr, Nth = G.Nth;
    const int j = (blockIdx.x * (FD_THREADS / 32) + (threadIdx.x >> 5)) * FD_COLS + lane - 1;
    if (j - lane + 1 > Nth) return;          // whole warps
    const int i0 = blockIdx.y * k.rows, i1 = min(i0 + k.rows, Nr + 1);
    const bool out = lane > 0 && j <= (G.full ? Nth - 1 : Nth);
    const bool in = j < Nth;                 // half th points
    const bool mid = out && in && (G.full || j >= 1);            // D^r, D^ph updated
    // column read: below column 0 the period's last, idle lanes the last
    const int jj = j < 0 ? (G.full ? Nth - 1 : 0) : min(j, Nth);
    const double dmp = damp_rows(k, i0, lane);
    const size_t ld = (size_t)G.ld, sz = k.T.sz;
    const double mfpi = -4.0 * M_PI;
    auto mean = [](double x, double y) { return half_of(x + y); };
    auto Din = [&](int c, size_t o, double d1) { return FIRST ? mean(__ldg(D0.p[c] + o), d1) : __ldg(D1.p[c] + o); };
    auto src = [&](int c, size_t o) { return FIRST ? mean(__ldg(S0.j[c] + o), __ldg(S1.j[c] + o)) : __ldg(S1.j[c] + o); };
    auto rho = [&](size_t o) { return FIRST ? mean(__ldg(S0.rho + o), __ldg(S1.rho + o)) : __ldg(S1.rho + o); };
    const int is = max(i0 - 1, 0);           // row i0 - 1's H_th, H_ph come first
    size_t o = (size_t)is * ld + jj;
    const double* T = k.T.m + o;
    auto tab = [&](int t) { return __ldg(T + (size_t)t * sz); };
    double Br = __ldg(B.p[0] + o), Dt = __ldg(D.p[1] + o), Dp = __ldg(D.p[2] + o), Bp = is > 0 ? __ldg(B.p[2] + o - ld) : __ldg(B.p[2] + o);
    double Htm = 0.0, Hpm = 0.0, rh = k.conserving ? 0.0 : rho((size_t)i0 * ld + jj);
    for (int i = is; i < i1; ++i, o += ld, T += ld) {
        const bool own = i >= i0;
        double Ht = 0.0, Hp = 0.0, Bpi = Bp, Brn = 0.0, Dtn = 0.0, Dpn = 0.0, Bt = 0.0;
        if (i < Nr) {
            const size_t on = o + ld;
            Bpi = __ldg(B.p[2] + o);
            Bt = __ldg(B.p[1] + o);
            Brn = __ldg(B.p[0] + on);
            Dtn = __ldg(D.p[1] + on);
            Dpn = __ldg(D.p[2] + on);
            Ht = fma(tab(F_HT_B), Bt, fma(tab(F_HT_D0), Dp, tab(F_HT_D1) * Dpn));
            Hp = fma(tab(F_HP_B), Bpi, fma(tab(F_HP_R0), Br, tab(F_HP_R1) * Brn));
            Hp = fma(tab(F_HP_T0), Dt, fma(tab(F_HP_T1), Dtn, Hp));
        }
        if (own) {
            // Bp: row i - 1 (row 0 at the lower end), Bpi: row i (row Nr - 1 at the upper end)
            const double Hr = fma(tab(F_HR_B), Br, fma(tab(F_HR_P0), Bp, tab(F_HR_P1) * Bpi));
            const double dn = __shfl_sync(0xffffffffu, dmp, i - i0), dh = __shfl_sync(0xffffffffu, dmp, 16 + i - i0);
            const double HrL = __shfl_up_sync(0xffffffffu, Hr, 1), HpL = __shfl_up_sync(0xffffffffu, Hp, 1);
            if (!FIRST && out) {
                if (in) put(H.p[0], o, j, G, Hr);
                if (i < Nr) put(H.p[1], o, j, G, Ht);
                if (i < Nr && in) put(H.p[2], o, j, G, Hp);
            }
            if (mid && i < Nr) {   // D^r (i+1/2, j)
                double J = (k.conserving ? mfpi : tab(F_JR)) * src(0, o);
                if (!k.conserving) {
                    const double rn = rho(o + ld);
                    J = fma(tab(F_JR0), rh, fma(tab(F_JR1), rn, J));
                    rh = rn;
                }
                const double d = FIRST ? __ldg(D1.p[0] + o) : 0.0;
                double v = fma(k.dt, fma(tab(F_DR), Hp - HpL, J), Din(0, o, d));
                if (!is_one(dh)) v *= dh;
                put(Dout.p[0], o, j, G, v);
                if (!G.full) {
                    if (j == 1) Dout.p[0][o - 1] = v;
                    if (j == Nth - 1) Dout.p[0][o + 1] = v;
                }
            }
            if (i >= 1 && i < Nr && out && in) {   // D^th (i, j+1/2)
                const double J = (k.conserving ? mfpi : tab(F_JT)) * src(1, o);
                double v = fma(k.dt, fma(-tab(F_DT), Hp - Hpm, J), Din(1, o, Dt));
                if (!is_one(dn)) v *= dn;
                put(Dout.p[1], o, j, G, v);
                if (i == 1) put(Dout.p[1], o - ld, j, G, v);
                if (i == Nr - 1) put(Dout.p[1], o + ld, j, G, v);
            }
            if (i >= 1 && i < Nr && mid) {   // D^ph (i, j)
                const double J = (k.conserving ? mfpi : tab(F_JP)) * src(2, o);
                const double c = fma(tab(F_DPR), Ht - Htm, fma(-tab(F_DPT), Hr - HrL, J));
                double v = fma(k.dt, c, Din(2, o, Dp));
                if (!is_one(dn)) v *= dn;
                put(Dout.p[2], o, j, G, v);
                if (i == 1) put(Dout.p[2], o - ld, j, G, v);
                if (i == Nr - 1) put(Dout.p[2], o + ld, j, G, v);
            }
            if (!G.full && out && (j == 0 || j == Nth)) Dout.p[2][o] = 0.0;
        }
        Htm = Ht;
        Hpm = Hp;
        Bp = Bpi;
        Br = Brn;
        Dt = Dtn;
        Dp = Dpn;
    }
}

}  // namespace fpic

using namespace fpic;

static Tabs tabs_of(const fpic_ctx* c)
{
    return Tabs{c->d_metric, c->metric_stride, c->ld};
}

extern "C" int fpic_sort(fpic_ctx* c, fpic_particles* p, void* stream)
{
    if (!c || !p) return set_error(FPIC_EINVAL, "fpic_sort: NULL argument");
    if (!c->has_grid) return set_error(FPIC_EINVAL, "fpic_sort: no grid set");
    if (p->n < 0 || p->n >= (1LL << 31)) return set_error(FPIC_EINVAL, "fpic_sort: n out of range");
    if (p->n == 0) return FPIC_OK;
    if (!particles_ok(p, true) || !p->w) return set_error(FPIC_EINVAL, "fpic_sort: NULL particle array");
    FPIC_CUDA(cudaSetDevice(c->device));
    Work w;
    int rc = work_layout(c, p->n, false, w);
    if (rc) return rc;
    return sort_impl(c, p, w, (cudaStream_t)stream);
}

namespace fpic {
static ff ff_host(double x)
{
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}

static BHff bh_ff(const BH& bh)
{
    return {ff_host(bh.twoM), ff_host(bh.a2), ff_host(1.0 / 3.0)};
}
}  // namespace fpic

extern "C" int fpic_deposit(fpic_ctx* c, fpic_particles* p, double* rho, double* jr, double* jth, double* jph,
                            void* stream)
{
    if (c && c->G.full) return set_error(FPIC_EINVAL, "fpic_deposit: not built for the full-theta domain");
    if (!c || !p || !rho || !jr || !jth || !jph) return set_error(FPIC_EINVAL, "fpic_deposit: NULL argument");
    if (!c->has_grid) return set_error(FPIC_EINVAL, "fpic_deposit: no grid set");
    if (p->n < 0 || p->n >= (1LL << 31)) return set_error(FPIC_EINVAL, "fpic_deposit: n out of range");
    if (p->n > 0 && (!particles_ok(p, true) || !p->w)) return set_error(FPIC_EINVAL, "fpic_deposit: NULL particle array");
    FPIC_CUDA(cudaSetDevice(c->device));
    cudaStream_t s = (cudaStream_t)stream;
    const long long n = p->n;
    const uint32_t C = (uint32_t)c->Nr * (uint32_t)c->Nth;
    Work w;
    int rc = work_layout(c, n > 0 ? n : 1, true, w);
    if (rc) return rc;
    if (n > 0) {
        rc = sort_impl(c, p, w, s, w.rec);
        if (rc) return rc;
    } else {
        FPIC_CUDA(cudaMemsetAsync(w.off, 0, 4 * ((size_t)C + 2), s));
    }
    PolyTab pt;
    int poly = 0;
    if (n > 0 && c->dep_lattice) {
        rc = poly_tables(c, pt, poly, s);
        if (rc) return rc;
    }
    // alive particles occupy [0, off[C]) after the sort; the count is read on the device
    DepK k{c->bh, bh_ff(c->bh), c->G, c->d_metric + (size_t)MT_N * c->metric_stride, p->r, p->th, p->ur, p->uth, p->uph, p->qm, p->w, n, w.rec, w.code};
    if (n > 0) {
        // rec/code for all n slots; removed particles (past off[C]) are never summed
        const int dt_ = c->dep_threads;
        const unsigned nb = (unsigned)((n + dt_ - 1) / dt_);
        if (!c->dep_lattice) k_dep_particle<<<nb, dt_, 0, s>>>(k);
        else if (poly == 5) k_dep_particle_poly<5><<<nb, dt_, 0, s>>>(k, pt);
        else if (poly == 6) k_dep_particle_poly<6><<<nb, dt_, 0, s>>>(k, pt);
        else k_dep_particle_ff<<<nb, dt_, 0, s>>>(k);
    }
    const unsigned cb = (unsigned)(((long long)C + DEP_CELL_WARPS - 1) / DEP_CELL_WARPS);
    if (poly) k_dep_cell<true><<<cb, 32 * DEP_CELL_WARPS, 0, s>>>(w.rec, w.code, w.off, w.part, n, C);
    else k_dep_cell<false><<<cb, 32 * DEP_CELL_WARPS, 0, s>>>(w.rec, w.code, w.off, w.part, n > 0 ? n : 1, C);
    NodeK nk{c->Nr, c->Nth, c->ld, w.part, C, tabs_of(c), rho, jr, jth, jph};
    k_dep_node<<<dim3(1, c->Nr + 1), 256, 0, s>>>(nk);
    FPIC_CUDA(cudaGetLastError());
    return FPIC_OK;
}

namespace fpic {
// ---------------------------------------------------------------------------
// Charge-conserving deposit (an extension; the paper's deposit is not and
// relies on the cleaning of Sec. 2.4)
// ---------------------------------------------------------------------------
// A move from x^n to x^{n+1} with linear (area) node weights S = S_r S_th,
// split Esirkepov's way on the 3 x 3 window of integer nodes spanned by the
// two stencils: W_r = dS_r <S_th>, W_th = <S_r> dS_th (<.> the mean of old
// and new), charge crossing the dual face between window nodes x and x+1 in
// +r: -Q sum_{x' <= x} W_r(x', y) (alike in th).  Window partials (30 per
// particle: Q S^new and Q <S> (dph/dt)_mid on 3 x 3 nodes, 2 x 3 r faces,
// 3 x 2 th faces) are summed per window-base cell in particle-index order,
// then gathered per node / face in a fixed order: bitwise reproducible.
// Normalised by the Yee cell (2 pi sqrtg dr_dual dth_dual) so that sqrtg
// (rho^{n+1} - rho^n) + dt Yee-div(sqrtg J) = 0 at every node.
//
// A move inside one cell (all but a few per cent at a PIC step) has only 12
// partials that are not zero, products of the two positions' cell fractions;
// it is keyed to its cell, a move across a boundary to a second set of
// buckets, so that k_cdep_particle works through each kind densely, one
// thread per particle, and k_cdep_cell adds the records up.  FP64-pipe
// bound: with one warp per cell, its 30 partials by every lane and a
// reduction tree, a cell of 16 particles left half the lanes idle:
// 4.0e6 particles on 512 x 512 3604 us, then 842 (particles, 86 % of the pipe,
// 113 FP64 operations each; some 435 with 43, see phdot_x) + 188 (cells).
enum { CD_Q = 0, CD_P = 9, CD_R = 18, CD_T = 24, CD_SLOTS = 30 };
// rows of a move inside its cell: Q and P at node (x, y) in row x + 2 y, the r
// face's charge at th node y, the th face's at r node x
enum { CI_Q = 0, CI_P = 4, CI_R = 8, CI_T = 10, CI_ROWS = 12 };

struct CDepK {
    int Nr, Nth, ld;
    GridDev G;
    BH bh;
    long long n;
    const double *r0, *t0, *ur0, *ut0, *up0;
    const uint8_t* alive0;
    const double *r1, *t1, *ur1, *ut1, *up1, *qm, *w;
    const double* trig;      // sin tn[0..Nth], then cos tn[0..Nth]
};

__device__ __forceinline__ void cd_lin(const GridDev& G, double r, double t, int& i, double& fr, int& j, double& ft)
{
    const float lr = __logf(f32_est(r));
    locate(G.rn, G.irn, G.Nr + 1, r, (lr - G.lr0) * G.ilr, i, fr);
    locate(G.tn, G.itn, G.Nth + 1, t, (f32_est(t) - G.t0) * G.it, j, ft);
}

// Bucket of each particle alive before the move: its cell, or C + the window
// base cell of a move across a boundary (2 C: skipped / removed).
__global__ void k_cdep_keys(CDepK k, uint32_t* key, uint32_t* count, uint32_t C, long long* n_skip)
{
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const bool valid = p < k.n;
    uint32_t kk = 2 * C;
    if (valid && k.alive0[p]) {
        int ia, ja, ib, jb;
        double f;
        cd_lin(k.G, k.r0[p], k.t0[p], ia, f, ja, f);
        cd_lin(k.G, k.r1[p], k.t1[p], ib, f, jb, f);
        if (abs(ia - ib) > 1 || abs(ja - jb) > 1) atomicAdd((unsigned long long*)n_skip, 1ull);
        else kk = (uint32_t)min(ia, ib) * (uint32_t)k.Nth + (uint32_t)min(ja, jb) + (ia == ib && ja == jb ? 0u : C);
    }
    if (valid) key[p] = kk;
    count_key(count, kk, valid);
}

// coordinate dph/dt = alpha gamma^{ph j} u_j / Gamma on integer mantissas
// (xf.cuh), the metric as in rhs_x: in FP64 (cd_phdot_f64) the two states' took
// 70 of k_cdep_particle's 113 FP64 instructions, on a pipe 86 % busy with 18 %
// of the issue slots used (conserving deposit of 4.0e6 particles on 512^2 1225 ->
// 818 us).  False as rhs_x is.
FPIC_HD bool phdot_x(const BH& bh, double r_, double s, double c, double ur_, double ut_, double up_, xf& v)
{
    const double z[7] = {c, ur_, ut_, up_, bh.a, bh.a2, bh.twoM};
    unsigned big = 0;
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        const unsigned h = (unsigned)(x_bits(z[i]) >> 32) & 0x7fffffffu;
        big = big > h ? big : h;
    }
    const unsigned hr = (unsigned)(x_bits(r_) >> 32), hs = (unsigned)(x_bits(s) >> 32);
    if (big >= 0x7ff00000u || hr - 0x00100000u >= 0x7fe00000u || hs - 0x00100000u >= 0x7fe00000u) return false;
    const xf r = x_from_pos(r_), sx = x_from_pos(s), ur = x_from(ur_), ut = x_from(ut_), up = x_from(up_);
    const xf a = x_from(bh.a), one = x_pow2(0), s2 = x_sqr(sx);
    const xf rho2 = x_norm(x_add(x_sqr(r), x_mul(x_from(bh.a2), x_sqr(x_from(c)))));
    const xf t = x_rcp(x_mul(rho2, s2)), irho2 = x_norm(x_mul(t, s2));
    const xf alpha = x_rsqrt(x_add(one, x_mul(x_mul(x_from(bh.twoM), irho2), r)));
    const xf g1 = x_norm(x_add(x_mul(x_mul(a, s2), ur), up)), iu = x_mul(x_sqr(alpha), ur), tu = x_norm(x_mul(t, up));
    const xf W = x_norm(x_add(x_mul(x_mul(a, ur), x_add(g1, up)), x_sqr(ut)));
    const xf G2 = x_norm(x_add3(one, x_mul(iu, ur), x_add(x_mul(W, irho2), x_mul(tu, up))));
    if (G2.m <= 0) return false;
    v = x_norm(x_mul(x_mul(alpha, x_rsqrt(G2)), x_add(x_mul(x_mul(a, irho2), ur), tu)));
    return true;
}

static __device__ __noinline__ double cd_phdot_f64(const BH& bh, double r, double s, double c, double ur, double ut,
                                                   double up)
{
    const double s2 = s * s, rho2 = fma(bh.a2, c * c, r * r);
    const double gpp = rcp_nr(rho2 * s2), irho2 = gpp * s2;
    const double alpha = rsqrt_nr(fma(bh.twoM * irho2, r, 1.0));
    const double iu = (alpha * alpha) * ur, tu = gpp * up, g1 = fma(bh.a * s2, ur, up);
    const double Q = fma(fma(bh.a * ur, g1 + up, ut * ut), irho2, tu * up);
    const double iG = rsqrt_nr(fma(iu, ur, 1.0 + Q));
    return alpha * fma(bh.a * irho2, ur, tu) * iG;
}

// The sum of both states' dph/dt, sin/cos th by angle addition from the
// tabulated node tn[j] of each one's cell.
__device__ __forceinline__ double cd_phdots(const CDepK& k, uint32_t p, const double r[2], const double t[2],
                                            const int j[2])
{
    xf v[2];
    double d[2];
    bool ok = true;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        double s, c;
        sincos_near(k.G.tn[j[q]], k.trig[j[q]], k.trig[k.G.Nth + 1 + j[q]], t[q], s, c);
        const double ur = q ? k.ur1[p] : k.ur0[p], ut = q ? k.ut1[p] : k.ut0[p], up = q ? k.up1[p] : k.up0[p];
        d[q] = 0.0;
        if (!phdot_x(k.bh, r[q], s, c, ur, ut, up, v[q])) {
            ok = false;
            v[q] = {0, XF_ZERO_E};
            d[q] = cd_phdot_f64(k.bh, r[q], s, c, ur, ut, up);
        }
    }
    const double x = x_to(x_add(v[0], v[1]));
    return ok ? x : x + (d[0] + d[1]);
}

// The records' buffer holds CDEP_CHUNK sorted entries (16 GB of 30 rows) at most,
// and fewer where the memory left does not hold that many: the rest take it in
// turns, each chunk's cell sums added to the ones before.  (240 bytes a particle
// are 72 GB at 3e8, which would not fit beside them.)  In turns a deposit is some
// 10 % longer -- 6.4e7 particles on 1024^2 10.8 ms at once, 12.0 in four chunks:
// the moves across boundaries, last in order, add to every cell once more.
constexpr long long CDEP_CHUNK = 67000000, CDEP_CHUNK_MIN = 1000000;

// One thread per sorted entry a0 .. a0 + m - 1: entries below off[C] are moves
// inside their cell (CI_ROWS records), the rest up to off[2 C] the general ones
// (CD_SLOTS).
__global__ void __launch_bounds__(128) k_cdep_particle(const __grid_constant__ CDepK k,
                                                       const uint32_t* __restrict__ off,
                                                       const uint32_t* __restrict__ perm, double* __restrict__ rec,
                                                       long long a0, long long m, uint32_t C)
{
    const long long t = blockIdx.x * 128LL + threadIdx.x, a = a0 + t;
    if (t >= m || a >= (long long)off[2 * (size_t)C]) return;
    const uint32_t p = perm[a];
    const bool inside = a < (long long)off[C];
    int ia, ja, ib, jb;
    double fra, fta, frb, ftb;
    const double r0 = k.r0[p], t0 = k.t0[p], r1 = k.r1[p], t1 = k.t1[p];
    cd_lin(k.G, r0, t0, ia, fra, ja, fta);
    cd_lin(k.G, r1, t1, ib, frb, jb, ftb);
    const double Q = k.w[p] * k.qm[p];
    const double rr[2] = {r0, r1}, tt[2] = {t0, t1};
    const int jj[2] = {ja, jb};
    const double Qh = 0.25 * Q * cd_phdots(k, p, rr, tt, jj);         // Q (dph/dt)_mid / 2
    rec += t;
    auto put = [&](int row, double v) { rec[row * m] = v; };
    if (inside) {
        const double qx = Q * frb, qc = fma(-Q, frb, Q);
        put(CI_Q + 0, fma(-qc, ftb, qc));
        put(CI_Q + 1, fma(-qx, ftb, qx));
        put(CI_Q + 2, qc * ftb);
        put(CI_Q + 3, qx * ftb);
        const double sx = fra + frb, sy = fta + ftb, px = Qh * sx;
        const double p11 = Qh * fma(fra, fta, frb * ftb), p01 = fma(Qh, sy, -p11);
        put(CI_P + 0, fma(2.0, Qh, -px) - p01);
        put(CI_P + 1, px - p11);
        put(CI_P + 2, p01);
        put(CI_P + 3, p11);
        const double qr = Q * (frb - fra), qt = Q * (ftb - fta);
        const double r1h = half_of(qr) * sy, t1h = half_of(qt) * sx;
        put(CI_R + 0, qr - r1h);
        put(CI_R + 1, r1h);
        put(CI_T + 0, qt - t1h);
        put(CI_T + 1, t1h);
        return;
    }
    // window weights by selects (registers, no indexed local arrays)
    const int da = ia - min(ia, ib), db = ib - min(ia, ib), ea = ja - min(ja, jb), eb = jb - min(ja, jb);
    double Sra[3], Srb[3], Sta[3], Stb[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
        Sra[x] = x == da ? 1.0 - fra : (x == da + 1 ? fra : 0.0);
        Srb[x] = x == db ? 1.0 - frb : (x == db + 1 ? frb : 0.0);
        Sta[x] = x == ea ? 1.0 - fta : (x == ea + 1 ? fta : 0.0);
        Stb[x] = x == eb ? 1.0 - ftb : (x == eb + 1 ? ftb : 0.0);
    }
#pragma unroll
    for (int x = 0; x < 3; ++x) {
        const double q = Q * Srb[x];
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            put(CD_Q + 3 * x + y, q * Stb[y]);
            put(CD_P + 3 * x + y, Qh * fma(Sra[x], Sta[y], Srb[x] * Stb[y]));
        }
    }
#pragma unroll
    for (int y = 0; y < 3; ++y) {
        const double sSt = Sta[y] + Stb[y];
        double s_ = 0.0;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            s_ = fma(0.5 * (Srb[x] - Sra[x]), sSt, s_);
            put(CD_R + 3 * x + y, -Q * s_);
        }
    }
#pragma unroll
    for (int x = 0; x < 3; ++x) {
        const double aSr = 0.5 * (Sra[x] + Srb[x]);
        double s_ = 0.0;
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            s_ = fma(aSr, Stb[y] - Sta[y], s_);
            put(CD_T + 2 * x + y, -Q * s_);
        }
    }
}

// One warp per cell: the 12 rows of its inside moves (32 particles at a time
// through shared memory, lane 2 row + parity sums its row over every other pair
// of particles), then lane q < 30 slot q of its general moves; both in a fixed
// order, a group of 32 by itself (the inside moves as a tree, neighbours first, as
// electrons and positrons alternate): as many additions as one after the other
// in shorter chains (rho of 60 particles a cell 9e-16 -> 2.7e-16 off).  Of the entries a0 .. a0 + m - 1; LATER: a chunk
// after the first, which adds to the sums of the cells it has entries of (a block
// looks at CDEP_CELLS neighbours and leaves if they have none).
constexpr int CDEP_WARPS = 8, CDEP_CELLS = 64;
template <bool LATER>
__global__ void __launch_bounds__(32 * CDEP_WARPS) k_cdep_cell(const double* __restrict__ rec,
                                                               const uint32_t* __restrict__ off, uint32_t a0,
                                                               uint32_t m, double* __restrict__ part, uint32_t C)
{
    __shared__ double sv[CDEP_WARPS][CI_ROWS * DEP_CELL_LD];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double* v = sv[wid];
    const int row = min(lane >> 1, CI_ROWS - 1), par = lane & 1;
    // entry a's place in the chunk
    const auto at = [&](uint32_t a) { return min(LATER ? (a > a0 ? a - a0 : 0u) : a, m); };
    const long long first = blockIdx.x * (long long)(LATER ? CDEP_CELLS : CDEP_WARPS);
    const long long last = LATER ? min(first + CDEP_CELLS, (long long)C) : (long long)C;
    if (LATER && at(off[first]) == at(off[last]) && at(off[(size_t)C + first]) == at(off[(size_t)C + last])) return;
    long long cell = first + wid;
    if (cell >= last) return;               // whole warps
    do {
        const uint32_t b0 = at(off[cell]), b1 = at(off[cell + 1]), c0 = at(off[(size_t)C + cell]),
                       c1 = at(off[(size_t)C + cell + 1]);
        if (b0 == b1 && c0 == c1) {             // an empty cell
            if (!LATER && lane < CD_SLOTS) part[(size_t)lane * C + cell] = 0.0;
            continue;
        }
        double acc = 0.0;
        for (uint32_t base = b0; base < b1; base += 32) {
            const uint32_t cnt = min(32u, b1 - base);
            const bool live = (uint32_t)lane < cnt;
            double x[CI_ROWS];
#pragma unroll
            for (int q = 0; q < CI_ROWS; ++q) x[q] = live ? __ldg(rec + (size_t)q * m + base + lane) : 0.0;
            __syncwarp();                       // the previous group's reads are done
#pragma unroll
            for (int q = 0; q < CI_ROWS; ++q) v[q * DEP_CELL_LD + lane] = x[q];
            __syncwarp();
            const double* u = v + row * DEP_CELL_LD + 2 * par;   // particles past the group's end hold zeros
            const auto four = [&](int k) { return (u[k] + u[k + 1]) + (u[k + 4] + u[k + 5]); };
            double t = four(0);
            if (cnt > 8) t += four(8);
            if (cnt > 16) t += cnt > 24 ? four(16) + four(24) : four(16);
            acc += t;
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        double g = 0.0;
        const int slot = min(lane, CD_SLOTS - 1);
        const double* rs = rec + (size_t)slot * m;
        for (uint32_t a = c0; a < c1;) {
            double t = 0.0;
            for (const uint32_t e = min(a + 32u, c1); a < e; ++a) t += __ldg(rs + a);
            g += t;
        }
        // the inside row that belongs to this lane's slot, if any
        int src = -1;
        if (slot < CD_R) {
            const int q = slot % 9, x = q / 3, y = q % 3;
            if (x < 2 && y < 2) src = (slot < CD_P ? CI_Q : CI_P) + x + 2 * y;
        } else if (slot < CD_T) {
            if (slot - CD_R < 2) src = CI_R + (slot - CD_R);
        } else if (slot == CD_T || slot == CD_T + 2) {
            src = CI_T + ((slot - CD_T) >> 1);
        }
        const double in = __shfl_sync(0xffffffffu, acc, 2 * max(src, 0));
        if (lane < CD_SLOTS) {
            double* o = part + (size_t)lane * C + cell;
            const double sum = src >= 0 ? in + g : g;
            *o = LATER ? *o + sum : sum;
        }
    } while (LATER && (cell += CDEP_WARPS) < last);
}

__device__ __forceinline__ double cd_dual_r(const GridDev& G, int i)
{
    return (i == G.Nr ? G.rn[G.Nr] : G.rh[i]) - (i == 0 ? G.rn[0] : G.rh[i - 1]);
}

__device__ __forceinline__ double cd_dual_t(const GridDev& G, int j)
{
    return (j == G.Nth ? M_PI : G.th[j]) - (j == 0 ? 0.0 : G.th[j - 1]);
}

// per node / face: the partials of the window cells covering it, fixed order
__global__ void k_cdep_node(CDepK k, Tabs T, const double* __restrict__ part, uint32_t C, double dt, double* rho,
                            double* Jr, double* Jt, double* Jp)
{
    const int i = blockIdx.y;
    const GridDev& G = k.G;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j <= k.Nth; j += gridDim.x * blockDim.x) {
        const size_t o = (size_t)i * k.ld + j;
        double Q = 0.0, Pp = 0.0, Fr = 0.0, Ft = 0.0;
        for (int x = 0; x < 3; ++x)
            for (int y = 0; y < 3; ++y) {
                const int ci = i - x, cj = j - y;
                if (ci < 0 || ci >= k.Nr || cj < 0 || cj >= k.Nth) continue;
                const size_t cell = (size_t)ci * k.Nth + cj;
                Q += part[(size_t)(CD_Q + 3 * x + y) * C + cell];
                Pp += part[(size_t)(CD_P + 3 * x + y) * C + cell];
                if (x < 2) Fr += part[(size_t)(CD_R + 3 * x + y) * C + cell];
                if (y < 2) Ft += part[(size_t)(CD_T + 2 * x + y) * C + cell];
            }
        const double drd = cd_dual_r(G, i), dtd = cd_dual_t(G, j);
        const double vol = 2.0 * M_PI * T.at(T_SG0, i, j) * drd * dtd;
        rho[o] = vol > 0.0 ? Q / vol : 0.0;
        Jp[o] = vol > 0.0 ? Pp / vol : 0.0;
        if (i < k.Nr) Jr[o] = Fr / (dt * 2.0 * M_PI * T.at(T_SG1, i, j) * dtd);
        else Jr[o] = 0.0;
        if (j < k.Nth) Jt[o] = Ft / (dt * 2.0 * M_PI * T.at(T_SG2, i, j) * drd);
        else Jt[o] = 0.0;
    }
}
}  // namespace fpic

extern "C" int fpic_deposit_conserving(fpic_ctx* c, const fpic_particles* before, const fpic_particles* after,
                                       double dt, double* rho, double* jr, double* jth, double* jph,
                                       long long* n_skipped, void* stream)
{
    if (c && c->G.full) return set_error(FPIC_EINVAL, "fpic_deposit_conserving: not built for the full-theta domain");
    if (!c || !before || !after || !rho || !jr || !jth || !jph)
        return set_error(FPIC_EINVAL, "fpic_deposit_conserving: NULL argument");
    if (!c->has_grid) return set_error(FPIC_EINVAL, "fpic_deposit_conserving: no grid set");
    if (before->n != after->n || after->n < 0) return set_error(FPIC_EINVAL, "fpic_deposit_conserving: n mismatch");
    if (!(std::isfinite(dt)) || dt == 0.0) return set_error(FPIC_EINVAL, "fpic_deposit_conserving: dt must be finite and nonzero");
    const long long n = after->n;
    if (n > 0 && (!before->r || !before->th || !before->ur || !before->uth || !before->uph || !before->alive ||
                  !after->r || !after->th || !after->ur || !after->uth || !after->uph || !after->qm || !after->w))
        return set_error(FPIC_EINVAL, "fpic_deposit_conserving: NULL particle array");
    if (n >= (1LL << 32)) return set_error(FPIC_EINVAL, "fpic_deposit_conserving: more than 2^32 particles");
    FPIC_CUDA(cudaSetDevice(c->device));
    cudaStream_t s = (cudaStream_t)stream;
    const long long C = (long long)c->Nr * c->Nth;
    Work w;
    void* part_v = nullptr;     // per-cell window partials (CD_SLOTS x C), a chunk's records (CD_SLOTS x chunk)
    const long long nn = n > 0 ? n : 1;
    // entries at a time; fewer where the records do not fit the memory left
    const long long most = c->cdep_chunk ? c->cdep_chunk : CDEP_CHUNK;
    long long chunk = nn < most ? nn : most;
    int rc;
    while ((rc = work_layout(c, nn, false, w, (size_t)CD_SLOTS * (C + chunk) * sizeof(double), &part_v, 2)) == FPIC_ENOMEM &&
           chunk > CDEP_CHUNK_MIN)
        c->cdep_chunk = chunk = chunk / 4 > CDEP_CHUNK_MIN ? chunk / 4 : CDEP_CHUNK_MIN;
    if (rc) return rc;
    double* part = (double*)part_v;
    double* rec = part + (size_t)CD_SLOTS * C;
    CDepK k{c->Nr, c->Nth, c->ld, c->G, c->bh, n, before->r, before->th, before->ur, before->uth, before->uph,
            before->alive, after->r, after->th, after->ur, after->uth, after->uph, after->qm, after->w,
            c->d_metric + (size_t)MT_N * c->metric_stride};
    // count and cursor follow one another
    FPIC_CUDA(cudaMemsetAsync(w.count, 0, (char*)(w.cursor + 2 * (size_t)C + 2) - (char*)w.count, s));
    FPIC_CUDA(cudaMemsetAsync(c->d_cnt + CNT_ERR, 0, sizeof(long long), s));
    const unsigned nb = (unsigned)((n + 255) / 256);
    if (n > 0) k_cdep_keys<<<nb, 256, 0, s>>>(k, w.key, w.count, (uint32_t)C, c->d_cnt + CNT_ERR);
    rc = scan_u32(w.count, w.off, w.bsum, 2 * C + 1, s);
    if (rc) return rc;
    if (n > 0) k_scatter<<<nb, 256, 0, s>>>(w.key, w.off, w.cursor, w.perm, n);
    k_bucket_rank<2><<<(unsigned)((C * 32 + 255) / 256), 256, 0, s>>>(w.off, w.perm, w.perm2, (uint32_t)C);
    for (long long a0 = 0; a0 < nn; a0 += chunk) {
        const long long m = nn - a0 < chunk ? nn - a0 : chunk;
        if (n > 0) k_cdep_particle<<<(unsigned)((m + 127) / 128), 128, 0, s>>>(k, w.off, w.perm2, rec, a0, m, (uint32_t)C);
        if (a0 == 0)
            k_cdep_cell<false><<<(unsigned)((C + CDEP_WARPS - 1) / CDEP_WARPS), 32 * CDEP_WARPS, 0, s>>>(
                rec, w.off, 0, (uint32_t)m, part, (uint32_t)C);
        else
            k_cdep_cell<true><<<(unsigned)((C + CDEP_CELLS - 1) / CDEP_CELLS), 32 * CDEP_WARPS, 0, s>>>(
                rec, w.off, (uint32_t)a0, (uint32_t)m, part, (uint32_t)C);
    }
    k_cdep_node<<<dim3((unsigned)((c->Nth + 1 + 255) / 256), c->Nr + 1), 256, 0, s>>>(k, tabs_of(c), part,
                                                                                     (uint32_t)C, dt, rho, jr,
                                                                                     jth, jph);
    FPIC_CUDA(cudaGetLastError());
    if (n_skipped) {
        long long v = 0;
        FPIC_CUDA(cudaMemcpyAsync(&v, c->d_cnt + CNT_ERR, sizeof(long long), cudaMemcpyDeviceToHost, s));
        FPIC_CUDA(cudaStreamSynchronize(s));
        *n_skipped = v;
    }
    return FPIC_OK;
}

namespace fpic {
// ---------------------------------------------------------------------------
// Divergence cleaning (Sec. 2.4, Eq. phi)
// ---------------------------------------------------------------------------
// (1/sqrtg) d_k (sqrtg gamma^kl d_l phi) = (1/sqrtg) d_j (sqrtg D^j) - 4 pi rho at
// the integer nodes i = 1 .. Nr-1, j = 0 .. Nth, multiplied by sqrtg at the
// node: the left side is the sum over the four faces of sqrtg gamma^kk d_k phi
// differences over the dual widths (the Yee divergence's own fluxes), the
// pole faces carry no flux, phi = 0 on the radial end rows.  Jacobi form
// phi <- sum_f c_f phi_f - b with c_f = face coefficient / sum of the face
// coefficients and b = right side / the same sum, both built once.
struct CleanK {
    int Nr, Nth, ld;
    GridDev G;
    Tabs T;                  // metric tables at the Yee points
    double2 *cr, *ct;        // per node (library scratch): (c_r1, c_r0), (c_t1, c_t0)
    double *nb;              // and -b
};

__global__ void k_clean_setup(CleanK k, const double* __restrict__ Dr, const double* __restrict__ Dt,
                              const double* __restrict__ rho)
{
    const int i = blockIdx.y + 1;                   // 1 .. Nr-1
    const GridDev& G = k.G;
    const Tabs& T = k.T;
    const double idr = G.irh[i - 1], ir1 = G.irn[i] * idr, ir0 = G.irn[i - 1] * idr;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j <= k.Nth; j += gridDim.x * blockDim.x) {
        const size_t o = (size_t)i * k.ld + j;
        const bool up = j < k.Nth, dn = j > 0;
        const double idth = up && dn ? G.ith[j - 1] : rcp_nr((up ? G.th[j] : M_PI) - (dn ? G.th[j - 1] : 0.0));
        const double sr1 = T.at(T_SG1, i, j), sr0 = T.at(T_SG1, i - 1, j);
        const double st1 = up ? T.at(T_SG2, i, j) : 0.0, st0 = dn ? T.at(T_SG2, i, j - 1) : 0.0;
        const double rhs = (sr1 * Dr[o] - sr0 * Dr[o - k.ld]) * idr +
                           ((up ? st1 * Dt[o] : 0.0) - (dn ? st0 * Dt[o - 1] : 0.0)) * idth -
                           4.0 * M_PI * T.at(T_SG0, i, j) * rho[o];
        const double cr1 = sr1 * T.at(T_URR1, i, j) * ir1;
        const double cr0 = sr0 * T.at(T_URR1, i - 1, j) * ir0;
        const double ct1 = up ? st1 * T.at(T_UTT2, i, j) * (G.itn[j] * idth) : 0.0;
        const double ct0 = dn ? st0 * T.at(T_UTT2, i, j - 1) * (G.itn[j - 1] * idth) : 0.0;
        const double inv = rcp_nr(cr1 + cr0 + ct1 + ct0);
        k.cr[o] = make_double2(cr1 * inv, cr0 * inv);
        k.ct[o] = make_double2(ct1 * inv, ct0 * inv);
        k.nb[o] = -rhs * inv;
    }
}

// One Jacobi sweep over the interior nodes (phi_in -> phi_out); the radial
// end rows stay zero in both buffers.  A warp takes two rows of 32 theta
// columns; neighbours come from L1 and L2.  Four fused multiply-adds a node
// (the sum starts from -b): FP64-pipe bound at best, 6.7 us a sweep on 1024 x
// 1024.  What stands in the way is latency: a sweep is a few microseconds of
// work between two launches.  Hence short blocks (3 to 16 rows a warp measured
// 5 to 30 % slower), the coefficients loaded before the wait for the previous
// sweep (programmatic dependent launch inside the graph of sweeps): a
// cleaning of 500 sweeps 6564 -> 4360 us on 1024 x 1024, 2195 -> 727 us on
// 64 x 64.
constexpr int JAC_WARPS = 4, JAC_ROWS = 2;          // warps of a block, rows of a warp
__global__ void __launch_bounds__(32 * JAC_WARPS, 7) k_jacobi(CleanK k, const double* phi_in, double* phi_out)
{
    const int j = min((int)(blockIdx.x * 32 + (threadIdx.x & 31)), k.Nth);       // idle lanes repeat the last column
    const int i = 1 + ((int)blockIdx.y * JAC_WARPS + (int)(threadIdx.x >> 5)) * JAC_ROWS;
    if (i >= k.Nr) return;
    const size_t ld = k.ld, o0 = (size_t)i * ld + j, o1 = i + 1 < k.Nr ? o0 + ld : o0;   // a last odd row twice
    const double2 cr0 = __ldg(k.cr + o0), ct0 = __ldg(k.ct + o0), cr1 = __ldg(k.cr + o1), ct1 = __ldg(k.ct + o1);
    const double nb0 = __ldg(k.nb + o0), nb1 = __ldg(k.nb + o1);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // neighbours beyond the poles: any finite value, their coefficients are zero
    const int jl = j > 0 ? 1 : 0, jr = j < k.Nth ? 1 : 0;
    const double dn0 = phi_in[o0 - ld], up0 = phi_in[o0 + ld], l0 = phi_in[o0 - jl], r0 = phi_in[o0 + jr];
    const double dn1 = phi_in[o1 - ld], up1 = phi_in[o1 + ld], l1 = phi_in[o1 - jl], r1 = phi_in[o1 + jr];
    double v0 = fma(cr0.y, dn0, nb0), v1 = fma(cr1.y, dn1, nb1);
    v0 = fma(cr0.x, up0, v0);
    v1 = fma(cr1.x, up1, v1);
    v0 = fma(ct0.x, r0, v0);
    v1 = fma(ct1.x, r1, v1);
    v0 = fma(ct0.y, l0, v0);
    v1 = fma(ct1.y, l1, v1);
    phi_out[o0] = v0;
    phi_out[o1] = v1;
}

// D^i -= gamma^ij d_j phi: D^r at (i+1/2, j), D^th at (i, j+1/2), D^ph at
// (i, j) with d_r phi the mean of the two adjacent half-point differences
// (one-sided on the end rows).
__global__ void k_clean_correct(CleanK k, const double* __restrict__ phi, double* Dr, double* Dt, double* Dp)
{
    const int i = blockIdx.y;                       // 0 .. Nr
    const GridDev& G = k.G;
    const Tabs& T = k.T;
    const double iu = i < k.Nr ? G.irn[i] : 0.0, id = i > 0 ? G.irn[i - 1] : 0.0;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j <= k.Nth; j += gridDim.x * blockDim.x) {
        const size_t o = (size_t)i * k.ld + j;
        const double up = i < k.Nr ? (phi[o + k.ld] - phi[o]) * iu : 0.0;
        const double dn = i > 0 ? (phi[o] - phi[o - k.ld]) * id : 0.0;
        const double mean = (i > 0 && i < k.Nr) ? 0.5 * (up + dn) : up + dn;
        if (i < k.Nr) Dr[o] -= T.at(T_URR1, i, j) * up;
        if (j < k.Nth) Dt[o] -= T.at(T_UTT2, i, j) * ((phi[o + 1] - phi[o]) * G.itn[j]);
        Dp[o] -= T.at(T_URP0, i, j) * mean;
    }
}

}  // namespace fpic

namespace fpic {
// ---------------------------------------------------------------------------
// Pair injection (Sec. 3.3, 3.4)
// ---------------------------------------------------------------------------
// Every cell whose centre radius lies in [r_lo, r_hi] gets an e-/e+ pair
// when e n < mult e n_GJ: e n = sum of w |q/m| over the cell's alive
// particles (taken in particle-index order from the stable bucket order, so
// the sum is the same on every run) over the cell's proper volume V,
// e n_GJ = |Omega_h B^z| / 4 pi with B^z = B^r cos th - r sin th B^th at the
// centre.  The pair sits at one point of the cell, each particle with the
// weight that makes the pair's density n0 n_GJ; pairs are appended in cell
// order, e- then e+, while they fit.
struct InjK {
    int Nr, Nth, ld;
    GridDev G;
    BH bh;
    double Om, r_lo, r_hi, mult, n0, qm_e, B0pot;
    const double *Br, *Bth, *draws;
    const double *w, *qm;                    // existing particles
    const uint32_t *off, *perm;              // cell buckets, particle-index order
    uint32_t* flag;                          // per cell 0 / 1
    uint8_t* flags8;                         // optional copy for the caller
    double* wpair;                           // per cell: weight of each new particle
};

__global__ void k_inject_flag(InjK k)
{
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= (long long)k.Nr * k.Nth) return;
    const int i = (int)(c / k.Nth), j = (int)(c - (long long)i * k.Nth);
    uint32_t inj = 0;
    double wp = 0.0;
    const double rc = k.G.rh[i];
    if (rc >= k.r_lo && rc <= k.r_hi) {
        double S = 0.0;
        for (uint32_t q = k.off[c]; q < k.off[c + 1]; ++q) {
            const uint32_t p = k.perm[q];
            S = __dadd_rn(S, __dmul_rn(k.w[p], fabs(k.qm[p])));   // product rounded, then added
        }
        const double V = 2.0 * M_PI * trap16_dev(k.bh, k.G.rn[i], k.G.rn[i + 1], k.G.tn[j], k.G.tn[j + 1]);
        const size_t o = (size_t)i * k.ld + j;
        const double br = 0.5 * (k.Br[o] + k.Br[o + k.ld]);
        const double bt = 0.5 * (k.Bth[o] + k.Bth[o + 1]);
        double sn, cs;
        sincos(k.G.th[j], &sn, &cs);
        const double Bz = br * cs - rc * sn * bt;
        const double gj = fabs(k.Om * Bz) / (4.0 * M_PI);
        inj = S / V < k.mult * gj ? 1u : 0u;
        wp = k.n0 * gj * V / (2.0 * k.qm_e);
    }
    k.flag[c] = inj;
    if (k.flags8) k.flags8[c] = (uint8_t)inj;
    k.wpair[c] = wp;
}

__global__ void k_inject_write(InjK k, fpic_particles P, const uint32_t* __restrict__ pos, long long cap)
{
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= (long long)k.Nr * k.Nth || !k.flag[c]) return;
    const long long m = P.n + 2LL * pos[c];
    if (m + 2 > cap) return;
    const int i = (int)(c / k.Nth), j = (int)(c - (long long)i * k.Nth);
    const double* d = k.draws + 9 * c;
    const double r = k.G.rn[i] + d[0] * (k.G.rn[i + 1] - k.G.rn[i]);
    const double t = k.G.tn[j] + d[1] * (k.G.tn[j + 1] - k.G.tn[j]);
    const double ph = 2.0 * M_PI * d[2];
    double sn, cs;
    sincos(t, &sn, &cs);
    Geo g;
    geo_eval(k.bh, r, sn, cs, g);
    const double L11 = sqrt(g.grr), L31 = g.grp / L11, L22 = sqrt(g.gtt);
    const double L33 = sqrt(fma(-L31, L31, g.gpp));
    const double wp = k.wpair[c];
    for (int s = 0; s < 2; ++s) {
        const double* u = d + 3 + 3 * s;
        const double z[6] = {r, t, ph, L11 * u[0], L22 * u[1], fma(L31, u[0], L33 * u[2])};
        const long long q = m + s;
        const double qm = s == 0 ? -k.qm_e : k.qm_e;
        P.r[q] = z[0]; P.th[q] = z[1]; P.ph[q] = z[2];
        P.ur[q] = z[3]; P.uth[q] = z[4]; P.uph[q] = z[5];
        P.qm[q] = qm;
        P.w[q] = wp;
        P.alive[q] = 1;
        P.scheme[q] = 0;
        P.iters[q] = 0;
        if (P.cell) P.cell[q] = (uint32_t)c;
        double kin, pot;
        h_parts(k.bh, z, qm, k.B0pot, kin, pot);
        P.H0[q] = kin - pot;
        P.Hn[q] = kin - pot;
        P.D0[q] = fabs(kin) + fabs(pot);
    }
}
}  // namespace fpic

extern "C" int fpic_inject_pairs(fpic_ctx* c, fpic_particles* p, long long capacity, const double* Br,
                                 const double* Bth, const fpic_inject_params* prm, const double* draws,
                                 unsigned char* flags, long long* wanted, long long* n_new, void* stream)
{
    if (c && c->G.full) return set_error(FPIC_EINVAL, "fpic_inject_pairs: not built for the full-theta domain");
    if (!c || !p || !Br || !Bth || !prm || !draws || !n_new)
        return set_error(FPIC_EINVAL, "fpic_inject_pairs: NULL argument");
    if (!c->has_grid) return set_error(FPIC_EINVAL, "fpic_inject_pairs: no grid set");
    if (p->n < 0 || capacity < p->n) return set_error(FPIC_EINVAL, "fpic_inject_pairs: need 0 <= n <= capacity");
    if (!particles_ok(p, true) || !p->w) return set_error(FPIC_EINVAL, "fpic_inject_pairs: NULL particle array");
    if (!(prm->qm_e > 0.0) || !(prm->n0 > 0.0) || !(prm->multiplicity >= 0.0) || !(prm->r_lo <= prm->r_hi))
        return set_error(FPIC_EINVAL, "fpic_inject_pairs: need qm_e > 0, n0 > 0, multiplicity >= 0, r_lo <= r_hi");
    const long long n = p->n;
    const long long C = (long long)c->Nr * c->Nth;
    if (n + 2 * C > 0xffffffffLL) return set_error(FPIC_EINVAL, "fpic_inject_pairs: more than 2^32 particles");
    FPIC_CUDA(cudaSetDevice(c->device));
    cudaStream_t s = (cudaStream_t)stream;
    Work w;
    int rc = work_layout(c, n > C + 2 ? n : C + 2, false, w);
    if (rc) return rc;
    FPIC_CUDA(cudaMemsetAsync(w.count, 0, 4 * ((size_t)C + 2), s));
    FPIC_CUDA(cudaMemsetAsync(w.cursor, 0, 4 * ((size_t)C + 2), s));
    const unsigned nb = (unsigned)((n + 255) / 256);
    if (n > 0) k_keys<<<nb, 256, 0, s>>>(c->G, p->r, p->th, p->alive, w.key, nullptr, w.count, n, (uint32_t)C);
    rc = scan_u32(w.count, w.off, w.bsum, C + 1, s);
    if (rc) return rc;
    if (n > 0) k_scatter<<<nb, 256, 0, s>>>(w.key, w.off, w.cursor, w.perm, n);
    k_bucket_rank<1><<<(unsigned)((C * 32 + 255) / 256), 256, 0, s>>>(w.off, w.perm, w.perm2, (uint32_t)C);
    const double r_h = c->r_h;
    InjK k{c->Nr, c->Nth, c->ld, c->G, c->bh, c->a / (2.0 * c->M * r_h), prm->r_lo, prm->r_hi, prm->multiplicity,
           prm->n0, prm->qm_e, prm->B0pot, Br, Bth, draws, p->w, p->qm, w.off, w.perm2, w.flag, flags, w.tmp};
    const unsigned cb = (unsigned)((C + 255) / 256);
    k_inject_flag<<<cb, 256, 0, s>>>(k);
    rc = scan_u32(w.flag, w.pos, w.bsum, C, s);
    if (rc) return rc;
    k_inject_write<<<cb, 256, 0, s>>>(k, *p, w.pos, capacity);
    FPIC_CUDA(cudaGetLastError());
    uint32_t K = 0;
    FPIC_CUDA(cudaMemcpyAsync(&K, w.pos + C, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    FPIC_CUDA(cudaStreamSynchronize(s));
    const long long room = (capacity - n) / 2;
    if (wanted) *wanted = (long long)K;
    *n_new = n + 2 * ((long long)K < room ? (long long)K : room);
    return FPIC_OK;
}

namespace fpic {
// Eq. (Pbz) on the sphere r = rh[i]: P = (1/2) sum_j (E_th H_ph - E_ph H_th)
// dth_j with each product at the cell centre (rh[i], th_{j+1/2}) from its
// staggered neighbours (E_th averaged in r, H_th in th, E_ph over the four
// nodes).  One block; each thread sums a fixed stride of cells and the block
// sums in a fixed tree, so the result is bitwise reproducible.
__global__ void __launch_bounds__(256) k_bz_power(int Nth, int ld, const double* __restrict__ tn, const double* Eth,
                                                  const double* Eph, const double* Hth, const double* Hph, int i,
                                                  double* out)
{
    __shared__ double part[256];
    double acc = 0.0;
    for (int j = threadIdx.x; j < Nth; j += 256) {
        const size_t o = (size_t)i * ld + j, o1 = o + ld;
        const double et = 0.5 * (Eth[o] + Eth[o1]);
        const double ep = 0.25 * ((Eph[o] + Eph[o + 1]) + (Eph[o1] + Eph[o1 + 1]));
        const double ht = 0.5 * (Hth[o] + Hth[o + 1]);
        acc = fma(fma(et, Hph[o], -ep * ht), tn[j + 1] - tn[j], acc);
    }
    part[threadIdx.x] = acc;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = 0.5 * part[0];
}
}  // namespace fpic

extern "C" int fpic_bz_power(fpic_ctx* c, const fpic_fields* f, int i, double* out, void* stream)
{
    if (c && c->G.full) return set_error(FPIC_EINVAL, "fpic_bz_power: not built for the full-theta domain");
    if (!c || !f || !out) return set_error(FPIC_EINVAL, "fpic_bz_power: NULL argument");
    if (!c->has_grid) return set_error(FPIC_EINVAL, "fpic_bz_power: no grid set");
    if (i < 0 || i >= c->Nr) return set_error(FPIC_EINVAL, "fpic_bz_power: half-r index %d outside [0, %d)", i, c->Nr);
    if (!f->E[1] || !f->E[2] || !f->H[1] || !f->H[2]) return set_error(FPIC_EINVAL, "fpic_bz_power: NULL E or H array");
    FPIC_CUDA(cudaSetDevice(c->device));
    k_bz_power<<<1, 256, 0, (cudaStream_t)stream>>>(c->Nth, c->ld, c->G.tn, f->E[1], f->E[2], f->H[1], f->H[2], i,
                                                    out);
    FPIC_CUDA(cudaGetLastError());
    return FPIC_OK;
}

extern "C" int fpic_div_clean(fpic_ctx* c, double* const D[3], const double* rho, int n_iter, double* phi,
                              void* stream)
{
    if (c && c->G.full) return set_error(FPIC_EINVAL, "fpic_div_clean: not built for the full-theta domain");
    if (!c || !D || !D[0] || !D[1] || !D[2] || !rho) return set_error(FPIC_EINVAL, "fpic_div_clean: NULL argument");
    if (!c->has_grid) return set_error(FPIC_EINVAL, "fpic_div_clean: no grid set");
    if (n_iter < 0) return set_error(FPIC_EINVAL, "fpic_div_clean: n_iter < 0");
    FPIC_CUDA(cudaSetDevice(c->device));
    cudaStream_t s = (cudaStream_t)stream;
    const size_t sz = (size_t)(c->Nr + 1) * c->ld;
    // scratch: 5 coefficient arrays and two phi buffers
    int rc = ensure_scratch2(c, 7 * sz * sizeof(double) + 256);
    if (rc) return rc;
    double* base = (double*)c->d_scratch2;
    CleanK k{c->Nr, c->Nth, c->ld, c->G, tabs_of(c), (double2*)base, (double2*)base + sz, base + 4 * sz};
    double* pa = base + 5 * sz;
    double* pb = base + 6 * sz;
    FPIC_CUDA(cudaMemsetAsync(pa, 0, 2 * sz * sizeof(double), s));
    if (c->Nr >= 2) {
        const unsigned gx = (unsigned)((c->Nth + 1 + 255) / 256);
        k_clean_setup<<<dim3(gx, c->Nr - 1), 256, 0, s>>>(k, D[0], D[1], rho);
        const dim3 jg((unsigned)((c->Nth + 32) / 32),
                      (unsigned)((c->Nr - 1 + JAC_WARPS * JAC_ROWS - 1) / (JAC_WARPS * JAC_ROWS)));
        auto sweeps = [&](cudaStream_t st, bool chained) -> int {
            double *x = base + 5 * sz, *y = base + 6 * sz;
            cudaLaunchAttribute at{};
            at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
            at.val.programmaticStreamSerializationAllowed = 1;
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = jg;
            cfg.blockDim = dim3(32 * JAC_WARPS);
            cfg.stream = st;
            cfg.attrs = &at;
            for (int it = 0; it < n_iter; ++it) {
                cfg.numAttrs = chained && it > 0 ? 1 : 0;    // a sweep after a sweep of the same graph
                FPIC_CUDA(cudaLaunchKernelEx(&cfg, k_jacobi, k, (const double*)x, y));
                double* t = x;
                x = y;
                y = t;
            }
            return 0;
        };
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        FPIC_CUDA(cudaStreamIsCapturing(s, &cap));
        if (n_iter < 8 || cap != cudaStreamCaptureStatusNone) {
            rc = sweeps(s, false);  // short chains, or the caller is recording a graph itself
            if (rc) return rc;
        } else {
            // hundreds of short launches: replay them as one graph
            if (!c->clean_exec || c->clean_key_base != base || c->clean_key_Nr != c->Nr ||
                c->clean_key_Nth != c->Nth || c->clean_key_iter != n_iter) {
                if (c->clean_exec) FPIC_CUDA(cudaGraphExecDestroy(c->clean_exec));
                c->clean_exec = nullptr;
                int rc2 = ensure_copy_stream(c);
                if (rc2) return rc2;
                cudaGraph_t g = nullptr;
                FPIC_CUDA(cudaStreamBeginCapture(c->copy_stream, cudaStreamCaptureModeThreadLocal));
                rc = sweeps(c->copy_stream, true);
                const cudaError_t ec = cudaStreamEndCapture(c->copy_stream, &g);
                if (rc) {
                    if (g) cudaGraphDestroy(g);
                    return rc;
                }
                FPIC_CUDA(ec);
                cudaError_t e = cudaGraphInstantiate(&c->clean_exec, g, 0);
                cudaGraphDestroy(g);
                FPIC_CUDA(e);
                c->clean_key_base = base;
                c->clean_key_Nr = c->Nr;
                c->clean_key_Nth = c->Nth;
                c->clean_key_iter = n_iter;
            }
            FPIC_CUDA(cudaGraphLaunch(c->clean_exec, s));
        }
        if (n_iter & 1) {
            double* t = pa;
            pa = pb;
            pb = t;
        }
    }
    k_clean_correct<<<dim3((unsigned)((c->Nth + 1 + 255) / 256), c->Nr + 1), 256, 0, s>>>(k, pa, D[0], D[1], D[2]);
    if (phi) FPIC_CUDA(cudaMemcpyAsync(phi, pa, sz * sizeof(double), cudaMemcpyDeviceToDevice, s));
    FPIC_CUDA(cudaGetLastError());
    return FPIC_OK;
}

extern "C" int fpic_fdtd_step(fpic_ctx* c, fpic_fields* f, const fpic_fdtd_params* prm, int stage, void* stream)
{
    if (!c || !f || !prm) return set_error(FPIC_EINVAL, "fpic_fdtd_step: NULL argument");
    if (!c->has_grid) return set_error(FPIC_EINVAL, "fpic_fdtd_step: no grid set");
    if (stage != 1 && stage != 2) return set_error(FPIC_EINVAL, "fpic_fdtd_step: stage must be 1 or 2");
    if (!std::isfinite(prm->dt) || !std::isfinite(prm->chi0) || prm->chi0 < 0.0 ||
        (prm->chi0 > 0.0 && !(prm->r_max > prm->r_abs)))
        return set_error(FPIC_EINVAL, "fpic_fdtd_step: bad dt or absorbing-layer parameters");
    for (int k = 0; k < 3; ++k) {
        const void* need[] = {f->B0[k], f->B1[k], f->D0[k], f->D1[k], f->j0[k], f->j1[k], f->E[k], f->H[k],
                              f->Bh[k], f->Dw[k]};
        for (const void* q : need)
            if (!q) return set_error(FPIC_EINVAL, "fpic_fdtd_step: NULL field array");
    }
    if (!f->rho0 || !f->rho1) return set_error(FPIC_EINVAL, "fpic_fdtd_step: NULL rho array");
    FPIC_CUDA(cudaSetDevice(c->device));
    cudaStream_t s = (cudaStream_t)stream;
    // rows a warp walks: the first row's auxiliary field is worked out twice,
    // so as many as keep 16 warps on every SM, 16 at most
    const long long cols = (c->Nth + FD_COLS) / FD_COLS;
    int rows = 16;
    while (rows > 1 && cols * ((c->Nr + rows) / rows) < 16LL * c->sm_count) rows >>= 1;
    const FK k{rows, c->G, tabs_of(c), prm->dt, prm->chi0, prm->lambda, prm->r_abs, prm->r_max, prm->conserving};
    const dim3 grid((unsigned)((cols + FD_THREADS / 32 - 1) / (FD_THREADS / 32)), (unsigned)((c->Nr + rows) / rows));
    auto c3 = [](double* const a[3]) { return C3{{a[0], a[1], a[2]}}; };
    auto p3 = [](double* const a[3]) { return P3{{a[0], a[1], a[2]}}; };
    if (stage == 1) {
        // [1] E^{n+1} = alpha <D>^{n+1} + beta x B^{n+1}, [2] B^{n+3/2} = <B>^{n+1/2} - dt curl E^{n+1}
        k_step_B<true><<<grid, FD_THREADS, 0, s>>>(k, c3(f->D0), c3(f->D1), c3(f->B0), c3(f->B1), c3(f->B1),
                                                   p3(f->E), p3(f->Bh));
        // [3] E^{n+3/2}, [4] B^{n+2} = B^{n+1} - dt curl E^{n+3/2}  (into B0)
        k_step_B<false><<<grid, FD_THREADS, 0, s>>>(k, c3(f->D0), c3(f->D1), c3(f->B0), c3(f->B1), c3(f->Bh),
                                                    p3(f->E), p3(f->B0));
    } else {
        const Src S0{{f->j0[0], f->j0[1], f->j0[2]}, f->rho0}, S1{{f->j1[0], f->j1[1], f->j1[2]}, f->rho1};
        // [7] H^{n+3/2} = alpha B^{n+3/2} - beta x D^{n+3/2}, [8] D^{n+2} = <D>^{n+1} + dt [curl H - 4 pi <J>^{n+3/2}]
        k_step_D<true><<<grid, FD_THREADS, 0, s>>>(k, c3(f->D0), c3(f->D1), c3(f->D1), c3(f->Bh), S0, S1, p3(f->H),
                                                   p3(f->Dw));
        // [9] H^{n+2} = alpha B^{n+2} - beta x D^{n+2}, [10] D^{n+5/2} = D^{n+3/2} + dt [curl H - 4 pi J^{n+2}]  (into D0)
        k_step_D<false><<<grid, FD_THREADS, 0, s>>>(k, c3(f->D0), c3(f->D1), c3(f->Dw), c3(f->B0), S0, S1, p3(f->H),
                                                    p3(f->D0));
    }
    FPIC_CUDA(cudaGetLastError());
    return FPIC_OK;
}
