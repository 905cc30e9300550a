// recur_cluster.cu -- the BDCD s-step recurrence (eq. bdcd-sstep, Algorithm 4)
// on one thread-block cluster, in super-blocks of up to 32 rows.
//
// The inner system is L Delta = -g_S with L the block lower triangle of G
// (G_jt = Kss_jt / lambda + m [S_j = S_t]).  It is solved in FP32 and refined
// once: Delta0 from an FP32 block forward substitution, the residual
// rho = -g_S - L Delta0 with every product split exactly (TwoProd) and summed
// in double-single arithmetic (~2^-44 relative), Delta1 from a second FP32
// substitution on rho, Delta = Delta0 + Delta1.  That is FP64-accurate for the
// well-conditioned blocks of K-RR while avoiding GB300's slow FP64 pipe.
//
// Consecutive blocks are grouped into super-blocks of q = 32 / b blocks
// (Bs = q b <= 32 rows, one row per lane).  bdcd_prep_kernel inverts the
// diagonal part L_JJ of every super-block at once (Gauss-Jordan with one
// thread per entry; L_JJ is block lower triangular with SPD diagonal blocks,
// so no pivoting; one CTA per super-block) while a second set of CTAs marks
// repeated indices and links their occurrences, so a chain step is
// Delta_J = L_JJ^-1 r_J after r_J -= L_JT Delta_T for every earlier T: the
// block forward substitution with the steps inside a super-block regrouped
// into one matrix-vector product.
//
// The sb^2/2 Gram entries do not fit one SM's shared memory and one SM reads
// L2 at only ~40-60 B/clock, so the super-blocks are dealt to the P CTAs of a
// cluster, two per CTA, folded (CTA c owns J = c and 2P-1-c, which balances
// the triangle); each CTA copies its rows' Gram panels (Bs x Bs, row-major)
// once by 2-D TMA.  Per own super-block a CTA runs three warps:
//   round-0 warp: applies Delta0_T as it arrives (T < J), forms Delta0_J
//                 and sends it to every CTA, completing the receiver's
//                 per-step mbarrier;
//   residual warp: accumulates the double-single residual of the rows
//                 panel by panel as the Delta0_T arrive, Delta0_J last,
//                 which gives rho_J;
//   round-1 warp: applies Delta1_T as it arrives and once rho_J is ready
//                 forms Delta1_J, sends it and writes Delta = Delta0 + Delta1.
// The refinement chain thus runs a little behind the first one instead of
// after it.
//
// What bounds it is the latency of one step of the chain: Delta_{J-1} arrives,
// one 32 x 32 product, Delta_J leaves.  So the panel rows (and those of
// L_JJ^-1 and L_JJ^-1 L_{J,J-1}) are in registers before the wait, the
// residual is no work of the chain's warps, and a send goes to the two CTAs
// that need it next as 16-byte remote stores and to the others as one bulk
// copy each.  With 128 remote stores a send (1.8-3 k cycles to issue, in rank
// order), the residual in the chain's warp (8-14 k cycles between Delta0_J and
// rho_J) and the panels, inverses and masks copied through registers before
// the start (17 k cycles) 1024 coordinates took 43 us; now 22.  Panel rows are
// read as float4 chunks in a lane-rotated order (conflict-free).  Every wait is
// bounded; on expiry the kernel records DEV_TIMEOUT, skips its remaining waits
// and still lets every store addressed to it land (bounded) before it leaves.
#include "dcd_internal.cuh"
#include "ptx.cuh"

#include <map>
#include <mutex>

namespace dcd {
namespace {

// warps (slot = warp & 1): 0-1 round 0, 2-3 round 1, 6-7 residual (on the schedulers of round 1, which
// waits for it); 4-5 only help with the set-up
constexpr int CL_THREADS = 256;
constexpr int CL_SLOTS = 2;      // own super-blocks per CTA
constexpr int CL_PMAX = 16;      // CTAs per cluster (non-portable size)
constexpr int CL_NSUP_MAX = 2 * CL_PMAX;
constexpr size_t CL_SMEM_MAX = 224 * 1024;
constexpr unsigned long long CL_WAIT_NS = 2000000000ull;
constexpr int NLOCAL = 3 * CL_SLOTS;  // per slot: diagonal panel, other panels, rho ready
constexpr int PREP_THREADS = 256;

struct ClGeom {
    int q, Bs, nsup;
};

__host__ __device__ inline ClGeom cl_geom(int nblk, int b)
{
    ClGeom G;
    G.q = b >= 32 ? 1 : 32 / b;
    G.Bs = G.q * b;
    G.nsup = (nblk + G.q - 1) / G.q;
    return G;
}

// super-block of own slot k of CTA c (folded over 2P)
__host__ __device__ inline int cl_own(int k, int c, int P) { return k == 0 ? c : 2 * P - 1 - c; }

// rows of super-block J
__host__ __device__ inline int cl_rows(int J, int Bs, int sb)
{
    const int r = sb - J * Bs;
    return r < Bs ? r : Bs;
}

struct ClLayout {
    size_t recv, xs, ns, dmask, dsend, rbuf, rho, bars, gdata, ps, total;
    int nown;
};

__host__ __device__ inline size_t al16(size_t v) { return (v + 15) & ~(size_t)15; }

// Layout of CTA c.  Everything other CTAs address (recv, bars) sits at the
// same offset in every CTA; the per-CTA Gram panels are last, from the first
// 128-byte boundary at or after gdata (TMA destinations).  Own slot k keeps
// its J+1 panels (T = 0..J) in order.
__host__ __device__ inline ClLayout cl_layout(int nblk, int b, int P, int c)
{
    const ClGeom G = cl_geom(nblk, b);
    const size_t sb = (size_t)nblk * b;
    ClLayout L;
    size_t cur = 0;
    L.recv = cur;
    cur = al16(cur + 2 * sb * 4);
    L.xs = cur;
    cur = al16(cur + (size_t)CL_SLOTS * 32 * 32 * 4);
    L.ns = cur;
    cur = al16(cur + (size_t)CL_SLOTS * 32 * 32 * 4);
    L.dmask = cur;
    cur = al16(cur + (size_t)CL_SLOTS * CL_NSUP_MAX * 32 * 4);
    L.dsend = cur;
    cur = al16(cur + (size_t)2 * CL_SLOTS * 32 * 4);
    L.rbuf = cur;
    cur = al16(cur + (size_t)2 * CL_SLOTS * 32 * 4);
    L.rho = cur;
    cur = al16(cur + (size_t)CL_SLOTS * 32 * 8);
    L.bars = cur;
    cur = al16(cur + ((size_t)2 * G.nsup + NLOCAL) * 8);
    L.gdata = cur;
    L.ps = ((size_t)G.Bs * G.Bs * 4 + 127) & ~(size_t)127;
    size_t panels = 0;
    L.nown = 0;
    for (int k = 0; k < CL_SLOTS; ++k) {
        const int J = cl_own(k, c, P);
        if (J >= G.nsup || (k == 1 && J == cl_own(0, c, P))) break;
        panels += (size_t)J + 1;
        L.nown = k + 1;
    }
    L.total = L.gdata + 128 + panels * L.ps;
    return L;
}

// double-single accumulation of an exact product (p, e) into (hi, lo)
__device__ __forceinline__ void ds_add(float &hi, float &lo, float p, float e)
{
    const float s = hi + p;
    const float bp = s - hi;
    const float err = (hi - (s - bp)) + (p - bp);
    hi = s;
    lo += err + e;
}

__device__ __forceinline__ void ds_prod(float &hi, float &lo, float kv, float dv)
{
    const float pp = kv * dv;
    ds_add(hi, lo, pp, fmaf(kv, dv, -pp));
}

// Row `lane` of a panel of BS columns (20, 24, 28 or 32) in registers, as float4 chunks from chunk
// `lane` onwards (mod BS / 4), so the lanes of a quarter-warp read distinct banks, of the row and of
// the vector alike.
template <int BS> struct PanelRow {
    static constexpr int NC = BS / 4;
    float4 a[NC];
    __device__ __forceinline__ static int chunk(int lane, int j)
    {
        const int m = lane % NC + j;
        return m >= NC ? m - NC : m;
    }
    __device__ __forceinline__ void load(const float *pr, int lane)
    {
#pragma unroll
        for (int j = 0; j < NC; ++j) a[j] = *(const float4 *)(pr + 4 * chunk(lane, j));
    }
    // FUSED: by FMAs; else every product rounded by itself, the sums that panel_dot_ds has in its high parts
    template <bool FUSED> __device__ __forceinline__ float dot(const float *v, int lane) const
    {
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            const float4 x = *(const float4 *)(v + 4 * chunk(lane, j));
            s0 = FUSED ? fmaf(a[j].x, x.x, s0) : __fadd_rn(s0, __fmul_rn(a[j].x, x.x));
            s1 = FUSED ? fmaf(a[j].y, x.y, s1) : __fadd_rn(s1, __fmul_rn(a[j].y, x.y));
            s2 = FUSED ? fmaf(a[j].z, x.z, s2) : __fadd_rn(s2, __fmul_rn(a[j].z, x.z));
            s3 = FUSED ? fmaf(a[j].w, x.w, s3) : __fadd_rn(s3, __fmul_rn(a[j].w, x.w));
        }
        return (s0 + s1) + (s2 + s3);
    }
};

// The same dot product over the row's first ncol columns (a multiple of 4) as a double-single pair,
// each product exact (TwoProd).
__device__ __forceinline__ void panel_dot_ds(const float *pr, const float *v, int lane, int ncol, float &hi, float &lo)
{
    const int nc = ncol >> 2;
    const int m0 = nc == 8 ? (lane & 7) : lane % nc;
    float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f, h2 = 0.f, l2 = 0.f, h3 = 0.f, l3 = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (j < nc) {
            int m = m0 + j;
            m -= m >= nc ? nc : 0;
            const float4 a = *(const float4 *)(pr + 4 * m), x = *(const float4 *)(v + 4 * m);
            ds_prod(h0, l0, a.x, x.x);
            ds_prod(h1, l1, a.y, x.y);
            ds_prod(h2, l2, a.z, x.z);
            ds_prod(h3, l3, a.w, x.w);
        }
    }
    ds_add(h0, l0, h1, l1);
    ds_add(h2, l2, h3, l3);
    ds_add(h0, l0, h2, l2);
    hi = h0;
    lo = l0;
}

// sum of v over the set bits of mask
__device__ __forceinline__ float mask_sum(uint32_t mask, const float *v)
{
    float s = 0.f;
    while (mask) {
        s += v[__ffs(mask) - 1];
        mask &= mask - 1;
    }
    return s;
}

// Warp-uniform.  REMOTE: bytes from other CTAs complete the barrier.
template <bool REMOTE>
__device__ __forceinline__ bool wait_bar(uint64_t *bar, volatile int *abort_flag, int *err)
{
    bool ok = REMOTE ? ptx::mbar_test_cluster(bar, 0) : ptx::mbar_test(bar, 0);
    if (__all_sync(0xffffffffu, ok)) return true;
    ok = !*abort_flag && (REMOTE ? ptx::mbar_wait_cluster_bounded(bar, 0, CL_WAIT_NS)
                                 : ptx::mbar_wait_bounded(bar, 0, CL_WAIT_NS));
    if (!__all_sync(0xffffffffu, ok)) {
        if ((threadIdx.x & 31) == 0 && !*abort_flag) {
            *abort_flag = 1;
            set_error(err, DEV_TIMEOUT);
        }
        return false;
    }
    return true;
}

// ---------------------------------------------------------------------------
// Per super-block J (one CTA of 8 warps; lane j, rows i0 + 8 r):
//   M[J][T][p]: bit q set when position T*Bs + q precedes row J*Bs + p and
//          holds the same index (T <= J): the repeats that the m I term of
//          G couples across overlapping blocks;
//   X[J] = L_JJ^-1 (32 x 32 row-major, FP32; rows and columns past the
//          super-block's rows hold the identity), by Gauss-Jordan on
//          [L_JJ | I] (a thread owns columns j and j+32 of its rows; the
//          matrix is double-buffered so a pivot step needs one barrier); a
//          pivot that is not positive and finite records DEV_NOT_SPD;
//   N[J] = X_J L_{J,J-1} (J >= 1) with L_{J,J-1} = K_{J,J-1} / lambda + m D,
//          D the repeat pattern between J and J-1: the whole coupling of
//          super-block J to its predecessor in one matrix, so that a chain
//          step is Delta_J = X_J r'_J - N_J Delta_{J-1}.
__global__ void __launch_bounds__(PREP_THREADS)
    bdcd_prep_kernel(const float *Kss, int64_t ldk, const int32_t *S, int nblk, int b, float inv_lam, float mf,
                     float *X, float *N, uint32_t *M, int32_t *next, int *err)
{
    constexpr int RPT = 32 / (PREP_THREADS / 32);  // rows per thread
    __shared__ float a[2][32][65];
    __shared__ int sIJ[32], sIT[CL_NSUP_MAX * 32];
    __shared__ int bad, nxt[32];
    const ClGeom G = cl_geom(nblk, b);
    const int Bs = G.Bs, sb = nblk * b;
    const bool links = (int)blockIdx.x >= G.nsup;  // the second half of the grid: masks and links
    const int J = links ? (int)blockIdx.x - G.nsup : (int)blockIdx.x;
    const int base = J * Bs, rows = cl_rows(J, Bs, sb);
    const int i0 = threadIdx.x >> 5, j = threadIdx.x & 31;  // rows i0 + 8 r
    if (threadIdx.x == 0) bad = 0;
    if (threadIdx.x < 32) nxt[threadIdx.x] = INT32_MAX;
    for (int e = threadIdx.x; e < sb; e += PREP_THREADS) sIT[e] = S[e];
    __syncthreads();
    if (links) {
        // next[row]: the next position holding the same index (-1: none); warp i0 scans the
        // positions row + 1 + i0, row + 9 + i0, ... up to its first match, the minimum wins
        if (j < rows) {
            const int row = base + j, key = sIT[row];
            for (int q = row + 1 + i0; q < sb; q += PREP_THREADS / 32)
                if (sIT[q] == key) {
                    atomicMin(&nxt[j], q);
                    break;
                }
        }
        // repeat masks: (T, p = j) for T = i0 + 8 r <= J
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            const int T = i0 + 8 * r;
            if (T <= J) {
                const int key = j < rows ? sIT[base + j] : -1, row = base + j, tb = T * Bs, tr = cl_rows(T, Bs, sb);
                uint32_t mask = 0;
                for (int q = 0; q < tr; ++q)
                    if (sIT[tb + q] == key && tb + q < row) mask |= 1u << q;
                M[((size_t)J * CL_NSUP_MAX + T) * 32 + j] = mask;
            }
        }
        __syncthreads();
        if (threadIdx.x < rows) next[base + threadIdx.x] = nxt[threadIdx.x] == INT32_MAX ? -1 : nxt[threadIdx.x];
        return;
    }
    if (threadIdx.x < 32) sIJ[threadIdx.x] = threadIdx.x < rows ? sIT[base + threadIdx.x] : -1;
    // [L_JJ | I]
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        const int i = i0 + 8 * r;
        float v = (i == j) ? 1.f : 0.f;
        if (i < rows && j < rows) {
            v = 0.f;
            if (j / b <= i / b)
                v = Kss[(int64_t)(base + i) * ldk + base + j] * inv_lam + (sIT[base + i] == sIT[base + j] ? mf : 0.f);
        }
        a[0][i][j] = v;
        a[0][i][j + 32] = (i == j) ? 1.f : 0.f;
    }
    __syncthreads();
    int cur = 0;
    for (int k = 0; k < 32; ++k) {
        const float piv = a[cur][k][k];
        if (!(piv > 0.f) || !(piv < INFINITY)) {  // the same value in every thread
            if (threadIdx.x == 0) bad = 1;
            break;
        }
        const float ip = __frcp_rn(piv);  // = 1.f / piv (both correctly rounded)
        const float p0 = a[cur][k][j] * ip, p1 = a[cur][k][j + 32] * ip;
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            const int i = i0 + 8 * r;
            const float f = a[cur][i][k];
            a[cur ^ 1][i][j] = (i == k) ? p0 : fmaf(-f, p0, a[cur][i][j]);
            a[cur ^ 1][i][j + 32] = (i == k) ? p1 : fmaf(-f, p1, a[cur][i][j + 32]);
        }
        cur ^= 1;
        __syncthreads();
    }
    __syncthreads();
    if (bad) {
        if (threadIdx.x == 0) set_error(err, DEV_NOT_SPD);
        return;
    }
#pragma unroll
    for (int r = 0; r < RPT; ++r) X[(size_t)J * 1024 + (i0 + 8 * r) * 32 + j] = a[cur][i0 + 8 * r][j + 32];
    if (J == 0) return;
    // N_J = X_J (K_{J,J-1} / lambda + m D): B[t][c] in the other buffer, then row i of X times column j of B
    const int pb = (J - 1) * Bs;
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        const int t = i0 + 8 * r;
        float v = 0.f;
        if (t < rows && j < Bs)
            v = Kss[(int64_t)(base + t) * ldk + pb + j] * inv_lam + (sIJ[t] == sIT[pb + j] ? mf : 0.f);
        a[cur ^ 1][t][j] = v;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        const int i = i0 + 8 * r;
        float n = 0.f;
#pragma unroll 8
        for (int t = 0; t < 32; ++t) n = fmaf(a[cur][i][32 + t], a[cur ^ 1][t][j], n);
        N[(size_t)J * 1024 + i * 32 + j] = n;
    }
}

// ---------------------------------------------------------------------------
struct ClWarp {            // what a warp of own super-block J works with
    int P, c, J, slot, sb, nsup, b, rows, lane;
    int prow;              // the lane's row of a panel (lanes past Bs: a valid one)
    float inv_lam, mf;
    double lambda, mdiag;
    float *recv;           // [round][sb]: Delta_round as received
    const float *pan;      // panels T = 0 .. J, pstride floats apart
    size_t pstride;
    const float *xs, *ns;  // L_JJ^-1 and L_JJ^-1 L_{J,J-1}, 32 x 32 row-major
    const uint32_t *dm;    // repeat masks [T][lane]
    uint32_t nz;           // bit T: dm[T] is not all zero
    double rhs;
    double *rho;           // [32]
    uint64_t *bars, *dbar, *pbar, *rbar;
    volatile int *abort_flag;
    int *err;
};

// The residual rho_J = rhs - L_{J, T<=J} Delta0 (double-single products; FP64 repeat term).
template <int BS>
__device__ void cl_residual(const ClWarp &w)
{
    constexpr int NC = BS / 4;
    const int lane = w.lane;
    float hi = 0.f, lo = 0.f;
    bool alive = w.J == 0 || wait_bar<false>(w.pbar, w.abort_flag, w.err);
    for (int T = 0; T < w.J && alive; ++T) {
        PanelRow<BS> p;
        p.load(w.pan + (size_t)T * w.pstride + w.prow * BS, lane);
        if (!wait_bar<true>(&w.bars[T], w.abort_flag, w.err)) {
            alive = false;
            break;
        }
        const float *v = w.recv + T * BS;
        float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f, h2 = 0.f, l2 = 0.f, h3 = 0.f, l3 = 0.f;
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            const float4 x = *(const float4 *)(v + 4 * PanelRow<BS>::chunk(lane, j));
            ds_prod(h0, l0, p.a[j].x, x.x);
            ds_prod(h1, l1, p.a[j].y, x.y);
            ds_prod(h2, l2, p.a[j].z, x.z);
            ds_prod(h3, l3, p.a[j].w, x.w);
        }
        ds_add(h0, l0, h1, l1);
        ds_add(h2, l2, h3, l3);
        ds_add(h0, l0, h2, l2);
        ds_add(hi, lo, h0, l0);
    }
    alive = alive && wait_bar<false>(w.dbar, w.abort_flag, w.err);
    alive = alive && wait_bar<true>(&w.bars[w.J], w.abort_flag, w.err);
    if (alive && lane < w.rows) {
        const float *own = w.recv + w.J * BS;
        float h, l;  // the diagonal panel: the blocks up to this row's block
        panel_dot_ds(w.pan + (size_t)w.J * w.pstride + lane * BS, own, lane, (lane / w.b + 1) * w.b, h, l);
        ds_add(hi, lo, h, l);
        double dmv = (double)own[lane];
        for (uint32_t nz = w.nz; nz; nz &= nz - 1) {  // repeats are rare
            const int T = __ffs(nz) - 1;
            uint32_t mask = w.dm[T * 32 + lane];
            while (mask) {
                dmv += (double)w.recv[T * BS + __ffs(mask) - 1];
                mask &= mask - 1;
            }
        }
        w.rho[lane] = w.rhs - (((double)hi + (double)lo) / w.lambda + w.mdiag * dmv);
    }
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(w.rbar);  // always: the round-1 warp gives up if this one did
}

// The chain of round r.  All updates but the one from J-1 give r'_J; Delta_J = X_J r'_J - N_J
// Delta_{J-1} with N_J = X_J L_{J,J-1}, X_J r'_J formed while Delta_{J-1} is on its way.
// Returns whether Delta_J (d) was formed and sent.
template <int BS>
__device__ bool cl_chain(const ClWarp &w, int r, float *ds, float *rb, float &d)
{
    constexpr int Bs = BS;
    const int lane = w.lane, J = w.J;
    float *rv = w.recv + (size_t)r * w.sb;
    uint64_t *bars = w.bars + r * w.nsup;
    // the CTAs in the order in which they need Delta_J: owners of J + 1, J + 2, ...
    auto dest = [&](int k) {
        int q = w.slot == 1 ? w.c - 1 - k : w.c == w.P - 1 ? w.c - k : w.c + 1 + k;
        q += q < 0 ? w.P : 0;
        return q >= w.P ? q - w.P : q;
    };
    // lanes 0 .. 15: 16 bytes each to the first two; lanes 16 + k: a bulk copy to number 2 + k
    const int nd = lane < 16 ? lane >> 3 : lane - 14, part = lane & 7;
    const bool to = nd < w.P, sends = to && lane < 16 && 4 * part < w.rows, bulk = to && lane >= 16;
    const uint32_t rank = (uint32_t)dest(to ? nd : 0);
    const uint32_t raddr = ptx::mapa(ptx::su32(rv + J * Bs + (lane < 16 ? 4 * part : 0)), rank);
    const uint32_t rbar = ptx::mapa(ptx::su32(&bars[J]), rank);

    float rr = r == 0 ? (float)w.rhs : 0.f;  // round 0: the right-hand side minus updates; round 1: sum of updates
    bool alive = J == 0 || wait_bar<false>(w.pbar, w.abort_flag, w.err);
    PanelRow<BS> pr;
    PanelRow<32> xr;
    PanelRow<BS> nr;
    xr.load(w.xs + lane * 32, lane);
    if (J > 0) nr.load(w.ns + lane * 32, lane);
    for (int T = 0; T + 1 < J && alive; ++T) {
        pr.load(w.pan + (size_t)T * w.pstride + w.prow * Bs, lane);
        if (!wait_bar<true>(&bars[T], w.abort_flag, w.err)) {
            alive = false;
            break;
        }
        const float *dt = rv + T * Bs;
        const float sd = (w.nz >> T) & 1u ? mask_sum(lane < w.rows ? w.dm[T * 32 + lane] : 0u, dt) : 0.f;
        if (r == 0) rr -= pr.template dot<false>(dt, lane) * w.inv_lam + w.mf * sd;
        else rr += pr.template dot<true>(dt, lane) * w.inv_lam + w.mf * sd;
    }
    if (r == 1 && alive) {
        alive = wait_bar<false>(w.rbar, w.abort_flag, w.err);
        if (alive && lane < w.rows) rr = (float)w.rho[lane] - rr;
    }
    d = 0.f;
    if (alive) {
        rb[lane] = lane < w.rows ? rr : 0.f;
        __syncwarp();
        d = xr.template dot<true>(rb, lane);
    }
    if (alive && J > 0) {
        alive = wait_bar<true>(&bars[J - 1], w.abort_flag, w.err);
        if (alive) d -= nr.template dot<true>(rv + (J - 1) * Bs, lane);
    }
    if (!alive) return false;
    ds[lane] = lane < w.rows ? d : 0.f;
    __syncwarp();
    if (sends) ptx::st_async_v4(raddr, *(const float4 *)(ds + 4 * part), rbar);
    ptx::fence_proxy_async();
    __syncwarp();
    if (bulk) ptx::bulk_s2cluster(raddr, ds, (uint32_t)(w.rows * 4), rbar);
    return true;
}

template <int BS>
__global__ void __launch_bounds__(CL_THREADS, 1)
    bdcd_cluster_kernel(const __grid_constant__ CUtensorMap kmap, const int32_t *S, const float *X,
                        const float *Ng, const uint32_t *Mg, const int32_t *nextg, int nblk, int b, double lambda,
                        double mdiag, double *g, int rounds, double *delta, double *w64, float *w32, double *alpha,
                        uint64_t *ctr, uint64_t ctr_advance, const double *rhs_in, ClusterRhs x, int trig_sup, int *err)
{
    extern __shared__ __align__(16) unsigned char sm[];
    const int P = (int)gridDim.x;  // the grid is one cluster
    const int c = (int)ptx::cluster_ctarank();
    const ClGeom G = cl_geom(nblk, b);
    constexpr int Bs = BS;
    const int nsup = G.nsup, sb = nblk * b;
    const ClLayout L = cl_layout(nblk, b, P, c);
    float *recv = (float *)(sm + L.recv);          // [round][sb]: Delta_round as received
    float *xsa = (float *)(sm + L.xs);             // [slot][32][32]: L_JJ^-1, row-major
    float *nsa = (float *)(sm + L.ns);             // [slot][32][32]: L_JJ^-1 L_{J,J-1}, row-major
    uint32_t *dmask = (uint32_t *)(sm + L.dmask);  // [slot][T][lane]
    float *dsend = (float *)(sm + L.dsend);        // [round][slot][32]: own Delta_J
    float *rbufa = (float *)(sm + L.rbuf);         // [round][slot][32]: r_J before the product
    double *rhoa = (double *)(sm + L.rho);         // [slot][32]
    uint64_t *bars = (uint64_t *)(sm + L.bars);    // [round][J], then the local barriers
    uint64_t *lb = bars + 2 * nsup;
    const uint32_t goff = ptx::su32(sm + L.gdata);
    unsigned char *gd = sm + L.gdata + ((128u - (goff & 127u)) & 127u);
    __shared__ int abort_flag_s;
    __shared__ double rhs_pre[CL_SLOTS * 32];
    volatile int *abort_flag = &abort_flag_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int slot = warp & 1, role = warp >> 1;
    const int nown = L.nown;
    // A kernel launched after this one as a programmatic dependent (the fused block, on the SMs
    // this cluster leaves free) may start its set-up and tensor-core products once every CTA has
    // signalled; it waits for this grid to finish before it reads the coefficients or the
    // gradient.  The CTA owning super-block trig_sup signals when its round-0 Delta is out (the
    // kernels forked beside the chain have the other SMs until then); every other CTA at once, or,
    // with a part of the gradient not yet in g (x), when it has read its right-hand side: such a
    // dependent may write g once every CTA has signalled.
    const bool trig_own = trig_sup >= 0 && (trig_sup == cl_own(0, c, P) || (nown > 1 && trig_sup == cl_own(1, c, P)));

    if (tid == 0 && !x.x && !trig_own) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // ---- set-up: barriers and Gram panels (warp 0), right-hand sides (warps 1, 2), inverses and
    // repeat masks (the others, by asynchronous copies) ----
    if (warp == 0) {
        for (int i = lane; i < 2 * nsup + NLOCAL; i += 32)
            ptx::mbar_init(&bars[i], 1);
        if (lane == 0) abort_flag_s = 0;
        ptx::mbar_init_fence();
        __syncwarp();
        for (int i = lane; i < rounds * nsup; i += 32) {
            const int r = i >= nsup ? 1 : 0, J = i - r * nsup;
            ptx::mbar_expect_tx(&bars[i], (uint32_t)(cl_rows(J, Bs, sb) * 4));
        }
        if (lane < nown) {
            const int J = cl_own(lane, c, P);
            if (J > 0) ptx::mbar_expect_tx(&lb[3 * lane + 1], (uint32_t)(J * Bs * Bs * 4));
            ptx::mbar_expect_tx(&lb[3 * lane + 0], (uint32_t)(Bs * Bs * 4));
        }
        __syncwarp();
        size_t base = 0;
        for (int k = 0; k < nown; ++k) {  // panel T of own super-block k
            const int J = cl_own(k, c, P);
            if (lane <= J)
                ptx::tma_load_2d(gd + (base + lane) * L.ps, &kmap, &lb[3 * k + (lane == J ? 0 : 1)], lane * Bs, J * Bs);
            base += (size_t)J + 1;
        }
    } else if (warp <= CL_SLOTS) {
        const int k = warp - 1, J = k < nown ? cl_own(k, c, P) : 0, p = J * Bs + lane;
        if (k < nown && lane < cl_rows(J, Bs, sb)) {
            double v = 0.0;
            if (rhs_in) {
                v = rhs_in[p];
            } else {
                const int32_t row = S[p];
                if (x.x) {  // with the part of the gradient not yet in g
                    int q = x.link[p];
                    for (int h = 0; h < x.nx; ++h) v += x.x[(int64_t)h * x.ldx + p];
                    if (q >= 0) {  // rare: the previous step's positions that hold this row, in order
                        double sum = 0.0;
                        for (; q >= 0; q = x.next[q]) sum += x.delta[q];
                        v += mdiag * sum;
                    }
                }
                v = -(g[row] + v);
            }
            rhs_pre[k * 32 + lane] = v;
        }
        if (x.x) {
            asm volatile("barrier.cta.sync 1, %0;" ::"n"(32 * CL_SLOTS) : "memory");
            if (warp == 1 && lane == 0 && !trig_own) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        }
    } else {
        constexpr int NT = CL_THREADS - 32 * (1 + CL_SLOTS);
        const int t = tid - 32 * (1 + CL_SLOTS);
        for (int k = 0; k < nown; ++k) {
            const int J = cl_own(k, c, P);
            for (int e = t; e < 256; e += NT) {
                ptx::cp_async16(xsa + k * 1024 + 4 * e, X + (size_t)J * 1024 + 4 * e);
                if (J > 0) ptx::cp_async16(nsa + k * 1024 + 4 * e, Ng + (size_t)J * 1024 + 4 * e);
            }
            for (int e = t; e < (J + 1) * 8; e += NT)
                ptx::cp_async16(dmask + k * CL_NSUP_MAX * 32 + 4 * e, Mg + (size_t)J * CL_NSUP_MAX * 32 + 4 * e);
        }
        ptx::cp_async_wait_all();
    }
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");

    const int J = slot < nown ? cl_own(slot, c, P) : -1;
    ClWarp w;
    w.P = P;
    w.c = c;
    w.J = J;
    w.slot = slot;
    w.sb = sb;
    w.nsup = nsup;
    w.b = b;
    w.rows = J >= 0 ? cl_rows(J, Bs, sb) : 0;
    w.lane = lane;
    w.prow = lane < Bs ? lane : Bs - 1;
    w.inv_lam = (float)(1.0 / lambda);
    w.mf = (float)mdiag;
    w.lambda = lambda;
    w.mdiag = mdiag;
    w.recv = recv;
    w.pan = (const float *)(gd + (slot == 0 ? 0 : (size_t)cl_own(0, c, P) + 1) * L.ps);
    w.pstride = L.ps / 4;
    w.xs = xsa + slot * 1024;
    w.ns = nsa + slot * 1024;
    w.dm = dmask + slot * CL_NSUP_MAX * 32;
    w.rhs = lane < w.rows ? rhs_pre[slot * 32 + lane] : 0.0;
    w.rho = rhoa + slot * 32;
    w.bars = bars;
    w.dbar = &lb[3 * slot + 0];
    w.pbar = &lb[3 * slot + 1];
    w.rbar = &lb[3 * slot + 2];
    w.abort_flag = abort_flag;
    w.err = err;
    uint32_t seen = 0;  // lane T: the masks of panel T together
    if (lane <= J)
        for (int q = 0; q < 8; ++q) {
            const uint4 v = *(const uint4 *)(w.dm + lane * 32 + 4 * ((lane + q) & 7));
            seen |= v.x | v.y | v.z | v.w;
        }
    w.nz = __ballot_sync(0xffffffffu, seen != 0);
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // every CTA's barriers expect their bytes

    if (J >= 0 && role == 3 && rounds > 1) cl_residual<BS>(w);
    if (J >= 0 && role < rounds) {
        const int r = role;  // the round this warp runs
        float d;
        const bool sent = cl_chain<BS>(w, r, dsend + (r * CL_SLOTS + slot) * 32, rbufa + (r * CL_SLOTS + slot) * 32, d);
        if (r == 0 && J == trig_sup && lane == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        // Delta = the sum over the rounds
        const bool have = sent && (r == 0 || wait_bar<true>(&bars[J], abort_flag, err));
        if (have && r == rounds - 1 && lane < w.rows) {
            const int row = J * Bs + lane;
            const double dd = (r == 1 ? (double)recv[row] : 0.0) + (double)d, dw = dd / lambda;
            delta[row] = dd;
            if (w64) w64[row] = dw;
            if (w32) w32[row] = (float)dw;
        }
    }
    // every Delta addressed to this CTA, and every panel copy, lands before it leaves
    if (tid == 0) {
        for (int k = 0; k < nown; ++k) {
            const unsigned long long lim = *abort_flag ? 10000000ull : CL_WAIT_NS;
            bool ok = ptx::mbar_wait_bounded(&lb[3 * k + 0], 0, lim);
            if (cl_own(k, c, P) > 0) ok = ptx::mbar_wait_bounded(&lb[3 * k + 1], 0, lim) && ok;
            if (!ok && !*abort_flag) {
                *abort_flag = 1;
                set_error(err, DEV_TIMEOUT);
            }
        }
        for (int i = 0; i < rounds * nsup; ++i) {
            const unsigned long long lim = *abort_flag ? 10000000ull : CL_WAIT_NS;
            if (!ptx::mbar_wait_cluster_bounded(&bars[i], 0, lim) && !*abort_flag) {
                *abort_flag = 1;
                set_error(err, DEV_TIMEOUT);
            }
        }
    }
    __syncthreads();
    // a6 for the own rows, now that every Delta has landed here: a row holding the first occurrence
    // of its index adds Delta (over the rounds) of all occurrences, in position order, to alpha and
    // mdiag times that to g (the same sums, in the same order, as the sorted update)
    if (alpha && !*abort_flag && J >= 0 && role == 0 && lane < cl_rows(J, Bs, sb)) {
        const int row = J * Bs + lane;
        bool head = true;
        for (int T = 0; T <= J; ++T) head = head && dmask[slot * CL_NSUP_MAX * 32 + T * 32 + lane] == 0;
        if (head) {
            auto dsum = [&](int q) {
                double d = 0.0;
                for (int r = 0; r < rounds; ++r) d += (double)recv[(size_t)r * sb + q];
                return d;
            };
            double sum = dsum(row);
            for (int q = nextg[row]; q > row; q = nextg[q]) sum += dsum(q);
            const int32_t i = S[row];
            alpha[i] += sum;
            g[i] += mdiag * sum;
        }
    }
    if (alpha && tid == 0 && c == 0 && ctr) *ctr += ctr_advance;
    ptx::cluster_sync();  // no CTA leaves while another may still address it
}

// super-blocks have 20, 24, 28 or 32 rows (b a multiple of 4, at most 32)
auto cluster_kernel(int bs)
{
    return bs == 32 ? bdcd_cluster_kernel<32> : bs == 28 ? bdcd_cluster_kernel<28> : bs == 24 ? bdcd_cluster_kernel<24>
                                                                                             : bdcd_cluster_kernel<20>;
}

bool cluster_fits(int P, size_t smem, int bs)
{
    auto kfn = cluster_kernel(bs);
    if (cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CL_SMEM_MAX) != cudaSuccess)
        return false;
    if (cudaFuncSetAttribute(kfn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)P, 1, 1);
    cfg.blockDim = dim3(CL_THREADS, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)P;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kfn, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n >= 1;
}

// two super-blocks per CTA
int cluster_ctas(int nsup) { return (nsup + 1) / 2; }

size_t cluster_smem(int nblk, int b, int P)
{
    size_t smem = 0;
    for (int c = 0; c < P; ++c) {
        const ClLayout L = cl_layout(nblk, b, P, c);
        if (L.total > smem) smem = L.total;
    }
    return smem;
}

}  // namespace

// Cluster size for nblk blocks of size b (0: the cluster path does not apply).
int recur_cluster_size(int nblk, int b, int rounds)
{
    if (b % 4 != 0 || b > 32 || rounds < 1 || rounds > 2 || nblk < 1) return 0;
    const ClGeom G = cl_geom(nblk, b);
    if (G.nsup > CL_NSUP_MAX) return 0;
    // one occupancy query per shape (a map: batched solves mix shapes)
    static std::mutex mu;
    static std::map<long long, int> cache;
    const long long key = ((long long)nblk << 20) | ((long long)b << 4) | rounds;
    std::lock_guard<std::mutex> lock(mu);
    const auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    const int P = cluster_ctas(G.nsup);
    const size_t smem = cluster_smem(nblk, b, P);
    const bool ok = smem <= CL_SMEM_MAX && cluster_fits(P, smem, G.Bs);
    cache[key] = ok ? P : 0;
    return ok ? P : 0;
}

size_t recur_cluster_scratch_bytes(int64_t nblk, int b)
{
    if (b % 4 != 0 || b > 32) return 0;
    const ClGeom G = cl_geom((int)nblk, b);
    if (G.nsup > CL_NSUP_MAX) return 0;
    return 2 * (size_t)G.nsup * 1024 * 4 + (size_t)G.nsup * CL_NSUP_MAX * 32 * 4 + (size_t)nblk * b * 4;
}

// The two halves of launch_recur_cluster: the prep kernel (inverses,
// couplings, repeat masks, links; it needs only Kss and S, so a step's prep
// may run ahead of the previous step's chain) and the chain.
cudaError_t launch_recur_cluster_prep(const float *Kss, int64_t ldk, const int32_t *S, int nblk, int b, double lambda,
                                      double mdiag, void *scratch, int *err, cudaStream_t st)
{
    const ClGeom G = cl_geom(nblk, b);
    if (((uintptr_t)scratch & 15) != 0) return cudaErrorInvalidValue;
    float *X = (float *)scratch;
    float *N = X + (size_t)G.nsup * 1024;
    uint32_t *M = (uint32_t *)(N + (size_t)G.nsup * 1024);
    int32_t *next = (int32_t *)(M + (size_t)G.nsup * CL_NSUP_MAX * 32);
    bdcd_prep_kernel<<<(unsigned)(2 * G.nsup), PREP_THREADS, 0, st>>>(Kss, ldk, S, nblk, b, (float)(1.0 / lambda),
                                                                     (float)mdiag, X, N, M, next, err);
    return cudaGetLastError();
}

const int32_t *recur_cluster_next(const void *scratch, int nblk, int b)
{
    const ClGeom G = cl_geom(nblk, b);
    return (const int32_t *)((const float *)scratch + 2 * (size_t)G.nsup * 1024 + (size_t)G.nsup * CL_NSUP_MAX * 32);
}

cudaError_t launch_recur_cluster_chain(const float *Kss, int64_t ldk, const int32_t *S, int nblk, int b, int P,
                                       double lambda, double mdiag, double *g, int rounds, void *scratch,
                                       double *delta, double *w64, float *w32, const FusedUpdate *upd, int *err,
                                       cudaStream_t st, const double *rhs, int trig_sup, const ClusterRhs *x, int prio)
{
    const ClGeom G = cl_geom(nblk, b);
    const int sb = nblk * b;
    if ((ldk * 4) % 16 != 0 || ((uintptr_t)Kss & 15) != 0 || ((uintptr_t)scratch & 15) != 0)
        return cudaErrorInvalidValue;
    float *X = (float *)scratch;
    float *N = X + (size_t)G.nsup * 1024;
    uint32_t *M = (uint32_t *)(N + (size_t)G.nsup * 1024);
    int32_t *next = (int32_t *)(M + (size_t)G.nsup * CL_NSUP_MAX * 32);
    CUtensorMap kmap;
    if (!make_map_f32_2d(&kmap, Kss, sb, sb, ldk, G.Bs, G.Bs)) return cudaErrorInvalidValue;
    auto kfn = cluster_kernel(G.Bs);
    static bool attrs[4] = {false, false, false, false};
    bool &attr = attrs[(32 - G.Bs) / 4];
    cudaError_t e;
    if (!attr) {
        e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CL_SMEM_MAX);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(kfn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)P, 1, 1);
    cfg.blockDim = dim3(CL_THREADS, 1, 1);
    cfg.dynamicSmemBytes = cluster_smem(nblk, b, P);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)P;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributePriority;
    at[1].val.priority = prio;
    cfg.attrs = at;
    cfg.numAttrs = prio ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kfn, kmap, S, (const float *)X, (const float *)N, (const uint32_t *)M,
                              (const int32_t *)next, nblk, b, lambda, mdiag, g, rounds, delta, w64, w32,
                              upd ? upd->alpha : (double *)nullptr, upd ? upd->ctr : (uint64_t *)nullptr,
                              upd ? upd->ctr_advance : (uint64_t)0, rhs, x ? *x : ClusterRhs{}, trig_sup, err);
}

cudaError_t launch_recur_cluster(const float *Kss, int64_t ldk, const int32_t *S, int nblk, int b, int P,
                                 double lambda, double mdiag, double *g, int rounds, void *scratch, double *delta,
                                 double *w64, float *w32, const FusedUpdate *upd, int *err, cudaStream_t st,
                                 const double *rhs)
{
    cudaError_t e = launch_recur_cluster_prep(Kss, ldk, S, nblk, b, lambda, mdiag, scratch, err, st);
    if (e != cudaSuccess) return e;
    return launch_recur_cluster_chain(Kss, ldk, S, nblk, b, P, lambda, mdiag, g, rounds, scratch, delta, w64, w32, upd,
                                      err, st, rhs);
}

// The largest diagonal panel (in blocks) one cluster launch solves: the
// blocked recurrence for longer chains runs panels of this size.
int recur_cluster_panel_blocks(int b, int rounds)
{
    if (b % 4 != 0 || b > 32) return 0;
    const int q = cl_geom(1, b).q;
    for (int nsup = CL_NSUP_MAX; nsup >= 2; nsup -= 2)
        if (recur_cluster_size(nsup * q, b, rounds) > 0) return nsup * q;
    return 0;
}

}  // namespace dcd
