// Contour filter of problems with B = I from one Krylov space per column.
//
// For B = I every shifted system of a contour pass, (z_e I - A) y_e = b, has
// the same right-hand side and the same Krylov spaces K_k(A, b), whatever the
// node z_e (shift invariance; Frommer, "BiCGStab(l) for families of shifted
// linear systems", 2003; for COCG, Takayama, Hoshi, Sogabe, Zhang and Fujiwara,
// Phys. Rev. B 73, 165108, 2006).
// COCG started at zero returns the iterate y_k in K_k whose residual is
// orthogonal (without conjugation) to K_k, so with the real orthonormal
// Lanczos basis V_k of K_k and T_k = V_k^T A V_k, beta_1 = ||b||,
//     y_{e,k} = V_k u_e,  (z_e I - T_k) u_e = beta_1 e_1,
//     ||r_{e,k}|| = beta_{k+1} |(u_e)_k|,
// for A real symmetric and b real: one real three-term recurrence replaces one
// complex COCG per node, and every (node, column) pair still stops at its own
// step, the one at which its own COCG would.  The filter then is
//     Q = X rho(Lambda) + V_K g,   g = sum_e Re(c_e u_e)   (K x columns, real),
// one combination of the stored basis.  Bytes per element and step in the
// filter's real type: 7 (below) instead of 20 per node.
//
// One cooperative launch does a whole contour pass.  Columns are cut into
// tiles of 8, 4, 2 or 1 16-byte lanes per row (a thread owns one lane of a
// row).  A team of CTAs takes one tile at a time from a queue:
//   init     u_1 = b, ||b||
//   A(j)     s = A v_j - beta_j v_{j-1} (v = u / beta), partial sums of v_j^T s
//   B(j)     u_{j+1} = s - alpha_j v_j, partial sums of ||u_{j+1}||^2
//   check    the team's first CTA advances the pivots of z_e - T_j for every
//            (node, column) pair and finds the pairs that are done
//   solve    u_e by the UL factors of z_e - T (FP64), summed over the nodes
//   combine  Q = X rho(Lambda) + sum_j g_j u_j
// with a barrier of the team's CTAs after init, A and B; no host round trip and
// no launch between.  Two forms:
//   resident  every CTA owns a contiguous range of rows and keeps its part of
//             u_j and u_{j-1} (then s, then u_{j+1}) in shared memory; only the
//             neighbours outside the range and the stored basis are global.
//             A small problem is one CTA per tile with no barrier at all.
//   cached    blocks of rows dealt out in turn, everything in global memory,
//             two CTAs per SM, all tiles at once: for problems whose ranges do
//             not fit, or where the sums of the resident form's many narrow
//             tiles cost more than the traffic.
// A and the shifts are multiplied by a power of two that brings A's largest
// entry near 1 (krylov_scale; the solutions by the same factor at the end), and
// the pivots of z_e - T_j are carried in the filter's real type: no square
// leaves its range for matrices of any size, and a pair of an FP64 pass stops
// where FP64 recurrences stop it.
// What bounds it (GB300, 2.07 GHz).  Cached, 7-point 64^3, 150 float columns:
// 20 ms a pass of 80 steps and 222 (node, step) pairs against 154 ms with COCG
// per node (a call that has to map the bases' 13.6 GB takes 26 ms among others
// and 49 alone, with the memory at hand 20.6); a step moves 0.94 GB, A 130 us (3.6 TB/s: the gather's reads
// through L2, 21 bytes an element, and too few loads in flight), B 88 us (5.4
// TB/s, DRAM), the two sums 30 us.  Resident, one CTA per 4-column tile
// (n = 1000): 6.3 us a step, the entries' exchange and two block sums; FP64
// 32^3: 76 us a step, of which the FP64 ALU needs 40.  Narrow tiles were
// measured against wide ones at n = 5917 (37 columns, 40 steps): 4 columns x 15
// CTAs 0.41 ms of steps, 4 x 1 0.71, 32 x 64 0.52.
// Tried on 64^3 and not kept: u_j alone in shared memory (26 ms), the same with
// shared loads split from global ones by a vote per entry (32 ms) or by
// predicates (37 ms), 1,024 threads per CTA (34 ms), the resident form with 16
// columns (28 ms: its sums take 12 us of a 32 us step).
// Sums are deterministic: fixed rows per thread, fixed order of threads and
// CTAs.  Single-precision sums are carried as unevaluated pairs (TwoSum), so a
// dot product loses little beyond its products' rounding; GB300's FP64 ALU is
// too slow for per-thread sums.
#include <algorithm>
#include <cmath>

#include "feast_internal.cuh"
#include "team.cuh"

namespace feast {

static constexpr int kLzThreads = 512;
static constexpr int kLzWarps = kLzThreads / 32;
static constexpr int kLzMaxLanes = 8;                       // 16-byte lanes per tile row: 8, 4, 2 or 1
static constexpr int kLzGrain = 16;                         // rows of a CTA: a multiple of this
static constexpr int kLzChunk = 8;                          // entries per packed chunk
static constexpr int kLzSmem = 216 * 1024;                  // shared memory for a CTA's rows of u_j and u_{j-1}

// Rows of each CTA's range in the staged form, for a problem of n rows: the
// packed entries, the shared memory and the kernel all go by it.
__host__ __device__ inline int krylov_rpc(int n, int nc) { return ((n + nc - 1) / nc + kLzGrain - 1) / kLzGrain * kLzGrain; }

static constexpr int kLzFar = 3;  // of a row's eight entries, those always read from global memory

template <typename T> struct LzVec;
template <> struct LzVec<float> { using type = float4; };
template <> struct LzVec<double> { using type = double2; };

template <typename T>
union LzPack {
    typename LzVec<T>::type v;
    T e[16 / sizeof(T)];
};

// ---------------------------------------------------------------- sums
// A running sum: a pair h + l of the exact sum's leading parts (float), or a
// plain double.
template <typename T> struct LzSum;
template <> struct LzSum<float> {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void add(float x)
    {
        const float t = h + x, b = t - h;
        l += (h - (t - b)) + (x - b);
        h = t;
    }
    __device__ __forceinline__ void add(const LzSum& o)
    {
        add(o.h);
        l += o.l;
    }
    __device__ __forceinline__ LzSum xor_lane(int m) const
    {
        LzSum o;
        o.h = __shfl_xor_sync(0xffffffffu, h, m);
        o.l = __shfl_xor_sync(0xffffffffu, l, m);
        return o;
    }
    __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};
template <> struct LzSum<double> {
    double h = 0.0;
    __device__ __forceinline__ void add(double x) { h += x; }
    __device__ __forceinline__ void add(const LzSum& o) { h += o.h; }
    __device__ __forceinline__ LzSum xor_lane(int m) const
    {
        LzSum o;
        o.h = __shfl_xor_sync(0xffffffffu, h, m);
        return o;
    }
    __device__ __forceinline__ double value() const { return h; }
};

// A (node, column) pair while it iterates: its shift (scaled), pivot of z_e - T_j,
// (|r| / |b|)^2; in FP64, where a division is a long chain that every CTA of the
// team waits for, also 1 / |pivot|^2.
template <typename T>
struct alignas(sizeof(T) == 4 ? 32 : 16) LzPair {
    double zr;
    T zi, re, im, f2, rd;
};

// ---------------------------------------------------------------- packed rows
template <typename T> __device__ __forceinline__ void lz_entries(const int4* __restrict__ ent, int c, int (&j)[kLzChunk], T (&a)[kLzChunk]);
template <> __device__ __forceinline__ void lz_entries<float>(const int4* __restrict__ ent, int c, int (&j)[kLzChunk], float (&a)[kLzChunk])
{
#pragma unroll
    for (int u = 0; u < kLzChunk / 2; ++u) {
        const int4 v = __ldg(ent + (c >> 1) + u);
        j[2 * u] = v.x;
        a[2 * u] = __int_as_float(v.y);
        j[2 * u + 1] = v.z;
        a[2 * u + 1] = __int_as_float(v.w);
    }
}
template <> __device__ __forceinline__ void lz_entries<double>(const int4* __restrict__ ent, int c, int (&j)[kLzChunk], double (&a)[kLzChunk])
{
#pragma unroll
    for (int u = 0; u < kLzChunk; ++u) {
        const int4 v = __ldg(ent + c + u);
        j[u] = v.x;
        a[u] = __hiloint2double(v.w, v.z);
    }
}

// 16 bytes at p, or zero; stays where it is written, ahead of its use.
__device__ __forceinline__ float4 lz_load(bool on, const float4* p)
{
    float4 v;
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %4, 0;\n\t"
        "mov.f32 %0, 0f00000000;\n\tmov.f32 %1, 0f00000000;\n\tmov.f32 %2, 0f00000000;\n\tmov.f32 %3, 0f00000000;\n\t"
        "@p ld.global.v4.f32 {%0, %1, %2, %3}, [%5];\n}"
        : "=&f"(v.x), "=&f"(v.y), "=&f"(v.z), "=&f"(v.w)
        : "r"((int)on), "l"(p));
    return v;
}
__device__ __forceinline__ double2 lz_load(bool on, const double2* p)
{
    double2 v;
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t"
        "mov.f64 %0, 0d0000000000000000;\n\tmov.f64 %1, 0d0000000000000000;\n\t"
        "@p ld.global.v2.f64 {%0, %1}, [%3];\n}"
        : "=&d"(v.x), "=&d"(v.y)
        : "r"((int)on), "l"(p));
    return v;
}

// The eight packed entries of a row, held by its LPR lanes (K = 8 / LPR each).
template <typename T, int LPR> struct LzEntry;
template <int LPR> struct LzEntry<float, LPR> {
    static constexpr int K = kLzChunk / LPR;
    int2 e[K];
    __device__ __forceinline__ void load(bool on, const int4* __restrict__ ent, size_t row, int l)
    {
        if constexpr (K == 1) {
            e[0] = on ? __ldg((const int2*)ent + row * kLzChunk + l) : make_int2(0, 0);
        } else {
#pragma unroll
            for (int u = 0; u < K / 2; ++u) {
                const int4 v = on ? __ldg(ent + row * (kLzChunk / 2) + l * (K / 2) + u) : make_int4(0, 0, 0, 0);
                e[2 * u] = make_int2(v.x, v.y);
                e[2 * u + 1] = make_int2(v.z, v.w);
            }
        }
    }
    __device__ __forceinline__ int col(int u) const
    {
        if constexpr (LPR == 1) return e[u].x;
        else return __shfl_sync(0xffffffffu, e[u % K].x, u / K, LPR);
    }
    __device__ __forceinline__ float val(int u) const
    {
        if constexpr (LPR == 1) return __int_as_float(e[u].y);
        else return __int_as_float(__shfl_sync(0xffffffffu, e[u % K].y, u / K, LPR));
    }
};
template <int LPR> struct LzEntry<double, LPR> {
    static constexpr int K = kLzChunk / LPR;
    int4 e[K];
    __device__ __forceinline__ void load(bool on, const int4* __restrict__ ent, size_t row, int l)
    {
#pragma unroll
        for (int u = 0; u < K; ++u) e[u] = on ? __ldg(ent + row * kLzChunk + l * K + u) : make_int4(0, 0, 0, 0);
    }
    __device__ __forceinline__ int col(int u) const
    {
        if constexpr (LPR == 1) return e[u].x;
        else return __shfl_sync(0xffffffffu, e[u % K].x, u / K, LPR);
    }
    __device__ __forceinline__ double val(int u) const
    {
        if constexpr (LPR == 1) return __hiloint2double(e[u].w, e[u].z);
        else
            return __hiloint2double(__shfl_sync(0xffffffffu, e[u % K].w, u / K, LPR),
                                    __shfl_sync(0xffffffffu, e[u % K].z, u / K, LPR));
    }
};

// Rows of a CTA: a contiguous range (resident form), or blocks of kLzBlock
// rows dealt out in turn, so that the CTAs sweep the tile together and a row's
// far neighbours are still in L2.
static constexpr int kLzBlock = 256;

template <bool RES, int PASS>
__device__ __forceinline__ int lz_row(int t, int slot, int r0, int c, int nc)
{
    if (RES) return r0 + slot + t * PASS;
    constexpr int PB = kLzBlock / PASS;  // passes per block
    return ((t / PB) * nc + c) * kLzBlock + (t % PB) * PASS + slot;
}

template <typename T, int LPR, bool RES>
__global__ void __launch_bounds__(kLzThreads, RES ? 1 : 2) krylov_filter(KrylovArgs a)
{
    constexpr int N = 16 / sizeof(T);          // columns per thread
    constexpr int COLS = LPR * N;              // columns per tile
    constexpr int PASS = kLzThreads / LPR;     // rows per pass of the CTA
    constexpr int PARTS = kLzThreads / COLS;
    static_assert(RES || LPR == kLzMaxLanes, "the cached form has one width");
    using V = typename LzVec<T>::type;
    using S = LzSum<T>;
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ S red[kLzThreads];
    __shared__ T s_al[COLS], s_inv[COLS], s_bt[COLS];
    __shared__ int s_unit;
    __shared__ double s_zs;  // factor of A and the shifts
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int l = tid & (LPR - 1), slot = tid / LPR;
    const int nc = a.nc, team = blockIdx.x / nc, c = blockIdx.x - team * nc;
    unsigned* bar = a.bar + (size_t)team * 32;
    volatile int* mail = a.mail + (size_t)team * 32;  // [0] next unit, [1] all pairs of the tile done
    unsigned target = 0;
    V* basis = (V*)(a.basis + (size_t)team * a.team_bytes);
    const size_t sv = a.slot_vecs;  // vectors of 16 bytes per basis slot
    S* part = (S*)a.part + (size_t)team * 2 * nc * COLS;
    double* al_g = a.coef + (size_t)team * 2 * (a.maxit + 2) * COLS;  // alpha_j, row j
    double* bt_g = al_g + (size_t)(a.maxit + 2) * COLS;               // beta_{j+1}, row j
    T* g_g = (T*)a.g + (size_t)team * a.maxit * COLS;
    const int npair = COLS * a.ne;
    LzPair<T>* pst = (LzPair<T>*)a.pair + (size_t)team * npair;
    int* kst = a.kstop + (size_t)team * npair;    // step at which the pair stopped, -1 while it iterates
    double2* piv = a.piv + (size_t)team * COLS * a.nl * a.maxit;

    // sum over the team's CTAs of per-thread sums acc[N] of the thread's
    // columns; the totals arrive in red[0..COLS) of every CTA, column tid in
    // thread tid.  buf: 0 or 1, alternating.
    auto team_total = [&](S (&acc)[N], int buf) -> bool {
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1)
#pragma unroll
            for (int q = 0; q < N; ++q) acc[q].add(acc[q].xor_lane(o));
        if (lane < LPR)
#pragma unroll
            for (int q = 0; q < N; ++q) red[warp * COLS + lane * N + q] = acc[q];
        __syncthreads();
        S s;
        if (tid < COLS)
            for (int w = 0; w < kLzWarps; ++w) s.add(red[w * COLS + tid]);
        if (nc > 1) {
            if (tid < COLS) part[((size_t)buf * nc + c) * COLS + tid] = s;
            if (!team_sync(bar, target, nc, a.err, a.limit)) return false;
            const int col = tid % COLS, p = tid / COLS;
            S t;
#pragma unroll 4
            for (int k = p; k < nc; k += PARTS) t.add(part[((size_t)buf * nc + k) * COLS + col]);
            red[p * COLS + col] = t;
            __syncthreads();
            if (tid < COLS) {
                s = red[tid];
                const int np = min(PARTS, nc);
                for (int k = 1; k < np; ++k) s.add(red[k * COLS + tid]);
            }
        } else {
            __syncthreads();
        }
        if (tid < COLS) red[tid] = s;
        return true;
    };

    int unit = team;
    while (unit < a.nunits) {
        const int2 un = a.units ? a.units[unit] : make_int2(0, unit);
        const FiltProb& P = a.probs[un.x];
        const int n = P.n, g = un.y, m0 = P.m0;
        const int mk = P.mk ? min(*P.mk, m0) : m0;
        if (tid == 0) s_zs = krylov_scale(*P.amax);  // read after the sums of init
        const int rpc = krylov_rpc(n, nc);
        const int r0 = RES ? min(n, c * rpc) : 0;
        const int rows = RES ? min(n, r0 + rpc) - r0 : 0;
        const int rend = RES ? r0 + rows : n;
        V* xcur = (V*)dsm;                       // resident form: the CTA's rows of u_j
        V* xold = (V*)dsm + (size_t)rpc * LPR;   // and of u_{j-1}, then s, then u_{j+1}
        int nt;  // passes of this CTA
        if (RES) {
            nt = (rows + PASS - 1) / PASS;
        } else {
            const int nblk = (n + kLzBlock - 1) / kLzBlock;
            nt = nblk > c ? (nblk - c + nc - 1) / nc * (kLzBlock / PASS) : 0;
        }
        const int4* __restrict__ ent = (const int4*)P.apk;
        const int* __restrict__ app = P.app;
        const int col0 = g * COLS + l * N;  // the thread's first column
        // element of the FP64 blocks: row-major, or the real (even row) or imaginary
        // part (odd row) of a complex block
        auto elem = [&](int i, int col) {
            return P.q_off + (a.cplx ? ((size_t)(i >> 1) * m0 + col) * 2 + (i & 1) : (size_t)i * m0 + col);
        };
        auto row_of = [&](int t) { return lz_row<RES, PASS>(t, slot, r0, c, nc); };

        // ---- init: u_1 = b
        S acc[N];
        for (int t = 0; t < nt; ++t) {
            const int i = row_of(t);
            if (i >= rend) continue;
            LzPack<T> x;
#pragma unroll
            for (int q = 0; q < N; ++q) {
                x.e[q] = col0 + q < mk ? (T)a.R[elem(i, col0 + q)] : T(0);
                acc[q].add(x.e[q] * x.e[q]);
            }
            basis[(size_t)i * LPR + l] = x.v;
            if (RES) xcur[(i - r0) * LPR + l] = x.v;
        }
        if (!team_total(acc, 1)) return;
        if (tid < COLS) {
            const double b2 = red[tid].value();
            const bool live = g * COLS + tid < mk && b2 > 0.0 && b2 < 1.7e308;
            const T b = live ? (T)sqrt(b2) : T(0);
            const bool ok = b > T(0);
            s_bt[tid] = T(0);
            s_inv[tid] = ok ? T(1) / b : T(0);
            if (c == 0) {
                bt_g[tid] = (double)b;
                // the pairs of this column: pivot, relative residual, stop step
                for (int e = 0; e < a.ne; ++e) {
                    pst[e * COLS + tid] = {P.zw[4 * e] * s_zs, (T)(P.zw[4 * e + 1] * s_zs), T(0), T(0), T(1), T(0)};
                    kst[e * COLS + tid] = ok ? -1 : 0;
                }
            }
        }
        if (c == 0 && tid == 0) mail[1] = 0;
        __syncthreads();
        T inv[N], cb[N];  // 1 / beta_j; beta_j / beta_{j-1}
#pragma unroll
        for (int q = 0; q < N; ++q) {
            inv[q] = s_inv[l * N + q];
            cb[q] = T(0);
        }

        int k = 0;  // steps done
        for (int j = 1; j <= a.maxit; ++j) {
            const V* uj = basis + (size_t)(j - 1) * sv + l;              // u_j
            const V* up = basis + (size_t)(j > 1 ? j - 2 : 0) * sv + l;  // u_{j-1}
            V* sj = basis + (size_t)j * sv + l;                          // u_{j+1} (cached form: s before)
            // ---- A(j)
#pragma unroll
            for (int q = 0; q < N; ++q) acc[q] = S();
            // s of a row from its gathered sum; d[q] += v s
            auto finish = [&](int i, LzPack<T>& sum, const LzPack<T>& pv, const LzPack<T>& ov, T (&d)[N]) {
#pragma unroll
                for (int q = 0; q < N; ++q) {
                    sum.e[q] = fma(-cb[q], pv.e[q], inv[q] * sum.e[q]);
                    d[q] = fma(inv[q] * ov.e[q], sum.e[q], d[q]);
                }
                if (RES) xold[(i - r0) * LPR + l] = sum.v;
                else sj[(size_t)i * LPR] = sum.v;
            };
            if (RES || a.one_chunk) {
                // Rows of eight packed entries (krylov_pack).  The last kLzFar
                // entries, where the far neighbours are, load from global memory one
                // pair of rows ahead, the entries themselves two; the first ones are
                // the row's near neighbours, in shared memory in the resident form.
                using E = LzEntry<T, LPR>;
                constexpr int kNear = kLzChunk - kLzFar;
                const bool whole = RES && nc == 1;  // every row is in shared memory
                auto entry = [&](int t, E& e) {
                    const int i = row_of(t);
                    e.load(t < nt && i < rend, ent, (size_t)i, l);
                };
                struct Ahead {
                    LzPack<T> x[kLzFar], pv;
                };
                auto ahead = [&](int t, const E& e, Ahead& f) {
                    if (!whole) {
#pragma unroll
                        for (int u = 0; u < kLzFar; ++u) {
                            const int x = e.col(kNear + u);
                            f.x[u].v = lz_load(x >= 0, uj + (size_t)x * LPR);
                        }
                    }
                    if (!RES) {
                        const int i = row_of(t);
                        f.pv.v = lz_load(j > 1 && t < nt && i < rend, up + (size_t)i * LPR);
                    }
                };
                auto row = [&](int t, const E& e, Ahead& f, T (&d)[N]) {
                    const int i = row_of(t);
                    const bool ok = t < nt && i < rend;
                    LzPack<T> x[kNear], sum;
                    const int own = e.col(0);
                    if (RES && !__any_sync(0xffffffffu, own < 0)) {  // every near neighbour in the own range
#pragma unroll
                        for (int u = 0; u < kNear; ++u) {
                            const int r = u ? e.col(u) : own;
#pragma unroll
                            for (int q = 0; q < N; ++q) x[u].e[q] = T(0);
                            if (r >= 0) x[u].v = xcur[r * LPR + l];
                        }
                    } else {
                        const bool in = RES && own >= 0;
#pragma unroll
                        for (int u = 0; u < kNear; ++u) {
                            const int r = u ? e.col(u) : (own >= 0 ? own : ~own);
#pragma unroll
                            for (int q = 0; q < N; ++q) x[u].e[q] = T(0);
                            if (r >= 0) x[u].v = uj[(size_t)(in ? r0 + r : r) * LPR];
                        }
                    }
                    if (whole) {
#pragma unroll
                        for (int u = 0; u < kLzFar; ++u) {
                            const int r = e.col(kNear + u);
#pragma unroll
                            for (int q = 0; q < N; ++q) f.x[u].e[q] = T(0);
                            if (r >= 0) f.x[u].v = xcur[r * LPR + l];
                        }
                    }
                    if (RES) {
#pragma unroll
                        for (int q = 0; q < N; ++q) f.pv.e[q] = T(0);
                        if (j > 1 && ok) f.pv.v = xold[(i - r0) * LPR + l];
                    }
#pragma unroll
                    for (int q = 0; q < N; ++q) sum.e[q] = T(0);
#pragma unroll
                    for (int u = 0; u < kLzChunk; ++u) {
                        const T av = e.val(u);
#pragma unroll
                        for (int q = 0; q < N; ++q) sum.e[q] = fma(av, u < kNear ? x[u].e[q] : f.x[u - kNear].e[q], sum.e[q]);
                    }
                    if (ok) finish(i, sum, f.pv, x[0], d);  // entry 0 is the row's own value
                };
                if constexpr (RES && LPR >= 4) {
                    E ea, eb, na, nb;
                    entry(0, ea);
                    entry(1, eb);
                    entry(2, na);
                    entry(3, nb);
                    Ahead fa, fb;
                    ahead(0, ea, fa);
                    ahead(1, eb, fb);
                    for (int t = 0; t < nt; t += 2) {
                        E ma, mb;
                        entry(t + 4, ma);
                        entry(t + 5, mb);
                        Ahead ga, gb;
                        ahead(t + 2, na, ga);
                        ahead(t + 3, nb, gb);
                        T d[N];
    #pragma unroll
                        for (int q = 0; q < N; ++q) d[q] = T(0);
                        row(t, ea, fa, d);
                        row(t + 1, eb, fb, d);
    #pragma unroll
                        for (int q = 0; q < N; ++q) acc[q].add(d[q]);
                        ea = na;
                        eb = nb;
                        na = ma;
                        nb = mb;
                        fa = ga;
                        fb = gb;
                    }
                } else {  // narrow tiles hold more entries per lane: one row at a time
                    E e, ne;
                    entry(0, e);
                    for (int t = 0; t < nt; ++t) {
                        entry(t + 1, ne);
                        Ahead f;
                        ahead(t, e, f);
                        T d[N];
#pragma unroll
                        for (int q = 0; q < N; ++q) d[q] = T(0);
                        row(t, e, f, d);
#pragma unroll
                        for (int q = 0; q < N; ++q) acc[q].add(d[q]);
                        e = ne;
                    }
                }
            } else {
                for (int t = 0; t < nt; ++t) {
                    const int i = row_of(t);
                    if (i >= rend) continue;
                    LzPack<T> sum, pv, ov;
#pragma unroll
                    for (int q = 0; q < N; ++q) sum.e[q] = pv.e[q] = T(0);
                    if (j > 1) pv.v = up[(size_t)i * LPR];
                    ov.v = uj[(size_t)i * LPR];
                    const int c1 = __ldg(app + i + 1);
                    for (int cc = __ldg(app + i); cc < c1; cc += kLzChunk) {
                        int jc[kLzChunk];
                        T ac[kLzChunk];
                        lz_entries<T>(ent, cc, jc, ac);
                        LzPack<T> x[kLzChunk];
#pragma unroll
                        for (int u = 0; u < kLzChunk; ++u) {
#pragma unroll
                            for (int q = 0; q < N; ++q) x[u].e[q] = T(0);
                            if (jc[u] >= 0) x[u].v = uj[(size_t)jc[u] * LPR];
                        }
#pragma unroll
                        for (int u = 0; u < kLzChunk; ++u)
#pragma unroll
                            for (int q = 0; q < N; ++q) sum.e[q] = fma(ac[u], x[u].e[q], sum.e[q]);
                    }
                    T d[N];
#pragma unroll
                    for (int q = 0; q < N; ++q) d[q] = T(0);
                    finish(i, sum, pv, ov, d);
#pragma unroll
                    for (int q = 0; q < N; ++q) acc[q].add(d[q]);
                }
            }
            if (!team_total(acc, 0)) return;
            if (mail[1]) break;  // every pair of the tile stopped at step j - 1 or before (uniform in the team)
            if (tid < COLS) {
                const T al = (T)red[tid].value();
                s_al[tid] = al;
                if (c == 0) al_g[(size_t)j * COLS + tid] = (double)al;
            }
            __syncthreads();
            k = j;
            if (j == a.maxit) break;
            // ---- B(j)
            T ai[N];
#pragma unroll
            for (int q = 0; q < N; ++q) {
                ai[q] = s_al[l * N + q] * inv[q];
                acc[q] = S();
            }
            constexpr int U = 4;  // rows in flight per thread
            for (int t0 = 0; t0 < nt; t0 += U) {
                LzPack<T> s[U], ov[U];
                T d[N];
#pragma unroll
                for (int q = 0; q < N; ++q) d[q] = T(0);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = row_of(t0 + u);
                    if (t0 + u < nt && i < rend) {
                        s[u].v = RES ? xold[(i - r0) * LPR + l] : sj[(size_t)i * LPR];
                        ov[u].v = RES ? xcur[(i - r0) * LPR + l] : uj[(size_t)i * LPR];
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = row_of(t0 + u);
                    if (t0 + u < nt && i < rend) {
#pragma unroll
                        for (int q = 0; q < N; ++q) {
                            s[u].e[q] = fma(-ai[q], ov[u].e[q], s[u].e[q]);
                            d[q] = fma(s[u].e[q], s[u].e[q], d[q]);
                        }
                        sj[(size_t)i * LPR] = s[u].v;
                        if (RES) xold[(i - r0) * LPR + l] = s[u].v;
                    }
                }
#pragma unroll
                for (int q = 0; q < N; ++q) acc[q].add(d[q]);
            }
            if (RES) {
                V* x = xcur;
                xcur = xold;
                xold = x;
            }
            if (!team_total(acc, 1)) return;
            if (tid < COLS) {
                const double b2 = red[tid].value();
                const T b = (T)sqrt(b2);
                const T iv = s_inv[tid];
                const bool fine = b > T(sizeof(T) == 4 ? 1e-37 : 1e-300);
                s_bt[tid] = b * iv;  // beta_{j+1} / beta_j
                s_inv[tid] = fine ? T(1) / b : T(0);
                if (c == 0) bt_g[(size_t)j * COLS + tid] = (double)b;
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < N; ++q) {
                cb[q] = s_bt[l * N + q];
                inv[q] = s_inv[l * N + q];
            }
            // ---- check: the next pivot and residual of every pair of the tile
            if (c == 0) {
                int more = 0;
                for (int pr = tid; pr < npair; pr += kLzThreads) {
                    if (kst[pr] >= 0) continue;
                    const int cl = pr % COLS;
                    const LzPair<T> st = pst[pr];
                    const T bn = (T)bt_g[(size_t)j * COLS + cl], bj = (T)bt_g[(size_t)(j - 1) * COLS + cl];
                    T dr = (T)(st.zr - (double)s_al[cl]), di = st.zi;
                    if (j > 1) {
                        const T w = sizeof(T) == 8 ? bj * bj * st.rd : bj * bj / (st.re * st.re + st.im * st.im);
                        dr -= w * st.re;
                        di += w * st.im;
                    }
                    const T dd = dr * dr + di * di;
                    const T rd = sizeof(T) == 8 ? T(1) / dd : T(0);
                    const T f2 = st.f2 * (sizeof(T) == 8 ? bn * bn * rd : bn * bn / dd);
                    if (!(dd > T(0)) || !isfinite(f2)) {
                        kst[pr] = j - 1;  // no usable step: keep the last iterate
                    } else if ((double)f2 <= a.tol2) {
                        kst[pr] = j;
                    } else {
                        pst[pr] = {st.zr, st.zi, dr, di, f2, rd};
                        more = 1;
                    }
                }
                more = __syncthreads_or(more);
                if (tid == 0 && !more) mail[1] = 1;
            }
        }

        // ---- stop steps of the pairs still iterating; iteration counts
        if (c == 0) {
            for (int pr = tid; pr < npair; pr += kLzThreads) {
                int ks = kst[pr];
                if (ks < 0) {
                    kst[pr] = ks = k;
                    if (a.capped) atomicAdd(a.capped, 1);
                }
                atomicMax(a.iter_max + (size_t)un.x * a.nbatch + (pr / COLS) / a.nbp, max(ks, 1));
            }
            if (tid == 0 && a.work) atomicAdd(a.work, (unsigned long long)k);
        }
        if (!team_sync(bar, target, nc, a.err, a.limit)) return;

        // ---- solve: warp per column, lane per node (chunks of nl nodes)
        for (int cl = warp * nc + c; cl < COLS; cl += nc * kLzWarps) {  // spread over the SMs: FP64 is scarce
            const int m = g * COLS + cl;
            double2* pv = piv + (size_t)cl * a.nl * a.maxit;
            const double b1 = bt_g[cl];
            for (int e0 = 0; e0 < a.ne; e0 += a.nl) {
                const int e = e0 + lane;
                const bool mine = lane < a.nl && e < a.ne;
                const int ks = mine ? kst[e * COLS + cl] : 0;
                double zr = 0.0, zi = 1.0, cr = 0.0, ci = 0.0;
                if (mine && m < m0) {
                    zr = P.zw[4 * e];
                    zi = P.zw[4 * e + 1];
                    const double wr = P.zw[4 * e + 2], wi = P.zw[4 * e + 3];
                    cr = wr;
                    ci = wi;
                    if (a.rii) {
                        const double dr = zr - P.lam[m], d2 = dr * dr + zi * zi;
                        cr = (wr * dr + wi * zi) / d2;
                        ci = (wi * dr - wr * zi) / d2;
                    }
                    const double zs = s_zs;  // (z - A)^{-1} = zs (zs z - zs A)^{-1}
                    zr *= zs;
                    zi *= zs;
                    cr *= zs;
                    ci *= zs;
                }
                int kmax = ks;
                for (int o = 16; o > 0; o >>= 1) kmax = max(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
                // reciprocal UL pivots w_j = 1 / (z - alpha_j - beta_{j+1}^2 w_{j+1}), last step first
                double2 w = make_double2(0.0, 0.0);
                double al = kmax > 0 ? al_g[(size_t)kmax * COLS + cl] : 0.0, bn = 0.0;
                for (int j = kmax; j >= 1; --j) {
                    // the next step's coefficients load behind this step's arithmetic
                    const double al2 = j > 1 ? al_g[(size_t)(j - 1) * COLS + cl] : 0.0, bn2 = bt_g[(size_t)(j - 1) * COLS + cl];
                    if (j <= ks) {
                        const double b2 = j < ks ? bn * bn : 0.0;
                        const double dr = zr - al - b2 * w.x, di = zi - b2 * w.y;
                        const double r = 1.0 / (dr * dr + di * di);
                        w = make_double2(dr * r, -di * r);
                        pv[(size_t)(j - 1) * a.nl + lane] = w;
                    }
                    al = al2;
                    bn = bn2;
                }
                // u_1 = beta_1 w_1, u_{j+1} = beta_{j+1} w_{j+1} u_j; g_j = sum_e Re(c_e u_j)
                double2 u = make_double2(b1, 0.0);
                constexpr int kAhead = 4;  // steps loaded ahead
                double2 wq[kAhead];
                double bq[kAhead];
                auto ahead = [&](int j, int q) {
                    bq[q] = j <= k ? bt_g[(size_t)(j - 1) * COLS + cl] : 0.0;
                    wq[q] = j <= ks ? pv[(size_t)(j - 1) * a.nl + lane] : make_double2(0.0, 0.0);
                };
#pragma unroll
                for (int q = 0; q < kAhead; ++q) ahead(1 + q, q);
                for (int j0 = 1; j0 <= k; j0 += kAhead) {
#pragma unroll
                    for (int q = 0; q < kAhead; ++q) {
                        const int j = j0 + q;
                        const double2 wj = wq[q];
                        const double bj = bq[q], s = j > 1 ? bj : 1.0;
                        ahead(j + kAhead, q);
                        double v = 0.0;
                        if (j <= ks) {
                            const double ur = s * (wj.x * u.x - wj.y * u.y), ui = s * (wj.x * u.y + wj.y * u.x);
                            u = make_double2(ur, ui);
                            v = cr * ur - ci * ui;
                        }
                        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                        if (lane == 0 && j <= k) {
                            const double gv = bj > 0.0 ? v / bj : 0.0;  // coefficient of u_j = beta_j v_j
                            T* gp = g_g + (size_t)(j - 1) * COLS + cl;
                            *gp = (T)(e0 ? (double)*gp + gv : gv);
                        }
                    }
                }
            }
        }
        if (!team_sync(bar, target, nc, a.err, a.limit)) return;

        // ---- combine
        if (c == 0 && tid == 0) mail[0] = a.nteams + (int)atomicAdd(a.queue, 1u);  // the team's next unit
        double rq[N];
#pragma unroll
        for (int q = 0; q < N; ++q) {
            rq[q] = 0.0;
            if (a.rii && col0 + q < mk) {
                const double lm = P.lam[col0 + q];
                for (int f = 0; f < a.ne; ++f) {
                    const double fr = P.zw[4 * f] - lm, fi = P.zw[4 * f + 1];
                    rq[q] += (P.zw[4 * f + 2] * fr + P.zw[4 * f + 3] * fi) / (fr * fr + fi * fi);
                }
            }
        }
        auto put = [&](int i, const LzPack<T>& sum) {
#pragma unroll
            for (int q = 0; q < N; ++q)
                if (col0 + q < m0) {
                    const size_t o = elem(i, col0 + q);
                    double v = 0.0;
                    if (col0 + q < mk) v = (a.rii ? rq[q] * a.X[o] : 0.0) + (double)sum.e[q];
                    a.Q[o] = v;
                }
        };
        for (int t = 0; t < nt; t += 2) {  // two rows share the coefficients' loads
            const int ia = row_of(t), ib = row_of(t + 1);
            const bool okb = t + 1 < nt && ib < rend;
            if (ia >= rend) continue;
            LzPack<T> sa, sb;
#pragma unroll
            for (int q = 0; q < N; ++q) sa.e[q] = sb.e[q] = T(0);
            const V* ua = basis + (size_t)ia * LPR + l;
            const V* ub = basis + (size_t)(okb ? ib : ia) * LPR + l;
            const V* g0 = (const V*)g_g + l;
#pragma unroll(RES ? 8 : 4)
            for (int j = 0; j < k; ++j) {
                LzPack<T> xa, xb, gv;
                xa.v = ua[(size_t)j * sv];
                xb.v = ub[(size_t)j * sv];
                gv.v = g0[(size_t)j * LPR];
#pragma unroll
                for (int q = 0; q < N; ++q) {
                    // a column that stopped has no coefficient: its later vectors may hold anything
                    sa.e[q] = gv.e[q] != T(0) ? fma(gv.e[q], xa.e[q], sa.e[q]) : sa.e[q];
                    sb.e[q] = gv.e[q] != T(0) ? fma(gv.e[q], xb.e[q], sb.e[q]) : sb.e[q];
                }
            }
            put(ia, sa);
            if (okb) put(ib, sb);
        }
        if (!team_sync(bar, target, nc, a.err, a.limit)) return;  // the basis may be overwritten now
        if (tid == 0) s_unit = mail[0];
        __syncthreads();
        unit = s_unit;
    }
}

// ---------------------------------------------------------------- packed rows
// *wide: rows that need more than eight entries (their own row's included,
// stored or not).  *amax: the largest |v| (the bits of doubles >= 0 are ordered
// as they are; a NaN comes out as one).
__global__ void __launch_bounds__(256) krylov_scan(int n, const int* __restrict__ ia, const int* __restrict__ ja, int* wide,
                                                   int parts, const double* __restrict__ v, unsigned long long* amax)
{
    unsigned long long most = 0;
    const size_t end = (size_t)ia[n] * parts;  // not all that the arrays may hold
    for (size_t p = (size_t)ia[0] * parts + blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < end;
         p += (size_t)gridDim.x * blockDim.x) {
        const unsigned long long x = (unsigned long long)__double_as_longlong(fabs(v[p]));
        if (x > most) most = x;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, most, o);
        if (x > most) most = x;
    }
    __shared__ unsigned long long s_most[8];
    if ((threadIdx.x & 31) == 0) s_most[threadIdx.x >> 5] = most;
    __syncthreads();
    if (threadIdx.x == 0) {  // atomics on one address queue up: one per CTA
        for (int i = 1; i < 8; ++i) most = max(most, s_most[i]);
        if (most > *(volatile unsigned long long*)amax) atomicMax(amax, most);
    }
    if (!ja) return;
    int w = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int p0 = ia[i], len = ia[i + 1] - p0;
        bool own = len > kLzChunk;
        for (int p = 0; p < len && !own; ++p) own = ja[p0 + p] == i;
        w |= len + (own ? 0 : 1) > kLzChunk;
    }
    if (__syncthreads_or(w) && threadIdx.x == 0) *wide = 1;
}

cudaError_t launch_krylov_scan(int n, int nnz, const int* ia, const int* ja, int* wide, int parts, const double* v, double* amax,
                               cudaStream_t s)
{
    const int grid = (int)std::max(1LL, std::min<long long>((std::max(n, nnz) + 255LL) / 256, num_sms() * 2));
    krylov_scan<<<grid, 256, 0, s>>>(n, ia, ja, wide, parts, v, (unsigned long long*)amax);
    count_launches(1);
    return cudaGetLastError();
}

// Rows of at most eight entries as eight packed (position, value) entries at
// 8 i: the own row first (value 0 when not stored), the neighbours inside the
// row's range of rpc rows from the front, the others from the end backwards,
// padding (position -1, value 0) between; values multiplied by the filter's
// scale.  The last kLzFar positions are rows;
// the others are rows relative to the range when all of them lie in it, else
// (and for rpc 0) rows, and the own position is stored as ~row to say so.
// Eight threads per row.
template <typename E>
__global__ void __launch_bounds__(256) krylov_pack(int n, int rpc, const int* __restrict__ ia, const int* __restrict__ ja,
                                                   const double* __restrict__ av, const double* __restrict__ amax,
                                                   E* __restrict__ out)
{
    const double sc = krylov_scale(*amax);
    const int l = threadIdx.x & 7;
    const unsigned mine = 0xffu << (threadIdx.x & 24);
    for (int i0 = blockIdx.x * (blockDim.x / 8); i0 < n; i0 += gridDim.x * (blockDim.x / 8)) {
        const int i = i0 + threadIdx.x / 8;
        if (i >= n) continue;  // whole groups of eight
        const int lo = rpc > 0 ? i / rpc * rpc : 0, p0 = ia[i], len = ia[i + 1] - p0;
        const int jj = l < len ? ja[p0 + l] : -1;
        const double v = l < len ? av[p0 + l] * sc : 0.0;
        const unsigned has = __ballot_sync(mine, jj == i) & mine;
        const int d = has ? (__ffs(has) - 1) & 7 : -1;  // the own row's (first) entry
        const bool near = jj >= 0 && l != d && rpc > 0 && (unsigned)(jj - lo) < (unsigned)rpc;
        const bool far = jj >= 0 && l != d && !near;
        const unsigned nb = (__ballot_sync(mine, near) & mine) >> (threadIdx.x & 24);
        const unsigned fb = (__ballot_sync(mine, far) & mine) >> (threadIdx.x & 24);
        const unsigned below = (1u << l) - 1u;
        const int nn = __popc(nb), nf = __popc(fb);
        const bool local = rpc > 0 && nf <= kLzFar;
        E* o = out + (size_t)i * kLzChunk;
        auto put = [&](int at, int row, double val) {
            const int pos = row < 0 ? -1 : (at >= kLzChunk - kLzFar ? row : (local ? row - lo : (at ? row : ~row)));
            if constexpr (sizeof(E) == 8) o[at] = make_int2(pos, __float_as_int((float)val));
            else o[at] = make_int4(pos, 0, __double2loint(val), __double2hiint(val));
        };
        if (l == d || (d < 0 && l == 0)) put(0, i, d >= 0 ? v : 0.0);
        if (near) put(1 + __popc(nb & below), jj, v);
        if (far) put(kLzChunk - 1 - __popc(fb & below), jj, v);
        if (l > nn && l < kLzChunk - nf) put(l, -1, 0.0);
    }
}

cudaError_t launch_krylov_pack(int n, int rpc, const int* ia, const int* ja, const double* av, const double* amax, bool fp64,
                               void* out, cudaStream_t s)
{
    const int grid = std::max(1, std::min((n + 31) / 32, num_sms() * 16));
    if (fp64) krylov_pack<int4><<<grid, 256, 0, s>>>(n, rpc, ia, ja, av, amax, (int4*)out);
    else krylov_pack<int2><<<grid, 256, 0, s>>>(n, rpc, ia, ja, av, amax, (int2*)out);
    count_launches(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- complex Hermitian matrices
// Lanczos on a Hermitian A has real coefficients, so it is real Lanczos on the
// real symmetric operator that takes (Re x, Im x) to (Re A x, Im A x).  Rows 2 i
// and 2 i + 1 of that operator hold row i's entries as (2 j, Re a), (2 j + 1,
// -Im a) and (2 j, Im a), (2 j + 1, Re a), padded to chunks of eight at pp.
template <typename E, typename V2>
__global__ void __launch_bounds__(256) krylov_pack_hermitian(int n, const int* __restrict__ ia, const int* __restrict__ ja,
                                                             const V2* __restrict__ av, const int* __restrict__ pp,
                                                             const double* __restrict__ amax, E* __restrict__ out)
{
    const double sc = krylov_scale(*amax);
    const int lane = threadIdx.x & 31, nw = (gridDim.x * blockDim.x) >> 5;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += nw) {
        const int p0 = ia[i], len = ia[i + 1] - p0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c0 = pp[2 * i + h], c1 = pp[2 * i + h + 1];
            for (int t = c0 + lane; t < c1; t += 32) {
                const int q = (t - c0) >> 1, im = (t - c0) & 1;
                int j = -1;
                double v = 0.0;
                if (q < len) {
                    j = 2 * ja[p0 + q] + im;
                    const V2 a = av[p0 + q];
                    v = sc * (im == h ? (double)a.x : (h ? (double)a.y : -(double)a.y));
                }
                if constexpr (sizeof(E) == 8) out[t] = make_int2(j, __float_as_int((float)v));
                else out[t] = make_int4(j, 0, __double2loint(v), __double2hiint(v));
            }
        }
    }
}

cudaError_t launch_krylov_pack_hermitian(int n, const int* ia, const int* ja, const double2* av, const int* pp,
                                         const double* amax, bool fp64, void* out, cudaStream_t s)
{
    const int grid = std::max(1, std::min((n + 7) / 8, num_sms() * 16));
    if (fp64) krylov_pack_hermitian<int4><<<grid, 256, 0, s>>>(n, ia, ja, av, pp, amax, (int4*)out);
    else krylov_pack_hermitian<int2><<<grid, 256, 0, s>>>(n, ia, ja, av, pp, amax, (int2*)out);
    count_launches(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- plan and launch
int krylov_rows(int n, int nc) { return krylov_rpc(n, nc); }

int krylov_item_rows(const KrylovPlan& k) { return k.resident ? 32 / k.lanes : kLzBlock; }

// Bytes of Krylov bases that the teams of a pass may hold together: the number of
// tiles taken at once is limited by it, one team has what it needs whatever that
// is.  At 64^3 with 150 columns (2.7 GB a tile) all five tiles at once measured 21
// to 24 ms a pass, one after the other 27; the limit lies just above those five.
static constexpr double kKrylovMany = 16e9;

// Microseconds of one step of a tile of an n-row problem, by the measured parts of a step on
// GB300: a pass of 512 lanes through both phases (resident 1.2, cached 2.9 with
// two CTAs per SM, each times 4 in FP64), and the two sums of a step (2.2 within
// a CTA; 6 across a team and more with its size).
static double krylov_tile_cost(const KrylovPlan& k, bool fp64, int n)
{
    const int rows = k.resident ? krylov_rpc(n, k.nc) : ((n + kLzBlock - 1) / kLzBlock + k.nc - 1) / k.nc * kLzBlock;
    const double passes = std::ceil((double)rows * k.lanes / kLzThreads);
    return 1.8 + passes * (k.resident ? 1.2 : 2.9) * (fp64 ? 4.0 : 1.0) + (k.nc == 1 ? 2.2 : 6.0 + 0.035 * k.nc);
}

// Steps a problem of n rows may take: its Krylov spaces have at most n
// dimensions, and a pair that eight times as many steps (and a thousand) have not
// brought to its tolerance is at its rounding level.  Without this a cap that
// stands for "none" (fpm(46) = 10^6) planned 17 GB for 100 rows and mapped them in
// every filter call (36 ms; now 0.03 GB and 1.5, one COCG per node takes 8.1).
static int krylov_steps(int n, int maxit) { return (int)std::min<long long>(maxit, 8LL * n + 1000); }

// The parts of a plan that follow from its width, for problems of at most n rows.
static double krylov_size(KrylovPlan& k, bool fp64, int lanes, int n, int ne, int maxit)
{
    maxit = krylov_steps(n, maxit);
    k.lanes = lanes;
    k.cols = lanes * (fp64 ? 2 : 4);
    k.nl = std::min(ne, 32);
    k.maxit = maxit;
    k.ne = ne;
    k.slot_vecs = (size_t)n * lanes;
    k.team_bytes = ((size_t)maxit + 1) * k.slot_vecs * 16;
    return (double)k.team_bytes + (double)k.cols * k.nl * 16.0 * maxit + (double)k.cols * (24.0 * maxit + 52.0 * ne);
}

KrylovPlan krylov_plan(bool fp64, bool resident, int n, int m, int ne, int maxit, double max_bytes)
{
    KrylovPlan best;
    const int sms = num_sms(), ctas = resident ? sms : 2 * sms;
    for (int lanes = kLzMaxLanes; lanes >= 1; lanes /= 2) {
        if (!resident && lanes != kLzMaxLanes) break;
        KrylovPlan k;
        k.resident = resident;
        const double per_team = krylov_size(k, fp64, lanes, n, ne, maxit);
        if (per_team > max_bytes) continue;
        const int units = (m + k.cols - 1) / k.cols;
        const int fit = (int)std::max(1.0, kKrylovMany / per_team);
        for (int t = 1; t <= std::min({units, fit, sms}); ++t)
            for (const bool one : {true, false}) {  // one CTA per team, or as many as there are
                k.teams = t;
                k.nc = one ? 1 : std::max(1, std::min(ctas / t, (n + 63) / 64));
                k.rpc = resident ? krylov_rpc(n, k.nc) : 0;
                if ((size_t)k.rpc * lanes * 32 > kLzSmem) continue;
                k.cost = ((units + t - 1) / t) * krylov_tile_cost(k, fp64, n);
                if (best.teams == 0 || k.cost < best.cost) best = k;
            }
    }
    return best;
}

// Plan for a set of problems (np of them, n[i] rows and m[i] columns) whose
// tiles the teams take from one queue; teams = 0 when the largest does not fit.
KrylovPlan krylov_plan_set(bool fp64, bool resident, int np, const int* n, const int* m, int ne, int maxit, double max_bytes)
{
    KrylovPlan best;
    const int ctas = resident ? num_sms() : 2 * num_sms(), maxn = *std::max_element(n, n + np);
    for (int lanes = kLzMaxLanes; lanes >= 1; lanes /= 2) {
        if (!resident && lanes != kLzMaxLanes) break;
        KrylovPlan k;
        k.resident = resident;
        const double per_team = krylov_size(k, fp64, lanes, maxn, ne, maxit);
        if (per_team > max_bytes) continue;
        long long units = 0;
        for (int i = 0; i < np; ++i) units += (m[i] + k.cols - 1) / k.cols;
        for (k.nc = 1; k.nc <= ctas; k.nc *= 2) {
            k.rpc = resident ? krylov_rpc(maxn, k.nc) : 0;
            if ((size_t)k.rpc * lanes * 32 > kLzSmem) continue;
            k.teams = (int)std::min<double>({(double)(ctas / k.nc), (double)units, std::max(1.0, max_bytes / per_team)});
            double sum = 0.0, longest = 0.0;
            for (int i = 0; i < np; ++i) {
                const double us = krylov_tile_cost(k, fp64, n[i]);
                sum += us * ((m[i] + k.cols - 1) / k.cols);
                longest = std::max(longest, us);
            }
            k.cost = std::max(longest, sum / k.teams + 0.5 * longest);
            if (best.teams == 0 || k.cost < best.cost) best = k;
        }
    }
    return best;
}

// The plan's device memory from base (nullptr: only the size), 256-byte aligned pieces.
size_t krylov_layout(const KrylovPlan& k, char* base, KrylovArgs& a)
{
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* p = base ? base + off : nullptr;
        off += (bytes + 255) & ~(size_t)255;
        return p;
    };
    const size_t nt = k.teams, mi = k.maxit;
    a.nteams = k.teams;
    a.nc = k.nc;
    a.ne = k.ne;
    a.nl = k.nl;
    a.maxit = k.maxit;
    a.slot_vecs = k.slot_vecs;
    a.team_bytes = k.team_bytes;
    a.basis = take(nt * k.team_bytes);
    a.part = take(nt * 2 * k.nc * k.cols * 8);
    a.coef = (double*)take(nt * 2 * (mi + 2) * k.cols * sizeof(double));
    a.g = take(nt * mi * k.lanes * 16);
    a.pair = take(nt * k.cols * k.ne * sizeof(LzPair<double>));
    a.kstop = (int*)take(nt * k.cols * k.ne * sizeof(int));
    a.piv = (double2*)take(nt * k.cols * k.nl * mi * sizeof(double2));
    a.bar = (unsigned*)take((nt + 1) * 128);  // team counters, then the unit queue
    a.mail = (int*)take(nt * 128);
    a.queue = a.bar ? a.bar + nt * 32 : nullptr;
    return off;
}

size_t krylov_smem(int rpc, int lanes) { return (size_t)rpc * lanes * 32; }

template <typename T, int LPR, bool RES>
static cudaError_t krylov_launch(KrylovArgs a, int grid, size_t smem, cudaStream_t s)
{
    auto kern = krylov_filter<T, LPR, RES>;
    if (smem > 0) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kLzSmem);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {&a};
    count_launches(1);
    return cudaLaunchCooperativeKernel((void*)kern, dim3(grid), dim3(kLzThreads), args, smem, s);
}

template <typename T>
static cudaError_t krylov_launch_t(const KrylovArgs& a, int lanes, bool resident, int grid, size_t smem, cudaStream_t s)
{
    if (!resident) return krylov_launch<T, kLzMaxLanes, false>(a, grid, 0, s);
    switch (lanes) {
    case 8: return krylov_launch<T, 8, true>(a, grid, smem, s);
    case 4: return krylov_launch<T, 4, true>(a, grid, smem, s);
    case 2: return krylov_launch<T, 2, true>(a, grid, smem, s);
    default: return krylov_launch<T, 1, true>(a, grid, smem, s);
    }
}

cudaError_t launch_krylov_filter(const KrylovArgs& a, const KrylovPlan& p, bool fp64, cudaStream_t s)
{
    const int grid = a.nteams * a.nc;
    const size_t smem = krylov_smem(p.rpc, p.lanes);
    return fp64 ? krylov_launch_t<double>(a, p.lanes, p.resident, grid, smem, s)
                : krylov_launch_t<float>(a, p.lanes, p.resident, grid, smem, s);
}

}  // namespace feast
