// Reduced dense eigensolver of the Rayleigh-Ritz step (FEAST v4.0 guide,
// Sec. 1.1: the reduced problem is a small dense generalized symmetric
// eigenproblem A_Q v = lambda B_Q v, solved in FP64).
//
// Symmetric eigen-decomposition: two-sided cyclic Jacobi with the
// round-robin ("circle method") pair ordering, so each round rotates mp/2
// disjoint pairs at once.  Rotation of the pair (p,q) (Golub & Van Loan,
// symmetric Schur decomposition): tau = (a_qq - a_pp)/(2 a_pq),
// t = sign(tau)/(|tau| + sqrt(1+tau^2)), c = 1/sqrt(1+t^2), s = t c, and
// A <- J^T A J with J = [[c, s], [-s, c]] on columns (p, q).  Applying J_k^T
// on the left and J_l on the right of every 2x2 block (k,l) at once lets one
// thread update one block with no further synchronisation.
//
// GB300 has little FP64 throughput per SM, so the rounds are spread over many
// CTAs of one cooperative launch, with one grid barrier per round; the
// barrier spins on a global counter with a clock-based time limit and raises
// an error flag instead of hanging.
//
// Generalized problem, first route: D = diag(B_Q)^{-1/2}, D B_Q D = L L^T
// (one-CTA Cholesky), S = D L^{-T}, Jacobi on S^T A_Q S = W Lambda W^T,
// V = S W.  Taken when every pivot is positive and ||L^{-1}||_F^2 <= 1e8.
// Second route (B_Q singular or ill conditioned):
// D = diag(B_Q)^{-1/2}, Jacobi on D B_Q D = U diag(d) U^T,
// keep d_i > 1e-14 max d, S = D U_k diag(d_k)^{-1/2}, Jacobi on S^T A_Q S =
// W Lambda W^T, V = S W (V^T B_Q V = I).  Dropped directions stay in the
// m x m arrays as exact zero columns of S and get a sentinel eigenvalue, so
// they sort last and the live count mk is the number of non-sentinel values.
#include <atomic>

#include <algorithm>

#include "chol.cuh"
#include "feast_internal.cuh"
#include "team.cuh"

namespace feast {

static constexpr double kSentinel = 1e300;
static constexpr int kMaxSweeps = 60;
static constexpr int kEigThreads = 256;

static constexpr int kMaxHalf = 4096;  // m <= 8192

struct JacWork {
    unsigned count;  // barrier arrivals
    int err;
    int sweeps;
    int status;
    int again[2];  // a sweep left an entry above the threshold
};

struct JacTask {
    int m;
    double *A, *A2, *V, *lam, *Vout;
};
struct JacArgs {
    const BProb* pr;  // batch: the problems, their work areas and Ritz values
    double *bwork, *blam;
    JacTask one;
    int ntask, nteams, nc;
    JacWork* work;  // [nteams], zeroed
    long long limit;
};

// Spin limit of the barriers in SM clock cycles (about two seconds at
// 2 GHz); feast_set_wait_limit changes it for the launches that follow.
static constexpr long long kDefaultSpinCycles = 4000000000LL;
static std::atomic<long long> g_spin_cycles{kDefaultSpinCycles};
long long wait_limit_cycles() { return g_spin_cycles.load(); }

// round-robin partner table: slot 0 holds player 0, slot s >= 1 holds
// player 1 + ((s - 1 + r) mod (mp - 1)); pair k is (slot k, slot mp-1-k)
__device__ __forceinline__ int rr_player(int slot, int r, int mp)
{
    const int x = slot + r;  // r < mp - 1
    return slot == 0 ? 0 : (x < mp ? x : x - (mp - 1));
}

// Rotation of the pair (p, q): t near the smaller root of
// f(t) = b t^2 + d t - b, b = apq, d = aqq - app (scaled near 1): the root in
// single precision and one Newton step in FP64 (about 1e-13 of b is left), and
// c = 1 / sqrt(1 + t^2), s = t c to FP64 (a single-precision seed and the
// first two terms of the binomial series), so the rotation is orthogonal to rounding although it leaves
// -c^2 f(t) in the place of apq.  Twelve FP64 operations instead of two
// divisions and two square roots, which held every round up while all CTAs
// computed all angles.
__device__ __forceinline__ void jac_rotation(double d, double b, double& c, double& s, double& t)
{
    const float df = (float)d, bf = (float)b, h = 0.5f * df;
    const float x = df == 0.0f ? 1.0f : copysignf(1.0f, h) * (bf / (fabsf(h) + sqrtf(fmaf(h, h, bf * bf))));
    t = (double)x;
    t = fma(-fma(fma(b, t, d), t, -b), (double)(1.0f / fmaf(2.0f * bf, x, df)), t);
    const double y = fma(t, t, 1.0);
    const double r = (double)rsqrtf((float)y);
    const double e = fma(-y * r, r, 1.0);
    c = fma(r * e, fma(0.375, e, 0.5), r);
    s = t * c;
}

// Cyclic Jacobi of one matrix by a team of CTAs, one barrier per round: every
// CTA computes all mp/2 rotations of the round itself (identical inputs and
// code, so identical angles) into shared memory, then its share of the 2x2
// blocks from the current copy of A into the other copy, so no CTA writes what
// another still reads.  Of two blocks that mirror each other one is computed
// and written twice.  A round is a chain of latencies (at m = 150 with 90 CTAs
// 1.2 us of loads and angles, 1.2 the blocks, 1.7 the barrier; FP64
// operations take some 100 cycles one after the other): the entries of a
// thread's first block and of its first pair of V load together with those of
// the angles, its place in the round's table is worked out once, and V, whose
// rows belong to one CTA each, is updated between the CTA's arrival at the
// barrier and its wait.  7.7 us a round before, 4.6 with V ahead of the barrier
// (m = 150: 4.79 ms of a reduced problem), 4.1 now (4.44).  A sweep ends with a look for
// entries above the threshold, so no whole sweep is spent on finding none.
// Rotation tables in dynamic shared memory: c, s, t (doubles), p, q (ints).
// Tasks: `one` (pr == nullptr) or the batch's active problems in turn.
__global__ void __launch_bounds__(kEigThreads) jacobi_team(JacArgs a)
{
    extern __shared__ double rsh[];
    __shared__ double sred[kEigThreads];
    const int nc = a.nc, team = blockIdx.x / nc, cta = blockIdx.x - team * nc;
    JacWork* w = a.work + team;
    unsigned target = 0;
    const int gtid = cta * blockDim.x + threadIdx.x, gsz = nc * blockDim.x;
    for (int task = team; task < a.ntask; task += a.nteams) {
        int m = a.one.m;
        double *A = a.one.A, *A2 = a.one.A2, *V = a.one.V, *lam = a.one.lam, *Vout = a.one.Vout;
        if (a.pr) {
            const BProb& P = a.pr[task];
            if (!P.active) continue;
            m = P.m;
            const size_t mm = (size_t)m * m;
            double* W0 = a.bwork + P.w_off;  // layout of b_reduce_prep (k_batch.cu)
            A = W0 + 4 * mm;
            A2 = W0 + mm;
            V = W0 + 5 * mm;
            Vout = W0 + 2 * mm;
            lam = a.blam + P.l_off;
        }
        const int mp = m + (m & 1), half = mp / 2;
        double* rc = rsh;
        double* rs = rc + half;
        double* rt = rs + half;
        int* rp = (int*)(rt + half);
        int* rq = rp + half;
        for (long long idx = gtid; idx < (long long)m * m; idx += gsz) V[idx] = (idx / m == idx % m) ? 1.0 : 0.0;
        double fr = 0.0;  // the largest entry, the same in every CTA
        for (int idx = threadIdx.x; idx < m * m; idx += blockDim.x)
            if (fabs(A[idx]) < 1e299) fr = fmax(fr, fabs(A[idx]));  // sentinels excluded
        sred[threadIdx.x] = fr;
        __syncthreads();
        for (int o = blockDim.x / 2; o > 0; o >>= 1) {
            if (threadIdx.x < o) sred[threadIdx.x] = fmax(sred[threadIdx.x], sred[threadIdx.x + o]);
            __syncthreads();
        }
        const double big = sred[0];
        if (cta == 0 && threadIdx.x == 0) w->again[0] = w->again[1] = 0;
        if (!team_sync(&w->count, target, nc, &w->err, a.limit)) return;
        const double sc = big > 1e-300 && big < 1e300 ? ldexp(1.0, -ilogb(big)) : 1.0;
        // |x| above 1.1e-16 sqrt(|xp xq|) and the floor of 1e-18 of the matrix, all
        // scaled by sc: the largest entry is near 1, nothing under- or overflows
        auto above = [](float x, float xp, float xq) {
            return fabsf(x) > 1e-18f && x * x > 1.21e-32f * fabsf(xp) * fabsf(xq);
        };
        double* cur = A;
        double* nxt = A2;
        // every unordered pair of pairs {k, l} once, with no gaps inside a warp: row
        // k, then l = k + 1, k + 2, ... around the circle; the diagonal blocks, whose
        // arithmetic differs, after all the others
        const int ncol = half / 2, nblk = half * (ncol + 1);
        auto block = [&](int idx, int& k, int& l) {
            if (idx >= half * ncol) {
                k = l = idx - half * ncol;
                return idx < nblk;
            }
            k = idx / ncol;
            const int d = idx - k * ncol + 1;
            l = k + d < half ? k + d : k + d - half;
            return 2 * d < half || k < half / 2;
        };
        auto pair = [&](int k, int r, int& p, int& q) {
            p = rr_player(k, r, mp);
            q = rr_player(mp - 1 - k, r, mp);
            if (p > q) {
                const int t = p;
                p = q;
                q = t;
            }
        };
        // a thread's first block (k, l) and first pair of a row of V
        int k0 = 0, l0 = 0;
        const bool has = block(gtid, k0, l0);
        // V's rows go to the CTAs in turn: no other CTA reads them before the end
        const int vitems = cta < m ? ((m - 1 - cta) / nc + 1) * half : 0;
        const bool hasv = (int)threadIdx.x < vitems;
        const int i0 = cta + (int)threadIdx.x / half * nc, kv0 = (int)threadIdx.x % half;
        int sweep = 0;
        for (; sweep < kMaxSweeps && mp >= 2; ++sweep) {
            for (int r = 0; r < mp - 1; ++r) {
                double x00 = 0.0, x01 = 0.0, x10 = 0.0, x11 = 0.0, vp = 0.0, vq = 0.0;
                auto load = [&](int p, int q, int pp, int qq) {
                    x00 = __ldcg(cur + (size_t)p * m + pp);
                    x01 = qq < m ? __ldcg(cur + (size_t)p * m + qq) : 0.0;
                    x10 = q < m ? __ldcg(cur + (size_t)q * m + pp) : 0.0;
                    x11 = q < m && qq < m ? __ldcg(cur + (size_t)q * m + qq) : 0.0;
                };
                if (has) {
                    int p, q, pp, qq;
                    pair(k0, r, p, q);
                    pair(l0, r, pp, qq);
                    load(p, q, pp, qq);
                }
                if (hasv) {
                    int p, q;
                    pair(kv0, r, p, q);
                    vp = __ldcg(V + (size_t)i0 * m + p);
                    vq = q < m ? __ldcg(V + (size_t)i0 * m + q) : 0.0;
                }
                for (int k = threadIdx.x; k < half; k += blockDim.x) {
                    int p, q;
                    pair(k, r, p, q);
                    double c = 1.0, sn = 0.0, t = 0.0;
                    if (q < m) {
                        const double apq = __ldcg(cur + (size_t)p * m + q);
                        const double app = __ldcg(cur + (size_t)p * m + p), aqq = __ldcg(cur + (size_t)q * m + q);
                        const double b = apq * sc, xp = app * sc, xq = aqq * sc;
                        if (above((float)b, (float)xp, (float)xq)) jac_rotation(xq - xp, b, c, sn, t);
                    }
                    rc[k] = c;
                    rs[k] = sn;
                    rt[k] = t;
                    rp[k] = p;
                    rq[k] = q;
                }
                __syncthreads();
                for (int idx = gtid; idx < nblk; idx += gsz) {
                    int k = k0, l = l0;
                    if (idx == gtid ? !has : !block(idx, k, l)) continue;
                    const int p = rp[k], q = rq[k], pp = rp[l], qq = rq[l];
                    const bool qv = q < m, qqv = qq < m;
                    if (idx != gtid) load(p, q, pp, qq);
                    if (k == l) {
                        // diagonal block, with f(t): app - t apq + c^2 t f, aqq + t apq - c^2 t f, -c^2 f
                        const double t = rt[k];
                        const double e = rc[k] * rc[k] * fma(fma(x01, t, x11 - x00), t, -x01);
                        const double ta = fma(-t, e, t * x01);
                        nxt[(size_t)p * m + p] = x00 - ta;
                        if (qv) {
                            nxt[(size_t)q * m + q] = x11 + ta;
                            nxt[(size_t)p * m + q] = nxt[(size_t)q * m + p] = -e;
                        }
                        continue;
                    }
                    const double ck = rc[k], sk = rs[k], cl = rc[l], sl = rs[l];
                    // rows: new row p = c row p - s row q ; new row q = s row p + c row q
                    const double y00 = ck * x00 - sk * x10, y01 = ck * x01 - sk * x11;
                    const double y10 = sk * x00 + ck * x10, y11 = sk * x01 + ck * x11;
                    // columns: new col p' = c col p' - s col q' ; new col q' = s col p' + c col q'
                    const double z00 = cl * y00 - sl * y01, z01 = sl * y00 + cl * y01;
                    const double z10 = cl * y10 - sl * y11, z11 = sl * y10 + cl * y11;
                    nxt[(size_t)p * m + pp] = z00;
                    nxt[(size_t)pp * m + p] = z00;
                    if (qqv) {
                        nxt[(size_t)p * m + qq] = z01;
                        nxt[(size_t)qq * m + p] = z01;
                    }
                    if (qv) {
                        nxt[(size_t)q * m + pp] = z10;
                        nxt[(size_t)pp * m + q] = z10;
                    }
                    if (qv && qqv) {
                        nxt[(size_t)q * m + qq] = z11;
                        nxt[(size_t)qq * m + q] = z11;
                    }
                }
                team_arrive(&w->count, target, nc);
                for (int idx = threadIdx.x; idx < vitems; idx += blockDim.x) {  // behind the other CTAs' arrivals
                    const bool own = idx == (int)threadIdx.x;
                    const int i = own ? i0 : cta + idx / half * nc, k = own ? kv0 : idx % half;
                    const double sk = rs[k];
                    if (sk == 0.0) continue;
                    const double ck = rc[k];
                    const int p = rp[k], q = rq[k];
                    if (!own) {
                        vp = __ldcg(V + (size_t)i * m + p);
                        vq = __ldcg(V + (size_t)i * m + q);
                    }
                    V[(size_t)i * m + p] = ck * vp - sk * vq;
                    V[(size_t)i * m + q] = sk * vp + ck * vq;
                }
                if (!team_wait(&w->count, target, nc, &w->err, a.limit)) return;
                double* tmp = cur;
                cur = nxt;
                nxt = tmp;
            }
            // entries still above the threshold?
            int more = 0;
            for (int idx = gtid; idx < m * m; idx += gsz) {
                const int i = idx / m, j = idx % m;
                if (j <= i) continue;
                const double x = __ldcg(cur + idx);
                if (above((float)(x * sc), (float)(__ldcg(cur + (size_t)i * m + i) * sc), (float)(__ldcg(cur + (size_t)j * m + j) * sc)))
                    more = 1;
            }
            if (__syncthreads_or(more) && threadIdx.x == 0) w->again[sweep & 1] = 1;
            if (!team_sync(&w->count, target, nc, &w->err, a.limit)) return;
            const int go = *(volatile int*)&w->again[sweep & 1];
            if (!go) break;  // same decision in every CTA
            // the other flag is read next; nobody reads it before the next barrier
            if (cta == 0 && threadIdx.x == 0) *(volatile int*)&w->again[(sweep & 1) ^ 1] = 0;
        }
        // ascending order: rank of each diagonal entry (ties by index)
        double* dg = rsh;  // rotation tables are free: m doubles and m ranks fit
        int* rank = (int*)(dg + mp);
        __syncthreads();
        for (int i = threadIdx.x; i < m; i += blockDim.x) dg[i] = __ldcg(cur + (size_t)i * m + i);
        __syncthreads();
        for (int i = threadIdx.x; i < m; i += blockDim.x) {
            const double li = dg[i];
            int k = 0;
            for (int j = 0; j < m; ++j) k += (dg[j] < li) || (dg[j] == li && j < i);
            rank[i] = k;
            if (cta == 0) lam[k] = li;
        }
        __syncthreads();
        for (long long idx = gtid; idx < (long long)m * m; idx += gsz) {
            const int row = (int)(idx / m), i = (int)(idx % m);
            Vout[(size_t)row * m + rank[i]] = __ldcg(V + idx);
        }
        if (gtid == 0) {
            w->sweeps = sweep;
            w->status = sweep >= kMaxSweeps ? -1 : 0;
        }
        __syncthreads();
    }
}

static size_t rot_smem(int m)
{
    const int half = (m + (m & 1)) / 2;
    return (size_t)half * (3 * sizeof(double) + 2 * sizeof(int));
}

size_t jacobi_work_bytes(int m)
{
    return 1024 + sizeof(JacWork) + 2 * sizeof(double) * (size_t)m * m;
}

// CTAs of a team, within `most`.
static int jacobi_ctas(int m, int most)
{
    // a warp instruction holds the FP64 pipe for 16 cycles, so the blocks are
    // spread until a CTA has few warps of them
    const long long half = (m + 1) / 2, work = half * (half / 2 + 1);
    return (int)std::max(1LL, std::min<long long>((work + 31) / 32, most));
}

static cudaError_t launch_jacobi(JacArgs a, int m, cudaStream_t s)
{
    const size_t smem = rot_smem(m);
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(jacobi_team, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    a.limit = wait_limit_cycles();
    void* args[] = {&a};
    count_launches(1);
    return cudaLaunchCooperativeKernel((void*)jacobi_team, dim3(a.nteams * a.nc), dim3(kEigThreads), args, smem, s);
}

size_t jacobi_batch_bytes(int np) { return sizeof(JacWork) * (size_t)std::min(np, num_sms()); }

cudaError_t launch_jacobi_batch(const BProb* pr, int np, int maxm, double* lam, double* bwork, void* work, cudaStream_t s)
{
    JacArgs a = {};
    a.pr = pr;
    a.ntask = np;
    a.nteams = std::min(np, num_sms());
    a.nc = jacobi_ctas(maxm, num_sms() / a.nteams);
    a.blam = lam;
    a.bwork = bwork;
    a.work = (JacWork*)work;
    const cudaError_t e = cudaMemsetAsync(work, 0, sizeof(JacWork) * a.nteams, s);
    return e != cudaSuccess ? e : launch_jacobi(a, maxm, s);
}

int jacobi_batch_failed(const void* host_work, int np)
{
    const JacWork* w = (const JacWork*)host_work;
    for (int t = 0; t < std::min(np, num_sms()); ++t)
        if (w[t].err) return 1;
    return 0;
}

static char* align256(char* p) { return (char*)(((uintptr_t)p + 255) & ~(uintptr_t)255); }

// A (m x m, row-major) is destroyed; lam ascending; V row-major eigenvectors
// in columns.  m <= 8192 (the rotation tables of a round sit in shared
// memory); larger m returns -3.
int jacobi_eig_dev(int m, double* A, double* lam, double* V, void* work, cudaStream_t s, int* sweeps_host)
{
    if (m > 2 * kMaxHalf) return -3;
    char* p = align256((char*)work);
    JacWork* w = (JacWork*)p;
    p = align256(p + sizeof(JacWork));
    double* A2 = (double*)p;
    p = align256(p + sizeof(double) * (size_t)m * m);
    double* Vw = (double*)p;
    if (cudaMemsetAsync(w, 0, sizeof(JacWork), s) != cudaSuccess) return -3;
    JacArgs a = {};
    a.ntask = a.nteams = 1;
    a.nc = jacobi_ctas(m, num_sms());
    a.one = {m, A, A2, Vw, lam, V};
    a.work = w;
    if (launch_jacobi(a, m, s) != cudaSuccess) return -3;
    if (sweeps_host) {
        JacWork h;
        if (cudaMemcpyAsync(&h, w, sizeof(JacWork), cudaMemcpyDeviceToHost, s) != cudaSuccess) return -3;
        if (cudaStreamSynchronize(s) != cudaSuccess) return -3;
        *sweeps_host = h.sweeps;
        if (h.err) return -2;
        if (h.status) return -1;
    }
    return 0;
}

// ---------------------------------------------------------------- products of the reduced matrices
// C = A B (TA = 0) or A^T B with C symmetric, its part on and above the diagonal
// mirrored (TA = 1); all m x m.  A thread per element, 16 x 16 tiles: about
// (m / 16)^2 CTAs, where the 64 x 64 tiles of the n x m products would leave
// most of the chip idle (m = 150: 200 us, here 14).
template <int TA>
__global__ void __launch_bounds__(256) rg_product(int m, const double* __restrict__ A, const double* __restrict__ B,
                                                  double* __restrict__ C)
{
    __shared__ double sa[16][17], sb[16][17];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int i0 = blockIdx.y * 16, j0 = blockIdx.x * 16;
    if (TA && j0 < i0) return;
    double s = 0.0;
    for (int k0 = 0; k0 < m; k0 += 16) {
        const int ai = TA ? k0 + ty : i0 + ty, aj = TA ? i0 + tx : k0 + tx;
        const double av = ai < m && aj < m ? __ldg(A + (size_t)ai * m + aj) : 0.0;
        if (TA) sa[tx][ty] = av;
        else sa[ty][tx] = av;
        sb[ty][tx] = k0 + ty < m && j0 + tx < m ? __ldg(B + (size_t)(k0 + ty) * m + j0 + tx) : 0.0;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 16; ++k) s = fma(sa[ty][k], sb[k][tx], s);
        __syncthreads();
    }
    const int i = i0 + ty, j = j0 + tx;
    if (i >= m || j >= m || (TA && j < i)) return;
    C[(size_t)i * m + j] = s;
    if (TA) C[(size_t)j * m + i] = s;
}

template <int TA>
static cudaError_t launch_rg_product(int m, const double* A, const double* B, double* C, cudaStream_t s)
{
    const unsigned t = (unsigned)((m + 15) / 16);
    rg_product<TA><<<dim3(t, t), 256, 0, s>>>(m, A, B, C);
    count_launches(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- generalized problem
__global__ void rg_scale(int m, const double* Aq, const double* Bq, double* At, double* Bt, double* dsc)
{
    const long long total = (long long)m * m;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(idx / m), j = (int)(idx % m);
        const double bi = Bq[(size_t)i * m + i], bj = Bq[(size_t)j * m + j];
        const double di = bi > 0.0 ? 1.0 / sqrt(bi) : 0.0, dj = bj > 0.0 ? 1.0 / sqrt(bj) : 0.0;
        Bt[idx] = 0.5 * (Bq[(size_t)i * m + j] + Bq[(size_t)j * m + i]) * di * dj;
        At[idx] = 0.5 * (Aq[(size_t)i * m + j] + Aq[(size_t)j * m + i]);
        if (j == 0) dsc[i] = di;
    }
}

// S[r][c] = dsc[r] U[r][c] / sqrt(d_c) for kept c (d_c > 1e-14 max d), else 0.
__global__ void rg_basis(int m, const double* d, const double* U, const double* dsc, double* S, int* mk)
{
    const double dmax = d[m - 1];
    const long long total = (long long)m * m;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int r = (int)(idx / m), c = (int)(idx % m);
        const bool keep = dmax > 0.0 && d[c] > 1e-14 * dmax;
        S[idx] = keep ? dsc[r] * U[idx] / sqrt(d[c]) : 0.0;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        int k = 0;
        for (int c = 0; c < m; ++c) k += (dmax > 0.0 && d[c] > 1e-14 * dmax);
        *mk = k;
    }
}

// Dropped directions (zero columns of S) get the sentinel on the diagonal.
__global__ void rg_sentinel(int m, const double* S, double* C)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < m; c += gridDim.x * blockDim.x) {
        bool zero = true;
        for (int r = 0; r < m && zero; ++r) zero = S[(size_t)r * m + c] == 0.0;
        if (zero) C[(size_t)c * m + c] = kSentinel;
    }
}

// Cholesky route: factor B~ = L L^T in shared memory when (m^2 + 2m) doubles
// fit, else in the global scratch G; S = D X^T with X = L^{-1};
// status = 0 when accepted (and *mk = m), 1 otherwise.
static constexpr int kCholThreads = 1024;
static constexpr size_t kCholSmemMax = 216 * 1024;

__global__ void __launch_bounds__(kCholThreads) rg_cholinv(int m, const double* __restrict__ Bt,
                                                           const double* __restrict__ dsc, double* __restrict__ S,
                                                           double* G, int use_smem, int* status, int* mk)
{
    extern __shared__ double sh[];
    __shared__ double red[kCholThreads];
    double* M = use_smem ? sh : G;
    double* xd = M + (size_t)m * m;
    double* cj = xd + m;
    for (int idx = threadIdx.x; idx < m * m; idx += blockDim.x) M[idx] = Bt[idx];
    __syncthreads();
    const bool ok = cta_chol_inv(m, M, xd, cj, red);
    if (ok) {
        for (int idx = threadIdx.x; idx < m * m; idx += blockDim.x) {
            const int r = idx / m, c = idx % m;
            S[idx] = c > r ? dsc[r] * M[chol_inv_at(m, c, r)] : (c == r ? dsc[r] * xd[r] : 0.0);
        }
    }
    if (threadIdx.x == 0) {
        *status = ok ? 0 : 1;
        if (ok) *mk = m;
    }
}

static size_t chol_bytes(int m) { return ((size_t)m * m + 2 * (size_t)m) * sizeof(double); }

size_t reduced_work_bytes(int m)
{
    const size_t mm = (size_t)m * m * sizeof(double);
    return 8 * (mm + 256) + (m * sizeof(double) + 256) * 2 + jacobi_work_bytes(m) + chol_bytes(m) + 512 + 1024;
}

// lam[m] (ascending, sentinels >= 1e299 last), V row-major m x m, *mk (device).
// Synchronises the stream to check the two Jacobi runs.  Returns 0, -3 when
// a Jacobi run did not converge or its grid barrier timed out, -4 on a CUDA
// error.
int reduced_gev_dev(int m, const double* Aq, const double* Bq, double* lam, double* V, int* mk, void* work,
                    cudaStream_t s)
{
    int sweeps = 0;
    const size_t mm = (size_t)m * m;
    char* p = align256((char*)work);
    auto take = [&](size_t bytes) { char* q = p; p = align256(p + bytes); return q; };
    double* At = (double*)take(mm * 8);
    double* Bt = (double*)take(mm * 8);
    double* U = (double*)take(mm * 8);
    double* S = (double*)take(mm * 8);
    double* T1 = (double*)take(mm * 8);
    double* C = (double*)take(mm * 8);
    double* W = (double*)take(mm * 8);
    double* d = (double*)take(m * 8);
    double* dsc = (double*)take(m * 8);
    void* jw = take(jacobi_work_bytes(m));
    double* G = (double*)take(chol_bytes(m));
    int* cst = (int*)take(256);
    const int blocks = (int)((mm + 255) / 256 < 1024 ? (mm + 255) / 256 : 1024);
    rg_scale<<<blocks, 256, 0, s>>>(m, Aq, Bq, At, Bt, dsc);
    count_launches(2);  // scale, Cholesky
    if (cudaGetLastError() != cudaSuccess) return -4;
    const int use_smem = chol_bytes(m) <= kCholSmemMax;
    if (use_smem && cudaFuncSetAttribute(rg_cholinv, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)chol_bytes(m)) != cudaSuccess)
        return -4;
    rg_cholinv<<<1, kCholThreads, use_smem ? chol_bytes(m) : 0, s>>>(m, Bt, dsc, S, G, use_smem, cst, mk);
    if (cudaGetLastError() != cudaSuccess) return -4;
    int hst = 1;
    if (cudaMemcpyAsync(&hst, cst, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess) return -4;
    if (cudaStreamSynchronize(s) != cudaSuccess) return -4;
    if (hst == 0) {
        if (launch_rg_product<0>(m, At, S, T1, s) != cudaSuccess) return -4;
        if (launch_rg_product<1>(m, S, T1, C, s) != cudaSuccess) return -4;
        const int st = jacobi_eig_dev(m, C, lam, W, jw, s, &sweeps);
        if (st) return st == -3 ? -4 : -3;
        if (launch_rg_product<0>(m, S, W, V, s) != cudaSuccess) return -4;
        return 0;
    }
    count_launches(2);  // basis, sentinel
    int st = jacobi_eig_dev(m, Bt, d, U, jw, s, &sweeps);
    if (st) return st == -3 ? -4 : -3;
    rg_basis<<<blocks, 256, 0, s>>>(m, d, U, dsc, S, mk);
    if (cudaGetLastError() != cudaSuccess) return -4;
    if (launch_rg_product<0>(m, At, S, T1, s) != cudaSuccess) return -4;
    if (launch_rg_product<1>(m, S, T1, C, s) != cudaSuccess) return -4;
    rg_sentinel<<<(m + 255) / 256, 256, 0, s>>>(m, S, C);
    if (cudaGetLastError() != cudaSuccess) return -4;
    st = jacobi_eig_dev(m, C, lam, W, jw, s, &sweeps);
    if (st) return st == -3 ? -4 : -3;
    if (launch_rg_product<0>(m, S, W, V, s) != cudaSuccess) return -4;
    return 0;
}

}  // namespace feast

extern "C" long long feast_set_wait_limit(long long cycles)
{
    return feast::g_spin_cycles.exchange(cycles >= 1 ? cycles : feast::kDefaultSpinCycles);
}
