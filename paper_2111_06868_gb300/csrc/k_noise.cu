// k_noise.cu -- kernels of the noisy-simulation paths (HybridQ Sec. 5).
//
//   * k_rdm<R, K> (K <= 2): the reduced density matrix of K qubits of a pure
//     state, rho_ab = sum_y psi(y, a) conj(psi(y, b)) over the indices y of
//     the other qubits, in one read of the state.  Pure-state sampling of a
//     Kraus channel (Sec. 5) takes its branch probabilities from it:
//     p_i = ||K_i psi||^2 = Tr(K_i rho K_i^dag).
//   * k_window (n >= 4): one or two state-dependent channels per pass: the
//     branches picked on the device from the partial sums of the launch before
//     and caller-drawn uniforms, the renormalised operators applied, the next
//     window's reduced density matrix summed from what is written.
//   * k_kraus_pick, k_apply_sel (n < 4): the same channel by channel from
//     k_rdm's partial sums.
// Each thread sums its share of a complex64 state in FP32 with a compensation
// term, 8 products per addition (complex128 in FP64).  k_rdm: the CTA sums in
// FP64, one CTA joins the CTAs' sums; at most two CTAs per SM, so that few
// partial sums reach that join.  k_window: see there; one CTA per SM.  All
// joins run in a fixed order.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "hq_cp_async.cuh"
#include "hq_fault.cuh"
#include "hq_internal.cuh"

namespace hq {

constexpr int kNoiseThreads = 256;
constexpr int kRdmUnroll = 4;

template <typename R, int K> struct RdmParam {
    int64_t toff[1 << K];  // flat offset of local index a (qubits[0] = MSB)
    int fixed[K];          // flat bits of the K qubits, ascending
    int free_bits;         // n - K
};

// entries (a, b), a <= b, of the upper triangle in row order
template <int K> __host__ __device__ constexpr int rdm_entries() { return (1 << K) * ((1 << K) + 1) / 2; }

template <typename R, int K>
__global__ void __launch_bounds__(kNoiseThreads) k_rdm(const RdmParam<R, K> p, const typename C2<R>::type *__restrict__ psi,
                                                       int64_t groups, double *__restrict__ partials)
{
    using T2 = typename C2<R>::type;
    constexpr int D = 1 << K, NE = rdm_entries<K>();
    // per-thread sums in R; in FP32 each carries a compensation term (Kahan),
    // so that the FP64 pipe is used once per thread, not once per chunk
    R ar[NE], ai[NE], cr[NE], ci[NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) ar[e] = ai[e] = cr[e] = ci[e] = 0;
    auto add = [](R &sum, R &comp, R x) {
        if constexpr (sizeof(R) == 4) {
            const R y = x - comp;
            const R t = sum + y;
            comp = (t - sum) - y;
            sum = t;
        } else {
            sum += x;
        }
    };
    const int64_t stride = int64_t(gridDim.x) * blockDim.x * kRdmUnroll;
    for (int64_t f0 = int64_t(blockIdx.x) * blockDim.x * kRdmUnroll + threadIdx.x; f0 < groups; f0 += stride) {
        T2 v[kRdmUnroll][D];
#pragma unroll
        for (int u = 0; u < kRdmUnroll; ++u) {
            const int64_t f = f0 + int64_t(u) * blockDim.x;
            if (f < groups) {
                uint64_t x = uint64_t(f);
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    const int b = p.fixed[j];
                    x = ((x >> b) << (b + 1)) | (x & ((uint64_t(1) << b) - 1));
                }
#pragma unroll
                for (int a = 0; a < D; ++a) v[u][a] = psi[int64_t(x) + p.toff[a]];
            } else {
#pragma unroll
                for (int a = 0; a < D; ++a) v[u][a].x = v[u][a].y = 0;
            }
        }
        // v_a conj(v_b), summed over the chunk in R, then joined in FP64
        int e = 0;
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
            for (int b = a; b < D; ++b, ++e) {
                R sr = 0, si = 0;
#pragma unroll
                for (int u = 0; u < kRdmUnroll; ++u) {
                    sr += v[u][a].x * v[u][b].x + v[u][a].y * v[u][b].y;
                    si += v[u][a].y * v[u][b].x - v[u][a].x * v[u][b].y;
                }
                add(ar[e], cr[e], sr);
                add(ai[e], ci[e], si);
            }
    }
#pragma unroll
    for (int e = 0; e < NE; ++e) {
        const double sr = block_sum(double(ar[e]) - double(cr[e]));
        const double si = block_sum(double(ai[e]) - double(ci[e]));
        if (threadIdx.x == 0) {
            partials[(int64_t(blockIdx.x) * NE + e) * 2] = sr;
            partials[(int64_t(blockIdx.x) * NE + e) * 2 + 1] = si;
        }
    }
}

// one CTA: out[j] = sum over the nparts partial vectors of entry j (fixed order)
__global__ void __launch_bounds__(kNoiseThreads) k_noise_final(const double *__restrict__ partials, int nparts,
                                                               int width, double *__restrict__ out)
{
    for (int j = 0; j < width; ++j) {
        double v = 0;
        for (int i = threadIdx.x; i < nparts; i += blockDim.x) v += partials[int64_t(i) * width + j];
        const double s = block_sum(v);
        if (threadIdx.x == 0) out[j] = s;
    }
}

template <typename R, int K> static RdmParam<R, K> rdm_param(int n, const int *qubits)
{
    constexpr int D = 1 << K;
    RdmParam<R, K> p;
    std::memset(&p, 0, sizeof(p));
    for (int j = 0; j < K; ++j) p.fixed[j] = n - 1 - qubits[j];
    std::sort(p.fixed, p.fixed + K);
    for (int a = 0; a < D; ++a) {
        int64_t off = 0;
        for (int j = 0; j < K; ++j)
            if ((a >> (K - 1 - j)) & 1) off += int64_t(1) << (n - 1 - qubits[j]);
        p.toff[a] = off;
    }
    p.free_bits = n - K;
    return p;
}

// at most two CTAs per SM: enough loads in flight for HBM, and few partial
// sums for the one-CTA pass that joins them
template <typename R, int K> static int rdm_grid(int n)
{
    const int64_t per_cta = int64_t(kNoiseThreads) * kRdmUnroll;
    return int(std::min<int64_t>(2 * sm_count(), grid_for((const void *)k_rdm<R, K>, kNoiseThreads, 0,
                                                          ((int64_t(1) << (n - K)) + per_cta - 1) / per_cta)));
}

// per-CTA partial sums (rdm_grid<R, K>(n) rows of 2 * rdm_entries<K>() doubles)
template <typename R, int K>
static hq_status rdm_partials(const void *state, int n, const int *qubits, double *partials, cudaStream_t s)
{
    const RdmParam<R, K> p = rdm_param<R, K>(n, qubits);
    k_rdm<R, K><<<rdm_grid<R, K>(n), kNoiseThreads, 0, s>>>(p, (const typename C2<R>::type *)state,
                                                             int64_t(1) << p.free_bits, partials);
    return cuda_status("k_rdm", cudaGetLastError());
}

template <typename R, int K>
static hq_status run_rdm(const void *state, int n, const int *qubits, double *out_host, cudaStream_t s)
{
    constexpr int D = 1 << K, NE = rdm_entries<K>();
    const int grid = rdm_grid<R, K>(n);
    const int width = 2 * NE;
    double *scratch = nullptr;
    if (injected_alloc_failure() ||
        !scratch_alloc((void **)&scratch, sizeof(double) * (size_t(grid) + 1) * width, s))
        return HQ_ERR_ALLOC;
    hq_status rc = rdm_partials<R, K>(state, n, qubits, scratch, s);
    double *out_dev = scratch + size_t(grid) * width;
    if (rc == HQ_OK) {
        k_noise_final<<<1, kNoiseThreads, 0, s>>>(scratch, grid, width, out_dev);
        rc = cuda_status("k_noise_final", cudaGetLastError());
    }
    std::vector<double> tri(width);
    if (rc == HQ_OK)
        rc = cuda_status("copy result",
                         cudaMemcpyAsync(tri.data(), out_dev, sizeof(double) * width, cudaMemcpyDeviceToHost, s));
    scratch_free(scratch, s);
    if (rc == HQ_OK) rc = cuda_status("sync", cudaStreamSynchronize(s));
    if (rc != HQ_OK) return rc;
    int e = 0;
    for (int a = 0; a < D; ++a)
        for (int b = a; b < D; ++b, ++e) {
            out_host[2 * (a * D + b)] = tri[2 * e];
            out_host[2 * (a * D + b) + 1] = tri[2 * e + 1];
            out_host[2 * (b * D + a)] = tri[2 * e];
            out_host[2 * (b * D + a) + 1] = -tri[2 * e + 1];
        }
    return HQ_OK;
}

hq_status launch_rdm(const void *state, int n, hq_dtype dt, const int *qubits, int k, double *out_host,
                     cudaStream_t s)
{
    if (dt == HQ_C64) return k == 1 ? run_rdm<float, 1>(state, n, qubits, out_host, s)
                                    : run_rdm<float, 2>(state, n, qubits, out_host, s);
    return k == 1 ? run_rdm<double, 1>(state, n, qubits, out_host, s) : run_rdm<double, 2>(state, n, qubits, out_host, s);
}

// ----------------------------------------------------------------------------
// Pure-state sampling of a Kraus channel
// ----------------------------------------------------------------------------
// Device side of a state-dependent channel: k_rdm's partial sums -> the
// branch (one CTA) -> the renormalised operator applied.  `sel` holds the
// chosen operator (2 D^2 doubles) and, after it, 1.0 when that operator is
// the identity to rounding (then nothing is applied).  The gates that come
// right before the channel on the same qubits are not applied on their own:
// their product A is folded in, the branch probabilities taken from
// A rho A^dag (rho of the state before them) and K_i A / sqrt(p_i) applied,
// one read of the state and one read-write instead of two more passes.
constexpr int kMaxKraus = 64;
struct PickArgs {
    const double *partials;
    int nparts, width, D, nK;
    const double *K;  // nK row-major D x D complex matrices, interleaved re/im
    const double *G;  // their Gram matrices K^dag K
    const double *A;  // the absorbed gates' product (D x D; the identity when none)
    const double *u;  // the uniform in [0, 1)
    int *chosen;
    double *sel;
    int *status;      // set to 1 when every p_i is 0
};

// D = 2^K: the thread-0 part below works on arrays of fixed size (in
// registers, loops unrolled)
template <int D>
__global__ void __launch_bounds__(kNoiseThreads) k_kraus_pick(const PickArgs a)
{
    constexpr int W = 2 * rdm_entries<2>();  // widest partial-sum row
    __shared__ double tri[W];
    // the operators, their Gram matrices and the absorbed gates, staged by
    // the whole CTA (thread 0 then reads shared memory, not global memory)
    __shared__ double sK[kMaxKraus * 2 * 16], sG[kMaxKraus * 2 * 16], sA[2 * 16];
    {
        const int n2 = a.nK * 2 * a.D * a.D;
        for (int i = threadIdx.x; i < n2; i += blockDim.x) {
            sK[i] = a.K[i];
            sG[i] = a.G[i];
        }
        for (int i = threadIdx.x; i < 2 * a.D * a.D; i += blockDim.x) sA[i] = a.A[i];
    }
    // the columns of the partial sums, by one warp: rows per lane, then a
    // shuffle tree (GB300's FP64 pipe is slow enough that every FP64 warp
    // instruction counts: the other warps only stage the matrices)
    if (threadIdx.x < 32) {
        double v[W];
#pragma unroll
        for (int j = 0; j < W; ++j) v[j] = 0;
        for (int i = threadIdx.x; i < a.nparts; i += 32)
#pragma unroll
            for (int j = 0; j < W; ++j)
                if (j < a.width) v[j] += a.partials[int64_t(i) * a.width + j];
#pragma unroll
        for (int j = 0; j < W; ++j)
            if (j < a.width) {  // the same for every lane
                double x = v[j];
                for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
                if (threadIdx.x == 0) tri[j] = x;
            }
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    constexpr int DD = D * D;
    double r0r[D][D], r0i[D][D];
#pragma unroll
    for (int x = 0, e = 0; x < D; ++x)
#pragma unroll
        for (int y = x; y < D; ++y, ++e) {
            r0r[x][y] = r0r[y][x] = tri[2 * e];
            r0i[x][y] = tri[2 * e + 1];
            r0i[y][x] = -tri[2 * e + 1];
        }
    // rho = A rho0 A^dag: T = A rho0, then rho[x][y] = sum_z T[x][z] conj(A[y][z])
    double tr_[D][D], ti_[D][D], rr[D][D], ri[D][D];
#pragma unroll
    for (int x = 0; x < D; ++x)
#pragma unroll
        for (int y = 0; y < D; ++y) {
            double sr = 0, si = 0;
#pragma unroll
            for (int z = 0; z < D; ++z) {
                const double ar = sA[2 * (x * D + z)], ai = sA[2 * (x * D + z) + 1];
                sr += ar * r0r[z][y] - ai * r0i[z][y];
                si += ar * r0i[z][y] + ai * r0r[z][y];
            }
            tr_[x][y] = sr;
            ti_[x][y] = si;
        }
#pragma unroll
    for (int x = 0; x < D; ++x)
#pragma unroll
        for (int y = 0; y < D; ++y) {
            double sr = 0, si = 0;
#pragma unroll
            for (int z = 0; z < D; ++z) {
                const double br = sA[2 * (y * D + z)], bi = -sA[2 * (y * D + z) + 1];
                sr += tr_[x][z] * br - ti_[x][z] * bi;
                si += tr_[x][z] * bi + ti_[x][z] * br;
            }
            rr[x][y] = sr;
            ri[x][y] = si;
        }
    // p_i = Tr(K rho K^dag) = Tr(rho K^dag K) = sum_rc rho[r][c] G[c][r]
    // (computed again where it is needed, rather than kept in an array
    // indexed at run time)
    auto prob = [&](int i) {
        const double *G = sG + size_t(i) * 2 * DD;
        double t = 0;
#pragma unroll
        for (int r = 0; r < D; ++r)
#pragma unroll
            for (int c = 0; c < D; ++c) t += rr[r][c] * G[2 * (c * D + r)] - ri[r][c] * G[2 * (c * D + r) + 1];
        return fmax(t, 0.0);
    };
    double total = 0;
    for (int i = 0; i < a.nK; ++i) total += prob(i);
    if (!(total > 0)) {
        *a.status = 1;
        *a.chosen = -1;
        a.sel[2 * DD] = 1.0;
        return;
    }
    // the first i whose cumulative probability exceeds u * total (the last
    // nonzero one if rounding leaves none)
    const double target = *a.u * total;
    int pick = -1;
    double cum = 0, ppick = 0;
    for (int i = 0; i < a.nK; ++i) {
        const double pi = prob(i);
        cum += pi;
        if (pi > 0) {
            pick = i;
            ppick = pi;
            if (cum > target) break;
        }
    }
    const double sc = 1.0 / sqrt(ppick);
    const double *Kp = sK + size_t(pick) * 2 * DD;
    bool identity = true;
#pragma unroll
    for (int r = 0; r < D; ++r)
#pragma unroll
        for (int c = 0; c < D; ++c) {
            // (K_pick A)[r][c] / sqrt(p_pick)
            double mr = 0, mi = 0;
#pragma unroll
            for (int z = 0; z < D; ++z) {
                const double kr = Kp[2 * (r * D + z)], ki = Kp[2 * (r * D + z) + 1];
                const double ar = sA[2 * (z * D + c)], ai = sA[2 * (z * D + c) + 1];
                mr += kr * ar - ki * ai;
                mi += kr * ai + ki * ar;
            }
            mr *= sc;
            mi *= sc;
            a.sel[2 * (r * D + c)] = mr;
            a.sel[2 * (r * D + c) + 1] = mi;
            // |m - delta| <= 4 eps, compared squared (no hypot on the slow FP64 pipe)
            const double dr = mr - (r == c ? 1.0 : 0.0);
            identity = identity && dr * dr + mi * mi <= 16.0 * 2.220446049250313e-16 * 2.220446049250313e-16;
        }
    a.sel[2 * DD] = identity ? 1.0 : 0.0;
    *a.chosen = pick;
}

template <typename R, int K>
__global__ void __launch_bounds__(kNoiseThreads) k_apply_sel(const RdmParam<R, K> p, const double *__restrict__ sel,
                                                             typename C2<R>::type *__restrict__ psi, int64_t groups)
{
    using T2 = typename C2<R>::type;
    constexpr int D = 1 << K;
    if (sel[2 * D * D] != 0.0) return;  // the identity
    T2 m[D][D];
#pragma unroll
    for (int r = 0; r < D; ++r)
#pragma unroll
        for (int c = 0; c < D; ++c) {
            m[r][c].x = R(sel[2 * (r * D + c)]);
            m[r][c].y = R(sel[2 * (r * D + c) + 1]);
        }
    const int64_t stride = int64_t(gridDim.x) * blockDim.x * kRdmUnroll;
    for (int64_t f0 = int64_t(blockIdx.x) * blockDim.x * kRdmUnroll + threadIdx.x; f0 < groups; f0 += stride) {
        T2 v[kRdmUnroll][D];
        int64_t base[kRdmUnroll];
#pragma unroll
        for (int u = 0; u < kRdmUnroll; ++u) {
            const int64_t f = f0 + int64_t(u) * blockDim.x;
            base[u] = -1;
            if (f < groups) {
                uint64_t x = uint64_t(f);
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    const int b = p.fixed[j];
                    x = ((x >> b) << (b + 1)) | (x & ((uint64_t(1) << b) - 1));
                }
                base[u] = int64_t(x);
#pragma unroll
                for (int a = 0; a < D; ++a) v[u][a] = psi[base[u] + p.toff[a]];
            }
        }
#pragma unroll
        for (int u = 0; u < kRdmUnroll; ++u) {
            if (base[u] < 0) continue;
#pragma unroll
            for (int r = 0; r < D; ++r) {
                T2 acc;
                acc.x = acc.y = 0;
#pragma unroll
                for (int c = 0; c < D; ++c) cmac(acc, m[r][c], v[u][c]);
                psi[base[u] + p.toff[r]] = acc;
            }
        }
    }
}

template <typename R, int K>
static hq_status sample_on_device(void *state, int n, const int *qubits, PickArgs a, cudaStream_t s)
{
    hq_status st = rdm_partials<R, K>(state, n, qubits, const_cast<double *>(a.partials), s);
    if (st != HQ_OK) return st;
    a.nparts = rdm_grid<R, K>(n);
    a.width = 2 * rdm_entries<K>();
    a.D = 1 << K;
    k_kraus_pick<1 << K><<<1, kNoiseThreads, 0, s>>>(a);
    if ((st = cuda_status("k_kraus_pick", cudaGetLastError())) != HQ_OK) return st;
    const RdmParam<R, K> p = rdm_param<R, K>(n, qubits);
    const int64_t groups = int64_t(1) << p.free_bits;
    const int64_t per_cta = int64_t(kNoiseThreads) * kRdmUnroll;
    const int agrid = grid_for((const void *)k_apply_sel<R, K>, kNoiseThreads, 0, (groups + per_cta - 1) / per_cta);
    k_apply_sel<R, K><<<agrid, kNoiseThreads, 0, s>>>(p, a.sel, (typename C2<R>::type *)state, groups);
    return cuda_status("k_apply_sel", cudaGetLastError());
}

// ----------------------------------------------------------------------------
// Windows: one or two state-dependent channels per trip through the state
//
// Two one-qubit channels on different qubits, with nothing but absorbed gates
// between them, need one joint reduced density matrix: the first channel's
// probabilities come from its partial trace, the second's from the same matrix
// after the operator picked for the first,
//   rho2[b][b'] = sum_cc' (M^dag M)[c'][c] rho[(c, b)][(c', b')].
// k_window picks (every CTA for itself, from the partial sums of the launch
// before: no extra launch, no CTA waits for another), applies both operators
// to its groups and, from the amplitudes it writes, sums the reduced density
// matrix of the next window's qubits.  So a channel costs half of one read and
// write of the state instead of a read, a one-CTA pick and a read and write.
// A thread holds 16 amplitudes: all values of this window's two qubits and of
// the next one's (a qubit that a window lacks is replaced by any other bit).
// Bound: HBM (two channels at n = 24: 268 MB, 40 us at the copy bandwidth; a
// launch takes 74 us, the mean of a trajectory's 156 serialised ones, where
// three launches per channel took 101), with about 5 us of FP64 latency per
// launch for the pick; complex128 the FP64 pipe.
// ----------------------------------------------------------------------------
constexpr int kWindowRow = 20;  // sums per CTA: 10 complex entries of the upper triangle
struct WindowParam {
    int64_t off[16];   // flat offset of local index 4 a + b (a: this window's qubits, b: the next one's; first qubit
                       // most significant)
    int fixed[4];      // the four bits, ascending
    int free_bits;     // n - 4
    int na, nb;        // qubits of this window (0: nothing to apply) and of the next (0: nothing to sum)
    int nch;           // channels of this window: 2 one-qubit ones, or 1 on na qubits
    const double *K[2], *G[2], *A[2], *u[2];  // per channel: as in PickArgs
    int nK[2];
    int *chosen[2];
    int *status;
    const double *in;  // partial sums for this window: `rows` rows of kWindowRow
    int rows;
    double *out;       // partial sums for the next window, one row per CTA
};

// One warp: the branch of a channel on D levels with reduced density matrix
// rho0 (shared memory, D x D complex), its renormalised operator times the
// absorbed gates in M (FP64, shared memory); true when that is the identity to
// rounding.  The matrix products take one lane per entry (FP64 instructions are
// what they cost, whatever the lanes do); the sums run in k_kraus_pick's order.
template <int D>
__device__ __forceinline__ bool window_pick(const double *rho0, const double *K, const double *G, const double *A,
                                            double u, int nK, double *T, double *prob, double *M, int *chosen,
                                            int *status, bool report)
{
    constexpr int DD = D * D;
    const int lane = threadIdx.x & 31, x = (lane % DD) / D, y = lane % D;
    double sr = 0, si = 0;
#pragma unroll
    for (int z = 0; z < D; ++z) {  // T = A rho0
        const double ar = A[2 * (x * D + z)], ai = A[2 * (x * D + z) + 1];
        const double br = rho0[2 * (z * D + y)], bi = rho0[2 * (z * D + y) + 1];
        sr += ar * br - ai * bi;
        si += ar * bi + ai * br;
    }
    __syncwarp();
    if (lane < DD) T[2 * lane] = sr, T[2 * lane + 1] = si;
    __syncwarp();
    sr = si = 0;
#pragma unroll
    for (int z = 0; z < D; ++z) {  // rho = T A^dag
        const double ar = T[2 * (x * D + z)], ai = T[2 * (x * D + z) + 1];
        const double br = A[2 * (y * D + z)], bi = -A[2 * (y * D + z) + 1];
        sr += ar * br - ai * bi;
        si += ar * bi + ai * br;
    }
    __syncwarp();
    if (lane < DD) T[2 * lane] = sr, T[2 * lane + 1] = si;
    __syncwarp();
    for (int i = lane; i < nK; i += 32) {  // p_i = Tr(rho K_i^dag K_i)
        const double *g = G + size_t(i) * 2 * DD;
        double t = 0;
#pragma unroll
        for (int r = 0; r < D; ++r)
#pragma unroll
            for (int c = 0; c < D; ++c)
                t += T[2 * (r * D + c)] * g[2 * (c * D + r)] - T[2 * (r * D + c) + 1] * g[2 * (c * D + r) + 1];
        prob[i] = fmax(t, 0.0);
    }
    __syncwarp();
    double total = 0;
    for (int i = 0; i < nK; ++i) total += prob[i];
    int pick = -1;
    double cum = 0, ppick = 0;
    const double target = u * total;
    for (int i = 0; i < nK; ++i) {
        const double pi = prob[i];
        cum += pi;
        if (pi > 0) {
            pick = i;
            ppick = pi;
            if (cum > target) break;
        }
    }
    if (!(total > 0)) pick = -1;
    double mr = x == y ? 1.0 : 0.0, mi = 0;
    if (pick >= 0) {
        // (rsqrt: at most 0.51 ulp off, 0.29 on average, over 2^23 values each in [2^-20, 1), [0.9, 1.1] and
        // [2^-300, 2^300]; 1.0 / sqrt: 1.49 and 0.44 to 0.50)
        const double sc = rsqrt(ppick);
        const double *Kp = K + size_t(pick) * 2 * DD;
        mr = 0;
#pragma unroll
        for (int z = 0; z < D; ++z) {  // (K_pick A)[x][y] / sqrt(p_pick)
            const double kr = Kp[2 * (x * D + z)], ki = Kp[2 * (x * D + z) + 1];
            const double ar = A[2 * (z * D + y)], ai = A[2 * (z * D + y) + 1];
            mr += kr * ar - ki * ai;
            mi += kr * ai + ki * ar;
        }
        mr *= sc;
        mi *= sc;
    }
    const double dr = mr - (x == y ? 1.0 : 0.0);
    const bool one = dr * dr + mi * mi <= 16.0 * 2.220446049250313e-16 * 2.220446049250313e-16;
    const bool identity = __all_sync(0xffffffffu, one);
    if (lane < DD) M[2 * lane] = mr, M[2 * lane + 1] = mi;
    __syncwarp();
    if (report && lane == 0) {
        *chosen = pick;
        if (pick < 0) *status = 1;
    }
    return identity;
}

// Sums of a window kernel.  complex64: a thread hands over its compensated FP32 sum as a pair; inside the CTA the pairs
// are joined in three-float sums (error-free additions, Knuth's two-sum: 70 bits and more, so no less than FP64's 53),
// and the CTA's sums and those of all CTAs are FP64.  Joined as doubles from the threads on, the 20 sums of each of the
// 16 warps were 21 of a launch's 83 us (an FP64 instruction takes a GB300 SM's quarter 64 cycles whatever its lanes do).
template <typename R> struct ThreadSum;
template <> struct ThreadSum<float> {
    float h, l;
};
template <> struct ThreadSum<double> {
    double h;
};
__device__ __forceinline__ ThreadSum<float> thread_sum(float sum, float comp, float scale)
{
    const float h = sum - comp;
    return {h * scale, ((sum - h) - comp) * scale};
}
__device__ __forceinline__ ThreadSum<double> thread_sum(double sum, double, double) { return {sum}; }

template <typename R> struct Sum;
template <> struct Sum<float> {
    float a, b, c;  // a + b + c, each about 2^-24 of the one before
};
template <> struct Sum<double> {
    double a;
};
// x + y = result + err exactly
__device__ __forceinline__ float two_sum(float x, float y, float &err)
{
    const float t = x + y, z = t - x;
    err = (x - (t - z)) + (y - z);
    return t;
}
__device__ __forceinline__ void sum_add(Sum<float> &s, float a, float b, float c)
{
    float d, e, g;
    s.a = two_sum(s.a, a, d);
    s.b = two_sum(s.b, d, e);
    s.b = two_sum(s.b, b, g);
    s.c += (e + g) + c;
}
__device__ __forceinline__ void sum_start(Sum<float> &s, ThreadSum<float> t) { s = {t.h, t.l, 0.f}; }
__device__ __forceinline__ void sum_start(Sum<double> &s, ThreadSum<double> t) { s = {t.h}; }
__device__ __forceinline__ void sum_add(Sum<float> &s, ThreadSum<float> t) { sum_add(s, t.h, t.l, 0.f); }
__device__ __forceinline__ void sum_add(Sum<double> &s, ThreadSum<double> t) { s.a += t.h; }
__device__ __forceinline__ double sum_value(Sum<float> s) { return double(s.a) + (double(s.b) + double(s.c)); }
__device__ __forceinline__ double sum_value(Sum<double> s) { return s.a; }
// lane 0: the sum over the warp
__device__ __forceinline__ void warp_join(Sum<float> &s)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float a = __shfl_down_sync(0xffffffffu, s.a, o), b = __shfl_down_sync(0xffffffffu, s.b, o),
                    c = __shfl_down_sync(0xffffffffu, s.c, o);
        sum_add(s, a, b, c);
    }
}
__device__ __forceinline__ void warp_join(Sum<double> &s)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s.a += __shfl_down_sync(0xffffffffu, s.a, o);
}

// (v0, v1) <- m (v0, v1), m row-major 2 x 2; complex64 with packed FMAs in cmac's order
__device__ __forceinline__ float2 swap_halves(float2 v) { return make_float2(v.y, v.x); }
__device__ __forceinline__ double2 swap_halves(double2 v) { return make_double2(v.y, v.x); }
__device__ __forceinline__ void apply_pair(const float2 *m, float2 &v0, float2 &v1)
{
    const float2 w0 = swap_halves(v0), w1 = swap_halves(v1);
    auto row = [&](const float2 a, const float2 b) {
        float2 o = pk_mul(make_float2(a.x, a.x), v0);
        o = pk_fma(make_float2(-a.y, a.y), w0, o);
        o = pk_fma(make_float2(b.x, b.x), v1, o);
        return pk_fma(make_float2(-b.y, b.y), w1, o);
    };
    const float2 o0 = row(m[0], m[1]), o1 = row(m[2], m[3]);
    v0 = o0;
    v1 = o1;
}
__device__ __forceinline__ void apply_pair(const double2 *m, double2 &v0, double2 &v1)
{
    double2 o0, o1;
    o0.x = o0.y = o1.x = o1.y = 0;
    cmac(o0, m[0], v0);
    cmac(o0, m[1], v1);
    cmac(o1, m[2], v0);
    cmac(o1, m[3], v1);
    v0 = o0;
    v1 = o1;
}
// acc += (a.x b.x, a.y b.y)
__device__ __forceinline__ void mac2(float2 &acc, float2 a, float2 b) { acc = pk_fma(a, b, acc); }
__device__ __forceinline__ void mac2(double2 &acc, double2 a, double2 b)
{
    acc.x = fma(a.x, b.x, acc.x);
    acc.y = fma(a.y, b.y, acc.y);
}

constexpr int kWindowOps = 64;  // doubles of K (and of G) that are staged in shared memory

// one CTA per SM: few partial sums to read back (152 rows instead of 304: the pick's FP64 additions halve twice over)
// (512 threads; complex128 on states with few groups of 16 amplitudes, bound by the FP64 latency of an SM quarter's
// warps: 128, so that the groups reach four times as many SMs: a channel alone, n = 14 / 18 / 19, 102 / 106 / 118 us with
// 512 threads, 72 / 77 / 94 with 128; k_rdm, k_kraus_pick and k_apply_sel took 87 / 92 / 119)
constexpr int kWindowMany = 512, kWindowFew = 128;

template <typename R, int TH>
__global__ void __launch_bounds__(TH, 1) k_window(const __grid_constant__ WindowParam p,
                                                              typename C2<R>::type *__restrict__ psi)
{
    using T2 = typename C2<R>::type;
    __shared__ double s_part[TH / 32][kWindowRow];
    __shared__ Sum<R> s_sum[kWindowRow];
    __shared__ double s_rho[32], s_one[32], s_T[32], s_prob[kMaxKraus], s_M[2][32];
    __shared__ T2 s_m[2][16];
    __shared__ double s_op[2][3][kWindowOps], s_u[2];  // K, G, A of each channel
    __shared__ int s_identity[2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t groups = int64_t(1) << p.free_bits, stride = int64_t(gridDim.x) * blockDim.x;
    auto spread = [&](int64_t f) {
        int64_t x = f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int b = p.fixed[j];
            x = ((x >> b) << (b + 1)) | (x & ((int64_t(1) << b) - 1));
        }
        return x;
    };
    // complex64: a thread's groups come through its own slots of shared memory (cp.async; nobody else reads them, so
    // no barrier), two groups in flight: the first two under the pick, the later ones under the groups before them.
    // Three stages: a stage is filled again only after the arithmetic on what was read from it.
    constexpr bool kStaged = sizeof(R) == 4;
    extern __shared__ __align__(16) unsigned char s_stage[];
    T2 *const slot = reinterpret_cast<T2 *>(s_stage) + threadIdx.x;  // [stage][16][TH]
    T2 v[16];
    int64_t f = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    int stage = 0;
    auto fetch = [&](int64_t g, int to) {
        if (g < groups) {
            const T2 *const from = psi + spread(g);
#pragma unroll
            for (int i = 0; i < 16; ++i) cp_async8(slot + (16 * to + i) * TH, from + p.off[i]);
        }
        cp_async_commit();
    };
    if constexpr (kStaged) {
        fetch(f, 0);
        fetch(f + stride, 1);
    }
    // small operators staged by the CTA while its first warps read the sums
    for (int x = 0; x < p.nch; ++x) {
        const int DD = p.nch == 2 || p.na == 1 ? 4 : 16, n2 = p.nK[x] * 2 * DD;
        if (n2 <= kWindowOps)
            for (int i = threadIdx.x; i < n2; i += blockDim.x) {
                s_op[x][0][i] = p.K[x][i];
                s_op[x][1][i] = p.G[x][i];
            }
        if (int(threadIdx.x) < 2 * DD) s_op[x][2][threadIdx.x] = p.A[x][threadIdx.x];
        if (threadIdx.x == 0) s_u[x] = *p.u[x];
    }
    if (p.na > 0) {
        // the CTAs' sums, in a fixed order: rows warp by warp, one column per lane
        const int width = p.na == 1 ? 6 : kWindowRow;
        double part = 0;
        if (lane < width)
            for (int r = warp; r < p.rows; r += TH / 32) part += p.in[int64_t(r) * kWindowRow + lane];
        if (lane < kWindowRow) s_part[warp][lane] = part;
        __syncthreads();
        if (warp == 0) {
            double t = 0;
            if (lane < width)
                for (int w = 0; w < TH / 32; ++w) t += s_part[w][lane];
            // upper triangle -> full matrix
            const int D = 1 << p.na;
            if (lane < width) {
                int e = lane >> 1, r = 0;
                while (e >= D - r) e -= D - r, ++r;
                const int c = r + e, im = lane & 1;
                s_rho[2 * (r * D + c) + im] = t;
                if (r != c) s_rho[2 * (c * D + r) + im] = im ? -t : t;
            }
            __syncwarp();
            bool id0, id1 = true;
            const bool report = blockIdx.x == 0;
            const int DD = p.nch == 2 || p.na == 1 ? 4 : 16;
            const double *K[2], *G[2];
            for (int x = 0; x < 2; ++x) {
                const bool staged = p.nK[x] * 2 * DD <= kWindowOps;
                K[x] = staged ? s_op[x][0] : p.K[x];
                G[x] = staged ? s_op[x][1] : p.G[x];
            }
            if (p.nch == 1) {
                id0 = p.na == 1 ? window_pick<2>(s_rho, K[0], G[0], s_op[0][2], s_u[0], p.nK[0], s_T, s_prob, s_M[0],
                                                 p.chosen[0], p.status, report)
                                : window_pick<4>(s_rho, K[0], G[0], s_op[0][2], s_u[0], p.nK[0], s_T, s_prob, s_M[0],
                                                 p.chosen[0], p.status, report);
            } else {
                // the first qubit's partial trace
                if (lane < 8) {
                    const int a = (lane >> 2) & 1, a2 = (lane >> 1) & 1, im = lane & 1;
                    s_one[2 * (2 * a + a2) + im] =
                        s_rho[2 * (4 * (2 * a) + 2 * a2) + im] + s_rho[2 * (4 * (2 * a + 1) + 2 * a2 + 1) + im];
                }
                __syncwarp();
                id0 = window_pick<2>(s_one, K[0], G[0], s_op[0][2], s_u[0], p.nK[0], s_T, s_prob, s_M[0], p.chosen[0],
                                     p.status, report);
                // Q = M^dag M, then the second qubit's matrix after the first operator
                const int x = (lane >> 1) & 1, y = lane & 1;
                double qr = 0, qi = 0;
#pragma unroll
                for (int z = 0; z < 2; ++z) {
                    const double ar = s_M[0][2 * (2 * z + x)], ai = -s_M[0][2 * (2 * z + x) + 1];
                    const double br = s_M[0][2 * (2 * z + y)], bi = s_M[0][2 * (2 * z + y) + 1];
                    qr += ar * br - ai * bi;
                    qi += ar * bi + ai * br;
                }
                __syncwarp();
                if (lane < 4) s_T[2 * lane] = qr, s_T[2 * lane + 1] = qi;
                __syncwarp();
                double sr = 0, si = 0;
#pragma unroll
                for (int c = 0; c < 2; ++c)
#pragma unroll
                    for (int c2 = 0; c2 < 2; ++c2) {
                        const double ar = s_T[2 * (2 * c2 + c)], ai = s_T[2 * (2 * c2 + c) + 1];
                        const int e = 2 * (4 * (2 * c + x) + 2 * c2 + y);
                        const double br = s_rho[e], bi = s_rho[e + 1];
                        sr += ar * br - ai * bi;
                        si += ar * bi + ai * br;
                    }
                __syncwarp();
                if (lane < 4) s_one[2 * lane] = sr, s_one[2 * lane + 1] = si;
                __syncwarp();
                id1 = window_pick<2>(s_one, K[1], G[1], s_op[1][2], s_u[1], p.nK[1], s_T, s_prob, s_M[1], p.chosen[1],
                                     p.status, report);
            }
            if (lane < 16) {
                s_m[0][lane].x = R(s_M[0][2 * lane]);
                s_m[0][lane].y = R(s_M[0][2 * lane + 1]);
                s_m[1][lane].x = R(s_M[1][2 * lane]);
                s_m[1][lane].y = R(s_M[1][2 * lane + 1]);
            }
            if (lane == 0) s_identity[0] = id0, s_identity[1] = id1;
        }
        __syncthreads();
    }
    const bool ap0 = p.na > 0 && !s_identity[0], ap1 = p.na > 0 && p.nch == 2 && !s_identity[1];
    const bool wide = p.na == 2 && p.nch == 1;

    // sums of the next window's matrix, as in k_rdm
    constexpr int NE = 10;
    R ar[NE], ai[NE], cr[NE], ci[NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) ar[e] = ai[e] = cr[e] = ci[e] = 0;
    auto add = [](R &sum, R &comp, R x) {
        if constexpr (sizeof(R) == 4) {
            const R y = x - comp;
            const R t = sum + y;
            comp = (t - sum) - y;
            sum = t;
        } else {
            sum += x;
        }
    };
    while (f < groups) {
        T2 *const base = psi + spread(f);
        if constexpr (kStaged) {
            cp_async_wait<1>();
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = slot[(16 * stage + i) * TH];
            fetch(f + 2 * stride, stage == 0 ? 2 : stage - 1);
            stage = stage == 2 ? 0 : stage + 1;
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = base[p.off[i]];
        }
        if (ap0 || ap1) {
            if (wide) {
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    T2 o[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        o[r].x = o[r].y = 0;
#pragma unroll
                        for (int c = 0; c < 4; ++c) cmac(o[r], s_m[0][4 * r + c], v[4 * c + b]);
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r) v[4 * r + b] = o[r];
                }
            } else {
                if (ap0) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) apply_pair(s_m[0], v[i], v[i + 8]);
                }
                if (ap1) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int j = (i & 3) | ((i & 4) << 1);
                        apply_pair(s_m[1], v[j], v[j + 4]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) base[p.off[i]] = v[i];
        }
        if (p.nb == 2) {
            int e = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b)
#pragma unroll
                for (int b2 = b; b2 < 4; ++b2, ++e) {
                    T2 re, im;
                    re.x = re.y = im.x = im.y = 0;
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const T2 s = v[4 * a + b], t = v[4 * a + b2];
                        mac2(re, s, t);
                        if (b != b2) mac2(im, swap_halves(s), t);
                    }
                    add(ar[e], cr[e], re.x + re.y);
                    if (b != b2) add(ai[e], ci[e], im.x - im.y);
                }
        } else if (p.nb == 1) {
            int e = 0;
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int b2 = b; b2 < 2; ++b2, ++e) {
#pragma unroll
                    for (int half = 0; half < 8; half += 4) {  // 8 products per compensated addition, as in k_rdm
                        T2 re, im;
                        re.x = re.y = im.x = im.y = 0;
#pragma unroll
                        for (int a = half; a < half + 4; ++a) {  // a: this window's qubits and the replaced one
                            const T2 s = v[4 * (a >> 1) + 2 * b + (a & 1)], t = v[4 * (a >> 1) + 2 * b2 + (a & 1)];
                            mac2(re, s, t);
                            if (b != b2) mac2(im, swap_halves(s), t);
                        }
                        add(ar[e], cr[e], re.x + re.y);
                        if (b != b2) add(ai[e], ci[e], im.x - im.y);
                    }
                }
        }
        f += stride;
    }
    if constexpr (kStaged) cp_async_wait<0>();
    if (p.nb == 0) return;
    // every thread's sums to shared memory; lane by lane over the warps, then each sum's 32 lanes by shuffles (fixed
    // order; five shuffle levels of all 20 sums in every warp took 3 us).  The barrier also tells whether a sum of the
    // CTA is so large that joining it in FP32 could overflow: then all of them are scaled down first.
    bool huge = false;
    if constexpr (sizeof(R) == 4) {
#pragma unroll
        for (int e = 0; e < NE; ++e) huge = huge || fabsf(ar[e]) >= 0x1p100f || fabsf(ai[e]) >= 0x1p100f;
    }
    huge = __syncthreads_or(huge);
    const R scale = huge ? R(0x1p-16) : R(1);
    ThreadSum<R> *const all = reinterpret_cast<ThreadSum<R> *>(s_stage);  // [warp][sum][lane]
    const int width = p.nb == 1 ? 6 : kWindowRow;
#pragma unroll
    for (int e = 0; e < NE; ++e)
        if (2 * e < width) {
            all[(warp * kWindowRow + 2 * e) * 32 + lane] = thread_sum(ar[e], cr[e], scale);
            all[(warp * kWindowRow + 2 * e + 1) * 32 + lane] = thread_sum(ai[e], ci[e], scale);
        }
    __syncthreads();
    for (int j = warp; j < width; j += TH / 32) {
        Sum<R> t;
        sum_start(t, all[j * 32 + lane]);
        for (int w = 1; w < TH / 32; ++w) sum_add(t, all[(w * kWindowRow + j) * 32 + lane]);
        warp_join(t);
        if (lane == 0) s_sum[j] = t;
    }
    __syncthreads();
    if (int(threadIdx.x) < width)
        p.out[int64_t(blockIdx.x) * kWindowRow + threadIdx.x] =
            sum_value(s_sum[threadIdx.x]) * (huge ? 0x1p16 : 1.0);
}

static int window_threads(int n, hq_dtype dt)
{
    return dt == HQ_C128 && (int64_t(1) << (n - 4)) <= int64_t(sm_count()) * 2 * kWindowFew ? kWindowFew : kWindowMany;
}
static int window_grid(int n, hq_dtype dt)
{
    const int64_t groups = int64_t(1) << (n - 4);
    const int threads = window_threads(n, dt);
    return int(std::min<int64_t>(sm_count(), (groups + threads - 1) / threads));
}

// the bits a window kernel works on: this window's qubits a, the next one's b, others in the place of missing ones
static void window_bits(WindowParam &p, int n, int na, const int *qa, int nb, const int *qb)
{
    int bit[4];
    uint64_t used = 0;
    for (int j = 0; j < na; ++j) used |= uint64_t(1) << (bit[j] = n - 1 - qa[j]);
    for (int j = 0; j < nb; ++j) used |= uint64_t(1) << (bit[2 + j] = n - 1 - qb[j]);
    int top = n - 1;
    auto other = [&]() {  // a high bit: neighbouring threads keep neighbouring amplitudes
        while ((used >> top) & 1) --top;
        used |= uint64_t(1) << top;
        return top;
    };
    for (int j = na; j < 2; ++j) bit[j] = other();
    for (int j = nb; j < 2; ++j) bit[2 + j] = other();
    for (int i = 0; i < 16; ++i) {
        p.off[i] = 0;
        for (int j = 0; j < 4; ++j)
            if ((i >> (3 - j)) & 1) p.off[i] += int64_t(1) << bit[j];
    }
    std::copy(bit, bit + 4, p.fixed);
    std::sort(p.fixed, p.fixed + 4);
    p.free_bits = n - 4;
    p.na = na;
    p.nb = nb;
}

template <typename R, int TH> static hq_status launch_window_as(const WindowParam &p, void *state, int grid, cudaStream_t s)
{
    // complex64: three stages of groups; then (and in complex128 only) the threads' sums
    const size_t smem = std::max(sizeof(R) == 4 ? size_t(3) * 16 * TH * sizeof(float2) : size_t(0),
                                 size_t(TH) * kWindowRow * sizeof(ThreadSum<R>));
    occupancy((const void *)k_window<R, TH>, TH, smem);  // (sets the kernel's shared-memory limit)
    k_window<R, TH><<<grid, TH, smem, s>>>(p, (typename C2<R>::type *)state);
    return cuda_status("k_window", cudaGetLastError());
}
static hq_status launch_window(const WindowParam &p, void *state, int n, hq_dtype dt, cudaStream_t s)
{
    const int grid = window_grid(n, dt);
    if (dt == HQ_C64) return launch_window_as<float, kWindowMany>(p, state, grid, s);
    if (window_threads(n, dt) == kWindowFew) return launch_window_as<double, kWindowFew>(p, state, grid, s);
    return launch_window_as<double, kWindowMany>(p, state, grid, s);
}

// K^dag K as a row-major D x D complex matrix
static void gram(int D, const double *K, double *G)
{
    for (int r = 0; r < D; ++r)
        for (int c = 0; c < D; ++c) {
            double gr = 0, gi = 0;
            for (int m = 0; m < D; ++m) {
                // conj(K[m][r]) * K[m][c]
                const double ar = K[2 * (m * D + r)], ai = -K[2 * (m * D + r) + 1];
                const double br = K[2 * (m * D + c)], bi = K[2 * (m * D + c) + 1];
                gr += ar * br - ai * bi;
                gi += ar * bi + ai * br;
            }
            G[2 * (r * D + c)] = gr;
            G[2 * (r * D + c) + 1] = gi;
        }
}

// c when G = c I within 1e-12 of G's largest entry, else -1
static double scalar_of(int D, const double *G)
{
    double mx = 0;
    for (int i = 0; i < 2 * D * D; ++i) mx = std::max(mx, std::fabs(G[i]));
    const double c = G[0], tol = 1e-12 * std::max(mx, 1e-300);
    for (int r = 0; r < D; ++r)
        for (int cc = 0; cc < D; ++cc) {
            const double wr = r == cc ? c : 0.0;
            if (std::fabs(G[2 * (r * D + cc)] - wr) > tol || std::fabs(G[2 * (r * D + cc) + 1]) > tol) return -1.0;
        }
    return c;
}

hq_status run_trajectory(void *state, int n, hq_dtype dt, const hq_noisy_op *ops, int nops, const double *u,
                         int *chosen, const hq_config *cfg, cudaStream_t s)
{
    // Channels whose Kraus operators all have K^dag K = p_i I (Pauli channels)
    // are sampled here from p_i alone: the chosen, renormalised operator joins
    // the run of gates (nothing at all when it is the identity).  The others
    // are sampled on the device from the state.
    struct Dev { int op, ch; size_t koff, goff, aoff; };
    std::vector<Dev> dev;
    std::vector<double> hostbuf;  // K then G of each device-sampled channel, then their uniforms
    std::vector<std::vector<double>> kept;  // renormalised operators the gate runs point into
    // 0 gate, 1 host-sampled (applied), 2 host-sampled identity, 3 device,
    // 4 absorbed into the next device-sampled channel
    std::vector<int> plan(nops, 0);
    std::vector<int> pick_of(nops, -1);
    std::vector<const double *> mat_of(nops, nullptr);  // the matrix applied for plans 0 and 1
    int nch = 0;
    std::vector<double> G;
    for (int i = 0; i < nops; ++i) {
        if (ops[i].nkraus == 0) {
            mat_of[i] = ops[i].matrix;
            continue;
        }
        const int D = 1 << ops[i].k, nK = ops[i].nkraus;
        const size_t msz = size_t(2) * D * D;
        G.assign(msz * nK, 0.0);
        bool mixture = true;
        std::vector<double> p(nK);
        for (int j = 0; j < nK; ++j) {
            gram(D, ops[i].matrix + j * msz, G.data() + j * msz);
            p[j] = scalar_of(D, G.data() + j * msz);
            mixture = mixture && p[j] >= 0;
        }
        if (mixture) {
            double total = 0;
            for (double v : p) total += v;
            if (!(total > 0)) {
                set_last_error_text("hq_run_trajectory: a channel whose Kraus operators are all zero");
                return HQ_ERR_ARG;
            }
            const double target = u[nch] * total;
            int pick = -1;
            double cum = 0;
            for (int j = 0; j < nK; ++j) {
                cum += p[j];
                if (p[j] > 0) pick = j;
                if (cum > target && p[j] > 0) {
                    pick = j;
                    break;
                }
            }
            std::vector<double> m(ops[i].matrix + pick * msz, ops[i].matrix + (pick + 1) * msz);
            const double sc = 1.0 / std::sqrt(p[pick]);
            bool identity = true;
            for (int r = 0; r < D; ++r)
                for (int c = 0; c < D; ++c) {
                    m[2 * (r * D + c)] *= sc;
                    m[2 * (r * D + c) + 1] *= sc;
                    identity = identity && std::hypot(m[2 * (r * D + c)] - (r == c ? 1.0 : 0.0),
                                                      m[2 * (r * D + c) + 1]) <= 4.0 * 2.220446049250313e-16;
                }
            plan[i] = identity ? 2 : 1;
            pick_of[i] = pick;
            if (chosen) chosen[nch] = pick;
            kept.push_back(std::move(m));
            if (!identity) mat_of[i] = kept.back().data();
        } else {
            plan[i] = 3;
            Dev d{i, nch, hostbuf.size(), 0, 0};
            hostbuf.insert(hostbuf.end(), ops[i].matrix, ops[i].matrix + msz * nK);
            d.goff = hostbuf.size();
            hostbuf.insert(hostbuf.end(), G.begin(), G.end());
            // absorb the operators applied right before, on the same qubits in
            // the same order (identity branches in between apply nothing):
            // A = M_last ... M_first
            std::vector<double> A(msz, 0.0), T(msz);
            for (int r = 0; r < D; ++r) A[2 * (r * D + r)] = 1.0;
            for (int j = i - 1; j >= 0; --j) {
                if (plan[j] == 2) continue;
                if (plan[j] != 0 && plan[j] != 1) break;
                if (ops[j].k != ops[i].k) break;
                bool same = true;
                for (int q = 0; q < ops[i].k; ++q) same = same && ops[j].qubits[q] == ops[i].qubits[q];
                if (!same) break;
                const double *M = mat_of[j];  // A <- A M (M came before the ops already in A)
                for (int r = 0; r < D; ++r)
                    for (int c = 0; c < D; ++c) {
                        double tr = 0, ti = 0;
                        for (int z = 0; z < D; ++z) {
                            const double ar = A[2 * (r * D + z)], ai = A[2 * (r * D + z) + 1];
                            const double mr = M[2 * (z * D + c)], mi = M[2 * (z * D + c) + 1];
                            tr += ar * mr - ai * mi;
                            ti += ar * mi + ai * mr;
                        }
                        T[2 * (r * D + c)] = tr;
                        T[2 * (r * D + c) + 1] = ti;
                    }
                A.swap(T);
                plan[j] = 4;
            }
            d.aoff = hostbuf.size();
            hostbuf.insert(hostbuf.end(), A.begin(), A.end());
            dev.push_back(d);
        }
        ++nch;
    }
    // device workspace: operator data, uniforms, partial sums, the selected
    // operator, chosen indices, status
    const size_t uoff = hostbuf.size();
    for (const Dev &d : dev) hostbuf.push_back(u[d.ch]);
    // (n < 4: the per-channel kernels; a window kernel's threads hold four qubits)
    const bool windows = n >= 4;
    const int width = windows ? kWindowRow : 2 * rdm_entries<2>();  // doubles per row
    const int grid = windows ? window_grid(n, dt)
                   : std::max(dt == HQ_C64 ? std::max(rdm_grid<float, 1>(n), rdm_grid<float, 2>(n))
                                           : std::max(rdm_grid<double, 1>(n), rdm_grid<double, 2>(n)), 1);
    // two sets of partial sums: a window kernel writes the next one's while other CTAs still read its own
    const size_t nd = hostbuf.size() + size_t(2) * grid * width + 2 * 16 + 1;
    const size_t bytes = nd * sizeof(double) + sizeof(int) * (dev.size() + 1);
    char *ws = nullptr;
    if (!dev.empty()) {
        if (injected_alloc_failure() || !scratch_alloc((void **)&ws, bytes, s)) return HQ_ERR_ALLOC;
        hq_status cs = upload_async(ws, hostbuf.data(), sizeof(double) * hostbuf.size(), s);
        if (cs == HQ_OK)
            cs = cuda_status("clear chosen", cudaMemsetAsync(ws + nd * sizeof(double), 0, sizeof(int) * (dev.size() + 1), s));
        if (cs != HQ_OK) {
            scratch_free(ws, s);
            return cs;
        }
    }
    double *dbuf = reinterpret_cast<double *>(ws);
    double *partials = dbuf ? dbuf + hostbuf.size() : nullptr;
    double *sel = partials ? partials + size_t(2) * grid * width : nullptr;
    int *chosen_dev = ws ? reinterpret_cast<int *>(ws + nd * sizeof(double)) : nullptr;
    int *status_dev = chosen_dev ? chosen_dev + dev.size() : nullptr;

    hq_status st = HQ_OK;
    std::vector<hq_gate> run;
    size_t di = 0;
    auto flush = [&]() -> hq_status {
        if (run.empty()) return HQ_OK;
        hq_status r = hq_apply_blocks(state, n, dt, run.data(), int(run.size()), cfg, s);
        run.clear();
        return r;
    };
    // windows of device-sampled channels (k_window)
    size_t done = 0;      // channels before this one are in launched windows
    bool fed = false;     // the partial sums of the next window are there
    int side = 0;         // the set that holds them
    auto applied_between = [&](int x) {  // an operator applied between channels x and x + 1
        for (int j = dev[x].op + 1; j < dev[x + 1].op; ++j)
            if (plan[j] == 0 || plan[j] == 1) return true;
        return false;
    };
    auto shares_qubit = [&](int x, int y) {
        const hq_noisy_op &a = ops[dev[x].op], &b = ops[dev[y].op];
        for (int i = 0; i < a.k; ++i)
            for (int j = 0; j < b.k; ++j)
                if (a.qubits[i] == b.qubits[j]) return true;
        return false;
    };
    auto window_end = [&](size_t x) {  // last channel of the window that starts with channel x
        const bool two = x + 1 < dev.size() && ops[dev[x].op].k == 1 && ops[dev[x + 1].op].k == 1 &&
                         !shares_qubit(int(x), int(x) + 1) && !applied_between(int(x));
        return int(x) + (two ? 1 : 0);
    };
    for (int i = 0; i < nops && st == HQ_OK; ++i) {
        if (plan[i] == 0 || plan[i] == 1) {
            hq_gate g;
            std::memset(&g, 0, sizeof(g));
            g.k = ops[i].k;
            for (int j = 0; j < g.k; ++j) g.qubits[j] = ops[i].qubits[j];
            g.matrix = mat_of[i];
            run.push_back(g);
        }
        if (plan[i] != 3) continue;
        if (windows) {
            if (di < done) {  // the second channel of the window before
                ++di;
                continue;
            }
            if ((st = flush()) != HQ_OK) break;
            const int last = window_end(di);
            // the next window's sums ride along when nothing is applied between and the qubits differ
            int next_end = -1;
            if (last + 1 < int(dev.size()) && !applied_between(last)) {
                next_end = window_end(last + 1);
                for (int x = int(di); x <= last; ++x)
                    for (int y = last + 1; y <= next_end; ++y)
                        if (shares_qubit(x, y)) next_end = -1;
            }
            auto qubits_of = [&](int first, int end, int *q) {
                int k = 0;
                for (int x = first; x <= end; ++x)
                    for (int j = 0; j < ops[dev[x].op].k; ++j) q[k++] = ops[dev[x].op].qubits[j];
                return k;
            };
            int qa[2], qb[2];
            const int na = qubits_of(int(di), last, qa);
            WindowParam w;
            if (!fed) {
                std::memset(&w, 0, sizeof(w));
                window_bits(w, n, 0, nullptr, na, qa);
                w.out = partials + size_t(side) * grid * width;
                st = launch_window(w, state, n, dt, s);
                if (st != HQ_OK) break;
            }
            std::memset(&w, 0, sizeof(w));
            const int nb = next_end < 0 ? 0 : qubits_of(last + 1, next_end, qb);
            window_bits(w, n, na, qa, nb, qb);
            w.nch = last - int(di) + 1;
            for (int x = 0; x < w.nch; ++x) {
                const Dev &d = dev[di + x];
                w.K[x] = dbuf + d.koff;
                w.G[x] = dbuf + d.goff;
                w.A[x] = dbuf + d.aoff;
                w.u[x] = dbuf + uoff + di + x;
                w.nK[x] = ops[d.op].nkraus;
                w.chosen[x] = chosen_dev + di + x;
            }
            w.status = status_dev;
            w.in = partials + size_t(side) * grid * width;
            w.rows = grid;
            side ^= 1;
            w.out = partials + size_t(side) * grid * width;
            st = launch_window(w, state, n, dt, s);
            fed = nb > 0;
            done = size_t(last) + 1;
            ++di;
            continue;
        }
        if ((st = flush()) != HQ_OK) break;
        const Dev &d = dev[di];
        PickArgs a;
        std::memset(&a, 0, sizeof(a));
        a.partials = partials;
        a.nK = ops[i].nkraus;
        a.K = dbuf + d.koff;
        a.G = dbuf + d.goff;
        a.A = dbuf + d.aoff;
        a.u = dbuf + uoff + di;
        a.chosen = chosen_dev + di;
        a.sel = sel;
        a.status = status_dev;
        if (dt == HQ_C64)
            st = ops[i].k == 1 ? sample_on_device<float, 1>(state, n, ops[i].qubits, a, s)
                               : sample_on_device<float, 2>(state, n, ops[i].qubits, a, s);
        else
            st = ops[i].k == 1 ? sample_on_device<double, 1>(state, n, ops[i].qubits, a, s)
                               : sample_on_device<double, 2>(state, n, ops[i].qubits, a, s);
        ++di;
    }
    if (st == HQ_OK) st = flush();
    if (!ws) return st;
    std::vector<int> back(dev.size() + 1, 0);
    if (st == HQ_OK)
        st = cuda_status("copy chosen", cudaMemcpyAsync(back.data(), chosen_dev, sizeof(int) * back.size(),
                                                        cudaMemcpyDeviceToHost, s));
    scratch_free(ws, s);
    if (st == HQ_OK) st = cuda_status("sync", cudaStreamSynchronize(s));
    if (st != HQ_OK) return st;
    if (back[dev.size()]) {
        set_last_error_text("hq_run_trajectory: every Kraus operator of a channel annihilates the state");
        return HQ_ERR_ARG;
    }
    if (chosen)
        for (size_t j = 0; j < dev.size(); ++j) chosen[dev[j].ch] = back[j];
    return HQ_OK;
}

}  // namespace hq
