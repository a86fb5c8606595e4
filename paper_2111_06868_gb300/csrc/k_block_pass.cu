// k_block_pass.cu -- passes of dense 3- and 4-qubit blocks (complex64): several
// blocks per trip through HBM.
//
// A pass holds a tile of 2^L amplitudes in shared memory (the lowest bits as
// contiguous runs, plus higher bits, as k_runs.cu chooses them), multiplies up
// to NB blocks of K qubits into it one after another and writes it back.  The
// blocks are the gates of a list fused as Sec. 3.1's compress does (HybridQ,
// arXiv 2111.06868), products in double on the host.  The multiply is
// k_gather_pair's: a thread takes whole groups, a row of the product is two
// sums of packed FMAs whose matrix operands are constant-bank words of the
// parameter block (the blocks are unrolled, so every entry has a fixed place).
//
// Why blocks and not the gates themselves (k_runs): a random-circuit layer costs
// about 4 FMAs per gate and amplitude either way, but the register runs spend as
// many integer-pipe moves as FMAs, and a block's body is nothing but FMAs.
//
// Bound: the FP32 pipe and the issue slots (n = 26, K = 3: issue 62 %, FMA pipe 53 % busy); 8 K = 3 blocks need 1.9
// ms of FMAs at n = 28 against 0.63 ms of HBM time per pass.
// n = 28, 785-gate fSim circuit: 87 ms in register runs, 54.7 in 139 three-qubit blocks (25 passes).  Lists of
// 4-qubit blocks, n = 28: 64.1 ms one launch per block (k_gather_pair), 59.3 in passes; 3-qubit blocks n = 24: 3.72 -> 2.00
// ms, n = 12: 213 -> 67 us.
#include <cmath>
#include <cstring>
#include <vector>

#include "hq_block_pass.cuh"
#include "hq_cp_async.cuh"
#include "hq_internal.cuh"

namespace hq {

namespace {

constexpr int kBpThreads = 256;
constexpr int kBpCopies = 16;  // 16-byte copies of a 2^13 tile per thread

template <int K, int NB> struct BlockPassParam {
    int n, L, c, nb;
    uint8_t hi[16];        // flat bits of the tile's positions c.., ascending
    int asc[NB][K];        // tile positions of each block's qubits, ascending
    int off[NB][1 << K];   // swizzled byte offset of local index r (bit j of r: position asc[j])
    ulonglong2 a[NB][1 << K][1 << K];  // (re, re), (im, im)
};

// XOR of the low four bits with every higher group of four: linear, 16 lanes on positions of different residue
// modulo 4 hit different banks
__host__ __device__ __forceinline__ int bswz(int i) { return i ^ ((i >> 4) & 15) ^ ((i >> 8) & 15) ^ ((i >> 12) & 15); }

__device__ __forceinline__ unsigned long long b_mul(unsigned long long x, unsigned long long y)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(x), "l"(y));
    return d;
}
__device__ __forceinline__ unsigned long long b_fma(unsigned long long x, unsigned long long y, unsigned long long z)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(x), "l"(y), "l"(z));
    return d;
}

template <int K, int NB>
__global__ void __launch_bounds__(kBpThreads, 3) k_block_pass(const __grid_constant__ BlockPassParam<K, NB> p,
                                                                          float2 *__restrict__ state)
{
    constexpr int D = 1 << K;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *const tile = reinterpret_cast<float2 *>(smem_raw);
    __shared__ int64_t s_off[kBpCopies];  // flat offset of a thread's k-th copy from its first
    const int L = p.L, c = p.c, nh = L - c, TS = 1 << L;
    auto offset = [&](int i) {  // tile index -> flat offset; additive over disjoint bits
        int64_t off = i & ((1 << c) - 1);
        for (int q = 0; q < nh; ++q)
            if ((i >> (c + q)) & 1) off += int64_t(1) << p.hi[q];
        return off;
    };
    constexpr int STEP = 2 * kBpThreads;
    const int copies = TS / STEP;  // L >= 9
    const int first = threadIdx.x * 2;
    const int64_t off_first = offset(first);
    if (int(threadIdx.x) < copies) s_off[threadIdx.x] = offset(threadIdx.x * STEP);
    __syncthreads();
    const int s_first = bswz(first);
    const int64_t ntiles = int64_t(1) << (p.n - L);
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        int64_t base = t << c;
        for (int q = 0; q < nh; ++q) {
            const int b = p.hi[q];
            base = ((base >> b) << (b + 1)) | (base & ((int64_t(1) << b) - 1));
        }
        float2 *const g = state + base + off_first;
#pragma unroll 4
        for (int k = 0; k < copies; ++k) {
            const float2 *src = g + s_off[k];
            const int s = s_first ^ bswz(k * STEP);
            if (s & 1) {  // the pair's amplitudes trade places
                cp_async8(&tile[s], src);
                cp_async8(&tile[s ^ 1], src + 1);
            } else {
                cp_async16(&tile[s], src);
            }
        }
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            if (b < p.nb) {
#pragma unroll 1
                for (int grp = threadIdx.x; grp < (TS >> K); grp += kBpThreads) {
                    int i0 = grp;
#pragma unroll
                    for (int j = 0; j < K; ++j) {
                        const int q = p.asc[b][j];
                        i0 = ((i0 >> q) << (q + 1)) | (i0 & ((1 << q) - 1));
                    }
                    const int a0 = bswz(i0) * int(sizeof(float2));
                    unsigned long long v[D];
#pragma unroll
                    for (int r = 0; r < D; ++r)
                        v[r] = *reinterpret_cast<const unsigned long long *>(smem_raw + (a0 ^ p.off[b][r]));
#pragma unroll
                    for (int r = 0; r < D; ++r) {
                        unsigned long long A = b_mul(p.a[b][r][0].x, v[0]), B = b_mul(p.a[b][r][0].y, v[0]);
#pragma unroll
                        for (int x = 1; x < D; ++x) {
                            A = b_fma(p.a[b][r][x].x, v[x], A);
                            B = b_fma(p.a[b][r][x].y, v[x], B);
                        }
                        float ax, ay, bx, by;
                        asm("mov.b64 {%0, %1}, %2;" : "=f"(ax), "=f"(ay) : "l"(A));
                        asm("mov.b64 {%0, %1}, %2;" : "=f"(bx), "=f"(by) : "l"(B));
                        *reinterpret_cast<float2 *>(smem_raw + (a0 ^ p.off[b][r])) = make_float2(ax - by, ay + bx);
                    }
                }
                __syncthreads();
            }
        }
#pragma unroll 4
        for (int k = 0; k < copies; ++k) {
            const int s = s_first ^ bswz(k * STEP);
            float4 w = *reinterpret_cast<const float4 *>(&tile[s & ~1]);
            if (s & 1) w = make_float4(w.z, w.w, w.x, w.y);
            *reinterpret_cast<float4 *>(g + s_off[k]) = w;
        }
        __syncthreads();
    }
}

// M (2^K x 2^K on the K bits of `blk`) <- gate * M
void multiply_in(TileBlock &blk, int K, int n, const hq_gate &g)
{
    const int D = 1 << K, k = g.k, KD = 1 << k;
    int at[HQ_MAX_K];  // local bit of the gate's qubit j
    int all = 0;
    for (int j = 0; j < k; ++j) {
        const int b = n - 1 - g.qubits[j];
        for (int x = 0; x < blk.k; ++x)
            if (blk.bit[x] == b) at[j] = x;
        all |= 1 << at[j];
    }
    int idx[16];
    double in[32];
    for (int r = 0; r < KD; ++r) {
        idx[r] = 0;
        for (int j = 0; j < k; ++j)
            if ((r >> (k - 1 - j)) & 1) idx[r] |= 1 << at[j];
    }
    for (int x0 = 0; x0 < D; ++x0) {
        if (x0 & all) continue;
        for (int col = 0; col < D; ++col) {
            for (int r = 0; r < KD; ++r) {
                in[2 * r] = blk.m[2 * ((x0 | idx[r]) * D + col)];
                in[2 * r + 1] = blk.m[2 * ((x0 | idx[r]) * D + col) + 1];
            }
            for (int r = 0; r < KD; ++r) {
                double sr = 0, si = 0;
                for (int c = 0; c < KD; ++c) {
                    const double mr = g.matrix[2 * (r * KD + c)], mi = g.matrix[2 * (r * KD + c) + 1];
                    if (mr == 0.0 && mi == 0.0) continue;
                    sr += mr * in[2 * c] - mi * in[2 * c + 1];
                    si += mr * in[2 * c + 1] + mi * in[2 * c];
                }
                blk.m[2 * ((x0 | idx[r]) * D + col)] = sr;
                blk.m[2 * ((x0 | idx[r]) * D + col) + 1] = si;
            }
        }
    }
}

void identity_block(TileBlock &blk, int K, uint64_t qubits)
{
    const int D = 1 << K;
    blk.k = 0;
    for (uint64_t q = qubits; q; q &= q - 1) blk.bit[blk.k++] = __builtin_ctzll(q);
    std::memset(blk.m, 0, sizeof(double) * size_t(2 * D * D));
    for (int r = 0; r < D; ++r) blk.m[2 * (r * D + r)] = 1.0;
}

// Whether the product can stand in FP32 for its gates one after another: the
// largest part of every column (that is not all zero) within 2^-64 .. 2^64.  Gates
// far from unitary (scaled by 1e25, say) make products outside FP32's range
// (overflow to infinity, flush to 0) although every state between them is inside.
bool float_range(const TileBlock &blk, int K)
{
    const int D = 1 << K;
    for (int c = 0; c < D; ++c) {
        double mx = 0;
        bool number = true;
        for (int r = 0; r < D; ++r)
            for (int x = 0; x < 2; ++x) {
                const double v = std::fabs(blk.m[2 * (r * D + c) + x]);
                number = number && v <= 0x1p64;  // (false for NaN)
                mx = std::max(mx, v);
            }
        if (!number || (mx != 0.0 && mx < 0x1p-64)) return false;
    }
    return true;
}

// sc.set: the qubits of each block; sc.member: the block of each listed gate
void group_in_tile(int n, int K, const hq_gate *gates, const std::vector<int> &list, BlockScratch &sc)
{
    sc.set.clear();
    sc.member.clear();
    for (int g : list) {
        uint64_t q = 0;
        for (int j = 0; j < gates[g].k; ++j) q |= uint64_t(1) << (n - 1 - gates[g].qubits[j]);
        // the latest block that shares a qubit when the union fits, else the first later one that fits, else a new one
        int i = int(sc.set.size()) - 1, to = -1;
        while (i >= 0 && !(sc.set[size_t(i)] & q)) --i;
        if (i >= 0 && __builtin_popcountll(sc.set[size_t(i)] | q) <= K) to = i;
        for (int j = i + 1; to < 0 && j < int(sc.set.size()); ++j)
            if (__builtin_popcountll(sc.set[size_t(j)] | q) <= K) to = j;
        if (to < 0) {
            sc.set.push_back(0);
            to = int(sc.set.size()) - 1;
        }
        sc.set[size_t(to)] |= q;
        sc.member.push_back(to);
    }
}

// The listed gates (a valid order, every qubit in the tile T, none wider than K) fused into blocks of exactly K
// qubits; emit(block) for each in order, until one returns an error.
template <typename Emit>
hq_status fuse_in_tile(int n, int K, uint64_t T, const hq_gate *gates, const std::vector<int> &list, BlockScratch &sc,
                       Emit emit)
{
    group_in_tile(n, K, gates, list, sc);
    TileBlock blk;
    hq_status st = HQ_OK;
    for (size_t b = 0; b < sc.set.size() && st == HQ_OK; ++b) {
        // a block of fewer qubits is widened by the tile's highest other bits (identity there)
        uint64_t set = sc.set[b];
        for (int x = 63; x >= 0 && __builtin_popcountll(set) < K; --x)
            if (((T >> x) & 1) && !((set >> x) & 1)) set |= uint64_t(1) << x;
        identity_block(blk, K, set);
        for (size_t i = 0; i < list.size(); ++i)
            if (sc.member[i] == int(b)) multiply_in(blk, K, n, gates[list[i]]);
        if (float_range(blk, K)) {
            st = emit(blk);
            continue;
        }
        // the product leaves FP32's range where its gates need not: one block per gate
        for (size_t i = 0; i < list.size() && st == HQ_OK; ++i)
            if (sc.member[i] == int(b)) {
                identity_block(blk, K, set);
                multiply_in(blk, K, n, gates[list[i]]);
                st = emit(blk);
            }
    }
    return st;
}

template <int K, int NB>
hq_status launch_blocks(void *state, int n, int L, uint64_t T, const hq_gate *gates, const std::vector<int> &list,
                        BlockScratch &sc, cudaStream_t s)
{
    constexpr int D = 1 << K;
    BlockPassParam<K, NB> p;
    p.n = n;
    p.L = L;
    p.nb = 0;
    int pos[HQ_MAX_N], m = 0, c = 0;
    while (c < n && ((T >> c) & 1)) ++c;
    p.c = c;
    for (int b = 0; b < n; ++b)
        if ((T >> b) & 1) {
            if (m >= c) p.hi[m - c] = uint8_t(b);
            pos[b] = m++;
        }
    auto launch = [&]() -> hq_status {
        const size_t smem = sizeof(float2) << L;
        const void *fn = (const void *)k_block_pass<K, NB>;
        const int grid = grid_for(fn, kBpThreads, smem, int64_t(1) << (n - L));
        k_block_pass<K, NB><<<grid, kBpThreads, smem, s>>>(p, (float2 *)state);
        p.nb = 0;
        return cuda_status("k_block_pass", cudaGetLastError());
    };
    // NB blocks at a time: the first launch runs while the host multiplies the next ones
    hq_status st = fuse_in_tile(n, K, T, gates, list, sc, [&](const TileBlock &blk) -> hq_status {
        const int b = p.nb++;
        for (int j = 0; j < K; ++j) p.asc[b][j] = pos[blk.bit[j]];  // (ascending as the flat bits are)
        for (int r = 0; r < D; ++r) {
            int i = 0;
            for (int j = 0; j < K; ++j)
                if ((r >> j) & 1) i |= 1 << p.asc[b][j];
            p.off[b][r] = bswz(i) * int(sizeof(float2));
            for (int x = 0; x < D; ++x) {
                const double *e = blk.m + 2 * (r * D + x);
                const float re[2] = {float(e[0]), float(e[0])}, im[2] = {float(e[1]), float(e[1])};
                std::memcpy(&p.a[b][r][x].x, re, 8);
                std::memcpy(&p.a[b][r][x].y, im, 8);
            }
        }
        return p.nb == NB ? launch() : HQ_OK;
    });
    return st == HQ_OK && p.nb > 0 ? launch() : st;
}

}  // namespace

int count_in_tile(int n, int K, const hq_gate *gates, const std::vector<int> &list, BlockScratch &sc)
{
    group_in_tile(n, K, gates, list, sc);
    return int(sc.set.size());
}

hq_status launch_block_pass(void *state, int n, int L, uint64_t T, int K, const hq_gate *gates,
                            const std::vector<int> &list, BlockScratch &sc, cudaStream_t s)
{
    if (K == 3) return launch_blocks<3, kBlocks3>(state, n, L, T, gates, list, sc, s);
    return launch_blocks<4, kBlocks4>(state, n, L, T, gates, list, sc, s);
}

}  // namespace hq
