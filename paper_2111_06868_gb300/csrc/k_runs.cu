// k_runs.cu -- lists of narrow gates in passes: many gates per trip through HBM.
//
// HybridQ (arXiv 2111.06868) Sec. 4.2 applies the gates of a circuit one after
// another.  One launch per gate reads and writes the whole state for a few
// multiply-adds per amplitude (a dense one-qubit gate: 16 or 32 bytes for 8
// FMAs), and on a small state it is a launch for microseconds of work.  Here a
// run of consecutive gates is grouped into passes: a pass holds a tile of 2^L
// amplitudes (the lowest bits as contiguous runs, plus higher bits chosen for
// the gates at hand) in shared memory, applies every gate whose qubits allow it
// and writes the tile back.
//
//   * What a gate asks of the tile: only the bits it mixes.  A diagonal gate
//     mixes none (its phase follows from the amplitude's index, wherever its
//     bits are), a controlled one-target gate only its target.
//   * Inside a pass the gates form register runs: a run fixes up to RP tile
//     bits, a thread loads the 2^RP amplitudes that differ in them (RP = 4 for
//     complex64, 3 for complex128: 32 registers), applies all gates of the run
//     to them and stores them back: one trip through shared memory and one
//     barrier per run instead of per gate.
//   * Gates only ever move past gates they share no qubit with, so the product
//     is the same; every gate is the same multiply-add chain as in k_apply.cu.
//
// Products with an exactly zero real or imaginary part of a matrix entry are left out (sqrt(X), sqrt(Y), H, RY: half
// of the multiply-adds; phases 1, -1, +-i: none), and an exchange of two qubits (SWAP, fSim(pi/2, phi)) only renames
// register bits.
//
// What bounds it: complex64 instruction issue (n=26, ncu: 57 % issue, integer pipe 60 % of its half rate: the
// moves that a packed FMA's crosswise operand needs and shared-memory addresses; DRAM 16 %), complex128 the FP64 pipe.
// Tried and slower, n=28 circuit (785 gates): 8 amplitudes per thread 123 ms, scalar FMAs 120 ms, packed real and
// scalar imaginary products 94 ms, 512 threads at 64 registers 102 ms, two CTAs per SM 95 ms, against 87 ms.
// From 23 qubits on (and for 3- and 4-qubit gates) a complex64 pass may instead fuse its gates into dense blocks
// (k_block_pass.cu); the kind that does more work per time is chosen pass by pass, and the gates' own kernels where their
// estimated time is below that of the pass (own_kernels_faster).
// Per-gate circuits, against one launch per gate: n=28 complex64 depth 20 fSim 528 -> 87 ms (55 in blocks), n=20
// depth 16 CZ 1.53 -> 0.25 ms of device time, n=12 complex128 depth 10 1.06 -> 0.20 ms.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "hq_block_pass.cuh"
#include "hq_cp_async.cuh"
#include "hq_internal.cuh"

namespace hq {

namespace {

// ----------------------------------------------------------------------------
// the plan of one pass, passed to the kernel by value
// ----------------------------------------------------------------------------
constexpr int kMaxRuns = 36;    // register runs
constexpr int kMaxOps = 120;    // gates
constexpr int kMaxPool = 352;   // complex matrix entries
constexpr int kMaxAux = 256;    // bytes of diagonal gates' bit descriptions
constexpr int kMaxTile = 13;    // bits of a tile
constexpr int kMaxCopies = 32;  // 16-byte copies of a tile per thread

enum OpKind : uint8_t {
    OP_U1 = 0,    // dense 2 x 2 on register position var, where all controls are 1
    OP_U2 = 1,    // dense 4 x 4 on the register position pair var
    OP_D2 = 2,    // a phase for each value of the pair var
    OP_PH = 3,    // a phase where all controls are 1 (var: controls among the register positions)
    OP_DG = 4,    // a diagonal gate of k qubits by its table
    OP_BLK = 5    // a 3- or 4-qubit gate that only a pass of dense blocks takes (k_block_pass.cu)
};

// zero parts of a 2 x 2 matrix (sqrt(Y), H, RY: real; sqrt(X), RX: real diagonal, imaginary off it; sqrt(W): real
// diagonal): their products are left out
enum U1Class : uint8_t { U1_FULL = 0, U1_REAL = 1, U1_REAL_IMAG = 2, U1_REAL_FULL = 3 };
// phases that cost no multiplication
enum PhaseKind : uint8_t { PHASE_ANY = 0, PHASE_ONE = 1, PHASE_MINUS = 2, PHASE_I = 3 };  // I: i or -i

// register position pairs (p < q) by number: 01 02 03 12 13 23
inline int pair_no(int p, int q) { return p == 0 ? q - 1 : p == 1 ? q + 1 : 5; }

// gate bodies: U1 + 4 position + class, PH + mask of register bits, U2 and D2 + pair
enum OpCode : uint8_t { CODE_U1 = 0, CODE_PH = 16, CODE_U2 = 32, CODE_D2 = 38, CODE_DG = 44 };

struct alignas(16) RunOp {
    uint8_t code;    // the gate body (op_code)
    uint8_t var;     // U1, PH: 1 when there are controls to test
    uint8_t k;       // DG: qubits
    uint8_t flags;   // OP_U1: which parts of the matrix are zero (U1Class); OP_PH: 1 for the phase -1
    uint16_t mat;    // first entry in the pool, in bytes
    uint16_t lmask;  // OP_U1, OP_PH: control bits among the tile's bits; OP_DG: first byte in aux;
                     // OP_D2: 4 bits per entry (PhaseKind)
    uint64_t omask;               // control bits outside the tile (flat)
};
struct RunDesc {
    uint8_t reg[4];    // tile position each register bit is loaded from
    uint8_t out[4];    // and stored to: exchanges of two qubits only rename register bits
    uint8_t thr[12];   // tile position of each thread-index bit (31: unused)
    uint16_t op0, op1;
};

template <typename R> struct Traits;
template <> struct Traits<float> {
    static constexpr int RP = 4, NB = 4;  // register positions; 8-byte slots per bank row (log2)
};
template <> struct Traits<double> {
    static constexpr int RP = 3, NB = 3;
};

template <typename R> struct PassParam {
    int n, L, c, nruns, nops, npool, naux, pad;
    uint8_t hi[16];  // flat bits of the tile's positions c.., ascending
    RunDesc run[kMaxRuns];
    RunOp op[kMaxOps];
    uint8_t aux[kMaxAux];
    typename C2<R>::type pool[kMaxPool];
};

// Tile element i lives at slot rswz(i): the low NB bits are XORed with every
// higher group of NB bits, so 2^NB accesses that differ in bits of pairwise
// different position modulo NB hit different banks; linear over XOR.
template <int NB> __host__ __device__ __forceinline__ int rswz(int i)
{
    constexpr int m = (1 << NB) - 1;
    return i ^ ((i >> NB) & m) ^ ((i >> (2 * NB)) & m) ^ ((i >> (3 * NB)) & m) ^ (NB == 3 ? ((i >> 12) & m) : 0);
}

// ----------------------------------------------------------------------------
// gate bodies on a thread's register amplitudes
// ----------------------------------------------------------------------------
// A complex64 amplitude stays one 64-bit register pair (re low, im high) from its load to its store: the packed
// FMAs take and give such pairs, and as a float2 every gate body would end in moves back to common registers.
template <typename R> struct Amp;
template <> struct Amp<float> {
    using type = unsigned long long;
    using entry = ulonglong2;  // a matrix entry in the pool: (re, re), (-im, im)
    static __device__ __forceinline__ entry make(float2 m)
    {
        entry e;
        asm("mov.b64 %0, {%1, %1};" : "=l"(e.x) : "f"(m.x));
        asm("mov.b64 %0, {%1, %2};" : "=l"(e.y) : "f"(-m.y), "f"(m.y));
        return e;
    }
};
template <> struct Amp<double> {
    using type = double2;
    using entry = double2;
    static __device__ __forceinline__ double2 make(double2 m) { return m; }
};

using a64 = unsigned long long;
__device__ __forceinline__ a64 p_mul(a64 x, a64 y)
{
    a64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(x), "l"(y));
    return d;
}
__device__ __forceinline__ a64 p_fma(a64 x, a64 y, a64 z)
{
    a64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(x), "l"(y), "l"(z));
    return d;
}
__device__ __forceinline__ a64 yx(a64 v) { return (v << 32) | (v >> 32); }
__device__ __forceinline__ bool nonzero(double v) { return (__double_as_longlong(v) << 1) != 0; }

// acc[] (+)= m * v[] over N amplitudes; First: acc starts here; Re, Im: parts of m that are not known to be zero
template <int N, bool First, bool Re = true, bool Im = true>
__device__ __forceinline__ void macs(a64 (&acc)[N], const ulonglong2 m, const a64 (&v)[N])
{
#pragma unroll
    for (int i = 0; i < N; ++i) {
        if (Re) acc[i] = First ? p_mul(m.x, v[i]) : p_fma(m.x, v[i], acc[i]);
        if (Im) acc[i] = First && !Re ? p_mul(m.y, yx(v[i])) : p_fma(m.y, yx(v[i]), acc[i]);
    }
}
// complex128: every part is tested (the same for every thread: no divergence), an FP64 multiply-add costs
// 16 cycles of the SM's pipe
template <int N, bool First, bool Re = true, bool Im = true>
__device__ __forceinline__ void macs(double2 (&acc)[N], const double2 m, const double2 (&v)[N])
{
    if (First) {
#pragma unroll
        for (int i = 0; i < N; ++i) acc[i].x = acc[i].y = 0;
    }
    if (Re && nonzero(m.x)) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            acc[i].x = fma(m.x, v[i].x, acc[i].x);
            acc[i].y = fma(m.x, v[i].y, acc[i].y);
        }
    }
    if (Im && nonzero(m.y)) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            acc[i].x = fma(-m.y, v[i].y, acc[i].x);
            acc[i].y = fma(m.y, v[i].x, acc[i].y);
        }
    }
}
__device__ __forceinline__ a64 cprod(const ulonglong2 m, const a64 v) { return p_fma(m.y, yx(v), p_mul(m.x, v)); }
__device__ __forceinline__ double2 cprod(const double2 m, const double2 v) { return cmul(m, v); }
__device__ __forceinline__ a64 negate(a64 v) { return p_mul(v, 0xbf800000bf800000ull); }  // times (-1, -1): one FMA-pipe instruction
__device__ __forceinline__ double2 negate(double2 v) { return make_double2(-v.x, -v.y); }
// (0 + i y) v for an entry whose imaginary part y is +-1: complex128 without an FP64 product
__device__ __forceinline__ a64 times_iy(const ulonglong2 m, a64 v) { return p_mul(m.y, yx(v)); }
__device__ __forceinline__ double2 times_iy(const double2 m, double2 v)
{
    return m.y > 0 ? make_double2(-v.y, v.x) : make_double2(v.y, -v.x);
}

template <typename R, int P, int CLS, int NA>
__device__ __forceinline__ void op_u1_class(typename Amp<R>::type (&a)[NA],
                                      const typename Amp<R>::entry *m)
{
    using T2 = typename Amp<R>::type;
    constexpr int H = NA / 2;
    constexpr int STEP = H < 4 ? H : 4;  // pairs per batch
    constexpr bool DI = CLS == U1_FULL || sizeof(R) == 8, OR = CLS != U1_REAL_IMAG || sizeof(R) == 8, OI = CLS != U1_REAL || sizeof(R) == 8;
    const auto m00 = m[0], m01 = m[1], m10 = m[2], m11 = m[3];
#pragma unroll
    for (int b = 0; b < H; b += STEP) {
        T2 v0[STEP], v1[STEP], o0[STEP], o1[STEP];
#pragma unroll
        for (int i = 0; i < STEP; ++i) {
            const int g = b + i, j = ((g >> P) << (P + 1)) | (g & ((1 << P) - 1));
            v0[i] = a[j];
            v1[i] = a[j | (1 << P)];
        }
        // both products of v0, then both of v1: the last ones can write over their inputs
        macs<STEP, true, true, DI>(o0, m00, v0);
        macs<STEP, true, OR, OI>(o1, m10, v0);
        macs<STEP, false, OR, OI>(o0, m01, v1);
        macs<STEP, false, true, DI>(o1, m11, v1);
#pragma unroll
        for (int i = 0; i < STEP; ++i) {
            const int g = b + i, j = ((g >> P) << (P + 1)) | (g & ((1 << P) - 1));
            a[j] = o0[i];
            a[j | (1 << P)] = o1[i];
        }
    }
}

// group g's base among the register amplitudes, positions P < Q clear
template <int P, int Q> __device__ __forceinline__ constexpr int pair_base(int g)
{
    const int x = ((g >> P) << (P + 1)) | (g & ((1 << P) - 1));
    return ((x >> Q) << (Q + 1)) | (x & ((1 << Q) - 1));
}

template <typename R, int P, int Q, int NA>
__device__ __forceinline__ void op_u2(typename Amp<R>::type (&a)[NA],
                                      const typename Amp<R>::entry *m)
{
    using T2 = typename Amp<R>::type;
    constexpr int NG = NA / 4, STEP = NG < 2 ? NG : 2;
#pragma unroll
    for (int b = 0; b < NG; b += STEP) {
        T2 v[4][STEP], o[4][STEP];
#pragma unroll
        for (int i = 0; i < STEP; ++i)
#pragma unroll
            for (int r = 0; r < 4; ++r) v[r][i] = a[pair_base<P, Q>(b + i) | ((r & 1) << P) | ((r >> 1) << Q)];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            macs<STEP, true>(o[r], m[4 * r], v[0]);
            macs<STEP, false>(o[r], m[4 * r + 1], v[1]);
            macs<STEP, false>(o[r], m[4 * r + 2], v[2]);
            macs<STEP, false>(o[r], m[4 * r + 3], v[3]);
        }
#pragma unroll
        for (int i = 0; i < STEP; ++i)
#pragma unroll
            for (int r = 0; r < 4; ++r) a[pair_base<P, Q>(b + i) | ((r & 1) << P) | ((r >> 1) << Q)] = o[r][i];
    }
}

// entry r of m on the amplitudes whose bits Q, P are r; kinds: 4 bits per entry (PhaseKind)
template <typename R, int P, int Q, int NA>
__device__ __forceinline__ void op_d2(typename Amp<R>::type (&a)[NA],
                                      const typename Amp<R>::entry *m, int kinds)
{
    constexpr int NG = NA / 4;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int kind = (kinds >> (4 * r)) & 15;
        if (kind == PHASE_ONE) continue;
        if (kind == PHASE_ANY) {
            const auto d = m[r];
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const int j = pair_base<P, Q>(g) | ((r & 1) << P) | ((r >> 1) << Q);
                a[j] = cprod(d, a[j]);
            }
        } else {
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const int j = pair_base<P, Q>(g) | ((r & 1) << P) | ((r >> 1) << Q);
                a[j] = kind == PHASE_MINUS ? negate(a[j]) : times_iy(m[r], a[j]);
            }
        }
    }
}

// a phase on the amplitudes whose register bits MASK are all 1
template <typename R, int MASK, int NA>
__device__ __forceinline__ void op_ph(typename Amp<R>::type (&a)[NA],
                                      const typename Amp<R>::entry d, bool minus)
{
    if (minus) {
#pragma unroll
        for (int j = 0; j < NA; ++j)
            if ((j & MASK) == MASK) a[j] = negate(a[j]);
    } else {
#pragma unroll
        for (int j = 0; j < NA; ++j)
            if ((j & MASK) == MASK) a[j] = cprod(d, a[j]);
    }
}

// one gate body per case; Q: the highest register position it uses
#define HQ_CASE(Q, CODE, ...)                             \
    case CODE:                                            \
        if constexpr ((Q) < RP) __VA_ARGS__;              \
        break

template <typename R, int RP>
__device__ __forceinline__ void apply_op(const RunOp &op, typename Amp<R>::type (&a)[1 << RP], int i0,
                                         uint64_t base, const typename Amp<R>::entry *pool, const uint8_t *aux)
{
    constexpr int NA = 1 << RP;
    const auto *m = reinterpret_cast<const typename Amp<R>::entry *>(reinterpret_cast<const char *>(pool) + op.mat);
    if (op.var && ((i0 & op.lmask) != op.lmask || (base & op.omask) != op.omask)) return;  // a control is 0
    switch (op.code) {
    HQ_CASE(0, CODE_U1 + 0, op_u1_class<R, 0, 0>(a, m));
    HQ_CASE(0, CODE_U1 + 1, op_u1_class<R, 0, 1>(a, m));
    HQ_CASE(0, CODE_U1 + 2, op_u1_class<R, 0, 2>(a, m));
    HQ_CASE(0, CODE_U1 + 3, op_u1_class<R, 0, 3>(a, m));
    HQ_CASE(1, CODE_U1 + 4, op_u1_class<R, 1, 0>(a, m));
    HQ_CASE(1, CODE_U1 + 5, op_u1_class<R, 1, 1>(a, m));
    HQ_CASE(1, CODE_U1 + 6, op_u1_class<R, 1, 2>(a, m));
    HQ_CASE(1, CODE_U1 + 7, op_u1_class<R, 1, 3>(a, m));
    HQ_CASE(2, CODE_U1 + 8, op_u1_class<R, 2, 0>(a, m));
    HQ_CASE(2, CODE_U1 + 9, op_u1_class<R, 2, 1>(a, m));
    HQ_CASE(2, CODE_U1 + 10, op_u1_class<R, 2, 2>(a, m));
    HQ_CASE(2, CODE_U1 + 11, op_u1_class<R, 2, 3>(a, m));
    HQ_CASE(3, CODE_U1 + 12, op_u1_class<R, 3, 0>(a, m));
    HQ_CASE(3, CODE_U1 + 13, op_u1_class<R, 3, 1>(a, m));
    HQ_CASE(3, CODE_U1 + 14, op_u1_class<R, 3, 2>(a, m));
    HQ_CASE(3, CODE_U1 + 15, op_u1_class<R, 3, 3>(a, m));
    HQ_CASE(0, CODE_PH + 0, op_ph<R, 0>(a, m[0], op.flags != 0));
    HQ_CASE(0, CODE_PH + 1, op_ph<R, 1>(a, m[0], op.flags != 0));
    HQ_CASE(1, CODE_PH + 2, op_ph<R, 2>(a, m[0], op.flags != 0));
    HQ_CASE(1, CODE_PH + 3, op_ph<R, 3>(a, m[0], op.flags != 0));
    HQ_CASE(2, CODE_PH + 4, op_ph<R, 4>(a, m[0], op.flags != 0));
    HQ_CASE(2, CODE_PH + 5, op_ph<R, 5>(a, m[0], op.flags != 0));
    HQ_CASE(2, CODE_PH + 6, op_ph<R, 6>(a, m[0], op.flags != 0));
    HQ_CASE(3, CODE_PH + 8, op_ph<R, 8>(a, m[0], op.flags != 0));
    HQ_CASE(3, CODE_PH + 9, op_ph<R, 9>(a, m[0], op.flags != 0));
    HQ_CASE(3, CODE_PH + 10, op_ph<R, 10>(a, m[0], op.flags != 0));
    HQ_CASE(3, CODE_PH + 12, op_ph<R, 12>(a, m[0], op.flags != 0));
    HQ_CASE(1, CODE_U2 + 0, op_u2<R, 0, 1>(a, m));
    HQ_CASE(2, CODE_U2 + 1, op_u2<R, 0, 2>(a, m));
    HQ_CASE(3, CODE_U2 + 2, op_u2<R, 0, 3>(a, m));
    HQ_CASE(2, CODE_U2 + 3, op_u2<R, 1, 2>(a, m));
    HQ_CASE(3, CODE_U2 + 4, op_u2<R, 1, 3>(a, m));
    HQ_CASE(3, CODE_U2 + 5, op_u2<R, 2, 3>(a, m));
    HQ_CASE(1, CODE_D2 + 0, op_d2<R, 0, 1>(a, m, op.lmask));
    HQ_CASE(2, CODE_D2 + 1, op_d2<R, 0, 2>(a, m, op.lmask));
    HQ_CASE(3, CODE_D2 + 2, op_d2<R, 0, 3>(a, m, op.lmask));
    HQ_CASE(2, CODE_D2 + 3, op_d2<R, 1, 2>(a, m, op.lmask));
    HQ_CASE(3, CODE_D2 + 4, op_d2<R, 1, 3>(a, m, op.lmask));
    HQ_CASE(3, CODE_D2 + 5, op_d2<R, 2, 3>(a, m, op.lmask));
    default: {
        // aux: 2^RP table offsets of the register bits, then per qubit (in the table's order, most
        // significant first) 0..15 a tile position, 64 + b a flat bit outside the tile, 255 a register bit
        const uint8_t *x = aux + op.lmask;
        int t = 0;
        for (int j = 0; j < op.k; ++j) {
            const int w = x[NA + j];
            int bit = 0;
            if (w < 16) bit = (i0 >> w) & 1;
            else if (w != 255) bit = int((base >> (w - 64)) & 1);
            t |= bit << (op.k - 1 - j);
        }
#pragma unroll
        for (int j = 0; j < NA; ++j) a[j] = cprod(m[t + x[j]], a[j]);
    }
    }
}

// ----------------------------------------------------------------------------
// the pass kernel
// ----------------------------------------------------------------------------
constexpr int kRunThreads = 256;

template <typename R> constexpr size_t pass_smem(int L)
{
    return (sizeof(typename C2<R>::type) << L) + sizeof(typename Amp<R>::entry) * kMaxPool +
           sizeof(RunDesc) * kMaxRuns + sizeof(RunOp) * (kMaxOps + 1) + kMaxAux;
}

template <typename R, int RP>
__global__ void __launch_bounds__(kRunThreads, 3) k_runs(const __grid_constant__ PassParam<R> p,
                                                         typename C2<R>::type *__restrict__ state)
{
    using T2 = typename C2<R>::type;
    using A = typename Amp<R>::type;
    using PE = typename Amp<R>::entry;
    constexpr int NA = 1 << RP, NB = Traits<R>::NB;
    constexpr int V = 16 / int(sizeof(T2));  // amplitudes per 16-byte copy
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = p.L, c = p.c, nh = L - c;
    T2 *const tile = reinterpret_cast<T2 *>(smem_raw);
    PE *const pool = reinterpret_cast<PE *>(smem_raw + (sizeof(T2) << L));
    RunOp *const ops = reinterpret_cast<RunOp *>(pool + kMaxPool);
    RunDesc *const runs = reinterpret_cast<RunDesc *>(ops + kMaxOps + 1);
    uint8_t *const aux = reinterpret_cast<uint8_t *>(runs + kMaxRuns);
    __shared__ int64_t s_off[kMaxCopies];  // flat offset of a thread's k-th 16-byte copy from its first

    for (int i = threadIdx.x; i < p.npool; i += blockDim.x) pool[i] = Amp<R>::make(p.pool[i]);
    for (int i = threadIdx.x; i < p.nops; i += blockDim.x) ops[i] = p.op[i];
    for (int i = threadIdx.x; i < p.nruns; i += blockDim.x) runs[i] = p.run[i];
    for (int i = threadIdx.x; i < p.naux; i += blockDim.x) aux[i] = p.aux[i];
    // tile index -> flat offset; additive over disjoint bits
    auto offset = [&](int i) {
        int64_t off = i & ((1 << c) - 1);
        for (int q = 0; q < nh; ++q)
            if ((i >> (c + q)) & 1) off += int64_t(1) << p.hi[q];
        return off;
    };
    const int step = blockDim.x * V, copies = (1 << L) / step > 0 ? (1 << L) / step : 1;
    const int i_first = threadIdx.x * V;
    const bool copier = i_first < (1 << L);
    const int64_t off_first = offset(i_first & ((1 << L) - 1));
    if (threadIdx.x < copies) s_off[threadIdx.x] = offset(threadIdx.x * step);
    __syncthreads();

    const int64_t ntiles = int64_t(1) << (p.n - L);
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        int64_t base = t << c;
        for (int q = 0; q < nh; ++q) {
            const int b = p.hi[q];
            base = ((base >> b) << (b + 1)) | (base & ((int64_t(1) << b) - 1));
        }
        T2 *const g = state + base + off_first;
        const int s_first = rswz<NB>(i_first);
        if (copier)
            for (int k = 0; k < copies; ++k) {
                const T2 *src = g + s_off[k];
                const int s = s_first ^ rswz<NB>(k * step);
                if (V == 2 && (s & 1)) {  // the pair's amplitudes trade places
                    cp_async8(&tile[s], src);
                    cp_async8(&tile[s ^ 1], src + 1);
                } else {
                    cp_async16(&tile[s], src);
                }
            }
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
        for (int u = 0; u < p.nruns; ++u) {
            const RunDesc &rd = runs[u];
            const int op0 = rd.op0, op1 = rd.op1;
#pragma unroll 1
            for (int w = threadIdx.x; w < (1 << (L - RP)); w += blockDim.x) {
                int i0 = 0;
#pragma unroll
                for (int q = 0; q < kMaxTile - RP; ++q) i0 |= ((w >> q) & 1) << rd.thr[q];
                A a[NA];
                // byte offsets of the register amplitudes: the thread's slot XOR the register bits' slots
                const int a0 = rswz<NB>(i0) * int(sizeof(T2));
                {
                    int e[RP], adr[NA];
#pragma unroll
                    for (int q = 0; q < RP; ++q) e[q] = rswz<NB>(1 << rd.reg[q]) * int(sizeof(T2));
                    adr[0] = a0;
#pragma unroll
                    for (int j = 1; j < NA; ++j) {
                        const int low = j & (-j), q = low == 1 ? 0 : low == 2 ? 1 : low == 4 ? 2 : 3;
                        adr[j] = adr[j ^ low] ^ e[q];
                    }
#pragma unroll
                    for (int j = 0; j < NA; ++j) a[j] = *reinterpret_cast<const A *>(smem_raw + adr[j]);
                }
                RunOp op = ops[op0];
#pragma unroll 1
                for (int o = op0; o < op1; ++o) {
                    const RunOp next = ops[o + 1];  // in flight under this gate (slot kMaxOps exists)
                    apply_op<R, RP>(op, a, i0, uint64_t(base), pool, aux);
                    op = next;
                }
                {
                    int e[RP], adr[NA];
#pragma unroll
                    for (int q = 0; q < RP; ++q) e[q] = rswz<NB>(1 << rd.out[q]) * int(sizeof(T2));
                    adr[0] = a0;
#pragma unroll
                    for (int j = 1; j < NA; ++j) {
                        const int low = j & (-j), q = low == 1 ? 0 : low == 2 ? 1 : low == 4 ? 2 : 3;
                        adr[j] = adr[j ^ low] ^ e[q];
                    }
#pragma unroll
                    for (int j = 0; j < NA; ++j) *reinterpret_cast<A *>(smem_raw + adr[j]) = a[j];
                }
            }
            __syncthreads();
        }
        if (copier)
            for (int k = 0; k < copies; ++k) {
                const int s = s_first ^ rswz<NB>(k * step);
                float4 v = *reinterpret_cast<const float4 *>(&tile[V == 2 ? s & ~1 : s]);
                if (V == 2 && (s & 1)) v = make_float4(v.z, v.w, v.x, v.y);
                *reinterpret_cast<float4 *>(g + s_off[k]) = v;
            }
        __syncthreads();
    }
}

// ----------------------------------------------------------------------------
// planning (host)
// ----------------------------------------------------------------------------
constexpr uint64_t kNever = uint64_t(1) << 63;  // in Item::need: not for register runs

// One gate as the planner sees it.
struct Item {
    OpKind kind;
    bool wide;          // not for this path: applied on its own
    uint8_t nb, pool, aux;
    uint8_t bit[HQ_MAX_K];  // flat bits of its qubits, in their order
    int8_t target;      // OP_U1: index of the target in bit[]
    uint8_t flags;
    bool swap;          // OP_D2: exchange the two qubits first
    uint16_t keep;      // OP_U2: bit 4 r + c set where the entry is not an exact zero
    uint64_t all, need; // flat bits; those that a register run mixes
    double touched;     // share of the state that its own kernel reads and writes (below 1: k_ctrl)
    bool perm;          // OP_BLK: one nonzero entry per row
    double m[8];        // matrix entries (U1: 2x2, D2 and PH: phases); OP_U2 and OP_DG read the gate's own
};

double magnitude(const double *e)
{
    if (e[1] == 0.0) return std::fabs(e[0]);
    if (e[0] == 0.0) return std::fabs(e[1]);
    return std::hypot(e[0], e[1]);
}

uint8_t u1_class(const double *m)
{
    if (m[1] != 0.0 || m[7] != 0.0) return U1_FULL;
    if (m[3] == 0.0 && m[5] == 0.0) return U1_REAL;
    if (m[2] == 0.0 && m[4] == 0.0) return U1_REAL_IMAG;
    return U1_REAL_FULL;
}

int phase_kind(const double *e)
{
    if (e[1] == 0.0) return e[0] == 1.0 ? PHASE_ONE : e[0] == -1.0 ? PHASE_MINUS : PHASE_ANY;
    if (e[0] == 0.0) return e[1] == 1.0 || e[1] == -1.0 ? PHASE_I : PHASE_ANY;
    return PHASE_ANY;
}

// The share of the state that k_ctrl would read and write for this gate (1: not a controlled gate, or one that
// k_ctrl does not take): half per control above the 32-byte sector.  Costs only, so without control_split's exact
// tolerance.
double touched_share(int n, const hq_gate &g, bool diagonal, int sector_bits)
{
    const int k = g.k, K = 1 << k;
    int ctrl = K - 1;  // index bits that are 1 wherever the matrix differs from the identity
    for (int r = 0; r < K && ctrl; ++r)
        for (int c = diagonal ? r : 0; c < (diagonal ? r + 1 : K) && ctrl; ++c) {
            const double *e = g.matrix + 2 * (r * K + c);
            if (std::fabs(e[0] - (r == c ? 1.0 : 0.0)) > 1e-15 || std::fabs(e[1]) > 1e-15) ctrl &= r & c;
        }
    if (k - __builtin_popcount(unsigned(ctrl)) > kMaxCtrlTargets) return 1.0;
    double share = 1.0;
    for (int j = 0; j < k; ++j)
        if (((ctrl >> (k - 1 - j)) & 1) && n - 1 - g.qubits[j] >= sector_bits) share *= 0.5;
    return share;
}

// max_block: the widest dense gate that a pass of blocks may take (2: none); sector_bits: flat bits within 32 bytes
void classify(int n, const hq_gate &g, int max_block, int sector_bits, Item &it)
{
    const int k = g.k, K = 1 << k;
    const double *m = g.matrix;
    it.touched = 1.0;
    it.perm = false;
    it.wide = false;
    it.nb = uint8_t(k);
    it.all = it.need = 0;
    it.aux = 0;
    it.flags = 0;
    it.swap = false;
    it.target = 0;
    for (int j = 0; j < k; ++j) {
        it.bit[j] = uint8_t(n - 1 - g.qubits[j]);
        it.all |= uint64_t(1) << it.bit[j];
    }
    if (is_diagonal(k, m)) {
        it.touched = touched_share(n, g, true, sector_bits);
        bool phase = k <= 2;
        for (int r = 0; phase && r < K - 1; ++r)
            phase = m[2 * (r * K + r)] == 1.0 && m[2 * (r * K + r) + 1] == 0.0;
        if (phase) {
            it.kind = OP_PH;
            it.pool = 1;
            it.m[0] = m[2 * (K * K - 1)];
            it.m[1] = m[2 * (K * K - 1) + 1];
            it.flags = it.m[0] == -1.0 && it.m[1] == 0.0;
        } else {
            it.kind = OP_DG;
            it.pool = uint8_t(K);
            it.aux = uint8_t(16 + k);
        }
        return;
    }
    if (k == 1) {
        it.kind = OP_U1;
        it.pool = 4;
        it.need = it.all;
        std::memcpy(it.m, m, sizeof(double) * 8);
        it.flags = u1_class(it.m);
        return;
    }
    if (k > 2) {
        it.kind = OP_BLK;
        it.wide = k > max_block;
        it.pool = 0;
        it.need = it.all | kNever;
        if (it.wide) return;
        it.touched = touched_share(n, g, false, sector_bits);
        it.perm = true;
        for (int r = 0; r < K && it.perm; ++r) {
            int nz = 0;
            for (int c = 0; c < K && nz < 2; ++c) nz += m[2 * (r * K + c)] != 0.0 || m[2 * (r * K + c) + 1] != 0.0;
            it.perm = nz == 1;
        }
        return;
    }
    // k = 2: a controlled gate, an exchange with phases, or dense.  Entries within 4 FP64 epsilon of the largest
    // magnitude of 0 (or of the identity) count as exact, as in control_split and is_monomial.
    double mx = 0;
    for (int e = 0; e < 16; ++e) mx = std::max(mx, magnitude(m + 2 * e));
    const double tiny = 4.0 * 2.220446049250313e-16 * mx;
    auto is = [&](int r, int c, double v) {
        const double d[2] = {m[2 * (4 * r + c)] - v, m[2 * (4 * r + c) + 1]};
        return magnitude(d) <= tiny;
    };
    for (int j = 0; j < 2; ++j) {
        const int bit = 2 >> j;
        bool ctrl = true;
        for (int r = 0; r < 4 && ctrl; ++r)
            for (int c = 0; c < 4 && ctrl; ++c)
                if (!(r & bit) || !(c & bit)) ctrl = is(r, c, r == c ? 1.0 : 0.0);
        if (!ctrl) continue;
        const int tb = 3 ^ bit;
        it.kind = OP_U1;
        if (n - 1 - g.qubits[j] >= sector_bits) it.touched = 0.5;
        it.pool = 16;  // 4, or 16 when the control is among the register bits
        it.target = int8_t(1 - j);
        it.need = uint64_t(1) << it.bit[1 - j];
        for (int r = 0; r < 2; ++r)
            for (int c = 0; c < 2; ++c) {
                const int e = 4 * (bit | (r ? tb : 0)) + (bit | (c ? tb : 0));
                it.m[2 * (2 * r + c)] = m[2 * e];
                it.m[2 * (2 * r + c) + 1] = m[2 * e + 1];
            }
        it.flags = u1_class(it.m);
        return;
    }
    it.need = it.all;
    int perm[4];
    const bool mono = is_monomial(2, m, perm);
    if (mono && perm[0] == 0 && perm[1] == 2 && perm[2] == 1 && perm[3] == 3) {
        it.kind = OP_D2;
        it.swap = true;
        it.pool = 4;
        for (int r = 0; r < 4; ++r) {
            it.m[2 * r] = m[2 * (4 * r + perm[r])];
            it.m[2 * r + 1] = m[2 * (4 * r + perm[r]) + 1];
        }
        return;
    }
    it.kind = OP_U2;
    it.pool = 16;
    it.keep = 0xffff;
    if (mono) {
        it.keep = 0;
        for (int r = 0; r < 4; ++r) it.keep |= uint16_t(1u << (4 * r + perm[r]));
    }
}

// The gates of one segment as queues per flat bit: a gate may run when it is
// at the head of the queue of each of its bits.
struct Queues {
    const std::vector<Item> &it;
    int n;
    std::vector<int> next;             // gate ids, bit by bit
    int beg[HQ_MAX_N + 1], len[HQ_MAX_N];
    int head[HQ_MAX_N];

    Queues(const std::vector<Item> &items, int n_, int g0, int g1) : it(items), n(n_)
    {
        std::memset(len, 0, sizeof(len));
        for (int g = g0; g < g1; ++g)
            for (int j = 0; j < it[g].nb; ++j) ++len[it[g].bit[j]];
        beg[0] = 0;
        for (int b = 0; b < n; ++b) beg[b + 1] = beg[b] + len[b];
        next.resize(size_t(beg[n]));
        int at[HQ_MAX_N];
        for (int b = 0; b < n; ++b) at[b] = beg[b], head[b] = 0;
        for (int g = g0; g < g1; ++g)
            for (int j = 0; j < it[g].nb; ++j) next[size_t(at[it[g].bit[j]]++)] = g;
    }
    int front(const int *h, int b) const { return h[b] < len[b] ? next[size_t(beg[b] + h[b])] : -1; }
    bool ready(const int *h, int g) const
    {
        for (int j = 0; j < it[g].nb; ++j)
            if (front(h, it[g].bit[j]) != g) return false;
        return true;
    }
};

struct Budget {
    int ops = 0, pool = 0, aux = 0;
    bool fits(const Item &i) const
    {
        return ops + 1 <= kMaxOps && pool + i.pool <= kMaxPool && aux + i.aux <= kMaxAux;
    }
    void add(const Item &i)
    {
        ++ops;
        pool += i.pool;
        aux += i.aux;
    }
};

// What a gate asks of the tile: the bits it mixes (K = 0: register runs), or all of its bits (dense blocks of K
// qubits).
uint64_t need_of(const Item &i, int K)
{
    if (!K) return i.need;
    return i.nb <= K ? i.all : i.all | kNever;
}

// Runs every gate that can run with the tile bits T, starting from the bits in
// `from`; returns the points gained (3 per gate of two or more needed bits, 1
// otherwise) and appends the gates to out when given.
int absorb(const Queues &q, int *head, uint64_t T, uint64_t from, int K, Budget &bud, std::vector<int> *out)
{
    int points = 0;
    while (from) {
        const int b = __builtin_ctzll(from);
        const int g = q.front(head, b);
        if (g < 0 || (need_of(q.it[g], K) & ~T) || !bud.fits(q.it[g]) || !q.ready(head, g)) {
            from &= from - 1;
            continue;
        }
        const Item &i = q.it[g];
        for (int j = 0; j < i.nb; ++j) ++head[i.bit[j]];
        from |= i.all;
        if (!K) bud.add(i);
        const uint64_t need = need_of(i, K);
        points += (need & (need - 1)) ? 3 : 1;
        if (out) out->push_back(g);
    }
    return points;
}

template <typename R>
void put_entry(PassParam<R> &p, int at, const double *e)
{
    p.pool[at].x = R(e[0]);
    p.pool[at].y = R(e[1]);
}

// What planning a pass writes; as BlockScratch, reserved for a whole segment before its first launch: a list that runs
// out of host memory leaves the state after one of its gates, not amid a pass's reordered ones.
struct PlanScratch {
    std::vector<int> todo, rest, taken, blist;
    BlockScratch block;
    void reserve(size_t gates)
    {
        for (std::vector<int> *v : {&todo, &rest, &taken, &blist}) v->reserve(gates);
        block.reserve(gates);
    }
};

// Groups the pass's gates (sc.todo, in a valid order) into register runs and writes the
// kernel's parameters.  T: the tile's flat bits (L of them, the lowest c
// contiguous).  False when the runs do not fit (the caller then shortens the
// list).
template <typename R, int RP>
bool compile_pass(PassParam<R> &p, int n, int L, uint64_t T, const std::vector<Item> &it, const hq_gate *gates,
                  PlanScratch &sc)
{
    std::vector<int> &list = sc.todo, &rest = sc.rest, &taken = sc.taken;
    constexpr int NB = Traits<R>::NB, NA = 1 << RP;
    p.n = n;
    p.L = L;
    int c = 0;
    while (c < n && ((T >> c) & 1)) ++c;
    p.c = c;
    int pos[HQ_MAX_N];  // flat bit -> tile position
    int m = 0;
    for (int b = 0; b < n; ++b) {
        pos[b] = -1;
        if ((T >> b) & 1) {
            if (m >= c) p.hi[m - c] = uint8_t(b);
            pos[b] = m++;
        }
    }
    p.nruns = p.nops = p.npool = p.naux = 0;
    while (!list.empty()) {
        if (p.nruns == kMaxRuns) return false;
        // first fit in order: a gate joins when its mixed bits fit the run and nothing it
        // depends on was left out
        uint64_t regs = 0, blocked = 0;
        RunDesc &rd = p.run[p.nruns++];
        const int first = p.nops;
        taken.clear();
        rest.clear();
        for (int g : list) {
            const Item &i = it[g];
            const uint64_t want = regs | i.need;
            if ((i.all & blocked) || __builtin_popcountll(want) > RP) {
                blocked |= i.all;
                rest.push_back(g);
            } else {
                regs = want;
                taken.push_back(g);
            }
        }
        list.swap(rest);
        // fill up to RP register positions, highest tile positions first (lanes then keep the low ones)
        uint64_t rpos = 0;
        for (uint64_t x = regs; x; x &= x - 1) rpos |= uint64_t(1) << pos[__builtin_ctzll(x)];
        for (int q = L - 1; q >= 0 && __builtin_popcountll(rpos) < RP; --q) rpos |= uint64_t(1) << q;
        int rank[kMaxTile];  // tile position -> register position
        int nr = 0;
        for (int q = 0; q < L; ++q) {
            rank[q] = -1;
            if ((rpos >> q) & 1) {
                rd.reg[nr] = uint8_t(q);
                rank[q] = nr++;
            }
        }
        for (int q = nr; q < 4; ++q) rd.reg[q] = 0;
        for (int q = 0; q < 4; ++q) rd.out[q] = rd.reg[q];
        // thread bits: the first NB on positions of different residue (no bank conflicts), the rest ascending
        uint64_t left = ((uint64_t(1) << L) - 1) & ~rpos;
        int nt = 0;
        unsigned residues = 0;
        for (int q = 0; q < L && nt < NB; ++q)
            if (((left >> q) & 1) && !((residues >> (q % NB)) & 1)) {
                residues |= 1u << (q % NB);
                rd.thr[nt++] = uint8_t(q);
                left &= ~(uint64_t(1) << q);
            }
        for (; left; left &= left - 1) rd.thr[nt++] = uint8_t(__builtin_ctzll(left));
        for (; nt < 12; ++nt) rd.thr[nt] = 31;
        for (int g : taken) {
            const Item &i = it[g];
            RunOp &o = p.op[p.nops++];
            o.code = CODE_DG;
            o.var = 0;
            o.k = i.nb;
            o.flags = i.flags;
            o.mat = uint16_t(p.npool * int(sizeof(typename Amp<R>::entry)));
            o.lmask = 0;
            o.omask = 0;
            if (i.kind == OP_DG) {
                o.lmask = uint16_t(p.naux);
                uint8_t *x = p.aux + p.naux;
                for (int j = 0; j < NA; ++j) {
                    int off = 0;
                    for (int s = 0; s < i.nb; ++s) {
                        const int tp = pos[i.bit[s]];
                        if (tp >= 0 && rank[tp] >= 0 && ((j >> rank[tp]) & 1)) off |= 1 << (i.nb - 1 - s);
                    }
                    x[j] = uint8_t(off);
                }
                for (int s = 0; s < i.nb; ++s) {
                    const int tp = pos[i.bit[s]];
                    x[NA + s] = tp < 0 ? uint8_t(64 + i.bit[s]) : rank[tp] >= 0 ? uint8_t(255) : uint8_t(tp);
                }
                p.naux += NA + i.nb;
                const int K = 1 << i.nb;
                for (int r = 0; r < K; ++r) put_entry(p, p.npool++, gates[g].matrix + 2 * (r * K + r));
                continue;
            }
            if (i.kind == OP_PH) {
                int mask = 0;
                for (int s = 0; s < i.nb; ++s) {
                    const int tp = pos[i.bit[s]];
                    if (tp < 0) o.omask |= uint64_t(1) << i.bit[s];
                    else if (rank[tp] >= 0) mask |= 1 << rank[tp];
                    else o.lmask |= uint16_t(1 << tp);
                }
                o.var = o.lmask || o.omask;
                o.code = uint8_t(CODE_PH + mask);
                put_entry(p, p.npool++, i.m);
                continue;
            }
            if (i.kind == OP_U1) {
                const int t = i.target;
                const int rt = rank[pos[i.bit[t]]];
                if (i.nb == 2) {
                    const int cb = i.bit[1 - t], cp = pos[cb];
                    if (cp >= 0 && rank[cp] >= 0) {
                        // the control is a register bit too: the 4 x 4 matrix
                        const int rc = rank[cp], lo = std::min(rt, rc), hi = std::max(rt, rc);
                        o.code = uint8_t(CODE_U2 + pair_no(lo, hi));
                        for (int r = 0; r < 4; ++r)
                            for (int s = 0; s < 4; ++s) {
                                const int tr = rt == lo ? r & 1 : r >> 1, cr = rt == lo ? r >> 1 : r & 1;
                                const int ts = rt == lo ? s & 1 : s >> 1, cs = rt == lo ? s >> 1 : s & 1;
                                double e[2] = {0.0, 0.0};
                                if (cr && cs) e[0] = i.m[2 * (2 * tr + ts)], e[1] = i.m[2 * (2 * tr + ts) + 1];
                                else if (r == s) e[0] = 1.0;
                                put_entry(p, p.npool++, e);
                            }
                        continue;
                    }
                    o.var = 1;
                    if (cp < 0) o.omask = uint64_t(1) << cb;
                    else o.lmask = uint16_t(1 << cp);
                }
                // (complex128 bodies test every part themselves)
                o.code = uint8_t(CODE_U1 + 4 * rt + (sizeof(R) == 4 ? i.flags : U1_FULL));
                for (int e = 0; e < 4; ++e) put_entry(p, p.npool++, i.m + 2 * e);
                continue;
            }
            if (i.swap) {
                // each of the two qubits is in the other's register bit from here on
                int &a = rank[pos[i.bit[0]]], &b = rank[pos[i.bit[1]]];
                std::swap(rd.out[a], rd.out[b]);
                std::swap(a, b);
            }
            // two mixed bits: kernel index r = 2 [upper register bit] + [lower one]; the gate's own index has
            // bit[0] on top
            const int r0 = rank[pos[i.bit[0]]], r1 = rank[pos[i.bit[1]]];
            const bool flip = r0 < r1;  // bit[0] is the lower register bit
            o.code = uint8_t((i.kind == OP_D2 ? CODE_D2 : CODE_U2) + pair_no(std::min(r0, r1), std::max(r0, r1)));
            auto own = [&](int r) { return flip ? ((r & 1) << 1) | (r >> 1) : r; };
            if (i.kind == OP_D2) {
                o.lmask = 0;
                for (int r = 0; r < 4; ++r) {
                    put_entry(p, p.npool++, i.m + 2 * own(r));
                    o.lmask |= uint16_t(phase_kind(i.m + 2 * own(r)) << (4 * r));
                }
            } else {
                const double zero[2] = {0.0, 0.0};
                for (int r = 0; r < 4; ++r)
                    for (int s = 0; s < 4; ++s) {
                        const int e = 4 * own(r) + own(s);
                        put_entry(p, p.npool++, (i.keep >> e) & 1 ? gates[g].matrix + 2 * e : zero);
                    }
            }
        }
        rd.op0 = uint16_t(first);
        rd.op1 = uint16_t(p.nops);
    }
    return true;
}

// Time of a gate in register runs and of a dense block in a block pass, ms at n = 28 (from whole circuits of 785 gates:
// in runs 66.5 with CZ and 87 with fSim, in 139 three-qubit blocks 54.7, in 77 four-qubit blocks 59; QFT in runs); a
// pass cannot take less than its read and write of the state.
double run_cost(const Item &i)
{
    switch (i.kind) {
    case OP_PH: return 0.05;
    case OP_D2: return 0.13;
    case OP_U2: return 0.22;
    case OP_BLK: return i.nb == 3 ? 0.39 : 0.77;
    default: return 0.10;
    }
}
double block_cost(int K) { return K == 3 ? 0.39 : 0.77; }

// complex64: the time of a gate on its own kernel, us.  Measured, n = 28 / 24 / 22 / 20: X 670 / 47 / 12 / 6.2, a
// permutation of four qubits 703 / 49 / 13 / 6.3, a dense four-qubit gate 860 / 59 / 16 / 8; controlled gates by what k_ctrl
// touches: CNOT 376 / 21 / 7 / 4.3, a controlled SWAP 375 / 22 / 8.6 / 4.6, Toffoli 180-224 / 11-14 / 6.2 / 4.2, one with
// three controls 145 / 9 / 7.5 / 7.4 (the last ones by the host).
double own_time(const Item &i, double us_per_ms)
{
    const double full = i.kind == OP_BLK && i.nb == 4 && !i.perm ? 0.86 : 0.69;
    const double ms = i.touched < 1.0 ? 0.04 + 0.63 * i.touched : full;  // n = 28
    return std::max(4.2, 3.0 + us_per_ms * ms);
}

// complex128: the same for a gate in register runs and on its own kernel (ms at n = 28; FP64 multiply-adds at two per
// clock and SM, 0.46 ms for one per amplitude; a read and write of the state 1.26 ms).  Measured at n = 22: a CNOT 43 us on
// k_ctrl and 100 in runs (its 4 x 4 form tests every part), a dense two-qubit gate 154 and 157.
double own_cost_128(const Item &i)
{
    switch (i.kind) {
    case OP_PH: return i.nb == 1 ? 1.85 : 0.5;
    case OP_U1: return i.nb == 2 ? 2.75 : 3.9;
    case OP_U2: return 9.8;
    default: return i.kind == OP_DG ? 0.1 + 1.8 * i.touched : 1.9;
    }
}
double run_cost_128(const Item &i)
{
    auto parts = [&](int n) {  // nonzero parts of the first n entries
        int c = 0;
        for (int e = 0; e < 2 * n; ++e) c += i.m[e] != 0.0;
        return c;
    };
    switch (i.kind) {
    case OP_PH: return i.flags ? 0.1 : 0.5;
    case OP_U1: return i.nb == 2 ? 6.4 : 0.5 * parts(4);
    case OP_U2: return 10.0;
    case OP_D2: return 0.25 * parts(4);
    default: return 2.0;
    }
}
constexpr double kPassFloor = 0.75;
constexpr double kPassLaunch = 7.0;  // us of a pass beside that (three gates of one qubit, n = 20: 9.8 us)
// Below this size lists without 3- or 4-qubit gates stay on register runs (depth-12 CZ circuits, runs / blocks: n=25
// 4.88 / 3.99 ms, n=23 1.28 / 1.20 ms; below, the plan of the blocks and their products cost the host more than that).
constexpr int kBlockMinQubits = 23;

// Tile bits and the length of its contiguous runs.  A larger tile takes more gates per pass; a smaller one gives
// the SMs more tiles of a small state (and complex128, bound by the two FP64 lanes of an SM, wants all SMs).
// Measured, us per random grid circuit (tile / run bits):
//   complex64   n=12  12/5 56   11/4 54   9/4 60      n=18  13/5 231  12/4 138  11/4 120  10/4 133
//               n=20  13/5 309  12/4 246  11/4 306    n=22  13/5 771  12/4 672  11/4 885
//               n=24  13/5 2730 13/6 2853 12/4 2849   n=26  13/5 10047  12/4 10282  11/4 13533
//   complex128  n=12  10/4 350  9/3 209  8/3 197  7/3 216    n=16  10/4 577  9/3 354  8/3 349  (4 amplitudes per thread)
//               n=18  12/4 1755  11/4 922  10/4 928  9/3 1193
//               n=20  11/4 2723  10/4 2449  9/3 2670         n=23  12/4 21449  11/4 20833  10/4 21338
template <typename R> void tile_shape(int n, int &L, int &cmin)
{
    if (sizeof(R) == 4) L = n >= 23 ? 13 : n >= 19 ? 12 : 11;
    else L = n >= 21 ? 11 : n >= 17 ? 10 : 8;
    cmin = L == 13 ? 5 : L == 8 ? 3 : 4;
    L = std::min(L, n);
    cmin = std::min(cmin, L);
}

// Up to this size complex128 passes take 4 amplitudes per thread instead of 8: an FP64 instruction takes a quarter of an
// SM 64 cycles whatever its lanes do, so a small state wants its gates on as many warps as it can fill (4 / 8: n=12 197
// / 238 us, n=16 349 / 404; n=18 1427 / 927).
constexpr int kFewQubits128 = 16;

// The gates [g0, g1) of the list, none of them wide, pass by pass.
enum PassKind { PASS_RUNS, PASS_BLOCKS, PASS_SINGLE };
template <typename R, int RP> struct Segment {
    const std::vector<Item> &it;
    const hq_gate *gates;
    Queues q;
    int n, L, cmin, left;
    int K = 0;              // width of dense blocks, 0: none
    std::vector<int> list;  // the gates of the current pass, in a valid order
    PlanScratch sc;
    uint64_t T = 0;         // its tile (PASS_RUNS, PASS_BLOCKS)

    Segment(const std::vector<Item> &items, const hq_gate *gs, int n_, int g0, int g1)
        : it(items), gates(gs), q(items, n_, g0, g1), n(n_), left(g1 - g0)
    {
        list.reserve(size_t(left));
        sc.reserve(size_t(left));
        tile_shape<R>(n, L, cmin);
        if (sizeof(R) == 4 && L >= kBlockTileMin) {
            if (n >= kBlockMinQubits) K = 3;
            for (int g = g0; g < g1; ++g)
                if (it[size_t(g)].kind == OP_BLK) K = std::max<int>(K, it[size_t(g)].nb);
        }
    }

    // The tile's bits and the gates of a pass: the contiguous low bits, then, as long as there is room, the ones that
    // let the most gates in per added bit.  kind: 0 for register runs, else the width of dense blocks.
    void grow(int kind, int *head, std::vector<int> &out, uint64_t &tile)
    {
        const uint64_t every = (uint64_t(1) << n) - 1;
        out.clear();
        Budget bud;
        tile = n == L ? every : (uint64_t(1) << cmin) - 1;
        absorb(q, head, tile, every, kind, bud, &out);
        while (__builtin_popcountll(tile) < L) {
            const int room = L - __builtin_popcountll(tile);
            uint64_t best = 0;
            double top = 0;
            for (int b = 0; b < n; ++b) {
                const int g = q.front(head, b);
                if (g < 0) continue;
                const uint64_t add = need_of(it[size_t(g)], kind) & ~tile;
                if (!add || (add & kNever) || __builtin_ctzll(add) != b || __builtin_popcountll(add) > room ||
                    !q.ready(head, g))
                    continue;
                int h[HQ_MAX_N];
                std::memcpy(h, head, sizeof(int) * size_t(n));
                Budget b2 = bud;
                const double gain =
                    double(absorb(q, h, tile | add, add, kind, b2, nullptr)) / __builtin_popcountll(add);
                if (gain > top) top = gain, best = add;
            }
            if (!best) break;
            tile |= best;
            absorb(q, head, tile, best, kind, bud, &out);
        }
        for (int b = 0; b < n && __builtin_popcountll(tile) < L; ++b) tile |= uint64_t(1) << b;
    }

    bool two_with_a_dense_one() const
    {
        return list.size() == 2 && (it[size_t(list[0])].kind == OP_U2 || it[size_t(list[1])].kind == OP_U2);
    }

    // Whether the gates of the pass in `list` are done sooner one launch each (estimated times).
    bool own_kernels_faster(PassKind kind)
    {
        if (list.size() == 1) return true;
        if constexpr (sizeof(R) == 4) {
            // launches long enough to count: a list of Toffoli gates, n = 28, takes 0.41 ms each in blocks, 0.18 to 0.22 on
            // k_ctrl.  A pass with little work in it does not hide all of that under its copies (n = 28: three CZ
            // 0.87, three one-qubit gates 1.01, two Toffoli gates 1.03 ms).
            if (n < 20) return false;
            const double ms = std::ldexp(1e3, n - 28);  // us here of a ms at n = 28
            double own = 0, cost = 0, launches = 1;
            for (int g : list) {
                const Item &i = it[size_t(g)];
                own += own_time(i, ms);
                // (a diagonal gate by its table: 0.185 of three qubits, 0.3 of six)
                if (kind == PASS_RUNS) cost += i.kind == OP_DG ? 0.1 + 0.03 * i.nb : run_cost(i);
            }
            if (kind == PASS_BLOCKS) {
                const int count = count_in_tile(n, K, gates, list, sc.block), per = K == 3 ? kBlocks3 : kBlocks4;
                launches = (count + per - 1) / per;
                cost = block_cost(K) * count;
            }
            return own <= kPassLaunch * launches + ms * std::max(cost, kPassFloor * launches + std::min(cost, 0.4));
        } else if (n <= 9) {
            // one CTA: a gate takes its FP64 latency (16 permutations of two qubits, n = 6 / 9: 83 / 80 us in runs, 66 in
            // launches; two CNOT, n = 8: 10.6 and 8.2)
            double own = 0, run = 4.0;
            for (int g : list) {
                const Item &i = it[size_t(g)];
                own += i.kind == OP_U2 && i.keep == 0xffff ? 6.2 : 4.1;
                run += i.kind == OP_U2 ? 4.9 : i.kind == OP_U1 && i.nb == 2 ? 3.3 : 1.0;
            }
            return own <= run || two_with_a_dense_one();
        } else if (n < 17) {
            return two_with_a_dense_one();
        } else {
            // where the FP64 work of the gates is what counts, a pass saves nothing (n >= 22: a pass of three CZ 2.4 at n =
            // 24 and 2.6 at n = 26, the three on k_ctrl 2.0 and 1.7)
            double own = 0, run = 0, light = 0;
            for (int g : list) {
                const Item &i = it[size_t(g)];
                own += own_cost_128(i), run += run_cost_128(i);
                light += i.kind == OP_PH && i.nb == 2 ? 0.3 : i.kind == OP_U1 && i.nb == 2 ? 0.55 : 1.0;
            }
            return (n >= 20 && light <= 1.0) || std::max(n >= 22 ? 2.4 : 1.3, run) >= 0.95 * own;
        }
    }

    // The next pass: register runs (into p), dense blocks (list and T), or single gates cheaper on their own kernels.
    PassKind next(PassParam<R> &p)
    {
        int saved[HQ_MAX_N];
        std::memcpy(saved, q.head, sizeof(int) * size_t(n));
        grow(0, q.head, list, T);
        PassKind kind = PASS_RUNS;
        if (K) {
            // the kind that does more work per time (work: what the gates cost in register runs)
            int head[HQ_MAX_N];
            std::memcpy(head, saved, sizeof(int) * size_t(n));
            std::vector<int> &blist = sc.blist;
            uint64_t btile = 0;
            grow(K, head, blist, btile);
            double runs = 0, work = 0;
            for (int g : list) runs += run_cost(it[size_t(g)]);
            for (int g : blist) work += run_cost(it[size_t(g)]);
            const double rate = list.empty() ? 0.0 : runs / std::max(kPassFloor, runs);
            if (!blist.empty() &&
                work / std::max(kPassFloor, block_cost(K) * count_in_tile(n, K, gates, blist, sc.block)) > rate) {
                kind = PASS_BLOCKS;
                list.swap(blist);
                T = btile;
                std::memcpy(q.head, head, sizeof(int) * size_t(n));
            }
        }
        if (own_kernels_faster(kind)) kind = PASS_SINGLE;
        auto compiled = [&]() {
            sc.todo = list;
            return compile_pass<R, RP>(p, n, L, T, it, gates, sc);
        };
        while (kind == PASS_RUNS && !compiled()) {
            // too many runs: a shorter pass (the first half of the list is a valid order of its own)
            list.resize(list.size() / 2);
            std::memcpy(q.head, saved, sizeof(int) * size_t(n));
            for (int g : list)
                for (int j = 0; j < it[size_t(g)].nb; ++j) ++q.head[it[size_t(g)].bit[j]];
        }
        left -= int(list.size());
        return kind;
    }
};

template <typename R, int RP>
hq_status run_segment(void *state, int n, const std::vector<Item> &it, const hq_gate *gates, int g0, int g1,
                      int engine, cudaStream_t s)
{
    using T2 = typename C2<R>::type;
    const hq_dtype dt = sizeof(R) == 4 ? HQ_C64 : HQ_C128;
    Segment<R, RP> seg(it, gates, n, g0, g1);
    PassParam<R> p;
    while (seg.left > 0) {
        hq_status st = HQ_OK;
        switch (seg.next(p)) {
        case PASS_SINGLE:
            for (int g : seg.list)
                if ((st = launch_gate(state, n, dt, gates[g].k, gates[g].qubits, gates[g].matrix, 1, engine, s)) != HQ_OK)
                    return st;
            break;
        case PASS_BLOCKS:
            st = launch_block_pass(state, n, seg.L, seg.T, seg.K, gates, seg.list, seg.sc.block, s);
            break;
        default: {
            const size_t smem = pass_smem<R>(p.L);
            const int threads = std::max(32, std::min(kRunThreads, 1 << (p.L - RP)));
            const void *fn = (const void *)k_runs<R, RP>;
            const int grid = grid_for(fn, kRunThreads, smem, int64_t(1) << (n - p.L));
            k_runs<R, RP><<<grid, threads, smem, s>>>(p, (T2 *)state);
            st = cuda_status("k_runs", cudaGetLastError());
        }
        }
        if (st != HQ_OK) return st;
    }
    return HQ_OK;
}

// Gates planned at a time: bounds the plan's memory; a list of any length runs.
constexpr int kMaxSegment = 4096;

template <typename R>
hq_status run_list(void *state, int n, const hq_gate *gates, int G, int engine, cudaStream_t s)
{
    const hq_dtype dt = sizeof(R) == 4 ? HQ_C64 : HQ_C128;
    std::vector<Item> it;
    for (int first = 0; first < G; first += kMaxSegment) {
        const int cnt = std::min(kMaxSegment, G - first);
        const hq_gate *const gs = gates + first;
        it.resize(size_t(cnt));
        int L = 0, c = 0;
        tile_shape<R>(n, L, c);
        // (4-qubit blocks: below 20 qubits their own kernel is faster, n=18 115 against 123 us for 19 blocks)
        const int max_block = sizeof(R) == 4 && L >= kBlockTileMin ? (n >= 20 ? 4 : 3) : 2;
        for (int g = 0; g < cnt; ++g) classify(n, gs[g], max_block, sizeof(R) == 4 ? 2 : 1, it[size_t(g)]);
        for (int g = 0; g < cnt;) {
            int e = g;
            while (e < cnt && !it[size_t(e)].wide) ++e;
            hq_status st = HQ_OK;
            if (e - g > 1) {
                constexpr int RP = Traits<R>::RP, FEW = sizeof(R) == 8 ? 2 : RP;
                st = n <= kFewQubits128 ? run_segment<R, FEW>(state, n, it, gs, g, e, engine, s)
                                        : run_segment<R, RP>(state, n, it, gs, g, e, engine, s);
            } else {
                e = g + 1;
                st = launch_gate(state, n, dt, gs[g].k, gs[g].qubits, gs[g].matrix, 1, engine, s);
            }
            if (st != HQ_OK) return st;
            g = e;
        }
    }
    return HQ_OK;
}

}  // namespace

hq_status launch_gate_list(void *state, int n, hq_dtype dt, const hq_gate *gates, int G, int engine, cudaStream_t s)
{
    const int least = dt == HQ_C64 ? Traits<float>::RP : Traits<double>::RP;
    if (G >= 2 && n >= least) {
        try {
            if (dt == HQ_C64) return run_list<float>(state, n, gates, G, engine, s);
            return run_list<double>(state, n, gates, G, engine, s);
        } catch (const std::bad_alloc &) {
            set_last_error_text("gate passes: out of host memory");
            return HQ_ERR_ALLOC;
        }
    }
    for (int g = 0; g < G; ++g) {
        hq_status st = launch_gate(state, n, dt, gates[g].k, gates[g].qubits, gates[g].matrix, 1, engine, s);
        if (st != HQ_OK) return st;
    }
    return HQ_OK;
}

}  // namespace hq
