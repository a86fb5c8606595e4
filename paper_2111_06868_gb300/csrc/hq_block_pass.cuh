// hq_block_pass.cuh -- passes of dense 3- and 4-qubit blocks over a tile
// (k_block_pass.cu), planned by k_runs.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/hq.h"

namespace hq {

constexpr int kBlockTileMin = 9, kBlockTileMax = 13;  // tile bits a block pass takes
constexpr int kBlocks3 = 8, kBlocks4 = 4;  // blocks of 3 and of 4 qubits per launch
struct TileBlock {
    int k;
    int bit[4];        // flat bits, ascending; bit j of the matrix's index is bit[j]
    double m[2 * 256]; // 2^k x 2^k complex, row-major
};

// What planning and fusing a pass writes: reserved for every gate of a list's segment before its first launch, so that
// no pass allocates.
struct BlockScratch {
    std::vector<uint64_t> set;
    std::vector<int> member;
    void reserve(size_t gates)
    {
        set.reserve(gates);
        member.reserve(gates);
    }
};

// The number of blocks of at most K = 3 or 4 qubits that the listed gates (a valid order, none wider than K) make.
int count_in_tile(int n, int K, const hq_gate *gates, const std::vector<int> &list, BlockScratch &sc);
// The listed gates, every qubit in the tile T of L bits, fused into blocks of K qubits and applied in order to a
// complex64 state.
hq_status launch_block_pass(void *state, int n, int L, uint64_t T, int K, const hq_gate *gates,
                            const std::vector<int> &list, BlockScratch &sc, cudaStream_t s);

}  // namespace hq
