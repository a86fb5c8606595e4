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

// The listed gates (a valid order, every qubit in the tile T, none wider than
// K = 3 or 4) fused into blocks of exactly K qubits.
void fuse_in_tile(int n, int K, uint64_t T, const hq_gate *gates, const std::vector<int> &list,
                  std::vector<TileBlock> &blocks);
// The number of blocks that makes.
int count_in_tile(int n, int K, const hq_gate *gates, const std::vector<int> &list);
// The blocks in order on a complex64 state, tiles of the L bits T.
hq_status launch_block_pass(void *state, int n, int L, uint64_t T, int K, std::vector<TileBlock> &blocks,
                            cudaStream_t s);

}  // namespace hq
