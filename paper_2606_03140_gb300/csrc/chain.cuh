// Chains of symmetric products over all subgraphs in one launch (see chain.cu).
#pragma once
#include "dense.cuh"

namespace sedacs {

constexpr int kMaxChain = 96;      // products per launch (longer chains are split)

// One product  out = alpha A B + beta I + g1 C1 + g2 C2  of symmetric matrices kept as upper
// 128x128 tiles, over every subgraph.  Offsets are bytes from the arena base to the slot's plane 0
// (a, b, out, out2) or master (outm, c1, c2); -1: absent.  With out2 the first output is alpha A B
// alone and the second alpha2 A B + beta I + g1 C1 + g2 C2.
struct ChainOp {
  long long a, b, out, out2, outm, c1, c2;
  float alpha, beta, g1, g2, alpha2;
  int pad;
};

// One upper 128x128 tile of a subgraph's matrix.
struct alignas(16) ChainTile {
  long long el;        // element offset of the subgraph in every square slot
  int mat, tm, tn;
  int n_pad, n_real;
  int pad;
};

struct ChainParams {
  ChainOp op[kMaxChain];
  uint8_t* arena;
  const ChainTile* tiles;    // upper tiles of every subgraph, grouped by subgraph
  const int* win;            // window w holds the tiles [win[w], win[w + 1])
  unsigned* done;            // per subgraph: epilogue warps finished (cleared before the launch)
  int* err;
  long long plane;           // bytes between the planes of a square slot
  int n_ops, n_win;
};

// planes: 2 = the two-plane fp16 format, 3 = three bf16 planes.  n_work tiles; p.done is cleared here
// (n_sub words) when the chain holds more than one product.
cudaError_t launch_chain(const ChainParams& p, int planes, int n_work, int n_sub, cudaStream_t s);

// About how many tiles a window of subgraphs holds on this device (see chain.cu).
cudaError_t chain_window_tiles(int* tiles);

}  // namespace sedacs
