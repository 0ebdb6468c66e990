// Query rows of one attention CTA: the whole sequence's (one block), or a block of 64
// prompt rows, whose context also holds the local rows before it.
#pragma once

#include "kernels.h"

namespace chimera {

struct QueryBlock {
  int b, row0;         // sequence, first row of q / out
  int nctx, nq, nloc;  // context rows, query rows and local rows of this block
  __device__ QueryBlock(const AttnParams& p, int z) {
    if (p.q_blocks <= 1) {
      b = z;
      row0 = b * p.q_rows;
      nctx = p.n_ctx[b];
      nq = p.nq_dev ? p.nq_dev[b] : p.nq;
      nloc = p.n_local_dev ? p.n_local_dev[b] : p.n_local;
      return;
    }
    // the last blocks see the most keys: they start first
    b = z / p.q_blocks;
    const int j0 = (p.q_blocks - 1 - z % p.q_blocks) * 64;
    row0 = b * p.q_rows + j0;
    nctx = p.n_ctx[b] + j0;
    nq = max(0, min(64, p.nq_dev[b] - j0));
    nloc = max(0, min(64, p.n_local_dev[b] - j0));
  }
};

}  // namespace chimera
