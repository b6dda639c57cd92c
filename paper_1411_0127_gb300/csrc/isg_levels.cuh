// isg_levels.cuh -- the levels of whole colour passes, made ahead of their use by
// the resident blocks of isg_resident.cu, for ensembles with few RNG streams
// (isg_amsc.cu).
#pragma once

#include "isg_common.cuh"

namespace isg {

// Pass p's levels of part k (rows k rpb ..) of stream t are 2 cw words from
// lv + p pass_words + (t parts + k) 2 cw on: the lo and the hi bit stream, cw
// words each, or level bytes (take_levels).  Their first draw is bit (draw) 0;
// of MT19937, whose blocks run on over the passes, bit p D mod 32 (draw p D mod
// 16 of level bytes), D being the stream's draws of a pass.
struct LevelsPlan {
    int kind = 0, parts = 0, rpb = 0, nblocks = 0, cw = 0;
    bool bytes = false;
    size_t smem = 0, pass_words = 0;
    size_t state_bytes = 0;   // of the copy of the states that launch() needs, or 0
    void* jumps = nullptr;

    // g: size, partition and kind of the lattice; false where it does not fit.
    bool make(const isg_sim& g);
    // npass passes from the states gen.rng / gen.rng_pos on, which are left
    // after them.  gen: L, half, R, S, rows, cmp, rng, rng_pos, mt.
    cudaError_t launch(const FlipArgs& gen, uint32_t* rng_copy, uint32_t* lv, int npass, cudaStream_t s) const;
    void clear();
};

}  // namespace isg
