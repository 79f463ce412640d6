// kg_stages.h -- the order in which one warp feeds a ring of S shared-memory
// stages with nt tiles by bulk asynchronous copies.  Plain C++ beside the
// kernels, so that the order can be tested without a GPU.
#pragma once

#ifdef __CUDACC__
#define KG_STAGE_FN __device__ __forceinline__
#else
#define KG_STAGE_FN inline
#endif

namespace kg {

// Tiles [0, min(S, nt)) are in flight already.  landed(t): tile t's copy has
// arrived; freed(t): its readers are done with the stage; both wait for a
// bounded time and return false when that runs out.  issue(t) starts the copy
// of tile t into its stage, t % S.
//
// A tile is issued only into a stage whose copy has landed and whose readers
// are done, so a stage never has two copies in flight.  Nothing is issued
// after a wait that ran out, and whatever was issued is waited for before the
// return: a block that ended earlier would leave copies writing into shared
// memory that belongs to the next block.  False when any wait ran out.
template <class Landed, class Freed, class Issue>
KG_STAGE_FN bool feed_stages(int nt, int S, Landed landed, Freed freed, Issue issue) {
    bool ok = true;
    int t = nt < S ? nt : S;
    while (ok && t < nt) {
        ok = landed(t - S) && freed(t - S);
        if (ok) issue(t++);
    }
    for (int u = t > S ? t - S : 0; u < t; ++u) ok = landed(u) && ok;
    return ok;
}

}  // namespace kg
