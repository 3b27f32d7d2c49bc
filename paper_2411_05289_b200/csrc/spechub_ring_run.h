// The order of events of a ring of stages that one consumer fills and empties: plain control flow, without a GPU in it.
#pragma once

#ifdef __CUDACC__
#define SPECHUB_RING_FN __device__ __forceinline__
#else
#define SPECHUB_RING_FN inline
#endif

namespace spechub {

// `chunks` chunks through STAGES stages, the first STAGES of them already requested.  wait(c): has chunk c arrived (a
// bounded wait)?  take(c): out of its stage; then the stage's next chunk is requested, request(c); use(c).  A chunk that
// does not arrive ends the run: it is not taken, none behind it is, nothing more is requested, and what is still on its
// way is waited for once more (no copy may land in the stages when they are somebody else's).  Whether all arrived.
template <int STAGES, class WAIT, class TAKE, class REQUEST, class USE>
SPECHUB_RING_FN bool ring_run(int chunks, WAIT wait, TAKE take, REQUEST request, USE use) {
#ifdef __CUDACC__
#pragma unroll 1
#endif
    for (int c = 0; c < chunks; ++c) {
        if (!wait(c)) {
            for (int d = c; d < c + STAGES && d < chunks; ++d) wait(d);
            return false;
        }
        take(c);
        if (c + STAGES < chunks) request(c + STAGES);
        use(c);
    }
    return true;
}

}  // namespace spechub
