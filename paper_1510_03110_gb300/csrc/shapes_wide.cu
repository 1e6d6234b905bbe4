// shapes_wide.cu -- the reductions of the shapes 12,6 20,10 20,20 24,12 with a team of four warps
// per subproblem, for levels with few chunks: a level of a few hundred chunks leaves most warps
// of the chip idle when each chunk is one warp's, and its time is the serial chain of one chunk.
#define MHE_TEAM 128
#include "kernels.cuh"

namespace mhe {

int shapes_wide(WideEntry* out, int cap)
{
    int k = 0;
    if (k < cap) out[k++] = make_wide<12, 6>();
    if (k < cap) out[k++] = make_wide<20, 10>();
    if (k < cap) out[k++] = make_wide<20, 20>();
    if (k < cap) out[k++] = make_wide<24, 12>();
    return k;
}

}  // namespace mhe
