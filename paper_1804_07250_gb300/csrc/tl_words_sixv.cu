// Builds of the word kernel for six-vertex configurations.
#include "tl_words_kernel.cuh"

namespace tl {

const void* words_kernel_sixv(bool count, int threads, int slots, bool fixed)
{
    return count ? words_build<LAT_SIXV, THR_TABLE, true>(threads, slots, fixed)
                 : words_build<LAT_SIXV, THR_TABLE, false>(threads, slots, fixed);
}

// This file's debug word (failures, then the id, index and bound of the
// first failed check); cudaErrorNotSupported in the normal build.
int dbg_fetch_words_sixv(unsigned long long* out, bool clear)
{
#ifdef TL_DEBUG
    return tl_dbg_fetch(out, clear);
#else
    (void)out;
    (void)clear;
    return (int)cudaErrorNotSupported;
#endif
}

}  // namespace tl
