// Builds of the word kernel for dominoes.
#include "tl_words_kernel.cuh"

namespace tl {

const void* words_kernel_domino(int tk, int threads, int slots, bool fixed)
{
    return tk == THR_SITE ? words_build<LAT_DOMINO, THR_SITE, false>(threads, slots, fixed)
                          : words_build<LAT_DOMINO, THR_SCALAR, false>(threads, slots, fixed);
}

// This file's debug word (failures, then the id, index and bound of the
// first failed check); cudaErrorNotSupported in the normal build.
int dbg_fetch_words_domino(unsigned long long* out, bool clear)
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
