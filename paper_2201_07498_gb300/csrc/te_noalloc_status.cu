// te_noalloc_status.cu - the status words of te_spmv_noalloc's calls.
//
// In managed memory of their own, so that the call allocates nothing, not even
// page-locked host memory: host and kernels use the same address, and a word
// that no kernel writes is never moved.  In a translation unit of their own: a
// module with managed variables is loaded with the context, and the 4 MiB scratch
// array beside the kernels is not to be.
#include "te_internal.h"

namespace te {

static __device__ __managed__ int g_noalloc_status[NA_DEVICES * NA_SLOTS * 2];

int* noalloc_status_words() { return g_noalloc_status; }

}  // namespace te
