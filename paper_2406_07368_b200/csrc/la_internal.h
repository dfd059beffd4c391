/* Entry points shared by the library and its Python binding only; not part of include/la.h. */
#ifndef LA_B200_INTERNAL_H_
#define LA_B200_INTERNAL_H_

#include "la.h"

#ifdef __cplusplus
extern "C" {
#endif

/* la_commit for output buffers whose contents nobody has seen yet: where the flag of a buffer is set, a sequence that
 * the kernel skips (malformed tree) gets -1 in its whole path row / 0 as its length instead of being left alone. */
enum { LA_FRESH_PATH = 1, LA_FRESH_LEN = 2 };
la_status la_commit_fresh(la_ctx* ctx, int32_t B, int32_t N, const void* k, const void* v, const int32_t* parent,
                          const int32_t* accept_node, la_state* st /*host struct*/, int32_t* path_out,
                          int32_t* commit_len, int fresh, void* stream);

#ifdef __cplusplus
}
#endif
#endif /* LA_B200_INTERNAL_H_ */
