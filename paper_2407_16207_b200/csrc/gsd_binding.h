/* What libgsd exports for its Python binding only: calls of gsd.h in the form the binding hands on.  Not part of
 * the ABI. */
#ifndef GSD_BINDING_H_
#define GSD_BINDING_H_

#include "gsd.h"

#ifdef __cplusplus
extern "C" {
#endif

/* gsd_draft_expand with the entries of new_frontier behind the first new_frontier_len[b] set to -1 (a tensor
 * filled with -1 beforehand costs the caller 5 us and the device a launch). */
int gsd_binding_draft_expand(const float* logits, const int32_t* frontier, const int32_t* frontier_len,
                             int32_t* tokens, int32_t* tree_parent, int32_t* merge_to, uint8_t* leaf,
                             float* prob, int32_t* num_nodes, int32_t* new_frontier,
                             int32_t* new_frontier_len, const gsd_draft_params* p, void* workspace,
                             size_t workspace_bytes, int32_t* status, void* stream);

#ifdef __cplusplus
}
#endif
#endif
