/*
 * lbm_forms.h -- the form in which lbm_step runs the steps of a domain (no counterpart in
 * the paper).
 */
#ifndef LBM_FORMS_H_
#define LBM_FORMS_H_

#include "lbm.h"

#ifdef __cplusplus
extern "C" {
#endif

/* L2 prefetch distance in tiles that the plain step kernel of this handle runs with: the one
 * that lbm_set_prefetch or lbm_autotune fixed, or the one that follows the state's size
 * (lbm_info_t.prefetch_tiles is the storage type's default then). LBM_E_INVAL for a NULL
 * argument. */
lbm_status lbm_prefetch_in_effect(const lbm_handle* h, int* tiles);

/* Steps that the handle has taken in the form which runs many steps of a small domain in one
 * launch (lbm_step), since lbm_create. LBM_E_INVAL for a NULL argument. */
lbm_status lbm_resident_steps(const lbm_handle* h, long long* steps);

/* Failure-detection test hook. In the next launch that takes many steps of a small domain
 * (lbm_step), block `block` does nothing, and a wait of the others gives up after `polls`
 * tries (about half a microsecond each, rounded up to 1024) instead of about a second. Its neighbours' waits
 * run out; nothing faults or hangs. The next synchronising call then returns
 * LBM_E_TIMEOUT, after which lbm_step refuses to run until a re-init. LBM_E_INVAL if the
 * domain takes one launch per step, for a block it does not have or polls < 1. */
lbm_status lbm_test_stall_resident(lbm_handle* h, int block, int polls);

#ifdef __cplusplus
}
#endif
#endif /* LBM_FORMS_H_ */
