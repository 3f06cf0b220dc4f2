/*
 * lbm_arrays.h -- lbm_init_fields for callers whose five fields are separate host arrays.
 */
#ifndef LBM_ARRAYS_H_
#define LBM_ARRAYS_H_

#include "lbm.h"

#ifdef __cplusplus
extern "C" {
#endif

/* lbm_init_fields from rho, u_x, u_y, u_z, p as five host arrays [z][y][x] of `dtype`
 * (LBM_DT_F32 or LBM_DT_F64), each copied to the device as it is (no array of all five
 * on the host). Same result and errors; LBM_E_INVAL for a NULL array. */
lbm_status lbm_init_fields_arrays(lbm_handle* h, const void* const fields[5], int dtype);

#ifdef __cplusplus
}
#endif
#endif /* LBM_ARRAYS_H_ */
