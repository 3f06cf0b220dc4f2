/*
 * lbm_spectral.h -- device passes around the FFTs of the spectral diagnostics (Sec. 3.2:
 * Eq. 7 with curl and divergence taken spectrally, and the shell-averaged energy
 * spectrum). paper_2608_13437_gb300/spectral.py calls them between its transforms.
 *
 * All pointers are device memory of the current CUDA device, FP64, contiguous. A "half
 * spectrum" of a real (nz, ny, nx) field is the (nz, ny, nx/2 + 1) complex array of an
 * unnormalised real-to-complex transform. Work is queued on cuda_stream (a cudaStream_t,
 * NULL for the default stream); no call waits for it. LBM_E_INVAL for a NULL pointer or a
 * size outside 1 ... 2^31 - 1 points; LBM_E_CUDA if a launch fails.
 */
#ifndef LBM_SPECTRAL_H_
#define LBM_SPECTRAL_H_

#include "lbm.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Spectra wh[2] of (curl u)_x + i (curl u)_y and (curl u)_z + i div u over the whole
 * (nz, ny, nx) grid, divided by the number of points, from the unnormalised spectrum zh of
 * u_x + i u_y over the whole grid and the half spectrum ch of u_z (a complex transform
 * carries two real fields). k0 = 2 pi / box side; the Nyquist wavenumber of an even axis
 * counts as 0 (no derivative of that mode of a real field). */
lbm_status lbm_spectral_curl_div(const void* zh, const void* ch, void* wh, int nx, int ny, int nz,
                                 double k0, void* cuda_stream);

/* out[0] = mean of m |w|^2, out[1] = mean of m d^2 over n points, from the complex fields
 * w[2][n] = (w_x + i w_y, w_z + i d) in physical space and the temperature T[n]; m = mu,
 * or Sutherland's law with t = T/T_ref if sutherland. out must hold LBM_SPECTRAL_DOUBLES
 * doubles (scratch). */
#define LBM_SPECTRAL_DOUBLES (2 + 2 * 1216)
lbm_status lbm_spectral_dissipation(const void* w, const double* T, long long n, double mu,
                                    double T_ref, int sutherland, double* out, void* cuda_stream);

/* Adds |u_b / N|^2 / 2 of all N modes of the three components (zh, ch as above) to the shells
 * e[round(|m|)] (m: integer wavenumber vector); e must be zeroed, and nshell = 1 + the
 * largest shell of the grid (lbm_spectral_shell_count, at most 6000). */
int lbm_spectral_shell_count(int nx, int ny, int nz);
lbm_status lbm_spectral_shells(const void* zh, const void* ch, int nx, int ny, int nz, double* e,
                               int nshell, void* cuda_stream);

#ifdef __cplusplus
}
#endif
#endif /* LBM_SPECTRAL_H_ */
