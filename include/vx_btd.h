/*
 * vx_btd.h -- C ABI of the batched block-tridiagonal solve of the per-ray Newton systems.
 *
 * Where it sits in the method. The radial transport sweeps of Marek et al. (arXiv:1404.1719) are
 * implicit in time and run ray by ray; each ray's step is a non-linear system in the zone unknowns,
 * solved by Newton-Raphson iterations with an explicitly built Jacobian and a direct solve of the
 * linearised system (sec. 2.1). A radial difference scheme couples a zone only to its neighbours,
 * so for the zones k = 0 .. n-1 of one ray, with m unknowns per zone, that linear system reads
 *
 *     A_k x_{k-1} + B_k x_k + C_k x_{k+1} = d_k        (A_0 and C_{n-1} are not read).
 *
 * The pair-process source derivatives of vx_rates_spectral (blocks d(j0, chi0)/dJ and
 * d(j1, chi1)/dH of the partner spectrum) are part of B_k in such a system; the radial flux terms
 * make A_k and C_k. Rays are independent (sec. 2.2) and are solved in one call.
 *
 * Method (GB300: FP32 arithmetic, FP64 only where accuracy needs it). Block LU along the ray
 * without pivoting across zones: D_0 = B_0, D_k = B_k - A_k G_{k-1} with G_k = D_k^{-1} C_k,
 * each D_k inverted with partial pivoting inside the block. The factorisation is done in FP32 from
 * FP32 copies of the blocks, one CTA per ray, its matrix products on the tensor cores (TF32 with each
 * operand split into two parts, three products: about FP32 accuracy); D_k^{-1} and G_k are kept. Where
 * rays are few, a ray is eliminated from both ends at once by two CTAs, or in segments of its zones by a
 * CTA each and then the system of the segments' last zones (chosen by n_rays, n_zones and m, so a
 * ray's last bits depend on the batch it is in); if a pivot fails there, or entries of D^{-1} C or the like
 * exceed 4, the ray is done again from its first zone on. Then
 * the ray is solved by matrix-vector products with those, y_k = D_k^{-1} (d_k - A_k y_{k-1}) forward and
 * x_k = y_k - G_k x_{k+1} backward, and
 * n_refine sweeps of iterative refinement follow, each from the FP64 residual d - M x of the
 * caller's FP64 blocks; one or two more in a ray with an ill-conditioned block (its largest pivot more than 24 or 256
 * times the smallest), which is not cut into segments either: inverses would leave it further off than elimination
 * does. If these leave a residual of more than 0.03^(n_refine + 2) of rhs (at least 1e-10), the ray is eliminated in
 * FP64 instead, slowly: about 0.85 ms a zone at m = 84. For a ray whose Schur complements are well conditioned (e.g.
 * block rows diagonally dominant) every sweep gains a factor of about cond x 1e-7, so two sweeps reach FP64 accuracy at
 * moderate condition numbers. The reduction order is fixed: the results of a batch are
 * reproducible run to run.
 *
 * Conventions (as in vx_rates.h): arrays are dense, row-major FP64 unless stated; device pointers
 * are CUDA global memory of the current device, owned by the caller; the library never retains a
 * caller pointer after a call returns. Calls are asynchronous on `stream`; argument checks happen
 * on the host before anything is launched, and a rejected call returns VX_ERR_INVALID_ARG and
 * writes nothing. A handle is not thread-safe.
 */
#ifndef VX_BTD_H
#define VX_BTD_H

#include "vx_rates.h" /* vx_status, vx_stream, vx_status_string, vx_last_error */

#ifdef __cplusplus
extern "C" {
#endif

typedef struct vx_btd vx_btd;

#define VX_BTD_MAX_M 128      /* unknowns per zone */
#define VX_BTD_MAX_REFINE 8

/* Creates a solver for m unknowns per zone (1 .. VX_BTD_MAX_M) and batches of at most max_zones
 * zones (>= 0), with n_refine FP64 refinement sweeps (0 .. VX_BTD_MAX_REFINE; 0 leaves the FP32
 * solution, but in rays with ill-conditioned blocks). Allocates the device workspace: 12 m (m + 7) + 4 (m + 7) + 12 m + 20
 * bytes per zone at most, and, for max_zones of 40 or more and m up to 116, what rays in segments take besides:
 * 4 m (m + 7) for each zone that
 * 4 min(max_zones, 16384) exceeds 3 max_zones by (none from 21,846 zones on), and 36 m^2 + 300 m + 76 per SM. Without
 * the memory for that, rays are not cut into segments. *out is set to NULL on failure. Errors: VX_ERR_INVALID_ARG,
 * VX_ERR_OOM, VX_ERR_CUDA. */
vx_status vx_btd_create(int m, long long max_zones, int n_refine, vx_btd **out);

/* The same for calls of min_rays rays (>= 1) or more: where such calls are never cut into segments (min_rays above
 * a fifth of the SMs), the memory for that is not taken. Calls of fewer rays are solved all the same, as a whole. */
vx_status vx_btd_create_rays(int m, long long max_zones, int n_refine, int min_rays, vx_btd **out);

/* Solves every ray. n_rays >= 0; n_zones = the total zone count, 0 .. max_zones.
 *   ray_offsets: device int32 [n_rays + 1]; ray r owns zones ray_offsets[r] .. ray_offsets[r+1]-1.
 *                Must start at 0, not decrease and end at n_zones (checked on the device: if not,
 *                nothing is solved, x is left unwritten and the numeric flag is raised).
 *   A, B, C:     device FP64 [n_zones][m][m], the sub-diagonal, diagonal and super-diagonal blocks
 *                of each zone's block row (A of a ray's first zone and C of its last are not read).
 *   d:           device FP64 [n_zones][m], right-hand sides.
 *   x:           device FP64 [n_zones][m], the solution (written; must not overlap d or the blocks).
 * A ray with a zero or non-finite pivot gets NaN in x and raises the numeric flag (vx_btd_check).
 * Errors: VX_ERR_INVALID_ARG (NULL handle or pointers with n_zones > 0, a pointer that is not device
 * (or managed) memory, offsets not 4-byte or FP64 arrays not 8-byte aligned, n_rays < 0, n_zones
 * out of range, x overlapping an input), VX_ERR_CUDA. Nothing is launched then. */
vx_status vx_btd_solve(vx_btd *h, int n_rays, long long n_zones, const int *ray_offsets, const double *A,
                       const double *B, const double *C, const double *d, double *x, vx_stream stream);

/* Synchronises `stream` and returns VX_ERR_NUMERIC if a solve since the last check met a zero or
 * non-finite pivot or invalid ray offsets (then clears the flag), else VX_OK. */
vx_status vx_btd_check(vx_btd *h, vx_stream stream);

/* Frees the handle and its workspace (NULL is a no-op). */
void vx_btd_destroy(vx_btd *h);

#ifdef __cplusplus
}
#endif

#endif /* VX_BTD_H */
