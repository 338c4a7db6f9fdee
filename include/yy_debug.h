/*
 * yy_debug.h - test hooks of libyy (not needed by applications).
 *
 * Fault injection is done on the host only: a hook makes the library's
 * own allocation wrapper report failure so the error paths can be exercised
 * without touching the GPU's state.
 */
#ifndef YY_DEBUG_H
#define YY_DEBUG_H

#ifdef __cplusplus
extern "C" {
#endif

/* Make the n-th following device allocation made by the library fail with
 * YY_ERR_OOM (n = 0: the next one).  A negative n disables the hook.  Not
 * thread-safe; process-wide. */
void yy_debug_fail_alloc_after(int n);

/* The scale 2^-q under which YY_FP64_OZAKI writes the trig table
 * trig[2 l_max + 1][columns] (host memory; 1, then cos and sin of order 1, 2, ...) as
 * digits whose sums are exact: q, or -1 where no scale that it tries is (yy_grid_prepare
 * then gives YY_ERR_NOT_SUPPORTED); -2: invalid argument.  Host only. */
int yy_debug_oz_trig_scale(const double *trig, int l_max, int columns);

#ifdef __cplusplus
}
#endif

#endif /* YY_DEBUG_H */
