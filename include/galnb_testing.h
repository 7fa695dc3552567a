/*
 * galnb_testing.h -- test hooks of libgalnb.so, kept out of the public
 * interface in galnb.h.  They exercise failure paths that normal inputs never
 * reach; an application has no use for them.
 */
#ifndef GALNB_TESTING_H
#define GALNB_TESTING_H

#include "galnb.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Failure path of the tensor-core convolutions (no counterpart in the
 * paper): runs one forward pass on zeros in which the first convolution's
 * halo barriers expect 16 bytes more than its TMA loads deliver, so none of
 * its halo waits can complete.  Each bounded wait (1 s) runs out, the kernel
 * drains its copies and MMAs, frees TMEM and exits, and the call returns
 * GNB_ETIMEOUT; the network and the CUDA context stay usable.  Takes a few
 * seconds.  Errors: GNB_EINVAL (NULL, or the mma.sync path selected). */
int gnb_unet_test_wait_timeout(gnb_unet *net);

/* Out of device memory: after `after` further device allocations of the
 * context the next one fails, once, as cudaMalloc does without memory left
 * (the call that made it returns GNB_ENOMEM); -1 puts this off.  Returns what
 * was left of the former count (-1: no failure was due, or it has happened;
 * -2: NULL context). */
int64_t gnb_test_fail_alloc(gnb_ctx *ctx, int64_t after);

/* A bounded wait of the radix sort that runs out: the context's next sort
 * starts with its pass `pass` (the key's byte, 0 .. 7; the particles' sort
 * takes 2 .. 7) marked as given up.  The later passes do nothing and the call
 * returns GNB_ETIMEOUT.  -1 puts this off.  Errors: GNB_EINVAL. */
int gnb_test_sort_give_up(gnb_ctx *ctx, int pass);

/* The tile plan of the network's tensor-core 3^3 forward convolutions: number
 * `plan` of each layer's list of supported plans instead of the rule's (or the
 * autotuner's) choice, where the list is that long; -1 gives the choice back
 * to the rule.  Returns the longest list's length, or GNB_EINVAL. */
int gnb_unet_test_set_plan(gnb_unet *net, int plan);

/* y[i] = 10^x[i] as the remap forms its voxel weights (host arrays of n
 * doubles).  Errors: GNB_EINVAL, GNB_ENOMEM, GNB_ECUDA. */
int gnb_test_exp10(int64_t n, const double *x, double *y);

#ifdef __cplusplus
}
#endif

#endif /* GALNB_TESTING_H */
