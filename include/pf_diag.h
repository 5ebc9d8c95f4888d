/*
 * pf_diag.h -- diagnostic entry points of libpf.so for tests of what a
 * filter's results do not show.  They are not part of the particle-learning
 * method: the paper has no counterpart.  The failure handling is exercised
 * without faulting or hanging a GPU, by making one of the library's bounded
 * device waits run out on purpose.
 */
#ifndef PF_DIAG_H
#define PF_DIAG_H

#include <stddef.h>
#include <stdint.h>

#include "pf.h"

#ifdef __cplusplus
extern "C" {
#endif

/* pf_cdf (the exact fixed-point CDF of float weights, a single-pass scan with
 * decoupled look-back over 4096-element tiles) with test settings of the
 * look-back's bounded wait.  The tile that takes ticket `withhold_tile`
 * publishes neither its aggregate nor its prefix, so the next tile polls its
 * status word until `spin_limit` polls have passed, gives up and raises the
 * timeout bit of the error word; the call then returns PF_ERR_TIMEOUT and
 * Q_dev holds no valid CDF.  withhold_tile = 0xffffffff withholds nothing
 * (the call is then pf_cdf with a wait of spin_limit polls; pf_cdf itself
 * waits up to 2^22 polls).  Every wait is bounded, so the call always
 * returns, and nothing persists between calls: a later pf_cdf on the same
 * stream works normally.  Arguments otherwise as pf_cdf (device pointers,
 * n in [1, 2^26], spin_limit >= 1); synchronises `stream`. */
pf_status pf_diag_cdf_wait(const float* w_dev, uint64_t n, uint32_t withhold_tile,
                           uint32_t spin_limit, uint64_t* Q_dev, void* stream);

/* How a handle takes one block of device memory from its allocator callbacks,
 * on the host alone (the addresses are not used): *raw is what free must get
 * back, *start the block's first byte, at a multiple of 32. */
pf_status pf_diag_block(pf_alloc_fn alloc, pf_free_fn free, void* ctx, size_t bytes, void** raw,
                        void** start);

/* The correctly rounded arithmetic that the kernels use in place of the
 * compiler's division and square root, element by element on device arrays of
 * n values (8-byte aligned).  op 0..8: binary32, n even, the values taken in
 * pairs: 0 1/a, 1 a/b, 2 sqrt a, 3 sqrt a one value at a time, 4 a/b of the
 * predictive weights (any operands), 5 and 6 a/b of the inverse-gamma draws for
 * shapes below and from 2^60, 7 1/(a+b) and 8 sqrt((a b) (1/(a+b))) of the
 * propagation.  op 16, 17: binary64 a/b and sqrt a.  Synchronises `stream`. */
pf_status pf_diag_arith(int op, const void* a, const void* b, void* out, uint64_t n, void* stream);

#ifdef __cplusplus
}
#endif

#endif /* PF_DIAG_H */
