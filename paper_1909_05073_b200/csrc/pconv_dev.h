/*
 * Development entry points of the PCONV library.  They exist only in a library compiled with
 * -DPCONV_DEV (build.py: build(dev=True) -> libpconv_dev.so) and are not part of the public ABI
 * in include/pconv.h; none has a counterpart in the paper.  The development build is otherwise the
 * same code: it adds phase timestamps to the tiled kernel, lets the environment force a launch
 * plan (PCONV_FORCE_ZS / PCONV_FORCE_KS), and can make one bounded wait of a launch run out so
 * that the give-up path -- status word, skipped work, common exit, Tensor Memory handed back --
 * can be exercised without faulting or hanging anything.
 */
#ifndef PCONV_DEV_H_
#define PCONV_DEV_H_

#include "../../include/pconv.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Synchronises the device and copies the first n_words (<= PCONV_TRACE_WORDS) 64-bit trace words
 * of the handle to the HOST: timestamps of the tiled kernel's phases (nanoseconds of the global
 * timer for words 0-10, SM cycles for 11-12; each word's meaning is listed where the kernel
 * writes it). */
#define PCONV_TRACE_WORDS 14
pconv_status pconv_trace_read(const pconv_handle* h, unsigned long long* words_host, int n_words);

/* From now on, in every tiled-kernel launch on the current device, one producer thread leaves out
 * its arrival for chunk `chunk` (counted inside a CTA's chunk range) on the stage's "full"
 * barrier, and every bounded wait gives up after `spin_limit` tries (each try suspends the warp
 * for at most 200 ns) instead of the normal limit.  The consumers of that chunk then run out of
 * patience, record wait id 2 in the status word, skip their remaining work and leave through the
 * common exit; the launch produces no valid output.  chunk < 0 switches the behaviour off and
 * restores the normal limit.  Synchronises the device. */
pconv_status pconv_dev_withhold(int chunk, unsigned spin_limit);

/* Launch plans of the dense tensor-core kernel worked out by this process so far (a call that finds its
 * plan already made adds none). */
long long pconv_dev_dense_plans(void);

/* The dense kernel's plan for a shape on a device of 148 SMs of which `cluster_sms` can hold clusters (host
 * arithmetic, needs no device).  rows: the input is position rows.  prune = 0: every candidate is costed.
 * fields[14]: tiles of an item, filters of a tile, CTAs, split, cluster, equal parts of a tile, tiles, channel steps,
 * activation stages, weight slots, shared memory bytes, Tensor Memory columns of an accumulator set, workspace
 * bytes, a CTA's share.  PCONV_ERR_UNSUPPORTED if there is none. */
pconv_status pconv_dev_dense_plan(int c_out, int c_in, int stride, int storage, int tap_mask, int n, int h_in, int w_in,
                                  int pool, int rows, size_t ws_bytes, int cluster_sms, int prune, int* fields,
                                  double* cycles);

/* The kernel a default forward of this shape takes: 0 the sparse one, 1 the dense one from NCHW, 2 the dense one on
 * position rows.  rows: 0 there is no room for position rows, 1 there is, 2 they are there already. */
int pconv_dev_path(const pconv_handle* h, int n, int h_in, int w_in, int pool, int rows, size_t ws_bytes);

/* Layers of a stack that the dense kernel runs. */
int pconv_dev_stack_dense_layers(const pconv_stack* s);

/* Clears the handle's sticky status word (pconv_device_status reports PCONV_OK again until the
 * next abandoned wait).  Synchronises the device. */
pconv_status pconv_dev_clear_status(const pconv_handle* h);

#ifdef __cplusplus
}
#endif
#endif /* PCONV_DEV_H_ */
