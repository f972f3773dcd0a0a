/*
 * tahq_testing.h -- entry points of libtahq for its tests and its benchmark, kept apart from the codec's
 * C ABI (tahq.h).  None of them has a counterpart in the paper; a caller of the codec needs none of them.
 */
#ifndef TAHQ_TESTING_H
#define TAHQ_TESTING_H

#include "tahq.h"

#ifdef __cplusplus
extern "C" {
#endif

/*
 * Self-test of the library's bounded device-side waits (the paper has no counterpart).  Launches a two-CTA
 * kernel in which one CTA waits, as the offset look-back of decode does, for a count that is never
 * published.  The wait gives up after its fixed number of polls (about a second), the kernel returns, and
 * the device status word at d_ws[0..4) reads TAHQ_DEV_TIMEOUT; the CUDA context stays usable.  d_ws: at
 * least 32 KiB of device memory.
 */
tahq_status tahq_selftest_wait_timeout(void *d_ws, size_t ws_cap, tahq_stream stream);

/* Number of kernels the last tahq_encode / tahq_decode call of this thread enqueued. */
int tahq_last_launch_count(void);

/*
 * Per-kernel timing for benchmarks (off by default; the record list is guarded by a mutex, the switch is
 * process-wide; the paper has no counterpart).
 * tahq_profile(1) clears earlier records and makes every following kernel launch of the library be
 * bracketed by two CUDA events on its stream; tahq_profile(0) stops recording.
 * tahq_profile_read waits for the recorded events, writes up to max_records kernel names
 * (32 bytes each, NUL-terminated, into `names`) and their durations in milliseconds (into `ms`),
 * in launch order, clears the records and returns how many were written.  Host pointers.
 */
void tahq_profile(int enable);
int tahq_profile_read(char *names, float *ms, int max_records);

/*
 * Timeline of the kernels of a call, for benchmarks (off by default; process-wide; not thread-safe).  d_buf is a
 * device buffer of 64 unsigned 64-bit words, or NULL to switch the recording off.  While it is set, every
 * encode/decode kernel k (0 clear, 1 scores, 2 selection, 3 quantise + pack, 4 its outlier pass, 5 decode, 6 its
 * outlier pass) records into words 4k .. 4k+2 the smallest global-timer value at which one of its CTAs was resident,
 * the smallest at which one got past the wait for the kernel in front, and the largest at which one of its warps
 * finished (atomic min / min / max: the caller presets the words to all-ones / all-ones / zero).
 */
void tahq_trace(void *d_buf);

#ifdef __cplusplus
}
#endif
#endif /* TAHQ_TESTING_H */
