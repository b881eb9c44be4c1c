/*
 * sva_debug.h -- test and tuning aids exported by libsva.so next to the public calls of sva.h.
 *
 * Unlike everything in sva.h these three calls keep PROCESS-GLOBAL state (host variables and two device
 * variables per loaded library): a setting stays in force for every later launch of the process
 * until it is set back.  They are meant for single-threaded test and bench programs.  The paper has no
 * counterpart.
 */
#ifndef SVA_DEBUG_H_
#define SVA_DEBUG_H_

#ifdef __cplusplus
extern "C" {
#endif

/*
 * Cycle counter of the attention kernel.  buf: DEVICE buffer of at least 320 int64 (the caller zeroes it), or
 * NULL to switch the counter off again.  While set, every attention launch does an atomicMax of its CTAs'
 * elapsed SM cycles (clock64 from kernel entry to tear-down) into buf[319]: the cycle count of the longest
 * CTA, i.e. of the launch, independent of the SM clock (cycles / time = the clock the launch really ran at).
 */
void sva_debug_set_prof_buffer(void* buf);

/*
 * Kernel behaviour switches for the next launches (0 = normal operation).
 *   bit 4: test aid: the K producer withholds a row's tiles after the first, so that a bounded pipeline wait
 *          runs out and the kernel takes its give-up path (SVA_DEV_TIMEOUT) -- nothing faults or hangs.
 *   bit 5: measurement aid: the one-call forms (but the 4-bit one) read a transposed copy of V that they make first, as the two-step form
 *          does, instead of V where it lies; they then need sva_attn_workspace_bytes() (the remainder: its own query, asked meanwhile);
 *   bit 6: test aid: the one-launch routing of small problems asks for clusters of 32 CTAs, which no device holds, so that the
 *          call goes the way it goes in a partition of the device that is too small for its clusters;
 *   bit 7: test aid: the remainder call masks the kept blocks of a block-mean tile by looking them up in the CSR
 *          (the form that serves more than 1024 key blocks) even where the kept-block bit masks would serve;
 *   bit 8: test aid: the kernel of the first-order term's block covariances withholds a part of its V tile, and
 *   bit 9: the one that adds them up withholds every column tile of a CTA after its first, so that bounded waits run out.
 */
void sva_debug_set_mode(int bits);

/*
 * Test aid: the number of SM cycles a device-side wait may last before its CTA gives up (default 3e9, at most 4e9: larger
 * values count as that; cycles <= 0 restores the default).  Synchronous (two small host-to-device copies on the current device).
 * Returns 0 on success.
 */
int sva_debug_set_wait_limit(long long cycles);

#ifdef __cplusplus
}
#endif
#endif /* SVA_DEBUG_H_ */
