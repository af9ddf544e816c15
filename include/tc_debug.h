/*
 * tc_debug.h -- test hooks of libtc (see tc.h): failure paths, work counters.
 *
 * The paper has no counterpart: these calls exist so that tests can drive
 * the library's error paths without faulting or hanging a GPU, and see what a
 * call's kernels do.  The hooks change process-wide (allocation failures,
 * scans) or per-device (waits) state and are not meant for production use;
 * tc_debug_reset() undoes all of them.
 */
#ifndef TC_DEBUG_H
#define TC_DEBUG_H

#include <stdint.h>

#include "tc.h"

#ifdef __cplusplus
extern "C" {
#endif

/*
 * Bounded device waits, made to run out.  The preprocessing kernels wait
 * (spin) on status words that earlier tiles of the same launch publish
 * (decoupled look-back); every such wait gives up after a bounded number of
 * iterations, records the failure in the call's error word, and the call
 * returns TC_ERR_TIMEOUT with nothing computed from incomplete data (later
 * kernels of the call return at entry).  On the CURRENT device:
 *   spin_limit        iterations before a wait gives up (default 2^24)
 *   unpublished_tile  >= 0: the radix-sort tile with this number never
 *                     publishes its status, so the tiles after it wait on a
 *                     word that nothing sets and give up after spin_limit
 *                     iterations (meanwhile every call sorts by radix passes,
 *                     the small ones too that otherwise sort by counting);
 *                     < 0: every tile publishes (default)
 * Synchronises the device.  Returns TC_ERR_CUDA if the device rejects it.
 */
tc_status tc_debug_set_wait_limit(uint32_t spin_limit, int32_t unpublished_tile);

/*
 * The same for the offset scans, the waits that every call has: tile `tile`
 * (4096 vertices each) of the scan of the forward lists (scan 0) or of the
 * partner groups (scan 1) never publishes its status; tile < 0: all of that
 * scan do (default).  Process-wide, for calls made and engines created from
 * now on (an engine keeps what it was created with).
 */
tc_status tc_debug_set_unpublished_scan(int32_t scan, int32_t tile);

/*
 * Allocation failures, injected on the host: of the library's next device
 * allocations (workspaces, engine buffers, host-call staging), the first
 * `skip` succeed and the `count` after them fail as if the device were out
 * of memory (the call returns TC_ERR_OOM and releases what it had taken).
 * count <= 0 turns injection off.  Process-wide.
 */
tc_status tc_debug_fail_allocations(int32_t skip, int32_t count);

/*
 * What the counting kernels of one tc_count (per_vertex == 0) or
 * tc_count_per_vertex call do for this graph, counted over the very groups and
 * streams of that call by one more kernel (tc_count_work reports a split of its
 * own, see tc.h).  Vertices of equal degree class may come in any order, so the
 * counters of calls that sort by counting can differ a little from call to call.
 *   partners         edges left to an intersection, over all groups
 *   lookups          list entries streamed through hash tables
 *   inserts          list entries hashed
 *   bitmap_pairs     partners of `partners` that are intersected by bitmaps of
 *                    the top ranks too (512 bytes each)
 *   triangles        T
 *   dense_vertices   size of the hub set counted on the tensor cores (0: none)
 *   dense_triangles  triangles counted there
 * Same arguments and errors as those calls; synchronises `stream`.
 */
typedef struct tc_run_work {
  int64_t partners;
  int64_t lookups;
  int64_t inserts;
  int64_t bitmap_pairs;
  uint64_t triangles;
  uint64_t dense_triangles;
  int32_t dense_vertices;
  int32_t pad_;
} tc_run_work;
tc_status tc_debug_run_work(const int32_t *src, const int32_t *dst, int64_t m, int32_t n,
                            int32_t per_vertex, tc_stream_t stream, tc_run_work *out);

/* Default wait limit and no unpublished tiles on the current device, and no
 * injected allocation failures. */
tc_status tc_debug_reset(void);

#ifdef __cplusplus
}
#endif

#endif /* TC_DEBUG_H */
