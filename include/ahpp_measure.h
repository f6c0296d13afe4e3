/*
 * Measurement helpers of the AHPP library: device rates that roofline
 * reports divide by, and what a loaded graph was laid out as.  They live in the
 * same shared library as the query API (include/ahpp.h), whose status codes they
 * return.
 */
#ifndef AHPP_MEASURE_H
#define AHPP_MEASURE_H

#include "ahpp.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Row-access peak of a device, for roofline reporting (no graph needed).
 * The batched kernel moves its data as random 128-byte rows (32 queries x
 * FP32 of one node); once a table fits in L2 the L2 -> SM path, not HBM,
 * bounds those accesses.  This measures the rate, in rows per second, of
 * random 128-byte row gathers from (op 0) or float4 row reductions into
 * (op 1) a zero-filled device table of table_bytes (rounded down to 128-byte
 * rows), best of five launches after a warm-up.  Allocates and frees the
 * table itself and restores the caller's current device.  AHPP_EINVAL for
 * op not 0/1, table_bytes outside [128, 8 GiB], device < 0 or a NULL output;
 * AHPP_ENOMEM if the table cannot be allocated; AHPP_ECUDA otherwise. */
int ahpp_row_access_peak(int device, uint64_t table_bytes, int op, double *rows_per_s);

/* What the library built from a graph's arrays (graph_bytes of ahpp_graph_info)
 * for its pull rounds. */
typedef struct {
    uint64_t layout_bytes;               /* device bytes of the layouts, on top of graph_bytes */
    uint32_t cluster_blocks;             /* blocks of the one cluster that runs a single query (small
                                            graphs), 0: the whole-GPU kernel does */
    uint32_t cluster_smem_bytes;         /* shared memory of each of them */
} ahpp_layout_info;
int ahpp_get_layout_info(const ahpp_graph *g, ahpp_layout_info *info);

#ifdef __cplusplus
}
#endif

#endif /* AHPP_MEASURE_H */
