// gbx_device.cuh -- the device-side data model of the move kernels: tile size, the copy
// and fold descriptors, segment and fold-record layouts.  Everything a move kernel reads
// is defined here or in gbx_move.cu.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#define GBX_TILE 1024                    // chunks per tile (block * unroll)
#define GBX_MAGIC_SHIFT 21               // (2 * GBX_TILE) * GBX_TILE: see unit_of
#define GBX_TERM_GROUP (1ull << 63)      // fold term: first term of a group
#define GBX_TERM_BUFB (1ull << 62)       // fold term: reads buffer B (else A)
#define GBX_TERM_MASK ((1ull << 62) - 1)
// fold row record: a = output byte offset | GBX_ROW_SINGLE; b = the row's only term when
// GBX_ROW_SINGLE is set, else (first term index << 24) | term count
#define GBX_ROW_SINGLE (1ull << 63)
#define GBX_ROW_CNT_BITS 24

#define GBX_ERR_NONE 0x7fffffff          // device error word: "no error yet"

// Buffer roles of an op's pointers (for re-binding).
enum { ROLE_SRC = 0, ROLE_DST = 1, ROLE_AGG = 2, ROLE_NONE = 3 };

struct Seg {
    int64_t v0;       // first element of the segment in the op's element space
    int64_t dst_off;  // byte offset of the segment's first destination element
    int64_t src_off;  // byte offset of the source base (contiguous: of the first element)
    int64_t idx_off;  // >= 0: element k reads index idx[idx_off + k]; < 0: contiguous
};

struct CopyDesc {
    const char *src;
    char *dst;
    const Seg *segs;
    const int32_t *idx;
    const int64_t *tile_seg;  // ntiles + 1: segment holding each tile's first element
    int64_t nseg, nelem, nchunks, ntiles, elem_size;
    int32_t vec, cpe, cpe_shift;  // chunks per element; log2 of it, or -1
    uint32_t cpe_magic;           // ceil(2^GBX_MAGIC_SHIFT / cpe), for cpe <= GBX_TILE
    uint64_t cpe_magic64;         // ceil(2^64 / cpe) when cpe is not a power of two
    int32_t src_role, dst_role;
    // flat form (when set): destinations are one contiguous run from dst_flat0 and element
    // e reads source element flat_idx[e]; no segment search
    int32_t flat;
    const int32_t *flat_idx;
    int64_t dst_flat0;
    int32_t bulk_dst;   // dst is device memory: the bulk-copy engine may write the run
    // flat form with two sources: an index with bit 31 set reads src2 (e.g. the receive
    // aggregate) instead of src
    const char *src2;
    int32_t src2_role;
    // two-index flat form (flat == 3): element e also writes destination element flat_didx[e]
    const int32_t *flat_didx;
    // bulk form (flat == 8): contiguous pieces moved by the bulk-copy engine
    const struct BulkTask *bulk;
    int64_t nbulk;
    // scatter form (flat == 9) of a two-index copy whose pairs (flat_idx, flat_didx) are sorted
    // by source: the sources are read a window at a time by the bulk-copy engine and
    // scattered from shared memory by the threads
    const struct ScatterPiece *scat;
    int64_t nscat;
    // window form (flat == 15) of a flat gather with one chunk per element: the elements grouped by
    // source window, each window read by the bulk-copy engine and gathered from shared memory
    const struct WinPiece *win;
    const uint16_t *win_idx;      // per slot: element of the window
    const uint2 *win_grp;         // per 32 slots: run starts (bit mask), runs started before
    const int32_t *win_run;       // per run: destination element minus slot
    int64_t nwin;
    int32_t win_elems;            // source elements per window: 1024 or 2048
    int32_t win_lead, win_lead2;  // address of src / src2 modulo 16, or -1: host memory
    // the waiting kernels (bulk, scatter, stream, window): the request's status word (host-mapped memory,
    // read by gbx_wait / gbx_test), set to 1 when a bounded wait gave up and 2 when a piece
    // failed its in-kernel check; and the spin limit of their main waits (the waits that
    // drain copies already in flight keep GBX_WAIT_LIMIT)
    int *status;
    int32_t wait_limit;
};
#define GBX_WAIT_LIMIT (1 << 22)

// One window of a scatter-form copy: the source elements of sorted pairs m0 .. m0+n-1 lie in
// nrun runs of contiguous source bytes, run r at [src + run_off[r], src + run_off[r] +
// run_len[r]) (16-byte multiples, ascending, disjoint, inside [src, src + len), len at most
// GBX_SCAT_WIN); the gaps between runs hold no pair's source and are not read.
#define GBX_SCAT_RUNS 24
#define GBX_SCAT_GAP 1024   // gaps up to this many bytes are read with their run
struct ScatterPiece {
    int64_t src, m0;
    int32_t len, n, nrun, pad;
    uint16_t run_off[GBX_SCAT_RUNS], run_len[GBX_SCAT_RUNS];
};

// One piece of a window-form gather: its n slots k = 0 .. n-1 (at p * GBX_WIN_N + k in win_idx, for
// piece p) read element win_idx of the `bytes` source bytes at `src` (of src2 when buf is set)
// and write destination element win_run[run] + k, run = the number of run starts up to k minus
// one (runs of piece p at p * GBX_WIN_RUNS).
struct WinPiece {
    int64_t src;
    int32_t bytes, n, nrun, buf, pad[2];
};
#define GBX_WIN_N 2048        // slots per piece
#define GBX_WIN_RUNS 1024     // runs per piece at most

// One piece of a bulk-form copy: len bytes (a multiple of 16, at most GBX_BULK_BYTES) from
// byte src of the op's source to byte dst of its destination, both 16-byte aligned.
struct BulkTask {
    int64_t src, dst, len;
};
#define GBX_BULK_BYTES 32768             // bytes per bulk piece (one shared-memory stage)
#define GBX_BULK_STAGES 4                // stages per CTA of the bulk kernel
// scatter form: a stage holds one source window of GBX_SCAT_WIN bytes, then the window's
// source indices and its destination indices (at most GBX_SCAT_MAXN pairs, each index copy
// rounded out to 16-byte boundaries, so the index arrays carry 4 elements of padding)
#define GBX_SCAT_WIN 16384
#define GBX_SCAT_MAXN (GBX_SCAT_WIN / 16)
#define GBX_SCAT_IDX (GBX_SCAT_MAXN * 4 + 16)
#define GBX_SCAT_STAGE (GBX_SCAT_WIN + 2 * GBX_SCAT_IDX)
#define GBX_FLAT_SRC2 0x80000000u

struct FoldDesc {
    char *out;
    const char *bufA;
    const char *bufB;
    const int64_t *row_ptr;   // nrows + 1 (setup and validation)
    const int64_t *row_out;   // byte offset of each row's output element (setup and validation)
    const longlong2 *rec;     // nrows packed row records (the kernel's view)
    const int64_t *terms;     // byte offset | GBX_TERM_GROUP | GBX_TERM_BUFB
    int64_t nrows, nchunks, ntiles, elem_size;
    int32_t vec, cpe, cpe_shift;
    uint32_t cpe_magic;
    uint64_t cpe_magic64;
    int32_t dtype, accumulate;
    int32_t out_role, a_role, b_role;
    // window form (fold form 2): the rows of one-chunk elements cut into pieces (see FoldPiece)
    const struct FoldPiece *wpiece;
    const uint16_t *wpos, *wbase, *wrowout;
    const uint8_t *wrowcnt;
    const uint2 *wgrp;
    const uint32_t *wrun, *wgroup;
    int64_t nwpiece;
    int32_t wgroups;          // some row has more than one group
    int *status;              // the request's status word (see CopyDesc)
    int32_t wait_limit;
};

// One piece of a window-form fold: rows row0 .. row0 + nrow - 1, n terms in all, gathered in source
// order.  Slot k of piece p (tables at p * GBX_WFOLD_N) reads source element
// (wrun[run] & 0x7fffffff) - GBX_WFOLD_N + k of bufA (bufB where bit 31 of the run is set; runs of
// piece p at p * GBX_WFOLD_RUNS) and puts it at place wpos[k].  The rows are taken in order of
// their length, 32 to a slice: term m of row r (in that order) has place wbase[r / 32] + 32 * m +
// r % 32, its row wrowcnt[r] terms, summed in order into output element out0 + wrowout[r]; bit i of
// wgroup: the term at place i starts a group.  (wbase and wgroup of piece p at p * GBX_WFOLD_N / 32.)
struct FoldPiece {
    int64_t row0, out0;
    int32_t nrow, n, nrun, pad;
};
#define GBX_WFOLD_N 4096
#define GBX_WFOLD_RUNS 2048
#define GBX_WFOLD_ROW 64      // terms per row at most
