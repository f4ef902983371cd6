// gbx_move.cu -- the exchange's data-movement kernels (the hot path).
//
// gbx_copy_kernel: for every element e of a copy op, with s = elem_size,
//     dst[seg.dst_off + k*s .. +s) = src[seg.src_off + sel*s .. +s),  k = e - seg.v0,
//     sel = idx[seg.idx_off + k] (gather through the send index list) or k (contiguous)
//   This one kernel is the pack + block copy + unpack of the standard neighbourhood
//   all-to-all-v (MPI Advance section 2.2: every message, packed by its send list and
//   unpacked at its receive displacement, in one pass) and each step of the
//   locality-aware form (direct copy, gather into node-pair aggregates, one block per
//   node pair, redistribution).  Bytes are copied as opaque vectors: bit-exact.
// gbx_fold_kernel: for every row of a fold op,
//     out[row] (+)= fold over the row's groups, in order, of (fold over the group's terms)
//   with IEEE round-to-nearest adds in the payload type: the reverse exchange.
//
// Both kernels walk tiles of GBX_TILE chunks (chunk = one `vec`-byte vector) with a
// grid-stride loop; a launch may cover several ops (patterns), found by binary search
// over the tile prefix, so uneven patterns share one grid.  Consecutive threads handle
// consecutive chunks: destination writes are fully coalesced 16-byte stores, source
// reads are 16-byte vector gathers of whole elements.  No shared memory, no barriers,
// no waits: a launch always terminates.
//
// Every kernel takes its ops in one of two ways (template parameter L).  A launch of one op
// carries the op's descriptor by value (OneOp, read from the constant bank): no load of a
// descriptor pointer and then of its fields stands between the start of the kernel and its
// first index load, and a rebind only changes the next launch's argument.  A pooled launch
// (OpList, the batches) reads a list of descriptors in device memory.  Measured together with
// dependent launches and untimed events (start + wait, before and after): 3,072 8-byte points
// 13.7 -> 11.8 us, a 3-launch locality exchange of 78 k 24-byte points 20.3 -> 14.1, 2.6 M 24-byte
// records 46.6 -> 35.0, 1.7 M 8-byte values under datatypes 22.6 -> 16.8, 2^20-row SpMV halo fp64
// 41.1 -> 39.0, forward + backward of the fp32 one through autograd 230 -> 196.
#include "gbx_internal.cuh"

template <int VEC> struct VecT;
template <> struct VecT<16> { typedef uint4 T; };
template <> struct VecT<8> { typedef uint2 T; };
template <> struct VecT<4> { typedef unsigned int T; };
template <> struct VecT<2> { typedef unsigned short T; };
template <> struct VecT<1> { typedef unsigned char T; };

// Payload loads are plain ld.global: within a chain of dependent launches the payload may be
// written (by the launch before) after this kernel has started, which the non-coherent path does
// not allow for.  Indices and descriptors, fixed at init, use it.  (With the descriptor in the
// constant bank the two run equally fast, and so did L1::no_allocate, L2 prefetch hints and
// evict-first stores.)
template <int VEC>
__device__ __forceinline__ typename VecT<VEC>::T ldv(const char *p) {
    return *reinterpret_cast<const typename VecT<VEC>::T *>(p);
}
template <int VEC>
__device__ __forceinline__ void stv(char *p, typename VecT<VEC>::T v) {
    *reinterpret_cast<typename VecT<VEC>::T *>(p) = v;
}

// Largest op index whose tile range starts at or before t.
__device__ __forceinline__ int find_op(const int64_t *__restrict__ prefix, int nops, int64_t t) {
    int lo = 0, hi = nops - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(prefix + mid) <= t) lo = mid; else hi = mid - 1;
    }
    return lo;
}

template <typename D>
struct OneOp {
    static constexpr bool single = true;
    D d;
    int64_t ntiles;
    __device__ __forceinline__ int64_t tiles() const { return ntiles; }
    __device__ __forceinline__ const D *first() const { return &d; }
    __device__ __forceinline__ const D *at(int64_t t, int64_t &lt) const {
        lt = t;
        return &d;
    }
    __device__ __forceinline__ int count() const { return 1; }
    __device__ __forceinline__ const D *op(int) const { return &d; }
};

// A walk over a launch's tiles in ascending order: the descriptor of the tile's op.
template <typename L> struct Cursor;
template <typename D>
struct Cursor<OneOp<D>> {
    const OneOp<D> &l;
    __device__ __forceinline__ explicit Cursor(const OneOp<D> &list) : l(list) {}
    __device__ __forceinline__ const D &at(int64_t t, int64_t &lt) {
        lt = t;
        return l.d;
    }
};

template <typename D>
struct OpList {
    static constexpr bool single = false;
    const D *const *ops;
    const int64_t *prefix;
    int nops;
    int64_t ntiles;
    __device__ __forceinline__ int64_t tiles() const { return ntiles; }
    __device__ __forceinline__ const D *first() const { return ops[0]; }
    // the op whose tiles hold tile t of the launch, and the tile's number in that op
    __device__ __forceinline__ const D *at(int64_t t, int64_t &lt) const {
        const int op = nops > 1 ? find_op(prefix, nops, t) : 0;
        lt = nops > 1 ? t - __ldg(prefix + op) : t;
        return ops[op];
    }
    __device__ __forceinline__ int count() const { return nops; }
    __device__ __forceinline__ const D *op(int i) const { return ops[i]; }
};

// (The descriptor is held by value: the fields that the kernel uses stay in registers until the walk
// comes to another op.  Read through the pointer, they are loaded again after every store and
// wait, the async gather's 12 fields twice per unit, from an L1 that the gathers flush: 512^3
// stencil halo, one op in a list, 773 us; held, 606.)
template <typename D>
struct Cursor<OpList<D>> {
    const OpList<D> &l;
    D d;
    int64_t lo = 0, hi = 0;   // tiles of d's op
    __device__ __forceinline__ explicit Cursor(const OpList<D> &list) : l(list) {}
    __device__ __forceinline__ const D &at(int64_t t, int64_t &lt) {
        if (t >= hi) {
            const int op = l.nops > 1 ? find_op(l.prefix, l.nops, t) : 0;
            lo = l.nops > 1 ? __ldg(l.prefix + op) : 0;
            hi = l.nops > 1 ? __ldg(l.prefix + op + 1) : l.ntiles;
            d = *l.ops[op];
        }
        lt = t - lo;
        return d;
    }
};

// The launches of one request form a chain of programmatic dependent launches: a kernel lets
// the next one of the chain start its set-up as soon as all of its own blocks run
// (pdl_trigger), and touches payload only after the one before it has finished
// (pdl_wait).  Both do nothing in a launch without that attribute.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// dep: the launch depends on the one before it in the stream (its chain's), as above
template <typename L>
static cudaError_t launch(void (*f)(const L), int grid, int block, size_t smem, cudaStream_t st, bool dep, const L &l) {
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)block);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &a;
    c.numAttrs = dep ? 1 : 0;
    return cudaLaunchKernelEx(&c, f, l);
}

// Unit (element or row) that holds local chunk x of a tile whose first chunk is a chunk of unit 0:
// x < GBX_TILE + cpe - 1.  Units of at most a tile: magic = ceil(2^21 / cpe), exact for x < 2048;
// of a longer one a tile holds parts of two at most.  No branch: three ways by kind of cpe (shift,
// multiply, divide) cost the 512^3 stencil halo 557 us where this takes 548, 606 and 580 with the
// descriptor in device memory, where the compiler cannot know the branches to be uniform (2.6 M
// 24-byte records: 34.3 and 33.0).
__device__ __forceinline__ uint32_t unit_of(uint32_t x, int cpe, uint32_t magic) {
    return cpe > GBX_TILE ? (uint32_t)(x >= (uint32_t)cpe) : (x * magic) >> GBX_MAGIC_SHIFT;
}

// First unit of the tile (or part of one) whose first chunk is c0: computed, so that no load of a
// tile table stands before the index load (three launches over 78 k 24-byte points: 14.1 -> 13.6 us;
// with a hardware division instead of the 64-bit reciprocal, exact here for every c0 < 2^64 / cpe,
// 2.6 M 24-byte records took 37.1 us, 35.0 with the table).
template <typename D>
__device__ __forceinline__ int64_t first_unit(const D *d, int64_t c0) {
    return d->cpe_shift >= 0 ? c0 >> d->cpe_shift : (int64_t)__umul64hi((uint64_t)c0, d->cpe_magic64);
}

// ------------------------------------------------------------------------ copy
// flat form: destinations contiguous from dst_flat0, element e reads source element
// flat_idx[e]; the index load is the only dependency of the data load
template <int VEC, int U>
__device__ __forceinline__ void copy_tile_flat(const CopyDesc *__restrict__ d, int64_t t) {
    typedef typename VecT<VEC>::T V;
    constexpr int B = GBX_TILE / U;
    const int cpe = d->cpe;
    const uint32_t magic = d->cpe_magic;
    const int64_t e0 = first_unit(d, t * GBX_TILE);
    const uint32_t r0 = (uint32_t)(t * GBX_TILE - e0 * cpe);
    const int64_t left = d->nchunks - t * GBX_TILE;
    const int64_t s = d->elem_size;
    const int32_t *__restrict__ g = d->flat_idx;
    int64_t soff[U], doff[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
        const uint32_t x = r0 + (uint32_t)(u * B) + threadIdx.x;
        const uint32_t el = unit_of(x, cpe, magic);
        const int64_t j = (int64_t)(x - el * (uint32_t)cpe) * VEC;
        const int64_t e = e0 + el;
        const bool ok = (int64_t)(u * B + threadIdx.x) < left;
        const uint32_t gi = ok ? (uint32_t)__ldg(g + e) : 0u;
        // bit 31 selects the second source; offsets stay below 2^63 so the bit survives
        soff[u] = (((int64_t)(gi & ~GBX_FLAT_SRC2)) * s + j) | ((int64_t)(gi >> 31) << 62);
        doff[u] = d->dst_flat0 + e * s + j;
    }
    V val[U];
#pragma unroll
    for (int u = 0; u < U; u++)
        if ((int64_t)(u * B + threadIdx.x) < left) {
            const char *base = (soff[u] >> 62) ? d->src2 : d->src;
            val[u] = ldv<VEC>(base + (soff[u] & ((1ll << 62) - 1)));
        }
#pragma unroll
    for (int u = 0; u < U; u++)
        if ((int64_t)(u * B + threadIdx.x) < left) stv<VEC>(d->dst + doff[u], val[u]);
}

// two-index flat form: element e reads source element flat_idx[e] (bit 31 = second source)
// and writes destination element flat_didx[e]
template <int VEC, int U>
__device__ __forceinline__ void copy_tile_flat2(const CopyDesc *__restrict__ d, int64_t t) {
    typedef typename VecT<VEC>::T V;
    constexpr int B = GBX_TILE / U;
    const int cpe = d->cpe;
    const uint32_t magic = d->cpe_magic;
    const int64_t e0 = first_unit(d, t * GBX_TILE);
    const uint32_t r0 = (uint32_t)(t * GBX_TILE - e0 * cpe);
    const int64_t left = d->nchunks - t * GBX_TILE;
    const int64_t s = d->elem_size;
    int64_t soff[U], doff[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
        const uint32_t x = r0 + (uint32_t)(u * B) + threadIdx.x;
        const uint32_t el = unit_of(x, cpe, magic);
        const int64_t j = (int64_t)(x - el * (uint32_t)cpe) * VEC;
        const int64_t e = e0 + el;
        const bool ok = (int64_t)(u * B + threadIdx.x) < left;
        const uint32_t gi = ok ? (uint32_t)__ldg(d->flat_idx + e) : 0u;
        const int64_t go = ok ? (int64_t)__ldg(d->flat_didx + e) : 0;
        soff[u] = (((int64_t)(gi & ~GBX_FLAT_SRC2)) * s + j) | ((int64_t)(gi >> 31) << 62);
        doff[u] = go * s + j;
    }
    V val[U];
#pragma unroll
    for (int u = 0; u < U; u++)
        if ((int64_t)(u * B + threadIdx.x) < left) {
            const char *base = (soff[u] >> 62) ? d->src2 : d->src;
            val[u] = ldv<VEC>(base + (soff[u] & ((1ll << 62) - 1)));
        }
#pragma unroll
    for (int u = 0; u < U; u++)
        if ((int64_t)(u * B + threadIdx.x) < left) stv<VEC>(d->dst + doff[u], val[u]);
}

// Software-pipelined flat forms for a single-op persistent launch: the index loads of the
// block's next tile are issued while the current tile's payload loads are in flight, so the
// payload loads no longer wait for a full index round trip.  FORM 1: flat gather, 3: two-index.
template <int VEC, int U, int FORM>
__device__ __forceinline__ void flat_indices(const CopyDesc *__restrict__ d, int64_t t, uint32_t (&gi)[U],
                                             int32_t (&gd)[U], int64_t (&e)[U], int64_t (&j)[U], bool (&ok)[U]) {
    constexpr int B = GBX_TILE / U;
    const int cpe = d->cpe;
    const uint32_t magic = d->cpe_magic;
    const int64_t e0 = first_unit(d, t * GBX_TILE);
    const uint32_t r0 = (uint32_t)(t * GBX_TILE - e0 * cpe);
    const int64_t left = d->nchunks - t * GBX_TILE;
#pragma unroll
    for (int u = 0; u < U; u++) {
        const uint32_t x = r0 + (uint32_t)(u * B) + threadIdx.x;
        const uint32_t el = unit_of(x, cpe, magic);
        j[u] = (int64_t)(x - el * (uint32_t)cpe) * VEC;
        e[u] = e0 + el;
        ok[u] = (int64_t)(u * B + threadIdx.x) < left;
        gi[u] = ok[u] ? (uint32_t)__ldg(d->flat_idx + e[u]) : 0u;
        if (FORM == 3) gd[u] = ok[u] ? __ldg(d->flat_didx + e[u]) : 0;
    }
}

// NC: payload through the non-coherent path, in launches that never depend on the one before (lists):
// with the descriptor in device memory it is 551 us against 589 (512^3 stencil halo), read from the
// constant bank the two are equal.
template <int VEC, int U, int FORM, bool NC>
__device__ __forceinline__ void copy_flat_pipelined(const CopyDesc *__restrict__ d, int64_t ntiles) {
    typedef typename VecT<VEC>::T V;
    const int64_t s = d->elem_size;
    int64_t t = blockIdx.x;
    if (t >= ntiles) return;
    uint32_t gi[U];
    int32_t gd[U];
    int64_t e[U], j[U];
    bool ok[U];
    flat_indices<VEC, U, FORM>(d, t, gi, gd, e, j, ok);
    pdl_wait();
    for (;;) {
        const int64_t tn = t + gridDim.x;
        V val[U];
        int64_t doff[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            doff[u] = (FORM == 3 ? (int64_t)gd[u] * s : d->dst_flat0 + e[u] * s) + j[u];
            if (ok[u]) {
                const char *base = (gi[u] & GBX_FLAT_SRC2) ? d->src2 : d->src;
                const char *p = base + (int64_t)(gi[u] & ~GBX_FLAT_SRC2) * s + j[u];
                val[u] = NC ? __ldg(reinterpret_cast<const V *>(p)) : ldv<VEC>(p);
            }
        }
        bool okc[U];
#pragma unroll
        for (int u = 0; u < U; u++) okc[u] = ok[u];
        if (tn < ntiles) flat_indices<VEC, U, FORM>(d, tn, gi, gd, e, j, ok);
#pragma unroll
        for (int u = 0; u < U; u++)
            if (okc[u]) stv<VEC>(d->dst + doff[u], val[u]);
        if (tn >= ntiles) break;
        t = tn;
    }
}

template <int VEC, int U>
__device__ __forceinline__ void copy_tile(const CopyDesc *__restrict__ d, int64_t t) {
    typedef typename VecT<VEC>::T V;
    constexpr int B = GBX_TILE / U;
    const Seg *__restrict__ segs = d->segs;
    const int cpe = d->cpe;
    const uint32_t magic = d->cpe_magic;
    const int64_t e0 = first_unit(d, t * GBX_TILE);
    const uint32_t r0 = (uint32_t)(t * GBX_TILE - e0 * cpe);
    const int64_t left = d->nchunks - t * GBX_TILE;   // chunks of this op from the tile start
    const int64_t slo = __ldg(d->tile_seg + t);
    const int64_t shi = __ldg(d->tile_seg + t + 1);

    int64_t e[U], pos[U];
    uint32_t j[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
        const uint32_t x = r0 + (uint32_t)(u * B) + threadIdx.x;
        const uint32_t el = unit_of(x, cpe, magic);
        j[u] = x - el * (uint32_t)cpe;
        e[u] = e0 + el;
        pos[u] = slo;
    }
    // branch-free search: largest segment in [slo, shi] starting at or before e[u]
    const int64_t span = shi - slo;
    int64_t step = 1;
    while (step <= span) step <<= 1;
    for (step >>= 1; step > 0; step >>= 1) {
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t cand = pos[u] + step;
            if (cand <= shi && __ldg(&segs[cand].v0) <= e[u]) pos[u] = cand;
        }
    }
    const int64_t s = d->elem_size;
    const int32_t *__restrict__ idx = d->idx;
#pragma unroll
    for (int u = 0; u < U; u++) {   // e[u] := source byte offset, pos[u] := destination byte offset
        const Seg *sg = segs + pos[u];
        const int64_t k = e[u] - __ldg(&sg->v0);
        const int64_t io = __ldg(&sg->idx_off);
        const bool ok = (int64_t)(u * B + threadIdx.x) < left;
        const int64_t sel = (io >= 0 && ok) ? (int64_t)__ldg(idx + io + k) : k;
        e[u] = __ldg(&sg->src_off) + sel * s + (int64_t)j[u] * VEC;
        pos[u] = __ldg(&sg->dst_off) + k * s + (int64_t)j[u] * VEC;
    }
    V val[U];
#pragma unroll
    for (int u = 0; u < U; u++)
        if ((int64_t)(u * B + threadIdx.x) < left) val[u] = ldv<VEC>(d->src + e[u]);
#pragma unroll
    for (int u = 0; u < U; u++)
        if ((int64_t)(u * B + threadIdx.x) < left) stv<VEC>(d->dst + pos[u], val[u]);
}

// Every op of a launch has vector width VEC and one form, FLAT 0: segment form, 1: flat form,
// 3: two-index flat form.
// GBX_COPY_OCC (threads per SM the register budget must allow; 0 = no constraint) trades
// registers for resident warps.
#ifndef GBX_COPY_OCC
#define GBX_COPY_OCC 0
#endif
template <int VEC, int U, int FLAT, typename L>
__global__ void __launch_bounds__(GBX_TILE / U, GBX_COPY_OCC ? GBX_COPY_OCC / (GBX_TILE / U) : 1)
gbx_copy_kernel(const __grid_constant__ L list) {
    pdl_trigger();
    pdl_wait();
    for (int64_t t = blockIdx.x; t < list.tiles(); t += gridDim.x) {
        int64_t lt;
        const CopyDesc *d = list.at(t, lt);
        if (FLAT == 1) copy_tile_flat<VEC, U>(d, lt);
        else if (FLAT == 3) copy_tile_flat2<VEC, U>(d, lt);
        else copy_tile<VEC, U>(d, lt);
    }
}

// Pipelined flat forms (descriptor flat = 5: gather, 7: two-index), one op per launch,
// persistent grid; launch bounds keep two full waves of threads resident (<= 32 registers).
template <int VEC, int U, int FORM, typename L>
__global__ void __launch_bounds__(GBX_TILE / U, 2 * U) gbx_copy_pipe_kernel(const __grid_constant__ L list) {
    pdl_trigger();
    copy_flat_pipelined<VEC, U, FORM, !L::single>(list.first(), list.tiles());
}

// ------------------------------------------------------------------------ bulk
// Bulk form: contiguous pieces moved through shared memory by the bulk-copy engine.  One
// thread per CTA drives a ring of GBX_BULK_STAGES buffers: a piece is loaded with
// cp.async.bulk (completion counted on the stage's mbarrier), stored back with a bulk store,
// and a stage is refilled once the store before it has read it, so several pieces per CTA
// are always in flight.  Every mbarrier wait is bounded (the main waits by the op's
// wait_limit, the drain waits by GBX_WAIT_LIMIT): a wait that gives up records status 1 for
// every op of the launch (gbx_raise), waits (bounded again) for the stage loads still in
// flight and for the stores, and leaves the kernel.
__device__ int gbx_bulk_status;

// Records a status code (1: a bounded wait gave up, 2: a piece failed its check) in the
// process-wide word and in the status word of every op of the launch: a launch that gives up
// leaves pieces of any of its ops unfinished, so each request it serves must report it.
template <typename L>
__device__ __noinline__ void gbx_raise(const L &list, int code) {
    atomicExch(&gbx_bulk_status, code);
    for (int i = 0; i < list.count(); i++) {
        int *w = list.op(i)->status;
        if (w) *reinterpret_cast<volatile int *>(w) = code;
    }
    __threadfence_system();
}

__device__ __forceinline__ bool bulk_wait(uint32_t bar, uint32_t parity, int limit = GBX_WAIT_LIMIT) {
    for (int it = 0; it < limit; it++) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

template <typename L>
__global__ void __launch_bounds__(32) gbx_bulk_kernel(const __grid_constant__ L list) {
    extern __shared__ __align__(128) unsigned char gbx_bulk_smem[];
    __shared__ __align__(8) uint64_t bar[GBX_BULK_STAGES];
    pdl_trigger();
    if (threadIdx.x != 0) return;
    constexpr int S = GBX_BULK_STAGES;
    const int64_t ntasks = list.tiles();
    const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(gbx_bulk_smem);
    const uint32_t sbar = (uint32_t)__cvta_generic_to_shared(bar);
    for (int q = 0; q < S; q++) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sbar + 8 * q) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    char *dst_of[S];
    uint32_t len_of[S], parity[S];
    bool pend[S];
#pragma unroll
    for (int q = 0; q < S; q++) {
        parity[q] = 0;
        pend[q] = false;
        dst_of[q] = nullptr;
        len_of[q] = 0;
    }
    // pieces from the last to the first: what the step before wrote last is still in L2 (2^20-row SpMV
    // halo, locality form, 53.0 -> 52.2 us; 256^3 stencil 105.8 -> 105.0)
    auto load = [&](int q, int64_t task) {
        const int64_t t = ntasks - 1 - task;
        int64_t lt;
        const CopyDesc *d = list.at(t, lt);
        const BulkTask k = d->bulk[lt];
        const uint32_t b = sbar + 8 * q, len = (uint32_t)k.len;
        // pieces were validated at init; a piece that is not a whole number of aligned 16-byte
        // units within one stage is recorded and skipped
        if (k.len <= 0 || k.len > GBX_BULK_BYTES || ((k.len | k.src | k.dst |
                                                      (int64_t)(uintptr_t)d->src | (int64_t)(uintptr_t)d->dst) & 15)) {
            gbx_raise(list, 2);
            dst_of[q] = nullptr;
            len_of[q] = 0;
            pend[q] = false;
            return;
        }
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(len) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(sbuf + q * GBX_BULK_BYTES), "l"(d->src + k.src), "r"(len), "r"(b)
                     : "memory");
        dst_of[q] = d->dst + k.dst;
        len_of[q] = len;
        pend[q] = true;
    };
    pdl_wait();
#pragma unroll
    for (int q = 0; q < S; q++) {
        const int64_t t = blockIdx.x + (int64_t)q * gridDim.x;
        if (t < ntasks) load(q, t);
    }
    const int limit = list.first()->wait_limit;
    bool failed = false;
    for (int64_t k = 0;; k++) {
        const int64_t t = blockIdx.x + k * gridDim.x;
        if (t >= ntasks) break;
        const int q = (int)(k % S);
        if (pend[q]) {
            if (!bulk_wait(sbar + 8 * q, parity[q], limit)) {
                failed = true;
                break;
            }
            parity[q] ^= 1u;
            pend[q] = false;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                         ::"l"(dst_of[q]), "r"(sbuf + q * GBX_BULK_BYTES), "r"(len_of[q])
                         : "memory");
        }
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        // refill the previous piece's stage once its store has read it
        if (k >= 1) {
            const int64_t tn = blockIdx.x + (k - 1 + S) * gridDim.x;
            if (tn < ntasks) {
                asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                load((int)((k - 1) % S), tn);
            }
        }
    }
    if (failed) {
        gbx_raise(list, 1);
        for (int q = 0; q < S; q++)
            if (pend[q]) bulk_wait(sbar + 8 * q, parity[q]);
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Allows `bytes` of dynamic shared memory to both ways of launching a kernel.
static cudaError_t smem_attr(void (*one)(const OneOp<CopyDesc>), void (*pooled)(const OpList<CopyDesc>), int bytes) {
    cudaError_t e = cudaFuncSetAttribute(one, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    return e == cudaSuccess ? cudaFuncSetAttribute(pooled, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) : e;
}

int gbx_bulk_prepare(void) {
    cudaError_t e = smem_attr(gbx_bulk_kernel<OneOp<CopyDesc>>, gbx_bulk_kernel<OpList<CopyDesc>>,
                              GBX_BULK_STAGES * GBX_BULK_BYTES);
    return e == cudaSuccess ? GBX_SUCCESS : GBX_ERR_CUDA;
}

// ----------------------------------------------------------------- scatter
// Scatter form of a two-index copy whose pairs are sorted by source: each piece is a window of
// the source.  Warp 0 is the producer: its lane 0 has the bulk-copy engine read a window's
// runs of source elements (the gaps between them are not read) and the window's source and
// destination indices into one of S shared-memory stages, completing on the stage's "full"
// mbarrier.  The other warps are consumers: they wait on "full", scatter the window's elements
// from shared memory to their destinations with 16-byte stores, and release the stage on its
// "empty" mbarrier (one arrival per consumer warp), which the producer waits on before
// refilling it.  No CTA-wide barrier is crossed after setup, so a slow warp holds back only
// its own stage.  Every wait is bounded: a consumer that gives up raises `abort`, the producer
// then stops issuing, waits (bounded) for the copies it has in flight, and every warp leaves.
template <int NT, int S, typename L>
__global__ void __launch_bounds__(NT) gbx_scatter_kernel(const __grid_constant__ L list) {
    const int64_t npieces = list.tiles();
    pdl_trigger();
    constexpr int NC = NT - 32;          // consumer threads
    constexpr int NCW = NC / 32;         // consumer warps: arrivals that release a stage
    extern __shared__ __align__(128) unsigned char gbx_scatter_smem[];
    __shared__ __align__(8) uint64_t full[S], empty[S];
    __shared__ ScatterPiece piece_s[S];
    __shared__ __align__(16) ScatterPiece next_s;   // the producer's next piece, fetched ahead
    __shared__ const CopyDesc *desc_s[S];
    __shared__ volatile int abort_flag;
    const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(gbx_scatter_smem);
    const uint32_t sfull = (uint32_t)__cvta_generic_to_shared(full);
    const uint32_t sempty = (uint32_t)__cvta_generic_to_shared(empty);
    if (threadIdx.x == 0) {
        for (int q = 0; q < S; q++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sfull + 8 * q) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sempty + 8 * q), "r"(NCW) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    __syncthreads();   // the only CTA-wide barrier
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        if (lane != 0) return;
        // ---------------------------------------------------------------- producer
        auto fetch = [&](int64_t t, const CopyDesc *&d) {   // piece t into next_s, asynchronously
            int64_t lt;
            d = list.at(t, lt);
            const char *g = reinterpret_cast<const char *>(d->scat + lt);
            const uint32_t sl = (uint32_t)__cvta_generic_to_shared(&next_s);
#pragma unroll
            for (int i = 0; i < (int)sizeof(ScatterPiece) / 16; i++)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sl + 16 * i), "l"(g + 16 * i) : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        int64_t last[S];   // last piece issued on each stage (-1: none)
#pragma unroll
        for (int q = 0; q < S; q++) last[q] = -1;
        bool stop = false;
        const CopyDesc *d = nullptr;
        const int limit = list.first()->wait_limit;
        if (blockIdx.x < npieces) fetch(blockIdx.x, d);
        pdl_wait();
        for (int64_t k = 0;; k++) {
            const int64_t t = blockIdx.x + k * gridDim.x;
            if (t >= npieces) break;
            const int q = (int)(k % S);
            if (k >= S && !bulk_wait(sempty + 8 * q, (uint32_t)((k / S - 1) & 1), limit)) {
                abort_flag = 1;
                stop = true;
                break;
            }
            if (abort_flag) {
                stop = true;
                break;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // consumers' reads before the refill
            asm volatile("cp.async.wait_all;" ::: "memory");
            ScatterPiece P = next_s;
            const CopyDesc *pd = d;
            const int64_t tn = t + gridDim.x;
            if (tn < npieces) fetch(tn, d);   // the next piece's descriptor, while this one loads
            const int64_t i0 = (P.m0 * 4) & ~(int64_t)15, i1 = ((P.m0 + P.n) * 4 + 15) & ~(int64_t)15;
            bool good = P.len > 0 && P.len <= GBX_SCAT_WIN && P.n > 0 && P.n <= GBX_SCAT_MAXN && P.m0 >= 0 &&
                        P.nrun > 0 && P.nrun <= GBX_SCAT_RUNS &&
                        ((P.src | (int64_t)(uintptr_t)pd->src | (int64_t)(uintptr_t)pd->flat_idx |
                          (int64_t)(uintptr_t)pd->flat_didx) & 15) == 0;
            uint32_t bytes = 0;
            for (int r = 0; good && r < P.nrun; r++) {
                const uint32_t o = P.run_off[r], l = P.run_len[r];
                good = ((o | l) & 15) == 0 && l > 0 && o + l <= (uint32_t)P.len;
                bytes += l;
            }
            const uint32_t fb = sfull + 8 * q;
            if (!good) {   // validated at init; recorded, and the consumers skip it
                gbx_raise(list, 2);
                P.n = 0;
                piece_s[q] = P;
                if (!L::single) desc_s[q] = pd;
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(fb) : "memory");
                continue;
            }
            piece_s[q] = P;
            if (!L::single) desc_s[q] = pd;
            const uint32_t ilen = (uint32_t)(i1 - i0), stage = sbuf + q * GBX_SCAT_STAGE;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(bytes + 2 * ilen)
                         : "memory");
            for (int r = 0; r < P.nrun; r++)
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(stage + P.run_off[r]), "l"(pd->src + P.src + P.run_off[r]),
                             "r"((uint32_t)P.run_len[r]), "r"(fb)
                             : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(stage + GBX_SCAT_WIN), "l"(reinterpret_cast<const char *>(pd->flat_idx) + i0),
                         "r"(ilen), "r"(fb)
                         : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(stage + GBX_SCAT_WIN + GBX_SCAT_IDX),
                         "l"(reinterpret_cast<const char *>(pd->flat_didx) + i0), "r"(ilen), "r"(fb)
                         : "memory");
            last[q] = k;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (stop) {   // leave no copy in flight: wait (bounded) for the last one issued on each stage
            gbx_raise(list, 1);
            for (int q = 0; q < S; q++)
                if (last[q] >= 0) bulk_wait(sfull + 8 * q, (uint32_t)((last[q] / S) & 1));
        }
        return;
    }
    // -------------------------------------------------------------------- consumers
    const int ct = threadIdx.x - 32;
    const int limit = list.first()->wait_limit;
    pdl_wait();
    for (int64_t k = 0;; k++) {
        const int64_t t = blockIdx.x + k * gridDim.x;
        if (t >= npieces) break;
        const int q = (int)(k % S);
        if (!bulk_wait(sfull + 8 * q, (uint32_t)((k / S) & 1), limit)) {
            abort_flag = 1;
            break;
        }
        const CopyDesc *d = L::single ? list.first() : desc_s[q];
        const int64_t src0 = piece_s[q].src, m0 = piece_s[q].m0;
        const int s = (int)d->elem_size, cpe = s >> 4, len = piece_s[q].len, n = piece_s[q].n;
        const unsigned char *win = gbx_scatter_smem + q * GBX_SCAT_STAGE;
        const int32_t *ps = reinterpret_cast<const int32_t *>(win + GBX_SCAT_WIN) + (m0 & 3);
        const int32_t *pdst = reinterpret_cast<const int32_t *>(win + GBX_SCAT_WIN + GBX_SCAT_IDX) + (m0 & 3);
        char *dst = d->dst;
        for (int i = ct; i < n * cpe; i += NC) {
            const int j = i / cpe, c = i - j * cpe;
            const int64_t w = (int64_t)ps[j] * s - src0 + c * 16;
            if (w < 0 || w + 16 > len) {   // validated at init; recorded and skipped
                gbx_raise(list, 2);
                continue;
            }
            const uint4 v = *reinterpret_cast<const uint4 *>(win + w);
            stv<16>(dst + (int64_t)pdst[j] * s + c * 16, v);
        }
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sempty + 8 * q) : "memory");
        if (abort_flag) break;
    }
}

// Shapes of the scatter kernel, chosen by the launch's block value: threads per CTA (one
// producer warp plus consumers), stages per CTA and CTAs per SM (each shape fills about
// 192 KB of shared memory per SM).
struct ScatShape { int nt, stages, per_sm; };
static ScatShape scatter_shape(int block) {
    if (block <= 128) return {288, 2, 4};
    if (block <= 256) return {288, 4, 2};
    if (block <= 512) return {544, 4, 2};
    return {1024, 8, 1};
}

template <typename L>
static cudaError_t scatter_launch(int block, int grid, cudaStream_t st, bool dep, const L &l) {
    const ScatShape h = scatter_shape(block);
    const size_t smem = (size_t)h.stages * GBX_SCAT_STAGE;
    if (h.stages == 2) return launch(gbx_scatter_kernel<288, 2, L>, grid, 288, smem, st, dep, l);
    if (h.nt == 288) return launch(gbx_scatter_kernel<288, 4, L>, grid, 288, smem, st, dep, l);
    if (h.nt == 544) return launch(gbx_scatter_kernel<544, 4, L>, grid, 544, smem, st, dep, l);
    return launch(gbx_scatter_kernel<1024, 8, L>, grid, 1024, smem, st, dep, l);
}

template <int NT, int S>
static cudaError_t scatter_attr() {
    return smem_attr(gbx_scatter_kernel<NT, S, OneOp<CopyDesc>>, gbx_scatter_kernel<NT, S, OpList<CopyDesc>>,
                     S * GBX_SCAT_STAGE);
}

int gbx_scatter_prepare(void) {
    cudaError_t e = scatter_attr<288, 2>();
    if (e == cudaSuccess) e = scatter_attr<288, 4>();
    if (e == cudaSuccess) e = scatter_attr<544, 4>();
    if (e == cudaSuccess) e = scatter_attr<1024, 8>();
    return e == cudaSuccess ? GBX_SUCCESS : GBX_ERR_CUDA;
}

// ------------------------------------------------------------------ stream
// Stream form of the flat copies (FORM 1: gather into a contiguous destination run; FORM 3:
// two-index gather-scatter): the same tiles of GBX_TILE chunks, but the per-element index
// arrays, the only data whose addresses are known in advance, are streamed into a ring of S
// shared-memory stages by the bulk-copy engine, so that the payload loads never wait for an
// index load from memory.  Warp 0 is the producer: its lane 0 finds the op of the CTA's next
// tile, has the bulk-copy engine copy the tile's index range (rounded out to 16-byte
// boundaries; the index arrays carry 4 entries of padding) into a stage, completing on the
// stage's "full" mbarrier, and refills a stage once the consumers have released it on its
// "empty" mbarrier.  The other warps are consumers: per tile, each thread gathers U chunks
// (all loads issued before the stores) reading the indices from shared memory.  No CTA-wide
// barrier after setup; every wait is bounded as in the scatter kernel (a consumer that gives
// up raises `abort`, the producer stops issuing and drains its copies in flight).
#define GBX_STREAM_IDX ((GBX_TILE + 8) * 4)   // bytes of one index array per stage

template <int VEC, int FORM, int NT, int S, int U, int PS, bool ONE, typename L>
__global__ void __launch_bounds__(NT, PS) gbx_stream_kernel(const __grid_constant__ L list) {
    const int64_t ntiles = list.tiles();
    pdl_trigger();
    typedef typename VecT<VEC>::T V;
    constexpr int NC = NT - 32, NCW = NC / 32;
    constexpr int STAGE = GBX_STREAM_IDX * (FORM == 3 ? 2 : 1);
    extern __shared__ __align__(128) unsigned char gbx_stream_smem[];
    __shared__ __align__(8) uint64_t full[S], empty[S];
    __shared__ const CopyDesc *desc_s[S];
    __shared__ int64_t tile_s[S], efirst_s[S], ebase_s[S];
    __shared__ volatile int abort_flag;
    const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(gbx_stream_smem);
    const uint32_t sfull = (uint32_t)__cvta_generic_to_shared(full);
    const uint32_t sempty = (uint32_t)__cvta_generic_to_shared(empty);
    if (threadIdx.x == 0) {
        for (int q = 0; q < S; q++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sfull + 8 * q) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sempty + 8 * q), "r"(NCW) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    __syncthreads();   // the only CTA-wide barrier
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int limit = list.first()->wait_limit;
    if (warp == 0) {
        if (lane != 0) return;
        // ---------------------------------------------------------------- producer
        int64_t last[S];   // last tile issued on each stage (-1: none)
#pragma unroll
        for (int q = 0; q < S; q++) last[q] = -1;
        bool stop = false;
        for (int64_t k = 0;; k++) {
            const int64_t t = blockIdx.x + k * gridDim.x;
            if (t >= ntiles) break;
            const int q = (int)(k % S);
            if (k >= S && !bulk_wait(sempty + 8 * q, (uint32_t)((k / S - 1) & 1), limit)) {
                abort_flag = 1;
                stop = true;
                break;
            }
            if (abort_flag) {
                stop = true;
                break;
            }
            int64_t lt;
            const CopyDesc *d = list.at(t, lt);
            const int64_t c0 = lt * GBX_TILE;
            const int64_t c1 = min(d->nchunks, c0 + GBX_TILE);
            const int64_t e_first = first_unit(d, c0), e_last = first_unit(d, c1 - 1);
            const int64_t e_al = e_first & ~(int64_t)3, e_end = (e_last + 4) & ~(int64_t)3;
            const uint32_t bytes = (uint32_t)((e_end - e_al) * 4);
            const uint32_t fb = sfull + 8 * q, stage = sbuf + q * STAGE;
            if (!L::single) desc_s[q] = d;
            tile_s[q] = lt;
            efirst_s[q] = e_first;
            const uintptr_t al = (uintptr_t)d->flat_idx | (FORM == 3 ? (uintptr_t)d->flat_didx : 0);
            if ((al & 15) || bytes > GBX_STREAM_IDX || c1 <= c0) {   // validated at init; recorded, skipped
                gbx_raise(list, 2);
                ebase_s[q] = -1;
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(fb) : "memory");
                continue;
            }
            ebase_s[q] = e_al;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // consumers' reads before the refill
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb),
                         "r"(bytes * (FORM == 3 ? 2u : 1u))
                         : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(stage), "l"(d->flat_idx + e_al), "r"(bytes), "r"(fb)
                         : "memory");
            if (FORM == 3)
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(stage + GBX_STREAM_IDX), "l"(d->flat_didx + e_al), "r"(bytes), "r"(fb)
                             : "memory");
            last[q] = k;
        }
        if (stop) {   // leave no copy in flight: wait (bounded) for the last one issued on each stage
            gbx_raise(list, 1);
            for (int q = 0; q < S; q++)
                if (last[q] >= 0) bulk_wait(sfull + 8 * q, (uint32_t)((last[q] / S) & 1));
        }
        return;
    }
    // -------------------------------------------------------------------- consumers
    const int ct = threadIdx.x - 32;
    pdl_wait();
    for (int64_t k = 0;; k++) {
        const int64_t t = blockIdx.x + k * gridDim.x;
        if (t >= ntiles) break;
        const int q = (int)(k % S);
        if (!bulk_wait(sfull + 8 * q, (uint32_t)((k / S) & 1), limit)) {
            abort_flag = 1;
            break;
        }
        const int64_t e_al = ebase_s[q];
        if (ONE && e_al >= 0) {
            // ONE (every op of the launch has one chunk per element, elem_size == VEC): chunk x
            // of the tile is element e0 + x, every offset a multiple of VEC
            const CopyDesc *d = L::single ? list.first() : desc_s[q];
            const int64_t e0 = efirst_s[q];
            const int left = (int)min((int64_t)GBX_TILE, d->nchunks - tile_s[q] * GBX_TILE);
            const int32_t *is = reinterpret_cast<const int32_t *>(gbx_stream_smem + q * STAGE) + (e0 - e_al);
            const int32_t *ids =
                reinterpret_cast<const int32_t *>(gbx_stream_smem + q * STAGE + GBX_STREAM_IDX) + (e0 - e_al);
            const char *src = d->src, *src2 = d->src2;
            char *dst = d->dst;
            char *dtile = dst + (FORM == 3 ? 0 : d->dst_flat0 + e0 * VEC);
            for (int base = 0; base < left; base += NC * U) {
                V val[U];
                int32_t di[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int x = base + u * NC + ct;
                    if (x < left) {
                        const uint32_t gi = (uint32_t)is[x];
                        if (FORM == 3) di[u] = ids[x];
                        const char *b = (gi & GBX_FLAT_SRC2) ? src2 : src;
                        val[u] = ldv<VEC>(b + (int64_t)(gi & ~GBX_FLAT_SRC2) * VEC);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int x = base + u * NC + ct;
                    if (x < left) stv<VEC>(FORM == 3 ? dst + (int64_t)di[u] * VEC : dtile + (int64_t)x * VEC, val[u]);
                }
            }
        } else if (!ONE && e_al >= 0) {
            const CopyDesc *d = L::single ? list.first() : desc_s[q];
            const int cpe = d->cpe;
            const uint32_t magic = d->cpe_magic;
            const int64_t s = d->elem_size, e0 = efirst_s[q], c0 = tile_s[q] * GBX_TILE;
            const int left = (int)min((int64_t)GBX_TILE, d->nchunks - c0);
            const uint32_t r0 = (uint32_t)(c0 - e0 * cpe);   // chunk of element e0 where the tile starts
            const int32_t *is = reinterpret_cast<const int32_t *>(gbx_stream_smem + q * STAGE);
            const int32_t *ids = reinterpret_cast<const int32_t *>(gbx_stream_smem + q * STAGE + GBX_STREAM_IDX);
            const char *src = d->src, *src2 = d->src2;
            char *dst = d->dst;
            for (int base = 0; base < left; base += NC * U) {
                V val[U];
                int64_t doff[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int x = base + u * NC + ct;
                    if (x < left) {
                        const uint32_t xx = r0 + (uint32_t)x;
                        const uint32_t el = unit_of(xx, cpe, magic);
                        const int64_t j = (int64_t)(xx - el * (uint32_t)cpe) * VEC;
                        const int64_t e = e0 + el;
                        const int w = (int)(e - e_al);   // < GBX_TILE + 8: inside the stage's copy
                        const uint32_t gi = (uint32_t)is[w];
                        doff[u] = (FORM == 3 ? (int64_t)ids[w] * s : d->dst_flat0 + e * s) + j;
                        const char *b = (gi & GBX_FLAT_SRC2) ? src2 : src;
                        val[u] = ldv<VEC>(b + (int64_t)(gi & ~GBX_FLAT_SRC2) * s + j);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; u++)
                    if (base + u * NC + ct < left) stv<VEC>(dst + doff[u], val[u]);
            }
        }
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sempty + 8 * q) : "memory");
        if (abort_flag) break;
    }
}

// Shapes of the stream kernel, chosen by the launch's block value: threads per CTA (one
// producer warp plus consumers), stages, chunks per consumer thread per pass, CTAs per SM
// (the launch bounds hold the registers to what that many CTAs need; shared memory per SM
// is at most 4 x 4 x 8,256 = 132 KB).
// Block 128 selects the narrow shape, 160 threads x 4 stages (3 for two-index copies) x 8
// CTAs per SM with 8 chunks per thread in flight: offered only where every op has one chunk
// per element (ONE) of at most 8 bytes, whose kernel fits its 48 registers; the tuner never
// gives it other ops.
struct StreamShape { int nt, stages, u, per_sm; };
static StreamShape stream_shape(int block) {
    if (block <= 128) return {160, 4, 8, 8};
    if (block <= 256) return {288, 4, 4, 4};
    return {544, 6, 2, 2};
}

template <int VEC, int FORM, bool ONE, typename L>
static cudaError_t stream_launch_v(int block, int grid, cudaStream_t st, bool dep, const L &l) {
    const StreamShape h = stream_shape(block);
    constexpr int SC = FORM == 3 ? 3 : 4;   // stages of the narrow shape
    const size_t smem = (size_t)(h.nt == 160 ? SC : h.stages) * GBX_STREAM_IDX * (FORM == 3 ? 2 : 1);
    if (h.nt == 160) {
        if constexpr (ONE && VEC <= 8)
            return launch(gbx_stream_kernel<VEC, FORM, 160, SC, 8, 8, ONE, L>, grid, 160, smem, st, dep, l);
        else
            return cudaErrorInvalidValue;   // never chosen: only one-chunk ops of vectors up to 8 bytes
    }
    if (h.nt == 288) return launch(gbx_stream_kernel<VEC, FORM, 288, 4, 4, 4, ONE, L>, grid, 288, smem, st, dep, l);
    return launch(gbx_stream_kernel<VEC, FORM, 544, 6, 2, 2, ONE, L>, grid, 544, smem, st, dep, l);
}

template <int VEC, typename L>
static cudaError_t stream_launch_f(int flat, int block, int grid, cudaStream_t st, bool dep, const L &l) {
    switch (flat) {
        case 10: return stream_launch_v<VEC, 1, false>(block, grid, st, dep, l);
        case 11: return stream_launch_v<VEC, 3, false>(block, grid, st, dep, l);
        case 12: return stream_launch_v<VEC, 1, true>(block, grid, st, dep, l);
        default: return stream_launch_v<VEC, 3, true>(block, grid, st, dep, l);
    }
}

// flat 10 / 11: the stream forms; 12 / 13: the same when every op of the launch has one chunk
// per element (the kernel then skips the element / chunk split)
template <typename L>
static cudaError_t stream_launch(int vec, int flat, int block, int grid, cudaStream_t st, bool dep, const L &l) {
    switch (vec) {
        case 16: return stream_launch_f<16>(flat, block, grid, st, dep, l);
        case 8: return stream_launch_f<8>(flat, block, grid, st, dep, l);
        case 4: return stream_launch_f<4>(flat, block, grid, st, dep, l);
        default: return cudaErrorInvalidValue;   // the stream form is offered for vectors of 4..16 bytes
    }
}

template <int VEC, int FORM, int NT, int S, int U, int PS, bool ONE>
static cudaError_t stream_attr_k() {
    return smem_attr(gbx_stream_kernel<VEC, FORM, NT, S, U, PS, ONE, OneOp<CopyDesc>>,
                     gbx_stream_kernel<VEC, FORM, NT, S, U, PS, ONE, OpList<CopyDesc>>,
                     S * GBX_STREAM_IDX * (FORM == 3 ? 2 : 1));
}

template <int VEC, int FORM, bool ONE>
static cudaError_t stream_attr_o() {
    cudaError_t e = stream_attr_k<VEC, FORM, 288, 4, 4, 4, ONE>();
    if (e == cudaSuccess) e = stream_attr_k<VEC, FORM, 544, 6, 2, 2, ONE>();
    if constexpr (ONE && VEC <= 8)
        if (e == cudaSuccess) e = stream_attr_k<VEC, FORM, 160, FORM == 3 ? 3 : 4, 8, 8, ONE>();
    return e;
}

template <int VEC, int FORM>
static cudaError_t stream_attr_v() {
    cudaError_t e = stream_attr_o<VEC, FORM, false>();
    return e == cudaSuccess ? stream_attr_o<VEC, FORM, true>() : e;
}

int gbx_stream_prepare(void) {
    cudaError_t e = stream_attr_v<16, 1>();
    if (e == cudaSuccess) e = stream_attr_v<16, 3>();
    if (e == cudaSuccess) e = stream_attr_v<8, 1>();
    if (e == cudaSuccess) e = stream_attr_v<8, 3>();
    if (e == cudaSuccess) e = stream_attr_v<4, 1>();
    if (e == cudaSuccess) e = stream_attr_v<4, 3>();
    return e == cudaSuccess ? GBX_SUCCESS : GBX_ERR_CUDA;
}

// ------------------------------------------------------------ async gather
// Async form of the flat gather of 16-byte chunks (destinations one contiguous run): every warp
// gathers its chunks straight into shared memory (cp.async, one chunk per lane and step) and
// has the bulk-copy engine write them out as one contiguous store, through a ring of S stages
// of its own.  A unit is 32 * K consecutive chunks of the op's tiles; a warp keeps the loads of
// S - 2 units in flight while the store of the unit before them drains, and loads a unit's
// indices one unit ahead.  The gathers hold no registers and the stores no load / store slots,
// so the bytes in flight per SM are set by the ring (192 KB) and not by the register file
// (32 KB with one chunk per thread at full occupancy).  A warp waits only for copies it has
// issued itself (cp.async.wait_group), never on a flag.  Bound by HBM: 512^3 stencil halo (64-byte
// points, 3.57 GB of whole 128-byte lines) 549 us = 6.5 TB/s of line traffic; flat form 543-589 us,
// stream form 573, register-pipelined form 590-617.  More bytes in flight are not better: of the
// shapes the one of 48 KB per CTA takes 549 us, those of 64 KB 574 and 597 at the 3 CTAs per SM that they
// are launched with (548 and 550 at 2.4 and 2).  They stay for smaller exchanges, where they are level with it
// or ahead (256^3 halo 70 us in all three, its locality form 109 and 110, 113 with 48 KB).
// Chunks of 4 and 8 bytes gain nothing (2^20-row SpMV halo
// 45 us, stream form 38: a request per line and element bounds them, not bytes in flight).
// Destinations in host memory (bulk_dst = 0) are stored by the lanes.
template <int K, int S, int NW, int PS, typename L>
__global__ void __launch_bounds__(NW * 32, PS) gbx_agather_kernel(const __grid_constant__ L list) {
    constexpr int D = S - 2;                      // units of loads in flight
    constexpr int UNIT = 32 * K, SUB = GBX_TILE / UNIT;
    extern __shared__ __align__(128) unsigned char gbx_agather_smem[];
    pdl_trigger();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint4 *ring = reinterpret_cast<uint4 *>(gbx_agather_smem) + warp * S * UNIT;
    const uint32_t sring = (uint32_t)__cvta_generic_to_shared(ring);
    const int64_t stride = (int64_t)gridDim.x * NW, nunits = list.tiles() * SUB;
    int64_t u = (int64_t)blockIdx.x * NW + warp;  // next unit to load
    int64_t us = u;                               // next unit to store

    Cursor<L> loads(list), stores(list);
    // unit x: its op, its first chunk c0, the element e0 that holds it and the chunk r0 in it
    auto locate = [&](int64_t x, int64_t &c0, int64_t &e0, uint32_t &r0) -> const CopyDesc & {
        int64_t lt;
        const CopyDesc &d = loads.at(x / SUB, lt);
        c0 = lt * GBX_TILE + (x % SUB) * UNIT;
        e0 = first_unit(&d, c0);
        r0 = (uint32_t)(c0 - e0 * d.cpe);
        return d;
    };
    uint32_t gi[K];   // indices of the next unit's chunks (0 past the op's end)
    auto indices = [&](int64_t x) {
        int64_t c0, e0;
        uint32_t r0;
        const CopyDesc &d = locate(x, c0, e0, r0);
        const int64_t left = d.nchunks - c0;
        const int32_t *g = d.flat_idx + e0;
#pragma unroll
        for (int k = 0; k < K; k++) {
            const int x0 = k * 32 + lane;
            gi[k] = x0 < left ? (uint32_t)__ldg(g + unit_of(r0 + (uint32_t)x0, d.cpe, d.cpe_magic)) : 0u;
        }
    };
    if (u < nunits) indices(u);
    pdl_wait();
    for (int i = 0; us < nunits; i++) {
        if (u < nunits) {
            const int q = i % S;
            if (i >= S) {   // the last store from this stage has read it
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                __syncwarp();
            }
            int64_t c0, e0;
            uint32_t r0;
            const CopyDesc &d = locate(u, c0, e0, r0);
            const int64_t left = d.nchunks - c0, s = d.elem_size;
#pragma unroll
            for (int k = 0; k < K; k++) {
                const int x0 = k * 32 + lane;
                if (x0 < left) {
                    const uint32_t xx = r0 + (uint32_t)x0;
                    const uint32_t j = xx - unit_of(xx, d.cpe, d.cpe_magic) * (uint32_t)d.cpe;
                    const char *b = (gi[k] & GBX_FLAT_SRC2) ? d.src2 : d.src;
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                                 ::"r"(sring + (uint32_t)((q * UNIT + x0) * 16)),
                                 "l"(b + (int64_t)(gi[k] & ~GBX_FLAT_SRC2) * s + (int64_t)(j * 16))
                                 : "memory");
                }
            }
            u += stride;
            if (u < nunits) indices(u);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (i < D) continue;
        asm volatile("cp.async.wait_group %0;" ::"n"(D) : "memory");   // unit us has landed
        const int q = (i - D) % S;
        int64_t lt;
        const CopyDesc &d = stores.at(us / SUB, lt);
        const int64_t c0 = lt * GBX_TILE + (us % SUB) * UNIT;
        const int n = (int)min((int64_t)UNIT, d.nchunks - c0);   // (0 or less: past the op's last chunk)
        us += stride;
        if (n > 0) {
            char *out = d.dst + d.dst_flat0 + c0 * 16;
            if (d.bulk_dst) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0)
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                                 ::"l"(out), "r"(sring + (uint32_t)(q * UNIT * 16)), "r"((uint32_t)(n * 16))
                                 : "memory");
            } else {
                for (int x = lane; x < n; x += 32) stv<16>(out + (int64_t)x * 16, ring[q * UNIT + x]);   // its own chunks
            }
        }
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");   // one store group per unit
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Shapes of the async gather, chosen by the launch's block value: steps per unit, stages, warps
// per CTA, CTAs per SM (each fills 192 KB of shared memory per SM).
template <typename L>
static cudaError_t agather_launch(int block, int grid, cudaStream_t st, bool dep, const L &l) {
    if (block <= 128) return launch(gbx_agather_kernel<8, 4, 4, 3, L>, grid, 128, 65536, st, dep, l);
    if (block <= 256) return launch(gbx_agather_kernel<4, 6, 4, 4, L>, grid, 128, 49152, st, dep, l);
    return launch(gbx_agather_kernel<4, 4, 8, 3, L>, grid, 256, 65536, st, dep, l);
}

static int agather_per_sm(int block) { return block <= 128 || block > 256 ? 3 : 4; }

template <int K, int S, int NW, int PS>
static cudaError_t agather_attr() {
    return smem_attr(gbx_agather_kernel<K, S, NW, PS, OneOp<CopyDesc>>, gbx_agather_kernel<K, S, NW, PS, OpList<CopyDesc>>,
                     NW * S * K * 512);
}

int gbx_agather_prepare(void) {
    cudaError_t e = agather_attr<8, 4, 4, 3>();
    if (e == cudaSuccess) e = agather_attr<4, 6, 4, 4>();
    if (e == cudaSuccess) e = agather_attr<4, 4, 8, 3>();
    return e == cudaSuccess ? GBX_SUCCESS : GBX_ERR_CUDA;
}

// ------------------------------------------------------------------ window
// Window form of a flat gather of elements of VEC bytes (tables: WinPiece).  Warp 0 is the
// producer: per piece it has the bulk-copy engine read the source window and the piece's tables
// into one of S shared-memory stages, completing on the stage's "full" mbarrier.  The consumer
// warps pick the elements out of the window and store them: 32 consecutive slots of a piece per
// warp and step, whose destinations are runs of consecutive elements.  The element index costs 2
// bytes and its share of a run instead of 4, every source line is read whole by the copy
// engine, and no load of a single element goes through L1.  That is what bounds the other forms
// here: a request to L2 and an L1 line for every scattered element (2^20-row SpMV halo, 10.8 M
// elements of 8 bytes: L1-to-L2 requests 55 %, DRAM 27 % of peak).  Start and wait of the halo took 39.0 us
// in the best of them and takes 30.3 (fp32, repeated on the same buffers: 30.9 -> 18.6), its locality form
// 63.5 -> 52.3, a start of 16 uneven patterns 115 -> 80.  Now the requests of short destination runs weigh
// most, then the producer's work per piece.  Waits bounded as in the stream form.
// Sources off a 16-byte boundary (SHIFT): a window lies as far from a boundary in its stage as in the
// source, so that the engine reads all of it but the partial 16-byte units at its ends, which the
// producer's lanes copy.  2^20-row halo from such a source: 33 us fp64 and 28 fp32, 99 and 89 where
// the lanes copy whole windows, as they do without SHIFT, and from host memory.  A kernel of its own, as the few
// instructions more per piece cost the others time (fp32 halo in locality form 37.0 -> 37.7 us).
#define GBX_WIN_LEAD(shift) ((shift) ? 16 : 0)   // room before a window
#define GBX_WIN_TABLES (GBX_WIN_N * 2 + GBX_WIN_N / 32 * 8 + GBX_WIN_RUNS * 4)

template <int VEC, int WE, int NT, int S, int PS, bool SHIFT, typename L>
__global__ void __launch_bounds__(NT, PS) gbx_window_kernel(const __grid_constant__ L list) {
    typedef typename VecT<VEC>::T V;
    constexpr int NCW = NT / 32 - 1, U = 4;
    constexpr int WB = WE * VEC, STAGE = WB + GBX_WIN_LEAD(SHIFT) + GBX_WIN_TABLES;
    constexpr int OFF_IDX = WB + GBX_WIN_LEAD(SHIFT), OFF_GRP = OFF_IDX + GBX_WIN_N * 2, OFF_RUN = OFF_GRP + GBX_WIN_N / 32 * 8;
    extern __shared__ __align__(128) unsigned char gbx_window_smem[];
    __shared__ __align__(8) uint64_t full[S], empty[S];
    __shared__ char *dst_s[S];
    __shared__ int n_s[S], lead_s[SHIFT ? S : 1];
    __shared__ volatile int abort_flag;
    pdl_trigger();
    const int64_t npieces = list.tiles();
    const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(gbx_window_smem);
    const uint32_t sfull = (uint32_t)__cvta_generic_to_shared(full);
    const uint32_t sempty = (uint32_t)__cvta_generic_to_shared(empty);
    if (threadIdx.x == 0) {
        for (int q = 0; q < S; q++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sfull + 8 * q) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sempty + 8 * q), "r"(NCW) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    __syncthreads();   // the only CTA-wide barrier
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int limit = list.first()->wait_limit;
    if (warp == 0) {
        // ---------------------------------------------------------------- producer (whole warp)
        int64_t last[S];
#pragma unroll
        for (int q = 0; q < S; q++) last[q] = -1;
        bool stop = false;
        int64_t lt = 0;
        const CopyDesc *d = list.first();
        WinPiece P = {};
        if (blockIdx.x < npieces) {
            d = list.at(blockIdx.x, lt);
            P = d->win[lt];
        }
        pdl_wait();
        for (int64_t k = 0;; k++) {
            const int64_t t = blockIdx.x + k * gridDim.x;
            if (t >= npieces) break;
            const int q = (int)(k % S);
            bool go = k < S || bulk_wait(sempty + 8 * q, (uint32_t)((k / S - 1) & 1), limit);
            go = __all_sync(0xffffffffu, go && !abort_flag);
            if (!go) {
                abort_flag = 1;
                stop = true;
                break;
            }
            const uint32_t fb = sfull + 8 * q, stage = sbuf + q * STAGE;
            const char *src = (P.buf ? d->src2 : d->src) + P.src;
            const bool good = P.n > 0 && P.n <= GBX_WIN_N && P.nrun > 0 && P.nrun <= GBX_WIN_RUNS && P.bytes > 0 && P.bytes <= WB;
            // window byte o lies at lead + o of the stage; the engine reads [head, head + b16), the lanes the rest
            const int wl = P.buf ? d->win_lead2 : d->win_lead;
            const uint32_t lead = SHIFT && wl > 0 ? (uint32_t)wl : 0u, head = SHIFT ? min((uint32_t)P.bytes, (16u - lead) & 15u) : 0u;
            const uint32_t b16 = (SHIFT ? wl >= 0 : wl == 0) ? ((uint32_t)P.bytes - head) & ~15u : 0u;
            unsigned char *win = gbx_window_smem + q * STAGE + lead;
            if (good) {
                if (SHIFT && lane * VEC < head) *reinterpret_cast<V *>(win + lane * VEC) = ldv<VEC>(src + lane * VEC);
                for (uint32_t o = head + b16 + lane * VEC; o < (uint32_t)P.bytes; o += 32 * VEC)
                    *reinterpret_cast<V *>(win + o) = ldv<VEC>(src + o);
            }
            __syncwarp();
            if (lane == 0) {
                dst_s[q] = d->dst + d->dst_flat0;
                n_s[q] = good ? P.n : 0;
                if (SHIFT) lead_s[q] = (int)lead;
                if (!good) {   // validated at init; recorded, skipped
                    gbx_raise(list, 2);
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(fb) : "memory");
                } else {
                    const int64_t slot = lt * GBX_WIN_N;
                    const uint32_t ib = ((uint32_t)P.n * 2 + 15) & ~15u, gb = (((uint32_t)P.n + 31) / 32 * 8 + 15) & ~15u,
                                   rb = ((uint32_t)P.nrun * 4 + 15) & ~15u;
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // consumers' reads before the refill
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb),
                                 "r"(b16 + ib + gb + rb)
                                 : "memory");
                    if (b16)
                        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                     ::"r"(stage + lead + head), "l"(src + head), "r"(b16), "r"(fb) : "memory");
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(stage + OFF_IDX), "l"(d->win_idx + slot), "r"(ib), "r"(fb) : "memory");
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(stage + OFF_GRP), "l"(d->win_grp + slot / 32), "r"(gb), "r"(fb) : "memory");
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(stage + OFF_RUN), "l"(d->win_run + lt * GBX_WIN_RUNS), "r"(rb), "r"(fb) : "memory");
                    last[q] = k;
                }
            }
            const int64_t tn = t + gridDim.x;
            if (tn < npieces) {
                d = list.at(tn, lt);
                P = d->win[lt];
            }
        }
        if (stop && lane == 0) {   // leave no copy in flight: wait (bounded) for the last one on each stage
            gbx_raise(list, 1);
            for (int q = 0; q < S; q++)
                if (last[q] >= 0) bulk_wait(sfull + 8 * q, (uint32_t)((last[q] / S) & 1));
        }
        return;
    }
    // -------------------------------------------------------------------- consumers
    const uint32_t upto = 0xffffffffu >> (31 - lane);   // this lane and the ones before it
    pdl_wait();
    for (int64_t k = 0;; k++) {
        const int64_t t = blockIdx.x + k * gridDim.x;
        if (t >= npieces) break;
        const int q = (int)(k % S);
        if (!bulk_wait(sfull + 8 * q, (uint32_t)((k / S) & 1), limit)) {
            abort_flag = 1;
            break;
        }
        const unsigned char *stage = gbx_window_smem + q * STAGE;
        const V *win = reinterpret_cast<const V *>(stage + (SHIFT ? lead_s[q] : 0));
        const uint16_t *idx = reinterpret_cast<const uint16_t *>(stage + OFF_IDX);
        const uint2 *grp = reinterpret_cast<const uint2 *>(stage + OFF_GRP);
        const int32_t *run = reinterpret_cast<const int32_t *>(stage + OFF_RUN);
        const int n = n_s[q], ng = (n + 31) >> 5;
        char *dst = dst_s[q];
        for (int g0 = warp - 1; g0 < ng; g0 += NCW * U) {
            V val[U];
            int32_t e[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int g = g0 + u * NCW, x = g * 32 + lane;
                if (x < n) {
                    const uint2 m = grp[g];
                    e[u] = run[m.y + __popc(m.x & upto) - 1] + x;
                    val[u] = win[idx[x]];
                }
            }
#pragma unroll
            for (int u = 0; u < U; u++)
                if ((g0 + u * NCW) * 32 + lane < n) stv<VEC>(dst + (int64_t)e[u] * VEC, val[u]);
        }
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sempty + 8 * q) : "memory");
        if (abort_flag) break;
    }
}

// Shapes of the window kernel, chosen by the launch's block value: threads per CTA, stages, CTAs
// per SM (about 200 KB of shared memory per SM), by the bytes of a window.
template <int WB> struct WinShape;
template <> struct WinShape<4096> { static constexpr int S0 = 2, P0 = 8, S1 = 3, P1 = 5, S2 = 6, P2 = 2; };
template <> struct WinShape<8192> { static constexpr int S0 = 2, P0 = 6, S1 = 3, P1 = 4, S2 = 6, P2 = 2; };
template <> struct WinShape<16384> { static constexpr int S0 = 2, P0 = 4, S1 = 2, P1 = 4, S2 = 4, P2 = 2; };

template <int VEC, int WE, bool SHIFT, typename L>
static cudaError_t window_launch_v(int block, int grid, cudaStream_t st, bool dep, const L &l) {
    typedef WinShape<VEC * WE> H;
    constexpr size_t B = VEC * WE + GBX_WIN_LEAD(SHIFT) + GBX_WIN_TABLES;
    if (block <= 128) return launch(gbx_window_kernel<VEC, WE, 160, H::S0, H::P0, SHIFT, L>, grid, 160, H::S0 * B, st, dep, l);
    if (block <= 256) return launch(gbx_window_kernel<VEC, WE, 288, H::S1, H::P1, SHIFT, L>, grid, 288, H::S1 * B, st, dep, l);
    return launch(gbx_window_kernel<VEC, WE, 544, H::S2, H::P2, SHIFT, L>, grid, 544, H::S2 * B, st, dep, l);
}

template <int WB> static int win_per_sm(int block) {
    return block <= 128 ? WinShape<WB>::P0 : block <= 256 ? WinShape<WB>::P1 : WinShape<WB>::P2;
}
static int window_per_sm(int vec, int wide, int block) {
    const int wb = vec * (wide ? 2048 : 1024);
    return wb == 4096 ? win_per_sm<4096>(block) : wb == 8192 ? win_per_sm<8192>(block) : win_per_sm<16384>(block);
}

template <int VEC, int WE, typename L>
static cudaError_t window_launch_s(int shift, int block, int grid, cudaStream_t st, bool dep, const L &l) {
    return shift ? window_launch_v<VEC, WE, true>(block, grid, st, dep, l) : window_launch_v<VEC, WE, false>(block, grid, st, dep, l);
}

// code: the launch code (15, + 32 for the wide windows, + 128 for sources off a 16-byte boundary)
template <typename L>
static cudaError_t window_launch(int vec, int code, int block, int grid, cudaStream_t st, bool dep, const L &l) {
    const int wide = code >> 5 & 1, shift = code >> 7 & 1;
    if (vec == 8)
        return wide ? window_launch_s<8, 2048>(shift, block, grid, st, dep, l) : window_launch_s<8, 1024>(shift, block, grid, st, dep, l);
    if (vec == 4)
        return wide ? window_launch_s<4, 2048>(shift, block, grid, st, dep, l) : window_launch_s<4, 1024>(shift, block, grid, st, dep, l);
    return cudaErrorInvalidValue;   // offered for elements of 4 and 8 bytes
}

template <int VEC, int WE, int NT, int S, int PS, bool SHIFT>
static cudaError_t window_attr_k() {
    return smem_attr(gbx_window_kernel<VEC, WE, NT, S, PS, SHIFT, OneOp<CopyDesc>>,
                     gbx_window_kernel<VEC, WE, NT, S, PS, SHIFT, OpList<CopyDesc>>,
                     S * (VEC * WE + GBX_WIN_LEAD(SHIFT) + GBX_WIN_TABLES));
}
template <int VEC, int WE, bool SHIFT>
static cudaError_t window_attr_s() {
    typedef WinShape<VEC * WE> H;
    cudaError_t e = window_attr_k<VEC, WE, 160, H::S0, H::P0, SHIFT>();
    if (e == cudaSuccess) e = window_attr_k<VEC, WE, 288, H::S1, H::P1, SHIFT>();
    if (e == cudaSuccess) e = window_attr_k<VEC, WE, 544, H::S2, H::P2, SHIFT>();
    return e;
}
template <int VEC, int WE>
static cudaError_t window_attr() {
    const cudaError_t e = window_attr_s<VEC, WE, false>();
    return e == cudaSuccess ? window_attr_s<VEC, WE, true>() : e;
}

int gbx_window_prepare(void) {
    cudaError_t e = window_attr<8, 1024>();
    if (e == cudaSuccess) e = window_attr<8, 2048>();
    if (e == cudaSuccess) e = window_attr<4, 1024>();
    if (e == cudaSuccess) e = window_attr<4, 2048>();
    return e == cudaSuccess ? GBX_SUCCESS : GBX_ERR_CUDA;
}

int gbx_bulk_status_take(int *status) {
    int zero = 0;
    GBX_CUDA_TRY(cudaMemcpyFromSymbol(status, gbx_bulk_status, sizeof(int)));
    GBX_CUDA_TRY(cudaMemcpyToSymbol(gbx_bulk_status, &zero, sizeof(int)));
    return GBX_SUCCESS;
}

// ------------------------------------------------------------------------ fold
// Payload vectors: the CUDA vector type of `VEC` bytes of T, added component-wise with
// IEEE round-to-nearest adds (never contracted, never reassociated).
template <typename T, int VEC> struct PackT;
template <> struct PackT<double, 16> { typedef double2 T; };
template <> struct PackT<double, 8> { typedef double T; };
template <> struct PackT<float, 16> { typedef float4 T; };
template <> struct PackT<float, 8> { typedef float2 T; };
template <> struct PackT<float, 4> { typedef float T; };

__device__ __forceinline__ double2 padd(double2 a, double2 b) { return make_double2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y)); }
__device__ __forceinline__ double padd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float4 padd(float4 a, float4 b) {
    return make_float4(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z), __fadd_rn(a.w, b.w));
}
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y)); }
__device__ __forceinline__ float padd(float a, float b) { return __fadd_rn(a, b); }

template <typename P>
__device__ __forceinline__ P pload(const char *p) { return *reinterpret_cast<const P *>(p); }   // (as ldv)

template <typename T, int VEC, int U>
__device__ __forceinline__ void fold_tile(const FoldDesc *__restrict__ d, int64_t t) {
    typedef typename PackT<T, VEC>::T PK;
    constexpr int B = GBX_TILE / U;
    const int cpe = d->cpe;
    const uint32_t magic = d->cpe_magic;
    const int64_t e0 = first_unit(d, t * GBX_TILE);
    const uint32_t r0 = (uint32_t)(t * GBX_TILE - e0 * cpe);
    const int64_t left = d->nchunks - t * GBX_TILE;
    const int64_t *__restrict__ terms = d->terms;
    // one 16-byte record per row: most rows have a single term, which it holds inline
    int64_t oa[U], ob[U];
    uint32_t jv[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
        const uint32_t x = r0 + (uint32_t)(u * B) + threadIdx.x;
        const uint32_t el = unit_of(x, cpe, magic);
        jv[u] = (x - el * (uint32_t)cpe) * VEC;
        const bool ok = (int64_t)(u * B + threadIdx.x) < left;
        if (ok) {
            const longlong2 r = __ldg(d->rec + e0 + el);
            oa[u] = r.x;
            ob[u] = r.y;
        } else {
            oa[u] = 0;
            ob[u] = 0;
        }
    }
    PK res[U];
    bool multi = false;
#pragma unroll
    for (int u = 0; u < U; u++) {
        if ((uint64_t)oa[u] & GBX_ROW_SINGLE) {
            const uint64_t w = (uint64_t)ob[u];
            res[u] = pload<PK>(((w & GBX_TERM_BUFB) ? d->bufB : d->bufA) + (int64_t)(w & GBX_TERM_MASK) + jv[u]);
        } else if ((int64_t)(u * B + threadIdx.x) < left) {
            multi = true;
        }
    }
    if (multi) {
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (((uint64_t)oa[u] & GBX_ROW_SINGLE) || (int64_t)(u * B + threadIdx.x) >= left) continue;
            const int64_t b = (int64_t)((uint64_t)ob[u] >> GBX_ROW_CNT_BITS);
            const int64_t n = (int64_t)((uint64_t)ob[u] & ((1ull << GBX_ROW_CNT_BITS) - 1));
            PK grp, tot;
            bool has = false;
            for (int64_t m = 0; m < n; m++) {
                const uint64_t w = (uint64_t)__ldg(terms + b + m);
                const PK x = pload<PK>(((w & GBX_TERM_BUFB) ? d->bufB : d->bufA) + (int64_t)(w & GBX_TERM_MASK) + jv[u]);
                if (m == 0) {
                    grp = x;
                } else if (w & GBX_TERM_GROUP) {
                    tot = has ? padd(tot, grp) : grp;
                    has = true;
                    grp = x;
                } else {
                    grp = padd(grp, x);
                }
            }
            res[u] = has ? padd(tot, grp) : grp;
        }
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
        if ((int64_t)(u * B + threadIdx.x) >= left) continue;
        PK *o = reinterpret_cast<PK *>(d->out + (oa[u] & (int64_t)~GBX_ROW_SINGLE) + jv[u]);
        PK r = res[u];
        if (d->accumulate) r = padd(*o, r);
        *o = r;
    }
}

// Stream form of the fold (the reverse exchange's sums): the fold's tiles, with each tile's
// row records and its rows' term lists (both contiguous ranges, the terms rounded out to
// 16-byte boundaries; the term arrays carry 2 entries of padding) copied into a ring of S
// shared-memory stages by the bulk-copy engine from one producer lane, completing on the
// stage's "full" mbarrier.  Each consumer thread then holds one chunk of one row: it reads
// the record and terms from shared memory and issues up to GBX_SFOLD_K gradient loads of
// the row at once before adding them in the row's fixed order, so a row costs one memory
// latency instead of two per term.  A tile whose terms do not fit a stage reads them from
// global memory.  Waits bounded as in the stream copy.
#define GBX_SFOLD_REC ((GBX_TILE + 2) * 16)   // bytes of records per stage
#define GBX_SFOLD_TERMS 2048                   // term entries per stage
#define GBX_SFOLD_STAGE (GBX_SFOLD_REC + GBX_SFOLD_TERMS * 8)
// gradient loads in flight per thread: 8 of 4 or 8 bytes, 4 of 16 bytes (the registers of
// 2 CTAs of 544 threads per SM)

template <typename T, int VEC, int NT, int S, int PS, typename L>
__global__ void __launch_bounds__(NT, PS) gbx_sfold_kernel(const __grid_constant__ L list) {
    const int64_t ntiles = list.tiles();
    pdl_trigger();
    typedef typename PackT<T, VEC>::T PK;
    constexpr int NC = NT - 32, NCW = NC / 32;
    constexpr int GBX_SFOLD_K = VEC == 16 ? 4 : 8;
    extern __shared__ __align__(128) unsigned char gbx_sfold_smem[];
    __shared__ __align__(8) uint64_t full[S], empty[S];
    __shared__ const FoldDesc *desc_s[S];
    __shared__ int64_t tile_s[S], rfirst_s[S], tbase_s[S];
    __shared__ volatile int abort_flag;
    const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(gbx_sfold_smem);
    const uint32_t sfull = (uint32_t)__cvta_generic_to_shared(full);
    const uint32_t sempty = (uint32_t)__cvta_generic_to_shared(empty);
    if (threadIdx.x == 0) {
        for (int q = 0; q < S; q++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sfull + 8 * q) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sempty + 8 * q), "r"(NCW) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    __syncthreads();   // the only CTA-wide barrier
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int limit = list.first()->wait_limit;
    if (warp == 0) {
        if (lane != 0) return;
        // ---------------------------------------------------------------- producer
        int64_t last[S];
#pragma unroll
        for (int q = 0; q < S; q++) last[q] = -1;
        bool stop = false;
        for (int64_t k = 0;; k++) {
            const int64_t t = blockIdx.x + k * gridDim.x;
            if (t >= ntiles) break;
            const int q = (int)(k % S);
            if (k >= S && !bulk_wait(sempty + 8 * q, (uint32_t)((k / S - 1) & 1), limit)) {
                abort_flag = 1;
                stop = true;
                break;
            }
            if (abort_flag) {
                stop = true;
                break;
            }
            int64_t lt;
            const FoldDesc *d = list.at(t, lt);
            const int64_t c0 = lt * GBX_TILE, c1 = min(d->nchunks, c0 + GBX_TILE);
            const int64_t r_first = first_unit(d, c0), r_last = first_unit(d, c1 - 1);
            const uint32_t rbytes = (uint32_t)((r_last - r_first + 1) * 16);
            const int64_t tb = __ldg(d->row_ptr + r_first), te = __ldg(d->row_ptr + r_last + 1);
            const int64_t tb_al = tb & ~(int64_t)1, te_al = (te + 1) & ~(int64_t)1;
            const bool inl = (te_al - tb_al) <= GBX_SFOLD_TERMS;
            const uint32_t tbytes = inl ? (uint32_t)((te_al - tb_al) * 8) : 0u;
            const uint32_t fb = sfull + 8 * q, stage = sbuf + q * GBX_SFOLD_STAGE;
            if (!L::single) desc_s[q] = d;
            tile_s[q] = lt;
            rfirst_s[q] = r_first;
            tbase_s[q] = inl ? tb_al : -1;
            const uintptr_t al = (uintptr_t)d->rec | (uintptr_t)d->terms;
            if ((al & 15) || rbytes > GBX_SFOLD_REC || c1 <= c0) {   // validated at init; recorded, skipped
                gbx_raise(list, 2);
                rfirst_s[q] = -1;
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(fb) : "memory");
                continue;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(rbytes + tbytes)
                         : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(stage), "l"(d->rec + r_first), "r"(rbytes), "r"(fb)
                         : "memory");
            if (tbytes)
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(stage + GBX_SFOLD_REC), "l"(d->terms + tb_al), "r"(tbytes), "r"(fb)
                             : "memory");
            last[q] = k;
        }
        if (stop) {
            gbx_raise(list, 1);
            for (int q = 0; q < S; q++)
                if (last[q] >= 0) bulk_wait(sfull + 8 * q, (uint32_t)((last[q] / S) & 1));
        }
        return;
    }
    // -------------------------------------------------------------------- consumers
    const int ct = threadIdx.x - 32;
    pdl_wait();
    for (int64_t k = 0;; k++) {
        const int64_t t = blockIdx.x + k * gridDim.x;
        if (t >= ntiles) break;
        const int q = (int)(k % S);
        if (!bulk_wait(sfull + 8 * q, (uint32_t)((k / S) & 1), limit)) {
            abort_flag = 1;
            break;
        }
        const int64_t r_first = rfirst_s[q];
        if (r_first >= 0) {
            const FoldDesc *d = L::single ? list.first() : desc_s[q];
            const int cpe = d->cpe;
            const uint32_t magic = d->cpe_magic;
            const int64_t c0 = tile_s[q] * GBX_TILE, tb_al = tbase_s[q];
            const int left = (int)min((int64_t)GBX_TILE, d->nchunks - c0);
            const uint32_t r0 = (uint32_t)(c0 - r_first * cpe);
            const longlong2 *rs = reinterpret_cast<const longlong2 *>(gbx_sfold_smem + q * GBX_SFOLD_STAGE);
            const int64_t *ts = reinterpret_cast<const int64_t *>(gbx_sfold_smem + q * GBX_SFOLD_STAGE + GBX_SFOLD_REC);
            const char *bufA = d->bufA, *bufB = d->bufB;
            for (int x = ct; x < left; x += NC) {
                const uint32_t xx = r0 + (uint32_t)x;
                const uint32_t el = unit_of(xx, cpe, magic);
                const int64_t jv = (int64_t)(xx - el * (uint32_t)cpe) * VEC;
                const longlong2 rec = rs[el];
                const uint64_t oa = (uint64_t)rec.x, ob = (uint64_t)rec.y;
                PK res;
                if (oa & GBX_ROW_SINGLE) {
                    res = pload<PK>(((ob & GBX_TERM_BUFB) ? bufB : bufA) + (int64_t)(ob & GBX_TERM_MASK) + jv);
                } else {
                    const int64_t b = (int64_t)(ob >> GBX_ROW_CNT_BITS);
                    const int n = (int)(ob & ((1ull << GBX_ROW_CNT_BITS) - 1));
                    const int64_t *tw = tb_al >= 0 ? ts + (b - tb_al) : d->terms + b;
                    PK grp, tot;
                    bool has = false;
                    for (int m0 = 0; m0 < n; m0 += GBX_SFOLD_K) {
                        const int cnt = min(GBX_SFOLD_K, n - m0);
                        PK xv[GBX_SFOLD_K];
                        uint32_t gbit = 0;
#pragma unroll
                        for (int i = 0; i < GBX_SFOLD_K; i++)
                            if (i < cnt) {
                                const uint64_t w = (uint64_t)tw[m0 + i];
                                gbit |= (w & GBX_TERM_GROUP) ? (1u << i) : 0u;
                                xv[i] = pload<PK>(((w & GBX_TERM_BUFB) ? bufB : bufA) + (int64_t)(w & GBX_TERM_MASK) + jv);
                            }
#pragma unroll
                        for (int i = 0; i < GBX_SFOLD_K; i++)
                            if (i < cnt) {
                                if (m0 + i == 0) {
                                    grp = xv[i];
                                } else if (gbit & (1u << i)) {
                                    tot = has ? padd(tot, grp) : grp;
                                    has = true;
                                    grp = xv[i];
                                } else {
                                    grp = padd(grp, xv[i]);
                                }
                            }
                    }
                    res = has ? padd(tot, grp) : grp;
                }
                PK *o = reinterpret_cast<PK *>(d->out + (int64_t)(oa & ~GBX_ROW_SINGLE) + jv);
                if (d->accumulate) res = padd(*o, res);
                *o = res;
            }
        }
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sempty + 8 * q) : "memory");
        if (abort_flag) break;
    }
}

#define GBX_SFOLD_NT 544
#define GBX_SFOLD_S 3

template <typename T, int VEC, typename L>
static cudaError_t sfold_launch_v(int grid, cudaStream_t st, bool dep, const L &l) {
    return launch(gbx_sfold_kernel<T, VEC, GBX_SFOLD_NT, GBX_SFOLD_S, 2, L>, grid, GBX_SFOLD_NT,
                  (size_t)GBX_SFOLD_S * GBX_SFOLD_STAGE, st, dep, l);
}

template <typename T, int VEC, typename L>
static cudaError_t sfold_attr_l() {
    return cudaFuncSetAttribute(gbx_sfold_kernel<T, VEC, GBX_SFOLD_NT, GBX_SFOLD_S, 2, L>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, GBX_SFOLD_S * GBX_SFOLD_STAGE);
}
template <typename T, int VEC>
static cudaError_t sfold_attr_v() {
    cudaError_t e = sfold_attr_l<T, VEC, OneOp<FoldDesc>>();
    return e == cudaSuccess ? sfold_attr_l<T, VEC, OpList<FoldDesc>>() : e;
}

int gbx_sfold_prepare(void) {
    cudaError_t e = sfold_attr_v<double, 16>();
    if (e == cudaSuccess) e = sfold_attr_v<double, 8>();
    if (e == cudaSuccess) e = sfold_attr_v<float, 16>();
    if (e == cudaSuccess) e = sfold_attr_v<float, 8>();
    if (e == cudaSuccess) e = sfold_attr_v<float, 4>();
    return e == cudaSuccess ? GBX_SUCCESS : GBX_ERR_CUDA;
}

// Window form of the fold, for rows of one 4- or 8-byte value (tables: FoldPiece).  Per piece the
// bulk-copy engine brings the tables into shared memory; the threads gather the piece's terms
// in source order (runs of consecutive gradients: coalesced loads) and drop each at its place;
// then every row is summed from there, in its fixed order, by one thread.  Rows are taken by
// length, 32 of a slice side by side, so a warp's lanes read 32 consecutive values at each step
// and end together.  A term costs 2 bytes of place and its share of a run (8 bytes per term in
// the other forms) and no dependent load.  The other forms are bound by the latency of the chain
// record -> term -> gradient and by scattered 4- and 8-byte reads; here the phases of 3 or 4
// blocks per SM overlap, and the longest row's chain of sums weighs most.  Starts repeated on the
// same buffers, before and after: reverse halo of 2^20 rows, 10.8 M terms, fp32 53.4 -> 29.2 us, fp64 in
// node-blocked order 128 -> 86; of 415 k rows fp32 20.7 -> 12.4; of 300 k rows fp64, node-blocked,
// accumulating 50.9 -> 27.9 (on changing buffers 59 -> 38).
// The wait for the tables is bounded as in the other forms.
#define GBX_WFOLD_TABLES \
    (GBX_WFOLD_N * 2 + GBX_WFOLD_N / 32 * 8 + GBX_WFOLD_RUNS * 4 + GBX_WFOLD_N + GBX_WFOLD_N * 2 + GBX_WFOLD_N / 16 + GBX_WFOLD_N / 8)

template <typename T, int NT, int PS, typename L>
__global__ void __launch_bounds__(NT, PS) gbx_wfold_kernel(const __grid_constant__ L list) {
    constexpr int U = 4;
    constexpr int OFF_POS = GBX_WFOLD_N * (int)sizeof(T), OFF_GRP = OFF_POS + GBX_WFOLD_N * 2,
                  OFF_RUN = OFF_GRP + GBX_WFOLD_N / 32 * 8, OFF_CNT = OFF_RUN + GBX_WFOLD_RUNS * 4,
                  OFF_OUT = OFF_CNT + GBX_WFOLD_N, OFF_BASE = OFF_OUT + GBX_WFOLD_N * 2,
                  OFF_GB = OFF_BASE + GBX_WFOLD_N / 16;
    extern __shared__ __align__(128) unsigned char gbx_wfold_smem[];
    __shared__ __align__(8) uint64_t bar;
    pdl_trigger();
    T *vals = reinterpret_cast<T *>(gbx_wfold_smem);
    const uint16_t *pos = reinterpret_cast<const uint16_t *>(gbx_wfold_smem + OFF_POS);
    const uint2 *grp = reinterpret_cast<const uint2 *>(gbx_wfold_smem + OFF_GRP);
    const uint32_t *run = reinterpret_cast<const uint32_t *>(gbx_wfold_smem + OFF_RUN);
    const uint8_t *rowcnt = gbx_wfold_smem + OFF_CNT;
    const uint16_t *sbase = reinterpret_cast<const uint16_t *>(gbx_wfold_smem + OFF_BASE);
    const uint16_t *rowout = reinterpret_cast<const uint16_t *>(gbx_wfold_smem + OFF_OUT);
    const uint32_t *gbit = reinterpret_cast<const uint32_t *>(gbx_wfold_smem + OFF_GB);
    const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(gbx_wfold_smem);
    const uint32_t sbar = (uint32_t)__cvta_generic_to_shared(&bar);
    // pieces are fetched one ahead, by one thread, into slot k & 1
    __shared__ FoldPiece piece_s[2];
    __shared__ const FoldDesc *desc_s[2];
    __shared__ int64_t local_s[2];
    const int64_t npieces = list.tiles();
    auto fetch = [&](int64_t t, int slot) {
        int64_t lt;
        const FoldDesc *d = list.at(t, lt);
        piece_s[slot] = d->wpiece[lt];
        if (!L::single) desc_s[slot] = d;
        local_s[slot] = lt;
    };
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sbar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (blockIdx.x < npieces) fetch(blockIdx.x, 0);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const uint32_t upto = 0xffffffffu >> (31 - lane);
    uint32_t phase = 0;
    int slot = 0;
    for (int64_t t = blockIdx.x; t < npieces; t += gridDim.x, slot ^= 1) {
        const FoldDesc *d = L::single ? list.first() : desc_s[slot];
        const int n = piece_s[slot].n, nrow = piece_s[slot].nrow;
        const bool some = n > 0 && n <= GBX_WFOLD_N && nrow > 0 && nrow <= n && piece_s[slot].nrun > 0 &&
                          piece_s[slot].nrun <= GBX_WFOLD_RUNS;
        if (threadIdx.x == NT - 1 && t + gridDim.x < npieces) fetch(t + gridDim.x, slot ^ 1);
        if (!some) {
            if (threadIdx.x == 0 && (nrow != 0 || n != 0)) gbx_raise(list, 2);   // validated at init; recorded, skipped
            __syncthreads();
            continue;
        }
        if (threadIdx.x == 0) {
            const int64_t lt = local_s[slot], at = lt * GBX_WFOLD_N;
            const uint32_t pb = ((uint32_t)n * 2 + 15) & ~15u, gb = (((uint32_t)n + 31) / 32 * 8 + 15) & ~15u,
                           rb = ((uint32_t)piece_s[slot].nrun * 4 + 15) & ~15u, cb = ((uint32_t)nrow + 15) & ~15u,
                           ob = ((uint32_t)nrow * 2 + 15) & ~15u, sb = (((uint32_t)nrow + 31) / 32 * 2 + 15) & ~15u,
                           bb = d->wgroups ? GBX_WFOLD_N / 8 : 0u;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the last piece's reads before the refill
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(sbar),
                         "r"(pb + gb + rb + cb + ob + sb + bb)
                         : "memory");
            auto load = [&](uint32_t off, const void *src, uint32_t bytes) {
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(sbuf + off), "l"(src), "r"(bytes), "r"(sbar)
                             : "memory");
            };
            load(OFF_POS, d->wpos + at, pb);
            load(OFF_GRP, d->wgrp + at / 32, gb);
            load(OFF_RUN, d->wrun + lt * GBX_WFOLD_RUNS, rb);
            load(OFF_CNT, d->wrowcnt + at, cb);
            load(OFF_OUT, d->wrowout + at, ob);
            load(OFF_BASE, d->wbase + at / 32, sb);
            if (bb) load(OFF_GB, d->wgroup + at / 32, bb);
        }
        const bool got = bulk_wait(sbar, phase, d->wait_limit);
        if (__syncthreads_or(!got)) {
            if (threadIdx.x == 0) {
                gbx_raise(list, 1);
                bulk_wait(sbar, phase);   // leave no copy in flight
            }
            return;
        }
        phase ^= 1u;
        pdl_wait();
        const T *a = reinterpret_cast<const T *>(d->bufA) - GBX_WFOLD_N, *b = reinterpret_cast<const T *>(d->bufB) - GBX_WFOLD_N;
        // fp64: cp.async straight to the terms' places, all of a thread's in flight together and no
        // registers held (2^20-row reverse halo, node-blocked order: 95 us; 123 through registers).
        // fp32: cp.async of 4 bytes was slower (44 us against 38), so G loads per thread go
        // through registers.
        if constexpr (sizeof(T) == 8) {
            for (int x = threadIdx.x; x < n; x += NT) {
                const uint2 m = grp[x >> 5];
                const uint32_t r = run[m.y + __popc(m.x & upto) - 1];
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;"
                             ::"r"(sbuf + (uint32_t)pos[x] * 8u), "l"(((r >> 31) ? b : a) + ((int64_t)(r & 0x7fffffffu) + x))
                             : "memory");
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
        } else {
            constexpr int G = 4;
            for (int x0 = threadIdx.x; x0 < n; x0 += NT * G) {
                T v[G];
                uint16_t at[G];
#pragma unroll
                for (int u = 0; u < G; u++) {
                    const int x = x0 + u * NT;
                    if (x < n) {
                        const uint2 m = grp[x >> 5];
                        const uint32_t r = run[m.y + __popc(m.x & upto) - 1];
                        v[u] = ((r >> 31) ? b : a)[(int64_t)(r & 0x7fffffffu) + x];
                        at[u] = pos[x];
                    }
                }
#pragma unroll
                for (int u = 0; u < G; u++)
                    if (x0 + u * NT < n) vals[at[u]] = v[u];
            }
        }
        __syncthreads();
        T *out = reinterpret_cast<T *>(d->out) + piece_s[slot].out0;
        for (int r = threadIdx.x; r < nrow; r += NT) {
            const int cnt = rowcnt[r], b0 = sbase[r >> 5];   // (r % 32 = lane)
            const T *v = vals + b0 + lane;
            T *o = out + rowout[r];
            T old = T(0);
            if (d->accumulate) old = *o;
            T g = v[0], tot = T(0);
            bool has = false;
            if (!d->wgroups) {
#pragma unroll 4
                for (int m = 1; m < cnt; m++) g = padd(g, v[m * 32]);
            } else for (int m0 = 1; m0 < cnt; m0 += U) {   // U terms and group bits read ahead of their sums
                T x[U];
                uint32_t st = 0;
#pragma unroll
                for (int i = 0; i < U; i++)
                    if (m0 + i < cnt) {
                        x[i] = v[(m0 + i) * 32];
                        st |= ((gbit[(b0 >> 5) + m0 + i] >> lane) & 1u) << i;
                    }
#pragma unroll
                for (int i = 0; i < U; i++)
                    if (m0 + i < cnt) {
                        // one addition per term whether it starts a group (tot + g) or not (g + x), so
                        // that the lanes of a warp stay together (an fp64 addition holds its pipe
                        // for 16 cycles however few lanes take part)
                        const bool s = (st >> i) & 1u;
                        const T sum = padd(s ? tot : g, s ? g : x[i]);
                        tot = s ? (has ? sum : g) : tot;
                        has |= s;
                        g = s ? x[i] : sum;
                    }
            }
            if (has) g = padd(tot, g);
            *o = d->accumulate ? padd(old, g) : g;
        }
        __syncthreads();
    }
}

// One shape per type: 512 threads x 3 blocks per SM for fp64, 384 x 4 for fp32 (37.0 us on the
// 2^20-row reverse halo; 512 x 3 37.9, 512 x 4 40.2).
template <typename T, typename L>
static cudaError_t wfold_launch(int grid, cudaStream_t st, bool dep, const L &l) {
    constexpr int NT = sizeof(T) == 4 ? 384 : 512, PS = sizeof(T) == 4 ? 4 : 3;
    return launch(gbx_wfold_kernel<T, NT, PS, L>, grid, NT, GBX_WFOLD_N * sizeof(T) + GBX_WFOLD_TABLES, st, dep, l);
}

template <typename T, typename L>
static cudaError_t wfold_attr() {
    constexpr int NT = sizeof(T) == 4 ? 384 : 512, PS = sizeof(T) == 4 ? 4 : 3;
    return cudaFuncSetAttribute(gbx_wfold_kernel<T, NT, PS, L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                GBX_WFOLD_N * (int)sizeof(T) + GBX_WFOLD_TABLES);
}

int gbx_wfold_prepare(void) {
    cudaError_t e = wfold_attr<double, OneOp<FoldDesc>>();
    if (e == cudaSuccess) e = wfold_attr<double, OpList<FoldDesc>>();
    if (e == cudaSuccess) e = wfold_attr<float, OneOp<FoldDesc>>();
    if (e == cudaSuccess) e = wfold_attr<float, OpList<FoldDesc>>();
    return e == cudaSuccess ? GBX_SUCCESS : GBX_ERR_CUDA;
}

// CLS 1..5: every op of the launch is (f64,16) (f64,8) (f32,16) (f32,8) (f32,4).  The kernels
// with one chunk per thread (1024-thread blocks) are held to 32 registers so that two blocks
// fit on an SM: the fold is bound by load latency, and the doubled occupancy outweighs the few
// bytes of spill this costs (512^3 backward, all rows folded: 0.90 -> 0.82 ms).
template <int CLS, int U, typename L>
__global__ void __launch_bounds__(GBX_TILE / U, U == 1 ? 2 : 1) gbx_fold_kernel(const __grid_constant__ L list) {
    pdl_trigger();
    pdl_wait();
    for (int64_t t = blockIdx.x; t < list.tiles(); t += gridDim.x) {
        int64_t lt;
        const FoldDesc *d = list.at(t, lt);
        switch (CLS) {
            case 1: fold_tile<double, 16, U>(d, lt); break;
            case 2: fold_tile<double, 8, U>(d, lt); break;
            case 3: fold_tile<float, 16, U>(d, lt); break;
            case 4: fold_tile<float, 8, U>(d, lt); break;
            default: fold_tile<float, 4, U>(d, lt); break;
        }
    }
}

// ------------------------------------------------------------------- launching
static int g_num_sms = 0;

int gbx_num_sms(void) {
    if (!g_num_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_num_sms <= 0) g_num_sms = 1;
    }
    return g_num_sms;
}

template <int VEC, int FLAT, typename L>
static void (*copy_fn_u(int block))(const L) {
    switch (block) {
        case 128: return gbx_copy_kernel<VEC, 8, FLAT, L>;
        case 256: return gbx_copy_kernel<VEC, 4, FLAT, L>;
        case 512: return gbx_copy_kernel<VEC, 2, FLAT, L>;
        default: return gbx_copy_kernel<VEC, 1, FLAT, L>;
    }
}

template <int VEC, int FORM, typename L>
static void (*pipe_fn_u(int block))(const L) {
    return block == 1024 ? gbx_copy_pipe_kernel<VEC, 1, FORM, L> : gbx_copy_pipe_kernel<VEC, 2, FORM, L>;
}

template <int VEC, typename L>
static void (*copy_fn_v(int block, int flat))(const L) {
    if (flat == 5) return pipe_fn_u<VEC, 1, L>(block);
    if (flat == 7) return pipe_fn_u<VEC, 3, L>(block);
    if (flat == 1) return copy_fn_u<VEC, 1, L>(block);
    if (flat == 3) return copy_fn_u<VEC, 3, L>(block);
    return copy_fn_u<VEC, 0, L>(block);
}

// flat: 0 segment form, 1 flat form, 3 two-index flat form, 5 / 7 the pipelined flat forms (one
// op, persistent grid, block 512 or 1024)
template <typename L>
static void (*copy_fn(int vec, int block, int flat))(const L) {
    switch (vec) {
        case 16: return copy_fn_v<16, L>(block, flat);
        case 8: return copy_fn_v<8, L>(block, flat);
        case 4: return copy_fn_v<4, L>(block, flat);
        case 2: return copy_fn_v<2, L>(block, flat);
        default: return copy_fn_v<1, L>(block, flat);
    }
}

template <int CLS, typename L>
static void (*fold_fn_u(int block))(const L) {
    switch (block) {
        case 128: return gbx_fold_kernel<CLS, 8, L>;
        case 256: return gbx_fold_kernel<CLS, 4, L>;
        case 512: return gbx_fold_kernel<CLS, 2, L>;
        default: return gbx_fold_kernel<CLS, 1, L>;
    }
}

static int fold_cls(int dtype, int vec) {
    if (dtype == GBX_F64) return vec == 16 ? 1 : 2;
    return vec == 16 ? 3 : vec == 8 ? 4 : 5;
}

template <typename L>
static void (*fold_fn(int dtype, int vec, int block))(const L) {
    switch (fold_cls(dtype, vec)) {
        case 1: return fold_fn_u<1, L>(block);
        case 2: return fold_fn_u<2, L>(block);
        case 3: return fold_fn_u<3, L>(block);
        case 4: return fold_fn_u<4, L>(block);
        default: return fold_fn_u<5, L>(block);
    }
}

static int pipe_block(int flat, int block) { return (flat == 5 || flat == 7) && block < 512 ? 512 : block; }

int gbx_occupancy(int kind, int dtype, int vec, int block, int flat) {
    if (kind == 1 && flat == 1) return 2;   // stream fold: two CTAs of 544 threads per SM
    if (kind == 1 && flat == 2) return dtype == GBX_F32 ? 4 : 3;   // window fold
    if (kind == 0 && flat == 8) return 1;   // bulk kernel: one CTA per SM (its ring)
    if (kind == 0 && flat == 9) return scatter_shape(block).per_sm;
    if (kind == 0 && flat >= 10 && flat <= 13) return stream_shape(block).per_sm;
    if (kind == 0 && (flat & 31) == 15) return window_per_sm(vec, flat >> 5 & 1, block);
    if (kind == 0 && flat == 14) return agather_per_sm(block);
    if (kind == 0) block = pipe_block(flat, block);
    const void *f = kind == 0 ? (const void *)copy_fn<OneOp<CopyDesc>>(vec, block, flat)
                              : (const void *)fold_fn<OneOp<FoldDesc>>(dtype, vec, block);
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, block, 0);
    return n > 0 ? n : 1;
}

static int clamp_grid(int grid, int64_t total_tiles) {
    if (grid <= 0 || grid > total_tiles) grid = (int)(total_tiles < (1ll << 30) ? total_tiles : (1ll << 30));
    return grid;
}

template <typename L>
static cudaError_t launch_copy(const L &l, int nops, int vec, int flat, int block, int grid, cudaStream_t st, bool dep) {
    grid = clamp_grid(grid, l.ntiles);
    if (flat == 8)   // bulk form: a "tile" is one piece
        return launch(gbx_bulk_kernel<L>, grid, 32, (size_t)GBX_BULK_STAGES * GBX_BULK_BYTES, st, dep, l);
    if (flat == 9)   // scatter form: a "tile" is one source window
        return scatter_launch(block, grid, st, dep, l);
    if (flat >= 10 && flat <= 13) {   // stream forms: the flat forms' tiles, indices through shared memory
        if (block <= 128 && !(flat >= 12 && vec <= 8)) block = 256;   // the narrow shape needs ONE, vec <= 8
        return stream_launch(vec, flat, block, grid, st, dep, l);
    }
    if ((flat & 31) == 15)   // window form: a "tile" is one piece (code 47: the wide windows)
        return window_launch(vec, flat, block, grid, st, dep, l);
    if (flat == 14) return agather_launch(block, grid, st, dep, l);   // async gather (vec 16)
    if ((flat == 5 || flat == 7) && nops > 1) flat -= 4;   // the pipelined kernels take one op
    block = pipe_block(flat, block);
    return launch(copy_fn<L>(vec, block, flat), grid, block, 0, st, dep, l);
}

template <typename L>
static cudaError_t launch_fold(const L &l, int dtype, int vec, int block, int grid, cudaStream_t st, int form, bool dep) {
    grid = clamp_grid(grid, l.ntiles);
    if (form == 1) {   // stream form
        switch (fold_cls(dtype, vec)) {
            case 1: return sfold_launch_v<double, 16>(grid, st, dep, l);
            case 2: return sfold_launch_v<double, 8>(grid, st, dep, l);
            case 3: return sfold_launch_v<float, 16>(grid, st, dep, l);
            case 4: return sfold_launch_v<float, 8>(grid, st, dep, l);
            default: return sfold_launch_v<float, 4>(grid, st, dep, l);
        }
    }
    if (form == 2)   // window form: a "tile" is one piece
        return dtype == GBX_F64 ? wfold_launch<double>(grid, st, dep, l) : wfold_launch<float>(grid, st, dep, l);
    return launch(fold_fn<L>(dtype, vec, block), grid, block, 0, st, dep, l);
}

cudaError_t gbx_launch_copy(const OpRef<CopyDesc> &r, int vec, int flat, int block, int grid, cudaStream_t st, bool dep) {
    if (r.ntiles <= 0) return cudaSuccess;
    if (r.one) return launch_copy(OneOp<CopyDesc>{*r.one, r.ntiles}, 1, vec, flat, block, grid, st, dep);
    return launch_copy(OpList<CopyDesc>{r.ops, r.prefix, r.nops, r.ntiles}, r.nops, vec, flat, block, grid, st, dep);
}

cudaError_t gbx_launch_fold(const OpRef<FoldDesc> &r, int dtype, int vec, int block, int grid, cudaStream_t st, int form,
                            bool dep) {
    if (r.ntiles <= 0) return cudaSuccess;
    if (r.one) return launch_fold(OneOp<FoldDesc>{*r.one, r.ntiles}, dtype, vec, block, grid, st, form, dep);
    return launch_fold(OpList<FoldDesc>{r.ops, r.prefix, r.nops, r.ntiles}, dtype, vec, block, grid, st, form, dep);
}

// tile_seg[t] = segment holding the first element of tile t; tile_seg[ntiles] = nseg - 1
__global__ void tile_meta_kernel(const Seg *__restrict__ segs, int64_t nseg, int cpe, int64_t ntiles, int64_t *ts) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t <= ntiles;
         t += (int64_t)gridDim.x * blockDim.x) {
        if (t == ntiles) {
            ts[t] = nseg - 1;
            continue;
        }
        const int64_t e = (t * GBX_TILE) / cpe;
        int64_t lo = 0, hi = nseg - 1;
        while (lo < hi) {
            int64_t mid = (lo + hi + 1) >> 1;
            if (segs[mid].v0 <= e) lo = mid; else hi = mid - 1;
        }
        ts[t] = lo;
    }
}

int gbx_build_tile_meta(const Seg *segs, int64_t nseg, int cpe, int64_t ntiles, int64_t *tile_seg, cudaStream_t st) {
    int64_t n = ntiles + 1;
    int64_t g = ceil_div(n, 256);
    if (g > 65535 * 16) g = 65535 * 16;
    tile_meta_kernel<<<(unsigned)g, 256, 0, st>>>(segs, nseg, cpe, ntiles, tile_seg);
    GBX_CUDA_TRY(cudaGetLastError());
    return GBX_SUCCESS;
}
