// wg_launch.h -- host-side launchers of the sm_103a kernels (one translation
// unit per kernel family; the host engine only sees these declarations).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace wg {

// Records `msg` as the calling thread's wg_last_error() and returns `code`.
int set_error(int code, const char* msg);

struct Stage;
struct Dev;
struct Inst;
struct RowJob;
struct TriJob;
struct SgJob;
struct MsdJob;
struct RowInst;
struct SgInst;

// sorted-array stages (wg_kern_sort.cu); K = uint32_t or unsigned long long
template <typename K> void launch_sort_hist(Stage* st, int grid, cudaStream_t s);
// dbits: digit width of the pass plan (8 picks the whole-byte-digit kernel)
template <typename K> void launch_sort_pass(Stage* st, int grid, cudaStream_t s, uint32_t dbits);
// every pass of segments of at most kSegSortMaxTiles tiles, one CTA per segment
// (st0: the first pass's stage; the later passes' stages follow it)
template <typename K> void launch_sort_seg(Stage* st0, int grid, cudaStream_t s, uint32_t dbits,
                                           int items, bool wide);  // keys per thread: 16 or 8
template <typename K> void launch_unique_diff(Stage* st, int grid, cudaStream_t s);
template <typename K> void launch_merge(Stage* st, int grid, cudaStream_t s);
// tile: merged keys per fused-pass tile, FuseTile<K>::T or half of it
template <typename K> void launch_diff_merge(Stage* st, int grid, cudaStream_t s, uint32_t tile);
// mode 0: merge-path splits of a (Full, candidates) / (Full, delta) stage;
// mode 1: join-slab owner of each emit tile.  `tile` = outputs per tile.
template <typename K>
void launch_partition(Stage* consumer, int mode, uint32_t tile, int grid, cudaStream_t s);
template <typename K> int occupancy_sort(int which);  // 0 hist, 1 pass, 2 uniq, 3 merge, 4 fused,
                                                      // 5 fused with half tiles, 6 / 7 segment sort
                                                      // of 16 / 8 keys per thread

// sort of a large array by its top digit first (wg_kern_msd.cu), in three steps
template <typename K> void launch_msd_sort(const MsdJob& J, int step, int sms, cudaStream_t s);

// join and engine control (wg_kern_join.cu)
// tile: delta tuples per count tile, kTileD or kTileD / 2
template <typename K> void launch_join_count(Stage* st, int grid, cudaStream_t s, uint32_t tile);
template <typename K> void launch_join_emit(Stage* st, int grid, cudaStream_t s, uint32_t tile);
template <typename K> void launch_tri_probe(Stage* st, int grid, cudaStream_t s);
void launch_fuse_mark(Dev* dv, int grid, cudaStream_t s);
void launch_fuse_list(Dev* dv, int grid, cudaStream_t s);
template <typename K> void launch_fuse_copy(Stage* st, int grid, cudaStream_t s, uint32_t tile);
template <typename K> void launch_join_emit_hash(Stage* st, int grid, cudaStream_t s);
template <typename K>
void launch_hash_build(const K* E, unsigned long long ne, uint32_t w, unsigned long long* T,
                       unsigned long long mask, int grid, cudaStream_t s);
template <typename K> int occupancy_join(int which);  // 0 count, 1 emit, 2 triangle probe,
                                                      // 3 count with half tiles
// one warp waiting on a status word that is never published (bounded wait self-test)
struct Ctl;
void launch_selftest_wait(const unsigned long long* status, Ctl* ctl, unsigned long long* out,
                          cudaStream_t s);
// the same wait in the allocation-free sort's control block (wg_noalloc.cu)
int noalloc_selftest_wait(cudaStream_t s);
void launch_plan_delta(Dev* dv, cudaStream_t s);
void launch_plan_cand(Dev* dv, cudaStream_t s);
void launch_plan_merge(Dev* dv, cudaStream_t s);
void launch_plan_post(Dev* dv, cudaStream_t s);
void launch_plan_side(Dev* dv, cudaStream_t s);
void launch_xseg_build(Dev* dv, cudaStream_t s);
template <typename K>
void launch_init_diag(Inst* inst, uint32_t first, uint32_t count, void* dpool, cudaStream_t s);

// row-by-row closure (wg_kern_rows.cu); id_bytes: 2 for at most 2^16 vertices, else 4
int occupancy_rows(int id_bytes, uint32_t vwords);
void launch_rows(const RowJob& J, int id_bytes, int grid, cudaStream_t s);
// writes a single query's instance and clears `bytes` (a multiple of 16) of scratch
void launch_row_begin(const RowJob& J, const RowInst& I, const SgInst& G, void* clear,
                      size_t bytes, int sms, cudaStream_t s);
void launch_rows_small(const RowJob& J, int grid, cudaStream_t s);
void launch_row_plan(const RowJob& J, uint32_t n_inst, cudaStream_t s);
template <typename K> void launch_row_expand(const RowJob& J, int grid, cudaStream_t s);
double row_candidate_ns(uint32_t vwords);
// two-paths from every source: paths (nv zeros before), out: their maximum and sum (zeros)
template <typename K>
void launch_row_paths(const K* E, uint32_t ne, uint32_t w, const uint32_t* off, const uint32_t* adj,
                      uint32_t* paths, unsigned long long* out, int grid, cudaStream_t s);
// adjacency units of a relation: their number, and the layout of vertex records
// (16 bytes each), out-edge bit set (words), further units (16 bytes each), bit set
// of the vertices with several parents (words; followed by as many of scratch)
size_t row_units(uint64_t ne, uint32_t nv, int id_bytes);
template <typename K>
void launch_row_layout(const K* E, uint32_t ne, uint32_t w, const uint32_t* off,
                       const uint32_t* adj, uint32_t nv, void* rec, uint32_t* ns, uint32_t words,
                       void* units, uint32_t* mp, int id_bytes, int grid, cudaStream_t s);

// same-generation over rows (wg_kern_sg.cu): every iteration, and the row counts
int occupancy_sg(int id_bytes, uint32_t vwords);
cudaError_t launch_sg(const SgJob& J, int id_bytes, int grid, int sms, cudaStream_t s);

// triangle counting by set intersection (wg_kern_tri.cu): transpose and count
template <typename K>
void launch_tri(const K* E, uint32_t ne, uint32_t w, const TriJob& J, int sms, cudaStream_t s);

// relation load and result extraction
template <typename K>
void launch_rank_edges(const uint32_t* src, const uint32_t* dst, unsigned long long n,
                       const uint32_t* V, uint32_t nv, uint32_t w, K* keys, int grid,
                       cudaStream_t s);
template <typename K>
void launch_csr(const K* E, unsigned long long ne, uint32_t nv, uint32_t w, uint32_t* off,
                uint32_t* adj, int grid, cudaStream_t s);
template <typename K>
void launch_result_map(const K* F, unsigned long long n, uint32_t w, const uint32_t* V,
                       unsigned long long* out, int grid, cudaStream_t s);
// adds the digest of the n tuples F (ranks mapped to ids through V) to *out
template <typename K>
void launch_result_digest(const K* F, unsigned long long n, uint32_t w, const uint32_t* V,
                          unsigned long long* out, int grid, cudaStream_t s);

}  // namespace wg
