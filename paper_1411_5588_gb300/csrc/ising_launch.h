// Host-side launchers of the Ising-film kernels (internal to the library).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "ising_device.cuh"

namespace isg {

// Grid update kernels: threads per block and blocks per SM.  A thread has a
// column of column_len(items) words, items being the launch shape: GRID_1 (1)
// one, GRID_Q (0) two, GRID_2 (2) four.  A word of a column costs five loads
// instead of seven and no address set-up, but a launch then has a quarter of
// the threads and four words one after another in each: per sweep, no records,
// one / two / four words take 45.5 / 38.1 / 40.3 us on 120x240x1600, and 5.9 / 6.1 /
// 12.3 us on 32x96x64.
//
// Forms: columns by masks (single films without a bulk field), columns by
// look-ups (single films in one, and most film sets, whose walls would otherwise
// take seven masks: 320 films of 32x96x64 60.1 us per sweep by masks, 53.7 by look-ups,
// in a field 85.7 and 52.8), one word by masks drawn ahead, and one word by
// look-ups (kLookBlocks).
//
// The blocks per SM are the most whose registers hold each variant without a
// spill: 128 threads are a warp on each scheduler, whose register file grants
// 64 a thread at eight blocks, 72 at seven, 80 at six, 96 at five.
constexpr uint32_t kFilmThreads = 128;
enum : uint32_t { kFormColumns = 0, kFormColumnsLook = 1, kFormWord = 2, kFormWordLook = 3 };
constexpr int film_min_blocks(int rows, bool meas, uint32_t form) {
  return form == kFormWord || form == kFormWordLook ? (rows == 4 ? 5 : meas ? 7 : 8)
         : form == kFormColumnsLook                 ? (meas ? 6 : 7)
                                                    : rows > 1 || meas ? 5 : 6;
}
constexpr int multi_min_blocks(uint32_t form, bool meas, bool pack) {
  return form == kFormWord       ? (pack ? (meas ? 5 : 6) : 8)
         : form == kFormWordLook ? (meas ? 5 : 6)
                                 : meas ? 4 : 5;
}
__host__ __device__ constexpr uint32_t column_len(uint32_t items) {
  return items == 1 ? 1 : items == 2 ? 4 : 2;
}
// Blocks from which a launch of one word per thread is made by look-ups where
// most of its words are general: more than a wave (152 SMs, eight blocks each).
// Below it the chain counts, and seven masks drawn ahead are no slower.  Films
// in a bulk field, per sweep, masks / look-ups: 864 blocks 10.7 / 12.2 us, 1024
// blocks 12.7 / 12.7, 5625 blocks 68.1 / 45.6.
constexpr uint32_t kWaveWords = 8 * 152 * kFilmThreads;
constexpr uint32_t kLookBlocks = kWaveWords / kFilmThreads + 1;
// Whether film d's words are short: rows of one word of at most five calls, packed
// or not.
inline bool short_words(const FilmDesc& d) { return d.W == 1 && d.last_calls <= 5; }
// Form of a film set's launch: `words` words in all, `brief` of them short,
// `general` of films in a bulk field.  In columns, sets of short words go by masks
// (40 films of 64x512x32 44.9 us per sweep, by look-ups 51.2; of 128x512x16 55.2 and
// 57.3; 64 of 64x129x40 24.4 and 28.4), all others by look-ups: blocks by masks
// beside blocks by look-ups, in sets of thin and thick films, thrash the
// instruction cache (the line-tension set, 62% short, 45.7 us by look-ups, 52.5
// mixed).
inline uint32_t set_form(uint32_t items, uint32_t grid, uint64_t words, uint64_t brief, uint64_t general) {
  const bool look = 2 * general > words;
  if (items == 1) return look && grid >= kLookBlocks ? kFormWordLook : kFormWord;
  return !look && 8 * brief > 7 * words ? kFormColumns : kFormColumnsLook;
}
constexpr int kMeasureBlock = 256;

// Items a measurement block covers per layer before another block is added;
// layers of fewer than kMeasureItemsPerBlock / 2 words are grouped, up to
// kMeasureMaxLpu of them per block.
constexpr uint32_t kMeasureItemsPerBlock = 4 * kMeasureBlock;
constexpr uint32_t kMeasureMaxLpu = 64;

// The film's per-layer record accumulators (int64 pairs: magnetisation,
// bonds; Lx of them) follow its measurement partial sums in the same area.
__host__ __device__ inline uint64_t acc_offset(const FilmDesc& d) {
  return d.part_off + 2ull * d.Lx * d.meas_bpl;
}

// Work of a half-sweep of film d with a row per word, in words of eight calls (a
// word is its Philox calls, and about two more in loads and decisions).
inline uint64_t row_work(const FilmDesc& d) {
  return (uint64_t)d.Lx * d.Ly * d.W * ((d.W == 1 ? d.last_calls : 8u) + 2) / 10;
}
// Rows that a thin film packs to a word in launches of `work` words of eight calls
// (row_work of all their films), side by side.  Packed words are fewer
// instructions per site, but a chain of all their rows' calls in a fraction of
// the threads: they pay once the work fills the GPU for a wave (four rows), or
// three fifths of one (two).  Per sweep, a word per row / packed: four rows 65536
// rows (128x512x16, 0.17 waves) 6.3 / 12.4 us, 262144 (256x1024x16, 0.67) 10.6 /
// 14.1, 327680 (0.84) 12.0 / 14.4, 524288 (1.35) 17.0 / 14.4, 16 and 32 films of
// 64x256x16 (0.67 and 1.35) 10.4 / 12.9 and 20.0 / 17.3, twenty films of the
// line-tension set (1.08) 25.6 / 19.8; two rows 65536 (128x512x32, 0.25) 6.1 / 9.4,
// 153600 (0.59) 7.3 / 10.1, 196608 (0.76) 9.0 / 9.2, 262144 (1.01) 12.2 / 10.0.  Two
// rows only in films of at least kPack2Rows: a set of small ones is bound by its
// chains (the beta-integration set's films of 1200-3000 rows lose 6% packed, the
// line-tension set's of 13824 gain).
constexpr uint32_t kPack2Rows = 8192;
inline uint32_t grid_pack(const FilmDesc& d, uint64_t work) {
  if (d.sl_pack == 4) return work > kWaveWords ? 4u : 1u;
  return d.sl_pack == 2 && d.Lx * d.Ly >= kPack2Rows && 5 * work > 3 * kWaveWords ? 2u : 1u;
}

// Columns of a film in the grid update kernels (of words, or of packed words of
// `pack` rows): the pairs, then the rows between the first and the last, those
// of the first and the last layer before the others.  By masks a wall's words
// take half as long again to draw, and a block of them outlasts the others, so
// its columns are those of the next shorter shape (wall_short; 96x192x384 on
// GRID_Q: 9.9 us per sweep without, 8.5 with).  By look-ups all words cost alike
// (320 films of 32x96x64 on GRID_2: 53.7 us, 55.2 with shorter ones).
__host__ __device__ inline uint32_t wall_items(const FilmDesc& d, uint32_t items) {
  return !d.wall_short ? items : items == 2 ? 0u : 1u;
}
__host__ __device__ inline uint32_t grid_columns(const FilmDesc& d, uint32_t items) {
  const uint32_t walls = d.Lx < 2 ? d.Lx : 2u;
  return walls * d.cols[wall_items(d, items)] + (d.Lx - walls) * d.cols[items];
}
__host__ __device__ inline uint32_t grid_items(const FilmDesc& d, uint32_t items) {
  return d.W * (d.Lx + grid_columns(d, items));
}
__host__ __device__ inline uint32_t update_blocks(const FilmDesc& d, uint32_t items) {
  return (grid_items(d, items) + kFilmThreads - 1) / kFilmThreads;
}

// Words a half-sweep's launch updates for film d, and the most for which, without
// a measurement, a launch takes one word per thread: it is the shorter launch,
// columns are the higher rate.  Per sweep, one word / columns of two (one film):
// 245760 words 15.7 / 16.6 us, 524288 33.2 / 28.2; one word / columns of four (a
// batch's two lanes): 122880 words each 18.0 / 23.2, 245760 33.5 / 28.1, 491520
// 67.3 / 53.7, 806400 110 / 88.  Film sets cross over a little below the line.
constexpr uint64_t kOneWordAutoWords = 1ull << 18;
inline uint64_t launch_words(const FilmDesc& d) { return (uint64_t)d.Lx * (d.Ly / d.pack) * d.W; }

// Measurement blocks of one film.
inline uint32_t meas_units(const FilmDesc& d) {
  return d.meas_lpu > 1 ? (d.Lx + d.meas_lpu - 1) / d.meas_lpu : d.Lx * d.meas_bpl;
}

// The form of a film's tables that its cost and its slab's size depend on: 1 where
// the inner layers take three masks, 0 where they take seven.
inline uint32_t table_form(const FilmDesc& d) { return d.cls[0].sym; }

// Resident path: one CTA holds the film in shared memory for a whole run of
// sweeps, records included (the slab kernel with C = 1).  Films up to
// kResidentMaxSites spins whose planes and layer sums fit in
// kResidentMaxSmem bytes qualify; larger ones use the per-half-sweep grid.
// Chosen automatically, without a measurement, up to kResidentAutoSites; the
// cluster path from there up to kClusterAutoSites.  Per sweep on GB300, a record
// every sweep, resident / cluster of 8 / best grid: 8^3 2.3 / 2.6 / 8.4 us,
// 16x48x32 5.7 / 3.3 / 8.4, 32^3 7.8 / 3.6 / 7.6, 32x64x64 - / 5.6 / 8.9; without
// records the grid draws level at 32x96x64 (6.0 / 6.0 us).
constexpr uint64_t kResidentMaxSites = 1ull << 16;
constexpr uint64_t kResidentAutoSites = 1ull << 10;
constexpr uint64_t kClusterAutoSites = 3ull << 15;
constexpr uint64_t kResidentOnlySites = 1ull << 15;
constexpr uint32_t kResidentMaxSmem = 48u * 1024u;

// Slab path: a thread-block cluster of C CTAs (C <= kClusterMaxSize) holds one
// film in distributed shared memory for a whole call of sweeps, each CTA a
// slab of ceil(Lx / C) layers or one fewer.  kSlabThreads is the most threads
// a CTA runs on columns, kTaskThreads the most on tasks (slab_tasks_fit);
// kClusterMaxSmem the most dynamic shared memory it takes.
constexpr uint32_t kSlabThreads = 640;
constexpr uint32_t kTaskThreads = 640;
constexpr uint32_t kClusterMaxSize = 8;
constexpr uint32_t kClusterMaxSmem = 200u * 1024u;

// Rows per word of film d on clusters of C CTAs: thin films pack (sl_pack)
// unless the words, one row each, are few enough (128) for four drawing lanes and
// a deciding thread each in one turn: a packed word then only lengthens the
// chain of Philox calls.
__host__ __device__ inline uint32_t slab_rows(const FilmDesc& d, uint32_t C) {
  const uint64_t words = (uint64_t)((d.Lx + C - 1) / C) * d.Ly * d.W;
  return words <= 128 ? 1u : d.sl_pack;
}
// Philox calls of a word of film d in a slab of R rows per word.
inline uint32_t slab_calls(const FilmDesc& d, uint32_t R) { return d.W == 1 ? R * d.last_calls : 8u; }
// Work of a slab's half-sweep in words of eight calls: a word is its calls, and
// about two more in loads and decisions.  Without a measurement a film takes the
// slab path up to kClusterAutoWords of them per CTA, and up to twice that with a
// record every sweep, which costs the grid some 3.4 us and the cluster 0.4.  Per
// sweep, no records / a record each, cluster / one word per thread: 256
// (4x128x128) 5.9 / 6.2 and 5.6 / 9.1 us, 384 (3x128x192) 6.5 / 6.8 and 5.3 / 8.8,
// 490 (64x153x10) 7.5 / 8.0 and 5.2 / 8.4, 512 (2x128x256) 7.6 / 8.0 and 5.2 / 8.7.
constexpr uint64_t kClusterAutoWords = 256;
inline uint64_t slab_work(const FilmDesc& d, uint32_t C) {
  const uint32_t rows = slab_rows(d, C);
  return (uint64_t)((d.Lx + C - 1) / C) * (d.Ly / rows) * d.W * (slab_calls(d, rows) + 2) / 10;
}
// Columns of a slab (the largest of the cluster's) over at most tmax threads:
// each layer's G groups (words, W of them per group) in equal columns of
// `len` >= 2 steps, as short as one turn of the threads allows; with more than
// tmax columns of whole layers, threads take several in turn.
struct SlabShape {
  uint32_t len, turns, threads;
};
__host__ __device__ inline SlabShape slab_shape(const FilmDesc& d, uint32_t C, uint32_t tmax) {
  const uint32_t G = d.Ly / slab_rows(d, C), per = (d.Lx + C - 1) / C * d.W;
  uint32_t n = tmax / per;  // columns per layer and word
  if (n < 1) n = 1;
  SlabShape o;
  o.len = (G + n - 1) / n;
  if (o.len < 2) o.len = 2;
  const uint32_t cols = per * ((G + o.len - 1) / o.len);
  o.turns = (cols + tmax - 1) / tmax;
  o.threads = ((cols + o.turns - 1) / o.turns + 31) / 32 * 32;
  if (o.threads > tmax) o.threads = tmax;
  return o;
}

// Device arrays describing the films of a launch.
struct LaunchSet {
  FilmDesc* films = nullptr;         // n_films descriptors
  uint32_t* owner_upd = nullptr;     // virtual update block -> film
  uint32_t* owner_meas = nullptr;    // virtual measurement block -> film
  LaunchHdr* hdr = nullptr;          // sizes
};

// items: the launch shape, matching the owner table's block size; form: set_form's.
// Records:
// with accumulate (colour 1) the films that record after sweep k add their
// record sums into their accumulators in part; with rec_done > 0 (colour 0) the
// films that recorded after rec_done sweeps have that record written into
// their rings in records by this launch (the chunk's last record goes through
// launch_record instead).  pack: some film of the launch packs rows
// (FilmDesc::pack > 1).  first: the chunk's first launch, whose predecessor may
// still be advancing the films' sweep counters.
cudaError_t launch_update(const LaunchSet& L, uint32_t grid, uint32_t* pool, uint32_t colour, uint32_t k,
                          uint32_t items, uint32_t form, bool pack, int64_t* part, int64_t* records, bool accumulate,
                          uint32_t rec_done, bool first, cudaStream_t st);
// One half-sweep of a single film whose descriptor (with `sweep` absolute) is
// passed by value; acc (colour 1 of a recorded sweep, else null): the film's
// accumulators.
cudaError_t launch_update_film(const FilmDesc& d, uint32_t* pool, uint32_t colour, uint32_t sweep, uint32_t items,
                               int64_t* acc, cudaStream_t st);
// Records of the films that record after `done` sweeps of the chunk, from the
// accumulators the half-sweep 1 launch filled (which it clears).
cudaError_t launch_record(const LaunchSet& L, uint32_t grid, int64_t* part, int64_t* records, uint32_t done,
                          cudaStream_t st);
cudaError_t launch_measure(const LaunchSet& L, uint32_t grid, uint32_t fin_grid, const uint32_t* pool,
                           int64_t* part, int64_t* records, uint32_t done, int force, int64_t* direct,
                           cudaStream_t st);
cudaError_t launch_advance(const LaunchSet& L, uint32_t grid, uint32_t n_sweeps, cudaStream_t st);
cudaError_t launch_init(const FilmDesc& f, uint32_t* pool, int kind, uint32_t flip_lo, int flip_all,
                        cudaStream_t st);
cudaError_t launch_pack(const FilmDesc& f, uint32_t* pool, const int8_t* s, cudaStream_t st);
cudaError_t launch_unpack(const FilmDesc& f, const uint32_t* pool, int8_t* s, cudaStream_t st);
// Dynamic shared memory of a film on the resident path, 0 if it does not qualify.
uint32_t resident_smem_bytes(const FilmDesc& d);
// Dynamic shared memory of a CTA of film d on the cluster-resident path with
// clusters of C CTAs, 0 if the film does not qualify (C out of range, fewer
// layers than C, or too large).
uint32_t cluster_smem_bytes(const FilmDesc& d, uint32_t C);
// CTAs of the cluster path that share one SM (1..kClusterMaxPerSm): the launch
// pads each CTA's shared memory so that no more than per_sm fit on an SM.
constexpr uint32_t kClusterMaxPerSm = 2;
// Threads per CTA for film d with clusters of C CTAs, per_sm CTAs per SM: the
// slab's columns (slab_shape) over at most kSlabThreads / per_sm threads, or its
// draw tasks over at most kTaskThreads / per_sm (a multiple of 32).
uint32_t cluster_threads(const FilmDesc& d, uint32_t C, uint32_t per_sm, bool tasks);
// Whether the film takes the task form (its words few enough, and they and the
// masks fit a CTA's shared memory), and the dynamic shared memory of either form.
// Both depend on the film's geometry and on table_form.
bool slab_tasks_fit(const FilmDesc& d, uint32_t C);
uint32_t slab_dyn_bytes(const FilmDesc& d, uint32_t C, bool tasks);
// Clusters of C CTAs (smem_bytes of dynamic shared memory needed and threads
// each, per_sm of them per SM) that one GPU can hold at once (0: such a
// launch cannot run), or -1 on a CUDA error.  Sets the kernel's attributes and
// *smem_launch, the padded shared memory to launch with: a launch needs no
// further queries (six calls, some 5 us of host time).
int cluster_capacity(uint32_t C, uint32_t per_sm, uint32_t smem_bytes, uint32_t threads, bool tasks,
                     uint32_t* smem_launch);
// n_sweeps sweeps (with their records) of films on the cluster path:
// n_clusters clusters of C CTAs, cluster i sweeping the films list[n_clusters +
// 1 + j], j in [list[i], list[i + 1]), one after another (list: device memory;
// null: cluster i sweeps film i).  Every listed film must qualify for C (tasks:
// for slab_tasks_fit), threads cover the largest, and smem_launch is
// cluster_capacity's for these.  The kernel advances each descriptor's sweep
// and rec_next.
cudaError_t launch_cluster(FilmDesc* films, const uint32_t* list, uint32_t n_clusters, uint32_t C,
                           uint32_t smem_launch, uint32_t threads, bool tasks, uint32_t* pool, int64_t* records,
                           uint32_t n_sweeps, cudaStream_t st);
// Checked builds: the out-of-range access counters (returns 1); other
// builds return 0 with both zero; -1 on a CUDA error.
int read_oob_counters(unsigned long long* count, unsigned long long* first);
// The same for the allocation-free measurement kernel (ising_noalloc.cu).
int read_noalloc_oob_counters(unsigned long long* count, unsigned long long* first);
int update_blocks_per_sm();
int measure_blocks_per_sm();

}  // namespace isg
