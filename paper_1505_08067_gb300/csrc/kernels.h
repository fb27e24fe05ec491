// Host-side launch interface of the device kernels in kernels.cu.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include "fft_core.h"
#include "fft_join.h"

namespace gbfft {

// The joined kernels (joined.cuh): both passes of a four-step transform, or of
// 2D frames, in one launch.
constexpr uint32_t kJoinPolls = 1u << 21;  // about a second before a wait gives up
constexpr int kStatusGaveUp = 1;           // status word: a bounded wait gave up
constexpr int kStatusCounters = 2;         // and: a joined launch's counters were not its own
struct JoinDesc {
  const cf* tw1;  // w_L^j of the first pass's length, and of the second's
  const cf* tw2;
  JoinOrder o;
  unsigned* ctr;  // 2 + 2 ring counters, zero between launches
  int* status;
  uint32_t polls;  // kJoinPolls, or fewer in a test of the waits
  // frames: log2 rows and columns, elements of the whole batch
  int lr, lc;
  int64_t total;
  // first-pass tiles are prefetched into L2 when `mapped`: for transforms by a
  // tensor map of the input viewed as rows of N2 elements in boxes of G1
  // columns; frames only need a 16-byte-aligned input
  int mapped;
  alignas(64) unsigned char tmap_in[128];
};
struct JoinedLaunch {
  const void* fn = nullptr;  // null: the plan's passes run as launches of their own
  bool frames = false;
  const void* second = nullptr;  // passes apart (join_apart): fn is the first, this the second
  size_t second_smem = 0;
  int max_grid = 0;          // resident blocks
  int block = 0;
  size_t smem = 0;
  int tile_log = 0;
  int n1 = 0, n2 = 0, g1 = 0, box_rows = 0;
  JoinDesc d{};
};
// Kernel (apart: kernels) for transforms of 2^logn, or frames of 2^lr x 2^lc in
// tiles of 2^tile_log, its opt-in shared memory, resident blocks and tiles per unit.
cudaError_t prepare_joined(int logn, bool apart, bool inverse, int sm_count, JoinedLaunch* j);
cudaError_t prepare_joined_frames(int lr, int lc, int tile_log, bool inverse, int sm_count,
                                  JoinedLaunch* j);
// `batch` transforms or frames; `work`: the ring of a four-step plan.
cudaError_t launch_joined(const JoinedLaunch& j, int64_t batch, const void* in, void* out,
                          void* work, cudaStream_t st);
// Tensor map (128 bytes) over `rows` rows of `cols` complex64 elements at `p`,
// boxes of box_cols x box_rows; false if `p` or the driver does not allow it.
// (esz: bytes per element, 8 or 4)
bool encode_rows_map(const void* p, int64_t cols, int64_t rows, int box_cols, int box_rows,
                     unsigned char (&map)[128], int esz = 8);

// Job table of a coalesced launch (see stockham_grouped): up to kMaxGroup jobs
// of one contiguous single-pass shape, each with its own buffers.
constexpr int kMaxGroup = 64;
struct GroupEntry {
  const cf* in;
  cf* out;
  int64_t tile_begin;  // first tile of this job in the launch
  int64_t tiles;       // tiles of this job
  int64_t count;       // transforms of this job
};
struct GroupTable {
  int n;
  GroupEntry e[kMaxGroup];
};

// A launch that may start while the kernel before it in the stream finishes
// (programmatic stream serialization; after anything but a kernel it is an
// ordinary launch); the kernel waits for it (grid_wait) before it touches global
// memory.  Without it a dependent launch begins about 2 us after the last block
// of the kernel before: N = 1024 x 64 4.14 -> 2.64 us per call back to back,
// 2^20 x 1 (two launches) 16.4 -> 11.3, 4096 x 8192 frame 223.8 -> 219.1.
template <class... A>
inline cudaError_t launch_early(const void* fn, int grid, int block, size_t smem, cudaStream_t st,
                                const A&... args) {
  if (!fn) return cudaErrorInvalidValue;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &a;
  c.numAttrs = 1;
  void* p[] = {const_cast<void*>(static_cast<const void*>(&args))...};
  const cudaError_t e = cudaLaunchKernelExC(&c, fn, p);
  if (e != cudaSuccess) (void)cudaGetLastError();
  return e;
}

// Everything needed to launch one stockham_pass.
struct PassLaunch {
  PassDesc d;
  int R;            // elements per thread (register radix): 2, 4, 8 or 16
  int lmap, smap;   // thread maps of the load (and middle) stages and of the store
  int grid, block;  // grid size (tiles are grid-strided) and threads per block
  size_t smem;      // dynamic shared memory in bytes
  const void* fn = nullptr;  // resolved kernel (specialised or generic)
  bool specialised = false;
  int lines = 0;             // a line kernel (resolve_lines): log2 of its tile, one per block
  bool has_staged = false;   // a staged kernel exists for this shape (see below)
  int persistent_grid = 0;   // nonzero: grid capped at resident blocks (L2-prefetch variant)
  int ctas_per_sm = 0;       // persistent kernels: resident blocks per SM the grid assumes
  struct StagedLaunchData {
    const void* fn = nullptr;
    int grid = 0, block = 0;
    int max_grid = 0;  // resident blocks per SM x SMs (persistent grid)
    size_t smem = 0;
    bool map_in = false;   // input in column tiles (tensor-map box loads possible)
    bool map_out = false;  // output in column tiles (tensor-map box stores possible)
    bool tmap = false;     // use tensor maps where the layout allows
  } staged;
};

// The staged kernel for a pass (one contiguous transform or G columns per
// block, TMA copy of the next tile); used when the source is 16-byte aligned.
using StagedLaunch = PassLaunch::StagedLaunchData;

// Fills `s` if a staged kernel exists for this pass shape (contiguous
// transforms, or column tiles of a strided pass) and thread maps.
bool resolve_staged(const PassDesc& d, int lmap, int smap, bool generic_only, StagedLaunch* s);
// Opt-in shared memory and a persistent grid of (blocks per SM) x SMs.
cudaError_t prepare_staged(StagedLaunch& s, int64_t tiles, int sm_count);
cudaError_t launch_staged(const StagedLaunch& s, const PassDesc& d, const void* in, void* out,
                          cudaStream_t st);
// Encodes d.tmap_in (map_in) and d.tmap_out (map_out) for column tiles over
// `in` / `out` and sets d.tmap_*_ok; false if neither could be encoded (the
// pass's layout or the driver does not allow it).
bool encode_cols_maps(PassDesc& d, bool map_in, bool map_out, const void* in, void* out);

// Kernel for this pass shape: a compile-time specialisation when one matches,
// else the generic kernel for (R, maps).
const void* resolve_kernel(int R, int lmap, int smap, const PassDesc& d, bool generic_only,
                           bool* specialised);

// Tensor-core class kernel for length 2^logL (4, 8, 12) and FFT_PREC_TC_*:
// the warp-level MMA form.
const void* resolve_tc(int logL, int prec);
// The tcgen05 form for length 2^logL (4 .. 14); *smem = the shared memory it
// needs (the plan may ask for more to bound the CTAs per SM).
const void* resolve_umma(int logL, int prec, size_t* smem);
// Tensor-memory columns one tcgen05 block of length 2^logL allocates.
int umma_tmem_cols(int logL);
// Blocks of `fn` one SM holds at once by its registers, shared memory and
// threads (from the kernel's attributes and the device's limits), and by
// tensor memory when tmem_cols > 0 (512 columns per SM).
cudaError_t resident_blocks(const void* fn, int block, size_t smem, int tmem_cols, int* blocks);
// The tcgen05 form of the FP16 class with complex32 input and output.
const void* resolve_umma_c32(int logL, size_t* smem);
// The tcgen05 column forms (first and second pass of four-step plans) for
// lengths 2^7 .. 2^10; io16: complex32.
const void* resolve_umma_cols1(int logL, int prec, int io16);
const void* resolve_umma_cols2(int logL, int prec, int io16);
// Tensor map of a first pass's input (d.tmap_in; sets d.tmap_in_ok): `rows`
// rows of 2^le elements of `esz` bytes, boxes of `cols` x `box_rows`.
void encode_tc_cols_map(PassDesc& d, const void* in, int64_t rows, int le, int esz, int cols,
                        int box_rows);
// The kernel of a tensor-core pass of the given variant (0 tcgen05, 1 warp MMA);
// io16: complex32 input and output (tcgen05, FP16 only).
inline const void* resolve_tc_pass(int logL, int prec, int variant, int io16 = 0) {
  size_t sm = 0;
  if (io16) return variant == 0 && prec == 1 ? resolve_umma_c32(logL, &sm) : nullptr;  // FP16
  return variant == 1 ? resolve_tc(logL, prec) : resolve_umma(logL, prec, &sm);
}

// Six-step transposes (transpose.cu): per batch entry, rows x cols -> cols x
// rows, optionally multiplying element (r, c) by exp(sign 2 pi i r c / 2^logN)
// first (logN > 0); complex64, or complex32 with h16.  rows and cols are
// multiples of 32.
cudaError_t launch_transpose(const void* in, void* out, int64_t batch, int64_t rows, int64_t cols,
                             int logN, int sign, int h16, int sm_count, cudaStream_t st);

// The short-line kernel of a contiguous pass of 2^logL points (lines.cu): sets
// fn, block and smem; false if there is none.
bool resolve_lines(int logL, PassLaunch* l);
// The same for the column pass of frames of 2^logL rows (lines.cu).
bool resolve_cols(int logL, PassLaunch* l);
// The same for fast convolution (conv_lines.cu): contiguous lines, and the
// columns of frames.
bool resolve_conv_lines(int logL, PassLaunch* l);
bool resolve_conv_cols(int logL, PassLaunch* l);

// Per-kernel attributes a launch needs (opt-in shared memory); call once after
// resolving, before the first launch_pass.
cudaError_t prepare_launch(PassLaunch& p);

cudaError_t launch_pass(const PassLaunch& p, const void* in, void* out, cudaStream_t st);
cudaError_t occupancy(const PassLaunch& p, int* ctas_per_sm);
// Times one Stockham stage in isolation (see stage_bench).
cudaError_t launch_stage_bench(int R, const PassDesc& d, int Ns, int reps, int grid, int block,
                               size_t smem, void* sink, cudaStream_t st);
// One launch over the jobs of `gt` with the generic row kernel of R elements
// per thread; d0 is the pass descriptor of one job (tables, shape, strides).
cudaError_t launch_grouped(int R, const PassDesc& d0, const GroupTable& gt, int grid, int block,
                           size_t smem, cudaStream_t st);
// The same for a pass of the short-line kernels (l.lines; GroupEntry::tiles count
// tiles of 2^l.lines elements).
cudaError_t launch_grouped_lines(const PassLaunch& l, const GroupTable& gt, cudaStream_t st);
cudaError_t launch_copy(const void* in, void* out, int64_t count, int64_t in_stride,
                        int64_t out_stride, cudaStream_t st);
// Twiddle tables (planner.h: TwSegment) at out + off, all in one launch.
struct TwiddleTable {
  int64_t off, count, den, mult;
  int mode, r;
};
struct TwiddleList {
  int n;
  TwiddleTable t[40];
};
cudaError_t launch_twiddle_list(void* out, const TwiddleList& list, cudaStream_t st);
cudaError_t launch_twiddle_gen(void* out, int64_t count, int64_t den, int mode, int r,
                               int64_t mult, cudaStream_t st);

}  // namespace gbfft
