// Internal declarations shared by the C-ABI layer (api.cpp) and the kernels.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "hh.h"
#include "zpair.h"

// FP16 storage scales a channel group by the smallest power of two that maps
// its largest |value| to at most this code (so to more than half of it), and
// every value down to ~7e-9 of the maximum is a normal half.
#define HH_FP16_CODE_MAX 16384.0f

// Volume layouts.
//  LINEAR: x fastest, element (k*ny + j)*nx + i (the export / interchange
//          layout).
//  ZPAIR: the grid with a one-voxel halo: voxel (i,j,k) sits at padded
//          coordinates (I,J,K) = (i+1, j+1, k+1), and the halo (0 or n+1 on
//          some axis) holds a copy of the nearest grid voxel, so a trilinear
//          sample clamped to the edge needs no index clamps. Two slices are
//          interleaved: element (K>>1)*pair + J*row + 2*I + (K&1). A cell then
//          needs one base element and one select (the step to the next slice);
//          the next row and the next column are constant strides. Against 2x2x2
//          bricks (a select per axis, an address per corner) the march of a
//          256^3 FP32 1080p frame at h_max takes 330 instead of 359 us, of a
//          384^3 FP16 4K view 1657 instead of 1883; a plain x-fastest order
//          takes 333 and 1604, but its lines of eight voxels in a row spread a
//          cell over more of them (32 views of a 512^3 FP16 volume: 11.1 ms
//          against 10.0, and 10.1 for the bricks).
//          The strides' residues spread a warp's corner load, the same corner
//          of 32 neighbouring cells, over the L1's bank groups and tag banks
//          (the start of the next row or pair of slices must not fold onto this
//          one's). Measured over paddings of 0 to 42 elements: pair = 2 (mod
//          16), and row = 6 (mod 8) on FP32 storage (1080p view of a dense 256^3
//          volume 365 us; 376 at 12 (mod 16), 470 at 8), 12 (mod 16) on FP16 (32
//          views of a 512^3 volume 9.13 ms against 9.15 to 9.60).
// zpair.h has the strides and the corner addresses.
enum { HH_LAYOUT_LINEAR = 0, HH_LAYOUT_ZPAIR = 1 };

struct hh_volume_s {
    int nx, ny, nz;
    int storage;        // hh_storage
    int layout;         // HH_LAYOUT_*
    unsigned row, pair; // ZPAIR strides (elements)
    float h_kernel;
    void* data;         // float4 (FP32) or ushort4 of halves (FP16) per voxel
    size_t bytes;       // the packed field's bytes as reported: grid and halo, axes padded to even
    // ZPAIR: the free-corner mask and its build scratch follow the data in the
    // same allocation. free_dev: one bit per element in the layout's own order
    // (bit b & 31 of word b >> 5 for element b), set when the element's voxel
    // and its +1 neighbours on each axis hold no stored nonzero value, so that
    // a sample whose first corner is that voxel reads eight zeros. nz_dev: one
    // bit per grid column i, padded row J and slice K (bit i & 31 of word (K *
    // rows + J) * nz_words + (i >> 5), rows = ny + 2 rounded up to even), set
    // when the voxel holds a nonzero value. sparse_dev: nonzero when the mask is
    // worth testing (see free_mask_kernel). Null for LINEAR volumes.
    size_t mask_off;    // bytes from data to free_dev
    unsigned nz_words;
    unsigned* free_dev;
    unsigned* nz_dev;
    unsigned* sparse_dev;
    float* scales_dev;  // [2] = {s_n, s_g} on the device (1, 1 for FP32)
    unsigned* max_dev;  // [2] = bit patterns of max|dn|, max|g| (FP16 build)
    float* rho_dev;     // density scratch for particle builds (nullable)
    float4* sorted_dev; // particles binned by cell, for grids larger than L2 (nullable)
    int64_t sorted_cap; // particles sorted_dev holds
    unsigned* bins_dev; // 2 x bin count counters of the binning (nullable)
    int n_bins;         // bins of bins_dev
    int device;
};

namespace hh {

extern std::atomic<uint64_t> g_launches;

inline void count_launch(uint64_t n = 1) { g_launches.fetch_add(n, std::memory_order_relaxed); }

// Error reporting shared by the C-ABI entry points (defined in api.cpp): set
// the calling thread's hh_last_error() message and return the status.
hh_status fail(hh_status st, const char* fmt, ...);
hh_status cuda_fail(cudaError_t e, const char* what);
hh_status ok();

// Device (cudaMalloc) and pinned host (cudaMallocHost) allocations of the
// library, counted; HH_FAIL_ALLOC_AT=k fails the k-th one (defined in
// api.cpp). The free functions accept NULL.
cudaError_t dev_alloc(void** p, size_t bytes);
void dev_free(void* p);
cudaError_t host_alloc(void** p, size_t bytes);
void host_free(void* p);
int64_t live_allocations();

// Argument checks shared by the trace entry points (defined in api.cpp).
hh_status check_params(const hh_step_params* P);
hh_status check_camera(const hh_camera& c, int i);
hh_status check_background(const hh_background* bg);

// Launches a kernel of a build-and-march chain (zero, splat, field, mask,
// march) as a programmatic dependent of the one before it in the stream: its
// blocks may take their places while that one, all of whose blocks have called
// release_next() or ended, is still running, and wait in await_previous() until
// it has completed and its writes are visible. It hides the launch and the start of
// the blocks: 1 to 3 us a launch (build of 16,384 particles on 96^3 30.3 against
// 23.6 us, of 262,144 on 256^3 170 against 161, on FP16 194.6 against 183.7;
// allocation-free build on 128^3 46.0 against 39.9). A kernel launched so calls
// await_previous() before it touches memory that the stream's earlier work may
// have written or may still read, and at least one of its threads always does:
// then its completion implies theirs. After anything but such a kernel the
// launch is an ordinary one.
template <typename... P, typename... A>
void launch_next(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t s, A... args) {
    cudaLaunchConfig_t config = {};
    config.gridDim = grid;
    config.blockDim = block;
    config.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    config.attrs = attr;
    config.numAttrs = 1;
    cudaLaunchKernelEx(&config, kernel, static_cast<P>(args)...);
}

#ifdef __CUDACC__
__device__ __forceinline__ void await_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
// The next kernel in the stream may start once every block has called this.
__device__ __forceinline__ void release_next() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// p, for loads that the compiler must not move above await_previous() (it may
// move a read-only load past anything that p does not depend on).
template <typename T>
__device__ __forceinline__ T* after_wait(T* p) {
    asm volatile("" : "+l"(p) :: "memory");
    return p;
}
#endif

// Kernel launchers. Each returns the launch status (cudaGetLastError()).
// launch_splat also clears the two words at max_bits (nullable), for the field
// pass of an FP16 volume that follows.
cudaError_t launch_splat(const float4* xyzm, int64_t n, int nx, int ny, int nz, float h,
                         float* rho, unsigned* max_bits, cudaStream_t s);

// Counting sort of particles by cubic cell (splat_bin_count bins, x-fastest)
// into `sorted` (n float4), using `bins` (2 x splat_bin_count unsigned) as
// counters; the splat of the sorted copy keeps its reductions within a few
// cells at a time.
int splat_bin_count(int nx, int ny, int nz);
cudaError_t launch_bin_particles(const float4* xyzm, int64_t n, int nx, int ny, int nz,
                                 unsigned* bins, float4* sorted, cudaStream_t s);

// max_clear: the volume's max_dev is zero (launch_splat cleared it).
cudaError_t launch_field(const float* rho, int nx, int ny, int nz, float K, hh_volume_s* vol,
                         bool max_clear, cudaStream_t s);

cudaError_t launch_export(const hh_volume_s* vol, float4* dst, cudaStream_t s);

// View records for a caller-managed device view table (the server's jobs):
// build_view_table fills n records of view_record_bytes() each in host memory
// for tile width tile_w and returns the total tile count (-1 if too many).
size_t view_record_bytes();
int build_view_table(const hh_camera* cams, const hh_view_out* outs, int n, int tile_w,
                     void* host_records);

// The render server's persistent worker (ray-level continuous batching).
// The host publishes requests ("jobs") into a device queue while the worker
// runs; its warps take 32-pixel tiles of the oldest job that still has some,
// and the warp that finishes a job's last tile raises the job's flag in
// host-mapped memory. Jobs are numbered from 0 since the queue's last reset;
// the host resets the queue only while no worker runs.
struct ServeJob {
    const void* vol;      // the frame's volume data (ZPAIR)
    const float* scales;  // its FP16 scales on the device
    const unsigned* sparse;  // whether its free-corner mask is worth testing
    int view_begin;       // first record of the job in the view table
    int n_views;
    int n_tiles;          // tiles of all its views (view tile_begin is job-relative)
    int seq;              // the job's number; a slot holding another number is not written yet
};

// Exit reasons of a worker launch (host_ctl[1]).
enum { HH_WORKER_IDLE = 1, HH_WORKER_STOPPED = 2 };
// Values of a job's host flag.
enum { HH_JOB_DONE = 1, HH_JOB_FAILED = 2 };

struct ServeWorkerArgs {
    const ServeJob* jobs;       // job table (device)
    const void* views;          // view records (device), view_record_bytes() apart
    unsigned* claimed;          // per job: tiles handed out (from HH_JOB_CLAIM_FAILED up: failed)
    unsigned* done;             // per job: tiles finished
    const int* n_jobs;          // jobs published (device; written by host copies)
    int* first_open;            // lowest job that may still have tiles to hand out
    const int* stop;            // non-zero: leave when idle (device; written by a host copy)
    int* idle_warps;            // warps of this launch that count themselves idle
    int* leave;                 // set once every started warp is idle: the launch leaves
    int* started_warps;         // warps of this launch that have started (all three zeroed per launch)
    volatile unsigned* host_done;  // per job, host-mapped: HH_JOB_DONE / HH_JOB_FAILED
    volatile int* host_ctl;     // host-mapped: [1] exit reason
    int tile_w;
    unsigned long long idle_ns;   // a warp leaves after this long with an empty queue
    unsigned long long entry_ns;  // a published job's entry missing this long fails it
};
// A failed job's claim counter is ORed with this bit: every later claim then
// reads as beyond the job's tiles (jobs hold fewer than 2^30 tiles, and fewer
// than 2^31 claims follow).
#define HH_JOB_CLAIM_FAILED 0x80000000u

// Resident blocks per SM of the worker for a launch shape, and its launch
// (VolArgs from `like`: dims, storage, schedule, background; the volume data
// and scales come from each job).
int serve_worker_blocks_per_sm(const hh_volume_s* like, const hh_step_params& P, int threads);
cudaError_t launch_serve_worker(const hh_volume_s* like, const hh_step_params& P,
                                const hh_background& bg, const ServeWorkerArgs& W, int blocks,
                                int threads, cudaStream_t s);

cudaError_t launch_trace(const hh_volume_s* vol, const hh_camera& cam,
                         const hh_step_params& P, const hh_background& bg,
                         const hh_view_out& out, cudaStream_t s);

}  // namespace hh
