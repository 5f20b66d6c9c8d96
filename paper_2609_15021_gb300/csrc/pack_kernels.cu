// pack_kernels.cu -- gather (pack) and scatter (unpack) kernels between the
// paged KV pool and packed chunks, for sm_103a.
//
// Paper Sec. 3.2: storing a prefix gathers its KV pages into the host tier's
// packed chunk, loading scatters the chunk back into freshly allocated pages.
// This is pure byte movement bound by memory bandwidth (HBM for device chunks
// and staging, the host link for mapped pinned chunks), so it runs on the
// load/store units with 16-byte vectors; no tensor cores are involved.
//
// Work unit: one batch, 4 KiB of one plane -- one (chunk, layer, K|V) -- handled
// by one warp, kInflight 16-byte vectors per lane; in large launches a few
// batches.  The chunk side of a
// plane is one contiguous extent in [token][head][row] order, so a unit is
// contiguous there whatever the page and row sizes are, and its vectors are
// found on the page side ([head][token] order for HND, [token][head] for NHD)
// one by one: vector -> row -> (token, head) -> page of the block table ->
// address.  A lane finds its first vector by divisions by launch constants
// (FastDiv) and the others by steps of 32 vectors, with carries.  A unit may
// start and end inside a row or a page and may span pages.
//
// Out-of-range block-table entries skip their vectors (a pack writes zeros)
// and lower a device error word (atomicMin of the logical block index);
// nothing traps.

#include <algorithm>

#include "copy16.cuh"
#include "kvx_internal.h"

namespace kvx {
namespace {

constexpr int kBatchVectors = 32 * kInflight;  // 4 KiB
// Where HBM bounds a launch of more batches than this (32 MiB, about two for
// each warp the GPU holds), a unit is two batches.  Packing 1 GB of 16-token
// pages with one head of 256-byte rows took 337 us with units of one batch, 322
// of two, 333 of four; with 8 heads 316, 300 and 306; packing 4 MB 9, 9 and 13 us.
constexpr int64_t kBatchesApart = 8192;
// Taken from a queue, a unit is up to 4 batches as long as every warp gets 24
// units, and 8 where every warp gets 64 of these (the last units end apart).  A
// 32k-token restore of the 27B shape (8.3 GB) takes 39,377 us with 8, 39,391 with
// 4, 39,430 with 1 and 39,419 with 32; storing 400 MB 2,095 us with 4, 2,097 with 8
// and 2,110 with 32, one chunk (65 MB) 342 us with 1, 344 with 4, 346 with 8.
constexpr int64_t kQueueBatches = 4, kQueueUnits = 24;
constexpr int64_t kLargeBatches = 8, kLargeUnits = 64;

__device__ __forceinline__ uint32_t div_by(uint32_t n, const FastDiv& f) {
  return f.d == 1 ? n : (uint32_t)__umul64hi(f.m, n);
}
__device__ __forceinline__ uint64_t div_by(uint64_t n, const FastDiv& f) {
  return n >> 32 ? n / f.d : div_by((uint32_t)n, f);
}

// What bounds it: the host link where the chunks are mapped host memory, HBM
// where they are in device memory; either needs enough loads on their way.
// Over the link a launch runs on some of the SMs, and these get unequal shares of
// the link: which SMs they are, and so which CTAs fall behind, differs from one
// GPU to another.  With units dealt out in advance a 1 GB restore took 4850 us
// or up to 4955 (a store 5295 or up to 5370), depending on the GPU and the
// number of CTAs; taking units from a queue it takes 4846 to 4849 (5294) on all
// of them, with 48 CTAs as with 96.
// Measured on GB300, launches back to back, 32 layers, 16-token HND pages, 8 heads
// of head_dim 128 bf16 unless stated; in brackets the same call when a unit was a
// page half, read row by row (vector by vector where a row was no power of two):
//   restore over the link, 1 GB: 4736 us (4741); head_dim 96, 256 MB: 1217 us
//     (1331); one 128-byte head: 1223 us (1260)
//   restore, 4 MB: 24 us (28; head_dim 96: 24, 104); 1 MB: 8 us (17; 10, 57), since
//     4 KiB units put 256 warps on 1 MB where 32 of them made eight round trips each
//   store over the link, 1 GB: 5168 us (5169); head_dim 96, 256 MB: 1326 us (1492);
//     one 128-byte head: 1332 us (1414); 1 MB 9 us (8; head_dim 96: 10, 27)
//   pack / unpack in device memory, 1 GB: 297 / 296 us, 6.9 TB/s (305 / 307);
//     head_dim 96: 300 / 303 us (478 / 452); one 128-byte head: 350 / 357 (609 / 608)
//   the same of NHD pages, whose halves were straight copies (32 KiB unless stated;
//     the TMA engine takes them unless told not to), 16 MB: 8 / 8 us (9 / 9), 64 MB,
//     which L2 holds: 21 / 21 (19 / 19), 1 GB: 297 / 293 (305 / 305); halves of 8 KiB,
//     16 MB: 8 / 8 (6 / 6), 1 GB: 307 / 310 (307 / 304); of 128 KiB (this kernel's by
//     default), 16 MB: 8 / 8 (14 / 14), 64 MB: 21 / 21 (32 / 33), 1 GB: 295 / 293 (309 / 309)
// Dealt out in advance over the link a unit is one batch: units of eight took 4945
// us for the 1 GB restore and 5370 for the store, and equal shares of 26,368 B, so
// that a warp's last batch is not whole, 95 us for a 16 MB restore instead of 83.
// 80 registers, 3 CTAs per SM; at 64 it spills 48 bytes, and unpacking 1 GB into
// HBM takes 310 us.
// LINK, for launches over the host link: the page-side addresses of a batch are
// all worked out before its data is waited for.  The table entries are then on
// their way together with a restore's loads from the host, and a store's loads
// wait for one trip to the table, not for eight: restores of up to 80 MB take 0.5
// to 1 us less than with the addresses worked out vector by vector (in replayed
// graphs 4 MB 21.4 us against 22.4), stores 0 to 0.3.  A restore's addresses spill
// 80 bytes at 80 registers, which costs nothing over the link; with 96 it spills
// none, but a GEMM beside it keeps 2 to 3 % less of its rate.  In device memory other warps hide the
// trips, and spilling costs: unpacking 1 GB with one head 333 us against 313.
template <int DIR, bool LINK>
__global__ void __launch_bounds__(kThreads, 3) move_kernel(const __grid_constant__ MoveParams p) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t nwarps = gridDim.x * (kThreads / 32);
  uint32_t job_begin = 0;
  int j = 0;
  uint32_t u = (blockIdx.x * kThreads + threadIdx.x) >> 5;
  while (u < p.total_units) {
    uint32_t next = u;  // taken now, so that the answer is there when this unit is done
    if (p.units.taken && lane == 0) next = atomicAdd(p.units.taken, 1u) - p.units.base;
    while (u >= p.jobs[j].unit_end) {  // warp-uniform; units ascend per warp
      job_begin = p.jobs[j].unit_end;
      ++j;
    }
    const Job& J = p.jobs[j];
    const uint32_t plane = (u - job_begin) / J.units_per_plane;  // (layer - l0) * 2 + kv
    const uint64_t vectors = (uint64_t)J.tokens * p.H * p.by_row.d;  // of the plane
    const uint64_t first = (uint64_t)(u - job_begin - plane * J.units_per_plane) * p.unit_vectors + lane;
    // this lane's vectors: nv of them, 32 apart (none past the end of the plane)
    int nv = first >= vectors ? 0 : (int)(min((uint64_t)p.unit_vectors, vectors - first + 31) >> 5);
    uint8_t* ck = J.chunk + (plane * vectors + first) * 16;
    uint8_t* base = p.layer_base[J.l0 + (plane >> 1)] + (plane & 1 ? p.page_bytes >> 1 : 0);
    // place of the first vector: column of its row, head, token of its page, page
    // of its logical block, table entry
    const uint64_t row = div_by(first, p.by_row), tok = div_by(row, p.by_heads);
    const uint32_t page = div_by((uint32_t)tok, p.by_block), gp = J.first_sub + page;
    uint32_t col = (uint32_t)(first - row * p.by_row.d), h = (uint32_t)(row - tok * p.H);
    uint32_t sp = (uint32_t)tok - page * p.B, e = div_by(gp, p.by_group), sub = gp - e * p.ppb;
    const int32_t* entries = p.table + J.first_entry;
    uint32_t bad = ~0u;  // lowest entry out of range whose page begins in this lane's vectors
    for (; nv > 0; nv -= kInflight, ck += kInflight * 512) {
      uint4 data[kInflight];
      uint8_t* page_side[kInflight];  // null: no page to move to or from
      if (DIR == kUnpack) {
#pragma unroll
        for (int i = 0; i < kInflight; ++i)
          if (i < nv) data[i] = ld16(ck + i * 512);
      }
#pragma unroll
      for (int i = 0; i < kInflight; ++i) {
        if (i < nv) {
          const uint32_t entry = (uint32_t)__ldg(entries + e);
          const bool ok = entry < p.entries;
          const int64_t in_page = (int64_t)(h * p.head_step + sp * p.tok_step) * p.R + col * 16;
          uint8_t* pg = base + ((int64_t)entry * p.ppb + sub) * p.page_bytes + in_page;
          if (LINK) {
            page_side[i] = ok ? pg : nullptr;
          } else if (DIR == kPack) {
            data[i] = make_uint4(0, 0, 0, 0);
            if (ok) data[i] = ld16(pg);
          } else if (ok) {
            st16(pg, data[i]);
          }
          bad = !ok && in_page == 0 ? min(bad, e) : bad;
        }
        // 32 vectors on
        col += p.step_col;
        h += p.step_head;
        sp += p.step_tok;
        sub += p.step_sub;
        e += p.step_entry;
        if (col >= p.by_row.d) col -= p.by_row.d, ++h;
        if (h >= p.H) h -= p.H, ++sp;
        if (sp >= p.B) sp -= p.B, ++sub;
        if (sub >= p.ppb) sub -= p.ppb, ++e;
      }
      if (LINK) {
#pragma unroll
        for (int i = 0; i < kInflight; ++i) {
          if (DIR == kPack) data[i] = make_uint4(0, 0, 0, 0);
          if (i < nv && page_side[i]) {
            if (DIR == kPack)
              data[i] = ld16(page_side[i]);
            else
              st16(page_side[i], data[i]);
          }
        }
      }
      if (DIR == kPack) {
#pragma unroll
        for (int i = 0; i < kInflight; ++i)
          if (i < nv) st16(ck + i * 512, data[i]);
      }
    }
    // reported once for each plane, by the page's first vector
    if (bad != ~0u) atomicMin(p.err, (long long)(J.first_entry + bad));
    u = nwarps + (p.units.taken ? __shfl_sync(0xffffffffu, next, 0) : u);
  }
  if (!p.units.taken) return;
  __syncthreads();  // the warps of this CTA have taken their last units, and have the answers
  if (threadIdx.x == 0 && atomicAdd(p.units.taken + 1, 1u) - p.units.done_base == gridDim.x - 1)
    asm volatile("st.relaxed.sys.global.u32 [%0], %1;" ::"l"(p.units.done), "r"(p.units.ticket) : "memory");
}

using MoveKernel = void (*)(MoveParams);
MoveKernel kernel_of(int dir, bool link) {
  if (dir == kPack) return link ? move_kernel<kPack, true> : move_kernel<kPack, false>;
  return link ? move_kernel<kUnpack, true> : move_kernel<kUnpack, false>;
}

}  // namespace

int64_t cut_units(MoveParams* p, bool link, int64_t queue_warps) {
  const auto vectors = [p](const Job& J) { return (int64_t)J.tokens * p->H * p->by_row.d; };
  int64_t batches = 0;  // of the launch
  for (int32_t i = 0; i < p->n_jobs; ++i) batches += 2ll * p->jobs[i].nl * vectors(p->jobs[i]) / kBatchVectors;
  int64_t per_unit = !link && batches > kBatchesApart ? 2 : 1;
  if (queue_warps > 0) {
    per_unit = std::max<int64_t>(1, std::min(kQueueBatches, batches / (kQueueUnits * queue_warps)));
    if (batches >= kLargeBatches * kLargeUnits * queue_warps) per_unit = kLargeBatches;
  }
  p->unit_vectors = (uint32_t)(per_unit * kBatchVectors);
  p->total_units = 0;
  for (int32_t i = 0; i < p->n_jobs; ++i) {
    Job& J = p->jobs[i];
    J.units_per_plane = (int32_t)((vectors(J) + p->unit_vectors - 1) / p->unit_vectors);
    p->total_units += 2ll * J.nl * J.units_per_plane;
    J.unit_end = p->total_units;
  }
  constexpr int64_t kWarps = kThreads / 32;
  return (p->total_units + kWarps - 1) / kWarps;
}

cudaError_t launch_move(int dir, bool link, const MoveParams& p, int grid, cudaStream_t s) {
  kernel_of(dir, link)<<<grid, kThreads, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t load_move_kernels() {
  // cudaFuncGetAttributes makes CUDA load a kernel that lazy loading has not loaded yet
  cudaFuncAttributes a;
  for (int dir : {kPack, kUnpack})
    for (bool link : {false, true}) {
      const cudaError_t e = cudaFuncGetAttributes(&a, kernel_of(dir, link));
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

int link_ctas_per_sm(int dir) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel_of(dir, true), kThreads, 0) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return n > 0 ? n : 1;
}

}  // namespace kvx
