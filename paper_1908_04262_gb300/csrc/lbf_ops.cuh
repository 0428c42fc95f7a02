// lbf_ops.cuh -- launch layer: one Ops object per (lattice, storage) pair
// turns the host runtime's requests into kernel launches on a stream.
#pragma once
#include <cuda_runtime.h>

#include "lbf_common.cuh"
#include "lbf_ops_api.h"
#include "lbf_convert.cuh"
#include "lbf_geom.cuh"
#include "lbf_label.cuh"
#include "lbf_mlp_kappa.cuh"
#include "lbf_stream.cuh"

namespace lbf {

inline unsigned blocks_for(long long n, int b) { return (unsigned)((n + b - 1) / b); }

// full-lattice launches: blocks of B threads along x, one block row per (y, z)
inline int row_block(const Params &p) { return p.nx >= 96 ? 128 : (p.nx > 32 ? 64 : 32); }
inline dim3 row_grid(const Params &p) {
  const int b = row_block(p);
  return dim3((unsigned)((p.nx + b - 1) / b), (unsigned)p.ny, (unsigned)p.nz);
}

template <int D, class S>
struct OpsImpl final : Ops {
  using R = typename ST<S>::R;
  static constexpr int B = 256;

  // the root sort holds up to 16384 roots (64 KB) in shared memory
  OpsImpl() { cudaFuncSetAttribute(k_sort_roots, cudaFuncAttributeMaxDynamicSharedMemorySize, 16384 * (int)sizeof(int)); }

  void init_fill(const Params &p, int par, double h, cudaStream_t s) override {
    k_init_fill<D, S><<<row_grid(p), row_block(p), 0, s>>>(p, par, h);
  }
  void init_cells(const Params &p, int par, const uint8_t *t, const double *rho, const double *u,
                  const double *a, const double *c, cudaStream_t s) override {
    k_init_cells<D, S><<<row_grid(p), row_block(p), 0, s>>>(p, par, t, rho, u, a, c);
  }
  void separate(const Params &p, int par, cudaStream_t s) override {
    k_separate_mark<D><<<row_grid(p), row_block(p), 0, s>>>(p);
    k_separate_apply<D, S><<<row_grid(p), row_block(p), 0, s>>>(p, par);
  }
  void nearwall(const Params &p, cudaStream_t s) override { k_nearwall<D><<<row_grid(p), row_block(p), 0, s>>>(p); }
  void nucleate(const Params &p, int par, const double *c, double R0, cudaStream_t s) override {
    const int x0 = (int)floor(c[0] - R0 - 1.0), x1 = (int)ceil(c[0] + R0 + 1.0);
    const int y0 = (int)floor(c[1] - R0 - 1.0), y1 = (int)ceil(c[1] + R0 + 1.0);
    const int z0 = D == 3 ? (int)floor(c[2] - R0 - 1.0) : 0, z1 = D == 3 ? (int)ceil(c[2] + R0 + 1.0) : 0;
    const int bx = x1 - x0 + 1, by = y1 - y0 + 1, bz = z1 - z0 + 1;
    const long long cnt = (long long)bx * by * bz;
    k_nucleate<D, S><<<blocks_for(cnt, B), B, 0, s>>>(p, par, c[0], c[1], D == 3 ? c[2] : 0.0, R0, x0, y0,
                                                        z0, bx, by, bz);
  }
  // whether a grid of so many blocks (four warps each) could meet a list long
  // enough to be packed (see for_segment_cells)
  template <bool EARLY> static bool packs(const Params &p, int blocks) {
    return segs_pack<EARLY>((long long)((p.nx + 31) / 32) * p.ny * p.nz, 4ll * blocks);
  }
  template <bool WALLED, int SEGS> void exchange_as(const Params &p, int par, cudaStream_t s) {
    par ? k_exchange<D, S, 1, WALLED, SEGS><<<p.warp_blocks, 128, 0, s>>>(p)
        : k_exchange<D, S, 0, WALLED, SEGS><<<p.warp_blocks, 128, 0, s>>>(p);
  }
  template <bool WALLED> void exchange_walled(const Params &p, int par, cudaStream_t s) {
    if constexpr (sizeof(S) >= 4)
      exchange_as<WALLED, SEGS_TWO>(p, par, s);
    else if (packs<true>(p, p.warp_blocks))
      exchange_as<WALLED, SEGS_ONE>(p, par, s);
    else
      exchange_as<WALLED, SEGS_SINGLE>(p, par, s);
  }
  void exchange(const Params &p, int par, cudaStream_t s) override {
    p.walled ? exchange_walled<true>(p, par, s) : exchange_walled<false>(p, par, s);
  }
  void build_ilist(const Params &p, cudaStream_t s) override {
    cudaMemsetAsync(p.icount, 0, sizeof(int), s);
    cudaMemsetAsync(p.segcount, 0, sizeof(int), s);
    k_build_ilist<<<row_grid(p), row_block(p), 0, s>>>(p);
  }
  // (the collision model is a template parameter: the BGK sweep keeps its
  // registers)
  void stream_liquid(const Params &p, int par, cudaStream_t s) override {
    const dim3 g = row_grid(p);
    const int b = row_block(p);
    if (p.coll == 2)
      par ? k_stream_liquid<D, S, 1, 2><<<g, b, 0, s>>>(p) : k_stream_liquid<D, S, 0, 2><<<g, b, 0, s>>>(p);
    else if (p.coll == 1)
      par ? k_stream_liquid<D, S, 1, 1><<<g, b, 0, s>>>(p) : k_stream_liquid<D, S, 0, 1><<<g, b, 0, s>>>(p);
    else if (p.walled)
      par ? k_stream_liquid<D, S, 1, 0, true><<<g, b, 0, s>>>(p)
          : k_stream_liquid<D, S, 0, 0, true><<<g, b, 0, s>>>(p);
    else
      par ? k_stream_liquid<D, S, 1, 0><<<g, b, 0, s>>>(p) : k_stream_liquid<D, S, 0, 0><<<g, b, 0, s>>>(p);
  }
  template <int COLL, bool WALLED, int SEGS> void interface_segs(const Params &p, int par, cudaStream_t s) {
    par ? k_stream_interface<D, S, 1, COLL, WALLED, SEGS><<<p.list_blocks, 128, 0, s>>>(p)
        : k_stream_interface<D, S, 0, COLL, WALLED, SEGS><<<p.list_blocks, 128, 0, s>>>(p);
  }
  template <int COLL, bool WALLED> void interface_as(const Params &p, int par, cudaStream_t s) {
    if constexpr (sizeof(S) >= 4)
      interface_segs<COLL, WALLED, SEGS_TWO>(p, par, s);
    else if (packs<sizeof(S) == 8>(p, p.list_blocks))
      interface_segs<COLL, WALLED, SEGS_ONE>(p, par, s);
    else
      interface_segs<COLL, WALLED, SEGS_SINGLE>(p, par, s);
  }
  void stream_interface(const Params &p, int par, cudaStream_t s) override {
    if (p.coll == 2)
      interface_as<2, false>(p, par, s);
    else if (p.coll == 1)
      interface_as<1, false>(p, par, s);
    else if (p.walled)
      interface_as<0, true>(p, par, s);
    else
      interface_as<0, false>(p, par, s);
  }
  void convert_mark(const Params &p, cudaStream_t s) override { k_conv_mark<D><<<p.list_blocks, 128, 0, s>>>(p); }
  void convert_excess(const Params &p, int par, cudaStream_t s) override {
    const int post = 1 - par;
    k_conv_compute<D, S><<<p.list_blocks, 128, 0, s>>>(p, post);
    k_conv_apply<D, S><<<p.list_blocks, 128, 0, s>>>(p, post);
  }
  void convert_finalize(const Params &p, cudaStream_t s) override {
    k_conv_finalize<D><<<p.list_blocks, 128, 0, s>>>(p);
  }
  void label_prep(const Params &p, cudaStream_t s) override {
    k_label_prep<<<blocks_for(p.cap, B), B, 0, s>>>(p);
  }
  void label_forest(const Params &p, cudaStream_t s) override {
    const dim3 tg((unsigned)((p.nx + Tile<D>::TX - 1) / Tile<D>::TX), (unsigned)((p.ny + Tile<D>::TY - 1) / Tile<D>::TY),
                  (unsigned)((p.nz + Tile<D>::TZ - 1) / Tile<D>::TZ));
    // tile loops on a grid of two or four blocks per SM (a block of the
    // graph's patch steps then costs one short wave)
    const unsigned ntiles = tg.x * tg.y * tg.z;
    const unsigned two = p.tile_blocks > 0 ? (unsigned)p.tile_blocks : ntiles;
    const unsigned gm = two < ntiles ? two : ntiles, g = 2 * two < ntiles ? 2 * two : ntiles;
    k_uf_local<D><<<g, TILE_THREADS, 0, s>>>(p);
    k_uf_merge<D><<<gm, MERGE_THREADS, 0, s>>>(p);
    k_uf_compress<D><<<g, TILE_THREADS, 0, s>>>(p);
    int P = 1;
    while (P < p.cap) P <<= 1;
    k_sort_roots<<<1, 1024, P * sizeof(int), s>>>(p);
  }
  void label_relabel(const Params &p, cudaStream_t s) override {
    // four blocks per SM for the patch's short lists; the full relabelling
    // walks every segment of the lattice with them (carving a nucleus, which
    // labels in full: 256^3 1.00 ms a call, 128^3 0.30; with 16 blocks per SM
    // 1.01 and 0.30)
    k_relabel<D, R><<<p.list_blocks, 128, 0, s>>>(p);
  }
  void bubble_update(const Params &p, cudaStream_t s) override { k_bubble_update<<<1, 1024, 0, s>>>(p); }
  void label_check(const Params &p, cudaStream_t s) override {
    k_label_check<D><<<p.list_blocks, 128, 0, s>>>(p);
    k_root_scan<D><<<SCAN_BLOCKS, SCAN_THREADS, 0, s>>>(p);
  }
  void label_sync(const Params &p, cudaStream_t s) override { k_label_sync<<<p.list_blocks, 128, 0, s>>>(p); }
  void geometry(const Params &p, cudaStream_t s) override {
    k_geometry<D, R><<<p.warp_blocks, 128, 0, s>>>(p);
    if (p.kappa_hf) k_hf_kappa<D, R><<<p.list_blocks, 128, 0, s>>>(p);
  }
  void mlp_kappa(const Params &p, const void *img, cudaStream_t s) override {
    // up to two CTAs of 128 cells per SM (list_blocks holds 4 per SM);
    // each holds 128 of the SM's 512 tensor-memory columns, and no more
    // than four fit on an SM by their shared memory
    if constexpr (D == 3 && sizeof(R) == 8)
      mlp_kappa_f64(p, img, p.list_blocks / 2, s);
    else if (D == 3)
      k_mlp_kappa<D, R><<<p.list_blocks / 2, MLP_THREADS, sizeof(tc::Tile), s>>>(p, (const tc::Image *)img);
  }
  void mlp_harvest(const Params &p, float *x, float *y, int *cells, int cap, int *count, cudaStream_t s) override {
    if (D == 3) k_mlp_harvest<D, R><<<p.warp_blocks, 128, 0, s>>>(p, x, y, cells, cap, count);
  }
  void disjoining(const Params &p, cudaStream_t s) override {
    k_disjoining<D, R><<<p.list_blocks, 128, 0, s>>>(p);
  }
  void rank(const Params &p, cudaStream_t s) override {
    k_rank<<<blocks_for(p.cap, RANK_THREADS), RANK_THREADS, 0, s>>>(p.told.root, p.told.count, p.rank);
  }
  void fields(const Params &p, int par, unsigned mask, void *const (&out)[11], int dtype, cudaStream_t s) override {
    FieldPtrs f;
    for (int k = 0; k < 11; ++k) f.p[k] = out[k];
    if (mask >> FLD_LABEL & 1u) rank(p, s);
    k_fields<D, S><<<row_grid(p), row_block(p), 0, s>>>(p, par, mask, f, dtype);
  }
  void ledger(const Params &p, int par, double *acc, unsigned long long *counts, cudaStream_t s) override {
    k_ledger<D, S><<<row_grid(p), row_block(p), 0, s>>>(p, par, acc, counts);
  }
};

}  // namespace lbf
