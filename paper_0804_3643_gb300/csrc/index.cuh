// index.cuh -- launchers of the stage-0 and translation kernels (index.cu).
#pragma once
#include "common.cuh"

namespace plast {

cudaError_t launch_check_codes(const int8_t* codes, int64_t n, int hi, int* bad, cudaStream_t st);
// Codes into the sentinel-filled padded bank, checked against [0, hi].
cudaError_t launch_build_pad(const int8_t* codes, const int64_t* seq_off, int32_t n_seqs, int64_t n_res, int hi,
                             int8_t* pad, int* bad, cudaStream_t st);
// Stage-0 index as a counting sort in two digits of the key (index.cu): the
// padded bank in chunks of 8192 positions, `group` chunks a group.
struct IndexShape {
  int64_t n_chunks, n_groups, group;
  int64_t per;  // chunks a CTA counts; divides group
};
IndexShape index_shape(int64_t n_pad);     // n_pad > 0
int64_t index_cells(const IndexShape& sh); // of the count tables; off: their exclusive scan
cudaError_t launch_index_hist(const int8_t* pad, int64_t n_pad, const IndexShape& sh, int32_t* hist,
                              cudaStream_t st);
cudaError_t launch_index_key_off(const int64_t* off, const IndexShape& sh, int64_t* key_off, cudaStream_t st);
// by_pos, by_lo: room for every word (at most one per residue)
cudaError_t launch_index_split(const int8_t* pad, int64_t n_pad, const IndexShape& sh, const int64_t* off,
                               uint32_t* by_pos, uint8_t* by_lo, cudaStream_t st);
cudaError_t launch_index_fill(const int8_t* pad, const IndexShape& sh, const int64_t* off, const uint32_t* by_pos,
                              const uint8_t* by_lo, uint32_t* pos, int8_t* nb, cudaStream_t st);
// blk[i] = the sequence at padded position i * SEQ_BLK, i <= n_pad / SEQ_BLK
cudaError_t launch_block_seq(const int64_t* pad_off, int32_t n_seqs, int64_t n_pad, int32_t* blk, cudaStream_t st);
cudaError_t launch_export_pos(const uint32_t* pos, int64_t n, const int64_t* pad_off, int32_t n_seqs, int32_t* out,
                              cudaStream_t st);
cudaError_t launch_translate6(const uint8_t* dna, const int64_t* contig_off, int32_t n_contigs, const int64_t* seq_off,
                              int64_t n_aa, int8_t* aa, cudaStream_t st);

}  // namespace plast
