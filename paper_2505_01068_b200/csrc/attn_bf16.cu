// bf16 IM attention for sm_100a: TMA-fed, register-resident online softmax on mma.sync tiles.
//
// Decomposition (paper, Section "Inner Decomposition for Efficiency"): a CTA owns one tile of query
// rows of one modality segment of one sample and walks only the key tiles of the segment(s) the
// Interlaced Mask opens for that block row, and only up to the sample's valid length.  Closed blocks
// and padded keys are never loaded, multiplied or exponentiated.
//
// Layout: a CTA covers a column slice of CW features (= CW/HD heads) so that one TMA box row is a whole
// 128-byte (or 64/32-byte) line shared by all heads of the slice; warp w works on head (w % G).  With
// head_dim 8 the tensor-core shapes fit exactly: S = Q K^T is mma.m16n8k8 (K = head_dim) and O += P V is
// mma.m16n8k16 (N = head_dim); the score accumulators are reused in registers as the A operand of P V.
#include "attn_bf16_tile.cuh"
#include "attn_bf16_kernel.cuh"
#include "attn_bf16_host.cuh"
