// sf_seqscan.h -- the S = 1 path by sorts and scans (sf_seqscan.cu).
#pragma once

#include "sf_internal.h"

namespace sfk {

// Updates per launch; a sketch eligible for the path keeps a workspace for one piece in its scratch.
constexpr uint32_t kSeqPiece = 131072;
// Narrower sketches run the one-warp window kernel (sf_seq.cu) and need no workspace.
constexpr uint32_t kSeqScanMinW = 1024;
// Calls of at most two 32-update windows run the window kernel too: 16.5 us for 32 updates and 24.7 for 64,
// a tenth of them deletions, against 32.9 and 31.9 here; at 100 it is 43 against 35, and grows by 0.27 us
// an update (d = 4, w = 4,096, z = 16).
constexpr uint32_t kSeqScanMinN = 64;
// Control word counting the blocks that have left the launch (the last one resets the barrier).
constexpr uint32_t kCtrlSeqDone = 4;

// A Fat counter's index in its row is a 32-bit sort key.
inline bool seq_scan_eligible(uint32_t w, uint32_t z) { return w >= kSeqScanMinW && (uint64_t)w * z < (1ull << 32); }

uint64_t seq_scan_workspace_bytes(uint32_t d);

// Any mix of insertions and deletions, one at a time: keys and ops as in SeqArgs, ws a workspace of
// seq_scan_workspace_bytes(d) bytes (16-byte aligned), ctrl the sketch's control words.
cudaError_t launch_seq_scan(const SketchDesc& s, const uint8_t* keys, const int8_t* ops, int32_t op_const, uint64_t n,
                            void* ws, uint32_t* ctrl, int num_sms, cudaStream_t st);

}  // namespace sfk
