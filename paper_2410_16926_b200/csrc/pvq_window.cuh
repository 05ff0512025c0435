// Windowed tables for wide codes (pvq_decode_window.cu, pvq_encode_window.cu): layout and host interface.
//
// As in SearchLayout, with q = N(n+1,k) - r the coordinate of a position (n dimensions behind it) follows
// from where q falls among the thresholds T_n[2k'] = N(n+1,k'), T_n[2k'+1] = N(n+1,k') + N(n,k'), and the next
// position's q is q + E_n[m], E_n[m] = N(n,k') - T_n[m].  A table of all thresholds of all rows is too large for
// shared memory when codes are wide.  But the pulses k' left after a position hardly ever stray far
// from their mean: a row keeps only the window klo..khi outside of which no more than a share eps of all
// codes lies on either side.  A path that leaves the window somewhere is found out (see `last` below); those
// positions are searched in the count table's sections in global memory.
//
// Rows are taken in blocks of four positions.  A block's numbers are kept left-aligned: multiplied by the power
// of two that brings the largest q of the block to the top of its `words` 32-bit words.  The top two words
// (three from N = 128 on, whose windows span more than 56 bits) then hold the leading bits of q whatever the row;
// as an fp32, truncated, they are the key that numbers a bucket.  From one block to the next q is shifted left by `delta` bits.
//
// Block b in memory (block_off[b], a multiple of 16 bytes):
//     head     four 16-byte records (WinRow), one a row; then four words: klo of the position before minus klo of the
//              position, a byte each (first position lowest); delta; klo and khi - klo, a byte each (first
//              position highest, as the encoder's points are packed)
//     E        four rows, each `words` planes of `plane` 32-bit words: word w (lowest first) of
//              entry m - 2 klo of the row, modulo 2^(32 words)
//     buckets  four tables, 4 bytes a bucket, indexed by the key relative to `base` (its low 24 bits are c, the rest
//              is the same for the whole bucket).  With m0 the local index of the first threshold that a q of the bucket
//              can be at or below, and c0 that threshold's c if it lies in the bucket (else all ones): the entry is what added
//              to the relative key leaves m0 in the top byte, plus one iff c > c0, and all ones in the other
//              three iff c = c0.  The last entry of a table catches every key outside the window (relative
//              keys are cut off at `last`): it leaves 255, which makes the pulses left grow, and that is
//              seen.  (The read of E at 255 stays within the block.)
#pragma once
#include <memory>

#include "pvq_internal.cuh"

namespace pvq {

constexpr int kWinRows = 256, kWinBlocks = kWinRows / 4, kWinWords = 24;

__host__ __device__ constexpr int win_key_words(int N) { return N > 64 ? 3 : 2; }

struct WinRow {
    uint32_t base;     // key of the first bucket's start
    uint32_t last;     // relative key of the entry for keys outside the window
    uint32_t shift;    // relative key >> shift is the bucket
    uint32_t buckets;  // byte offset of the row's bucket table in its block
};
constexpr uint32_t kWinHead = 96;  // bytes of a block's head
constexpr uint32_t kWinDlo4 = 64, kWinDelta = 68, kWinKlo4 = 72, kWinWidth4 = 76;

struct WinArgs {
    const uint8_t* data;
    const uint8_t* thr;                  // thresholds (aligned), laid out like E; read when key bits are the same
    uint32_t block_off[kWinBlocks + 1];  // the last one: bytes in all
    uint32_t thr_off[kWinBlocks];
    uint8_t up[kWinBlocks];              // bits by which its numbers are multiplied
    uint8_t words[kWinBlocks];
    uint8_t blocks_of[33];               // blocks_of[w]: blocks done in w words or more
    int16_t klo[kWinRows];
    uint32_t typical[kWinWords];                // q of a code whose path stays in the middle of the windows
};

struct WinTables {
    WinArgs args;
    int plane;           // entries of a plane: 96 (N = 64, tables that fit shared memory) or 192 (others), 160 (N = 128, 256)
    uint32_t max_block;  // bytes of the largest block
    uint32_t max_rows;   // ... of its head and its four rows of E
};

// Bytes of a block's head and E, which is all that the encoder reads.
__host__ __device__ constexpr uint32_t win_rows_bytes(int words, int plane) { return kWinHead + 16u * words * plane; }

// The settings with windowed kernels: codes of 5 to 8 words at group size 64, 9 to 12 at 128, 24 at 256 (decoding only).
// Those are the widths up to 4 direction bits a value at N = 64 and 3 at N = 128 and 256 that workloads here have; the
// tables suit others too (with up to 255 pulses, or 160 thresholds a row), but every width is kernels of its own.
constexpr bool has_window_tables(int N, int W, int K) {
    return (N == 64 && W >= 5 && W <= 8 && K <= 255) || (N == 128 && W >= 9 && W <= 12 && K <= 255) || (N == 256 && W == 24);
}

// The tables for (N,K) on the current device for a launch on `stream`, or null (never built here, or no such kernel).
// They stay while the holder is held (until the launch is enqueued: freeing waits for the kernels that read them), and
// for good once they have been handed out for a launch that a stream capture records.
std::shared_ptr<const WinTables> window_tables(int N, int K, cudaStream_t stream);
// Builds them, once per device and (N,K): called when a count table is built, off the hot path.  The tables of at most
// kWinKept (N,K) are kept per device; for one more the oldest that no capture has used are freed, by the thread that builds.
// Failing to build (all are in captures, no memory) is not an error: the calls take the kernels without.
constexpr int kWinKept = 8;
void build_window_tables(int N, int K, cudaStream_t stream);

// PVQ_ERR_UNSUPPORTED: no tables or no kernel for it; the caller walks
int launch_decode_window(const BatchArgs& args, int N, int W, cudaStream_t stream);
int launch_encode_window(const BatchArgs& args, int dtype, int N, int W, cudaStream_t stream);

}  // namespace pvq
