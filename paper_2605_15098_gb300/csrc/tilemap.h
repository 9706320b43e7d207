// A tile's gather as a few tensor copies.
//
// The tile's local qubits form runs of neighbouring physical bits.  The state
// is described to the copy engine as a dense array whose dimensions begin
// where a local run begins: dimension i holds the index bits from run i up to
// the next run, the local run lowest, so a box that takes the whole run in
// every dimension is the tile, in the order of its slots (ascending physical
// bit), and the tile's global bits are the box's coordinates.  Five
// dimensions hold the five lowest runs; the bits of any further run are the
// tile's highest slots, so each of their values is one copy of its own into
// its own part of the tile.
#pragma once

#include <cuda.h>

#include <cstdint>

#include "common.h"

namespace sv {

constexpr int kTileDims = 5;

// The box coordinates and the copies of one tile, in 8-byte words (a
// complex128 amplitude is two words: word bit 0 is a local bit).
struct TileBox {
    int8_t pos[kTileDims];      // first word bit of the dimension
    int8_t next;                // bits of the runs beyond the dimensions (2^next copies)
    int8_t ext[kMaxTileQubits + 1];  // their word bits
    uint32_t mask[kTileDims];   // dimension size - 1
    uint32_t copy_bytes;        // bytes of one copy
};

// Describe tiles of 2^k amplitudes of `amp_bytes` bytes at the physical bits
// slot_phys (ascending) of a state of 2^n amplitudes at `amps`.
sv_status tile_map(void *amps, int n, int k, const int *slot_phys, size_t amp_bytes, CUtensorMap *map,
                   TileBox *box);

// The dimensions alone (host only, no CUDA call): sizes, byte strides and box
// widths of the tensor, and the coordinates' record.
struct TileDims {
    uint64_t size[kTileDims], stride[kTileDims];
    uint32_t width[kTileDims];
};
void tile_dims(int n, int k, const int *slot_phys, size_t amp_bytes, TileDims *dims, TileBox *box);

}  // namespace sv
