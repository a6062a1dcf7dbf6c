// Marching-cubes case table (built on the host, copied to the device).
#pragma once

#include <cstdint>

namespace bcmc {

constexpr int kMaxTriPerCell = 5;   // the rule in mc_tables.cu never needs more (checked when built)

struct McTables {
    uint8_t num_tri[256];
    uint8_t tri_edges[256][16];      // 3 edge numbers per triangle, kMaxTriPerCell triangles
    int max_tri;
};

// What the emission reads of the table, laid out for it.  A table triangle
// is a row (rows of a case are consecutive); its three corners are cut edges
// of the cell, each named by its lower sample (relative to the cell's lower
// corner) and its axis.  The samples of a block's 5x5x5 window are staged
// unpadded: sample (x, y, z) at x + 5y + 25z.
constexpr int kCaseTriangles = 820;  // triangles of all 256 cases together (checked when built)
constexpr int kWindow = 125;         // samples of a block's window
constexpr int kTileBlocks = 4;       // blocks an emitting warp stages at a time, one window after another

struct alignas(16) EmitTables {
    uint16_t info[256];                     // per case: byte offset of its first row (13 bits) | triangles << 13
    uint16_t corner[kCaseTriangles][4];     // byte offset of the lower sample | byte step to the upper one << 8
    uint16_t coord[kTileBlocks * kWindow][4];   // staged sample: its x, y, z as half floats
};

void build_emit_tables(const McTables &t, EmitTables *e);

// Returns false if the rule produced something inconsistent (never expected).
bool build_mc_tables(McTables *t);

}  // namespace bcmc
