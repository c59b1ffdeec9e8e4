// Token-ordered key lists of the causal SA branch (sa_order.cu): geometry, layout, launch.
#pragma once
#include "sa_common.cuh"

namespace sa {

constexpr int kOrderTile = 128;    // queries per tile, keys per block

// Groups of `slots` consecutive slots, dealt to slots / 128 query tiles by token.
struct OrderGeom {
  int slots, span;         // slots of a group; slots of its windows' union
  int groups, tiles;       // of a sequence
  int blocks, pitch;       // most key blocks of a tile; tokens between two groups' lists
};

struct OrderView {
  int32_t *q, *k, *tiles;  // [B, tiles, 128] query tokens; [B, groups, pitch] key tokens; [B, tiles] blocks
  uint4* bits;             // [B, tiles, blocks, 128]: what a row sees of a block, one bit per key
};

// Whether the SA branch of such a problem can walk token-ordered lists, and their geometry.  Depends on
// nothing that a part of a batch or of the KV heads changes: a sequence has the same bits in either.
bool order_geom(int n, int d, int w, uint32_t flags, OrderGeom* g);
size_t order_bytes(int B, const OrderGeom& g);
OrderView order_view(void* ws, int B, const OrderGeom& g);
cudaError_t launch_order(const int32_t* perm, int B, int n, int w, uint32_t flags, const OrderGeom& g,
                         const OrderView& v, cudaStream_t st);

}  // namespace sa
