// The portal table (csrc/geom_portals.h) of a geometry finalized in a context of the library.
#include <cstring>

#include "g4n_internal.h"

extern "C" long long portals_of(g4n_ctx *ctx, int geom, int32_t *out) {
  const std::vector<int32_t> &t = ctx->geoms[geom]->portal;
  if (out) std::memcpy(out, t.data(), t.size() * sizeof(int32_t));
  return (long long)t.size();
}
