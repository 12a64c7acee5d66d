// Shared-memory plan of the persistent layer kernel (host code only).
#pragma once
#include <algorithm>

#include "host.hpp"
#include "layer_stack.cuh"

namespace bpd {

// Shared-memory plan of the persistent kernel for a session whose widest pass has `rows` rows; `budget` bytes per
// CTA.  Returns false when the working buffers and a ring that holds at least the two largest tiles do not fit.
// lean: the kernel's variant (1: short sequences, 2: one long sequence, 3: one short sequence, 0: general).
inline bool stack_plan(const Config& c, int rows, int nb, int ppr, int cross_rows, bool long_seq, int lean, size_t budget,
                       stack::Layout* out) {
  const int NT = rows > 8 ? 2 : 1, RP = NT * 8;
  const stack::Geo g = stack::make_geo(c.d, c.H, c.d_ff, c.n_dec, cross_rows, lean == 2 || lean == 3);
  auto up = [](size_t v, size_t a) { return (v + a - 1) / a * a; };
  size_t off = 0;
  stack::Layout L;
  memset(&L, 0, sizeof(L));
  auto take = [&](size_t bytes) { const size_t at = off; off = up(off + bytes, 128); return (int)at; };
  L.x = take((size_t)RP * g.ks * 4);
  L.xh = take((size_t)RP * g.ks * 2);
  L.xl = take((size_t)RP * g.ks * 2);
  L.oh = take((size_t)RP * 128);
  L.ol = take((size_t)RP * 128);
  const bool split = lean == 2 || lean == 3;
  const size_t states = (size_t)fused::kC * rows * stack::kState * 4;
  L.hid = take(std::max((size_t)fused::kC * 2 * RP * g.UPR * 2, split ? states : 0));
  const size_t chunk = std::max((size_t)NT * 3 * fused::kDH * 4, (size_t)g.UPR * RP * 4);
  const size_t window = lean == 2 ? stack::kLongKeys : stack::kShortKeys;
  if (split) {
    // scores share the outbox, the ranks' states the hidden planes (see share_states)
    L.outbox = L.sc = take(std::max(fused::kC * chunk, (size_t)16 * (window + 4) * 4));
    L.inbox = take(fused::kC * chunk);
    L.lvl2 = L.hid;
    L.qp = take((size_t)3 * 16 * (attn::kPitch + stack::kLongCross + 8) * 2);
    L.kv = take(window * 256);
    L.attn = take(48 * 4);
    L.wst = L.lvl1 = L.attn;
  } else {
    L.outbox = take(fused::kC * chunk);
    L.inbox = take(fused::kC * chunk);
    L.attn = take(sizeof(AttnSmem<fused::kDH, stack::kWarps>));
    L.wst = take((size_t)stack::kWarps * NT * stack::kState * 4);
    const size_t lvl = long_seq ? states : 0;
    L.lvl1 = take(lvl);
    L.lvl2 = take(lvl);
  }
  L.kvq = take((size_t)RP * 512);
  L.stats = take((size_t)fused::kC * fused::kMaxRows * 2 * 4 + 4 * fused::kMaxRows * 4);
  L.pt = take((size_t)nb * ppr * 4);
  L.layers = take((size_t)c.n_dec * sizeof(stack::LayerPtrs));
  L.misc = take(sizeof(stack::Ctl));
  const size_t work = off;
  int largest = 0, second = 0, per_layer = 0;
  if (g.ntl > stack::kMaxTiles) return false;
  for (int i = 0; i < g.ntl; ++i) {
    const int b = stack::make_tile(g, i, cross_rows, c.d, 0, 0).bytes;
    per_layer += b;
    if (b > largest) { second = largest; largest = b; } else if (b > second) second = b;
  }
  if (work + 1024 > budget) return false;
  size_t ring = std::min((budget - work) / 1024 * 1024, (size_t)per_layer * c.n_dec);
  if (ring < (size_t)largest + second) return false;
  L.ring_bytes = (int)ring;
  int* fields[] = {&L.x, &L.xh, &L.xl, &L.oh, &L.ol, &L.hid, &L.outbox, &L.inbox, &L.kvq, &L.stats, &L.attn, &L.wst, &L.lvl1,
                   &L.lvl2, &L.pt, &L.layers, &L.misc, &L.kv, &L.qp, &L.sc};
  for (int* f : fields) *f += (int)ring;
  L.total = (int)(ring + work);
  *out = L;
  return true;
}

}  // namespace bpd
