// Host-side schedule of the solver's blocks (the program that blk_stream and blk_sweeps in
// dp_blk.cuh run): which rows form a block, which blocks may run at the same time, and which warp
// runs which.
#include <algorithm>
#include <cstring>
#include <vector>

#include "dp_kernels.h"

namespace {

struct Op {
  int type, idx, mask, a, b, slot, live, weight;
  std::vector<int> deps, users;
  int path = 0;   // rows on the longest chain of blocks from this one to the end of the sweep
  int level = -1, warp = 0;
};

}  // namespace

// Fills T's block fields and the program (32-bit words of the blob the kernels copy to shared
// memory). Returns false when the robot has more blocks or levels than the stream format holds.
bool plan_blocks(DevTopo& T, std::vector<int32_t>& blob) {
  T.cslot = T.nslots;
  for (int j = 0; j < T.nj; ++j) T.jslot[j] = T.jlim[j] = T.jmot[j] = -1;
  for (int s = T.nslots - 1; s >= 0; --s) {
    if (T.skind[s] == RK_JLIN && T.ssub[s] == 0) T.jslot[T.sidx[s]] = (int16_t)s;
    if (T.skind[s] == RK_LIMIT) T.jlim[T.sidx[s]] = (int16_t)s;
    if (T.skind[s] == RK_MOTOR) T.jmot[T.sidx[s]] = (int16_t)s;
    if (T.skind[s] >= RK_GN) T.cslot = s;
  }
  // Warps: eight for the compiled topologies (the quadruped has 8 joints, 9 bodies, 8 contacts; two
  // warps a scheduler also hide each other's latencies), four for the other robots, which are mostly
  // smaller: two such CTAs fit on an SM. A large one loses little by it: 9728 quadrupeds without their
  // compiled topology, ten steps of ten sweeps, 1.11 + 3.54 ms (rollout, reverse) on four warps, with it
  // 0.93 + 3.61 on eight.
  const int nw = T.blk_nw = T.topo_id != 0 ? 8 : 4;
  // Blocks: a row joins the block of its item when that block is the last one on every body the
  // row touches (so the block's rows are adjacent for both bodies), else it starts a new block.
  std::vector<Op> ops;
  std::vector<int> last(T.nb, -1);
  for (int o = 0; o < T.nslots; ++o) {
    const int s = T.order[o], kind = T.skind[s], idx = T.sidx[s], a = T.sa[s], b = T.sb[s];
    int type, bit, slot, live = -1;
    switch (kind) {
      case RK_JLIN: type = 0; bit = T.ssub[s]; slot = T.jslot[idx]; break;
      case RK_JANG: type = 0; bit = 3 + T.ssub[s]; slot = T.jslot[idx]; break;
      case RK_LIMIT: type = 1; bit = 0; slot = s; live = idx; break;
      case RK_MOTOR: type = 2; bit = 0; slot = s; break;
      default: {
        const bool pair = kind >= RK_PN;
        type = pair ? 4 : 3;
        bit = kind == RK_GN || kind == RK_PN ? 0 : 1 + T.ssub[s];
        slot = T.cslot + 3 * ((pair ? T.ns : 0) + idx);
        live = T.nj + (pair ? T.ns : 0) + idx;
      }
    }
    int k = -1;
    bool join = true;
    for (int body : {a, b}) {
      if (body < 0) continue;
      if (last[body] < 0 || (k >= 0 && last[body] != k)) { join = false; break; }
      k = last[body];
    }
    if (k < 0 || !join || ops[k].type != type || ops[k].idx != idx || type == 1 || type == 2) {
      Op n{};
      n.type = type; n.idx = idx; n.a = a; n.b = b; n.slot = slot; n.live = live;
      k = (int)ops.size();
      for (int body : {a, b}) {
        if (body < 0) continue;
        const int d = last[body];
        if (d >= 0 && std::find(n.deps.begin(), n.deps.end(), d) == n.deps.end()) n.deps.push_back(d);
        last[body] = k;
      }
      ops.push_back(n);
      for (int d : ops[k].deps) ops[d].users.push_back(k);
    }
    ops[k].mask |= 1 << bit;
    if (type != 1) ++ops[k].weight;  // limits are seldom active: no weight
  }
  const int n = (int)ops.size();
  if (n > 63 || n == 0) return false;
  if (T.topo_id != 0)  // (true of every compiled topology: their reverse blocks are written for whole items)
    for (const Op& o : ops)
      if ((o.type == 0 && o.mask != 31) || o.type == 4 || (o.type == 3 && o.mask != 7)) return false;
  for (int k = n - 1; k >= 0; --k) {
    for (int u : ops[k].users) ops[k].path = std::max(ops[k].path, ops[u].path);
    ops[k].path += ops[k].weight;
  }
  // Levels: the ready blocks with the longest remaining chains first, each on the least loaded
  // warp; a block that would make the level longer than its most urgent block waits.
  int done = 0, nlev = 0;
  std::vector<std::vector<int>> runs[8];
  while (done < n) {
    std::vector<int> ready;
    for (int k = 0; k < n; ++k) {
      if (ops[k].level >= 0) continue;
      bool ok = true;
      for (int d : ops[k].deps) ok &= ops[d].level >= 0 && ops[d].level < nlev;
      if (ok) ready.push_back(k);
    }
    std::stable_sort(ready.begin(), ready.end(), [&](int x, int y) { return ops[x].path > ops[y].path; });
    int load[8] = {0}, cnt[8] = {0};
    const int cap = std::max(1, ops[ready[0]].weight);
    for (int g = 0; g < nw; ++g) runs[g].emplace_back();
    for (int k : ready) {
      // the first warp of the level rotates: the warps of a level's most urgent blocks were idle in the
      // one before, and load their next record while they wait for its barrier
      const int first = nlev * 3 % nw;
      int w = first;
      for (int q = 1; q < nw; ++q) {
        const int g = (first + q) % nw;
        if (load[g] < load[w] || (load[g] == load[w] && cnt[g] < cnt[w])) w = g;
      }
      if (cnt[w] > 0 && load[w] + ops[k].weight > cap) continue;
      ops[k].level = nlev;
      ops[k].warp = w;
      load[w] += ops[k].weight;
      ++cnt[w];
      runs[w][nlev].push_back(k);
      ++done;
    }
    if (++nlev > 32) return false;
  }
  // blob: descriptors grouped by warp and level, then the level table (bytes), the bodies' item
  // lists, the live flags and the streams
  std::vector<uint8_t> b;
  std::vector<uint8_t> lev(nw * (nlev + 1));
  std::vector<int32_t> desc;
  int pos = 0;
  for (int w = 0; w < nw; ++w) {
    for (int l = 0; l < nlev; ++l) {
      lev[w * (nlev + 1) + l] = (uint8_t)pos;
      for (int k : runs[w][l]) {
        const Op& o = ops[k];
        desc.push_back(o.type | (o.mask << 8));
        desc.push_back(0);
        desc.push_back((o.slot & 0xffff) | (o.live * 65536));
        desc.push_back((o.a + 1) | ((o.b + 1) << 8) | (o.idx << 16));
        ++pos;
      }
    }
    lev[w * (nlev + 1) + nlev] = (uint8_t)pos;
  }
  b.resize(desc.size() * 4);
  std::memcpy(b.data(), desc.data(), b.size());
  T.blk_lev = (int)b.size();
  b.insert(b.end(), lev.begin(), lev.end());
  // items touching each body, in slot order: type (0 joint, 1 contact, 2 pair) << 6 | side b << 5 | index
  T.blk_inc0 = (int)b.size();
  std::vector<uint8_t> inc, first;
  for (int body = 0; body < T.nb; ++body) {
    first.push_back((uint8_t)inc.size());
    for (int j = 0; j < T.nj; ++j) {
      if (T.ja[j] == body) inc.push_back((uint8_t)j);
      if (T.jb[j] == body) inc.push_back((uint8_t)(0x20 | j));
    }
    for (int q = 0; q < T.ns; ++q)
      if (T.sbody[q] == body) inc.push_back((uint8_t)(0x40 | q));
    for (int p = 0; p < T.np; ++p) {
      if (T.sbody[T.pk[p]] == body) inc.push_back((uint8_t)(0x80 | p));
      if (T.sbody[T.pl[p]] == body) inc.push_back((uint8_t)(0xa0 | p));
    }
    if (inc.size() > 255) return false;
  }
  first.push_back((uint8_t)inc.size());
  b.insert(b.end(), first.begin(), first.end());
  T.blk_inc = (int)b.size();
  b.insert(b.end(), inc.begin(), inc.end());
  while (b.size() % 4) b.push_back(0);
  T.blk_words = (int)b.size() / 4;
  T.blk_live = (int)b.size();
  T.blk_stream_len = n + nlev + 2;
  T.blk_stream = T.blk_live + T.nj + T.ns + T.np;
  T.blk_bytes_total = T.blk_stream + nw * T.blk_stream_len;
  T.blk_nops = n;
  T.blk_nlev = nlev;
  T.blk_single = n == 1;
  blob.assign(T.blk_words, 0);
  std::memcpy(blob.data(), b.data(), b.size());
  return true;
}
