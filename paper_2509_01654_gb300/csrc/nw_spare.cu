// nw_spare.cu -- the list of nw_spare.h.  Blocks are freed outside the lock:
// cudaFree may wait for the device.
#include <cuda_runtime.h>

#include <map>
#include <mutex>
#include <vector>

#include "nw_spare.h"

namespace nw {
namespace {

struct Block {
  const void* owner;
  int device;
  void* p;
  size_t bytes;
};
std::mutex mu;
std::vector<Block> blocks;  // oldest first
std::map<int, int> contexts;  // by device

// takes out what `pick` says, at most `most` blocks, and frees it
template <class Pick>
bool drop(Pick pick, size_t most) {
  std::vector<void*> out;
  {
    std::lock_guard<std::mutex> lock(mu);
    for (size_t i = 0; i < blocks.size() && out.size() < most;) {
      if (!pick(blocks[i])) {
        ++i;
        continue;
      }
      out.push_back(blocks[i].p);
      blocks.erase(blocks.begin() + (std::ptrdiff_t)i);
    }
  }
  for (void* p : out) cudaFree(p);
  return !out.empty();
}

}  // namespace

void* spare_take(const void* owner, int device, size_t bytes, size_t most, size_t* have) {
  std::lock_guard<std::mutex> lock(mu);
  size_t best = blocks.size();
  for (size_t i = 0; i < blocks.size(); ++i) {
    const Block& b = blocks[i];
    if (b.device != device || (owner && b.owner != owner) || b.bytes < bytes || b.bytes > most) continue;
    if (best == blocks.size() || b.bytes < blocks[best].bytes) best = i;
  }
  if (best == blocks.size()) return nullptr;
  void* const p = blocks[best].p;
  *have = blocks[best].bytes;
  blocks.erase(blocks.begin() + (std::ptrdiff_t)best);
  return p;
}

void spare_give(const void* owner, int device, void* p, size_t bytes) {
  if (bytes > kSpareBytes) {
    cudaFree(p);
    return;
  }
  for (bool room = false; !room;) {
    size_t total = 0, count = 0;
    {
      std::lock_guard<std::mutex> lock(mu);
      for (const Block& b : blocks) {
        total += b.device == device ? b.bytes : 0;
        count += b.owner == owner ? 1 : 0;
      }
      room = total + bytes <= kSpareBytes && count < kSpareBlocks;
      if (room) blocks.push_back({owner, device, p, bytes});
    }
    if (room) break;
    if (count >= kSpareBlocks) drop([&](const Block& b) { return b.owner == owner; }, 1);
    else drop([&](const Block& b) { return b.device == device; }, 1);
  }
}

size_t spare_held(const void* owner) {
  std::lock_guard<std::mutex> lock(mu);
  size_t n = 0;
  for (const Block& b : blocks) n += b.owner == owner ? b.bytes : 0;
  return n;
}

bool spare_drop_oldest(const void* owner) {
  return drop([&](const Block& b) { return b.owner == owner; }, 1);
}
bool spare_drop_device(int device) {
  return drop([&](const Block& b) { return b.device == device; }, (size_t)-1);
}


void spare_open(int device) {
  std::lock_guard<std::mutex> lock(mu);
  ++contexts[device];
}
void spare_close(const void* owner, int device) {
  bool last = false;
  {
    std::lock_guard<std::mutex> lock(mu);
    last = --contexts[device] <= 0;
    for (Block& b : blocks)
      if (b.owner == owner) b.owner = nullptr;
  }
  if (last) spare_drop_device(device);
}

}  // namespace nw
