// The order in which the one-pass attention's operands go through its ring, as plain arithmetic (no CUDA,
// so that it can be compiled and checked on the host).
#pragma once

#ifdef __CUDACC__
#define UAD_HD __host__ __device__ __forceinline__
#else
#define UAD_HD inline
#endif

namespace uad {

constexpr int kRingChunk = 128;   // keys of a chunk: K in kp pieces of its head dims, Vt in two halves of 64 keys

// K of chunk 0; then per chunk c the K of chunk c + 1 (S runs a chunk ahead of P V) and the Vt of chunk c.
struct AttnRing {
  int kp, nck;   // K pieces of a chunk, chunks

  UAD_HD int total() const { return kp + (nck - 1) * (kp + 2) + 2; }
  UAD_HD int k_entry(int c, int piece) const { return c == 0 ? piece : kp + (c - 1) * (kp + 2) + piece; }
  UAD_HD int v_entry(int c, int half) const { return kp + c * (kp + 2) + (c + 1 < nck ? kp : 0) + half; }

  struct Entry {
    bool k;            // K, else Vt
    int chunk, part;   // of that chunk: K piece, or half of its keys
  };
  UAD_HD Entry at(int e) const {
    if (e < kp) return {true, 0, e};
    const int f = e - kp, g = f / (kp + 2), c = g < nck - 1 ? g : nck - 1, r = f - c * (kp + 2);
    if (c + 1 < nck && r < kp) return {true, c + 1, r};
    return {false, c, c + 1 < nck ? r - kp : r};
  }
  // One past the last key that an entry holds.
  UAD_HD static int end_key(Entry e) {
    return e.k ? (e.chunk + 1) * kRingChunk : e.chunk * kRingChunk + (e.part + 1) * (kRingChunk / 2);
  }
  // How many of the first `slots` entries may be requested before the kernel that writes the chunk's own keys has
  // finished: with two chunks of prefix keys, K of both and the Vt of the first.
  UAD_HD int early(int slots, int prefix) const {
    if (prefix < 2 * kRingChunk) return 0;
    const int safe = 2 * kp + 2, n = slots < safe ? slots : safe;
    return n < total() ? n : total();
  }
};

}  // namespace uad
