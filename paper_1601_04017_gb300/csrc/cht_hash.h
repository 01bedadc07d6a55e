// Hashes of keys.  Device code in the kernels; plain functions where a host
// compiler includes it.
#pragma once

#ifdef __CUDACC__
#define CHT_HASH_FN __device__ __forceinline__
#else
#define CHT_HASH_FN inline
#endif

namespace cht {

// fmix64, the 64-bit finalizer of MurmurHash3 (Appleby, public domain).
CHT_HASH_FN unsigned long long fmix64(unsigned long long x) {
    x ^= x >> 33;
    x *= 0xff51afd7ed558ccdull;
    x ^= x >> 33;
    x *= 0xc4ceb9fe1a85ec53ull;
    x ^= x >> 33;
    return x;
}

// A key's slot among 2^n in shared memory (mask = 2^n - 1), to be probed
// linearly: low bits of fmix64.  Every bit of the key counts, so ids shifted
// left, aligned addresses and packed pairs spread like random keys (1.5 looks a
// key at half load), and a window sorted by the home (the top bits) does too.
// The folding's time is in its looks, not in the hash: 2^24 insertOrUpdates of 1024 ids
// shifted by 25 bits take 0.28 ms, with a hash of two 32-bit multiplies whose
// low bits miss the key's high ones 2.74 ms; dense ids 0.27 and 0.25 ms.  (The high bits of one 64-bit
// multiply: 0.20 to 0.28 ms on those, but one stride in a hundred takes 12 looks
// a key and more.)
CHT_HASH_FN unsigned int slot_hash(unsigned long long key, unsigned int mask) {
    return static_cast<unsigned int>(fmix64(key)) & mask;
}

}  // namespace cht
