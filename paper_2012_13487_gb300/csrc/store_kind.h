#pragma once
namespace fedbm {

// Storage forms of the distribution state.  Plain forms store f itself; the
// deviation forms store q with f_i = w_i (1 + s_k q_i), s_k a per-element
// power-of-two scale, and compute in FP32.
enum StoreKind { kStoreF64 = 0, kStoreF32 = 1, kStoreBF16 = 2, kStoreF16 = 3 };

}  // namespace fedbm
