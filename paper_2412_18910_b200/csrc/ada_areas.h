// What the pass kernel keeps in the area of its activation buffers between the products of a QKV phase and the attention phase
// that follows (also compiled on the host, tests/areas_model.cpp):
//
//   sums   from byte 0: one row of 256 floats per pass row, written and read by all worker warps in the phase's epilogue
//   keys   from kKeysAt: per worker warp 16 keys, then 16 values, copied there for the attention phase; below them that phase keeps
//          the rows of q, and of new keys and values, which it stages after the grid barrier
//
// A warp's first keys and values may be requested early: as soon as the products are complete where the sums end below the keys,
// else when every worker warp has read its sums.
#pragma once
#ifndef __CUDACC__
#define __host__
#define __device__
#endif

namespace ada {

constexpr int kSumsRowBytes = 256 * 4;
constexpr int kKeysAt = 4 * 16 * 128 * 2;              // q hi, q lo, new keys, new values: 16 rows of 128 halves each
constexpr int kKeysWarpBytes = 2 * 16 * 128 * 2;
__host__ __device__ constexpr bool keys_clear_of_sums(int TP) { return TP * kSumsRowBytes <= kKeysAt; }   // (up to 16 padded rows)

}  // namespace ada
