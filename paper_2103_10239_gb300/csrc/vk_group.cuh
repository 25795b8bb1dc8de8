// vk_group.cuh -- exact k-nearest selection by a group of GS lanes, shared by
// the 2D and the 3D search: hits are appended to the group's list in shared
// memory by ballot, a nearly full list keeps its k best by (int64 squared
// distance, id), and the search radius follows.
#pragma once
#include <climits>

#include "vk_internal.cuh"

namespace vk {

namespace {

template <int CAP>
struct GroupList {
  unsigned long long d[CAP];
  int32_t slot[CAP];
};

template <int KC> struct GroupCfg { static constexpr int CAP = KC <= 12 ? 64 : KC <= 17 ? 96 : 160; };

// All lanes of the group call every function.
template <int GS, int CAP>
struct GroupTop {
  GroupList<CAP>& L;
  const int32_t* __restrict__ ids;
  unsigned mask;      // the group's lanes
  int shift, gl;      // its first lane, the lane's number in it
  int32_t self;
  int k, cnt;
  unsigned long long tau;
  uint32_t n_cand;

  // the lanes whose candidate q counts (squared distance D <= tau) add it
  __device__ __forceinline__ void append(bool hit, unsigned long long D, int64_t q) {
    const unsigned m = (__ballot_sync(mask, hit) & mask) >> shift;
    if (hit) {
      const int at = cnt + __popc(m & ((1u << gl) - 1u));
      L.d[at] = D;
      L.slot[at] = (int32_t)q;
    }
    cnt += __popc(m);
    if (cnt > CAP - GS) compact();
  }

  // the k best of the list by (D, id), in order, through put(rank, D, slot)
  template <class F>
  __device__ __forceinline__ void rank(F put) {
    constexpr int E = (CAP + GS - 1) / GS;
    __syncwarp(mask);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int i = gl + e * GS;
      if (e * GS >= cnt) break;
      int r = INT_MAX;
      unsigned long long D = 0;
      int32_t q = 0;
      if (i < cnt) {
        D = L.d[i];
        q = L.slot[i];
        r = 0;
        for (int j = 0; j < cnt; ++j) {
          const unsigned long long Dj = L.d[j];
          bool before = Dj < D;
          if (Dj == D && j != i) before = __ldg(ids + L.slot[j]) < __ldg(ids + q);
          r += before ? 1 : 0;
        }
      }
      put(e, r, D, q);
    }
  }

  __device__ __forceinline__ void compact() {
    constexpr int E = (CAP + GS - 1) / GS;
    int rk[E];
    unsigned long long dk[E];
    int32_t qk[E];
#pragma unroll
    for (int e = 0; e < E; ++e) rk[e] = INT_MAX;
    rank([&](int e, int r, unsigned long long D, int32_t q) {
      rk[e] = r;
      dk[e] = D;
      qk[e] = q;
    });
    __syncwarp(mask);
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (rk[e] < k) {
        L.d[rk[e]] = dk[e];
        L.slot[rk[e]] = qk[e];
      }
    __syncwarp(mask);
    cnt = min(cnt, k);
    if (cnt == k) tau = L.d[k - 1];
  }

};

}  // namespace

}  // namespace vk
