// Traversal of all primitives along a ray with pooled leaf steps, and the transmittance (Sec. 5.3,
// Eq. 7) of one ray by it: device code shared by the queries, the renderer and the batch server.
#pragma once

#include "ugp_gauss.cuh"
#include "ugp_trace.cuh"

namespace ugp {

struct TrStats {
  unsigned n_nodes, n_prims;
  uint8_t st;
};

constexpr int kTrLeafQ = 10;  // primitives a lane may hold back (top of its stack column)

// Visits every primitive whose clipped interval over [t0, t1] may meet [t0, t_far] (t_far <= t1).
// `stk` points at this thread's column of a shared-memory stack with `stride` between levels and
// `owner` at its entry of a shared int array (its neighbours in the warp are the other lanes' entries).
// The whole warp calls together (lanes without a ray pass live = false) and runs in steps: a node
// step visits one node per lane and holds back the primitives it meets (up to kTrLeafQ, kept at
// the top of the stack column); a leaf step, taken once the lanes hold a primitive for each of
// them (or a queue is nearly full or a traversal is over), spreads the held-back primitives over
// the lanes, one per lane whichever ray it belongs to. The kernels are bound by instruction issue (ALU
// pipe): one packed warp sum per step instead of six votes, one erf for an interval whose two ends are
// the ellipsoid's, and the shared recomputation of ill-conditioned hits took 1,000,003 light-sample rays
// in a 1M-primitive room from 3.42 to 3.04 ms.
//
// With kOneScene all rays share the scene, whose fields then come from the constant bank.
//
// `P` collects the hits:
//   leaf(bool ok, const PrimHit& h, int o, int off, int mine)   called by all lanes in a leaf step: this lane's
//       primitive is hit (ok) by the ray of lane o; those of one ray are on neighbouring lanes, this lane's
//       own ray's from lane off on, of the `mine` that were waiting as many as there are lanes
//   bool enough()    after it, by lanes whose primitives were taken: nothing more can matter
//   kNearFirst       children are visited nearest first
//   kInOrder         a ray's primitives are handed to leaf() in the order in which the ray met them
static_assert(kTrLeafQ < 16, "queue lengths are summed from four bit planes");
//
// With kGroup, 1 << lg neighbouring lanes share a ray (its arguments are the same on all of them): the
// stack columns of a group are one stack, and a node step takes a node per lane from its top, nearest in
// the group's first lane. (Above half of the rows, which 4 lanes have 76 of, the stack holds at most 3 lanes + kStackMax
// entries: those of the last step of all lanes, then three a level of one path.) A launch of few rays is bound by the chain of dependent steps of its longest
// ray, and this shortens the chain, where spreading the rays over the warps left most lanes idle (figures at
// tr_group).
template <bool kGroup, bool kOneScene, class P>
static __device__ __forceinline__ void tr_walk(const TraceScene& sc, const Ray& ray, float t0, float t1, float t_far,
                                               int ex, int* stk, int stride, int* owner, TrStats& ts, bool live,
                                               int lg, P& pol) {
  constexpr unsigned mask = 0xffffffffu;
  const int lane = int(threadIdx.x) & 31;
  const unsigned below_me = (1u << lane) - 1u;
  int sp = 0, node = 0, nq = 0;
  bool tdone = !(live && sc.n_prims > 0 && t0 < t_far), done = tdone;
  constexpr int kRows = kTrStack - kTrLeafQ;  // of the stack in shared memory
  int* lq = stk + kRows * stride;
  int deep[kStackMax - kRows];
  // the group: its first lane, its lanes, its stack (entry i in row i >> lg of column i & (lanes - 1))
  const int gsize = kGroup ? 1 << lg : 1, gbase = lane & ~(gsize - 1);
  const unsigned glanes = (gsize == 32 ? ~0u : (1u << gsize) - 1u) << gbase;
  int* const gstk = stk - (lane - gbase);
  auto at = [&](int i) -> int& { return gstk[(i >> lg) * stride + (i & (gsize - 1))]; };
  const int grows = kRows << lg;  // the group's entries in shared memory
  if (kGroup) {
    if (lane == gbase) at(0) = 0;
    sp = 1;  // entries of the group's stack (with a lane per ray: below the current node)
  }
  __syncwarp(mask);
  for (;;) {
    // one packed sum: held-back primitives (9 bits), lanes at work, lanes that need a leaf step (a
    // node step may add four held-back primitives: it runs only while every lane has room)
    const int mine = done ? 0 : nq;
    const bool need_leaf = !done && (nq > kTrLeafQ - 4 || (tdone && nq > 0));
    const unsigned sums = __reduce_add_sync(mask, unsigned(mine) | (done ? 0u : 1u << 9) | (need_leaf ? 1u << 15 : 0u));
    if (((sums >> 9) & 63u) == 0u) break;
    const int total = int(sums & 511u);
    if (total >= 32 || (sums >> 15) != 0u) {
      // each lane's exclusive prefix of the queue lengths (below 16) from four bit planes
      const unsigned p0 = __ballot_sync(mask, (mine & 1) != 0), p1 = __ballot_sync(mask, (mine & 2) != 0),
                     p2 = __ballot_sync(mask, (mine & 4) != 0), p3 = __ballot_sync(mask, (mine & 8) != 0);
      // lane i takes item i of the queues laid end to end
      const int off = __popc(p0 & below_me) + 2 * __popc(p1 & below_me) + 4 * __popc(p2 & below_me) +
                      8 * __popc(p3 & below_me);
      const unsigned starts = __reduce_or_sync(mask, (mine > 0 && off < 32) ? (1u << off) : 0u);
      const bool work = lane < total;
      // the k-th lane with queued primitives, by a table the owners fill
      int* owner_of = owner - lane;
      if (mine > 0) owner_of[__popc((p0 | p1 | p2 | p3) & below_me)] = lane;
      __syncwarp(mask);
      const int o = work ? owner_of[__popc(starts & (0xffffffffu >> (31 - lane))) - 1] : lane;
      const int off_o = __shfl_sync(mask, off, o);
      const int nq_o = __shfl_sync(mask, mine, o);
      Ray ro;
      ro.o = make_float3(__shfl_sync(mask, ray.o.x, o), __shfl_sync(mask, ray.o.y, o), __shfl_sync(mask, ray.o.z, o));
      ro.d = make_float3(__shfl_sync(mask, ray.d.x, o), __shfl_sync(mask, ray.d.y, o), __shfl_sync(mask, ray.d.z, o));
      ro.inv = make_float3(0.f, 0.f, 0.f);  // not used by the primitive test
      ro.inv_dd = __shfl_sync(mask, ray.inv_dd, o);
      const float t0o = __shfl_sync(mask, t0, o), t1o = __shfl_sync(mask, t1, o);
      const int exo = __shfl_sync(mask, ex, o);
      const float4 *prims = sc.prims, *wlo = sc.wlo;
      float k2 = sc.k2;
      if (!kOneScene) {
        prims = reinterpret_cast<const float4*>(__shfl_sync(mask, reinterpret_cast<unsigned long long>(prims), o));
        wlo = reinterpret_cast<const float4*>(__shfl_sync(mask, reinterpret_cast<unsigned long long>(wlo), o));
        k2 = __shfl_sync(mask, k2, o);
      }
      PrimHit h;
      const int slot = work ? lq[(P::kInOrder ? lane - off_o : nq_o - 1 - (lane - off_o)) * stride + (o - lane)] : 0;
      const bool ok = prim_test_of<true>(work, prims, wlo, slot, ro, t0o, t1o, k2, exo, h);
      pol.leaf(ok, h, o, off, mine);
      __syncwarp(mask);
      if (kGroup || mine > 0) {
        nq = mine - min(mine, max(0, 32 - off));
        if (P::kInOrder && nq > 0 && nq < mine)  // at most one ray keeps some, the last that had its turn
          for (int k = 0; k < nq; ++k) lq[k * stride] = lq[(k + mine - nq) * stride];
        if (pol.enough()) {
          done = true;
          nq = 0;
        }
      }
    } else if (kGroup) {
      // ---- node step of groups: all lanes together (one node, by the first lane, once the stack is half full: it
      // then grows by three a level, as a single lane's does, and may go on in that lane's local memory)
      const int k0 = lane - gbase, m = tdone || done ? 0 : min(sp, sp > grows / 2 ? 1 : gsize);
      const bool act = k0 < m;
      if (act) {
        if (__builtin_expect(sp > grows, 0)) node = deep[sp - 1 - grows];
        else node = at(sp - 1 - k0);
      }
      sp -= m;
      float tk[4] = {INFINITY, INFINITY, INFINITY, INFINITY};
      int rk[4] = {-1, -1, -1, -1};
      int nk = 0;
      int inv = act && unsigned(node) >= unsigned(sc.n_nodes) ? -1 : 0;  // see valid_ref
      if (act && inv == 0) {
        float en[4];
        int ch[4];
        const unsigned hm = node4_test(sc.nodes4, node, ray, t0, t_far, en, ch);
        ++ts.n_nodes;
#pragma unroll
        for (int k = 3; k >= 0; --k) {
          if (!((hm >> k) & 1u)) continue;
          if (ch[k] < 0) {
            if (unsigned(~ch[k]) >= unsigned(sc.n_prims)) {
              inv = ch[k];
              continue;
            }
            ++ts.n_prims;
            lq[nq * stride] = ~ch[k];  // nq <= kTrLeafQ - 4 here: a node adds at most four
            ++nq;
          } else {
            tk[k] = en[k];
            rk[k] = ch[k];
            ++nk;
          }
        }
        sort4(tk, rk);
      }
      // the children go on the stack, those of the group's first lane on top, the nearest of each last
      const unsigned b0 = __ballot_sync(mask, (nk & 1) != 0) & glanes, b1 = __ballot_sync(mask, (nk & 2) != 0) & glanes,
                     b2 = __ballot_sync(mask, (nk & 4) != 0) & glanes;
      const unsigned above = lane == 31 ? 0u : ~0u << (lane + 1);
      const int pushed = __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2);
      const int base = sp + __popc(b0 & above) + 2 * __popc(b1 & above) + 4 * __popc(b2 & above);
      const bool g_bad = (__ballot_sync(mask, !valid_ref(inv)) & glanes) != 0u;
      const bool full = sp + pushed > grows + (kStackMax - kRows);
      if (m > 0 && (g_bad || full)) {
        ts.st = g_bad ? UGP_RAY_BAD_NODE : UGP_RAY_STACK_OVERFLOW;
        tdone = true;
        nq = 0;
      } else if (m > 0) {
        if (__builtin_expect(sp + pushed > grows, 0)) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (rk[k] >= 0) {  // hits are sorted first
              const int i = base + nk - 1 - k;
              if (i < grows) at(i) = rk[k];
              else deep[i - grows] = rk[k];
            }
        } else {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (rk[k] >= 0) at(base + nk - 1 - k) = rk[k];
        }
        sp += pushed;
        if (sp == 0) tdone = true;
      }
      __syncwarp(mask);
    } else if (!done && !tdone) {
      if (unsigned(node) >= unsigned(sc.n_nodes)) {
        ts.st = UGP_RAY_BAD_NODE;
        tdone = true;
        nq = 0;
      } else {
        float en[4];
        int ch[4];
        const unsigned hm = node4_test(sc.nodes4, node, ray, t0, t_far, en, ch);
        ++ts.n_nodes;
        float tk[4];
        int rk[4];
        int nk = 0;
        int inv = 0;
#pragma unroll
        for (int k = 3; k >= 0; --k) {
          tk[k] = INFINITY;
          rk[k] = -1;
          if (!((hm >> k) & 1u)) continue;
          if (ch[k] < 0) {
            // a primitive's slot is checked here (its record is loaded by slot); a child node's
            // index is checked when it is visited
            if (unsigned(~ch[k]) >= unsigned(sc.n_prims)) {
              inv = ch[k];
              continue;
            }
            ++ts.n_prims;
            lq[nq * stride] = ~ch[k];  // nq <= kTrLeafQ - 4 here: a node adds at most four
            ++nq;
          } else {
            tk[k] = en[k];
            rk[k] = ch[k];
            ++nk;
          }
        }
        if (P::kNearFirst || rk[0] < 0) sort4(tk, rk);  // at least, the first is one that was hit
        if (!valid_ref(inv)) {
          ts.st = UGP_RAY_BAD_NODE;
          tdone = true;
          nq = 0;
        } else if (nk > 0) {
          // rare, and apart from the plain pushes: 1,000,003 light-sample rays in a 1M-primitive room take 2.74 ms
          // (2.75 with no rows beyond shared memory), with a comparison at each push 2.82
          if (sp + nk - 1 > kRows) {
            if (sp + nk - 1 > kStackMax) {
              ts.st = UGP_RAY_STACK_OVERFLOW;
              tdone = true;
              nq = 0;
            } else {
#pragma unroll
              for (int k = 3; k >= 1; --k)
                if (rk[k] >= 0) {
                  if (sp < kRows) stk[sp * stride] = rk[k];
                  else deep[sp - kRows] = rk[k];
                  ++sp;
                }
              node = rk[0];
            }
          } else {
#pragma unroll
            for (int k = 3; k >= 1; --k)
              if (rk[k] >= 0) {
                stk[sp * stride] = rk[k];
                ++sp;
              }
            node = rk[0];
          }
        } else if (sp == 0) {
          tdone = true;
        } else {
          --sp;
          if (__builtin_expect(sp >= kRows, 0)) node = deep[sp - kRows];
          else node = stk[sp * stride];
        }
      }
    }
    if (tdone && nq == 0) done = true;
  }
}

// Returns tau = 1/2 sum_k I_k(clip_k) over [t0, t1], stopping once it reaches 1 (then T = 0).
// The sum is kept in 64-bit fixed point (units of 2^-40), so it is the same in any traversal
// order and whichever lanes test a ray's primitives (terms below 2^-41 are dropped: under 1e-10
// in tau for a few hundred of them); nearest-child-first only makes the early exit come sooner.
// `acc` points at this thread's entry of a shared array of sums; each lane of a leaf step adds its
// primitive's term to the owner's with a shared-memory atomic. Other arguments as for tr_walk.
struct DepthSum {
  static constexpr bool kNearFirst = true, kInOrder = false;
  static constexpr float kScale = 1099511627776.f;  // 2^40
  static constexpr unsigned long long kOne = 1ull << 40;
  unsigned long long* acc;  // the warp's sums; a group's is its first lane's
  int first;                // ~(lanes per ray - 1)
  __device__ void leaf(bool ok, const PrimHit& h, int o, int, int) {
    if (ok)
      atomicAdd(acc + (o & first),
                (unsigned long long)__float2ll_rn(fminf(fmaxf(hit_half_integral(h), 0.f), 2.f) * kScale));
  }
  __device__ bool enough() const {  // saturated: T = 0 whatever follows
    return *reinterpret_cast<volatile unsigned long long*>(acc + (int(threadIdx.x) & 31 & first)) >= kOne;
  }
};
template <bool kGroup = false, bool kOneScene = true>
static __device__ float tr_optical_depth(const TraceScene& sc, const Ray& ray, float t0, float t1, int ex,
                                         int* stk, int stride, unsigned long long* acc, int* owner, TrStats& ts,
                                         bool live, int lg = 0) {
  const int lane = int(threadIdx.x) & 31;
  DepthSum pol{acc - lane, kGroup ? -(1 << lg) : -1};
  *acc = 0ull;
  tr_walk<kGroup, kOneScene>(sc, ray, t0, t1, t1, ex, stk, stride, owner, ts, live, lg, pol);
  __syncwarp();
  const unsigned long long a = pol.acc[lane & pol.first];
  return a >= DepthSum::kOne ? 1.f : float(a) * (1.f / DepthSum::kScale);
}

}  // namespace ugp
