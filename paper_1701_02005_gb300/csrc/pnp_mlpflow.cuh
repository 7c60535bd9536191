// The order in which the MMA thread of a network kernel (k_mlp_tc.cu) waits and
// issues, as templates over the operations themselves, so that the host can run it
// with waits that run out; and how the weight gradients' CTAs are shared out.
//
// Both flows end in o.drain(), whatever ended the loop: it commits everything the thread has
// issued to a barrier that nothing else uses and waits for that (bounded).  A barrier
// of the loop cannot serve: a layer whose second half was never handed over has MMAs
// that no commit covers, and the phase of a barrier whose last use is unknown may be
// one that completed long ago.  The tensor memory is freed after these return.
#pragma once

#ifdef __CUDACC__
#define PNP_FLOW __device__ __forceinline__
#else
#define PNP_FLOW inline
#endif

namespace pnp {

// All tiles of a CTA: the layers forward, and (train) the data gradients back to the
// first layer.  The first layer's K comes in one piece, the others' in halves as they
// are handed over.
template <int LAYERS, bool TRAIN, typename Ops>
PNP_FLOW bool flow_network(Ops& o, int first, int ntiles, int step) {
  unsigned phase = 0;
  bool ok = true;
  for (int tile = first; tile < ntiles && ok; tile += step) {
    for (int l = 0; l < LAYERS && ok; ++l, phase ^= 1u) {
      if (!(ok = o.ready(0, phase))) break;
      if (l == 0 && !(ok = o.ready(1, phase))) break;
      o.forward(l, 0);
      if (l > 0) {
        if (!(ok = o.ready(1, phase))) break;
        o.forward(l, 1);
      }
      o.commit();
    }
    if (TRAIN)
      for (int l = LAYERS - 1; l > 0 && ok; --l, phase ^= 1u) {
        if (!(ok = o.ready(0, phase) && o.ready(1, phase))) break;
        o.backward(l);
        o.commit();
      }
  }
  return o.drain() && ok;
}

// The weight gradients' ntl tiles through a ring of STAGES slots, RUN tiles to a sum,
// the sums in two TMEM blocks by turns.
template <int STAGES, int RUN, typename Ops>
PNP_FLOW bool flow_wgrad(Ops& o, int ntl) {
  bool ok = true;
  for (int n = 0; n < ntl; ++n) {
    const int q = n % STAGES, g = n / RUN;
    if (n % RUN == 0 && g >= 2 && !(ok = o.freed(g & 1, ((g >> 1) - 1) & 1))) break;
    if (!(ok = o.full(q, (n / STAGES) & 1))) break;
    o.product(q, g & 1, n % RUN != 0);
    o.commit_slot(q);
    if (n % RUN == RUN - 1 || n == ntl - 1) o.commit_sum(g & 1);
  }
  return o.drain() && ok;
}

// How `ctas` CTAs, one per SM, share the layers' tiles, given the shares of `full` of
// them: in proportion, at least one each, and no layer more than of `full` (the partial
// sums are laid out for those).
template <int N>
inline void share_ctas(const int (&of_full)[N], int full, int ctas, int (&out)[N]) {
  ctas = ctas < full ? ctas : full;
  int left = ctas;
  for (int l = 0; l < N; ++l) {
    out[l] = of_full[l] * ctas / full;
    if (out[l] < 1) out[l] = 1;
    left -= out[l];
  }
  for (int l = 0; left > 0; l = (l + 1) % N)
    if (out[l] < of_full[l]) {
      ++out[l];
      --left;
    }
}

}  // namespace pnp
