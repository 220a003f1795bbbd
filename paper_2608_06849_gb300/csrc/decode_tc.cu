// The stream-K instances of the tcgen05 decode kernel and the host's choices
// for it.
#include <algorithm>

#include "decode_tc.cuh"

namespace aoh {

using namespace dtc;

bool decode_uses_tc(int D, int G) { return D == 128 && ((G >= 1 && G <= 8) || G == 16); }

bool decode_on_tc(int D, int G) {
  return decode_uses_tc(D, G) || (D == 64 && (G == 1 || G == 2 || G == 4 || G == 7 || G == 8));
}

int decode_tc_item_cost(long long total_rows, int n_ctas, int num_sms) {
  if (total_rows >= kItemCostMaxShare * n_ctas) return 0;
  return n_ctas < num_sms ? kItemCostFewCtas : kItemCost;
}

void reuse_tc_weights(int G, int* gather_w, int* ring_w) {
  (void)G;
  *gather_w = 3;
  *ring_w = 2;
}

// One CTA per SM; small steps use fewer, at least 512 rows each.
// At least 512 rows (four tiles) per CTA, so that small steps keep few
// partials per item (an item spread over more than kGroup CTAs needs the
// second merge level); once that fills half the GPU, every SM streams.
int decode_tc_ctas(long long total_rows, int num_sms) {
  const long long by_rows = (total_rows + 511) / 512;
  long long p = by_rows >= num_sms / 2 ? num_sms : by_rows;
  return p < 1 ? 1 : (int)p;
}

namespace {

// Clusters of C CTAs that `n` items of `rows` rows need at k tiles a CTA.
long long clusters_for(long long n, long long rows, int C, int k) {
  const long long per = (long long)kBN * C * k;
  return n * ((rows + per - 1) / per);
}

}  // namespace

// The cluster split serves steps of up to 32 items whose longest CTA then has
// few more tiles than an even share over all SMs. It spares a step the switch
// of items inside a CTA, the two merge levels through global memory and the
// length update at its end, worth about kSpared tiles (a tile is 0.8-1.4 us);
// with more items the whole clusters fit the rows less evenly. Measured, B=1
// and 28/4 heads of which 2 stream (S = 128, W = 2048), us a step as a layer
// of a graph, stream-K / clusters of 2 / 4 / 8 / 16: 1K 13.9 / 8.5 / 6.4 / 6.1 /
// 6.2, 2K 13.1 / 9.5 / 7.8 / 7.7 / 6.7, 4K 12.5 / 10.5 / 8.7 / 8.2 / 7.4, 16K
// 17.2 / 13.4 / 11.3 / 10.8 / 11.9, 32K 18.6 / 17.8 / 14.1 / 13.9 / 16.1, 128K
// 35.1 / 34.0 / 31.4 / - / -, 256K (W = 4096) 54.0 / 52.7 / 50.2 / - / -; B=4, 16
// items: 1K 14.3 / 9.0 / 7.0, 16K 25.6 / 20.7 / 20.5; B=4, 32/8 heads, 32 items: 1K
// 15.6 / 10.5 / 9.0, 4K 15.9 / 14.9 / 15.3, 16K 33.0 / - / - (-: not taken, the
// clusters that run at once do not hold the rows within kSpared tiles).
//
// Among the sizes and tiles a CTA: a step costs its k tiles (0.8 us each here), a
// global exchange (1.3 us, 2 tiles) unless one cluster holds each item, and
// another round trip (1 tile) for every eight clusters of an item beyond eight; a
// tile more is cheaper than the exchange (4,097 rows on 16 CTAs: 9.0 us with two
// clusters of 2 tiles, 8.7 with one of 3). Clusters of 2 leave
// more of them to that exchange, and are taken only above 16 items, where the
// larger sizes run out of clusters.
void decode_tc_split(DecodeArgs& a, const CacheGeom& g, long long longest, long long total_rows, int num_sms) {
  constexpr int kSpared = 6;
  a.row_keys = g.D == 64 ? 2 : 1;
  long long ring = std::min<long long>(longest, (long long)g.S + g.W);
  longest = (longest + a.row_keys - 1) / a.row_keys;
  ring = (ring + a.row_keys - 1) / a.row_keys;
  total_rows = (total_rows + a.row_keys - 1) / a.row_keys;
  a.cluster = 0;
  a.n_ctas = decode_tc_ctas(total_rows, num_sms);
  a.item_cost = decode_tc_item_cost(total_rows, a.n_ctas, num_sms);
  const long long n_r = (long long)g.B * g.n_r, n_s = (long long)g.B * g.n_s;
  const long long widest = g.n_r > 0 ? longest : ring;
  if (n_r + n_s > dec::kClusterItems || widest * (n_r + n_s) > (1ll << 30)) return;
  const long long even = (n_r * longest + n_s * ring + (long long)kBN * num_sms - 1) / ((long long)kBN * num_sms);
  double best = 1e30;
  for (int C = dec::kClusterMax; C >= (n_r + n_s > 16 ? 2 : 4); C /= 2) {
    const int most = decode_tc_max_clusters(C);
    if (n_r + n_s > most) continue;
    for (int k = 1; k <= even + kSpared; ++k) {
      const long long need = clusters_for(n_r, longest, C, k) + clusters_for(n_s, ring, C, k);
      if (need > most) continue;
      const long long parts = clusters_for(1, widest, C, k);
      const double cost = k + (parts > 1 ? 2.0 : 0.0) + (double)((parts - 1) / 8) + (C == 16 ? 0.6 : 0.0);
      if (cost < best) {
        best = cost;
        a.cluster = C;
        a.n_ctas = C * (int)need;
      }
    }
  }
}

// The reuse step (a.idx set) launches the variant with gather warps.
cudaError_t launch_decode_tc(const DecodeArgs& a, cudaStream_t s) {
  if (a.idx != nullptr) return launch_decode_tc_reuse(a, s);
  if (a.geom.D == 64) return launch_decode_tc64(a, s);
  if (a.cluster > 0) return launch_decode_tc_cluster(a, a.cluster, s);
  return launch_mode<128, kStream>(a, 1, s);
}

}  // namespace aoh
