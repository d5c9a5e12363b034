// Which leaves of which layers of a stack run together (rt_leaf_group.cu): a leaf is ready when the layer below has finished it and its own
// layer the one before.  Plain C++, so that it can be walked through on the host.
#pragma once

namespace rt {

constexpr int kWaveBand = 16;            // layers that run side by side at most; deeper stacks run band after band

// Of the ready leaves those with the most still to come after them in a row (of their layer and the layers above) go first, of equal ones the deepest
// layer's.  A launch costs a pass over the layers of the band, whatever the number of leaves.
struct WaveOrder {
  int n_layers, n_leaves, done[kWaveBand];
  WaveOrder(int layers, int leaves) : n_layers(layers), n_leaves(leaves), done{} {}
  // The next launch: up to `places` (layer, leaf) pairs; 0 when all leaves are done.
  int next(int places, int* layer, int* leaf) {
    int n = 0;
    for (int l = 0; l < n_layers; ++l) {
      if (done[l] == n_leaves || (l > 0 && done[l - 1] <= done[l])) continue;
      const int sum = l + done[l];       // the smaller, the more is to come
      int i = n < places ? n++ : places;
      for (; i > 0 && sum <= layer[i - 1] + leaf[i - 1]; --i)
        if (i < places) { layer[i] = layer[i - 1]; leaf[i] = leaf[i - 1]; }
      if (i < places) { layer[i] = l; leaf[i] = done[l]; }
    }
    for (int i = 0; i < n; ++i) ++done[layer[i]];
    return n;
  }
};

// How many launches that takes: a band's leaves one after the other through its layers, or as many as fill the places, which fill and drain one by one.
// (8 layers of 5 leaves in 4 places 13, of 64 leaves in 6 places 91.)
inline long long wave_launches(int n_layers, int n_leaves, int places) {
  const int at_once = n_layers < n_leaves ? n_layers : n_leaves, p = places < at_once ? places : at_once;
  const long long chain = (long long)n_layers + n_leaves - 1, full = ((long long)n_layers * n_leaves + p - 1) / p + p - 1;
  return chain > full ? chain : full;
}

}  // namespace rt
