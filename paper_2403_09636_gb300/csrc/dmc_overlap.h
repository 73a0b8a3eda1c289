// Which decode launches of a cache may overlap the launch before them. Host only.
#pragma once

namespace dmc {

// A decode launch may overlap the tail of the kernel before it on its stream
// (programmatic dependent launch) only if that kernel was this cache's decode of
// other layers, none of this launch's among them: its prologue reads slot counts, page
// table and pages (the tensor-core kernel those of its first two layers), which this
// cache's prefill and decode of those layers write. The cache's latest call is known
// here in host order, so it is the kernel before it on the stream only if it went to
// the same one; after a call on another stream the kernel before may be anything,
// an earlier call for the same layers among them.
struct DecodeOrder {
  int lo = 0, hi = 0;  // layers [lo, hi) of the latest call that wrote the cache if it was a decode, else empty
  const void* stream = nullptr;  // of that call

  // A decode of layers [layer0, layer0 + nlayers) comes next: may it overlap?
  // one_stream: the handle stands for one stream (cudaStreamPerThread does not).
  bool next_decode(int layer0, int nlayers, const void* s, bool one_stream) {
    const bool ok = hi > lo && one_stream && s == stream && (layer0 + nlayers <= lo || layer0 >= hi);
    lo = layer0;
    hi = layer0 + nlayers;
    stream = s;
    return ok;
  }
  // Any other call that writes the cache comes next.
  void other() { lo = hi = 0; }
};

}  // namespace dmc
