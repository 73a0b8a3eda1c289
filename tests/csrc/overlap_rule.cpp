// The decode overlap rule (dmc_overlap.h) as a C function for the CPU test: call i
// is a decode of layers [layer0[i], layer0[i] + nlayers[i]) on stream[i], or, with
// nlayers[i] = 0, another call; may[i] = 1 where a decode may overlap.
#include "dmc_overlap.h"

extern "C" void dmc_overlap_rule(int n, const int* layer0, const int* nlayers, const long long* stream,
                                 const int* one_stream, int* may) {
  dmc::DecodeOrder order;
  for (int i = 0; i < n; ++i) {
    may[i] = 0;
    if (nlayers[i] == 0)
      order.other();
    else
      may[i] = order.next_decode(layer0[i], nlayers[i], reinterpret_cast<const void*>(stream[i]), one_stream[i] != 0);
  }
}
