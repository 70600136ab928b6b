// Local density peaks of a level's groups (peaks.cu).
#pragma once
#include "cells.cuh"

// Cell-sorted particles and their group labels for one level.
struct PeakArgs {
  CellGrid grid;
  const int4* spos;
  const long long* ssig;
  const uint64_t* sid;
  const int* slab;  // group label per cell-sorted particle (-1: none)
  uint32_t b2;
  int n;            // cell-sorted particles
};

// The peaks of every segment, grouped by segment (unordered within one):
// peaks off[g] .. off[g + 1] - 1 belong to segment g.
struct PeakList {
  uint32_t* off;    // nseg + 1
  int4* pos;        // position, and the cell-sorted index in w
  long long* sig;   // kernel sum
  uint64_t* id;
  uint8_t* out;     // scratch of the nucleus loop: no longer eligible
};

// Members gs[0 .. m) (cell-sorted indices, seg[k] the segment of member k)
// whose kernel sum is above T_min and that no denser member of the same
// segment within b comes before (Sec. 2.2.2 step 2): fills P, whose arrays are
// allocated here from ws (which keeps them) unless P brings arrays of at
// least m peaks.
//
// beater (one entry per cell-sorted particle) links the levels: with
// `first`, every member above T_test is tested and beater[s] receives one
// particle that beats s (-1: none, s is a peak); without it, a member whose
// recorded beater shares its label is no peak, one without a beater is a
// peak, and only the others (their beater is in another segment) are tested.
int peaks_find(const PeakArgs& a, const uint32_t* gs, const uint32_t* seg, int m, int nseg, long long T_min,
               long long T_test, bool first, int* beater, PeakList& P, Workspace& ws, cudaStream_t st);
