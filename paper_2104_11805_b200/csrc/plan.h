// Rules of the launches that need no device: plain host code, so that they can be looked at without one.
#pragma once

namespace sdnn_plan {

// Whole networks in one launch (vector.cuh): CTAs of the cluster, and rows a CTA works on at once; CTA r has the rows r * VECTOR_BLOCK
// .. of every VECTOR_CTAS * VECTOR_BLOCK.
constexpr int VECTOR_CTAS = 16, VECTOR_BLOCK = 64;
// CTAs that have rows of a net of n neurons.  Only these exchange activations: see vector.cuh.
constexpr int vector_ctas(int n) { return n > (VECTOR_CTAS - 1) * VECTOR_BLOCK ? VECTOR_CTAS : (n + VECTOR_BLOCK - 1) / VECTOR_BLOCK; }

}  // namespace sdnn_plan
