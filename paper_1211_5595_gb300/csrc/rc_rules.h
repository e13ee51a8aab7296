// Host-side rules that choose the form of a launch from its sizes. Plain C++
// without CUDA types, so that they can be compiled and tested by themselves.
#pragma once

namespace rc {

// CTAs of a persistent launch that takes `chunks` pieces of work from a queue,
// one CTA per SM: as many as there are SMs or chunks. A CTA of the 2-D table's
// gradient runs two or three groups, each with its own chunk, but an SM for
// each chunk comes first (128x128x96, 32 x 256 table, one 128^2 view of 64
// chunks: 748 us packed three to a CTA, 674 spread; 2 x 2 table 735 and 615).
inline int persistent_ctas(int chunks, int sms) { return chunks < sms ? chunks : sms; }

}  // namespace rc
