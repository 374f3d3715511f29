// context_id.h -- whether something looked up or created in a CUDA context, and
// kept between calls with the context's id, may be used again.  Host code.
#pragma once

namespace titan {

// An id of 0 means that the driver gives none: nothing kept can then be trusted to
// belong to the context current now.
constexpr bool same_context(unsigned long long kept, unsigned long long now) { return now != 0 && kept == now; }

}  // namespace titan
