// Exact Gram pass, FP32 storage.
#include "xgram.cuh"

namespace ql {
template ql_status xgram_pass1<float>(const GramCall&, const GramWs&);
}  // namespace ql
