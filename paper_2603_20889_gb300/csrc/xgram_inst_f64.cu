// Exact Gram pass, FP64 storage.
#include "xgram.cuh"

namespace ql {
template ql_status xgram_pass1<double>(const GramCall&, const GramWs&);
}  // namespace ql
