// Between the sources of this library: the attention call and its workspace query where no more than `limit` bytes of scratch can be
// had.  With num_kv_splits = 0 the library's own cut is made as fine as fits; nothing else differs from the entry points in vpp.h.
#pragma once
#include "../../include/vpp.h"

namespace vpp {
size_t workspace_size_within(const vpp_chunk_attn_args* args, size_t limit);
vpp_status chunk_attn_fwd_within(const vpp_chunk_attn_args* args, vpp_stream_t stream, size_t limit);
}  // namespace vpp
