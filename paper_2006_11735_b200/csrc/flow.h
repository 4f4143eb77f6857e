// The general form of a stack of layers (kernel_flow.cu), behind iconv_plan_stack.
#pragma once

#include "plan.h"

struct iconv_flow_s;

namespace iconv {

int flow_plan(const iconv_stack_layer *layers, int n, iconv_flow_s **out);
void flow_destroy(iconv_flow_s *s);
size_t flow_sync_bytes(const iconv_flow_s *s);
int flow_forward(const iconv_flow_s *s, void *sync, cudaStream_t stream);

}  // namespace iconv
