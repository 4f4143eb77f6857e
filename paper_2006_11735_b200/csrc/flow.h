// The general form of a stack of layers (kernel_flow.cu), behind iconv_plan_stack.
#pragma once

#include "plan.h"

struct iconv_flow_s;

namespace iconv {

// Why the layers cannot run as one launch on their tensors, or NULL: a layer reads what an earlier layer writes only as its
// exact output slice, and none writes what it or an earlier layer uses, by whatever pointer.  Host only.
const char *stack_aliases(const iconv_stack_layer *layers, int n);
int stack_layer_refused(int rc, int i);      // puts the layer's index before the reason why iconv_plan refused it
int flow_plan(const iconv_stack_layer *layers, int n, iconv_flow_s **out);
void flow_destroy(iconv_flow_s *s);
size_t flow_sync_bytes(const iconv_flow_s *s);
int flow_forward(const iconv_flow_s *s, void *sync, cudaStream_t stream);      // ICONV_ERR_UNSUPPORTED: its CTAs cannot all be resident, nothing is enqueued
const iconv_plan_t *flow_layer(const iconv_flow_s *s, int i);                  // the plan of one of its layers
int cooperative_launch_status(cudaError_t e, const char *what);                // the status of a cooperative launch that returned e

}  // namespace iconv
