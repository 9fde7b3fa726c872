// The streaming stencil kernels of degree 2 (a translation unit of their own: they
// are the slowest to compile).
#include "wm_stream.h"

template int wm_stream_run<2>(int, const StreamArgs&);
