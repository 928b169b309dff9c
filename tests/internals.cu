// Access to a context's internal settings (for test_gpu_small_clusters.py).
#include "../paper_2505_10857_gb300/csrc/nswe_internal.h"

extern "C" int get_max_cluster(nswe_ctx c) { return c->max_cluster; }
extern "C" void set_max_cluster(nswe_ctx c, int ctas) { c->max_cluster = ctas; }
