// Host-side helpers of the library with C names, for tests/test_host_helpers.py.
#include "../paper_2508_07424_gb300/csrc/pff_host.cuh"

extern "C" void map_pages(void *p, size_t bytes) { pff::map_pages(p, bytes); }
