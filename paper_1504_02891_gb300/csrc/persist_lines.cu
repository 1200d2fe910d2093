// persist_lines.cu -- the persistent float32 Algorithm 1 launch with line
// transforms.
#include "persist_lines.cuh"
