// plain_b.cu -- the plain form's transform kernels for N >= 4096
#include "plain_step.cuh"

namespace qt {
const PlainOps *plain_ops_b(int N)
{
    switch (N) {
    case 4096: return plain_ops<4096>();
    case 8192: return plain_ops<8192>();
    case 16384: return plain_ops<16384>();
    default: return nullptr;
    }
}
} // namespace qt
