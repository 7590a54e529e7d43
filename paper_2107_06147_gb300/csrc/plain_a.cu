// plain_a.cu -- the plain form's transform kernels for N <= 2048
#include "plain_step.cuh"

namespace qt {
const PlainOps *plain_ops_a(int N)
{
    switch (N) {
    case 16: return plain_ops<16>();
    case 32: return plain_ops<32>();
    case 64: return plain_ops<64>();
    case 128: return plain_ops<128>();
    case 256: return plain_ops<256>();
    case 512: return plain_ops<512>();
    case 1024: return plain_ops<1024>();
    case 2048: return plain_ops<2048>();
    default: return nullptr;
    }
}
} // namespace qt
