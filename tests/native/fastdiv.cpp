// The constants of the kernels' divisions (csrc/hpt_internal.h) compiled with the host compiler, for the tests.
#include "hpt_internal.h"

using namespace hpt;

extern "C" void constants(int d, unsigned *mul, int *shift)
{
    const FastDiv f = make_fastdiv(d);
    *mul = f.mul;
    *shift = f.shift;
}
