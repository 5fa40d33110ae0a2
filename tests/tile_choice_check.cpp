// Drives rule_config of bf_choice.h; built and run by tests/test_host_logic_tiles.py with
// g++ against the CUDA headers only.  Arguments: prec ns na nx nz sms alone shares peers.
#include <cstdio>
#include <cstdlib>

#include "bf_choice.h"

int main(int, char **v)
{
    const int prec = std::atoi(v[1]), ns = std::atoi(v[2]), na = std::atoi(v[3]), nx = std::atoi(v[4]),
              nz = std::atoi(v[5]), sms = std::atoi(v[6]), peers = std::atoi(v[9]);
    std::printf("%d\n", bfi::rule_config(prec, ns, na, bfi::image_tiles(nx, nz), sms, std::atoi(v[7]) != 0,
                                         std::atoi(v[8]) != 0, peers));
    return 0;
}
