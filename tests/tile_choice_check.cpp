// Drives rule_config and pairs_room of bf_choice.h; built and run by
// tests/test_host_logic_tiles.py with g++ against the CUDA headers only.  Arguments: prec ns
// na nx nz sms alone shares peers; or cap peers fixed, for the rooms of all the peers.
#include <cstdio>
#include <cstdlib>

#include "bf_choice.h"

int main(int n, char **v)
{
    if (n == 4) {
        const int cap = std::atoi(v[1]), all = std::atoi(v[2]);
        for (int k = 0; k < all; ++k)
            std::printf("%d\n", bfi::pairs_room(cap, k, all, std::atoi(v[3]) != 0));
        return 0;
    }
    const int prec = std::atoi(v[1]), ns = std::atoi(v[2]), na = std::atoi(v[3]), nx = std::atoi(v[4]),
              nz = std::atoi(v[5]), sms = std::atoi(v[6]), peers = std::atoi(v[9]);
    std::printf("%d\n", bfi::rule_config(prec, ns, na, bfi::image_tiles(nx, nz), sms, std::atoi(v[7]) != 0,
                                         std::atoi(v[8]) != 0, peers));
    return 0;
}
