// The list of diagonals D = K2 - K1 = (dk, dn) of the tensor-core exchange
// kernels: (D, -D) pairs in the order dn = 0, 1, ... with dk inner, so that a
// diagonal read as the A operand is read as the B operand soon after.
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "g4_internal.h"

// Position of diagonal (dk, dn) in the list; dn = 0 is listed once per pair
// (pos0, a table of Nc entries); mk = (-)dk.
__device__ __forceinline__ int diag_pos(int dk, int dn, int mk, int Nc, const int* pos0) {
    if (dn > 0) return Nc + (dn - 1) * 2 * Nc + 2 * dk;
    if (dn < 0) return Nc + (-dn - 1) * 2 * Nc + 2 * mk + 1;
    return pos0[dk];
}

// The list itself, and the lengths of its items: 2 for a pair, 1 for D = -D.
inline void diag_list(const G4Dims& d, std::vector<int2>& dl, std::vector<int>& itemlen) {
    for (int dn = 0; dn < d.Nw2; ++dn)
        for (int dk = 0; dk < d.Nc; ++dk) {
            const int kx = dk % d.Lx, ky = dk / d.Lx;
            const int mk = (d.Lx - kx) % d.Lx + d.Lx * ((d.Ly - ky) % d.Ly);
            if (dn == 0) {
                if (mk < dk) continue;
                dl.push_back(make_int2(dk, 0));
                if (mk != dk) {
                    dl.push_back(make_int2(mk, 0));
                    itemlen.push_back(2);
                } else {
                    itemlen.push_back(1);
                }
            } else {
                dl.push_back(make_int2(dk, dn));
                dl.push_back(make_int2(mk, -dn));
                itemlen.push_back(2);
            }
        }
}
