// Host check of the GEMM epilogue's column arithmetic (tc_common.cuh): for every
// output width the pieces of 8 columns that the tiles store cover each column once
// and none beyond the output.  Prints the number of mismatches; exits non-zero on any.
#include <cstdio>
#include <vector>

#include "tc_common.cuh"

using namespace fsi::tc;

int main()
{
    int bad = 0;
    for (int N = 1; N <= 256; ++N) {
        const int BN = gemm_tile_columns(N);
        if (BN % 16 || BN > kGemmMaxBN) ++bad;
        std::vector<int> stored(N, 0);
        for (int n0 = 0; n0 < N; n0 += BN)
            for (int c8 = 0; c8 * 8 < BN; ++c8) {
                const int j0 = n0 + 8 * c8, nc = gemm_piece_columns(j0, N);
                if (nc < 0 || nc > 8) ++bad;
                for (int j = j0; j < j0 + nc; ++j) {
                    if (j >= N) ++bad;
                    else ++stored[j];
                }
            }
        for (int c : stored) bad += c != 1;
    }
    std::printf("mismatches %d\n", bad);
    return bad != 0;
}
