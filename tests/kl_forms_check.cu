// Host check of the FP32 contraction's choice of tiles (no GPU needed): over the sizes of
// a served run and of the benchmark, no SM goes without a tile that the next narrower
// tile would give it in the same single wave, a grid fits its launch, and the largest calls
// keep the widest tile.  Built and run by tests/test_kl_forms.py.
#include "../paper_1907_12334_gb300/csrc/field.cu"
#include <cstdio>
using namespace msg;

int main()
{
    int n = 0, idle = 0, big = 0;
    for (int64_t npts : {1, 100, 128, 129, 400, 1175, 2048, 4000, 8385, 20000, 33153, 263169})
        for (int64_t S : {1, 8, 31, 33, 64, 100, 200, 364, 600, 1000, 2048})
            for (int M : {1, 20, 64, 150, 206, 300, 400, 4096}) {
                const KlForm f = kl_f32_form(npts, M, S);
                ++n;
                if (f.TR > 2 && kl_f32_tiles(npts, S, f.TR / 2) <= 152) {
                    if (idle++ < 20) printf("idle SMs: %ld points, %ld samples, %d terms: TR %d\n", (long)npts, (long)S, M, f.TR);
                }
                if (kl_f32_tiles(npts, S, 8) >= 20 * 152 && f.TR != 8) ++big;
            }
    printf("%d calls, %d leave SMs idle, %d large ones in narrow tiles\n", n, idle, big);
    return idle || big;
}
