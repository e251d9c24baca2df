// Reads descriptors (one per line: N C_in H W C_out KH KW stride_h stride_w pad_h pad_w dilation_h dilation_w groups) and prints what the
// library's host code makes of each: the variant, whether an instantiation runs its configuration, the workspace.  Host code only.
#include <stdio.h>

#include "../paper_2006_09791_b200/csrc/gconv_internal.h"

int main() {
    int v[14];
    for (;;) {
        for (int i = 0; i < 14; ++i)
            if (scanf("%d", &v[i]) != 1) return 0;
        gconv_desc* d = nullptr;
        if (gconv_desc_create_2d(&d, v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], v[9], v[10], v[11], v[12], v[13]) != GCONV_OK) {
            printf("refused\n");
            continue;
        }
        const bool tc = gconv::igemm_supported(d->s);
        printf("%d %d %zu\n", d->variant, !tc || gconv::igemm_runnable(d->s, 0, 148) ? 1 : 0, tc ? gconv::igemm_scratch_bytes(d->s) : (size_t)0);
        gconv_desc_destroy(d);
    }
}
