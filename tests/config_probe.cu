// Reads descriptors (one per line: N C_in H W C_out KH KW stride_h stride_w pad_h pad_w dilation_h dilation_w groups) and prints what the
// library's host code makes of each: the variant, whether an instantiation runs its configuration, the workspace, and for the staged FP32
// kernel whether its shared memory holds what the kernel puts there (-1: the one-thread-per-output kernel runs), the parts a batch of host
// buffers is cut into, and those after the descriptor has been set to the generic variant, and of the tensor-core configuration: CTAs that
// share a tile's channels, whether its tiles are row boxes, and filters a tile (0 where the variant does not apply).  Host code only.
#include <stdio.h>

#include "../paper_2006_09791_b200/csrc/gconv_internal.h"

// Buffers as the kernel addresses them, in 64 bits: patches [NI][CC][PH][pitch], weights [CC * taps][BM], the table of tap offsets, and over
// them the partial sums of a split tile.
static int staging_fits(const gconv::Shape& s, const gconv::ConvCfg& c) {
    const long long taps = (long long)s.KH * s.KW, BM = (long long)c.TM * c.WM, BN = 32ll * c.TN * c.WN, sw = s.stride_w;
    const long long columns = c.vec ? c.PW + 3 : ((long long)c.PW + sw - 1) / sw * sw;          // of a staged row, with the columns it is shifted by
    const long long patch = (long long)c.NI * c.CC * c.PH * c.pitch, weights = c.CC * taps * BM;
    const bool pw_ok = c.PW == (c.TW - 1) * sw + (long long)(s.KW - 1) * s.dilation_w + 1 && c.PH == (c.TH - 1ll) * s.stride + (long long)(s.KH - 1) * s.dilation + 1;
    return pw_ok && c.pitch >= columns && (long long)c.plane == (long long)c.PH * c.pitch && c.phase * sw == c.pitch && c.in_floats >= patch && c.w_floats >= weights &&
           (long long)c.smem >= 4 * (c.stages * ((long long)c.in_floats + c.w_floats) + c.CC * taps) && (c.split == 1 || (long long)c.smem >= 4 * BM * BN) &&
           c.smem <= 224 * 1024 && c.ctas > 0;
}

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
        gconv::ConvCfg c;
        const int staged = gconv::conv_config(d->s, 148, c) ? staging_fits(d->s, c) : -1;
        const int variant = d->variant, parts = gconv::host_parts(d);
        gconv_desc_set_variant(d, GCONV_VARIANT_DIRECT_GENERIC);
        gconv::IgemmCfg ig = {};
        if (tc) ig = gconv::igemm_config(d->s, 148);
        printf("%d %d %zu %d %d %d %d %d %d\n", variant, !tc || gconv::igemm_runnable(d->s, 0, 148) ? 1 : 0, tc ? gconv::igemm_scratch_bytes(d->s) : (size_t)0, staged, parts,
               gconv::host_parts(d), ig.spl ? ig.split : 0, ig.rowbox, ig.Kt);
        gconv_desc_destroy(d);
    }
}
