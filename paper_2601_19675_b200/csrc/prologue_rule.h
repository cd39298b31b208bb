// The shape of the prologue launch of the small-batch forward and the kernel that runs it (rotate.cu).  Plain C++ (no CUDA), so that
// it is testable by itself.
#pragma once

namespace lopro {

struct PrologueShape {
    int tpr;        // tokens of a row CTA
    int row_ctas;   // of one layer and one group of eight tokens: the rows of B, `tpr` tokens each
    int rot_ctas;   // and the rotation's
    int groups;     // groups of eight tokens
    bool staged;    // a token's row of x is staged in shared memory
    bool pairs;     // two rows of B per CTA
    bool deep;      // the passes over a row in flight together
    bool common;    // the kernel that takes tpr as an argument, not the one made for it
};

// r_pad: padded rank (0: no low-rank term); layers: of the launch; fp8: the FP8 low-rank record; other_product: not in front of the
// kernels of stream.cu, warps.cu and tall.cu; sms: multiprocessors (read only where a row CTA has eight tokens, i.e. with five and more).
inline PrologueShape prologue_shape(int d_in, int r_pad, int T, int layers, bool fp8, bool other_product, int sms) {
    PrologueShape s;
    const int live = T < 8 ? T : 8, nchunks = (d_in + 255) / 256;
    s.groups = (T + 7) / 8;
    // Tokens per row CTA: as few as it takes to fill the multiprocessors -- with one group of tokens a CTA per (row, token) is best
    // (256 CTAs for 4096 columns, rank 32, 8 tokens), with several groups about one CTA per multiprocessor --, and no more than there
    // are: the loads, products and sums of absent tokens are not free (4096 -> 11008 twice, rank 128, 1 token with the loop of eight
    // 19.4 us, of one 17.1; eight experts 4096 -> 14336, rank 32, a row each 54.8 and 51.2).
    const int want = T <= 8 ? 256 : 120;
    s.tpr = 1;
    while (s.tpr < live) s.tpr *= 2;
    while (s.tpr > 1 && r_pad * ((live + s.tpr - 1) / s.tpr) * s.groups * layers < want) s.tpr /= 2;
    s.row_ctas = r_pad * ((live + s.tpr - 1) / s.tpr);
    // rotation: a token's row of x is staged in shared memory and gathered from there; with very few (token,
    // chunk) pairs the gather straight from global memory, warp = token, is as fast (measured: 6.1 against 6.3 us
    // per layer forward for one token and 4096 columns, 15.4 against 16.9 us for 8 tokens and 11008 columns)
    s.staged = nchunks * live * s.groups > 64;
    // More than eight tokens: two rows of B per CTA and half the tokens (as many CTAs as before), or all eight tokens where
    // that leaves more than one CTA per multiprocessor and all loads of x are in flight at once: fewer reads of x.  Whole
    // forwards with one row, two rows and half the tokens, two rows and all of them: 2048 -> 1024, 128 rows, 32 tokens 11.9 us,
    // 11.3, 10.6; 16 tokens (128 CTAs in the last form) 6.8, 6.5, 7.4; 4096 -> 4096, 64 rows, 32 tokens 14.3, 13.5, 13.4.  A
    // kernel of its own: it takes other numbers of registers.
    s.pairs = s.staged && s.groups > 1 && s.tpr >= 4 && !fp8 && (long long)d_in * 2 <= 48 * 1024;
    if (s.pairs) {
        if (s.tpr == 8 && d_in <= 4096 && s.row_ctas * s.groups * layers > 2 * sms) s.row_ctas /= 2;
        else s.tpr /= 2;
    }
    // Few tokens of long rows: the passes over a row in flight together (11008 -> 4096 at 8 tokens 13.7 -> 13.4 us for the whole
    // forward, FP8 record at 5 tokens 14.9 -> 14.5, 8192 columns 9.2 -> 9.1; 5120 columns 10.8 -> 11.0, so not there; also a kernel
    // of its own, for its registers).
    s.deep = s.groups == 1 && d_in >= 8192;
    s.rot_ctas = s.staged ? live * ((nchunks + 7) / 8) : nchunks;
    // A kernel per number of tokens of a row CTA: with one or two it takes 54 to 92 registers instead of 96 to 128, and the CTAs of the
    // next launch find room beside it (with kernels of their own throughout: decoder layer 4096, 4 sequences 69.4 -> 60.3 us, 2048, 6
    // sequences 50.6 -> 43.9, 11008 -> 4096 at 8 tokens 14.0 -> 12.9, graphs of 4096 -> 4096 at 1 token 6.5 -> 6.1; the same by single
    // calls, where the two launches cost the host more than that, 5.8 and 6.0).  The common kernel stays
    //  * for two rows of B per CTA and a layer alone (4096 -> 4096 at 16 tokens 8.5 and 9.0, 4096 -> 11008 12.7 and 13.4);
    //  * for long rows of the FP8 record: 11008 -> 4096 at 1, 2, 3, 4 and 5 tokens, ranks 16 to 64, 12.5 to 14.0 us and 13.0 to 14.3 alone,
    //    within one percent either way as part of a decoder layer.  With folded factors it gains as much on most long rows alone (8192 to
    //    14336 columns, 1 to 4 tokens 0 to 4 percent; at 8 tokens it loses as often), but costs the layer around it more: decoder
    //    layer 4096 of 1 and 4 sequences 63.9 us and 65.5, 60.3 and 62.2, 3072 with a gate of 10240 at 2 sequences 51.4 and 53.4;
    //  * in front of products whose CTAs leave no room for others anyhow: vector-quantized layers 4096 -> 4096 at 2 and 4 tokens
    //    12.2 and 13.4 us, 12.3 and 12.6 (others gain up to 2.5 percent).
    // Layers alone that lose by their own kernels, and win as part of a decoder layer: one or two tokens whose product goes in runs of
    // row tiles (5120 -> 5120, rank 64, 2 tokens 8.9 and 9.3; decoder layer 5120 80.9 and 77.6), 9 to 16 tokens of rank 16 (512 -> 4096,
    // 16 tokens 4.6 and 5.2; decoder layer 1024 of 16 sequences 37.8 and 36.8, 4096 of 12 84.2 and 80.5).
    const int ctas = (s.row_ctas + s.rot_ctas) * s.groups;
    s.common = other_product || (s.pairs && layers == 1) || (s.deep && fp8);
    // The loop of eight tokens by itself takes 165 registers, so that a multiprocessor holds one CTA, against two of the common kernel:
    // only where the last row CTA of the launch is among the first that start (the rotation's CTAs come after the rows' and end soon).
    // 4096 -> 4096, FP8 record, 16 tokens by itself and in common: rank 64 (the last row CTA is number 144) 10.1 us and 10.5, 80 (176)
    // 11.6 and 10.6, 128 (272) 12.7 and 11.1; 512 -> 4096, 32 tokens, rank 32 (134) 6.9 and 7.4, 64 (262) 8.5 and 7.9; three layers
    // 4096 -> 4096, rank 128, 8 tokens 17.9 and 16.2.  With two rows of B per CTA and for long rows it has nothing over the common kernel.
    if (s.tpr == 8 && (s.pairs || s.deep || ctas * layers - s.rot_ctas > sms)) s.common = true;
    return s;
}

}  // namespace lopro
