// How the tensor-core projections cut their work: K-splits, pipeline stages, accumulators and accumulation segments.  Host
// arithmetic on sizes only, without CUDA types, so that the rules can be checked where there is no GPU.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace river {

constexpr int kTcBM = 128;      // output features per tile (UMMA M)
constexpr int kTcBK = 64;       // K per stage: 64 bf16 = one 128-byte swizzle row
constexpr int kW4Super = 4;     // k-blocks per raw code tile: 4 x 32 bytes of codes per row
constexpr int kW4RawBufs = 2;
constexpr uint32_t kW4RawBytes = kTcBM * 128;  // one raw code tile
constexpr uint32_t kW4ACols = kTcBK / 2;       // TMEM columns of one A tile: 64 f16 per row, two per column

constexpr size_t kSmSmem = 228 * 1024;
constexpr int kTcMostSplits = 8;   // CTAs of a cluster
constexpr int kTcHalvesRows = 64;  // operand rows up to which two CTAs' double accumulators (4 np columns each) share an SM
constexpr size_t kCtaFixed = 1024 + 1024 + 256;  // per CTA: system reserve, alignment slack, barriers

// K-splits per tile: fill whole waves of the CTA slots, keep at least four 64-wide k-blocks per split; no split at
// all when there is a tile for every SM.  The kernel is memory-bound, so what matters is that all CTAs are resident
// together and every SM slot streams.
inline int tc_pick_splits(int num_sms, int tiles, int kb_total, int slots, int min_kb = 4) {
    int best = 1;
    double best_eff = 0.0;
    if (tiles >= num_sms) return 1;  // every SM has a tile of its own: splitting only adds reductions
    for (int s = 1; s <= kTcMostSplits; ++s) {
        if (s > 1 && kb_total / s < min_kb) break;
        const int ctas = tiles * s, waves = (ctas + slots - 1) / slots;
        const double eff = (double)ctas / ((double)waves * slots);
        if (eff > best_eff + 0.02) { best_eff = eff; best = s; }
    }
    return best;
}

inline size_t tc_stage_bytes(int np) { return (size_t)kTcBM * kTcBK * 2 + 2 * (size_t)np * kTcBK * 2; }
// pipeline stages with `occ` CTAs per SM (0: they do not fit)
inline int tc_stages_at(int np, int occ) {
    const size_t stage = tc_stage_bytes(np), room = std::min<size_t>(kSmSmem / occ, 227 * 1024);
    return room < kCtaFixed + 2 * stage ? 0 : (int)std::min<size_t>(occ == 1 ? 8 : occ == 2 ? 4 : 3, (room - kCtaFixed) / stage);
}
// hi | lo as one operand doubles the accumulator columns; all CTAs of a launch that can be resident on an SM get their tensor memory
// at once
inline int tc_cols(int np, int occ, int *wide) {
    int cols = 32;
    while (cols < 2 * np) cols <<= 1;
    *wide = (2 * np <= 256 && occ * cols <= 512) ? 1 : 0;
    if (!*wide) { cols = 32; while (cols < np) cols <<= 1; }
    return cols;
}

// tc_gemm_kernel: CTAs per SM and K-splits.  `decode`: the rows are a decode step's (not a prefill pass's).  `most_kb`: the most
// k-blocks that one accumulator may sum (0: as many as it comes to); 0 splits: no plan keeps to it.
struct TcPlan { int occ, splits, halves; };
inline TcPlan tc_plan(int num_sms, int np, int tiles, int K, bool allow_split, bool decode, int most_kb = 0) {
    TcPlan p{};
    // CTAs per SM: two with three stages each, or three with two when that puts more CTAs of one wave to work (while
    // one CTA drains its accumulator and takes part in the cluster reduction the others keep the weight stream going);
    // one with deep stages when the operand tiles are too large for that.
    p.occ = tc_stages_at(np, 2) ? 2 : 1;
    p.splits = tc_pick_splits(num_sms, tiles, K / kTcBK, num_sms * p.occ);
    if (p.occ == 2 && tc_stages_at(np, 3) && allow_split) {
        const int s3 = tc_pick_splits(num_sms, tiles, K / kTcBK, num_sms * 3);
        if (tiles * s3 > tiles * p.splits && tiles * s3 <= num_sms * 3) { p.occ = 3; p.splits = s3; }
    }
    // Decode steps of up to 64 operand rows: one CTA per SM, in the shared memory of half an SM, where it still has a long
    // enough run of k-blocks: the other half takes the CTAs of the projection behind this one (and of the dequantising kernel
    // beside it), which set up and request their first weights while this grid drains.  8B-class shape, 64 rows: two or three
    // CTAs per SM 2083 us a step (8 blocks), so 2005; with fewer than a dozen k-blocks per CTA (1B-class shape, 8 rows) more
    // CTAs win (1118 against 1224-1337), and so they do in prefill (58 positions, 2 blocks: 589 against 596 us).  The run of
    // k-blocks is summed in two halves, whose accumulators fit twice into an SM's tensor memory up to 64 rows.
    if (p.occ >= 2 && allow_split && tiles < num_sms && decode && np <= kTcHalvesRows) {
        const int s1 = tc_pick_splits(num_sms, tiles, K / kTcBK, num_sms);
        if (s1 >= 2 && K / kTcBK / s1 >= 12) { p.splits = s1; p.occ = 2; p.halves = 1; }
    }
    if (!allow_split) p.splits = 1;
    // A bound on the sums: two accumulators where they fit, and then as few splits as keep to it - more of them, in whole waves of
    // CTAs, only add reductions (one 8B-class block's pass that ends on 5 rows: gate/up in 2 splits 268 us, in 5 278).
    const int kb = K / kTcBK;
    if (most_kb && ((kb + p.splits - 1) / p.splits + p.halves) / (1 + p.halves) > most_kb) {
        p.occ = tc_stages_at(np, 2) ? 2 : 1;
        p.halves = p.occ == 2 && np <= kTcHalvesRows ? 1 : 0;
        p.splits = std::max(p.splits, (kb - 1) / (most_kb << p.halves) + 1);
        if (p.splits > kTcMostSplits) p.splits = 0;
    }
    return p;
}

// tc_gemm_w4_kernel: stages (an even number: the two dequantisation warps of a lane quarter alternate), CTAs per SM, K-splits
// in whole raw tiles, accumulators.  hi | lo as one operand (`wide`) and `most_kb` as above.
struct W4Plan { int occ, n_stages, splits, wide, sets, cols; };  // cols: tensor-memory columns per CTA (occ * cols > 512: does not fit)
inline W4Plan w4_plan(int num_sms, int np, int tiles, int K, bool decode, int most_kb = 0) {
    W4Plan p{};
    const size_t stage = 2 * (size_t)np * kTcBK * 2;  // the activations' hi and lo tiles; the A tiles are in tensor memory
    const size_t raw = (size_t)kW4RawBufs * kW4RawBytes;
    // two CTAs per SM (16 dequantisation warps) when two stages fit in half of the shared memory
    const bool two = 2 * stage + raw + 4096 <= 110 * 1024;
    p.occ = two ? 2 : 1;
    p.n_stages = two ? (int)std::min<size_t>(4, (110 * 1024 - raw - 4096) / stage)
                     : (int)std::max<size_t>(2, std::min<size_t>(4, (214 * 1024 - raw) / stage));
    p.n_stages &= ~1;
    auto cols_for = [&](int acc) { int cols = 32; while (cols < acc + p.n_stages * (int)kW4ACols) cols <<= 1; return cols; };
    p.wide = (2 * np <= 256 && p.occ * cols_for(2 * np) <= 512) ? 1 : 0;
    p.sets = 1;
    // in raw tiles of four k-blocks: at least four per split, two when K is so short that four would allow only two
    // splits (measured on the 1B shape, K = 2048: 2 -> 4 splits 35 -> 31 us per layer for QKV, 33 -> 27 us for O)
    const int raw_tiles = K / (kTcBK * kW4Super), min_raw = raw_tiles <= 8 ? 2 : 4;
    p.splits = tc_pick_splits(num_sms, tiles, raw_tiles, num_sms * p.occ, min_raw);
    // Decode steps: splits for one CTA per SM, the rest of the SM belongs to tc_gemm_kernel's CTAs beside this grid and to the
    // next projection's (1B-class, 8 rows 1120 -> 1109 us a step) - where the longer run can be summed in two accumulators of
    // half of it each, so that no sum inside the tensor cores takes more inputs: its error grows with their number (8B-class QKV on
    // exact weights against 64-bit arithmetic: 1.5e-7 split over every slot, 2.0e-7 with one accumulator and half the splits, 1.1e-7
    // with two).  That is up to 32 operand rows: 2 x 2 np columns beside four A tiles are the 256 that one accumulator takes as well.
    // With fewer than eight raw tiles the clusters this asks for cost more than they bring (tiny shape, 77 rows 149.8 -> 152.4),
    // and in prefill passes they do whatever K is (8B-class, 20 positions on the exit layers 524 -> 541).
    if (two && decode && raw_tiles >= 8) {
        const int s1 = tc_pick_splits(num_sms, tiles, raw_tiles, num_sms, min_raw);
        if (s1 >= p.splits) p.splits = s1;
        else if (p.wide && p.occ * cols_for(4 * np) <= 512 && (raw_tiles + s1 - 1) / s1 <= 2 * ((raw_tiles + p.splits - 1) / p.splits)) {
            p.splits = s1;
            p.sets = 2;
        }
    }
    if (most_kb && (raw_tiles + p.splits - 1) / p.splits * kW4Super > most_kb * p.sets) {  // (as in tc_plan)
        p.sets = p.wide && p.occ * cols_for(4 * np) <= 512 ? 2 : 1;
        const int most_raw = most_kb * p.sets / kW4Super;
        p.splits = most_raw ? std::max(p.splits, (raw_tiles - 1) / most_raw + 1) : 0;
        if (p.splits > kTcMostSplits) p.splits = 0;
    }
    p.cols = cols_for(p.sets * (p.wide ? 2 * np : np));
    return p;
}

// Where tc_gemm_w4_kernel looks, before the grids before it are through, whether it will have rows (and may request its codes at once):
// the entry of n_riv to read, or -1 for the rows of the pass.  `at`: the entry that describes the rows of this block; `settled`: it was
// written before the block before this one, so it may be read; `before`: the entry before it, whose count is no higher; `all`: the host
// knows that every row is on the exit layers.  Steps write an entry per block (at = l - 1, never settled), passes whose depths the host
// knows only those behind blocks that rows leave at: every other entry holds whatever an earlier step left there.  Short passes in a
// context that had not decoded, entry at - 1 / this, us: mini shape, 118 positions, depth 3 of 6 388 / 381, tiny shape, 100 positions,
// depth 3 of 4 213 / 210.
inline int exit_rows_hint(bool all, int at, int before, bool settled) { return all ? -1 : settled ? at : before; }

// Operand rows per CTA of a step with np of them, from its widest projection (`tiles` 128-feature tiles, K inputs).  A small model's weight
// tiles and K-splits are CTAs for a fraction of the chip (mini shape: 24 for QKV), each of which then finishes all the rows alone; so
// the rows are dealt out as well, 16 to 64 to a CTA, while all CTAs of the widest projection find a place at once, two to an SM.  (The
// 1B and 8B shapes fill the chip with their weights: there every row tile would only stream them again.)  The K-splits, and so what
// one accumulator sums, stay those of all rows together.  Mini shape, us a block of a 118-row prompt, one tile / tiles of 32: QKV 24 /
// 11, O 12 / 10, gate/up 18 / 10, down 15 / 8; the prompt 587 / 409.
inline int tc_row_tile(int num_sms, int np, int tiles, int K, bool decode) {
    const int splits = tc_plan(num_sms, np, tiles, K, true, decode).splits;
    for (int nt = 16; nt <= 64 && nt < np; nt *= 2)
        if (tiles * splits * ((np + nt - 1) / nt) <= 2 * num_sms) return nt;
    return np;
}
// The plan for np rows, in the shared and tensor memory of CTAs that take nt of them.
inline W4Plan w4_row_plan(W4Plan p, int np, int nt) {
    if (nt >= np) return p;
    const size_t stage = 2 * (size_t)nt * kTcBK * 2, raw = (size_t)kW4RawBufs * kW4RawBytes;
    p.occ = 2;
    p.n_stages = (int)std::min<size_t>(4, (110 * 1024 - raw - 4096) / stage) & ~1;
    p.wide = 1;
    p.cols = 32;
    while (p.cols < p.sets * 2 * nt + p.n_stages * (int)kW4ACols) p.cols <<= 1;
    return p;
}

inline size_t tc_smem_bytes(int n_pad, int n_stages) {  // (the finished tile reuses the stages: the launch checks the fit)
    return 1024 + (size_t)n_stages * tc_stage_bytes(n_pad) + sizeof(uint64_t) * (2 * n_stages + 1) + 64;
}
inline size_t tc_w4_smem_bytes(int n_pad, int n_stages) {
    const size_t stage = 2 * (size_t)n_pad * kTcBK * 2;
    return 1024 + (size_t)n_stages * stage + (size_t)kW4RawBufs * kW4RawBytes + sizeof(uint64_t) * (2 * n_stages + 2 * kW4RawBufs + 1) + 64;
}

// Tensor memory: a grid starts once the CTAs of the grids before it have their columns (tc_gemm_kernel), so an allocation that has to wait
// is a delay and no more.  Inside a step it need not wait: whatever mix of its projections' launches fits into an SM's shared memory fits
// into its 512 columns, and requests are padded until it does.  (The LM head of a prefill pass has the prompt ends' rows, not the
// pass's: beside the dequantising CTAs of a pass of 193 to 224 rows its own may wait.)
struct TcFootprint { size_t smem; int cols; };
constexpr size_t kTcTwoSmem = 90 * 1024;  // two such CTAs leave no room for a third of any launch
// tc_gemm_kernel with np operand rows per CTA: two CTAs per SM, with one accumulator or two, three; or the one that fits.
inline int tc_footprints(int np, TcFootprint *out /* [3] */) {
    int n = 0, wide;
    for (int occ = tc_stages_at(np, 2) ? 2 : 1; occ <= 3; ++occ) {
        const int st = tc_stages_at(np, occ);
        if (!st) break;
        out[n].smem = tc_smem_bytes(np, st);
        out[n++].cols = tc_cols(np, occ, &wide);
        if (occ == 2 && np <= kTcHalvesRows) {
            out[n].smem = std::max(out[n - 1].smem, kTcTwoSmem);
            out[n].cols = 2 * out[n - 1].cols;
            ++n;
        }
        if (occ == 1) break;
    }
    return n;
}
// The most columns that CTAs of these footprints may ask of one SM.
inline int most_columns(const TcFootprint *fp, int n, size_t room = kSmSmem) {
    if (!n) return 0;
    int most = 0;
    for (int i = 0; i * fp[0].smem <= room; ++i) most = std::max(most, i * fp[0].cols + most_columns(fp + 1, n - 1, room - i * fp[0].smem));
    return most;
}
// What a step with np operand rows, nt per CTA, launches on tc_gemm_kernel (the LM head may have all rows in a CTA).
inline int step_footprints(int np, int nt, TcFootprint *out /* [6] */) {
    int n = tc_footprints(nt, out);
    if (nt == np) return n;
    const int n0 = n;
    n += tc_footprints(np, out + n);
    for (int i = n0; i < n; ++i) out[i].smem = std::max(out[i].smem, kTcTwoSmem);
    return n;
}
// Shared memory that a CTA of tc_gemm_w4_kernel asks for: its own, no more than p.occ of them, and the rule above beside the CTAs of
// tc_gemm_kernel of the same step; 0: there is none.
inline size_t w4_smem_request(const W4Plan &p, int np, int nt) {
    if (p.occ * p.cols > 512) return 0;
    TcFootprint fp[7];
    const int n = step_footprints(np, nt, fp);
    TcFootprint &mine = fp[n] = {std::max(tc_w4_smem_bytes(nt, p.n_stages), kSmSmem / (p.occ + 1) + 1024), p.cols};
    while (most_columns(fp, n + 1) > 512) {
        mine.smem += 4096;
        if (mine.smem > kSmSmem / p.occ - 1024) return 0;
    }
    return mine.smem;
}

// tc_gemm_wide_kernel: k-blocks per accumulation segment.  1024 inputs, 512 where K is short, and never more than the longest
// sum that the batch kernels' K-splits make of the same projection in passes of `pass_rows` rows (1B-class shape: 256 inputs for
// O and gate/up, 384 for QKV; 8B-class: 1024 for all), since the error of a sum inside the tensor cores grows with its length:
// cache of 300 positions, mini shape, against 64-bit arithmetic 5.5e-4 with 512 inputs everywhere, 5.06e-4 so, as in short
// passes; logits of 1000 positions, 1B-class blocks, 1.78e-4 and 1.72e-4.  It costs 1-2 % of a prompt on those shapes.
inline int tc_wide_segment(int num_sms, int pass_rows, int tiles, int K, bool f16) {
    const int np = std::min(256, (pass_rows + 15) / 16 * 16), kb = K / kTcBK;
    int run;
    if (f16) {
        const int splits = w4_plan(num_sms, np, tiles, K, false).splits, raw = kb / kW4Super;
        run = (raw + splits - 1) / splits * kW4Super;
    } else {
        const int splits = tc_plan(num_sms, np, tiles, K, true, false).splits;
        run = (kb + splits - 1) / splits;
    }
    return std::min(K >= 4096 ? 16 : 8, run);
}

// Long passes of small models: where a projection has few features (O and down) its tiles keep no more than half of the pairs busy,
// each with the whole run of k-blocks; then it goes to tc_gemm_kernel instead, 64 rows to a CTA, in as many K-splits as keep every
// sum as short as the pair kernel's (two accumulators per CTA) - if its CTAs all find a place at once.  0: not so.  us a prompt, all
// projections on the pair kernel / so: mini, full depth 256 rows 463 / 418, 512 499 / 470, 1024 590 / 563; five of six blocks on the
// exit layers 535 / 507, 608 / 563, 676 / 662; d 1024, full depth 256 rows 388 / 335, 512 436 / 396.  (Fewer than 16 k-blocks are
// no run to split.)
constexpr int kTcPassRows = 64;
inline int tc_pass_splits(int num_sms, int pass_rows, int tiles, int K, bool f16, int n) {
    const int row_tiles = (n + kTcPassRows - 1) / kTcPassRows, kb = K / kTcBK, splits = (kb - 1) / (2 * tc_wide_segment(num_sms, pass_rows, tiles, K, f16)) + 1;
    return tiles <= 8 && kb >= 16 && tiles / 2 * row_tiles <= num_sms / 4 && splits <= kTcMostSplits && tiles * splits * row_tiles <= 2 * num_sms ? splits : 0;
}

// Whether the last block of a long pass runs behind QKV (O, gate / up, down; f16: on the exit layers) on the kernels of decode steps,
// for `ends` prompt ends.  Those put every SM to work on a few rows, by K-splits, where the pair kernel has a pair per 256 features
// and every exit-layer matrix is expanded for it first; their time grows with the rows sooner.  And only where every sum inside the
// tensor cores stays as short as the pair kernel's (up to four rows on the backbone never enter them): with the batch kernels' own
// plans the logits of 20 ends behind one 8B-class block are 1.04e-5 from 64-bit arithmetic (8.4e-6 on the exit layers), on the pair
// kernel 9.9e-6 (7.6e-6), with this bound 9.6e-6 (7.2e-6).  Passes of 512 positions through one block, us, pair kernel / so:
//   ends             5         16        32        48        64        96
//   8B   backbone  383/268   384/268   387/276   394/296   407/316   (down: 224 k-blocks, 8 splits x 2 accumulators x 16 up to 64 rows)
//        exit      566/298   565/299   573/309   (two accumulators up to 32 rows)
//   3072 backbone  271/198   271/198   275/207   284/223   293/237   317/316
//        exit      357/224   357/224   362/237   370/258   380/274   406/314
//   1B   backbone  242/168   241/167   244/176   250/193   258/203   277/272   (128: 293/309)
//        exit      288/179   286/177   292/184   299/204   309/218   328/242
//   mini backbone  133/108   132/110   139/116   150/126   149/134   159/153   (128: 170/172)
//        exit      144/122   147/124   151/132   164/137   162/145   172/162
constexpr int kTcEndsMost = 96;
inline bool tc_ends_fit(int num_sms, int pass_rows, int ends, int d, int qdim, int F, bool f16) {
    if (ends <= 4 && !f16) return true;
    const int np = (ends + 15) / 16 * 16, shapes[3][2] = {{d / kTcBM, qdim}, {F / 64, d}, {d / kTcBM, F}};
    for (const auto &[tiles, K] : shapes) {
        const int most = tc_wide_segment(num_sms, pass_rows, tiles, K, f16);
        if (!(f16 ? w4_plan(num_sms, np, tiles, K, false, most).splits : tc_plan(num_sms, np, tiles, K, true, false, most).splits)) return false;
    }
    return ends <= kTcEndsMost;
}

// Rows from which a prefill pass that the batch kernels could take as well (up to `max_rows` rows, 256 at most) is a long one.
// `exit_blocks` of its L blocks have rows on the exit layers.  The pair kernel's time hardly depends on the rows up to 256 - its
// tiles fill the chip late, and every exit-layer matrix is expanded first - the batch kernels' grows with them, the later the wider
// the blocks.  Measured, batch / pair kernels, us (blocks on the exit layers / all, 1 prompt):
//   mini 0/6      129 rows 642 / 490
//   d 1024 0/4    160: 460 / 462   176: 481 / 467      3/4  176: 513 / 535   192: 540 / 534
//   1B 0/3        144: 553 / 647   145: 933 / 645      2/3  176: 771 / 779   192: 785 / 778
//   d 3072 0/3    144: 636 / 707   145: 1018 / 708     2/3  176: 890 / 904   192: 919 / 907
//   8B 0/2        160: 783 / 820   176: 851 / 838      1/2  208: 879 / 1036  256: 1019 / 1056   257 (two passes): 1206 / 1132
inline int tc_long_pass_rows(int d, int L, int exit_blocks, int max_rows) {
    const int base = d >= 4096 ? 160 : d >= 1024 ? 144 : 128, more = d >= 4096 ? 220 : d >= 1024 ? 60 : 0;
    return std::min(base + more * exit_blocks / L, std::min(max_rows, 256)) + 1;
}

// Where the batch kernels' rows are dealt out over CTAs (tc_row_tile), a short pass is the faster one for longer: up to this many rows,
// where the mini shape's tiles become wider than 32 rows.  (The tiny shape's stay narrow, and its short passes ahead up to 256.)
// Batch / pair kernels (O and down of the latter by tc_pass_splits), us, 1 prompt:
//   tiny 0/4   129 rows 209 / 239   145: 206 / 239   176: 209 / 237   192: 209 / 236   200: 216 / 242   224: 218 / 241   256: 224 / 240
//        3/4   129: 231 / 275       145: 224 / 277   176: 231 / 276   192: 232 / 276   200: 239 / 279   224: 240 / 277   256: 246 / 278
//   mini 0/6   129: 365 / 396       145: 372 / 396   176: 377 / 399   192: 384 / 402   200: 453 / 406   224: 462 / 409   256: 476 / 410
//        5/6   129: 411 / 486       145: 408 / 485   176: 417 / 486   192: 421 / 488   200: 479 / 493   224: 489 / 494   256: 494 / 497
constexpr int kTcTiledPassRows = 192;
inline int tc_tiled_pass_rows(int num_sms, int tiles, int K) {
    return tc_row_tile(num_sms, kTcTiledPassRows, tiles, K, false) < kTcTiledPassRows ? kTcTiledPassRows : 0;
}

// Attention of a long pass's n rows, which see `seen` positions in all: the tcgen05 kernel where they look back far enough on average, at
// 128 positions (below, its tiles are mostly padding: 1B-class, 5 prompts of 160 positions 1017 against 995 us, 4 of 240 level), at 64
// where the warp-level kernel's CTAs, 16 positions and a KV head each, are one per SM at most, so that one's walk over the keys is the
// time it takes (mini shape, 5 prompts of 160 479 against 505, 4 of 240 500 against 550; of 90 460 against 456).
inline bool tc_long_attention(int num_sms, int warp_ctas, int n, long long seen) { return seen >= (warp_ctas <= num_sms ? 64LL : 128LL) * n; }

}  // namespace river
