// Job descriptor shared by the host planner and the walk kernels.
//
// A job is one generalized BB/FG sum (Eq. bbfgrepeated) in canonical form:
//   * K product columns, each with multiplicity 1 (repeated columns are
//     expanded by the planner, so the product length equals K);
//   * one pinned row (delta = +1, Sec. 2.2) folded into the base column sums;
//   * nrows digit rows; digit j has radix R_j = M_j + 1 and counts the -1
//     entries Delta_j among the M_j copies of that row (Eq. Deltak).  The
//     first nbin digits are binary (M_j = 1) and vary fastest.
// The addend index i in [0, C), C = prod_j R_j, is read as a mixed-radix
// number (digit 0 least significant) and mapped to the reflected n-ary Gray
// code of Sec. 2.2; each addend is
//     (-1)^{sum Delta} prod_j C(M_j, Delta_j) * prod_col c_col
// with c_col = c0_col - sum_j Delta_j * (2 a_j,col).
//
// kind == BS_KIND_PERM   : one output, sum * 2^{scale_exp}
// kind == BS_KIND_MINORS : K outputs, output l = sum over addends of
//                          (-1)^.. C(..) prod_{col != l} c_col, scaled by
//                          2^{colexp[l]} (Laplace minors, one column removed).
#pragma once
#include <stdint.h>

#define BS_KIND_PERM 0
#define BS_KIND_MINORS 1

#define BS_MAX_COLS 48     // product columns per job
#define BS_MAX_DIGITS 48   // digit rows per job
#define BS_MAX_PHOTONS 48  // n = sum of multiplicities

struct bs_job {
    uint64_t C;            // number of addends = prod of radices
    uint64_t task_begin;   // first global warp-task index of this job
    uint32_t ntasks;       // warp tasks in this launch: 32 (or 16) chunks of 2^log2L addends each
    uint32_t task_offset;  // job-local number of this launch's first task (a launch may walk a slice)
    int32_t K;             // product columns
    int32_t nrows;         // digit rows
    int32_t nbin;          // leading binary digits
    int32_t kind;          // BS_KIND_PERM or BS_KIND_MINORS
    int32_t log2L;         // chunk length exponent (one chunk per lane per task)
    int32_t out_index;     // perm: output slot; minors: first of K output slots
    int32_t n;             // photons of the formula (prefactor 2^(1-n))
    int32_t prec;          // BS_PREC_*: which kernels walk the job
    int64_t data_off;      // complex elements: c0[KP] then 2a[nrows][KP], KP = BS_ROW_STRIDE(K)
    int64_t meta_off;      // ints, see BS_META_* below
    int64_t partial_off;   // double-double complex slots: ntasks * (perm ? 1 : K)
    int64_t src_off;       // source matrix: element offset of entry (0, 0)
    int32_t src_ld;        // source leading dimension (complex elements)
    int32_t src_trans;     // 1: formula row r / column c read source (c, r)
    int32_t formula;       // BS_JOB_BBFG (0), BS_JOB_RYSER or BS_JOB_NW (plain permanents, FP64)
    int32_t walk_log2;     // a warp task walks 2^walk_log2 consecutive tasks of the cut, summed in one slot
    int32_t fold_log2;     // the reduce kernel adds 2^fold_log2 consecutive slots first (bs_cut)
    int32_t reseed_log2;   // FP32 jobs: > 0 re-seeds the column sums from the matrix every 2^reseed_log2
                           // steps inside a chunk as well (0: at chunk starts only)
};

#define BS_MAX_GROUP 16  // most tasks of a group (2^walk_log2, 2^fold_log2)

// Formula of a job (see bs_perm_formula).  Ryser and Nijenhuis-Wilf jobs
// walk the columns of the matrix as binary digits with the rows as product
// columns; the walk kernels are the same, only packing and prefactor differ.
#define BS_JOB_BBFG 0
#define BS_JOB_RYSER 1
#define BS_JOB_NW 2

// Integer metadata of a job, at meta_off (int32 units; meta_off even):
//   radix[nrows]        digit radices R_j = M_j + 1 (binary digits first)
//   digit_src[nrows]    source row of each digit
//   col_src[K]          source column of each product column
//   colexp[K]           power-of-two column scale chosen by the pack kernel
//   pinned_src          source row of the pinned (delta = +1) row
//   split               1: a column has parts of its own scale (pack kernel)
//   binom[]             uint64 table written by the pack kernel: for each
//                       digit j in order, C(M_j, d) for d = 0..M_j
//                       (nrows + n - 1 entries in all)
// colexp values: the exponent e of the column's scale, how far the bound of its
// imaginary part lies below that of its real part (d > 0) or above it (d < 0;
// both scaled alike: 0), and marks of a part with an entry that is not finite.
#define BS_COLEXP(e, d) (((e) + 2048) | (((d) + 1024) << 12))
#define BS_COLEXP_E(x) (((x) & 4095) - 2048)
#define BS_COLEXP_D(x) ((((x) >> 12) & 2047) - 1024)
#define BS_COLEXP_NAN_RE (1 << 24)
#define BS_COLEXP_NAN_IM (1 << 25)
#define BS_META_RADIX(jb) ((jb).meta_off)
#define BS_META_DIGIT_SRC(jb) ((jb).meta_off + (jb).nrows)
#define BS_META_COL_SRC(jb) ((jb).meta_off + 2 * (jb).nrows)
#define BS_META_COLEXP(jb) ((jb).meta_off + 2 * (jb).nrows + (jb).K)
#define BS_META_PINNED(jb) ((jb).meta_off + 2 * (jb).nrows + 2 * (jb).K)
#define BS_META_SPLIT(jb) (BS_META_PINNED(jb) + 1)
#define BS_META_BINOM(jb) ((jb).meta_off + 2 * (jb).nrows + 2 * (jb).K + 2)
#define BS_META_SIZE(nrows, K, n) (2 * (nrows) + 2 * (K) + 2 + 2 * ((nrows) + (n)))

// Row stride of the packed matrix c0 / 2a: K rounded up to a multiple of 4,
// the width KB of the bucket kernel that walks the job (inside a kernel the
// stride is the compile-time KB), so FP32 rows are whole 16-byte column pairs
// and every bucket column has a slot.  Pad columns are neutral: rows hold
// zeros and c0 holds the value 1, so a pad column's sum stays exactly 1 and
// leaves every product unchanged.
#define BS_ROW_STRIDE(K) ((((K) + 3) / 4) * 4)
// Double-float minors: K rounded up to a multiple of 8 (the DF bucket width).
#define BS_ROW_STRIDE_DF(K) ((((K) + 7) / 8) * 8)
#define BS_ROW_STRIDE_P(K, prec, kind) (BS_DF_MINORS(prec, kind) ? BS_ROW_STRIDE_DF(K) : BS_ROW_STRIDE(K))
// Double-float permanents run in the FP64 kernels' fixed point, which is more
// accurate (2^-63 of a column's bound against 2^-44) and faster at every width
// than products on the FP32 pipe were (calls: 12 x 12 98 -> 55 us, 20 x 20
// 160 -> 105, 24 x 24 645 -> 480, 26 x 26 2.63 -> 1.80 ms, 30 x 30 34.8 -> 28.9
// ms).  Only double-float minors have kernels of their own: at 30 columns they
// take 38.7 ms where the fixed point takes 49.0.
#define BS_DF_MINORS(prec, kind) ((prec) == BS_PREC_DF && (kind) == BS_KIND_MINORS)

// Task partials of the fixed-point kernels are in units of 2^-BS_FIX_BIAS of the
// product of the column bounds, so that addends far below it keep their
// digits; the reduce kernel takes the factor out.
#define BS_FIX_BIAS 512
#define BS_FIXED(prec, kind) ((prec) == BS_PREC_FP64 || ((prec) == BS_PREC_DF && (kind) == BS_KIND_PERM))

// Precision of a job: the kernel family that walks it.
//   FP64: 64-bit fixed point (walk_fix.cuh; data in pairs of 64-bit integers);
//   FP32: single-precision packed pairs (data in complex floats);
//   DF:   minors in double-float (float pairs, exact fixed-point column sums;
//         data in 16-byte units like FP64), permanents as FP64.
#define BS_PREC_FP64 0
#define BS_PREC_FP32 1
#define BS_PREC_DF 2
#define BS_NPREC 3

// Double-double complex partial: re = (re_hi, re_lo), im = (im_hi, im_lo).
struct bs_zdd {
    double re_hi, re_lo, im_hi, im_lo;
};

// Device status word values (written by kernels, read by the host).
#define BS_STATUS_OK 0
#define BS_STATUS_TIMEOUT 1
#define BS_STATUS_BADJOB 2
