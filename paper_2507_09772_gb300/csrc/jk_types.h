// Plain-data records shared by the host planner (nvcc/g++) and the
// runtime-compiled integral kernels (NVRTC). No includes: NVRTC compiles this
// file without the CUDA toolkit headers.
#pragma once

// One significant shell pair (a, b), oriented so that the shell type of a
// (l, then nprim) is >= that of b. Pairs of one pair class are stored
// contiguously, grouped by molecule and sorted by descending Q inside a
// molecule, so that a ket scan can stop at the first Q that fails the bound.
// 16-byte alignment: records that lanes gather load as 16-byte vectors
struct alignas(16) JkPair {
    int a, b;          // global shell indices
    int mol;           // molecule index
    int pp_off;        // first primitive pair (na*nb of them, a-major)
    int a_ao, b_ao;    // molecule-local Cartesian AO offsets
    int a_loc, b_loc;  // molecule-local shell indices (density-max table)
    double Q;          // Schwarz factor sqrt(max |(mu nu|mu nu)|)
    double ABx, ABy, ABz;  // A - B (horizontal recurrence)
    float Qf;              // Q rounded to FP32 (the FP32 screening path)
    float padf;
};

// What a kernel reads of every candidate ket: one 16-byte vector for the
// screening (32 candidates in a row are four lines; the JkPair records would be
// 20), and a 64-byte record for a quartet in FP32 (the first half) or two
// floats. Arrays aligned with the pairs.
struct alignas(16) JkKetScr {
    float Qf;
    int a_loc, b_loc;
    int pad;
};
struct alignas(16) JkRec {
    int pp_off, a_ao, b_ao;
    int same;                // a == b
    float ABxf, AByf, ABzf, ABxl, AByl, ABzl;   // A - B rounded to FP32, and what the rounding left
    float Axh, Axl, Ayh, Ayl, Azh, Azl;   // centre A in two floats
};

// Per primitive pair (alpha_i on a, beta_j on b), p = alpha + beta:
//   P    = (alpha A + beta B) / p
//   PA   = P - A
//   K    = c_i c_j exp(-alpha beta |A-B|^2 / p) / p
//   inv2p = 1 / (2 p)
//   q    = primitive Schwarz factor sqrt(max |(ij|ij)|) (coefficients
//          included); a shell pair's primitive pairs are sorted by q,
//          largest first, so primitive loops can stop at the first
//          q_ij q_kl Dmax at or below the primitive threshold
struct alignas(16) JkPrimPair64 {
    double Px, Py, Pz, p;
    double PAx, PAy, PAz, K;
    double inv2p, q;
    float qf, padf;   // qf: q rounded to FP32 (the primitive screen compares in FP32)
    double pad2;
};
struct alignas(16) JkPrimPair32 {
    float Px, Py, Pz, p;
    float PAx, PAy, PAz, K;
    float inv2p, q, pad1, pad2;
};

// The same in two-float arithmetic (x = xh + xl, 48 bits): the split tier,
// which forms P - Q as (P - A) + (A - C) - (Q - C): the difference of the
// absolute centres would carry 2^-49 of their distance from the origin, which
// the tightest products (exponents of thousands) turn into 1e-12 of the integral.
struct alignas(16) JkPrimPairDf {
    float ph, pl, Kh, Kl;
    float PAxh, PAxl, PAyh, PAyl, PAzh, PAzl;
    float i2ph, i2pl, q, pad[3];
};

// Per molecule of a handle.
struct JkMol {
    const double *D;   // n_dm x nao x nao (Cartesian)
    const float2 *D2;  // the same as two floats, read by the split tier (nullptr when it does not run)
    double qmax2;      // largest Q squared (0: no quartets in two floats)
    const float *D32;  // the same rounded to FP32, read by the FP32 tier (nullptr when it does not run)
    double *J;         // half-matrix accumulator X, symmetrised after the build
    double *K;         // half-matrix accumulator Y
    int nao;           // Cartesian functions
    int nsh;           // shells
    long long dmax_off;  // offset of this molecule's nsh x nsh block-max table
};

struct JkRouterDev;
struct JkPairFeat;

// Bound up to which a molecule's FP64-tier quartets run in two floats: split x
// max Q^2 x the largest density element the screening uses (dmol), at least
// split_min; 0 (none) where the largest |D| itself (dreal; infinite for a
// density that is not finite) or the largest product with an integral is not
// well inside the FP32 range: sums of products of integrals and density
// elements are formed in it, and halves below 1.2e-38 are lost.
__device__ __forceinline__ double jk_split_threshold(double split, double split_min, double qmax2, double dmol, double dreal)
{
    const double s = qmax2 * dreal;
    if (!(dreal > 1e-15 && dreal < 1e15 && s > 1e-20 && s < 1e30)) return 0.0;
    return fmax(split_min, __dmul_rn(__dmul_rn(split, qmax2), dmol));
}

// splitmix64 (Steele, Lea and Flood, OOPSLA 2014): counter-based random bits.
__host__ __device__ __forceinline__ unsigned long long jk_mix64(unsigned long long z)
{
    z += 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// One class pair (bra pair class, ket pair class) of a launch. A launch runs
// every class pair that shares a kernel (angular momenta and fragment shape),
// whatever its primitive counts.
struct JkSub {
    const JkPair *bra;           // pairs of the bra class
    const JkPair *ket;           // pairs of the ket class
    const JkKetScr *ket_scr;     // aligned with ket
    const JkRec *ket_rec, *bra_rec;
    const int *ket_beg;          // per molecule: first ket index in the ket class
    const int *ket_end;          // per molecule: one past the last
    const JkPairFeat *bra_feat;  // aligned with bra / ket
    const JkPairFeat *ket_feat;
    int nbra;
    int same_class;              // ket class == bra class: ket index >= bra index
    int nab, ncd;                // primitive pairs of a bra / ket pair
    int chunk;                   // kets per work item
    int split, split_ab;         // work items that share the primitive quartets: in all, and by the bra's pairs
    int group;                   // launch it belongs to
    int launch;                  // class pair index: statistics, routed lists
    int seed;                    // bra i belongs to part (i + seed) % part_count of a partitioned build
    double tight;                // factor of the split threshold for its angular momenta
};

// A work item: the candidates [kb, ke) of the ket class for one bra pair, and
// of the primitive pairs of the bra number s % split_ab, + split_ab, ... and of
// the ket number s / split_ab, + split / split_ab, ... (J and K are linear in
// them); sub = class pair + s * 2^23 (at most 80 shell types, 5.2 million class
// pairs, and 256 shares).
struct alignas(16) JkItem {
    int sub, bra, kb, ke;
};

// A band quartet the learned router released from the FP64 tier: bra pair
// `item` of the class pair's bra class, ket pair `ket` of its ket class, and
// the density factor its screening used. The FP32 list kernel (MODE 3) of
// the class pair evaluates it.
struct alignas(16) JkRouted {
    int item, ket;
    float dmq;
    int pad;
};

// Arguments of one launch (passed by value).
struct JkClassArgs {
    const JkSub *subs;           // the class pairs of the launch
    int nsub;
    const JkItem *items;         // work items, listed per build by jk_plan_kernel
    const unsigned long long *nitems;
    unsigned long long *work;    // work counter (zeroed before the launch)
    const JkPrimPair64 *pp64;
    const JkPrimPair32 *pp32;
    const JkPrimPairDf *ppdf;
    const JkMol *mols;
    const double *dmax;          // block max |D| tables, all molecules
    const float *dmax32;         // the same rounded to FP32
    const double *dmax_mol;      // per molecule: max over its table
    const double *rys64;         // FP64 Rys tables
    const float *rys32;          // FP32 Rys tables
    const float *rysdf;          // two-float Rys tables
    double prim_eps;             // skip primitive quartets with q_ij q_kl Dmax <= prim_eps
    double omega;                // |w| of the range-separated operator (OP 1, 2)
    unsigned long long *stats;   // per class pair (stride stat_stride): [0] quartets, [1] primitive quartets, [2] routed
    int stat_stride;
    int *err;                    // device error word
    double lo, hi;               // keep a quartet iff lo < Q_ab Q_cd Dmax <= hi
    // the split threshold of a molecule, split x max Q^2 x max |D| and at least
    // split_min, narrows that range: split_side 1 raises lo to it (the FP64
    // tier), -1 lowers hi to it (the split tier), 0 leaves the range alone
    double split, split_min;
    int split_side;
    // FP32 screening (scr32 = 1, used when the build's cutoff is >= 1e-30 so
    // that no product of interest leaves the FP32 range): the same bounds and
    // the band in FP32; every tier of a build evaluates them identically
    int scr32;
    float lo32, hi32, tau32, band_hi32, prim_eps32;
    int with_j, with_k;          // which outputs (and density blocks) to use
    int use_dmax;                // 0: screen with Dmax := 1
    int ndm;
    // learned router (MODE 1) and label logging (MODE 2)
    const JkRouterDev *router;
    double tau;                  // band (tau, band_hi]
    double band_hi;
    int tier;                    // 0: this launch is the FP64 tier, 1: FP32
    float *log_x;                // MODE 2: features (12 per sample)
    float *log_y;                // MODE 2: labels
    unsigned long long *log_n;   // MODE 2: band quartets seen; those with a key up to log_keep (may exceed log_cap)
    long long log_cap;
    unsigned long long log_keep; // a band quartet is written iff the key of its shells is at most this
    unsigned long long *log_key; // the keys of the written ones, or nullptr
    // routed builds: the FP64 tier (MODE 1) appends the band quartets the
    // router releases to their class pair's list (rlist + roff[launch], while
    // it has room: rcap[launch]; a quartet that finds it full stays in FP64);
    // the FP32 list kernel (MODE 3) evaluates min(rcount[launch], rcap[launch])
    // entries of each of its class pairs
    JkRouted *rlist;
    unsigned long long *rcount;
    const long long *roff, *rcap;
    // 1: the FP32 tier evaluates the large-T (Gauss-Hermite) roots and
    // weights in FP64 and rounds them to FP32
    int asym64;
    // 1: the FP32 tier widens its contributions to FP64 with integer bit
    // operations; 0: with the conversion instruction
    int widen_int;
};

// Arguments of the Schwarz (diagonal-quartet) launch of one pair class.
struct JkSchwarzArgs {
    const JkPair *pairs;
    const JkPrimPair64 *pp64;
    const double *rys64;
    double *Qout;                // one per pair
    int npair;
};

// Bits of the device error word. Only the density check sets one today; no
// kernel of the library waits on another kernel or on the host.
#define JK_ERR_DEV_NAN 4
