// Descriptors of the mixed-radix passes (fft_mixed.cuh): any cycle lengths, any
// element type, one pattern per launch, grouped launches and the single-launch
// queue alike.
//
// Three kinds of tile, all transformed in shared memory by the same stages:
//
//   row    T rows of the logical LB x nD array (the DFT over the last cycle);
//          with a split last cycle the rows of a tile are adjacent lambda_a,
//          which are adjacent input slots, so the tile is held [element][row]
//          and the lanes of its box loads and stores run along the rows;
//   column T adjacent workspace columns (the DFTs over the other cycles), held
//          [row][column];
//   whole  T complete signals of m points each (every cycle in one tile): the
//          box side is read and written in slot order through a table of tile
//          positions, so such a transform is one launch without a workspace.
#pragma once
#include <stdint.h>

#include "fft_plan.hpp"

namespace pfft {

enum MixKind { MIX_ROW = 0, MIX_COL = 1, MIX_WHOLE = 2 };

constexpr int kMixMaxStages = 16;
constexpr int kMixPoints = 16;  // points a thread holds between the barriers of a stage, at most
// Register butterflies reach radix 16; primes from 17 up are direct stages, and so
// are 11 and 13 in a complex128 pencil that needs more than 11 or 13 points a thread.
constexpr int kMixMinDirect = 17;
constexpr int kMixDirect = 2048;  // marks the radix of such a stage (one comparison tells the kernel)
// Output pairs of one work item of a direct stage: kMixWide when every item
// has a thread of its own, else kMixNarrow with at most kMixItems per thread;
// kMixNarrow either way in complex128 (mix_direct_pairs).
constexpr int kMixWide = 6, kMixNarrow = 4, kMixItems = 3;
// Order in which the stages of the register radices run (mix_stages).
constexpr int kMixOrder[15] = {15, 13, 11, 9, 16, 14, 12, 10, 8, 7, 6, 5, 4, 3, 2};
template <typename C>
constexpr int kMixThreads = sizeof(C) == 8 ? 1024 : 512;
// Dynamic shared memory of a grouped tile: the 227 KB per CTA less room for the
// static copies of the descriptors (batch_kernels.cu checks that they fit).
constexpr int kMixGroupedSmem = 227 * 1024 - 8192;
constexpr int kMixThreadsC64 = 1024, kMixThreadsC128 = 512;

// One radix stage along one axis.  Tile positions of a butterfly (low, j, hi):
// base + (j + r aR) sig -> base + ((j - k) R + k + r Ns) sig, k = j mod Ns,
// base = hi blk + low, low < sig, j < aR, blk = aR R sig; sig is the axis's
// stride in the tile (the columns of a tile are strides below every axis).
// Tiles are padded from the first stage along the fastest axis on: when its
// radix R1 is even, its outputs j R1 + r would meet in few banks, so `pad`
// elements (one pencil position) follow every R1 of them from there.  R1 divides
// every later step, so all accesses of a stage stay affine in r: istep and ostep
// are the padded steps, ipad / opad the padding per pad unit (0: not padded).
// The workspace side of a row tile visits the elements in the order of the column
// positions, which may put every lane into the same bank: there the padding is by
// a unit of its own (MixDesc::ws_in, ws_out), which divides the step of the first
// stage's inputs or of the last one's outputs.
struct MixStage {
  int R;        // plus kMixDirect for a direct stage of a radix below kMixMinDirect
  int aR, sig, Ns, blk;
  int istep, ostep, ipad, opad;
  int tw;       // twiddles of the stage in the stage table: [b][k] (MixTableArgs); direct stages: the radix
  int gen;      // direct stages: offset of g^t mod R (R - 1 ints) in the integer table
  int twstep;   // direct stages: step of the root table per unit of exp(-2 pi i / (Ns R))
  FastDiv div_in, div_out;  // by the pad units of the inputs and of the outputs
  FastDiv div_sig, div_aR, div_Ns, div_nb;  // div_nb: direct stages, butterflies of the tile
};

struct alignas(16) MixDesc {
  int kind, lay;  // lay 1: the tile is [element][row] (row tiles of a split last cycle)
  int d, ts;
  int L, T, logT, n;  // pencil length, pencils per tile, points of the tile
  int nD, LB, m, batch;
  int groups;         // tiles per signal (whole tiles: of the batch)
  int nthreads, smem_bytes;
  int pad;            // padding of the finished tile: position x at x + pad (x / pad unit)
  FastDiv div_pad;    // by the pad unit (R1 positions of the fastest axis)
  int ws_in, ws_out;  // row tiles in [row][element] order: pad units of the workspace side (0: as without)
  int pitch_in, pitch_out;  // their distances of the rows
  const int *psin, *psout;  // row tiles: padded element position of each column position
  int dir_off;        // tables of the direct stages after the tile (elements)
  int nstages;
  int tw_n;           // order of the root table
  int load_mode, store_mode, conj_in, conj_out;
  int in_sel, out_sel;  // grouped launches: in / out are byte offsets into base[in_sel] / base[out_sel]
  double scale;
  const void* in;
  void* out;
  const int *Atab, *Btab, *Ctab, *Etab, *PIinv;
  const int *map_in, *map_out;  // whole tiles: tile position of box slot s (input box, output box)
  const void* tw;               // roots exp(-2 pi i t / tw_n)
  const void* stw;              // stage table
  const int* gtab;              // integer table of the direct stages
  const void *fs_lo, *fs_hi;    // phases of a split last cycle (fft_plan.hpp)
  int fs_na;
  FastDiv fs_div;
  FastDiv divnD, divL;
  int nsub, sub_n[kMaxSub], alpha[kMaxSub];
  FastDiv sub_div[kMaxSub];
  BoxDesc boxH, boxG;
  MixStage st[kMixMaxStages];
};
static_assert(sizeof(MixDesc) % 16 == 0, "descriptors are copied in 16-byte pieces");

// Stage twiddles: entry (s, b, k) = exp(-2 pi i k 2^b / (Ns R)), or, for the
// stages of fused_dft (fused), factor b of its levels: exp(-2 pi i (k + c Ns) /
// (Ns 2^l)), b = fused_first(l) + c.
struct MixTableArgs {
  int n, total;
  int fused[kMixMaxStages];
  int R[kMixMaxStages], Ns[kMixMaxStages], off[kMixMaxStages + 1];
};

// Sets the sides of a call (load and store map) in a row tile's descriptor: the
// workspace side has its own padding.
inline void mix_sides(MixDesc& a, int load, int store) {
  a.load_mode = load;
  a.store_mode = store;
  if (load == MAP_WS && a.ws_in) {
    MixStage& s = a.st[0];
    s.ipad = 1;
    s.istep += s.istep / a.ws_in;
    s.div_in.init(uint32_t(a.ws_in));
  }
  if (store == MAP_WS && a.ws_out) {
    MixStage& s = a.st[a.nstages - 1];
    s.opad = 1;
    s.ostep = s.Ns * s.sig;
    s.ostep += s.ostep / a.ws_out;
    s.div_out.init(uint32_t(a.ws_out));
  }
}

// Host-side launchers (fft_mixed_c64.cu, fft_mixed_c128.cu, fft_support.cu).
int launch_mixed_c64(const MixDesc& a, cudaStream_t s);
int launch_mixed_c128(const MixDesc& a, cudaStream_t s);
int launch_mixed_tables(void* tab, const MixTableArgs& t, int dtype, cudaStream_t s);
int launch_whole_maps(const MixDesc& a, const int* PI, int* map_in, int* map_out, cudaStream_t s);

}  // namespace pfft
