// pc_screen.h -- screened pricing launches: paths of a barrier contract that
// are decided by a few early bridge nodes leave before the walk.
//
// The bridge computes the last date first and bisects, so the values at the
// last date, the middle and the quarter dates need four nodes.  For a program
// that is one whole-loop barrier (result: a literal if the test holds on any
// date of a range, else a payoff), a path whose test holds on one of those
// dates has the literal as its payoff, whatever the other dates hold.  The
// screen computes the four dates of every path (the walk's nodes, normals and
// roundings, so the decision is the walk's own), writes the literal for the
// decided paths and lists the others; the pricing kernel then walks the
// listed paths only, full warps of them, and writes their payoffs; the totals
// kernel sums the payoffs tile by tile as an unscreened launch does.  Payoffs
// and sums are bit-identical.
#pragma once

#include "pc_internal.h"

namespace pc {

constexpr int kScreenNodes = 4;  // the last date, the middle, the quarters
struct Screen {
  float wl[kScreenNodes], wr[kScreenNodes], sd[kScreenNodes];
  uint32_t op[kScreenNodes];        // bridge op numbers
  float A[kScreenNodes][4];         // drifts (ModelDev::A) at the nodes' dates
  int32_t test[kScreenNodes];       // 1: the date is in the loop's range
  XInsn cond;                       // the loop's condition
  float literal;
  float *payoffs;                   // [n_paths]
  uint32_t *list, *count;           // undecided paths (any order), their number (zeroed before)
};

// Fills everything but the buffers; false when the program is not one
// whole-loop barrier of plain tests or the model is too short.
bool screen_program(const Program &p, const ModelHost &H, Screen &s);
// An estimate of the fraction of paths the screen decides, from each watched
// underlying's largest probability p to pass its level on a screened date
// (closed form): 0.8 (1 - prod (1 - p)).  (Three underlyings, correlation 0.4
// to 0.6, one year, 70 %: 0.12 to 0.31 estimated, 0.17 to 0.38 decided.)
double screen_fraction(const ModelHost &H, const Screen &s);

// The screen; *s.count must be zero.
cudaError_t launch_screen(const PriceArgs &a, const Screen &s, int sm_count, cudaStream_t st);
cudaError_t launch_totals(const PriceArgs &a, const float *payoffs, int sm_count, cudaStream_t st);

// A launch is screened when its walk is long (underlyings x dates x paths:
// about 0.2 ms of it; the screen's three extra launches take about 12 us and
// its nodes 2 % of a daily walk) and at least this fraction is decided.
constexpr double kScreenWork = 1.2e8, kScreenFraction = 0.05;
// (Portfolio plans are not screened: their contracts are smaller and run
// beside each other, and three launches in a row a branch took 1.68 ms where
// one took 1.45.)
constexpr int kScreenDates = 64;
constexpr uint64_t kScreenPaths = uint64_t(1) << 26;  // 8 bytes of scratch a path

}  // namespace pc
