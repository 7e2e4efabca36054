// The ring of B stages of k_kernel_eval_tc_ta, in plain C++ so that its rules can
// be checked on the host: column tile j (of a CTA's own) takes the fillings
// j KP .. j KP + KP - 1, KP = ceil(KB / 2) of them, filling t goes into stage
// ta_stage(t), and tile j's fillings are waited for by its issuing thread alone.
//
// A wait for a parity passes as soon as the barrier is in a phase of the other
// parity, the phase before the awaited one included.  The two issuers share the
// ring, so one barrier per stage would not do: the thread that waits for filling
// t may not have waited for filling t - kTaStages, and if that copy is still
// under way its wait for the next parity passes at once (copies are not ordered
// among themselves).  Each filling therefore has a barrier of its own, used once,
// in phase 0: there is no earlier phase to mistake.  The stages' empty barriers
// have one waiter, the thread that copies, which waits for every phase in turn.
#pragma once

namespace wmc {

constexpr int kTaStages = 5;    // stages of two 64-K blocks
constexpr int kTaMaxKB = 8;     // 64-K blocks of a tile
constexpr int kTaMaxTiles = 5;  // column tiles of a CTA
constexpr int kTaIssuers = 2;   // issuing threads: column tile j is thread j % kTaIssuers's
constexpr int kTaFills = kTaMaxTiles * ((kTaMaxKB + 1) / 2);

constexpr int ta_stage(int t) { return t % kTaStages; }
constexpr int ta_full_bar(int t) { return t; }
constexpr unsigned ta_full_parity(int) { return 0u; }
// the wait before filling t (t >= kTaStages): the MMAs of filling t - kTaStages
constexpr unsigned ta_empty_parity(int t) { return (unsigned)((t / kTaStages - 1) & 1); }

}  // namespace wmc
