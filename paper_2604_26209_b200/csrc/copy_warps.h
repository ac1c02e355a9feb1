// Which decode launches under the own-branch mask get warps of their own for the K and V copies.  Plain C++: the host tests compile it too.
#pragma once

namespace hpd {

// What the host knows of a step.  How long the documents are and how many branches still live is known on the device only, so the rule
// below goes by averages; it decides about time, never about results.
struct StepSize {
    int n_docs, max_rows, total_prefix;
    int G, Hkv, D;
    int n_sm, work_cap, part_cap;    // SMs; work items and partial rows that the workspace holds
    int new_tokens;                  // every branch has a cached token: the call sees those of this step
};
struct AverageUnit { long long units; int branches, keys; };

// The units of a step whose documents all have the average number of rows and tokens, by the table kernel's plan: 128 / G rows of a document
// and one kv head each, and where those are fewer than SMs, chunks of 16384 tokens, 8192, ... 512 until they are not.
inline AverageUnit average_unit(const StepSize& s)
{
    const int per_unit = 128 / s.G, rows = (s.max_rows - 1) / s.n_docs + 1, tokens = s.total_prefix / s.n_docs;
    const long long items = static_cast<long long>(s.n_docs) * ((rows - 1) / per_unit + 1);
    AverageUnit u{items * s.Hkv, rows < per_unit ? rows : per_unit, tokens};
    for (int chunk = 16384; chunk >= 512 && u.units < s.n_sm; chunk >>= 1) {
        const long long chunks = tokens > chunk ? (tokens - 1) / chunk + 1 : 1;
        if (items * chunks > s.work_cap || (chunks > 1 && s.max_rows * chunks > s.part_cap)) break;
        u.units = items * chunks * s.Hkv;
        u.keys = tokens < chunk ? tokens : chunk;
    }
    return u;
}

// A unit's copies are one per branch, half of D and cache, about 100 cycles each for a warp; what four more warps take is registers of the
// softmax warps.  us with / without them:
//   at most one unit an SM, where the copy warps of the idle pipeline help: the call at 4 branches a unit 14.3 / 13.9, 24 17.6 / 18.6, 32
//     20.7 / 22.1, 128 (a head a group) 29.5 / 46.3; the step breaks even at 18 to 22 branches of D = 128 and at 22 to 28 of D = 64;
//   several units an SM, where they only take: 24 branches and chunks of 512 keys 29.5 / 27.0, 32 and 128 keys 19.9 / 18.9; but units that
//     pack many columns against few keys still wait for their copies: 48 branches and 512 keys 33.4 / 35.4, 1024 keys 39.1 / 37.3; 90 and
//     1024 48.3 / 51.4, 2048 63.7 / 62.1; 128 and 2048 72.7 / 71.7 (3000 tokens) and 84.8 / 85.8 (4000), 4000 keys 119 / 131.
//     The line lies at 13 keys a branch, 20 at D = 64 (52 branches and 1024 keys), and 96 branches take them always;
//   four units an SM and more: short units of 32 branches gain a little too (960 units, 128 keys 54.5 / 56.1, a step 76.8 / 80.2, 512 keys 100.6 /
//     103.1, 2048 keys 202 / 198; but 480 units of 128 keys 32.8 / 31.1).
//   A call that does not see the step's tokens is as a rule one over a block's rows without branch caches: nothing to pack (6144 rows over
//     128 tokens 42.2 / 36.3, 96 rows 10.0 / 8.8), so it never takes them.
inline bool copy_warps_pay(const StepSize& s)
{
    if (!s.new_tokens || static_cast<long long>(s.n_docs) * s.Hkv > s.n_sm) return false;
    const AverageUnit u = average_unit(s);
    if (u.units <= s.n_sm) return u.branches >= 22;
    if (u.units >= 4ll * s.n_sm && u.branches >= 32 && u.keys <= 16 * u.branches) return true;
    return u.branches >= 40 && (u.branches >= 96 || u.keys <= (s.D == 128 ? 13 : 20) * u.branches);
}

}  // namespace hpd
