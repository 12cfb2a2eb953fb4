// Whose turn a stage of the pair kernel is, for the kernel and (as plain C++) for the model of its barriers in the tests.
//
// The converter groups take the stages of a launch in turn: stage g is group g % 4's, in T', in the tiles and across them.  A group
// waits by parity for the MMAs of stage g - 5 (the ring has five places).  That is right if it knows those of stage g - 10 to be complete,
// since its turn before waited for stage g - 9, and those of stage g to be still to come, since they need its own arrival.
//   Packed tiles have a ring of their own, of four slots, and a tile is one stage or two.  A group has a turn of every tile, or of every second
// one, so that it has seen the tile whose slot a tile takes over, four before it, if that belongs to the same output tile.  From one output
// tile to the next the stages without a packed tile (or half a packed tile at the end) shift the turns: a group may not have seen that
// tile, and then waits for the MMAs of stage g - 5 first.  They have read what was expanded from it, since its stages lie five back or more
// (four back lies the group's own).
#pragma once
#include <stdint.h>

#include "handover.h"

namespace slim {

constexpr int kTurnGroups = 4, kTurnPlaces = 5, kTurnSlots = 4;

// The first stage at or behind `base` that is the group's, counted from there.
SLIM_BOTH int first_turn(int group, int base) { return (group - base) & (kTurnGroups - 1); }

// From which stage of an output tile on (`nth` of its pair; `sparse` stages, `per_tile` of a packed tile, then `dense` ones) a group has seen the
// packed tile whose slot the stage's takes over.
SLIM_BOTH int seen_from(int nth, int sparse, int dense, int per_tile) {
    return nth == 0 || (dense % kTurnGroups == 0 && sparse % per_tile == 0) ? 0 : kTurnSlots * per_tile;
}

}  // namespace slim
