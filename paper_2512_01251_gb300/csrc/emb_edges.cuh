// Sizes of the edge table of the watertight check (host arithmetic alone).
//
// An edge takes a slot of one of its vertices, or a place in the overflow table.  A closed
// list has 3T/2 undirected edges over about T/2 vertices, and a few percent of them overflow
// (more where a few vertices hold most edges); a list that is not closed has up to 3T.  Large
// lists are tried first with a small overflow table and bounded probes; the table that
// decides has room for all 3T edges at three quarters full, so that a probe always ends.
#pragma once
#include <stdint.h>

#define EDGE_PROBES 128      // of an overflow table without room for every edge
#define EDGE_SMALL (1 << 16)  // triangles up to which it gets room for every edge at once

struct EdgePlan {
    bool slots;    // slots by vertex: not for a list with more than 2T vertices (a closed one has about T/2)
    bool all;      // room for every edge: the table cannot fill up
    uint64_t cap;  // entries of the overflow table, a power of two
};

// attempt 0, and 1 after a table without room for every edge has filled up.
static inline EdgePlan emb_edge_plan(int64_t V, int64_t T, int attempt)
{
    EdgePlan P;
    P.slots = V <= 2 * T;
    P.all = attempt > 0 || !P.slots || T <= EDGE_SMALL;
    const uint64_t want = (uint64_t)(P.all ? 4 * T : T / 2);
    P.cap = 1024;
    while (P.cap < want) P.cap <<= 1;
    return P;
}
