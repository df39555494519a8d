"""Writes ws_units.inc: a lane schedule of the trailing update of a
right-looking tile Cholesky by one warp.  The persistent row kernel
(rows_ws.cu), which used it, now factors left-looking on tensor-core tiles and
includes no schedule; the table and its generator are kept as the subject of
the schedule and algorithm tests.

In the blocked right-looking Cholesky of one row's bordered matrix (g x g
tiles of 8 x 8), panel p leaves the trailing tiles (I, J), p < J <= I < g, to
be updated as A_IJ -= L_Ip L_Jp^T.  A consumer warp does this in units of
half a tile (columns 4h .. 4h + 3 of tile (I, J)), one unit per lane per
round.  Every unit streams 40 128-bit shared-memory accesses (the two
L rows, the A rows read and written), and a 128-bit access is served eight
lanes at a time: if two of those eight lanes touch different 16-byte words
in the same bank, the access takes one more pass through the memory.

The tiles sit 68 floats apart in tidx order (tile (I, J) at
68 (I (I + 1) / 2 + J)) with row r at 8 r + 4 (r / 4), as the kernel lays
them out.  Which units share an eight-lane group then decides the passes, so
for every panel this script groups the units eight at a time greedily (each
next unit the one that adds the fewest passes), improves the grouping by
random pair swaps that never add passes, and emits four groups per round.
The result depends only on g and a fixed seed; run it to regenerate the
file:

    python gen_ws_units.py > ws_units.inc

Entry format: 0xFFFF for an idle lane, else I | J << 4 | h << 8.
"""
import collections
import random

TILE_F = 68
G_MIN, G_MAX = 2, 16  # K = 8 .. 127 gives g = ceil((K + 1) / 8) = 2 .. 16
IDLE = 0xFFFF
SEED = 20170512  # one random stream for every grid, drawn in order of g


def trow(r):
    return 8 * r + 4 * (r >> 2)


def tile_base(I, J):
    return TILE_F * (I * (I + 1) // 2 + J)


def passes(addrs):
    """Memory passes of one eight-lane group of 128-bit accesses (float
    offsets, 4-aligned): the largest number of distinct 16-byte words that
    fall into one bank group of four banks."""
    groups = collections.defaultdict(set)
    for a in addrs:
        groups[(a >> 2) & 7].add(a)
    return max((len(s) for s in groups.values()), default=0)


def group_cost(units, p):
    if not units:
        return 0
    c = 0
    for jj in range(4):  # L_Jp rows 4h .. 4h + 3
        for q in (0, 4):
            c += passes([tile_base(J, p) + trow(4 * h) + 8 * jj + q for (I, J, h) in units])
    for ii in range(8):
        for q in (0, 4):  # L_Ip row ii
            c += passes([tile_base(I, p) + trow(ii) + q for (I, J, h) in units])
        # A_IJ row ii, columns 4h .. 4h + 3: read and written
        c += 2 * passes([tile_base(I, J) + trow(ii) + 4 * h for (I, J, h) in units])
    return c


def units_of(g, p):
    return [(I, J, h) for I in range(p + 1, g) for J in range(p + 1, I + 1) for h in (0, 1)]


def schedule(g, p, rng, swaps=4000):
    rest = units_of(g, p)
    groups = []
    while rest:
        grp = []
        while len(grp) < 8 and rest:
            best = min(rest, key=lambda u: (group_cost(grp + [u], p), u))
            grp.append(best)
            rest.remove(best)
        groups.append(grp)
    cost = [group_cost(x, p) for x in groups]
    if len(groups) > 1:
        for _ in range(swaps):
            a, b = rng.randrange(len(groups)), rng.randrange(len(groups))
            if a == b:
                continue
            ia, ib = rng.randrange(len(groups[a])), rng.randrange(len(groups[b]))
            ga, gb = groups[a][:], groups[b][:]
            ga[ia], gb[ib] = gb[ib], ga[ia]
            ca, cb = group_cost(ga, p), group_cost(gb, p)
            if ca + cb <= cost[a] + cost[b]:
                groups[a], groups[b], cost[a], cost[b] = ga, gb, ca, cb
    lanes = []
    for grp in groups:
        lanes += [I | (J << 4) | (h << 8) for (I, J, h) in grp] + [IDLE] * (8 - len(grp))
    lanes += [IDLE] * (-len(lanes) % 32)
    return lanes, sum(cost)


def main():
    rng = random.Random(SEED)
    flat, starts = [], []
    for g in range(G_MIN, G_MAX + 1):
        row = []
        for p in range(g):
            row.append(len(flat) // 32)
            lanes, _ = schedule(g, p, rng) if p < g - 1 else ([], 0)
            flat += lanes
        row.append(len(flat) // 32)
        starts.append(row)
    print("// Generated by gen_ws_units.py: lane schedule of the trailing update")
    print("// (entry I | J << 4 | h << 8, 0xFFFF idle; 32 entries per round).")
    print(f"constexpr int kWsUnitGMin = {G_MIN}, kWsUnitGMax = {G_MAX};")
    print(f"__device__ const unsigned short kWsUnits[{len(flat)}] = {{")
    for i in range(0, len(flat), 16):
        print("  " + ", ".join(f"0x{v:04x}" for v in flat[i:i + 16]) + ",")
    print("};")
    width = G_MAX + 1
    print("// first round of panel p for g: kWsUnitRound[g - kWsUnitGMin][p], p = 0 .. g")
    print(f"__device__ const unsigned short kWsUnitRound[{G_MAX - G_MIN + 1}][{width}] = {{")
    for row in starts:
        print("  {" + ", ".join(str(v) for v in row + [row[-1]] * (width - len(row))) + "},")
    print("};")


if __name__ == "__main__":
    main()
