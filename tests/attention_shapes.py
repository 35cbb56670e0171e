"""Shapes for each route that the tensor-core attention has, at the sizes where the route's division of labour
has edges: (route, (B, N, L, P, Hq, Hkv), head dimension), routes as attention_routes.py names them on a device of
148 multiprocessors (test_attention_routes.py holds this table to the library's plan)."""

SHAPES = [
    # two, four and eight thread blocks to an M-tile: a key tile each, one block with one more, odd and even
    # shares, M-tiles with few rows, ragged heads, block keys over one key tile for some M-tiles and two for others
    ("cluster of 2", (2, 3, 7, 700, 66, 1), 128), ("cluster of 2", (2, 3, 7, 771, 66, 1), 128),
    ("cluster of 2", (1, 2, 32, 640, 66, 1), 128), ("cluster of 2", (1, 3, 7, 1400, 130, 2), 128),
    ("cluster of 2", (2, 3, 7, 384, 66, 1), 64), ("cluster of 2", (2, 3, 7, 500, 70, 1), 64),
    ("cluster of 2", (1, 2, 32, 2000, 37, 37), 64),
    ("cluster of 4", (1, 1, 7, 384, 66, 1), 128), ("cluster of 4", (1, 1, 7, 385, 66, 1), 128),
    ("cluster of 4", (1, 3, 7, 2700, 16, 16), 128), ("cluster of 4", (1, 3, 40, 3000, 28, 4), 128),
    ("cluster of 4", (1, 8, 32, 2700, 16, 16), 128), ("cluster of 4", (1, 4, 100, 2600, 7, 1), 128),
    ("cluster of 4", (1, 1, 7, 384, 66, 1), 64), ("cluster of 4", (1, 1, 7, 900, 16, 16), 64),
    ("cluster of 4", (2, 8, 32, 768, 6, 6), 64), ("cluster of 4", (1, 8, 32, 1000, 16, 16), 64),
    ("cluster of 8", (1, 1, 7, 896, 66, 1), 128), ("cluster of 8", (1, 1, 7, 897, 66, 1), 128),
    ("cluster of 8", (1, 4, 17, 2700, 7, 1), 128), ("cluster of 8", (1, 2, 100, 2600, 7, 1), 128),
    ("cluster of 8", (1, 1, 7, 900, 2, 1), 64), ("cluster of 8", (1, 3, 17, 893, 28, 4), 64),
    # one thread block to an M-tile: one key tile, two, three; several rounds
    ("one tile", (1, 2, 3, 0, 128, 1), 128), ("one tile", (1, 2, 16, 100, 100, 1), 128),
    ("one tile", (1, 2, 16, 200, 100, 1), 128), ("one tile", (2, 9, 32, 100, 40, 40), 128),
    ("one tile", (1, 2, 3, 20, 128, 1), 64), ("one tile", (1, 4, 16, 130, 70, 1), 64),
    # two M-tiles to a thread block, the last one without rows
    ("two tiles", (2, 9, 32, 300, 35, 35), 128), ("two tiles", (2, 9, 32, 100, 35, 35), 64),
    # ... in full rounds, what is left in a second launch: every other or fourth of its blocks or pairs without an
    # M-tile, groups of one, two and three heads
    ("two tiles, then pair", (5, 8, 25, 50, 64, 64), 128), ("two tiles, then pair", (3, 7, 36, 40, 150, 50), 128),
    ("two tiles, then one tile", (2, 7, 60, 20, 150, 50), 128), ("two tiles, then one tile", (2, 10, 30, 50, 90, 90), 128),
    ("two tiles, then pair", (5, 8, 25, 50, 64, 64), 64), ("two tiles, then one tile", (2, 10, 30, 50, 90, 90), 64),
    # a pair of thread blocks to an M-tile: 63 rows of 64 in each, the ring of stages several times round
    ("pair", (1, 3, 17, 893, 28, 4), 128), ("pair", (1, 9, 17, 637, 28, 4), 64), ("pair", (1, 9, 34, 1533, 28, 4), 64),
    ("pair", (1, 8, 32, 768, 24, 24), 64), ("pair", (1, 1, 4, 0, 1, 1), 64)]

# The maximum of a row grows from key tile to key tile: accumulators are rescaled, partials of very different
# reference maxima merged.
GROWING = [("cluster of 2", (2, 3, 7, 771, 66, 1), 128), ("cluster of 4", (1, 3, 7, 2700, 16, 16), 128),
           ("cluster of 2", (2, 3, 7, 1284, 66, 1), 64), ("cluster of 4", (1, 1, 7, 1400, 16, 16), 64),
           ("cluster of 8", (1, 1, 7, 2000, 2, 1), 64), ("pair", (1, 8, 40, 1157, 24, 12), 64),
           ("pair", (1, 3, 17, 893, 28, 4), 128), ("one tile", (1, 9, 16, 700, 60, 60), 64),
           ("two tiles", (2, 9, 32, 300, 35, 35), 64)]

# Layers of a model, one after the other.
CHAINS = [("pair", (1, 8, 32, 512, 16, 16), 128), ("pair", (3, 5, 20, 777, 24, 8), 64),
          ("one tile", (2, 9, 32, 100, 40, 40), 128), ("cluster of 2", (2, 3, 7, 771, 66, 1), 128),
          ("cluster of 4", (1, 1, 7, 900, 16, 16), 64), ("cluster of 8", (1, 4, 17, 2700, 7, 1), 128),
          ("two tiles", (2, 9, 32, 300, 35, 35), 128), ("two tiles, then pair", (5, 8, 32, 256, 32, 32), 128),
          ("two tiles, then one tile", (2, 7, 60, 20, 150, 50), 128)]
