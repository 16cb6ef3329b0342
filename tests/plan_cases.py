"""Layers whose tests depend on the plan the library makes for them; test_plan_host.py holds the library to it without a GPU, the GPU tests run them."""

RANDOM, MAGNITUDE, RESCALED = 0, 1, 2
TWO_PASS, DENSE = 0, 2

# The kernel for narrow groups: the layer, the pattern, binary16 - accumulators of a unit, units of the busiest multiprocessor, operand stages. More
# units than stages: a stage is used again (twice as many: every barrier of the ring has seen both phases); more than two: so is an accumulator.
NARROW = [
    # B, H, W, C, R, S, stride, pad, groups, n, m, scheme, fp16, (accumulators, units, stages)
    ((96, 40, 40, 32, 3, 3, 1, 1, 2, 2, 4, MAGNITUDE, False), (1, 9, 4)),
    ((60, 64, 64, 32, 3, 3, 1, 1, 2, 2, 4, RANDOM, True), (4, 4, 2)),       # largest units
    ((256, 28, 28, 32, 3, 3, 1, 1, 2, 2, 4, RANDOM, False), (3, 4, 3)),
    ((200, 28, 28, 32, 3, 3, 1, 1, 2, 2, 8, RESCALED, True), (2, 5, 4)),
    ((60, 28, 28, 96, 3, 3, 1, 1, 3, 2, 16, MAGNITUDE, True), (1, 6, 4)),   # groups of 32, a last block of one
    ((250, 31, 33, 32, 3, 3, 2, 1, 2, 1, 4, RESCALED, True), (1, 5, 4)),    # four parities, uneven images
    ((3, 26, 27, 96, 3, 3, 2, 1, 3, 2, 32, RESCALED, False), (1, 1, 4)),    # ... of groups of 32, pruned in groups of 32
    ((2, 9, 12, 96, 3, 3, 1, 1, 3, 2, 32, RESCALED, True), (1, 1, 4)),      # groups of 32 held by two lanes, rescaled
    ((2, 9, 12, 48, 5, 5, 1, 2, 3, 2, 8, RANDOM, True), (1, 1, 4)),         # 25 taps
    ((40, 7, 7, 112, 3, 3, 1, 1, 7, 2, 4, RESCALED, True), (1, 1, 4)),
    ((3, 13, 27, 112, 3, 3, 2, 1, 7, 2, 16, RANDOM, True), (1, 1, 4)),
]

# The same kind of layer where the other path is the faster one: filters and images with a long reach, many taps
NARROW_ELSEWHERE = [
    (5, 76, 76, 416, 7, 1, 1, 0, 26, 2, 4, RANDOM),
    (12, 75, 144, 240, 3, 3, 1, 1, 15, 1, 8, RANDOM),
    (98, 37, 37, 224, 7, 1, 1, 0, 14, 2, 16, RANDOM),
    (26, 80, 80, 288, 3, 3, 1, 1, 9, 2, 8, RANDOM),
    (237, 16, 16, 80, 5, 5, 1, 2, 5, 1, 8, RANDOM),
    (3, 56, 56, 512, 7, 1, 1, 0, 16, 2, 32, RANDOM),
    (2, 9, 12, 96, 5, 5, 1, 2, 3, 2, 32, RESCALED),   # (groups of 32: two stages of 25 taps leave no room for dL/dO)
]

# Compressed operands against block-diagonal filters (other widths, other channel counts on the two sides): several blocks of 128 channels, the last
# one partly filled, so that a tile visits a window of them
BLOCK_DIAGONAL = [
    # B, H, W, Cin, Cout, R, S, stride, pad, groups, n, m, scheme, (route)
    ((3, 14, 14, 384, 384, 3, 3, 1, 1, 8, 2, 8, MAGNITUDE), 0),
    ((3, 14, 14, 160, 160, 3, 3, 1, 1, 20, 2, 4, RANDOM), 0),
    ((2, 20, 20, 160, 320, 3, 3, 2, 1, 10, 1, 16, RESCALED), 2),
    ((2, 20, 20, 384, 384, 3, 3, 2, 1, 8, 2, 8, RANDOM), 2),
    ((3, 7, 7, 384, 384, 3, 3, 1, 1, 8, 2, 4, RANDOM), 0),
    ((2, 28, 28, 240, 480, 3, 3, 1, 1, 15, 2, 16, MAGNITUDE), 0),
    ((4, 8, 8, 480, 480, 3, 3, 2, 1, 10, 2, 8, RESCALED), 0),
]

# Four output parities in one launch: the layer; whether its last round is dealt out strip by strip, whether a row of strips lies below the
# images of the smaller parities
PARITIES = [
    # B, H, W, Cin, Cout, R, S, pad
    ((2, 18, 49, 128, 192, 3, 3, 1), False, False),
    ((3, 12, 12, 192, 64, 3, 3, 0), False, False),
    ((1, 40, 24, 64, 64, 5, 5, 2), False, False),
    ((2, 22, 30, 128, 128, 2, 3, 1), False, False),
    ((5, 14, 14, 320, 256, 3, 3, 1), False, False),
    ((1, 9, 64, 64, 128, 3, 3, 1), False, False),
    ((24, 56, 56, 64, 128, 3, 3, 1), False, False),
    ((1, 65, 48, 64, 128, 3, 3, 1), False, True),
    ((10, 56, 56, 64, 128, 3, 3, 1), True, False),
]
