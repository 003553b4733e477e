"""Volumes and boxes (X Y Z) for which the direct engine takes its 16-row tiles: every box width with a
kernel of its own and two without, with one and with several splits of the tap planes, none a whole
number of tiles; the last stages its planes in rows. tests/test_box_plan_host.py checks that the tiling
rule chooses them so."""

TALL_TILES = [
    ((34, 61, 74), (1, 3, 1)), ((1, 73, 57), (1, 7, 3)), ((3, 108, 89), (3, 19, 1)), ((3, 60, 39), (3, 13, 3)),
    ((73, 67, 45), (5, 5, 1)), ((6, 76, 41), (5, 13, 3)), ((34, 93, 52), (7, 5, 1)), ((7, 41, 54), (7, 25, 3)),
    ((41, 57, 73), (9, 5, 1)), ((11, 91, 49), (9, 5, 3)), ((38, 61, 73), (11, 5, 1)), ((41, 46, 25), (11, 11, 5)),
    ((99, 79, 27), (13, 7, 1)), ((47, 73, 29), (13, 11, 3)), ((33, 59, 88), (15, 9, 1)), ((94, 25, 25), (15, 7, 7)),
    ((102, 34, 60), (17, 11, 1)), ((48, 76, 15), (17, 11, 5)), ((34, 84, 63), (19, 15, 1)), ((108, 63, 9), (21, 11, 7)),
    ((80, 299, 58), (25, 159, 1)),
]
