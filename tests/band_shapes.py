"""Batches of one bucket (queries of 511-513 bases, scores beyond a packed lane's) and
the band engine's lanes and slots their plan takes."""
from paper_2301_09310_gb300.synth import ScoringParams

# band, pairs, lanes per pair, slots per lane: every compiled shape, and both sides of the
# counts and bands where the rule changes
SHAPES = [
    (8, 12000, 2, 32), (31, 9729, 2, 32), (31, 9728, 4, 32), (16, 4864, 8, 26), (32, 9000, 4, 32),
    (63, 4865, 4, 32), (64, 3000, 8, 26), (103, 2433, 8, 26), (104, 2433, 8, 32), (127, 5000, 8, 32),
    (103, 2432, 16, 14), (111, 1217, 16, 14), (112, 2432, 16, 26), (128, 3000, 16, 26), (207, 1217, 16, 26),
    (208, 1217, 16, 32), (255, 4000, 16, 32), (100, 1216, 32, 8), (127, 300, 32, 8), (128, 1216, 32, 14),
    (223, 700, 32, 14), (224, 1216, 32, 26), (415, 2000, 32, 26), (416, 500, 32, 32), (511, 1500, 32, 32),
]

# the row keys' range: the most a row's maximum falls, plus the match score, just inside
# and just outside of what the shape's lanes leave
KEY_EDGES = [
    (ScoringParams(1, -59, 20, 1, 100, 0, -1), 3000, True),
    (ScoringParams(1, -60, 20, 1, 100, 0, -1), 3000, False),
    (ScoringParams(2, -4, 21, 1, 300, 50, -1), 400, True),
    (ScoringParams(2, -4, 22, 1, 300, 50, -1), 400, False),
    (ScoringParams(1, -3, 5, 1, 31, 0, -91), 10000, True),
    (ScoringParams(1, -3, 5, 1, 31, 0, -92), 10000, False),
]
