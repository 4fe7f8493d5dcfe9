"""The autotuner's choice of a class: the default kernel unless a candidate is
faster by more than repeated runs differ."""
from paper_2207_00514_gb300 import tune


def test_choice():
    other = {"traversal": 1, "block_size": 256, "leaf_size": 1}
    assert tune.DEFAULT in tune.candidates("single")
    for ms, expected in ((0.99, tune.DEFAULT), (0.97, other), (1.2, tune.DEFAULT)):
        chosen = tune.choose([(ms, other), (1.0, tune.DEFAULT), (3.0, {"traversal": 2})])
        assert chosen == (min(ms, 1.0) if expected is other else 1.0, expected, 1.0)
    batched = [(1.0, o) for o in tune.candidates("batched")]
    assert tune.choose(batched)[1] == tune.DEFAULT
