"""The bounded table of plans keeps what was asked for last and stays bounded."""
from paper_2504_06881_b200 import inputs, tconv


def test_table_is_bounded_and_makes_each_entry_once():
    made = []
    t = tconv.KeptPlans(lambda k: made.append(k) or k, most=8)
    for k in range(20):
        assert t.get(k, k) == k and t.get(k, k) == k
        assert len(t.table) <= 8
    assert made == list(range(20))


def test_plan_follows_the_descriptor():
    d = inputs.layer(2, 3, 9, 10, 5, stride=2, pad=1, mode="compound")
    p = tconv.plan_of(d)
    assert p.y == (2, 5) + inputs.output_hw(d) and p.winner_bytes == tconv.tconv_winner_bytes(d)
    assert tconv.plan_of(dict(d)) is p
    d["N"] = 3                                     # a plain dict may change: its plan is looked up by content
    assert tconv.plan_of(d).y[0] == 3
    assert tconv.plan_of(dict(d, pad_mode="neutral")) is not tconv.plan_of(d)
