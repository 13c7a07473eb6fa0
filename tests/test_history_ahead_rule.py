"""The rule for the history term ahead of the selection's end where no selection precedes the attention kernel (hf_dispatch.h)."""
from tests.test_dispatch_rules import rules  # noqa: F401  (fixture)


def test_not_without_a_selection_in_front(rules):  # noqa: F811
    """Attention on lists that are there before the call has nothing to form the term ahead of."""
    for block in (16, 64, 128):
        for units in (1, 12, 147, 148, 149, 300, 444):
            assert not rules.ahead(block, units, 0, 148)
    assert rules.ahead(128, 12, 1, 148)
