"""Stage times of a profiled pass: the row updates of enacted prefixes are
reported under "cross", once for every round on connection rows that sorted
moves, and every stage that a pass runs has its time."""
import pytest

import snngen

pytestmark = pytest.mark.gpu


def test_row_updates_have_their_stage():
    import __graft_entry__ as g
    g.build()
    from paper_2609_07577_gb300 import HGraph
    G = HGraph.from_hypergraph(snngen.by_name("cfg3s"))   # enacts moves on levels with rows
    try:
        G.profile(True)
        G.partition()
        st, logs = G.stage_times(), G.round_logs()
    finally:
        G.close()
    with_moves = [r for r in logs if r["n_props"] > 0]
    assert st["cross"]["calls"] == sum(r["rows"] for r in with_moves) > 0
    assert st["cross"]["ms"] > 0
    assert st["sortmoves"]["calls"] == st["replay"]["calls"] == len(with_moves)
