"""Workspace sizes of the group-by (host only)."""
import paper_2606_24647_gb300 as px


def test_workspace_never_shrinks_and_holds_a_claim_slot_per_group():
    L = px.load()
    before = 0
    for e in range(0, 31):
        for mg in (2**e - 1, 2**e, 2**e + 1, 2**e + 2**e // 2):
            if not 1 <= mg < 2**31:
                continue
            need = L.px_groupby_ws_bytes(0, mg)
            assert need >= before, mg
            # state, key and output row of a slot; accumulators and a flag of an entry
            assert need > (4 + 8 + 4) * (mg + 1) + (8 * 8 + 1) * mg, mg
            assert L.px_join_probe_agg_ws_bytes(0, mg) == need
            before = need
    assert L.px_groupby_ws_bytes(0, 2**31 - 1) >= before
