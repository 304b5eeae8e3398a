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


def test_workspace_is_about_what_the_claim_table_and_the_dense_result_take():
    """The hash mode's table, of any capacity, needs little more than the other modes: their
    claim table (a power of two of at least two slots per group, 16 bytes each) and dense
    result (65 bytes per group)."""
    L = px.load()
    for mg in (5000, 8192, 100_000, 125_000, 131_072, 131_073, 10**6, 2**20, 2**20 + 1, 10**7, 2**30):
        slots = 1024
        while slots < 2 * mg:
            slots *= 2
        assert L.px_groupby_ws_bytes(0, mg) < 1.15 * (16 * slots + 65 * mg) + 700_000, mg
