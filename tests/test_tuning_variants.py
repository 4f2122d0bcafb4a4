"""What heat_tuning_variant says of each variant (host only): fused are the
one-kernel Chronopoulos-Gear iterations and nothing else, and the default
variant, whose meshes may be held on the chip, is told from both them and the
plain form of its shape."""


def test_fused_and_on_chip_variants_are_told_apart():
    import __graft_entry__
    __graft_entry__._build_module().build()
    import paper_1905_07622_gb300.api as api
    info = [api.heat_tuning_variant(v) for v in range(api.heat_tuning_num_variants())]
    assert [v for v, i in enumerate(info) if i["fused"]] == [9, 10, 11, 12, 13, 14]
    assert all(i["stages"] == 0 for i in info if i["fused"])
    assert [v for v, i in enumerate(info) if i["stages"] < 0] == [0]
    shape = ("seg_width", "rows", "warps")
    assert [info[0][k] for k in shape] == [info[15][k] for k in shape] and info[15]["stages"] == 0
