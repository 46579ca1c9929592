"""hef_debug_inject belongs to the bounds-checked build: the regular build refuses
it (HEF_ERR_UNSUPPORTED) and says why (CPU only)."""


def test_regular_build_refuses_injected_conditions():
    import paper_2511_06600_gb300 as hef
    L = hef.lib()
    for what in (0, 1, 2):
        assert L.hef_debug_inject(what) == -6
    assert b"bounds-checked" in L.hef_last_error()
