"""The binding remembers workspace sizes; the hooks that change the planner's choice must leave no old one behind."""
import pytest

from paper_2311_00368_b200 import build as b2sp_build


@pytest.mark.parametrize("hook,value,sizes", [("debug_force_k_splits", 1, (4096, 4096, 0, 128, 1_600_000)),
                                              ("debug_force_partition", 1, (8192, 8192, 0, 128, 10_000_000))])
def test_a_size_asked_for_while_a_hook_is_set_is_not_kept(monkeypatch, hook, value, sizes):
    b2sp_build.build()
    from paper_2311_00368_b200 import binding as b
    args = (b.OP_SPMM, *sizes, b.ALGO_TILE)
    remembered = lambda: b._workspace_need(*args, b._planner_setting)
    real = getattr(b.lib, "b2sp_" + hook)

    class Lib:
        """The library, with another thread's question arriving just before the hook takes effect."""
        def __getattr__(self, name):
            if name != "b2sp_" + hook:
                return getattr(lib, name)

            def call(x):
                remembered()
                real(x)
            return call

    lib = b.lib
    monkeypatch.setattr(b, "lib", Lib())
    try:
        for v in (value, 0):
            getattr(b, hook)(v)
            assert remembered() == b.workspace_bytes(*args)
    finally:
        real(0)
