"""Every global name that a function of bench.py loads exists (the workloads need a GPU and do not run here)."""
import builtins
import dis
import types

import bench


def _loads(code):
    for ins in dis.get_instructions(code):
        if ins.opname in ("LOAD_GLOBAL", "LOAD_NAME"):
            yield ins.argval
    for const in code.co_consts:
        if isinstance(const, types.CodeType):
            yield from _loads(const)


def test_functions_load_no_unknown_name():
    unknown = {(f.__name__, n) for f in vars(bench).values() if isinstance(f, types.FunctionType) and f.__module__ == "bench"
               for n in _loads(f.__code__) if n not in vars(bench) and not hasattr(builtins, n)}
    assert not unknown
