"""Every name that bench.py's functions use exists: its workloads take minutes
on a GPU, and a name that is missing shows only at the end of one."""
import builtins
import os
import symtable

BENCH = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "bench.py")


def unresolved():
    """(function, name) of every global name read in a function of bench.py
    that neither the module nor the builtins define."""
    with open(BENCH) as fh:
        top = symtable.symtable(fh.read(), BENCH, "exec")
    known = set(top.get_identifiers()) | set(dir(builtins)) | {"__file__", "__name__"}
    out = set()

    def walk(table, function):
        for child in table.get_children():
            inner = function or child.get_name()
            out.update((inner, s.get_name()) for s in child.get_symbols()
                       if s.is_global() and s.is_referenced() and s.get_name() not in known)
            walk(child, inner)

    walk(top, "")
    return out


def test_the_batch_workload_uses_no_missing_name():
    assert not {n for f, n in unresolved() if f == "run_batch"}


def test_no_function_of_the_benchmark_uses_a_missing_name():
    assert not unresolved()
