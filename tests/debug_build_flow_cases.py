"""More parity cases for the debug build of the library (debug_build_cases.py
says what it checks): the forms that the cases there do not reach.  Run as a
process of its own by tests/test_gpu_debug_build.py."""
from debug_build_cases import _build, cubic, oracle, square


def main():
    from paper_2505_05919_gb300 import _capi
    assert _capi.lib_path() == _build.DEBUG_LIB and _capi.cvf_debug_checks()
    for L in (2, 9, 12, 34, 51, 52, 70):           # the dataflow sweep of cubes
        cubic(L, 5, -1)
    for L, kw in ((34, {}), (64, dict(rng_words=2)), (130, {})):   # the layered schedule's launches
        square(L, 7, tiles=0, schedule=oracle.SCHED_LAYERED, **kw)
    print("debug build: all cases match, no index check failed")


if __name__ == "__main__":
    main()
