"""The build: device code must come out the same in every build of one source, so that figures can be compared."""
from paper_2003_12811_gb300 import build as B


def test_device_code_is_not_cut_differently_from_build_to_build():
    """nvcc's own parallel compilation partitions the device code anew in every run (the spills of one kernel then
    differ from build to build); the build compiles translation units side by side instead."""
    flags = list(B.NVCC_FLAGS)
    for _, _, macros in B.UNITS:
        flags += macros
    assert not any(f.startswith("--split-compile") or f.startswith("-split-compile") for f in flags)


def test_units_cover_every_precision_and_order_once():
    got = sorted(m for src, _, m in B.UNITS if src == "sbp_ops.cu")
    want = sorted([f"-DSBP_T={t}", f"-DSBP_O={o}"] + (["-DSBP_BATCH"] if t == "float" else [])
                  for t in ("float", "double") for o in (2, 4, 6))
    assert got == want
    assert len({name for _, name, _ in B.UNITS}) == len(B.UNITS)
