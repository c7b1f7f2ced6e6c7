"""The autotuner times no configuration twice: the shared-memory batch no longer
changes a launch, so no two candidates differ in it alone, and none names one."""


def test_candidates_are_different_launches():
    from paper_2506_12727_gb300 import build
    build.build()
    from paper_2506_12727_gb300 import autotune
    launches = [(tile, ppt) for tile, ppt, _ in autotune.CANDIDATES]
    assert len(set(launches)) == len(launches)
    assert all(batch == 0 for _, _, batch in autotune.CANDIDATES)
