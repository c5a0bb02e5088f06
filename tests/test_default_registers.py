"""The instances of the pair kernels that a call without a tuning launches compile for
sm_103a without register spills, and fit their block into the SM's registers.  Needs
nvcc, not a GPU."""
import pytest

from test_build_registers import ptxas_report  # noqa: F401 (the fixture)

# FP32: 640 threads in both modes, on orthogonal and skewed cells, with images or a
# cutoff (k_pair) and without (k_pair_open).  FP64: energies 512 threads, E + v 256, or
# 384 on skewed cells.
KEYS = [("k_pairIfLi%dELi640ELb%dE" % (m, s), 640) for m in (0, 1) for s in (0, 1)]
KEYS += [("k_pair_openILi%dELi640ELb%dE" % (m, s), 640) for m in (0, 1) for s in (0, 1)]
KEYS += [("k_pairIdLi0ELi512ELb%dE" % s, 512) for s in (0, 1)]
KEYS += [("k_pairIdLi1ELi256ELb0E", 256), ("k_pairIdLi1ELi384ELb1E", 384)]


@pytest.mark.parametrize("key,threads", KEYS)
def test_no_spills(ptxas_report, key, threads):  # noqa: F811
    hits = [v for k, v in ptxas_report.items() if key in k]
    assert len(hits) == 1, (key, sorted(ptxas_report))
    assert hits[0].get("spill", 0) == 0, (key, hits[0])
    assert hits[0]["regs"] * threads <= 65536, (key, hits[0])
