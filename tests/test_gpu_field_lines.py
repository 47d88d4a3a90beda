"""The field calls at sizes either side of the lines between their kernels and
between the cluster sizes of many targets (one to eight CTAs, by the load of the
busiest SM), against the FP64 oracle."""
import pytest

from tests import test_gpu_probe_field as probe

pytestmark = pytest.mark.gpu
md = probe.md


@pytest.mark.parametrize("alloc", [True, False])
@pytest.mark.parametrize("nt,ns", [(8192, 12001), (10000, 8200), (12000, 9001), (14000, 17000),
                                   (16383, 8195), (20000, 16100), (28000, 8193), (30323, 9000),
                                   (32768, 8200)])
def test_clusters_of_many_targets(md, nt, ns, alloc):
    probe.test_field_and_potential_follow_oracle(md, nt, ns, alloc)


@pytest.mark.parametrize("nt,ns", [(100000, 520), (100000, 1300), (50000, 600), (300000, 510),
                                   (400000, 300), (130000, 500)])
def test_few_sources_at_many_targets(md, nt, ns):
    probe.test_field_and_potential_follow_oracle(md, nt, ns, True)
