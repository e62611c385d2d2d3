"""Tensor-core GEMMs run without thread-block clusters: no CTA writes into
another's shared memory (replicas run one process per GPU with this library).
The knob that chose the cluster size keeps its place and its former values."""
import pathlib

import pytest
import torch

from paper_2402_17660_gb300 import synth
from paper_2402_17660_gb300.tnet import TensorNet, tuning_knobs

CLUSTER = 7


def test_no_kernel_source_loads_into_other_ctas():
    import paper_2402_17660_gb300
    root = pathlib.Path(paper_2402_17660_gb300.__file__).parent / "csrc"
    for f in sorted(root.iterdir()):
        text = f.read_text()
        assert "multicast" not in text and "clusterDim" not in text, f.name
    assert tuning_knobs()[CLUSTER] == ("tc_cluster", [1, 2, 4])   # the default first


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs CUDA")
@pytest.mark.parametrize("precision", [1, 2])
def test_former_cluster_values_are_accepted_and_change_nothing(precision):
    from tests.gpu_helpers import DEV, gpu_energy_forces
    s = synth.random_cluster(90, seed=5)
    m = TensorNet(synth.init_weights(synth.ModelShape(), seed=0), max_atoms=90, max_pairs=90 * 89,
                  precision=precision, device=DEV)
    assert m.get_tuning()[CLUSTER] == 1
    E0, F0 = gpu_energy_forces(m, s)
    for v in (2, 4):
        knobs = m.get_tuning()
        knobs[CLUSTER] = v
        m.set_tuning(knobs)
        assert m.get_tuning()[CLUSTER] == v
        E1, F1 = gpu_energy_forces(m, s)
        assert (E1 == E0).all() and (F1 == F0).all()
    with pytest.raises(Exception):
        knobs[CLUSTER] = 3
        m.set_tuning(knobs)


def test_every_message_form_is_listed_once():
    assert tuning_knobs()[6] == ("message_kernel", [3, 1, 4])   # 3 and the former 0 are the same kernels


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs CUDA")
def test_former_message_form_is_accepted_and_runs_like_its_equal():
    from tests.gpu_helpers import DEV, gpu_energy_forces
    s = synth.random_cluster(90, seed=5)
    m = TensorNet(synth.init_weights(synth.ModelShape(), seed=0), max_atoms=90, max_pairs=90 * 89, device=DEV)
    knobs = m.get_tuning()
    assert knobs[6] == 3
    E0, F0 = gpu_energy_forces(m, s)
    m.set_tuning(knobs[:6] + [0] + knobs[7:])
    assert m.get_tuning()[6] == 0
    E1, F1 = gpu_energy_forces(m, s)
    assert (E1 == E0).all() and (F1 == F0).all()
