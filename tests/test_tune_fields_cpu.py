"""The autotuner's choices are ones that the workload's kernels have (no GPU)."""
import inputs
from paper_2302_00414_gb300 import tune as TU


def test_two_dimensional_searches_have_no_prefetch():
    """No d = 2 spread copies ahead; the field only keeps a batch off the persistent form."""
    assert "prefetch" not in TU.CANDIDATES_2D
    assert TU.CANDIDATES_3D["prefetch"] == [1, 2]


def test_cached_choices_are_read_without_fields_of_other_kernels(tmp_path):
    path = str(tmp_path / "tuning.json")
    d2, d3 = [(16, inputs.random_points(1000, 2, 5))], [(16, inputs.random_points(1000, 3, 5))]
    TU.save_cache({TU.signature(s, 4, "fp32", 1): {"tune": {"branches": 4, "prefetch": 2}, "default_ms": 1.0, "tuned_ms": 0.8}
                   for s in (d2, d3)}, path)
    assert TU.tuned_choice(None, None, d2, None, 4, "fp32", 1, cache_path=path)["tune"] == {"branches": 4}
    assert TU.tuned_choice(None, None, d3, None, 4, "fp32", 1, cache_path=path)["tune"] == {"branches": 4, "prefetch": 2}


def test_shipped_choices():
    for key, entry in TU.load_cache().items():
        assert set(entry["tune"]) <= set(TU.CANDIDATES_2D if key.startswith("d2") else TU.CANDIDATES_3D)
