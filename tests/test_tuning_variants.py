"""A stored batch variant is only used while its index means the same (phases per block, pixels per thread):
a table without the variants, or written for others, is tuned again."""
from types import SimpleNamespace

import torch

from paper_2301_04259_gb300 import _build, tuning


def test_table_of_other_variants_is_tuned_again(tmp_path, monkeypatch):
    _build.build()
    from paper_2301_04259_gb300 import soap
    calls, chosen = [], []
    variants = [soap.soap_batch_variant_info(v) for v in range(soap.soap_batch_num_variants())]
    monkeypatch.setattr(soap, "soap_get_star_info", lambda ctx: SimpleNamespace(n_taps=27))
    monkeypatch.setattr(soap, "soap_batch_autotune",
                        lambda *a, **k: calls.append(1) or (2, [1.0] * len(variants)))
    monkeypatch.setattr(soap, "soap_batch_set_variant", lambda ctx, v: chosen.append(v))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda d: "GPU X")
    star = SimpleNamespace(n_px=16834, mu_values=[0.1] * 20, grid_n=150)
    path = tmp_path / "t.json"

    def tune():
        return tuning.tune_batch(None, star, [], [], [], SimpleNamespace(device=0), path=path)["source"]
    # an index stored before the key said what the variants are
    tuning.save_table(path, {tuning.tuning_key(16834, 27, 20, 150, "GPU X"): {"variant": 5, "ms": []}})
    assert tune() == "autotune" and tune() == "cache" and len(calls) == 1
    monkeypatch.setattr(soap, "soap_batch_variant_info", lambda v: (variants[v][0], 2))
    assert tune() == "autotune" and len(calls) == 2
    assert chosen == [2, 2, 2]
