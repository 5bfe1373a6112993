"""Properties of the CUDA sources themselves (no GPU)."""
from pathlib import Path

CSRC = Path(__file__).resolve().parents[1] / "paper_2503_07526_gb300" / "csrc"


def test_no_tma_multicast():
    """The one library is loaded by every rank of a run over several GPUs, where
    TMA loads with cluster multicast are not used in any form."""
    named = [p.name for p in sorted(CSRC.iterdir()) if "multicast" in p.read_text().lower()]
    assert named == []
