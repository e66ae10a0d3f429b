"""Variants of the kernels that the library chooses by sizes and types: parity with the oracle where each one's range
begins and ends."""
import pytest

from paper_2502_11417_b200 import synth
from parity import full_parity

pytestmark = pytest.mark.gpu

PACED = synth.FLAG_MIGRATION | synth.FLAG_PACING


@pytest.mark.parametrize("n", [1, 255, 257, 3000])
@pytest.mark.parametrize("buffer_tokens", [0, 1, 2, 11, 12, 200])
def test_handoff_search_by_one_thread_and_by_a_warp(n, buffer_tokens):
    # 20 tokens/s consumption against a server whose slowest token takes 42 ms: every token gains 8 ms or more, so the
    # search looks at (buffer - 1) * 50 / 8 + 1 tokens (64 is the last that one thread takes); a device generates at 40/s
    w = synth.tiny_workload(7 + n, n, max_prompt=300, max_out=500)
    w.servers = [synth.server(tbt_s=0.035, jitter=0.2)]
    w.devices = [synth.device(500.0, 40.0, jitter=0.05)]
    dear = [synth.device(500.0, 40.0, jitter=0.05, c_prefill=5e-3, c_decode=5e-3)]
    for devices in (w.devices, dear):
        w.devices = devices
        full_parity(w, [synth.policy(b, r_c=20.0, t_m_s=buffer_tokens * 0.05, mig_threshold=th, flags=PACED)
                        for b in (0.3, 1.0) for th in (0.0, 0.1)], select=False, tag=f"search {buffer_tokens}")
