"""The kernels bench.py names for the storage modes the library reports."""
import bench
import workloads as wl


def test_kernel_names():
    chain = wl.serial_chains(B=2, T=1, n=12).model          # FP64: too long for the four-warp rollout
    assert bench.kernel_flops(chain, ("pipelined", "aligned_pipelined_global"))[::2] == ("k_rollout_pipe", "k_wbackward_pipe")
    kf, ff, _, _ = bench.kernel_flops(chain, ("pipelined_team", "aligned_pipelined_shared"))
    assert kf == "k_wrollout_team" and ff == bench.flops_per_system_step(chain, "wfwd")
    quad = wl.quadruped(B=2, T=1).model
    assert bench.kernel_flops(quad, ("floating_global", "floating_pipelined_global"))[::2] == ("k_wrollout", "k_wbackward_pipe")
    feet = wl.quadruped(B=2, T=1, contacts=True).model
    assert bench.kernel_flops(feet, ("global", "global"))[::2] == ("k_rollout_contact", "k_backward_contact")
