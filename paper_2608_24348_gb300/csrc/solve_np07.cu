// solve_np07.cu -- persistent solver kernels for order N = 6 (up to 8 problems).
#include "solver.cuh"

int sem_solve_launch_np7(const SolveParams<8> &p, int mode, int sms, cudaStream_t s)
{
    switch (mode) {
        case MODE_F64: return launch_solve<8, MODE_F64, 7>(p, sms, s);
        case MODE_F64N: return launch_solve<8, MODE_F64N, 7>(p, sms, s);
        case MODE_F32: return launch_solve<8, MODE_F32, 7>(p, sms, s);
        case MODE_TC: return launch_solve<8, MODE_TC, 7>(p, sms, s);
        default: return SEM_ERR_ARG;
    }
}

int sem_solve_tables_np7(const double *D) { return solver_upload_tables(7, D); }
