// solve_ordered_c.cu -- the ordered solver of Taylor-Green steps, N + 1 in {3, 6, 9}.
#include "solver_ordered.cuh"

int sem_solve_ordered_c(const SolveParams<8> &p, int n, int sms, cudaStream_t s)
{
    switch (n) {
        case 3: return ordered::launch<3>(p, sms, s);
        case 6: return ordered::launch<6>(p, sms, s);
        case 9: return ordered::launch<9>(p, sms, s);
        default: return SEM_ERR_ARG;
    }
}

int sem_solve_ordered_tables_c(int n, const double *D) { return solver_upload_tables(n, D); }
